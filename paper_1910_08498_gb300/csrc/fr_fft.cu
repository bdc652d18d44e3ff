// fr_fft.cu -- the volume's inverse transform for S = 64 and 128 (below), and the
// images' 2D transforms for S = 64, 128, 256: a kernel over the
// rows (real to complex) and one over the columns that also centres the image and
// converts to the insertion's dtype.
//
// The general path (cuFFT rows, cuFFT columns, then a staging pass) moves the
// spectra through HBM three times; here the columns' kernel does the staging's
// work.  1100 real images of 256^2, centred, to FP16: 323 -> 203 us.  For 1016 images
// the rows take 94 us (80 us of HBM traffic; 97 with the partners of the last step
// exchanged through shared memory, whose data pipe was 88 % busy; S = 64, 1500
// images: 25 -> 23 us in all), the columns 97 us (60 us of HBM traffic; two CTAs of
// 90 KB an SM; narrower blocks, three CTAs of 68 KB, took 123).
//
// Transforms by Cooley-Tukey with two factors (N = N1 N2): a thread takes N1 points
// n2 + N2 n1, transforms them in registers (radix 4 and 2 steps), multiplies by
// W_N^(n2 k1), exchanges through shared memory and transforms N2 points for one k1;
// its outputs are k1 + N1 k2.  Twiddles come from a table of W_S per CTA (sincospif,
// correctly reduced).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "fr_internal.h"

namespace fr {
namespace {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }  // a * -i

// forward DFTs in place, outputs in natural order
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d) {
  const float2 s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = mul_mi(csub(b, d));
  a = cadd(s0, s2);
  b = cadd(s1, s3);
  c = csub(s0, s2);
  d = csub(s1, s3);
}
constexpr float kC8 = 0.70710678118654752f;                              // cos(pi / 4)
constexpr float kC16 = 0.92387953251128674f, kS16 = 0.38268343236508977f;  // cos, sin(pi / 8)

__device__ __forceinline__ void dft(float2 (&v)[8]) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4(e0, e1, e2, e3);
  dft4(o0, o1, o2, o3);
  o1 = make_float2(kC8 * (o1.x + o1.y), kC8 * (o1.y - o1.x));   // * W_8
  o2 = mul_mi(o2);
  o3 = make_float2(kC8 * (o3.y - o3.x), -kC8 * (o3.x + o3.y));  // * W_8^3
  v[0] = cadd(e0, o0), v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1), v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2), v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3), v[7] = csub(e3, o3);
}

__device__ __forceinline__ void dft(float2 (&v)[16]) {
  // 4 x 4: columns n2, twiddles W_16^(n2 k1), rows
#pragma unroll
  for (int j = 0; j < 4; ++j) dft4(v[j], v[4 + j], v[8 + j], v[12 + j]);
  const float2 w1 = make_float2(kC16, -kS16), w2 = make_float2(kC8, -kC8), w3 = make_float2(kS16, -kC16);
  v[5] = cmul(v[5], w1);
  v[6] = cmul(v[6], w2);
  v[7] = cmul(v[7], w3);
  v[9] = cmul(v[9], w2);
  v[10] = mul_mi(v[10]);
  v[11] = cmul(v[11], make_float2(-kC8, -kC8));
  v[13] = cmul(v[13], w3);
  v[14] = cmul(v[14], make_float2(-kC8, -kC8));
  v[15] = cmul(v[15], make_float2(-kC16, kS16));
  float2 o[16];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    dft4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
#pragma unroll
    for (int m = 0; m < 4; ++m) o[k + 4 * m] = v[4 * k + m];
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = o[i];
}

// W_S^i = exp(-2 pi i / S), i < S
template <int S>
__device__ __forceinline__ void fill_twiddles(float2 *tw) {
  for (int i = threadIdx.x; i < S; i += blockDim.x) {
    float s, c;
    sincospif(2.0f * (float)i / (float)S, &s, &c);
    tw[i] = make_float2(c, -s);
  }
}

// ---- rows: M = S / 2 complex points z[n] = x[2n] + i x[2n + 1], M = 16 M2 (8 M2
// for M = 32), M2 threads a row; X[k] = (Z[k] + conj Z[M - k]) / 2 - (i / 2) W_S^k
// (Z[k] - conj Z[M - k]), k = 0 .. M
template <int S>
struct RowShape {
  static constexpr int M = S / 2, N1 = M == 32 ? 8 : 16, M2 = M / N1;  // M2 threads a row: 4 or 8
  static constexpr int T = 256, ROWS = T / M2;
  // float2 per group of M2 points and per row in shared memory: a half warp's
  // rows and groups fall on different bank pairs
  static constexpr int GP = M2 + 1, PITCH = M2 == 8 ? 152 : (N1 == 16 ? 84 : 52);
  static_assert(PITCH >= N1 * GP && PITCH >= M, "row buffer");
};

template <int S>
__global__ void __launch_bounds__(RowShape<S>::T) fft_rows_kernel(const float2 *__restrict__ real,
                                                                  long long rows,
                                                                  float2 *__restrict__ out) {
  using SH = RowShape<S>;
  constexpr int M = SH::M, N1 = SH::N1, M2 = SH::M2, NX = M + 1;
  extern __shared__ __align__(16) unsigned char raw[];
  float2 *tw = reinterpret_cast<float2 *>(raw);
  float2 *buf = tw + S;
  const int t = threadIdx.x % M2, rl = threadIdx.x / M2;
  const long long row = (long long)blockIdx.x * SH::ROWS + rl;
  const bool in = row < rows;
  float2 v[N1];
  const float2 *src = real + (in ? row : 0) * M + t;
#pragma unroll
  for (int k = 0; k < N1; ++k) v[k] = __ldg(src + M2 * k);
  fill_twiddles<S>(tw);
  __syncthreads();
  float2 *b = buf + rl * SH::PITCH;
  dft(v);
#pragma unroll
  for (int k = 0; k < N1; ++k) b[k * SH::GP + t] = k ? cmul(v[k], tw[2 * t * k]) : v[0];  // W_M = W_S^2
  __syncwarp();
  // N1 transforms of M2 points, N1 / M2 a thread (M2 = 8, N1 = 16: two; M2 = 4, N1
  // = 8 or 16: two or four)
  constexpr int J = N1 / M2;
  float2 u[J][M2];
#pragma unroll
  for (int j = 0; j < J; ++j)
#pragma unroll
    for (int n = 0; n < M2; ++n) u[j][n] = b[(t + j * M2) * SH::GP + n];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    if constexpr (M2 == 8) dft(u[j]);
    else dft4(u[j][0], u[j][1], u[j][2], u[j][3]);
  }
  // Z[k], k = t + M2 j + N1 n, is u[j][n]; its partner Z[M - k] is lane (M2 - t) % M2's
  // u[J - 1 - j][M2 - 1 - n], but lane 0's partners are its own.  By shuffles: half the
  // shared-memory wavefronts of another exchange.
  const int peer = (threadIdx.x & 31 & ~(M2 - 1)) | ((M2 - t) & (M2 - 1));
  float2 *dst = out + row * NX;
#pragma unroll
  for (int j = 0; j < J; ++j)
#pragma unroll
    for (int n = 0; n < M2; ++n) {
      const float2 z = u[j][n], g = u[J - 1 - j][M2 - 1 - n];
      const float2 own = j ? u[(J - j) % J][M2 - 1 - n] : u[0][(M2 - n) % M2];
      float2 y = make_float2(__shfl_sync(0xffffffffu, g.x, peer), __shfl_sync(0xffffffffu, g.y, peer));
      if (t == 0) y = own;
      const int k = t + M2 * j + N1 * n;
      // X[k] = e - i q, e = (Z[k] + conj Z[M - k]) / 2, q = W^k (Z[k] - conj Z[M - k]) / 2
      const float2 e = make_float2(0.5f * (z.x + y.x), 0.5f * (z.y - y.y));
      const float2 q = cmul(make_float2(0.5f * (z.x - y.x), 0.5f * (z.y + y.y)), tw[k]);
      if (in) dst[k] = make_float2(e.x + q.y, e.y - q.x);
    }
  if (in && t == 0) dst[M] = make_float2(u[0][0].x - u[0][0].y, 0.f);
}

// ---- columns: S points, S = N1 N2, of CB columns a CTA; centring and conversion
template <int S>
struct ColShape {
  static constexpr int NX = S / 2 + 1;
  static constexpr int N1 = S == 64 ? 8 : 16, N2 = S / N1;  // 8 x 8, 16 x 8, 16 x 16
  static constexpr int NB = S == 256 ? 3 : 1;               // column blocks of an image
  static constexpr int CB = NX / NB;                        // 33, 65, 43 columns (odd: no bank conflicts)
  static_assert(CB * NB == NX && (CB & 1), "whole column blocks");
  static constexpr int T = 352;
};

template <int S, int F16>
__global__ void __launch_bounds__(ColShape<S>::T, 2)
fft_cols_kernel(const float2 *spec, int center, void *out) {
  using SH = ColShape<S>;
  constexpr int NX = SH::NX, N1 = SH::N1, N2 = SH::N2, CB = SH::CB, T = SH::T;
  extern __shared__ __align__(16) unsigned char raw[];
  float2 *tw = reinterpret_cast<float2 *>(raw);
  float2 *buf = tw + S;  // [S][CB]
  const int c0 = (blockIdx.x % SH::NB) * CB;
  const size_t img = (size_t)(blockIdx.x / SH::NB) * S * NX;
  const float2 *src = spec + img + c0;
  fill_twiddles<S>(tw);
  __syncthreads();
  for (int q = threadIdx.x; q < N2 * CB; q += T) {
    const int t = q / CB, c = q - t * CB;
    float2 v[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) v[k] = src[(size_t)(t + N2 * k) * NX + c];
    dft(v);
#pragma unroll
    for (int k = 0; k < N1; ++k)
      buf[(k * N2 + t) * CB + c] = k ? cmul(v[k], tw[(t * k) & (S - 1)]) : v[0];
  }
  __syncthreads();
  for (int q = threadIdx.x; q < N1 * CB; q += T) {
    const int k1 = q / CB, c = q - k1 * CB;
    float2 v[N2];
#pragma unroll
    for (int n = 0; n < N2; ++n) v[n] = buf[(k1 * N2 + n) * CB + c];
    dft(v);
#pragma unroll
    for (int k = 0; k < N2; ++k) {
      const int j = k1 + N1 * k;
      float2 w = v[k];
      // the image origin moved from pixel (0, 0) to (S/2, S/2): (-1)^(kx + j)
      if (center && ((c0 + c + j) & 1)) w = make_float2(-w.x, -w.y);
      const size_t o = img + (size_t)j * NX + c0 + c;
      if (F16) reinterpret_cast<__half2 *>(out)[o] = __floats2half2_rn(w.x, w.y);
      else reinterpret_cast<float2 *>(out)[o] = w;
    }
  }
}

// ---- the volume's inverse transform, S = 64 and 128, in two kernels: weighting and
// the z lines; then a plane a CTA, its y lines and its x lines (complex to real).
//
// A plane's CTA holds it in shared memory: 74 KB at S = 128, 4 times that at 256, which
// does not fit.  The data fit in L2, so what counts is the number of passes and the latency of
// each; the general path takes four (weighting, then cuFFT's three).  S = 128: 9.7 +
// 20.6 us in four launches -> 12.8 + 7.5 us.  The z kernel waits for the six sums' 27
// MB (4 us of HBM traffic); with 16 points a thread instead of 8, and half the warps,
// it took 14.4 us, with the loads behind a branch a point 19.9.
// The transforms are the forward ones above, applied to the conjugate of F.  Column
// kx = S / 2 is zero and left out.
template <int S>
struct VolShape {
  static constexpr int M = S / 2;                   // columns kept
  static constexpr int Z1 = 8, Z2 = S / Z1;         // z lines: Z2 threads of Z1 points
  static constexpr int CB = S == 64 ? 16 : 32;      // columns of a CTA of the z lines
  static constexpr int TZ = Z2 * CB;
  static constexpr int N1 = S == 64 ? 8 : 16, N2 = 8;  // y lines
  static constexpr int TP = N2 * M;                 // threads of a plane's CTA
  static constexpr int R1 = 8, R2 = M / R1;         // x lines: R2 threads of R1 points
  // float2 per group of R2 points and per row of a plane in shared memory: a half
  // warp's rows and groups fall on different bank pairs
  static constexpr int GP = R2 + 1, P = S == 64 ? 52 : 72;
  static_assert(N1 * N2 == S && P >= M && P >= R1 * GP, "volume lines");
};

template <int S>
__global__ void __launch_bounds__(VolShape<S>::TZ)
volume_z_kernel(const Geom g, const float *__restrict__ acc, size_t plane, float w_clip, float inv_n,
                float2 *__restrict__ spec) {
  using V = VolShape<S>;
  constexpr int M = V::M, N1 = V::Z1, N2 = V::Z2, CB = V::CB, NB = M / CB;
  __shared__ float2 tw[S], buf[S * CB];
  const int jy = blockIdx.x / NB, c0 = (blockIdx.x % NB) * CB;
  const int ky = jy < M ? jy : jy - S;
  const int t = threadIdx.x / CB, c = threadIdx.x % CB;
  const int kx = c0 + c;
  // conj(F) at (kx, ky, kz), 0 on the Nyquist planes.  All points' sums are read first,
  // without a branch, so that the reads are in flight together; those of the mirrored
  // point -v join where it is stored (the first few columns).
  float2 v[N1];
  float w[N1];
  // point k is kz = t + N2 k, less S from k = N1 / 2 on: plane kz + S / 2
  const float *p = acc + ((size_t)t * g.D + (size_t)(ky + M)) * g.NXa + (size_t)(kx - g.xa0);
  const size_t dz = (size_t)N2 * g.D * g.NXa;
#pragma unroll
  for (int k = 0; k < N1; ++k) {
    const float *q = p + (size_t)((k + N1 / 2) % N1) * dz;
    v[k] = make_float2(q[0] + q[3 * plane], q[plane] + q[4 * plane]);
    w[k] = q[2 * plane] + q[5 * plane];
  }
  if (-kx >= g.xa0) {
    const float *pm = acc + ((size_t)(S - t) * g.D + (size_t)(M - ky)) * g.NXa + (size_t)(-kx - g.xa0);
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      const float *q = pm - (size_t)((k + N1 / 2) % N1) * dz;
      v[k].x += q[0] + q[3 * plane];
      v[k].y -= q[plane] + q[4 * plane];
      w[k] += q[2 * plane] + q[5 * plane];
    }
  }
#pragma unroll
  for (int k = 0; k < N1; ++k) {
    const float s = inv_n / fmaxf(w[k], w_clip);
    const bool nyquist = jy == M || (k == N1 / 2 && t == 0);
    v[k] = nyquist ? make_float2(0.f, 0.f) : make_float2(v[k].x * s, -(v[k].y * s));
  }
  fill_twiddles<S>(tw);
  __syncthreads();
  dft(v);
#pragma unroll
  for (int k = 0; k < N1; ++k) buf[(k * N2 + t) * CB + c] = k ? cmul(v[k], tw[(t * k) & (S - 1)]) : v[0];
  __syncthreads();
  if (t < N1) {
    float2 u[N2];
#pragma unroll
    for (int n = 0; n < N2; ++n) u[n] = buf[(t * N2 + n) * CB + c];
    dft(u);
#pragma unroll
    for (int k = 0; k < N2; ++k) spec[((size_t)(t + N1 * k) * S + jy) * M + c0 + c] = u[k];
  }
}

template <int S>
__global__ void __launch_bounds__(VolShape<S>::TP)
volume_plane_kernel(const float2 *__restrict__ spec, float2 *__restrict__ out) {
  using V = VolShape<S>;
  constexpr int M = V::M, N1 = V::N1, N2 = V::N2, R1 = V::R1, R2 = V::R2, GP = V::GP, P = V::P;
  extern __shared__ __align__(16) unsigned char raw[];
  float2 *tw = reinterpret_cast<float2 *>(raw);
  float2 *buf = tw + S;  // [S][P]
  spec += (size_t)blockIdx.x * S * M;
  out += (size_t)blockIdx.x * S * M;
  {
    const int t = threadIdx.x / M, c = threadIdx.x % M;
    float2 v[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) v[k] = spec[(t + N2 * k) * M + c];
    fill_twiddles<S>(tw);
    __syncthreads();
    dft(v);
#pragma unroll
    for (int k = 0; k < N1; ++k) buf[(k * N2 + t) * P + c] = k ? cmul(v[k], tw[(t * k) & (S - 1)]) : v[0];
    __syncthreads();
    float2 u[N1 / N2][N2];
#pragma unroll
    for (int i = 0; i < N1 / N2; ++i)
#pragma unroll
      for (int n = 0; n < N2; ++n) u[i][n] = buf[((t + N2 * i) * N2 + n) * P + c];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N1 / N2; ++i) {
      dft(u[i]);
#pragma unroll
      for (int k = 0; k < N2; ++k) buf[(t + N2 * i + N1 * k) * P + c] = u[i][k];
    }
    __syncthreads();
  }
  // x lines: with Y the row and W = W_S, x[2n] + i x[2n + 1] is the transform over M
  // points of E + i O, E[k] = Y[k] + conj Y[M - k], O[k] = (Y[k] - conj Y[M - k]) W^k;
  // Y[M] = 0, and Y[0] counts by its real part
  const int t = threadIdx.x % R2;
  for (int row = threadIdx.x / R2; row < S; row += V::TP / R2) {
    float2 *b = buf + row * P;
    float2 v[R1];
#pragma unroll
    for (int n = 0; n < R1; ++n) {
      const int k = t + R2 * n;
      float2 y = b[k], z = make_float2(0.f, 0.f);
      if (k) z = b[M - k];
      else y.y = 0.f;
      const float2 o = cmul(make_float2(y.x - z.x, y.y + z.y), tw[k]);
      v[n] = make_float2(y.x + z.x - o.y, y.y - z.y + o.x);
    }
    __syncwarp();
    dft(v);
#pragma unroll
    for (int k = 0; k < R1; ++k) b[k * GP + t] = k ? cmul(v[k], tw[2 * t * k]) : v[0];  // W_M = W_S^2
    __syncwarp();
#pragma unroll
    for (int j = 0; j < R1 / R2; ++j) {
      float2 u[R2];
#pragma unroll
      for (int n = 0; n < R2; ++n) u[n] = b[(t + j * R2) * GP + n];
      if constexpr (R2 == 8) dft(u);
      else dft4(u[0], u[1], u[2], u[3]);
#pragma unroll
      for (int n = 0; n < R2; ++n) out[row * M + t + j * R2 + R1 * n] = u[n];
    }
  }
}

template <int S>
cudaError_t run_volume(const Geom &g, const float *acc, size_t plane, float w_clip, float2 *spec,
                       float *out, cudaStream_t st) {
  using V = VolShape<S>;
  // the plane kernel stores pairs of floats (cuFFT refuses such an output too)
  if (reinterpret_cast<uintptr_t>(out) % sizeof(float2)) return cudaErrorInvalidValue;
  const size_t smem = (size_t)(S + S * V::P) * sizeof(float2);
  auto pk = volume_plane_kernel<S>;
  cudaError_t e = allow_dynamic_smem((const void *)pk, smem);
  if (e != cudaSuccess) return e;
  const float inv_n = 1.0f / ((float)S * (float)S * (float)S);
  volume_z_kernel<S><<<S * (V::M / V::CB), V::TZ, 0, st>>>(g, acc, plane, w_clip, inv_n, spec);
  pk<<<S, V::TP, smem, st>>>(spec, reinterpret_cast<float2 *>(out));
  return cudaGetLastError();
}

template <int S>
cudaError_t run(const float *real, float2 *spec, int m, int center, void *out, int f16,
                cudaStream_t st) {
  using R = RowShape<S>;
  using C = ColShape<S>;
  const size_t rs = (size_t)(S + R::ROWS * R::PITCH) * sizeof(float2);
  const size_t csm = (size_t)(S + S * C::CB) * sizeof(float2);
  const long long rows = (long long)m * S;
  auto rk = fft_rows_kernel<S>;
  auto ck = f16 ? fft_cols_kernel<S, 1> : fft_cols_kernel<S, 0>;
  cudaError_t e = allow_dynamic_smem((const void *)rk, rs);
  if (e == cudaSuccess) e = allow_dynamic_smem((const void *)ck, csm);
  if (e != cudaSuccess) return e;
  rk<<<(unsigned)((rows + R::ROWS - 1) / R::ROWS), R::T, rs, st>>>(
      reinterpret_cast<const float2 *>(real), rows, spec);
  ck<<<(unsigned)m * C::NB, C::T, csm, st>>>(spec, center, out);
  return cudaGetLastError();
}

}  // namespace

bool fft_volume_here(int S) { return S == 64 || S == 128; }

cudaError_t fft_volume(const Geom &g, const float *acc, size_t plane, float w_clip, float2 *spec,
                       float *out, cudaStream_t st) {
  return g.S == 64 ? run_volume<64>(g, acc, plane, w_clip, spec, out, st)
                   : run_volume<128>(g, acc, plane, w_clip, spec, out, st);
}

bool fft_images_here(int S) { return S == 64 || S == 128 || S == 256; }

cudaError_t fft_images(int S, const float *real, float2 *spec, int m, int center, void *out,
                       int f16, cudaStream_t st) {
  switch (S) {
    case 64: return run<64>(real, spec, m, center, out, f16, st);
    case 128: return run<128>(real, spec, m, center, out, f16, st);
    case 256: return run<256>(real, spec, m, center, out, f16, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fr
