// fr_gather2.cuh -- the direct-drain gather insertion kernel.
//
// A warp owns a footprint of 8 x 8 x 8 voxels (4 x 8 x 8 in the fold columns),
// culls the images of its work unit into a list, and accumulates (image, voxel)
// items into shared-memory partial sums that are folded into HBM with TwoSum;
// warps never wait for one another.  Per list entry (an image, in one of the two
// orientations of its half plane):
//
//  * patch: the pixels that the footprint's voxels can meet, a rectangle of at
//    most PW x PW stored pixels, are copied into one of the warp's two
//    shared-memory patches while the previous entry is evaluated (cp.async;
//    FP16 pixels go through registers and are converted on the way).  A row of
//    20 eight-byte pixels puts pixel (x, y) in bank pair x + 4 y modulo 16, so
//    that any 4 x 4 block of pixels is free of bank conflicts;
//  * item generation: a lane computes the run of z levels of each of its
//    columns that lie within a of the plane (u_z is linear in z) and writes one
//    8-bit tag per item (column, z level) at positions from a warp scan;
//  * evaluation: 32 items a round, one per lane: u = R^T v from the footprint
//    centre's compensated projection, the 4 x 4 candidate box at rint(u - 1.5)
//    (it covers [u - a, u + a] for every a < 2; for 2 <= a <= 2.5 the 5 x 5 box
//    at rint(u - 2), for a < 3 the 6 x 6 box at rint(u - 2.5)), clamped into the
//    patch (rows and columns moved in by the clamp lie outside the blob and are
//    masked), its pixels from the patch, the Chebyshev weight polynomial in
//    x = 2 r^2 / a^2 - 1 for two candidates at a time with packed FP32x2 FMAs
//    (masked to 0 outside r <= a), and the complex and weight sums added to the
//    voxel's partial sums with plain loads and stores: the items of one entry
//    are distinct voxels.
//
// What bounds it.  Reading the boxes straight from global memory through L1 cost
// 128 data-pipe wavefronts a round (32 boxes lie in about nine image rows) and
// kept that pipe 90 % busy at 63 % issue: 13.4 ms for 5000 FP32 images of 256^2.
// From the patches a round costs about 50, and one 512-voxel footprint a warp
// (137 items an entry) halves the work per entry against 256 voxels; with an
// entry's last half round on two lanes an item and 14 candidates a box: 8.4 ms; with
// the phase counters in a kernel of their own: 8.2 ms; with the split units' sums in
// slabs (exact and repeatable; see g2_flush_slab) and 32 units an SM: 8.4 ms.
// Now the instructions bound it: 71 % issue, of which a quarter are packed FMAs
// that hold the FMA pipe for two cycles (58 % busy); shared memory 59 %.  About a
// quarter of the time is per-entry work (copies 0.6 ms, tags 0.2, records 0.2).
//
// Half planes.  A stored pixel k sits at R k or, point-reflected and
// conjugated, at -R k.  An image whose patch lies in k_x > 0 (or its mirror)
// makes one list entry: as stored, or with the in-plane axes negated (u -> -u)
// and the sums conjugated.  One whose patch crosses k_x = 0 makes both, and
// each item is evaluated once per half it reaches.  Away from the fold columns
// every point of the extended plane within a of the voxel has (R c)_x > 0, so
// a column c_x > 0 receives the stored pixel c, a column c_x < 0 the stored -c
// conjugated, and the column c_x = 0 both (0, c_y) and, conjugated, (0, -c_y):
// exactly what the two entries read.  The main bricks tile x >= floor(a) + 1.
// The fold columns |x| <= floor(a), where the fold predicate itself has to be
// evaluated per pixel, have units of their own (FOLD), in footprints 4 (8) columns
// wide so that three of four (five of eight) lanes hold fold columns: there a stored
// pixel k counts in the entry as stored when it is not folded and in the reflected
// entry when it is (exact sign of R00 k_x + R01 k_y, found once per pixel of the patch
// and kept as one bit).  Polynomial weights only.
//
// The blob's edge r <= a is decided in FP32, but for the fold columns of a >= 2
// (g2_ties): a candidate within rounding of it may fall on the wrong side and costs
// b(a) = 1 / I0(alpha), 2.9e-6 at alpha = 15.
#pragma once

#include "fr_gather.cuh"

namespace fr {

constexpr int G2_ENTRIES = 16;  // records built and processed at a time
constexpr int G2_REC = 16;      // floats of a record

// Geometry of the warp footprint FW x 8 x 8 and of its pixel patches, for
// KB x KB candidate boxes (KB = 4: a < 2, 5: a <= 2.5, 6: a < 3).
template <int FW, int KB>
struct G2Shape {
  static constexpr int FH = 8, ZC = 8;
  static constexpr int NC = FW * FH / 32;               // columns per lane
  static constexpr int WV = FW * FH * ZC;               // voxels
  static constexpr float HX = 0.5f * (FW - 1), HY = 0.5f * (FH - 1), HZ = 0.5f * (ZC - 1);
  // a box reaches KB / 2 pixels past u, and u lies within the footprint's
  // radius (6.07; 5.17 for FW = 4) of the centre: at most 17 (KB = 5: 18, KB = 6:
  // 19; FW = 4: 15) columns
  static constexpr int PW = (FW == 8 ? 13 : 11) + KB;   // patch columns and rows
  static constexpr int XC = PW > 16 ? PW - 16 : 0;      // columns past the first 16
  static constexpr int PITCH = 20;                      // = 4 modulo 16 eight-byte banks
  static constexpr int PATCH = PW * PITCH;              // pixels of a patch
  static_assert(PW <= PITCH && XC <= 3, "patch rows");
};

// Per-warp shared memory: records, partial sums, patches, image list, fold
// bits, tags.
template <int FW, int KB, int FOLD>
__host__ __device__ constexpr size_t gather2_warp_smem(int chunk) {
  using SH = G2Shape<FW, KB>;
  return ((size_t)G2_REC * G2_ENTRIES * 4 + (size_t)3 * SH::WV * 4 + (size_t)2 * SH::PATCH * 8 +
          (size_t)chunk * 4 + (FOLD ? (size_t)2 * SH::PITCH * 4 : 0) + (size_t)(SH::WV + 32) + 15) &
         ~(size_t)15;
}

__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// x . x - 1 for a nearly unit vector, to a few ulp of the difference
__device__ __forceinline__ float dot3_less_one(float x, float y, float z) {
  float hi, lo;
  dot3_dd(x, y, z, x, y, z, hi, lo);
  return (hi - 1.0f) + lo;
}

// Candidates of a fold column's box within rounding of the blob edge (FP32 r^2
// within 1e-5 a^2 of a^2), decided as the real numbers do: with a lattice
// distance a (a = 2, or a signed permutation for the rotation) the DC pixel
// and others sit there for every image.  k0: the box's first stored pixel.  x by g2_box's
// operations: a candidate that rounding put into the band there and out of it here was
// lost (a = 2.00001, signed permutations: two voxels of each image, b(a) each).
template <int PITCH, int KB>
__device__ __noinline__ void g2_ties(const float2 *cp, const float2 *p, float dx, float dy,
                                     float uz2, float cs, float sq, const unsigned *rows, int shift,
                                     const float4 e1, const float4 e2, int3 v, int2 k0, float a,
                                     float &ar, float &ai, float &aw) {
  const float U = fmaf(cs, uz2, -1.0f);
  for (int r = 0; r < KB; ++r)
    for (int j = 0; j < KB; ++j) {
      const float d = sq * (dx - (float)j), ey = dy - (float)r;
      const float x = fmaf(d, d, fmaf(cs * ey, ey, U));
      if (fabsf(x - 1.0f) > 2e-5f || !((rows[r] >> (shift + j)) & 1u) ||
          !exact_r2_le_a2(v.x, v.y, v.z, e1.x, e1.y, e1.z, e2.x, e2.y, e2.z, k0.x + j, k0.y + r, a))
        continue;
      float w = cp[POLY_N - 1].x;
      for (int k = POLY_N - 2; k >= 0; --k) w = fmaf(w, fminf(x, 1.0f), cp[k].x);
      const float2 q = p[r * PITCH + j];
      ar = fmaf(w, q.x, ar);
      ai = fmaf(w, q.y, ai);
      aw += w;
    }
}

// The KB x KB box of an item: pixels p[l * PITCH + j], u at (dx, dy) from pixel
// (0, 0), u_z^2 = uz2; returns the sums of w p (complex) and of w over the
// candidates with r <= a.  FOLD: candidate (j, l) counts only if bit j of
// rows[l] >> shift is set; with KB > 4 (a >= 2) candidates within rounding of
// the blob edge are left out, and whether there are any is returned (g2_ties).
// ROWS < KB: only the box's first ROWS rows.
template <int PITCH, int KB, int FOLD, int ROWS = KB>
__device__ __forceinline__ bool g2_box(const float2 *cp, const float2 *p, float dx, float dy,
                                       float uz2, float cs, float sq, float &ar, float &ai,
                                       float &aw, const unsigned *rows, int shift) {
  constexpr int NP = POLY_N, RP = KB == 4 ? ROWS : 3, NX = (RP * KB + 1) / 2;
  // cp: coefficient pairs (c_k, c_k), kernel-parameter constants
  // scaled column offsets sq (dx - j): x = (sq dx)^2 + cs (dy^2 + u_z^2) - 1
  float d[KB];
#pragma unroll
  for (int j = 0; j < KB; ++j) d[j] = sq * (dx - (float)j);
  const float U = fmaf(cs, uz2, -1.0f);
  ar = 0.f;
  ai = 0.f;
  aw = 0.f;
  bool ties = false;
#pragma unroll
  for (int r0 = 0; r0 < ROWS; r0 += RP) {
    // all polynomials of RP rows advance together: eight or nine independent
    // chains of packed FMAs (row by row the FMA pipe waits for their latency).
    // With a constant as its third operand a packed FMA runs at the full rate
    // (74 TFLOP/s measured; with three register pairs 44), so only the
    // polynomial is packed.  Unpacked it took 9.5 ms instead of 8.7 (S = 256, n =
    // 5000): 32 % more instructions at 83 % issue.
    // Candidate (r, j) of the rows is half i % 2 of pair i / 2, i = r KB + j.  The fold
    // columns' 5 x 5 box (2 <= a <= 2.5) takes 8 + 5 pairs, the 6 x 6 box 9 + 9: an insert
    // of 777 images, S = 96, a = 2.5, 588 -> 546 us.
    const int nc = (ROWS - r0 < RP ? ROWS - r0 : RP) * KB;  // a constant, unrolled
    float2 x[NX], h[NX];
#pragma unroll
    for (int i = 0; i < 2 * NX; ++i) {
      const float ey = dy - (float)(r0 + i / KB), dj = d[i % KB];
      const float xv = i < nc ? fmaf(dj, dj, fmaf(cs * ey, ey, U)) : 0.f;
      if (i & 1) x[i / 2].y = xv;
      else x[i / 2].x = xv;
    }
#pragma unroll
    for (int i = 0; i < NX; ++i)
      if (2 * i < nc) h[i] = __ffma2_rn(cp[NP - 1], x[i], cp[NP - 2]);
#pragma unroll
    for (int k = NP - 3; k >= 0; --k)
#pragma unroll
      for (int i = 0; i < NX; ++i)
        if (2 * i < nc) h[i] = __ffma2_rn(h[i], x[i], cp[k]);
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      if (r * KB >= nc) continue;
      const unsigned m = FOLD ? rows[r0 + r] >> shift : 0u;
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        const int i = r * KB + j;
        const float2 xx = x[i / 2], hh = h[i / 2];
        const float xv = i & 1 ? xx.y : xx.x, w = i & 1 ? hh.y : hh.x;
        const float2 q = p[(r0 + r) * PITCH + j];
        bool in = xv <= 1.0f;
        if (FOLD) in = in && ((m >> j) & 1u);
        if (FOLD && KB > 4) {
          const bool tie = fabsf(xv - 1.0f) <= 2e-5f;
          ties = ties || tie;
          in = in && !tie;
        }
        // predicated accumulation: no select, and no pixel outside the blob is used
        if (in) {
          ar = fmaf(w, q.x, ar);
          ai = fmaf(w, q.y, ai);
          aw += w;
        }
      }
    }
  }
  return ties;
}

// The 4 x 4 box of an item outside the fold columns, in 14 candidates: of the four
// corner pixels at most two, neighbours, lie within a < 2 of u.  (Opposite ones: the
// squared distances add up to dx^2 + (3 - dx)^2 + dy^2 + (3 - dy)^2 >= 9 > 2 a^2.)
// They are on the side of the box that u is nearest to: with e = |dx - 1.5| >= |dy -
// 1.5| a corner of the far column is at least (1.5 + e)^2 + (1.5 - e)^2 >= 4.5 away.
template <int PITCH>
__device__ __forceinline__ void g2_box14(const float2 *cp, const float2 *p, float dx, float dy,
                                         float uz2, float cs, float sq, float &ar, float &ai,
                                         float &aw) {
  constexpr int NP = POLY_N;
  float d[4], Y[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = sq * (dx - (float)k);
  const float U = fmaf(cs, uz2, -1.0f);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float ey = dy - (float)k;
    Y[k] = fmaf(cs * ey, ey, U);
  }
  // the two corners: distance m from u's near side, nn and nn - 3 along it
  const float gx = fabsf(dx - 1.5f), gy = fabsf(dy - 1.5f);
  const bool side = gx > gy;  // a column's two corners, else a row's
  const float m = 1.5f - fmaxf(gx, gy), V = fmaf(cs * m, m, U);
  const float nn = side ? dy : dx, n0 = sq * nn, n1 = sq * (nn - 3.0f);
  const int ca = side ? (dx < 1.5f ? 0 : 3) : (dy < 1.5f ? 0 : 3 * PITCH);
  const float2 *pa = p + ca, *pb = pa + (side ? 3 * PITCH : 3);
  float2 x[7], h[7];
  x[0] = make_float2(fmaf(d[1], d[1], Y[0]), fmaf(d[2], d[2], Y[0]));
#pragma unroll
  for (int r = 1; r < 3; ++r) {
    x[2 * r - 1] = make_float2(fmaf(d[0], d[0], Y[r]), fmaf(d[1], d[1], Y[r]));
    x[2 * r] = make_float2(fmaf(d[2], d[2], Y[r]), fmaf(d[3], d[3], Y[r]));
  }
  x[5] = make_float2(fmaf(d[1], d[1], Y[3]), fmaf(d[2], d[2], Y[3]));
  x[6] = make_float2(fmaf(n0, n0, V), fmaf(n1, n1, V));
#pragma unroll
  for (int i = 0; i < 7; ++i) h[i] = __ffma2_rn(cp[NP - 1], x[i], cp[NP - 2]);
#pragma unroll
  for (int k = NP - 3; k >= 0; --k)
#pragma unroll
    for (int i = 0; i < 7; ++i) h[i] = __ffma2_rn(h[i], x[i], cp[k]);
  ar = 0.f;
  ai = 0.f;
  aw = 0.f;
  auto add = [&](float xv, float w, const float2 q) {
    if (xv <= 1.0f) {
      ar = fmaf(w, q.x, ar);
      ai = fmaf(w, q.y, ai);
      aw += w;
    }
  };
  add(x[0].x, h[0].x, p[1]);
  add(x[0].y, h[0].y, p[2]);
#pragma unroll
  for (int r = 1; r < 3; ++r) {
    const float2 *q = p + r * PITCH;
    add(x[2 * r - 1].x, h[2 * r - 1].x, q[0]);
    add(x[2 * r - 1].y, h[2 * r - 1].y, q[1]);
    add(x[2 * r].x, h[2 * r].x, q[2]);
    add(x[2 * r].y, h[2 * r].y, q[3]);
  }
  add(x[5].x, h[5].x, p[3 * PITCH + 1]);
  add(x[5].y, h[5].y, p[3 * PITCH + 2]);
  add(x[6].x, h[6].x, *pa);
  add(x[6].y, h[6].y, *pb);
}

// The 5 x 5 box of an item outside the fold columns (2 <= a <= 2.5), in 23
// candidates: of the corners only the two on the near side (see g2_box14: opposite
// corners' squared distances add up to at least 16 > 2 a^2, a far corner is at least
// 8 away).  Its origin rint(u - 2) leaves out at most a pixel at distance exactly
// 2.5 along an axis, for u = (k + 1/2, m) in the image's plane: no voxel is seen there,
// as |u|^2 would be an integer and 1/4, and |u| = |v| for a rotation.
template <int PITCH>
__device__ __forceinline__ void g2_box23(const float2 *cp, const float2 *p, float dx, float dy,
                                         float uz2, float cs, float sq, float &ar, float &ai,
                                         float &aw) {
  constexpr int NP = POLY_N;
  float d[5], Y[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) d[k] = sq * (dx - (float)k);
  const float U = fmaf(cs, uz2, -1.0f);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float ey = dy - (float)k;
    Y[k] = fmaf(cs * ey, ey, U);
  }
  // the two corners: distance m from u's near side, nn and nn - 4 along it
  const float gx = fabsf(dx - 2.0f), gy = fabsf(dy - 2.0f);
  const bool side = gx > gy;  // a column's two corners, else a row's
  const float m = 2.0f - fmaxf(gx, gy), V = fmaf(cs * m, m, U);
  const float nn = side ? dy : dx, n0 = sq * nn, n1 = sq * (nn - 4.0f);
  const int ca = side ? (dx < 2.0f ? 0 : 4) : (dy < 2.0f ? 0 : 4 * PITCH);
  const float2 *pa = p + ca, *pb = pa + (side ? 4 * PITCH : 4);
  ar = 0.f;
  ai = 0.f;
  aw = 0.f;
  auto add = [&](float xv, float w, const float2 q) {
    if (xv <= 1.0f) {
      ar = fmaf(w, q.x, ar);
      ai = fmaf(w, q.y, ai);
      aw += w;
    }
  };
  auto at = [&](int r, int c) { return fmaf(d[c], d[c], Y[r]); };
  // two passes of six packed polynomials (the last one's second half repeats)
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    float2 x[6], h[6];
    if (pass == 0) {
      x[0] = make_float2(at(0, 1), at(0, 2));
      x[1] = make_float2(at(0, 3), at(1, 0));
      x[2] = make_float2(at(1, 1), at(1, 2));
      x[3] = make_float2(at(1, 3), at(1, 4));
      x[4] = make_float2(at(2, 0), at(2, 1));
      x[5] = make_float2(at(2, 2), at(2, 3));
    } else {
      x[0] = make_float2(at(2, 4), at(3, 0));
      x[1] = make_float2(at(3, 1), at(3, 2));
      x[2] = make_float2(at(3, 3), at(3, 4));
      x[3] = make_float2(at(4, 1), at(4, 2));
      x[4] = make_float2(at(4, 3), fmaf(n0, n0, V));
      x[5] = make_float2(fmaf(n1, n1, V), 2.0f);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) h[i] = __ffma2_rn(cp[NP - 1], x[i], cp[NP - 2]);
#pragma unroll
    for (int k = NP - 3; k >= 0; --k)
#pragma unroll
      for (int i = 0; i < 6; ++i) h[i] = __ffma2_rn(h[i], x[i], cp[k]);
    const float2 *r0 = p, *r1 = p + PITCH, *r2 = p + 2 * PITCH, *r3 = p + 3 * PITCH, *r4 = p + 4 * PITCH;
    if (pass == 0) {
      add(x[0].x, h[0].x, r0[1]), add(x[0].y, h[0].y, r0[2]);
      add(x[1].x, h[1].x, r0[3]), add(x[1].y, h[1].y, r1[0]);
      add(x[2].x, h[2].x, r1[1]), add(x[2].y, h[2].y, r1[2]);
      add(x[3].x, h[3].x, r1[3]), add(x[3].y, h[3].y, r1[4]);
      add(x[4].x, h[4].x, r2[0]), add(x[4].y, h[4].y, r2[1]);
      add(x[5].x, h[5].x, r2[2]), add(x[5].y, h[5].y, r2[3]);
    } else {
      add(x[0].x, h[0].x, r2[4]), add(x[0].y, h[0].y, r3[0]);
      add(x[1].x, h[1].x, r3[1]), add(x[1].y, h[1].y, r3[2]);
      add(x[2].x, h[2].x, r3[3]), add(x[2].y, h[2].y, r3[4]);
      add(x[3].x, h[3].x, r4[1]), add(x[3].y, h[3].y, r4[2]);
      add(x[4].x, h[4].x, r4[3]), add(x[4].y, h[4].y, *pa);
      add(x[5].x, h[5].x, *pb);
    }
  }
}

// Clear a warp's partial sums (16-byte aligned).
template <int WV>
__device__ __forceinline__ void g2_clear(float *s_acc, int lane) {
#pragma unroll 4
  for (int i = lane; i < 3 * WV / 4; i += 32)
    reinterpret_cast<float4 *>(s_acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Put a warp's partial sums (s_acc: [3][WV], slot (y FW + x) 8 + z) into its slab, the
// folds-th time: FP32 sums first, an FP32 pair by TwoSum when there are more.  The
// merge after the launch adds the slabs of a brick's units to the accumulators in the
// units' order, so the result rounds nothing away and is the same bits in every run.
// (The units' FP32 sums added with atomics instead: 100 equal images left W 9e-7 off,
// and most bricks are split.  Atomics into an FP64 scratch cost 11 % at S = 128.)
template <int WV>
__device__ __noinline__ void g2_flush_slab(const float *s_acc, float *slab, int folds) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const float4 *src = reinterpret_cast<const float4 *>(s_acc);
  float4 *hi = reinterpret_cast<float4 *>(slab), *lo = hi + 3 * WV / 4;
#pragma unroll 4
  for (int i = lane; i < 3 * WV / 4; i += 32) {
    float4 s = src[i];
    if (folds > 0) {  // a slab of six planes (see slab_once)
      float4 h = hi[i], l = folds > 1 ? lo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      dd_add(h.x, l.x, s.x);
      dd_add(h.y, l.y, s.y);
      dd_add(h.z, l.z, s.z);
      dd_add(h.w, l.w, s.w);
      lo[i] = l;
      s = h;
    }
    hi[i] = s;
  }
  __syncwarp();
}

// Fold a warp's partial sums into HBM: straight into the double-float accumulators
// (error-free TwoSum) when the warp is the only writer of its voxels, else, where there
// are no slabs, into the float4 scratch with atomics (merged after the launch).  The
// loads of four z levels are issued together: one after the other, their latency made a
// flush take four times as long.
template <int FW, int KB>
__device__ __noinline__ void g2_flush(const InsertArgs &args, const float *s_acc, int fx0, int fy0,
                                      int z0, bool to_scratch) {
  using SH = G2Shape<FW, KB>;
  constexpr int WV = SH::WV, ZC = SH::ZC, ZG = 4;
  const Geom &g = args.g;
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll 1
  for (int k = 0; k < SH::NC * ZC / ZG; ++k) {
    const int col = (k / (ZC / ZG)) * 32 + lane, t0 = k % (ZC / ZG) * ZG;
    const int vx = fx0 + col % FW, vy = fy0 + col / FW;
    if (vx > g.H || vy > g.H) continue;
    float s[3][ZG];  // four z levels of the three sums, as 16-byte groups
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float4 q = *reinterpret_cast<const float4 *>(s_acc + c * WV + col * ZC + t0);
      s[c][0] = q.x, s[c][1] = q.y, s[c][2] = q.z, s[c][3] = q.w;
    }
    const size_t slice = (size_t)g.D * g.NXa;
    const size_t v0 = ((size_t)(z0 + t0 + g.H) * g.D + (size_t)(vy + g.H)) * g.NXa + (size_t)(vx - g.xa0);
    if (to_scratch) {
      float4 *q = args.scratch + v0;
#pragma unroll
      for (int t = 0; t < ZG; ++t, q += slice)
        if (z0 + t0 + t <= g.H && (s[0][t] != 0.f || s[1][t] != 0.f || s[2][t] != 0.f))
          atomicAdd(q, make_float4(s[0][t], s[1][t], s[2][t], 0.f));
    } else {
      float h[3 * ZG], l[3 * ZG];
#pragma unroll
      for (int t = 0; t < ZG; ++t)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const bool in = z0 + t0 + t <= g.H;
          const float *q = args.acc + c * args.plane + v0 + t * slice;
          h[3 * t + c] = in ? q[0] : 0.f;
          l[3 * t + c] = in ? q[3 * args.plane] : 0.f;
        }
#pragma unroll
      for (int t = 0; t < ZG; ++t) {
        if (z0 + t0 + t > g.H || (s[0][t] == 0.f && s[1][t] == 0.f && s[2][t] == 0.f)) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float *q = args.acc + c * args.plane + v0 + t * slice;
          dd_add(h[3 * t + c], l[3 * t + c], s[c][t]);
          q[0] = h[3 * t + c];
          q[3 * args.plane] = l[3 * t + c];
        }
      }
    }
  }
  __syncwarp();
}

// The warp footprints of a BX x BY x BZ brick, FW x 8 x 8 voxels each.
template <int BX, int BY, int BZ, int FW>
__host__ __device__ constexpr int g2_warps() {
  return (BX / FW) * (BY / 8) * (BZ / 8);
}

// One warp's share of one work unit (see gather_warp for the unit word).
// args: the batch's arguments; cst: the arguments its launch shares (geometry,
// weight polynomial, list capacity) and images the batch's images, both read
// in the inner loops; block: the unit's slab, if it is split.  FOLD = 0: the bricks
// tile x >= floor(a) + 1; FOLD = 1: they tile x >= -floor(a) and only the fold
// columns |x| <= floor(a) are computed, with the fold predicate tested per candidate.
template <int BX, int BY, int BZ, int F16, int KB = 4, int FW = 8, int FOLD = 0, int PROF = 0>
__device__ __forceinline__ void gather2_warp(const InsertArgs &args, const InsertArgs &cst,
                                             const void *images, unsigned char *wsmem,
                                             const int4 unit, const int block, const int warp) {
  using SH = G2Shape<FW, KB>;
  constexpr int FH = SH::FH, ZC = SH::ZC, WV = SH::WV, PW = SH::PW, PITCH = SH::PITCH,
                NC = SH::NC, XC = SH::XC;
  static_assert((FW == 8 || FW == 4) && BX % FW == 0 && BY % FH == 0 && BZ % ZC == 0,
                "warp footprints are 8 x 8 x 8 or 4 x 8 x 8 voxels");
  constexpr float HB = 0.5f * KB;  // a box reaches HB pixels past u
  constexpr int ESZ = F16 ? 4 : 8;
  constexpr float HX = SH::HX, HY = SH::HY, HZ = SH::HZ;
  constexpr unsigned FULL = 0xffffffffu;
  const Geom &g = cst.g;
  int lane;  // read once: the special register is slow
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  const int wx = warp % (BX / FW), wy = warp / (BX / FW) % (BY / FH), wz = warp / (BX / FW * (BY / FH));
  const int fx0 = (FOLD ? g.xa0 : 1 - g.xa0) + unit.x * BX + wx * FW;
  const int fy0 = -g.H + unit.y * BY + wy * FH;
  const int z0 = -g.H + unit.z * BZ + wz * ZC;
  const int lcap = cst.chunk;
  if (lcap < 32 || lcap > 128) {  // the image list holds lcap entries
    if (lane == 0) set_err(args.err, DERR_RANGE);
    return;
  }
  if (fx0 > g.H || fy0 > g.H || z0 > g.H) return;  // no voxel of the volume
  float4 *s_rec = reinterpret_cast<float4 *>(__builtin_assume_aligned(wsmem, 16));  // [G2_ENTRIES][4]
  float *s_acc = reinterpret_cast<float *>(s_rec + G2_REC / 4 * G2_ENTRIES);        // [3][WV]
  float2 *s_patch = reinterpret_cast<float2 *>(s_acc + 3 * WV);                     // [2][PATCH]
  int *s_idx = reinterpret_cast<int *>(s_patch + 2 * SH::PATCH);                    // [lcap]
  unsigned *s_bits = reinterpret_cast<unsigned *>(s_idx + lcap);                    // FOLD: [2][PITCH]
  unsigned char *s_tag = reinterpret_cast<unsigned char *>(s_bits + (FOLD ? 2 * PITCH : 0));  // [WV + 32]

  const int split = unit.w & 0xffff, nsplit = (unit.w >> 16) & 0x3fff;
  const bool to_scratch = nsplit > 1 || ((unit.w >> 30) & 1);
  const int img0 = (int)((long long)args.n * split / nsplit);
  const int img1 = (int)((long long)args.n * (split + 1) / nsplit);
  const float cx = fx0 + HX, cy = fy0 + HY, cz = z0 + HZ;  // footprint centre
  const float a_plane = g.a + 1e-4f;  // conservative |u_z| <= a test
  const float cs = 2.0f / g.a2, sq = sqrtf(cs);  // the weight polynomial's argument scales
  const unsigned char *imgs = reinterpret_cast<const unsigned char *>(images);
  const size_t img_stride = (size_t)g.S * g.NX * ESZ;
  const unsigned lt = (1u << lane) - 1u;
  // the lane's columns (x, y), (x, y + 32 / FW): offsets from the centre, last
  // z level inside the volume (-1: the column is outside)
  const float dvx = (float)(lane % FW) - HX, dvy = (float)(lane / FW) - HY;
  int tmax[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int vx = fx0 + lane % FW, vy = fy0 + lane / FW + c * (32 / FW);
    tmax[c] = vx <= g.H && vy <= g.H && (!FOLD || vx <= -g.xa0) ? min(ZC - 1, g.H - z0) : -1;
  }

  int folds = 0;  // of the sums into the slab
  auto flush = [&]() {
    if (to_scratch && args.slab) {
      if (folds > 0 && args.slab_planes < 6) {  // no room for a pair; slab_once rules it out
        if (lane == 0) set_err(args.err, DERR_RANGE);
        return;
      }
      const size_t b = (size_t)block + warp * (WV / SLAB_BLOCK);
      g2_flush_slab<WV>(s_acc, args.slab + b * (size_t)(SLAB_BLOCK * args.slab_planes), folds++);
    } else {
      g2_flush<FW, KB>(args, s_acc, fx0, fy0, z0, to_scratch);
    }
  };
  g2_clear<WV>(s_acc, lane);
  __syncwarp();
  // PROF: phase counters (fr_options.debug bit 1), cycles of cull, item generation
  // with the patches (PH_QUEUE), evaluation rounds (PH_DRAIN_FAST) and flushes, item
  // and round counts, added by lane 0.  In kernels of their own: tests of a flag cost
  // the others 12 registers and 3 % (2500 images of 256^2: 4.29 -> 4.17 ms without;
  // 1000 of 128^2: 584 -> 564 us; 777 of 96^2, a = 2.5: 608 -> 588 us)
  const bool prof = PROF && args.phase != nullptr;
  auto tick = [&]() -> long long { return prof ? clock64() : 0; };
  auto count = [&](int what, long long v) {
    if (prof && lane == 0) atomicAdd(args.phase + what, (unsigned long long)v);
  };
  auto clocked = [&](int what, long long since) {
    if (prof && lane == 0) atomicAdd(args.phase + what, (unsigned long long)(clock64() - since));
  };
  const long long t_start = tick();
  const float reach = (float)g.H + g.a + 1e-2f;  // the extended plane spans [-H, H]^2

  // Records of listed images from `head` on, one image per lane, one record
  // per half plane whose pixels the footprint can meet (each half plane's
  // pixels lie in k_x >= 0 of the orientation):
  //   plane normal, u_z of the centre | first in-plane axis, fractional u_x |
  //   second in-plane axis, fractional u_y |
  //   first patch pixel relative to the centre's integer part and patch size
  //   (bytes px, py, pw, ph), first patch pixel (px | py << 16), image, flags
  //   (bit 0: reflected, bit 1: the image has records for both half planes)
  // Takes as many images as have G2_ENTRIES records; returns their number, ne
  // the number of records.
  auto build = [&](int head, int nl, int &ne) -> int {
    const bool have = lane < G2_ENTRIES && head + lane < nl;
    int i = 0;
    bool direct = false, refl = false;
    float e1x = 0, e1y = 0, e1z = 0, e2x = 0, e2y = 0, e2z = 0, mx = 0, my = 0, mz = 0;
    float fx = 0, fy = 0, uz = 0, sx = 0, sy = 0;
    int cxi = 0, cyi = 0;
    if (have) {
      i = s_idx[head + lane];
      const float *R = args.rot + 9 * (size_t)i;
      e1x = __ldg(R + 0); e1y = __ldg(R + 3); e1z = __ldg(R + 6);
      e2x = __ldg(R + 1); e2y = __ldg(R + 4); e2z = __ldg(R + 7);
      mx = __ldg(R + 2);  my = __ldg(R + 5);  mz = __ldg(R + 8);
      float hxx, lx, hyy, ly, hzz, lz;
      dot3_dd(e1x, e1y, e1z, cx, cy, cz, hxx, lx);
      dot3_dd(e2x, e2y, e2z, cx, cy, cz, hyy, ly);
      dot3_dd(mx, my, mz, cx, cy, cz, hzz, lz);
      if (args.ortho) {
        // An FP32 rotation is orthonormal only to 6e-8, which moves u by up to 6e-8
        // |c| from the coordinates of c on e1, e2 and its distance from their plane:
        // corrected to first order in R^T R - 1, formed without cancellation.
        const float d11 = dot3_less_one(e1x, e1y, e1z), d22 = dot3_less_one(e2x, e2y, e2z),
                    d33 = dot3_less_one(mx, my, mz);
        float d12, d13, d23, l12, l13, l23;
        dot3_dd(e1x, e1y, e1z, e2x, e2y, e2z, d12, l12);
        dot3_dd(e1x, e1y, e1z, mx, my, mz, d13, l13);
        dot3_dd(e2x, e2y, e2z, mx, my, mz, d23, l23);
        d12 += l12;
        d13 += l13;
        d23 += l23;
        lx -= fmaf(d11, hxx, d12 * hyy);
        ly -= fmaf(d12, hxx, d22 * hyy);
        lz -= fmaf(d13, hxx, fmaf(d23, hyy, 0.5f * d33 * hzz));
      }
      const float rx = rintf(hxx), ry = rintf(hyy);
      fx = (hxx - rx) + lx;  // hxx - rx is exact
      fy = (hyy - ry) + ly;
      uz = hzz + lz;
      sx = fabsf(e1x) * HX + fabsf(e1y) * HY + fabsf(e1z) * HZ;
      sy = fabsf(e2x) * HX + fabsf(e2y) * HY + fabsf(e2z) * HZ;
      const bool in = fabsf(hxx) <= reach + sx && fabsf(hyy) <= reach + sy;
      direct = in && hxx + sx + g.a + 1e-2f >= 0.f;
      refl = in && hxx - sx - g.a - 1e-2f <= 0.f;
      const float far = 4096.0f;  // bounds for inputs that are no rotation
      cxi = (int)fminf(fmaxf(rx, -far), far);
      cyi = (int)fminf(fmaxf(ry, -far), far);
    }
    const unsigned bd = __ballot_sync(FULL, direct), br = __ballot_sync(FULL, refl);
    int o = __popc(bd & lt) + __popc(br & lt);
    const int mine = (direct ? 1 : 0) + (refl ? 1 : 0);
    const unsigned taken = __ballot_sync(FULL, have && o + mine <= G2_ENTRIES);
    const int images_taken = __popc(taken);  // o + mine ascends: the first images
    ne = __popc(bd & taken) + __popc(br & taken);
    if (have && o + mine <= G2_ENTRIES) {
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (h == 0 ? direct : refl) {
          const float sg = h ? -1.f : 1.f;
          const float ffx = sg * fx, ffy = sg * fy;
          const int ccx = h ? -cxi : cxi, ccy = h ? -cyi : cyi;
          // pixels that the boxes can reach, inside the stored half plane [0, H]
          // x [-H, H - 1]; at least one whole box, at most PW x PW
          const float far = 4096.0f, wx_ = sx + (HB + 0.01f), wy_ = sy + (HB + 0.01f);
          const int lox = ccx + (int)fminf(fmaxf(ceilf(ffx - wx_), -far), far);
          const int hix = ccx + (int)fminf(fmaxf(floorf(ffx + wx_), -far), far);
          const int loy = ccy + (int)fminf(fmaxf(ceilf(ffy - wy_), -far), far);
          const int hiy = ccy + (int)fminf(fmaxf(floorf(ffy + wy_), -far), far);
          const int px = max(0, min(lox, g.H + 1 - PW)), py = max(-g.H, min(loy, g.H - PW));
          const int pw = min(max(min(hix, g.H) - px + 1, KB), min(PW, g.H + 1 - px));
          const int ph = min(max(min(hiy, g.H - 1) - py + 1, KB), min(PW, g.H - py));
          const int rpx = max(-127, min(px - ccx, 127)), rpy = max(-127, min(py - ccy, 127));
          s_rec[o * 4 + 0] = make_float4(mx, my, mz, uz);
          s_rec[o * 4 + 1] = make_float4(sg * e1x, sg * e1y, sg * e1z, ffx);
          s_rec[o * 4 + 2] = make_float4(sg * e2x, sg * e2y, sg * e2z, ffy);
          reinterpret_cast<int4 *>(s_rec)[o * 4 + 3] =
              make_int4((rpx & 255) | ((rpy & 255) << 8) | (pw << 16) | (ph << 24),
                        (px & 0xffff) | (py << 16), i, h | (mine == 2 ? 2 : 0));
          ++o;
        }
      }
    }
    __syncwarp();
    return images_taken;
  };

  // Patch copies: 16 columns x 2 rows a step (rows past the patch repeat its
  // last row), then the columns past 16 (4, 2 or 1 of them, 32 pixels a step).
  constexpr int RG = (PW + 1) / 2, XL = XC == 3 ? 4 : XC == 2 ? 2 : 1, XR = XC == 0 ? 0 : (PW * XL + 31) / 32;
  const int xc = lane % XL, xr = lane / XL;
  const int pc = lane & 15, pr = lane >> 4;
  const int row_bytes = g.NX * ESZ;
  __half2 stage[F16 ? RG + XR : 1];
  // start copying the patch of entry li (FP32: into its patch; FP16: into registers)
  auto fetch = [&](int li) {
    const int4 q = reinterpret_cast<const int4 *>(s_rec)[li * 4 + 3];
    const int pw = (q.x >> 16) & 255, ph1 = (int)((unsigned)q.x >> 24) - 1;
    const int px = q.y & 0xffff, py = q.y >> 16;
    const unsigned char *img = imgs + (size_t)(unsigned)q.z * img_stride + px * ESZ;
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(s_patch + (li & 1) * SH::PATCH)) +
                         (pr * PITCH + pc) * 8;
    const int c0 = min(pc, pw - 1) * ESZ;
    if (py < 0 && py + ph1 >= 0) {  // storage wraps at k_y = 0
#pragma unroll
      for (int r = 0; r < RG; ++r) {
        const int ky = py + min(2 * r + pr, ph1);
        const unsigned char *src = img + (ky + (ky < 0 ? g.S : 0)) * row_bytes + c0;
        if (F16) stage[r] = __ldg(reinterpret_cast<const __half2 *>(src));
        else if (2 * r + 1 < PW || pr == 0) cp_async8(dst + 2 * r * PITCH * 8, src);
      }
    } else {
      const unsigned char *first = img + (py + (py < 0 ? g.S : 0)) * row_bytes + c0;
#pragma unroll
      for (int r = 0; r < RG; ++r) {
        const unsigned char *src = first + (size_t)((unsigned)min(2 * r + pr, ph1) * (unsigned)row_bytes);
        if (F16) stage[r] = __ldg(reinterpret_cast<const __half2 *>(src));
        else if (2 * r + 1 < PW || pr == 0) cp_async8(dst + 2 * r * PITCH * 8, src);
      }
    }
    if (XC > 0 && pw > 16) {
      const int cx = min(16 + xc, pw - 1) - 16;
#pragma unroll
      for (int k = 0; k < XR; ++k) {
        const int row = xr + k * (32 / XL), ky = py + min(row, ph1);
        const unsigned char *src = img + (ky + (ky < 0 ? g.S : 0)) * row_bytes + (16 + cx) * ESZ;
        if (F16) stage[RG + k] = __ldg(reinterpret_cast<const __half2 *>(src));
        else if (row < PW && xc < XC)
          cp_async8(dst + (row * PITCH + 16 + xc - pr * PITCH - pc) * 8, src);
      }
    }
  };
  // FP16: convert the staged pixels into entry li's patch
  auto land = [&](int li, int pw) {
    float2 *dst = s_patch + (li & 1) * SH::PATCH + pr * PITCH + pc;
#pragma unroll
    for (int r = 0; r < RG; ++r)
      if (2 * r + 1 < PW || pr == 0) dst[2 * r * PITCH] = __half22float2(stage[r]);
    if (XC > 0 && pw > 16) {
#pragma unroll
      for (int k = 0; k < XR; ++k) {
        const int row = xr + k * (32 / XL);
        if (row < PW && xc < XC)
          dst[row * PITCH + 16 + xc - pr * PITCH - pc] = __half22float2(stage[RG + k]);
      }
    }
  };

  // one entry: its items, then their rounds
  auto entry = [&](int li, int ne) {
    const long long tq = tick();
    const float4 q0 = s_rec[li * 4], q1 = s_rec[li * 4 + 1], q2 = s_rec[li * 4 + 2];
    const int4 q3 = reinterpret_cast<const int4 *>(s_rec)[li * 4 + 3];
    const int rpx = (int)(signed char)(q3.x & 255), rpy = (int)(signed char)((q3.x >> 8) & 255);
    const int pw = (q3.x >> 16) & 255, ph = (int)((unsigned)q3.x >> 24);
    const float lox = (float)rpx, hix = (float)(rpx + pw - KB);
    const float loy = (float)rpy, hiy = (float)(rpy + ph - KB);
    const float2 *patch = s_patch + (li & 1) * SH::PATCH;
    if (F16) {
      land(li, pw);
      if (li + 1 < ne) fetch(li + 1);
    }
    if (FOLD) {
      // one bit per patch pixel, whether it counts in this entry.  In a row the
      // sign of R00 k_x + R01 k_y changes at most once: lane r finds where in
      // row r with five exact evaluations.
      if (lane < PW) {
        const bool refl = (q3.w & 1) != 0;
        const float r00 = refl ? -q1.x : q1.x, r01 = refl ? -q2.x : q2.x;
        const int px = q3.y & 0xffff, py = q3.y >> 16;
        const bool up = r00 < 0.f;  // the predicate (folded) turns true along the row, else false
        int t = 0;                  // columns before the turn, 0 .. 31 (not unrolled: the code is cold)
#pragma unroll 1
        for (int s = 16; s > 0; s >>= 1)
          if (fold_pred(r00, r01, px + t + s - 1, py + lane) != up) t += s;
        const unsigned before = t > 30 ? 0x7fffffffu : (1u << t) - 1u;
        const unsigned folded = up ? ~before : before;
        s_bits[(li & 1) * PITCH + lane] = refl ? folded : ~folded;
      }
    }
    // z levels t of each column with |u_z| <= a, u_z = b + m_z t: t within a /
    // |m_z| of -b / m_z (a_plane's margin covers the rounding of the quotients,
    // and of an m_z too small to divide by)
    const float iz = __fdividef(1.0f, fabsf(q0.z) < 1e-6f ? 1e-6f : q0.z), az = a_plane * fabsf(iz);
    float b = fmaf(q0.z, -HZ, fmaf(q0.y, dvy, fmaf(q0.x, dvx, q0.w)));
    int cnt[NC], first[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const float tc = b * iz;
      int tl = max(__float2int_ru(-tc - az), 0), th = min(__float2int_rd(az - tc), tmax[c]);
      if (q3.w & 2) {
        // only the items whose box reaches this entry's half plane: u_x >= -a
        // (lox is the column k_x = 0 here)
        const float bx = fmaf(q1.z, -HZ, fmaf(q1.y, dvy + c * (32 / FW), fmaf(q1.x, dvx, q1.w)));
        const float ez = fabsf(q1.z) < 1e-6f ? 1e-6f : q1.z;
        const float tb = (lox - a_plane - bx) * __fdividef(1.0f, ez);
        if (ez > 0.f) tl = max(tl, __float2int_ru(tb));
        else th = min(th, __float2int_rd(tb));
      }
      first[c] = tl;
      cnt[c] = max(th - tl + 1, 0);
      b = fmaf(q0.y, (float)(32 / FW), b);
    }
    // positions: all first columns, then all second ones
    int incl = NC == 2 ? cnt[0] | (cnt[NC - 1] << 16) : cnt[0];
#pragma unroll
    for (int s = 1; s < 32; s <<= 1)
      asm volatile(
          "{\n\t.reg .s32 r;\n\t.reg .pred p;\n\t"
          "shfl.sync.up.b32 r|p, %0, %1, 0, 0xffffffff;\n\t"
          "@p add.s32 %0, %0, r;\n\t}"
          : "+r"(incl)
          : "r"(s));
    const int tot = __shfl_sync(FULL, incl, 31);
    const int tot0 = tot & 0xffff, total = tot0 + (tot >> 16);
    // a tag is its slot less its position, modulo 256
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int p = c == 0 ? (NC == 2 ? incl & 0xffff : incl) - cnt[0]
                           : (tot & 0xffff) + (incl >> 16) - cnt[c];
      const unsigned char tag = (unsigned char)(lane * ZC + first[c] - p);
#pragma unroll
      for (int s = 0; s < ZC; ++s)
        if (s < cnt[c]) s_tag[p + s] = tag;
    }
    if (!F16) {
      // this entry's patch has landed; the next one's buffer is free
      cp_async_wait_all();
      __syncwarp();
      if (li + 1 < ne) fetch(li + 1);
    } else {
      __syncwarp();
    }
    clocked(PH_QUEUE, tq);
    count(PH_ITEMS_FAST, total);
    const long long td = tick();
    const float sgn = (q3.w & 1) ? -1.f : 1.f;
    // patch address of a pixel: at pixel (ox, oy) relative to the centre's
    // integer part it is ox + PITCH oy, plus 1.5 2^23 whose significand bits
    // arrive with it
    const float kM = 8388608.0f, kR = 12582912.0f;
    const unsigned base = (unsigned)-(rpy * PITCH + rpx) - 0x4b400000u;
    // an item: where its box is and u relative to it
    struct Item {
      int slot;
      const float2 *p;
      float dx, dy, uz2;
      const unsigned *rows;
      int shift, row;
    };
    auto locate = [&](unsigned tag, int h) -> Item {
      Item it;
      // the slot: of the first columns up to position tot0, of the second after
      const int slot = (int)((tag + h) & 255) + (NC == 2 && h >= tot0 ? 256 : 0);
      it.slot = slot;
      // voxel offsets from the centre: bit fields of the slot placed in the
      // significand of 2^23, scaled and shifted (exactly)
      const float sdz = (__int_as_float(0x4b000000 | (slot & (ZC - 1))) - kM) - HZ;
      const float sdx = fmaf(__int_as_float(0x4b000000 | (slot & ((FW - 1) * ZC))), 1.0f / ZC,
                             -(kM / ZC + HX));
      const float sdy = fmaf(__int_as_float(0x4b000000 | (slot & ((FH - 1) * FW * ZC))),
                             1.0f / (ZC * FW), -(kM / (ZC * FW) + HY));
      const float uz = fmaf(q0.z, sdz, fmaf(q0.y, sdy, fmaf(q0.x, sdx, q0.w)));
      const float ux = fmaf(q1.z, sdz, fmaf(q1.y, sdy, fmaf(q1.x, sdx, q1.w)));
      const float uy = fmaf(q2.z, sdz, fmaf(q2.y, sdy, fmaf(q2.x, sdx, q2.w)));
      // box origin: the nearest integer to u - 1.5 (2.5; by adding 1.5 2^23), clamped
      constexpr float HO = HB - 0.5f;
      const float ox = fminf(fmaxf(__fadd_rn(__fadd_rn(ux - HO, kR), -kR), lox), hix);
      const float oy = fminf(fmaxf(__fadd_rn(__fadd_rn(uy - HO, kR), -kR), loy), hiy);
      it.p = patch + (__float_as_uint(fmaf(oy, (float)PITCH, __fadd_rn(ox, kR))) + base);
      it.dx = ux - ox;
      it.dy = uy - oy;
      it.uz2 = uz * uz;
      it.rows = s_bits;
      it.shift = it.row = 0;
      if (FOLD) {
        it.shift = (int)(ox - lox);
        it.row = (int)(oy - loy);
        it.rows += (li & 1) * PITCH + it.row;
      }
      return it;
    };
    // one round ahead: the tags are loaded (their buffer is a round longer)
    unsigned next = s_tag[lane];
    // the last round of at most 16 items takes two lanes an item, two rows of the
    // box each (half of all entries end in one: 137 items on average)
    constexpr bool HALF = KB == 4 && !FOLD;
    int left = total;
#pragma unroll 1
    for (int h = lane; left > (HALF ? 16 : 0); h += 32, left -= 32) {
      const Item it = locate(next, h);
      next = s_tag[h + 32];
      // the partial sums, read before the box: no other item of the entry adds to them
      const float tr = s_acc[it.slot], ti = s_acc[WV + it.slot], tw = s_acc[2 * WV + it.slot];
      float ar, ai, aw;
      bool ties = false;
      if (KB == 4 && !FOLD)
        g2_box14<PITCH>(cst.poly2, it.p, it.dx, it.dy, it.uz2, cs, sq, ar, ai, aw);
      else if (KB == 5 && !FOLD)
        g2_box23<PITCH>(cst.poly2, it.p, it.dx, it.dy, it.uz2, cs, sq, ar, ai, aw);
      else
        ties = g2_box<PITCH, KB, FOLD>(cst.poly2, it.p, it.dx, it.dy, it.uz2, cs, sq, ar, ai, aw,
                                       it.rows, it.shift);
      if (FOLD && KB > 4 && ties)
        g2_ties<PITCH, KB>(cst.poly2, it.p, it.dx, it.dy, it.uz2, cs, sq, it.rows, it.shift, q1, q2,
                           make_int3(fx0 + (it.slot / ZC) % FW, fy0 + it.slot / (ZC * FW), z0 + it.slot % ZC),
                           make_int2((q3.y & 0xffff) + it.shift, (q3.y >> 16) + it.row), g.a, ar, ai, aw);
      if (h < total) {
        s_acc[it.slot] = tr + ar;
        s_acc[WV + it.slot] = fmaf(sgn, ai, ti);
        s_acc[2 * WV + it.slot] = tw + aw;
      }
    }
    if (HALF && left > 0) {
      const int h = total - left + (lane & 15), half = lane >> 4;
      const Item it = locate(s_tag[h], h);
      const float tr = s_acc[it.slot], ti = s_acc[WV + it.slot], tw = s_acc[2 * WV + it.slot];
      float ar, ai, aw;
      g2_box<PITCH, KB, FOLD, KB / 2>(cst.poly2, it.p + half * (KB / 2 * PITCH), it.dx,
                                      it.dy - (float)(half * (KB / 2)), it.uz2, cs, sq, ar, ai, aw,
                                      it.rows + half * (KB / 2), it.shift);
      ar += __shfl_xor_sync(FULL, ar, 16);
      ai += __shfl_xor_sync(FULL, ai, 16);
      aw += __shfl_xor_sync(FULL, aw, 16);
      if (lane < left) {
        s_acc[it.slot] = tr + ar;
        s_acc[WV + it.slot] = fmaf(sgn, ai, ti);
        s_acc[2 * WV + it.slot] = tw + aw;
      }
    }
    __syncwarp();
    count(PH_ROUNDS, (total + 31) / 32);
    clocked(PH_DRAIN_FAST, td);
  };

  int nl = 0;           // listed images
  int since_flush = 0;  // images listed since the last flush
  // plane normals of the next 32 images, loaded one step ahead
  float nx = 0.f, ny = 0.f, nz = 0.f;
  auto load_normals = [&](int i) {
    if (i < img1) {
      const float *R = args.rot + 9 * (size_t)i;
      nx = __ldg(R + 2);
      ny = __ldg(R + 5);
      nz = __ldg(R + 8);
    }
  };
  load_normals(img0 + lane);
  for (int cs0 = img0;; cs0 += 32) {
    const bool last = cs0 >= img1;
    if (!last) {
      // cull: an image is listed if its plane passes within a of the footprint box
      const long long tc = tick();
      const int i = cs0 + lane;
      const float d = nx * cx + ny * cy + nz * cz;
      const float supp = fabsf(nx) * HX + fabsf(ny) * HY + fabsf(nz) * HZ;
      const bool keep = i < img1 && fabsf(d) <= g.a + supp + 1e-3f;
      load_normals(i + 32);
      const unsigned bk = __ballot_sync(FULL, keep);
      if (keep) s_idx[nl + __popc(bk & lt)] = i;
      nl += __popc(bk);
      __syncwarp();
      clocked(PH_CULL, tc);
    }
    // the next step lists at most 32 images
    if (nl > lcap - 32 || (last && nl > 0)) {
      for (int head = 0; head < nl;) {
        int ne = 0;
        head += build(head, nl, ne);
        count(PH_LIST_IMAGES, ne);
        if (ne > 0) fetch(0);
        for (int li = 0; li < ne; ++li) entry(li, ne);
      }
      since_flush += nl;
      nl = 0;
      if (since_flush > GATHER_FLUSH - lcap) {
        const long long tf = tick();
        flush();
        g2_clear<WV>(s_acc, lane);
        __syncwarp();
        clocked(PH_FLUSH, tf);
        since_flush = 0;
      }
    }
    if (last) break;
  }
  const long long tf = tick();
  if (since_flush) flush();
  if (to_scratch && args.slab) {
    if (slab_once(args.n, nsplit)) {  // one FP32 sum, no state to read: zeros if no image came
      if (folds == 0) flush();
    } else if (lane == 0) {
      args.slab_state[block + warp * (WV / SLAB_BLOCK)] = min(folds, 2);
    }
  }
  clocked(PH_FLUSH, tf);
  clocked(PH_WARP_CYCLES, t_start);
}

// Bricks of the fold columns: one footprint wide (three fold columns for a < 2,
// five for 2 <= a < 3), 32 x 8.
template <int KB>
__host__ __device__ constexpr int g2_fold_width() {
  return KB == 4 ? 4 : 8;
}
constexpr int G2_FOLD_BY = 32, G2_FOLD_BZ = 8;

// Dynamic shared memory of a launch: a warp of the main or the fold columns.
template <int KB>
__host__ __device__ constexpr size_t gather2_smem(int chunk) {
  const size_t m = gather2_warp_smem<8, KB, 0>(chunk),
               f = gather2_warp_smem<g2_fold_width<KB>(), KB, 1>(chunk);
  return m > f ? m : f;
}

// Work unit k of a launch without a unit list: split k / (bricks) of brick k %
// (bricks) of those that tile x in [x0, x1], of as many splits as its expected
// images (brick_unit_loads' estimate) over unit_share; false if it has fewer.  The
// last splits come first: only the bricks around the centre have them, whose units
// take longest, and the launch ends on units of the outer bricks (S = 64, 200
// images: 91 -> 81 us a call; 1000 images: 288 -> 273).
template <int BX, int BY, int BZ>
__device__ __forceinline__ bool g2_implicit_unit(const InsertArgs &args, int x0, int x1, int k,
                                                 int4 &unit) {
  const Geom &g = args.g;
  const int nbx = (x1 - x0 + BX) / BX, nby = (g.D + BY - 1) / BY, nbz = (g.D + BZ - 1) / BZ;
  const int b = k % (nbx * nby * nbz), s = args.unit_most - 1 - k / (nbx * nby * nbz);
  const int bx = b % nbx, by = b / nbx % nby, bz = b / (nbx * nby);
  const float hx = 0.5f * (BX - 1), hy = 0.5f * (BY - 1), hz = 0.5f * (BZ - 1);
  const float cx = x0 + bx * BX + hx, cy = -g.H + by * BY + hy, cz = -g.H + bz * BZ + hz;
  const float d = sqrtf(cx * cx + cy * cy + cz * cz), r = g.a + sqrtf(hx * hx + hy * hy + hz * hz);
  const float load = args.n * ((d <= r ? 1.0f : r / d) + 0.02f);
  const int ns = max(1, min((int)ceilf(load / args.unit_share), args.unit_most));
  unit = make_int4(bx, by, bz, s | (ns << 16) | (1 << 30));
  return s < ns;
}

// A unit's brick, packed, and split word as gather2_warp takes them.
__device__ __forceinline__ int4 g2_unpack(int brick, int word) {
  return make_int4(brick & 1023, (brick >> 10) & 1023, (brick >> 20) & 1023, word);
}

// One warp per CTA: after the nfold units of the fold columns (the few heavy ones
// first), CTA b takes footprint b % W of work unit args.units[b / W] (W footprints
// a brick).  Warps of one brick never wait for one another, but a CTA holds its
// shared memory until its last warp ends: with two and four warps a CTA 17 % of
// the resident warp slots stood idle.  Both kinds of unit in one launch: as a
// second kernel on a side stream the fold columns cost a fork and a join.  Shared
// memory holds 16 CTAs an SM, so the registers are bounded for 16 (a bound for 24, 80
// registers, spilled: 8.5 ms instead of 8.2 for 5000 images of 256^2).  KB: what the
// launch's geometry and shared memory are for (4, or 6 for a >= 2), KBM: width of the
// boxes (5 for 2 <= a <= 2.5).
template <int BX, int BY, int BZ, int F16, int KB = 4, int KBM = KB, int PROF = 0>
__global__ void __launch_bounds__(32, 16)
gather2_kernel(const __grid_constant__ InsertArgs args) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int FW = g2_fold_width<KB>(), W = g2_warps<BX, BY, BZ, 8>(),
                WF = g2_warps<FW, G2_FOLD_BY, G2_FOLD_BZ, FW>();
  const Geom &g = args.g;
  const int nf = args.nfold * WF;
  const bool fold = (int)blockIdx.x < nf;
  const int b = fold ? blockIdx.x : blockIdx.x - nf, k = fold ? b / WF : b / W;
  int4 unit;
  int block = 0;
  if (args.units) {
    const int4 q = fold ? args.fold[k] : args.units[k];
    unit = g2_unpack(q.x, q.w);
    block = q.y;
  } else if (fold ? !g2_implicit_unit<FW, G2_FOLD_BY, G2_FOLD_BZ>(args, g.xa0, -g.xa0, k, unit)
                  : !g2_implicit_unit<BX, BY, BZ>(args, 1 - g.xa0, g.H, k, unit)) {
    return;
  }
  if (fold)
    gather2_warp<FW, G2_FOLD_BY, G2_FOLD_BZ, F16, KBM, FW, 1, PROF>(args, args, args.images, smem, unit,
                                                                   block, b % WF);
  else
    gather2_warp<BX, BY, BZ, F16, KBM, 8, 0, PROF>(args, args, args.images, smem, unit, block, b % W);
}

// Several batches in one launch: work items p.items[k] = {bx | by << 10 | bz <<
// 20, split word, batch | slot << 24, slab} of batch p.descs[batch], first those of the
// fold columns; geometry, weight polynomial and list capacity, common to the launch's
// batches, are read from p.base (kernel parameters: constant operands in the
// inner loops), the batch's own arguments (rotations, volume) from its
// descriptor.
template <int BX, int BY, int BZ, int F16, int KB = 4, int KBM = KB>
__global__ void __launch_bounds__(32, 16)
gather2_multi_kernel(const __grid_constant__ MultiLaunch p) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int FW = g2_fold_width<KB>(), W = g2_warps<BX, BY, BZ, 8>(),
                WF = g2_warps<FW, G2_FOLD_BY, G2_FOLD_BZ, FW>();
  const int nf = p.nfold * WF, b = (int)blockIdx.x - nf;
  const int4 it = p.items[b < 0 ? (int)blockIdx.x / WF : p.nfold + b / W];
  const int4 unit = g2_unpack(it.x, it.y);
  const InsertArgs &args = p.descs[it.z & 0xffffff];
  const void *images = p.images[(unsigned)it.z >> 24];
  if (b < 0)
    gather2_warp<FW, G2_FOLD_BY, G2_FOLD_BZ, F16, KBM, FW, 1>(args, p.base, images, smem, unit, it.w,
                                                             (int)(blockIdx.x % WF));
  else
    gather2_warp<BX, BY, BZ, F16, KBM>(args, p.base, images, smem, unit, it.w, b % W);
}

}  // namespace fr
