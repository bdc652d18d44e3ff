"""GPU parity of the direct-drain gather at the edges of its pixel patches.

A patch holds at most 19 x 19 stored pixels, copied 16 columns and 2 rows at a
time and clamped into the half plane.  The sizes put every edge inside small
volumes: images narrower than a patch (S = 8 .. 30), row lengths S/2 + 1 that
are even (16-byte rows) and odd, patches that wrap at k_y = 0 and cross
k_x = 0, footprints cut by the volume's border, an odd number of images, and
blobs from less than one voxel to the widest 6-wide box.  Tolerance: the
library's parity bar (2e-5 of the largest value, FP32 accumulation of at most
40 images; FP16 images against the oracle fed the rounded values)."""
import numpy as np
import pytest
import torch

from paper_1910_08498_gb300 import _lib as L
from paper_1910_08498_gb300 import inputs
from tests.helpers import TOL_F32, gpu_insert, oracle_insert, rel_err, worst

pytestmark = pytest.mark.gpu


def _batch(S, n, seed):
    img, rot = inputs.make_batch(S, n, seed)
    perm = inputs.proper_signed_permutations()
    rot[:5] = perm[[0, 5, 11, 17, 22]]  # planes along the axes: runs of every z level or none
    return img, rot


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("a", [0.6, 1.0, 1.5, 1.999, 2.0, 2.25, 2.5, 2.51, 2.999])
@pytest.mark.parametrize("S", [8, 10, 14, 16, 18, 30, 32, 34, 46])
def test_patch_edges_match_oracle(S, a, f16):
    a = float(np.float32(a))
    batches = [_batch(S, 33, 7 * S)]
    V, W, _ = gpu_insert(S, batches, a=a, tuning=False, f16=f16)
    Vr, Wr, _ = oracle_insert(S, batches, a=a, f16=f16)
    assert rel_err(V, Vr) <= TOL_F32, worst(V, Vr, S)
    assert rel_err(W, Wr) <= TOL_F32, worst(W, Wr, S)


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("a", [0.6, 1.0, 1.5, 1.9, 2.5, 2.999])
@pytest.mark.parametrize("S,n", [(8, 1), (8, 40), (10, 3), (16, 17), (30, 33), (46, 15), (64, 130), (64, 400),
                                 (46, 700), (64, 640)])
def test_no_allocation_call_matches_oracle(S, n, a, f16):
    """Batches and radii that keep the scatter (small ones, a = 1), and the
    gather with units worked out by the CTAs themselves.  700 images: FP32 sums
    of a voxel's about 700 terms, within the bar by the scatter's own test of
    1024-image sub-batches."""
    a = float(np.float32(a))
    img, rot = inputs.make_batch(S, n, 11 * S + n)
    perm = inputs.proper_signed_permutations()
    rot[:min(n, 3)] = perm[[3, 9, 20]][:min(n, 3)]
    V = torch.zeros((S + 1) ** 3, dtype=torch.complex64, device="cuda")
    W = torch.zeros((S + 1) ** 3, dtype=torch.float32, device="cuda")
    dev = (inputs.to_half(img) if f16 else img).cuda()
    assert L.fr_insert_noalloc(S, dev, rot.cuda(), V, W, a=a, alpha=15.0) == L.FR_OK
    Vr, Wr, _ = oracle_insert(S, [(img, rot)], a=a, f16=f16)
    Vn, Wn = V.cpu().numpy(), W.cpu().numpy()
    assert rel_err(Vn, Vr) <= TOL_F32, worst(Vn, Vr, S)
    assert rel_err(Wn, Wr) <= TOL_F32, worst(Wn, Wr, S)


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("a", [1.9, 2.5, 2.999])
@pytest.mark.parametrize("config", [47, 49])
def test_phase_counting_kernel_computes_the_same_sums(config, a, f16):
    """The counters run in kernels of their own; 12 images are not split, so the
    sums of two runs are the same bits."""
    if a >= 2:
        config = -1  # the default's wide boxes
    S, n = 30, 12
    img, rot = _batch(S, n, 3)
    out = []
    for debug in (0, 2):
        ctx = L.fr_create(S, float(np.float32(a)), 15.0, 0, 10000)
        try:
            L.fr_set_options(ctx, tuning=0, forced_config=config, debug=debug)
            L.fr_insert(ctx, (inputs.to_half(img) if f16 else img).cuda(), rot.cuda())
            V = torch.empty((S + 1) ** 3, dtype=torch.complex64, device="cuda")
            W = torch.empty((S + 1) ** 3, dtype=torch.float32, device="cuda")
            L.fr_finalize(ctx, V, W)
            out.append((V.cpu(), W.cpu(), sum(L.fr_debug_phase_counters(ctx).values())))
        finally:
            L.fr_destroy(ctx)
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == 0 and out[1][2] > 0


def test_pixels_outside_the_blob_do_not_reach_a_voxel():
    """One infinite pixel: only the voxels within the radius of it are not finite."""
    S = 32
    img, rot = inputs.make_batch(S, 2, 5)
    img[1, 3, 7] = complex(float("inf"), 0.0)
    V, W, _ = gpu_insert(S, [(img, rot)], tuning=False)
    q = rot[1].double() @ torch.tensor([7.0, 3.0, 0.0], dtype=torch.float64)
    if rot[1, 0, 0] * 7 + rot[1, 0, 1] * 3 < 0:
        q = -q
    D, H = S + 1, S // 2
    g = np.arange(D) - H
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    r2 = (x - float(q[0])) ** 2 + (y - float(q[1])) ** 2 + (z - float(q[2])) ** 2
    a2 = float(np.float32(1.9)) ** 2
    inside = (r2 <= a2 - 1e-4).ravel()
    outside = (r2 > a2 + 1e-4).ravel()
    assert not np.isfinite(V[inside]).any()
    assert np.isfinite(V[outside]).all()
    assert np.isfinite(W).all()


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("a", [1.9, 2.5, 2.999])
def test_split_units_sums_are_not_rounded(a, f16):
    """100 copies of one image: around the centre a unit takes two.  Its FP32 sum of at
    most four terms (an image meets a voxel in up to two records) takes three roundings,
    the single image's sum one, the export one: 5 x 2^-24 of a voxel's W; 50 units'
    sums added in FP32 round 49 times more."""
    S, n, a = 32, 100, float(np.float32(a))
    img, rot = inputs.make_batch(S, 1, 9)
    _, W1, _ = gpu_insert(S, [(img, rot)], a=a, tuning=False, f16=f16)
    _, W, _ = gpu_insert(S, [(img.repeat(n, 1, 1), rot.repeat(n, 1, 1))], a=a, tuning=False, f16=f16)
    g = np.abs(np.arange(S + 1) - S // 2) <= 2
    near = (g[:, None, None] & g[:, None] & g).ravel()
    assert W1[near].max() > 0
    err = np.abs(W[near] - n * W1[near])
    assert np.all(err <= 5 * 2.0 ** -24 * n * W1[near]), np.max(err / np.maximum(n * W1[near], 1e-30))


@pytest.mark.parametrize("S,n,a", [(64, 640, 1.9), (48, 300, 2.25), (40, 200, 2.9), (16, 20000, 1.9)])
def test_split_units_give_the_same_bits_every_time(S, n, a):
    """The units of a brick are summed in their order (20,000 images: units that fold
    their sums into their slab more than once)."""
    img, rot = _batch(S, n, 13)
    runs = [gpu_insert(S, [(img, rot)], a=float(np.float32(a)), tuning=False) for _ in range(3)]
    for V, W, _ in runs[1:]:
        assert np.array_equal(V, runs[0][0]) and np.array_equal(W, runs[0][1])
    Vr, Wr, _ = oracle_insert(S, [(img, rot)], a=float(np.float32(a)))
    assert rel_err(runs[0][0], Vr) <= TOL_F32 and rel_err(runs[0][1], Wr) <= TOL_F32


@pytest.mark.parametrize("a", [2.0, 2.00001, 5 ** 0.5, 2.236079, 8 ** 0.5, 2.8284414])
def test_fold_columns_decide_the_edge_band_once(a):
    """Signed permutations put whole lattices of candidates at the blob's edge, or 1e-5
    a^2 inside it, where the box leaves them to the exact decision; alpha = 0 gives
    each the weight 1."""
    S, a = 24, float(np.float32(a))
    rot = inputs.proper_signed_permutations()
    img, _ = inputs.make_batch(S, rot.shape[0], 21)
    V, W, _ = gpu_insert(S, [(img, rot)], a=a, alpha=0.0, tuning=False)
    Vr, Wr, _ = oracle_insert(S, [(img, rot)], a=a, alpha=0.0)
    assert rel_err(V, Vr) <= TOL_F32, worst(V, Vr, S)
    assert rel_err(W, Wr) <= TOL_F32, worst(W, Wr, S)
