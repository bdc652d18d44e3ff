"""fr_insert_noalloc: the insertion entry point that allocates no device memory.

The file name sorts last so that, in a full run, these tests also execute
after every other test has used the library on the same device.

* GPU: two calls in a row into zeroed caller-owned V, W give, within the
  FP32 tolerance, what the FP64 oracle gives for the two seeded batches (and
  what the context entry point gives), at the largest size the fixed scratch
  holds and with the largest blob radius (the scratch filled to its last
  cell); FP16 images within the FP16 bound; a call after the one-time setup
  changes the device's free memory by nothing.
* CPU: sizes above the fixed scratch are rejected with FR_ERR_NOALLOC_LIMIT
  before any CUDA call.
"""
import numpy as np
import pytest
import torch

from paper_1910_08498_gb300 import _lib as L
from paper_1910_08498_gb300 import inputs
from tests.helpers import A32, ALPHA, TOL_F16, TOL_F32, gpu_insert, oracle_insert, rel_err, worst


def test_noalloc_rejects_sizes_beyond_its_scratch():
    lib = L.lib()
    S = L.FR_NOALLOC_MAX_S + 2
    rc = lib.fr_insert_noalloc(S, 1.9, 15.0, None, L.FR_F32, None, 10, None, None, None)
    assert rc == L.FR_ERR_NOALLOC_LIMIT
    assert b"fr_insert_noalloc" in lib.fr_error_string(rc)
    # odd and tiny sizes keep their usual statuses
    assert lib.fr_insert_noalloc(63, 1.9, 15.0, None, L.FR_F32, None, 10, None, None, None) == \
        L.FR_ERR_UNSUPPORTED
    assert lib.fr_insert_noalloc(6, 1.9, 15.0, None, L.FR_F32, None, 10, None, None, None) == \
        L.FR_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("a", [A32, 2.5, 2.9])
def test_noalloc_two_calls_match_oracle(a):
    a = float(np.float32(a))
    S = L.FR_NOALLOC_MAX_S
    b1 = inputs.make_batch(S, 300, 41)
    b2 = inputs.make_batch(S, 257, 42)
    Vr, Wr, _ = oracle_insert(S, [b1, b2], a=a, alpha=ALPHA)
    Vc, Wc, _ = gpu_insert(S, [b1, b2], a=a, alpha=ALPHA, tuning=False)

    D3 = (S + 1) ** 3
    V = torch.zeros(D3, dtype=torch.complex64, device="cuda")
    W = torch.zeros(D3, dtype=torch.float32, device="cuda")
    for img, rot in (b1, b2):
        rc = L.fr_insert_noalloc(S, img.cuda(), rot.cuda(), V, W, a=a, alpha=ALPHA)
        assert rc == L.FR_OK
    torch.cuda.synchronize()
    Vn = V.cpu().numpy().astype(np.complex128)
    Wn = W.cpu().numpy().astype(np.float64)
    assert rel_err(Vn, Vr) <= TOL_F32, (rel_err(Vn, Vr), worst(Vn, Vr, S))
    assert rel_err(Wn, Wr) <= TOL_F32, (rel_err(Wn, Wr), worst(Wn, Wr, S))
    # and the context entry point on the same batches
    assert rel_err(Vn, Vc) <= TOL_F32 and rel_err(Wn, Wc) <= TOL_F32
    # voxels the fold never reaches stay exactly zero
    H = S // 2
    xa0 = -int(np.floor(np.float32(a)))
    Wg = Wn.reshape(S + 1, S + 1, S + 1)
    assert not Wg[:, :, : xa0 + H].any()


@pytest.mark.gpu
def test_noalloc_call_after_setup_allocates_nothing():
    S = 32
    img, rot = inputs.make_batch(S, 64, 43)
    img, rot = img.cuda(), rot.cuda()
    D3 = (S + 1) ** 3
    V = torch.zeros(D3, dtype=torch.complex64, device="cuda")
    W = torch.zeros(D3, dtype=torch.float32, device="cuda")
    L.fr_insert_noalloc(S, img, rot, V, W)  # first call on the device: one-time setup
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    L.fr_insert_noalloc(S, img, rot, V, W)
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free1 == free0
    # two identical calls: W is twice one call's W
    W1 = torch.zeros_like(W)
    V1 = torch.zeros_like(V)
    L.fr_insert_noalloc(S, img, rot, V1, W1)
    torch.cuda.synchronize()
    assert rel_err(W.cpu().numpy(), 2 * W1.cpu().numpy().astype(np.float64)) <= TOL_F32


@pytest.mark.gpu
def test_noalloc_fp16_images():
    """FP16-stored images through the no-allocation entry point: within the
    FP16 bound of the oracle fed the FP32 values, within the FP32 bound of
    the oracle fed the FP16-rounded values."""
    S = L.FR_NOALLOC_MAX_S
    img, rot = inputs.make_batch(S, 200, 44)
    Vr, Wr, _ = oracle_insert(S, [(img, rot)])
    V16, W16, _ = oracle_insert(S, [(img, rot)], f16=True)
    D3 = (S + 1) ** 3
    V = torch.zeros(D3, dtype=torch.complex64, device="cuda")
    W = torch.zeros(D3, dtype=torch.float32, device="cuda")
    assert L.fr_insert_noalloc(S, inputs.to_half(img).cuda(), rot.cuda(), V, W, a=A32,
                               alpha=ALPHA) == L.FR_OK
    torch.cuda.synchronize()
    Vn = V.cpu().numpy().astype(np.complex128)
    Wn = W.cpu().numpy().astype(np.float64)
    assert rel_err(Vn, Vr) <= TOL_F16 and rel_err(Wn, Wr) <= TOL_F16
    assert rel_err(Vn, V16) <= TOL_F32 and rel_err(Wn, W16) <= TOL_F32


def _lattice_rotations(n):
    """Rotations by the 3-4-5 angle about each axis, turned by the signed
    permutations: for a^2 = 3.6 pixels lie at distance a from voxels, to rounding,
    all over the volume."""
    c, s = 0.6, 0.8
    turns = [np.array(m) for m in ([[c, -s, 0], [s, c, 0], [0, 0, 1]], [[1, 0, 0], [0, c, -s], [0, s, c]],
                                   [[c, 0, s], [0, 1, 0], [-s, 0, c]])]
    perms = inputs.proper_signed_permutations().double().numpy()
    rots = [p @ t for t in turns for p in perms]
    return torch.tensor(np.stack([rots[i % len(rots)] for i in range(n)]), dtype=torch.float32)


def _noalloc(S, img, rot, a, alpha):
    V = torch.zeros((S + 1) ** 3, dtype=torch.complex64, device="cuda")
    W = torch.zeros((S + 1) ** 3, dtype=torch.float32, device="cuda")
    assert L.fr_insert_noalloc(S, img.cuda(), rot.cuda(), V, W, a=a, alpha=alpha) == L.FR_OK
    return V.cpu().numpy().astype(np.complex128), W.cpu().numpy().astype(np.float64)


@pytest.mark.gpu
@pytest.mark.parametrize("alpha", [0.0, 2.0, 8.0, 15.0])
@pytest.mark.parametrize("a,lattice", [(3.6 ** 0.5, True), (A32, False), (6.4 ** 0.5, True)])
def test_noalloc_decides_the_blob_edge_for_every_taper(a, lattice, alpha):
    """b(a) = 1 / I0(alpha) is 1 at alpha = 0: a candidate at the blob's edge that
    is decided wrongly then costs a whole pixel.  Sizes and radii at which the
    gather is the faster kernel."""
    S, n = L.FR_NOALLOC_MAX_S, 400
    a = float(np.float32(a))
    img, rot = inputs.make_batch(S, n, 45)
    if lattice:
        rot = _lattice_rotations(n)
    V, W = _noalloc(S, img, rot, a, alpha)
    Vr, Wr, _ = oracle_insert(S, [(img, rot)], a=a, alpha=alpha)
    assert rel_err(V, Vr) <= TOL_F32, worst(V, Vr, S)
    assert rel_err(W, Wr) <= TOL_F32, worst(W, Wr, S)


@pytest.mark.gpu
@pytest.mark.parametrize("tail", [20, 300])
def test_noalloc_sub_batches_of_both_kernels(tail):
    """A full sub-batch by the gather, then a tail that is small enough for the
    scatter or large enough for the gather."""
    S, n = L.FR_NOALLOC_MAX_S, 1024 + tail
    img, rot = inputs.make_batch(S, n, 46)
    V, W = _noalloc(S, img, rot, A32, ALPHA)
    Vr, Wr, _ = oracle_insert(S, [(img, rot)])
    assert rel_err(V, Vr) <= TOL_F32, worst(V, Vr, S)
    assert rel_err(W, Wr) <= TOL_F32, worst(W, Wr, S)


_SETUP_CHILD = """
import torch
from paper_1910_08498_gb300 import _lib as L
from paper_1910_08498_gb300 import inputs

def args(S, n, f16):
    img, rot = inputs.make_batch(S, n, 47)
    img = (inputs.to_half(img) if f16 else img).cuda()
    return S, img, rot.cuda(), torch.zeros((S + 1) ** 3, dtype=torch.complex64, device="cuda"), \
        torch.zeros((S + 1) ** 3, dtype=torch.float32, device="cuda")

small = args(16, 4, False)
calls = [(args(64, 400, f16), a) for f16 in (False, True) for a in (1.9, 2.25, 2.9)]
calls += [(args(32, 30, f16), a) for f16 in (False, True) for a in (1.9, 2.25)]
L.fr_insert_noalloc(*small)  # the first call on the device: all of the setup
torch.cuda.synchronize()
free0, _ = torch.cuda.mem_get_info()
for c, a in calls:
    L.fr_insert_noalloc(*c, a=a)
    torch.cuda.synchronize()
    print(free0 - torch.cuda.mem_get_info()[0])
"""


@pytest.mark.gpu
def test_noalloc_first_call_is_the_whole_setup():
    """In a fresh process, after one small call (which runs the scatter): calls of
    every kernel variant load no code, so that they change no free memory."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _SETUP_CHILD], cwd=root, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=root, CUDA_MODULE_LOADING="LAZY"))
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["0"] * 10, r.stdout


@pytest.mark.gpu
def test_noalloc_call_can_be_captured():
    """The gather's call in a graph, replayed into the same V, W."""
    S, n = L.FR_NOALLOC_MAX_S, 300
    img, rot = inputs.make_batch(S, n, 48)
    V, W = _noalloc(S, img, rot, A32, ALPHA)
    img, rot = img.cuda(), rot.cuda()
    Vg = torch.zeros((S + 1) ** 3, dtype=torch.complex64, device="cuda")
    Wg = torch.zeros((S + 1) ** 3, dtype=torch.float32, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        L.fr_insert_noalloc(S, img, rot, Vg, Wg, a=A32, alpha=ALPHA)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert rel_err(Vg.cpu().numpy(), 2 * V) <= TOL_F32 and rel_err(Wg.cpu().numpy(), 2 * W) <= TOL_F32
