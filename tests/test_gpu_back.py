"""The way back at the edges of its kernels: rsc_reconstruct's two layouts
(16-byte pieces or single entries), its longest codes, missing steps, weights
outside the range of its FP32 accumulator and entries that cancel;
rsc_synthesize's tiles of 128 and 32 patches and of up to 128 pixels."""
import ctypes

import numpy as np
import pytest

from oracle import basis as obasis, ksvd
from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


def _gpu_reconstruct(rsc, d, R, atom, angle, coef, shift=0):
    """shift: floats by which the output misses a 16-byte boundary."""
    import torch
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    t = [torch.from_numpy(v).cuda() for v in (atom, angle, coef)]
    P, K = atom.shape
    n = P * d[0].size
    buf = torch.full((n + 4,), np.nan, dtype=torch.float32, device="cuda")
    out = buf[shift:shift + n]
    vp = ctypes.c_void_p
    assert rsc.load_library().rsc_reconstruct(
        vp(dic.handle), P, K, *[vp(v.data_ptr()) for v in t], vp(out.data_ptr()),
        vp(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + n:]).all()
    dic.close()
    return out.cpu().numpy().reshape((P,) + d.shape[1:])


def _codes(P, K, M, R, seed):
    rng = np.random.default_rng(seed)
    atom = rng.integers(-1, M, (P, K)).astype(np.int32)
    angle = np.where(atom < 0, -1, rng.integers(0, R, (P, K))).astype(np.int32)
    return atom, angle, np.where(atom < 0, 0.0, rng.standard_normal((P, K)))


@pytest.mark.parametrize("shape", [
    # (M, J, kmax, R, K, P, shift)
    (5, 6, 8, 64, 5, 1, 0), (5, 6, 8, 64, 5, 17, 0), (5, 6, 8, 64, 5, 33, 2),
    (4, 5, 9, 33, 3, 50, 0), (3, 4, 16, 128, 16, 40, 0), (3, 30, 16, 7, 1, 19, 0),
    (6, 3, 0, 1, 2, 16, 0)], ids=str)
def test_reconstruct_edges(rsc, shape):
    """The accumulator is exact to 2^-41 of a power of two below 5 sum |a_i|
    (twenty terms and more), the result is rounded once: within 2^-23 of the
    value plus 2^-38 sum |a_i|."""
    M, J, kmax, R, K, P, shift = shape
    d = synth.make_dictionary(M, J, kmax, 700 + M)
    atom, angle, coef = _codes(P, K, M, R, 800 + P)
    coef[::4] *= 1e-6
    got = _gpu_reconstruct(rsc, d, R, atom, angle, coef, shift)
    ref = ksvd.reconstruct(d, R, atom, angle, coef)
    tol = 2.0 ** -23 * np.abs(ref) + 2.0 ** -38 * np.abs(coef).sum(1)[:, None, None, None]
    assert np.all(np.abs(got - ref) <= tol)
    assert np.all(got[:, 0, :, 1] == 0.0)


def test_reconstruct_weights_out_of_range_and_cancelling(rsc):
    """Weights far from 1 or not finite give what FP64 rounded to float32
    gives; terms that cancel to 1e-9 keep FP64's accuracy (2^-50 of the terms
    here, against 2^-41 of the FP32 accumulator)."""
    M, J, kmax, R, K = 4, 6, 8, 16, 2
    d = synth.make_dictionary(M, J, kmax, 90)
    atom = np.tile(np.array([[1, 2]], np.int32), (9, 1))
    angle = np.tile(np.array([[3, 5]], np.int32), (9, 1))
    coef = np.array([[1e-30, 2e-31], [1e30, -2e29], [1e-300, 1.0], [0.0, 0.0], [np.inf, 1.0],
                     [np.nan, 1.0], [1e200, 1.0], [3e38, 3e38], [1.0, -1.0 + 1e-9]])
    atom[8], angle[8] = 1, 3  # the same steered atom twice: 1e-9 of it is left
    got = _gpu_reconstruct(rsc, d, R, atom, angle, coef)
    fin = [0, 1, 2, 3, 8]
    ref = ksvd.reconstruct(d, R, atom[fin], angle[fin], coef[fin])
    with np.errstate(over="ignore"):
        r32 = ref.astype(np.float32)
    tol = np.spacing(np.abs(r32)).astype(np.float64)
    tol[4] += 2.0 ** -50
    assert np.all(np.abs(got[fin] - ref) <= tol)
    assert np.all(got[3] == 0.0)
    assert np.isnan(got[5][1:]).all() and not np.isfinite(got[4][1:]).any()
    assert np.isinf(got[6][1:]).all()


@pytest.mark.parametrize("shape", [
    # (N, J, kmax, P): four pixels; tiles of 104 pixels; three tiles; partial
    # tiles of 32 and of 128 patches
    (2, 1, 0, 3), (3, 1, 1, 40), (11, 6, 8, 1), (11, 6, 8, 33), (11, 6, 8, 19457 + 128),
    (13, 5, 6, 129), (21, 10, 12, 65), (21, 10, 12, 20000)], ids=str)
def test_synthesize_edges(rsc, shape):
    """n FP32 multiply-adds per pixel: within n 2^-24 sum |X c| (and the
    rounding of X), the imaginary parts of k = 0 ignored."""
    import torch
    N, J, kmax, P = shape
    rng = np.random.default_rng(P)
    c = rng.standard_normal((P, kmax + 1, J, 2)).astype(np.float32)
    c[:, 0, :, 1] = np.nan
    b = rsc.Basis(N, J, kmax)
    got = rsc.synthesize(b, torch.from_numpy(c).cuda()).cpu().numpy()
    b.close()
    c[:, 0, :, 1] = 0.0
    idx = np.unique(np.r_[np.arange(min(P, 64)), np.arange(max(0, P - 160), P)])
    ref = obasis.synthesize(c[idx], N, J, kmax)
    X = np.stack([obasis.synthesize(e, N, J, kmax)[0] for e in
                  np.eye(c[0].size).reshape(-1, 1, kmax + 1, J, 2)])
    X[1:2 * J:2] = 0.0
    bound = np.abs(c[idx].reshape(len(idx), -1)).astype(np.float64) @ np.abs(X)
    n = J * (2 * kmax + 1)
    assert np.all(np.abs(got[idx] - ref) <= (n + 4) * 2.0 ** -24 * bound + 1e-30)
