"""The coding errors of the K-SVD update at and past the ends of FP32's range:
the list of largest-error patches (rsc_ksvd_accumulate) holds the FP64 sum
rounded once to float32, infinity where it does not fit, and orders the
patches by it, so that the reset of an unused atom takes the same patch as in
FP64."""
import numpy as np
import pytest

from oracle import ksvd
from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J, kmax", [(6, 8), (1, 0), (10, 12)])
@pytest.mark.parametrize("scales", [
    # about 1: the FP32 path; past FLT_MAX for some; subnormal; zero
    [1.0, 3.0, 0.5, 2.0], [1.0, 1e25, 1e18, 1e30], [1e-19, 1.01e-19, 1e-21, 2e-22],
    [0.0, 1e-23, 0.0, 1.0]], ids=str)
def test_largest_coding_errors(cuda_ok, J, kmax, scales):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    P, R, M = 64, 8, 3
    d = synth.make_dictionary(M, J, kmax, 60)
    x = synth.make_patches(d, P, 2, 0.1, 61)[0].astype(np.float64)
    x = (x * np.resize(scales, P)[:, None, None, None]).astype(np.float32)
    # half the patches uncoded, half coded with a tenth of their size
    atom = np.where(np.arange(P)[:, None] < P // 2, -1, 1).astype(np.int32)
    angle = np.where(atom < 0, -1, 3).astype(np.int32)
    coef = np.where(atom < 0, 0.0, 0.1 * np.resize(scales, P)[:, None])
    res = x.astype(np.float64) - ksvd.reconstruct(d, R, atom, angle, coef)
    err = (ksvd.pack(res) ** 2).sum(1)
    with np.errstate(over="ignore"):
        want = err.astype(np.float32)
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    codes = {"atom": torch.from_numpy(atom).cuda(), "angle_idx": torch.from_numpy(angle).cuda(),
             "coef": torch.from_numpy(coef).cuda()}
    acc = rsc.ksvd_accumulate(dic, torch.from_numpy(x).cuda(), codes)
    top, idx = acc["top_err"].cpu().numpy(), acc["top_idx"].cpu().numpy()
    assert sorted(idx.tolist()) == list(range(P))
    # residuals in double-float (2^-44), the sum rounded once (2^-24, half a
    # unit of the subnormals)
    exact = err[idx]
    fin = np.isfinite(want[idx])
    assert np.array_equal(np.isinf(top), ~fin)
    assert np.all(np.abs(top[fin] - exact[fin]) <= exact[fin] * (2.0 ** -24 + 2.0 ** -40) + 2.0 ** -150)
    key = np.where(np.isinf(top), np.inf, top)
    assert np.all(key[:-1] >= key[1:])
    same = key[:-1] == key[1:]
    assert np.all(idx[:-1][same] < idx[1:][same])
    dic.close()
