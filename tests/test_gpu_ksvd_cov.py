"""Covariances of the K-SVD update (rsc_ksvd_accumulate) at the edges of the
tensor-core kernel: sample counts around its stages of 64 and windows of 320,
several slices of an atom, packed lengths up to 112 and the lengths, angle
counts and scales that the CUDA cores keep."""
import numpy as np
import pytest

from paper_1806_04374_gb300 import synth

from test_oracle_ksvd import _direct_columns

pytestmark = pytest.mark.gpu

# C_m against FP64 numpy, relative to its norm: entries exact to 2^-46 of the
# largest of their row, products to 2^-50, sums in double-float (2^-47 an
# addition, some tens of them): below 2^-40.
TOL = 1e-12

CASES = [
    # (name, M, J, kmax, R, K, P, scale): P samples and more for atom 0
    ("one_sample", 2, 6, 8, 16, 1, 1, 1.0),
    ("stage_less_one", 2, 6, 8, 64, 2, 63, 1.0),
    ("stage", 2, 6, 8, 33, 2, 64, 1.0),
    ("stage_and_one", 2, 6, 8, 64, 2, 65, 1.0),
    ("window", 2, 5, 8, 60, 2, 320, 1.0),
    ("window_and_one", 2, 6, 8, 64, 2, 321, 1.0),
    ("slices", 3, 6, 8, 64, 3, 2700, 1.0),
    ("n112", 2, 16, 3, 32, 2, 200, 1.0),
    ("n112_kmax0", 3, 112, 0, 4, 2, 200, 1.0),
    ("n8", 3, 8, 0, 1, 2, 150, 1.0),
    ("n114_cuda_cores", 2, 6, 9, 32, 2, 150, 1.0),
    ("large_factor_table_cuda_cores", 2, 3, 16, 128, 2, 150, 1.0),
    ("small_scale", 3, 6, 8, 16, 2, 150, 1e-9),
    ("tiny_scale_cuda_cores", 3, 6, 8, 16, 2, 150, 1e-15),
    ("huge_scale_cuda_cores", 3, 6, 8, 16, 2, 150, 1e17),
]


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_covariances(rsc, case):
    import torch
    _, M, J, kmax, R, K, P, scale = case
    rng = np.random.default_rng(P + M)
    d = synth.make_dictionary(M, J, kmax, 300 + P)
    x, _ = synth.make_patches(d, P, 2, 0.1, 400 + P)
    x = (x * scale).astype(np.float32)
    # atom 0 in every patch, at one place or two; the others at random
    atom = np.concatenate([np.zeros((P, 1), np.int32),
                           rng.integers(-1, M - 1, (P, K - 1)).astype(np.int32)], 1)
    angle = np.where(atom < 0, -1, rng.integers(0, R, (P, K))).astype(np.int32)
    coef = np.where(atom < 0, 0.0, rng.standard_normal((P, K)) * scale)
    coef[::5] *= 30.0
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    codes = {"atom": torch.from_numpy(atom).cuda(), "angle_idx": torch.from_numpy(angle).cuda(),
             "coef": torch.from_numpy(coef).cuda()}
    xd = torch.from_numpy(x).cuda()
    out = rsc.ksvd_accumulate(dic, xd, codes, ntop=0)
    again = rsc.ksvd_accumulate(dic, xd, codes, ntop=0)
    torch.cuda.synchronize()
    assert rsc.rsc_dict_check(dic.handle) == 0
    assert torch.equal(out["C"], again["C"])
    C, cnt = out["C"].cpu().numpy(), out["count"].cpu().numpy()
    for m in range(M):
        assert cnt[m] == (atom == m).any(1).sum()
        if cnt[m] == 0:
            assert not C[m].any()
            continue
        Y = _direct_columns(x, d.astype(np.float64), R, atom, angle, coef, m)
        ref = Y @ Y.T
        assert np.linalg.norm(C[m] - ref) <= TOL * np.linalg.norm(ref), m
        assert np.array_equal(C[m], C[m].T)
    dic.close()
