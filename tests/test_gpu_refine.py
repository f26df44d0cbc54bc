"""The FP16 path's per-patch kernels at the edges of their layouts: warps of
32 patches with a ragged end, rows of 112 and 256 slots, steered rows stored
for half the angles (even R) or all of them (odd R), and dictionaries whose
Gram table is too large to be kept (entries computed per harmonic)."""
import numpy as np
import pytest

from paper_1806_04374_gb300 import synth

from parity import check
from test_gpu_parity import run_gpu

pytestmark = pytest.mark.gpu

# The weights solve a K x K system whose entries are double-float inner
# products (2^-44 relative); random atoms keep its condition number below
# 10^4, so they agree with the oracle's FP64 weights to 2^-44 10^4 < 1e-9.
TOL = 1e-9

CASES = [
    # (name, M, J, kmax, R, K, P)
    ("paired_one_patch", 16, 6, 8, 32, 5, 1),
    ("paired_K8_ragged_warp", 16, 6, 8, 32, 8, 33),
    ("paired_no_gram_table", 760, 6, 8, 60, 3, 31),
    # odd-harmonic half over 48 slots: plain rows, even R (odd slots change sign)
    ("plain_even_R_odd_J", 12, 5, 9, 16, 8, 65),
    ("plain_odd_R_K8", 12, 6, 8, 33, 8, 63),
    ("plain_no_gram_table", 760, 6, 8, 61, 3, 31),
    ("long_even_R_K8", 20, 10, 12, 32, 8, 129),
    ("long_odd_R_odd_J", 20, 7, 16, 15, 6, 34),
    ("long_kmax0", 30, 130, 0, 4, 4, 33),
]


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_layout_edges(rsc, case):
    _, M, J, kmax, R, K, P = case
    d = synth.make_dictionary(M, J, kmax, 5000 + M + R)
    x, _ = synth.make_patches(d, P, 4, 0.1, 6000 + P)
    x[:, 0, :, 1] = np.nan  # the imaginary parts of k = 0 are ignored
    g = run_gpu(rsc, x, d, R, K, "f16")
    x[:, 0, :, 1] = 0.0
    check(x, d, R, K, g, TOL)


@pytest.mark.parametrize("J,kmax,R", [(6, 8, 32), (6, 8, 33), (10, 12, 16)],
                         ids=["paired", "plain", "long"])
def test_patches_of_a_warp(rsc, J, kmax, R):
    """32 patches a warp, or 4 to 28 in small calls: the same bits."""
    import torch
    d = synth.make_dictionary(9, J, kmax, 77)
    x, _ = synth.make_patches(d, 80_000, 3, 0.1, 78)
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    xd = torch.from_numpy(x).cuda()
    whole = rsc.encode(dic, xd, 3, "f16")
    for lo, hi in ((0, 1), (1, 1000), (1000, 13_200), (13_200, 80_000)):
        part = rsc.encode(dic, xd[lo:hi].contiguous(), 3, "f16")
        for k, v in part.items():
            assert torch.equal(v, whole[k][lo:hi]), (k, lo)
    dic.close()
