"""The FP32 path with an odd number of angles up to 31 (one angle a lane) in
blocks of 8 and of 20 warps, with copies of atoms, pruned, and as the hand-off
of the FP16 path."""
import numpy as np
import pytest

from paper_1806_04374_gb300 import synth

from parity import check
from test_gpu_parity import run_gpu

pytestmark = pytest.mark.gpu

# as in the other tests of this path: double-float inner products, condition
# numbers below 10^4
TOL = 1e-9


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


@pytest.mark.parametrize("case", [
    # (M, J, kmax, R, K, P, copies of each atom, precision)
    (33, 6, 8, 31, 4, 40, 1, "fp32"), (33, 6, 8, 31, 4, 2600, 1, "fp32"),
    (65, 5, 7, 15, 5, 40, 1, "fp32"), (7, 6, 8, 1, 3, 2600, 1, "fp32"), (40, 6, 8, 17, 16, 40, 1, "fp32"),
    (40, 6, 8, 31, 4, 40, 2, "fp32"), (48, 6, 8, 15, 3, 40, 6, "fp32"),
    (33, 6, 8, 31, 4, 40, 1, "fp32_prune"), (40, 6, 8, 31, 4, 40, 8, "f16"),
], ids=str)
def test_odd_angles(rsc, case):
    M, J, kmax, R, K, P, copies, precision = case
    d = synth.make_dictionary(M // copies, J, kmax, 7100 + M + R)
    d = np.concatenate([d] * copies)
    x, _ = synth.make_patches(d, P, min(4, K), 0.1, 8100 + P)
    g = run_gpu(rsc, x, d, R, K, precision)
    check(x, d, R, K, g, TOL)


@pytest.mark.parametrize("R", [31, 33, 64, 128])
def test_codes_do_not_depend_on_the_patches_before(rsc, R):
    """A warp chooses the pass over the scores by its last step: patches near
    pairs of equal atoms and others, in turn, in reverse and apart, are coded
    the same, bit for bit."""
    import torch
    d = synth.make_dictionary(24, 6, 8, 7300)
    d = np.concatenate([d, d[:8]])
    P = 8000
    near, _ = synth.make_patches(d[:8], P, 2, 0.05, 7301)
    far, _ = synth.make_patches(d[8:24], P, 2, 0.05, 7302)
    x = torch.from_numpy(np.where((np.arange(P) % 7 < 3)[:, None, None, None], near, far)).cuda()
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    got = rsc.encode(dic, x, 3, "fp32")
    back = rsc.encode(dic, x.flip(0).contiguous(), 3, "fp32")
    part = rsc.encode(dic, x[:500].contiguous(), 3, "fp32")
    for k in got:
        assert torch.equal(got[k], back[k].flip(0)), k
        assert torch.equal(got[k][:500], part[k]), k
    dic.close()
