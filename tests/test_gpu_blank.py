"""Patches of zeros (blank windows) among others: no code, no error and no
hand-off, whatever the dictionary's size; patches whose squares underflow or with
a not-a-number are no blank ones."""
import numpy as np
import pytest

from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M, J, kmax, R", [(16, 6, 8, 16), (64, 6, 8, 64), (16, 6, 8, 33), (16, 10, 12, 32)])
def test_blank_patches(cuda_ok, M, J, kmax, R):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    P = 300
    d = synth.make_dictionary(M, J, kmax, 5)
    x = torch.from_numpy(synth.make_patches(d, P, 2, 0.1, 6)[0]).cuda()
    i = torch.arange(P, device="cuda")
    blank = (i % 3 == 1) | (i >= 200) & (i < 240)
    x[blank] = 0.0
    x[blank, 0, :, 1] = 7.0  # the imaginary parts of k = 0 are ignored
    tiny = (i % 30 == 3) & ~blank
    x[tiny] *= 1e-30
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    rsc.rsc_dict_fallback_count(dic.handle)
    got = rsc.encode(dic, x, 3, "f16")
    torch.cuda.synchronize()
    assert rsc.rsc_dict_check(dic.handle) == 0
    assert rsc.rsc_dict_fallback_count(dic.handle) < P // 10  # (100 and more blank ones)
    assert (got["atom"][blank] == -1).all() and (got["angle_idx"][blank] == -1).all()
    for k in ("angle", "coef", "resid_norm2"):
        assert (got[k][blank] == 0).all(), k
    # the others as in a call without blank patches
    rest = rsc.encode(dic, x[~blank].contiguous(), 3, "f16")
    for k in got:
        assert torch.equal(got[k][~blank], rest[k]), k
    assert (got["atom"][tiny][:, 0] >= 0).all()
    x[1, 2, 1, 0] = float("nan")
    assert torch.isnan(rsc.encode(dic, x, 3, "f16")["resid_norm2"][1])
    dic.close()
