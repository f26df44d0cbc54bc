"""A wait of the K-SVD covariance kernel that runs out (1 ns, set by
rsc_dict_set_limits) without faulting the GPU: rsc_dict_check reports it, the
covariance is not a number instead of an unfinished sum, rksvd.learn raises
before a checkpoint is written, and the next call with the default limit is
right again."""
import os

import pytest

from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(cuda_ok):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    M, R, K, P = 5, 16, 2, 2000
    d = torch.from_numpy(synth.make_dictionary(M, 6, 8, 51)).cuda()
    x = torch.from_numpy(synth.make_patches(d.cpu().numpy(), P, 2, 0.1, 52)[0]).cuda()
    dic = rsc.Dictionary(d, R)
    codes = rsc.encode(dic, x, K, "fp32")
    yield rsc, dic, d, x, codes, R, K
    dic.close()


def test_covariance_timeout_is_reported_and_marked(case):
    import torch
    rsc, dic, d, x, codes, R, K = case
    good = rsc.ksvd_accumulate(dic, x, codes, ntop=0)
    assert rsc.rsc_dict_check(dic.handle) == 0
    assert rsc.rsc_dict_set_limits(dic.handle, 1, 0) == 0
    bad = rsc.ksvd_accumulate(dic, x, codes, ntop=0)
    assert rsc.rsc_dict_check(dic.handle) == rsc.RSC_ERR_TIMEOUT
    assert rsc.rsc_dict_check(dic.handle) == 0
    # every atom's covariance is whole or not a number throughout
    lost = [bool(torch.isnan(c).all()) for c in bad["C"]]
    assert any(lost)
    for m, gone in enumerate(lost):
        assert gone or torch.equal(bad["C"][m], good["C"][m])
    new, _ = rsc.ksvd_update(dic, x, codes)
    assert rsc.rsc_dict_check(dic.handle) == rsc.RSC_ERR_TIMEOUT
    assert torch.isnan(new).any()
    with pytest.raises(rsc.RscError):  # such atoms make no dictionary
        rsc.Dictionary(new, R)
    assert rsc.rsc_dict_set_limits(dic.handle, 0, 0) == 0
    again = rsc.ksvd_accumulate(dic, x, codes, ntop=0)
    assert rsc.rsc_dict_check(dic.handle) == 0
    assert torch.equal(again["C"], good["C"])


def test_learning_raises_before_the_checkpoint(case, monkeypatch, tmp_path):
    rsc, _, d, x, _, R, K = case
    from paper_1806_04374_gb300 import rksvd

    class Hurried(rsc.Dictionary):
        def __init__(self, *a):
            super().__init__(*a)
            rsc.rsc_dict_set_limits(self.handle, 1, 0)

    monkeypatch.setattr(rksvd, "Dictionary", Hurried)
    ck = str(tmp_path / "c.npz")
    with pytest.raises(rsc.RscError) as e:
        rksvd.learn(x, d, R, K, 2, precision="fp32", checkpoint=ck)
    assert e.value.status == rsc.RSC_ERR_TIMEOUT
    assert not os.path.exists(ck)
