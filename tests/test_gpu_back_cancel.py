"""rsc_reconstruct where an entry's terms cancel: down to 2^-30 of the sum of
weights, on both sides of the kernel's line between its FP32 accumulators and
FP64, an entry is its FP64 value rounded to FP32.  Patches without a code and
with weights below FP32's range are zeros."""
import numpy as np
import pytest

from oracle import ksvd
from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(d, R, atom, angle, coef):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), R)
    got = rsc.reconstruct(dic, {"atom": torch.from_numpy(atom).cuda(),
                                "angle_idx": torch.from_numpy(angle).cuda(),
                                "coef": torch.from_numpy(coef).cuda()}).cpu().numpy()
    dic.close()
    return got


@pytest.mark.parametrize("K, J, kmax, R", [(2, 6, 8, 64), (5, 6, 8, 64), (16, 6, 8, 32), (8, 5, 9, 33)])
def test_cancelling_entries(cuda_ok, K, J, kmax, R):
    M, P = 12, 3000
    rng = np.random.default_rng(K)
    d = synth.make_dictionary(M, J, kmax, 40 + K)
    atom = np.stack([rng.choice(M, K, replace=K > M) for _ in range(P)]).astype(np.int32)
    angle = rng.integers(0, R, (P, K)).astype(np.int32)
    coef = rng.standard_normal((P, K))
    # one entry of every patch is brought to `target` by its last weight
    k, j = rng.integers(1, kmax + 1, P), rng.integers(0, J, P)
    c = rng.integers(0, 2, P)
    part = ksvd.reconstruct(d, R, atom[:, :-1], angle[:, :-1], coef[:, :-1])
    last = ksvd.reconstruct(d, R, atom[:, -1:], angle[:, -1:], np.ones((P, 1)))
    at = (np.arange(P), k, j, c)
    target = np.exp2(-rng.uniform(8, 30, P)) * np.abs(coef).sum(1) * rng.choice([-1, 1], P)
    with np.errstate(divide="ignore"):
        w = (target - part[at]) / last[at]
    ok = np.abs(w) < 8.0
    coef[ok, -1] = w[ok]
    assert ok.sum() > P // 2
    got = _run(d, R, atom, angle, coef)
    ref = ksvd.reconstruct(d, R, atom, angle, coef)
    small = np.abs(ref[at]) / np.abs(coef).sum(1)
    for lo, hi in [(-12, -10), (-16, -14), (-20, -18), (-24, -22), (-28, -26)]:
        assert ((small > 2.0 ** lo) & (small < 2.0 ** hi)).sum() > 50
    # one rounding to FP32 (2^-24) and 2^-27 of the entry, the bound of the
    # accumulators at their line; the FP64 sums themselves 2^-49 of the weights
    tol = (2.0 ** -24 + 2.0 ** -27) * np.abs(ref) + 2.0 ** -49 * np.abs(coef).sum(1)[:, None, None, None]
    assert np.all(np.abs(got - ref) <= tol)


def test_nothing_coded(cuda_ok):
    d = synth.make_dictionary(5, 6, 8, 77)
    atom = np.full((40, 3), -1, np.int32)
    coef = np.zeros((40, 3))
    atom[20:, 1] = 2
    coef[20:30, 1] = 1e-60  # below FP32
    got = _run(d, 16, atom, np.where(atom < 0, -1, 3).astype(np.int32), coef)
    assert np.all(got == 0.0)
