"""The covariance of many equal columns with the largest slices that there
are, where every window's sums of order 3 pass 2^24: nothing of them is lost.
Columns are the patches themselves (weight 0, one angle, harmonic 0 alone), so
that C is known exactly."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _value(b0, b1, b2, b3):
    """b0 2^-8 + b1 2^-16 + b2 2^-24 + b3 2^-32, a float32 (b3 0 or 128)."""
    v = np.float32(b0 / 2.0 ** 8 + b1 / 2.0 ** 16 + b2 / 2.0 ** 24 + b3 / 2.0 ** 32)
    assert Fraction(float(v)) == Fraction(b0, 2 ** 8) + Fraction(b1, 2 ** 16) + \
        Fraction(b2, 2 ** 24) + Fraction(b3, 2 ** 32)
    return v


@pytest.mark.parametrize("P", [319, 960, 1000])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20])
def test_equal_columns(cuda_ok, P, scale):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    J = 4
    # 64,000 units of order 3 a sample and more, 320 of them 2.05e7; one column
    # in 64 makes the sums off the diagonal odd
    col = [_value(127, 127, 126, 128), _value(126, 127, 126, 128), _value(-127, -127, -126, -128),
           _value(127, 126, 126, 128)]
    odd = [_value(121, 1, 2, 0), _value(3, 5, 99, 0), _value(-7, 121, 4, 0), _value(5, -78, 1, 0)]
    x = np.zeros((P, 1, J, 2), np.float32)
    x[:, 0, :, 0] = np.where((np.arange(P) % 64 == 61)[:, None], odd, col)
    x *= np.float32(scale)
    d = np.zeros((1, 1, J, 2), np.float32)
    d[0, 0, :, 0] = 0.5
    dic = rsc.Dictionary(torch.from_numpy(d).cuda(), 1)
    zero = torch.zeros((P, 1), dtype=torch.int32, device="cuda")
    C = rsc.ksvd_accumulate(dic, torch.from_numpy(x).cuda(), {
        "atom": zero, "angle_idx": zero, "coef": zero.double()}, ntop=0)["C"][0].cpu().numpy()
    dic.close()
    y = [[Fraction(float(v)) for v in r] for r in x[:, 0, :, 0]]
    for i in range(J):
        for j in range(J):
            ref = sum(r[i] * r[j] for r in y)
            # slices are exact here, products kept down to 2^-53, the rest of
            # the sums (2^-30 of the whole) in FP32: 2^-49 with the last rounding
            assert abs(Fraction(float(C[i, j])) - ref) <= abs(ref) * Fraction(1, 2 ** 49), (i, j)


@pytest.mark.parametrize("P", [1, 65, 321])
def test_every_slice_counts(cuda_ok, P):
    """Columns sqrt(2) x (weight 0, one angle): 48 bits each, cut into six
    slices of 8.  A column is off by 2^-46 of itself (double-float: the product
    with sqrt(2) 2^-47, its constant 2^-48) and its slices by 2^-48 of its row's
    largest, so C by 2^-45 of the sum of moduli and 2^-47 of the products of the
    largest; one slice left out shows 2^-42."""
    import torch
    import paper_1806_04374_gb300 as rsc
    from oracle import ksvd
    from paper_1806_04374_gb300 import synth
    rsc.load_library()
    J, kmax = 6, 8
    x = np.random.default_rng(P).standard_normal((P, kmax + 1, J, 2)).astype(np.float32)
    x[:, 0, :, 1] = 0.0
    dic = rsc.Dictionary(torch.from_numpy(synth.make_dictionary(1, J, kmax, 3)).cuda(), 1)
    zero = torch.zeros((P, 1), dtype=torch.int32, device="cuda")
    C = rsc.ksvd_accumulate(dic, torch.from_numpy(x).cuda(), {
        "atom": zero, "angle_idx": zero, "coef": zero.double()}, ntop=0)["C"][0].cpu().numpy()
    dic.close()
    y = ksvd.pack(x)
    a, most = np.abs(y), np.abs(y).max(0)
    tol = 2.0 ** -45 * (a.T @ a) + 2.0 ** -47 * P * np.outer(most, most)
    assert np.all(np.abs(C - y.T @ y) <= tol)
