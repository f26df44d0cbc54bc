"""The FP32 scoring path where its branches meet: angles in pairs (even R, one
or two a lane) or single (odd R), block sizes for few and for many patches,
lane-parallel factor updates up to K = 16, and runner-ups inside the window
(copies of an atom), which repeat a step's scores with a top-4 a lane."""
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
    # (name, M, J, kmax, R, K, P, copies of each atom)
    ("one_atom_one_angle", 1, 6, 8, 1, 1, 5, 1),
    ("two_angles", 5, 6, 8, 2, 3, 33, 1),
    ("odd_31", 33, 6, 8, 31, 4, 40, 1),
    ("odd_33", 31, 5, 7, 33, 4, 40, 1),
    ("odd_127", 12, 6, 8, 127, 4, 40, 1),
    ("even_62_ragged_chunk", 65, 6, 8, 62, 5, 40, 1),
    ("even_66_two_a_lane", 20, 6, 8, 66, 5, 40, 1),
    ("even_128_kmax12", 20, 10, 12, 128, 5, 40, 1),
    ("even_64_kmax16", 20, 4, 16, 64, 4, 40, 1),
    ("odd_63_kmax16", 20, 4, 16, 63, 4, 40, 1),
    ("kmax0_long", 40, 300, 0, 1, 4, 20, 1),
    ("K16", 40, 6, 8, 32, 16, 40, 1),
    ("many_patches", 8, 6, 8, 32, 3, 2600, 1),
    ("many_patches_K16", 40, 6, 8, 32, 16, 2600, 1),
    ("twins", 40, 6, 8, 64, 4, 40, 2),
    ("twins_odd_R", 40, 6, 8, 33, 4, 40, 2),
    ("six_copies", 48, 6, 8, 64, 3, 40, 6),
]


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_branches(rsc, case):
    _, M, J, kmax, R, K, P, copies = case
    d = synth.make_dictionary(M // copies, J, kmax, 7000 + M + R)
    d = np.concatenate([d] * copies)
    x, _ = synth.make_patches(d, P, min(4, K), 0.1, 8000 + P)
    g = run_gpu(rsc, x, d, R, K, "fp32")
    check(x, d, R, K, g, TOL)
