"""rsc_synthesize in small calls (a thread per output) and in tiles: the same
pixels, bit for bit, on both sides of the line between them."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(11, 6, 8), (21, 10, 12), (9, 5, 8), (33, 6, 8), (10, 5, 8), (5, 2, 2)], ids=str)
def test_small_calls_equal_tiles(cuda_ok, shape):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    N, J, kmax = shape
    b = rsc.Basis(N, J, kmax)
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    line = 256 * nsm // b.npix
    c = torch.randn((line + 40, kmax + 1, J, 2), device="cuda")
    c[:, 0, :, 1] = float("nan")  # ignored
    whole = rsc.synthesize(b, c)
    assert torch.isfinite(whole).all()
    for P in (1, 7, line, line + 1):
        assert torch.equal(rsc.synthesize(b, c[:P].contiguous()), whole[:P]), P
    b.close()
