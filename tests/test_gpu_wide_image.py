"""Projection of images so wide that a window's pixel offsets (row times width
plus column) pass 2^31: the tensor-core kernels' tables hold 32 bits, so such
images take their 64-bit offsets.  One row of windows, 10 GB an image; the
windows at either end and around the middle are those of the image cut there,
bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N, extra", [(11, 12_345), (21, 12_345), (11, -200), (21, -200)])
def test_offsets_past_32_bits(cuda_ok, N, extra):
    import torch
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    # the last offset is (N - 1) w + N - 1: 2^31 lies `extra` columns off
    w = 2 ** 31 // (N - 1) + extra
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 24 GB of device memory")
    b = rsc.Basis(N, 2, 0)  # four floats a window
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    img = torch.empty((N, w), dtype=torch.float32, device="cuda")
    for row in img:
        row.uniform_(-1.0, 1.0, generator=g)
    got = rsc.project(b, img)
    assert got.shape[0] == w - N + 1
    for c in (0, 127, w // 2, w - N + 1 - 300):
        part = rsc.project(b, img[:, c:c + 300 + N - 1].contiguous())
        assert torch.equal(got[c:c + 300], part), c
    b.close()
    del img, got
    torch.cuda.empty_cache()
