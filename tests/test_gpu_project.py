"""The tensor-core projections at the edges of their tiles: 1 to 129 windows,
padded pixels and outputs of every kind, images of one row or column of
windows, and tiles that span several images of different widths."""
import numpy as np
import pytest

from oracle import basis as obasis
from paper_1806_04374_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsc(cuda_ok):
    import paper_1806_04374_gb300 as rsc
    rsc.load_library()
    return rsc


@pytest.mark.parametrize("case", [
    # (N, J, kmax, window rows, window columns): 9 to 113 pixels, 16 to 128 outputs
    (3, 2, 3, 5, 7), (4, 2, 4, 1, 128), (6, 4, 5, 3, 43), (9, 4, 8, 129, 1), (10, 6, 8, 1, 127),
    (11, 6, 8, 1, 1), (11, 6, 8, 40, 130), (12, 8, 7, 2, 64),
    # 137 to 489 pixels: 3 to 8 K-blocks, the last one of 9 to 61 pixels
    (13, 6, 8, 1, 1), (13, 6, 8, 3, 43), (16, 8, 10, 1, 129), (21, 10, 12, 12, 150), (25, 10, 12, 129, 1),
], ids=str)
def test_project_tiles(rsc, case):
    """fp16 hi + lo products summed in FP32: every product is off by 2^-21 at
    most (two operands to 2^-22, lo * lo left out), every one of the 3 npix / 16
    accumulations by 2^-22 of the sum of moduli."""
    import torch
    N, J, kmax, nr, nc = case
    rng = np.random.default_rng(100 * N + nc)
    img = (rng.standard_normal((nr + N - 1, nc + N - 1)) *
           np.exp2(rng.integers(-6, 7, (nr + N - 1, 1)))).astype(np.float32)
    b = rsc.Basis(N, J, kmax)
    got = rsc.project(b, torch.from_numpy(img).cuda()).cpu().numpy()
    ref = obasis.project(img, N, J, kmax)
    assert got.shape == ref.shape
    # moduli: the operator's columns from the projections of single pixels
    rows, cols = np.divmod(np.arange(N * N), N)
    op = np.stack([obasis.project(e, N, J, kmax)[0] for e in np.eye(N * N).reshape(-1, N, N)])
    win = np.stack([img[r:r + nr, c:c + nc].ravel() for r, c in zip(rows, cols)], 1)
    bound = np.abs(win).astype(np.float64) @ np.abs(op).reshape(N * N, -1)
    tol = (2.0 ** -20 + (3 * b.npix / 16 + 8) * 2.0 ** -22) * bound
    assert np.all(np.abs(got - ref).reshape(bound.shape) <= tol)
    b.close()


@pytest.mark.parametrize("shape", [(11, 6, 8), (21, 10, 12)], ids=str)
def test_tiles_across_images_code_like_single_images(rsc, shape):
    """A window's coefficients do not depend on the tile that it falls in: the
    codes of many small images in one call (tiles of several images and
    widths) are those of the images projected alone, bit for bit."""
    import torch
    N, J, kmax = shape
    rng = np.random.default_rng(N)
    sizes = [(N, N), (N + 3, N + 40), (N - 1, 50), (N + 200, N), (N + 12, N + 12), (N, N + 300),
             (N + 1, N + 2)] + [(N + int(h), N + int(w)) for h, w in rng.integers(0, 9, (30, 2))]
    imgs = [torch.from_numpy(synth.make_line_image(h, w, 0.02, 900 + i)).cuda()
            for i, (h, w) in enumerate(sizes)]
    dic = rsc.Dictionary(torch.from_numpy(synth.make_dictionary(12, J, kmax, 17)).cuda(), 16)
    b = rsc.Basis(N, J, kmax)
    got = rsc.encode_images(dic, b, imgs, 3, "f16")
    x = torch.cat([rsc.project(b, im) for im in imgs])
    ref = rsc.encode(dic, x, 3, "f16")
    for k in ref:
        assert torch.equal(got[k], ref[k]), k
    dic.close()
    b.close()
