"""The end of a call: canvas rows to dense images at every alignment of the
destination rows and around the pieces a warp takes (2048 bytes), beside
images that stay untouched; bytes equal to the oracle's."""
import numpy as np
import pytest

from paper_1306_5390_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("rows,cols", [(5, 15), (9, 16), (7, 17), (40, 31), (33, 2047), (12, 2048), (11, 2063),
                                       (9, 2064), (8, 4111), (3, 70)])
@pytest.mark.parametrize("offset", [0, 1, 6, 15])
def test_rows_at_every_alignment(oracle_mod, torch_cuda, rows, cols, offset):
    from paper_1306_5390_gb300 import hgrms
    img = synth.random_image(rows, cols, 100 * rows + cols)
    ref, k_ref, _ = oracle_mod.denoise(img, 3, 1, 3)
    n = rows * cols
    buf = torch_cuda.full((2 * n + 64,), 77, dtype=torch_cuda.uint8, device="cuda")
    with hgrms.Denoiser(0) as d:
        for batch in (False, True):
            buf.fill_(77)
            views = [buf[offset:offset + n].view(rows, cols)]
            if batch:
                views.append(buf[offset + n + 3:offset + 2 * n + 3].view(rows, cols))
            for v in views:
                v.copy_(torch_cuda.from_numpy(img))
            ks = d.denoise_batch(views, 3, 1, 3) if batch else [d.denoise(views[0], 3, 1, 3)]
            assert ks == [k_ref] * len(views)
            for v in views:
                assert np.array_equal(v.cpu().numpy(), ref)
            rest = buf.cpu().numpy().copy()
            rest[offset:offset + n] = 77
            if batch:
                rest[offset + n + 3:offset + 2 * n + 3] = 77
            assert (rest == 77).all()
