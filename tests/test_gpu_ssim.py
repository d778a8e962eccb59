"""The separable FP64 SSIM kernel at the edges of its 128-column blocks and of
its rows per block, against the plain FP64 window sums."""
import numpy as np
import pytest

from oracle import metrics
from pcad_inputs import greyscale_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


# the window just fits; one block of columns and one more; a remainder; tall
@pytest.mark.parametrize("H,W", [(11, 11), (11, 138), (12, 139), (300, 14), (77, 395),
                                 (600, 1100)])
def test_ssim_at_block_edges(pc, H, W):
    rng = np.random.default_rng(H + W)
    L = 256
    clean = greyscale_scene(H, H, W, L, n_shapes=5)
    est = np.clip(clean + rng.normal(0, 15.0, (H, W)), 0, L - 1).astype(np.float32)
    psnr, ssim = pc.pcad_metrics(est, clean, L)
    # FP64 sums of 121 products of values in [0, 1] and one division: 1e-12 each side
    assert abs(ssim - metrics.ssim(est.astype(np.float64), clean, L)) < 1e-11
    assert abs(psnr - metrics.psnr(est.astype(np.float64), clean, L)) < 1e-9
