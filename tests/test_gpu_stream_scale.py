"""The streaming step has no size of its own: without a source and with walls at 0 K a state scaled by a power of
two steps to the scaled result, bit for bit, down to slopes near 1e-12, where the products of the limiter are
still normal numbers (a regularisation of van Albada's denominator may not reach them)."""
import numpy as np
import pytest

from tests.support import fused_TL, gpu_ctx, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, (37, 21, 1), [DIF, SPE, ISO, DIF, PER, PER]),
                                      (2, (34, 8, 1), [PER, PER, SPE, ISO, PER, PER]),
                                      (3, (13, 9, 6), [SPE, ISO, PER, PER, DIF, SPE])])
def test_scaled_state(dim, n, bc, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, nb=3)
    out = []
    for scale in (1.0, 2.0 ** -41):
        ctx = gpu_ctx(cfg, limiter=limiter, kernel=bte.BTE_KERNEL_GENERIC)
        z, y, x = np.meshgrid(*(np.arange(m) for m in n[::-1]), indexing="ij")
        f = 1.0 + np.random.default_rng(3).random(ctx.shape[:2])[..., None, None, None]
        # differences of one to a few times the scale along every axis, curved enough to limit
        e = f * (10 + 1.1 * x + 1.3 * y + 1.2 * z + 0.04 * (x + y + z) ** 2)
        bte.bte_set_state(ctx, e.astype(np.float32) * np.float32(scale))
        TL0 = fused_TL(ctx).copy()
        bte.bte_step(ctx, 1)
        out.append([a.astype(np.float64) / scale for a in (TL0, bte.bte_get_state(ctx), fused_TL(ctx))])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
