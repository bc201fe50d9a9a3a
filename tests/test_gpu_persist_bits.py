"""The persistent kernel's bits: digests of the state and T_L after 20 steps with a source, by every wall, for one band a
block and several, rows off and on its groups of four.  Up to 16 bands they are those of the kernel that keeps bare
rows, one cell a thread (which still runs where the padded rows do not fit)."""
import hashlib

import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import gpu_ctx, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


DIGESTS = {  # (cells, bands, directions): by limiter
    (6, 40, 8): ("8df1810f5b827bbe", "d1503039ad142521", "ab0bf013df262eb1"),
    (37, 3, 10): ("ec968f64084732f1", "bd0d52cce1813f39", "ba206866e291771e"),
    (100, 10, 16): ("44d6e17052e956d9", "b9bbd17857364fbb", "269636a5cc863961"),
    (130, 17, 8): ("faaf2d2ad1a656a1", "4c9e072e09dd2c3e", "5a006574265dc75e"),
    (600, 1, 16): ("0e5eb36b19926b1b", "510c11422aded205", "46f29c2219c49d5b"),
}
WALLS = {100: [DIF, ISO], 37: [SPE, DIF], 130: [PER, PER], 6: [DIF, DIF], 600: [ISO, SPE]}


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("nx,nb,nd", sorted(DIGESTS))
def test_persistent_bits(nx, nb, nd, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(1, (nx, 1, 1), WALLS[nx] + [PER] * 4, Tw=[0.3, -0.2, 0, 0, 0, 0], nb=nb, quad=("gl1d", nd))
    ctx = gpu_ctx(cfg, limiter=limiter, kernel=bte.BTE_KERNEL_PERSISTENT)
    rng = np.random.default_rng(5)
    bte.bte_set_state(ctx, (inputs.random_state(ctx.shape, 63) * 1e4).astype(np.float32))
    bte.bte_set_source(ctx, (rng.random((1, 1, nx)) * 1e17).astype(np.float32), np.linspace(1.0, 0.3, 20))
    bte.bte_step(ctx, 20)
    h = hashlib.sha256(bte.bte_get_state(ctx).tobytes() + bte.bte_lattice_temperature(ctx).tobytes())
    assert h.hexdigest()[:16] == DIGESTS[nx, nb, nd][limiter]
