"""Thread counts of the persistent kernel: more wall tasks than cells, and rows beyond 512 cells, against the oracle
at the parity tests' 1e-5."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import fused_TL, oracle_problem, rel_linf, run_both, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("nx,bc,nb,nd", [(5, [DIF, SPE], 100, 8), (2, [ISO, DIF], 40, 64), (4, [PER, PER], 100, 16),
                                         (8, [DIF, DIF], 17, 64), (513, [DIF, ISO], 2, 16), (580, [SPE, DIF], 1, 8),
                                         (802, [PER, PER], 1, 16)])
def test_persistent_threads(nx, bc, nb, nd):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(1, (nx, 1, 1), bc + [PER] * 4, Tw=[0.3, -0.2, 0, 0, 0, 0], nb=nb, quad=("gl1d", nd))
    P = oracle_problem(cfg)
    e0 = inputs.random_state(P.shape, 63) * 1e4
    Q = (np.random.default_rng(3).random((1, 1, nx)) * 1e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 5, Q, np.linspace(1.0, 0.3, 5), kernel=bte.BTE_KERNEL_PERSISTENT)
    assert rel_linf(g, eo) <= 1e-5 and rel_linf(fused_TL(ctx), oTL) <= 1e-5
