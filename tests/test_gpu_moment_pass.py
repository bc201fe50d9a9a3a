"""The moment pass of an uploaded FP32 state: T_L has the bits of the sum over the directions in order, for
every cell count and every wall, in 2-D and 3-D as in 1-D (whose pass takes a thread a cell and band): a
1-D context with the same directions, fed one row, is the reference.  The wall values are compared through
the next step of the generic update, at the parity tests' 1e-5."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import fused_TL, gpu_ctx, oracle_problem, rel_linf, run_both, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("dim,n,bc,quad", [(2, (3, 3, 1), [DIF, DIF, DIF, DIF, PER, PER], (1, 1)),
                                           (2, (96, 40, 1), [SPE, DIF, DIF, ISO, PER, PER], (2, 3)),
                                           (2, (37, 29, 1), [DIF, ISO, PER, PER, PER, PER], (3, 3)),
                                           (3, (7, 6, 5), [DIF, DIF, DIF, DIF, DIF, DIF], (2, 2)),
                                           (3, (9, 5, 7), [PER, PER, DIF, SPE, ISO, DIF], (3, 2))])
def test_lattice_temperature_bits(dim, n, bc, quad):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, nb=3, quad=("octant",) + quad)
    P = oracle_problem(cfg)
    e = (inputs.random_state(P.shape, 81) * 1e4).astype(np.float32)
    ctx = gpu_ctx(cfg)
    bte.bte_set_state(ctx, e)
    TL = fused_TL(ctx)
    s, w = bte.bte_get_quadrature(ctx)
    line = dict(cfg, dim=1, n=(P.ncell, 1, 1), quad=("explicit", s, w), bc=[ISO, ISO] + [PER] * 4)
    one = gpu_ctx(line, kernel=bte.BTE_KERNEL_GENERIC)
    bte.bte_set_state(one, e.reshape(P.nb, P.nd, 1, 1, P.ncell))
    assert np.array_equal(TL.reshape(-1), fused_TL(one).reshape(-1))
    # the diffuse-wall values of the upload, which one step reads
    ctx, g, gTL, eo, oTL = run_both(cfg, e, 1)
    assert rel_linf(g, eo) <= 1e-5
