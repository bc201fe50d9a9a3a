"""The register-streaming forward kernel (2-D and 3-D grids of any shape, FP32) where its geometry has
edges: rows of two cells to a few warps (odd rows' last pair overlaps the one before), fewer rows than a
strip holds and ragged last strips, two and three slices, every wall type on every axis, a periodic
jump, and a number of directions its parts do not divide, against the FP64 oracle on the state, T_L and
the wall values (which the second step reads).  The tolerance is the parity tests', 1e-5 relative
L-inf."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import fused_TL, gpu_ctx, oracle_problem, rel_linf, run_both, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3
TW = [0.3, -0.2, 0.1, 0.4, -0.3, 0.2]
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


GRIDS = [
    (2, (2, 2, 1), [ISO, DIF, SPE, ISO, PER, PER]),
    (2, (3, 3, 1), [DIF, SPE, ISO, DIF, PER, PER]),
    (2, (5, 4, 1), [PER, PER, DIF, SPE, PER, PER]),
    (2, (66, 5, 1), [SPE, ISO, PER, PER, PER, PER]),
    (2, (131, 9, 1), [DIF, DIF, DIF, DIF, PER, PER]),
    (3, (2, 3, 2), [SPE, SPE, DIF, ISO, ISO, DIF]),
    (3, (7, 2, 3), [ISO, DIF, PER, PER, SPE, SPE]),
    (3, (34, 5, 3), [PER, PER, SPE, DIF, DIF, ISO]),
    (3, (67, 6, 5), [DIF, SPE, ISO, SPE, PER, PER]),
    (3, (64, 9, 4), [SPE, ISO, DIF, DIF, SPE, DIF]),
]


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("dim,n,bc", GRIDS)
def test_stream_fp32(dim, n, bc, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=3, quad=("octant", 3, 3))
    P = oracle_problem(cfg, limiter)
    e0 = inputs.random_state(P.shape, 41) * 1e4
    Q = (np.random.default_rng(3).random((P.nz, P.ny, P.nx)) * 1e17).astype(np.float32)
    amps = np.linspace(1.0, 0.3, 4)
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 4, Q, amps, limiter=limiter, kernel=bte.BTE_KERNEL_GENERIC)
    assert ctx.info.kernel == bte.BTE_KERNEL_GENERIC
    assert rel_linf(g, eo) <= TOL and rel_linf(gTL, oTL) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


@pytest.mark.parametrize("dim,n,axis", [(2, (6, 7, 1), 0), (2, (35, 5, 1), 1), (3, (8, 5, 6), 2)])
def test_stream_periodic_jump(dim, n, axis):
    from paper_2306_14181_gb300 import bte
    bc = [PER, PER] + [DIF, ISO] * 2
    bc[2 * axis] = bc[2 * axis + 1] = PER
    for a in range(dim, 3):
        bc[2 * a] = bc[2 * a + 1] = PER
    jump = [0.0, 0.0, 0.0]
    jump[axis] = 0.7
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=2, jump=jump)
    P = oracle_problem(cfg)
    e0 = inputs.random_state(P.shape, 43) * 1e4
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 3, kernel=bte.BTE_KERNEL_GENERIC)
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


def test_stream_repeats_bitwise():
    """Strips and pairs that overlap are computed twice: the same bits every time."""
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(3, (37, 6, 5), [DIF, SPE, ISO, DIF, DIF, ISO], Tw=TW, nb=3)
    P = oracle_problem(cfg)
    e0 = (inputs.random_state(P.shape, 44) * 1e4).astype(np.float32)
    out = []
    for _ in range(2):
        ctx = gpu_ctx(cfg, kernel=bte.BTE_KERNEL_GENERIC)
        bte.bte_set_state(ctx, e0)
        bte.bte_step(ctx, 5)
        out.append((bte.bte_get_state(ctx).copy(), bte.bte_lattice_temperature(ctx).copy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
