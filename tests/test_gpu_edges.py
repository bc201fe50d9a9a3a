"""Edge sizes of the kernels that split their work by size: the FP64 moments (three direction rules,
storages, cell counts off the block), the moment pass and the implicit sweep (rows of one and two
register chunks and longer, odd rows), the 1-D forward kernels (two cells up, bands and directions off
the block), the persistent film kernel (rows off its groups of four, more bands than CTAs, a state only
its flat form fits), and the tiled kernel's rows shorter than its instance and next to specular x walls.
Tolerances are those of the parity tests: 1e-5 relative L-inf for FP32 states, 2e-3 on T_L for 16-bit
codes, 1e-12 for FP64 sums over an FP32 state (a 16-bit state is read back in FP32: 2^-24 a value, summed
with weights of one sign, 1e-6 of the largest)."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import fused_TL, gpu_ctx, oracle_problem, rel_linf, run_both, small_cfg
from tests.test_gpu_adjoint import _gpu_adjoint, _setup

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3
TW = [0.3, -0.2, 0.1, 0.4, -0.3, 0.2]
TOL, TOL16 = 1e-5, 2e-3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("dim,n,quad", [(1, (5, 1, 1), ("gl1d", 8)), (1, (257, 1, 1), ("gl1d", 272)),
                                        (2, (7, 5, 1), ("octant", 2, 3)), (2, (64, 5, 1), ("octant", 6, 6)),
                                        (3, (5, 3, 3), ("octant", 3, 2)), (3, (33, 4, 2), ("octant", 2, 2))])
def test_moments(dim, n, quad, storage):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, [ISO, DIF] * dim + [PER] * (6 - 2 * dim), Tw=TW, nb=3, quad=quad)
    P = oracle_problem(cfg)
    ctx = gpu_ctx(cfg, storage=storage, kernel=bte.BTE_KERNEL_GENERIC)
    if storage == 0:
        bte.bte_set_state(ctx, (inputs.random_state(P.shape, 51) * 1e4).astype(np.float32))
    else:
        bte.bte_init_temperature(ctx, np.random.default_rng(2).random(P.ncell) - 0.2)
        bte.bte_step(ctx, 3)
    e = np.asarray(bte.bte_get_values(ctx), dtype=np.float64)
    T, TL, q = bte.bte_moments(ctx)
    To, TLo, qo = P.moments(e)
    tol = 1e-12 if storage == 0 else 1e-6
    assert rel_linf(T, To) <= tol and rel_linf(TL, TLo) <= tol
    if storage == 0:
        assert rel_linf(q, qo) <= 1e-12


@pytest.mark.parametrize("dim,n,bc", [
    (2, (2, 3, 1), [ISO, DIF, SPE, ISO, PER, PER]), (2, (127, 4, 1), [DIF, SPE, ISO, DIF, PER, PER]),
    (2, (132, 5, 1), [PER, PER, DIF, SPE, PER, PER]), (2, (255, 3, 1), [SPE, ISO, PER, PER, PER, PER]),
    (2, (256, 3, 1), [DIF, DIF, DIF, DIF, PER, PER]), (2, (260, 3, 1), [ISO, SPE, SPE, DIF, PER, PER]),
    (3, (6, 3, 4), [SPE, DIF, PER, PER, ISO, DIF]), (3, (132, 3, 2), [PER, PER, DIF, ISO, SPE, SPE])])
def test_implicit_rows(dim, n, bc):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=3)
    P = oracle_problem(cfg)
    rng = np.random.default_rng(31)
    e0 = (P.equilibrium(rng.uniform(-0.5, 0.5, (P.nz, P.ny, P.nx))) * (1 + 0.2 * rng.standard_normal(P.shape))).astype(np.float32)
    ctx = gpu_ctx(cfg)
    bte.bte_set_state(ctx, e0)
    bte.bte_sis_iterate(ctx, 2)
    eo = e0.astype(np.float64)
    for _ in range(2):
        eo = P.sis_iteration(eo, None)
    assert rel_linf(bte.bte_get_state(ctx), eo) <= TOL
    # the FP32 moment pass of the new state
    assert rel_linf(fused_TL(ctx), P.lattice_temperature(eo)) <= TOL


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("nx,bc,nb,nd", [(2, [ISO, DIF], 1, 8), (3, [DIF, SPE], 3, 8), (5, [SPE, ISO], 2, 10),
                                         (257, [PER, PER], 3, 34), (300, [DIF, DIF], 5, 16)])
def test_1d_step(nx, bc, nb, nd, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(1, (nx, 1, 1), bc + [PER] * 4, Tw=TW, nb=nb, quad=("gl1d", nd))
    P = oracle_problem(cfg, limiter)
    e0 = inputs.random_state(P.shape, 61) * 1e4
    Q = (np.random.default_rng(3).random((1, 1, nx)) * 1e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 4, Q, np.linspace(1.0, 0.3, 4), limiter=limiter, kernel=bte.BTE_KERNEL_GENERIC)
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("nx,bc", [(2, [ISO, DIF]), (37, [SPE, ISO]), (257, [DIF, DIF])])
def test_1d_step_16bit(nx, bc, storage):
    cfg = small_cfg(1, (nx, 1, 1), bc + [PER] * 4, Tw=TW, nb=3)
    P = oracle_problem(cfg)
    Q = (np.random.default_rng(9).random((1, 1, nx)) * 2e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, np.zeros(P.shape), 60, Q, storage=storage, rounding=1 if storage == 2 else 0, seed=5)
    scale = max([np.max(np.abs(oTL))] + [abs(t) for t, b in zip(TW, bc) if b in (ISO, DIF)])
    assert np.max(np.abs(gTL - oTL)) / scale <= TOL16


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("nx,bc,nb,nd", [(2, [ISO, DIF], 1, 8), (3, [DIF, SPE], 3, 8), (4, [PER, PER], 2, 8),
                                         (5, [SPE, SPE], 17, 10), (33, [DIF, ISO], 18, 8), (130, [SPE, DIF], 2, 96),
                                         (1100, [PER, PER], 2, 8), (100, [DIF, ISO], 1, 272)])
def test_persistent_rows(nx, bc, nb, nd, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(1, (nx, 1, 1), bc + [PER] * 4, Tw=TW, nb=nb, quad=("gl1d", nd))
    P = oracle_problem(cfg, limiter)
    e0 = inputs.random_state(P.shape, 63) * 1e4
    Q = (np.random.default_rng(3).random((1, 1, nx)) * 1e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 5, Q, np.linspace(1.0, 0.3, 5), limiter=limiter,
                                    kernel=bte.BTE_KERNEL_PERSISTENT)
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL
    # the wall values it leaves are those the next call starts from
    bte.bte_step(ctx, 1)
    eo = P.run(eo, 1, Q, np.linspace(1.0, 0.3, 5), n0=5)
    assert rel_linf(bte.bte_get_state(ctx), eo) <= TOL


TILED = [(2, (100, 9, 1), [SPE, DIF, ISO, SPE, PER, PER]), (2, (64, 19, 1), [ISO, SPE, PER, PER, PER, PER]),
         (2, (256, 5, 1), [SPE, SPE, DIF, ISO, PER, PER]), (2, (136, 7, 1), [SPE, SPE, SPE, SPE, PER, PER]),
         (3, (96, 9, 7), [SPE, SPE, DIF, SPE, ISO, DIF]), (3, (40, 5, 8), [SPE, ISO, PER, PER, SPE, SPE]),
         (3, (32, 10, 13), [DIF, SPE, PER, PER, DIF, ISO])]


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("dim,n,bc", TILED)
def test_specular_x_and_short_rows(dim, n, bc, kernel):
    """The tiled kernel, and what the default choice runs in its place on these grids."""
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=3)
    P = oracle_problem(cfg)
    ctx, g, gTL, eo, oTL = run_both(cfg, inputs.random_state(P.shape, 71) * 1e4, 3, kernel=kernel)
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("dim,n,bc", TILED)
def test_specular_x_and_short_rows_16bit(dim, n, bc, storage):
    n = (n[0] // 8 * 8, n[1], n[2])
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=3)
    P = oracle_problem(cfg)
    Q = (np.random.default_rng(9).random((P.nz, P.ny, P.nx)) * 2e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, np.zeros(P.shape), 30, Q, storage=storage, kernel=2,
                                    rounding=1 if storage == 2 else 0, seed=5)
    scale = max([np.max(np.abs(oTL))] + [abs(t) for t, b in zip(TW, bc) if b in (ISO, DIF)])
    assert np.max(np.abs(gTL - oTL)) / scale <= TOL16


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("dim,n,bc", [TILED[1], TILED[2], TILED[4], (2, (37, 21, 1), [DIF, SPE, ISO, DIF, PER, PER]),
                                      (2, (2, 4, 1), [PER, PER, SPE, DIF, PER, PER]),
                                      (3, (13, 5, 2), [SPE, ISO, PER, PER, DIF, SPE])])
def test_adjoint_by_default(dim, n, bc, limiter):
    """The streaming adjoint, after tiled, streaming and (minmod) generic forward steps."""
    cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, limiter, 0, 6)
    J, gQ, gt = _gpu_adjoint(ctx, Q, amps, dT0, p, 6, ckpt=2)
    Jo, gQo, gto = P.adjoint(P.equilibrium(np.asarray(dT0, np.float32).astype(np.float64)), 6, p, Q, amps)
    assert abs(J - Jo) <= 1e-5 * abs(Jo)
    assert rel_linf(gQ, gQo) <= 1e-4 and rel_linf(gt, gto) <= 1e-4
