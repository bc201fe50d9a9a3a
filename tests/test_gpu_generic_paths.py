"""The two kernels grids of one or two 1-D bands and 16-bit states off the tiled kernel's shapes run: the split 1-D
step gives the generic step's bits, and the generic step's direction groups repeat theirs.

The split step runs with one or two bands, the generic one with more: the same bands followed by bands of 1e-30 of
their heat capacity, which no sum of the first ones feels, are the same problem on the generic step."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import gpu_ctx, oracle_problem, rel_linf, run_both, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3
TW = [0.3, -0.2, 0.1, 0.4, -0.3, 0.2]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("storage,rounding", [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("nx,bc,nb,nd,limiter", [
    (2, [ISO, DIF], 1, 8, 2), (3, [DIF, SPE], 2, 10, 1), (37, [SPE, ISO], 2, 34, 2), (37, [DIF, DIF], 1, 34, 0),
    (257, [DIF, DIF], 2, 34, 2), (300, [PER, PER], 1, 272, 1), (256, [DIF, ISO], 1, 512, 2)])
def test_split_step_is_the_generic_step(nx, bc, nb, nd, limiter, storage, rounding):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(1, (nx, 1, 1), bc + [PER] * 4, Tw=TW, nb=nb, quad=("gl1d", nd))
    rng = np.random.default_rng(17)
    e0 = (inputs.random_state((nb, nd, 1, 1, nx), 23) * 1e4).astype(np.float32)
    Q = (rng.random((1, 1, nx)) * 1e17).astype(np.float32)
    dT0 = rng.random(nx) - 0.3
    out = []
    for extra in (0, 3 - nb):
        c = dict(cfg, nb=nb + extra)
        c["C"], c["v"], c["tau"] = (np.concatenate([cfg[x], np.repeat(cfg[x][-1:] * f, extra)])
                                    for x, f in (("C", 1e-30), ("v", 1.0), ("tau", 1.0)))
        ctx = gpu_ctx(c, limiter=limiter, kernel=bte.BTE_KERNEL_GENERIC, storage=storage, rounding=rounding, seed=5)
        if storage == 0:
            bte.bte_set_state(ctx, np.concatenate([e0, np.repeat(e0[-1:] * np.float32(1e-30), extra, axis=0)]))
        else:
            bte.bte_init_temperature(ctx, dT0)
        bte.bte_set_source(ctx, Q, np.linspace(1.0, 0.3, 6))
        bte.bte_step(ctx, 6)
        state = bte.bte_get_state(ctx)[:nb].copy()
        out.append((state.view(np.uint16 if storage else np.uint32), bte.bte_lattice_temperature(ctx).copy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("dim,n,bc,quad,storage", [
    (1, (40, 1, 1), [DIF, ISO, PER, PER, PER, PER], ("gl1d", 8), 0),
    (1, (300, 1, 1), [SPE, DIF, PER, PER, PER, PER], ("gl1d", 70), 0),
    (1, (70, 1, 1), [DIF, ISO, PER, PER, PER, PER], ("gl1d", 34), 2),
    (2, (37, 9, 1), [SPE, DIF, ISO, DIF, PER, PER], ("octant", 3, 3), 1),
    (3, (7, 6, 5), [DIF, SPE, ISO, DIF, DIF, ISO], ("octant", 2, 2), 1),
    (3, (13, 5, 4), [PER, PER, SPE, DIF, DIF, ISO], ("octant", 3, 2), 2)])
def test_generic_direction_groups(dim, n, bc, quad, storage):
    """Grids that still run the generic step and split its directions over thread groups: two runs are bitwise
    equal, and match the oracle (the parity tests' 1e-5, and 2e-3 on T_L for 16-bit codes)."""
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=3, quad=quad)
    P = oracle_problem(cfg)
    Q = (np.random.default_rng(9).random((P.nz, P.ny, P.nx)) * 2e17).astype(np.float32)
    e0 = np.zeros(P.shape) if storage else inputs.random_state(P.shape, 19) * 1e4
    out = []
    for _ in range(2):
        ctx, g, gTL, eo, oTL = run_both(cfg, e0, 30 if storage else 6, Q, storage=storage, kernel=bte.BTE_KERNEL_GENERIC,
                                        rounding=1 if storage == 2 else 0, seed=5)
        out.append((g.copy(), bte.bte_lattice_temperature(ctx).copy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    if storage == 0:
        assert rel_linf(g, eo) <= 1e-5
    else:
        scale = max([np.max(np.abs(oTL))] + [abs(t) for t, b in zip(TW, bc) if b in (ISO, DIF)])
        assert np.max(np.abs(gTL - oTL)) / scale <= 2e-3
