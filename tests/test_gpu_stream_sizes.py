"""The register-streaming forward kernel at the edges of its geometry, on grids large enough to run it (smaller ones run
the generic kernel): two and three rows, cells or slices, odd rows whose last pair overlaps the one before, ragged
last strips, every wall on every axis, a number of directions its parts do not divide, and the sizes on either side
of the line between the two kernels.  Against the FP64 oracle at the parity tests' 1e-5 relative L-inf; the adjoint's
end state is bte_step's bit for bit."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import fused_TL, gpu_ctx, oracle_problem, rel_linf, run_both, small_cfg
from tests.test_gpu_adjoint import _gpu_adjoint, _setup

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


def streams(n, nb, nd):
    """The rule of bte_create."""
    nc = n[0] * n[1] * n[2]
    return nc ** 2 * nb * (min(nd, 32) / 32) ** 2 >= (2.5e7 if n[2] == 1 else 1.2e8)


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("dim,n,bc", [
    (2, (2, 511, 1), [ISO, DIF, SPE, ISO, PER, PER]), (2, (3, 341, 1), [DIF, SPE, ISO, DIF, PER, PER]),
    (2, (511, 2, 1), [PER, PER, DIF, SPE, PER, PER]), (2, (341, 3, 1), [SPE, ISO, PER, PER, PER, PER]),
    (2, (66, 17, 1), [SPE, ISO, PER, PER, PER, PER]), (2, (131, 9, 1), [DIF, DIF, DIF, DIF, PER, PER]),
    (3, (2, 34, 34), [SPE, SPE, DIF, ISO, ISO, DIF]), (3, (34, 2, 34), [ISO, DIF, PER, PER, SPE, SPE]),
    (3, (34, 33, 2), [PER, PER, SPE, DIF, DIF, ISO]), (3, (3, 3, 250), [DIF, SPE, ISO, SPE, PER, PER]),
    (3, (67, 6, 6), [DIF, SPE, ISO, SPE, PER, PER]), (3, (35, 13, 5), [SPE, ISO, DIF, DIF, SPE, DIF])])
def test_shapes(dim, n, bc, limiter):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=24, quad=("octant", 3, 3))
    assert streams(n, 24, 72)
    P = oracle_problem(cfg, limiter)
    e0 = inputs.random_state(P.shape, 41) * 1e4
    Q = (np.random.default_rng(3).random((P.nz, P.ny, P.nx)) * 1e17).astype(np.float32)
    ctx, g, gTL, eo, oTL = run_both(cfg, e0, 3, Q, np.linspace(1.0, 0.3, 3), limiter=limiter, kernel=bte.BTE_KERNEL_GENERIC)
    assert rel_linf(g, eo) <= TOL and rel_linf(gTL, oTL) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


@pytest.mark.parametrize("dim,n,axis", [(2, (41, 35, 1), 0), (2, (35, 41, 1), 1), (3, (19, 13, 10), 2)])
def test_periodic_jump(dim, n, axis):
    from paper_2306_14181_gb300 import bte
    bc = [DIF, ISO] * dim + [PER] * (6 - 2 * dim)
    bc[2 * axis] = bc[2 * axis + 1] = PER
    cfg = small_cfg(dim, n, bc, Tw=TW, nb=24, jump=[0.7 if a == axis else 0.0 for a in range(3)])
    assert streams(n, 24, 32)
    P = oracle_problem(cfg)
    ctx, g, gTL, eo, oTL = run_both(cfg, inputs.random_state(P.shape, 43) * 1e4, 3, kernel=bte.BTE_KERNEL_GENERIC)
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


# the last size of the generic kernel and the first of the streaming one
@pytest.mark.parametrize("dim,n,nb", [(2, (37, 33, 1), 16), (2, (37, 34, 1), 16), (3, (21, 21, 6), 16), (3, (21, 19, 7), 16)])
def test_either_side_of_the_line(dim, n, nb):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, [SPE, DIF, ISO, DIF, DIF, SPE], Tw=TW, nb=nb)
    assert streams(n, nb, 32) == (n in ((37, 34, 1), (21, 19, 7)))
    P = oracle_problem(cfg)
    e0 = (inputs.random_state(P.shape, 44) * 1e4).astype(np.float32)
    out = []
    for _ in range(2):
        ctx, g, gTL, eo, oTL = run_both(cfg, e0, 5, kernel=bte.BTE_KERNEL_GENERIC)
        out.append((g.copy(), bte.bte_lattice_temperature(ctx).copy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert rel_linf(g, eo) <= TOL and rel_linf(fused_TL(ctx), oTL) <= TOL


@pytest.mark.parametrize("limiter", [1, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, (67, 54, 1), [DIF, SPE, ISO, DIF, PER, PER]),
                                      (3, (21, 20, 19), [SPE, ISO, DIF, DIF, DIF, SPE])])
def test_adjoint_ends_where_the_steps_end(dim, n, bc, limiter):
    from paper_2306_14181_gb300 import bte
    assert streams(n, 2, 32)
    out = []
    for adjoint in (True, False):
        cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, limiter, 0, 7)
        if adjoint:
            _, _, gt = _gpu_adjoint(ctx, Q, amps, dT0, p, 7, ckpt=3)
            assert np.array_equal(gt, _gpu_adjoint(ctx, Q, amps, dT0, p, 7, ckpt=7)[2])
        else:
            bte.bte_init_temperature(ctx, dT0.reshape(-1))
            bte.bte_set_source(ctx, Q, amps)
            bte.bte_step(ctx, 7)
        end = [bte.bte_get_state(ctx).copy(), bte.bte_lattice_temperature(ctx).copy()]
        bte.bte_step(ctx, 1)
        out.append(end + [bte.bte_get_state(ctx).copy()])
    assert all(np.array_equal(x, y) for x, y in zip(*out))
