"""Which kernels bte_adjoint runs, and that the choice shows in no result: gradients of the default choice
are those of the explicit one, bit for bit (sums that cancel form dJ/dlog tau, so that any other
order of the same operations moves it by up to 1e-3), rows without an instance of a kernel run the next one,
and the context ends where bte_step ends.  Tolerances against the oracle are those of the parity tests: 1e-5
on J, 1e-4 on the gradients."""
import numpy as np
import pytest

from tests.support import rel_linf
from tests.test_gpu_adjoint import _gpu_adjoint, _setup

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, (64, 3, 1), [ISO, SPE, DIF, ISO, PER, PER]),
                                      (2, (64, 9, 1), [SPE, SPE, ISO, DIF, PER, PER]),
                                      (3, (64, 3, 5), [SPE, ISO, PER, PER, DIF, SPE])])
def test_rows_without_a_tiled_adjoint(dim, n, bc, kernel):
    """64-cell rows step forward on the tiled kernel; the adjoint has no instance for them."""
    cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, 2, kernel, 6)
    J, gQ, gt = _gpu_adjoint(ctx, Q, amps, dT0, p, 6, ckpt=2)
    Jo, gQo, gto = P.adjoint(P.equilibrium(np.asarray(dT0, np.float32).astype(np.float64)), 6, p, Q, amps)
    assert abs(J - Jo) <= 1e-5 * abs(Jo)
    assert rel_linf(gQ, gQo) <= 1e-4 and rel_linf(gt, gto) <= 1e-4


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("limiter", [0, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, (96, 9, 1), [SPE, SPE, ISO, DIF, PER, PER]),
                                      (2, (128, 13, 1), [PER, PER, SPE, DIF, PER, PER]),
                                      (2, (256, 6, 1), [DIF, SPE, PER, PER, PER, PER]),
                                      (3, (128, 5, 6), [ISO, DIF, SPE, SPE, PER, PER]),
                                      (3, (128, 10, 7), [SPE, SPE, PER, PER, DIF, ISO]),
                                      # 3-D rows below 112 cells: bte_step streams by default
                                      (3, (96, 10, 7), [SPE, SPE, PER, PER, DIF, ISO]),
                                      (3, (80, 6, 5), [DIF, ISO, SPE, SPE, PER, PER])])
def test_default_gradients_are_the_tiled_ones(dim, n, bc, limiter, storage):
    out = []
    for kernel in (0, 2):
        cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, limiter, kernel, 6, storage=storage)
        out.append(_gpu_adjoint(ctx, Q, amps, dT0, p, 6, ckpt=2))
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])


# dJ/dlog tau (two bands) by (dimension, limiter, storage): the wall pass with every stored value rounded by
# itself, as the general ghost routine forms them
WALL_BITS = {
    (2, 2, 1): ('-0x1.e5ccc4b97b2dcp-19', '-0x1.40b018d511635p-15'),
    (2, 2, 2): ('-0x1.e5217e0565c43p-19', '-0x1.422e3a6622496p-15'),
    (3, 1, 1): ('0x1.b143abb1d0bf3p-16', '0x1.ae105c2fe4c33p-15'),
    (3, 1, 2): ('0x1.b1336a0abe11ap-16', '0x1.ad99317dff515p-15'),
    (3, 2, 1): ('0x1.b1fcddc9a9e13p-16', '0x1.b76ae6124b1d8p-15'),
    (3, 2, 2): ('0x1.b20796b0b0ca5p-16', '0x1.b7d99614000d9p-15'),
}


@pytest.mark.parametrize("dim,limiter,storage", sorted(WALL_BITS))
def test_16bit_wall_pass_rounds_each_operation(dim, limiter, storage):
    n, bc = {2: ((96, 9, 1), [SPE, SPE, ISO, DIF, PER, PER]), 3: ((96, 10, 7), [SPE, ISO, DIF, SPE, DIF, ISO])}[dim]
    cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, limiter, 2, 6, storage=storage)
    _, _, gt = _gpu_adjoint(ctx, Q, amps, dT0, p, 6, ckpt=2)
    assert tuple(float(x).hex() for x in gt) == WALL_BITS[dim, limiter, storage]


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, (128, 9, 1), [SPE, DIF, ISO, DIF, PER, PER]),
                                      (2, (37, 21, 1), [DIF, SPE, ISO, DIF, PER, PER]),
                                      (3, (64, 6, 5), [SPE, ISO, PER, PER, DIF, SPE]),
                                      (3, (13, 5, 4), [SPE, ISO, DIF, DIF, DIF, SPE])])
def test_end_state_is_that_of_the_steps(dim, n, bc, limiter):
    """By default, streamed or not: the state, T_L and the wall values (one more step) of bte_step, bit for
    bit; nothing changes in a call of no steps; a repeated call gives the same gradients."""
    from paper_2306_14181_gb300 import bte
    out = []
    for adjoint in (True, False):
        cfg, P, ctx, Q, amps, dT0, p = _setup(dim, n, bc, limiter, 0, 7)
        if adjoint:
            first = _gpu_adjoint(ctx, Q, amps, dT0, p, 7, ckpt=3)
            again = _gpu_adjoint(ctx, Q, amps, dT0, p, 7, ckpt=3)
            assert first[0] == again[0] and np.array_equal(first[2], again[2])
        else:
            bte.bte_init_temperature(ctx, dT0.reshape(-1))
            bte.bte_set_source(ctx, Q, amps)
            bte.bte_step(ctx, 7)
        end = [bte.bte_get_state(ctx).copy(), bte.bte_lattice_temperature(ctx).copy()]
        J, _, _ = bte.bte_adjoint(ctx, 0, p, 0)
        assert abs(J - float(np.sum(p.reshape(-1) * end[1].astype(np.float64)))) <= 1e-12 * abs(J)
        bte.bte_step(ctx, 1)
        end.append(bte.bte_get_state(ctx).copy())
        out.append(end)
    assert all(np.array_equal(x, y) for x, y in zip(*out))
