"""The FP64 moments of a state that holds one infinity or NaN: the call returns its error, and T, T_L and the flux
it copied out are non-finite in that cell, with the sign the sum has, and the oracle's in every other (1e-12, and 1e-6
for 16-bit codes, as for finite states)."""
import numpy as np
import pytest

from paper_2306_14181_gb300 import inputs
from tests.support import gpu_ctx, oracle_problem, rel_linf, small_cfg

pytestmark = pytest.mark.gpu

ISO, DIF, SPE, PER = 0, 1, 2, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_14181_gb300 import build
    build.build()


CODES = {0: {"inf": np.inf, "-inf": -np.inf, "nan": np.nan}, 1: {"inf": np.inf, "-inf": -np.inf, "nan": np.nan},
         2: {"inf": 0x7f80, "-inf": 0xff80, "nan": 0x7fc0}}


@pytest.mark.parametrize("value", ["inf", "-inf", "nan"])
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("dim,n,explicit", [(1, (37, 1, 1), False), (2, (7, 5, 1), False), (3, (5, 4, 3), True)])
def test_moments_mark_the_cell(dim, n, explicit, storage, value):
    from paper_2306_14181_gb300 import bte
    cfg = small_cfg(dim, n, [ISO, DIF] * dim + [PER] * (6 - 2 * dim), nb=3)  # gl1d 8, octant 2 x 2
    P = oracle_problem(cfg)
    if explicit:
        cfg["quad"] = ("explicit",) + tuple(bte.bte_get_quadrature(gpu_ctx(cfg)))
    ctx = gpu_ctx(cfg, storage=storage)
    nb, nd = ctx.shape[:2]
    if storage == 0:
        bte.bte_set_state(ctx, (inputs.random_state(ctx.shape, 51) * 1e4).astype(np.float32))
    else:
        bte.bte_init_temperature(ctx, np.random.default_rng(2).random(int(np.prod(n))))
        bte.bte_step(ctx, 2)
    To, TLo, qo = P.moments(np.asarray(bte.bte_get_values(ctx), np.float64))
    ref = np.zeros(ctx.info.ncell, np.float32)
    codes = bte.bte_get_state(ctx, ref=ref).reshape(nb, nd, -1).copy()
    cell, d = ctx.info.ncell - 2, nd // 2 + 1
    codes[1, d, cell] = CODES[storage][value]
    bte.bte_set_state(ctx, codes, ref if storage else None)
    T, TL, q = (np.zeros(ctx.info.ncell * m) for m in (1, 1, 3))
    dp = bte._dp
    assert bte.load().bte_moments(ctx.handle, dp(T), dp(TL), dp(q)) == bte.BTE_ENONFINITE
    for t in (T, TL):
        assert np.isnan(t[cell]) if value == "nan" else t[cell] == float(value)
    assert not np.any(np.isfinite(q.reshape(3, -1)[:dim, cell]))
    assert np.all(np.isfinite(q.reshape(3, -1)[:, np.arange(T.size) != cell]))
    tol = 1e-12 if storage == 0 else 1e-6
    rest = np.arange(ctx.info.ncell) != cell
    assert rel_linf(T[rest], To.reshape(-1)[rest]) <= tol and rel_linf(TL[rest], TLo.reshape(-1)[rest]) <= tol
    with pytest.raises(bte.BteError):
        bte.bte_energy(ctx)
