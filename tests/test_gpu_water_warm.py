"""The warm-started water path (k_water_warm: FP32 start, FP64 evaluations) against the oracle.

Tolerances are those of the general path's parity tests: forces 1e-9 of the largest, populations and
cell energies 1e-10; the positions are the GPU's own, so nothing accumulates.
"""
import numpy as np
import pytest

import cavmd_synth as cs
from oracle import dftb as OD

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2512_03277_gb300 as P
    P.load_library()
    return P


def _check(ctx, params, species, order):
    """The last evaluation against the oracle at the context's own positions; its SCC iterations."""
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    n = ctx.n_cells
    pos = st["r"].reshape(n, 3, 3)[:, order]
    ref = OD.dftb(params, species, pos)
    F, q = ev["F_dftb"].reshape(n, 3, 3)[:, order], ev["q_pop"].reshape(n, 3)[:, order]
    assert np.abs(F - ref["F"]).max() < 1e-9 * np.abs(ref["F"]).max()
    assert np.abs(q - ref["q"]).max() < 1e-10
    assert np.abs(ev["E_cell"] - ref["E"]).max() < 1e-10
    return ev["scc_iters"]


# around the five waters of a warp and the ten of a block, one cell, and several blocks
@pytest.mark.parametrize("n", [1, 4, 5, 6, 9, 11, 20, 333])
@pytest.mark.parametrize("fast", [False, True])
def test_warm_steps_match_the_oracle(P, n, fast):
    """fast: momenta three times and a time step twice as large, so that the overlap of some waters
    changes by more than the warm path takes (0.2) and they go through the general solve, beside
    others that do not. (Every overlap stays positive definite along this trajectory.)"""
    w = cs.make_workload("c2", n_cells=n, n_modes=8)
    o = P.default_options()
    if fast:
        w["system"].p *= np.where(np.arange(n) % 2 == 0, 3.0, 1.0).repeat(3)[:, None]
        o.dt *= 2.0
    ctx = P.Context(w["system"], w["params"], w["modes"], o)
    for step in range(3):
        ctx.cavmd_step(1)
        it = _check(ctx, w["params"], [0, 1, 1], [0, 1, 2])
        if not fast:
            assert it.max() <= 4
        elif step == 0 and n >= 4:
            assert it.max() > 4 > it.min()   # both ways were taken


def test_other_orders_take_the_general_path(P):
    """Hydrogen first: not the warm path's order, the same physics."""
    w = cs.make_workload("c2", n_cells=12, n_modes=8)
    sy = w["system"]
    perm = (3 * np.arange(12)[:, None] + np.array([1, 0, 2])).ravel()
    sy.species, sy.r, sy.p = sy.species[perm], sy.r[perm], sy.p[perm]
    ctx = P.Context(sy, w["params"], w["modes"])
    for _ in range(2):
        ctx.cavmd_step(1)
        it = _check(ctx, w["params"], [0, 1, 1], [1, 0, 2])
        assert it.max() > 4
