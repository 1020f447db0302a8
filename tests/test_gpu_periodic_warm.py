"""The warm path of the periodic kernels after many steps (mixing inside the occupied and virtual blocks,
the block sweeps that undo it, blocks sharing a k-grid cell) against the periodic oracle, at the
context's own positions. Tolerances: those of the parity tests (forces 1e-9 of the largest,
populations and cell energies 1e-10)."""
import numpy as np
import pytest

import cavmd_synth as cs
from oracle import periodic as PR

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("waters,grid,steps", [(12, 1, 60), (3, 1, 3), (2, 2, 40), (2, 3, 3)])
def test_many_warm_steps_match_the_oracle(waters, grid, steps):
    import paper_2512_03277_gb300 as P
    rng = np.random.default_rng(17)
    side = (waters / 33.0) ** (1.0 / 3.0) * 10.0 * cs.ANGSTROM if waters > 2 else 8.5
    cent = np.zeros((3, 3))
    cent[:, 0] = [200.0, 400.0, 600.0]
    kw = {} if waters > 2 else {"d_min": 4.0, "d_atom": 2.8}
    sy, lat = cs.periodic_water_cells(rng, cent, n_waters=waters, side=side, **kw)
    sy.p = cs.mb_momenta(rng, sy)
    o = P.default_options()
    for k in range(3):
        o.kgrid[k] = grid
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o, lattice=lat)
    ctx.cavmd_step(steps)
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    assert ev["scc_iters"].max() <= 4
    for c in range(sy.n_cells):
        s = slice(sy.cell_offset[c], sy.cell_offset[c + 1])
        if grid == 1:
            ref = PR.dftb_periodic(pa, sy.species[s], st["r"][s], lat)
        else:
            ref = PR.dftb_periodic_k(pa, sy.species[s], st["r"][s], lat, (grid, grid, grid))
        assert np.abs(ev["F_dftb"][s] - ref["F"]).max() < 1e-9 * np.abs(ref["F"]).max()
        assert np.abs(ev["q_pop"][s] - ref["q"]).max() < 1e-10
        assert abs(ev["E_cell"][c] - ref["E"]) < 1e-10 * max(1.0, abs(ref["E"]))
