"""Cells that leave the warm-started path, beside others that stay on it, and the widest k-point
problems, against the oracles at the context's own positions. Tolerances: those of the parity tests
(forces 1e-9 of the largest, populations and cell energies 1e-10)."""
import numpy as np
import pytest

import cavmd_synth as cs
from oracle import dftb as OD
from oracle import periodic as PR

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2512_03277_gb300 as P
    P.load_library()
    return P


def _check(ctx, sy, solve):
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    cells = [slice(sy.cell_offset[c], sy.cell_offset[c + 1]) for c in range(sy.n_cells)]
    refs = [solve(sy.species[s], st["r"][s]) for s in cells]
    largest = max(np.abs(ref["F"]).max() for ref in refs)
    for c, (s, ref) in enumerate(zip(cells, refs)):
        assert np.abs(ev["F_dftb"][s] - ref["F"]).max() < 1e-9 * largest
        assert np.abs(ev["q_pop"][s] - ref["q"]).max() < 1e-10
        assert abs(ev["E_cell"][c] - ref["E"]) < 1e-10 * max(1.0, abs(ref["E"]))
    return ev["scc_iters"]


def _periodic(waters, n, seed=17):
    rng = np.random.default_rng(seed)
    side = (waters / 33.0) ** (1.0 / 3.0) * 10.0 * cs.ANGSTROM if waters > 2 else 8.5
    cent = np.zeros((n, 3))
    cent[:, 0] = 200.0 * np.arange(1, n + 1)
    kw = {} if waters > 2 else {"d_min": 4.0, "d_atom": 2.8}
    sy, lat = cs.periodic_water_cells(rng, cent, n_waters=waters, side=side, **kw)
    sy.p = cs.mb_momenta(rng, sy)
    return sy, lat


def _solver(pa, lat, grid):
    if tuple(grid) == (1, 1, 1):
        return lambda sp, r: PR.dftb_periodic(pa, sp, r, lat)
    return lambda sp, r: PR.dftb_periodic_k(pa, sp, r, lat, tuple(grid))


# the Gamma point; two points (blocks of a cluster: one or two); fourteen points (several blocks a cell, of which
# the first takes the cell over)
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 1, 1), (3, 3, 3)])
def test_periodic_cells_that_leave_the_warm_path(P, grid):
    """Every second cell's momenta four times and the time step twice as large: the overlap of those
    cells changes by more than the warm path takes."""
    sy, lat = _periodic(2, 4)
    sy.p *= np.repeat(np.where(np.arange(4) % 2 == 0, 4.0, 1.0), np.diff(sy.cell_offset))[:, None]
    o = P.default_options()
    o.dt *= 2.0
    o.kgrid[:] = grid
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o, lattice=lat)
    for step in range(2):
        ctx.cavmd_step(1)
        it = _check(ctx, sy, _solver(pa, lat, grid))
        if step == 0:
            assert it.max() > 4 > it.min()   # both ways were taken


def test_clusters_that_leave_the_warm_path(P):
    rng = np.random.default_rng(7)
    sizes = [6, 1, 8, 2, 3, 10, 4]
    sy = cs.cluster_batch(rng, sizes, np.zeros((len(sizes), 3)))
    sy.p = cs.mb_momenta(rng, sy)
    sy.p *= np.repeat(np.where(np.arange(len(sizes)) % 2 == 0, 3.0, 1.0), np.diff(sy.cell_offset))[:, None]
    o = P.default_options()
    o.dt *= 2.0
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o)

    def solve(sp, r):
        ref = OD.dftb(pa, sp, r[None])
        return {k: ref[k][0] for k in ("F", "q", "E")}

    for step in range(2):
        ctx.cavmd_step(1)
        it = _check(ctx, sy, solve)
        if step == 0:
            assert it.max() > 4 > it.min()


def test_warm_steps_of_wide_k_points(P):
    """Twenty-two waters, 132 orbitals: real forms of 264 rows, beyond the 256 of the smaller kernel."""
    sy, lat = _periodic(22, 2)
    o = P.default_options()
    o.kgrid[:] = (2, 1, 1)
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o, lattice=lat)
    ctx.cavmd_step(2)
    assert _check(ctx, sy, _solver(pa, lat, (2, 1, 1))).max() <= 4


@pytest.mark.parametrize("grid", [(1, 1, 1), (3, 3, 3)])
def test_displaced_copies_that_leave_the_warm_path(P, grid):
    """A displacement of 0.3 bohr changes the overlap by more than the warm path takes: copies go through the
    general path from their cell's basis. Tolerance: populations to 1e-10 times positions of a few bohr over
    the displacement, for the two ends of a difference. (At 0.5 bohr two overlaps are not positive definite.)"""
    sy, lat = _periodic(2, 2)
    o = P.default_options()
    o.kgrid[:] = grid
    o.charge_model = 1       # forward finite differences
    o.fd_step = 0.3
    pa = cs.load_water_params()
    mo = cs.line_modes(8, 1000.0, 0.001, k_max=0.01)
    ctx = P.Context(sy, pa, mo, o, lattice=lat)
    b = ctx.cavmd_get_eval()["b"].reshape(-1, 3)
    for c in range(sy.n_cells):
        s = slice(sy.cell_offset[c], sy.cell_offset[c + 1])
        ref = PR.born_fd_periodic(pa, sy.species[s], sy.r[s], lat, np.array(mo.pol), h=0.3, kgrid=grid)
        assert np.abs(b[s] - ref).max() < 2 * 1e-10 * 20.0 / 0.3
