"""The warm-started paths leave nothing of the residual that passed their convergence test in the
charges: against the oracle converged to 2e-14, at the context's own positions.

Tolerance: scc_tol (1e-12) bounds the change that is left when the test passes, and the paths take that
change themselves, to a tenth: 1e-13, and half of it again for the rounding of both sides and the
oracle's own residual. (A general iteration ends likewise: it moves the basis after its test.)"""
import numpy as np
import pytest

import cavmd_synth as cs
from oracle import dftb as OD
from oracle import periodic as PR

pytestmark = pytest.mark.gpu

TOL = 1.5e-13


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2512_03277_gb300 as P
    P.load_library()
    return P


def test_waters(P):
    w = cs.make_workload("c2", n_cells=3000, n_modes=16)
    ctx = P.Context(w["system"], w["params"], w["modes"])
    ctx.cavmd_step(4)
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    ref = OD.dftb(w["params"], [0, 1, 1], st["r"].reshape(-1, 3, 3), tol=2e-14, forces=False)
    assert np.abs(ev["q_pop"].reshape(-1, 3) - ref["q"]).max() < TOL


def test_clusters(P):
    rng = np.random.default_rng(5)
    sizes = list(rng.integers(1, 11, size=96))
    sy = cs.cluster_batch(rng, sizes, np.zeros((len(sizes), 3)))
    sy.p = cs.mb_momenta(rng, sy)
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01))
    ctx.cavmd_step(4)
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    for c in range(sy.n_cells):
        s = slice(sy.cell_offset[c], sy.cell_offset[c + 1])
        ref = OD.dftb(pa, sy.species[s], st["r"][None, s], tol=2e-14, forces=False)
        assert np.abs(ev["q_pop"][s] - ref["q"][0]).max() < TOL


def test_periodic_cells(P):
    rng = np.random.default_rng(17)
    cent = np.zeros((4, 3))
    cent[:, 0] = 200.0 * np.arange(1, 5)
    sy, lat = cs.periodic_water_cells(rng, cent, n_waters=33, side=10.0 * cs.ANGSTROM)
    sy.p = cs.mb_momenta(rng, sy)
    pa = cs.load_water_params()
    ctx = P.Context(sy, pa, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), lattice=lat)
    ctx.cavmd_step(3)
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    for c in range(sy.n_cells):
        s = slice(sy.cell_offset[c], sy.cell_offset[c + 1])
        ref = PR.dftb_periodic(pa, sy.species[s], st["r"][s], lat, tol=2e-14, forces=False)
        assert np.abs(ev["q_pop"][s] - ref["q"]).max() < TOL


def test_fast_waters_keep_their_electrons(P):
    """Momenta 2.5 times and a time step twice as large: rotations at the edge of the warm path leave the
    largest overlap defects E that it takes. The populations of a water sum to 2 tr(C_o^T S C_o) = 8.

    Tolerance: with the norm of E below 5e-4, what the correction leaves out (35/128 E^4) is below 1.7e-14
    and FP32 rounds its last terms by 6e-15: 2 sqrt(4) 2.3e-14 on the trace, and 1e-14 for the sums."""
    w = cs.make_workload("c2", n_cells=4000, n_modes=16)
    w["system"].p *= 2.5
    o = P.default_options()
    o.dt *= 2.0
    ctx = P.Context(w["system"], w["params"], w["modes"], o)
    ctx.cavmd_step(1)
    ev = ctx.cavmd_get_eval()
    warm = ev["scc_iters"] <= 4
    assert warm.sum() > 100
    assert np.abs(ev["q_pop"].reshape(-1, 3).sum(1) - 8.0)[warm].max() < 1.02e-13
