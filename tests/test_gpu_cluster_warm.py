"""The warm-started path of the cluster kernel (FP32 start, FP64 evaluations) against the oracle, at
the context's own positions. Tolerances: those of the parity tests (forces 1e-9 of the largest,
populations and cell energies 1e-10)."""
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


def _check(ctx, params, sy):
    ev, st = ctx.cavmd_get_eval(), ctx.cavmd_get_state()
    cells = [slice(sy.cell_offset[c], sy.cell_offset[c + 1]) for c in range(sy.n_cells)]
    refs = [OD.dftb(params, sy.species[s], st["r"][None, s]) for s in cells]
    largest = max(np.abs(ref["F"]).max() for ref in refs)
    for c, (s, ref) in enumerate(zip(cells, refs)):
        assert np.abs(ev["F_dftb"][s] - ref["F"][0]).max() < 1e-9 * largest
        assert np.abs(ev["q_pop"][s] - ref["q"][0]).max() < 1e-10
        assert abs(ev["E_cell"][c] - ref["E"][0]) < 1e-10 * max(1.0, abs(ref["E"][0]))
    return ev["scc_iters"]


# one water to the largest cell (10 waters, 60 orbitals), both thread groups, an idle half of the last block
@pytest.mark.parametrize("sizes", [[2], [1, 5, 6], [1, 2, 3, 4, 5], [6, 7, 8, 9, 10, 3, 4]])
@pytest.mark.parametrize("fast", [False, True])
def test_warm_steps_match_the_oracle(P, sizes, fast):
    """fast: a time step twice as large and every second cluster's momenta doubled, so that some leave
    the warm path's range (an overlap change of 0.2) beside others that stay in it."""
    rng = np.random.default_rng(7)
    sy = cs.cluster_batch(rng, sizes, np.zeros((len(sizes), 3)))
    sy.p = cs.mb_momenta(rng, sy)
    o = P.default_options()
    if fast:
        o.dt *= 2.0
        sy.p *= np.repeat(np.where(np.arange(len(sizes)) % 2 == 0, 2.0, 1.0), np.diff(sy.cell_offset))[:, None]
    params = cs.load_water_params()
    ctx = P.Context(sy, params, cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o)
    for _ in range(3):
        ctx.cavmd_step(1)
        it = _check(ctx, params, sy)
        if not fast:
            assert it.max() <= 4


def test_mixed_compositions(P):
    """Cells other than water clusters: hydrogen and oxygen molecules, and a lone hydrogen molecule's
    two orbitals, in one batch with a water."""
    sp = [[1, 1], [0, 0], [0, 1, 1], [1, 1, 1, 1]]
    pos = [[[0, 0, 0], [0, 0, 1.6]], [[0, 0, 0], [0.3, 2.4, 0.1]],
           cs.water_reference_geometry(), [[0, 0, 0], [0, 0, 1.5], [6, 0, 0], [6, 0.2, 1.6]]]
    params = cs.load_water_params()
    keep = []
    for s, r in zip(sp, pos):   # those whose oracle solution exists (a closed shell with a gap)
        try:
            OD.dftb(params, s, np.array(r, float)[None])
            keep.append((s, r))
        except (OD.SCCError, np.linalg.LinAlgError):
            pass
    assert len(keep) >= 3
    off = np.cumsum([0] + [len(s) for s, _ in keep]).astype(np.int32)
    sy = cs.System(species=np.concatenate([s for s, _ in keep]).astype(np.int32), cell_offset=off,
                   r=np.concatenate([np.array(r, float) for _, r in keep]), p=np.zeros((off[-1], 3)),
                   R_ref=np.zeros((len(keep), 3)))
    ctx = P.Context(sy, params, cs.line_modes(8, 1000.0, 0.001, k_max=0.01))
    for _ in range(2):
        ctx.cavmd_step(1)
        _check(ctx, params, sy)
