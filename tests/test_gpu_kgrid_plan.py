"""The k-grid's workspace where the allocator has little memory: fewer cells in flight, the same results."""
import ctypes as C

import numpy as np
import pytest

import cavmd_synth as cs

pytestmark = pytest.mark.gpu


def _run(P, B, torch, limit):
    """Sixty two-water cells on 3 x 3 x 3 with an allocator that refuses requests above `limit` bytes."""
    rng = np.random.default_rng(17)
    cent = np.zeros((60, 3))
    cent[:, 0] = 200.0 * np.arange(1, 61)
    sy, lat = cs.periodic_water_cells(rng, cent, n_waters=2, side=8.5, d_min=4.0, d_atom=2.8)
    sy.p = cs.mb_momenta(rng, sy)
    sy.p[:60] *= 4.0    # some of the first ten cells leave the warm path
    o = P.default_options()
    o.dt *= 2.0
    o.kgrid[:] = (3, 3, 3)
    refused = []

    def alloc(nbytes, user):
        if nbytes > limit:
            refused.append(nbytes)
            return 0
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0)

    def free(ptr, user):
        torch.cuda.caching_allocator_delete(ptr)

    keep = B.ALLOC_FN(alloc), B.FREE_FN(free)
    o.dev_alloc, o.dev_free = keep
    ctx = P.Context(sy, cs.load_water_params(), cs.line_modes(8, 1000.0, 0.001, k_max=0.01), o, torch_memory=False,
                    lattice=lat)
    ctx.cavmd_step(1)
    ev = ctx.cavmd_get_eval()
    assert ctx.cavmd_last_error() == ""
    ctx.cavmd_destroy()
    return ev, refused


def test_fewer_cells_in_flight_when_memory_is_short():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2512_03277_gb300 as P
    from paper_2512_03277_gb300 import cavmd as B
    P.load_library()
    full, none = _run(P, B, torch, 1 << 40)
    few, refused = _run(P, B, torch, 12 << 20)   # a cell takes about half a MB
    assert not none and refused
    assert full["scc_iters"].max() > 4 > full["scc_iters"].min()
    for k in ("F_dftb", "q_pop", "E_cell", "M", "scc_iters"):
        assert np.array_equal(full[k], few[k]), k
    with pytest.raises(B.CavmdError):            # not even one
        _run(P, B, torch, 1 << 16)
