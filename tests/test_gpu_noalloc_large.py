"""The allocation-free field and kick above 524,288 cells, where its blocks take 32 cells instead of
16, and on both sides of that line: ragged last blocks, empty cells, cells of one to three atoms.

Tolerances: a field is three products summed in FP64, so 4 ulp of the largest sum of their magnitudes;
a momentum two multiply-adds on it; the kinetic energy, a sum of positive terms, 1e-12 of itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LINE = 524288


@pytest.mark.parametrize("n", [LINE - 3, LINE, LINE + 1, LINE + 37])
def test_kick_around_the_block_size_line(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2512_03277_gb300 as P
    from paper_2512_03277_gb300 import cavmd as B
    P.load_library()
    rng = np.random.default_rng(3)
    m, tau = 3, 0.7
    nat = rng.integers(0, 4, n)
    off = np.concatenate([[0], np.cumsum(nat)]).astype(np.int32)
    na = int(off[-1])
    U, W = rng.normal(size=(m, n)), rng.normal(size=m)
    F, b, p = (rng.normal(size=(na, 3)) for _ in range(3))
    im = rng.uniform(0.1, 1.0, na)
    t = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in
         dict(off=off, U=U, W=W, F=F, b=b, im=im, p=p).items()}
    E = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    ek = torch.empty(1, dtype=torch.float64, device="cuda")
    B.cavmd_field_kick_noalloc(n, m, t["off"].data_ptr(), t["U"].data_ptr(), t["W"].data_ptr(), t["F"].data_ptr(),
                               t["b"].data_ptr(), t["im"].data_ptr(), tau, t["p"].data_ptr(), E.data_ptr(),
                               ek.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    e = W @ U
    e_tol = 4 * 2.0 ** -52 * (np.abs(W) @ np.abs(U)).max()
    assert np.abs(E.cpu().numpy() - e).max() <= e_tol
    ref = p + e[np.repeat(np.arange(n), nat)][:, None] * b + tau * F
    got = t["p"].cpu().numpy()
    assert np.abs(got - ref).max() <= np.abs(b).max() * e_tol + 4 * 2.0 ** -52 * np.abs(ref).max()
    kin = 0.5 * np.sum(im[:, None] * got * got)
    assert abs(ek.item() - kin) < 1e-12 * kin
