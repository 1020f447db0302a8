"""The work a user of this library has it do, as timed cases.

Every trajectory case is one segment of a run: cavmd_step(steps), then the read-out a program takes
at the end of a segment (the energies, the cell dipoles, the photon coordinates and the nuclear
state). The sizes are the workloads of cavmd_synth (c1..c5 and the periodic 33-water cells), with
odd and trimmed sizes beside them. Two cases call the library's other entry points: the fit of the
Born-charge network, and the allocation-free field and kick on device arrays.

exact() restates the method in plain 64-bit NumPy (generalised eigenproblems by LAPACK, charges
mixed to 1e-13), from the formulas of include/cavmd.h and the same inputs.
"""
import math

import numpy as np
import torch

import cavmd_synth as cs
import paper_2512_03277_gb300 as P
from paper_2512_03277_gb300 import cavmd as B

KB = 3.166811563e-6
DT = 0.5 * cs.FS


def listed():
    return [
        # config 1, the smallest system: eight waters in a 1D cavity, a long run of short steps
        # (latency of the launches and of one water's serial chain)
        dict(name="box_8w_16m", kind="waters", cells=8, kx=16, ky=0, charges="mulliken", mixed=False, steps=30, acf=0),
        # config 2: 4096 waters, 512 line modes, plain FP64, spectra accumulated on the device and read
        dict(name="slab_4096w_512m", kind="waters", cells=4096, kx=512, ky=0, charges="mulliken", mixed=False,
             steps=25, acf=256),
        # the paper's own dipole derivative (forward finite differences every third step), at a ragged
        # trimmed size of config 2
        dict(name="born_fd_1237w_302m", kind="waters", cells=1237, kx=302, ky=0, charges="born_fd", mixed=False,
             steps=9, acf=0),
        # mode functions that follow the centres of mass, on the tensor-core coupling
        dict(name="moving_8191w_1024m", kind="waters", cells=8191, kx=32, ky=32, charges="born_mlp", mixed=True,
             steps=6, acf=0, moving=True),
        # config 4: the learned Born charges with the mixed-precision coupling
        dict(name="learned_16384w_1024m", kind="waters", cells=16384, kx=32, ky=32, charges="born_mlp", mixed=True,
             steps=10, acf=0),
        # config 5: the full-scale angle-resolved run, spectra accumulated on the device
        dict(name="full_262144w_8192m", kind="waters", cells=262144, kx=64, ky=128, charges="born_mlp", mixed=True,
             steps=50, acf=1024),
        # config 3 trimmed: a few hundred uneven clusters (the last wave of the persistent launch counts)
        dict(name="clusters_301c_256m", kind="clusters", cells=301, kx=16, ky=16, mixed=True, steps=4),
        # config 3: uneven clusters in bulk
        dict(name="clusters_16384c_4096m", kind="clusters", cells=16384, kx=64, ky=64, mixed=True, steps=2),
        # the paper's system: periodic cubes of 33 waters, Gamma point
        dict(name="periodic_304c_33w", kind="periodic", cells=304, waters=33, kx=512, ky=0, kgrid=1, steps=1),
        # the paper's 3 x 3 x 3 k-grid, on smaller cubes of the same density
        dict(name="kgrid_24c_8w", kind="periodic", cells=24, waters=8, kx=128, ky=0, kgrid=3, steps=1),
        # one pass of the network's fit: loss and gradient over the set, and its predictions
        dict(name="network_fit_20001w", kind="network", cells=20001),
        # the allocation-free field and kick on a caller's device arrays
        dict(name="field_kick_16384c_1024m", kind="field_kick", cells=16384, kx=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["waters", "waters", "waters", "clusters", "periodic", "network", "field_kick"])
    if kind == "waters":
        mixed = rng.random() < 0.5
        cells = _log(rng, 8, 100000 if mixed else 20000)
        kx, ky = (rng.choice([8, 16, 32, 64]), rng.choice([8, 16, 32, 64])) if mixed else (2 * _log(rng, 8, 300), 0)
        charges = rng.choice(["mulliken", "born_mlp"] if mixed else ["mulliken", "born_fd", "born_mlp"])
        steps = 9 if charges == "born_fd" else rng.choice([3, 10, 20])
        c = dict(kind=kind, cells=cells, kx=kx, ky=ky, charges=charges, mixed=mixed, steps=steps,
                 acf=rng.choice([0, 64]))
        if mixed and rng.random() < 0.25:
            c["moving"] = True
        return c
    if kind == "clusters":
        k = rng.choice([8, 16, 32])
        return dict(kind=kind, cells=_log(rng, 20, 8000), kx=k, ky=k, mixed=rng.random() < 0.5, steps=2)
    if kind == "periodic":
        grid = rng.choice([1, 1, 2, 3])
        waters = rng.randint(4, 33 if grid == 1 else 8)
        return dict(kind=kind, cells=rng.randint(1, 150 if grid == 1 else 30), waters=waters, kx=2 * rng.randint(8, 150),
                    ky=0, kgrid=grid, steps=1)
    if kind == "network":
        return dict(kind=kind, cells=_log(rng, 100, 50000))
    return dict(kind=kind, cells=_log(rng, 50, 30000), kx=_log(rng, 10, 1000))


# ------------------------------------------------------------------------------------- inputs

def _momenta(rng, system):
    """Maxwell-Boltzmann momenta at 300 K without centre-of-mass motion of any cell."""
    m = np.array(cs.MASS_AMU)[system.species] * cs.AMU
    off = system.cell_offset
    v = rng.normal(size=(system.n_atoms, 3)) * np.sqrt(KB * 300.0 / m)[:, None]
    pc = np.add.reduceat(m[:, None] * v, off[:-1], axis=0) / np.add.reduceat(m, off[:-1])[:, None]
    return m[:, None] * (v - np.repeat(pc, np.diff(off), axis=0))


def _rigid(rng, n):
    """n uniform random rotation matrices."""
    q = rng.normal(size=(n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                     [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                     [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]).transpose(2, 0, 1)


def _modes(case, line_length, waters):
    if case["ky"] == 0:
        if case["cells"] <= 16:      # the 1D cavity of config 1
            return cs.standing_modes(case["kx"], 2000.0, 0.002)
        return cs.line_modes(case["kx"], line_length, 0.001, k_max=10.0 * np.pi / line_length)
    side = math.sqrt(waters / cs.WATER_DENSITY / 30.0)
    return cs.grid_modes(case["kx"], case["ky"], 2 * np.pi / side, 2 * np.pi / side, 2000.0, 0.001)


def _inputs(case, seed):
    """(system, modes, lattice) of a trajectory case."""
    rng = np.random.default_rng(seed)
    n = case["cells"]
    lattice = None
    if case["kind"] == "waters":
        length = n / cs.WATER_DENSITY / 900.0
        if case["ky"]:
            side = math.sqrt(n / cs.WATER_DENSITY / 30.0)
            box = (side, side, 30.0)
        else:
            box = (2000.0, 0.0, 0.0) if n <= 16 else (length, 30.0, 30.0)
        centres = rng.uniform(size=(n, 3)) * np.array(box)
        pos = cs.water_batch(rng, centres)
        system = cs.System(species=np.tile(np.array([cs.ELEM_O, cs.ELEM_H, cs.ELEM_H], np.int32), n),
                           cell_offset=np.arange(0, 3 * n + 1, 3, dtype=np.int32), r=pos.reshape(-1, 3).copy(),
                           p=np.zeros((3 * n, 3)), R_ref=centres)
        modes = _modes(case, length, n)
    elif case["kind"] == "clusters":
        # (H2O)_1 .. (H2O)_8 at liquid density: rotated and newly disturbed copies of a pool of
        # packed clusters (packing every one of a large set anew takes minutes on the host)
        pool_n = 12
        pool = [cs.cluster_batch(rng, [w] * pool_n, np.zeros((pool_n, 3))).r.reshape(pool_n, 3 * w, 3)
                for w in range(1, 9)]
        sizes = np.random.default_rng(n).integers(1, 9, size=n)   # the case's own, whatever the seed
        off = np.concatenate([[0], np.cumsum(3 * sizes)]).astype(np.int32)
        side = math.sqrt(float(sizes.sum()) / cs.WATER_DENSITY / 30.0)
        centres = rng.uniform(size=(n, 3)) * np.array([side, side, 30.0])
        r = np.empty((off[-1], 3))
        for w in range(1, 9):
            at = np.flatnonzero(sizes == w)
            x = np.einsum("nij,naj->nai", _rigid(rng, len(at)), pool[w - 1][rng.integers(0, pool_n, len(at))])
            r[(off[at][:, None] + np.arange(3 * w)).ravel()] = (x + rng.normal(0.0, 0.01, x.shape)
                                                                + centres[at][:, None]).reshape(-1, 3)
        system = cs.System(species=np.tile(np.array([cs.ELEM_O, cs.ELEM_H, cs.ELEM_H], np.int32), off[-1] // 3),
                           cell_offset=off, r=r, p=np.zeros_like(r), R_ref=centres)
        modes = _modes(case, 0.0, float(sizes.sum()))
    else:
        w = case["waters"]
        side = (w / 33.0) ** (1.0 / 3.0) * 10.0 * cs.ANGSTROM
        pool_n = min(n, 8)
        pool, lattice = cs.periodic_water_cells(rng, np.zeros((pool_n, 3)), n_waters=w, side=side)
        x = pool.r.reshape(pool_n, 3 * w, 3)[np.arange(n) % pool_n]
        # the cube's own symmetries (axis permutations and reflections), and new displacements
        perm = np.array([[0, 1, 2], [0, 2, 1], [1, 0, 2], [1, 2, 0], [2, 0, 1], [2, 1, 0]])[rng.integers(0, 6, n)]
        x = np.take_along_axis(x, np.broadcast_to(perm[:, None, :], x.shape), axis=2)
        x = x * rng.choice([-1.0, 1.0], size=(n, 1, 3)) + rng.normal(0.0, 0.01, x.shape)
        centres = np.zeros((n, 3))
        centres[:, 0] = (np.arange(n) + 0.5) * side
        system = cs.System(species=np.tile(np.array([cs.ELEM_O, cs.ELEM_H, cs.ELEM_H], np.int32), n * w),
                           cell_offset=np.arange(0, 3 * w * n + 1, 3 * w, dtype=np.int32),
                           r=(x + centres[:, None]).reshape(-1, 3), p=np.zeros((3 * w * n, 3)), R_ref=centres)
        line = max(n, 16) * side
        modes = cs.line_modes(case["kx"], line, 0.001, k_max=10.0 * np.pi / line)
    system.p = _momenta(rng, system)
    return system, modes, lattice


def _network_inputs(case, seed):
    """Waters near their minimum, their net charges, and Born tensors that the fit is shown."""
    rng = np.random.default_rng(seed)
    n = case["cells"]
    r = cs.water_batch(rng, np.zeros((n, 3)), noise=0.06)
    Q = np.empty((n, 3))
    Q[:, 0] = rng.normal(-0.55, 0.03, n)
    Q[:, 1] = -0.5 * Q[:, 0] + rng.normal(0.0, 0.01, n)
    Q[:, 2] = -Q[:, 0] - Q[:, 1]
    Z = Q.reshape(-1, 1, 1) * np.eye(3) + rng.normal(0.0, 0.03, (3 * n, 3, 3))
    params = B.trained_born_mlp().astype(np.float64) * (1.0 + rng.normal(0.0, 0.05, B.MLP_NPARAMS))
    return r.reshape(-1, 3), Q.ravel(), Z, params.astype(np.float32)


def _kick_inputs(case, seed):
    rng = np.random.default_rng(seed)
    n, m = case["cells"], case["kx"]
    w = rng.normal(size=m) * 1e-3
    n_at = 3 * n
    F, b = rng.normal(size=(n_at, 3)) * 0.05, rng.normal(size=(n_at, 3)) * 0.4
    inv_mass = 1.0 / np.tile(np.array(cs.MASS_AMU)[[0, 1, 1]] * cs.AMU, n)
    p = rng.normal(size=(n_at, 3)) * 5.0
    U = np.cos(rng.uniform(0, 2 * np.pi, (m, 1)) + rng.uniform(0, 0.2, (m, 1)) * rng.uniform(0, 400.0, n))
    return U, w, F, b, inv_mass, p


# ------------------------------------------------------------------------------------- a pass

def prepare(case, seed):
    if case["kind"] == "network":
        r, Q, Z, params = _network_inputs(case, seed)
        net = B.BornMLP(params)
        net.cavmd_mlp_set_data(np.tile(np.array([cs.ELEM_O, cs.ELEM_H, cs.ELEM_H], np.int32), case["cells"]), r, Q, Z)
        return dict(kind="network", net=net)
    if case["kind"] == "field_kick":
        n, m = case["cells"], case["kx"]
        U, w, F, b, inv_mass, p = (torch.from_numpy(x).cuda() for x in _kick_inputs(case, seed))
        off = torch.arange(0, 3 * n + 1, 3, dtype=torch.int32, device="cuda")
        return dict(kind="field_kick", n=n, m=m, off=off, U=U, w=w, F=F, b=b, inv_mass=inv_mass, p=p,
                    E=torch.empty(n, dtype=torch.float64, device="cuda"),
                    ek=torch.empty(1, dtype=torch.float64, device="cuda"))
    system, modes, lattice = _inputs(case, seed)
    o = P.default_options()
    if case.get("mixed"):
        o.precision = B.PREC_MIXED_BF16X3
    else:
        o.photon_init = P.PHOTON_ZERO    # photons at rest (configs 1 and 2); the mixed runs start relaxed
    charges = case.get("charges", "mulliken")
    o.charge_model = {"mulliken": B.CHARGE_MULLIKEN, "born_fd": B.CHARGE_BORN_FD,
                      "born_mlp": B.CHARGE_BORN_MLP}[charges]
    o.acf_lags = case.get("acf", 0)
    o.graph_chunk = min(case["steps"], 50)
    if case.get("moving"):
        o.mode_positions = 1
    if case.get("kgrid", 1) > 1:
        for k in range(3):
            o.kgrid[k] = case["kgrid"]
    ctx = P.Context(system, cs.load_water_params(), modes, o, lattice=lattice)
    if charges == "born_mlp":
        ctx.cavmd_load_born_mlp(B.trained_born_mlp())
    return dict(kind=case["kind"], ctx=ctx, mixed=bool(case.get("mixed")), steps=case["steps"],
                acf=0 < case.get("acf", 0) <= 256)


ENERGIES = ("e_kin", "e_dftb", "e_photon", "e_coupling", "e_dse", "e_photon_free", "e_total", "temperature")


def run(state):
    if state["kind"] == "network":
        loss, grad = state["net"].cavmd_mlp_loss_grad()
        Z = state["net"].cavmd_mlp_predict().astype(np.float32)   # a single-precision network in a double array
        return dict(loss=loss, grad=grad, Z=Z)
    if state["kind"] == "field_kick":
        s = state
        B.cavmd_field_kick_noalloc(s["n"], s["m"], s["off"].data_ptr(), s["U"].data_ptr(), s["w"].data_ptr(),
                                   s["F"].data_ptr(), s["b"].data_ptr(), s["inv_mass"].data_ptr(), 0.5 * DT,
                                   s["p"].data_ptr(), s["E"].data_ptr(), s["ek"].data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
        return dict(p=s["p"], E=s["E"], e_kin=s["ek"])
    ctx = state["ctx"]
    ctx.cavmd_step(state["steps"])
    obs = ctx.cavmd_observables()
    out = {k: obs[k] for k in ENERGIES + ("M", "q", "p", "D")}
    if state["mixed"]:   # the mixed-precision contraction gives D, and the photons it drives, to single precision
        out.update({k: out[k].astype(np.float32) for k in ("q", "p", "D")})
    frame = ctx.cavmd_get_state()
    out["r_nuc"], out["p_nuc"] = frame["r"], frame["p"]
    if state["acf"]:
        out["acf"] = ctx.cavmd_autocorrelation()[0]
    return out


def work(case):
    n = case["cells"]
    if case["kind"] == "network":
        at = 3 * n                            # positions, charges, targets in; predictions and gradient out
        per = 2 * (32 * 128 + 128 * 128 + 128 * 9)
        return {"bytes": at * (24 + 8 + 72 + 36) + 8 * B.MLP_NPARAMS, "flops": 4.0 * per * at}
    m = case["kx"] * max(1, case["ky"]) if "ky" in case else case["kx"]
    if case["kind"] == "field_kick":
        return {"bytes": 8.0 * (n * m + m + n * (4 * 9 + 3 + 1)), "flops": 2.0 * n * m + 40.0 * n}
    # a step: every occupied-virtual eigenproblem taken once with its self-consistency (5 passes of
    # 2 n^3), the mode contraction both ways (4 flops an element), the state read and written once
    waters = {"waters": 1.0, "clusters": 4.5}.get(case["kind"], float(case.get("waters", 1)))
    points, wide = (1, 1) if case.get("kgrid", 1) == 1 else ((case["kgrid"] ** 3 + 1) // 2, 4)
    n_orb = 6.0 * waters
    cube = n_orb ** 3 if case["kind"] != "clusters" else 216.0 * 8 * 9 * 9 * 8 / 32.0   # mean of w^3 over 1..8
    scf = n * points * wide * 10.0 * cube
    rows = 1.0 + (9.0 / 3.0 if case.get("charges") == "born_fd" else 0.0)
    net = 2 * (32 * 128 + 128 * 128 + 128 * 9) * 3.0 * n if case.get("charges") == "born_mlp" else 0.0
    both = 4.0 * n * m if not case["ky"] else 2 * 4.0 * n * 2 * case["kx"] * case["ky"]
    atoms = 3.0 * waters * n
    state = 8.0 * (atoms * 12 + n * (3 + points * wide * n_orb ** 2 * 2) + 8 * m)
    return {"bytes": case["steps"] * state, "flops": case["steps"] * (scf * rows + both + net)}


# --------------------------------------------------------------------- the method in 64 bits

def _radial(par, r, sk):
    a, b, c1, c2 = par
    x = (r - sk.r_cut + sk.taper) / sk.taper
    f = np.where(x <= 0, 1.0, np.where(x >= 1, 0.0, 0.5 * (1 + np.cos(np.pi * x))))
    df = np.where((x > 0) & (x < 1), -0.5 * np.pi / sk.taper * np.sin(np.pi * x), 0.0)
    e, poly = a * np.exp(-b * r), 1 + c1 * r + c2 * r * r
    return e * poly * f, e * ((c1 + 2 * c2 * r - b * poly) * f + poly * df)


class _Cells:
    """SCC-DFTB of a batch of cells of one composition: pos (B, nat, 3)."""

    def __init__(self, sk, species):
        self.sk, self.sp = sk, np.asarray(species)
        self.no = sk.norb[self.sp].astype(int)
        self.off = np.concatenate([[0], np.cumsum(self.no)])
        self.n = int(self.off[-1])
        self.at = np.repeat(np.arange(len(self.sp)), self.no)
        self.z = sk.zval[self.sp]
        self.nocc = int(round(self.z.sum())) // 2

    def _blocks(self, table, A, C, r, e, grad):
        """<A|C> block (B, na, nc) and its derivative along the vector from A to C (B, 3, na, nc)."""
        sk, ea, ec = self.sk, self.sp[A], self.sp[C]
        na, nc = self.no[A], self.no[C]
        blk = np.zeros((len(r), na, nc))
        g = np.zeros((len(r), 3, na, nc)) if grad else None
        eye = np.eye(3)
        de = (eye - e[:, :, None] * e[:, None, :]) / r[:, None, None]
        v, dv = _radial(table[ea, ec, 0], r, sk)
        blk[:, 0, 0] = v
        if grad:
            g[:, :, 0, 0] = dv[:, None] * e
        for on, t, sign in ((nc, table[ea, ec, 1], 1.0), (na, table[ec, ea, 1], -1.0)):
            if on != 4:
                continue
            v, dv = _radial(t, r, sk)
            d1 = sign * (de * v[:, None, None] + e[:, :, None] * e[:, None, :] * dv[:, None, None])
            if sign > 0:
                blk[:, 0, 1:] = e * v[:, None]
                if grad:
                    g[:, :, 0, 1:] = d1
            else:
                blk[:, 1:, 0] = -e * v[:, None]
                if grad:
                    g[:, :, 1:, 0] = d1
        if na == 4 and nc == 4:
            s, ds = _radial(table[ea, ec, 2], r, sk)
            p, dp = _radial(table[ea, ec, 3], r, sk)
            ee = e[:, :, None] * e[:, None, :]
            blk[:, 1:, 1:] = ee * (s - p)[:, None, None] + eye * p[:, None, None]
            if grad:
                dee = np.einsum("bki,bj->bkij", de, e) + np.einsum("bi,bkj->bkij", e, de)
                g[:, :, 1:, 1:] = (dee * (s - p)[:, None, None, None] + e[:, :, None, None] * (
                    ee * (ds - dp)[:, None, None] + eye * dp[:, None, None])[:, None])
        return blk, g

    def solve(self, pos, q0=None, forces=True):
        sk, n, nat, Bn = self.sk, self.n, len(self.sp), len(pos)
        H0, S = np.zeros((Bn, n, n)), np.tile(np.eye(n), (Bn, 1, 1))
        for a in range(nat):
            for k in range(self.no[a]):
                H0[:, self.off[a] + k, self.off[a] + k] = sk.onsite[self.sp[a], 1 if k else 0]
        d = pos[:, None] - pos[:, :, None]
        c = 2.0 / (sk.hubbard[self.sp][:, None] + sk.hubbard[self.sp][None])
        gam = 1.0 / np.sqrt((d * d).sum(-1) + c * c)
        pairs = []
        for A in range(nat):
            for C in range(A + 1, nat):
                v = pos[:, C] - pos[:, A]
                r = np.sqrt((v * v).sum(-1))
                e = v / r[:, None]
                sa, sc = slice(self.off[A], self.off[A + 1]), slice(self.off[C], self.off[C + 1])
                h, gh = self._blocks(sk.h0, A, C, r, e, forces)
                s, gs = self._blocks(sk.s, A, C, r, e, forces)
                H0[:, sa, sc], H0[:, sc, sa] = h, h.transpose(0, 2, 1)
                S[:, sa, sc], S[:, sc, sa] = s, s.transpose(0, 2, 1)
                pairs.append((A, C, r, e, sa, sc, gh, gs))
        Li = np.linalg.inv(np.linalg.cholesky(S))
        LiT = Li.transpose(0, 2, 1)

        def out_of(q):
            sh = np.einsum("bij,bj->bi", gam, q - self.z)[:, self.at]
            Hp = Li @ (H0 + 0.5 * S * (sh[:, :, None] + sh[:, None])) @ LiT
            eps, V = np.linalg.eigh(0.5 * (Hp + Hp.transpose(0, 2, 1)))
            Co = LiT @ V[:, :, :self.nocc]
            Pm = 2 * Co @ Co.transpose(0, 2, 1)
            return np.add.reduceat((Pm * S).sum(-1), self.off[:-1], axis=1), Pm, Co, eps

        q = np.tile(self.z, (Bn, 1)) if q0 is None else q0
        hist = []
        for it in range(300):   # Anderson mixing of the populations, every cell by itself
            qo, Pm, Co, eps = out_of(q)
            f = qo - q
            if np.abs(f).max() < 2e-13 or (it > 60 and np.abs(f).max() < 2e-12):
                break
            hist = (hist + [(q, f)])[-4:]
            dq, df = q, f
            if len(hist) > 1:
                dF = np.stack([f - h[1] for h in hist[:-1]], -1)
                dQ = np.stack([q - h[0] for h in hist[:-1]], -1)
                G = dF.transpose(0, 2, 1) @ dF
                G += 1e-13 * np.trace(G, axis1=1, axis2=2)[:, None, None] * np.eye(G.shape[1]) + 1e-300 * np.eye(G.shape[1])
                x = np.linalg.solve(G, dF.transpose(0, 2, 1) @ f[:, :, None])
                x = np.where(np.abs(x).max(1, keepdims=True) < 20, x, 0.0)
                dq, df = q - (dQ @ x)[:, :, 0], f - (dF @ x)[:, :, 0]
            q = dq + 0.6 * df
        q = qo
        out = {"q": q, "Q": self.z - q, "mu": np.einsum("ba,bak->bk", self.z - q, pos)}
        if not forces:
            return out
        dz = q - self.z
        sh = np.einsum("bij,bj->bi", gam, dz)
        W = 2 * (Co * eps[:, None, :self.nocc]) @ Co.transpose(0, 2, 1)
        E = (Pm * H0).sum((-1, -2)) + 0.5 * np.einsum("bi,bij,bj->b", dz, gam, dz)
        F = np.zeros_like(pos)
        for A, C, r, e, sa, sc, gh, gs in pairs:
            Pab = Pm[:, sa, sc]
            X = Pab * (0.5 * (sh[:, A] + sh[:, C]))[:, None, None] - W[:, sa, sc]
            g = 2 * (np.einsum("bij,bkij->bk", Pab, gh) + np.einsum("bij,bkij->bk", X, gs))
            g += (dz[:, A] * dz[:, C] * -r * gam[:, A, C] ** 3)[:, None] * e
            ar, br = sk.rep[self.sp[A], self.sp[C]]
            v, dv = _radial((ar, br, 0.0, 0.0), r, sk)
            E += v
            g += dv[:, None] * e
            F[:, C] -= g
            F[:, A] += g
        return {**out, "E": E, "F": F}


def _features(pos):
    """Network features and local frames of waters, pos (B, 3, 3): (B, 3, 32), (B, 3, 3, 3)."""
    Bn, rc = len(pos), 8.0
    X, R = np.zeros((Bn, 3, 32)), np.zeros((Bn, 3, 3, 3))
    for j in range(3):
        k, l = [a for a in range(3) if a != j]
        dk, dl = pos[:, k] - pos[:, j], pos[:, l] - pos[:, j]
        rk, rl = np.sqrt((dk * dk).sum(-1)), np.sqrt((dl * dl).sum(-1))
        fk, fl = 0.5 * (np.cos(np.pi * rk / rc) + 1), 0.5 * (np.cos(np.pi * rl / rc) + 1)
        for a, r, f in ((k, rk, fk), (l, rl, fl)):
            o = 11 * (a > 0)
            X[:, j, o:o + 11] += np.exp(-2.0 * (r[:, None] - (0.8 + 0.7 * np.arange(11))) ** 2) * f[:, None]
        cos = (dk * dl).sum(-1) / (rk * rl)
        rad = np.exp(-0.05 * (rk ** 2 + rl ** 2)) * fk * fl
        for zi, z in enumerate((1, 2, 4, 8)):
            for li, lam in enumerate((1.0, -1.0)):
                X[:, j, 22 + 2 * zi + li] = 2.0 ** (1 - z) * (1 + lam * cos) ** z * rad
        X[:, j, 30 + (j > 0)] = 1.0
        near = (rk <= rl)[:, None]
        d1, r1 = np.where(near, dk, dl), np.where(near[:, 0], rk, rl)
        d2 = np.where(near, dl, dk)
        e1 = d1 / r1[:, None]
        v = d2 - (d2 * e1).sum(-1)[:, None] * e1
        e2 = v / np.sqrt((v * v).sum(-1))[:, None]
        R[:, j] = np.stack([e1, e2, np.cross(e1, e2)], 1)
    return X, R


def _weights(params):
    """The network's parameters rounded to bfloat16, as float64 arrays."""
    f = torch.from_numpy(np.asarray(params, np.float32)).to(torch.bfloat16).double().numpy()
    out, o = [], 0
    for shape in ((128, 32), (128,), (128, 128), (128,), (9, 128), (9,)):
        out.append(f[o:o + math.prod(shape)].reshape(shape))
        o += math.prod(shape)
    return out


def _born(X, R, Q, weights):
    """Born tensors (B, 3, 3, 3) and what the gradient needs."""
    W1, b1, W2, b2, W3, b3 = weights
    z1 = X @ W1.T + b1
    h1 = z1 / (1 + np.exp(-z1))
    z2 = h1 @ W2.T + b2
    h2 = z2 / (1 + np.exp(-z2))
    T = (h2 @ W3.T + b3).reshape(X.shape[0], 3, 3, 3)
    Z = R.transpose(0, 1, 3, 2) @ T @ R
    return Z - Z.mean(1, keepdims=True) + Q[:, :, None, None] * np.eye(3), (z1, h1, z2, h2)


def _dsilu(z):
    s = 1 / (1 + np.exp(-z))
    return s * (1 + z * (1 - s))


class _Matter:
    def __init__(self, system, charges):
        self.off, self.sp, self.charges = np.asarray(system.cell_offset), np.asarray(system.species), charges
        sk = cs.load_water_params()
        self.mass = sk.mass[self.sp]
        self.cell = np.repeat(np.arange(len(self.off) - 1), np.diff(self.off))
        nat = np.diff(self.off)
        self.groups = [(_Cells(sk, self.sp[self.off[c[0]]:self.off[c[0] + 1]]), c)
                       for c in (np.flatnonzero(nat == a) for a in np.unique(nat))]
        self.q = np.zeros(len(self.sp))
        self.b = np.zeros((len(self.sp), 3))
        self.weights = _weights(B.trained_born_mlp()) if charges == "born_mlp" else None
        self.evals = 0

    def __call__(self, r):
        F, E, M = np.zeros_like(r), np.zeros(len(self.off) - 1), np.zeros(len(self.off) - 1)
        for cells, which in self.groups:
            nat = len(cells.sp)
            idx = self.off[which][:, None] + np.arange(nat)
            pos = r[idx]
            o = cells.solve(pos, None if self.evals == 0 else self.q[idx])
            F[idx], E[which], M[which], self.q[idx] = o["F"], o["E"], o["mu"][:, 0], o["q"]
            if self.charges == "mulliken":
                self.b[idx] = o["Q"][..., None] * np.array([1.0, 0.0, 0.0])
            elif self.charges == "born_mlp":
                X, R = _features(pos)
                self.b[idx] = _born(X, R, o["Q"], self.weights)[0][:, :, 0, :]
            elif self.evals % 3 == 0:
                h = 1e-3
                b = np.zeros(pos.shape)
                for j in range(nat):
                    for k in range(3):
                        moved = pos.copy()
                        moved[:, j, k] += h
                        b[:, j, k] = (cells.solve(moved, o["q"], False)["mu"][:, 0] - M[which]) / h
                self.b[idx] = b
        self.evals += 1
        return F, E, M


def _trajectory(case, seed):
    system, modes, _ = _inputs(case, seed)
    matter = _Matter(system, case.get("charges", "mulliken"))
    off, cell, mass = matter.off, matter.cell, matter.mass
    r, p = system.r.copy(), system.p.copy()
    w, lam, k = modes.omega, modes.lam, modes.k
    moving = bool(case.get("moving"))
    mc = np.add.reduceat(mass, off[:-1])

    def functions():
        R = np.add.reduceat(mass[:, None] * r, off[:-1], axis=0) / mc[:, None] if moving else system.R_ref
        ph = k @ R.T + modes.phi[:, None]
        return np.cos(ph), (np.sin(ph) if moving else None)

    u, s = functions()
    F, E, M = matter(r)
    D = lam * (u @ M)
    q, pq = (D / w if case.get("mixed") else np.zeros_like(D)), np.zeros_like(D)
    xs = [np.concatenate([q, [M.sum()]])]

    def half(tau):
        nonlocal p, q, pq
        c, y = D / w, q - D / w
        sn, cn = np.sin(w * tau), np.cos(w * tau)
        Y = lam * (y * sn + pq * (1 - cn) / w)
        p = p + tau * F + (u.T @ Y)[cell][:, None] * matter.b
        if moving:
            p = p + (mass / mc[cell] * M[cell])[:, None] * (-(s.T @ (Y[:, None] * k)))[cell]
        q, pq = c + y * cn + pq * sn / w, pq * cn - w * y * sn

    for _ in range(case["steps"]):
        half(0.5 * DT)
        r = r + DT * p / mass[:, None]
        if moving:
            u, s = functions()
        F, E, M = matter(r)
        D = lam * (u @ M)
        half(0.5 * DT)
        xs.append(np.concatenate([q, [M.sum()]]))
    kin = float((p * p / (2 * mass[:, None])).sum())
    ph = float((0.5 * pq ** 2 + 0.5 * (w * q - D) ** 2).sum())
    out = dict(e_kin=kin, e_dftb=float(E.sum()), e_photon=ph, e_coupling=float(-(w * q * D).sum()),
               e_dse=float(0.5 * (D * D).sum()), e_photon_free=float((0.5 * (pq ** 2 + (w * q) ** 2)).sum()),
               e_total=kin + float(E.sum()) + ph, temperature=2 * kin / (3 * len(mass) * KB), M=M, q=q, p=pq, D=D,
               r_nuc=r, p_nuc=p)
    if 0 < case.get("acf", 0) <= 256:
        x = np.array(xs)
        x, n = x - x.mean(0), len(xs)
        out["acf"] = np.zeros((x.shape[1], case["acf"]))
        for lag in range(min(n, case["acf"])):
            out["acf"][:, lag] = (x[lag:] * x[:n - lag]).sum(0) / (n - lag)
    return out


def exact(case, seed):
    if case["kind"] == "periodic":   # Ewald sums and 200-orbital problems in NumPy: minutes a pass
        return None
    if case["kind"] == "network":
        r, Q, Zref, params = _network_inputs(case, seed)
        wt = _weights(params)
        X, R = _features(r.reshape(-1, 3, 3))
        Q, Zref = Q.reshape(-1, 3), Zref.reshape(-1, 3, 3, 3)
        Z, (z1, h1, z2, h2) = _born(X, R, Q, wt)
        n = Z.shape[0] * 3
        gZ = 2 * (Z - Zref) / (9 * n)
        gZ = gZ - gZ.mean(1, keepdims=True)
        flat = lambda a: a.reshape(n, -1)  # noqa: E731
        gy = flat(R @ gZ @ R.transpose(0, 1, 3, 2))
        g2 = (gy @ wt[4]) * _dsilu(flat(z2))
        g1 = (g2 @ wt[2]) * _dsilu(flat(z1))
        grad = [g1.T @ flat(X), g1.sum(0), g2.T @ flat(h1), g2.sum(0), gy.T @ flat(h2), gy.sum(0)]
        return dict(loss=float(((Z - Zref) ** 2).sum() / (9 * n)), grad=np.concatenate([g.ravel() for g in grad]),
                    Z=Z.reshape(-1, 3, 3))
    if case["kind"] == "field_kick":
        U, w, F, b, inv_mass, p = _kick_inputs(case, seed)
        E = w @ U
        p = p + 0.5 * DT * F + np.repeat(E, 3)[:, None] * b
        return dict(p=p, E=E, e_kin=np.array([0.5 * (p * p * inv_mass[:, None]).sum()]))
    # the time of the restatement: eigenproblems of every cell, about nine charge iterations an evaluation
    rows = case["steps"] + 1 + (9 * (1 + case["steps"] // 3) if case.get("charges") == "born_fd" else 0)
    one = 8e-6 if case["kind"] == "waters" else 6e-4
    if case["cells"] * rows * 10 * one > 18.0 or case["cells"] * case["kx"] * max(1, case["ky"]) > 2.5e7:
        return None
    return _trajectory(case, seed)
