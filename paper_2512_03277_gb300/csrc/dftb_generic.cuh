// Batched SCC-DFTB for cells of any composition up to 64 orbitals, e.g. water clusters (H2O)_n
// with n <= 10 (6n orbitals), in one persistent launch per evaluation.
//
// The method is the one of the water kernel in dftb_kernel.cu (second-order SCC-DFTB, section
// "Computational details"): warm-started S-orthonormal basis, SCC iterations with Jacobi sweeps or
// the second-order occupied-virtual update, Anderson mixing, analytic forces. The mapping to the
// machine is made for matrices too large for a lane group, on a GPU whose FP64 pipe (2 FMA per
// clock per SM) is the only bottleneck, so what counts is the number of FP64 warp instructions:
//   * work items: a cell of more than 32 orbitals takes a whole 256-thread block, smaller cells
//     take 128 threads each, two per block (128 and 64 threads left the FP64 pipe 55 % busy with
//     eight warps per SM; these 65 %: 16,384 clusters 24 -> 19.5 ms with the pairs sorted by kind). A persistent grid pulls items from a queue ordered by
//     decreasing size, so large cells start first and small ones fill the tail;
//   * every matrix product spreads its output entries evenly over the cell's threads (R entries
//     per thread per pass, each summed over k in increasing order), so nearly every lane of
//     every FP64 instruction does useful work whatever the orbital count; the results do not
//     depend on R or on the grid size;
//   * per SCC iteration only what the update needs is formed: H C, the diagonal and the
//     occupied-virtual block of C^T H C, K^2 in its two diagonal blocks from the compact
//     occupied-virtual generator, C V, and S C_occ for the Mulliken populations;
//   * four n x n matrices per cell in shared memory: SH (the symmetric S in the strict lower
//     triangle, the symmetric H0 in the upper triangle and on the diagonal, since S_ii = 1),
//     C, A and Y, plus the compact generator and the warm path's n x n_occ buffer. A (H2O)_8 cell (48
//     orbitals) takes 108 KB, so two large cells share an SM.
#pragma once

#include "cavmd_internal.cuh"

namespace {

constexpr int GNHIST = 6;              // largest Anderson history (current + 5 previous iterates)
constexpr int G_MAX_SWEEPS = 40;            // default bound on the Jacobi sweeps of a cold start
constexpr double G_JACOBI_TOL = 1e-15;
constexpr double G_MIN_GAP = 1e-3;
constexpr double G_EIG_TOL = 1e-10;
constexpr float G_KMAX_PERT = 1e-4f;
constexpr int GW_FP32_ITERS = 5;       // warm path: bound on the FP32 Newton steps,
constexpr float GW_FP32_KTOL = 3e-5f;  // the rotation below which the next step would be FP32 rounding
constexpr float GW_ROT_MAX = 0.3f;     // the largest rotation taken (beyond: the general path)
constexpr int GW_EVALS = 8;            // and bound on the FP64 evaluations
constexpr float GW_ORTH_MAX = 3e-2f;   // norm of the overlap defect that the FP64 correction takes,
constexpr float GW_ORTH_ONCE = 5e-4f;  // above which it is repeated
constexpr float GW_ORTH_CUBE = 2e-5f;  // and above which its cubic term counts
constexpr float GW_ROT64_MAX = 1e-2f;  // norm of a rotation between FP64 evaluations,
constexpr float GW_ROT64_ONCE = 3e-4f; // and above which the correction follows it (below, C stays orthonormal to 3e-15)
constexpr float GW_GAP = 2e-3f;        // HOMO-LUMO gap (Hartree) the warm path needs, above G_MIN_GAP
constexpr int GW_CG_SLOW = 6;          // conjugate-gradient steps of the first Newton step that ask for a block sweep
constexpr int GW_BISECT = 6;           // tries for a level between the occupied and the empty ones
constexpr float GW_LAST_TOL = 0.1f;    // relative residual of the last solve, of a rotation below 1e-9
constexpr int GW_CG_ITERS = 40;        // bound on the conjugate-gradient steps of a Newton step
constexpr int BT = 256;                // threads per block
constexpr int TB = 256;                // threads per large cell
constexpr int TS = 128;                // threads per small cell (two per block)

// Shared-memory layout of one cell (byte offsets) for cells of at most nmax orbitals, amax atoms.
struct GLayout {
    int nmax, amax, pmax, xb;   // xb: doubles of XB (0: no warm path)
    unsigned SH, C, A, Y, Kc, XB, pos, gam, zv, q, qout, qst, shift, shl, hq, hf, red, diag, cs, invd, th, ints,
        total;
};

// Doubles of the warm path's n x n_occ buffer (three quarters of an n x (n + 1) matrix: water
// clusters need two thirds; cells with more occupied orbitals take the general path).
__host__ __device__ inline int g_xb(int nmax) { return (3 * nmax + 3) / 4 * (nmax + 1); }

__host__ __device__ inline GLayout g_layout(int nmax, int amax, int warm) {
    GLayout L;
    L.xb = warm ? g_xb(nmax) : 0;
    L.nmax = nmax;
    L.amax = amax;
    L.pmax = amax * (amax - 1) / 2 > 0 ? amax * (amax - 1) / 2 : 1;
    const int ld = nmax + 1;
    const unsigned mat = (unsigned)(nmax * ld + 8) * 8;   // 8 doubles of slack for clamped reads
    const unsigned ymat = mat > (unsigned)L.pmax * 32u ? mat : (unsigned)L.pmax * 32u;   // pair gradients fit too
    unsigned o = 0;
    L.SH = o; o += mat;
    L.C = o; o += ymat;   // C and Y swap roles: both can hold the pair gradients
    L.A = o; o += mat;
    L.Y = o; o += ymat;
    L.Kc = o; o += (unsigned)((nmax / 2) * ((nmax + 1) / 2) + 8) * 8;   // n_occ x n_virt <= n^2 / 4
    L.XB = o; o += (unsigned)L.xb * 8;
    L.pos = o; o += amax * 3 * 8;
    L.gam = o; o += amax * amax * 8;
    L.zv = o; o += amax * 8;
    L.q = o; o += amax * 8;
    L.qout = o; o += amax * 8;
    L.qst = o; o += amax * 8;
    L.shift = o; o += amax * 8;
    L.shl = o; o += amax * 8;
    L.hq = o; o += GNHIST * amax * 8;
    L.hf = o; o += GNHIST * amax * 8;
    L.red = o; o += nmax * 8;
    L.diag = o; o += nmax * 8;
    L.cs = o; o += (nmax / 2 + 1) * 16;
    L.invd = o; o += nmax * 8;
    L.th = o; o += GNHIST * 8;
    L.ints = o;
    // ints: spec[amax], atom_off[amax+1], orb_atom[nmax], occ_list[nmax], virt_list[nmax],
    //       occf[nmax], pp[nmax/2+1], pq[nmax/2+1], pa[pmax], pb[pmax], lst[amax], rk[amax], fl[8]
    o += (unsigned)(4 * amax + 1 + 4 * nmax + 2 * (nmax / 2 + 1) + 2 * L.pmax + 8) * 4;
    L.total = (o + 15u) & ~15u;
    return L;
}

// A group of T threads evaluating one cell: the whole block (T = BT), or one half of it
// (T = TS, named barrier 1 or 2).
template <int T>
struct Grp {
    int tid;
    int bar;
    int *vote;   // T/32 ints of shared scratch (halves only)
    __device__ __forceinline__ void sync() const {
        if (T == BT) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");
    }
    __device__ __forceinline__ bool all(bool p) const {
        if (T == BT) return __syncthreads_and(p) != 0;
        const bool w = __all_sync(CAVMD_FULL_MASK, p);
        sync();   // earlier readers of vote are done
        if ((tid & 31) == 0) vote[tid >> 5] = w;
        sync();
        bool r = true;
#pragma unroll
        for (int i = 0; i < T / 32; ++i) r = r && vote[i];
        return r;
    }
};

__device__ __forceinline__ void radial_g(const double *par, double r, const DevSK &sk, double &v, double &dv) {
    const double a = par[0], b = par[1], c1 = par[2], c2 = par[3];
    const double e = a * exp(-b * r);
    const double poly = fma(fma(c2, r, c1), r, 1.0);
    const double dpoly = fma(2.0 * c2, r, c1);
    const double x = (r - (sk.r_cut - sk.taper)) * sk.inv_taper;
    double f = 1.0, df = 0.0;
    if (x > 0.0) {
        if (x < 1.0) {
            double sn, cn;
            sincospi(x, &sn, &cn);
            f = 0.5 * (1.0 + cn);
            df = -0.5 * 3.141592653589793 * sk.inv_taper * sn;
        } else {
            f = 0.0;
        }
    }
    v = e * poly * f;
    dv = e * (fma(-b * poly, f, dpoly * f) + poly * df);
}

// Round-robin Jacobi schedule for even n: pair k of round r (0..n-2); index n-1 meets r.
__device__ __forceinline__ void g_pair(int k, int r, int n, int &p, int &q) {
    const int m = n - 1;
    if (k == 0) { p = r; q = m; return; }
    const int x = (r + k) % m, y = (r - k + m) % m;
    p = min(x, y);
    q = max(x, y);
}

// Rotation annihilating a_pq: angle from FP32, (c, s) normalised in FP64 by two Newton steps.
__device__ __forceinline__ void g_jacobi_cs(double app, double aqq, double apq, double &c, double &s) {
    const float d = d2f_steer(aqq - app);
    const float o = 2.0f * d2f_steer(apq);
    float t = 0.0f;
    if (o != 0.0f) t = o / (d + copysignf(sqrtf(fmaf(d, d, o * o)), d));
    const float cf = rsqrtf(fmaf(t, t, 1.0f));
    c = f2d_steer(cf);
    s = f2d_steer(t * cf);
    for (int it = 0; it < 2; ++it) {
        const double nrm = fma(c, c, s * s);
        const double f = fma(-0.5, nrm, 1.5);
        c *= f;
        s *= f;
    }
}

// Flattened dot products: for every entry e < n_out of this thread (e = tid, tid + T, ...),
// epi(e, sum_{k < nk} xb(e)[k xs] zb(e)[k zs]), the sum taken in increasing k. R entries per pass
// with independent accumulators; the last pass clamps its surplus entries to n_out - 1 and drops
// them.
template <int T, int R, typename XB, typename ZB, typename EPI>
__device__ __forceinline__ void flat(int tid, int n_out, int nk, int xs, int zs, XB xb, ZB zb, EPI epi) {
    for (int e0 = tid; e0 < n_out; e0 += T * R) {
        const double *xp[R];
        const double *zp[R];
        double acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = min(e0 + r * T, n_out - 1);
            xp[r] = xb(e);
            zp[r] = zb(e);
            acc[r] = 0.0;
        }
        for (int k = 0; k < nk; ++k) {
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(xp[r][k * xs], zp[r][k * zs], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (e0 + r * T < n_out) epi(e0 + r * T, acc[r]);
    }
}

// FP32 product in register tiles: for i < m, c < w, epi(i, c, sum_{k < K} X[i xi + k xk] Z[k zk + c zc]),
// TM x TN entries per thread (clamped at the edges, the surplus dropped).
template <int T, int TM, int TN, typename EPI>
__device__ __forceinline__ void ftile(int tid, int m, int w, int K, const float *X, int xi, int xk, const float *Z,
                                      int zk, int zc, EPI epi) {
    const int ni = (m + TM - 1) / TM, nc = (w + TN - 1) / TN;
    for (int t = tid; t < ni * nc; t += T) {
        const int tc = t / ni, i0 = (t - tc * ni) * TM, c0 = tc * TN;
        const float *xp[TM], *zp[TN];
        float acc[TM][TN];
#pragma unroll
        for (int r = 0; r < TM; ++r) xp[r] = X + min(i0 + r, m - 1) * xi;
#pragma unroll
        for (int c = 0; c < TN; ++c) zp[c] = Z + min(c0 + c, w - 1) * zc;
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c) acc[r][c] = 0.0f;
#pragma unroll 2
        for (int k = 0; k < K; ++k) {
            float x[TM], z[TN];
#pragma unroll
            for (int r = 0; r < TM; ++r) x[r] = xp[r][k * xk];
#pragma unroll
            for (int c = 0; c < TN; ++c) z[c] = zp[c][k * zk];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) acc[r][c] = fmaf(x[r], z[c], acc[r][c]);
        }
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c)
                if (i0 + r < m && c0 + c < w) epi(i0 + r, c0 + c, acc[r][c]);
    }
}

// Row i >= c and column c of entry e of the packed lower triangle (column by column) of an m x m
// matrix. A call, not inlined: it stands in the address functions of many products.
__device__ __noinline__ int2 g_lower(int e, int m) {
    const float b = 2.0f * (float)m + 1.0f;
    int c = (int)((b - sqrtf(fmaxf(b * b - 8.0f * (float)e, 0.0f))) * 0.5f);
    c = max(0, min(c, m - 1));
    while (c > 0 && c * m - c * (c - 1) / 2 > e) --c;
    while (c + 1 < m && (c + 1) * m - (c + 1) * c / 2 <= e) ++c;
    return make_int2(c + (e - (c * m - c * (c - 1) / 2)), c);
}

// What the warm path works on (shared memory of one cell, see GLayout).
struct GWarm {
    int n, nocc, nat, AM;
    double *SH, *A, *XB, *Kc, *gam, *zv, *q, *shift, *red;
    float *u, *dq, *ea, *eo, *scr;   // [n], [nat], [nat], [n], [8]: FP32 charges, shifts, reduction scratch
    float *moved;                    // [nat] the change of the charges under K
    const int *orb_atom, *atom_off;
    int *pp, *pq;                    // pairs and
    float *cs;                       // rotations of a Jacobi round
};

// Warm-started cell: the method of k_water_warm (dftb_kernel.cu) for matrices of any size.
//
// The general path below spends 10.8 FP64 iterations of about 3.2 n^3 multiply-adds on a cell, and
// FP64 multiply-adds are this kernel's bound. Here the previous basis (occupied columns first) is
// made orthonormal under the new overlap and moved by Newton steps of the orbital rotation in FP32
// (64 times the FP64 rate), each step solved by conjugate gradients on the orbital Hessian
//   K -> A_vv K - K A_oo + C_v^T dH(K) C_o,  dH = S o (e_A + e_B) / 2, e = gamma dq(K),
// preconditioned by the diagonal differences (3 to 7 iterations). Two steps reach FP32 rounding. Then
// in FP64: the orthonormal correction C (1 - E/2 + 3/8 E^2 - 5/16 E^3); evaluations of q(C), H(q), H C_o and the
// residual A_vo, each followed by the rotation C (1 + K + K^2/2) with K from the FP32 Hessian of this
// basis. Converged when every |A_vo| < G_EIG_TOL and the populations that A_vo implies to first
// order, q_out - q, are below scc_tol: two or three evaluations, about 9 n^3 FP64 multiply-adds with
// the correction. Nothing of the FP32 part but the starting basis and the approximate Hessian enters
// the result. Returns false, with SH untouched, for a cell that leaves the path's range (a large
// rotation or overlap change, a Hessian or gap that is not safely positive, no convergence): the
// general path takes it. On success: C (FP64, occupied columns first), q; shift and XB = H C_o of the charges
// before their last change `moved`.
// Measured (GB300, 16,384 clusters (H2O)_1..8 x 2 steps): 170 -> 48 ms, mean evaluations 2.0 against 10.8
// iterations; 301 clusters x 4 steps 20.2 -> 3.25 ms. Bound: the FP64 pipe (about 65 % busy).
template <int T>
__device__ bool g_warm(const DftbArgs &a, const GWarm &v, double *&C, double *&Y, const double *cw, const Grp<T> &g,
                       int &evals) {
    const int j = g.tid;
    const int n = v.n, no = v.nocc, nv = n - no, nat = v.nat, LD = n + 1, LF = n + 1, nn = n * n, nvo = nv * no;
    double *SH = v.SH, *A = v.A, *XB = v.XB;
    // FP32 matrices in the halves of the FP64 buffers, row-major with stride LF
    float *F0 = (float *)Y, *F1 = F0 + n * LF, *F2 = (float *)A, *F3 = F2 + n * LF;
    float *F4 = (float *)C, *F5 = F4 + n * LF;
    float *x = (float *)v.Kc, *r = x + nvo;   // K and the residual, [virtual][occupied]
    auto s_at = [&](int i, int k) -> double {
        const double lo = SH[k * LD + i], up = SH[i * LD + k];
        return i == k ? 1.0 : (i > k ? lo : up);
    };
    auto h0_at = [&](int i, int k) -> double {
        const double lo = SH[k * LD + i], up = SH[i * LD + k];
        return i <= k ? lo : up;
    };
    auto all = [&](bool p) { return g.all(p); };
    auto sum = [&](float s) -> float {   // over the group, in a fixed order
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(CAVMD_FULL_MASK, s, o);
        g.sync();
        if ((j & 31) == 0) v.scr[j >> 5] = s;
        g.sync();
        float t = v.scr[0];
#pragma unroll
        for (int w = 1; w < T / 32; ++w) t += v.scr[w];
        return t;
    };
    auto s32 = [&]() {
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            F2[c * LF + i] = d2f_steer(s_at(i, c));
        }
        g.sync();
    };
    // F1 = S F0 (S32 in F2)
    auto sc32 = [&]() {
        ftile<T, 3, 3>(j, n, n, n, F2, 1, LF, F0, LF, 1, [&](int i, int c, float t) { F1[i * LF + c] = t; });
        g.sync();
    };
    // A32 = F0^T H F0 into F2, H with the orbital half shifts eo (F3 holds H F0 on the way)
    auto a32 = [&]() {
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            F2[c * LF + i] = fmaf(d2f_steer(s_at(i, c)), v.eo[i] + v.eo[c], d2f_steer(h0_at(i, c)));
        }
        g.sync();
        ftile<T, 3, 3>(j, n, n, n, F2, 1, LF, F0, LF, 1, [&](int i, int c, float t) { F3[i * LF + c] = t; });
        g.sync();
        ftile<T, 3, 3>(j, n, n, n, F0, 1, LF, F3, LF, 1, [&](int i, int c, float t) { F2[i * LF + c] = t; });
        g.sync();
    };
    // populations moved by K = kv to first order, per atom into dq; uses F0 = C, F1 = S C and F3's tail
    constexpr int CQ = 3;   // rows per tile
    auto charges = [&](const float *kv) {
        float *part = F3 + 2 * nvo;
        const int ni = (n + CQ - 1) / CQ, nc = (no + 1) / 2;
        for (int t = j; t < ni * nc; t += T) {
            const int tc = t / ni, i0 = (t - tc * ni) * CQ, c0 = 2 * tc, c1 = min(2 * tc + 1, no - 1);
            float ax[CQ][2], as[CQ][2];
            const float *cp[CQ], *sp[CQ];
#pragma unroll
            for (int q = 0; q < CQ; ++q) {
                cp[q] = F0 + min(i0 + q, n - 1) * LF;
                sp[q] = F1 + min(i0 + q, n - 1) * LF;
                ax[q][0] = ax[q][1] = as[q][0] = as[q][1] = 0.0f;
            }
            for (int k = 0; k < nv; ++k) {
                const float k0 = kv[k * no + c0], k1 = kv[k * no + c1];
#pragma unroll
                for (int q = 0; q < CQ; ++q) {
                    const float cv = cp[q][no + k], sv = sp[q][no + k];
                    ax[q][0] = fmaf(cv, k0, ax[q][0]);
                    ax[q][1] = fmaf(cv, k1, ax[q][1]);
                    as[q][0] = fmaf(sv, k0, as[q][0]);
                    as[q][1] = fmaf(sv, k1, as[q][1]);
                }
            }
#pragma unroll
            for (int q = 0; q < CQ; ++q) {
                if (i0 + q >= n) continue;
                float s = fmaf(ax[q][0], sp[q][c0], cp[q][c0] * as[q][0]);
                if (c0 + 1 < no) s += fmaf(ax[q][1], sp[q][c1], cp[q][c1] * as[q][1]);
                part[tc * n + i0 + q] = s;
            }
        }
        g.sync();
        if (j < n) {
            float s = 0.0f;
            for (int t = 0; t < nc; ++t) s += part[t * n + j];
            v.u[j] = 2.0f * s;
        }
        g.sync();
        if (j < nat) {
            float s = 0.0f;
            for (int o = v.atom_off[j]; o < v.atom_off[j + 1]; ++o) s += v.u[o];
            v.dq[j] = s;
        }
        g.sync();
    };
    // half shifts of the orbitals from the atoms' charges dq
    auto half_shifts = [&]() {
        if (j < nat) {
            float s = 0.0f;
            for (int k = 0; k < nat; ++k) s = fmaf(d2f_steer(v.gam[j * v.AM + k]), v.dq[k], s);
            v.ea[j] = 0.5f * s;
        }
        g.sync();
        if (j < n) v.eo[j] = v.ea[v.orb_atom[j]];
        g.sync();
    };
    auto diag_of = [&](int e) -> float {
        const int vi = e / no, o = e - vi * no;
        return F2[(no + vi) * LF + no + vi] - F2[o * LF + o];
    };
    // K (in x) from the residual r (destroyed): Hessian K = r to a relative residual rel, by
    // preconditioned conjugate gradients. False when the Hessian is not positive along the way.
    int steps = 0;   // conjugate-gradient steps of the last solve
    auto newton = [&](float rel) -> bool {
        float *p = F3, *hp = F3 + nvo;
        float rz = 0.0f;
        steps = 0;
        if (j < nat) v.moved[j] = 0.0f;
        for (int e = j; e < nvo; e += T) {
            const float z = r[e] / diag_of(e);
            x[e] = 0.0f;
            p[e] = z;
            rz = fmaf(r[e], z, rz);
        }
        rz = sum(rz);
        const float stop = rel * rel * rz;
        if (!(rz < 1e30f) || !(rz >= 0.0f)) return false;
        for (int it = 0; it < GW_CG_ITERS && rz > stop; ++it) {
            ++steps;
            charges(p);
            half_shifts();
            ftile<T, 2, 2>(j, nv, no, nv, F2 + no * LF + no, LF, 1, p, no, 1,
                           [&](int i, int c, float t) { hp[i * no + c] = t; });
            ftile<T, 2, 2>(j, nv, no, no, p, no, 1, F2, LF, 1, [&](int i, int c, float t) { hp[i * no + c] -= t; });
            {   // C_v^T (e S C_o) + (S C_v)^T (e C_o): the same tiles, so each thread adds to its own entries
                const int ni = (nv + 1) / 2, nc = (no + 1) / 2;
                for (int t = j; t < ni * nc; t += T) {
                    const int tc = t / ni, i0 = 2 * (t - tc * ni), i1 = min(i0 + 1, nv - 1), c0 = 2 * tc, c1 = min(c0 + 1, no - 1);
                    float a00 = 0.f, a01 = 0.f, a10 = 0.f, a11 = 0.f;
                    for (int m = 0; m < n; ++m) {
                        const float *cr = F0 + m * LF, *sr = F1 + m * LF;
                        const float e = v.eo[m];
                        const float s0 = e * sr[c0], s1 = e * sr[c1], q0 = e * cr[c0], q1 = e * cr[c1];
                        const float v0 = cr[no + i0], v1 = cr[no + i1], w0 = sr[no + i0], w1 = sr[no + i1];
                        a00 = fmaf(v0, s0, fmaf(w0, q0, a00));
                        a01 = fmaf(v0, s1, fmaf(w0, q1, a01));
                        a10 = fmaf(v1, s0, fmaf(w1, q0, a10));
                        a11 = fmaf(v1, s1, fmaf(w1, q1, a11));
                    }
                    hp[i0 * no + c0] += a00;
                    if (c0 + 1 < no) hp[i0 * no + c1] += a01;
                    if (i0 + 1 < nv) hp[i1 * no + c0] += a10;
                    if (i0 + 1 < nv && c0 + 1 < no) hp[i1 * no + c1] += a11;
                }
            }
            g.sync();
            float ph = 0.0f;
            for (int e = j; e < nvo; e += T) ph = fmaf(p[e], hp[e], ph);
            ph = sum(ph);
            if (!(ph > 0.0f)) return false;
            const float al = rz / ph;
            if (j < nat) v.moved[j] = fmaf(al, v.dq[j], v.moved[j]);
            float rn = 0.0f;
            for (int e = j; e < nvo; e += T) {
                x[e] = fmaf(al, p[e], x[e]);
                const float q = fmaf(-al, hp[e], r[e]);
                r[e] = q;
                rn = fmaf(q, q / diag_of(e), rn);
            }
            rn = sum(rn);
            if (!(rn < 1e30f) || !(rn >= 0.0f)) return false;
            const float be = rn / rz;
            rz = rn;
            for (int e = j; e < nvo; e += T) p[e] = fmaf(be, p[e], r[e] / diag_of(e));
            g.sync();
        }
        g.sync();
        return true;
    };
    // second-order parts of the rotation: G[i][o] = 1/2 sum_v C[i][v] K_vo, G[i][no + v] = -1/2 sum_o C[i][o] K_vo
    auto second = [&](float *G, bool with_c) {
        ftile<T, 3, 2>(j, n, no, nv, F0 + no, LF, 1, x, no, 1, [&](int i, int c, float t) {
            G[i * LF + c] = fmaf(0.5f, t, with_c ? F0[i * LF + c] : 0.0f);
        });
        ftile<T, 3, 1>(j, n, nv, no, F0, LF, 1, x, 1, no, [&](int i, int c, float t) {
            G[i * LF + no + c] = fmaf(-0.5f, t, with_c ? F0[i * LF + no + c] : 0.0f);
        });
        g.sync();
    };

    // ---------------------------------------------------------------- FP32 start
    for (int e = j; e < nn; e += T) {
        const int c = e / n, i = e - c * n;
        F0[i * LF + c] = d2f_steer(cw[e]);
    }
    s32();
    for (int pass = 0; pass < 2; ++pass) {   // E is a few 1e-2 after one step: below 1e-6 after two passes
        sc32();
        float big = 0.0f;
        ftile<T, 3, 3>(j, n, n, n, F0, 1, LF, F1, LF, 1, [&](int i, int c, float t) {
            const float e = t - (i == c ? 1.0f : 0.0f);
            big = max_nan(big, fabsf(e));
            if (pass == 0) F3[i * LF + c] = e;
            else F4[i * LF + c] = fmaf(-0.5f, e, i == c ? 1.0f : 0.0f);
        });
        if (!all(big < 0.2f)) return false;   // a NaN too
        if (pass == 0) {
            g.sync();
            ftile<T, 3, 3>(j, n, n, n, F3, 1, LF, F3, LF, 1, [&](int i, int c, float t) {
                F4[i * LF + c] = fmaf(0.375f, t, fmaf(-0.5f, F3[i * LF + c], i == c ? 1.0f : 0.0f));
            });
        }
        g.sync();
        ftile<T, 3, 3>(j, n, n, n, F0, LF, 1, F4, LF, 1, [&](int i, int c, float t) { F5[i * LF + c] = t; });
        g.sync();
        for (int e = j; e < nn; e += T) {
            const int i = e / n, c = e - i * n;
            F0[i * LF + c] = F5[i * LF + c];
        }
        g.sync();
    }
    bool done = false;
    int first_steps = 0;
    for (int it = 0; it < GW_FP32_ITERS && !done; ++it) {
        if (it > 0) s32();
        sc32();
        if (j < n) {
            float s = 0.0f;
            for (int o = 0; o < no; ++o) s = fmaf(F0[j * LF + o], F1[j * LF + o], s);
            v.u[j] = 2.0f * s;
        }
        g.sync();
        if (j < nat) {
            float s = -d2f_steer(v.zv[j]);
            for (int o = v.atom_off[j]; o < v.atom_off[j + 1]; ++o) s += v.u[o];
            v.dq[j] = s;
        }
        g.sync();
        half_shifts();
        a32();
        for (int e = j; e < nvo; e += T) {
            const int vi = e / no, o = e - vi * no;
            r[e] = -0.5f * (F2[(no + vi) * LF + o] + F2[o * LF + no + vi]);
        }
        g.sync();
        if (!newton(it < 2 ? 3e-3f : 1e-2f)) return false;
        if (it == 0) first_steps = steps;
        float kmax = 0.0f;
        for (int e = j; e < nvo; e += T) kmax = max_nan(kmax, fabsf(x[e]));
        if (!all(kmax < GW_ROT_MAX)) return false;
        done = all(kmax < GW_FP32_KTOL);
        second(F4, true);
        ftile<T, 3, 2>(j, n, no, nv, F4 + no, LF, 1, x, no, 1, [&](int i, int c, float t) { F0[i * LF + c] += t; });
        ftile<T, 3, 1>(j, n, nv, no, F4, LF, 1, x, 1, no, [&](int i, int c, float t) { F0[i * LF + no + c] -= t; });
        g.sync();
    }
    if (!done) return false;
    // One Jacobi sweep inside each block when their off-diagonal part has grown enough to slow the solve
    // (see p_warm in dftb_periodic.cuh); any orthogonal mixing inside a block leaves the result alone.
    if (first_steps >= GW_CG_SLOW) {
        for (int b = 0; b < 2; ++b) {
            const int off = b ? no : 0, mb = b ? nv : no, me = mb + (mb & 1), half = me / 2;
            for (int e = j; e < mb * mb; e += T) {
                const int c = e / mb, i = e - c * mb;
                F3[e] = F2[(off + i) * LF + off + c];
                F4[e] = i == c ? 1.0f : 0.0f;
            }
            g.sync();
            for (int rd = 0; rd < me - 1; ++rd) {
                if (j < half) {
                    int pa, pb;
                    g_pair(j, rd, me, pa, pb);
                    float t = 0.0f;
                    if (pb < mb) {
                        const float d = F3[pb * mb + pb] - F3[pa * mb + pa], o = 2.0f * F3[pb * mb + pa];
                        if (o != 0.0f) t = o / (d + copysignf(sqrtf(fmaf(d, d, o * o)), d));
                    }
                    const float c = rsqrtf(fmaf(t, t, 1.0f));
                    v.pp[j] = pa;
                    v.pq[j] = pb;
                    v.cs[2 * j] = c;
                    v.cs[2 * j + 1] = t * c;
                }
                g.sync();
                for (int e = j; e < half * 2 * mb; e += T) {   // columns of the block and of the rotation
                    const int k = e / (2 * mb), rr = e - k * 2 * mb, pa = v.pp[k], pb = v.pq[k];
                    if (pb >= mb) continue;
                    float *base = rr < mb ? F3 : F4;
                    const int i = rr < mb ? rr : rr - mb;
                    const float xp = base[pa * mb + i], xq = base[pb * mb + i], c = v.cs[2 * k], sn = v.cs[2 * k + 1];
                    base[pa * mb + i] = fmaf(c, xp, -sn * xq);
                    base[pb * mb + i] = fmaf(sn, xp, c * xq);
                }
                g.sync();
                for (int e = j; e < half * mb; e += T) {   // rows of the block
                    const int k = e / mb, cc = e - k * mb, pa = v.pp[k], pb = v.pq[k];
                    if (pb >= mb) continue;
                    const float xp = F3[cc * mb + pa], xq = F3[cc * mb + pb], c = v.cs[2 * k], sn = v.cs[2 * k + 1];
                    F3[cc * mb + pa] = fmaf(c, xp, -sn * xq);
                    F3[cc * mb + pb] = fmaf(sn, xp, c * xq);
                }
                g.sync();
            }
            ftile<T, 3, 3>(j, n, mb, mb, F0 + off, LF, 1, F4, 1, mb, [&](int i, int c, float t) { F5[i * LF + c] = t; });
            g.sync();
            for (int e = j; e < n * mb; e += T) {
                const int i = e / mb, c = e - i * mb;
                F0[i * LF + off + c] = F5[i * LF + c];
            }
            g.sync();
        }
    }

    // ---------------------------------------------------------------- FP64 evaluations
    for (int e = j; e < nn; e += T) {
        const int c = e / n, i = e - c * n;
        C[c * LD + i] = f2d_steer(F0[i * LF + c]);
    }
    bool rough = true;   // the basis is orthonormal to FP32 only (or after a large rotation)
    const int most = min(a.max_iter, GW_EVALS);
    for (int it = 1; it <= most; ++it) {
        for (int pass = 0; rough; ++pass) {
            for (int e = j; e < nn; e += T) {
                const int c = e / n, i = e - c * n;
                A[c * LD + i] = s_at(i, c);
            }
            g.sync();
            flat<T, 4>(j, nn, n, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return C + (e / n) * LD; },
                       [&](int e, double t) { Y[(e / n) * LD + e % n] = t; });
            g.sync();
            // E = C^T S C - 1 into A, and in FP32 into XB
            float *E32 = (float *)XB, *Q32 = (float *)Y;
            float e2 = 0.0f;
            flat<T, 4>(j, n * (n + 1) / 2, n, 1, 1,
                       [&](int e) { return C + g_lower(e, n).x * LD; },
                       [&](int e) { return Y + g_lower(e, n).y * LD; }, [&](int e, double t) {
                           const int2 ic = g_lower(e, n);
                           const int i = ic.x, c = ic.y;
                           if (i == c) t -= 1.0;
                           A[c * LD + i] = t;
                           A[i * LD + c] = t;
                           const float f = d2f_steer(t);
                           E32[c * LF + i] = f;
                           E32[i * LF + c] = f;
                           e2 = fmaf(i == c ? 1.0f : 2.0f, f * f, e2);
                       });
            e2 = sum(e2);
            if (!(e2 < GW_ORTH_MAX * GW_ORTH_MAX) || pass == 3) return false;
            rough = e2 > GW_ORTH_ONCE * GW_ORTH_ONCE;
            g.sync();
            // 1 - E/2 + 3/8 E^2 - 5/16 E^3. The norm of E is 2e-6 as a rule, more after a large rotation; up to
            // GW_ORTH_ONCE FP32 rounds the last two terms by 6e-15, and the quartic one is 2e-14.
            ftile<T, 3, 3>(j, n, n, n, E32, 1, LF, E32, LF, 1, [&](int i, int c, float t) {
                A[c * LD + i] = fma(-0.5, A[c * LD + i], (i == c ? 1.0 : 0.0) + f2d_steer(0.375f * t));
                Q32[c * LF + i] = t;
            });
            g.sync();
            if (e2 > GW_ORTH_CUBE * GW_ORTH_CUBE) {
                ftile<T, 3, 3>(j, n, n, n, E32, 1, LF, Q32, 1, LF,
                               [&](int i, int c, float t) { A[c * LD + i] -= f2d_steer(0.3125f * t); });
                g.sync();
            }
            flat<T, 4>(j, nn, n, LD, 1, [&](int e) { return C + (e % n); }, [&](int e) { return A + (e / n) * LD; },
                       [&](int e, double t) { Y[(e / n) * LD + e % n] = t; });
            g.sync();
            double *t = C;
            C = Y;
            Y = t;
        }
        F0 = (float *)Y;
        F1 = F0 + n * LF;
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            A[c * LD + i] = s_at(i, c);
        }
        g.sync();
        flat<T, 4>(j, n * no, n, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return C + (e / n) * LD; },
                   [&](int e, double t) { XB[(e / n) * LD + e % n] = t; });
        g.sync();
        if (j < n) {
            double t = 0.0;
            for (int o = 0; o < no; ++o) t = fma(C[o * LD + j], XB[o * LD + j], t);
            v.red[j] = 2.0 * t;
        }
        g.sync();
        if (j < nat) {
            double t = 0.0;
            for (int o = v.atom_off[j]; o < v.atom_off[j + 1]; ++o) t += v.red[o];
            v.q[j] = t;
        }
        g.sync();
        if (j < nat) {
            double t = 0.0;
            for (int k = 0; k < nat; ++k) t = fma(v.gam[j * v.AM + k], v.q[k] - v.zv[k], t);
            v.shift[j] = t;
        }
        g.sync();
        if (j < n) v.eo[j] = 0.5f * d2f_steer(v.shift[v.orb_atom[j]]);
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            A[c * LD + i] = fma(0.5 * s_at(i, c), v.shift[v.orb_atom[i]] + v.shift[v.orb_atom[c]], h0_at(i, c));
        }
        g.sync();
        flat<T, 4>(j, n * no, n, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return C + (e / n) * LD; },
                   [&](int e, double t) { XB[(e / n) * LD + e % n] = t; });
        g.sync();
        bool small = true, finite = true;
        flat<T, 4>(j, nvo, n, 1, 1, [&](int e) { return C + (no + e / no) * LD; },
                   [&](int e) { return XB + (e % no) * LD; }, [&](int e, double t) {
                       if (!abs_lt(t, G_EIG_TOL)) small = false;
                       if (!abs_lt(t, 1.0)) finite = false;
                       r[e] = -d2f_steer(t);
                   });
        small = all(small);
        if (!all(finite)) return false;
        // the FP32 Hessian of this basis (over A and Y)
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            F0[i * LF + c] = d2f_steer(C[c * LD + i]);
        }
        s32();
        sc32();
        a32();
        bool conv = false;
        if (small) {   // q_out - q to first order: K0 = r / (A_vv - A_oo)
            for (int e = j; e < nvo; e += T) x[e] = r[e] / diag_of(e);
            g.sync();
            charges(x);
            conv = all(j >= nat || fabsf(v.dq[j]) < (float)a.scc_tol);
        }
        if (conv) {
            // aufbau and gap: tau - A_oo and A_vv - tau - GW_GAP positive definite (Cholesky pivots)
            float hi = -1e30f, lo = 1e30f;
            for (int o = 0; o < no; ++o) hi = fmaxf(hi, F2[o * LF + o]);
            for (int k = no; k < n; ++k) lo = fminf(lo, F2[k * LF + k]);
            // the diagonals bound tau (mixing inside the blocks moves the levels beyond them): bisection
            for (int t = 0;; ++t) {
                const float tau = 0.5f * (hi + lo);
                g.sync();
                for (int e = j; e < nn; e += T) {
                    const int i = e / n, c = e - i * n;
                    const float x = F2[i * LF + c];
                    F3[i * LF + c] = (i < no && c < no) ? (i == c ? tau : 0.0f) - x : x - (i == c ? tau + GW_GAP : 0.0f);
                }
                g.sync();
                bool occ = true, emp = true;
                for (int k = 0; k < n; ++k) {   // both blocks in turn; entries between them are not touched
                    const float d = F3[k * LF + k];
                    if (k < no) occ = occ && d > 0.0f; else emp = emp && d > 0.0f;
                    const int end = k < no ? no : n;
                    const float id = 1.0f / d;
                    for (int i = k + 1 + j; i < end; i += T) {
                        const float f = F3[i * LF + k] * id;
                        for (int c = k + 1; c <= i; ++c) F3[i * LF + c] = fmaf(-f, F3[c * LF + k], F3[i * LF + c]);
                    }
                    g.sync();
                }
                if (occ && emp) break;   // the same in every thread
                if (t == GW_BISECT || occ == emp) return false;
                if (occ) lo = tau; else hi = tau;
            }
        }
        if ((it == most && !conv) || !newton(conv ? GW_LAST_TOL : 1e-6f)) return false;
        if (conv) {
            // The residual that passed the test stays in no result: q takes the change that K makes and C_o becomes
            // C_o + C_v K, which changes A_oo = C_o^T H C_o to second order only. K is solved for, to a tenth: K0 in
            // its place would leave half of the residual, since the blocks of A are not diagonal. Largest error of
            // 400 clusters without and with this: charges 4.0e-13 and 2.2e-14, forces 1.0e-13 and 7.8e-15 (the
            // general path: 2.3e-13, 1.2e-14); 16,384 clusters x 2 steps take 46.1 and 48.3 ms.
            if (j < nat) v.q[j] += f2d_steer(v.moved[j]);
            if (a.n_disp == 0)
                ftile<T, 3, 2>(j, n, no, nv, F0 + no, LF, 1, x, no, 1,
                               [&](int i, int c, float t) { C[c * LD + i] += f2d_steer(t); });
            g.sync();
            evals = it;
            return true;
        }
        float k2 = 0.0f;
        for (int e = j; e < nvo; e += T) k2 = fmaf(x[e], x[e], k2);
        k2 = sum(k2);
        if (!(k2 < GW_ROT64_MAX * GW_ROT64_MAX)) return false;
        rough = k2 > GW_ROT64_ONCE * GW_ROT64_ONCE;
        // C (1 + K + K^2/2), as C_o + (C_v - (C_o K^T)/2) K and C_v - (C_o + (C_v K)/2) K^T
        second(F1, false);
        double Kd[4];   // this thread's entries of K: n_virt n_occ <= n^2 / 4, 1024 on 256 threads at n = 64, 256 on 128 at n = 32
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int e = j + t * T;
            Kd[t] = e < nvo ? f2d_steer(x[e]) : 0.0;
        }
        for (int e = j; e < nn; e += T) {
            const int c = e / n, i = e - c * n;
            A[c * LD + i] = C[c * LD + i] + f2d_steer(F1[i * LF + c]);
        }
        g.sync();
        double *K = v.Kc;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int e = j + t * T;
            if (e < nvo) K[e] = Kd[t];
        }
        g.sync();
        flat<T, 4>(j, n * no, nv, LD, no, [&](int e) { return A + no * LD + e % n; }, [&](int e) { return K + e / n; },
                   [&](int e, double t) { C[(e / n) * LD + e % n] += t; });
        flat<T, 4>(j, n * nv, no, LD, 1, [&](int e) { return A + e % n; }, [&](int e) { return K + (e / n) * no; },
                   [&](int e, double t) { C[(no + e / n) * LD + e % n] -= t; });
        g.sync();
    }
    return false;
}

// One cell (main evaluation, kd < 0) or one displaced copy of it (kd = displacement index),
// evaluated by the T threads of group g.
template <int T, int R>
__device__ void g_molecule(const DevSK &sk, const DftbArgs &a, const GLayout &L, unsigned char *sm, int cell,
                           int kd, const Grp<T> &g) {
    const int j = g.tid;
    const bool disp = kd >= 0;
    const int a0 = a.cell_offset[cell];
    const int nat = a.cell_offset[cell + 1] - a0;
    double *SH = (double *)(sm + L.SH), *A = (double *)(sm + L.A), *Kc = (double *)(sm + L.Kc);
    double *C = (double *)(sm + L.C), *Y = (double *)(sm + L.Y);   // swapped by the second-order update
    double(*pos)[3] = (double(*)[3])(sm + L.pos);
    double *gam = (double *)(sm + L.gam), *zv = (double *)(sm + L.zv), *q = (double *)(sm + L.q);
    double *qout = (double *)(sm + L.qout), *qst = (double *)(sm + L.qst);
    double *shift = (double *)(sm + L.shift), *shl = (double *)(sm + L.shl);
    double *hq = (double *)(sm + L.hq), *hf = (double *)(sm + L.hf), *red = (double *)(sm + L.red);
    double *diag = (double *)(sm + L.diag), *cs = (double *)(sm + L.cs), *invd = (double *)(sm + L.invd);
    double *th = (double *)(sm + L.th);
    int *spec = (int *)(sm + L.ints);
    int *atom_off = spec + L.amax;
    int *orb_atom = atom_off + L.amax + 1;
    int *occ_list = orb_atom + L.nmax;
    int *virt_list = occ_list + L.nmax;
    int *occf = virt_list + L.nmax;
    int *pp = occf + L.nmax;
    int *pq = pp + (L.nmax / 2 + 1);
    int *pa = pq + (L.nmax / 2 + 1);
    int *pb = pa + L.pmax;
    int *lst = pb + L.pmax;  // atoms with p orbitals, then those without, each in increasing order
    int *rk = lst + L.amax;  // position of an atom among those of its kind
    int *fl = rk + L.amax;   // 0 error bits, 2 iterations, 3 occupied orbitals, 4 orbitals, 6 atoms with p orbitals
    const int AM = L.amax;

    if (j < nat) {
        spec[j] = a.species[a0 + j];
        for (int k = 0; k < 3; ++k) pos[j][k] = a.r[3 * (a0 + j) + k];
        if (disp) {   // atom da, component dc, by +h (forward) or +-h (central pairs)
            const int kk = a.fd_central ? kd >> 1 : kd;
            const int da = kk / 3, dc = kk - 3 * (kk / 3);
            const double sg = (a.fd_central && (kd & 1)) ? -1.0 : 1.0;
            if (j == da) pos[j][dc] += sg * a.fd_h;
        }
    }
    g.sync();
    if (j == 0) {
        int o = 0;
        double nel = 0.0;
        for (int at = 0; at < nat; ++at) {
            atom_off[at] = o;
            const int no = sk.norb[spec[at]];
            for (int k = 0; k < no; ++k) orb_atom[o + k] = at;
            o += no;
            zv[at] = sk.zval[spec[at]];
            nel += zv[at];
        }
        atom_off[nat] = o;
        fl[0] = 0;
        fl[2] = 0;
        fl[3] = (int)(nel * 0.5 + 0.25);
        fl[4] = o;
    }
    if (j < nat) {
        const bool big = sk.norb[spec[j]] == 4;
        int same = 0, nbig = 0;
        for (int x = 0; x < nat; ++x) {
            const bool bx = sk.norb[spec[x]] == 4;
            nbig += bx;
            same += x < j && bx == big;
        }
        rk[j] = same;
        lst[big ? same : nbig + same] = j;
        if (j == 0) fl[6] = nbig;
    }
    g.sync();
    const int n = fl[4], nocc = fl[3], npair = nat * (nat - 1) / 2;
    // Pairs (A < B) by kind, so that the threads of a warp evaluate the same integrals: both atoms with p
    // orbitals (10 radial functions), one of them (4), neither (2).
    const int nb = fl[6], ns = nat - nb, p_bb = nb * (nb - 1) / 2, p_bs = p_bb + nb * ns;
    for (int pi = j; pi < npair; pi += T) {
        int x, y;
        if (pi >= p_bb && pi < p_bs) {
            const int u = pi - p_bb;
            x = lst[u / ns];
            y = lst[nb + u % ns];
        } else {
            const int u = pi < p_bb ? pi : pi - p_bs, o = pi < p_bb ? 0 : nb;
            int k = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)u)) * 0.5f);
            while (k * (k - 1) / 2 > u) --k;
            while ((k + 1) * k / 2 <= u) ++k;
            x = lst[o + u - k * (k - 1) / 2];
            y = lst[o + k];
        }
        pa[pi] = min(x, y);
        pb[pi] = max(x, y);
    }
    auto pair_of = [&](int x, int y) -> int {   // the pair's index
        const bool bx = lst[rk[x]] == x && rk[x] < nb, by = lst[rk[y]] == y && rk[y] < nb;
        if (bx != by) return p_bb + (bx ? rk[x] : rk[y]) * ns + (bx ? rk[y] : rk[x]);
        const int k = max(rk[x], rk[y]), i = min(rk[x], rk[y]);
        return (bx ? 0 : p_bs) + k * (k - 1) / 2 + i;
    };
    const int nv = n - nocc;
    const int LD = n + 1;   // n is even (closed shell), so the stride is odd
    const int nn = n * n;
    // S(i, k) and H0(i, k) from the shared buffer: column k below the diagonal, row k above it
    auto s_at = [&](int i, int k) -> double {
        const double lo = SH[k * LD + i], up = SH[i * LD + k];
        return i == k ? 1.0 : (i > k ? lo : up);
    };
    auto h0_at = [&](int i, int k) -> double {
        const double lo = SH[k * LD + i], up = SH[i * LD + k];
        return i <= k ? lo : up;
    };

    // ---------------------------------------------------------------- H0, S, gamma
    for (int e = j; e < nn; e += T) {
        const int c = e / n, i = e - c * n;
        double v = 0.0;
        if (i == c) {
            const int at = orb_atom[c], el = spec[at];
            v = (c == atom_off[at]) ? sk.onsite[el][0] : sk.onsite[el][1];
        }
        SH[c * LD + i] = v;
    }
    g.sync();
    for (int pi = j; pi < npair; pi += T) {
        const int PA = pa[pi], PB = pb[pi];
        const int eA = spec[PA], eB = spec[PB];
        const int oA = atom_off[PA], oB = atom_off[PB];
        const int na = sk.norb[eA], nb = sk.norb[eB];
        const double dx = pos[PB][0] - pos[PA][0], dy = pos[PB][1] - pos[PA][1], dz = pos[PB][2] - pos[PA][2];
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        const double ir = rsqrt_nr(r2);
        const double r = r2 * ir;
        const double ev[3] = {dx * ir, dy * ir, dz * ir};
        for (int t = 0; t < 2; ++t) {
            const double(*tab)[CAVMD_MAX_ELEM][4][4] = t == 0 ? sk.h0 : sk.s;
            // element (mu of A, nu of B), mu < nu: H0 in column nu, S in column mu
            auto put = [&](int mu, int nu, double v) {
                if (t == 0) SH[nu * LD + mu] = v; else SH[mu * LD + nu] = v;
            };
            double v, dv;
            radial_g(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
            put(oA, oB, v);
            if (nb == 4) {
                radial_g(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                for (int i = 0; i < 3; ++i) put(oA, oB + 1 + i, ev[i] * v);
            }
            if (na == 4) {
                radial_g(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                for (int i = 0; i < 3; ++i) put(oA + 1 + i, oB, -ev[i] * v);
            }
            if (na == 4 && nb == 4) {
                double vs, vp;
                radial_g(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dv);
                radial_g(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dv);
                const double dl = vs - vp;
                for (int i = 0; i < 3; ++i)
                    for (int k = 0; k < 3; ++k) put(oA + 1 + i, oB + 1 + k, fma(ev[i] * ev[k], dl, (i == k) ? vp : 0.0));
            }
        }
    }
    for (int e2 = j; e2 < nat * nat; e2 += T) {
        const int x = e2 / nat, y = e2 - x * nat;
        if (x == y) {
            gam[x * AM + y] = sk.hubbard[spec[x]];
        } else {
            const double dx = pos[y][0] - pos[x][0], dy = pos[y][1] - pos[x][1], dz = pos[y][2] - pos[x][2];
            gam[x * AM + y] = rsqrt_nr(fma(dx, dx, fma(dy, dy, fma(dz, dz, sk.gamma_c2[spec[x]][spec[y]]))));
        }
    }

    const long long coff = a.Cwarm_off ? a.Cwarm_off[cell] : (long long)cell * 36;
    const double *cw = a.Cwarm + coff;
    // ---------------------------------------------------------------- warm path
    bool warm = false;
    if (a.have_warm && nocc > 0 && nv > 0 && nocc * LD <= L.xb) {
        GWarm wv;
        wv.n = n; wv.nocc = nocc; wv.nat = nat; wv.AM = AM;
        wv.SH = SH; wv.A = A; wv.XB = (double *)(sm + L.XB); wv.Kc = Kc; wv.gam = gam; wv.zv = zv; wv.q = q;
        wv.shift = shift; wv.red = red;
        wv.u = (float *)diag; wv.dq = (float *)qout; wv.ea = (float *)shl; wv.eo = (float *)invd; wv.scr = (float *)th; wv.moved = (float *)hq;
        wv.orb_atom = orb_atom; wv.atom_off = atom_off;
        wv.pp = pp; wv.pq = pq; wv.cs = (float *)cs;
        g.sync();
        int evals = 0;
        warm = g_warm<T>(a, wv, C, Y, cw, g, evals);
        g.sync();
        if (warm && j == 0) fl[2] = evals;
        if (warm && j < nat) qst[j] = a.qpop[a0 + j];
        g.sync();
    }
    if (!warm) {
    // ---------------------------------------------------------------- warm-started S-orthonormal basis
    for (int e = j; e < nn; e += T) {   // coalesced copy of the previous eigenvectors
        const int c = e / n, i = e - c * n;
        C[c * LD + i] = a.have_warm ? cw[e] : (i == c ? 1.0 : 0.0);
    }
    if (j < nat) {
        if (a.have_warm) {   // predictor 2 q(t) - q(t - dt); displaced copies start from q(t)
            const double qt = a.qpop[a0 + j];
            qst[j] = qt;
            q[j] = disp ? qt : fma(2.0, qt, -a.qprev[a0 + j]);
        } else {
            q[j] = zv[j];
        }
    }
    g.sync();
    for (int e = j; e < nn; e += T) {   // S, full, into A
        const int c = e / n, i = e - c * n;
        A[c * LD + i] = s_at(i, c);
    }
    if (a.have_warm) {   // A = C^T S C
        g.sync();
        flat<T, R>(j, nn, n, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return C + (e / n) * LD; },
                   [&](int e, double v) { Y[(e / n) * LD + e % n] = v; });
        g.sync();
        flat<T, R>(j, nn, n, 1, 1, [&](int e) { return C + (e % n) * LD; }, [&](int e) { return Y + (e / n) * LD; },
                   [&](int e, double v) { A[(e / n) * LD + e % n] = v; });
    }
    g.sync();
    for (int k = 0; k < n; ++k) {   // Cholesky A = L L^T, right-looking, thread = column
        if (j == k) {
            double d = A[k * LD + k];
            if (!(d > 1e-300)) { atomicOr(&fl[0], ERRBIT_S_NOT_PD); d = 1.0; }
            const double y = rsqrt_nr(d);
            invd[k] = y;
            A[k * LD + k] = d * y;
            for (int i = k + 1; i < n; ++i) A[k * LD + i] *= y;
        }
        g.sync();
        if (j > k && j < n) {
            const double ljk = A[k * LD + j];
            for (int i = j; i < n; ++i) A[j * LD + i] = fma(-A[k * LD + i], ljk, A[j * LD + i]);
        }
        g.sync();
    }
    if (j < n) {   // C <- C L^-T, thread = row
        const int i = j;
        for (int c = 0; c < n; ++c) {
            double x = C[c * LD + i];
            for (int k = 0; k < c; ++k) x = fma(-C[k * LD + i], A[k * LD + c], x);
            C[c * LD + i] = x * invd[c];
        }
    }
    g.sync();

    // aufbau occupation from diag[]: occupied and virtual index lists in order of rank
    auto rank_occupation = [&]() {
        if (j < n) {
            const long long kj = order_key(diag[j]);
            int rank = 0;
            for (int i = 0; i < n; ++i) {
                const long long ki = order_key(diag[i]);
                rank += (ki < kj) || (ki == kj && i < j);
            }
            occf[j] = rank < nocc;
            if (rank < nocc) occ_list[rank] = j; else virt_list[rank - nocc] = j;
        }
    };

    // ---------------------------------------------------------------- SCC loop
    // Per iteration: H(q) into A; Y = H C; the diagonal of C^T Y, the occupation, the occupied-
    // virtual block of C^T Y and the compact generator K(v, o) = A_vo / (A_oo - A_vv). When every
    // generator entry is below KMAX the basis takes C <- C (I + K + K^2/2) (orthogonal to O(K^4));
    // otherwise the rest of A = C^T H C is formed and Jacobi sweeps move C (one per iteration when
    // warm started, to convergence on a cold start).
    int it;
    for (it = 1; it <= a.max_iter; ++it) {
        if (j < nat) {
            double sh = 0.0;
            for (int k = 0; k < nat; ++k) sh = fma(gam[j * AM + k], q[k] - zv[k], sh);
            shift[j] = sh;
        }
        g.sync();
        for (int e = j; e < nn; e += T) {   // H into A
            const int c = e / n, i = e - c * n;
            A[c * LD + i] = fma(0.5 * s_at(i, c), shift[orb_atom[i]] + shift[orb_atom[c]], h0_at(i, c));
        }
        g.sync();
        flat<T, R>(j, nn, n, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return C + (e / n) * LD; },
                   [&](int e, double v) { Y[(e / n) * LD + e % n] = v; });
        g.sync();
        flat<T, R>(j, n, n, 1, 1, [&](int e) { return C + e * LD; }, [&](int e) { return Y + e * LD; },
                   [&](int e, double v) { diag[e] = v; });
        g.sync();
        rank_occupation();
        g.sync();
        // occupied-virtual block of C^T H C (entry e: virtual index e % nv, occupied e / nv)
        bool small = true;
        float kmax = 0.0f;
        flat<T, R>(j, nocc * nv, n, 1, 1, [&](int e) { return C + virt_list[e % nv] * LD; },
                   [&](int e) { return Y + occ_list[e / nv] * LD; }, [&](int e, double v) {
                       const int vi = virt_list[e % nv], oi = occ_list[e / nv];
                       A[oi * LD + vi] = v;
                       A[vi * LD + oi] = v;
                       if (!abs_lt(v, G_EIG_TOL)) small = false;
                       float kf = d2f_steer(v) / d2f_steer(diag[oi] - diag[vi]);
                       if (!(fabsf(kf) <= 1e30f)) kf = 1e30f;   // degenerate or non-finite: Jacobi path
                       kmax = fmaxf(kmax, fabsf(kf));
                       Kc[e] = f2d_steer(kf);   // K(v, o) at [o][v]
                   });
        const bool eok = g.all(small);
        const bool cold_first = !a.have_warm && it == 1;
        const bool perturb = g.all(kmax < G_KMAX_PERT && !cold_first);
        if (perturb) {
            // V = I + K + K^2/2 into A: K(v, o) = Kc[o][v], K(o, v) = -Kc[o][v];
            // (K^2)(o1, o2) = -sum_v Kc[o1][v] Kc[o2][v], (K^2)(v1, v2) = -sum_o Kc[o][v1] Kc[o][v2]
            flat<T, R>(j, nocc * nocc, nv, 1, 1, [&](int e) { return Kc + (e % nocc) * nv; },
                       [&](int e) { return Kc + (e / nocc) * nv; }, [&](int e, double v) {
                           const int o1 = e % nocc, o2 = e / nocc;
                           A[occ_list[o2] * LD + occ_list[o1]] = fma(-0.5, v, o1 == o2 ? 1.0 : 0.0);
                       });
            flat<T, R>(j, nv * nv, nocc, nv, nv, [&](int e) { return Kc + (e % nv); },
                       [&](int e) { return Kc + (e / nv); }, [&](int e, double v) {
                           const int v1 = e % nv, v2 = e / nv;
                           A[virt_list[v2] * LD + virt_list[v1]] = fma(-0.5, v, v1 == v2 ? 1.0 : 0.0);
                       });
            for (int e = j; e < nocc * nv; e += T) {
                const int vi = virt_list[e % nv], oi = occ_list[e / nv];
                const double k = Kc[e];
                A[oi * LD + vi] = k;    // V(v, o) = K(v, o)
                A[vi * LD + oi] = -k;   // V(o, v) = K(o, v)
            }
            g.sync();
            flat<T, R>(j, nn, n, LD, 1, [&](int e) { return C + (e % n); }, [&](int e) { return A + (e / n) * LD; },
                       [&](int e, double v) { Y[(e / n) * LD + e % n] = v; });
            g.sync();
            double *t = C;
            C = Y;
            Y = t;
        } else {
            // the rest of C^T H C: the occupied and virtual diagonal blocks
            flat<T, R>(j, nocc * nocc, n, 1, 1, [&](int e) { return C + occ_list[e % nocc] * LD; },
                       [&](int e) { return Y + occ_list[e / nocc] * LD; },
                       [&](int e, double v) { A[occ_list[e / nocc] * LD + occ_list[e % nocc]] = v; });
            flat<T, R>(j, nv * nv, n, 1, 1, [&](int e) { return C + virt_list[e % nv] * LD; },
                       [&](int e) { return Y + virt_list[e / nv] * LD; },
                       [&](int e, double v) { A[virt_list[e / nv] * LD + virt_list[e % nv]] = v; });
            g.sync();
            // a cold start sweeps until the off-diagonal entries are below tolerance, at most `cap`
            // sweeps (then DEVICE_TIMEOUT); later iterations take one sweep
            const int cap = cold_first ? (a.max_sweeps > 0 ? a.max_sweeps : G_MAX_SWEEPS) : 1;
            for (int sweep = 0;; ++sweep) {
                bool off_small = true;
                for (int e = j; e < nn; e += T) {
                    const int c = e / n, i = e - c * n;
                    if (i != c && !abs_lt(A[c * LD + i], G_JACOBI_TOL)) off_small = false;
                }
                if (g.all(off_small)) break;
                if (sweep >= cap) {
                    if (cold_first && j == 0) atomicOr(&fl[0], ERRBIT_TIMEOUT);
                    break;
                }
                for (int rd = 0; rd < n - 1; ++rd) {
                    if (j < n / 2) {   // the rotations of this round
                        int p, qq;
                        g_pair(j, rd, n, p, qq);
                        double c, s;
                        g_jacobi_cs(A[p * LD + p], A[qq * LD + qq], A[qq * LD + p], c, s);
                        pp[j] = p;
                        pq[j] = qq;
                        cs[2 * j] = c;
                        cs[2 * j + 1] = s;
                    }
                    g.sync();
                    for (int e = j; e < n * (n / 2); e += T) {   // columns p, q of A and C, row i
                        const int k = e / n, i = e - k * n;
                        const int p = pp[k], qq = pq[k];
                        const double c = cs[2 * k], s = cs[2 * k + 1];
                        const double ap = A[p * LD + i], aq = A[qq * LD + i];
                        A[p * LD + i] = fma(c, ap, -s * aq);
                        A[qq * LD + i] = fma(s, ap, c * aq);
                        const double cp = C[p * LD + i], cq = C[qq * LD + i];
                        C[p * LD + i] = fma(c, cp, -s * cq);
                        C[qq * LD + i] = fma(s, cp, c * cq);
                    }
                    g.sync();
                    for (int e = j; e < n * (n / 2); e += T) {   // rows p, q of A, column c
                        const int k = e / n, c = e - k * n;
                        const int p = pp[k], qq = pq[k];
                        const double ck = cs[2 * k], sk_ = cs[2 * k + 1];
                        const double x = A[c * LD + p], y = A[c * LD + qq];
                        A[c * LD + p] = fma(ck, x, -sk_ * y);
                        A[c * LD + qq] = fma(sk_, x, ck * y);
                    }
                    g.sync();
                }
            }
            if (j < n) diag[j] = A[j * LD + j];
            g.sync();
            rank_occupation();
            g.sync();
        }
        // Mulliken populations: (P S)_ii = 2 sum_o C(i, o) (S C)(i, o); S C_occ into A
        for (int e = j; e < n * nocc; e += T) {
            const int o = e / n, i = e - o * n;
            const double *co = C + occ_list[o] * LD;
            double acc = 0.0;
            for (int k = 0; k < n; ++k) acc = fma(s_at(i, k), co[k], acc);
            A[o * LD + i] = acc;
        }
        g.sync();
        if (j < n) {
            double qo = 0.0;
            for (int o = 0; o < nocc; ++o) qo = fma(C[occ_list[o] * LD + j], A[o * LD + j], qo);
            red[j] = 2.0 * qo;
        }
        g.sync();
        const int NH = a.hist;   // ring of the last NH iterates
        const int hs = (it - 1) % NH;
        if (j < nat) {
            double qa = 0.0;
            for (int o = atom_off[j]; o < atom_off[j + 1]; ++o) qa += red[o];
            qout[j] = qa;
            shl[j] = shift[j];
            hq[hs * AM + j] = q[j];
            hf[hs * AM + j] = qa - q[j];
        }
        g.sync();
        bool conv = eok;
        for (int at = 0; at < nat; ++at)
            if (!abs_lt(hf[hs * AM + at], a.scc_tol)) conv = false;
        const int h = min(it, NH);
        if (!conv && j == 0) {
            // Anderson coefficients over the h - 1 previous iterates: normal equations in FP32 with
            // a small diagonal shift, solved by Cholesky (they only steer the iteration)
            float Mx[GNHIST - 1][GNHIST - 1], bv[GNHIST - 1], x[GNHIST - 1];
            const int m = h - 1;
            for (int u = 0; u < m; ++u) {
                const int hu = (hs + NH - 1 - u) % NH;
                float b = 0.f;
                for (int w = 0; w <= u; ++w) {
                    const int hw = (hs + NH - 1 - w) % NH;
                    float s = 0.f;
                    for (int at = 0; at < nat; ++at) {
                        const float du = d2f_steer(hf[hu * AM + at] - hf[hs * AM + at]);
                        const float dw = d2f_steer(hf[hw * AM + at] - hf[hs * AM + at]);
                        s = fmaf(du, dw, s);
                    }
                    Mx[u][w] = s;
                }
                for (int at = 0; at < nat; ++at)
                    b = fmaf(-d2f_steer(hf[hu * AM + at] - hf[hs * AM + at]), d2f_steer(hf[hs * AM + at]), b);
                bv[u] = b;
            }
            float dmax = 0.f;
            for (int u = 0; u < m; ++u) dmax = fmaxf(dmax, Mx[u][u]);
            bool ok = m > 0 && dmax > 0.f;
            for (int u = 0; u < m && ok; ++u) {   // lower Cholesky factor of M + 1e-6 max(diag) I, in place
                for (int w = 0; w <= u && ok; ++w) {
                    float s = Mx[u][w] + (u == w ? 1e-6f * dmax : 0.f);
                    for (int l = 0; l < w; ++l) s -= Mx[u][l] * Mx[w][l];
                    if (u == w) {
                        if (!(s > 0.f)) ok = false; else Mx[u][u] = sqrtf(s);
                    } else {
                        Mx[u][w] = s / Mx[w][w];
                    }
                }
            }
            if (ok) {
                for (int u = 0; u < m; ++u) {
                    float s = bv[u];
                    for (int l = 0; l < u; ++l) s -= Mx[u][l] * x[l];
                    x[u] = s / Mx[u][u];
                }
                for (int u = m - 1; u >= 0; --u) {
                    float s = x[u];
                    for (int l = u + 1; l < m; ++l) s -= Mx[l][u] * x[l];
                    x[u] = s / Mx[u][u];
                }
                for (int u = 0; u < m; ++u)
                    if (!(fabsf(x[u]) < 50.f)) ok = false;
            }
            for (int u = 0; u < GNHIST - 1; ++u) th[u] = (ok && u < m) ? f2d_steer(x[u]) : 0.0;
        }
        g.sync();
        if (j < nat) {
            if (conv) {
                q[j] = qout[j];
            } else {
                const double q0 = hq[hs * AM + j], f0 = hf[hs * AM + j];
                double qb = q0, fb = f0;
                for (int u = 0; u < h - 1; ++u) {
                    const int hu = (hs + NH - 1 - u) % NH;
                    qb = fma(th[u], hq[hu * AM + j] - q0, qb);
                    fb = fma(th[u], hf[hu * AM + j] - f0, fb);
                }
                q[j] = fma(a.beta, fb, qb);
            }
        }
        g.sync();   // the next iteration's shifts read every atom's charge
        if (conv) {   // the same value in every thread: all leave together
            if (j == 0) fl[2] = it;
            break;
        }
    }
    g.sync();
    if (j == 0 && it > a.max_iter) {
        atomicOr(&fl[0], ERRBIT_SCC_NOCONV);
        fl[2] = a.max_iter;
    }
    g.sync();
    }   // general path

    if (disp) {   // displaced copy: only the dipole of the converged charges
        if (j == 0) {
            double mu[3] = {0.0, 0.0, 0.0};
            for (int at = 0; at < nat; ++at) {
                const double Q = zv[at] - q[at];
                for (int k = 0; k < 3; ++k) mu[k] = fma(Q, pos[at][k] - pos[0][k], mu[k]);
            }
            a.M_disp[(long long)(a.fd_central ? 6 : 3) * a0 + kd] = fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
            if (fl[0]) atomicOr(a.status, (unsigned)fl[0]);
        }
        g.sync();
        return;
    }

    // ---------------------------------------------------------------- energy, forces, dipole
    const double *P = C, *W = SH;
    if (warm) {
        // W = 2 C_o A_oo C_o^T and P = 2 C_o C_o^T with A_oo = C_o^T (H C_o) of the last evaluation: A <- A_oo;
        // Y <- t = 2 A_oo C_o^T; A <- P and SH <- W, the entries above the diagonal (all that the pair
        // gradients read). Band energy: Tr P H0 = 2 Tr A_oo - sum_A q_A eps_A.
        const double *XB = (const double *)(sm + L.XB);
        double *cwo = a.Cwarm + coff;
        for (int e = j; e < nn; e += T) {
            const int c = e / n;
            cwo[e] = C[c * LD + (e - c * n)];
        }
        flat<T, R>(j, nocc * (nocc + 1) / 2, n, 1, 1,
                   [&](int e) { return C + g_lower(e, nocc).x * LD; },
                   [&](int e) { return XB + g_lower(e, nocc).y * LD; }, [&](int e, double v) {
                       const int2 ic = g_lower(e, nocc);
                       const int i = ic.x, c = ic.y;
                       A[c * LD + i] = v;
                       A[i * LD + c] = v;
                   });
        g.sync();
        if (j == 0) {
            double eb = 0.0;
            for (int o = 0; o < nocc; ++o) eb += A[o * LD + o];
            eb *= 2.0;
            // the shifts and A_oo are those of the charges q - moved; with 1/2 sum_A dq_A eps_A below this is the
            // energy there, which differs from that at q to second order
            const float *moved = (const float *)hq;
            for (int at = 0; at < nat; ++at) eb = fma(fma(0.5, f2d_steer(moved[at]), -q[at]), shift[at], eb);
            red[0] = eb;
        }
        // t(o, i) = 2 sum_p A_oo(o, p) C(i, p) into Y[i * LD + o]
        flat<T, R>(j, nocc * n, nocc, LD, LD, [&](int e) { return A + (e % nocc); }, [&](int e) { return C + (e / nocc); },
                   [&](int e, double v) { Y[(e / nocc) * LD + e % nocc] = 2.0 * v; });
        g.sync();
        if (n > 1) {   // entries (row c, column i), c < i: the strict lower triangle (i, c) transposed
            flat<T, R>(j, n * (n - 1) / 2, nocc, LD, LD,
                       [&](int e) { return C + g_lower(e, n - 1).x + 1; },
                       [&](int e) { return C + g_lower(e, n - 1).y; }, [&](int e, double v) {
                           const int2 ic = g_lower(e, n - 1);
                           A[(ic.x + 1) * LD + ic.y] = 2.0 * v;
                       });
            flat<T, R>(j, n * (n - 1) / 2, nocc, 1, LD,
                       [&](int e) { return Y + (g_lower(e, n - 1).x + 1) * LD; },
                       [&](int e) { return C + g_lower(e, n - 1).y; }, [&](int e, double v) {
                           const int2 ic = g_lower(e, n - 1);
                           SH[(ic.x + 1) * LD + ic.y] = v;
                       });
        }
        if (j < nat) shl[j] = shift[j];
        g.sync();
        P = A;
    } else {
    {   // eigenvectors for the next warm start
        double *cwo = a.Cwarm + coff;
        for (int e = j; e < nn; e += T) {   // occupied columns first, as the warm path reads them
            const int c = e / n, src = c < nocc ? occ_list[c] : virt_list[c - nocc];
            cwo[e] = C[src * LD + (e - c * n)];
        }
    }
    if (j < nat) {
        double sh = 0.0;
        for (int k = 0; k < nat; ++k) sh = fma(gam[j * AM + k], q[k] - zv[k], sh);
        shift[j] = sh;
    }
    // W = 2 C_occ (C_occ^T H C_occ) C_occ^T with the H of the last iteration and the whole occupied
    // block. Buffers: A <- H; Y <- T = H C_occ; A <- C_occ; C <- Aoo = C_occ^T T;
    // Y <- t = 2 Aoo C_occ^T; C <- P; SH <- W = C_occ t; Y <- pair gradients
    for (int e = j; e < nn; e += T) {
        const int c = e / n, i = e - c * n;
        A[c * LD + i] = fma(0.5 * s_at(i, c), shl[orb_atom[i]] + shl[orb_atom[c]], h0_at(i, c));
    }
    g.sync();
    flat<T, R>(j, n * nocc, n, LD, 1, [&](int e) { return A + (e % n); },
               [&](int e) { return C + occ_list[e / n] * LD; }, [&](int e, double v) { Y[(e / n) * LD + e % n] = v; });
    g.sync();
    for (int e = j; e < n * nocc; e += T) {
        const int o = e / n, i = e - o * n;
        A[o * LD + i] = C[occ_list[o] * LD + i];
    }
    g.sync();
    flat<T, R>(j, nocc * nocc, n, 1, 1, [&](int e) { return A + (e % nocc) * LD; },
               [&](int e) { return Y + (e / nocc) * LD; }, [&](int e, double v) { C[(e / nocc) * LD + e % nocc] = v; });
    g.sync();
    // t(o, i) = 2 sum_o2 Aoo(o, o2) C_occ(i, o2) into Y[i * LD + o]
    flat<T, R>(j, nocc * n, nocc, LD, LD, [&](int e) { return C + (e % nocc); }, [&](int e) { return A + (e / nocc); },
               [&](int e, double v) { Y[(e / nocc) * LD + e % nocc] = 2.0 * v; });
    if (j == 0 && nocc < n) {   // HOMO-LUMO gap of the last iteration
        double homo = -1e300, lumo = 1e300;
        for (int c = 0; c < n; ++c) {
            if (occf[c]) homo = fmax(homo, diag[c]); else lumo = fmin(lumo, diag[c]);
        }
        if (!(lumo - homo > G_MIN_GAP)) atomicOr(&fl[0], ERRBIT_ZERO_GAP);
    }
    g.sync();
    // P = 2 C_occ C_occ^T into C
    flat<T, R>(j, nn, nocc, LD, LD, [&](int e) { return A + (e % n); }, [&](int e) { return A + (e / n); },
               [&](int e, double v) { C[(e / n) * LD + e % n] = 2.0 * v; });
    g.sync();
    if (j < n) {   // band energy, per column in a fixed order
        double eb = 0.0;
        for (int i = 0; i < n; ++i) eb = fma(C[j * LD + i], h0_at(i, j), eb);
        red[j] = eb;
    }
    g.sync();
    // W(i, c) = sum_o C_occ(i, o) t(o, c) into SH
    flat<T, R>(j, nn, nocc, LD, 1, [&](int e) { return A + (e % n); }, [&](int e) { return Y + (e / n) * LD; },
               [&](int e, double v) { SH[(e / n) * LD + e % n] = v; });
    g.sync();
    P = C;
    }
    double *gp = Y, *ep = Y + 3 * L.pmax;
    for (int pi = j; pi < npair; pi += T) {
        const int PA = pa[pi], PB = pb[pi];
        const int eA = spec[PA], eB = spec[PB];
        const int oA = atom_off[PA], oB = atom_off[PB];
        const int na = sk.norb[eA], nb = sk.norb[eB];
        const double dx = pos[PB][0] - pos[PA][0], dy = pos[PB][1] - pos[PA][1], dz = pos[PB][2] - pos[PA][2];
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        const double ir = rsqrt_nr(r2);
        const double r = r2 * ir;
        const double e[3] = {dx * ir, dy * ir, dz * ir};
        const double hshift = 0.5 * (shl[PA] + shl[PB]);
        double gk[3] = {0.0, 0.0, 0.0};
        for (int t = 0; t < 2; ++t) {
            const double(*tab)[CAVMD_MAX_ELEM][4][4] = t == 0 ? sk.h0 : sk.s;
            // weights of the (A, B) block: P for H0, P (eps_A + eps_B)/2 - W for S
            auto wt = [&](int mu, int nu) -> double {
                const double pv = P[nu * LD + mu];
                return t == 0 ? pv : fma(pv, hshift, -W[nu * LD + mu]);
            };
            double v, dv;
            radial_g(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
            {
                const double w = wt(oA, oB) * dv;
                for (int k = 0; k < 3; ++k) gk[k] = fma(w, e[k], gk[k]);
            }
            if (nb == 4) {
                radial_g(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                double w[3], we = 0.0;
                for (int i = 0; i < 3; ++i) { w[i] = wt(oA, oB + 1 + i); we = fma(w[i], e[i], we); }
                for (int k = 0; k < 3; ++k) gk[k] += fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
            }
            if (na == 4) {
                radial_g(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                double w[3], we = 0.0;
                for (int i = 0; i < 3; ++i) { w[i] = wt(oA + 1 + i, oB); we = fma(w[i], e[i], we); }
                for (int k = 0; k < 3; ++k) gk[k] -= fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
            }
            if (na == 4 && nb == 4) {
                double vs, dvs, vp, dvp;
                radial_g(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dvs);
                radial_g(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dvp);
                double Wm[3][3], We[3] = {0, 0, 0}, WTe[3] = {0, 0, 0}, tr = 0.0;
                for (int i = 0; i < 3; ++i)
                    for (int k = 0; k < 3; ++k) Wm[i][k] = wt(oA + 1 + i, oB + 1 + k);
                for (int i = 0; i < 3; ++i) {
                    tr += Wm[i][i];
                    for (int k = 0; k < 3; ++k) {
                        We[i] = fma(Wm[i][k], e[k], We[i]);
                        WTe[k] = fma(Wm[i][k], e[i], WTe[k]);
                    }
                }
                double eWe = 0.0;
                for (int i = 0; i < 3; ++i) eWe = fma(e[i], We[i], eWe);
                const double dl = vs - vp, ddl = dvs - dvp;
                for (int k = 0; k < 3; ++k)
                    gk[k] += (We[k] + WTe[k] - 2.0 * eWe * e[k]) * dl * ir + eWe * e[k] * ddl + tr * e[k] * dvp;
            }
        }
        for (int k = 0; k < 3; ++k) gk[k] *= 2.0;
        const double gi = rsqrt_nr(fma(r, r, sk.gamma_c2[eA][eB]));
        const double dgam = -r * gi * gi * gi;
        const double qq = (q[PA] - zv[PA]) * (q[PB] - zv[PB]) * dgam;
        const double arep = sk.rep[eA][eB][0], brep = sk.rep[eA][eB][1];
        double erep = 0.0, derep = 0.0;
        if (arep != 0.0) {
            const double vr = arep * exp(-brep * r);
            const double x = (r - (sk.r_cut - sk.taper)) * sk.inv_taper;
            double f = 1.0, df = 0.0;
            if (x > 0.0) {
                if (x < 1.0) {
                    double sn, cn;
                    sincospi(x, &sn, &cn);
                    f = 0.5 * (1.0 + cn);
                    df = -0.5 * 3.141592653589793 * sk.inv_taper * sn;
                } else {
                    f = 0.0;
                }
            }
            erep = vr * f;
            derep = vr * (df - brep * f);
        }
        for (int k = 0; k < 3; ++k) gp[3 * pi + k] = gk[k] + (qq + derep) * e[k];
        ep[pi] = erep;
    }
    g.sync();
    if (j < nat) {
        double f[3] = {0.0, 0.0, 0.0}, er = 0.0;
        for (int x = 0; x < nat; ++x) {
            if (x == j) continue;
            const int pi = pair_of(x, j);
            const double sg = x < j ? -1.0 : 1.0;
            for (int k = 0; k < 3; ++k) f[k] = fma(sg, gp[3 * pi + k], f[k]);
            if (x < j) er += ep[pi];
        }
        hq[j] = er;   // the repulsion of the pairs whose second atom this is
        const int at = a0 + j;
        for (int k = 0; k < 3; ++k) a.F[3 * at + k] = f[k];
        a.qprev[at] = a.have_warm ? qst[j] : q[j];
        a.qpop[at] = q[j];
        if (a.Qout) a.Qout[at] = zv[j] - q[j];
        if (a.write_b) {
            const double Q = zv[j] - q[j];
            a.b[3 * at + 0] = Q * a.pol0;
            a.b[3 * at + 1] = Q * a.pol1;
            a.b[3 * at + 2] = Q * a.pol2;
        }
    }
    g.sync();
    if (j == 0) {
        double E = 0.0;
        if (warm) E = red[0];
        else
            for (int i = 0; i < n; ++i) E += red[i];
        double e2 = 0.0;   // sum_A dq_A eps_A (the shifts of the converged charges)
        for (int x = 0; x < nat; ++x) e2 = fma(q[x] - zv[x], shift[x], e2);
        E = fma(0.5, e2, E);
        for (int x = 0; x < nat; ++x) E += hq[x];
        double mu[3] = {0.0, 0.0, 0.0};
        for (int at = 0; at < nat; ++at) {
            const double Q = zv[at] - q[at];
            for (int k = 0; k < 3; ++k) mu[k] = fma(Q, pos[at][k] - pos[0][k], mu[k]);
        }
        a.E_cell[cell] = E;
        a.M_cell[cell] = fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
        a.iters[cell] = fl[2];
        if (fl[0]) atomicOr(a.status, (unsigned)fl[0]);
    }
    g.sync();
}

// Persistent grid over a queue of work units: units [0, n_big) are one large item each (the whole
// block), the rest take two small items (one per half of the block).
template <int R>
__global__ void __launch_bounds__(BT, 2) k_dftb_generic(const DevSK *__restrict__ skp, const DftbArgs a,
                                                     const int2 *__restrict__ items, int n_big, int n_small,
                                                     unsigned *__restrict__ queue, int nmax_b, int amax_b,
                                                     int nmax_s, int amax_s, int warm) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int next;
    __shared__ int vote[2][TS / 32];
    const DevSK &sk = *skp;
    const GLayout Lb = g_layout(nmax_b, amax_b, warm);
    const GLayout Ls = g_layout(nmax_s, amax_s, warm);
    const int n_units = n_big + (n_small + 1) / 2;
    const int half = threadIdx.x / TS;
    for (;;) {
        if (threadIdx.x == 0) next = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int w = next;
        __syncthreads();
        if (w >= n_units) break;
        if (w < n_big) {
            const int2 it = items[w];
            const Grp<TB> g{(int)threadIdx.x, 0, nullptr};
            g_molecule<TB, R>(sk, a, Lb, smem, it.x, it.y, g);
        } else {
            const int s = 2 * (w - n_big) + half;
            if (s < n_small) {
                const int2 it = items[n_big + s];
                const Grp<TS> g{(int)threadIdx.x - half * TS, 1 + half, vote[half]};
                g_molecule<TS, R>(sk, a, Ls, smem + half * Ls.total, it.x, it.y, g);
            }
        }
        __syncthreads();
    }
}

}  // namespace
