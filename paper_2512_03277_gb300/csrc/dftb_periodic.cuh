// Batched Gamma-point SCC-DFTB of periodic cells: the paper's per-molecule systems are cubic cells
// of 33 waters with periodic boundaries in all three directions and Gamma-point sampling (section
// "Computational details").
//
// What is computed (the textbook Gamma-point forms):
//   * H0 and S: the (A, B) block is the sum over lattice images T of the Slater-Koster block at
//     d = r_B + T - r_A, |d| < r_cut (for A = B the T = 0 term is the on-site block);
//   * gamma: Ewald lattice sum of 1/r (tin-foil boundary, neutralising background) plus the
//     Klopman-Ohno remainder 1/sqrt(r^2 + c^2) - 1/r over images with the cosine taper at r_cut,
//     and U_A on the diagonal. The real-space part is a matrix formed once per evaluation; the
//     reciprocal part acts on the charges through structure factors in every SCC iteration;
//   * the SCC loop, band + second-order + repulsion energy and its analytic gradient, every term
//     summed over the same images.
//
// Mapping to the machine. A 33-water cell has 198 orbitals: one 198 x 198 FP64 matrix is 313 KB,
// more than a block's shared memory, and GB300's FP64 pipe (2 FMA per clock per SM) is the only
// bottleneck. So each cell is one 256-thread block of a persistent grid (two per SM), its
// matrices live in a per-block global workspace (L2-resident while the cell runs), and every
// product stages k-chunks of its operands in shared memory and spreads its output entries
// evenly over the threads (8 per thread per pass, each summed over k in increasing order), so the
// results do not depend on the launch shape. Per SCC iteration only what the update needs is
// formed: H, Y = H C, the diagonal and the occupied-virtual block of C^T Y, and a rotation by the
// occupied-virtual generator K(v, o) = A_vo / (A_oo - A_vv): while some entry of K is 1e-4 or
// more, the Cayley rotation C <- C (I - K/2)^-1 (I + K/2), orthogonal to rounding for any K (two
// small Cholesky factorisations, I + X^T X / 4 and I + X X^T / 4, X = K_vo, and row solves);
// below that, C <- C (I + K + K^2/2), orthogonal to O(K^4), as two staged products. A cold start
// diagonalises C^T H C once by cyclic Jacobi sweeps; warm starts re-orthonormalise the previous
// step's C under the new overlap by a Cholesky factor of C^T S C, and their first iteration runs
// one Jacobi sweep inside the occupied and inside the virtual block: the diagonal denominators
// need those blocks nearly diagonal, and without the sweeps their off-diagonal part grows (a cold
// start leaves it large, then it drifts with every step; its norm over 132 nearly degenerate
// occupied orbitals reaches the gap) and the iteration count with it.
#pragma once

#include "cavmd_internal.cuh"

namespace {

constexpr int PT = 256;          // threads per block (one cell at a time)
constexpr int PE = 8;            // product entries per thread per pass
constexpr int KC = 24;           // contraction chunk staged in shared memory
constexpr int ZC = 80;           // columns of the second operand staged per pass
constexpr int PNMAX = 256;       // orbitals per cell
constexpr int PAMAX = 128;       // atoms per cell
constexpr int PHIST = 6;         // largest Anderson history
constexpr int P_MAX_SWEEPS = 40;   // default bound on the Jacobi sweeps of a cold start
constexpr double P_JACOBI_TOL = 1e-11;   // cold start: off-diagonal size where the sweeps stop
constexpr double P_MIN_GAP = 1e-3;
constexpr double P_EIG_TOL = 1e-10;
constexpr float P_KMAX_PERT = 1e-4f;      // generator size below which C (I + K + K^2/2) is used
constexpr int P_SWEEP_PERIOD = 1;         // warm steps between within-block Jacobi sweeps (every fourth
                                          // step measured slower: 13.6 SCC iterations instead of 11.9)
constexpr int P_SWEEP_ITERS = 12;         // or after an evaluation with more SCC iterations than this
constexpr double PI_D = 3.141592653589793;
constexpr int PW_FP32_ITERS = 5;        // warm path (p_warm): bound on the FP32 Newton steps,
constexpr float PW_FP32_KTOL = 3e-5f;   // the rotation below which the next step would be FP32 rounding
constexpr float PW_ROT_MAX = 0.3f;      // the largest rotation taken (beyond: the general path)
constexpr int PW_EVALS = 8;             // and bound on the FP64 evaluations
constexpr float PW_ORTH_MAX = 5e-4f;    // norm (over all k-points) of the overlap defect that the last FP64 correction takes,
constexpr float PW_ORTH_ONCE = 5e-4f;   // norm (of one k-point) above which another one follows
constexpr float PW_ORTH_CUBE = 2e-5f;   // and above which its cubic term counts
constexpr float PW_ROT64_MAX = 1e-2f;   // norm of a rotation between FP64 evaluations,
constexpr float PW_ROT64_ONCE = 3e-4f;  // and above which the correction follows it (below, C stays orthonormal to 3e-15)
constexpr float PW_GAP = 2e-3f;         // HOMO-LUMO gap (Hartree) the warm path needs, above P_MIN_GAP
constexpr int PW_CG_SLOW = 6;           // conjugate-gradient steps of the first Newton step that ask for a block sweep
constexpr int PW_BISECT = 6;            // tries for a level between the occupied and the empty ones
constexpr float PW_LAST_TOL = 0.1f;     // relative residual of the last solve, of a rotation below 1e-9
constexpr int PW_CG_ITERS = 60;         // bound on the conjugate-gradient steps of a Newton step

// Shared memory of one block; PN is the largest problem dimension (the orbitals of a cell at the
// Gamma point, twice that for the real form of a complex k-point problem).
template <int PN>
struct PSharedT {
    double Xs[KC * PN];
    double Zs[KC * ZC];
    double pos[PAMAX][3];
    double zv[PAMAX], q[PAMAX], qout[PAMAX], qst[PAMAX], dq[PAMAX], shift[PAMAX];
    double hq[PHIST][PAMAX], hf[PHIST][PAMAX];
    double diag[PN], red[PN], invd[PN];
    double cs[PN];               // Jacobi (c, s) of the rotations of one round
    double qk[PNMAX];            // k-grid: populations summed over the k-points of one iteration
    double hl[2];                // k-grid: highest occupied and lowest empty level over the k-points
    double th[PHIST];
    double gred[PT / 32][3];
    int spec[PAMAX], atom_off[PAMAX + 1], orb_atom[PNMAX];
    int lst[PAMAX];              // atoms with p orbitals, then those without
    int occ_list[PN], virt_list[PN], occf[PN];
    int pp[PN / 2], pq[PN / 2];
    int fl[8];                   // 0 error bits, 1 n, 2 iterations, 3 occupied orbitals, 5 atoms with p orbitals
    int vote[PT / 32];
};
using PShared = PSharedT<PNMAX>;
using PSharedK = PSharedT<2 * PNMAX>;

__device__ __forceinline__ bool blk_all(bool p) { return __syncthreads_and(p) != 0; }

__device__ __forceinline__ void cutoff_fn(double r, const DevSK &sk, double &f, double &df) {
    const double x = (r - (sk.r_cut - sk.taper)) * sk.inv_taper;
    f = 1.0;
    df = 0.0;
    if (x > 0.0) {
        if (x < 1.0) {
            double sn, cn;
            sincospi(x, &sn, &cn);
            f = 0.5 * (1.0 + cn);
            df = -0.5 * PI_D * sk.inv_taper * sn;
        } else {
            f = 0.0;
        }
    }
}

// V(r) = a exp(-b r) (1 + c1 r + c2 r^2) f_cut(r) and dV/dr.
__device__ __forceinline__ void radial_p(const double *par, double r, const DevSK &sk, double &v, double &dv) {
    const double a = par[0], b = par[1], c1 = par[2], c2 = par[3];
    const double e = a * exp(-b * r);
    const double poly = fma(fma(c2, r, c1), r, 1.0);
    const double dpoly = fma(2.0 * c2, r, c1);
    double f, df;
    cutoff_fn(r, sk, f, df);
    v = e * poly * f;
    dv = e * (fma(-b * poly, f, dpoly * f) + poly * df);
}

// Column of entry e of the packed lower triangle of an m x m matrix, stored column by column
// (column c holds rows c..m-1 and starts at c m - c (c - 1) / 2).
__device__ __forceinline__ int lower_col(int e, int m) {
    const float b = 2.0f * (float)m + 1.0f;
    int c = (int)((b - sqrtf(fmaxf(b * b - 8.0f * (float)e, 0.0f))) * 0.5f);
    c = max(0, min(c, m - 1));
    while (c > 0 && c * m - c * (c - 1) / 2 > e) --c;
    while (c + 1 < m && (c + 1) * m - (c + 1) * c / 2 <= e) ++c;
    return c;
}

// Block-wide product: out(i, c) = sum_{k < K} xa(i, k) za(k, c) for the entries of an m x w
// matrix (LOWER: the entries i >= c of an m x m one), the sum taken in increasing k; epi(i, c, v)
// receives each entry once. Passes of up to PT * PE entries in column order; each k-chunk of the
// m rows of X and of the pass's columns of Z is staged in shared memory first.
// XK: consecutive k of X are adjacent in memory (else consecutive i); ZK: consecutive k of Z are
// adjacent (else consecutive c). They only choose the staging order, for coalesced loads.
template <bool LOWER, bool XK, bool ZK, class SH, class XA, class ZA, class EPI>
__device__ void pprod(SH &sh, int m, int w, int K, XA xa, ZA za, EPI epi) {
    const int tid = threadIdx.x;
    const int n_out = LOWER ? m * (m + 1) / 2 : m * w;
    const int pe = LOWER ? PT * PE : min(PT * PE, m * (ZC - 2));
    for (int e0 = 0; e0 < n_out; e0 += pe) {
        const int e1 = min(e0 + pe, n_out);
        const int c_lo = LOWER ? lower_col(e0, m) : e0 / m;
        const int c_hi = LOWER ? lower_col(e1 - 1, m) : (e1 - 1) / m;
        const int ncol = c_hi - c_lo + 1;
        int ii[PE], cc[PE];
        double acc[PE];
#pragma unroll
        for (int r = 0; r < PE; ++r) {
            const int e = min(e0 + tid + r * PT, e1 - 1);
            int i, c;
            if (LOWER) {
                c = lower_col(e, m);
                i = c + (e - (c * m - c * (c - 1) / 2));
            } else {
                c = e / m;
                i = e - c * m;
            }
            ii[r] = i;
            cc[r] = c - c_lo;
            acc[r] = 0.0;
        }
        for (int k0 = 0; k0 < K; k0 += KC) {
            const int kc = min(KC, K - k0);
            __syncthreads();
            for (int idx = tid; idx < kc * m; idx += PT) {
                int kk, i;
                if (XK) { i = idx / kc; kk = idx - i * kc; } else { kk = idx / m; i = idx - kk * m; }
                sh.Xs[kk * m + i] = xa(i, k0 + kk);
            }
            for (int idx = tid; idx < kc * ncol; idx += PT) {
                int kk, cl;
                if (ZK) { cl = idx / kc; kk = idx - cl * kc; } else { kk = idx / ncol; cl = idx - kk * ncol; }
                sh.Zs[kk * ZC + cl] = za(k0 + kk, c_lo + cl);
            }
            __syncthreads();
            for (int kk = 0; kk < kc; ++kk) {
#pragma unroll
                for (int r = 0; r < PE; ++r) acc[r] = fma(sh.Xs[kk * m + ii[r]], sh.Zs[kk * ZC + cc[r]], acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < PE; ++r)
            if (e0 + tid + r * PT < e1) epi(ii[r], cc[r] + c_lo, acc[r]);
    }
    __syncthreads();
}

// In-place lower Cholesky factor of the m x m matrix A (column-major, leading dimension m; the
// lower triangle is read and written), right-looking with one thread per trailing column.
// Returns false (in every thread) when a pivot is not positive.
template <class SH>
__device__ bool pchol(double *A, int m, SH &sh) {
    const int j = threadIdx.x;
    if (j == 0) sh.fl[4] = 0;
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        if (j == 0) {
            double d = A[k * m + k];
            if (!(d > 1e-300)) { sh.fl[4] = 1; d = 1.0; }
            const double y = rsqrt_nr(d);
            sh.invd[k] = y;
            A[k * m + k] = d * y;
        }
        __syncthreads();
        const double y = sh.invd[k];
        for (int i = k + 1 + j; i < m; i += PT) A[k * m + i] *= y;
        __syncthreads();
        for (int jj = k + 1 + j; jj < m; jj += PT) {
            const double ljk = A[k * m + jj];
            for (int i = jj; i < m; ++i) A[jj * m + i] = fma(-A[k * m + i], ljk, A[jj * m + i]);
        }
        __syncthreads();
    }
    const bool ok = sh.fl[4] == 0;
    __syncthreads();
    return ok;
}

// Row solve x L^T = z (forward substitution) for one row of length m with stride xs, in place.
__device__ __forceinline__ void row_solve_lt(const double *L, int m, const double *invd, double *x, int xs) {
    for (int c = 0; c < m; ++c) {
        double v = x[c * xs];
        for (int k = 0; k < c; ++k) v = fma(-x[k * xs], L[k * m + c], v);
        x[c * xs] = v * invd[c];
    }
}

// Row solve x L L^T = z for one row (z, x of length m, strides zs and xs), L the lower factor
// above: forward u L^T = z, then backward x L = u. x may alias z.
__device__ __forceinline__ void row_solve_llt(const double *L, int m, const double *invd, const double *z, int zs,
                                              double *x, int xs) {
    for (int c = 0; c < m; ++c) {   // u_c = (z_c - sum_{k<c} u_k L(c, k)) / L(c, c)
        double v = z[c * zs];
        for (int k = 0; k < c; ++k) v = fma(-x[k * xs], L[k * m + c], v);
        x[c * xs] = v * invd[c];
    }
    for (int c = m - 1; c >= 0; --c) {   // x_c = (u_c - sum_{k>c} x_k L(k, c)) / L(c, c)
        double v = x[c * xs];
        for (int k = c + 1; k < m; ++k) v = fma(-x[k * xs], L[c * m + k], v);
        x[c * xs] = v * invd[c];
    }
}

// Round-robin Jacobi schedule for even n: pair k of round r (0..n-2); index n-1 meets r.
__device__ __forceinline__ void p_pair(int k, int r, int n, int &p, int &q) {
    const int m = n - 1;
    if (k == 0) { p = r; q = m; return; }
    const int x = (r + k) % m, y = (r - k + m) % m;
    p = min(x, y);
    q = max(x, y);
}

// Rotation annihilating a_pq: angle from FP32, (c, s) normalised in FP64 by two Newton steps.
__device__ __forceinline__ void p_jacobi_cs(double app, double aqq, double apq, double &c, double &s) {
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


// Device view of the periodic plan (by value).
struct PbcDev {
    double lat[9], inv[9];       // lattice vectors as rows; fractional coordinates f = r inv
    double alpha, bg, self_e;    // Ewald alpha, -pi / (alpha^2 V), -2 alpha / sqrt(pi)
    double r_real2;              // real-space cutoff squared
    int n_img, n_img_sk, n_g, nmax, amax;
    int n_g32, g_max;            // vectors that matter in FP32; largest |m| of a vector
    const int4 *gi;              // [n_g] the vectors' integer coordinates
    const double *img;           // [n_img][3] lattice translations by increasing length; the first
                                 // n_img_sk reach every image within r_cut
    const double *gw;            // [n_g][4] half-space reciprocal vectors G and 2 w_G
    double *work;                // per-block workspaces
    long long work_stride;       // doubles per block
    int nk;                      // k-grid: irreducible k-points (0: Gamma-point kernel)
    int cluster;                 // k-grid: blocks that share a cell
    int lean;                    // k-grid: workspaces without the warm path's part
    int late_pass;               // k-grid: 1 evaluates the items of `late` by the general path
    int *late;                   // k-grid, clusters: [1 + items] count and items that left the warm path
    const double *kpt;           // [nk][4] fractional k (units of the reciprocal rows) and weight
};

// Memory of one cell's evaluation (global workspace): the block's own work matrices, and what the
// blocks that share a cell hold in common (k-grid cells can take a cluster of blocks, one slice of the
// k-points each).
struct PbcMem {
    double *H, *Y, *P, *Xg, *Mo, *Mv;   // this block's, n2 doubles each
    double *sgf, *pbuf;                 // [n_g][2] structure factors; [nat][nat][4] pair gradients and energies
    long long pbuf_stride;              // from one block's pbuf to the next one's
    float *g32;                         // [nat][nat] the whole gamma matrix (with the reciprocal part) in FP32
    double *H0, *S;                     // Gamma: the matrices; k-grid: of the first k-point, 2 n2 apart
    float *kf;                          // k-grid: FP32 state of every k-point, 4 n2 floats apart
    double *gam, *csg;                  // real-space gamma; cos and sin of G . r
    double *pw;                         // this block's powers of the reciprocal phases
    double *Cd;                         // working bases of the warm path and of finite-difference copies
    double *xch;                        // [2][blocks][amax + 8] exchange between the blocks of a cell
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Every thread of every block of the cell; global writes before it are seen by the others after it.
__device__ __forceinline__ void cluster_barrier(int blocks) {
    if (blocks > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

// FP32 product in register tiles: epi(i, c, sum_{k < K} xa(i, k) za(k, c)) for i < m, c < w, each entry once.
// A block tile of 16 TM x 16 TN entries takes TM x TN per thread; chunks of 16 k are staged in shared
// memory, the next chunk's loads in flight meanwhile. Seven entries a side make 49 FMAs per 14 shared loads. XK (ZK): consecutive k of the operand are adjacent in
// memory (else consecutive i or c); they only choose the staging order.
template <int TM, int TN, bool XK, bool ZK, class SH, class XA, class ZA, class EPI>
__device__ __forceinline__ void fprod(SH &sh, int m, int w, int K, XA xa, ZA za, EPI epi) {
    constexpr int BM = 16 * TM, BN = 16 * TN, KF = 16, LX = BM + 1, LZ = BN + 1;
    constexpr int NX = KF * BM / PT, NZ = KF * BN / PT;
    static_assert(PT == 256 && KF * (LX + LZ) * 4 <= (int)sizeof(sh.Xs), "staging");
    float *Xs = reinterpret_cast<float *>(sh.Xs), *Zs = Xs + KF * LX;
    const int tid = threadIdx.x, ti = tid & 15, tc = tid >> 4;
    for (int c0 = 0; c0 < w; c0 += BN)
        for (int i0 = 0; i0 < m; i0 += BM) {
            float acc[TM][TN], px[NX], pz[NZ];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) acc[r][c] = 0.0f;
            auto load = [&](int k0) {
#pragma unroll
                for (int q = 0; q < NX; ++q) {
                    const int idx = tid + q * PT, kk = XK ? idx % KF : idx / BM, i = XK ? idx / KF : idx % BM;
                    px[q] = (i0 + i < m && k0 + kk < K) ? xa(i0 + i, k0 + kk) : 0.0f;
                }
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    const int idx = tid + q * PT, kk = ZK ? idx % KF : idx / BN, c = ZK ? idx / KF : idx % BN;
                    pz[q] = (c0 + c < w && k0 + kk < K) ? za(k0 + kk, c0 + c) : 0.0f;
                }
            };
            load(0);
            for (int k0 = 0; k0 < K; k0 += KF) {
                __syncthreads();
#pragma unroll
                for (int q = 0; q < NX; ++q) {
                    const int idx = tid + q * PT, kk = XK ? idx % KF : idx / BM, i = XK ? idx / KF : idx % BM;
                    Xs[kk * LX + i] = px[q];
                }
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    const int idx = tid + q * PT, kk = ZK ? idx % KF : idx / BN, c = ZK ? idx / KF : idx % BN;
                    Zs[kk * LZ + c] = pz[q];
                }
                __syncthreads();
                if (k0 + KF < K) load(k0 + KF);
#pragma unroll 4
                for (int kk = 0; kk < KF; ++kk) {
                    float x[TM], z[TN];
#pragma unroll
                    for (int r = 0; r < TM; ++r) x[r] = Xs[kk * LX + ti + 16 * r];
#pragma unroll
                    for (int c = 0; c < TN; ++c) z[c] = Zs[kk * LZ + tc + 16 * c];
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int c = 0; c < TN; ++c) acc[r][c] = fmaf(x[r], z[c], acc[r][c]);
                }
            }
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c)
                    if (i0 + ti + 16 * r < m && c0 + tc + 16 * c < w) epi(i0 + ti + 16 * r, c0 + tc + 16 * c, acc[r][c]);
        }
    __syncthreads();
}

// Atomic shifts eps_A = sum_B gamma_AB dq_B + the reciprocal part, from sh.dq into sh.shift.
template <class SH>
__device__ __noinline__ void p_shifts(SH &sh, const PbcDev &pl, const PbcMem &w, int nat) {
    const int j = threadIdx.x;
    for (int g = j; g < pl.n_g; g += PT) {
        double sc = 0.0, ss = 0.0;
        const double *t = w.csg + 2LL * g * nat;
        for (int at = 0; at < nat; ++at) {
            sc = fma(sh.dq[at], t[2 * at], sc);
            ss = fma(sh.dq[at], t[2 * at + 1], ss);
        }
        w.sgf[2 * g] = sc;
        w.sgf[2 * g + 1] = ss;
    }
    __syncthreads();
    // every thread: atom j % nat, a contiguous share of the vectors; the shares are added in order
    const int parts = PT / nat, part = j / nat, at = j - part * nat, per = (pl.n_g + parts - 1) / parts;
    if (part < parts) {
        const int g1 = min(pl.n_g, (part + 1) * per);
        double rr = 0.0;
        for (int g = part * per; g < g1; ++g) {
            const double *t = w.csg + 2LL * (g * nat + at);
            rr = fma(pl.gw[4 * g + 3], fma(t[0], w.sgf[2 * g], t[1] * w.sgf[2 * g + 1]), rr);
        }
        sh.Xs[j] = rr;
    }
    __syncthreads();
    if (j < nat) {
        double v = 0.0;
        for (int k = 0; k < nat; ++k) v = fma(w.gam[j * pl.amax + k], sh.dq[k], v);
        for (int q = 0; q < parts; ++q) v += sh.Xs[q * nat + j];
        sh.shift[j] = v;
    }
    __syncthreads();
}

// FP32 state of a k-point in the warm path: C, S C, C^T H C and K.
struct PState32 {
    float *C, *SC, *A, *x;
};

template <bool KG>
__device__ __forceinline__ PState32 p_state32(const PbcMem &wk, int kp, long long n2, int mm) {
    PState32 f;
    f.C = KG ? wk.kf + 4LL * kp * n2 : (float *)wk.P;
    f.SC = f.C + mm;
    f.A = KG ? f.C + 2 * mm : (float *)wk.Xg;
    f.x = f.A + mm;
    return f;
}

// The end of the warm path: the residual that passed its test stays in no result. With the rotation K that it
// asks for, q takes its change (moved), the shifts follow and C_o becomes C_o + C_v K. At the Gamma point half of
// the change C_o^T dH C_o of A_oo goes to Mv (a k-grid forms H anew). K is solved for, to a tenth: r / (A_vv - A_oo)
// in its place would leave half of the residual, since the blocks of A are not diagonal. Against 64 bits, 24 cells
// of 33 waters: forces 4.2e-14 -> 5.6e-15, charges 5.2e-13 -> 2.8e-14 (without this step -> with it). A call of its own,
// so that its registers are not p_warm's (inlined: 6,488 bytes of spill loads there instead of 3,772). 304 such cells: 73.5 -> 76.1 ms.
template <bool KG, class SH>
__device__ __noinline__ void p_settle(const DftbArgs &a, const PbcDev &pl, SH &sh, const PbcMem &wk, double *Cb,
                                      const float *moved, int n, int nocc, int nat, int rank, int blocks) {
    const int j = threadIdx.x;
    const int m = KG ? 2 * n : n, mo = KG ? 2 * nocc : nocc, mv = m - mo, mm = m * m;
    const long long n2 = (KG ? 4LL : 1LL) * pl.nmax * pl.nmax;
    if (j < nat) {
        sh.q[j] += f2d_steer(moved[j]);
        sh.dq[j] = sh.q[j] - sh.zv[j];
    }
    __syncthreads();
    if (a.n_disp > 0) return;   // a finite-difference copy needs only its charges
    for (int kp = rank; kp < (KG ? pl.nk : 1); kp += blocks) {
        const PState32 f = p_state32<KG>(wk, kp, n2, mm);
        double *C = Cb + (KG ? (long long)kp * mm : 0);
        fprod<5, 5, false, true>(sh, m, mo, mv, [&](int i, int k) { return f.C[(mo + k) * m + i]; },
                                 [&](int k, int c) { return f.x[c * mv + k]; },
                                 [&](int i, int c, float v) { C[(long long)c * m + i] += f2d_steer(v); });
    }
    if (!KG) {
        const PState32 f = p_state32<KG>(wk, 0, n2, mm);
        float *eo = (float *)sh.invd, *ea = (float *)sh.qst, *dA = (float *)wk.Mv;
        if (j < nat) {
            float s = 0.0f;
            for (int k = 0; k < nat; ++k) s = fmaf(wk.g32[k * nat + j], moved[k], s);
            ea[j] = 0.5f * s;
        }
        __syncthreads();
        for (int i = j; i < m; i += PT) eo[i] = ea[sh.orb_atom[i]];
        __syncthreads();
        fprod<5, 5, true, true>(sh, mo, mo, m, [&](int i, int k) { return f.C[i * m + k]; },
                                [&](int k, int c) { return eo[k] * f.SC[c * m + k]; },
                                [&](int i, int c, float v) { dA[c * mo + i] = v; });
    }
    p_shifts(sh, pl, wk, nat);
}

// Warm-started cell: the method of k_water_warm and g_warm (dftb_kernel.cu, dftb_generic.cuh) for the
// staged products of this kernel and for a set of k-points coupled by the charges.
//
// The general path spends about twelve FP64 iterations, Cholesky factors and Jacobi sweeps on iterates
// that are approximate until the last two. Here the previous bases (occupied columns first) are made
// orthonormal and moved by Newton steps of the orbital rotation in FP32, 64 times the FP64 rate; each
// step is solved by conjugate gradients over all k-points (inner product weighted like the energy) on
//   K_k -> A_vv K_k - K_k A_oo + C_v^T dH_k C_o,  dH = S o (e_A + e_B) / 2, e = gamma sum_k w_k dq(K_k).
// Then in FP64: C (1 - E/2 + 3/8 E^2 - 5/16 E^3), evaluations of q(C), H, H C_o and the residual A_vo, each followed
// by C (1 + K + K^2/2) with K from the FP32 Hessian of this basis; converged when every |A_vo| < P_EIG_TOL
// and the populations that A_vo implies to first order, q_out - q, are below scc_tol: two evaluations as a
// rule. Nothing of the FP32 part but the starting basis and the approximate Hessian enters the result.
// The stored bases Cs are only read; the path works in Cb (wk.Cd). Returns false (in every block of the cell)
// when the cell leaves the path's range, so that the general path starts from Cs. On success: Cb occupied
// columns first (each block its own k-points), sh.q, sh.dq and sh.shift (not for a finite-difference copy), and
// for the Gamma point Y = H C_o before the last change of the charges and in Mv (FP32) half of that change of A_oo.
// Measured (GB300, one step): 304 cells of 33 waters 263 -> 76 ms (with the image lists and the Ewald split),
// 24 cells of 8 waters on 3 x 3 x 3 232 -> 19.4 ms (with clusters of blocks); evaluations 11.8 -> 2.0. Bound: FP64
// products (7.5 n^3 multiply-adds a cell) and pair sums, the pipe about 65 % busy.
template <bool KG, class SH>
__device__ __noinline__ bool p_warm(const DftbArgs &a, const PbcDev &pl, SH &sh, const PbcMem &wk, const double *Cs,
                                    double *Cb, int n, int nocc, int nat, int rank, int blocks, int &evals) {
    const int j = threadIdx.x;
    const int m = KG ? 2 * n : n, mo = KG ? 2 * nocc : nocc, mv = m - mo, mm = m * m, mvo = mv * mo;
    const long long n2 = (KG ? 4LL : 1LL) * pl.nmax * pl.nmax;
    const int NKP = KG ? pl.nk : 1;
    double *H = wk.H, *Y = wk.Y;
    float *T0 = (float *)wk.Mo, *T1 = (float *)wk.Mv;   // m^2 floats of scratch each
    float *u = (float *)sh.red, *dqf = (float *)sh.qout, *ea = (float *)sh.qst, *eo = (float *)sh.invd;
    float *scr = (float *)sh.gred;
    double *H0 = wk.H0, *S = wk.S, *C = Cb;
    float *C32, *SC, *A32, *x, *r, *p, *hp;
    float wkp = 1.0f;
    auto set_k = [&](int kp) {
        if (KG) {
            H0 = wk.H0 + 2LL * kp * n2;
            S = H0 + n2;
            C = Cb + (long long)kp * mm;
            wkp = (float)pl.kpt[4 * kp + 3];
        }
        const PState32 f = p_state32<KG>(wk, kp, n2, mm);
        C32 = f.C;
        SC = f.SC;
        A32 = f.A;
        x = f.x;   // K, residual, search direction and its image: n_virt n_occ <= m^2 / 4 each
        r = x + mvo;
        p = r + mvo;
        hp = p + mvo;
    };
    int parity = 0;
    // sums over the blocks of the cell, in rank order; every block receives the same values
    auto exchange = [&](float *v, int cnt) {
        if (blocks > 1) {
            double *mine = wk.xch + ((long long)parity * blocks + rank) * (pl.amax + 8);
            for (int i = j; i < cnt; i += PT) mine[i] = v[i];
            cluster_barrier(blocks);
            for (int i = j; i < cnt; i += PT) {
                float s = 0.0f;
                for (int b = 0; b < blocks; ++b) s += (float)__ldcg(wk.xch + ((long long)parity * blocks + b) * (pl.amax + 8) + i);
                v[i] = s;
            }
            parity ^= 1;
        }
        __syncthreads();
    };
    auto total = [&](float s) -> float {   // over the block's threads, then over the blocks
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(CAVMD_FULL_MASK, s, o);
        __syncthreads();
        if ((j & 31) == 0) scr[1 + (j >> 5)] = s;
        __syncthreads();
        if (j == 0) {
            float t = 0.0f;
            for (int w = 0; w < PT / 32; ++w) t += scr[1 + w];
            scr[0] = t;
        }
        __syncthreads();
        exchange(scr, 1);
        return scr[0];
    };
    auto all = [&](bool ok) -> bool {
        const bool mine = blk_all(ok);
        if (blocks == 1) return mine;
        return total((j == 0 && !mine) ? 1.0f : 0.0f) == 0.0f;
    };
    auto atom_of = [&](int i) -> int { return sh.orb_atom[(KG && i >= n) ? i - n : i]; };
    // C32, SC and the half shifts eo give A32 = C^T H C (H C in T0 on the way)
    auto build_a = [&]() {
        fprod<7, 7, false, true>(sh, m, m, m,
                                 [&](int i, int k) { return fmaf(d2f_steer(S[(long long)k * m + i]), eo[i] + eo[k], d2f_steer(H0[(long long)k * m + i])); },
                                 [&](int k, int c) { return C32[c * m + k]; },
                                 [&](int i, int c, float v) { T0[c * m + i] = v; });
        fprod<7, 7, true, true>(sh, m, m, m, [&](int i, int k) { return C32[i * m + k]; },
                                [&](int k, int c) { return T0[c * m + k]; },
                                [&](int i, int c, float v) { A32[c * m + i] = v; });
    };
    auto build_sc = [&]() {
        fprod<7, 7, false, true>(sh, m, m, m, [&](int i, int k) { return d2f_steer(S[(long long)k * m + i]); },
                                 [&](int k, int c) { return C32[c * m + k]; },
                                 [&](int i, int c, float v) { SC[c * m + i] = v; });
    };
    // adds the k-point's part of the populations, 2 sum_o X(i, o) Z(i, o) per orbital, to u[0..n-1]
    auto add_orbitals = [&](int i, float s) {
        if (KG) u[i] = fmaf(0.5f * wkp, s, u[i]); else u[i] = s;
    };
    auto clear_u = [&]() {
        for (int i = j; i < n; i += PT) u[i] = 0.0f;
        __syncthreads();
    };
    auto to_atoms = [&]() {   // per-atom sums of u over the cell's blocks, into dqf
        __syncthreads();
        if (j < nat) {
            float s = 0.0f;
            for (int o = sh.atom_off[j]; o < sh.atom_off[j + 1]; ++o) s += u[o];
            dqf[j] = s;
        }
        __syncthreads();
        exchange(dqf, nat);
    };
    auto half_shifts = [&]() {
        if (j < nat) {
            float s = 0.0f;
            for (int k = 0; k < nat; ++k) s = fmaf(wk.g32[k * nat + j], dqf[k], s);
            ea[j] = 0.5f * s;
        }
        __syncthreads();
        for (int i = j; i < m; i += PT) eo[i] = ea[atom_of(i)];
        __syncthreads();
    };
    // populations moved by K = kv(kp) to first order (into dqf): X = C_v K, 2 sum_o [X SC_o + C_o (S X)]
    auto charges = [&](int which) {   // 0: x, 1: p
        clear_u();
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            const float *kv = which ? p : x;
            fprod<5, 5, false, true>(sh, m, mo, mv, [&](int i, int k) { return C32[(mo + k) * m + i]; },
                                     [&](int k, int c) { return kv[c * mv + k]; },
                                     [&](int i, int c, float v) { T0[c * m + i] = v * SC[c * m + i]; });
            fprod<5, 5, false, true>(sh, m, mo, mv, [&](int i, int k) { return SC[(mo + k) * m + i]; },
                                     [&](int k, int c) { return kv[c * mv + k]; },
                                     [&](int i, int c, float v) { T0[c * m + i] = fmaf(v, C32[c * m + i], T0[c * m + i]); });
            for (int i = j; i < n; i += PT) {
                float s = 0.0f;
                for (int o = 0; o < mo; ++o) s += T0[o * m + i];
                if (KG)
                    for (int o = 0; o < mo; ++o) s += T0[o * m + i + n];
                add_orbitals(i, 2.0f * s);
            }
            __syncthreads();
        }
        to_atoms();
    };
    auto diag_of = [&](int e) -> float { return A32[(mo + e % mv) * (m + 1)] - A32[(e / mv) * (m + 1)]; };
    // Hessian K = r (K in x, r destroyed) to a relative residual rel; false when it is not positive
    int steps = 0;   // conjugate-gradient steps of the last solve
    float *moved = (float *)sh.hq[0];   // the change of the atoms' charges under K
    auto newton = [&](float rel) -> bool {
        float rz = 0.0f;
        steps = 0;
        if (j < nat) moved[j] = 0.0f;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            for (int e = j; e < mvo; e += PT) {
                const float z = r[e] / diag_of(e);
                x[e] = 0.0f;
                p[e] = z;
                rz = fmaf(wkp * r[e], z, rz);
            }
        }
        rz = total(rz);
        const float stop = rel * rel * rz;
        if (!(rz < 1e30f) || !(rz >= 0.0f)) return false;
        for (int it = 0; it < PW_CG_ITERS && rz > stop; ++it) {
            ++steps;
            charges(1);
            half_shifts();
            float ph = 0.0f;
            for (int kp = rank; kp < NKP; kp += blocks) {
                set_k(kp);
                // A_vv p - p A_oo + C_v^T (e S C_o) + (S C_v)^T (e C_o), one product over the joined index
                fprod<5, 5, true, true>(
                    sh, mv, mo, mv + mo + 2 * m,
                    [&](int v, int k) -> float {
                        if (k < mv) return A32[(mo + v) * m + mo + k];
                        k -= mv;
                        if (k < mo) return -p[k * mv + v];
                        k -= mo;
                        return k < m ? C32[(mo + v) * m + k] : SC[(mo + v) * m + k - m];
                    },
                    [&](int k, int o) -> float {
                        if (k < mv) return p[o * mv + k];
                        k -= mv;
                        if (k < mo) return A32[o * m + k];
                        k -= mo;
                        return k < m ? eo[k] * SC[o * m + k] : eo[k - m] * C32[o * m + k - m];
                    },
                    [&](int v, int o, float t) { hp[o * mv + v] = t; });
                for (int e = j; e < mvo; e += PT) ph = fmaf(wkp * p[e], hp[e], ph);
            }
            ph = total(ph);
            if (!(ph > 0.0f)) return false;
            const float al = rz / ph;
            if (j < nat) moved[j] = fmaf(al, dqf[j], moved[j]);
            float rn = 0.0f;
            for (int kp = rank; kp < NKP; kp += blocks) {
                set_k(kp);
                for (int e = j; e < mvo; e += PT) {
                    x[e] = fmaf(al, p[e], x[e]);
                    const float q = fmaf(-al, hp[e], r[e]);
                    r[e] = q;
                    rn = fmaf(wkp * q, q / diag_of(e), rn);
                }
            }
            rn = total(rn);
            if (!(rn < 1e30f) || !(rn >= 0.0f)) return false;
            const float be = rn / rz;
            rz = rn;
            for (int kp = rank; kp < NKP; kp += blocks) {
                set_k(kp);
                for (int e = j; e < mvo; e += PT) p[e] = fmaf(be, p[e], r[e] / diag_of(e));
            }
            __syncthreads();
        }
        return true;
    };
    // T1: [C_o + C_v K / 2 | C_v - C_o K^T / 2] (with_c), or the second parts alone
    auto second = [&](bool with_c) {
        fprod<5, 5, false, true>(sh, m, mo, mv, [&](int i, int k) { return C32[(mo + k) * m + i]; },
                                 [&](int k, int c) { return x[c * mv + k]; }, [&](int i, int c, float v) {
                                     T1[c * m + i] = fmaf(0.5f, v, with_c ? C32[c * m + i] : 0.0f);
                                 });
        fprod<5, 5, false, false>(sh, m, mv, mo, [&](int i, int k) { return C32[k * m + i]; },
                                  [&](int k, int c) { return x[k * mv + c]; }, [&](int i, int c, float v) {
                                      T1[(mo + c) * m + i] = fmaf(-0.5f, v, with_c ? C32[(mo + c) * m + i] : 0.0f);
                                  });
    };

    // ---------------------------------------------------------------- gamma in FP32
    // The vectors are sorted by length: from n_g32 on their weights are below FP32 rounding of gamma. Slices of
    // 32 vectors are added in FP64 (in pbuf): a single FP32 sum over them all was 5e-7 off, enough for the
    // Hessian to ask for a third evaluation.
    for (int e = j; e < nat * nat; e += PT) wk.pbuf[e] = wk.gam[(e % nat) * pl.amax + e / nat];
    __syncthreads();
    for (int g0 = 0; g0 < pl.n_g32; g0 += 32) {
        const int k0 = 2 * g0;
        fprod<7, 7, false, false>(sh, nat, nat, 2 * min(32, pl.n_g32 - g0),
                                  [&](int A, int k) { return d2f_steer(wk.csg[2LL * ((long long)((k0 + k) >> 1) * nat + A) + (k & 1)]); },
                                  [&](int k, int B) {
                                      return d2f_steer(pl.gw[4 * ((k0 + k) >> 1) + 3]) *
                                             d2f_steer(wk.csg[2LL * ((long long)((k0 + k) >> 1) * nat + B) + (k & 1)]);
                                  },
                                  [&](int A, int B, float v) { wk.pbuf[B * nat + A] += f2d_steer(v); });
    }
    for (int e = j; e < nat * nat; e += PT) wk.g32[e] = __double2float_rn(wk.pbuf[e]);
    __syncthreads();

    // ---------------------------------------------------------------- FP32 start
    float big = 0.0f;
    for (int kp = rank; kp < NKP; kp += blocks) {
        set_k(kp);
        const double *from = Cs + (KG ? (long long)kp * mm : 0);
        for (int e = j; e < mm; e += PT) C32[e] = d2f_steer(from[e]);
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {
            build_sc();
            fprod<7, 7, true, true>(sh, m, m, m, [&](int i, int k) { return C32[i * m + k]; },
                                    [&](int k, int c) { return SC[c * m + k]; }, [&](int i, int c, float v) {
                                        const float e = v - (i == c ? 1.0f : 0.0f);
                                        big = max_nan(big, fabsf(e));
                                        if (pass == 0) T0[c * m + i] = e;
                                        else T1[c * m + i] = fmaf(-0.5f, e, i == c ? 1.0f : 0.0f);
                                    });
            if (pass == 0)
                fprod<7, 7, false, true>(sh, m, m, m, [&](int i, int k) { return T0[k * m + i]; },
                                         [&](int k, int c) { return T0[c * m + k]; }, [&](int i, int c, float v) {
                                             T1[c * m + i] = fmaf(0.375f, v, fmaf(-0.5f, T0[c * m + i], i == c ? 1.0f : 0.0f));
                                         });
            fprod<7, 7, false, true>(sh, m, m, m, [&](int i, int k) { return C32[k * m + i]; },
                                     [&](int k, int c) { return T1[c * m + k]; },
                                     [&](int i, int c, float v) { T0[c * m + i] = v; });
            for (int e = j; e < mm; e += PT) C32[e] = T0[e];
            __syncthreads();
        }
    }
    if (!all(big < 0.2f)) return false;
    bool done = false;
    int first_steps = 0;
    for (int it = 0; it < PW_FP32_ITERS && !done; ++it) {
        clear_u();
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            build_sc();
            for (int i = j; i < n; i += PT) {
                float s = 0.0f;
                for (int o = 0; o < mo; ++o) s = fmaf(C32[o * m + i], SC[o * m + i], s);
                if (KG)
                    for (int o = 0; o < mo; ++o) s = fmaf(C32[o * m + i + n], SC[o * m + i + n], s);
                add_orbitals(i, 2.0f * s);
            }
            __syncthreads();
        }
        to_atoms();
        if (j < nat) dqf[j] -= d2f_steer(sh.zv[j]);
        __syncthreads();
        half_shifts();
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            build_a();
            for (int e = j; e < mvo; e += PT) {
                const int v = e % mv, o = e / mv;
                r[e] = -0.5f * (A32[o * m + mo + v] + A32[(mo + v) * m + o]);
            }
            __syncthreads();
        }
        if (!newton(it < 2 ? 3e-3f : 1e-2f)) return false;
        if (it == 0) first_steps = steps;
        float kmax = 0.0f;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            for (int e = j; e < mvo; e += PT) kmax = max_nan(kmax, fabsf(x[e]));
            second(true);
            fprod<5, 5, false, true>(sh, m, mo, mv, [&](int i, int k) { return T1[(mo + k) * m + i]; },
                                     [&](int k, int c) { return x[c * mv + k]; },
                                     [&](int i, int c, float v) { C32[c * m + i] += v; });
            fprod<5, 5, false, false>(sh, m, mv, mo, [&](int i, int k) { return T1[k * m + i]; },
                                      [&](int k, int c) { return x[k * mv + c]; },
                                      [&](int i, int c, float v) { C32[(mo + c) * m + i] -= v; });
        }
        if (!all(kmax < PW_ROT_MAX)) return false;
        done = all(kmax < PW_FP32_KTOL);
    }
    if (!done) return false;
    // The rotations leave the occupied and the virtual blocks of C^T H C alone, and their off-diagonal part
    // grows with every step until the diagonal preconditioner is a poor one (100 cells of 17 waters: 11 ms a
    // step at first, 19 after 100 steps). When the solve shows it, one Jacobi sweep inside each block (FP32:
    // any orthogonal mixing inside a block leaves the result alone, and C is made orthonormal below).
    if (first_steps >= PW_CG_SLOW) {
        float *cs = (float *)sh.cs;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            for (int b = 0; b < 2; ++b) {
                const int off = b ? mo : 0, mb = b ? mv : mo, me = mb + (mb & 1), half = me / 2;
                for (int e = j; e < mb * mb; e += PT) {
                    const int c = e / mb, i = e - c * mb;
                    T0[e] = A32[(off + c) * m + off + i];
                    T1[e] = i == c ? 1.0f : 0.0f;
                }
                __syncthreads();
                for (int rd = 0; rd < me - 1; ++rd) {
                    if (j < half) {
                        int pa, pb;
                        p_pair(j, rd, me, pa, pb);
                        float t = 0.0f;
                        if (pb < mb) {
                            const float d = T0[pb * mb + pb] - T0[pa * mb + pa], o = 2.0f * T0[pb * mb + pa];
                            if (o != 0.0f) t = o / (d + copysignf(sqrtf(fmaf(d, d, o * o)), d));
                        }
                        const float c = rsqrtf(fmaf(t, t, 1.0f));
                        sh.pp[j] = pa;
                        sh.pq[j] = pb;
                        cs[2 * j] = c;
                        cs[2 * j + 1] = t * c;
                    }
                    __syncthreads();
                    for (int e = j; e < half * 2 * mb; e += PT) {   // columns of the block and of the rotation
                        const int k = e / (2 * mb), rr = e - k * 2 * mb, pa = sh.pp[k], pb = sh.pq[k];
                        if (pb >= mb) continue;
                        float *base = rr < mb ? T0 : T1;
                        const int i = rr < mb ? rr : rr - mb;
                        const float xp = base[pa * mb + i], xq = base[pb * mb + i], c = cs[2 * k], sn = cs[2 * k + 1];
                        base[pa * mb + i] = fmaf(c, xp, -sn * xq);
                        base[pb * mb + i] = fmaf(sn, xp, c * xq);
                    }
                    __syncthreads();
                    for (int e = j; e < half * mb; e += PT) {   // rows of the block
                        const int k = e / mb, cc = e - k * mb, pa = sh.pp[k], pb = sh.pq[k];
                        if (pb >= mb) continue;
                        const float xp = T0[cc * mb + pa], xq = T0[cc * mb + pb], c = cs[2 * k], sn = cs[2 * k + 1];
                        T0[cc * mb + pa] = fmaf(c, xp, -sn * xq);
                        T0[cc * mb + pb] = fmaf(sn, xp, c * xq);
                    }
                    __syncthreads();
                }
                fprod<5, 5, false, true>(sh, m, mb, mb, [&](int i, int k) { return C32[(off + k) * m + i]; },
                                         [&](int k, int c) { return T1[c * mb + k]; },
                                         [&](int i, int c, float v) { SC[c * m + i] = v; });
                for (int e = j; e < m * mb; e += PT) C32[off * m + e] = SC[e];
                __syncthreads();
            }
        }
    }

    // ---------------------------------------------------------------- FP64 evaluations
    for (int kp = rank; kp < NKP; kp += blocks) {
        set_k(kp);
        for (int e = j; e < mm; e += PT) C[e] = f2d_steer(C32[e]);
    }
    __syncthreads();
    bool rough = true;   // the bases are orthonormal to FP32 only (or after a large rotation)
    const int most = min(a.max_iter, PW_EVALS);
    for (int it = 1; it <= most; ++it) {
        if (rough) {
            float e2 = 0.0f;
            for (int kp = rank; kp < NKP; kp += blocks) {
                set_k(kp);
                bool again = true;
                for (int pass = 0; again; ++pass) {
                    float ek = 0.0f;   // this thread's share of the k-point's sum
                    pprod<false, false, true>(sh, m, m, m, [&](int i, int k) { return S[(long long)k * m + i]; },
                                              [&](int i, int c) { return C[(long long)c * m + i]; },
                                              [&](int i, int c, double v) { Y[(long long)c * m + i] = v; });
                    pprod<true, true, true>(sh, m, m, m, [&](int i, int k) { return C[(long long)i * m + k]; },
                                            [&](int k, int c) { return Y[(long long)c * m + k]; },
                                            [&](int i, int c, double v) {
                                                if (i == c) v -= 1.0;
                                                H[(long long)c * m + i] = v;
                                                H[(long long)i * m + c] = v;
                                                const float f = d2f_steer(v);
                                                T0[c * m + i] = f;
                                                T0[i * m + c] = f;
                                                ek = fmaf(i == c ? 1.0f : 2.0f, f * f, ek);
                                            });
                    // (a bound on every share bounds the sum)
                    again = pass < 2 && !blk_all(ek * PT < PW_ORTH_ONCE * PW_ORTH_ONCE);
                    if (!again) e2 += ek;
                    // 1 - E/2 + 3/8 E^2 - 5/16 E^3. The norm of E is 2e-6 (36 waters: 7e-6, 14 k-points: 2e-5) as a
                    // rule, more after a large rotation; up to PW_ORTH_ONCE FP32 rounds the last two terms by 6e-15,
                    // and the quartic one is 2e-14.
                    fprod<7, 7, false, true>(sh, m, m, m, [&](int i, int k) { return T0[k * m + i]; },
                                             [&](int k, int c) { return T0[c * m + k]; }, [&](int i, int c, float v) {
                                                 double &h = H[(long long)c * m + i];
                                                 h = fma(-0.5, h, (i == c ? 1.0 : 0.0) + f2d_steer(0.375f * v));
                                                 T1[c * m + i] = v;
                                             });
                    if (!blk_all(ek * PT < PW_ORTH_CUBE * PW_ORTH_CUBE))
                        fprod<7, 7, false, true>(sh, m, m, m, [&](int i, int k) { return T0[k * m + i]; },
                                                 [&](int k, int c) { return T1[c * m + k]; },
                                                 [&](int i, int c, float v) { H[(long long)c * m + i] -= f2d_steer(0.3125f * v); });
                    pprod<false, false, true>(sh, m, m, m, [&](int i, int k) { return C[(long long)k * m + i]; },
                                              [&](int k, int c) { return H[(long long)c * m + k]; },
                                              [&](int i, int c, double v) { Y[(long long)c * m + i] = v; });
                    for (int e = j; e < mm; e += PT) C[e] = Y[e];
                    __syncthreads();
                }
            }
            if (!(total(e2) < PW_ORTH_MAX * PW_ORTH_MAX)) return false;
        }
        // populations: 2 sum_o C(i, o) (S C)(i, o), weighted over the k-points
        for (int i = j; i < n; i += PT) sh.qk[i] = 0.0;
        __syncthreads();
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            pprod<false, false, true>(sh, m, mo, m, [&](int i, int k) { return S[(long long)k * m + i]; },
                                      [&](int k, int c) { return C[(long long)c * m + k]; },
                                      [&](int i, int c, double v) { Y[(long long)c * m + i] = v; });
            for (int i = j; i < n; i += PT) {
                double s = 0.0;
                for (int o = 0; o < mo; ++o) s = fma(C[(long long)o * m + i], Y[(long long)o * m + i], s);
                if (KG) {
                    for (int o = 0; o < mo; ++o) s = fma(C[(long long)o * m + i + n], Y[(long long)o * m + i + n], s);
                    sh.qk[i] = fma(pl.kpt[4 * kp + 3], s, sh.qk[i]);   // 0.5 w for the real form, 2 for the spin
                } else {
                    sh.qk[i] = 2.0 * s;
                }
            }
            __syncthreads();
        }
        if (j < nat) {
            double s = 0.0;
            for (int o = sh.atom_off[j]; o < sh.atom_off[j + 1]; ++o) s += sh.qk[o];
            sh.q[j] = s;
        }
        __syncthreads();
        if (blocks > 1) {
            double *mine = wk.xch + ((long long)parity * blocks + rank) * (pl.amax + 8);
            if (j < nat) mine[j] = sh.q[j];
            cluster_barrier(blocks);
            if (j < nat) {
                double s = 0.0;
                for (int b = 0; b < blocks; ++b) s += __ldcg(wk.xch + ((long long)parity * blocks + b) * (pl.amax + 8) + j);
                sh.q[j] = s;
            }
            parity ^= 1;
            __syncthreads();
        }
        if (j < nat) sh.dq[j] = sh.q[j] - sh.zv[j];
        __syncthreads();
        p_shifts(sh, pl, wk, nat);
        for (int i = j; i < m; i += PT) eo[i] = 0.5f * d2f_steer(sh.shift[atom_of(i)]);
        __syncthreads();
        bool small = true, finite = true;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            for (int e = j; e < mm; e += PT) {
                const int c = e / m, i = e - c * m;
                H[e] = fma(0.5 * S[e], sh.shift[atom_of(i)] + sh.shift[atom_of(c)], H0[e]);
            }
            __syncthreads();
            pprod<false, false, true>(sh, m, mo, m, [&](int i, int k) { return H[(long long)k * m + i]; },
                                      [&](int k, int c) { return C[(long long)c * m + k]; },
                                      [&](int i, int c, double v) { Y[(long long)c * m + i] = v; });
            pprod<false, true, true>(sh, mv, mo, m, [&](int v, int k) { return C[(long long)(mo + v) * m + k]; },
                                     [&](int k, int o) { return Y[(long long)o * m + k]; }, [&](int v, int o, double t) {
                                         if (!abs_lt(t, P_EIG_TOL)) small = false;
                                         if (!abs_lt(t, 1.0)) finite = false;
                                         r[o * mv + v] = -d2f_steer(t);
                                     });
            // the FP32 Hessian of this basis
            for (int e = j; e < mm; e += PT) C32[e] = d2f_steer(C[e]);
            __syncthreads();
            build_sc();
            build_a();
        }
        if (!all(finite)) return false;
        bool conv = false;
        float hi = -1e30f, lo = 1e30f;
        if (all(small)) {   // q_out - q to first order: K0 = r / (A_vv - A_oo)
            for (int kp = rank; kp < NKP; kp += blocks) {
                set_k(kp);
                for (int e = j; e < mvo; e += PT) x[e] = r[e] / diag_of(e);
                for (int i = 0; i < mo; ++i) hi = fmaxf(hi, A32[i * (m + 1)]);
                for (int i = mo; i < m; ++i) lo = fminf(lo, A32[i * (m + 1)]);
            }
            __syncthreads();
            charges(0);
            conv = blk_all(j >= nat || fabsf(dqf[j]) < (float)a.scc_tol);   // the same charges in every block
        }
        if (conv) {
            // aufbau and gap over all k-points: tau - A_oo and A_vv - tau - PW_GAP positive definite for a tau
            // between the highest occupied and the lowest empty diagonal (pivots of L D L^T)
            if (blocks > 1) {
                double *mine = wk.xch + ((long long)parity * blocks + rank) * (pl.amax + 8);
                if (j == 0) {
                    mine[0] = hi;
                    mine[1] = lo;
                }
                cluster_barrier(blocks);
                for (int b = 0; b < blocks; ++b) {
                    hi = fmaxf(hi, (float)__ldcg(wk.xch + ((long long)parity * blocks + b) * (pl.amax + 8)));
                    lo = fminf(lo, (float)__ldcg(wk.xch + ((long long)parity * blocks + b) * (pl.amax + 8) + 1));
                }
                parity ^= 1;
            }
            // the diagonals bound tau (mixing inside the blocks moves the levels beyond them): bisection
            for (int t = 0;; ++t) {
                const float tau = 0.5f * (hi + lo);
                bool occ = true, emp = true;
                for (int kp = rank; kp < NKP; kp += blocks) {
                    set_k(kp);
                    // a row bound first: diagonally dominant rows are enough
                    bool dom = true;
                    for (int i = j; i < m; i += PT) {
                        float off = 0.0f;
                        const int b0 = i < mo ? 0 : mo, b1 = i < mo ? mo : m;
                        for (int c = b0; c < b1; ++c)
                            if (c != i) off += fabsf(A32[c * m + i]);
                        const float d = i < mo ? tau - A32[i * (m + 1)] : A32[i * (m + 1)] - tau - PW_GAP;
                        dom = dom && d > off;
                    }
                    if (blk_all(dom)) continue;
                    for (int e = j; e < mm; e += PT) {
                        const int c = e / m, i = e - c * m;
                        T0[e] = (i < mo && c < mo) ? (i == c ? tau : 0.0f) - A32[e] : A32[e] - (i == c ? tau + PW_GAP : 0.0f);
                    }
                    __syncthreads();
                    for (int k = 0; k < m; ++k) {
                        const float d = T0[k * (m + 1)];
                        if (k < mo) occ = occ && d > 0.0f; else emp = emp && d > 0.0f;
                        const int end = k < mo ? mo : m;
                        const float id = 1.0f / d;
                        for (int c = k + 1 + (j >> 5); c < end; c += PT / 32) {   // a warp per column of the trailing block
                            const float f = T0[k * m + c] * id;
                            for (int i = c + (j & 31); i < end; i += 32) T0[c * m + i] = fmaf(-f, T0[k * m + i], T0[c * m + i]);
                        }
                        __syncthreads();
                    }
                }
                occ = all(occ);
                emp = all(emp);
                if (occ && emp) break;
                if (t == PW_BISECT || occ == emp) return false;
                if (occ) lo = tau; else hi = tau;
            }
        }
        // (a relative residual of 1e-6 left one cell in ten above scc_tol)
        if ((it == most && !conv) || !newton(conv ? PW_LAST_TOL : 1e-7f)) return false;
        if (conv) {
            p_settle<KG>(a, pl, sh, wk, Cb, moved, n, nocc, nat, rank, blocks);
            evals = it;
            return true;
        }
        float k2 = 0.0f;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            for (int e = j; e < mvo; e += PT) k2 = fmaf(x[e], x[e], k2);
        }
        k2 = total(k2);
        if (!(k2 < PW_ROT64_MAX * PW_ROT64_MAX)) return false;
        rough = k2 > PW_ROT64_ONCE * PW_ROT64_ONCE;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            // C (1 + K + K^2/2), as C_o + (C_v - (C_o K^T)/2) K and C_v - (C_o + (C_v K)/2) K^T; the half terms in FP32
            second(false);
            for (int e = j; e < mm; e += PT) H[e] = C[e] + f2d_steer(T1[e]);
            __syncthreads();
            pprod<false, false, true>(sh, m, mo, mv, [&](int i, int k) { return H[(long long)(mo + k) * m + i]; },
                                      [&](int k, int c) { return f2d_steer(x[c * mv + k]); },
                                      [&](int i, int c, double v) { C[(long long)c * m + i] += v; });
            pprod<false, false, false>(sh, m, mv, mo, [&](int i, int k) { return H[(long long)k * m + i]; },
                                       [&](int k, int c) { return f2d_steer(x[k * mv + c]); },
                                       [&](int i, int c, double v) { C[(long long)(mo + c) * m + i] -= v; });
        }
    }
    return false;
}

// Calls f(im) for the lattice images (of the first n_img) whose distance from the wrapped separation dw may be
// below sqrt(r2max), in increasing order. Each thread first marks its own images in FP32 (with a margin;
// f applies the exact test) and then visits those: the threads of a warp reach different images, and a plain
// loop would run f's long body for every image that any of them reaches.
template <class F>
__device__ __forceinline__ void pbc_images(const PbcDev &pl, const double *dw, int n_img, double r2max, F f) {
    const float x = d2f_steer(dw[0]), y = d2f_steer(dw[1]), z = d2f_steer(dw[2]);
    const float lim = fmaf(d2f_steer(r2max), 1.0001f, 1e-2f);
    for (int base = 0; base < n_img; base += 32) {
        unsigned mask = 0u;
        const int end = min(32, n_img - base);
        for (int b = 0; b < end; ++b) {
            const double *t = pl.img + 3 * (base + b);
            const float u = x + d2f_steer(t[0]), v = y + d2f_steer(t[1]), w = z + d2f_steer(t[2]);
            if (fmaf(u, u, fmaf(v, v, w * w)) < lim) mask |= 1u << b;
        }
        while (mask) {
            const int b = __ffs(mask) - 1;
            mask &= mask - 1u;
            f(base + b);
        }
    }
}

// Pair A <= B number t of a cell, by kind: both atoms with p orbitals, one of them, neither, then each atom
// with its own images. The threads of a warp then evaluate the same radial functions.
template <class SH>
__device__ __forceinline__ void pbc_pair(const SH &sh, int nat, int t, int &A, int &B) {
    const int nb = sh.fl[5], ns = nat - nb, p_bb = nb * (nb - 1) / 2, p_bs = p_bb + nb * ns, p_all = nat * (nat - 1) / 2;
    int x, y;
    if (t >= p_all) {
        x = y = t - p_all;
    } else if (t >= p_bb && t < p_bs) {
        const int u = t - p_bb;
        x = sh.lst[u / ns];
        y = sh.lst[nb + u % ns];
    } else {
        const int u = t < p_bb ? t : t - p_bs, o = t < p_bb ? 0 : nb;
        int k = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)u)) * 0.5f);
        while (k * (k - 1) / 2 > u) --k;
        while ((k + 1) * k / 2 <= u) ++k;
        x = sh.lst[o + u - k * (k - 1) / 2];
        y = sh.lst[o + k];
    }
    A = min(x, y);
    B = max(x, y);
}

// One cell, or (disp_k >= 0) one finite-difference copy of it: atom disp_k / 3 (central: disp_k / 6)
// moved along x, y or z by +h (central: +h and -h in turn), warm started from the cell's converged
// basis in a private copy, and only its dipole written (M_disp, the layout of the water kernels).
//
// KG: the cell sampled on a k-grid (the paper's Gamma point of a folded supercell). Each k-point of
// the irreducible list (k and -k give complex-conjugate problems) is a complex Hermitian problem
// H(k) c = e S(k) c, H(k)_{mu nu} = sum_T exp(i 2 pi f_k . n_T) h_{mu nu}(r_B + T - r_A), solved in its
// real form of twice the size, [[Re, -Im], [Im, Re]] (every level appears twice, so twice the
// occupied count is occupied): the same products, factorisations, sweeps and rotations as the
// Gamma point. The SCC iteration runs every k-point's update in turn and joins the populations,
// sum_k w_k Re (P(k) S(k)*)_{mu mu}, before the mixing; the band energy is sum_k w_k Re Tr P(k) H0(k)*
// and the forces use the real-space densities rho(T) = sum_k w_k Re[P(k)_{nu mu} exp(i 2 pi f_k . n_T)]
// (and the same for the energy-weighted density) image by image.
// `blocks` blocks (a cluster; one outside the k-grid) share the cell: each takes the k-points rank,
// rank + blocks, ... A cluster only takes the warm path: a cell that leaves it puts its item on the list pl.late
// and returns.
template <bool KG, class SH>
__device__ void p_cell(const DevSK &sk, const DftbArgs &a, const PbcDev &pl, SH &sh, const PbcMem &wk, int cell,
                       int disp_k, int rank, int blocks, int item) {
    const int j = threadIdx.x;
    const int a0 = a.cell_offset[cell];
    const int nat = a.cell_offset[cell + 1] - a0;
    const long long n2max = (KG ? 4LL : 1LL) * pl.nmax * pl.nmax;   // one problem matrix
    const bool disp = disp_k >= 0;
    const int NKP = KG ? pl.nk : 1;
    double *H0 = wk.H0, *S = wk.S;
    double *H = wk.H, *Y = wk.Y, *P = wk.P, *Xg = wk.Xg, *Mo = wk.Mo, *Mv = wk.Mv;
    double *gam = wk.gam, *csg = wk.csg, *sgf = wk.sgf, *pbuf = wk.pbuf;   // pbuf: [atom * nat + atom] gradient (3) + energy
    double *const C0 = a.Cwarm + a.Cwarm_off[cell];
    double *C = C0;

    if (j < nat) {
        sh.spec[j] = a.species[a0 + j];
        for (int k = 0; k < 3; ++k) sh.pos[j][k] = a.r[3 * (a0 + j) + k];
        if (disp) {
            const int kk = a.fd_central ? disp_k >> 1 : disp_k;
            const double sg = (a.fd_central && (disp_k & 1)) ? -1.0 : 1.0;
            if (j == kk / 3) sh.pos[j][kk % 3] += sg * a.fd_h;
        }
    }
    __syncthreads();
    if (j == 0) {
        int o = 0;
        double nel = 0.0;
        for (int at = 0; at < nat; ++at) {
            sh.atom_off[at] = o;
            const int no = sk.norb[sh.spec[at]];
            for (int k = 0; k < no; ++k) sh.orb_atom[o + k] = at;
            o += no;
            sh.zv[at] = sk.zval[sh.spec[at]];
            nel += sh.zv[at];
        }
        sh.atom_off[nat] = o;
        sh.fl[0] = 0;
        sh.fl[1] = o;
        sh.fl[2] = 0;
        sh.fl[3] = (int)(nel * 0.5 + 0.25);
    }
    if (j < nat) {
        const bool big = sk.norb[sh.spec[j]] == 4;
        int same = 0, nbig = 0;
        for (int x = 0; x < nat; ++x) {
            const bool bx = sk.norb[sh.spec[x]] == 4;
            nbig += bx;
            same += x < j && bx == big;
        }
        sh.lst[big ? same : nbig + same] = j;
        if (j == 0) sh.fl[5] = nbig;
    }
    __syncthreads();
    const int n = sh.fl[1], nocc = sh.fl[3];
    const int nv = n - nocc, nn = n * n;
    // the problem: orbitals (Gamma), or the real form of a k-point problem (KG)
    const int m = KG ? 2 * n : n, mo = KG ? 2 * nocc : nocc, mv = m - mo, mm = m * m;
    double *Cb = C0;   // the bases of the k-points, mm apart
    // point the problem's matrices at k-point kp
    auto set_k = [&](int kp) {
        if (KG) {
            H0 = wk.H0 + 2LL * kp * n2max;
            S = H0 + n2max;
            C = Cb + (long long)kp * mm;
        }
    };

    // ---------------------------------------------------------------- H0, S, real-space gamma
    if constexpr (KG) {
        // every k-point: H0(k), S(k) in real form; gamma (k-independent) with the first k-point
        const double rc2 = sk.r_cut * sk.r_cut;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            const bool first = kp == 0;
            const double fk[3] = {pl.kpt[4 * kp], pl.kpt[4 * kp + 1], pl.kpt[4 * kp + 2]};
            for (int e = j; e < mm; e += PT) {
                const int c = e / m, i = e - c * m;
                double h = 0.0, s = 0.0;
                if (i == c) {
                    const int io = i < n ? i : i - n;
                    const int at = sh.orb_atom[io], el = sh.spec[at];
                    h = (io == sh.atom_off[at]) ? sk.onsite[el][0] : sk.onsite[el][1];
                    s = 1.0;
                }
                H0[e] = h;
                S[e] = s;
            }
            __syncthreads();
            for (int t = j; t < nat * (nat + 1) / 2; t += PT) {   // pairs A <= B, by kind
                int A, B;
                pbc_pair(sh, nat, t, A, B);
                const int eA = sh.spec[A], eB = sh.spec[B];
                const int oA = sh.atom_off[A], oB = sh.atom_off[B];
                const int na = sk.norb[eA], nb = sk.norb[eB];
                double d[3], f[3], dw[3];
                for (int k = 0; k < 3; ++k) d[k] = sh.pos[B][k] - sh.pos[A][k];
                for (int k = 0; k < 3; ++k) f[k] = rint(fma(d[0], pl.inv[k], fma(d[1], pl.inv[3 + k], d[2] * pl.inv[6 + k])));
                for (int k = 0; k < 3; ++k) dw[k] = d[k] - fma(f[0], pl.lat[k], fma(f[1], pl.lat[3 + k], f[2] * pl.lat[6 + k]));
                double hr[16], hi[16], sr[16], si[16];
                for (int u = 0; u < 16; ++u) { hr[u] = 0.0; hi[u] = 0.0; sr[u] = 0.0; si[u] = 0.0; }
                double g_re = 0.0, g_sr = 0.0;
                const double c2 = sk.gamma_c2[eA][eB];
                if (first) {
                    pbc_images(pl, dw, pl.n_img, pl.r_real2, [&](int im) {   // real-space Ewald sum
                        const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                        const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                        if (!(r2 < pl.r_real2) || r2 == 0.0) return;
                        const double ir = rsqrt_nr(r2);
                        g_re = fma(erfc(pl.alpha * (r2 * ir)), ir, g_re);
                    });
                }
                pbc_images(pl, dw, pl.n_img_sk, rc2, [&](int im) {   // images within r_cut
                    const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                    const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                    if (!(r2 < rc2) || r2 == 0.0) return;
                    const double ir = rsqrt_nr(r2);
                    const double r = r2 * ir;
                    const double e[3] = {x0 * ir, x1 * ir, x2 * ir};
                    // the image's translation n_T = (its lattice coordinates) - f, and its phase
                    double ph = 0.0;
                    for (int k = 0; k < 3; ++k) {
                        const double nk_ = rint(fma(pl.img[3 * im], pl.inv[k], fma(pl.img[3 * im + 1], pl.inv[3 + k],
                                                                                     pl.img[3 * im + 2] * pl.inv[6 + k]))) - f[k];
                        ph = fma(fk[k], nk_, ph);
                    }
                    double sn, cs;
                    sincospi(2.0 * ph, &sn, &cs);
                    for (int tb = 0; tb < 2; ++tb) {
                        const double(*tab)[CAVMD_MAX_ELEM][4][4] = tb == 0 ? sk.h0 : sk.s;
                        double blk[16];
                        for (int u = 0; u < 16; ++u) blk[u] = 0.0;
                        double v, dv;
                        radial_p(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                        blk[0] = v;
                        if (nb == 4) {
                            radial_p(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                            for (int i = 0; i < 3; ++i) blk[1 + i] = e[i] * v;
                        }
                        if (na == 4) {
                            radial_p(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                            for (int i = 0; i < 3; ++i) blk[4 * (1 + i)] = -e[i] * v;
                        }
                        if (na == 4 && nb == 4) {
                            double vs, vp;
                            radial_p(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dv);
                            radial_p(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dv);
                            const double dl = vs - vp;
                            for (int i = 0; i < 3; ++i)
                                for (int k = 0; k < 3; ++k) blk[4 * (1 + i) + 1 + k] = fma(e[i] * e[k], dl, (i == k) ? vp : 0.0);
                        }
                        double *re = tb == 0 ? hr : sr, *imv = tb == 0 ? hi : si;
                        for (int u = 0; u < 16; ++u) {
                            re[u] = fma(cs, blk[u], re[u]);
                            imv[u] = fma(sn, blk[u], imv[u]);
                        }
                    }
                    if (first) {
                        double fc, dfc;
                        cutoff_fn(r, sk, fc, dfc);
                        g_sr = fma(rsqrt_nr(r2 + c2) - ir, fc, g_sr);
                    }
                });
                // complex block z (mu of A, nu of B) at row oA + mu, column oB + nu of [[Re, -Im], [Im, Re]],
                // and its Hermitian transpose; a block of an atom with its own images is Hermitian,
                // written as the mean of z and the conjugate transpose
                for (int mu = 0; mu < na; ++mu)
                    for (int nu = 0; nu < nb; ++nu) {
                        const int u = 4 * mu + nu, ut = 4 * nu + mu;
                        for (int tb = 0; tb < 2; ++tb) {
                            const double *re = tb == 0 ? hr : sr, *imv = tb == 0 ? hi : si;
                            double *M_ = tb == 0 ? H0 : S;
                            const double zr = A == B ? 0.5 * (re[u] + re[ut]) : re[u];
                            const double zi = A == B ? 0.5 * (imv[u] - imv[ut]) : imv[u];
                            const int row = oA + mu, col = oB + nu;
                            if (A == B) {
                                M_[(long long)col * m + row] += zr;
                                M_[(long long)(col + n) * m + row] -= zi;
                                M_[(long long)col * m + row + n] += zi;
                                M_[(long long)(col + n) * m + row + n] += zr;
                            } else {
                                M_[(long long)col * m + row] = zr;
                                M_[(long long)(col + n) * m + row] = -zi;
                                M_[(long long)col * m + row + n] = zi;
                                M_[(long long)(col + n) * m + row + n] = zr;
                                M_[(long long)row * m + col] = zr;
                                M_[(long long)(row + n) * m + col] = zi;
                                M_[(long long)row * m + col + n] = -zi;
                                M_[(long long)(row + n) * m + col + n] = zr;
                            }
                        }
                    }
                if (first) {
                    double gv = g_re + g_sr + pl.bg;
                    if (A == B) gv += sk.hubbard[eA] + pl.self_e;
                    gam[A * pl.amax + B] = gv;
                    gam[B * pl.amax + A] = gv;
                }
            }
            __syncthreads();
        }
    } else {
        for (int e = j; e < nn; e += PT) {
            const int c = e / n, i = e - c * n;
            double h = 0.0, s = 0.0;
            if (i == c) {
                const int at = sh.orb_atom[c], el = sh.spec[at];
                h = (c == sh.atom_off[at]) ? sk.onsite[el][0] : sk.onsite[el][1];
                s = 1.0;
            }
            H0[e] = h;
            S[e] = s;
        }
        __syncthreads();
        for (int t = j; t < nat * (nat + 1) / 2; t += PT) {   // pairs A <= B, by kind
            int A, B;
                pbc_pair(sh, nat, t, A, B);
            const int eA = sh.spec[A], eB = sh.spec[B];
            const int oA = sh.atom_off[A], oB = sh.atom_off[B];
            const int na = sk.norb[eA], nb = sk.norb[eB];
            double d[3], f[3], dw[3];
            for (int k = 0; k < 3; ++k) d[k] = sh.pos[B][k] - sh.pos[A][k];
            for (int k = 0; k < 3; ++k) f[k] = rint(fma(d[0], pl.inv[k], fma(d[1], pl.inv[3 + k], d[2] * pl.inv[6 + k])));
            for (int k = 0; k < 3; ++k) dw[k] = d[k] - fma(f[0], pl.lat[k], fma(f[1], pl.lat[3 + k], f[2] * pl.lat[6 + k]));
            double hb[16], sb[16];
            for (int u = 0; u < 16; ++u) { hb[u] = 0.0; sb[u] = 0.0; }
            double g_re = 0.0, g_sr = 0.0;
            const double c2 = sk.gamma_c2[eA][eB];
            const double rc2 = sk.r_cut * sk.r_cut;
            pbc_images(pl, dw, pl.n_img, pl.r_real2, [&](int im) {   // real-space Ewald sum
                const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                if (!(r2 < pl.r_real2) || r2 == 0.0) return;
                const double ir = rsqrt_nr(r2);
                g_re = fma(erfc(pl.alpha * (r2 * ir)), ir, g_re);
            });
            pbc_images(pl, dw, pl.n_img_sk, rc2, [&](int im) {   // images within r_cut
                const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                if (!(r2 < rc2) || r2 == 0.0) return;
                const double ir = rsqrt_nr(r2);
                const double r = r2 * ir;
                const double e[3] = {x0 * ir, x1 * ir, x2 * ir};
                for (int tb = 0; tb < 2; ++tb) {
                    const double(*tab)[CAVMD_MAX_ELEM][4][4] = tb == 0 ? sk.h0 : sk.s;
                    double *acc = tb == 0 ? hb : sb;
                    double v, dv;
                    radial_p(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                    acc[0] += v;
                    if (nb == 4) {
                        radial_p(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                        for (int i = 0; i < 3; ++i) acc[1 + i] = fma(e[i], v, acc[1 + i]);
                    }
                    if (na == 4) {
                        radial_p(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                        for (int i = 0; i < 3; ++i) acc[4 * (1 + i)] = fma(-e[i], v, acc[4 * (1 + i)]);
                    }
                    if (na == 4 && nb == 4) {
                        double vs, vp;
                        radial_p(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dv);
                        radial_p(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dv);
                        const double dl = vs - vp;
                        for (int i = 0; i < 3; ++i)
                            for (int k = 0; k < 3; ++k)
                                acc[4 * (1 + i) + 1 + k] += fma(e[i] * e[k], dl, (i == k) ? vp : 0.0);
                    }
                }
                double fc, dfc;
                cutoff_fn(r, sk, fc, dfc);
                g_sr = fma(rsqrt_nr(r2 + c2) - ir, fc, g_sr);
            });
            // block (mu of A, nu of B) at column oB + nu, row oA + mu, and its transpose; a block of an
            // atom with its own images is symmetric, written as the mean of the two halves
            for (int mu = 0; mu < na; ++mu)
                for (int nu = 0; nu < nb; ++nu) {
                    const double hv = A == B ? 0.5 * (hb[4 * mu + nu] + hb[4 * nu + mu]) : hb[4 * mu + nu];
                    const double sv = A == B ? 0.5 * (sb[4 * mu + nu] + sb[4 * nu + mu]) : sb[4 * mu + nu];
                    H0[(oB + nu) * n + oA + mu] += hv;
                    S[(oB + nu) * n + oA + mu] += sv;
                    if (A != B) {
                        H0[(oA + mu) * n + oB + nu] = hv;
                        S[(oA + mu) * n + oB + nu] = sv;
                    }
                }
            double gv = g_re + g_sr + pl.bg;
            if (A == B) gv += sk.hubbard[eA] + pl.self_e;
            gam[A * pl.amax + B] = gv;
            gam[B * pl.amax + A] = gv;
        }
    }
    // cos and sin of G . (r_A - r_0) for the reciprocal sum:
    // G = m0 b0 + m1 b1 + m2 b2: products of three powers of exp(i b . (r_A - r_0)), so a (vector, atom) takes
    // two complex products instead of a sincos. The powers: [axis][0..g_max][atom].
    {
        double2 *pw = reinterpret_cast<double2 *>(wk.pw);
        const int gm = pl.g_max + 1;
        for (int e = j; e < 3 * nat; e += PT) {
            const int ax = e / nat, at = e - ax * nat;
            const double turns = fma(sh.pos[at][0] - sh.pos[0][0], pl.inv[ax],
                                     fma(sh.pos[at][1] - sh.pos[0][1], pl.inv[3 + ax], (sh.pos[at][2] - sh.pos[0][2]) * pl.inv[6 + ax]));
            double sn, cn;
            sincospi(2.0 * turns, &sn, &cn);
            double x = 1.0, y = 0.0;
            for (int q = 0; q < gm; ++q) {
                pw[(ax * gm + q) * nat + at] = make_double2(x, y);
                const double u = fma(x, cn, -y * sn);
                y = fma(x, sn, y * cn);
                x = u;
            }
        }
        __syncthreads();
        for (int e = j + rank * PT; e < nat * pl.n_g; e += blocks * PT) {
            const int g = e / nat, at = e - g * nat;
            const int4 q = pl.gi[g];   // m0 >= 0 or the vector is the half space's; signs by conjugation
            double2 a0 = pw[abs(q.x) * nat + at], a1 = pw[(gm + abs(q.y)) * nat + at], a2 = pw[(2 * gm + abs(q.z)) * nat + at];
            a0.y = q.x < 0 ? -a0.y : a0.y;
            a1.y = q.y < 0 ? -a1.y : a1.y;
            a2.y = q.z < 0 ? -a2.y : a2.y;
            const double u = fma(a0.x, a1.x, -a0.y * a1.y), v = fma(a0.x, a1.y, a0.y * a1.x);
            csg[2LL * e] = fma(u, a2.x, -v * a2.y);
            csg[2LL * e + 1] = fma(u, a2.y, v * a2.x);
        }
    }
    cluster_barrier(blocks);

    // ---------------------------------------------------------------- warm path
    bool warm = false;
    int evals = 0;
    if (a.have_warm && mo > 0 && m > mo && !(KG && pl.late_pass)) {
        warm = p_warm<KG>(a, pl, sh, wk, C0, wk.Cd, n, nocc, nat, rank, blocks, evals);
        if (j < nat) sh.qst[j] = a.qpop[a0 + j];
        if (j == 0) sh.fl[2] = evals;
        __syncthreads();
    }
    if (!warm && blocks > 1) {
        if (rank == 0 && j == 0) pl.late[1 + atomicAdd(pl.late, 1)] = item;
        cluster_barrier(blocks);   // the workspace is the next cell's from here on
        return;
    }
    if (warm) {
        Cb = wk.Cd;
        if (!disp)
            for (int kp = rank; kp < NKP; kp += blocks)
                for (long long e = j; e < mm; e += PT) C0[(long long)kp * mm + e] = Cb[(long long)kp * mm + e];
    } else if (disp) {   // a private copy of the cell's basis: the cell and its other copies read the original
        for (long long e = j; e < (long long)NKP * mm; e += PT) wk.Cd[e] = C0[e];
        Cb = wk.Cd;
        __syncthreads();
    }
    C = Cb;
    // atomic shifts eps_A = sum_B gamma_AB dq_B + reciprocal part, from sh.dq
    auto shifts = [&]() { p_shifts(sh, pl, wk, nat); };
    auto build_h = [&]() {
        for (int e = j; e < mm; e += PT) {
            const int c = e / m, i = e - c * m;
            const int io = (KG && i >= n) ? i - n : i, co = (KG && c >= n) ? c - n : c;
            H[e] = fma(0.5 * S[e], sh.shift[sh.orb_atom[io]] + sh.shift[sh.orb_atom[co]], H0[e]);
        }
        __syncthreads();
    };
    auto rank_occupation = [&]() {
        for (int r = j; r < m; r += PT) {
            const long long kj = order_key(sh.diag[r]);
            int rank = 0;
            for (int i = 0; i < m; ++i) {
                const long long ki = order_key(sh.diag[i]);
                rank += (ki < kj) || (ki == kj && i < r);
            }
            sh.occf[r] = rank < mo;
            if (rank < mo) sh.occ_list[rank] = r; else sh.virt_list[rank - mo] = r;
        }
        __syncthreads();
    };
    auto Cat = [&](int i, int c) -> double { return C[c * m + i]; };
    // One cyclic Jacobi sweep on the block Ab = C_b^T Y_b of the columns list[0..m-1] (occupied or
    // virtual). It keeps the diagonal blocks of C^T H C diagonal, which the generator's diagonal
    // denominators need (the occupied-virtual rotations leave them alone, and within a block they
    // drift with every step). The rounds rotate Ab and accumulate the rotations in Vb (m x m,
    // starting from I); then C_b <- C_b Vb and Y_b <- Y_b Vb as staged products through H, which
    // is free until the next iteration builds it.
    // Workspaces it overwrites: Vb (the caller passes the density buffer P, free at this point:
    // P = 2 C_o C_o^T is formed later in the same iteration) and H (rebuilt at the start of the
    // next iteration). Neither may be read after a sweep before it is formed again.
    auto block_sweep = [&](const int *list, int mb, double *Ab, double *Vb) {
        pprod<false, true, true>(sh, mb, mb, m, [&](int i, int k) { return C[list[i] * m + k]; },
                                 [&](int k, int c) { return Y[list[c] * m + k]; },
                                 [&](int i, int c, double v) { Ab[c * mb + i] = v; });
        for (int e = j; e < mb * mb; e += PT) Vb[e] = (e / mb == e % mb) ? 1.0 : 0.0;
        __syncthreads();
        const int me = mb + (mb & 1), half = me / 2, span = 2 * mb;
        for (int rd = 0; rd < me - 1; ++rd) {
            if (j < half) {
                int p, qq;
                p_pair(j, rd, me, p, qq);
                double c = 1.0, s = 0.0;
                if (qq < mb) p_jacobi_cs(Ab[p * mb + p], Ab[qq * mb + qq], Ab[qq * mb + p], c, s);
                sh.pp[j] = p;
                sh.pq[j] = qq;
                sh.cs[2 * j] = c;
                sh.cs[2 * j + 1] = s;
            }
            __syncthreads();
            for (int e = j; e < half * span; e += PT) {   // columns p, q of Ab and Vb
                const int k = e / span, r = e - k * span;
                const int p = sh.pp[k], qq = sh.pq[k];
                if (qq >= mb) continue;
                const double c = sh.cs[2 * k], s = sh.cs[2 * k + 1];
                double *base = r < mb ? Ab : Vb;
                const int rr = r < mb ? r : r - mb;
                const double xp = base[p * mb + rr], yq = base[qq * mb + rr];
                base[p * mb + rr] = fma(c, xp, -s * yq);
                base[qq * mb + rr] = fma(s, xp, c * yq);
            }
            __syncthreads();
            for (int e = j; e < half * mb; e += PT) {   // rows p, q of Ab
                const int k = e / mb, cc = e - k * mb;
                const int p = sh.pp[k], qq = sh.pq[k];
                if (qq >= mb) continue;
                const double ck = sh.cs[2 * k], sk_ = sh.cs[2 * k + 1];
                const double x = Ab[cc * mb + p], y = Ab[cc * mb + qq];
                Ab[cc * mb + p] = fma(ck, x, -sk_ * y);
                Ab[cc * mb + qq] = fma(sk_, x, ck * y);
            }
            __syncthreads();
        }
        for (int t = 0; t < 2; ++t) {   // C_b <- C_b Vb, then Y_b <- Y_b Vb
            double *M_ = t == 0 ? C : Y;
            pprod<false, false, true>(sh, m, mb, mb, [&](int i, int k) { return M_[list[k] * m + i]; },
                                      [&](int k, int c) { return Vb[c * mb + k]; },
                                      [&](int i, int c, double v) { H[c * m + i] = v; });
            for (int e = j; e < m * mb; e += PT) {
                const int c = e / m, i = e - c * m;
                M_[list[c] * m + i] = H[e];
            }
            __syncthreads();
        }
        for (int r = j; r < mb; r += PT) sh.diag[list[r]] = Ab[r * mb + r];
        __syncthreads();
    };

    if (!warm) {
    // ---------------------------------------------------------------- S-orthonormal start
    if (j < nat) {
        if (a.have_warm) {   // predictor 2 q(t) - q(t - dt); a displaced copy starts from q(r)
            const double qt = a.qpop[a0 + j];
            sh.qst[j] = qt;
            sh.q[j] = disp ? qt : fma(2.0, qt, -a.qprev[a0 + j]);
        } else {
            sh.q[j] = sh.zv[j];
        }
    }
    __syncthreads();
    // Mo <- lower of C^T S C (Y = S C first), its Cholesky factor L, then C <- C L^-T (every k-point)
    for (int kp = 0; kp < NKP; ++kp) {
        set_k(kp);
        if (!a.have_warm)
            for (int e = j; e < mm; e += PT) C[e] = (e / m == e % m) ? 1.0 : 0.0;
        pprod<false, false, true>(sh, m, m, m, [&](int i, int k) { return S[k * m + i]; }, Cat,
                                  [&](int i, int c, double v) { Y[c * m + i] = v; });
        pprod<true, true, true>(sh, m, m, m, [&](int i, int k) { return C[i * m + k]; },
                                [&](int k, int c) { return Y[c * m + k]; }, [&](int i, int c, double v) { Mo[c * m + i] = v; });
        if (!pchol(Mo, m, sh) && j == 0) sh.fl[0] |= ERRBIT_S_NOT_PD;
        for (int r = j; r < m; r += PT) row_solve_lt(Mo, m, sh.invd, C + r, m);
        __syncthreads();
    }

    // Warm steps re-diagonalise the occupied and virtual blocks every P_SWEEP_PERIOD steps, and
    // after an evaluation that needed more than P_SWEEP_ITERS iterations (a cold start, or drift).
    const bool sweep_now = a.have_warm && ((a.step_counter && (*a.step_counter % P_SWEEP_PERIOD) == 0) ||
                                           a.iters[cell] > P_SWEEP_ITERS);

    // ---------------------------------------------------------------- SCC loop
    // Per iteration: shifts, H, Y = H C, the diagonal of C^T Y and the occupation by rank; then the
    // occupied-virtual block A_vo, the generator X(v, o) = A_vo / (A_oo - A_vv) (FP32: it only
    // steers) and the Cayley rotation
    //   C_o <- (2 C_o + C_v X) (I + X^T X / 4)^-1 - C_o,  C_v <- (2 C_v - C_o X^T) (I + X X^T / 4)^-1 - C_v,
    // which is C (I - K/2)^-1 (I + K/2) for the antisymmetric K with K_vo = X. A cold start instead
    // forms all of C^T H C and runs Jacobi sweeps on its first iteration. Then P = 2 C_o C_o^T,
    // the Mulliken populations and Anderson mixing.
    int it;
    for (it = 1; it <= a.max_iter; ++it) {
        if (j < nat) sh.dq[j] = sh.q[j] - sh.zv[j];
        __syncthreads();
        shifts();
        bool eok_all = true;
        if (KG) {
            for (int r = j; r < n; r += PT) sh.qk[r] = 0.0;
            if (j == 0) {
                sh.hl[0] = -1e300;
                sh.hl[1] = 1e300;
            }
        }
        for (int kp = 0; kp < NKP; ++kp) {   // each k-point's update (Gamma: the one problem)
        set_k(kp);
        build_h();
        pprod<false, false, true>(sh, m, m, m, [&](int i, int k) { return H[k * m + i]; }, Cat,
                                  [&](int i, int c, double v) { Y[c * m + i] = v; });
        for (int r = j; r < m; r += PT) {
            double dg = 0.0;
            for (int k = 0; k < m; ++k) dg = fma(C[r * m + k], Y[r * m + k], dg);
            sh.diag[r] = dg;
        }
        __syncthreads();
        bool eok = false;
        const bool cold_first = !a.have_warm && it == 1;
        if (cold_first) {
            // all of A = C^T H C into P, then Jacobi sweeps on A accumulated into C
            pprod<false, true, true>(sh, m, m, m, [&](int i, int k) { return C[i * m + k]; },
                                     [&](int k, int c) { return Y[c * m + k]; },
                                     [&](int i, int c, double v) { P[c * m + i] = v; });
            double *Am = P;
            const int cap = a.max_sweeps > 0 ? a.max_sweeps : P_MAX_SWEEPS;
            for (int sweep = 0;; ++sweep) {
                bool off_small = true;
                for (int e = j; e < mm; e += PT) {
                    const int c = e / m, i = e - c * m;
                    if (i != c && !abs_lt(Am[c * m + i], P_JACOBI_TOL)) off_small = false;
                }
                if (blk_all(off_small)) break;
                if (sweep >= cap) {   // the cold start's sweeps ran out: DEVICE_TIMEOUT
                    if (j == 0) sh.fl[0] |= ERRBIT_TIMEOUT;
                    break;
                }
                for (int rd = 0; rd < m - 1; ++rd) {
                    if (j < m / 2) {
                        int p, qq;
                        p_pair(j, rd, m, p, qq);
                        double c, s;
                        p_jacobi_cs(Am[p * m + p], Am[qq * m + qq], Am[qq * m + p], c, s);
                        sh.pp[j] = p;
                        sh.pq[j] = qq;
                        sh.cs[2 * j] = c;
                        sh.cs[2 * j + 1] = s;
                    }
                    __syncthreads();
                    for (int e = j; e < m * (m / 2); e += PT) {   // columns p, q of A and C, row i
                        const int k = e / m, i = e - k * m;
                        const int p = sh.pp[k], qq = sh.pq[k];
                        const double c = sh.cs[2 * k], s = sh.cs[2 * k + 1];
                        const double ap = Am[p * m + i], aq = Am[qq * m + i];
                        Am[p * m + i] = fma(c, ap, -s * aq);
                        Am[qq * m + i] = fma(s, ap, c * aq);
                        const double cp = C[p * m + i], cq = C[qq * m + i];
                        C[p * m + i] = fma(c, cp, -s * cq);
                        C[qq * m + i] = fma(s, cp, c * cq);
                    }
                    __syncthreads();
                    for (int e = j; e < m * (m / 2); e += PT) {   // rows p, q of A, column c
                        const int k = e / m, c = e - k * m;
                        const int p = sh.pp[k], qq = sh.pq[k];
                        const double ck = sh.cs[2 * k], sk_ = sh.cs[2 * k + 1];
                        const double x = Am[c * m + p], y = Am[c * m + qq];
                        Am[c * m + p] = fma(ck, x, -sk_ * y);
                        Am[c * m + qq] = fma(sk_, x, ck * y);
                    }
                    __syncthreads();
                }
            }
            for (int r = j; r < m; r += PT) sh.diag[r] = Am[r * m + r];
            __syncthreads();
            rank_occupation();
        } else {
            rank_occupation();
            if (sweep_now && it == 1) {   // first iteration after a geometry change
                double *const sweep_V = P;   // the rotation accumulator: P is formed later this iteration
                block_sweep(sh.occ_list, mo, Mo, sweep_V);
                block_sweep(sh.virt_list, mv, Mv, sweep_V);
            }
            bool small = true;
            float kmax = 0.0f;
            // A_vo (entry (v, o), v fastest) and the generator, stored X[o nv + v]
            pprod<false, true, true>(sh, mv, mo, m, [&](int v, int k) { return C[sh.virt_list[v] * m + k]; },
                                     [&](int k, int o) { return Y[sh.occ_list[o] * m + k]; },
                                     [&](int v, int o, double val) {
                                         if (!abs_lt(val, P_EIG_TOL)) small = false;
                                         const float den = d2f_steer(sh.diag[sh.occ_list[o]] - sh.diag[sh.virt_list[v]]);
                                         float kf = d2f_steer(val) / den;
                                         if (!(fabsf(kf) <= 1e3f)) kf = copysignf(1e3f, kf);
                                         kmax = fmaxf(kmax, fabsf(kf));
                                         Xg[o * mv + v] = f2d_steer(kf);
                                     });
            eok = blk_all(small);
            // X^T X and X X^T (lower triangles)
            pprod<true, true, true>(sh, mo, mo, mv, [&](int o1, int v) { return Xg[o1 * mv + v]; },
                                    [&](int v, int o2) { return Xg[o2 * mv + v]; },
                                    [&](int i, int c, double v) { Mo[c * mo + i] = v; });
            pprod<true, false, false>(sh, mv, mv, mo, [&](int v1, int o) { return Xg[o * mv + v1]; },
                                      [&](int o, int v2) { return Xg[o * mv + v2]; },
                                      [&](int i, int c, double v) { Mv[c * mv + i] = v; });
            if (blk_all(kmax < P_KMAX_PERT)) {
                // small generator: C <- C (I + K + K^2/2), orthogonal to O(K^4) (below 1e-16 here):
                //   C_o <- C_o (I - X^T X / 2) + C_v X,  C_v <- C_v (I - X X^T / 2) - C_o X^T,
                // each one staged product over the columns [C_o | C_v], into Y
                pprod<false, false, true>(
                    sh, m, mo, m,
                    [&](int i, int k) { return C[(k < mo ? sh.occ_list[k] : sh.virt_list[k - mo]) * m + i]; },
                    [&](int k, int o) {
                        if (k >= mo) return Xg[o * mv + (k - mo)];
                        return fma(-0.5, Mo[min(k, o) * mo + max(k, o)], k == o ? 1.0 : 0.0);
                    },
                    [&](int i, int o, double v) { Y[o * m + i] = v; });
                pprod<false, false, false>(
                    sh, m, mv, m,
                    [&](int i, int k) { return C[(k < mv ? sh.virt_list[k] : sh.occ_list[k - mv]) * m + i]; },
                    [&](int k, int v) {
                        if (k >= mv) return -Xg[(k - mv) * mv + v];
                        return fma(-0.5, Mv[min(k, v) * mv + max(k, v)], k == v ? 1.0 : 0.0);
                    },
                    [&](int i, int v, double val) { Y[(mo + v) * m + i] = val; });
                for (int e = j; e < mm; e += PT) {
                    const int c = e / m, i = e - c * m;
                    const int col = c < mo ? sh.occ_list[c] : sh.virt_list[c - mo];
                    C[col * m + i] = Y[e];
                }
                __syncthreads();
            } else {
            // I + X^T X / 4 and I + X X^T / 4 in place
            for (int e = j; e < mo * mo; e += PT) {
                const int c = e / mo, i = e - c * mo;
                if (i >= c) Mo[e] = fma(0.25, Mo[e], i == c ? 1.0 : 0.0);
            }
            for (int e = j; e < mv * mv; e += PT) {
                const int c = e / mv, i = e - c * mv;
                if (i >= c) Mv[e] = fma(0.25, Mv[e], i == c ? 1.0 : 0.0);
            }
            __syncthreads();
            // Z1 = 2 C_o + C_v X into Y[o n + i]; Z2 = 2 C_v - C_o X^T into Y[(nocc + v) n + i]
            pprod<false, false, true>(sh, m, mo, mv, [&](int i, int v) { return C[sh.virt_list[v] * m + i]; },
                                      [&](int v, int o) { return Xg[o * mv + v]; },
                                      [&](int i, int o, double v) { Y[o * m + i] = fma(2.0, C[sh.occ_list[o] * m + i], v); });
            pprod<false, false, false>(sh, m, mv, mo, [&](int i, int o) { return C[sh.occ_list[o] * m + i]; },
                                       [&](int o, int v) { return Xg[o * mv + v]; },
                                       [&](int i, int v, double val) {
                                           Y[(mo + v) * m + i] = fma(2.0, C[sh.virt_list[v] * m + i], -val);
                                       });
            pchol(Mo, mo, sh);
            for (int r = j; r < m; r += PT) row_solve_llt(Mo, mo, sh.invd, Y + r, m, Y + r, m);
            __syncthreads();
            if (mv > 0) {
                pchol(Mv, mv, sh);
                for (int r = j; r < m; r += PT) row_solve_llt(Mv, mv, sh.invd, Y + mo * m + r, m, Y + mo * m + r, m);
            }
            __syncthreads();
            for (int e = j; e < mm; e += PT) {
                const int c = e / m, i = e - c * m;   // c < mo: occupied column c, else virtual c - mo
                const int col = c < mo ? sh.occ_list[c] : sh.virt_list[c - mo];
                C[col * m + i] = Y[e] - C[col * m + i];
            }
            __syncthreads();
            }
        }
        // P = 2 C_o C_o^T (lower triangle) and the Mulliken populations
        pprod<true, false, false>(sh, m, m, mo, [&](int i, int o) { return C[sh.occ_list[o] * m + i]; },
                                  [&](int o, int c) { return C[sh.occ_list[o] * m + c]; },
                                  [&](int i, int c, double v) { P[c * m + i] = 2.0 * v; });
        for (int r = j; r < m; r += PT) {
            double qo = 0.0;
            for (int k = 0; k < m; ++k) {
                const int lo = min(r, k), hi = max(r, k);
                qo = fma(P[lo * m + hi], S[k * m + r], qo);
            }
            sh.red[r] = qo;
        }
        __syncthreads();
        if (KG) {   // the k-point's populations (both halves of the real form) and its frontier levels
            const double w = pl.kpt[4 * kp + 3];
            for (int r = j; r < n; r += PT) sh.qk[r] = fma(0.5 * w, sh.red[r] + sh.red[r + n], sh.qk[r]);
            if (j == 0 && mo < m) {
                double homo = -1e300, lumo = 1e300;
                for (int c = 0; c < m; ++c) {
                    if (sh.occf[c]) homo = fmax(homo, sh.diag[c]); else lumo = fmin(lumo, sh.diag[c]);
                }
                sh.hl[0] = fmax(sh.hl[0], homo);
                sh.hl[1] = fmin(sh.hl[1], lumo);
            }
            __syncthreads();
        }
        eok_all = eok_all && eok;
        }
        const int NH = a.hist;
        const int hs = (it - 1) % NH;
        if (j < nat) {
            double qa = 0.0;
            for (int o = sh.atom_off[j]; o < sh.atom_off[j + 1]; ++o) qa += KG ? sh.qk[o] : sh.red[o];
            sh.qout[j] = qa;
            sh.hq[hs][j] = sh.q[j];
            sh.hf[hs][j] = qa - sh.q[j];
        }
        __syncthreads();
        bool conv = eok_all;
        for (int at = 0; at < nat; ++at)
            if (!abs_lt(sh.hf[hs][at], a.scc_tol)) conv = false;
        const int h = min(it, NH);
        if (!conv && j == 0) {
            // Anderson coefficients over the h - 1 previous iterates: normal equations in FP32 with
            // a small diagonal shift, solved by Cholesky (they only steer the iteration)
            float Mx[PHIST - 1][PHIST - 1], bv[PHIST - 1], x[PHIST - 1];
            const int mh = h - 1;
            for (int u = 0; u < mh; ++u) {
                const int hu = (hs + NH - 1 - u) % NH;
                float b = 0.f;
                for (int w = 0; w <= u; ++w) {
                    const int hw = (hs + NH - 1 - w) % NH;
                    float sacc = 0.f;
                    for (int at = 0; at < nat; ++at) {
                        const float du = d2f_steer(sh.hf[hu][at] - sh.hf[hs][at]);
                        const float dw = d2f_steer(sh.hf[hw][at] - sh.hf[hs][at]);
                        sacc = fmaf(du, dw, sacc);
                    }
                    Mx[u][w] = sacc;
                }
                for (int at = 0; at < nat; ++at)
                    b = fmaf(-d2f_steer(sh.hf[hu][at] - sh.hf[hs][at]), d2f_steer(sh.hf[hs][at]), b);
                bv[u] = b;
            }
            float dmax = 0.f;
            for (int u = 0; u < mh; ++u) dmax = fmaxf(dmax, Mx[u][u]);
            bool ok = mh > 0 && dmax > 0.f;
            for (int u = 0; u < mh && ok; ++u) {
                for (int w = 0; w <= u && ok; ++w) {
                    float sacc = Mx[u][w] + (u == w ? 1e-6f * dmax : 0.f);
                    for (int l = 0; l < w; ++l) sacc -= Mx[u][l] * Mx[w][l];
                    if (u == w) {
                        if (!(sacc > 0.f)) ok = false; else Mx[u][u] = sqrtf(sacc);
                    } else {
                        Mx[u][w] = sacc / Mx[w][w];
                    }
                }
            }
            if (ok) {
                for (int u = 0; u < mh; ++u) {
                    float sacc = bv[u];
                    for (int l = 0; l < u; ++l) sacc -= Mx[u][l] * x[l];
                    x[u] = sacc / Mx[u][u];
                }
                for (int u = mh - 1; u >= 0; --u) {
                    float sacc = x[u];
                    for (int l = u + 1; l < mh; ++l) sacc -= Mx[l][u] * x[l];
                    x[u] = sacc / Mx[u][u];
                }
                for (int u = 0; u < mh; ++u)
                    if (!(fabsf(x[u]) < 50.f)) ok = false;
            }
            for (int u = 0; u < PHIST - 1; ++u) sh.th[u] = (ok && u < mh) ? f2d_steer(x[u]) : 0.0;
        }
        __syncthreads();
        if (j < nat) {
            if (conv) {
                sh.q[j] = sh.qout[j];
            } else {
                const double q0 = sh.hq[hs][j], f0 = sh.hf[hs][j];
                double qb = q0, fb = f0;
                for (int u = 0; u < h - 1; ++u) {
                    const int hu = (hs + NH - 1 - u) % NH;
                    qb = fma(sh.th[u], sh.hq[hu][j] - q0, qb);
                    fb = fma(sh.th[u], sh.hf[hu][j] - f0, fb);
                }
                sh.q[j] = fma(a.beta, fb, qb);
            }
        }
        __syncthreads();
        if (conv) {
            if (j == 0) sh.fl[2] = it;
            break;
        }
    }
    __syncthreads();
    if (j == 0 && it > a.max_iter) {
        sh.fl[0] |= ERRBIT_SCC_NOCONV;
        sh.fl[2] = a.max_iter;
    }
    __syncthreads();
    }   // general path
    if (disp) {   // a finite-difference copy: only its dipole
        if (j == 0 && rank == 0) {
            double mu[3] = {0.0, 0.0, 0.0};
            for (int at = 0; at < nat; ++at) {
                const double Q = sh.zv[at] - sh.q[at];
                for (int k = 0; k < 3; ++k) mu[k] = fma(Q, sh.pos[at][k] - sh.pos[0][k], mu[k]);
            }
            a.M_disp[(long long)(a.fd_central ? 6 : 3) * a0 + disp_k] =
                fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
            if (sh.fl[0]) atomicOr(a.status, (unsigned)sh.fl[0]);
        }
        cluster_barrier(blocks);
        return;
    }
    if (warm) {   // the basis has its occupied columns first
        for (int r = j; r < m; r += PT) {
            sh.occf[r] = r < mo;
            if (r < mo) sh.occ_list[r] = r; else sh.virt_list[r - mo] = r;
        }
        __syncthreads();
    }
    // stores a basis with its occupied columns first, as the warm path reads it
    auto store_sorted = [&]() {
        for (int e = j; e < mm; e += PT) {
            const int c = e / m, i = e - c * m;
            Y[e] = C[(c < mo ? sh.occ_list[c] : sh.virt_list[c - mo]) * m + i];
        }
        __syncthreads();
        for (int e = j; e < mm; e += PT) C[e] = Y[e];
        __syncthreads();
    };

    // ---------------------------------------------------------------- energy and forces
    if constexpr (KG) {
        // per k-point: H; Y = H C and the occupation by rank; Aoo = C_o^T Y_o (lower) into Mo;
        // t = 2 Aoo C_o^T into Mv; W = C_o t (lower) into H; P = 2 C_o C_o^T (lower) into P; then the
        // pair tasks with the k-point's phases, accumulated over the k-points (the k-independent
        // terms, second order and repulsion, with the first)
        if (j < nat) sh.dq[j] = sh.q[j] - sh.zv[j];
        __syncthreads();
        shifts();
        if (j == 0) {
            sh.hl[0] = -1e300;
            sh.hl[1] = 1e300;
        }
        double eb_t = 0.0;   // this thread's part of the band energy sum_k w_k Re Tr P(k) H0(k)*
        const double rc2 = sk.r_cut * sk.r_cut;
        for (int kp = rank; kp < NKP; kp += blocks) {
            set_k(kp);
            const bool first = kp == 0, fresh = kp == rank;
            const double wkp = pl.kpt[4 * kp + 3];
            const double fk[3] = {pl.kpt[4 * kp], pl.kpt[4 * kp + 1], pl.kpt[4 * kp + 2]};
            build_h();
            pprod<false, false, true>(sh, m, warm ? mo : m, m, [&](int i, int k) { return H[k * m + i]; }, Cat,
                                      [&](int i, int c, double v) { Y[c * m + i] = v; });
            if (!warm) {
                for (int r = j; r < m; r += PT) {
                    double dg = 0.0;
                    for (int k = 0; k < m; ++k) dg = fma(C[r * m + k], Y[r * m + k], dg);
                    sh.diag[r] = dg;
                }
                __syncthreads();
                rank_occupation();
                if (j == 0) {
                    for (int c = 0; c < m; ++c) {
                        if (sh.occf[c]) sh.hl[0] = fmax(sh.hl[0], sh.diag[c]); else sh.hl[1] = fmin(sh.hl[1], sh.diag[c]);
                    }
                }
            }
            pprod<true, true, true>(sh, mo, mo, m, [&](int o1, int k) { return C[sh.occ_list[o1] * m + k]; },
                                    [&](int k, int o2) { return Y[sh.occ_list[o2] * m + k]; },
                                    [&](int i, int c, double v) { Mo[c * mo + i] = v; });
            pprod<false, false, false>(sh, mo, m, mo,
                                       [&](int o, int o2) { return Mo[min(o, o2) * mo + max(o, o2)]; },
                                       [&](int o2, int c) { return C[sh.occ_list[o2] * m + c]; },
                                       [&](int o, int c, double v) { Mv[c * mo + o] = 2.0 * v; });
            pprod<true, false, true>(sh, m, m, mo, [&](int i, int o) { return C[sh.occ_list[o] * m + i]; },
                                     [&](int o, int c) { return Mv[c * mo + o]; },
                                     [&](int i, int c, double v) { H[c * m + i] = v; });
            pprod<true, false, false>(sh, m, m, mo, [&](int i, int o) { return C[sh.occ_list[o] * m + i]; },
                                      [&](int o, int c) { return C[sh.occ_list[o] * m + c]; },
                                      [&](int i, int c, double v) { P[c * m + i] = 2.0 * v; });
            for (int r = j; r < m; r += PT) {   // sum over the real form: 2 Re Tr P(k) H0(k)*
                double eb = 0.0;
                for (int i = r; i < m; ++i) eb = fma((i == r ? 1.0 : 2.0) * P[r * m + i], H0[r * m + i], eb);
                eb_t = fma(0.5 * wkp, eb, eb_t);
            }
            __syncthreads();
            const double *W = H;
            for (int t = j; t < nat * (nat + 1) / 2; t += PT) {   // pairs A <= B, by kind
                int A, B;
                pbc_pair(sh, nat, t, A, B);
                const int eA = sh.spec[A], eB = sh.spec[B];
                const int oA = sh.atom_off[A], oB = sh.atom_off[B];
                const int na = sk.norb[eA], nb = sk.norb[eB];
                double d[3], f[3], dw[3];
                for (int k = 0; k < 3; ++k) d[k] = sh.pos[B][k] - sh.pos[A][k];
                for (int k = 0; k < 3; ++k) f[k] = rint(fma(d[0], pl.inv[k], fma(d[1], pl.inv[3 + k], d[2] * pl.inv[6 + k])));
                for (int k = 0; k < 3; ++k) dw[k] = d[k] - fma(f[0], pl.lat[k], fma(f[1], pl.lat[3 + k], f[2] * pl.lat[6 + k]));
                const double hshift = 0.5 * (sh.shift[A] + sh.shift[B]);
                const double qq = sh.dq[A] * sh.dq[B];
                const double c2 = sk.gamma_c2[eA][eB];
                const double arep = sk.rep[eA][eB][0], brep = sk.rep[eA][eB][1];
                const double two_a_spi = 2.0 * pl.alpha * 0.5641895835477563;   // 2 alpha / sqrt(pi)
                double gk[3] = {0.0, 0.0, 0.0};
                double erep = 0.0;
                if (A != B && first) {
                    pbc_images(pl, dw, pl.n_img, pl.r_real2, [&](int im) {   // real-space Ewald gradient
                        const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                        const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                        if (!(r2 < pl.r_real2) || r2 == 0.0) return;
                        const double ir = rsqrt_nr(r2);
                        const double ar = pl.alpha * (r2 * ir);
                        const double rad = -qq * (erfc(ar) * ir + two_a_spi * exp(-ar * ar)) * ir * ir;
                        gk[0] = fma(rad, x0, gk[0]);
                        gk[1] = fma(rad, x1, gk[1]);
                        gk[2] = fma(rad, x2, gk[2]);
                    });
                }
                pbc_images(pl, dw, pl.n_img_sk, rc2, [&](int im) {   // images within r_cut
                    const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                    const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                    if (!(r2 < rc2) || r2 == 0.0) return;
                    const double ir = rsqrt_nr(r2);
                    const double r = r2 * ir;
                    const double e[3] = {x0 * ir, x1 * ir, x2 * ir};
                    double rad = 0.0;   // d/dr of the radial terms, along e
                    double fc, dfc;
                    cutoff_fn(r, sk, fc, dfc);
                    if (first) {
                        if (arep != 0.0) {
                            const double vr = arep * exp(-brep * r);
                            erep = fma(vr, fc, erep);
                            if (A != B) rad = fma(vr, dfc - brep * fc, rad);
                        }
                        if (A != B) {
                            const double gi = rsqrt_nr(r2 + c2);
                            const double s_ = gi - ir;
                            const double ds = fma(-r * gi, gi * gi, ir * ir);
                            rad = fma(qq, fma(ds, fc, s_ * dfc), rad);
                        }
                    }
                    if (A != B) {
                        double ph = 0.0;   // the image's phase 2 pi f_k . n_T
                        for (int k = 0; k < 3; ++k) {
                            const double nk_ = rint(fma(pl.img[3 * im], pl.inv[k], fma(pl.img[3 * im + 1], pl.inv[3 + k],
                                                                                         pl.img[3 * im + 2] * pl.inv[6 + k]))) - f[k];
                            ph = fma(fk[k], nk_, ph);
                        }
                        double sn, cs;
                        sincospi(2.0 * ph, &sn, &cs);
                        // band and overlap terms: weights rho(T) and rho(T) (eps_A + eps_B) / 2 - w(T) of the
                        // block, rho(T)_{mu nu} = w_k Re[P(k)_{nu mu} e^{i ph}] (mu of A < nu of B)
                        double g[3] = {0.0, 0.0, 0.0};
                        for (int tb = 0; tb < 2; ++tb) {
                            const double(*tab)[CAVMD_MAX_ELEM][4][4] = tb == 0 ? sk.h0 : sk.s;
                            auto wt = [&](int mu, int nu) -> double {
                                const double pr = P[(long long)mu * m + nu], pim = P[(long long)mu * m + n + nu];
                                const double rho = wkp * fma(pr, cs, -pim * sn);
                                if (tb == 0) return rho;
                                const double wr = W[(long long)mu * m + nu], wim = W[(long long)mu * m + n + nu];
                                return fma(rho, hshift, -wkp * fma(wr, cs, -wim * sn));
                            };
                            double v, dv;
                            radial_p(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                            {
                                const double w = wt(oA, oB) * dv;
                                for (int k = 0; k < 3; ++k) g[k] = fma(w, e[k], g[k]);
                            }
                            if (nb == 4) {
                                radial_p(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                                double w[3], we = 0.0;
                                for (int i = 0; i < 3; ++i) { w[i] = wt(oA, oB + 1 + i); we = fma(w[i], e[i], we); }
                                for (int k = 0; k < 3; ++k) g[k] += fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                            }
                            if (na == 4) {
                                radial_p(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                                double w[3], we = 0.0;
                                for (int i = 0; i < 3; ++i) { w[i] = wt(oA + 1 + i, oB); we = fma(w[i], e[i], we); }
                                for (int k = 0; k < 3; ++k) g[k] -= fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                            }
                            if (na == 4 && nb == 4) {
                                double vs, dvs, vp, dvp;
                                radial_p(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dvs);
                                radial_p(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dvp);
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
                                    g[k] += (We[k] + WTe[k] - 2.0 * eWe * e[k]) * dl * ir + eWe * e[k] * ddl + tr * e[k] * dvp;
                            }
                        }
                        for (int k = 0; k < 3; ++k) gk[k] = fma(2.0, g[k], gk[k]);
                    }
                    for (int k = 0; k < 3; ++k) gk[k] = fma(rad, e[k], gk[k]);
                });
                double *pb = pbuf + 4LL * (A * nat + B);
                if (fresh) {
                    pb[0] = gk[0];
                    pb[1] = gk[1];
                    pb[2] = gk[2];
                    pb[3] = A == B ? 0.5 * erep : erep;
                } else {
                    pb[0] += gk[0];
                    pb[1] += gk[1];
                    pb[2] += gk[2];
                }
            }
            __syncthreads();
            if (!warm) store_sorted();
        }
        if (!warm && j == 0 && mo < m && !(sh.hl[1] - sh.hl[0] > P_MIN_GAP)) sh.fl[0] |= ERRBIT_ZERO_GAP;
        // the band energy into sh.red[0] (the rest of the n entries zero), summed in thread order
        sh.cs[j] = eb_t;
        __syncthreads();
        if (j == 0) {
            double eb = 0.0;
            for (int t = 0; t < PT; ++t) eb += sh.cs[t];
            sh.red[0] = eb;
            if (rank > 0) sgf[0] = eb;   // (the structure factors are rank 0's to read from here on)
        }
        if (blocks > 1) {   // rank 0 adds the others' gradients and band energies, in rank order
            cluster_barrier(blocks);
            if (rank == 0) {
                const long long apart = wk.pbuf_stride;
                for (int e = j; e < nat * nat; e += PT)
                    if (e / nat <= e % nat)
                        for (int b = 1; b < min(blocks, NKP); ++b)
                            for (int k = 0; k < 3; ++k) pbuf[4LL * e + k] += __ldcg(pbuf + b * apart + 4LL * e + k);
                if (j == 0)
                    for (int b = 1; b < blocks; ++b) sh.red[0] += __ldcg(sgf + b * apart);
            }
        }
        for (int r = j; r < n; r += PT)
            if (r > 0) sh.red[r] = 0.0;
        __syncthreads();
    } else {
        // Shifts of the converged charges; H; T = H C_o into Y; Aoo = C_o^T T (lower) into Mo;
        // t = 2 Aoo C_o^T into Mv; W = C_o t (lower) into H; P = 2 C_o C_o^T (lower) into P.
        if (j < nat) sh.dq[j] = sh.q[j] - sh.zv[j];
        __syncthreads();
        if (!warm) {
            shifts();
            build_h();
            pprod<false, false, true>(sh, n, nocc, n, [&](int i, int k) { return H[k * n + i]; },
                                      [&](int k, int o) { return C[sh.occ_list[o] * n + k]; },
                                      [&](int i, int o, double v) { Y[o * n + i] = v; });
        }
        pprod<true, true, true>(sh, nocc, nocc, n, [&](int o1, int k) { return C[sh.occ_list[o1] * n + k]; },
                                [&](int k, int o2) { return Y[o2 * n + k]; },
                                [&](int i, int c, double v) {
                                    const float *dA = (const float *)Mv;
                                    Mo[c * nocc + i] = warm ? v + f2d_steer(dA[c * nocc + i] + dA[i * nocc + c]) : v;
                                });
        pprod<false, false, false>(sh, nocc, n, nocc,
                                   [&](int o, int o2) { return Mo[min(o, o2) * nocc + max(o, o2)]; },
                                   [&](int o2, int c) { return C[sh.occ_list[o2] * n + c]; },
                                   [&](int o, int c, double v) { Mv[c * nocc + o] = 2.0 * v; });
        pprod<true, false, true>(sh, n, n, nocc, [&](int i, int o) { return C[sh.occ_list[o] * n + i]; },
                                 [&](int o, int c) { return Mv[c * nocc + o]; },
                                 [&](int i, int c, double v) { H[c * n + i] = v; });
        pprod<true, false, false>(sh, n, n, nocc, [&](int i, int o) { return C[sh.occ_list[o] * n + i]; },
                                  [&](int o, int c) { return C[sh.occ_list[o] * n + c]; },
                                  [&](int i, int c, double v) { P[c * n + i] = 2.0 * v; });
        if (!warm && j == 0 && nocc < n) {   // HOMO-LUMO gap of the last iteration
            double homo = -1e300, lumo = 1e300;
            for (int c = 0; c < n; ++c) {
                if (sh.occf[c]) homo = fmax(homo, sh.diag[c]); else lumo = fmin(lumo, sh.diag[c]);
            }
            if (!(lumo - homo > P_MIN_GAP)) sh.fl[0] |= ERRBIT_ZERO_GAP;
        }
        if (!warm) store_sorted();
        if (j < n) {   // band energy sum P H0, by column of the lower triangle
            double eb = 0.0;
            for (int i = j; i < n; ++i) eb = fma((i == j ? 1.0 : 2.0) * P[j * n + i], H0[j * n + i], eb);
            sh.red[j] = eb;
        }
        __syncthreads();
        const double *W = H;
        // pair tasks A <= B: d/dr_B of every image term (band, overlap, second order, repulsion), and
        // the repulsion energy (an atom with its own images counts each image pair once)
        for (int t = j; t < nat * (nat + 1) / 2; t += PT) {   // pairs A <= B, by kind
            int A, B;
                pbc_pair(sh, nat, t, A, B);
            const int eA = sh.spec[A], eB = sh.spec[B];
            const int oA = sh.atom_off[A], oB = sh.atom_off[B];
            const int na = sk.norb[eA], nb = sk.norb[eB];
            double d[3], f[3], dw[3];
            for (int k = 0; k < 3; ++k) d[k] = sh.pos[B][k] - sh.pos[A][k];
            for (int k = 0; k < 3; ++k) f[k] = rint(fma(d[0], pl.inv[k], fma(d[1], pl.inv[3 + k], d[2] * pl.inv[6 + k])));
            for (int k = 0; k < 3; ++k) dw[k] = d[k] - fma(f[0], pl.lat[k], fma(f[1], pl.lat[3 + k], f[2] * pl.lat[6 + k]));
            const double hshift = 0.5 * (sh.shift[A] + sh.shift[B]);
            const double qq = sh.dq[A] * sh.dq[B];
            const double c2 = sk.gamma_c2[eA][eB];
            const double rc2 = sk.r_cut * sk.r_cut;
            const double arep = sk.rep[eA][eB][0], brep = sk.rep[eA][eB][1];
            const double two_a_spi = 2.0 * pl.alpha * 0.5641895835477563;   // 2 alpha / sqrt(pi)
            double gk[3] = {0.0, 0.0, 0.0};
            double erep = 0.0;
            if (A != B) {
                pbc_images(pl, dw, pl.n_img, pl.r_real2, [&](int im) {   // real-space Ewald gradient
                    const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                    const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                    if (!(r2 < pl.r_real2) || r2 == 0.0) return;
                    const double ir = rsqrt_nr(r2);
                    const double ar = pl.alpha * (r2 * ir);
                    const double rad = -qq * (erfc(ar) * ir + two_a_spi * exp(-ar * ar)) * ir * ir;
                    gk[0] = fma(rad, x0, gk[0]);
                    gk[1] = fma(rad, x1, gk[1]);
                    gk[2] = fma(rad, x2, gk[2]);
                });
            }
            pbc_images(pl, dw, pl.n_img_sk, rc2, [&](int im) {   // images within r_cut
                const double x0 = dw[0] + pl.img[3 * im], x1 = dw[1] + pl.img[3 * im + 1], x2 = dw[2] + pl.img[3 * im + 2];
                const double r2 = fma(x0, x0, fma(x1, x1, x2 * x2));
                if (!(r2 < rc2) || r2 == 0.0) return;
                const double ir = rsqrt_nr(r2);
                const double r = r2 * ir;
                const double e[3] = {x0 * ir, x1 * ir, x2 * ir};
                double rad = 0.0;   // d/dr of the radial terms, along e
                {
                    double fc, dfc;
                    cutoff_fn(r, sk, fc, dfc);
                    if (arep != 0.0) {
                        const double vr = arep * exp(-brep * r);
                        erep = fma(vr, fc, erep);
                        if (A != B) rad = fma(vr, dfc - brep * fc, rad);
                    }
                    if (A != B) {
                        const double gi = rsqrt_nr(r2 + c2);
                        const double s_ = gi - ir;
                        const double ds = fma(-r * gi, gi * gi, ir * ir);
                        rad = fma(qq, fma(ds, fc, s_ * dfc), rad);
                        // band and overlap terms: weights P and P (eps_A + eps_B) / 2 - W of the block
                        double g[3] = {0.0, 0.0, 0.0};
                        for (int tb = 0; tb < 2; ++tb) {
                            const double(*tab)[CAVMD_MAX_ELEM][4][4] = tb == 0 ? sk.h0 : sk.s;
                            auto wt = [&](int mu, int nu) -> double {   // mu of A < nu of B: lower entry (nu, mu)
                                const double pv = P[mu * n + nu];
                                return tb == 0 ? pv : fma(pv, hshift, -W[mu * n + nu]);
                            };
                            double v, dv;
                            radial_p(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                            {
                                const double w = wt(oA, oB) * dv;
                                for (int k = 0; k < 3; ++k) g[k] = fma(w, e[k], g[k]);
                            }
                            if (nb == 4) {
                                radial_p(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                                double w[3], we = 0.0;
                                for (int i = 0; i < 3; ++i) { w[i] = wt(oA, oB + 1 + i); we = fma(w[i], e[i], we); }
                                for (int k = 0; k < 3; ++k) g[k] += fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                            }
                            if (na == 4) {
                                radial_p(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                                double w[3], we = 0.0;
                                for (int i = 0; i < 3; ++i) { w[i] = wt(oA + 1 + i, oB); we = fma(w[i], e[i], we); }
                                for (int k = 0; k < 3; ++k) g[k] -= fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                            }
                            if (na == 4 && nb == 4) {
                                double vs, dvs, vp, dvp;
                                radial_p(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dvs);
                                radial_p(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dvp);
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
                                    g[k] += (We[k] + WTe[k] - 2.0 * eWe * e[k]) * dl * ir + eWe * e[k] * ddl + tr * e[k] * dvp;
                            }
                        }
                        for (int k = 0; k < 3; ++k) gk[k] = fma(2.0, g[k], gk[k]);
                    }
                }
                for (int k = 0; k < 3; ++k) gk[k] = fma(rad, e[k], gk[k]);
            });
            double *pb = pbuf + 4LL * (A * nat + B);
            pb[0] = gk[0];
            pb[1] = gk[1];
            pb[2] = gk[2];
            pb[3] = A == B ? 0.5 * erep : erep;
        }
        __syncthreads();
    }
    if (rank > 0) {
        cluster_barrier(blocks);
        return;
    }
    // reciprocal part: d/dr_A of 1/2 sum_G w_G |S(G)|^2 = dq_A sum_G w_G G (c_A S_s - s_A S_c), the vectors in
    // contiguous shares as in p_shifts
    const int gparts = PT / nat;
    {
        const int part = j / nat, at = j - part * nat, per = (pl.n_g + gparts - 1) / gparts;
        if (part < gparts) {
            const int g1 = min(pl.n_g, (part + 1) * per);
            double gr[3] = {0.0, 0.0, 0.0};
            for (int g = part * per; g < g1; ++g) {
                const double *t = csg + 2LL * (g * nat + at);
                const double amp = pl.gw[4 * g + 3] * fma(t[0], sgf[2 * g + 1], -t[1] * sgf[2 * g]);
                for (int k = 0; k < 3; ++k) gr[k] = fma(amp, pl.gw[4 * g + k], gr[k]);
            }
            for (int k = 0; k < 3; ++k) sh.Xs[3 * j + k] = gr[k];
        }
        __syncthreads();
    }
    if (j < nat) {
        double gr[3] = {0.0, 0.0, 0.0};
        for (int q = 0; q < gparts; ++q)
            for (int k = 0; k < 3; ++k) gr[k] += sh.Xs[3 * (q * nat + j) + k];
        double G[3];
        for (int k = 0; k < 3; ++k) G[k] = sh.dq[j] * gr[k];
        for (int A = 0; A < nat; ++A) {
            if (A == j) continue;
            const double *pb = pbuf + 4LL * (A < j ? A * nat + j : j * nat + A);
            const double sg = A < j ? 1.0 : -1.0;
            for (int k = 0; k < 3; ++k) G[k] = fma(sg, pb[k], G[k]);
        }
        const int at = a0 + j;
        for (int k = 0; k < 3; ++k) a.F[3 * at + k] = -G[k];
        a.qprev[at] = a.have_warm ? sh.qst[j] : sh.q[j];
        a.qpop[at] = sh.q[j];
        if (a.Qout) a.Qout[at] = sh.zv[j] - sh.q[j];
        if (a.write_b) {
            const double Q = sh.zv[j] - sh.q[j];
            a.b[3 * at + 0] = Q * a.pol0;
            a.b[3 * at + 1] = Q * a.pol1;
            a.b[3 * at + 2] = Q * a.pol2;
        }
    }
    if (j == 0) {
        double E = 0.0;
        for (int i = 0; i < n; ++i) E += sh.red[i];
        double e2 = 0.0;
        for (int x = 0; x < nat; ++x) e2 = fma(sh.dq[x], sh.shift[x], e2);
        E = fma(0.5, e2, E);
        for (int A = 0; A < nat; ++A)
            for (int B = A; B < nat; ++B) E += pbuf[4LL * (A * nat + B) + 3];
        double mu[3] = {0.0, 0.0, 0.0};
        for (int at = 0; at < nat; ++at) {
            const double Q = sh.zv[at] - sh.q[at];
            for (int k = 0; k < 3; ++k) mu[k] = fma(Q, sh.pos[at][k] - sh.pos[0][k], mu[k]);
        }
        a.E_cell[cell] = E;
        a.M_cell[cell] = fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
        a.iters[cell] = sh.fl[2];
        if (sh.fl[0]) atomicOr(a.status, (unsigned)sh.fl[0]);
    }
    cluster_barrier(blocks);
}

// Items of a launch: the cells, or the finite-difference copies of every cell (rows per cell).
__device__ __forceinline__ int pbc_rows(const DftbArgs &a, const PbcDev &pl) {
    return a.n_disp > 0 ? (a.fd_central ? 6 : 3) * pl.amax : 1;
}

__device__ __forceinline__ bool pbc_item(const DftbArgs &a, int rows, long long it, int &cell, int &row) {
    cell = (int)(it / rows);
    row = a.n_disp > 0 ? (int)(it - (long long)cell * rows) : -1;
    return row < (a.fd_central ? 6 : 3) * (a.cell_offset[cell + 1] - a.cell_offset[cell]);
}

// The workspace of one cell's evaluation: first what its blocks share, then each block's own part.
__device__ __forceinline__ PbcMem pbc_mem(const PbcDev &pl, bool kg, long long group, int rank, int blocks) {
    PbcMem w;
    const long long n2 = (kg ? 4LL : 1LL) * pl.nmax * pl.nmax, nk = kg ? pl.nk : 1, a2 = (long long)pl.amax * pl.amax;
    double *p = pl.work + group * pl.work_stride;
    w.H0 = p;
    w.S = p + n2;
    p += 2 * nk * n2;
    w.kf = (float *)p;
    if (kg && !pl.lean) p += 2 * nk * n2;
    w.gam = p; p += a2;
    w.csg = p; p += 2LL * pl.amax * pl.n_g;
    w.Cd = p;
    if (!pl.lean) p += nk * n2;
    w.xch = p; p += 2LL * blocks * (pl.amax + 8);
    const long long own = 6 * n2 + 2LL * pl.n_g + 4 * a2 + (a2 + 1) / 2 + 6LL * pl.amax * (pl.g_max + 1) + 1;
    p += rank * own;
    w.H = p; w.Y = p + n2; w.P = p + 2 * n2; w.Xg = p + 3 * n2; w.Mo = p + 4 * n2; w.Mv = p + 5 * n2;
    p += 6 * n2;
    w.sgf = p; p += 2LL * pl.n_g;
    w.pbuf = p; p += 4 * a2;
    w.g32 = (float *)p; p += (a2 + 1) / 2;
    w.pw = p + ((size_t)p & 8 ? 1 : 0);   // pairs of doubles
    w.pbuf_stride = own;
    return w;
}

// k-grid sampling: one cell (or copy) at a time per cluster of pl.cluster blocks, each with its slice of
// the k-points. SH: the shared-memory struct, MB: blocks per SM (problems up to 256 wide leave room for two).
template <class SH, int MB>
__global__ void __launch_bounds__(PT, MB) k_dftb_periodic_kg(const DevSK *__restrict__ skp, const DftbArgs a, const PbcDev pl) {
    extern __shared__ __align__(16) unsigned char p_smem[];
    SH &sh = *reinterpret_cast<SH *>(p_smem);
    const int rank = pl.cluster > 1 ? (int)cluster_rank() : 0, group = blockIdx.x / pl.cluster;
    const PbcMem wk = pbc_mem(pl, true, group, rank, pl.cluster);
    const int rows = pbc_rows(a, pl);
    const long long items = pl.late_pass ? pl.late[0] : (long long)rows * a.n_cells;
    for (long long at = group; at < items; at += gridDim.x / pl.cluster) {
        const long long it = pl.late_pass ? pl.late[1 + at] : at;
        int cell, row;
        if (pbc_item(a, rows, it, cell, row)) p_cell<true>(*skp, a, pl, sh, wk, cell, row, rank, pl.cluster, (int)it);
    }
}

}  // namespace
