// Batched second-order SCC-DFTB of small molecules, one group of NORB lanes per molecule.
//
// The paper evaluates -grad V_n, mu_n and the Mulliken charges of every cell on the fly with
// SCC-DFTB (section "Computational details"; Eq. dpj needs -grad V_n). This kernel evaluates
// many independent cells of one composition at once:
//
//   H0, S from Slater-Koster tables  ->  warm-started S-orthonormal basis C (Cholesky of C^T S C)
//   -> SCC loop: shifts eps_A = sum_B gamma_AB dq_B, H = H0 + 1/2 S o (eps_A + eps_B),
//      A = C^T H C, cyclic Jacobi on A (rotations applied to A and C), aufbau occupation,
//      P = 2 C_occ C_occ^T, Mulliken populations, Anderson-accelerated mixing
//   -> energy, analytic gradient (P dH0 + (P (eps_A+eps_B)/2 - W) dS + dgamma + dE_rep),
//      dipole M_n = pol . sum_A Q_A r_A and the Mulliken dipole derivative b_A = Q_A pol.
//
// Layout: lane j of a group owns column j of every NORB x NORB matrix, stored column-major in
// the group's shared-memory slot with an odd leading dimension. All groups of a warp advance in
// lock step (__syncwarp); a group whose charges have converged idles until the slowest group
// of its warp is done. The FP64 pipe bounds this kernel on GB300, so auxiliary quantities that
// only steer the iteration (rotation angles, mixing coefficients, convergence tests) are formed
// in FP32 or by integer comparisons, while every quantity that enters the result (rotations
// themselves, matrices, populations, energies, forces) is computed in FP64.
#include "cavmd_internal.cuh"

namespace {

constexpr int NHIST = 3;          // Anderson history (current + 2 previous iterates)
constexpr int MAX_SWEEPS = 24;    // default bound on the Jacobi sweeps of a cold start
constexpr double JACOBI_TOL = 1e-15;   // off-diagonal magnitude treated as converged (Hartree)
constexpr double MIN_GAP = 1e-3;       // closed-shell HOMO-LUMO threshold (Hartree)
constexpr double EIG_TOL = 1e-10;      // occupied-virtual coupling treated as converged (Hartree)
constexpr float KMAX_PERT = 1e-4f;     // largest generator entry for the second-order update
constexpr int W_FP32_ITERS = 6;         // warm waters: bound on the FP32 Newton steps,
constexpr float W_FP32_KTOL = 1e-6f;    // the rotation at which they stop (FP32 rounding moves C by as much),
constexpr float W_ROT_MAX = 0.3f;       // the largest rotation taken (beyond: the general solve)
constexpr int W_EVALS = 8;              // and bound on the FP64 evaluations
constexpr float W_ORTH_MAX = 3e-2f;     // norm of the overlap defect that the FP64 correction takes,
constexpr float W_ORTH_ONCE = 5e-4f;    // above which it is repeated
constexpr float W_ORTH_CUBE = 2e-5f;    // and above which its cubic term counts
constexpr float W_ROT64_MAX = 1e-2f;    // norm of a rotation between FP64 evaluations,
constexpr float W_ROT64_ONCE = 3e-4f;   // and above which the correction follows it
constexpr float W_GAP = 2e-3f;          // HOMO-LUMO gap (Hartree) the warm path needs, above MIN_GAP

// Scratch of one water in the warm path (k_water_warm). Matrices are row-major: the lane of orbital
// i owns row i and reads the others' rows as broadcasts.
struct __align__(16) WarmScratch {
    double C[36];       // basis, occupied columns first
    double X[36];       // S C, then H C_occ
    double E[22];       // overlap defects; later C_occ^T H C_occ and its product with the H rows of C
    double PW[18];      // density and energy-weighted density of the 9 interatomic entries
    double pop[6];      // orbital populations
    float Cf[6][8], Mf[6][8];   // FP32 basis; the column exchanged by a reduction
    float B[16];        // Mulliken charge response of the two hydrogens, [atom][virtual][occupied]
    float L[36];        // Cholesky factor of the orbital Hessian, rows of the lower triangle
    float av[8];        // occupied-virtual residual
    float popf[8];
};

template <int NAT, int NORB>
struct __align__(16) MolShared {
    static constexpr int LD = (NORB % 2 == 0) ? NORB + 1 : NORB;   // odd column stride
    static constexpr int NPAIR = NAT * (NAT - 1) / 2;
    double S[NORB * LD];
    double H0[NORB * LD];
    union {   // the general solve's matrices, or the warm water path's scratch
        struct {
            double A[NORB * LD];
            double C[NORB * LD];
            double Y[NORB * LD];
            double P[NORB * LD];
            double Hs[NORB * LD];   // H of the current SCC iteration
        };
        WarmScratch w;
    };
    double pos[NAT][3];
    double gam[NAT][NAT];
    double zv[NAT];
    double q[NAT];
    double qout[NAT];
    double shift[NAT];
    double hq[NHIST][NAT];
    double hf[NHIST][NAT];
    double qstart[NAT];   // q(t) of the previous step, for the predictor
    double red[NORB];
    double cs[NORB / 2 + 1][2];
    double invd[NORB];
    double hsh[NORB];     // half shift of the atom of each orbital
    float diagf[NORB];    // diagonal of A in FP32 (generator denominators)
    double gpair[NPAIR > 0 ? NPAIR : 1][3];
    double gpart[2][NPAIR > 0 ? NPAIR : 1][3];   // H0 and S parts of the pair gradients
    double epair[NPAIR > 0 ? NPAIR : 1];
    int occ_list[NORB];
    int virt_list[NORB];
    int occf[NORB];       // orbital column j is occupied
    int eok[NORB];        // occupied-virtual couplings of column j were below EIG_TOL
    int orb_atom[NORB];
    int atom_off[NAT + 1];
    int spec[NAT];
    int pa[NPAIR > 0 ? NPAIR : 1];
    int pb[NPAIR > 0 ? NPAIR : 1];
    int flag;
    int conv;
    int iters;
    int nocc;
};

__device__ __forceinline__ void radial(const double *par, double r, const DevSK &sk, double &v,
                                       double &dv) {
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

// Jacobi round-robin schedule for even n: in round r (0..n-2) index n-1 meets r and index j
// meets (2r - j) mod (n-1). Returns the partner of j and the pair slot (0 = the pair with n-1).
__device__ __forceinline__ int rr_partner(int j, int r, int n, int &slot) {
    const int m = n - 1;
    if (j == m) { slot = 0; return r; }
    if (j == r) { slot = 0; return m; }
    const int dlt = (j - r + m) % m;
    slot = min(dlt, m - dlt);
    return (r - dlt + m) % m;
}

__device__ __forceinline__ void rr_pair(int k, int r, int n, int &p, int &q) {
    const int m = n - 1;
    if (k == 0) { p = r; q = m; return; }
    const int x = (r + k) % m, y = (r - k + m) % m;
    p = min(x, y);
    q = max(x, y);
}

// Rotation (c, s) that annihilates a_pq: tan(phi) = t from the FP32 quadratic, then (c, s) made
// orthonormal in FP64 by two Newton steps on 1/sqrt(c^2 + s^2).
__device__ __forceinline__ void jacobi_cs(double app, double aqq, double apq, double &c, double &s) {
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

// The general SCC solve of the molecules of a warp that have not converged yet (m.conv = 0): the
// S-orthonormal basis (warm: the previous eigenvectors; cold: Cholesky of S), then the SCC loop.
// Leaves the basis in m.C, the occupation in occ_list and occf, the populations in m.q and the last
// iteration's H in m.Hs; sets m.conv, m.iters and the error bits of m.flag.
template <int NAT, int NORB>
__device__ __forceinline__ void scc_general(const DftbArgs &a, MolShared<NAT, NORB> &m, const bool lane_act,
                                            const int j, const int cell, const int a0, const bool disp) {
    constexpr int LD = MolShared<NAT, NORB>::LD;
    const bool act = lane_act && !m.conv;   // a molecule that is done keeps its state
    __syncwarp();
    // ---------------------------------------------------------------- warm-started S-orthonormal basis
    if (act) {
        if (a.have_warm) {
            const double *cw = a.Cwarm + (a.Cwarm_off ? a.Cwarm_off[cell] : (long long)cell * NORB * NORB);
            for (int i = 0; i < NORB; ++i) m.C[j * LD + i] = cw[j * NORB + i];
            // linear predictor 2 q(t) - q(t - dt) of the populations (q_prev equals q after a
            // cold start, so the first warm step starts from q(t) itself)
            if (j < NAT) {
                const double qt = a.qpop[a0 + j];
                m.qstart[j] = qt;
                m.q[j] = disp ? qt : fma(2.0, qt, -a.qprev[a0 + j]);   // displaced rows start at q(r)
            }
        } else {
            for (int i = 0; i < NORB; ++i) m.C[j * LD + i] = (i == j) ? 1.0 : 0.0;
            if (j < NAT) m.q[j] = m.zv[j];
        }
    }
    __syncwarp();
    // G = C^T S C  (in A)
    if (act) {
        if (a.have_warm) {
            double y[NORB];
#pragma unroll
            for (int i = 0; i < NORB; ++i) y[i] = 0.0;
            for (int k = 0; k < NORB; ++k) {
                const double ckj = m.C[j * LD + k];
#pragma unroll
                for (int i = 0; i < NORB; ++i) y[i] = fma(m.S[k * LD + i], ckj, y[i]);
            }
#pragma unroll
            for (int i = 0; i < NORB; ++i) m.Y[j * LD + i] = y[i];
        }
    }
    __syncwarp();
    if (act) {
        if (a.have_warm) {
            for (int i = 0; i < NORB; ++i) {
                double s = 0.0;
#pragma unroll
                for (int k = 0; k < NORB; ++k) s = fma(m.C[i * LD + k], m.Y[j * LD + k], s);
                m.A[j * LD + i] = s;
            }
        } else {
            for (int i = 0; i < NORB; ++i) m.A[j * LD + i] = m.S[j * LD + i];
        }
    }
    __syncwarp();
    // Cholesky G = L L^T, right-looking, lane = column (L in the lower triangle of A)
    for (int k = 0; k < NORB; ++k) {
        if (act && j == k) {
            double d = m.A[k * LD + k];
            if (!(d > 1e-300)) {
                m.flag |= ERRBIT_S_NOT_PD;
                d = 1.0;
            }
            const double y = rsqrt_nr(d);
            m.invd[k] = y;
            m.A[k * LD + k] = d * y;
            for (int i = k + 1; i < NORB; ++i) m.A[k * LD + i] *= y;
        }
        __syncwarp();
        if (act && j > k) {
            const double ljk = m.A[k * LD + j];
            for (int i = j; i < NORB; ++i) m.A[j * LD + i] = fma(-m.A[k * LD + i], ljk, m.A[j * LD + i]);
        }
        __syncwarp();
    }
    // C <- C L^-T (lane = row)
    if (act) {
        const int i = j;
        for (int c = 0; c < NORB; ++c) {
            double x = m.C[c * LD + i];
            for (int k = 0; k < c; ++k) x = fma(-m.C[k * LD + i], m.A[k * LD + c], x);
            m.C[c * LD + i] = x * m.invd[c];
        }
    }
    __syncwarp();

    // ---------------------------------------------------------------- SCC loop
    // Each iteration builds H(q) and A = C^T H C in the current S-orthonormal basis C and moves C
    // towards the eigenvectors of H. When the occupied-virtual couplings are small, C takes the
    // second-order exponential V = I + K + K^2/2 of the first-order generator
    // K_kj = A_kj / (A_jj - A_kk) over occupied-virtual pairs: V is orthogonal to O(K^4) and, like
    // a Jacobi sweep, squares the remaining coupling, at a third of the cost. Otherwise (the first
    // iteration after a geometry change, a cold start, a large charge change) C takes Jacobi
    // sweeps: one per iteration when warm started, to full convergence in the first iteration of a
    // cold start. Only occupied-virtual mixing changes P, so occupied-occupied couplings are left
    // to the final energy-weighted density, which uses the whole occupied block. The charges count
    // as converged once |q_out - q| < tol and every occupied-virtual coupling was below EIG_TOL
    // before the update.
    int it = 0;
    for (it = 1; it <= a.max_iter; ++it) {
        const bool work = act && !m.conv;
        if (work && j < NAT) {
            double sh = 0.0;
            for (int k = 0; k < NAT; ++k) sh = fma(m.gam[j][k], m.q[k] - m.zv[k], sh);
            m.shift[j] = sh;
        }
        __syncwarp();
        if (work) m.hsh[j] = 0.5 * m.shift[m.orb_atom[j]];
        __syncwarp();
        if (work) {   // H column j: H0 + S o (eps_A + eps_B)/2 (halving is exact, so this equals the
                      // product with the halved sum bit for bit)
            const double hj = m.hsh[j];
            for (int i = 0; i < NORB; ++i)
                m.Hs[j * LD + i] = fma(m.S[j * LD + i], m.hsh[i] + hj, m.H0[j * LD + i]);
        }
        __syncwarp();
        if (work) {   // Y = H C
            double y[NORB];
#pragma unroll
            for (int i = 0; i < NORB; ++i) y[i] = 0.0;
            for (int k = 0; k < NORB; ++k) {
                const double ckj = m.C[j * LD + k];
#pragma unroll
                for (int i = 0; i < NORB; ++i) y[i] = fma(m.Hs[k * LD + i], ckj, y[i]);
            }
#pragma unroll
            for (int i = 0; i < NORB; ++i) m.Y[j * LD + i] = y[i];
        }
        __syncwarp();
        // A = C^T H C = C^T Y is formed only where the iteration needs it: its diagonal (aufbau,
        // denominators) and its occupied-virtual block (generator, convergence), the latter as
        // (occupied, virtual) pair tasks spread over the lanes and stored symmetric. The Jacobi
        // path adds the other entries when it runs.
        if (work) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < NORB; ++k) s = fma(m.C[j * LD + k], m.Y[j * LD + k], s);
            m.A[j * LD + j] = s;
        }
        __syncwarp();
        // aufbau occupation from the diagonal of A
        if (work) {
            m.diagf[j] = d2f_steer(m.A[j * LD + j]);
            const long long kj = order_key(m.A[j * LD + j]);
            int rank = 0;
            for (int i = 0; i < NORB; ++i) {
                const long long ki = order_key(m.A[i * LD + i]);
                rank += (ki < kj) || (ki == kj && i < j);
            }
            m.occf[j] = rank < m.nocc;
            if (rank < m.nocc) m.occ_list[rank] = j;
            else m.virt_list[rank - m.nocc] = j;
        }
        __syncwarp();
        if (work) {   // occupied-virtual block
            const int nv = NORB - m.nocc;
            for (int t = j; t < m.nocc * nv; t += NORB) {
                const int oi = t / nv;
                const int o = m.occ_list[oi], v = m.virt_list[t - oi * nv];
                double s = 0.0;
#pragma unroll
                for (int k = 0; k < NORB; ++k) s = fma(m.C[v * LD + k], m.Y[o * LD + k], s);
                m.A[o * LD + v] = s;
                m.A[v * LD + o] = s;
            }
        }
        __syncwarp();
        // first-order occupied-virtual generator, column j, into Y (FP32: it only steers)
        // Only the entries of the other block (virtual rows of an occupied column, and conversely)
        // are non-zero; the loop visits just those.
        float kmax = 0.0f;
        unsigned same_mask = 0u, other_mask = 0u;
        if (work) {
            unsigned om = 0u;
#pragma unroll
            for (int k = 0; k < NORB; ++k) om |= (m.occf[k] ? 1u : 0u) << k;
            same_mask = m.occf[j] ? om : (~om & ((1u << NORB) - 1u));
            other_mask = ~same_mask & ((1u << NORB) - 1u);
#pragma unroll
            for (int k = 0; k < NORB; ++k) m.P[j * LD + k] = 0.0;   // K column j (P is free until the density)
            const float dj = m.diagf[j];
            bool small = true;
            for (unsigned om = other_mask; om; om &= om - 1u) {
                const int k = __ffs(om) - 1;
                const double akj = m.A[j * LD + k];
                if (!abs_lt(akj, EIG_TOL)) small = false;
                float kf = d2f_steer(akj) / (dj - m.diagf[k]);
                if (!(fabsf(kf) <= 1e30f)) kf = 1e30f;   // degenerate or non-finite: Jacobi path
                m.P[j * LD + k] = f2d_steer(kf);
                kmax = fmaxf(kmax, fabsf(kf));
            }
            m.eok[j] = small;
        }
        const bool cold_first = !a.have_warm && it == 1;
        const bool perturb = __all_sync(CAVMD_FULL_MASK, !work || (kmax < KMAX_PERT && !cold_first));
        __syncwarp();
        if (perturb) {
            double cn[NORB];
            if (work) {   // V column j = e_j + K e_j + K (K e_j) / 2, then C <- C V
                // (K^2)(i, j) vanishes for rows i of the other block; for rows of j's own block it sums
                // over the other block only: n_occ n_virt products per column, in increasing index
                // order (the skipped terms are exact zeros). The row sums go to A, free here.
                for (unsigned sm = same_mask; sm; sm &= sm - 1u) {
                    const int i = __ffs(sm) - 1;
                    double acc = 0.0;
                    for (unsigned om = other_mask; om; om &= om - 1u) {
                        const int mm = __ffs(om) - 1;
                        acc = fma(m.P[mm * LD + i], m.P[j * LD + mm], acc);
                    }
                    m.A[j * LD + i] = acc;
                }
                // (K + K^2 / 2) e_j; the identity part of V is C's own column, the start of C V
                double v[NORB];
#pragma unroll
                for (int i = 0; i < NORB; ++i)
                    v[i] = fma(0.5, ((same_mask >> i) & 1u) ? m.A[j * LD + i] : 0.0, m.P[j * LD + i]);
#pragma unroll
                for (int i = 0; i < NORB; ++i) cn[i] = m.C[j * LD + i];
                for (int k = 0; k < NORB; ++k) {
                    const double vk = v[k];
#pragma unroll
                    for (int i = 0; i < NORB; ++i) cn[i] = fma(m.C[k * LD + i], vk, cn[i]);
                }
            }
            __syncwarp();
            if (work) {
#pragma unroll
                for (int i = 0; i < NORB; ++i) m.C[j * LD + i] = cn[i];
            }
            __syncwarp();
        } else {
            // the sweeps need all of A: add the off-diagonal entries inside the occupied and the
            // virtual blocks (Y still holds H C), one (a, b) pair per task, stored symmetric
            if (work) {
                for (int t = j; t < NORB * (NORB - 1) / 2; t += NORB) {
                    int pa_ = 0, rem = t;
                    while (rem >= NORB - 1 - pa_) {
                        rem -= NORB - 1 - pa_;
                        ++pa_;
                    }
                    const int pb_ = pa_ + 1 + rem;
                    if (m.occf[pa_] == m.occf[pb_]) {
                        double s = 0.0;
#pragma unroll
                        for (int k = 0; k < NORB; ++k) s = fma(m.C[pa_ * LD + k], m.Y[pb_ * LD + k], s);
                        m.A[pb_ * LD + pa_] = s;
                        m.A[pa_ * LD + pb_] = s;
                    }
                }
            }
            __syncwarp();
            // a cold start sweeps until the off-diagonal entries are below tolerance, at most `cap`
            // sweeps (then DEVICE_TIMEOUT); later iterations take one sweep
            const int cap = cold_first ? (a.max_sweeps > 0 ? a.max_sweeps : MAX_SWEEPS) : 1;
            for (int sweep = 0;; ++sweep) {
                bool small = true;
                if (work) {
                    for (int i = 0; i < NORB; ++i)
                        if (i != j && !abs_lt(m.A[j * LD + i], JACOBI_TOL)) small = false;
                }
                if (__all_sync(CAVMD_FULL_MASK, small)) break;
                if (sweep >= cap) {
                    if (cold_first && work && !small) m.flag |= ERRBIT_TIMEOUT;
                    break;
                }
                for (int rd = 0; rd < NORB - 1; ++rd) {
                    int slot = 0;
                    const int pj = rr_partner(j, rd, NORB, slot);
                    const int p = min(j, pj), q = max(j, pj);
                    double c = 1.0, s = 0.0;
                    double na[NORB], nc[NORB];
                    if (work) {
                        jacobi_cs(m.A[p * LD + p], m.A[q * LD + q], m.A[q * LD + p], c, s);
                        const double cp = (j == p) ? c : s;       // new col j = cp * col p + cq * col q
                        const double cq = (j == p) ? -s : c;
#pragma unroll
                        for (int i = 0; i < NORB; ++i) {
                            na[i] = fma(cp, m.A[p * LD + i], cq * m.A[q * LD + i]);
                            nc[i] = fma(cp, m.C[p * LD + i], cq * m.C[q * LD + i]);
                        }
                    }
                    __syncwarp();
                    if (work) {
#pragma unroll
                        for (int i = 0; i < NORB; ++i) {
                            m.A[j * LD + i] = na[i];
                            m.C[j * LD + i] = nc[i];
                        }
                        if (j == p) {
                            m.cs[slot][0] = c;
                            m.cs[slot][1] = s;
                        }
                    }
                    __syncwarp();
                    if (work) {
#pragma unroll
                        for (int k = 0; k < NORB / 2; ++k) {
                            int pk, qk;
                            rr_pair(k, rd, NORB, pk, qk);
                            const double ck = m.cs[k][0], sk_ = m.cs[k][1];
                            const double x = m.A[j * LD + pk], y = m.A[j * LD + qk];
                            m.A[j * LD + pk] = fma(ck, x, -sk_ * y);
                            m.A[j * LD + qk] = fma(sk_, x, ck * y);
                        }
                    }
                    __syncwarp();
                }
            }
            if (work) {   // occupation after the sweeps
                const long long kj = order_key(m.A[j * LD + j]);
                int rank = 0;
                for (int i = 0; i < NORB; ++i) {
                    const long long ki = order_key(m.A[i * LD + i]);
                    rank += (ki < kj) || (ki == kj && i < j);
                }
                m.occf[j] = rank < m.nocc;
                if (rank < m.nocc) m.occ_list[rank] = j;
            }
            __syncwarp();
        }

        if (work) {   // P = 2 C_occ C_occ^T, column j, and (P S)_jj
            double pc[NORB];
#pragma unroll
            for (int i = 0; i < NORB; ++i) pc[i] = 0.0;
            for (int o = 0; o < m.nocc; ++o) {
                const int col = m.occ_list[o];
                const double w = 2.0 * m.C[col * LD + j];
#pragma unroll
                for (int i = 0; i < NORB; ++i) pc[i] = fma(w, m.C[col * LD + i], pc[i]);
            }
            double qo = 0.0;
#pragma unroll
            for (int i = 0; i < NORB; ++i) {
                m.P[j * LD + i] = pc[i];
                qo = fma(pc[i], m.S[j * LD + i], qo);
            }
            m.red[j] = qo;
        }
        __syncwarp();
        const int hs = (it - 1) % NHIST;
        if (work && j < NAT) {
            double qa = 0.0;
            for (int o = m.atom_off[j]; o < m.atom_off[j + 1]; ++o) qa += m.red[o];
            m.qout[j] = qa;
            m.hq[hs][j] = m.q[j];
            m.hf[hs][j] = qa - m.q[j];
        }
        __syncwarp();
        if (work) {
            // convergence test and Anderson coefficients (FP32: they only steer the iteration)
            bool conv = true;
            for (int at = 0; at < NAT; ++at)
                if (!abs_lt(m.hf[hs][at], a.scc_tol)) conv = false;
            for (int c = 0; c < NORB; ++c) conv = conv && m.eok[c];
            float th1 = 0.0f, th2 = 0.0f;
            const int h = min(it, NHIST);
            if (!conv && h >= 2) {
                const int h1 = (hs + NHIST - 1) % NHIST, h2 = (hs + NHIST - 2) % NHIST;
                float a11 = 0.f, a12 = 0.f, a22 = 0.f, b1 = 0.f, b2 = 0.f;
                for (int at = 0; at < NAT; ++at) {
                    const float f0 = d2f_steer(m.hf[hs][at]);
                    const float d1 = d2f_steer(m.hf[h1][at]) - f0;
                    const float d2 = h >= 3 ? d2f_steer(m.hf[h2][at]) - f0 : 0.f;
                    a11 = fmaf(d1, d1, a11);
                    a12 = fmaf(d1, d2, a12);
                    a22 = fmaf(d2, d2, a22);
                    b1 = fmaf(-d1, f0, b1);
                    b2 = fmaf(-d2, f0, b2);
                }
                const float det = a11 * a22 - a12 * a12;
                if (h >= 3 && det > 1e-6f * a11 * a22 && det > 0.f) {
                    th1 = (b1 * a22 - b2 * a12) / det;
                    th2 = (a11 * b2 - a12 * b1) / det;
                } else if (a11 > 0.f) {
                    th1 = b1 / a11;
                }
                if (!(fabsf(th1) < 50.f) || !(fabsf(th2) < 50.f)) { th1 = 0.f; th2 = 0.f; }
            }
            if (j < NAT) {
                if (conv) {
                    m.q[j] = m.qout[j];
                } else {
                    const int h1 = (hs + NHIST - 1) % NHIST, h2 = (hs + NHIST - 2) % NHIST;
                    const double t1 = f2d_steer(th1), t2 = f2d_steer(th2);
                    const double q0 = m.hq[hs][j], f0 = m.hf[hs][j];
                    double qb = q0, fb = f0;
                    if (h >= 2) { qb = fma(t1, m.hq[h1][j] - q0, qb); fb = fma(t1, m.hf[h1][j] - f0, fb); }
                    if (h >= 3) { qb = fma(t2, m.hq[h2][j] - q0, qb); fb = fma(t2, m.hf[h2][j] - f0, fb); }
                    m.q[j] = fma(a.beta, fb, qb);
                }
            }
            if (j == 0 && conv) {
                m.conv = 1;
                m.iters = it;
            }
        }
        __syncwarp();
        if (__all_sync(CAVMD_FULL_MASK, !act || m.conv)) break;
    }
    if (act && j == 0 && !m.conv) {
        m.flag |= ERRBIT_SCC_NOCONV;
        m.iters = a.max_iter;
    }
    __syncwarp();
}

template <int NAT, int NORB>
__global__ void __launch_bounds__(256, 1) dftb_kernel(const DevSK *__restrict__ skp, const DftbArgs a, const int gpw) {
    const DevSK &sk = *skp;
    using SM = MolShared<NAT, NORB>;
    constexpr int LD = SM::LD;
    // gpw <= 32 / NORB molecules per warp (fewer spreads a small batch over more warps)
    constexpr int NPAIR = SM::NPAIR;
    extern __shared__ __align__(16) unsigned char smem_raw[];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    const int g = lane / NORB;
    const int j = lane - g * NORB;
    const bool act = g < gpw;
    SM &m = reinterpret_cast<SM *>(smem_raw)[warp * gpw + (act ? g : 0)];
    const bool disp = a.n_disp > 0;                       // finite-difference rows
    const int n_rows = disp ? a.n_cells * a.n_disp : a.n_cells;
    const int idx = (blockIdx.x * wpb + warp) * gpw + g;
    const bool valid = act && idx < n_rows;
    const int ridx = min(idx, n_rows - 1);
    const int cidx = disp ? ridx / a.n_disp : ridx;
    const int cell = a.cell_list ? a.cell_list[cidx] : cidx;
    const int a0 = a.cell_offset[cell];

    // ---------------------------------------------------------------- load geometry, layout
    const bool open = a.E_open != nullptr && !disp;
    double p_new[3], r_new[3];
    if (act && j < NAT) {
        m.spec[j] = a.species[a0 + j];
        m.pos[j][0] = a.r[3 * (a0 + j) + 0];
        m.pos[j][1] = a.r[3 * (a0 + j) + 1];
        m.pos[j][2] = a.r[3 * (a0 + j) + 2];
        if (open) {   // opening half-flow: kick by tau F + E_n b, then drift (stored after the warp sync)
            const int at = a0 + j;
            const double e1 = a.E_open[cell], im = a.inv_mass[at];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                p_new[k] = fma(a.tau, a.F[3 * at + k], fma(e1, a.b[3 * at + k], a.p_open[3 * at + k]));
                r_new[k] = fma(a.dt * im, p_new[k], m.pos[j][k]);
                m.pos[j][k] = r_new[k];
            }
        }
        if (disp) {   // displaced copy: atom da, component dc, by +h (forward) or +-h (central)
            const int k = ridx - cidx * a.n_disp;
            const int kk = a.fd_central ? k >> 1 : k;
            const int da = kk / 3, dc = kk - 3 * (kk / 3);
            const double sg = (a.fd_central && (k & 1)) ? -1.0 : 1.0;
            if (j == da) m.pos[j][dc] += sg * a.fd_h;
        }
    }
    __syncwarp();   // every lane of the warp has read the state it kicks before any is stored
    if (open && valid && j < NAT) {
        const int at = a0 + j;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.p_open[3 * at + k] = p_new[k];
            a.r_open[3 * at + k] = r_new[k];
        }
    }
    if (act && j == 0) {
        int o = 0;
        double nel = 0.0;
        for (int at = 0; at < NAT; ++at) {
            m.atom_off[at] = o;
            const int no = sk.norb[m.spec[at]];
            for (int k = 0; k < no; ++k) m.orb_atom[o + k] = at;
            o += no;
            m.zv[at] = sk.zval[m.spec[at]];
            nel += m.zv[at];
        }
        m.atom_off[NAT] = o;
        m.nocc = (int)(nel * 0.5f + 0.25f);
        int pi = 0;
        for (int x = 0; x < NAT; ++x)
            for (int y = x + 1; y < NAT; ++y) { m.pa[pi] = x; m.pb[pi] = y; ++pi; }
        m.flag = 0;
        m.conv = 0;
        m.iters = 0;
    }
    __syncwarp();

    // ---------------------------------------------------------------- H0, S, gamma
    if (act) {
        const int at = m.orb_atom[j];
        const int e = m.spec[at];
        const double eps = (j == m.atom_off[at]) ? sk.onsite[e][0] : sk.onsite[e][1];
        for (int i = 0; i < NORB; ++i) {
            m.S[j * LD + i] = (i == j) ? 1.0 : 0.0;
            m.H0[j * LD + i] = (i == j) ? eps : 0.0;
        }
    }
    __syncwarp();
    if (act) {
        // one (pair, table) task per lane: the H0 and the S integrals of a pair on two lanes
        for (int task = j; task < 2 * NPAIR; task += NORB) {
            const int pi = task % NPAIR, t = task / NPAIR;
            const int A = m.pa[pi], B = m.pb[pi];
            const int eA = m.spec[A], eB = m.spec[B];
            const int oA = m.atom_off[A], oB = m.atom_off[B];
            const int na = sk.norb[eA], nb = sk.norb[eB];
            const double dx = m.pos[B][0] - m.pos[A][0];
            const double dy = m.pos[B][1] - m.pos[A][1];
            const double dz = m.pos[B][2] - m.pos[A][2];
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const double ir = rsqrt_nr(r2);
            const double r = r2 * ir;
            const double ev[3] = {dx * ir, dy * ir, dz * ir};
            {
                const double (*tab)[CAVMD_MAX_ELEM][4][4] = t == 0 ? sk.h0 : sk.s;
                double *X = t == 0 ? m.H0 : m.S;
                double v, dv;
                radial(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                X[oB * LD + oA] = v;
                X[oA * LD + oB] = v;
                if (nb == 4) {
                    radial(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                    for (int i = 0; i < 3; ++i) {
                        X[(oB + 1 + i) * LD + oA] = ev[i] * v;
                        X[oA * LD + oB + 1 + i] = ev[i] * v;
                    }
                }
                if (na == 4) {
                    radial(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                    for (int i = 0; i < 3; ++i) {
                        X[oB * LD + oA + 1 + i] = -ev[i] * v;
                        X[(oA + 1 + i) * LD + oB] = -ev[i] * v;
                    }
                }
                if (na == 4 && nb == 4) {
                    double vs, vp;
                    radial(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dv);
                    radial(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dv);
                    const double dl = vs - vp;
                    for (int i = 0; i < 3; ++i)
                        for (int k = 0; k < 3; ++k) {
                            const double val = fma(ev[i] * ev[k], dl, (i == k) ? vp : 0.0);
                            X[(oB + 1 + k) * LD + oA + 1 + i] = val;
                            X[(oA + 1 + i) * LD + oB + 1 + k] = val;
                        }
                }
            }
        }
        if (j < NAT) {
            for (int k = 0; k < NAT; ++k) {
                if (k == j) {
                    m.gam[j][k] = sk.hubbard[m.spec[j]];
                } else {
                    const double dx = m.pos[k][0] - m.pos[j][0];
                    const double dy = m.pos[k][1] - m.pos[j][1];
                    const double dz = m.pos[k][2] - m.pos[j][2];
                    m.gam[j][k] = rsqrt_nr(fma(dx, dx, fma(dy, dy, fma(dz, dz, sk.gamma_c2[m.spec[j]][m.spec[k]]))));
                }
            }
        }
    }
    __syncwarp();

    scc_general<NAT, NORB>(a, m, act, j, cell, a0, disp);

    if (disp) {   // finite-difference row: only the dipole of the converged charges
        if (valid && j == 0) {
            double mu[3] = {0.0, 0.0, 0.0};
            for (int at = 0; at < NAT; ++at) {
                const double Q = m.zv[at] - m.q[at];
                for (int k = 0; k < 3; ++k) mu[k] = fma(Q, m.pos[at][k] - m.pos[0][k], mu[k]);
            }
            a.M_disp[(long long)(a.fd_central ? 6 : 3) * a0 + (ridx - cidx * a.n_disp)] =
                fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
            if (m.flag) atomicOr(a.status, (unsigned)m.flag);
        }
        return;
    }
    // ---------------------------------------------------------------- energy, forces, dipole
    if (act && j < NAT) {
        double sh = 0.0;
        for (int k = 0; k < NAT; ++k) sh = fma(m.gam[j][k], m.q[k] - m.zv[k], sh);
        m.shift[j] = sh;
    }
    __syncwarp();
    // energy-weighted density W = 2 C_o (C_o^T H C_o) C_o^T with the H of the last iteration and the
    // whole occupied block (basis independent inside the occupied subspace)
    if (act) {   // Y = H C
        double y[NORB];
#pragma unroll
        for (int i = 0; i < NORB; ++i) y[i] = 0.0;
        for (int k = 0; k < NORB; ++k) {
            const double ckj = m.C[j * LD + k];
#pragma unroll
            for (int i = 0; i < NORB; ++i) y[i] = fma(m.Hs[k * LD + i], ckj, y[i]);
        }
#pragma unroll
        for (int i = 0; i < NORB; ++i) m.Y[j * LD + i] = y[i];
    }
    __syncwarp();
    if (act) {   // A = C^T Y
        double y[NORB];
        for (int i = 0; i < NORB; ++i) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < NORB; ++k) s = fma(m.C[i * LD + k], m.Y[j * LD + k], s);
            y[i] = s;
        }
        for (int i = 0; i < NORB; ++i) m.A[j * LD + i] = y[i];
    }
    __syncwarp();
    if (act) {   // W column j, band energy partial, HOMO-LUMO gap
        double t[NORB];
        for (int o = 0; o < m.nocc; ++o) {
            const int co = m.occ_list[o];
            double x = 0.0;
            for (int o2 = 0; o2 < m.nocc; ++o2) {
                const int c2 = m.occ_list[o2];
                x = fma(m.A[c2 * LD + co], m.C[c2 * LD + j], x);
            }
            t[o] = 2.0 * x;
        }
        double wc[NORB];
#pragma unroll
        for (int i = 0; i < NORB; ++i) wc[i] = 0.0;
        for (int o = 0; o < m.nocc; ++o) {
            const int co = m.occ_list[o];
            const double w = t[o];
#pragma unroll
            for (int i = 0; i < NORB; ++i) wc[i] = fma(w, m.C[co * LD + i], wc[i]);
        }
        double eb = 0.0;
#pragma unroll
        for (int i = 0; i < NORB; ++i) {
            m.Y[j * LD + i] = wc[i];
            eb = fma(m.P[j * LD + i], m.H0[j * LD + i], eb);
        }
        m.red[j] = eb;
        if (j == 0 && m.nocc < NORB) {
            double homo = -1e300, lumo = 1e300;
            for (int i = 0; i < NORB; ++i) {
                const double ei = m.A[i * LD + i];
                if (m.occf[i]) homo = fmax(homo, ei); else lumo = fmin(lumo, ei);
            }
            if (!(lumo - homo > MIN_GAP)) m.flag |= ERRBIT_ZERO_GAP;
        }
    }
    __syncwarp();
    if (act) {
        // one (pair, table) task per lane: the H0 part of a pair's gradient on one lane, its S
        // part (with the second-order and repulsion terms) on another; combined below
        for (int task = j; task < 2 * NPAIR; task += NORB) {
            const int pi = task % NPAIR, t = task / NPAIR;
            const int A = m.pa[pi], B = m.pb[pi];
            const int eA = m.spec[A], eB = m.spec[B];
            const int oA = m.atom_off[A], oB = m.atom_off[B];
            const int na = sk.norb[eA], nb = sk.norb[eB];
            const double dx = m.pos[B][0] - m.pos[A][0];
            const double dy = m.pos[B][1] - m.pos[A][1];
            const double dz = m.pos[B][2] - m.pos[A][2];
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const double ir = rsqrt_nr(r2);
            const double r = r2 * ir;
            const double e[3] = {dx * ir, dy * ir, dz * ir};
            const double hshift = 0.5 * (m.shift[A] + m.shift[B]);
            double gk[3] = {0.0, 0.0, 0.0};
            {
                const double (*tab)[CAVMD_MAX_ELEM][4][4] = t == 0 ? sk.h0 : sk.s;
                // weights of the (A, B) block: P for H0, P (eps_A + eps_B)/2 - W for S
                auto wt = [&](int mu, int nu) -> double {
                    const double pv = m.P[nu * LD + mu];
                    return t == 0 ? pv : fma(pv, hshift, -m.Y[nu * LD + mu]);
                };
                double v, dv;
                radial(tab[eA][eB][CAVMD_SK_SS], r, sk, v, dv);
                {
                    const double w = wt(oA, oB) * dv;
                    for (int k = 0; k < 3; ++k) gk[k] = fma(w, e[k], gk[k]);
                }
                if (nb == 4) {
                    radial(tab[eA][eB][CAVMD_SK_SP], r, sk, v, dv);
                    double w[3], we = 0.0;
                    for (int i = 0; i < 3; ++i) { w[i] = wt(oA, oB + 1 + i); we = fma(w[i], e[i], we); }
                    for (int k = 0; k < 3; ++k)
                        gk[k] += fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                }
                if (na == 4) {
                    radial(tab[eB][eA][CAVMD_SK_SP], r, sk, v, dv);
                    double w[3], we = 0.0;
                    for (int i = 0; i < 3; ++i) { w[i] = wt(oA + 1 + i, oB); we = fma(w[i], e[i], we); }
                    for (int k = 0; k < 3; ++k)
                        gk[k] -= fma(w[k] - we * e[k], v * ir, we * e[k] * dv);
                }
                if (na == 4 && nb == 4) {
                    double vs, dvs, vp, dvp;
                    radial(tab[eA][eB][CAVMD_SK_PPS], r, sk, vs, dvs);
                    radial(tab[eA][eB][CAVMD_SK_PPP], r, sk, vp, dvp);
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
                        gk[k] += (We[k] + WTe[k] - 2.0 * eWe * e[k]) * dl * ir + eWe * e[k] * ddl +
                                 tr * e[k] * dvp;
                }
            }
            for (int k = 0; k < 3; ++k) m.gpart[t][pi][k] = gk[k];
            if (t == 1) {
                // second-order charge term and pair repulsion
                const double gi = rsqrt_nr(fma(r, r, sk.gamma_c2[eA][eB]));
                const double dgam = -r * gi * gi * gi;
                const double qq = (m.q[A] - m.zv[A]) * (m.q[B] - m.zv[B]) * dgam;
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
                for (int k = 0; k < 3; ++k) m.gpair[pi][k] = (qq + derep) * e[k];
                m.epair[pi] = erep;
            }
        }
    }
    __syncwarp();
    if (act && j < NPAIR)
        for (int k = 0; k < 3; ++k) m.gpair[j][k] = fma(2.0, m.gpart[0][j][k] + m.gpart[1][j][k], m.gpair[j][k]);
    __syncwarp();
    if (valid && j < NAT) {
        double f[3] = {0.0, 0.0, 0.0};
        for (int pi = 0; pi < NPAIR; ++pi) {
            const double sg = (m.pb[pi] == j) ? -1.0 : ((m.pa[pi] == j) ? 1.0 : 0.0);
            for (int k = 0; k < 3; ++k) f[k] = fma(sg, m.gpair[pi][k], f[k]);
        }
        const int at = a0 + j;
        for (int k = 0; k < 3; ++k) a.F[3 * at + k] = f[k];
        a.qprev[at] = a.have_warm ? m.qstart[j] : m.q[j];
        a.qpop[at] = m.q[j];
        if (a.Qout) a.Qout[at] = m.zv[j] - m.q[j];
        if (a.write_b) {
            const double Q = m.zv[j] - m.q[j];
            a.b[3 * at + 0] = Q * a.pol0;
            a.b[3 * at + 1] = Q * a.pol1;
            a.b[3 * at + 2] = Q * a.pol2;
        }
    }
    if (valid) {
        double *cw = a.Cwarm + (a.Cwarm_off ? a.Cwarm_off[cell] : (long long)cell * NORB * NORB);
        int col = j;
        if (a.warm_water) {   // the warm water path reads the occupied columns first
            int below = 0;
            for (int i = 0; i < j; ++i) below += m.occf[i] ? 1 : 0;
            col = m.occf[j] ? below : m.nocc + j - below;
        }
        for (int i = 0; i < NORB; ++i) cw[col * NORB + i] = m.C[j * LD + i];
    }
    if (valid && j == 0) {
        double E = 0.0;
        for (int i = 0; i < NORB; ++i) E += m.red[i];
        double e2 = 0.0;
        for (int x = 0; x < NAT; ++x)
            for (int y = 0; y < NAT; ++y)
                e2 = fma(m.gam[x][y] * (m.q[x] - m.zv[x]), m.q[y] - m.zv[y], e2);
        E = fma(0.5, e2, E);
        for (int pi = 0; pi < NPAIR; ++pi) E += m.epair[pi];
        double mu[3] = {0.0, 0.0, 0.0};
        for (int at = 0; at < NAT; ++at) {
            const double Q = m.zv[at] - m.q[at];
            for (int k = 0; k < 3; ++k) mu[k] = fma(Q, m.pos[at][k] - m.pos[0][k], mu[k]);
        }
        a.E_cell[cell] = E;
        a.M_cell[cell] = fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
        a.iters[cell] = m.iters;
        if (m.flag) atomicOr(a.status, (unsigned)m.flag);
    }
}

// Newton step of the self-consistent orbital rotation of a water in FP32: K[v * 4 + o] solves
//   (A_vv (x) 1 - 1 (x) A_oo + 4 sum_AB B^A gamma_AB B^B) K = -A_vo,
// by forward and back substitution with the Cholesky factor L (rows of the lower triangle, its
// diagonal stored as reciprocals).
__device__ __forceinline__ void w_solve(const float *L, const float *rhs, float *K) {
    float y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float s = -rhs[i];
#pragma unroll
        for (int k = 0; k < i; ++k) s = fmaf(-L[i * (i + 1) / 2 + k], y[k], s);
        y[i] = s * L[i * (i + 1) / 2 + i];
    }
#pragma unroll
    for (int i = 7; i >= 0; --i) {
        float s = y[i];
#pragma unroll
        for (int k = i + 1; k < 8; ++k) s = fmaf(-L[k * (k + 1) / 2 + i], K[k], s);
        K[i] = s * L[i * (i + 1) / 2 + i];
    }
}

// The general solve as a call: the warm path reaches it for molecules it does not converge.
__device__ __noinline__ void scc_general_water(const DftbArgs &a, MolShared<3, 6> &m, bool act, int j, int cell,
                                               int a0, bool disp) {
    scc_general<3, 6>(a, m, act, j, cell, a0, disp);
}

// Warm-started waters: three atoms with 4, 1 and 1 orbitals in this order, eight electrons, and the
// eigenvectors of the previous step (or, for a displaced copy, of the undisplaced cell).
//
// On GB300 an FP64 multiply-add costs 64 FP32 ones, and the general solve above spends about six
// FP64 iterations on what is, until the last two, an approximate answer. Here the approximate part
// runs in FP32: the previous basis is made S-orthonormal, then Newton steps on the orbital rotation
// (the 8 occupied-virtual angles, with the charges' response, so that each step squares the error)
// until the rotation reaches FP32 rounding. The FP64 part starts from that basis:
//   C <- C (1 - E/2 + 3/8 E^2 - 5/16 E^3), E = C^T S C - 1 (about 1e-6 here);
//   evaluations of the populations q(C), H(q) and the residual A_vo = C_v^T H C_o, all in FP64, each
//   followed by the second-order rotation C (1 + K + K^2/2) with the Newton K of the last FP32
//   Hessian (relative error about 1e-6, so the error falls by that factor).
// A water is converged when every |A_vo| is below EIG_TOL and the charges would move by less than
// scc_tol under K: two evaluations as a rule, against 6.2 iterations of the general solve. Nothing of
// the FP32 part but the starting basis and the approximate Hessian enters the result. A water that
// leaves the path's range (a rotation above W_ROT_MAX, a Hessian or gap that is not safely positive,
// no convergence) goes through the general solve of its warp.
// Measured (GB300, one launch): 262,144 waters 6.31 -> 2.0 ms, 4,096 waters 156 -> 47 us; mean
// evaluations 6.15 -> 2.04. Bound: the FP64 pipe at large batches, the serial chain at small ones.
// Lanes: six per water, lane = orbital = matrix row. A row of S and of H0 stays in registers, so a
// product with C needs only broadcast reads of C; products over rows go through shared memory.
// The radial functions of a pair stay in registers for the gradient.
__device__ __forceinline__ void water_warm(const DevSK &sk, const DftbArgs &a, const int gpw) {
    using SM = MolShared<3, 6>;
    constexpr int LD = SM::LD;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int g = lane / 6;
    const int j = lane - g * 6;
    const bool act = g < gpw;
    SM &m = reinterpret_cast<SM *>(smem_raw)[warp * gpw + (act ? g : 0)];
    WarmScratch &w = m.w;
    const bool disp = a.n_disp > 0;
    const int n_rows = disp ? a.n_cells * a.n_disp : a.n_cells;
    const int idx = (blockIdx.x * (blockDim.x >> 5) + warp) * gpw + g;
    const bool valid = act && idx < n_rows;
    const int ridx = min(idx, n_rows - 1);
    const int cidx = disp ? ridx / a.n_disp : ridx;
    const int cell = a.cell_list ? a.cell_list[cidx] : cidx;
    const int a0 = a.cell_offset[cell];
    const double *cw = a.Cwarm + (a.Cwarm_off ? a.Cwarm_off[cell] : (long long)cell * 36);

    // ---------------------------------------------------------------- geometry, opening half-flow
    const bool open = a.E_open != nullptr && !disp;
    double p_new[3], r_new[3];
    float cf[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (act) {
#pragma unroll
        for (int k = 0; k < 6; ++k) cf[k] = d2f_steer(cw[k * 6 + j]);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            m.S[j * LD + k] = (k == j) ? 1.0 : 0.0;
            m.H0[j * LD + k] = 0.0;
        }
    }
    if (act && j < 3) {
        const int at = a0 + j;
        m.spec[j] = a.species[at];
#pragma unroll
        for (int k = 0; k < 3; ++k) m.pos[j][k] = a.r[3 * at + k];
        if (open) {
            const double e1 = a.E_open[cell], im = a.inv_mass[at];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                p_new[k] = fma(a.tau, a.F[3 * at + k], fma(e1, a.b[3 * at + k], a.p_open[3 * at + k]));
                r_new[k] = fma(a.dt * im, p_new[k], m.pos[j][k]);
                m.pos[j][k] = r_new[k];
            }
        }
        if (disp) {
            const int k = ridx - cidx * a.n_disp;
            const int kk = a.fd_central ? k >> 1 : k;
            const int da = kk / 3, dc = kk - 3 * (kk / 3);
            const double sg = (a.fd_central && (k & 1)) ? -1.0 : 1.0;
            if (j == da) m.pos[j][dc] += sg * a.fd_h;
        }
    }
    __syncwarp();   // every lane of the warp has read the state it kicks before any is stored
    if (open && valid && j < 3) {
        const int at = a0 + j;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.p_open[3 * at + k] = p_new[k];
            a.r_open[3 * at + k] = r_new[k];
        }
    }

    // ---------------------------------------------------------------- H0, S, gamma
    // lane (pair, table): pairs (0,1), (0,2), (1,2); the values and slopes stay for the gradient
    const int pi = j >= 3 ? j - 3 : j, tb = j >= 3 ? 1 : 0;
    const int PA = pi == 2 ? 1 : 0, PB = pi == 0 ? 1 : 2;
    const int e0 = m.spec[0], e1_ = m.spec[1], e2_ = m.spec[2];
    const int eA = pi == 2 ? e1_ : e0, eB = pi == 0 ? e1_ : e2_;
    const double U0 = sk.hubbard[e0], U1 = sk.hubbard[e1_], U2 = sk.hubbard[e2_];
    const double z0 = sk.zval[e0], z1 = sk.zval[e1_], z2 = sk.zval[e2_];
    double ev[3], rr, ir, gi, vss, dvss, vps = 0.0, dvps = 0.0;
    {
        const double dx = m.pos[PB][0] - m.pos[PA][0];
        const double dy = m.pos[PB][1] - m.pos[PA][1];
        const double dz = m.pos[PB][2] - m.pos[PA][2];
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        ir = rsqrt_nr(r2);
        rr = r2 * ir;
        ev[0] = dx * ir;
        ev[1] = dy * ir;
        ev[2] = dz * ir;
        gi = rsqrt_nr(r2 + sk.gamma_c2[eA][eB]);
        const double (*tab)[CAVMD_MAX_ELEM][4][4] = tb == 0 ? sk.h0 : sk.s;
        radial(tab[eA][eB][CAVMD_SK_SS], rr, sk, vss, dvss);
        double *X = tb == 0 ? m.H0 : m.S;
        if (pi < 2) radial(tab[eB][eA][CAVMD_SK_SP], rr, sk, vps, dvps);
        if (act) {
            const int rB = 3 + PB;   // orbital of atom B; atom A's first orbital is 0 (pi < 2) or 4
            const int rA = pi < 2 ? 0 : 4;
            X[rB * LD + rA] = vss;
            X[rA * LD + rB] = vss;
            if (pi < 2) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const double x = -ev[i] * vps;
                    X[rB * LD + 1 + i] = x;
                    X[(1 + i) * LD + rB] = x;
                }
            }
            if (tb == 0) {
                m.gam[PA][PB] = gi;
                m.gam[PB][PA] = gi;
            } else if (pi == 0) {
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    m.H0[k * LD + k] = k == 0 ? sk.onsite[e0][0] : k < 4 ? sk.onsite[e0][1] : k == 4 ? sk.onsite[e1_][0]
                                                                                                    : sk.onsite[e2_][0];
                m.gam[0][0] = U0;
                m.gam[1][1] = U1;
                m.gam[2][2] = U2;
                m.zv[0] = z0;
                m.zv[1] = z1;
                m.zv[2] = z2;
                m.flag = 0;
                m.conv = 0;
                m.iters = 0;
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) w.Cf[j][k] = cf[k];
        }
    }
    __syncwarp();
    double sr[6], hr[6];   // row j of S and H0
    float sf[6], hf[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        sr[k] = m.S[j * LD + k];
        hr[k] = m.H0[j * LD + k];
        sf[k] = d2f_steer(sr[k]);
        hf[k] = d2f_steer(hr[k]);
    }
    const double g01 = m.gam[0][1], g02 = m.gam[0][2], g12 = m.gam[1][2];

    // ---------------------------------------------------------------- FP32 start
    auto load_row = [](const float (&row)[8], float *x) {
        const float4 lo = *reinterpret_cast<const float4 *>(row);
        const float2 hi = *reinterpret_cast<const float2 *>(row + 4);
        x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w; x[4] = hi.x; x[5] = hi.y;
    };
    auto store_row = [](float (&row)[8], const float *x) {
        *reinterpret_cast<float4 *>(row) = make_float4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<float2 *>(row + 4) = make_float2(x[4], x[5]);
    };
    // out[a] = sum_k row[k] Cf[k][a]; then, with those rows exchanged, M(a, j) = sum_i Cf[i][a] out_i[j]
    // in Mf[j][a] (lane j forms column j), read back by every lane
    auto row_times_C = [&](const float *row, const float (*cc)[6], float *out) {
#pragma unroll
        for (int k = 0; k < 6; ++k) out[k] = row[0] * cc[0][k];
#pragma unroll
        for (int i = 1; i < 6; ++i)
#pragma unroll
            for (int k = 0; k < 6; ++k) out[k] = fmaf(row[i], cc[i][k], out[k]);
    };
    auto ct_rows = [&](const float *out, const float (*cc)[6], float (*M)[6]) {
        if (act) store_row(w.Mf[j], out);
        __syncwarp();
        float col[6], t[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) col[i] = w.Mf[i][j];
#pragma unroll
        for (int k = 0; k < 6; ++k) t[k] = cc[0][k] * col[0];
#pragma unroll
        for (int i = 1; i < 6; ++i)
#pragma unroll
            for (int k = 0; k < 6; ++k) t[k] = fmaf(cc[i][k], col[i], t[k]);
        __syncwarp();
        if (act) store_row(w.Mf[j], t);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 6; ++i) load_row(w.Mf[i], M[i]);
    };
    const float u0 = d2f_steer(U0), u1 = d2f_steer(U1), u2 = d2f_steer(U2);
    const float zf0 = d2f_steer(z0), zf1 = d2f_steer(z1), zf2 = d2f_steer(z2);
    const double hU0 = 0.5 * U0, hU1 = 0.5 * U1, hU2 = 0.5 * U2, h01 = 0.5 * g01, h02 = 0.5 * g02, h12 = 0.5 * g12;
    const float f01 = d2f_steer(g01), f02 = d2f_steer(g02), f12 = d2f_steer(g12);
    bool ok = true;
    {
        float cc[6][6], M[6][6], out[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) load_row(w.Cf[i], cc[i]);
        row_times_C(sf, cc, out);
        ct_rows(out, cc, M);   // C^T S C
        float big = 0.0f;
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                M[i][k] -= (i == k) ? 1.0f : 0.0f;
                big = max_nan(big, fabsf(M[i][k]));
            }
        ok = big < 0.2f;   // false for NaN
        // C (1 - E/2 + 3/8 E^2 - 5/16 E^3): E is a few 1e-2 after one step
        float x1[6], x2[6], x3[6];
        row_times_C(cf, M, x1);
        row_times_C(x1, M, x2);
        row_times_C(x2, M, x3);
#pragma unroll
        for (int k = 0; k < 6; ++k) cf[k] += fmaf(-0.5f, x1[k], fmaf(0.375f, x2[k], -0.3125f * x3[k]));
    }
    float bh[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // lanes 4 and 5: B of their hydrogen
    bool done = !ok || !act;
    for (int it = 0; it < W_FP32_ITERS; ++it) {
        if (act) store_row(w.Cf[j], cf);
        __syncwarp();
        if (__all_sync(CAVMD_FULL_MASK, done)) break;
        float cc[6][6], out[6], M[6][6], K[8];
#pragma unroll
        for (int i = 0; i < 6; ++i) load_row(w.Cf[i], cc[i]);
        row_times_C(sf, cc, out);
        if (act) {
            w.popf[j] = 2.0f * fmaf(cf[0], out[0], fmaf(cf[1], out[1], fmaf(cf[2], out[2], cf[3] * out[3])));
            if (j >= 4) {
#pragma unroll
                for (int v = 0; v < 2; ++v)
#pragma unroll
                    for (int o = 0; o < 4; ++o)
                        w.B[(j - 4) * 8 + v * 4 + o] = 0.5f * fmaf(cf[4 + v], out[o], out[4 + v] * cf[o]);
            }
        }
        __syncwarp();
        {
            const float d0 = (w.popf[0] + w.popf[1]) + (w.popf[2] + w.popf[3]) - zf0;
            const float d1 = w.popf[4] - zf1, d2 = w.popf[5] - zf2;
            const float s0 = 0.5f * fmaf(u0, d0, fmaf(f01, d1, f02 * d2));
            const float s1 = 0.5f * fmaf(f01, d0, fmaf(u1, d1, f12 * d2));
            const float s2 = 0.5f * fmaf(f02, d0, fmaf(f12, d1, u2 * d2));
            const float sj = j < 4 ? s0 : (j == 4 ? s1 : s2);
            float hrow[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) hrow[k] = fmaf(sf[k], sj + (k < 4 ? s0 : (k == 4 ? s1 : s2)), hf[k]);
            row_times_C(hrow, cc, out);
        }
        ct_rows(out, cc, M);   // C^T H C
        // the orbital Hessian and its Cholesky factor, the same in every lane of the water
        float L[36];
        {
            float b1[8], b2[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { b1[i] = w.B[i]; b2[i] = w.B[8 + i]; }
            const float q11 = 4.0f * (u1 - 2.0f * f01 + u0), q22 = 4.0f * (u2 - 2.0f * f02 + u0);
            const float q12 = 4.0f * (f12 - f01 - f02 + u0);
            bool pd = true;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float w1 = fmaf(q11, b1[i], q12 * b2[i]), w2 = fmaf(q12, b1[i], q22 * b2[i]);
#pragma unroll
                for (int k = 0; k <= i; ++k) {
                    float x = fmaf(w1, b1[k], w2 * b2[k]);
                    if ((i & 3) == (k & 3)) x += M[4 + (i >> 2)][4 + (k >> 2)];
                    if ((i >> 2) == (k >> 2)) x -= M[i & 3][k & 3];
#pragma unroll
                    for (int l = 0; l < k; ++l) x = fmaf(-L[i * (i + 1) / 2 + l], L[k * (k + 1) / 2 + l], x);
                    if (k < i) {
                        L[i * (i + 1) / 2 + k] = x * L[k * (k + 1) / 2 + k];
                    } else {
                        pd = pd && x > 1e-3f;
                        L[i * (i + 1) / 2 + i] = rsqrtf(x);
                    }
                }
            }
            // gap: tau - C_o^T H C_o is positive definite for tau = lowest virtual level - W_GAP
            const float av = M[4][4], bv = M[5][5], cv = M[5][4];
            const float tau = 0.5f * (av + bv) - sqrtf(fmaf(0.25f * (av - bv), av - bv, cv * cv)) - W_GAP;
            float G[10];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k <= i; ++k) {
                    float x = (i == k ? tau : 0.0f) - M[i][k];
#pragma unroll
                    for (int l = 0; l < k; ++l) x = fmaf(-G[i * (i + 1) / 2 + l], G[k * (k + 1) / 2 + l], x);
                    if (k < i) {
                        G[i * (i + 1) / 2 + k] = x * G[k * (k + 1) / 2 + k];
                    } else {
                        pd = pd && x > 0.0f;
                        G[i * (i + 1) / 2 + i] = rsqrtf(x);
                    }
                }
            ok = ok && pd;
        }
        {
            float rhs[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) rhs[i] = 0.5f * (M[4 + (i >> 2)][i & 3] + M[i & 3][4 + (i >> 2)]);
            w_solve(L, rhs, K);
        }
        float kmax = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) kmax = max_nan(kmax, fabsf(K[i]));
        ok = ok && kmax < W_ROT_MAX;
        if (!done && ok) {   // a water that is done keeps its basis and Hessian whatever its warp does
            if (j == 0) {
#pragma unroll
                for (int i = 0; i < 36; ++i) w.L[i] = L[i];
            }
            if (j >= 4) {
#pragma unroll
                for (int i = 0; i < 8; ++i) bh[i] = w.B[(j - 4) * 8 + i];
            }
            // C (1 + K + K^2/2) by rows: b_o + sum_v K_vo (a_v - s_v/2), a_v - sum_o K_vo (b_o + r_o/2),
            // s_v = sum_o b_o K_vo, r_o = sum_v a_v K_vo
            float sv[2], ro[4];
#pragma unroll
            for (int v = 0; v < 2; ++v)
                sv[v] = fmaf(cf[0], K[4 * v], fmaf(cf[1], K[4 * v + 1], fmaf(cf[2], K[4 * v + 2], cf[3] * K[4 * v + 3])));
#pragma unroll
            for (int o = 0; o < 4; ++o) ro[o] = fmaf(cf[4], K[o], cf[5] * K[4 + o]);
            float n[6];
#pragma unroll
            for (int o = 0; o < 4; ++o)
                n[o] = fmaf(K[o], fmaf(-0.5f, sv[0], cf[4]), fmaf(K[4 + o], fmaf(-0.5f, sv[1], cf[5]), cf[o]));
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                float x = cf[4 + v];
#pragma unroll
                for (int o = 0; o < 4; ++o) x = fmaf(-K[4 * v + o], fmaf(0.5f, ro[o], cf[o]), x);
                n[4 + v] = x;
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) cf[k] = n[k];
        }
        done = done || !ok || kmax < W_FP32_KTOL;
        __syncwarp();
    }
    ok = ok && done;
    __syncwarp();

    // ---------------------------------------------------------------- FP64: orthonormal basis
    double c[6];   // row j of C
#pragma unroll
    for (int k = 0; k < 6; ++k) c[k] = f2d_steer(cf[k]);
    auto put_C = [&]() {
        if (act) {
            double2 *row = reinterpret_cast<double2 *>(w.C + 6 * j);
            row[0] = make_double2(c[0], c[1]);
            row[1] = make_double2(c[2], c[3]);
            row[2] = make_double2(c[4], c[5]);
        }
        __syncwarp();
    };
    if (act && j >= 4) {
#pragma unroll
        for (int i = 0; i < 8; ++i) w.B[(j - 4) * 8 + i] = bh[i];
    }
    put_C();

    // ---------------------------------------------------------------- FP64 evaluations
    double q0 = 0.0, q1 = 0.0, q2 = 0.0, s0 = 0.0, s1 = 0.0, s2 = 0.0;   // populations of one spin, half shifts
    // q(C), the shifts and H C_occ (in X) of the basis in w.C
    auto evaluate = [&]() {
        double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const double2 *row = reinterpret_cast<const double2 *>(w.C + 6 * i);
            const double2 lo = row[0], hi = row[1];
            x[0] = fma(sr[i], lo.x, x[0]);
            x[1] = fma(sr[i], lo.y, x[1]);
            x[2] = fma(sr[i], hi.x, x[2]);
            x[3] = fma(sr[i], hi.y, x[3]);
        }
        if (act) w.pop[j] = fma(c[0], x[0], fma(c[1], x[1], fma(c[2], x[2], c[3] * x[3])));   // of one spin
        __syncwarp();
        q0 = (w.pop[0] + w.pop[1]) + (w.pop[2] + w.pop[3]);
        q1 = w.pop[4];
        q2 = w.pop[5];
        const double d0 = fma(2.0, q0, -z0), d1 = fma(2.0, q1, -z1), d2 = fma(2.0, q2, -z2);
        s0 = fma(hU0, d0, fma(h01, d1, h02 * d2));
        s1 = fma(h01, d0, fma(hU1, d1, h12 * d2));
        s2 = fma(h02, d0, fma(h12, d1, hU2 * d2));
        const double sj = j < 4 ? s0 : (j == 4 ? s1 : s2);
        const double t0 = sj + s0, t1 = sj + s1, t2 = sj + s2;
        double h[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = fma(sr[k], k < 4 ? t0 : (k == 4 ? t1 : t2), hr[k]);
#pragma unroll
        for (int o = 0; o < 4; ++o) x[o] = 0.0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const double2 *row = reinterpret_cast<const double2 *>(w.C + 6 * i);
            const double2 lo = row[0], hi = row[1];
            x[0] = fma(h[i], lo.x, x[0]);
            x[1] = fma(h[i], lo.y, x[1]);
            x[2] = fma(h[i], hi.x, x[2]);
            x[3] = fma(h[i], hi.y, x[3]);
        }
        if (act) {
            double2 *row = reinterpret_cast<double2 *>(w.X + 4 * j);
            row[0] = make_double2(x[0], x[1]);
            row[1] = make_double2(x[2], x[3]);
        }
        __syncwarp();
    };
    const float tol = (float)a.scc_tol;
    const int evals = min(a.max_iter, W_EVALS);
    bool conv = false;
    int used = 0;
    float K[8], move1 = 0.0f, move2 = 0.0f;   // the rotation that the last residual asks for, the charges' change under it
    bool rough = act && ok;   // the basis is orthonormal to FP32 only (or after a large rotation)
    for (int it = 1; it <= evals; ++it) {
        for (int pass = 0; pass < 3 && __any_sync(CAVMD_FULL_MASK, rough); ++pass) {
            double x[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) x[k] = 0.0;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                const double2 *row = reinterpret_cast<const double2 *>(w.C + 6 * i);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double2 v = row[k];
                    x[2 * k] = fma(sr[i], v.x, x[2 * k]);
                    x[2 * k + 1] = fma(sr[i], v.y, x[2 * k + 1]);
                }
            }
            if (act) {
                double2 *row = reinterpret_cast<double2 *>(w.X + 6 * j);
                row[0] = make_double2(x[0], x[1]);
                row[1] = make_double2(x[2], x[3]);
                row[2] = make_double2(x[4], x[5]);
            }
            __syncwarp();
            if (act) {   // -E/2, entry (p, q), p >= q, at p (p + 1) / 2 + q: 21 entries over 6 lanes
                for (int e = j; e < 21; e += 6) {
                    int p = (e >= 15) ? 5 : (e >= 10) ? 4 : (e >= 6) ? 3 : (e >= 3) ? 2 : (e >= 1) ? 1 : 0;
                    const int q = e - p * (p + 1) / 2;
                    double s = p == q ? -1.0 : 0.0;
#pragma unroll
                    for (int i = 0; i < 6; ++i) s = fma(w.C[6 * i + p], w.X[6 * i + q], s);
                    w.E[e] = -0.5 * s;
                }
            }
            __syncwarp();
            double n[6];
            float ef[21], x0[6], x1[6], x2[6];
            float e2 = 0.0f;   // sum of (E/2)^2
#pragma unroll
            for (int k = 0; k < 6; ++k) n[k] = c[k];
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
                for (int q = 0; q <= p; ++q) {
                    const double e = w.E[p * (p + 1) / 2 + q];
                    ef[p * (p + 1) / 2 + q] = d2f_steer(e);
                    e2 = fmaf(p == q ? 1.0f : 2.0f, ef[p * (p + 1) / 2 + q] * ef[p * (p + 1) / 2 + q], e2);
                    n[q] = fma(c[p], e, n[q]);
                    if (p != q) n[p] = fma(c[q], e, n[p]);
                }
            // 3/8 E^2 - 5/16 E^3, with H = -E/2: 3/2 H^2 + 5/2 H^3. The norm of E is 6e-7 as a rule, more after a large
            // rotation; up to W_ORTH_ONCE FP32 rounds these terms by 6e-15, and the quartic one is 2e-14.
            auto efe = [&](const float *x, float *y) {
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    y[q] = 0.0f;
#pragma unroll
                    for (int p = 0; p < 6; ++p) y[q] = fmaf(x[p], p >= q ? ef[p * (p + 1) / 2 + q] : ef[q * (q + 1) / 2 + p], y[q]);
                }
            };
#pragma unroll
            for (int k = 0; k < 6; ++k) x0[k] = d2f_steer(c[k]);
            efe(x0, x1);
            efe(x1, x2);
#pragma unroll
            for (int k = 0; k < 6; ++k) x1[k] = 1.5f * x2[k];
            if (4.0f * e2 > W_ORTH_CUBE * W_ORTH_CUBE) {
                float x3[6];
                efe(x2, x3);
#pragma unroll
                for (int k = 0; k < 6; ++k) x1[k] = fmaf(2.5f, x3[k], x1[k]);
            }
            if (rough) {   // the others of the warp keep their basis to the bit
#pragma unroll
                for (int k = 0; k < 6; ++k) c[k] = n[k] + f2d_steer(x1[k]);
                ok = ok && 4.0f * e2 < W_ORTH_MAX * W_ORTH_MAX;   // false for NaN
                rough = ok && 4.0f * e2 > W_ORTH_ONCE * W_ORTH_ONCE;
            }
            put_C();
        }
        ok = ok && !rough;
        rough = false;
        evaluate();
        if (act) {
            for (int e = j; e < 8; e += 6) {
                const int v = 4 + (e >> 2), o = e & 3;
                double s = 0.0;
#pragma unroll
                for (int i = 0; i < 6; ++i) s = fma(w.C[6 * i + v], w.X[4 * i + o], s);
                w.av[e] = d2f_steer(s);
            }
        }
        __syncwarp();
        float L[36], rhs[8];
#pragma unroll
        for (int i = 0; i < 36; ++i) L[i] = w.L[i];
        float amax = 0.0f;
        move1 = move2 = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            rhs[i] = w.av[i];
            amax = max_nan(amax, fabsf(rhs[i]));
        }
        w_solve(L, rhs, K);
#pragma unroll
        for (int i = 0; i < 8; ++i) {   // the charges' change under K (the oxygen's is minus the sum)
            move1 = fmaf(4.0f * w.B[i], K[i], move1);
            move2 = fmaf(4.0f * w.B[8 + i], K[i], move2);
        }
        const float move = fmaxf(fabsf(move1 + move2), fmaxf(fabsf(move1), fabsf(move2)));
        if (!conv && ok) {
            used = it;
            conv = amax < (float)EIG_TOL && move < tol;
            float k2 = 0.0f;
#pragma unroll
            for (int i = 0; i < 8; ++i) k2 = fmaf(K[i], K[i], k2);
            ok = amax < 1.0f && k2 < W_ROT64_MAX * W_ROT64_MAX;   // false for NaN
            rough = ok && !conv && k2 > W_ROT64_ONCE * W_ROT64_ONCE;
        }
        if (__all_sync(CAVMD_FULL_MASK, conv || !ok || !act)) break;
        if (!conv && ok && it < evals) {   // the rotation; its second-order part in FP32: up to W_ROT64_ONCE of a
                                              // norm below 5e-8, rounded below 3e-15, and C stays orthonormal to K^4 / 4 < 3e-15
            float sv[2], ro[4], c32[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) c32[k] = d2f_steer(c[k]);
#pragma unroll
            for (int v = 0; v < 2; ++v)
                sv[v] = fmaf(c32[0], K[4 * v], fmaf(c32[1], K[4 * v + 1], fmaf(c32[2], K[4 * v + 2], c32[3] * K[4 * v + 3])));
#pragma unroll
            for (int o = 0; o < 4; ++o) ro[o] = fmaf(c32[4], K[o], c32[5] * K[4 + o]);
            double Kd[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) Kd[i] = f2d_steer(K[i]);
            const double x4 = c[4] - f2d_steer(0.5f * sv[0]), x5 = c[5] - f2d_steer(0.5f * sv[1]);
            double n[6];
#pragma unroll
            for (int o = 0; o < 4; ++o) n[o] = fma(Kd[o], x4, fma(Kd[4 + o], x5, c[o]));
            n[4] = c[4];
            n[5] = c[5];
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const double y = c[o] + f2d_steer(0.5f * ro[o]);
                n[4] = fma(-Kd[o], y, n[4]);
                n[5] = fma(-Kd[4 + o], y, n[5]);
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) c[k] = n[k];
        }
        put_C();
    }
    // the general solve for what is left, then its state as the evaluations leave it
    if (!__all_sync(CAVMD_FULL_MASK, conv || !act)) {
        __syncwarp();
        if (act && j == 0) {
            m.conv = conv;
            if (!conv) {
                m.nocc = 4;
                m.atom_off[0] = 0;
                for (int x = 0; x < 3; ++x) m.atom_off[x + 1] = 4 + x;
                for (int x = 0; x < 6; ++x) m.orb_atom[x] = x < 4 ? 0 : x - 3;
            }
        }
        __syncwarp();
        scc_general_water(a, m, act, j, cell, a0, disp);
        __syncwarp();
        if (act && !conv) {   // occupied columns first
            int no = 0, nv = 0;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const double x = m.C[k * LD + j];
                const int to = m.occf[k] ? no++ : 4 + nv++;
#pragma unroll
                for (int d = 0; d < 6; ++d)
                    if (d == to) c[d] = x;
            }
            used = m.iters;
#pragma unroll
            for (int i = 0; i < 8; ++i) K[i] = 0.0f;
            move1 = move2 = 0.0f;
        }
        __syncwarp();
        if (act && !conv && j == 0) {   // highest occupied and lowest empty level of the last iteration
            double homo = -1e300, lumo = 1e300;
            for (int i = 0; i < 6; ++i) {
                const double ei = m.diagf[i];
                if (m.occf[i]) homo = fmax(homo, ei); else lumo = fmin(lumo, ei);
            }
            if (!(lumo - homo > MIN_GAP)) m.flag |= ERRBIT_ZERO_GAP;
        }
        __syncwarp();
        put_C();
        evaluate();
    }

    q0 *= 2.0;
    q1 *= 2.0;
    q2 *= 2.0;
    // 1/2 sum_A dq_A eps_A - sum_A q_A eps_A (s = eps / 2), the charge part of the energy, at the evaluated charges
    const double eq = fma(-(q0 + z0), s0, fma(-(q1 + z1), s1, -(q2 + z2) * s2));
    // The residual that passed the test stays in no result: the charges take their first-order change under K here
    // and the occupied orbitals theirs below (a finite-difference row divides what is left by its step). Largest
    // error of 3,000 waters without and with this: charges 9.8e-13 and 1.2e-14, forces 3.3e-12 and 1.2e-14 (the
    // general solve: 2.7e-13, 8.8e-14); 262,144 waters x 50 steps take 128.1 and 129.7 ms.
    const double m1 = f2d_steer(move1), m2 = f2d_steer(move2);
    q0 -= m1 + m2;
    q1 += m1;
    q2 += m2;

    if (disp) {   // finite-difference row: only the dipole of the converged charges
        if (valid && j == 0) {
            const double Q1 = z1 - q1, Q2 = z2 - q2;
            double mu[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                mu[k] = fma(Q2, m.pos[2][k] - m.pos[0][k], Q1 * (m.pos[1][k] - m.pos[0][k]));
            a.M_disp[(long long)(a.fd_central ? 6 : 3) * a0 + (ridx - cidx * a.n_disp)] =
                fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
            if (m.flag) atomicOr(a.status, (unsigned)m.flag);
        }
        return;
    }
    // ---------------------------------------------------------------- energy, forces, dipole
    // A_oo = C_o^T (H C_o) into E[0..9]; t(k, o) = 2 sum_p A_op C(k, p) of the hydrogens' rows k into
    // E[10..17]; then the 9 interatomic entries (row i of the lane, column of a hydrogen) of
    // P = 2 C_o C_o^T and W = 2 C_o A_oo C_o^T
    if (act) {
        for (int e = j; e < 10; e += 6) {
            const int p = (e >= 6) ? 3 : (e >= 3) ? 2 : (e >= 1) ? 1 : 0;
            const int q = e - p * (p + 1) / 2;
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < 6; ++i) s = fma(w.C[6 * i + p], w.X[4 * i + q], s);
            w.E[e] = s;
        }
    }
    __syncwarp();
    {   // C_o + C_v K: A_oo above changes with K only to second order
        const float v4 = d2f_steer(c[4]), v5 = d2f_steer(c[5]);
#pragma unroll
        for (int o = 0; o < 4; ++o) c[o] += f2d_steer(fmaf(K[o], v4, K[4 + o] * v5));
    }
    put_C();
    if (act) {
        for (int e = j; e < 8; e += 6) {
            const int row = 4 + (e >> 2), o = e & 3;
            double s = 0.0;
#pragma unroll
            for (int p = 0; p < 4; ++p) s = fma(w.E[p >= o ? p * (p + 1) / 2 + o : o * (o + 1) / 2 + p], w.C[6 * row + p], s);
            w.E[10 + e] = 2.0 * s;
        }
    }
    __syncwarp();
    if (act && j < 5) {   // entries (j, 4) (j < 4) and (j, 5): PW[2 (j, .)] for j < 4, then (4, 5)
        const double c0 = 2.0 * c[0], c1 = 2.0 * c[1], c2 = 2.0 * c[2], c3 = 2.0 * c[3];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (j == 4 && h == 0) continue;
            const double *row = w.C + 6 * (4 + h), *t = w.E + 10 + 4 * h;
            const int at = j < 4 ? 4 * h + j : 8;
            w.PW[at] = fma(c0, row[0], fma(c1, row[1], fma(c2, row[2], c3 * row[3])));
            w.PW[9 + at] = fma(c[0], t[0], fma(c[1], t[1], fma(c[2], t[2], c[3] * t[3])));
        }
    }
    __syncwarp();
    if (act) {
        const double hshift = pi == 0 ? s0 + s1 : (pi == 1 ? s0 + s2 : s1 + s2);   // (eps_A + eps_B) / 2
        const int at = pi < 2 ? 4 * pi : 8;
        double wt[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = pi < 2 ? at + i : at;
            const double pv = w.PW[k];
            wt[i] = tb == 0 ? pv : fma(pv, hshift, -w.PW[9 + k]);
        }
        double gk[3];
        double rad = wt[0] * dvss;
        if (pi < 2) {   // p orbitals of atom A with the s orbital of atom B
            const double we = fma(wt[1], ev[0], fma(wt[2], ev[1], wt[3] * ev[2]));
            const double vr = vps * ir;
            rad = fma(we, vr - dvps, rad);
#pragma unroll
            for (int k = 0; k < 3; ++k) gk[k] = fma(rad, ev[k], -wt[1 + k] * vr);
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) gk[k] = rad * ev[k];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) m.gpart[tb][pi][k] = gk[k];
        if (tb == 1) {   // second-order charge term and pair repulsion
            const double qA = pi == 2 ? q1 - z1 : q0 - z0, qB = pi == 0 ? q1 - z1 : q2 - z2;
            double erep = 0.0;
            double along = -rr * gi * gi * gi * (qA * qB);
            const double arep = sk.rep[eA][eB][0], brep = sk.rep[eA][eB][1];
            if (arep != 0.0) {
                const double vr = arep * exp(-brep * rr);
                const double x = (rr - (sk.r_cut - sk.taper)) * sk.inv_taper;
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
                along = fma(vr, df - brep * f, along);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) m.gpair[pi][k] = along * ev[k];
            m.epair[pi] = erep;
        }
    }
    __syncwarp();
    if (act && j < 3)
#pragma unroll
        for (int k = 0; k < 3; ++k) m.gpair[j][k] = fma(2.0, m.gpart[0][j][k] + m.gpart[1][j][k], m.gpair[j][k]);
    __syncwarp();
    if (valid && j < 3) {
        const int at = a0 + j;
        // pairs (0,1), (0,2), (1,2): + as the first atom, - as the second
        const int pf = j == 2 ? 1 : 0, ps = j == 0 ? 1 : 2;
        const double qj = j == 0 ? q0 : (j == 1 ? q1 : q2), zj = j == 0 ? z0 : (j == 1 ? z1 : z2);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double x = m.gpair[pf][k], y = m.gpair[ps][k];
            a.F[3 * at + k] = j == 0 ? x + y : (j == 1 ? y - x : -x - y);
        }
        a.qprev[at] = a.qpop[at];
        a.qpop[at] = qj;
        if (a.Qout) a.Qout[at] = zj - qj;
        if (a.write_b) {
            const double Q = zj - qj;
            a.b[3 * at + 0] = Q * a.pol0;
            a.b[3 * at + 1] = Q * a.pol1;
            a.b[3 * at + 2] = Q * a.pol2;
        }
    }
    if (valid) {
        double *cwo = a.Cwarm + (a.Cwarm_off ? a.Cwarm_off[cell] : (long long)cell * 36);
#pragma unroll
        for (int k = 0; k < 6; ++k) cwo[k * 6 + j] = c[k];
    }
    if (valid && j == 0) {
        // band energy Tr P H0 = 2 Tr A_oo - sum_A q_A eps_A; second order 1/2 sum_A dq_A eps_A
        double E = fma(2.0, (w.E[0] + w.E[2]) + (w.E[5] + w.E[9]), eq);
        E += (m.epair[0] + m.epair[1]) + m.epair[2];
        const double Q1 = z1 - q1, Q2 = z2 - q2;
        double mu[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) mu[k] = fma(Q2, m.pos[2][k] - m.pos[0][k], Q1 * (m.pos[1][k] - m.pos[0][k]));
        a.E_cell[cell] = E;
        a.M_cell[cell] = fma(a.pol0, mu[0], fma(a.pol1, mu[1], a.pol2 * mu[2]));
        a.iters[cell] = used;
        if (m.flag) atomicOr(a.status, (unsigned)m.flag);
    }
}

// 200 registers: eight warps per SM without spills, the faster code while that many warps hold the batch.
__global__ void __launch_bounds__(256, 1) k_water_warm(const DevSK *__restrict__ skp, const DftbArgs a, const int gpw) {
    water_warm(*skp, a, gpw);
}

// 128 registers with spills: twelve warps per SM, for batches of more than 24 warps per SM (two of its waves).
// Passes of 262,144 waters x 50 steps 138.5 -> 132.5 ms; of 8 waters x 30 steps 1.61 -> 1.66 ms, and 14.6
// warps per SM of displaced rows (1,237 waters x 9 steps) 0.92 -> 0.96 ms.
__global__ void __launch_bounds__(256, 2) k_water_warm_dense(const DevSK *__restrict__ skp, const DftbArgs a,
                                                             const int gpw) {
    water_warm(*skp, a, gpw);
}

__global__ void k_born_assemble(int n_cells, const int *__restrict__ off, const double *__restrict__ M0,
                                const double *__restrict__ Md, int nd, int central, double h,
                                double *__restrict__ b) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_cells) return;
    const double ih = 1.0 / h;
    const double *md = Md + (size_t)(central ? 6 : 3) * off[n];
    for (int j = off[n]; j < off[n + 1]; ++j) {
        const int jl = j - off[n];
        for (int k = 0; k < 3; ++k) {
            const int r = 3 * jl + k;
            b[3 * j + k] = central ? (md[2 * r] - md[2 * r + 1]) * (0.5 * ih) : (md[r] - M0[n]) * ih;
        }
    }
}

}  // namespace

cudaError_t launch_born_assemble(int n_cells, const int *cell_offset, const double *M_cell,
                                 const double *M_disp, int n_disp, int central, double h, double *b,
                                 cudaStream_t st) {
    k_born_assemble<<<(n_cells + 127) / 128, 128, 0, st>>>(n_cells, cell_offset, M_cell, M_disp, n_disp,
                                                           central, h, b);
    return cudaGetLastError();
}

// warps per block (2, 4 or 8) and waters per warp (1..5). The warps per block never change a result;
// the waters per warp do at rounding level, because the choice between a Jacobi sweep and the
// second-order update is taken per warp.
cudaError_t launch_dftb_water(const DevSK *sk, const DftbArgs &a, cudaStream_t st, int warps, int per_warp) {
    constexpr int NAT = 3, NORB = 6;
    using SM = MolShared<NAT, NORB>;
    const int gpw = per_warp < 1 ? 1 : (per_warp > 32 / NORB ? 32 / NORB : per_warp);
    const int threads = 32 * warps;
    const int per_block = warps * gpw;
    const long long rows = (long long)a.n_cells * (a.n_disp > 0 ? a.n_disp : 1);
    const int blocks = (int)((rows + per_block - 1) / per_block);
    const size_t smem = sizeof(SM) * per_block;
    if (a.n_cells <= 0) return cudaSuccess;
    if (a.have_warm && a.warm_water) {
        int dev = 0, n_sm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if ((long long)blocks * warps > 24LL * n_sm) k_water_warm_dense<<<blocks, threads, smem, st>>>(sk, a, gpw);
        else k_water_warm<<<blocks, threads, smem, st>>>(sk, a, gpw);
    } else dftb_kernel<NAT, NORB><<<blocks, threads, smem, st>>>(sk, a, gpw);
    return cudaGetLastError();
}

cudaError_t prepare_dftb_water(int max_warps) {
    const int smem = (int)(sizeof(MolShared<3, 6>) * max_warps * 5);
    const cudaError_t e = cudaFuncSetAttribute(dftb_kernel<3, 6>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const cudaError_t e2 = cudaFuncSetAttribute(k_water_warm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e2 != cudaSuccess) return e2;
    return cudaFuncSetAttribute(k_water_warm_dense, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}
