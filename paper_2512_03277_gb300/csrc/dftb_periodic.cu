// Gamma-point kernels of the periodic cells (dftb_periodic.cuh), the k-grid's launch plan, and the host side.
#include <algorithm>
#include <cmath>
#include <vector>

#include "dftb_periodic.cuh"

namespace {

// One block per cell, or (a.n_disp > 0) per finite-difference copy of a cell: (cell, row) items,
// rows_max = 3 (central: 6) x the largest atom count per cell.
__global__ void __launch_bounds__(PT, 2) k_dftb_periodic(const DevSK *__restrict__ skp, const DftbArgs a, const PbcDev pl) {
    extern __shared__ __align__(16) unsigned char p_smem[];
    PShared &sh = *reinterpret_cast<PShared *>(p_smem);
    const PbcMem wk = pbc_mem(pl, false, blockIdx.x, 0, 1);
    const int rows = pbc_rows(a, pl);
    for (long long it = blockIdx.x; it < (long long)rows * a.n_cells; it += gridDim.x) {
        int cell, row;
        if (pbc_item(a, rows, it, cell, row)) p_cell<false>(*skp, a, pl, sh, wk, cell, row, 0, 1, 0);
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Host side

namespace {

// Doubles of one cell's workspace (pbc_mem) for `cluster` blocks; lean: without the warm path's FP32 state and
// working bases.
size_t pbc_cell_doubles(const PbcPlan &p, int cluster, bool lean) {
    const size_t n2 = (p.nk > 0 ? 4 : 1) * (size_t)p.nmax * p.nmax, k = p.nk > 0 ? p.nk : 1, a2 = (size_t)p.amax * p.amax;
    const size_t own = 6 * n2 + 2 * (size_t)p.n_g + 4 * a2 + (a2 + 1) / 2 + 6 * (size_t)p.amax * (p.g_max + 1) + 1;
    return (lean ? 2 : p.nk > 0 ? 5 : 3) * k * n2 + a2 + 2 * (size_t)p.amax * p.n_g + 2 * (size_t)cluster * (p.amax + 8) +
           cluster * own + 32;
}

}  // namespace

size_t pbc_workspace_doubles(const PbcPlan &p) {
    const size_t warm = pbc_cell_doubles(p, p.cluster, false) * p.blocks;
    return p.nk > 0 ? std::max(warm, pbc_cell_doubles(p, 1, true) * p.alone) : warm;
}

bool shrink_dftb_periodic(PbcPlan &p) {
    if (p.blocks == 1 && (p.nk <= 0 || p.alone == 1)) return false;
    p.blocks = (p.blocks + 1) / 2;
    p.alone = (p.alone + 1) / 2;
    return true;
}

// The irreducible points of a Gamma-centred n1 x n2 x n3 grid: k and -k (modulo the reciprocal
// lattice) give complex-conjugate problems with the same populations and band energy, so each
// pair is kept once with weight 2 / (n1 n2 n3) (self-conjugate points: 1 / (n1 n2 n3)), the
// member with the smaller grid index. Rows: f1, f2, f3, weight.
std::vector<double> pbc_kpoints(const int *kgrid) {
    const int n1 = kgrid[0], n2 = kgrid[1], n3 = kgrid[2], N = n1 * n2 * n3;
    std::vector<double> out;
    for (int i = 0; i < n1; ++i)
        for (int j = 0; j < n2; ++j)
            for (int l = 0; l < n3; ++l) {
                const int ii = (n1 - i) % n1, jj = (n2 - j) % n2, ll = (n3 - l) % n3;   // -k on the grid
                const int idx = (i * n2 + j) * n3 + l, midx = (ii * n2 + jj) * n3 + ll;
                if (midx < idx) continue;
                out.push_back((double)i / n1);
                out.push_back((double)j / n2);
                out.push_back((double)l / n3);
                out.push_back((midx == idx ? 1.0 : 2.0) / N);
            }
    return out;
}

// Lattice images and reciprocal vectors for one lattice (rows a_i), and the Ewald constants. The
// splitting parameter is chosen so the half-space reciprocal list holds about 250 sqrt(n_atoms) vectors, at
// least 1000: the real-space sums cost n_atoms^2 / n_g error functions, the reciprocal ones n_atoms n_g
// products (99 atoms: 22 images a pair at 1000 vectors, 9 at 2500). Every term left out of either sum is
// below 1e-18 (erfc(6.5) and exp(-6.5^2)).
void plan_dftb_periodic(const double *lat, double r_cut, int n_atoms, PbcPlan &p, std::vector<double> &img,
                        std::vector<double> &gw, std::vector<int4> &gi) {
    for (int k = 0; k < 9; ++k) p.lat[k] = lat[k];
    const double a0 = lat[0], a1 = lat[1], a2 = lat[2], b0 = lat[3], b1 = lat[4], b2 = lat[5], c0 = lat[6],
                 c1 = lat[7], c2 = lat[8];
    const double det = a0 * (b1 * c2 - b2 * c1) - a1 * (b0 * c2 - b2 * c0) + a2 * (b0 * c1 - b1 * c0);
    // inverse (f = r inv with r a row vector): inv = lat^-1
    double inv[9];
    inv[0] = (b1 * c2 - b2 * c1) / det; inv[1] = (a2 * c1 - a1 * c2) / det; inv[2] = (a1 * b2 - a2 * b1) / det;
    inv[3] = (b2 * c0 - b0 * c2) / det; inv[4] = (a0 * c2 - a2 * c0) / det; inv[5] = (a2 * b0 - a0 * b2) / det;
    inv[6] = (b0 * c1 - b1 * c0) / det; inv[7] = (a1 * c0 - a0 * c1) / det; inv[8] = (a0 * b1 - a1 * b0) / det;
    for (int k = 0; k < 9; ++k) p.inv[k] = inv[k];
    const double V = std::fabs(det);
    const double EX = 6.5;
    const double pi = 3.141592653589793;
    // half-space count N ~ (4 pi / 3) (2 alpha EX)^3 V / (2 (2 pi)^3)  ->  alpha for N
    const double g_cube = std::max(1000.0, 250.0 * std::sqrt((double)n_atoms)) * 2.0 * std::pow(2.0 * pi, 3) * 3.0 / (4.0 * pi * V);
    const double alpha = std::cbrt(g_cube) / (2.0 * EX);
    p.alpha = alpha;
    p.bg = -pi / (alpha * alpha * V);
    p.self_e = -2.0 * alpha / std::sqrt(pi);
    const double r_real = std::max(EX / alpha, r_cut);
    p.r_real = r_real;
    // farthest point of a wrapped separation (fractional coordinates in [-1/2, 1/2]): a corner
    double hmax = 0.0;
    for (int s = 0; s < 8; ++s) {
        const double f0 = (s & 1) ? 0.5 : -0.5, f1 = (s & 2) ? 0.5 : -0.5, f2 = (s & 4) ? 0.5 : -0.5;
        double x[3];
        for (int k = 0; k < 3; ++k) x[k] = f0 * lat[k] + f1 * lat[3 + k] + f2 * lat[6 + k];
        hmax = std::max(hmax, std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]));
    }
    // heights across the faces: h_i = 1 / |column i of inv|
    int N[3];
    for (int i = 0; i < 3; ++i) {
        const double h = 1.0 / std::sqrt(inv[i] * inv[i] + inv[3 + i] * inv[3 + i] + inv[6 + i] * inv[6 + i]);
        N[i] = (int)std::ceil((r_real + hmax) / h) + 1;
    }
    // translations by increasing length (ties in the order generated); a wrapped separation
    // reaches an image within r_cut only through a translation shorter than r_cut + hmax
    struct Tr { double len, t[3]; };
    std::vector<Tr> trs;
    const double reach = r_real + hmax;
    for (int n0 = -N[0]; n0 <= N[0]; ++n0)
        for (int n1 = -N[1]; n1 <= N[1]; ++n1)
            for (int n2 = -N[2]; n2 <= N[2]; ++n2) {
                Tr t;
                for (int k = 0; k < 3; ++k) t.t[k] = n0 * lat[k] + n1 * lat[3 + k] + n2 * lat[6 + k];
                t.len = std::sqrt(t.t[0] * t.t[0] + t.t[1] * t.t[1] + t.t[2] * t.t[2]);
                if (t.len < reach) trs.push_back(t);
            }
    std::stable_sort(trs.begin(), trs.end(), [](const Tr &a, const Tr &b) { return a.len < b.len; });
    img.clear();
    p.n_img_sk = 0;
    for (const Tr &t : trs) {
        img.insert(img.end(), t.t, t.t + 3);
        if (t.len < r_cut + hmax) ++p.n_img_sk;
    }
    p.n_img = (int)(img.size() / 3);
    // reciprocal rows b_j = 2 pi (column j of inv), G = m b; half space: first nonzero m positive
    double B[9];
    for (int jx = 0; jx < 3; ++jx)
        for (int k = 0; k < 3; ++k) B[3 * jx + k] = 2.0 * pi * inv[3 * k + jx];
    const double g_max = 2.0 * alpha * EX;
    int M[3];
    for (int i = 0; i < 3; ++i) {   // heights of the reciprocal cell: 2 pi / |a_i|
        const double an = std::sqrt(lat[3 * i] * lat[3 * i] + lat[3 * i + 1] * lat[3 * i + 1] + lat[3 * i + 2] * lat[3 * i + 2]);
        M[i] = (int)std::ceil(g_max * an / (2.0 * pi)) + 1;
    }
    struct Vec { double g2, G[3], w2; int m[3]; };
    std::vector<Vec> vs;
    for (int m0 = -M[0]; m0 <= M[0]; ++m0)
        for (int m1 = -M[1]; m1 <= M[1]; ++m1)
            for (int m2 = -M[2]; m2 <= M[2]; ++m2) {
                const bool pos = m0 > 0 || (m0 == 0 && (m1 > 0 || (m1 == 0 && m2 > 0)));
                if (!pos) continue;
                double G[3];
                for (int k = 0; k < 3; ++k) G[k] = m0 * B[k] + m1 * B[3 + k] + m2 * B[6 + k];
                const double g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
                if (!(g2 < g_max * g_max)) continue;
                const double w = 4.0 * pi / V * std::exp(-g2 / (4.0 * alpha * alpha)) / g2;
                vs.push_back({g2, {G[0], G[1], G[2]}, 2.0 * w, {m0, m1, m2}});
            }
    std::stable_sort(vs.begin(), vs.end(), [](const Vec &x, const Vec &y) { return x.g2 < y.g2; });
    gw.clear();
    gi.clear();
    p.n_g32 = 0;
    p.g_max = 0;
    for (const Vec &v : vs) {
        gw.insert(gw.end(), {v.G[0], v.G[1], v.G[2], v.w2});
        gi.push_back(make_int4(v.m[0], v.m[1], v.m[2], 0));
        if (v.g2 < 4.0 * alpha * alpha * 18.0) ++p.n_g32;   // exp(-18) = 1.5e-8 of the weight at small G
        for (int k = 0; k < 3; ++k) p.g_max = std::max(p.g_max, std::abs(v.m[k]));
    }
    p.n_g = (int)(gw.size() / 4);
}

namespace {

bool kg_small(int nmax) { return 2 * nmax <= PNMAX; }   // the problems of the k-points fit the smaller struct

const void *kg_kernel(int nmax) { return kg_small(nmax) ? pbc_kg_small() : pbc_kg_large(); }

size_t kg_smem(int nmax) { return kg_small(nmax) ? sizeof(PShared) : sizeof(PSharedK); }

// Blocks of the k-grid kernel that can be resident at once as clusters of c.
cudaError_t kg_clusters(int nmax, int c, int *n) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = kg_smem(nmax);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n, kg_kernel(nmax), &cfg);
}

}  // namespace

// Blocks per cell and resident groups of blocks. The Gamma point takes two blocks per SM, a cell each.
// On a k-grid a cell's k-points are independent between the charge sums, so when the cells alone leave
// the chip idle a cluster of blocks shares each: the size that gives the fewest rounds of k-points,
// ceil(nk / c) ceil(n_cells / resident clusters of c), the smaller one on a tie (24 cells on 3 x 3 x 3:
// 14 points on 24 blocks before).
// A cold start takes the general path, one block per cell and SM, and so do cells that leave the warm path of a
// cluster: these are listed and evaluated by a launch of their own, so that no cluster's other blocks wait for them.
cudaError_t plan_dftb_periodic_launch(PbcPlan &p, int n_cells, int n_sm) {
    p.cluster = 1;
    p.alone = std::max(1, std::min(n_cells, n_sm));
    p.late = nullptr;
    if (p.nk <= 0) {
        p.blocks = std::max(1, std::min(n_cells, 2 * n_sm));
        return cudaSuccess;
    }
    long long best = -1;
    for (int c = 1; c <= std::min(8, p.nk); ++c) {
        int n = 0;
        const cudaError_t e = kg_clusters(p.nmax, c, &n);
        if (e != cudaSuccess) return e;
        if (n <= 0) continue;
        const long long rounds = (long long)((p.nk + c - 1) / c) * ((n_cells + n - 1) / n);
        if (best < 0 || rounds < best) {
            best = rounds;
            p.cluster = c;
            p.blocks = std::max(1, std::min(n_cells, n));
        }
    }
    if (best < 0) return cudaErrorInvalidConfiguration;
    // dense grids of large cells: at most 128 GiB of workspace, the blocks taking several cells in turn (and less
    // when the allocator has less: shrink_dftb_periodic)
    const size_t most = ((size_t)128 << 30) / 8;
    p.blocks = (int)std::max<size_t>(1, std::min<size_t>(p.blocks, most / pbc_cell_doubles(p, p.cluster, false)));
    p.alone = (int)std::max<size_t>(1, std::min<size_t>(p.alone, most / pbc_cell_doubles(p, 1, true)));
    return cudaSuccess;
}

cudaError_t prepare_dftb_periodic() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f, size_t smem) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
    set((const void *)k_dftb_periodic, sizeof(PShared));
    for (int nmax : {1, PNMAX}) set(kg_kernel(nmax), kg_smem(nmax));
    return e;
}

cudaError_t launch_dftb_periodic(const DevSK *sk_dev, const DftbArgs &a, const PbcPlan &p, cudaStream_t st) {
    if (a.n_cells <= 0) return cudaSuccess;
    PbcDev d;
    for (int k = 0; k < 9; ++k) { d.lat[k] = p.lat[k]; d.inv[k] = p.inv[k]; }
    d.alpha = p.alpha;
    d.bg = p.bg;
    d.self_e = p.self_e;
    d.r_real2 = p.r_real * p.r_real;
    d.n_img = p.n_img;
    d.n_img_sk = p.n_img_sk;
    d.n_g = p.n_g;
    d.n_g32 = p.n_g32;
    d.g_max = p.g_max;
    d.gi = p.d_gi;
    d.nmax = p.nmax;
    d.amax = p.amax;
    d.img = p.d_img;
    d.gw = p.d_gw;
    d.work = p.work;
    d.nk = p.nk;
    d.cluster = p.cluster;
    d.kpt = p.d_kpt;
    d.late = nullptr;
    d.late_pass = d.lean = 0;
    d.work_stride = (long long)pbc_cell_doubles(p, p.cluster, false);
    const long long items = a.n_disp > 0 ? (long long)a.n_cells * (a.fd_central ? 6 : 3) * p.amax : a.n_cells;
    const int groups = (int)std::min<long long>(items, p.blocks);
    if (p.nk > 0) {
        auto run = [&](int n, int nmax) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            cfg.gridDim = dim3(n * d.cluster);
            cfg.blockDim = dim3(PT);
            cfg.dynamicSmemBytes = kg_smem(nmax);
            cfg.stream = st;
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = d.cluster;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            void *args[] = {(void *)&sk_dev, (void *)&a, (void *)&d};
            return cudaLaunchKernelExC(&cfg, kg_kernel(nmax), args);
        };
        if (a.have_warm) {
            if (p.cluster == 1) return run(groups, p.nmax);
            d.late = p.late;
            cudaError_t e = cudaMemsetAsync(p.late, 0, sizeof(int), st);
            if (e == cudaSuccess) e = run(groups, p.nmax);
            if (e != cudaSuccess) return e;
            d.late_pass = 1;
        }
        // the general path, one block per cell with the wider kernel's registers: a cold start, or the late cells
        // (a finite-difference copy needs the working bases)
        d.cluster = 1;
        d.lean = a.n_disp == 0;
        d.work_stride = (long long)pbc_cell_doubles(p, 1, d.lean);
        const long long room = (long long)pbc_workspace_doubles(p) / d.work_stride;
        return run((int)std::min({items, room, (long long)p.alone}), PNMAX);
    }
    k_dftb_periodic<<<groups, PT, sizeof(PShared), st>>>(sk_dev, a, d);
    return cudaGetLastError();
}
