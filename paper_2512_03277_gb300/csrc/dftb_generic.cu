// The cluster kernel (dftb_generic.cuh) with four product entries per thread, its plan and its launch.
#include <algorithm>
#include <vector>

#include "dftb_generic.cuh"

namespace {

cudaError_t set_attr(const void *kernel, size_t smem, int &blocks_per_sm) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, kernel, BT, smem);
    return e;
}

}  // namespace

size_t dftb_generic_smem(int nmax_b, int amax_b, int nmax_s, int amax_s, int warm) {
    const size_t b = nmax_b > 0 ? g_layout(nmax_b, amax_b, warm).total : 0;
    const size_t s = nmax_s > 0 ? 2 * (size_t)g_layout(nmax_s, amax_s, warm).total : 0;
    return std::max(b, s);
}

void plan_dftb_generic(const int *cell_offset, const int *species, const int *norb_of_elem, int n_cells,
                       int n_disp_per_atom, GenericPlan &p, std::vector<int2> &items,
                       std::vector<int2> &disp_items) {
    std::vector<int> order(n_cells), norb(n_cells);
    for (int c = 0; c < n_cells; ++c) {
        int o = 0;
        for (int i = cell_offset[c]; i < cell_offset[c + 1]; ++i) o += norb_of_elem[species[i]];
        norb[c] = o;
        order[c] = c;
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return norb[x] > norb[y]; });
    p.nmax_b = p.amax_b = p.nmax_s = p.amax_s = 0;
    p.n_big = p.n_small = p.n_disp_big = p.n_disp_small = 0;
    items.clear();
    disp_items.clear();
    for (int c : order) {
        const int nat = cell_offset[c + 1] - cell_offset[c];
        const bool big = norb[c] > 32;
        int &nmax = big ? p.nmax_b : p.nmax_s, &amax = big ? p.amax_b : p.amax_s;
        nmax = std::max(nmax, norb[c]);
        amax = std::max(amax, nat);
        (big ? p.n_big : p.n_small) += 1;
        (big ? p.n_disp_big : p.n_disp_small) += n_disp_per_atom * nat;
        items.push_back(make_int2(c, -1));
        for (int k = 0; k < n_disp_per_atom * nat; ++k) disp_items.push_back(make_int2(c, k));
    }
    // cells of 64 orbitals with more than about 45 atoms leave no room for the warm path's buffer
    p.warm = 1;
    p.smem = dftb_generic_smem(p.nmax_b, p.amax_b, p.nmax_s, p.amax_s, 1);
    if (p.smem > GENERIC_SMEM_MAX) {
        p.warm = 0;
        p.smem = dftb_generic_smem(p.nmax_b, p.amax_b, p.nmax_s, p.amax_s, 0);
    }
    p.r_entries = 4;
    p.blocks_per_sm = 0;
}

cudaError_t prepare_dftb_generic(GenericPlan &p) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p.n_sm, cudaDevAttrMultiProcessorCount, dev);
    int b2 = 0, b4 = 0;
    if (e == cudaSuccess) e = set_attr(dftb_generic_kernel_r2(), p.smem, b2);
    if (e == cudaSuccess) e = set_attr((const void *)k_dftb_generic<4>, p.smem, b4);
    p.max_blocks_per_sm = std::max(1, std::min(b2, b4));
    if (p.blocks_per_sm <= 0 || p.blocks_per_sm > p.max_blocks_per_sm) p.blocks_per_sm = p.max_blocks_per_sm;
    return e;
}

// Evaluates the items of the plan: the cells, or their displaced copies when a.n_disp > 0.
cudaError_t launch_dftb_generic(const DevSK *sk, const DftbArgs &a, const GenericPlan &p, cudaStream_t st) {
    const bool disp = a.n_disp > 0;
    const int2 *items = disp ? p.disp_items : p.items;
    const int nb = disp ? p.n_disp_big : p.n_big, ns = disp ? p.n_disp_small : p.n_small;
    const int units = nb + (ns + 1) / 2;
    if (units <= 0) return cudaSuccess;
    unsigned *queue = p.queue + (disp ? 1 : 0);
    cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    const int grid = std::min(units, p.n_sm * std::max(p.blocks_per_sm, 1));
    const void *kernel = p.r_entries == 2 ? dftb_generic_kernel_r2() : (const void *)k_dftb_generic<4>;
    int nmax_b = p.nmax_b, amax_b = p.amax_b, nmax_s = p.nmax_s, amax_s = p.amax_s, n_big = nb, n_small = ns,
        warm = p.warm;
    void *args[] = {(void *)&sk, (void *)&a, (void *)&items, &n_big, &n_small, &queue, &nmax_b, &amax_b, &nmax_s, &amax_s,
                    &warm};
    return cudaLaunchKernel(kernel, dim3(grid), dim3(BT), args, p.smem, st);
}
