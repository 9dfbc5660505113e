// DynaComm DP of listed instances, 17 <= L <= 4096 (Eq. 8 / Algorithm 3 and
// Eq. 9 / Algorithm 4): the pass over the first passes' work lists (dp_mid.cu,
// dp_warp.cu, dp_deep.cu; the lists of L <= 16 are dp_small.cu's own), whose instances
// have values beyond the first pass's range or an optimum deeper than its kept columns. The
// method is in chain.cuh; this pass takes every value (64 bits) and keeps every
// column: one warp per instance with the table in shared memory up to L = 64, otherwise
// one CTA per instance with a table in the caller's workspace.
#include "chain.cuh"

namespace dc {

namespace {

struct GroupArgs {
    int64_t batch;
    int L;
    const int64_t *comp, *xfer, *dt;
    SolveOut out;
    const uint32_t *list_count, *list;
    unsigned char *tables;  // L > 64: the tables of the CTAs
    int vec;                // the cost rows are 16-byte aligned
};

template <bool FWD, int NJ>
__global__ void __launch_bounds__(kChainThreads, 1) group_kernel(GroupArgs a)
{
    const int L = a.L;
    int64_t *table = reinterpret_cast<int64_t *>(a.tables + size_t(blockIdx.x) * size_t(tri_cells(L)) * 8);
    pdl_wait();  // the first pass has finished its list
    const int64_t count = int64_t(*a.list_count);
    for (int64_t j = blockIdx.x; j < count; j += gridDim.x) {
        const int64_t i = int64_t(a.list[j]);
        if (!DC_CHECK(i >= 0 && i < a.batch)) continue;
        chain_solve<FWD, NJ>(i, L,
                             RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0},
                             __ldg(a.dt + i), a.out, KeptValues{table, L});
        __syncthreads();  // shared memory is read
    }
}

// L <= 64: one warp per instance, the table in shared memory, without the CTA form's
// barriers (some 6,000 listed instances of L = 16 took 51 us with that, 33 with this kernel
// on 4 warps per SM).
template <bool FWD>
__global__ void __launch_bounds__(32) list_warp_kernel(GroupArgs a)
{
    const int L = a.L;
    int64_t *table = &sh<int64_t>(chain_pair_bytes(64));
    if (threadIdx.x == 0) zero_row(0, 64);
    pdl_wait();  // the first pass has finished its list
    const int64_t count = int64_t(*a.list_count);
    for (int64_t j = blockIdx.x; j < count; j += gridDim.x) {
        const int64_t i = int64_t(a.list[j]);
        if (!DC_CHECK(i >= 0 && i < a.batch)) continue;
        chain_solve_warp<FWD, 1>(0, i, L,
                                 RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0},
                                 __ldg(a.dt + i), a.out, KeptValues{table, L});
        __syncwarp();  // shared memory is read
    }
}

template <bool FWD, int NJ>
cudaError_t launch_group_nj(const GroupArgs &a, int nt, int64_t grid, cudaStream_t stream)
{
    static DeviceCache attr;  // the kernel's shared-memory limit, raised once per device
    int done = 0;
    const cudaError_t e = attr.get(done, [](int &v) {
        v = 1;
        return cudaFuncSetAttribute(group_kernel<FWD, NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    int(chain_smem_most(DC_L_MAX)));
    });
    if (e != cudaSuccess) return e;
    // launched early: the CTAs wait in hardware until the first pass completes, so the
    // launch overlaps that pass's tail
    return launch_early(group_kernel<FWD, NJ>, grid, nt, chain_smem_bytes(a.L, 2 * NJ * nt), stream, a);
}

template <bool FWD>
cudaError_t launch_group_dir(const GroupArgs &a, int64_t grid, cudaStream_t stream)
{
    if (a.L <= kSmemTableLMax)
        return launch_early(list_warp_kernel<FWD>, grid, 32,
                            chain_pair_bytes(64) + size_t(tri_cells(a.L)) * 8, stream, a);
    // lists are short: two rows per thread, for the shortest column
    int nt = 32 * ((a.L + 63) / 64);
    if (nt > kChainThreads) nt = 32 * ((a.L + 127) / 128);
    // the test hook's warps, where four rows per thread cover the instance
    if (const int f = forced_warps(); f && a.L <= 128 * f) nt = 32 * f;
    return a.L <= 2 * nt ? launch_group_nj<FWD, 1>(a, nt, grid, stream)
                         : launch_group_nj<FWD, 2>(a, nt, grid, stream);
}

}  // namespace

cudaError_t launch_group(bool forward, int64_t batch, int L, const int64_t *comp,
                         const int64_t *xfer, const int64_t *dt, const SolveOut &out, const uint32_t *list_count, const uint32_t *list, void *tables,
                         int64_t grid, cudaStream_t stream)
{
    if (grid <= 0) return cudaSuccess;
    const bool vec = (L % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(xfer)) & 15u) == 0;
    const GroupArgs a{batch, L, comp, xfer, dt, out,
                      list_count, list, static_cast<unsigned char *>(tables), vec ? 1 : 0};
    return forward ? launch_group_dir<true>(a, grid, stream) : launch_group_dir<false>(a, grid, stream);
}

}  // namespace dc

DC_CHECKED_EXPORT(dp_group)
