// Warp-per-instance DynaComm DP for 17 <= L <= 192 (Eq. 8 / Algorithm 3 and Eq. 9 /
// Algorithm 4) by the method of chain.cuh: a column is one binary search per row, and
// there are no more columns than the optimum has segments, plus about one.
//
// Design (GB300):
//  * two rows per lane (L <= 64), four or six. The cost rows are read coalesced straight
//    into registers and scanned by shuffles, in 32 bits with a flag for sums past
//    2^31; the instances it marks run in 64 bits. A column's keys and b sit in the
//    warp's slice of shared memory; there are no CTA barriers;
//  * columns 2..8 are kept for the traceback in shared memory, 9..16 in a slot of the
//    workspace per resident warp; optima deeper than 17 segments, and instances whose
//    useful values span 2^32, go to the work list (dp_group.cu);
//  * the traceback finds Path[m][n], the first k with b[k] at least a bound, by one
//    ballot over the lanes' b;
//  * persistent warps take runs of instances from an atomic ticket, the next run
//    claimed while one is solved.
// Small batches of L <= 64 (use_solo) take one launch without tickets, work list or
// memset: solo_kernel keeps every column, in whole values, in shared memory, so one
// warp solves any instance to the end.
// Bound by integer issue: the searches, the scans and the per-column bookkeeping.
// Measured per direction against the looped thread-per-instance kernel that took
// L <= 256 before (every candidate of every column): 262,144 x 54 (ResNet-50) 185 us
// against 945; 20,000 x 128 80 us against 955; one instance of L = 54 23 us, launches
// included, against 88. Above L = 192 (eight rows per lane) the CTA-per-instance pass
// is as fast on large batches and faster on small ones: 3,000 x 200 66 us against 81.
#include "chain.cuh"

namespace dc {

int sm_count();  // SMs of the current device (dp_small.cu)

namespace {

constexpr int kShared = 8, kLast = 16;  // columns kept in shared memory, and in all
constexpr int kMaxWarpsPerSm = 64;
constexpr int64_t kSlotWarps = 152 * kMaxWarpsPerSm;  // slots of the workspace, at most

struct WarpArgs {
    int64_t batch;
    int L;
    const int64_t *comp, *xfer, *dt;
    SolveOut out;
    uint32_t *ticket;  // runs of instances taken so far (zero before the launch)
    uint32_t *list_count, *list;
    uint32_t *slots;  // columns 9..16, one slot per warp of the grid
    int run;          // instances per run
    int vec;          // the cost rows are 16-byte aligned
};

__host__ __device__ inline size_t warp_smem_bytes(int L)
{
    return (2 * chain_row_bytes(L) + size_t(kShared - 1) * L * 4 + 15) / 16 * 16;
}
__host__ __device__ inline int64_t warp_slot_words(int L) { return int64_t(kLast - kShared) * L; }

template <bool FWD, int NJ>
__global__ void __launch_bounds__(256, NJ == 1 ? 4 : NJ == 2 ? 3 : 2) warp_kernel(WarpArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = a.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned char *mine = smem + size_t(warp) * warp_smem_bytes(L);
    uint32_t *cols = reinterpret_cast<uint32_t *>(mine + 2 * chain_row_bytes(L));
    uint32_t *slot = a.slots + (int64_t(blockIdx.x) * nw + warp) * warp_slot_words(L);
    const int last = L - 1 < kLast ? L - 1 : kLast;
    pdl_trigger();
    auto claim = [&]() {
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(a.ticket, 1u);
        return v;
    };
    int64_t at = int64_t(__shfl_sync(0xffffffffu, claim(), 0)) * a.run;
    while (at < a.batch) {
        const uint32_t next = claim();
        const int64_t end = at + a.run < a.batch ? at + a.run : a.batch;
        for (int64_t i = at; i < end; ++i) {
            const bool solved = chain_solve_warp<FWD, NJ>(
                mine, i, L, RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0},
                __ldg(a.dt + i), a.out,
                [&](int64_t base, uint64_t range, bool &ok) {
                    ok = range < (uint64_t(1) << 32);
                    return KeptOffsets{cols, slot, L, kShared, last, base};
                });
            if (!solved && lane == 0) {
                const uint32_t p = atomicAdd(a.list_count, 1u);
                if (DC_CHECK(int64_t(p) < a.batch)) a.list[p] = uint32_t(i);
            }
            __syncwarp();  // the slice is read
        }
        at = int64_t(__shfl_sync(0xffffffffu, next, 0)) * a.run;
    }
}

template <bool FWD>
__global__ void __launch_bounds__(32) solo_kernel(WarpArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = a.L;
    const int64_t i = blockIdx.x;
    int64_t *table = reinterpret_cast<int64_t *>(smem + 2 * chain_row_bytes(L));
    if (i == 0 && threadIdx.x == 0) *a.list_count = 0u;  // nothing is left to a second pass
    chain_solve_warp<FWD, 1>(smem, i, L,
                             RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0},
                             __ldg(a.dt + i), a.out,
                             [&](int64_t, uint64_t, bool &) { return KeptValues{table, L}; });
}

inline size_t solo_smem_bytes(int L) { return 2 * chain_row_bytes(L) + size_t(tri_cells(L)) * 8; }

template <bool FWD, int NJ>
cudaError_t launch_warp_nj(WarpArgs a, cudaStream_t stream)
{
    static DeviceCache attr;  // the shared-memory limit, raised once per device
    int nw = 4;  // warps per CTA (any number works: the warps are independent)
    if (const int f = forced_warps()) nw = f;
    const size_t smem = size_t(nw) * warp_smem_bytes(a.L);
    int done = 0;
    cudaError_t e = attr.get(done, [](int &v) {
        v = 1;
        return cudaFuncSetAttribute(warp_kernel<FWD, NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    int(8 * warp_smem_bytes(64 * NJ)));
    });
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, warp_kernel<FWD, NJ>, 32 * nw, smem);
    if (e != cudaSuccess) return e;
    if (nb < 1) nb = 1;
    if (nb * nw > kMaxWarpsPerSm) nb = kMaxWarpsPerSm / nw;
    const int64_t warps = int64_t(sm_count()) * nb * nw;
    // runs of up to 16 instances, at least 8 per warp: one atomic per instance would
    // queue at the ticket (about 0.7 claims per ns), longer runs unbalance the end
    int64_t run = a.batch / (warps * 8);
    a.run = int(run < 1 ? 1 : run > 16 ? 16 : run);
    const int64_t runs = (a.batch + a.run - 1) / a.run;
    int64_t grid = (runs + nw - 1) / nw;
    if (grid > int64_t(sm_count()) * nb) grid = int64_t(sm_count()) * nb;
    if (grid > kSlotWarps / nw) grid = kSlotWarps / nw;
    warp_kernel<FWD, NJ><<<unsigned(grid), 32 * nw, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Whether one launch of solo_kernel solves the batch. It saves the memset and the list
// pass (about 4 us on the GPU, more on the host), and a warp per instance starts sooner
// than a thread per instance finishes (per direction, from a graph: one instance of
// L = 16 2.2 us against 6.5, of L = 54 2.3 against 8.2; 4,000 x 16 4.8 us against 27 with
// optima on the work list), but from a wave on it costs about 0.6 us per 1,000 instances:
// 16,000 x 8 10.4 us against 7.6-10.3; 32,000 x 16 19.4 against 30.5 and 32,000 x 32
// 21.9 against 35.7; 32,000 x 64, with 17.7 KB of shared memory a warp, 40.6 against 38.8.
bool use_solo(int64_t batch, int L)
{
    const int64_t most = L <= 8 ? 8000 : L <= 16 ? 24000 : L <= 48 ? 40000 : L <= 64 ? 20000 : 0;
    return batch <= most;
}

cudaError_t launch_solo(bool forward, int64_t batch, int L, const int64_t *comp,
                        const int64_t *xfer, const int64_t *dt, const SolveOut &out, uint32_t *list_count, cudaStream_t stream)
{
    const bool vec = (L % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(xfer)) & 15u) == 0;
    const WarpArgs a{batch, L, comp, xfer, dt, out,
                     nullptr, list_count, nullptr, nullptr, 1, vec ? 1 : 0};
    const size_t smem = solo_smem_bytes(L);  // 17.7 KB at L = 64
    if (forward)
        solo_kernel<true><<<unsigned(batch), 32, smem, stream>>>(a);
    else
        solo_kernel<false><<<unsigned(batch), 32, smem, stream>>>(a);
    return cudaGetLastError();
}

// Slots of the kept columns past shared memory: one per warp of the largest grid, and
// no more than the batch has instances (rounded up to whole CTAs of 8).
size_t warp_scratch_bytes(int64_t batch, int L)
{
    int64_t n = kSlotWarps;
    const int64_t need = (batch + 7) / 8 * 8;
    if (need < n) n = need;
    return size_t(n) * size_t(warp_slot_words(L)) * 4;
}

cudaError_t launch_warp(bool forward, int64_t batch, int L, const int64_t *comp,
                        const int64_t *xfer, const int64_t *dt, const SolveOut &out, uint32_t *ticket, uint32_t *list_count,
                        uint32_t *list, uint32_t *slots, cudaStream_t stream)
{
    const bool vec = (L % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(xfer)) & 15u) == 0;
    const WarpArgs a{batch, L, comp, xfer, dt, out,
                     ticket, list_count, list, slots, 1, vec ? 1 : 0};
    if (L <= 64) return forward ? launch_warp_nj<true, 1>(a, stream) : launch_warp_nj<false, 1>(a, stream);
    if (L <= 128) return forward ? launch_warp_nj<true, 2>(a, stream) : launch_warp_nj<false, 2>(a, stream);
    return forward ? launch_warp_nj<true, 3>(a, stream) : launch_warp_nj<false, 3>(a, stream);
}

}  // namespace dc

DC_CHECKED_EXPORT(dp_warp)
