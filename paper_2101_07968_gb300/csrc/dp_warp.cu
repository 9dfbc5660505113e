// Warp-per-instance DynaComm DP for 17 <= L <= 192 (Eq. 8 / Algorithm 3 and Eq. 9 /
// Algorithm 4) by the method of chain.cuh: a column is one binary search per row, and
// there are no more columns than the optimum has segments, plus about one.
//
// Design (GB300):
//  * two rows per lane (L <= 64), four or six. The cost rows are read coalesced straight
//    into registers and scanned by shuffles, in 32 bits with a flag for sums past
//    2^31; the instances it marks run in 64 bits. A column's keys and b sit in the
//    warp's slice of shared memory; there are no CTA barriers;
//  * columns 1..8 are kept for the traceback in shared memory, 9..24 in a slot of the
//    workspace per resident warp; optima deeper than 25 segments, and instances whose
//    useful values span 2^32 (see KeptWords), go to the work list (dp_group.cu);
//  * the traceback finds Path[m][n], the first k with b[k] at least a bound, by one
//    ballot over the lanes' b;
//  * persistent warps solve an equal share of the batch each, then runs of instances
//    from an atomic ticket, the next run claimed while one is solved.
// Small batches of L <= 64 (use_solo) take one launch without tickets, work list or
// memset: solo_kernel keeps every column, in whole values, in shared memory, so one
// warp solves any instance to the end.
// Bound by integer issue (0.7 of the slots while all warps run) and, on small batches, by
// the deepest instances at the end. Measured per direction against the looped
// thread-per-instance kernel that took L <= 256 before (every candidate of every
// column): 262,144 x 54 (ResNet-50) 155 us against 945; 20,000 x 128 45 us against 955.
// Above L = 192 (eight rows per lane) the CTA-per-instance pass is as fast on large
// batches and faster on small ones: 3,000 x 200 66 us against 81.
#include "chain.cuh"

namespace dc {

int sm_count();  // SMs of the current device (dp_small.cu)

namespace {

constexpr int kShared = 8, kLast = 24;  // columns kept in shared memory, and in all
constexpr int kMaxWarpsPerSm = 64;
constexpr int64_t kSlotWarps = 152 * kMaxWarpsPerSm;  // slots of the workspace, at most

struct WarpArgs {
    int64_t batch;
    int L;
    const int64_t *comp, *xfer, *dt;
    SolveOut out;
    uint32_t *ticket;  // runs of instances taken so far (zero before the launch)
    uint32_t *list_count, *list;
    uint32_t *slots;  // columns 9..24, one slot per warp of the grid
    int own;          // instances of each warp's own, before the ticket's
    int run;          // instances per run of the ticket
    int vec;          // the cost rows are 16-byte aligned
};

// K and b of 64 NJ rows, then the kept columns
__host__ __device__ inline int warp_smem_bytes(int L, int nj)
{
    return (chain_pair_bytes(64 * nj) + kShared * chain_stride(L) * 4 + 15) / 16 * 16;
}
__host__ __device__ inline int64_t warp_slot_words(int L) { return int64_t(kLast - kShared) * chain_stride(L); }

template <bool FWD, int NJ>
__global__ void __launch_bounds__(256, NJ == 1 ? 4 : NJ == 2 ? 3 : 2) warp_kernel(WarpArgs a)
{
    const int L = a.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int kb = warp * warp_smem_bytes(L, NJ), cols = kb + chain_pair_bytes(64 * NJ);
    if (lane == 0) zero_row(kb, 64 * NJ);
    uint32_t *slot = a.slots + (int64_t(blockIdx.x) * nw + warp) * warp_slot_words(L);
    const KeptWords kept{cols, slot, chain_stride(L), kShared, L - 1 < kLast ? L - 1 : kLast};
    pdl_trigger();
    auto claim = [&]() {
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(a.ticket, 1u);
        __syncwarp();  // see the end of chain_columns
        return v;
    };
    // first this warp's own share, then runs from the ticket (claimed one ahead)
    const int64_t gw = int64_t(blockIdx.x) * nw + warp;
    const int64_t shared_from = a.own * int64_t(gridDim.x) * nw;
    uint32_t next = claim();
    int64_t at = gw * a.own, end = at + a.own;
    for (;;) {
        const int64_t *crow = a.comp + at * L, *xrow = a.xfer + at * L;
        for (int64_t i = at; i < end; ++i, crow += L, xrow += L) {
            const bool solved = chain_solve_warp<FWD, NJ>(
                kb, i, L, RowLoader<FWD>{crow, xrow, L, a.vec != 0}, __ldg(a.dt + i), a.out, kept);
            if (!solved && lane == 0) {
                const uint32_t p = atomicAdd(a.list_count, 1u);
                if (DC_CHECK(int64_t(p) < a.batch)) a.list[p] = uint32_t(i);
            }
            __syncwarp();  // the slice is read
        }
        at = shared_from + int64_t(__shfl_sync(0xffffffffu, next, 0)) * a.run;
        if (at >= a.batch) break;
        end = at + a.run < a.batch ? at + a.run : a.batch;
        next = claim();
    }
}

template <bool FWD>
__global__ void __launch_bounds__(32) solo_kernel(WarpArgs a)
{
    const int L = a.L;
    const int64_t i = blockIdx.x;
    int64_t *table = &sh<int64_t>(chain_pair_bytes(64));
    if (threadIdx.x == 0) zero_row(0, 64);
    if (i == 0 && threadIdx.x == 0) *a.list_count = 0u;  // nothing is left to a second pass
    chain_solve_warp<FWD, 1>(0, i, L,
                             RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0},
                             __ldg(a.dt + i), a.out, KeptValues{table, L});
}

inline size_t solo_smem_bytes(int L) { return chain_pair_bytes(64) + size_t(tri_cells(L)) * 8; }

template <bool FWD, int NJ>
cudaError_t launch_warp_nj(WarpArgs a, cudaStream_t stream)
{
    static DeviceCache attr;  // the shared-memory limit, raised once per device
    int nw = 4;  // warps per CTA (any number works: the warps are independent)
    if (const int f = forced_warps()) nw = f;
    const size_t smem = size_t(nw) * warp_smem_bytes(a.L, NJ);
    int done = 0;
    cudaError_t e = attr.get(done, [](int &v) {
        v = 1;
        return cudaFuncSetAttribute(warp_kernel<FWD, NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    8 * warp_smem_bytes(64 * NJ, NJ));
    });
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, warp_kernel<FWD, NJ>, 32 * nw, smem);
    if (e != cudaSuccess) return e;
    if (nb < 1) nb = 1;
    if (nb * nw > kMaxWarpsPerSm) nb = kMaxWarpsPerSm / nw;
    int64_t grid = (a.batch + nw - 1) / nw;
    if (grid > int64_t(sm_count()) * nb) grid = int64_t(sm_count()) * nb;
    if (grid > kSlotWarps / nw) grid = kSlotWarps / nw;
    // The ticket takes about 1.2 claims per ns: with one claim per instance it alone took
    // 55 us for 65,536 instances of L = 54. So each warp starts with three quarters of an
    // equal share of its own, and only the rest comes from the ticket, in runs of up to 8,
    // for the balance at the end (without shares, single instances from the ticket: 20,011
    // x 129 113 us a direction against 107, 60,000 x 100 119 against 109).
    const int64_t warps = grid * nw, share = a.batch / warps;
    a.own = int(share >= 4 ? share * 3 / 4 : 0);
    const int64_t run = (a.batch - a.own * warps) / (warps * 2);
    a.run = int(run < 1 ? 1 : run > 8 ? 8 : run);
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
                     nullptr, list_count, nullptr, nullptr, 0, 1, vec ? 1 : 0};
    const size_t smem = solo_smem_bytes(L);  // 17.7 KB at L = 64
    if (forward)
        solo_kernel<true><<<unsigned(batch), 32, smem, stream>>>(a);
    else
        solo_kernel<false><<<unsigned(batch), 32, smem, stream>>>(a);
    return cudaGetLastError();
}

// Slots of the kept columns past shared memory: one per warp of the largest grid, and
// no more than the batch has instances (rounded up to whole CTAs of 8). The solo kernel
// keeps its columns on chip.
size_t warp_scratch_bytes(int64_t batch, int L)
{
    if (use_solo(batch, L)) return 0;
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
                     ticket, list_count, list, slots, 0, 1, vec ? 1 : 0};
    if (L <= 64) return forward ? launch_warp_nj<true, 1>(a, stream) : launch_warp_nj<false, 1>(a, stream);
    if (L <= 128) return forward ? launch_warp_nj<true, 2>(a, stream) : launch_warp_nj<false, 2>(a, stream);
    return forward ? launch_warp_nj<true, 3>(a, stream) : launch_warp_nj<false, 3>(a, stream);
}

}  // namespace dc

DC_CHECKED_EXPORT(dp_warp)
