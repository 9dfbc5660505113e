// CTA-per-instance DynaComm DP for 193 <= L <= 4096 (Eq. 8 / Algorithm 3 and
// Eq. 9 / Algorithm 4): the first pass over a deep batch. The method is in
// chain.cuh: O(L log L) per column, and no more columns than the optimum has
// segments, plus about one.
//
// Design (GB300):
//  * an instance per CTA of up to 32 warps, two or four rows per thread
//    (deep_threads): a column is one independent binary search per row in shared
//    memory, so every thread works in every column; a thread's searches run two at
//    a time to overlap their shared-memory latency, and the other CTAs of the SM
//    hide the rest; from 640 layers on it starts where the last column's ended;
//  * what bounds it: integer issue in the searches (L log2 L steps of 3 to 4
//    instructions a column) and the two CTA barriers of a column; the profiles are
//    read once (16 L bytes per instance and direction) and the columns kept for the
//    traceback stay in L2;
//  * a column is updated in place: every thread's results wait in registers for a
//    barrier, then they are written;
//  * 32-bit values where the instance's sums fit, otherwise 64-bit (two in five
//    instances of the deep chain), chosen per instance. Columns 1..64 are kept as
//    32-bit words, the first in shared memory, the rest in a slot of the workspace per
//    resident CTA; optima deeper than 65
//    segments, and the rare instances whose values do not fit (see KeptWords), go to
//    the work list (dp_group.cu, whole values, every column);
//  * persistent CTAs take instances from a per-launch ticket, and a long batch of
//    L > 256 is split into launches of four resident waves, so that kernels of other
//    streams get their turn on the GPU between them. The launches are chained by
//    programmatic dependent launch: each may fill the SMs as the one before drains.
//    A CTA claims a free slot from a bitmap for as long as it lives.
//
// Measured, both directions together: 16,384 instances of L = 1024 in 0.88 ms, and
// 383 of L = 1023 in 0.102 ms (1.65 and 0.21 ms with 64-bit values only, eight rows
// per thread and two key buffers; 532 and 20.5 ms for the fill of all L columns over
// every candidate).
#include "chain.cuh"

namespace dc {

int sm_count();  // SMs of the current device (dp_small.cu)

namespace {

// From this depth on a search first looks at the 32 keys from where it ended in the column
// before: 83 to 90 in 100 end there on the deep chain, in 6 steps instead of 10. Both
// directions: 5,000 x 2,047 824 us -> 754, 16,384 x 1,024 924 -> 880, 10,000 x 700 428 ->
// 417; but 24,000 x 512 564 -> 573, whose searches are 9 steps, and nothing at 300.
constexpr int kWindowMinL = 640;
constexpr int kSplitLMin = 256;  // longer batches are split into launches above this depth
constexpr int kSmemPerSm = 227 * 1024;
constexpr int kKeep = 64;  // columns 1..kKeep kept for the traceback

__host__ __device__ inline size_t slot_bytes(int L)
{
    const int last = L - 1 < kKeep ? L - 1 : kKeep;
    return (size_t(last) * chain_stride(L) * 4 + 255) / 256 * 256;
}

struct DeepArgs {
    int64_t lo, count;  // this launch solves instances lo .. lo + count - 1
    int L;
    const int64_t *comp, *xfer, *dt;
    SolveOut out;
    uint32_t *ticket;             // instances taken so far (zero before the launch)
    uint32_t *list_count, *list;  // instances left to the work-list pass
    uint32_t *busy;               // slot bitmap: bit set while a CTA holds the slot (zero before the first launch)
    unsigned char *slots;
    size_t slot_bytes;
    int nslots;
    int vec;     // the cost rows are 16-byte aligned
    int shared;  // kept columns in shared memory, the rest in the slot
};

// A free slot, or -1: at most one resident wave of CTAs lives at a time, over this
// launch and the next, and there are at least that many slots. Each bitmap word
// is tried from a free bit until one is won or none is left.
__device__ int claim_slot(uint32_t *busy, int nslots)
{
    const int nw = (nslots + 31) / 32;
    for (int p = 0; p < nw; ++p) {
        const int w = int((blockIdx.x / 32u + unsigned(p)) % unsigned(nw));
        const int nbits = min(32, nslots - 32 * w);
        const uint32_t full = nbits == 32 ? 0xffffffffu : ((1u << nbits) - 1u);
        uint32_t v = *reinterpret_cast<volatile uint32_t *>(busy + w);
        for (int tries = 0; tries < 32 && (v & full) != full; ++tries) {
            const int b = __ffs(int(~v & full)) - 1;
            const uint32_t old = atomicOr(busy + w, 1u << b);
            if (!(old & (1u << b))) return 32 * w + b;
            v = old | (1u << b);
        }
    }
    return -1;
}

template <bool FWD, int NJ, int WINDOW>
__global__ void __launch_bounds__(kChainThreads, 1) deep_kernel(DeepArgs a)
{
    __shared__ int s_slot;
    __shared__ uint32_t s_taken;
    const int L = a.L, tid = threadIdx.x;
    // the next launch of a split batch may start filling SMs as this one's CTAs
    // exit; it shares no data with this one
    pdl_trigger();
    if (tid == 0) s_slot = claim_slot(a.busy, a.nslots);
    __syncthreads();
    const int slot = s_slot;
    if (slot < 0 || !DC_CHECK(slot < a.nslots)) {  // every slot held (not expected):
        pdl_wait();                                // leave the instances to the other CTAs
        return;
    }
    uint32_t *at = reinterpret_cast<uint32_t *>(a.slots + size_t(slot) * a.slot_bytes);
    const int cols = int((chain_smem_bytes(L, 2 * NJ * int(blockDim.x)) + 15) / 16 * 16);
    const KeptWords kept{cols, at, chain_stride(L), a.shared, L - 1 < kKeep ? L - 1 : kKeep};
    for (;;) {
        if (tid == 0) s_taken = atomicAdd(a.ticket, 1u);
        __syncthreads();
        const uint32_t taken = s_taken;
        if (int64_t(taken) >= a.count) break;
        const int64_t i = a.lo + int64_t(taken);
        const bool solved = chain_solve<FWD, NJ, WINDOW>(
            i, L, RowLoader<FWD>{a.comp + i * L, a.xfer + i * L, L, a.vec != 0}, __ldg(a.dt + i),
            a.out, kept);
        if (!solved && tid == 0) {
            const uint32_t p = atomicAdd(a.list_count, 1u);
            if (DC_CHECK(int64_t(p) < a.lo + a.count)) a.list[p] = uint32_t(i);
        }
        __syncthreads();  // shared memory and s_taken are read
    }
    // release the slot, then finish no earlier than the previous launch of the
    // batch, so that a kernel waiting for the last launch waits for them all
    if (tid == 0) {
        __threadfence();
        atomicAnd(a.busy + slot / 32, ~(1u << (slot % 32)));
    }
    pdl_wait();
}

}  // namespace

size_t deep_slot_bytes(int L) { return slot_bytes(L); }

// Resident CTAs per SM for depth L: a bound from shared memory alone (the workspace
// is sized from it on the host, without a device query).
int64_t deep_slots_bound(int L)
{
    const size_t per = chain_smem_bytes(L, L) + 1024;  // the runtime reserves 1 KB per CTA
    int64_t n = int64_t((228 * 1024) / per);
    if (n > 32) n = 32;
    if (n < 1) n = 1;
    return 152 * n;
}

namespace {

// Threads per instance: four rows per thread (two row pairs, whose searches hide each
// other's latency) for long rows on a full GPU, two per thread otherwise, for shorter
// columns and tracebacks. Measured per direction, two rows against four: 40,000 x 300
// 296 us against 323, 383 x 1023 56 against 70, 2,432 x 1024 (256 warps per SM in all)
// 108 against 109, 4,864 x 1024 179 against 165, 24,000 x 512 299 against 275.
int deep_threads(int64_t count, int L, int sms)
{
    const int nt2 = 32 * ((L + 127) / 128), nt1 = 32 * ((L + 63) / 64);
    if (nt1 > kChainThreads) return nt2;
    return L <= 384 || count * (nt1 / 32) <= int64_t(sms) * 256 ? nt1 : nt2;
}

template <bool FWD, int NJ, int WINDOW>
cudaError_t launch_deep_nj(DeepArgs a, int nt, bool pdl, cudaStream_t stream)
{
    static DeviceCache attr;
    int done = 0;
    cudaError_t e = attr.get(done, [](int &v) {
        v = 1;
        return cudaFuncSetAttribute(deep_kernel<FWD, NJ, WINDOW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kSmemPerSm - 1024);
    });
    if (e != cudaSuccess) return e;
    // The kernel's 64 registers allow 1,024 threads on an SM; the shared memory that
    // leaves a CTA holds its first columns (9 at L = 1024), so that the traceback of
    // most instances does not wait for L2 at every step
    const size_t fixed = (chain_smem_bytes(a.L, 2 * NJ * nt) + 15) / 16 * 16;
    const int ctas = 1024 / nt > 32 ? 32 : 1024 / nt < 1 ? 1 : 1024 / nt;
    const size_t room = size_t(kSmemPerSm) / ctas - 1024, col = size_t(chain_stride(a.L)) * 4;
    a.shared = room > fixed ? int((room - fixed) / col) : 0;
    if (a.shared > a.L - 1) a.shared = a.L - 1;
    if (a.shared > kKeep) a.shared = kKeep;
    const size_t smem = fixed + a.shared * col;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, deep_kernel<FWD, NJ, WINDOW>, nt, smem);
    if (e != cudaSuccess) return e;
    int64_t grid = int64_t(nb < 1 ? 1 : nb) * sm_count();
    if (grid > a.nslots) grid = a.nslots;
    if (grid > a.count) grid = a.count;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(unsigned(grid));
    lc.blockDim = dim3(unsigned(nt));
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&lc, deep_kernel<FWD, NJ, WINDOW>, a);
}

template <bool FWD>
cudaError_t launch_deep_dir(const DeepArgs &a, bool pdl, cudaStream_t stream)
{
    int nt = deep_threads(a.count, a.L, sm_count());
    // the test hook's warps, where four rows per thread cover the instance
    if (const int f = forced_warps(); f && a.L <= 128 * f) nt = 32 * f;
    if (a.L < kWindowMinL)
        return a.L <= 2 * nt ? launch_deep_nj<FWD, 1, 0>(a, nt, pdl, stream)
                             : launch_deep_nj<FWD, 2, 0>(a, nt, pdl, stream);
    return a.L <= 2 * nt ? launch_deep_nj<FWD, 1, 32>(a, nt, pdl, stream)
                         : launch_deep_nj<FWD, 2, 32>(a, nt, pdl, stream);
}

// Instances per launch: four resident waves above L = 256, the whole batch below.
int64_t deep_per_launch(int64_t batch, int L)
{
    if (L <= kSplitLMin) return batch;
    const int64_t per = 4 * deep_slots_bound(L);
    if (per >= batch) return batch;
    const int64_t n = (batch + per - 1) / per;  // equal shares
    return (batch + n - 1) / n;
}

}  // namespace

int64_t deep_launches(int64_t batch, int L)
{
    if (batch <= 0) return 0;
    const int64_t per = deep_per_launch(batch, L);
    return (batch + per - 1) / per;
}

cudaError_t launch_deep(bool forward, int64_t batch, int L, const int64_t *comp,
                        const int64_t *xfer, const int64_t *dt, const SolveOut &out, uint32_t *tickets,
                        uint32_t *busy, uint32_t *list_count, uint32_t *list, void *slots,
                        int64_t nslots, cudaStream_t stream)
{
    if (batch <= 0) return cudaSuccess;
    const bool vec = (L % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(xfer)) & 15u) == 0;
    const int64_t per = deep_per_launch(batch, L);
    // every launch's ticket and every slot's flag start at zero (adjacent in the
    // workspace: the flags' words lie in the first nslots words)
    cudaError_t e = cudaMemsetAsync(busy, 0, size_t((nslots + 31) / 32) * 4, stream);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(tickets, 0, size_t(deep_launches(batch, L)) * 4, stream);
    if (e != cudaSuccess) return e;
    int64_t k = 0;
    for (int64_t lo = 0; lo < batch; lo += per, ++k) {
        const int64_t count = batch - lo < per ? batch - lo : per;
        DeepArgs a{lo, count, L, comp, xfer, dt, out,
                   tickets + k, list_count, list, busy, static_cast<unsigned char *>(slots),
                   slot_bytes(L), int(nslots), vec ? 1 : 0, 0};
        // the first launch waits for the memsets in stream order; later ones may
        // overlap the tail of the one before
        e = forward ? launch_deep_dir<true>(a, k > 0, stream)
                    : launch_deep_dir<false>(a, k > 0, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dc

DC_CHECKED_EXPORT(dp_deep)
