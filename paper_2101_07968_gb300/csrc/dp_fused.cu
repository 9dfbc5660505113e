// Generate-and-solve for 1 <= L <= 16 (dc_schedule_generated_batch, dc_step_batch): the
// short-L passes of dp_small.cu with each tile's rows drawn inside the kernel by the
// profile generator's device functions instead of being read from memory; small batches
// take one launch of the chain solver on drawn rows (fused_solo_kernel).
#include "chain.cuh"
#include "dp_small.cuh"

namespace dc {
namespace {

// ---------------------------------------------------------------------------
// Generate and solve in one pass (no profile round trip through HBM): each lane
// draws its instance's rows with the profile generator's own device functions
// into its row of the staging area, then the tile is solved as in dp_small.cu.
// Both directions come from one draw of the rows (fused_pair_kernel): the forward
// and backward U, V rows are derived from the staged rows and saved in the lane's
// slice, and one copy of the solve, with the direction as a runtime argument,
// runs once per direction (two unrolled copies overflow the instruction cache).
// Each direction has its own list pass, which regenerates the listed instances'
// rows.
// workspace: [0, 256) the two list counters and the tile ticket,
// [256, 256 + 8 batch) the two lists, then the generator's tables
inline size_t fused_tables_offset(int64_t batch) { return (256 + 8 * size_t(batch) + 255) / 256 * 256; }

struct FusedOut {
    SolveOut out[2];
    // STORE: the drawn profiles; pairs: 16-byte aligned
    int64_t *fc, *pt, *bc, *gt, *dt;
    int pairs;
    uint32_t *wide_count[2], *wide_list[2];
    uint32_t *ticket;  // tiles handed out (zero before the launch)
};

// The generator's lookup tables, copied once per call from the parameter block
// into the workspace: lanes index them with their own draws, which global loads
// serve in parallel where the parameter (constant) path serialises them.
struct GenTables {
    int64_t rate[kKnots + 1], bw[kKnots + 1];
    LayerRow layer[kFixedMax];
};

__global__ void __launch_bounds__(256) copy_tables_kernel(const __grid_constant__ GenParams g,
                                                          GenTables *t)
{
    const int nl = g.layer_mode == DC_LAYERS_FIXED ? g.L
                   : (g.layer_mode == DC_LAYERS_LOGUNIFORM ? kKnots + 1 : 0);
    if (g.rate_dist == DC_DIST_LOGUNIFORM)
        for (int j = threadIdx.x; j <= kKnots; j += blockDim.x) t->rate[j] = g.rate_knots[j];
    if (g.bw_dist == DC_DIST_LOGUNIFORM)
        for (int j = threadIdx.x; j <= kKnots; j += blockDim.x) t->bw[j] = g.bw_knots[j];
    for (int j = threadIdx.x; j < nl; j += blockDim.x) t->layer[j] = g.layer[j];
}

// Shared memory of a warp of the pair pass, per lane (lane-interleaved words):
// the backward U, V at [0, 2(L+1)), then the table, whose first 2(L+1) words hold
// the forward U, V until the forward solve loads them; the tile's staged rows
// (compute forward, compute backward, transfer, at the padded stride) overlap it
// all, being read before any of it is written.
template <int L>
struct Pair32 {
    static constexpr int kUV = 2 * (L + 1);
    static constexpr int kTab = Tab32<L>::kWords > kUV ? Tab32<L>::kWords : kUV;
    static constexpr int kSlotBytes = 32 * (kUV + kTab) * 4;
    static constexpr int kRowsBytes = 3 * 32 * Tab32<L>::kStride * 8;
    static constexpr int kBytes = kRowsBytes > kSlotBytes ? kRowsBytes : kSlotBytes;
};

// Both directions of each instance from one draw of its rows. STORE: a whole step, which
// also writes the profiles out, coalesced from the staged rows, and f_m of the decisions:
// the writes run under the solve (1,000,000 x 8: 99 us, 115 as a generator pass that
// writes and two solves that read; at L = 16 the solve binds and both take 204).
template <int L, bool STORE>
__global__ void __launch_bounds__(32, DC_SMALL_MINB)
    fused_pair_kernel(const __grid_constant__ GenParams g, const GenTables *t, const FusedOut o)
{
    using K = Tab32<L>;
    using P = Pair32<L>;
    constexpr int W = (L - 1 + 31) / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x;
    int64_t *stF = reinterpret_cast<int64_t *>(smem) + lane * K::kStride;
    int64_t *stB = stF + 32 * K::kStride;
    int64_t *stX = stB + 32 * K::kStride;
    int32_t *uvb = reinterpret_cast<int32_t *>(smem) + lane;  // backward U, V
    int32_t *lw = uvb + 32 * P::kUV;                           // table; forward U, V first
    const int64_t tiles = (g.batch + 31) / 32;
    pdl_trigger();
    auto solve_tile = [&](int64_t tile) {
        const int64_t i = tile * 32 + lane;
        const bool active = i < g.batch;
        const int64_t gi = g.inst0 + i;
        int64_t dti = 0;
        __syncwarp();  // every lane is done with the area (the previous tile's table)
        if (active && g.words) {
            // rolled: unrolled, the generator's divisions and the DP overflow the
            // instruction cache
            const WordDraws d = word_draws(g, t->rate, t->bw, gi);
            dti = d.dt;
#pragma unroll 1
            for (int l = 0; l < L; ++l) {
                int64_t wire, flops;
                uint32_t f, x;
                uint64_t b;
                layer_numerators(g, t->layer, gi, l, wire, flops);
                word_costs(g, d.rate, d.bw, uint64_t(wire), uint64_t(flops), f, b, x);
                stF[l] = int64_t(uint64_t(f));
                stB[l] = int64_t(b);
                stX[l] = int64_t(uint64_t(x));
            }
        } else if (active) {
            const InstanceDraws d = instance_draws(g, t->rate, t->bw, gi);
            dti = d.dt;
#pragma unroll 1
            for (int l = 0; l < L; ++l) {
                int64_t wire, flops, f, b, x;
                layer_numerators(g, t->layer, gi, l, wire, flops);
                wire_costs(g, d, uint64_t(wire), uint64_t(flops), f, b, x);
                stF[l] = f;
                stB[l] = b;
                stX[l] = x;
            }
        }
        if constexpr (STORE) {
            __syncwarp();
            const int64_t *sf = reinterpret_cast<const int64_t *>(smem);
            const int64_t *sb = sf + 32 * K::kStride, *sx = sb + 32 * K::kStride;
            const int rows = int(g.batch - tile * 32 < 32 ? g.batch - tile * 32 : 32);
            const int64_t o0 = tile * 32 * L;
            if (L % 2 == 0 && o.pairs) {
                constexpr int H = L / 2 > 0 ? L / 2 : 1;  // pairs per row
                for (int p = lane; p < rows * H; p += 32) {
                    const int r = p / H, at = r * K::kStride + 2 * (p - r * H);
                    const longlong2 x = *reinterpret_cast<const longlong2 *>(sx + at);
                    *reinterpret_cast<longlong2 *>(o.fc + o0 + 2 * p) = *reinterpret_cast<const longlong2 *>(sf + at);
                    *reinterpret_cast<longlong2 *>(o.bc + o0 + 2 * p) = *reinterpret_cast<const longlong2 *>(sb + at);
                    *reinterpret_cast<longlong2 *>(o.pt + o0 + 2 * p) = x;
                    *reinterpret_cast<longlong2 *>(o.gt + o0 + 2 * p) = x;
                }
            } else {
                for (int e = lane; e < rows * L; e += 32) {
                    const int r = e / L, at = r * K::kStride + (e - r * L);
                    o.fc[o0 + e] = sf[at];
                    o.bc[o0 + e] = sb[at];
                    o.pt[o0 + e] = sx[at];
                    o.gt[o0 + e] = sx[at];
                }
            }
            if (active) o.dt[i] = dti;
        }
        uint64_t xraw[2];
        bool wide[2];
        int st[2];
        {
            int32_t Uf[L + 1], Vf[L + 1], Ub[L + 1], Vb[L + 1];
            row_uv<L, true>(stF, stX, dti, Uf, Vf, xraw[0], wide[0], st[0]);
            row_uv<L, false>(stB, stX, dti, Ub, Vb, xraw[1], wide[1], st[1]);
            __syncwarp();  // rows read: the lanes' slices may be written
#pragma unroll
            for (int m = 0; m <= L; ++m) {
                lw[32 * m] = Uf[m];
                lw[32 * (L + 1 + m)] = Vf[m];
                uvb[32 * m] = Ub[m];
                uvb[32 * (L + 1 + m)] = Vb[m];
            }
        }
#pragma unroll 1
        for (int dir = 0; dir < 2; ++dir) {
            const bool fwd = dir == 0;
            const int32_t *uv = fwd ? lw : uvb;
            int32_t U[L + 1], V[L + 1];
#pragma unroll
            for (int m = 0; m <= L; ++m) {
                U[m] = uv[32 * m];
                V[m] = uv[32 * (L + 1 + m)];
            }
            // selected, not indexed by `dir`: an index would put the pairs on the stack
            const int std = fwd ? st[0] : st[1];
            const bool wd = fwd ? wide[0] : wide[1];
            const uint64_t xd = fwd ? xraw[0] : xraw[1];
            const SolveOut od = fwd ? o.out[0] : o.out[1];
            const bool done = solve_uv<L, STORE, kKeepCols>(fwd, active && std == DC_OK && !wd, U, V, int32_t(dti),
                                                 xd, lw, i, od);
            if (active && std != DC_OK) {
                write_failure(std, i, W, od);
            } else if (active && (wd || !done)) {
                uint32_t *count = fwd ? o.wide_count[0] : o.wide_count[1];
                uint32_t *list = fwd ? o.wide_list[0] : o.wide_list[1];
                const uint32_t at = atomicAdd(count, 1u);
                if (DC_CHECK(int64_t(at) < g.batch)) list[at] = uint32_t(i);
            }
        }
    };
    if constexpr (L >= kSplitMinL) {
        // tiles from a ticket, the next claimed while this one is solved
        auto claim = [&]() {
            uint32_t v = 0;
            if (lane == 0) v = atomicAdd(o.ticket, 1u);
            return v;
        };
        int64_t tile = int64_t(__shfl_sync(0xffffffffu, claim(), 0));
        while (tile < tiles) {
            const uint32_t next_raw = claim();
            solve_tile(tile);
            tile = int64_t(__shfl_sync(0xffffffffu, next_raw, 0));
        }
    } else {
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) solve_tile(tile);
    }
}

// The costs of one instance's rows in processing order, drawn (see RowLoader).
template <bool FWD>
struct DrawLoader {
    const GenParams &g;
    const LayerRow *layer;
    const InstanceDraws &d;
    int64_t gi;
    __device__ __forceinline__ void row(int r, uint64_t &c, uint64_t &x) const
    {
        c = x = 0;
        if (r > g.L) return;
        int64_t wire, flops, f, b, v;
        layer_numerators(g, layer, gi, FWD ? r - 1 : g.L - r, wire, flops);
        wire_costs(g, d, uint64_t(wire), uint64_t(flops), f, b, v);
        c = uint64_t(FWD ? f : b);
        x = uint64_t(v);
    }
    __device__ __forceinline__ void operator()(int r, uint64_t &c0, uint64_t &c1, uint64_t &x0,
                                               uint64_t &x1) const
    {
        row(r, c0, x0);
        row(r + 1, c1, x1);
    }
};

// Pass over one direction's list, rows regenerated (see small_list_kernel).
template <int L, bool FWD>
__global__ void __launch_bounds__(32 * List64<L, true>::kWarps)
    fused_list_kernel(const __grid_constant__ GenParams g, const GenTables *t, const FusedOut o)
{
    static_assert(Table<L, int64_t, L>::kWords >= 2 * L, "a lane's rows lie where its table will");
    constexpr int dir = FWD ? 0 : 1;
    pdl_wait();  // the passes ahead of this one have finished
    list_pass<L, true>(
        g.batch, int64_t(*o.wide_count[dir]), o.wide_list[dir],
        [&](int kb, int64_t i, const KeptValues &kept) {
            const InstanceDraws d = instance_draws(g, t->rate, t->bw, g.inst0 + i);
            chain_solve_warp<FWD, 1>(kb, i, L, DrawLoader<FWD>{g, t->layer, d, g.inst0 + i}, d.dt,
                                     o.out[dir], kept);
        },
        [&](bool active, int64_t i) {
            int64_t *row = &sh<int64_t>(8 * int(threadIdx.x)), dti = 0;
            if (active) {
                const InstanceDraws d = instance_draws(g, t->rate, t->bw, g.inst0 + i);
                dti = d.dt;
#pragma unroll 1
                for (int l = 0; l < L; ++l) {
                    int64_t wire, flops, f, b, x;
                    layer_numerators(g, t->layer, g.inst0 + i, l, wire, flops);
                    wire_costs(g, d, uint64_t(wire), uint64_t(flops), f, b, x);
                    row[32 * l] = FWD ? f : b;
                    row[32 * (L + l)] = x;
                }
            }
            list_solve_lane<L, FWD>(
                active, i, dti,
                [&](int col, int64_t &cv, int64_t &xv) {
                    cv = row[32 * col];
                    xv = row[32 * (L + col)];
                },
                o.out[dir]);
        });
}

template <int L, bool FWD>
cudaError_t launch_fused_list(const GenParams &g, const GenTables *t, const FusedOut &o,
                              cudaStream_t stream)
{
    static DeviceCache listers;
    return launch_list<L, true>(listers, g.batch, stream, fused_list_kernel<L, FWD>, g, t, o);
}

// Small batches, one launch: warp 0 of a CTA draws two instances' rows, one layer to a
// lane, and writes them out (STORE); then each of the four warps solves one instance in
// one direction with every column on chip, as solo_kernel does. The tables are read from
// the parameter block, where only the layers' lookups diverge. Bound by integer issue
// (drawn by each warp for itself, two layers to a lane, the kernel took twice as long).
constexpr int kSoloInstances = 2;
__host__ __device__ inline int fused_solo_bytes(int L)
{
    return chain_pair_bytes(64) + (int(tri_cells(L)) * 8 + 15) / 16 * 16;
}

// The costs of one instance's drawn rows in processing order (see RowLoader).
template <bool FWD>
struct DrawnLoader {
    const int64_t *comp, *xfer;  // shared memory, layer order
    int L;
    __device__ __forceinline__ void operator()(int r, uint64_t &c0, uint64_t &c1, uint64_t &x0,
                                               uint64_t &x1) const
    {
        c0 = c1 = x0 = x1 = 0;
        if (r > L) return;
        const int at = FWD ? r - 1 : L - r, next = FWD ? at + 1 : at - 1;
        c0 = uint64_t(comp[at]);
        x0 = uint64_t(xfer[at]);
        if (r < L) {
            c1 = uint64_t(comp[next]);
            x1 = uint64_t(xfer[next]);
        }
    }
};

template <bool STORE>
__global__ void __launch_bounds__(64 * kSoloInstances)
    fused_solo_kernel(const __grid_constant__ GenParams g, const FusedOut o)
{
    static_assert(kSoloInstances == 2 && kSmallLMax == 16, "a half warp draws an instance");
    __shared__ int64_t rows[kSoloInstances][3][kSmallLMax], dts[kSoloInstances];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, L = g.L;
    const int64_t i0 = int64_t(blockIdx.x) * kSoloInstances;
    if (warp == 0) {
        const int h = lane >> 4, l = lane & 15;
        const bool there = i0 + h < g.batch;
        const int64_t i = there ? i0 + h : i0, gi = g.inst0 + i;
        int64_t rate, bw;
        InstanceDraws d;
        base_draws(g, g.rate_knots, g.bw_knots, gi, rate, bw, d.dt);
        d.rate = uint64_t(rate);
        d.bw = uint64_t(bw);
        const uint64_t inv = ~uint64_t(0) / ((lane & 1) ? d.bw : d.rate);  // one division, not two
        d.mrate = __shfl_sync(0xffffffffu, inv, 16 * h);
        d.mbw = __shfl_sync(0xffffffffu, inv, 16 * h + 1);
        if (there && l < L) {
            int64_t wire, flops, f, b, x;
            layer_numerators(g, g.layer, gi, l, wire, flops);
            wire_costs(g, d, uint64_t(wire), uint64_t(flops), f, b, x);
            rows[h][0][l] = f;
            rows[h][1][l] = b;
            rows[h][2][l] = x;
            if (l == 0) dts[h] = d.dt;
            if constexpr (STORE) {
                const int64_t at = i * L + l;
                o.fc[at] = f;
                o.bc[at] = b;
                o.pt[at] = x;
                o.gt[at] = x;
                if (l == 0) o.dt[i] = d.dt;
            }
        }
        if (i0 == 0 && lane < 2) *(lane == 0 ? o.wide_count[0] : o.wide_count[1]) = 0u;  // nothing listed
    }
    const int kb = warp * fused_solo_bytes(L), h = warp >> 1;
    const KeptValues kept{&sh<int64_t>(kb + chain_pair_bytes(64)), L};
    if (lane == 0) zero_row(kb, 64);
    __syncthreads();
    if (i0 + h >= g.batch) return;
    if ((warp & 1) == 0)
        chain_solve_warp<true, 1>(kb, i0 + h, L, DrawnLoader<true>{rows[h][0], rows[h][2], L}, dts[h],
                                  o.out[0], kept);
    else
        chain_solve_warp<false, 1>(kb, i0 + h, L, DrawnLoader<false>{rows[h][1], rows[h][2], L}, dts[h],
                                   o.out[1], kept);
}

template <int L, bool STORE>
cudaError_t launch_fused_L(const GenParams &g, const GenTables *t, const FusedOut &o,
                           cudaStream_t stream)
{
    static DeviceCache resident;  // single-warp CTAs of the pair kernel per SM
    int per_sm = 0;
    cudaError_t le = resident.get(per_sm, [](int &n) {
        cudaError_t e = cudaFuncSetAttribute(fused_pair_kernel<L, STORE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Pair32<L>::kBytes);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fused_pair_kernel<L, STORE>, 32,
                                                             Pair32<L>::kBytes);
    });
    if (le != cudaSuccess) return le;
    const int64_t tiles = (g.batch + 31) / 32;
    int64_t grid = int64_t(sm_count()) * per_sm;
    if (grid > tiles) grid = tiles;
    fused_pair_kernel<L, STORE><<<unsigned(grid), 32, Pair32<L>::kBytes, stream>>>(g, t, o);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_fused_list<L, true>(g, t, o, stream);
    if (e != cudaSuccess) return e;
    return launch_fused_list<L, false>(g, t, o, stream);
}

}  // namespace

size_t fused_workspace_bytes(int64_t batch) { return fused_tables_offset(batch) + sizeof(GenTables); }

// Whether one launch of fused_solo_kernel takes the batch. The pair kernel's path is five
// launches, and a thread per instance is slow to finish; but the solo kernel takes 1.5 us
// per 1,000 instances, 3.5 to 5 where the layers' knots are looked up. Whole steps from a
// graph, solo against pair: one instance 6.2 us against 12-22; 4,096 x 8 (tiny) 10.3
// against 16.4, 4,096 x 16 (VGG-16) 12.3 against 20.8; 8,000 x 8 15.3 against 16.5, 8,000 x
// 16 18.5 against 28.8; 12,000 x 8 20.6 against 16.5. Log-uniform layers: 6,000 x 8 22.6
// against 24.5, x 16 34 against 45; 8,000 x 8 27.4 against 24.6.
bool use_fused_solo(int64_t batch, int layer_mode)
{
    return batch <= (layer_mode == DC_LAYERS_LOGUNIFORM ? 6000 : 8000);
}

// Generate-and-solve for 1 <= L <= 16; rows: where the profiles go, or null.
cudaError_t launch_fused(const GenParams &g, const SolveOut (&out)[2], const StepRows *rows,
                         void *workspace, cudaStream_t stream)
{
    const int64_t B = g.batch;
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    FusedOut o = {};
    for (int d = 0; d < 2; ++d) {
        o.out[d] = out[d];
        o.wide_count[d] = reinterpret_cast<uint32_t *>(ws) + d;
        o.wide_list[d] = reinterpret_cast<uint32_t *>(ws + 256) + d * B;
    }
    o.ticket = reinterpret_cast<uint32_t *>(ws) + 2;
    if (rows) {
        o.fc = rows->fc;
        o.pt = rows->pt;
        o.bc = rows->bc;
        o.gt = rows->gt;
        o.dt = rows->dt;
        o.pairs = ((reinterpret_cast<uintptr_t>(o.fc) | reinterpret_cast<uintptr_t>(o.pt) |
                    reinterpret_cast<uintptr_t>(o.bc) | reinterpret_cast<uintptr_t>(o.gt)) & 15u) == 0;
    }
    if (use_fused_solo(B, g.layer_mode)) {
        const unsigned grid = unsigned((B + kSoloInstances - 1) / kSoloInstances);
        const size_t smem = size_t(2 * kSoloInstances) * fused_solo_bytes(g.L);  // 8.5 KB at L = 16
        if (rows)
            fused_solo_kernel<true><<<grid, 64 * kSoloInstances, smem, stream>>>(g, o);
        else
            fused_solo_kernel<false><<<grid, 64 * kSoloInstances, smem, stream>>>(g, o);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(ws, 0, 3 * sizeof(uint32_t), stream);
    if (e != cudaSuccess) return e;
    GenTables *t = reinterpret_cast<GenTables *>(ws + fused_tables_offset(B));
    copy_tables_kernel<<<1, 256, 0, stream>>>(g, t);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
#define DC_FUSED_CASE(LL) \
    case LL:                                          \
        return rows ? launch_fused_L<LL, true>(g, t, o, stream) \
                    : launch_fused_L<LL, false>(g, t, o, stream);
    switch (g.L) {
        DC_FUSED_CASE(1) DC_FUSED_CASE(2) DC_FUSED_CASE(3) DC_FUSED_CASE(4)
        DC_FUSED_CASE(5) DC_FUSED_CASE(6) DC_FUSED_CASE(7) DC_FUSED_CASE(8)
        DC_FUSED_CASE(9) DC_FUSED_CASE(10) DC_FUSED_CASE(11) DC_FUSED_CASE(12)
        DC_FUSED_CASE(13) DC_FUSED_CASE(14) DC_FUSED_CASE(15) DC_FUSED_CASE(16)
        default: return cudaErrorInvalidValue;
    }
#undef DC_FUSED_CASE
}

}  // namespace dc

DC_CHECKED_EXPORT(dp_fused)
