// Seeded synthetic profile generator (stand-in for the real-time profiler of
// Sec. IV-A, which derives pt, fc, bc, gt and dt from a framework's profiler).
//
// Every value is a pure function of (seed, global instance index, field, layer),
// so any sub-range of a batch can be generated on its own. Integer-only on the
// device: SplitMix64 draws, multiply-high uniform integers, piecewise-linear
// log-uniform knots built on the host in double precision, and exact ceiling
// divisions by multiply-high with a per-instance reciprocal.
#include <algorithm>
#include <cmath>

#include "gen_device.cuh"

namespace dc {
namespace {

// Warp-level tiles of `ti` consecutive instances (32; fewer in small batches, so that
// the elements spread over more warps). Phase 1: lane j draws rate, bandwidth and
// latency of instance j and forms the two reciprocals (the instances' divisions run
// side by side). Phase 2: the warp walks the tile's ti * L (instance, layer) elements 32
// at a time, so the output rows are written coalesced. Only __syncwarp between the
// phases.
//
// WORDS: every cost is below 2^32 (all configurations here; see fill_gen_params):
// divisions in 32-bit steps (WordDiv), an instance's divisors in one 16-byte and one 4-byte
// load, a layer's numerators in one 16-byte load. SHARED: the knots and layer tables in
// shared memory; without it (small batches) lanes read the few entries they need from the
// parameters, which beats copying the tables in every CTA. Bound by the HBM writes on large
// batches (1,000,000 x 16, 520 MB: 84 us, 6.2 TB/s, with either division), by integer issue on
// short rows (1,000,000 x 8: 48 us, 53 with 64-bit divisions) and on log-uniform layers
// (16,384 x 1,024: 127 us, 376 with 64-bit divisions in tiles of 32).
constexpr int kGenWarps = 8;

template <bool SHARED, bool WORDS>
__global__ void __launch_bounds__(32 * kGenWarps, SHARED ? 5 : 1)
    gen_kernel(const __grid_constant__ GenParams g, int ti, int tw, int64_t *__restrict__ fc,
               int64_t *__restrict__ pt, int64_t *__restrict__ bc, int64_t *__restrict__ gt,
               int64_t *__restrict__ dt)
{
    extern __shared__ __align__(16) unsigned char dyn[];  // rate and bw knots, layer table
    __shared__ uint4 s_div[kGenWarps][32];     // WORDS: rate.dn, rate.v, bw.dn, bw.v; else rate, its reciprocal
    __shared__ uint4 s_div2[WORDS ? 1 : kGenWarps][32];  // else: bw, its reciprocal
    __shared__ uint32_t s_shift[WORDS ? kGenWarps : 1][32];
    const int L = g.L, t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
    int64_t *s_rate = reinterpret_cast<int64_t *>(dyn), *s_bw = s_rate + kKnots + 1;
    LayerRow *s_layer = reinterpret_cast<LayerRow *>(s_bw + kKnots + 1);
    if (SHARED) {
        const int nl = g.layer_mode == DC_LAYERS_FIXED ? L
                       : (g.layer_mode == DC_LAYERS_LOGUNIFORM ? kKnots + 1 : 0);
        if (g.rate_dist == DC_DIST_LOGUNIFORM)
            for (int j = t; j <= kKnots; j += blockDim.x) s_rate[j] = g.rate_knots[j];
        if (g.bw_dist == DC_DIST_LOGUNIFORM)
            for (int j = t; j <= kKnots; j += blockDim.x) s_bw[j] = g.bw_knots[j];
        for (int j = t; j < nl; j += blockDim.x) s_layer[j] = g.layer[j];
        __syncthreads();
    }
    // warp `sub` of the tw that share a tile takes every tw-th run of 32 elements
    const int sub = warp % tw, stride = 32 * tw;
    const int step_i = stride / L, step_l = stride % L;  // advance of (instance, layer) a step
    const int64_t tiles = (g.batch + ti - 1) / ti;
    for (int64_t tile = (int64_t(blockIdx.x) * nw + warp) / tw; tile < tiles;
         tile += int64_t(gridDim.x) * nw / tw) {
        const int64_t i0 = tile * ti;
        const int n_inst = int(g.batch - i0 < ti ? g.batch - i0 : ti);
        __syncwarp();  // previous tile done with the divisors
        if (lane < n_inst) {
            const int64_t i = i0 + lane;
            const int64_t *kr = SHARED ? s_rate : g.rate_knots, *kw = SHARED ? s_bw : g.bw_knots;
            if (WORDS) {
                const WordDraws d = word_draws(g, kr, kw, g.inst0 + i);
                s_div[warp][lane] = make_uint4(d.rate.dn, d.rate.v, d.bw.dn, d.bw.v);
                s_shift[warp][lane] = d.rate.s | (d.bw.s << 8);
                if (sub == 0) dt[i] = d.dt;
            } else {
                const InstanceDraws d = instance_draws(g, kr, kw, g.inst0 + i);
                *reinterpret_cast<ulonglong2 *>(&s_div[warp][lane]) = make_ulonglong2(d.rate, d.mrate);
                *reinterpret_cast<ulonglong2 *>(&s_div2[warp][lane]) = make_ulonglong2(d.bw, d.mbw);
                if (sub == 0) dt[i] = d.dt;
            }
        }
        __syncwarp();
        const int total = n_inst * L;
        const int e0 = 32 * sub + lane;
        int il = e0 / L, l = e0 - il * L;
        const int64_t o0 = i0 * L + e0;
        int64_t *pf = fc + o0, *pb = bc + o0, *px = pt + o0, *pg = gt + o0;
        for (int e = e0; e < total; e += stride) {
            int64_t wire, flops;
            layer_numerators(g, SHARED ? s_layer : g.layer, g.inst0 + i0 + il, l, wire, flops);
            if (WORDS) {
                const uint4 d = s_div[warp][il];
                const uint32_t s = s_shift[warp][il];
                uint32_t f, x;
                uint64_t b;
                word_costs(g, WordDiv{d.x, d.y, s & 0xffu}, WordDiv{d.z, d.w, s >> 8}, uint64_t(wire),
                           uint64_t(flops), f, b, x);
                *pf = int64_t(uint64_t(f));
                *pb = int64_t(b);
                *px = int64_t(uint64_t(x));
                *pg = int64_t(uint64_t(x));
            } else {
                const ulonglong2 r = *reinterpret_cast<const ulonglong2 *>(&s_div[warp][il]);
                const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(&s_div2[warp][il]);
                const InstanceDraws d{r.x, r.y, w.x, w.y, 0};
                int64_t f, b, x;
                wire_costs(g, d, uint64_t(wire), uint64_t(flops), f, b, x);
                *pf = f;
                *pb = b;
                *px = x;
                *pg = x;
            }
            pf += stride;
            pb += stride;
            px += stride;
            pg += stride;
            il += step_i;
            l += step_l;
            if (l >= L) {
                l -= L;
                ++il;
            }
        }
    }
}

int64_t knot(int64_t lo, int64_t hi, int j)
{
    if (j <= 0) return lo;
    if (j >= kKnots) return hi;
    const double x = double(j) / 512.0;
    const double y = std::log(double(hi) / double(lo));
    return int64_t(std::llround(double(lo) * std::exp(x * y)));
}

void knots(int64_t lo, int64_t hi, int64_t *out)
{
    for (int j = 0; j <= kKnots; ++j) out[j] = knot(lo, hi, j);
}

bool in_range(int64_t lo, int64_t hi, int64_t min_lo, int64_t max_hi)
{
    return lo >= min_lo && lo <= hi && hi <= max_hi;
}

}  // namespace

void fill_gen_params(const dc_profile_cfg *c, GenParams &g)
{
    g.batch = c->batch;
    g.inst0 = c->inst0;
    g.seed = c->seed;
    g.L = c->L;
    g.layer_mode = c->layer_mode;
    g.rate_dist = c->rate_dist;
    g.bw_dist = c->bw_dist;
    g.bwd_mult = c->bwd_flops_mult;
    g.bits = c->bits_per_param;
    g.rate_lo = c->rate_lo;
    g.rate_hi = c->rate_hi;
    g.bw_lo = c->bw_lo;
    g.bw_hi = c->bw_hi;
    g.dt_lo = c->dt_lo;
    g.dt_hi = c->dt_hi;
    g.params_lo = c->params_lo;
    g.params_hi = c->params_hi;
    g.flops_lo = c->flops_lo;
    g.flops_hi = c->flops_hi;
    // the largest numerators, and whether their costs, the quotients rounded up, all fit
    // 32 bits (word_costs rounds up in 32 bits: a quotient of 2^32 - 1 with a remainder
    // would come out 0)
    int64_t most_p = c->params_hi, most_f = c->flops_hi;
    if (c->layer_mode == DC_LAYERS_FIXED) {
        most_p = most_f = 0;
        for (int l = 0; l < c->L; ++l) {
            most_p = std::max(most_p, c->fixed_params[l]);
            most_f = std::max(most_f, c->fixed_flops[l]);
        }
    }
    auto fits = [](int64_t num, int64_t d) { return (num + d - 1) / d < (int64_t(1) << 32); };
    g.words = fits(int64_t(c->bits_per_param) * 1000 * most_p, c->bw_lo) &&
              fits(int64_t(c->bwd_flops_mult == 2 ? 1 : c->bwd_flops_mult) * most_f, c->rate_lo);
    if (c->rate_dist == DC_DIST_LOGUNIFORM) knots(c->rate_lo, c->rate_hi, g.rate_knots);
    if (c->bw_dist == DC_DIST_LOGUNIFORM) knots(c->bw_lo, c->bw_hi, g.bw_knots);
    if (c->layer_mode == DC_LAYERS_FIXED) {
        for (int l = 0; l < c->L; ++l) {
            g.layer[l] = LayerRow{c->fixed_params[l] * (int64_t(c->bits_per_param) * 1000),
                                  c->fixed_flops[l]};
        }
    } else if (c->layer_mode == DC_LAYERS_LOGUNIFORM) {
        for (int j = 0; j <= kKnots; ++j)
            g.layer[j] = LayerRow{knot(c->params_lo, c->params_hi, j), knot(c->flops_lo, c->flops_hi, j)};
    }
}

dc_status check_profile_cfg(const dc_profile_cfg *c)
{
    const int64_t cap = int64_t(1) << 40, rcap = (int64_t(1) << 31) - 1;
    if (c->L < 1 || c->L > DC_L_MAX || c->batch < 0 || c->inst0 < 0) return DC_ERR_BAD_CONFIG;
    if (c->inst0 + c->batch > (int64_t(1) << 44)) return DC_ERR_BAD_CONFIG;
    if (c->bwd_flops_mult < 1 || c->bwd_flops_mult > 16) return DC_ERR_BAD_CONFIG;
    if (c->bits_per_param < 1 || c->bits_per_param > 64) return DC_ERR_BAD_CONFIG;
    if (!in_range(c->rate_lo, c->rate_hi, 1, rcap) || !in_range(c->bw_lo, c->bw_hi, 1, rcap))
        return DC_ERR_BAD_CONFIG;
    if (!in_range(c->dt_lo, c->dt_hi, 0, cap)) return DC_ERR_BAD_CONFIG;
    if (c->rate_dist < 0 || c->rate_dist > 1 || c->bw_dist < 0 || c->bw_dist > 1)
        return DC_ERR_BAD_CONFIG;
    if (c->layer_mode == DC_LAYERS_FIXED) {
        if (c->L > kFixedMax) return DC_ERR_BAD_CONFIG;
        if (!c->fixed_params || !c->fixed_flops) return DC_ERR_NULL;
        for (int l = 0; l < c->L; ++l)
            if (!in_range(c->fixed_params[l], c->fixed_params[l], 0, cap) ||
                !in_range(c->fixed_flops[l], c->fixed_flops[l], 0, cap))
                return DC_ERR_BAD_CONFIG;
    } else if (c->layer_mode == DC_LAYERS_UNIFORM || c->layer_mode == DC_LAYERS_LOGUNIFORM) {
        const int64_t min_lo = c->layer_mode == DC_LAYERS_LOGUNIFORM ? 1 : 0;
        if (!in_range(c->params_lo, c->params_hi, min_lo, cap) ||
            !in_range(c->flops_lo, c->flops_hi, min_lo, cap))
            return DC_ERR_BAD_CONFIG;
    } else {
        return DC_ERR_BAD_CONFIG;
    }
    return DC_OK;
}

cudaError_t launch_gen(const dc_profile_cfg *c, int64_t *fc, int64_t *pt, int64_t *bc,
                       int64_t *gt, int64_t *dt, cudaStream_t stream)
{
    static thread_local GenParams g;  // 25 KB: kept off the caller's stack
    fill_gen_params(c, g);
    // Few instances and elements, and tables that lanes read at a few places only: no copy
    // of them (4,096 x 8: 3.4 us from a graph, 7.2 with the copy and tiles of 32; but the
    // log-uniform layer tables, read at 64 places a step, serialise: 11 times slower on
    // 16,384 x 1,024; and so do the knots, read once per instance, and fixed layers: 60,000 x
    // 1 7.8 us against 5.6 with the copy, 30,000 x 8 (AlexNet) 9.1 against 6.8, 20,000 x 8 7.3
    // against 6.4; but with drawn layers 20,000 x 13 7.2 against 8.3)
    const bool shared = c->batch * c->L > (int64_t(1) << 18) ||
                        c->batch > (c->layer_mode == DC_LAYERS_FIXED ? 16000 : 24000) ||
                        c->layer_mode == DC_LAYERS_LOGUNIFORM;
    // Tiles of 32 instances once they fill the GPU (8 warps per SM, 32 where a tile is long;
    // 4 where short rows share a copy of the tables: log-uniform 10,000 x 4 8.1 us against
    // 9.5 with 8, but 20,000 x 24 11.7 against 11.1), else smaller ones, down to 32 elements,
    // and for long rows several warps to an instance
    int ti = 32, tw = 1;
    const int fill = shared && c->L <= 16 ? 4 : 8;
    auto tiles_of = [&](int n) { return (c->batch + n - 1) / n; };
    while (ti > 1 && tiles_of(ti) < 152 * (ti * c->L >= 4096 ? 32 : fill) && ti / 2 * c->L >= 32) ti /= 2;
    while (ti == 1 && tw < 4 && c->batch * tw < 152 * 32 && c->L >= 128 * tw) tw *= 2;
    const int64_t warps = tiles_of(ti) * tw;
    if (!shared) {
        const unsigned blocks = unsigned((warps + 3) / 4);
        if (g.words)
            gen_kernel<false, true><<<blocks, 128, 0, stream>>>(g, ti, tw, fc, pt, bc, gt, dt);
        else
            gen_kernel<false, false><<<blocks, 128, 0, stream>>>(g, ti, tw, fc, pt, bc, gt, dt);
        return cudaGetLastError();
    }
    const size_t rows = c->layer_mode == DC_LAYERS_FIXED        ? size_t(c->L)
                        : c->layer_mode == DC_LAYERS_LOGUNIFORM ? size_t(kKnots + 1)
                                                                : 0;
    const size_t smem = 2 * (kKnots + 1) * 8 + rows * sizeof(LayerRow);  // at most 24.6 KB
    int64_t blocks = (warps + kGenWarps - 1) / kGenWarps;
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (g.words)
        gen_kernel<true, true><<<unsigned(blocks), 32 * kGenWarps, smem, stream>>>(g, ti, tw, fc, pt, bc, gt, dt);
    else
        gen_kernel<true, false><<<unsigned(blocks), 32 * kGenWarps, smem, stream>>>(g, ti, tw, fc, pt, bc, gt, dt);
    return cudaGetLastError();
}

}  // namespace dc
