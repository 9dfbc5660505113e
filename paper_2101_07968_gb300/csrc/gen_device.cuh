// Device side of the seeded profile generator, shared by the generator kernel
// and the fused generate-and-solve kernel: every value is a pure function of
// (seed, global instance index, field, layer), so any kernel can regenerate any
// instance's rows. Integer-only: SplitMix64 draws, multiply-high uniform
// integers, piecewise-linear log-uniform knots built on the host in double
// precision, and exact ceiling divisions by multiply-high with a per-divisor
// reciprocal.
#pragma once

#include "common.cuh"

namespace dc {

constexpr int kKnots = 512;
constexpr int kFixedMax = 1024;

// numerators of a layer (fixed tables: bits * 1000 * params and FLOPs), or one knot of
// each log-uniform layer table (params, FLOPs)
struct alignas(16) LayerRow {
    int64_t a, b;
};

struct GenParams {
    int64_t batch, inst0;
    uint64_t seed;
    int32_t L, layer_mode, rate_dist, bw_dist, bwd_mult, bits;
    int32_t words;  // every cost is below 2^32 (word_costs)
    int64_t rate_lo, rate_hi, bw_lo, bw_hi, dt_lo, dt_hi;
    int64_t params_lo, params_hi, flops_lo, flops_hi;
    int64_t rate_knots[kKnots + 1], bw_knots[kKnots + 1];
    LayerRow layer[kFixedMax];
};
static_assert(sizeof(GenParams) < 32000, "kernel parameter block limit");

__device__ __forceinline__ uint64_t splitmix(uint64_t seed, uint64_t ctr)
{
    uint64_t z = seed + (ctr + 1) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t counter(int64_t gi, int field, int layer)
{
    return (uint64_t(gi) << 20) | (uint64_t(field) << 12) | uint64_t(layer);
}

__device__ __forceinline__ int64_t uniform_int(int64_t lo, int64_t hi, uint64_t r)
{
    return lo + int64_t(__umul64hi(r, uint64_t(hi - lo) + 1u));
}

// the log-uniform draw r between the knots t0 = T(r >> 55) and t1 = T((r >> 55) + 1)
__device__ __forceinline__ int64_t between(int64_t t0, int64_t t1, uint64_t r)
{
    const uint64_t f = (r >> 23) & 0xffffffffull;
    return t0 + int64_t((uint64_t(t1 - t0) * f) >> 32);
}

template <typename Tab>
__device__ __forceinline__ int64_t loguniform(const Tab &knots, uint64_t r)
{
    const int j = int(r >> 55);
    return between(knots[j], knots[j + 1], r);
}

// Exact floor(a / d) and a mod d for 0 <= a < 2^62 and 1 <= d < 2^31 with
// m = floor((2^64-1)/d) precomputed once per divisor: q = mulhi(a, m) is floor(a/d) or
// one less, because a*m/2^64 >= a/d - a*(1 + ((2^64-1) mod d))/(d*2^64) > a/d - 1/4; one
// remainder step makes it exact.
__device__ __forceinline__ void floor_div(uint64_t a, uint64_t d, uint64_t m, uint64_t &q,
                                          uint64_t &r)
{
    q = __umul64hi(a, m);
    r = a - q * d;
    if (r >= d) {
        ++q;
        r -= d;
    }
}

__device__ __forceinline__ uint64_t ceil_div(uint64_t a, uint64_t d, uint64_t m)
{
    uint64_t q, r;
    floor_div(a, d, m, q, r);
    return q + (r != 0 ? 1u : 0u);
}

// The same for quotients below 2^32 (a < d * 2^32), in 32-bit steps: division of two
// words by one normalised word with its reciprocal v = floor((2^64-1)/dn) - 2^32, after
// Moeller and Granlund, "Improved division by invariant integers" (IEEE Trans. Comput.
// 60, 2011), Algorithm 4. About 11 instructions against 20.
struct WordDiv {
    uint32_t dn, v;  // d << s with the top bit set, its reciprocal
    uint32_t s;
};
__device__ __forceinline__ WordDiv word_div(uint32_t d)
{
    WordDiv w;
    w.s = uint32_t(__clz(int(d)));
    w.dn = d << w.s;
    w.v = uint32_t(~uint64_t(0) / w.dn);  // the quotient lies in [2^32, 2^33)
    return w;
}
// q = floor(a / d); r = (a mod d) << s
__device__ __forceinline__ void divide(uint64_t a, const WordDiv &w, uint32_t &q, uint32_t &r)
{
    const uint64_t u = a << w.s;
    const uint64_t t = uint64_t(w.v) * uint32_t(u >> 32) + u;
    q = uint32_t(t >> 32) + 1u;
    r = uint32_t(u) - q * w.dn;
    if (r > uint32_t(t)) {
        --q;
        r += w.dn;
    }
    if (r >= w.dn) {
        ++q;
        r -= w.dn;
    }
}

// Host: config checks, and the generator's parameter block for a valid config.
dc_status check_profile_cfg(const dc_profile_cfg *c);
void fill_gen_params(const dc_profile_cfg *c, GenParams &g);

// Generate-and-solve for 1 <= L <= 16 (dp_fused.cu), forward first, the profiles to
// `rows` unless it is null; workspace: fused_workspace_bytes(batch).
size_t fused_workspace_bytes(int64_t batch);
bool use_fused_solo(int64_t batch, int layer_mode);  // one launch takes the batch
struct StepRows {
    int64_t *fc, *pt, *bc, *gt, *dt;
};
cudaError_t launch_fused(const GenParams &g, const SolveOut (&out)[2], const StepRows *rows,
                         void *workspace, cudaStream_t stream);

// Rate, bandwidth and latency of global instance gi, with the reciprocals of rate and
// bandwidth: of floor_div, or of WordDiv.
struct InstanceDraws {
    uint64_t rate, mrate, bw, mbw;
    int64_t dt;
};
struct WordDraws {
    WordDiv rate, bw;
    int64_t dt;
};

template <typename Tab>
__device__ __forceinline__ void base_draws(const GenParams &g, const Tab &rate_knots,
                                           const Tab &bw_knots, int64_t gi, int64_t &rate,
                                           int64_t &bw, int64_t &dt)
{
    const uint64_t r_rate = splitmix(g.seed, counter(gi, 0, 0));
    const uint64_t r_bw = splitmix(g.seed, counter(gi, 1, 0));
    rate = g.rate_dist == DC_DIST_LOGUNIFORM ? loguniform(rate_knots, r_rate)
                                             : uniform_int(g.rate_lo, g.rate_hi, r_rate);
    bw = g.bw_dist == DC_DIST_LOGUNIFORM ? loguniform(bw_knots, r_bw)
                                         : uniform_int(g.bw_lo, g.bw_hi, r_bw);
    dt = uniform_int(g.dt_lo, g.dt_hi, splitmix(g.seed, counter(gi, 2, 0)));
}

template <typename Tab>
__device__ __forceinline__ InstanceDraws instance_draws(const GenParams &g, const Tab &rate_knots,
                                                        const Tab &bw_knots, int64_t gi)
{
    int64_t rate, bw;
    InstanceDraws d;
    base_draws(g, rate_knots, bw_knots, gi, rate, bw, d.dt);
    d.rate = uint64_t(rate);
    d.mrate = ~uint64_t(0) / uint64_t(rate);
    d.bw = uint64_t(bw);
    d.mbw = ~uint64_t(0) / uint64_t(bw);
    return d;
}

template <typename Tab>
__device__ __forceinline__ WordDraws word_draws(const GenParams &g, const Tab &rate_knots,
                                                const Tab &bw_knots, int64_t gi)
{
    int64_t rate, bw;
    WordDraws d;
    base_draws(g, rate_knots, bw_knots, gi, rate, bw, d.dt);
    d.rate = word_div(uint32_t(rate));
    d.bw = word_div(uint32_t(bw));
    return d;
}

// Wire bits per kbit/s (bits * 1000 * params) and FLOPs of layer l (0-based) of global
// instance gi; rows: the layer table (LayerRow).
__device__ __forceinline__ void layer_numerators(const GenParams &g, const LayerRow *rows,
                                                 int64_t gi, int l, int64_t &wire, int64_t &flops)
{
    if (g.layer_mode == DC_LAYERS_FIXED) {
        const longlong2 row = *reinterpret_cast<const longlong2 *>(rows + l);
        wire = row.x;
        flops = row.y;
        return;
    }
    const uint64_t rp = splitmix(g.seed, counter(gi, 3, l));
    const uint64_t rf = splitmix(g.seed, counter(gi, 4, l));
    int64_t params;
    if (g.layer_mode == DC_LAYERS_LOGUNIFORM) {
        const int jp = int(rp >> 55), jf = int(rf >> 55);
        params = between(rows[jp].a, rows[jp + 1].a, rp);
        flops = between(rows[jf].b, rows[jf + 1].b, rf);
    } else {
        params = uniform_int(g.params_lo, g.params_hi, rp);
        flops = uniform_int(g.flops_lo, g.flops_hi, rf);
    }
    wire = params * (int64_t(g.bits) * 1000);
}

// Forward compute, backward compute and transfer cost (pt = gt) of one layer; `wire` is
// bits * 1000 * params.
__device__ __forceinline__ void wire_costs(const GenParams &g, const InstanceDraws &d,
                                           uint64_t wire, uint64_t flops, int64_t &fc,
                                           int64_t &bc, int64_t &xfer)
{
    xfer = int64_t(ceil_div(wire, d.bw, d.mbw));
    if (g.bwd_mult == 2) {
        // flops = q*rate + r (0 <= r < rate): ceil(flops/rate) = q + (r > 0) and
        // ceil(2*flops/rate) = 2q + ceil(2r/rate) = 2q + (r > 0) + (2r > rate)
        uint64_t q, r;
        floor_div(uint64_t(flops), d.rate, d.mrate, q, r);
        const uint64_t up = r != 0 ? 1u : 0u;
        fc = int64_t(q + up);
        bc = int64_t(2 * q + up + (2 * r > d.rate ? 1u : 0u));
    } else {
        fc = int64_t(ceil_div(uint64_t(flops), d.rate, d.mrate));
        bc = int64_t(ceil_div(uint64_t(g.bwd_mult) * uint64_t(flops), d.rate, d.mrate));
    }
}

// The same costs where each of them is below 2^32 (with bwd_mult 2 the forward ones and
// the transfers): `wire` is bits * 1000 * params.
__device__ __forceinline__ void word_costs(const GenParams &g, const WordDiv &rate, const WordDiv &bw,
                                           uint64_t wire, uint64_t flops, uint32_t &fc,
                                           uint64_t &bc, uint32_t &xfer)
{
    uint32_t q, r;
    divide(wire, bw, q, r);
    xfer = q + (r != 0 ? 1u : 0u);
    divide(flops, rate, q, r);
    const uint32_t up = r != 0 ? 1u : 0u;
    fc = q + up;
    if (g.bwd_mult == 2) {  // as in wire_costs; 2 r > rate as r > rate - r, which do not wrap
        bc = 2 * uint64_t(q) + up + (r > rate.dn - r ? 1u : 0u);
    } else {
        divide(uint64_t(g.bwd_mult) * flops, rate, q, r);
        bc = uint64_t(q) + (r != 0 ? 1u : 0u);
    }
}

}  // namespace dc
