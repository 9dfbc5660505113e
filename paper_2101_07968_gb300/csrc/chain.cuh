// One instance of the DynaComm DP (Eq. 8 / Algorithm 3 and Eq. 9 / Algorithm 4)
// solved by a CTA in O(L log L) per segment count, in 64-bit arithmetic: the
// device code shared by the deep-chain pass (dp_deep.cu) and the work-list pass
// (dp_group.cu).
//
// With the layers in processing order, P the prefix of the transfer costs and C
// that of the compute costs, put
//   forward : V[m][n] = F[m][n] - C[m]              a = P, b = C, e = 0,  c_n = n*dt
//   backward: V[m][n] = B[m][n] - dt - P[m]         a = C, b = P, e = dt, c_n = 0
// Eq. 8 and Eq. 9 both become a bottleneck (min-max) recurrence,
//   V[m][1] = c_1 + a[m],
//   V[m][n] = min_k max(V[k][n-1] + e, c_n + a[m] - b[k]),   T_n = V[L][n] + e + b[L],
// in which the first operand does not depend on m and the second falls with k.
// The kernel computes, instead of V, the column
//   H[m][n] = min(H[m][n-1], min over every k in [1, L-1] of
//                            max(H[k][n-1] + e, c_n + a[m] - b[k])),  H[m][1] = V[m][1],
// that is, it also allows fewer segments than n, and steps that go back (k >= m).
//  * H[.][n] is non-decreasing in m, as a minimum of such functions: H + e + b is
//    sorted, and the minimum over k sits at the crossing of the two operands,
//    found by a binary search for the first k with H[k] + e + b[k] >= c_n + a[m].
//  * It gives the same optimum, segment count and decision. Take any chain of
//    steps that H allows and drop its surplus: a step that goes back, or a count
//    larger than the segments it stands for. The result is a real decision with
//    strictly fewer segments, and its makespan is no larger: dropping a step
//    starts the next segment at a later layer (a larger b) and lowers every later
//    segment's number by one, which lowers c forward and saves an e backward.
//    So min_n T_n is unchanged, and H[L][n] = V[L][n] at the lowest optimal count
//    s: a smaller H would be a decision with fewer than s segments and no larger
//    makespan. For the same reason H equals V, and an operand is at most the
//    cell only for a real step, at every cell that the traceback from (L, s)
//    visits.
//  * The traceback's Path[m][n], the lowest k that attains the cell v, is then the
//    first k with c_n + a[m] - b[k] <= v: the k that attains v satisfy it together
//    with H[k][n-1] + e <= v, the latter holds for a prefix of the k (H is sorted)
//    and the former for a suffix.
//  * Columns end early: column n+1 differs from column n only through k whose H
//    column n lowered, and such a k can lower the optimum only if H[k][n] + e <
//    H[L][n]. The fill stops after the first column without one (on the deep
//    chain after 6.2 columns on average, where the optimum has 5.6 segments), or
//    when c_n + a[L] - b[L-1], which bounds every later T, reaches the optimum.
// Values stay below 2^53 (the range check), so 64 bits hold every sum.
#pragma once

#include "common.cuh"

namespace dc {
namespace {

constexpr int kChainPairs = 4;             // row pairs per thread, at most
constexpr int kChainThreads = 512;         // threads per instance, at most
constexpr int kChainRows = 2 * kChainPairs;  // rows per thread, at most

// Shared memory of a CTA: two key buffers (H + e + b of a column, rows 1..L at
// 0..L-1) and b, then the decision words, the scan's partial sums and a few
// words that one thread publishes.
__host__ __device__ inline size_t chain_row_bytes(int L) { return size_t((L + 1) / 2) * 16; }
__host__ __device__ inline size_t chain_bits_bytes(int L)
{
    return (size_t(words_for(L)) * 4 + 15) / 16 * 16;
}
constexpr size_t kChainScratch = (2 * kChainPairs * (kChainThreads / 32) + 8 + 4) * 8;
__host__ __device__ inline size_t chain_smem_bytes(int L)
{
    return 3 * chain_row_bytes(L) + chain_bits_bytes(L) + kChainScratch;
}

// Threads per instance: the fewest warps that hold the rows (8 per thread), and
// more, down to one row pair per thread, while `count` instances leave the GPU's
// SMs with fewer than 16 warps each.
inline int chain_threads(int64_t count, int L, int sms)
{
    int nt = 32 * ((L + 32 * kChainRows - 1) / (32 * kChainRows));
    while (nt * 2 <= kChainThreads && nt * 2 < L && count * (nt / 32) < int64_t(sms) * 16) nt *= 2;
    return nt;
}

// Where H of column n >= 2 goes for the traceback. Offsets from H[1][1], which no
// value is below, in 32 bits (the caller has checked the range), or whole values.
struct KeptOffsets {
    uint32_t *at;
    int L, last;  // columns 2..last
    int64_t base;
    __device__ bool holds(int n) const { return n <= last; }
    __device__ void put(int n, int m, int64_t v) const
    {
        const int64_t j = int64_t(n - 2) * L + (m - 1);
        if (DC_CHECK(n >= 2 && n <= last && m >= 1 && m <= L))
            at[j] = uint32_t(min(uint64_t(v - base), uint64_t(0xffffffffu)));
    }
    __device__ int64_t get(int n, int m) const
    {
        if (!DC_CHECK(n >= 2 && n <= last && m >= 1 && m <= L)) return 0;
        return base + int64_t(at[int64_t(n - 2) * L + (m - 1)]);
    }
};
struct KeptValues {  // the triangle of cells m >= n, every column
    int64_t *at;
    int L;
    __device__ bool holds(int) const { return true; }
    __device__ void put(int n, int m, int64_t v) const
    {
        if (m >= n && DC_CHECK(n >= 1 && m <= L)) at[tri_index(L, m, n)] = v;
    }
    __device__ int64_t get(int n, int m) const
    {
        if (!DC_CHECK(n >= 1 && m >= n && m <= L)) return 0;
        return at[tri_index(L, m, n)];
    }
};

struct ChainOut {
    int64_t *makespan;
    uint32_t *bits;
    int32_t *nseg, *status;
};

// Number of keys below t among key[1..N] (key[k] at K[k-1], sorted), P the largest
// power of two <= N: the first probe splits [0, N] into two ranges of at most P
// values, the rest halve it. Two searches at once (independent load chains).
__device__ __forceinline__ void count_below2(const int64_t *K, int N, int P, int64_t t0,
                                             int64_t t1, int &p0, int &p1)
{
    const int64_t kp = K[P - 1];
    p0 = kp < t0 ? N - P + 1 : 0;
    p1 = kp < t1 ? N - P + 1 : 0;
    for (int st = P >> 1; st > 0; st >>= 1) {
        const int64_t k0 = K[p0 + st - 1], k1 = K[p1 + st - 1];
        if (k0 < t0) p0 += st;
        if (k1 < t1) p1 += st;
    }
}

// Solves instance i (rows crow, xrow of L costs) with the whole CTA. make_kept(base,
// range) gives the store of kept columns, or refuses by returning false; returns
// false, having written nothing, when the instance needs columns the store does not
// hold. `vec`: the rows are 16-byte aligned and L is even.
template <bool FWD, typename Kept, typename MakeKept>
__device__ bool chain_solve(unsigned char *smem, int64_t i, int L, const int64_t *crow,
                            const int64_t *xrow, int64_t dt, bool vec, const ChainOut &o,
                            MakeKept make_kept)
{
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
    const int W = words_for(L);
    const size_t rb = chain_row_bytes(L);
    int64_t *K0 = reinterpret_cast<int64_t *>(smem), *K1 = reinterpret_cast<int64_t *>(smem + rb);
    int64_t *B = reinterpret_cast<int64_t *>(smem + 2 * rb);
    uint32_t *bitsw = reinterpret_cast<uint32_t *>(smem + 3 * rb);
    uint64_t *tot = reinterpret_cast<uint64_t *>(smem + 3 * rb + chain_bits_bytes(L));
    uint32_t *orw = reinterpret_cast<uint32_t *>(tot + 2 * kChainPairs * (kChainThreads / 32));
    int64_t *s_aL = reinterpret_cast<int64_t *>(orw + 16);
    const int NJ = (L + 2 * NT - 1) / (2 * NT);  // row pairs per thread

    // ---- rows: pair j of this thread holds rows r, r+1 with r = 2 (j NT + tid) + 1
    uint64_t a[kChainPairs][2], b[kChainPairs][2];
    uint64_t any = uint64_t(dt);
#pragma unroll
    for (int j = 0; j < kChainPairs; ++j) {
        if (j < NJ) {
            const int r = 2 * (j * NT + tid) + 1;
            uint64_t c0 = 0, c1 = 0, x0 = 0, x1 = 0;
            if (r < L && vec) {
                const int at = FWD ? r - 1 : L - r - 1;
                const ulonglong2 c = *reinterpret_cast<const ulonglong2 *>(crow + at);
                const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(xrow + at);
                c0 = FWD ? c.x : c.y;
                c1 = FWD ? c.y : c.x;
                x0 = FWD ? x.x : x.y;
                x1 = FWD ? x.y : x.x;
            } else if (r <= L) {
                const int at = FWD ? r - 1 : L - r;
                c0 = uint64_t(__ldg(crow + at));
                x0 = uint64_t(__ldg(xrow + at));
                if (r < L) {
                    c1 = uint64_t(__ldg(crow + (FWD ? at + 1 : at - 1)));
                    x1 = uint64_t(__ldg(xrow + (FWD ? at + 1 : at - 1)));
                }
            }
            any |= c0 | c1 | x0 | x1;
            uint64_t sa = FWD ? x0 + x1 : c0 + c1, sb = FWD ? c0 + c1 : x0 + x1;
            const uint64_t ta = sa, tb = sb;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint64_t ua = __shfl_up_sync(0xffffffffu, sa, d);
                const uint64_t ub = __shfl_up_sync(0xffffffffu, sb, d);
                if (lane >= d) {
                    sa += ua;
                    sb += ub;
                }
            }
            if (lane == 31) {
                tot[j * NW + warp] = sa;
                tot[(NJ + j) * NW + warp] = sb;
            }
            a[j][0] = sa - ta + (FWD ? x0 : c0);
            a[j][1] = sa;
            b[j][0] = sb - tb + (FWD ? c0 : x0);
            b[j][1] = sb;
        }
    }
    const uint32_t hi = __reduce_or_sync(0xffffffffu, uint32_t(any >> 32));
    if (lane == 0) orw[warp] = hi;
    for (int w = tid; w < W; w += NT) bitsw[w] = 0u;
    __syncthreads();
    uint32_t all = 0;
    for (int w = 0; w < NW; ++w) all |= orw[w];
    uint64_t accA = 0, accB = 0;
    {
        int next = warp;
        int j = 0;
        uint64_t offA[kChainPairs] = {}, offB[kChainPairs] = {};
        for (int q = 0; q < NJ * NW; ++q) {
            if (q == next) {
#pragma unroll
                for (int u = 0; u < kChainPairs; ++u)
                    if (u == j) {
                        offA[u] = accA;
                        offB[u] = accB;
                    }
                ++j;
                next += NW;
            }
            accA += tot[q];
            accB += tot[NJ * NW + q];
        }
#pragma unroll
        for (int u = 0; u < kChainPairs; ++u) {
            a[u][0] += offA[u];
            a[u][1] += offA[u];
            b[u][0] += offB[u];
            b[u][1] += offB[u];
        }
    }
    // accA = a[L], accB = b[L]: the totals
    int st = DC_OK;
    if (all >> 31)
        st = DC_ERR_NEGATIVE;
    else if (all >> 20 || exceeds_range(L, dt, FWD ? accB : accA, FWD ? accA : accB))
        st = DC_ERR_RANGE;
    if (st != DC_OK) {
        if (tid == 0) {
            o.makespan[i] = -int64_t(st);
            if (o.nseg) o.nseg[i] = 0;
            if (o.status) o.status[i] = st;
        }
        for (int w = tid; w < W; w += NT) o.bits[i * W + w] = 0u;
        return true;
    }
    const int64_t e = FWD ? 0 : dt, h1 = FWD ? dt : 0;  // H[m][1] = h1 + a[m]
    const int64_t aL = int64_t(accA), bL = int64_t(accB);
#pragma unroll
    for (int j = 0; j < kChainPairs; ++j) {
        const int r = 2 * (j * NT + tid) + 1;
        if (j < NJ && r <= L) {  // row L + 1 of an odd L's last pair is padding
            *reinterpret_cast<ulonglong2 *>(B + r - 1) = make_ulonglong2(b[j][0], b[j][1]);
            *reinterpret_cast<ulonglong2 *>(K0 + r - 1) =
                make_ulonglong2(a[j][0] + b[j][0] + uint64_t(h1 + e), a[j][1] + b[j][1] + uint64_t(h1 + e));
            if (r == 1) *s_aL = int64_t(a[j][0]);
        }
    }
    __syncthreads();
    int64_t hL = h1 + aL;  // H[L][n] of the newest column
    const int64_t base = h1 + *s_aL;
    Kept kept;
    if (!make_kept(kept, base, uint64_t(hL - base))) return false;
    int s = 1;
    bool deep = false;  // the optimum lies beyond the kept columns

    // ---- columns 2..
    const int N = L - 1;
    int P = 1;
    while (P * 2 <= N) P *= 2;
    int64_t *K = K0, *Kn = K1;
    const int64_t bL1 = L > 1 ? B[L - 2] : 0;
    for (int n = 2; n <= L; ++n) {
        const int64_t c = FWD ? int64_t(n) * dt : 0;
        if (c + aL - bL1 >= hL) break;
        int64_t least = INT64_MAX;  // lowest H that this column lowered
#pragma unroll
        for (int j = 0; j < kChainPairs; ++j) {
            const int r = 2 * (j * NT + tid) + 1;
            if (j < NJ && r <= L) {
                const int64_t t0 = c + int64_t(a[j][0]), t1 = c + int64_t(a[j][1]);
                int p0, p1;
                count_below2(K, N, P, t0, t1, p0, p1);
                // k = p + 1 is the first with H + e + b >= t (row L when there is
                // none: H[L] lowers nothing), k = p the last below it (p = 0 gives
                // t, which lowers nothing)
                const longlong2 bb = *reinterpret_cast<const longlong2 *>(B + r - 1);
                const longlong2 kk = *reinterpret_cast<const longlong2 *>(K + r - 1);
                const int64_t o0 = kk.x - bb.x - e, o1 = kk.y - bb.y - e;
                const int64_t u0 = min(K[p0] - B[p0], t0 - (p0 > 0 ? B[p0 - 1] : 0));
                const int64_t u1 = min(K[p1] - B[p1], t1 - (p1 > 0 ? B[p1 - 1] : 0));
                const int64_t v0 = min(o0, u0), v1 = min(o1, u1);
                *reinterpret_cast<longlong2 *>(Kn + r - 1) = make_longlong2(v0 + e + bb.x, v1 + e + bb.y);
                if (v0 < o0) least = min(least, v0);
                if (r < L && v1 < o1) least = min(least, v1);
                if (kept.holds(n)) {
                    kept.put(n, r, v0);
                    if (r < L) kept.put(n, r + 1, v1);
                }
            }
        }
        __syncthreads();
        const int64_t h = Kn[L - 1] - bL - e;
        if (h < hL) {
            hL = h;
            s = n;
            if (n > 2 && !kept.holds(n - 1)) deep = true;
        }
        // another column only while a lowered H may still lower H[L]; e >= 0, so the
        // sentinel stays above every sum
        const bool more = least != INT64_MAX && least + e < hL;
        int64_t *sw = K;
        K = Kn;
        Kn = sw;
        if (!__syncthreads_or(more) || deep) break;
    }
    if (deep) return false;

    // ---- traceback by warp 0: Path[m][n] = the first k with b[k] >= c_n + a[m] - v.
    // a goes to the idle key buffer first.
#pragma unroll
    for (int j = 0; j < kChainPairs; ++j) {
        const int r = 2 * (j * NT + tid) + 1;
        if (j < NJ && r <= L)
            *reinterpret_cast<ulonglong2 *>(Kn + r - 1) = make_ulonglong2(a[j][0], a[j][1]);
    }
    __syncthreads();
    if (warp == 0) {
        int err = 0, m = L, n = s;
        int64_t v = hL;
        while (n > 1) {
            const int64_t thr = (FWD ? int64_t(n) * dt : 0) + Kn[m - 1] - v;
            int lo = 1, len = N;  // the answer lies in [lo, lo + len], lo + len: none
            while (len > 0) {
                const int step = (len + 31) / 32;
                const int k = lo + (lane + 1) * step - 1;  // last k of this lane's piece
                const bool hit = k >= lo + len || B[k - 1] >= thr;
                const unsigned bal = __ballot_sync(0xffffffffu, hit);
                if (bal == 0u) {  // the last piece ends the range, and none reaches thr
                    lo += len;
                    break;
                }
                const int q = __ffs(int(bal)) - 1;
                const int end = lo + len;
                lo += q * step;
                len = min(step - 1, end - lo);
            }
            const int k = lo;
            if (k < n - 1 || k >= m) {
                err = 1;
                break;
            }
            const int64_t hk = n == 2 ? h1 + Kn[k - 1] : kept.get(n - 1, k);
            if (hk + e > v) {
                err = 1;
                break;
            }
            if (lane == 0) bitsw[(k - 1) >> 5] |= 1u << ((k - 1) & 31);
            v = hk;
            m = k;
            n -= 1;
        }
        __syncwarp();
        if (lane == 0) {
            o.makespan[i] = err ? -int64_t(DC_ERR_INTERNAL) : hL + e + bL;
            if (o.nseg) o.nseg[i] = err ? 0 : s;
            if (o.status) o.status[i] = err ? DC_ERR_INTERNAL : DC_OK;
        }
        for (int w = lane; w < W; w += 32) o.bits[i * W + w] = err ? 0u : bitsw[w];
    }
    return true;
}

}  // namespace
}  // namespace dc
