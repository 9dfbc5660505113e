// One instance of the DynaComm DP (Eq. 8 / Algorithm 3 and Eq. 9 / Algorithm 4)
// solved by a warp or a CTA in O(L log L) per segment count: the device code shared
// by the warp-per-instance pass (dp_warp.cu), the CTA-per-instance pass (dp_deep.cu) and
// the work-list passes (dp_group.cu, dp_small.cu, the drawing one in dp_fused.cu).
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
// Values stay below 2^53 (the range check), so 64 bits hold every sum; an instance
// with a[L] + b[L] + (L + 1) dt < 2^31 runs in 32 bits.
#pragma once

#include "common.cuh"

namespace dc {
namespace {

// Shared memory is addressed by byte offsets from the CTA's dynamic shared memory, so
// that a load needs no address arithmetic beyond the search's own offset.
template <typename T>
__device__ __forceinline__ T &sh(int off)
{
    extern __shared__ __align__(16) unsigned char smem[];
    return *reinterpret_cast<T *>(smem + off);
}

// Arrays of the solver: K (the newest column's keys H + e + b) and b of rows 1, 2, ..,
// 8 bytes a row (the 32-bit form uses the first half of each array), with 16 bytes
// between them whose last 8 are zero: b of row 0.
__host__ __device__ constexpr int chain_rows_bytes(int rows) { return rows * 8; }
__host__ __device__ constexpr int chain_pair_bytes(int rows) { return 2 * chain_rows_bytes(rows) + 16; }

// The columns kept for the traceback, 1..last, as 32-bit words at a stride of
// chain_stride(L) cells; columns 1..shared in shared memory (from byte `sm`) and the
// rest in a slot of the workspace. A word is the value itself where values have 32
// bits, otherwise H[m][1] - H[m][n], which lies between 0 and min(a[L], b[L] + h1):
// H[m][n] is at least H[1][1], and at least c_n + a[m] - b[L].
__host__ __device__ inline int chain_stride(int L) { return (L + 1) & ~1; }
struct KeptWords {
    int sm;
    uint32_t *gm;
    int stride, shared, last;
    static constexpr bool kWhole = false;
    __device__ __forceinline__ bool holds(int n) const { return n <= last; }
    // cells (m, n), (m + 1, n), m odd; the second may be padding past an odd L
    template <typename T>
    __device__ __forceinline__ void put2(int n, int m, T v0, T v1) const
    {
        if (!DC_CHECK(n >= 1 && m >= 1 && m < stride)) return;
        const uint2 x = make_uint2(uint32_t(v0), uint32_t(v1));
        if (n <= shared)
            sh<uint2>(sm + 4 * ((n - 1) * stride + (m - 1))) = x;
        else if (n <= last)
            *reinterpret_cast<uint2 *>(gm + int64_t(n - 1 - shared) * stride + (m - 1)) = x;
    }
    template <typename T>
    __device__ __forceinline__ T get(int n, int m) const
    {
        if (!DC_CHECK(n >= 1 && n <= last && m >= 1 && m <= stride)) return T(0);
        return T(n <= shared ? sh<uint32_t>(sm + 4 * ((n - 1) * stride + (m - 1)))
                             : gm[int64_t(n - 1 - shared) * stride + (m - 1)]);
    }
};
// whole values, every column: the triangle of cells m >= n
struct KeptValues {
    int64_t *at;
    int L;
    static constexpr bool kWhole = true;
    __device__ __forceinline__ bool holds(int) const { return true; }
    template <typename T>
    __device__ __forceinline__ void put2(int n, int m, T v0, T v1) const
    {
        if (!DC_CHECK(n >= 1 && m >= 1 && m <= L)) return;
        if (m >= n) at[tri_index(L, m, n)] = int64_t(v0);
        if (m + 1 >= n && m + 1 <= L) at[tri_index(L, m + 1, n)] = int64_t(v1);
    }
    template <typename T>
    __device__ __forceinline__ T get(int n, int m) const
    {
        if (!DC_CHECK(n >= 1 && m >= n && m <= L)) return T(0);
        return T(at[tri_index(L, m, n)]);
    }
};
// whether KeptWords can hold the values of an instance in 64 bits
__device__ __forceinline__ bool words_hold(uint64_t aL, uint64_t bL, uint64_t h1)
{
    return min(aL, bL + h1) < (uint64_t(1) << 32);
}

template <typename T>
struct Pair;
template <>
struct Pair<int32_t> {
    using type = int2;
    static constexpr int32_t kMax = INT32_MAX;
    static __device__ __forceinline__ int2 make(int32_t x, int32_t y) { return make_int2(x, y); }
};
template <>
struct Pair<int64_t> {
    using type = longlong2;
    static constexpr int64_t kMax = INT64_MAX;
    static __device__ __forceinline__ longlong2 make(int64_t x, int64_t y) { return make_longlong2(x, y); }
};

// Searches for the sorted keys below t0 and t1, two at once (independent load chains):
// q = the byte offset of key p + 1, with p the number of keys below t.
//
// halve_from<STEP>: the count lies in [0, 2 STEP - 1] past q; keys that the caller
// padded with the largest value end it earlier. UPTO: p counts the keys up to t (the
// padding too where t is the largest value: t + 1, to search below it, would not exist).
template <typename T, int STEP, bool UPTO = false>
__device__ __forceinline__ void halve_from(T t0, T t1, int &q0, int &q1)
{
    constexpr int S = int(sizeof(T));
    const T k0 = sh<T>(q0 + (STEP - 1) * S), k1 = sh<T>(q1 + (STEP - 1) * S);
    if (UPTO ? k0 <= t0 : k0 < t0) q0 += STEP * S;
    if (UPTO ? k1 <= t1 : k1 < t1) q1 += STEP * S;
    if constexpr (STEP > 1) halve_from<T, STEP / 2, UPTO>(t0, t1, q0, q1);
}
// search_below: N keys from byte kb, P the largest power of two <= N: the first probe
// splits [0, N] into two ranges of at most P values, the rest halve it.
template <typename T>
__device__ __forceinline__ void search_below(int kb, int N, int P, T t0, T t1, int &q0, int &q1)
{
    constexpr int S = int(sizeof(T));
    const T kp = sh<T>(kb + (P - 1) * S);
    const int far = kb + (N - P + 1) * S;
    q0 = kp < t0 ? far : kb;
    q1 = kp < t1 ? far : kb;
    switch (P) {  // uniform
        case 2048: halve_from<T, 1024>(t0, t1, q0, q1); break;
        case 1024: halve_from<T, 512>(t0, t1, q0, q1); break;
        case 512: halve_from<T, 256>(t0, t1, q0, q1); break;
        case 256: halve_from<T, 128>(t0, t1, q0, q1); break;
        case 128: halve_from<T, 64>(t0, t1, q0, q1); break;
        default:
            for (int st = P >> 1; st > 0; st >>= 1) {
                const T k0 = sh<T>(q0 + (st - 1) * S), k1 = sh<T>(q1 + (st - 1) * S);
                if (k0 < t0) q0 += st * S;
                if (k1 < t1) q1 += st * S;
            }
    }
}

// First k in [lo, lo + len] for which pred holds, given that it holds from some k on
// and at lo + len (which is not asked); one warp, 32 probes a round.
template <typename Pred>
__device__ __forceinline__ int warp_first(int lo, int len, Pred pred)
{
    const int lane = threadIdx.x & 31;
    while (len > 0) {
        const int step = (len + 31) / 32;
        const int probe = lo + (lane + 1) * step - 1;  // last k of this lane's piece
        const bool hit = probe >= lo + len || pred(probe);
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if (bal == 0u) return lo + len;  // the last piece ends the range
        const int q = __ffs(int(bal)) - 1;
        const int end = lo + len;
        lo += q * step;
        len = min(step - 1, end - lo);
    }
    return lo;
}

// Columns 2.., the traceback and the outputs of instance i, from its prefixes:
// thread tid of NT holds rows r, r+1 with r = 2 (j NT + tid) + 1 as a[j], b[j] (rows
// past L hold the totals). WARP: one warp solves it (NT = 32), else the CTA. kb: byte
// of K; D: bytes from K to b, both arrays with room for 2 NJ NT rows. word: shared
// memory, W decision words, pub: two values that the CTA's last row publishes (both
// CTA only). WINDOW: keys that a search looks at first, from where it ended in the column
// before (0: none). Returns false, having written nothing, when the optimum needs columns
// that `kept` does not hold.
template <bool FWD, typename T, int NJ, bool WARP, int WINDOW, typename Kept>
__device__ __forceinline__ bool chain_columns(int kb, int D, uint32_t *word, T *pub, int tid, int NT,
                                              int64_t i, int L, T dt, const T (&a)[NJ][2],
                                              const T (&b)[NJ][2], T aL, T bL, const Kept &kept,
                                              const SolveOut &o)
{
    using P2 = Pair<T>;
    using Two = typename P2::type;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int S = int(sizeof(T));
    static_assert(!WARP || WINDOW == 0, "a warp searches the whole range");
    constexpr bool kDrop = S == 8 && !Kept::kWhole;  // kept words are H[m][1] - H[m][n]
    const int lane = tid & 31, W = words_for(L);
    const T e = FWD ? T(0) : dt, h1 = FWD ? dt : T(0);  // H[m][1] = h1 + a[m]
    T h[NJ][2];
    bool in[NJ][2];  // rows 1..L-1: the k of a step
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int r = 2 * (j * NT + tid) + 1;
        in[j][0] = r < L;
        in[j][1] = r + 1 < L;
        h[j][0] = h1 + a[j][0];
        h[j][1] = h1 + a[j][1];
        // keys from row L on end every search: they lower nothing
        sh<Two>(kb + D + (r - 1) * S) = P2::make(b[j][0], b[j][1]);
        sh<Two>(kb + (r - 1) * S) = P2::make(in[j][0] ? h[j][0] + e + b[j][0] : P2::kMax,
                                             in[j][1] ? h[j][1] + e + b[j][1] : P2::kMax);
        if (r <= L) kept.put2(1, r, kDrop ? T(0) : h[j][0], kDrop ? T(0) : h[j][1]);
    }
    if (WARP) __syncwarp(); else __syncthreads();
    T hL = h1 + aL;  // H[L] of the newest column
    int s = 1;
    bool deep = false;  // the optimum lies beyond the kept columns
    const int N = L - 1;
    const int P = 1 << (31 - __clz(N | 1));
    const T tail = N > 0 ? aL - sh<T>(kb + D + (N - 1) * S) : aL;  // a[L] - b[L-1]
    T c = FWD ? dt : T(0);
    // Where a row's search ended never moves back from one column to the next: its keys
    // fall or stay, and c does not fall. So from the third column on it starts there, and
    // the whole range is searched only when some lane has moved past the window.
    const int lim = kb + (2 * NJ * NT - WINDOW) * S;  // keys from row L on are the largest value
    int q[NJ][2];
    for (int n = 2; n <= L; ++n) {
        if (FWD) c += dt;
        if (c + tail >= hL) break;
        T v[NJ][2];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int r = 2 * (j * NT + tid) + 1;
            const T t0 = c + a[j][0], t1 = c + a[j][1];
            int q0 = kb, q1 = kb;
            bool search = true;
            if constexpr (WINDOW > 0) {
                if (n > 2) {
                    q0 = q[j][0];
                    q1 = q[j][1];
                    // backward, two in five warps have not moved at all
                    if (!FWD) search = __any_sync(kAll, sh<T>(q0) < t0 || sh<T>(q1) < t1);
                    if (search) {
                        q0 = min(q0, lim);
                        q1 = min(q1, lim);
                        search = __any_sync(kAll, sh<T>(q0 + (WINDOW - 1) * S) < t0 ||
                                                      sh<T>(q1 + (WINDOW - 1) * S) < t1);
                        if (!search) halve_from<T, WINDOW / 2>(t0, t1, q0, q1);
                    }
                }
            }
            if constexpr (WARP)
                halve_from<T, NJ == 1 ? 32 : NJ == 2 ? 64 : 128>(t0, t1, q0, q1);
            else if (search)
                search_below<T>(kb, N, P, t0, t1, q0, q1);
            if constexpr (WINDOW > 0) {
                q[j][0] = q0;
                q[j][1] = q1;
            }
            // k = p + 1, at q, is the first with H + e + b >= t, k = p the last below it
            // (p = 0 gives t, which lowers nothing)
            v[j][0] = min(min(h[j][0], sh<T>(q0) - sh<T>(q0 + D)), t0 - sh<T>(q0 + D - S));
            v[j][1] = min(min(h[j][1], sh<T>(q1) - sh<T>(q1 + D)), t1 - sh<T>(q1 + D - S));
            if (r <= L)
                kept.put2(n, r, kDrop ? h1 + a[j][0] - v[j][0] : v[j][0],
                          kDrop ? h1 + a[j][1] - v[j][1] : v[j][1]);
            if (!WARP && (r == L || r + 1 == L)) pub[n & 1] = r == L ? v[j][0] : v[j][1];
        }
        T hn;
        if (WARP) {
            // the last row that a lane holds is row L or past it (then it has row L's a, and
            // comes out the same)
            hn = __shfl_sync(kAll, v[NJ - 1][1], 31);
            __syncwarp();  // every lane has read column n-1 (a shuffle orders no memory)
        } else {
            __syncthreads();
            hn = pub[n & 1];
        }
        // another column only while a lowered H may still lower H[L] (rows from L on
        // never pass: their H is H[L])
        bool more = false;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int r = 2 * (j * NT + tid) + 1;
            more |= v[j][0] < h[j][0] && v[j][0] + e < hn;
            more |= v[j][1] < h[j][1] && v[j][1] + e < hn;
            h[j][0] = v[j][0];
            h[j][1] = v[j][1];
            sh<Two>(kb + (r - 1) * S) = P2::make(in[j][0] ? v[j][0] + e + b[j][0] : P2::kMax,
                                                 in[j][1] ? v[j][1] + e + b[j][1] : P2::kMax);
        }
        if (hn < hL) {
            hL = hn;
            s = n;
            if (n > 2 && !kept.holds(n - 1)) deep = true;
        }
        if (WARP) {
            __syncwarp();
            if (!__any_sync(kAll, more) || deep) break;
        } else {
            if (!__syncthreads_or(more) || deep) break;
        }
    }
    if (deep) return false;

    // ---- traceback by one warp: Path[m][n] = the first k with b[k] >= c_n + a[m] - v;
    // a goes to the key array first
    if (!WARP || s > 1) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            sh<Two>(kb + 2 * (j * NT + tid) * S) = P2::make(a[j][0], a[j][1]);
    }
    if (WARP) __syncwarp(); else __syncthreads();
    if (!WARP && tid >= 32) return true;
    int err = 0, m = L, n = s;
    T v = hL;
    uint32_t mine = 0u;  // WARP: lane w's decision word w
    // f_m of the decision, from its own segments: the largest over its segments j of
    // c_j + a[end] - b[start] + (s - j) e, then the same e + b[L] as T
    T span = T(0), later = T(0);
    T cn = FWD ? T(n) * dt : T(0);
    while (n > 1) {
        const T am = cn + sh<T>(kb + (m - 1) * S);
        const T thr = am - v;
        int k;
        if (WARP) {
            int below = 0;  // rows past L hold b[L] >= thr, or there is no such k
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                below += __popc(__ballot_sync(kAll, b[j][0] < thr)) + __popc(__ballot_sync(kAll, b[j][1] < thr));
            k = below + 1;
        } else {
            k = warp_first(1, N, [&](int q) { return sh<T>(kb + D + (q - 1) * S) >= thr; });
        }
        if (k < n - 1 || k >= m) {
            err = 1;
            break;
        }
        T hk = kept.template get<T>(n - 1, k);
        if (kDrop) hk = h1 + sh<T>(kb + (k - 1) * S) - hk;
        if (hk + e > v) {
            err = 1;
            break;
        }
        if (o.replay) {
            const T w = am - sh<T>(kb + D + (k - 1) * S) + later;
            span = n == s ? w : max(span, w);
            later += e;
        }
        const uint32_t bit = 1u << ((k - 1) & 31);
        if (WARP)
            mine |= lane == ((k - 1) >> 5) ? bit : 0u;
        else if (lane == 0)
            word[(k - 1) >> 5] |= bit;
        v = hk;
        m = k;
        n -= 1;
        if (FWD) cn -= dt;
    }
    if (o.replay) {
        const T first = h1 + later + (s > 1 ? sh<T>(kb + (m - 1) * S) : aL);  // the first segment
        span = s > 1 ? max(span, first) : first;
    }
    if (!WARP) __syncwarp();
    if (lane == 0) {
        if (o.replay) o.replay[i] = err ? -int64_t(DC_ERR_INTERNAL) : int64_t(span + e) + int64_t(bL);
        o.makespan[i] = err ? -int64_t(DC_ERR_INTERNAL) : int64_t(hL + e) + int64_t(bL);
        if (o.nseg) o.nseg[i] = err ? 0 : s;
        if (o.status) o.status[i] = err ? DC_ERR_INTERNAL : DC_OK;
    }
    if (WARP) {
        if (lane < W) o.bits[i * W + lane] = err ? 0u : mine;
        __syncwarp();  // lane 0 rejoins here and not somewhere in the next instance
    } else {
        for (int w = lane; w < W; w += 32) o.bits[i * W + w] = err ? 0u : word[w];
    }
    return true;
}

__device__ __forceinline__ void chain_failure(int st, int64_t i, int W, int tid, int NT, const SolveOut &o)
{
    if (tid == 0) {
        o.makespan[i] = -int64_t(st);
        if (o.nseg) o.nseg[i] = 0;
        if (o.status) o.status[i] = st;
        if (o.replay) o.replay[i] = -int64_t(st);
    }
    for (int w = tid; w < W; w += NT) o.bits[i * W + w] = 0u;
}

// Where an instance's costs come from: operator()(r, c0, c1, x0, x1) gives the compute
// and transfer costs of rows r, r+1 (r odd) in processing order, zero past L. This one
// reads its rows; vec: they are 16-byte aligned and L is even.
template <bool FWD>
struct RowLoader {
    const int64_t *crow, *xrow;
    int L;
    bool vec;
    __device__ __forceinline__ void operator()(int r, uint64_t &c0, uint64_t &c1, uint64_t &x0,
                                               uint64_t &x1) const
    {
        c0 = c1 = x0 = x1 = 0;
        if (r > L) return;
        if (vec) {
            const int at = FWD ? r - 1 : L - r - 1;
            const ulonglong2 c = __ldg(reinterpret_cast<const ulonglong2 *>(crow + at));
            const ulonglong2 x = __ldg(reinterpret_cast<const ulonglong2 *>(xrow + at));
            c0 = FWD ? c.x : c.y;
            c1 = FWD ? c.y : c.x;
            x0 = FWD ? x.x : x.y;
            x1 = FWD ? x.y : x.x;
        } else {
            const int at = FWD ? r - 1 : L - r, next = FWD ? at + 1 : at - 1;
            c0 = uint64_t(__ldg(crow + at));
            x0 = uint64_t(__ldg(xrow + at));
            if (r < L) {
                c1 = uint64_t(__ldg(crow + next));
                x1 = uint64_t(__ldg(xrow + next));
            }
        }
    }
};

// Inclusive prefixes over a warp's lanes of two values at once.
template <typename U>
__device__ __forceinline__ void scan2(U &sa, U &sb, int lane)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const U ua = __shfl_up_sync(0xffffffffu, sa, d), ub = __shfl_up_sync(0xffffffffu, sb, d);
        if (lane >= d) {
            sa += ua;
            sb += ub;
        }
    }
}

// b's row 0, for arrays with room for `rows` rows at byte kb.
__device__ __forceinline__ void zero_row(int kb, int rows)
{
    sh<int64_t>(kb + chain_rows_bytes(rows) + 8) = 0;
}

// --------------------------------------------------------------- warp per instance
// The same with a flag that gathers bit 31 of every partial sum: clear for all lanes
// when no sum of the prefix reached 2^31 (the operands of the first that does are
// below it, so it does not wrap).
__device__ __forceinline__ void scan2_flag(uint32_t &sa, uint32_t &sb, uint32_t &flag, int lane)
{
    flag |= sa | sb;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t ua = __shfl_up_sync(0xffffffffu, sa, d), ub = __shfl_up_sync(0xffffffffu, sb, d);
        if (lane >= d) {
            sa += ua;
            sb += ub;
        }
        flag |= sa | sb;
    }
}

// The prefixes of an instance's rows over a warp, NJ row pairs per lane (L <= 64 NJ, the
// row layout of chain_columns): go(a, b, aL, bL) gets them in int32_t where
// a[L] + b[L] + (L + 1) dt < 2^31, otherwise in int64_t, and its value is returned; bad(st)
// gets an input error's status.
template <bool FWD, int NJ, typename Load, typename Go, typename Bad>
__device__ __forceinline__ bool with_warp_prefix(int L, const Load &load, int64_t dt, Go go, Bad bad)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    uint64_t a[NJ][2], b[NJ][2];
    uint32_t hi = uint32_t(uint64_t(dt) >> 32), flag = uint32_t(dt);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int r = 2 * (32 * j + lane) + 1;
        if (FWD)
            load(r, b[j][0], b[j][1], a[j][0], a[j][1]);
        else
            load(r, a[j][0], a[j][1], b[j][0], b[j][1]);
        hi |= uint32_t((a[j][0] | a[j][1] | b[j][0] | b[j][1]) >> 32);
        flag |= uint32_t(a[j][0] | a[j][1] | b[j][0] | b[j][1]);
    }
    int32_t a32[NJ][2], b32[NJ][2];
    uint32_t aL32 = 0, bL32 = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        uint32_t sa = uint32_t(a[j][0]) + uint32_t(a[j][1]), sb = uint32_t(b[j][0]) + uint32_t(b[j][1]);
        scan2_flag(sa, sb, flag, lane);
        a32[j][0] = int32_t(aL32 + sa - uint32_t(a[j][1]));
        a32[j][1] = int32_t(aL32 + sa);
        b32[j][0] = int32_t(bL32 + sb - uint32_t(b[j][1]));
        b32[j][1] = int32_t(bL32 + sb);
        aL32 += __shfl_sync(kAll, sa, 31);  // below 2^31 + 2^31 where it matters
        bL32 += __shfl_sync(kAll, sb, 31);
        flag |= aL32 | bL32;
    }
    if (!__any_sync(kAll, (hi | (flag >> 31)) != 0u) &&
        uint64_t(aL32) + bL32 + uint64_t(L + 1) * uint64_t(dt) < (uint64_t(1) << 31))
        return go(a32, b32, int32_t(aL32), int32_t(bL32));
    // any other instance: 64-bit sums and the input checks
    uint64_t any = uint64_t(dt), aL = 0, bL = 0;
    int64_t a64[NJ][2], b64[NJ][2];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        any |= a[j][0] | a[j][1] | b[j][0] | b[j][1];
        uint64_t sa = a[j][0] + a[j][1], sb = b[j][0] + b[j][1];
        scan2(sa, sb, lane);
        a64[j][0] = int64_t(aL + sa - a[j][1]);
        a64[j][1] = int64_t(aL + sa);
        b64[j][0] = int64_t(bL + sb - b[j][1]);
        b64[j][1] = int64_t(bL + sb);
        aL += __shfl_sync(kAll, sa, 31);
        bL += __shfl_sync(kAll, sb, 31);
    }
    const uint32_t all = __reduce_or_sync(kAll, uint32_t(any >> 32));
    if (all >> 31) return bad(DC_ERR_NEGATIVE);
    if (all >> 20 || exceeds_range(L, dt, FWD ? bL : aL, FWD ? aL : bL)) return bad(DC_ERR_RANGE);
    return go(a64, b64, int64_t(aL), int64_t(bL));
}

// Solves instance i with one warp, NJ row pairs per lane (L <= 64 NJ). kb: byte of the
// warp's K, b beside it (chain_pair_bytes(64 NJ); the caller zeroes b's row 0 once with
// zero_row). Returns false, having written nothing, when the instance is left to the
// work list, as chain_solve does.
template <bool FWD, int NJ, typename Load, typename Kept>
__device__ __forceinline__ bool chain_solve_warp(int kb, int64_t i, int L, const Load &load,
                                                 int64_t dt, const SolveOut &o, const Kept &kept)
{
    constexpr int D = 64 * NJ * 8 + 16;
    const int lane = threadIdx.x & 31;
    return with_warp_prefix<FWD, NJ>(
        L, load, dt,
        [&](const auto &a, const auto &b, auto aL, auto bL) {
            using T = decltype(aL);
            if (sizeof(T) == 8 && !Kept::kWhole &&
                !words_hold(uint64_t(aL), uint64_t(bL), uint64_t(FWD ? dt : 0)))
                return false;
            return chain_columns<FWD, T, NJ, true, 0>(kb, D, static_cast<uint32_t *>(nullptr),
                                                   static_cast<T *>(nullptr), lane, 32, i, L, T(dt),
                                                   a, b, aL, bL, kept, o);
        },
        [&](int st) {
            chain_failure(st, i, words_for(L), lane, 32, o);
            return true;
        });
}

// ---------------------------------------------------------------- CTA per instance
constexpr int kChainThreads = 1024;  // threads per instance, at most
constexpr int kChainPairs = 2;       // row pairs per thread, at most

__host__ __device__ inline size_t chain_word_bytes(int L)
{
    return (size_t(words_for(L)) * 4 + 15) / 16 * 16;
}
// K and b with room for `rows` rows (2 NJ times the threads), the decision words, then the
// scan's partial sums, the warps' flags and two published values
constexpr size_t kChainScratch = size_t(2 * kChainPairs * (kChainThreads / 32)) * 8 + 32 * 4 + 16;
__host__ __device__ inline size_t chain_smem_bytes(int L, int rows)
{
    return chain_pair_bytes(rows) + chain_word_bytes(L) + kChainScratch;
}
// the most that any choice of threads takes at depth L: whole warps of one row pair
__host__ __device__ inline size_t chain_smem_most(int L) { return chain_smem_bytes(L, (L + 127) / 128 * 128); }

// The prefixes of an instance's rows over the whole CTA, in processing order (a, b and
// the row layout of chain_columns; 64-bit). tot, orw: scratch. One CTA barrier, which
// also publishes what the threads wrote to shared memory before. Returns the
// instance's status: DC_OK or its input error.
template <bool FWD, int NJ, typename Load>
__device__ __forceinline__ int cta_prefix(uint64_t *tot, uint32_t *orw, int L, const Load &load,
                                          int64_t dt, uint64_t (&a)[NJ][2], uint64_t (&b)[NJ][2],
                                          uint64_t &aL, uint64_t &bL)
{
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
    uint64_t any = uint64_t(dt);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int r = 2 * (j * NT + tid) + 1;
        uint64_t a0, a1, b0, b1;
        if (FWD)
            load(r, b0, b1, a0, a1);
        else
            load(r, a0, a1, b0, b1);
        any |= a0 | a1 | b0 | b1;
        uint64_t sa = a0 + a1, sb = b0 + b1;
        scan2(sa, sb, lane);
        if (lane == 31) {
            tot[j * NW + warp] = sa;
            tot[(NJ + j) * NW + warp] = sb;
        }
        a[j][0] = sa - a1;
        a[j][1] = sa;
        b[j][0] = sb - b1;
        b[j][1] = sb;
    }
    const uint32_t hi = __reduce_or_sync(0xffffffffu, uint32_t(any >> 32));
    if (lane == 0) orw[warp] = hi;
    __syncthreads();
    // every warp scans the partial sums: lane q holds those of warp q
    const uint32_t all = __reduce_or_sync(0xffffffffu, lane < NW ? orw[lane] : 0u);
    aL = 0;
    bL = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        uint64_t sa = lane < NW ? tot[j * NW + lane] : 0u, sb = lane < NW ? tot[(NJ + j) * NW + lane] : 0u;
        const uint64_t xa = sa, xb = sb;
        scan2(sa, sb, lane);
        const uint64_t oa = aL + __shfl_sync(0xffffffffu, sa - xa, warp);
        const uint64_t ob = bL + __shfl_sync(0xffffffffu, sb - xb, warp);
        a[j][0] += oa;
        a[j][1] += oa;
        b[j][0] += ob;
        b[j][1] += ob;
        aL += __shfl_sync(0xffffffffu, sa, 31);
        bL += __shfl_sync(0xffffffffu, sb, 31);
    }
    if (all >> 31) return DC_ERR_NEGATIVE;
    if (all >> 20 || exceeds_range(L, dt, FWD ? bL : aL, FWD ? aL : bL)) return DC_ERR_RANGE;
    return DC_OK;
}

// Solves instance i with the whole CTA, NJ row pairs per thread, keeping columns in
// `kept`. Returns false, having written nothing, when the instance is left to the work
// list: its values do not fit there, or its optimum needs a column it does not hold.
// WINDOW: see chain_columns.
template <bool FWD, int NJ, int WINDOW = 0, typename Load, typename Kept>
__device__ bool chain_solve(int64_t i, int L, const Load &load, int64_t dt, const SolveOut &o,
                            const Kept &kept)
{
    const int NT = blockDim.x, tid = threadIdx.x;
    const int W = words_for(L), rows = 2 * NJ * NT, D = chain_rows_bytes(rows) + 16;
    uint32_t *word = &sh<uint32_t>(chain_pair_bytes(rows));
    uint64_t *tot = &sh<uint64_t>(chain_pair_bytes(rows) + int(chain_word_bytes(L)));
    uint32_t *orw = reinterpret_cast<uint32_t *>(tot + 2 * kChainPairs * (kChainThreads / 32));
    unsigned char *pub = reinterpret_cast<unsigned char *>(orw + 32);

    if (tid == 0) zero_row(0, rows);
    for (int w = tid; w < W; w += NT) word[w] = 0u;
    uint64_t a[NJ][2], b[NJ][2], aL, bL;
    const int st = cta_prefix<FWD, NJ>(tot, orw, L, load, dt, a, b, aL, bL);
    if (st != DC_OK) {
        chain_failure(st, i, W, tid, NT, o);
        return true;
    }
    if (aL + bL + uint64_t(L + 1) * uint64_t(dt) < (uint64_t(1) << 31)) {
        int32_t a32[NJ][2], b32[NJ][2];
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a32[j][u] = int32_t(a[j][u]);
                b32[j][u] = int32_t(b[j][u]);
            }
        return chain_columns<FWD, int32_t, NJ, false, WINDOW>(0, D, word, reinterpret_cast<int32_t *>(pub), tid,
                                                      NT, i, L, int32_t(dt), a32, b32, int32_t(aL),
                                                      int32_t(bL), kept, o);
    }
    int64_t a64[NJ][2], b64[NJ][2];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a64[j][u] = int64_t(a[j][u]);
            b64[j][u] = int64_t(b[j][u]);
        }
    if (!Kept::kWhole && !words_hold(aL, bL, uint64_t(FWD ? dt : 0))) return false;
    return chain_columns<FWD, int64_t, NJ, false, WINDOW>(0, D, word, reinterpret_cast<int64_t *>(pub), tid, NT,
                                                  i, L, dt, a64, b64, int64_t(aL), int64_t(bL), kept, o);
}

}  // namespace
}  // namespace dc
