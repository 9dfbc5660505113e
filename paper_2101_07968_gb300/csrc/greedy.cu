// The paper's competing schedulers as batched kernels (Sec. II-C): greedy
// parameter scheduling of iBatch (Algorithm 1, forward) and greedy gradient
// scheduling of iPart (Algorithm 2, backward).
//
// Readings where the listings leave a choice open (the same as the oracle's):
//  * ties in "choose the one with minimum ..." keep the first candidate of the
//    listing's enumeration (positions ascending, Algorithm 2's n ascending);
//  * an empty Options set takes the position with the largest slack (the
//    condition's left side less its right side), the one closest to meeting it;
//  * Algorithm 1's first pair (D1, D2): among the pairs meeting the condition,
//    maximum first-segment compute, then minimum first transfer, then minimum
//    slack; with none meeting it, the largest slack; the loop runs while m < L;
//  * Algorithm 2's "estimated total execution time" is f_m, the backward replay.
//
// Prefix sums are non-decreasing, which makes each choice a search instead of the
// listings' enumerations:
//  * forward: D1 is valid iff dt + P[L] - P[D1] >= FC[D1] (take D2 = L), a prefix
//    of [1, L-1]; its largest FC is at the last valid D1 and the smallest P among
//    equal FC at the first D1 of that plateau (a lower D1 never has a larger
//    minimum slack). D2, and every later step, is the first x whose transfer
//    covers the compute (minimum slack), else the first x reaching P[L];
//  * backward: the positions x meeting k*dt + GT[m..L] >= BC[x..m-1] form a
//    suffix [x*, m-1]; the minimum slack is at x*; with none, the largest slack is
//    at m-1, extended down over zero-compute layers (ties keep the lowest x).
// Segment boundaries come in time order, so f_m is accumulated on the fly
// (forward: end_s = max(end_{s-1}, s*dt + P[b_s]) + FC[b_s] - FC[b_{s-1}];
// backward: link = max(link, BC[q..L]) + dt + GT of the segment).
//
// Three kernels, chosen in launch_greedy. One instance per thread scans its own rows: O(L)
// for Algorithm 1, O(L^2) for Algorithm 2, bound by the latency of its uncoalesced reads.
// One instance per warp (L <= 64) or per CTA has its prefix sums in registers and
// shared memory: Algorithm 1's one chain takes a search over all rows at once per step (a
// ballot, or 32 probes), and Algorithm 2's L - 1 chains, one per second position, run
// side by side with a binary search per step; both are bound by integer issue and by
// the longest chain of the warp.
// 65,537 x 54 (ResNet-50): forward 18 us and backward 80 us of kernel time (45 and 1,540
// one instance per thread, 127 backward with 64-bit prefixes, one chain per lane at a time).
#include "chain.cuh"

namespace dc {

int sm_count();  // SMs of the current device (dp_small.cu)

namespace {

__device__ __forceinline__ int instance_check(int L, const int64_t *c, const int64_t *x, int64_t dt,
                                              uint64_t &sc, uint64_t &sx)
{
    bool neg = dt < 0, big = (dt >> 52) != 0;
    sc = 0;
    sx = 0;
    for (int l = 0; l < L; ++l) {
        const int64_t cv = __ldg(c + l), xv = __ldg(x + l);
        neg |= (cv < 0) | (xv < 0);
        big |= ((cv | xv) >> 52) != 0;
        sc += uint64_t(cv);
        sx += uint64_t(xv);
    }
    if (neg) return DC_ERR_NEGATIVE;
    if (big || exceeds_range(L, dt, sc, sx)) return DC_ERR_RANGE;
    return DC_OK;
}

__device__ __forceinline__ void set_bit(uint32_t *w, int l) { w[(l - 1) >> 5] |= 1u << ((l - 1) & 31); }

// Algorithm 1. fc, pt: the instance's rows (layer l at index l-1).
__device__ void greedy_fwd(int L, const int64_t *fc, const int64_t *pt, int64_t dt, int64_t Ptot,
                           uint32_t *bits, int64_t *makespan)
{
    if (L < 2) {  // one segment
        *makespan = dt + __ldg(pt) + __ldg(fc);
        return;
    }
    // steps 1-4: D1 (and the prefix sums at it)
    int d1 = 0, plateau = 1;
    int64_t P = 0, FC = 0, P1 = 0, FC1 = 0, plateauP = 0, plateauFC = 0;
    for (int d = 1; d < L; ++d) {
        const int64_t f = __ldg(fc + d - 1);
        if (d == 1 || f != 0) {  // FC grows: a new plateau starts at d
            plateau = d;
            plateauP = P + __ldg(pt + d - 1);
            plateauFC = FC + f;
        }
        P += __ldg(pt + d - 1);
        FC += f;
        if (dt + Ptot - P < FC) break;  // valid D1 form a prefix
        d1 = plateau;
        P1 = plateauP;
        FC1 = plateauFC;
    }
    int64_t Pm, FCm;
    int m;
    if (d1 > 0) {
        // D2: the first x > D1 with dt + P[x] - P[D1] >= FC[D1] (exists: x = L)
        Pm = P1;
        FCm = FC1;
        m = d1;
        do {
            ++m;
            Pm += __ldg(pt + m - 1);
            FCm += __ldg(fc + m - 1);
        } while (dt + Pm - P1 < FC1);
    } else {
        // no pair meets the condition: the largest slack is D1 = 1 and D2 the
        // first x > 1 with P[x] = P[L]
        d1 = 1;
        P1 = __ldg(pt);
        FC1 = __ldg(fc);
        Pm = P1;
        FCm = FC1;
        m = 1;
        do {
            ++m;
            Pm += __ldg(pt + m - 1);
            FCm += __ldg(fc + m - 1);
        } while (Pm < Ptot);
    }
    // f_m over the segments fixed so far: [1, D1], [D1+1, D2]
    int64_t end = dt + P1 + FC1;
    end = max(end, 2 * dt + Pm) + (FCm - FC1);
    int s = 2;
    set_bit(bits, d1);
    int64_t FCn = FC1;
    while (m < L) {
        set_bit(bits, m);
        const int64_t cover = FCm - FCn;
        // the first x > m whose transfer covers `cover`; else the first x with
        // P[x] = P[L] (largest slack)
        int j = m, jg = -1;
        int64_t Px = Pm, FCx = FCm, Pg = 0, FCg = 0;
        bool ok = false;
        while (j < L) {
            ++j;
            Px += __ldg(pt + j - 1);
            FCx += __ldg(fc + j - 1);
            if (jg < 0 && Px == Ptot) {
                jg = j;
                Pg = Px;
                FCg = FCx;
            }
            if (dt + Px - Pm >= cover) {
                ok = true;
                break;
            }
        }
        if (!ok) {
            j = jg;
            Px = Pg;
            FCx = FCg;
        }
        ++s;
        end = max(end, int64_t(s) * dt + Px) + (FCx - FCm);
        FCn = FCm;
        m = j;
        Pm = Px;
        FCm = FCx;
    }
    *makespan = end;
}

// One chain of Algorithm 2 from second position n; returns its f_m and, when
// `bits` is given, sets its decision there. BCs, GTs: sums of bc, gt over
// layers n..L.
__device__ int64_t greedy_bwd_chain(int L, const int64_t *bc, const int64_t *gt, int64_t dt,
                                    int n, int64_t BCs, int64_t GTs, uint32_t *bits)
{
    // segment 1 holds layers L..n
    int64_t link = BCs + dt + GTs;  // f_m so far
    if (bits) set_bit(bits, L + 1 - n);
    int m = n;
    int64_t k = 1;
    while (m > 1) {
        const int64_t limit = k * dt + GTs;  // the listing's link estimate
        // x* = the lowest x in [1, m-1] with BC[x..m-1] <= limit
        int64_t s = 0, g = 0;
        int x = m;
        while (x > 1) {
            const int64_t b = __ldg(bc + x - 2);
            if (s + b > limit) break;
            s += b;
            g += __ldg(gt + x - 2);
            --x;
        }
        if (x == m) {  // none: the largest slack, x = m-1 and the zero-compute layers below
            s = __ldg(bc + m - 2);
            g = __ldg(gt + m - 2);
            x = m - 1;
            while (x > 1 && __ldg(bc + x - 2) == 0) {
                g += __ldg(gt + x - 2);
                --x;
            }
        }
        // segment m-1..x
        BCs += s;
        GTs += g;
        link = max(link, BCs) + dt + g;
        if (bits && x > 1) set_bit(bits, L + 1 - x);
        m = x;
        k += 1;
    }
    return link;
}

// Algorithm 2. bc, gt: the instance's rows in layer order 1..L.
__device__ void greedy_bwd(int L, const int64_t *bc, const int64_t *gt, int64_t dt, int64_t BCtot,
                           int64_t GTtot, uint32_t *bits, int64_t *makespan)
{
    if (L < 2) {
        *makespan = BCtot + dt + GTtot;
        return;
    }
    int best_n = 2;
    int64_t best = 0, BCs = BCtot, GTs = GTtot;
    for (int n = 2; n <= L; ++n) {
        BCs -= __ldg(bc + n - 2);  // layers n..L
        GTs -= __ldg(gt + n - 2);
        const int64_t t = greedy_bwd_chain(L, bc, gt, dt, n, BCs, GTs, nullptr);
        if (n == 2 || t < best) {
            best = t;
            best_n = n;
        }
    }
    BCs = BCtot;
    GTs = GTtot;
    for (int n = 2; n <= best_n; ++n) {
        BCs -= __ldg(bc + n - 2);
        GTs -= __ldg(gt + n - 2);
    }
    greedy_bwd_chain(L, bc, gt, dt, best_n, BCs, GTs, bits);
    *makespan = best;
}

template <bool FWD>
__global__ void __launch_bounds__(128) greedy_kernel(int64_t batch, int L,
                                                     const int64_t *__restrict__ comp,
                                                     const int64_t *__restrict__ xfer,
                                                     const int64_t *__restrict__ dt,
                                                     int64_t *__restrict__ makespan,
                                                     uint32_t *__restrict__ bits)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    const int W = words_for(L);
    uint32_t *w = bits + i * W;
    for (int q = 0; q < W; ++q) w[q] = 0u;
    const int64_t *c = comp + i * L, *x = xfer + i * L;
    const int64_t dti = __ldg(dt + i);
    uint64_t sc, sx;
    const int st = instance_check(L, c, x, dti, sc, sx);
    if (st != DC_OK) {
        makespan[i] = -int64_t(st);
        return;
    }
    if (FWD)
        greedy_fwd(L, c, x, dti, int64_t(sx), w, makespan + i);
    else
        greedy_bwd(L, c, x, dti, int64_t(sc), int64_t(sx), w, makespan + i);
}

struct GreedyArgs {
    int64_t batch;
    int L;
    const int64_t *comp, *xfer, *dt;
    int64_t *makespan;
    uint32_t *bits;
    int vec;  // the cost rows are 16-byte aligned
};

// Prefixes A, B of rows 0..L (chain.cuh's a and b), then the decision words, the
// scan's partial sums and flags, and the warps' best chains.
__host__ __device__ inline size_t greedy_row_bytes(int L) { return (size_t(L + 2) * 8 + 15) / 16 * 16; }
constexpr size_t kGreedyScratch = size_t(2 * kChainPairs * (kChainThreads / 32)) * 8 + 32 * 4 + 32 * 16;
__host__ __device__ inline size_t greedy_smem_bytes(int L)
{
    return 2 * greedy_row_bytes(L) + chain_word_bytes(L) + kGreedyScratch;
}

// Algorithm 1 by one warp.
template <typename T>
__device__ T greedy_forward_warp(const T *A, const T *B, int L, T dt, uint32_t *word)
{
    const T aL = A[L];
    auto mark = [&](int l) {
        if ((threadIdx.x & 31) == 0) set_bit(word, l);
    };
    const int last = warp_first(1, L - 1, [&](int d) { return A[d] + B[d] > dt + aL; }) - 1;
    int n = 1, m;
    if (last >= 1) {
        n = warp_first(1, last - 1, [&](int d) { return B[d] >= B[last]; });
        const T thr = A[n] + B[n] - dt;
        m = warp_first(n + 1, L - n - 1, [&](int x) { return A[x] >= thr; });
    } else {
        m = warp_first(2, L - 2, [&](int x) { return A[x] >= aL; });
    }
    mark(n);
    T pull = dt + dt, end = dt + A[n] + B[n];
    end = max(end, pull + A[m]) + (B[m] - B[n]);
    for (int step = 2; m < L && step <= L; ++step) {  // m grows every time
        mark(m);
        // the first x that covers the segment's compute, else the first with all transfers
        const T thr = min(A[m] + (B[m] - B[n]) - dt, aL);
        const int x = warp_first(m + 1, L - m - 1, [&](int q) { return A[q] >= thr; });
        pull += dt;
        end = max(end, pull + A[x]) + (B[x] - B[m]);
        n = m;
        m = x;
    }
    return end;
}

// One chain of Algorithm 2 whose first push holds the last p layers; visit(q) for
// every break. Returns its f_m.
template <typename T, typename Visit>
__device__ __forceinline__ T greedy_chain(const T *A, const T *B, int L, int P, T dt, int p, Visit visit)
{
    T link = A[p] + dt + B[p], sent = dt;
    visit(p);
    for (int step = p; p < L && step < L; ++step) {  // p grows every time
        // the longest segment whose compute the link estimate covers, else one layer
        // and the zero-compute layers after it
        const T lim = max(A[p] + sent + B[p], A[p + 1]);
        int q = p + 1;
        for (int st = P; st > 0; st >>= 1)
            if (q + st <= L && A[q + st] <= lim) q += st;
        link = max(link, A[q]) + dt + (B[q] - B[p]);
        sent += dt;
        p = q;
        if (p < L) visit(p);
    }
    return link;
}

// The chain again, for its decision. Not inlined: a second copy beside the loop over the
// chains takes registers from it (20,000 x 128 91 us with it inlined, 73 so).
template <typename T>
__device__ __noinline__ void mark_chain(const T *A, const T *B, int L, int P, T dt, int p, uint32_t *word)
{
    greedy_chain(A, B, L, P, dt, p, [&](int q) { set_bit(word, q); });
}

// Algorithm 2 by the CTA, two warps or more; the result in thread 0.
template <typename T>
__device__ T greedy_backward_cta(const T *A, const T *B, int L, T dt, uint32_t *word, longlong2 *best_of)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = blockDim.x >> 5;
    int P = 1;
    while (2 * P < L) P *= 2;
    T best = T(0);
    int at = 0;  // ties keep the longest first push (the lowest second position)
    for (int p = 1 + tid; p < L; p += int(blockDim.x)) {
        const T t = greedy_chain(A, B, L, P, dt, p, [](int) {});
        if (at == 0 || t <= best) {
            best = t;
            at = p;
        }
    }
    int64_t key = at ? int64_t(best) : INT64_MAX;
    int from = at;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const int64_t k = __shfl_xor_sync(0xffffffffu, key, d);
        const int f = __shfl_xor_sync(0xffffffffu, from, d);
        if (k < key || (k == key && f > from)) {
            key = k;
            from = f;
        }
    }
    if (lane == 0) best_of[warp] = make_longlong2(key, from);
    __syncthreads();
    for (int w = 0; w < NW; ++w) {
        const longlong2 o = best_of[w];
        if (o.x < key || (o.x == key && int(o.y) > from)) {
            key = o.x;
            from = int(o.y);
        }
    }
    if (tid == 0) mark_chain(A, B, L, P, dt, from, word);
    __syncthreads();
    return T(key);
}

template <bool FWD, typename T, int NJ>
__device__ void greedy_solve(unsigned char *smem, uint32_t *word, longlong2 *best_of, int64_t i,
                             const GreedyArgs &g, T dt, const uint64_t (&a)[NJ][2],
                             const uint64_t (&b)[NJ][2])
{
    const int L = g.L, tid = threadIdx.x, NT = blockDim.x, W = words_for(L);
    T *A = reinterpret_cast<T *>(smem), *B = reinterpret_cast<T *>(smem + greedy_row_bytes(L));
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int r = 2 * (j * NT + tid) + 1;
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (r + u <= L) {
                A[r + u] = T(a[j][u]);
                B[r + u] = T(b[j][u]);
            }
    }
    if (tid == 0) {
        A[0] = T(0);
        B[0] = T(0);
    }
    __syncthreads();
    T t = T(0);
    if (!FWD)
        t = greedy_backward_cta(A, B, L, dt, word, best_of);
    else if (tid < 32)
        t = greedy_forward_warp(A, B, L, dt, word);
    if (FWD) __syncwarp();
    if (tid < 32) {
        if (tid == 0) g.makespan[i] = int64_t(t);
        for (int w = tid; w < W; w += 32) g.bits[i * W + w] = word[w];
    }
}

// Algorithm 1 by one warp, two rows per lane (rows past L hold the totals). mine: lane
// w's decision word w. Returns f_m.
template <typename T>
__device__ __forceinline__ T greedy_forward_rows(int kb, int D, int L, T dt, const T (&a)[1][2],
                                                 const T (&b)[1][2], T aL, uint32_t &mine)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int S = int(sizeof(T));
    const int lane = threadIdx.x & 31, r = 2 * lane + 1;
    auto A = [&](int m) { return sh<T>(kb + (m - 1) * S); };
    auto B = [&](int m) { return sh<T>(kb + D + (m - 1) * S); };
    // the first row x past `from` with A[x] >= thr (thr <= A[L])
    auto first = [&](T thr, int from) {
        const int below = __popc(__ballot_sync(kAll, a[0][0] < thr)) + __popc(__ballot_sync(kAll, a[0][1] < thr));
        return max(below, from) + 1;
    };
    auto mark = [&](int l) { mine |= lane == ((l - 1) >> 5) ? 1u << ((l - 1) & 31) : 0u; };
    const T lim = dt + aL;
    const int last = __popc(__ballot_sync(kAll, r < L && a[0][0] + b[0][0] <= lim)) +
                     __popc(__ballot_sync(kAll, r + 1 < L && a[0][1] + b[0][1] <= lim));
    int n = 1, m;
    if (last >= 1) {
        const T bl = B(last);
        n = 1 + __popc(__ballot_sync(kAll, b[0][0] < bl)) + __popc(__ballot_sync(kAll, b[0][1] < bl));
        m = first(A(n) + B(n) - dt, n);
    } else {
        m = first(aL, 1);
    }
    mark(n);
    T pull = dt + dt, Bm = B(m), Am = A(m), Bn = B(n);
    T end = dt + A(n) + Bn;
    end = max(end, pull + Am) + (Bm - Bn);
    for (int step = 2; m < L && step <= L; ++step) {  // m grows every time
        mark(m);
        const int x = first(min(Am + (Bm - Bn) - dt, aL), m);
        pull += dt;
        Bn = Bm;
        Am = A(x);
        Bm = B(x);
        end = max(end, pull + Am) + (Bm - Bn);
        m = x;
    }
    return end;
}

// Algorithm 2 by one warp (L <= 64): lane l runs the chains whose first push holds the
// last l + 1 and l + 33 layers, both at once. The best chain's breaks go to its lane's
// `breaks`; returns f_m and that lane.
template <typename T>
__device__ __forceinline__ T greedy_backward_rows(int kb, int D, int L, T dt, T aL,
                                                  uint64_t &breaks, int &owner)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int S = int(sizeof(T));
    const int lane = threadIdx.x & 31;
    const int end = kb + L * S;  // where row L + 1 would be
    // chain u stands at row p; q: byte of row p + 1
    int q[2];
    T A[2], B[2], next[2], link[2];
    uint64_t mask[2] = {0, 0};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int p = min(lane + 32 * u + 1, L);
        q[u] = kb + p * S;
        A[u] = sh<T>(q[u] - S);
        B[u] = sh<T>(q[u] + D - S);
        next[u] = sh<T>(q[u]);
        link[u] = A[u] + dt + B[u];
    }
    const int own0 = q[0], own1 = q[1];
    T sent = dt;
    // a chain advances by a row or more each step, so L steps end them all
    for (int step = 1; step < L && __any_sync(kAll, q[0] < end || q[1] < end); ++step) {
        T lim[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool on = q[u] < end;
            const int p = (q[u] - kb) / S;  // 1..L
            mask[u] |= on ? uint64_t(1) << (p - 1) : uint64_t(0);
            // the longest segment whose compute the link estimate covers, else one layer
            // and the zero-compute layers after it; a finished chain stays at L
            lim[u] = on ? max(A[u] + sent + B[u], next[u]) : aL;
        }
        int n0 = kb, n1 = kb;
        halve_from<T, 32, true>(lim[0], lim[1], n0, n1);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool on = q[u] < end;
            // the search counts to 63 rows, and past L where the limit is the padding's value
            q[u] = aL <= lim[u] ? end : (u == 0 ? n0 : n1);
            const T a = sh<T>(q[u] - S), b = sh<T>(q[u] + D - S);
            next[u] = sh<T>(q[u]);
            link[u] = on ? max(link[u], a) + dt + (b - B[u]) : link[u];
            A[u] = a;
            B[u] = b;
        }
        sent += dt;
    }
    // least f_m, the longest first push on ties; chains that began at L are none
    int64_t best = INT64_MAX;
    int from = 0;
    if (own0 < end) {
        best = int64_t(link[0]);
        from = own0;
        breaks = mask[0];
    }
    if (own1 < end && int64_t(link[1]) <= best) {
        best = int64_t(link[1]);
        from = own1;
        breaks = mask[1];
    }
    owner = lane;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const int64_t ob = __shfl_xor_sync(kAll, best, d);
        const int of = __shfl_xor_sync(kAll, from, d), oo = __shfl_xor_sync(kAll, owner, d);
        if (ob < best || (ob == best && of > from)) {
            best = ob;
            from = of;
            owner = oo;
        }
    }
    return T(best);
}

template <bool FWD>
__global__ void __launch_bounds__(256, 5) greedy_warp_kernel(GreedyArgs g)
{
    constexpr int D = 64 * 8 + 16;
    const int L = g.L, W = words_for(L), lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int kb = int(threadIdx.x >> 5) * chain_pair_bytes(64);
    for (int64_t i = int64_t(blockIdx.x) * nw + (threadIdx.x >> 5); i < g.batch; i += int64_t(gridDim.x) * nw) {
        const int64_t dt = __ldg(g.dt + i);
        with_warp_prefix<FWD, 1>(
            L, RowLoader<FWD>{g.comp + i * L, g.xfer + i * L, L, g.vec != 0}, dt,
            [&](const auto &a, const auto &b, auto aL, auto bL) {
                using T = decltype(aL);
                using P2 = Pair<T>;
                using Two = typename P2::type;
                constexpr int S = int(sizeof(T));
                const int r = 2 * lane + 1;
                sh<Two>(kb + 2 * lane * S) = P2::make(r <= L ? a[0][0] : P2::kMax, r < L ? a[0][1] : P2::kMax);
                sh<Two>(kb + D + 2 * lane * S) = P2::make(b[0][0], b[0][1]);
                __syncwarp();
                uint32_t mine = 0u;
                T t;
                if (FWD) {
                    t = greedy_forward_rows<T>(kb, D, L, T(dt), a, b, aL, mine);
                } else {
                    uint64_t breaks = 0;
                    int owner = 0;
                    t = greedy_backward_rows<T>(kb, D, L, T(dt), aL, breaks, owner);
                    breaks = __shfl_sync(0xffffffffu, breaks, owner);
                    mine = lane == 0 ? uint32_t(breaks) : uint32_t(breaks >> 32);
                }
                if (lane == 0) g.makespan[i] = int64_t(t);
                if (lane < W) g.bits[i * W + lane] = mine;
                __syncwarp();
                return true;
            },
            [&](int st) {
                if (lane == 0) g.makespan[i] = -int64_t(st);
                if (lane < W) g.bits[i * W + lane] = 0u;
                __syncwarp();
                return true;
            });
    }
}

template <bool FWD, int NJ>
__global__ void __launch_bounds__(kChainThreads, 1) greedy_cta_kernel(GreedyArgs g)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = g.L, W = words_for(L), tid = threadIdx.x, NT = blockDim.x;
    uint32_t *word = reinterpret_cast<uint32_t *>(smem + 2 * greedy_row_bytes(L));
    uint64_t *tot = reinterpret_cast<uint64_t *>(smem + 2 * greedy_row_bytes(L) + chain_word_bytes(L));
    uint32_t *orw = reinterpret_cast<uint32_t *>(tot + 2 * kChainPairs * (kChainThreads / 32));
    longlong2 *best_of = reinterpret_cast<longlong2 *>(orw + 32);
    for (int64_t i = blockIdx.x; i < g.batch; i += gridDim.x) {
        const int64_t dt = __ldg(g.dt + i);
        for (int w = tid; w < W; w += NT) word[w] = 0u;
        uint64_t a[NJ][2], b[NJ][2], aL, bL;
        const int st = cta_prefix<FWD, NJ>(
            tot, orw, L, RowLoader<FWD>{g.comp + i * L, g.xfer + i * L, L, g.vec != 0}, dt, a, b, aL, bL);
        if (st != DC_OK) {
            if (tid == 0) g.makespan[i] = -int64_t(st);
            for (int w = tid; w < W; w += NT) g.bits[i * W + w] = 0u;
        } else if (aL + bL + uint64_t(L + 1) * uint64_t(dt) < (uint64_t(1) << 31)) {
            greedy_solve<FWD, int32_t, NJ>(smem, word, best_of, i, g, int32_t(dt), a, b);
        } else {
            greedy_solve<FWD, int64_t, NJ>(smem, word, best_of, i, g, dt, a, b);
        }
        __syncthreads();  // shared memory is read
    }
}

template <bool FWD, int NJ>
cudaError_t launch_greedy_cta(const GreedyArgs &g, int nt, cudaStream_t stream)
{
    static DeviceCache attr;  // the kernel's shared-memory limit, raised once per device
    int done = 0;
    cudaError_t e = attr.get(done, [](int &v) {
        v = 1;
        return cudaFuncSetAttribute(greedy_cta_kernel<FWD, NJ>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    int(greedy_smem_bytes(DC_L_MAX)));
    });
    if (e != cudaSuccess) return e;
    const size_t smem = greedy_smem_bytes(g.L);
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, greedy_cta_kernel<FWD, NJ>, nt, smem);
    if (e != cudaSuccess) return e;
    // four waves of CTAs, each walking every grid-th instance: chains differ in length
    int64_t grid = int64_t(nb < 1 ? 1 : nb) * sm_count() * 4;
    if (grid > g.batch) grid = g.batch;
    greedy_cta_kernel<FWD, NJ><<<unsigned(grid), nt, smem, stream>>>(g);
    return cudaGetLastError();
}

// One instance per thread where a warp's lanes are better used on 32 instances than on
// one short row. Forward: up to L = 22 (100,000 x 20: 38 us against 44 per warp; but 100,000
// x 24 38 against 32, x 32 61 against 32), at odd L, whose rows start all over a line, up to
// 25 on large batches (100,000 x 23 30.5 against 32.4, 200,000 x 25 58.0 against 58.8, but
// 60,000 x 25 25 against 22, 200,000 x 27 65 against 60), and above the warp kernel's rows up
// to 128 on large batches (100,000 x 100: 139 against 152 per CTA; but 10,000 x 100: 50
// against 39). Backward, quadratic in L per thread: up to L = 8, and up to 12 on large
// batches (500,000 x 12: 208 us against 284; 100,000 x 12 76 against 73). The warp kernel is
// slower on values past 32 bits, which the host cannot see: 200,000 x 28 forward 90 us, 70
// per thread (60 in 32 bits); 200,000 x 13 backward 159, 120 (117 in 32 bits).
template <bool FWD>
bool per_thread(int64_t batch, int L)
{
    if (FWD)
        return L <= 22 || (L <= 25 && L % 2 == 1 && batch >= 100000) ||
               (L > 64 && L <= 128 && batch >= 50000);
    return L <= 8 || (L <= 12 && batch >= 50000);
}

template <bool FWD>
cudaError_t launch_greedy(int64_t batch, int L, const int64_t *comp, const int64_t *xfer,
                          const int64_t *dt, int64_t *makespan, uint32_t *bits, cudaStream_t stream)
{
    if (per_thread<FWD>(batch, L)) {
        greedy_kernel<FWD><<<unsigned((batch + 127) / 128), 128, 0, stream>>>(batch, L, comp, xfer, dt,
                                                                             makespan, bits);
        return cudaGetLastError();
    }
    const bool vec = (L % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(comp) | reinterpret_cast<uintptr_t>(xfer)) & 15u) == 0;
    const GreedyArgs g{batch, L, comp, xfer, dt, makespan, bits, vec ? 1 : 0};
    if (L <= 64) {
        // one-warp CTAs until they fill the GPU, then four warps to a CTA in four waves
        const int nw = batch < int64_t(sm_count()) * 32 ? 1 : 4;
        int64_t grid = (batch + nw - 1) / nw;
        if (nw > 1 && grid > int64_t(sm_count()) * 10 * 4) grid = int64_t(sm_count()) * 10 * 4;
        greedy_warp_kernel<FWD><<<unsigned(grid), 32 * nw, nw * chain_pair_bytes(64), stream>>>(g);
        return cudaGetLastError();
    }
    const int nt = 32 * ((L + 63) / 64);
    return nt <= kChainThreads ? launch_greedy_cta<FWD, 1>(g, nt, stream)
                               : launch_greedy_cta<FWD, 2>(g, 32 * ((L + 127) / 128), stream);
}

}  // namespace
}  // namespace dc

extern "C" dc_status dc_greedy_forward_batch(int64_t batch, int32_t L, const int64_t *fc,
                                             const int64_t *pt, const int64_t *dt,
                                             int64_t *makespan, uint32_t *bits,
                                             cudaStream_t stream)
{
    const dc::NvtxRange nvtx("dc_greedy_forward_batch");
    if (batch < 0 || L < 1 || L > DC_L_MAX || batch > int64_t(0xffffffffll)) return DC_ERR_BAD_SHAPE;
    if (batch == 0) return DC_OK;
    if (!fc || !pt || !dt || !makespan || (!bits && dc::words_for(L) > 0)) return DC_ERR_NULL;
    return dc::launch_greedy<true>(batch, L, fc, pt, dt, makespan, bits, stream) == cudaSuccess
               ? DC_OK
               : DC_ERR_CUDA;
}

extern "C" dc_status dc_greedy_backward_batch(int64_t batch, int32_t L, const int64_t *bc,
                                              const int64_t *gt, const int64_t *dt,
                                              int64_t *makespan, uint32_t *bits,
                                              cudaStream_t stream)
{
    const dc::NvtxRange nvtx("dc_greedy_backward_batch");
    if (batch < 0 || L < 1 || L > DC_L_MAX || batch > int64_t(0xffffffffll)) return DC_ERR_BAD_SHAPE;
    if (batch == 0) return DC_OK;
    if (!bc || !gt || !dt || !makespan || (!bits && dc::words_for(L) > 0)) return DC_ERR_NULL;
    return dc::launch_greedy<false>(batch, L, bc, gt, dt, makespan, bits, stream) == cudaSuccess
               ? DC_OK
               : DC_ERR_CUDA;
}
