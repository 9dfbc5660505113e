// Device building blocks of the short-L (1 <= L <= 16) DP, shared by the dense
// and list passes (dp_small.cu) and the fused generate-and-solve passes
// (dp_fused.cu). The design notes are at the top of dp_small.cu.
#pragma once

#include "chain.cuh"
#include "gen_device.cuh"

namespace dc {

int sm_count();  // SMs of the current device (dp_small.cu)

namespace {


#ifndef DC_KEEP_COLS
#define DC_KEEP_COLS 4
#endif
#ifndef DC_SMALL_MINB
#define DC_SMALL_MINB 16  // resident single-warp CTAs per SM the registers must allow
#endif
// From this L on the dense and fused passes take their tiles from an atomic
// ticket; shorter rows take every grid-th tile, for which one atomic per tile costs
// more than the balance gains.
constexpr int kSplitMinL = 12;
// Whether the dense pass stages a tile beside its table, where the next one lands while
// this one is solved, or in the table's place: from kSplitMinL on, where a long solve
// hides the copies, and up to L = 6, where both are small enough for as many warps as the
// registers allow (1,000,000 instances per direction: L = 4 21.2 us against 23.5, 6 28.1
// against 30.8; but 7 39.7 against 36.0 and 8 37.7 against 33.9, with fewer warps).
__host__ __device__ constexpr bool staged_beside(int L) { return L <= 6 || L >= kSplitMinL; }
constexpr int kKeepCols = DC_KEEP_COLS;  // the 32-bit pass stores columns 2..kKeepCols

// index of stored cell (m, n), 2 <= n <= L-1, n <= m <= L
__host__ __device__ constexpr int cell2(int L, int m, int n)
{
    return (n - 2) * L - (n - 2) * (n - 1) / 2 + (m - n);
}

// Row stride of the staging buffer in int64 units. Odd L: the odd stride L, so
// that the 16 lanes of a half-warp reading 64-bit words of their own rows hit 16
// distinct bank pairs. Even L: rows are copied and read as 16-byte pairs, so the
// stride is even (16-byte aligned rows) and 2 mod 4, so that the 8 lanes of a
// quarter-warp reading 16 bytes of their own rows hit 8 distinct 4-bank groups.
__host__ __device__ constexpr int stage_stride(int L)
{
    return (L % 2 == 1) ? L : (L % 4 == 2 ? L : L + 2);
}

// A warp's table, per lane (values of type T, lane-interleaved): value 0 unused, the kept
// cells of columns 2..kLast at 1 + cell2 (a traceback step loads one value below a
// column's first cell, which stays inside the table), then U[0..L]; column 1 is not
// stored, being U shifted by a constant. KEEP: the last column kept, if there are as many.
template <int L, typename T, int KEEP>
struct Table {
    static constexpr int kLast = KEEP < L - 1 ? KEEP : L - 1;  // last stored column
    static constexpr int kCells = kLast >= 2 ? cell2(L, L, kLast) + 1 : 0;
    static constexpr int kOffU = 1 + kCells;
    static constexpr int kWords = kOffU + L + 1;
    static constexpr int kBytes = 32 * kWords * int(sizeof(T));
};

// Shared memory of a warp of the 32-bit pass: its table, and the tile's staging (comp and
// xfer rows at a padded stride, then dt), which either shares the table's area
// (kSharedBytes) or lies beside it (kSplitBytes), so that the next tile can land while
// this one is solved.
template <int L>
struct Tab32 : Table<L, int32_t, kKeepCols> {
    using Table<L, int32_t, kKeepCols>::kBytes;
    static constexpr int kStride = stage_stride(L);               // staging row stride (int64)
    static constexpr int kRowsBytes = 2 * 32 * kStride * 8;        // comp + xfer rows of a tile
    static constexpr int kSharedBytes = kRowsBytes > kBytes ? kRowsBytes : kBytes;
    static constexpr int kSplitBytes = kBytes + kRowsBytes + 32 * 8;  // table | rows | dt
};

template <typename T>
__device__ __forceinline__ T lds(const T *lane_base, int v) { return lane_base[32 * v]; }

// ---------------------------------------------------------------------------
// The 32-bit pass in shifted form. Every value is taken relative to the time
// the last pull (forward) or push (backward) of its cell can start, which turns
// a transition into one add-then-max and the minimum into 3-input mins: on
// GB300 both are single integer-ALU instructions (the DPX forms), so a transition
// costs 1.5 ALU-pipe instructions instead of 2.
//
// forward (P = transfer prefix, FC = compute prefix, G[k] = FC[L] - FC[k],
// Q[m] = dt + P[m]): with B = X - n*dt - P[m] + G[m] (X as above) and
// A[k] = B[k][n-1] + P[k],
//   B[m][n] + Q[m] = min_k max(G[k] + Q[m], A[k]),  A[m][1] = FC[L] + P[m],
//   X[L][n] = B[L][n] + n*dt + P[L];
// the next column's A[m] is that minimum less dt;
// backward (BC = compute prefix, NGT[k] = -(transfer prefix), U = BC - dt):
// with F = X - dt - S[m],
//   F[m][n] - dt = min_k max(U[m] + NGT[k], F[k][n-1]),  F[m][1] = BC[m],
//   X[L][n] = F[L][n] + dt + S[L];
// the next column's F[m] is that minimum plus dt.
// Both are min_k max(U[m] + V[k], C[k]) with a row constant U, the same in every
// column, and the previous column C in the max operand. Each candidate differs from Eq. 8/9's by a
// constant of its row, so every argmin is the same. All values and sums lie in
// [-2^31, 2^31) when the capped bound L*dt + sum(comp) + sum(capped xfer) is
// below 2^31; other instances take the work-list pass, which has the same form in 64
// bits (T). The table stores A (forward)
// or F (backward) for columns 1..kKeepCols and the row U (Q forward, BC - dt
// backward); V (G forward, NGT backward) stays in registers.

__device__ __forceinline__ int32_t add_max(int32_t a, int32_t b, int32_t c) { return __viaddmax_s32(a, b, c); }
__device__ __forceinline__ int64_t add_max(int64_t a, int64_t b, int64_t c) { return dmax(a + b, c); }
__device__ __forceinline__ int32_t add_min(int32_t a, int32_t b, int32_t c) { return __viaddmin_s32(a, b, c); }
__device__ __forceinline__ int64_t add_min(int64_t a, int64_t b, int64_t c) { return dmin(a + b, c); }
__device__ __forceinline__ int32_t min3(int32_t a, int32_t b, int32_t c) { return __vimin3_s32(a, b, c); }
__device__ __forceinline__ int64_t min3(int64_t a, int64_t b, int64_t c) { return dmin(dmin(a, b), c); }
template <typename T>
constexpr T kLeast = sizeof(T) == 4 ? T(INT32_MIN) : T(INT64_MIN);

// Minimum of c[0..cnt-1] (cnt a compile-time constant after unrolling): two
// chains of 3-input mins, so that each row has two independent dependency chains
// and the rows of a column interleave.
template <int N, typename T>
__device__ __forceinline__ T min_fold3(const T (&c)[N], int cnt)
{
    if (cnt == 1) return c[0];
    if (cnt == 2) return dmin(c[0], c[1]);
    T a = c[0], b = c[1];
    int j = 2;
#pragma unroll
    for (; j + 3 < cnt; j += 4) {
        a = min3(a, c[j], c[j + 1]);
        b = min3(b, c[j + 2], c[j + 3]);
    }
    if (j + 1 < cnt) return min3(min3(a, b, c[j]), c[j + 1], cnt > j + 2 ? c[j + 2] : c[j + 1]);
    if (j < cnt) return min3(a, b, c[j]);
    return dmin(a, b);
}

// The fill also keeps a cell's value of the column before when that is lower (fewer
// segments than n), which makes a column non-decreasing in m and changes neither the
// optimum, nor its segment count, nor any cell that the traceback visits (the argument
// is in chain.cuh). In return the columns end early: column n+1 can lower the optimum
// only through a cell that column n lowered below the optimum's own bound, and only if
// the last segment's bound U[L] + V[L-1] allows it. The warp stops after the first
// column in which no lane has such a cell: 4.0-4.1 columns of 16 on the VGG-16 batch
// (3.2 of 8 on AlexNet), where the deepest optimum of a warp has 4.0 segments. One
// direction of 1,000,000 VGG-16 instances: 62 us, 90 with all columns filled.
//
// The direction `fwd` is an argument: the dense passes pass a compile-time
// constant, which folds every choice below away; the fused pass solves both
// directions with one copy of this code. Every lane of the warp calls it; `run` is
// false for lanes without a 32-bit instance, whose values are not used.
template <int L, int KEEP, typename T>
__device__ __forceinline__ void fill_e(const bool fwd, const bool run, const T (&U)[L + 1],
                                       const T (&V)[L + 1], T dt, T fcL, T *lw, T &bestV, int &best_s)
{
    using K = Table<L, T, KEEP>;
    // forward: U = Q, V = G, col = A; backward: U = BC - dt, V = NGT, col = F
    const T dt2 = 2 * dt;
    const T c1 = fwd ? fcL - dt : dt;  // column 1 is U + c1
    const T sdt = fwd ? -dt : dt;      // column n is its minimum + sdt
    const T sold = fwd ? -dt : 0;      // column n - 1 in column n's terms, less column n - 1
    const T slim = fwd ? 0 : -dt;      // a cell of column n helps only below col[L] + slim
    const T uL = fwd ? U[L] : 0;       // row L's minimum less uL: B[L][n] or F[L][n] - dt
    const T step = fwd ? dt : 0, base = fwd ? 0 : dt2;
    const T tail = L > 1 ? U[L] + V[L - 1] : 0;  // no later minimum of row L is below it
    T col[L + 1];
#pragma unroll
    for (int m = 1; m <= L; ++m) col[m] = U[m] + c1;
    bestV = fwd ? fcL + dt : U[L] + dt2;
    best_s = 1;
#pragma unroll
    for (int n = 2; n <= L; ++n) {
        T lim = 0;
        bool more = false;
#pragma unroll
        for (int m = L; m >= n; --m) {  // descending: column n overwrites column n-1 in place
            const int cnt = m - n + 1;  // k = n-1 .. m-1
            const T u = U[m];
            T c[L];
#pragma unroll
            for (int j = 0; j < cnt; ++j) c[j] = add_max(u, V[n - 1 + j], col[n - 1 + j]);
            const T b = min_fold3<L>(c, cnt);
            const T old = col[m] + sold;
            col[m] = add_min(b, sdt, old);
            if (m == L) {
                if (col[m] < old) {  // strict: the lowest n wins ties
                    bestV = b - uL + n * step + base;  // X[L][n] - P[L] or X[L][n] - S[L]
                    best_s = n;
                }
                lim = col[m] + slim;
            } else {
                more |= col[m] < dmin(old, lim);
            }
            if (n <= K::kLast) lw[32 * (1 + cell2(L, m, n))] = col[m];
        }
        if (n < L && !__any_sync(0xffffffffu, run && more && tail < lim)) break;
    }
}

// Number of v[0..N-1] (non-increasing) above t: N a power of two, halved by selects.
// next: the first value that is not above, if any.
template <int N, typename T>
__device__ __forceinline__ int count_above(const T (&v)[N], T t, T &next)
{
    if constexpr (N == 1) {
        if (v[0] <= t) next = v[0];
        return v[0] > t ? 1 : 0;
    } else {
        constexpr int H = N / 2;
        const bool up = v[H - 1] > t;  // the first half lies above t
        T w[H];
#pragma unroll
        for (int j = 0; j < H; ++j) w[j] = up ? v[H + j] : v[j];
        if (!up) next = v[H - 1];
        return (up ? H : 0) + count_above<H>(w, t, next);
    }
}

__host__ __device__ constexpr int ceil_log2(int x) { return x <= 1 ? 0 : 1 + ceil_log2((x + 1) / 2); }

// The fill, the traceback and the outputs of one instance per lane in shifted form,
// from its U and V rows (forward: U = dt + capped transfer prefix, V = FC[L] - compute
// prefix; backward: U = compute prefix - dt, V = -capped transfer prefix) and the raw
// transfer sum. Every lane of the warp calls it; lanes with `run` false write nothing
// but their slice. REPLAY: o.replay takes f_m of the decision. Returns false (having
// written nothing) when the traceback needs a column the pass did not keep.
template <int L, bool REPLAY, int KEEP, typename T>
__device__ __forceinline__ bool solve_uv(const bool fwd, const bool run, const T (&U)[L + 1],
                                         const T (&V)[L + 1], T dt, uint64_t xraw, T *lw, int64_t i,
                                         const SolveOut &o)
{
    using K = Table<L, T, KEEP>;
    constexpr int W = (L - 1 + 31) / 32;
    const T fcL = V[0];  // forward: FC[L]
#pragma unroll
    for (int m = 0; m <= L; ++m) lw[32 * (K::kOffU + m)] = U[m];  // the traceback reads U[m]
    T bestV;
    int s;
    fill_e<L, KEEP>(fwd, run, U, V, dt, fcL, lw, bestV, s);
    if (!run) return true;
    if (s - 1 > K::kLast && s - 1 >= 2) return false;

    // from (L, s) step to the lowest k that attains the cell, set p_k / g_k, continue
    // at (k, n-1). That k is the first with U[m] + V[k] <= the cell (chain.cuh), found
    // by a binary search over V in registers.
    constexpr int kPad = 1 << ceil_log2(L > 2 ? L - 1 : 1);
    T vs[kPad];
#pragma unroll
    for (int j = 0; j < kPad; ++j) vs[j] = j + 1 < L ? V[j + 1] : kLeast<T>;
    uint32_t word = 0;
    int err = 0;
    int m = L, n = s;
    T target = fwd ? bestV - s * dt + U[L] : bestV - 2 * dt;  // B[L][s] + Q[L] or F[L][s] - dt
    const T off1 = fwd ? fcL - dt : dt;  // column 1 is U + off1 (not stored)
    // f_m of the decision from its own segments, in the cells' shifted terms: the
    // largest over its segments of U[end] + V[start] and the shift since, then the
    // first segment's U
    T span = kLeast<T>, later = 0;
    while (n > 1) {
        const int nm1 = n - 1;
        const T u = lds(lw, K::kOffU + m);
        T vk = kLeast<T>;
        const int k = 1 + count_above<kPad>(vs, target - u, vk);
        // cell (k, n-1) of a kept column is word base + k
        const int base = nm1 == 1 ? K::kOffU : 1 + cell2(L, 0, nm1);
        const int at = k < m ? k : m;  // inside the column
        const T fk = lds(lw, base + at) + (nm1 == 1 ? off1 : 0);
        if (k < nm1 || k >= m || fk > target) {  // cannot happen: the fill took this minimum
            err = 1;
            break;
        }
        word |= 1u << ((k - 1) & 31);
        if constexpr (REPLAY) {
            span = dmax(span, u + vk + later);
            later += fwd ? -dt : dt;
        }
        target = fwd ? fk + dt : fk - dt;  // the cell (k, n-1): B + Q[k] = A + dt, or F - dt
        m = k;
        n = nm1;
    }
    auto absolute = [&](T v) {  // both are at least 0
        return int64_t((sizeof(T) == 4 ? uint64_t(uint32_t(v)) : uint64_t(v)) + xraw);
    };
    o.makespan[i] = absolute(bestV);
    if (o.nseg) o.nseg[i] = s;
    if (o.status) o.status[i] = err ? DC_ERR_INTERNAL : DC_OK;
    if constexpr (REPLAY) {
        T f = bestV;  // s = 1: the one segment, dt + FC[L] or dt + BC[L]
        if (s > 1) {
            span = dmax(span, lds(lw, K::kOffU + m) + off1 + later - (fwd ? -dt : dt));
            f = fwd ? span - U[L] + s * dt : span + 2 * dt;
        }
        if (sizeof(T) == 4 || o.replay) o.replay[i] = err ? -int64_t(DC_ERR_INTERNAL) : absolute(f);
    }
    if (W > 0) o.bits[i * W] = word;
    return true;
}

// U and V from 64-bit prefix sums (the caller has checked T's range).
template <int L, bool FWD, typename T>
__device__ __forceinline__ void shifted_uv(const uint64_t (&Pc)[L + 1], const uint64_t (&Px)[L + 1],
                                           int64_t dti, T (&U)[L + 1], T (&V)[L + 1])
{
    const T dt = T(dti);
    const T fcL = T(Pc[L]);
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        U[m] = FWD ? dt + T(Px[m]) : T(Pc[m]) - dt;
        V[m] = FWD ? fcL - T(Pc[m]) : -T(Px[m]);
    }
}

// The row's U and V in 32-bit arithmetic, for the common row whose costs all lie
// in [0, 2^32) with every compute cost below 2^31 / L (then every compute sum is
// exact in 32 bits) and dt below 2^31. rc, rx: the row's costs in layer order.
// Returns false, computing nothing, for any other row: the caller takes the
// 64-bit route (which also classifies negative and out-of-range input). On true,
// `wide` says whether the capped bound L*dt + sum(comp) + sum(capped xfer) exceeds
// the shifted form's limit. Transfers are capped at the total compute as in
// row_prefix; the sums of capped transfers and raw transfers are kept in 64 bits.
template <int L, bool FWD>
__device__ __forceinline__ bool fast_uv(const int64_t *rc, const int64_t *rx, int64_t dti,
                                        int32_t (&U)[L + 1], int32_t (&V)[L + 1], uint64_t &xraw,
                                        bool &wide)
{
    constexpr int kCompBits = 31 - ceil_log2(L);
    uint32_t cl[L], xl[L];
    uint32_t hor = uint32_t(uint64_t(dti) >> 31), cor = 0u, tc = 0u;
    if constexpr (L % 2 == 0) {  // 16-byte rows: two costs per load
#pragma unroll
        for (int q = 0; q < L; q += 2) {
            const uint4 c = *reinterpret_cast<const uint4 *>(rc + q);
            const uint4 x = *reinterpret_cast<const uint4 *>(rx + q);
            const int r0 = FWD ? q : L - 1 - q, r1 = FWD ? q + 1 : L - 2 - q;
            cl[r0] = c.x;
            cl[r1] = c.z;
            xl[r0] = x.x;
            xl[r1] = x.z;
            hor |= c.y | x.y;
            hor |= c.w | x.w;
            cor |= c.x | c.z;
            tc += c.x + c.z;
        }
    } else {
#pragma unroll
        for (int r = 0; r < L; ++r) {
            const int col = FWD ? r : L - 1 - r;
            const uint2 c = *reinterpret_cast<const uint2 *>(rc + col);
            const uint2 x = *reinterpret_cast<const uint2 *>(rx + col);
            cl[r] = c.x;
            xl[r] = x.x;
            hor |= c.y | x.y;
            cor |= c.x;
            tc += c.x;
        }
    }
    if ((hor | (cor >> kCompBits)) != 0u) return false;
    uint32_t u = FWD ? uint32_t(dti) : 0u - uint32_t(dti), v = FWD ? tc : 0u;
    U[0] = int32_t(u);
    V[0] = int32_t(v);
    uint64_t px = 0, xr = 0;
#pragma unroll
    for (int r = 0; r < L; ++r) {
        const uint32_t xc = min(xl[r], tc);
        px += xc;
        xr += xl[r];
        if (FWD) {
            u += xc;
            v -= cl[r];
        } else {
            u += cl[r];
            v -= xc;
        }
        U[r + 1] = int32_t(u);
        V[r + 1] = int32_t(v);
    }
    xraw = xr;
    wide = uint64_t(L) * uint64_t(dti) + tc + px > uint64_t(kShiftedLimit);
    return true;
}

__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gmem_src)
{
    const uint32_t d = uint32_t(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    const uint32_t d = uint32_t(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Issue the copies of tile `base` (rows base..base+rows-1) into the staging area:
// 16-byte copies of cost pairs when L is even and both cost arrays are 16-byte
// aligned (`pairs`; every pair then starts on a 16-byte boundary on both sides),
// else 8-byte copies.
template <int L>
__device__ __forceinline__ void stage_tile(int64_t *stC, int64_t *stX, const int64_t *comp,
                                           const int64_t *xfer, int64_t base, int rows, int lane,
                                           bool pairs)
{
    constexpr int kStride = stage_stride(L);
    const int64_t *gC = comp + base * L;
    const int64_t *gX = xfer + base * L;
    if (L % 2 == 0 && pairs) {
        constexpr int H = L / 2 > 0 ? L / 2 : 1;  // pairs per row
        const int np = rows * H;
        for (int p = lane; p < np; p += 32) {
            const int r = p / H, cidx = 2 * (p - r * H);
            cp_async16(stC + r * kStride + cidx, gC + 2 * p);
            cp_async16(stX + r * kStride + cidx, gX + 2 * p);
        }
    } else {
        const int nel = rows * L;
        for (int e = lane; e < nel; e += 32) {
            const int r = e / L, cidx = e - r * L;
            cp_async8(stC + r * kStride + cidx, gC + e);
            cp_async8(stX + r * kStride + cidx, gX + e);
        }
    }
    cp_async_commit();
}

// Read this lane's row (processing order) into 64-bit prefix sums; flag bad
// input. Transfer costs are capped at the row's total compute: shifted by
// n*dt + (transfer prefix), every DP value lies in [0, total compute] and the
// recurrence sees transfer costs only through saturating differences, so the cap
// changes no comparison (same decision) and lowers the makespan by exactly
// sum(xfer) - sum(capped xfer), returned in `shift`.
template <int L, bool FWD, typename Src>
__device__ __forceinline__ void row_prefix(Src get, uint64_t (&Pc)[L + 1], uint64_t (&Px)[L + 1],
                                           uint64_t &xraw, bool &neg, bool &big)
{
    uint64_t tc = 0;
    xraw = 0;
#pragma unroll
    for (int r = 1; r <= L; ++r) {
        int64_t cv, xv;
        get(FWD ? r - 1 : L - r, cv, xv);
        neg |= (cv < 0) | (xv < 0);
        big |= ((cv | xv) >> 52) != 0;
        tc += uint64_t(cv);
        xraw += uint64_t(xv);
    }
    Pc[0] = 0;
    Px[0] = 0;
#pragma unroll
    for (int r = 1; r <= L; ++r) {
        int64_t cv, xv;
        get(FWD ? r - 1 : L - r, cv, xv);
        Pc[r] = Pc[r - 1] + uint64_t(cv);
        Px[r] = Px[r - 1] + (uint64_t(xv) < tc ? uint64_t(xv) : tc);
    }
}

// A staged row (rc, rx: its costs in layer order) to the 32-bit pass's U and V:
// fast_uv when the row fits, else 64-bit prefix sums with the input checks.
// st: DC_OK or the row's error; wide: the capped bound exceeds the shifted form's
// limit (the instance belongs to the 64-bit pass).
template <int L, bool FWD>
__device__ __forceinline__ void row_uv(const int64_t *rc, const int64_t *rx, int64_t dti,
                                       int32_t (&U)[L + 1], int32_t (&V)[L + 1], uint64_t &xraw,
                                       bool &wide, int &st)
{
    st = DC_OK;
    if (fast_uv<L, FWD>(rc, rx, dti, U, V, xraw, wide)) return;
    uint64_t Pc[L + 1], Px[L + 1];
    bool neg = dti < 0, big = (dti >> 52) != 0;
    row_prefix<L, FWD>(
        [&](int col, int64_t &cv, int64_t &xv) {
            cv = rc[col];
            xv = rx[col];
        },
        Pc, Px, xraw, neg, big);
    if (neg)
        st = DC_ERR_NEGATIVE;
    else if (big || uint64_t(L) * uint64_t(dti) + Pc[L] + xraw >= uint64_t(kRangeLimit))
        st = DC_ERR_RANGE;
    wide = uint64_t(L) * uint64_t(dti) + Pc[L] + Px[L] > kShiftedLimit;  // capped bound
    shifted_uv<L, FWD>(Pc, Px, dti, U, V);
}

// ---------------------------------------------------------------------------
// The pass over a first pass's list, every value in 64 bits and every column kept:
// instances with values past the shifted form's range or optima deeper than kKeepCols.
// A short list takes a warp per instance (chain.cuh), whose lanes share the work: it ends
// soonest. A longer one takes a lane per instance with the fill above, several times
// faster on a full GPU, up to the depth at which the unrolled 64-bit fill no longer fits
// the instruction cache; beyond it warps at a higher occupancy. DRAWN: the rows are drawn
// again, one layer after the other in the lane form.
// Measured, one direction of 1,000,000 log-uniform instances that all lie past 2^31, one
// warp per instance on 4 warps per SM (alone) / an unrolled fill of every column, a lane
// per instance / these rules: L = 4 3,430 us / 159 / 136, L = 8 5,150 / 424 / 340, L = 12
// 4,040 / 689 / 437, L = 15 4,150 / 1,001 / 986, L = 16 3,700 / 1,220 / 870-960; generated
// and solved at L = 12 with costs in nanoseconds, both directions, 3,270 / 2,434 / 690.
// Where the lines lie, 400,000 instances of which a part is listed, by warp against by lane:
// 608 of L = 12 25 us against 26, of L = 8 17 against 17-23; 1,500 27 against 27 and 20
// against 18-23; 3,000 30 against 28 and 22 against 19-24; of L = 6 14.2 against 13.6, 16.8
// against 13.6 and 19 against 14.3; at L = 2 and 4 never faster.
// All of L = 16: lanes 1,300 us, warps 870. All of L = 15: 990 against 900-1,050, but 580
// against 880-1,030 at L = 14. Drawn lists, 1,000,000 plain log-uniform instances (some
// thousand listed): L = 12 210 us by warp and 218 by lane, L = 15 261 and 277.
// Four single-warp CTAs per SM hold up the short calls least (L = 8, nothing listed: 15.2
// us against 16.4 with sixteen).
template <int L, bool DRAWN>
struct List64 {
    static constexpr bool kLanes = L <= (DRAWN ? 12 : 15);  // whether a list may take a lane per instance
    // lists up to here go by warp
    static constexpr int kByWarp = L <= 4 ? 0 : DRAWN ? 4864 : L <= 6 ? 1200 : 2432;
    static constexpr int kWarps = kLanes ? 1 : 4;               // warps per CTA
    static constexpr int kCtas = !kLanes ? 8 : DRAWN ? 16 : 4;  // CTAs per SM, at most
    static constexpr int kChainBytes = (chain_pair_bytes(64) + int(tri_cells(L)) * 8 + 15) / 16 * 16;
    static constexpr int kLaneBytes = kLanes ? Table<L, int64_t, L>::kBytes : 0;
    static constexpr int kSlice = kLaneBytes > kChainBytes ? kLaneBytes : kChainBytes;  // a warp's
    static constexpr int kBytes = kWarps * kSlice;
};

// Walks a list: by_warp(kb, i, kept) solves instance i with the warp, kb: byte of the warp's
// slice of shared memory; by_lane(active, i), called by every lane of the warp, an instance
// per lane where `active`.
template <int L, bool DRAWN, typename ByWarp, typename ByLane>
__device__ __forceinline__ void list_pass(int64_t batch, int64_t count, const uint32_t *list,
                                          ByWarp by_warp, ByLane by_lane)
{
    using K = List64<L, DRAWN>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kb = warp * K::kSlice;
    if (K::kByWarp > 0 && (!K::kLanes || count <= K::kByWarp)) {
        if (lane == 0) zero_row(kb, 64);
        const KeptValues kept{&sh<int64_t>(kb + chain_pair_bytes(64)), L};
        for (int64_t j = int64_t(blockIdx.x) * K::kWarps + warp; j < count;
             j += int64_t(gridDim.x) * K::kWarps) {
            const int64_t i = int64_t(list[j]);
            if (!DC_CHECK(i < batch)) continue;
            by_warp(kb, i, kept);
            __syncwarp();  // shared memory is read
        }
        return;
    }
    if constexpr (K::kLanes) {
        for (int64_t j0 = int64_t(blockIdx.x) * 32; j0 < count; j0 += int64_t(gridDim.x) * 32) {
            const bool listed = j0 + lane < count;
            const int64_t i = listed ? int64_t(list[j0 + lane]) : 0;
            by_lane(listed && DC_CHECK(i < batch), i);
        }
    }
}

// Host: launches a list kernel. The list's length is known on the device only; its CTAs
// are launched early and the surplus exits at once.
template <int L, bool DRAWN, typename... Params, typename... Args>
cudaError_t launch_list(DeviceCache &resident, int64_t batch, cudaStream_t stream,
                        void (*kernel)(Params...), const Args &...args)
{
    using K = List64<L, DRAWN>;
    int n = 0;
    const cudaError_t e = resident.get(n, [&](int &v) {
        const cudaError_t q =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, 32 * K::kWarps, K::kBytes);
        if (v > K::kCtas) v = K::kCtas;
        return q;
    });
    if (e != cudaSuccess) return e;
    const int64_t most = int64_t(sm_count()) * n, need = (batch + K::kWarps - 1) / K::kWarps;
    return launch_early(kernel, need < most ? need : most, 32 * K::kWarps, K::kBytes, stream, args...);
}

// One instance per lane: rows(col, comp, xfer) gives the costs of the lane's instance i, of
// latency dti, in layer order. Every lane of the warp calls it.
template <int L, bool FWD, typename Rows>
__device__ __forceinline__ void list_solve_lane(bool active, int64_t i, int64_t dti, Rows rows,
                                                const SolveOut &o)
{
    uint64_t Pc[L + 1] = {}, Px[L + 1] = {}, xraw = 0;
    bool neg = false, big = false;  // checked by the first pass
    if (active) row_prefix<L, FWD>(rows, Pc, Px, xraw, neg, big);
    int64_t U[L + 1], V[L + 1];
    shifted_uv<L, FWD>(Pc, Px, dti, U, V);
    solve_uv<L, true, L>(FWD, active, U, V, dti, xraw, &sh<int64_t>(8 * int(threadIdx.x)), i, o);
}

}  // namespace
}  // namespace dc
