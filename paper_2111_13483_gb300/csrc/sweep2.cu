// Two-level triangular sweeps (Eqs. 23, 24): the default for the Schur and null-field forms.
//
// A sweep is a chain: block row o needs its neighbour's result, and on GB300 each hand-over from
// one CTA to the next costs about 1.3 us of L2 round trips on top of the block product.  With one
// row per hand-over (the kinds of ops.cu) the chain of the 30,720-unknown sphere's 1,106 rows took
// 5.2 ms at 64 columns and 3.3 ms at one.  Here S2_K consecutive block rows form a
// super-row.  With L_SS the unit triangle of super-row S and L_SS^{-1} = I + N_S (N_S formed once
// per setup, k_s2_inverse), the sweep is
//   z_o = x_o - sum over the dependencies outside S,     o in S   (phase A)
//   y_o = z_o + sum over the members i of S before o of N_oi z_i  (phase B)
// so all rows of a super-row run side by side and the chain has two hand-overs per S2_K rows.  The
// backward sweep uses N_S^T (a second copy, so that both directions read rows contiguously).
//
// One CTA per block row and column group (S2_NW warps), rows taken from a ticket counter in sweep
// order.  Dependency t of the row belongs to warp t mod S2_NW, which walks its dependencies alone:
// coefficients through a ring of its own that cp.async fills with whole blocks or large pieces (staging
// them by element, eight columns at a time, cost 1.5 x), vector blocks one dependency ahead in
// registers, no CTA barrier until the warps' partial sums are added in warp order.  A row's
// newest dependencies (the previous super-row) fall on different warps.
//
// Hand-over: y and z of a sweep live in row-major buffers that start as all-ones words; a
// consumer reads a word until it is no longer all ones (a result that is that NaN pattern is
// stored as another NaN), so neither flags nor fences are needed, and a row that is never
// published ends every wait on it at the handle's bound.  A word has 64 bits and is an element of
// that size in the load and in the store (wait.cuh), so a half of it is never taken for a result.
//
// What binds it now: at one column the chain (69 super-rows of the 30,720-unknown sphere, 8.6 us each); at 64
// columns the instructions (two CTAs of eight warps per SM issue every other cycle, a fifth of them FMAs: blocks
// of 28 x 28 and rank-5 factors are short against their staging).  Measured on that sphere, per sweep, forward
// / backward: 64 columns 5.19 / 4.74 -> 2.88 / 2.37 ms, 16 columns 1.25 / 1.03 ms, one column 3.32 / 3.3 -> 0.60
// / 0.59 ms; FP64, one column, 7,680 unknowns: 3.65 / 3.59 -> 0.74 / 0.75 ms.  Super-rows of 8 took 0.77 ms at one
// column and 3.24 / 2.51 at 64, of 32 0.49 and 2.95 / 3.33 (N_S grows with the super-row, and so does the setup).
//
// Every output adds its terms in an order that depends on the plan alone (dependency, warp, piece),
// never on the columns of the launch or on the group width: a column's result is bitwise the same
// in any batch.
#include <algorithm>

#include "cplx.cuh"
#include "hm_internal.h"
#include "tile.cuh"
#include "wait.cuh"

namespace hm {

namespace {

constexpr int S2_NW = 8;       // warps per CTA
constexpr int S2_PIECE = 528;  // most entries of a piece of a block (forward dense blocks: see k_sweep2)
constexpr int S2_LR = 8;       // most factor columns in one piece of a low-rank block
constexpr int S2_RING = 4;     // most pieces staged ahead

// entries between the 16-byte boundary at or below p and p
template <class T> __device__ __forceinline__ int s2_rem(const T *p) { return sizeof(T) == 8 ? (int)((size_t)p >> 3 & 1) : 0; }

// A warp copies the 16-byte words that hold src[0 .. len) to dst (16-byte aligned; entry src[0] lands at
// dst + s2_rem(src)).  The words before and after belong to the same allocation (256-byte granules).
template <class T> __device__ __forceinline__ void s2_span(T *dst, const T *src, int len)
{
    const int rem = s2_rem(src), n = (int)(((rem + len) * sizeof(T) + 15) / 16);
    const char *g = (const char *)(src - rem);
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll 4
    for (int i = threadIdx.x & 31; i < n; i += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16 * i), "l"(g + 16 * i) : "memory");
}

// How a lane's outputs lie in a 64 x GW block: RL row lanes x CL column lanes, TC columns each; row
// lane l has the rows l + RL t.
template <int GW> struct S2Map {
    static constexpr int TC = GW < 4 ? GW : 4, CL = GW / TC, RL = 32 / CL, TR = 64 / RL, TH = TR / 2;   // TH: 32 rows
};

// a vector load of the hand-over buffers: words of 8 bytes, EPV entries
template <class T, int GW> struct S2Vec {
    static constexpr int EPV = sizeof(T) == 16 ? 1 : (GW > 1 ? 2 : 1);
    static constexpr bool WIDE = sizeof(T) * EPV == 16;
};
template <bool WIDE> __device__ __forceinline__ uint4 s2_ld(const void *p)
{
    if constexpr (WIDE) return ld_words2(p);
    const uint2 v = ld_word(p);
    return make_uint4(v.x, v.y, 0, 0);
}
__device__ __forceinline__ bool s2_stale(uint4 v) { return (v.x & v.y) == ~0u || (v.z & v.w) == ~0u; }

// the L2 cache fetches the bytes at p (rounded out to 16: arena allocations end on 256)
__device__ __forceinline__ void s2_prefetch(const void *p, size_t bytes)
{
    const size_t a = (size_t)p & ~(size_t)15, n = ((size_t)p + bytes + 15 & ~(size_t)15) - a;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)n) : "memory");
}

// The warp waits until the vectors at p (of the lanes that want one) are published; false when the
// wait ran out or another one had.
template <bool WIDE> __device__ __noinline__ bool s2_wait(const void *p, bool want, int *err)
{
    unsigned long long t0 = 0, bound = 0;
    for (int it = 1;; ++it) {
        if (!__any_sync(0xffffffffu, want && s2_stale(s2_ld<WIDE>(p)))) return true;
        if ((it & 7) == 0) {   // now and then: has another wait expired, or this one?
            if (__any_sync(0xffffffffu, *(volatile int *)err != 0)) return false;
            const unsigned long long t = gtimer();
            if (!t0) t0 = t, bound = wait_bound(err);
            else if (__any_sync(0xffffffffu, t - t0 > bound)) {
                if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, ERR_TIMEOUT);
                return false;
            }
        }
    }
}

// publishes a result: no 8-byte word of it is all ones
__device__ __forceinline__ void s2_publish(float2 *p, float2 v)
{
    unsigned a = __float_as_uint(v.x), b = __float_as_uint(v.y);
    if ((a & b) == ~0u) a = 0x7fffffffu;
    st_word(p, make_uint2(a, b));
}
__device__ __forceinline__ void s2_publish(double2 *p, double2 v)
{
    uint4 w = make_uint4((unsigned)__double2loint(v.x), (unsigned)__double2hiint(v.x), (unsigned)__double2loint(v.y),
                         (unsigned)__double2hiint(v.y));
    if ((w.x & w.y) == ~0u) w.y = 0x7fffffffu;
    if ((w.z & w.w) == ~0u) w.w = 0x7fffffffu;
    st_words2(p, w);
}

// One warp's reader of vector blocks: issue() starts the loads of rows [row, row + nc) of a
// hand-over buffer (columns of the group) into registers, finish() waits until every word is
// published and leaves them in ys[q * GW + c].
template <class T, int GW> struct S2Reader {
    typedef S2Vec<T, GW> V;
    static constexpr int VPR = GW / V::EPV;                       // vectors per row
    static constexpr int NMAX = sizeof(T) == 8 ? 4 : 8;           // vectors in registers: blocks of up to 32 rows at GW = 8
    static constexpr int NV = (64 * VPR + 31) / 32 < NMAX ? (64 * VPR + 31) / 32 : NMAX;
    const T *base;
    int64_t ld;
    uint4 v[NV];
    int row, cnt;

    __device__ __forceinline__ const T *at(int e) const
    {
        return base + (int64_t)(row + e / VPR) * ld + (e % VPR) * V::EPV;
    }
    __device__ __forceinline__ void load(int e0)
    {
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int e = e0 + u * 32;
            if (e < cnt) v[u] = s2_ld<V::WIDE>(at(e));
        }
    }
    __device__ __forceinline__ void issue(const T *b, int64_t ld_, int row_, int nc)
    {
        base = b;
        ld = ld_;
        row = row_;
        cnt = nc * VPR;
        load(threadIdx.x & 31);
    }
    __device__ __forceinline__ void finish(int *err, T *ys)
    {
        const int lane = threadIdx.x & 31;
        for (int p = 0; p < cnt; p += NV * 32) {
            if (p > 0) load(p + lane);
            for (;;) {
                int first = -1;   // the lane's first vector that is not published yet
#pragma unroll
                for (int u = NV - 1; u >= 0; --u)
                    if (p + lane + u * 32 < cnt && s2_stale(v[u])) first = u;
                if (!__any_sync(0xffffffffu, first >= 0)) break;
                if (!s2_wait<V::WIDE>(at(first < 0 ? 0 : p + lane + first * 32), first >= 0, err)) break;
                load(p + lane);
            }
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                const int e = p + lane + u * 32;
                if (e < cnt) {
                    if constexpr (V::WIDE) *(uint4 *)(ys + e * V::EPV) = v[u];
                    else *(uint2 *)(ys + e) = make_uint2(v[u].x, v[u].y);
                }
            }
        }
    }
};

template <class T, int GW> __device__ __forceinline__ void s2_row(const T *yp, T (&y)[S2Map<GW>::TC])
{
    if constexpr (sizeof(T) == 8 && S2Map<GW>::TC >= 2) {
#pragma unroll
        for (int c = 0; c < S2Map<GW>::TC; c += 2) {
            const float4 f = *(const float4 *)(yp + c);
            y[c].x = f.x;
            y[c].y = f.y;
            y[c + 1].x = f.z;
            y[c + 1].y = f.w;
        }
    } else {
#pragma unroll
        for (int c = 0; c < S2Map<GW>::TC; ++c) y[c] = yp[c];
    }
}

// acc(row, c) += sum over q < kl of ws[q * ldw + row] ys[q * GW + c], q ascending, for the rows of the first TRN
template <class T, int GW, int TRN>
__device__ __forceinline__ void s2_mac(T (&acc)[S2Map<GW>::TR][S2Map<GW>::TC], const T *ws, int ldw, const T *ys, int kl)
{
    typedef S2Map<GW> M;
    const int lane = threadIdx.x & 31;
    const T *wp = ws + lane % M::RL;
    const T *yp = ys + lane / M::RL * M::TC;
#pragma unroll 2
    for (int q = 0; q < kl; ++q) {
        T w[TRN], y[M::TC];
#pragma unroll
        for (int t = 0; t < TRN; ++t) w[t] = wp[q * ldw + t * M::RL];
        s2_row<T, GW>(yp + q * GW, y);
#pragma unroll
        for (int t = 0; t < TRN; ++t)
#pragma unroll
            for (int c = 0; c < M::TC; ++c) acc[t][c] = cfma(w[t], y[c], acc[t][c]);
    }
}
template <class T, int GW, int TRN = 1>
__device__ __forceinline__ void s2_mac_rows(T (&acc)[S2Map<GW>::TR][S2Map<GW>::TC], int no, const T *ws, int ldw,
                                            const T *ys, int kl)
{
    if constexpr (TRN == S2Map<GW>::TR) s2_mac<T, GW, TRN>(acc, ws, ldw, ys, kl);
    else if (no <= TRN * S2Map<GW>::RL) s2_mac<T, GW, TRN>(acc, ws, ldw, ys, kl);
    else s2_mac_rows<T, GW, TRN + 1>(acc, no, ws, ldw, ys, kl);
}

// The same for rows [r0, r0 + rn), which lie in the lanes' rows TI .. TI + TN - 1, of a block stored row by
// row, ws[(row - r0) * nc + q].  (Two steps per 16-byte load halve the bank conflicts of an even nc, but the
// longer code cost more in instruction fetches: 3.08 against 2.88 ms per 64-column forward sweep.)
template <class T, int GW, int TI, int TN>
__device__ __forceinline__ void s2_mac_t(T (&acc)[S2Map<GW>::TR][S2Map<GW>::TC], const T *ws, int r0, int rn, const T *ys,
                                         int nc)
{
    typedef S2Map<GW> M;
    const int lane = threadIdx.x & 31;
    const T *wp[TN];
    bool in[TN];
#pragma unroll
    for (int t = 0; t < TN; ++t) {
        const int row = (TI + t) * M::RL + lane % M::RL - r0;
        in[t] = row >= 0 && row < rn;
        wp[t] = ws + (in[t] ? row : 0) * nc;
    }
    const T *yp = ys + lane / M::RL * M::TC;
#pragma unroll 2
    for (int q = 0; q < nc; ++q) {
        T w[TN], y[M::TC];
#pragma unroll
        for (int t = 0; t < TN; ++t) {
            w[t] = wp[t][q];
            if (!in[t]) w[t] = czero(T());
        }
        s2_row<T, GW>(yp + q * GW, y);
#pragma unroll
        for (int t = 0; t < TN; ++t)
#pragma unroll
            for (int c = 0; c < M::TC; ++c) acc[TI + t][c] = cfma(w[t], y[c], acc[TI + t][c]);
    }
}
template <class T, int GW, int TI>
__device__ __forceinline__ void s2_mac_half(T (&acc)[S2Map<GW>::TR][S2Map<GW>::TC], const T *ws, int r0, int rn,
                                            const T *ys, int nc)
{
    typedef S2Map<GW> M;
    if constexpr (M::TH == 1) s2_mac_t<T, GW, TI, 1>(acc, ws, r0, rn, ys, nc);
    else if (r0 == TI * M::RL && rn <= M::RL) s2_mac_t<T, GW, TI, 1>(acc, ws, r0, rn, ys, nc);
    else s2_mac_t<T, GW, TI, 2>(acc, ws, r0, rn, ys, nc);
}

// tb[l * GW + c] = sum over q < nc of g[q + l * nc] ys[q * GW + c], l < lr.  Complex FP32: one lane per
// output, q ascending.  FP64: eight lanes per output (q = s, s + 8, ...; then a fixed tree), because a
// DFMA takes its scheduler 64 cycles however few lanes are active.
template <class T, int GW> __device__ __forceinline__ void s2_lowrank(const T *g, int nc, int lr, const T *ys, T *tb)
{
    const int lane = threadIdx.x & 31;
    if constexpr (sizeof(T) == 8) {
        for (int o = lane; o < lr * GW; o += 32) {
            const int l = o / GW, c = o % GW;
            T v = czero(T());
#pragma unroll 4
            for (int q = 0; q < nc; ++q) v = cfma(g[q + l * nc], ys[q * GW + c], v);
            tb[o] = v;
        }
    } else {
        const int s = lane & 7;
        for (int o0 = 0; o0 < lr * GW; o0 += 4) {
            const int o = o0 + (lane >> 3), l = o / GW, c = o % GW;
            T v = czero(T());
            if (o < lr * GW)
                for (int q = s; q < nc; q += 8) v = cfma(g[q + l * nc], ys[q * GW + c], v);
#pragma unroll
            for (int d = 4; d > 0; d >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, d);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, d);
            }
            if (s == 0 && o < lr * GW) tb[o] = v;
        }
    }
}

// Shared memory: per warp a ring of staged coefficient pieces, a vector area and the products of a
// low-rank piece; two CTAs per SM in complex FP32, one in FP64.
template <class T, int GW> struct S2Smem {
    static constexpr int R = sizeof(T) == 16 ? (GW > 1 ? 1520 : 1664) : GW > 4 ? 1088 : GW > 1 ? 1344 : 1600;   // ring entries
    static constexpr int WARP = R + 64 * GW + S2_LR * GW;
    static constexpr size_t BYTES = sizeof(T) * (size_t)WARP * S2_NW;
    static constexpr int CTAS = BYTES <= 112 * 1024 ? 2 : 1;
};

// One block row and column group (see the file comment).  rows[o] and deps are the plan of the
// direction; N the rows of I + N_S or of its transpose; Y, Z the hand-over buffers.
template <class T, int GW, bool FWD>
__global__ void __launch_bounds__(32 * S2_NW, S2Smem<T, GW>::CTAS)
    k_sweep2(int nb, const S2Row *rows, const int4 *deps, const T *W, const T *N, const T *x, T *y, int n, int nrhs, int G,
             int *ticket, T *Y, T *Z, int *err)
{
    typedef S2Map<GW> M;
    typedef S2Smem<T, GW> SM;
    extern __shared__ unsigned char smraw[];
    __shared__ int s_t;
    if (threadIdx.x == 0) s_t = atomicAdd(ticket, 1) + 1;   // the counter starts at all ones
    __syncthreads();
    const int pos = s_t / G, g = s_t % G;
    if (pos >= nb) return;
    const int o = FWD ? pos : nb - 1 - pos;
    if (held_back(err, o)) return;
    const S2Row R = rows[o];
    const int no = R.no, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c0 = g * GW, ncol = nrhs - c0;
    const int64_t ldy = (int64_t)G * GW;
    Y += c0;
    Z += c0;
    T *const sm = (T *)smraw, *const wb = sm + w * SM::WARP, *const yb = wb + SM::R, *const tb = yb + 64 * GW;
    __shared__ int4 s_meta[S2_NW][S2_RING];
    // the thread's outputs e = tid + 256 u: column e % GW, row e / GW
    constexpr int NO = (64 * GW + 32 * S2_NW - 1) / (32 * S2_NW);
    T xv[NO];
#pragma unroll
    for (int u = 0; u < NO; ++u) {
        const int e = threadIdx.x + u * 32 * S2_NW, c = e % GW, r = e / GW;
        xv[u] = e < no * GW && c < ncol ? x[R.ro + r + (int64_t)(c0 + c) * n] : czero(T());
    }
    T acc[M::TR][M::TC];
    auto clear = [&]() {
#pragma unroll
        for (int t = 0; t < M::TR; ++t)
#pragma unroll
            for (int c = 0; c < M::TC; ++c) acc[t][c] = czero(T());
    };
    auto put_partial = [&]() {   // the warp's sums into its vector area
#pragma unroll
        for (int t = 0; t < M::TR; ++t) {
            const int r = lane % M::RL + t * M::RL;
            if (r < no)
#pragma unroll
                for (int c = 0; c < M::TC; ++c) yb[r * GW + lane / M::RL * M::TC + c] = acc[t][c];
        }
    };
    auto partial = [&](int e, int nw) {   // output e summed over the first nw warps
        T v = czero(T());
        for (int q = 0; q < nw; ++q) {
            const T a = sm[q * SM::WARP + SM::R + e];
            v.x += a.x;
            v.y += a.y;
        }
        return v;
    };
    S2Reader<T, GW> rd;
    // ---- phase A: the dependencies outside the super-row
    auto commit = []() { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
    if (threadIdx.x == 0 && R.zlen > 0) s2_prefetch(N + R.noff, sizeof(T) * (size_t)R.zlen * no);
    clear();
    {
        const int nd = R.ext > w ? (R.ext - w + S2_NW - 1) / S2_NW : 0;
        int4 dl = make_int4(0, 0, 0, 0);
        // The next piece to stage: entries [src, src + len) of dependency di of this warp (first row `row`, nc rows,
        // rank r, -1 dense).  Backward dense (no x nc) and low rank: columns [q0, q0 + kl); forward dense (nc x no, so
        // the row's blocks lie column by column): the columns of the rows [q0, q0 + kl).
        int di = -1, row = 0, nc = 0, r = 0, q0 = 0, kl = 0, step = 0, tot = 0;
        const T *base = W;
        auto next = [&]() {   // false past the last
            q0 += kl;
            if (q0 >= tot) {
                do {
                    if (++di >= nd) return false;
                    if ((di & 31) == 0) {   // the plan entries of this warp's next 32 dependencies, one per lane
                        const int t = w + S2_NW * (di + lane);
                        if (t < R.ext) {
                            dl = __ldg(deps + (FWD ? R.p0 + t : R.p0 - t));
                            const int n1 = dl.w & 0xffff, r1 = dl.w >> 16, len = r1 < 0 ? no * n1 : r1 * (no + n1);
                            const T *b = W + (int64_t)((unsigned long long)(unsigned)dl.y << 32 | (unsigned)dl.x);
                            if (len > 0) s2_prefetch(b, sizeof(T) * (size_t)len);
                        }
                    }
                    const int s = di & 31;
                    const unsigned lo = __shfl_sync(0xffffffffu, dl.x, s), hi = __shfl_sync(0xffffffffu, dl.y, s);
                    base = W + (int64_t)((unsigned long long)hi << 32 | lo);
                    row = __shfl_sync(0xffffffffu, dl.z, s);
                    const int nr = __shfl_sync(0xffffffffu, dl.w, s);
                    nc = nr & 0xffff;
                    r = nr >> 16;
                } while (r == 0);   // a block truncated to zero
                q0 = 0;
                if (r > 0) {
                    tot = r;
                    step = min(S2_LR, S2_PIECE / (no + nc));
                } else if (FWD) {
                    tot = no;
                    step = 32 * nc <= SM::R - 2 ? 32 : 16;
                } else {
                    tot = nc;
                    step = S2_PIECE / no;
                }
            }
            kl = min(step, tot - q0);
            return true;
        };
        int head = 0, tail = 0, out = 0, staged = 0;   // ring: next free entry, oldest piece, pieces in it
        bool cand = next();
        auto produce = [&]() {   // stage pieces while they fit
            while (cand && out < S2_RING) {
                // low rank, W_kj ~ P Q^T, P (n_k x r) then Q (n_j x r): forward (j = o) H = Q, G = P; backward (k = o)
                // H = P, G = Q; the columns [q0, q0 + kl) of H, then those of G
                const T *s1 = base + (r > 0 ? (FWD ? nc * r : 0) + q0 * no : FWD ? q0 * nc : q0 * no);
                const T *s2 = base + (FWD ? 0 : no * r) + q0 * nc;
                const int l1 = r > 0 ? kl * no : FWD ? kl * nc : kl * no, l2 = r > 0 ? kl * nc : 0;
                const int m1 = s2_rem(s1), z1 = l1 + m1 + 1 & ~1, m2 = s2_rem(s2), z2 = r > 0 ? l2 + m2 + 1 & ~1 : 0;
                const int sz = z1 + z2;
                if (out == 0) head = tail = 0;
                int at = head;
                if (head >= tail && out > 0 ? head + sz > SM::R : false) at = 0;
                if (out > 0 && at < tail && at + sz >= tail) return;   // no room yet
                if (out > 0 && at == tail) return;
                s2_span(wb + at, s1, l1);
                if (r > 0) s2_span(wb + at + z1, s2, l2);
                commit();
                if (lane == 0)
                    s_meta[w][staged & S2_RING - 1] =
                        make_int4(row, nc | (at + m1) << 16, r > 0 ? at + z1 + m2 : -1, q0 << 16 | kl << 1 | (int)(q0 == 0));
                head = at + sz;
                ++out;
                ++staged;
                cand = next();
            }
        };
        produce();
        __syncwarp();
        if (staged > 0) rd.issue(Y, ldy, s_meta[w][0].x, s_meta[w][0].y & 0xffff);
        for (int done = 0; out > 0; ++done) {
            if (out == 1) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            else if (out == 2) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            else if (out == 3) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
            else asm volatile("cp.async.wait_group 3;\n" ::: "memory");
            __syncwarp();
            const int4 m = s_meta[w][done & S2_RING - 1];
            const int mn = m.y & 0xffff, mq0 = m.w >> 16, mkl = m.w >> 1 & 0x7fff;
            const T *buf = wb + (m.y >> 16);
            if (m.w & 1) {   // a new dependency: its vector block
                rd.finish(err, yb);
                __syncwarp();
            }
            if (out > 1) {   // the loads of the next one
                const int4 mx = s_meta[w][done + 1 & S2_RING - 1];
                if (mx.w & 1) rd.issue(Y, ldy, mx.x, mx.y & 0xffff);
            }
            const T *ys = yb + mq0 * GW;
            if (m.z >= 0) {
                s2_lowrank<T, GW>(wb + m.z, mn, mkl, yb, tb);
                __syncwarp();
                ys = tb;
            }
            if (FWD && m.z < 0) {
                if (mq0 < 32) s2_mac_half<T, GW, 0>(acc, buf, mq0, mkl, yb, mn);
                else s2_mac_half<T, GW, M::TH>(acc, buf, mq0, mkl, yb, mn);
            } else
                s2_mac_rows<T, GW>(acc, no, buf, no, ys, mkl);
            __syncwarp();   // the piece's ring entries are free
            const bool alone = out == 1;
            --out;
            if (out > 0) tail = s_meta[w][done + 1 & S2_RING - 1].y >> 16 & ~1;
            produce();
            if (alone && out > 0) {   // the next piece was not staged above
                __syncwarp();
                const int4 mx = s_meta[w][done + 1 & S2_RING - 1];
                if (mx.w & 1) rd.issue(Y, ldy, mx.x, mx.y & 0xffff);
            }
        }
    }
    // the first pieces of N, whose coefficients do not wait on anything
    const int kc = no <= 33 ? 16 : 8, ns = (R.zlen + kc - 1) / kc;
    int nat[2] = {0, 0};   // entry of each half of the ring where the piece's first coefficient lies
    auto stage_n = [&](int s, int half) {
        if (s < ns) {
            const T *src = N + R.noff + (int64_t)s * kc * no;
            s2_span(wb + half * (SM::R / 2), src, min(kc, R.zlen - s * kc) * no);
            nat[half] = half * (SM::R / 2) + s2_rem(src);
        }
        commit();
    };
    stage_n(w, 0);
    put_partial();
    __syncthreads();
    T *const Zo = Z + R.ro * ldy, *const Yo = Y + R.ro * ldy;
#pragma unroll
    for (int u = 0; u < NO; ++u) {
        const int e = threadIdx.x + u * 32 * S2_NW;
        if (e < no * GW) {
            const T v = partial(e, min(S2_NW, R.ext));
            xv[u].x -= v.x;
            xv[u].y -= v.y;
            const int64_t at = (int64_t)(e / GW) * ldy + e % GW;
            s2_publish(Zo + at, xv[u]);
            if (ns == 0) s2_publish(Yo + at, xv[u]);
        }
    }
    // ---- phase B: the members of the super-row that come before this row
    if (ns > 0) {
        __syncthreads();   // the partial sums are read before the vector areas are reused
        clear();
        if (w < ns) rd.issue(Z, ldy, R.zrow + w * kc, min(kc, R.zlen - w * kc));
        auto slab = [&](int s, int half) {
            const int sn = s + S2_NW;
            stage_n(sn, half ^ 1);
            rd.finish(err, yb);
            if (sn < ns) rd.issue(Z, ldy, R.zrow + sn * kc, min(kc, R.zlen - sn * kc));
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            __syncwarp();
            s2_mac_rows<T, GW>(acc, no, wb + nat[half], no, yb, min(kc, R.zlen - s * kc));
            __syncwarp();
        };
        for (int s = w; s < ns; s += 2 * S2_NW) {
            slab(s, 0);
            if (s + S2_NW < ns) slab(s + S2_NW, 1);
        }
        put_partial();
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NO; ++u) {
            const int e = threadIdx.x + u * 32 * S2_NW;
            if (e < no * GW) {
                const T v = partial(e, min(S2_NW, ns));
                xv[u].x += v.x;
                xv[u].y += v.y;
                s2_publish(Yo + (int64_t)(e / GW) * ldy + e % GW, xv[u]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < NO; ++u) {
        const int e = threadIdx.x + u * 32 * S2_NW, c = e % GW;
        if (e < no * GW && c < ncol) y[R.ro + e / GW + (int64_t)(c0 + c) * n] = xv[u];
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// deps[0][p] (gather list of the forward sweep) and deps[1][e] (S_k lists) of k_sweep2: where the
// coefficient block is, its dependency's first row, its rows and rank
__global__ void k_s2_deps(int ne, const int *ridx, const int *rent, const int *sidx, const int *boff, const int *size,
                          const int64_t *cbo, const int *crk, int4 *fwd, int4 *bwd)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
    auto entry = [&](int ent, int dep) {
        const unsigned long long off = (unsigned long long)cbo[ent];
        return make_int4((int)(unsigned)off, (int)(unsigned)(off >> 32), boff[dep],
                         (int)((unsigned)crk[ent] << 16 | (unsigned)size[dep]));
    };
    fwd[e] = entry(rent[e], ridx[e]);
    bwd[e] = entry(e, sidx[e]);
}

// N_S = L_SS^{-1} - I, one CTA per S2_IC columns of a block column j of its super-row: with L_im = W_mi^T as the
// sweeps apply it (a compressed block expanded), N_ij = -(L_ij + sum over j < m < i of L_im N_mj), i ascending.
// Written twice: row i of N (n_i x the rows before it in the super-row) and row j of N^T (n_j x the rows after
// it).  The recurrence over i is serial, its columns are not: whole block columns per CTA took 5.7 ms of the FP64 setup
// of the 1,920-unknown sphere.
constexpr int S2_IC = 8;
template <class T>
__global__ void __launch_bounds__(256) k_s2_inverse(int nb, const int *size, const int *boff, const int *sptr,
                                                    const int *sidx, const int64_t *cbo, const int *crk, const T *W,
                                                    const int64_t *off0, const int64_t *off1, T *N, T *NT)
{
    extern __shared__ unsigned char smraw[];
    T *Ls = (T *)smraw, *Ns = Ls + 64 * 65;   // Ls[r * 65 + q] = L_im(r, q), Ns[q + c * 65] = N_mj(q, c0 + c)
    const int j = blockIdx.x, b0 = j / S2_K * S2_K, b1 = min(nb, b0 + S2_K), nj = size[j];
    const int c0 = blockIdx.y * S2_IC, ncol = min(S2_IC, nj - c0);
    if (ncol <= 0) return;
    constexpr int NO = 64 * S2_IC / 256;
    for (int i = j + 1; i < b1; ++i) {
        const int ni = size[i], len = ni * ncol;
        T acc[NO];
#pragma unroll
        for (int u = 0; u < NO; ++u) acc[u] = czero(T());
        for (int m = j; m < i; ++m) {
            int e = -1;   // entry of block (m, i), if S_m holds i (S_m is sorted: at most S2_K - 1 entries to look at)
            for (int p = sptr[m]; p < sptr[m + 1] && sidx[p] <= i; ++p)
                if (sidx[p] == i) e = p;
            if (e < 0) continue;
            const int nm = size[m], r = crk[e];
            const T *B = W + cbo[e];
            __syncthreads();   // the previous product is done with the tiles; N_mj of these columns is written
            for (int x = threadIdx.x; x < nm * ni; x += blockDim.x) {
                const int q = x % nm, rr = x / nm;
                T v;
                if (r < 0) v = B[x];
                else {
                    v = czero(T());
                    for (int l = 0; l < r; ++l) v = cfma(B[q + l * nm], B[nm * r + rr + l * ni], v);
                }
                Ls[rr * 65 + q] = v;
            }
            if (m > j)
                for (int x = threadIdx.x; x < nm * ncol; x += blockDim.x) {
                    const int q = x % nm, c = x / nm;
                    Ns[q + c * 65] = N[off0[m] + q + (int64_t)(boff[j] - boff[b0] + c0 + c) * nm];
                }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < NO; ++u) {
                const int x = threadIdx.x + u * 256;
                if (x < len) {
                    const int rr = x % ni, c = x / ni;
                    if (m == j) {
                        acc[u] = Ls[rr * 65 + c0 + c];
                        continue;
                    }
                    for (int q = 0; q < nm; ++q) acc[u] = cfma(Ls[rr * 65 + q], Ns[q + c * 65], acc[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < NO; ++u) {
            const int x = threadIdx.x + u * 256;
            if (x < len) {
                const int rr = x % ni, c = c0 + x / ni;
                const T v = {-acc[u].x, -acc[u].y};
                N[off0[i] + rr + (int64_t)(boff[j] - boff[b0] + c) * ni] = v;
                NT[off1[j] + c + (int64_t)(boff[i] - boff[j + 1] + rr) * nj] = v;
            }
        }
        __syncthreads();
    }
}

template <class T> size_t s2_buf_bytes(int n) { return 256 + 2 * sizeof(T) * (size_t)n * (sizeof(T) == 16 ? 16 : 64); }

// the direction's block rows as k_sweep2 walks them
std::vector<S2Row> s2_rows(const Plan &P, bool fwd, const std::vector<int64_t> &off)
{
    std::vector<S2Row> rows(P.nb);
    for (int o = 0; o < P.nb; ++o) {
        const int b0 = o / S2_K * S2_K, b1 = std::min(P.nb, b0 + S2_K);
        S2Row &R = rows[o];
        R.ro = P.boff[o];
        R.no = P.size[o];
        R.noff = off[o];
        const int lo = fwd ? P.rptr[o] : P.sptr[o], hi = fwd ? P.rptr[o + 1] : P.sptr[o + 1];
        int inside = 0;
        for (int p = lo; p < hi; ++p) inside += fwd ? P.ridx[p] >= b0 : P.sidx[p] < b1;
        R.p0 = fwd ? lo : hi - 1;   // walked upwards / downwards, the members of the super-row last
        R.ext = hi - lo - inside;
        R.zrow = fwd ? P.boff[b0] : P.boff[o + 1];
        R.zlen = fwd ? P.boff[o] - P.boff[b0] : P.boff[b1] - P.boff[o + 1];
    }
    return rows;
}

template <class T> cudaError_t s2_build(hm_ctx *h, const T *W)
{
    const Plan &P = h->plan;
    const int ne = (int)P.sidx.size();
    cudaStream_t st = h->stream;
    cudaError_t e;
    if (!h->s2.buf) {
        std::vector<int64_t> off[2];
        int64_t len = 0;
        off[0].resize(P.nb), off[1].resize(P.nb);
        for (int i = 0; i < P.nb; ++i) {
            off[0][i] = len;
            len += (int64_t)P.size[i] * (P.boff[i] - P.boff[i / S2_K * S2_K]);
        }
        int64_t len1 = 0;
        for (int j = 0; j < P.nb; ++j) {
            off[1][j] = len1;
            len1 += (int64_t)P.size[j] * (P.boff[std::min(P.nb, j / S2_K * S2_K + S2_K)] - P.boff[j + 1]);
        }
        h->s2.bytes = 2 * (Arena::rounded(sizeof(S2Row) * P.nb) + Arena::rounded(sizeof(int64_t) * P.nb) +
                           Arena::rounded(sizeof(int4) * std::max(ne, 1)) +
                           Arena::rounded(sizeof(T) * (size_t)std::max<int64_t>(len, 1))) +
                      Arena::rounded(s2_buf_bytes<T>(P.n));
        if (!h->arena.room(h->s2.bytes)) return cudaErrorMemoryAllocation;
        for (int d = 0; d < 2; ++d) {
            const std::vector<S2Row> rows = s2_rows(P, d == 0, off[d]);
            if ((e = h->arena.alloc((void **)&h->s2.rows[d], sizeof(S2Row) * P.nb)) ||
                (e = h->arena.alloc((void **)&h->s2.off[d], sizeof(int64_t) * P.nb)) ||
                (e = h->arena.alloc((void **)&h->s2.deps[d], sizeof(int4) * std::max(ne, 1))) ||
                (e = h->arena.alloc(&h->s2.N[d], sizeof(T) * (size_t)std::max<int64_t>(len, 1))) ||
                (e = cudaMemcpyAsync(h->s2.rows[d], rows.data(), sizeof(S2Row) * P.nb, cudaMemcpyHostToDevice, st)) ||
                (e = cudaMemcpyAsync(h->s2.off[d], off[d].data(), sizeof(int64_t) * P.nb, cudaMemcpyHostToDevice, st)) ||
                (e = cudaStreamSynchronize(st)))
                return e;
        }
        if ((e = h->arena.alloc(&h->s2.buf, s2_buf_bytes<T>(P.n)))) return e;
    }
    const size_t smem = sizeof(T) * (64 + S2_IC) * 65;
    const int maxn = *std::max_element(P.size.begin(), P.size.end());
    static DeviceOnce attr;
    if (attr.need()) {
        if ((e = cudaFuncSetAttribute(k_s2_inverse<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
        attr.done();
    }
    if (ne > 0)
        HM_LAUNCH(h, K_PANEL,
                  k_s2_deps<<<(ne + 255) / 256, 256, 0, st>>>(ne, h->d_ridx, h->d_rent, h->d_sidx, h->d_boff, h->d_size,
                                                              h->d_cboff, h->d_crank, h->s2.deps[0], h->s2.deps[1]));
    HM_LAUNCH(h, K_PANEL,
              k_s2_inverse<T><<<dim3(P.nb, (maxn + S2_IC - 1) / S2_IC), 256, smem, st>>>(P.nb, h->d_size, h->d_boff, h->d_sptr, h->d_sidx, h->d_cboff,
                                                       h->d_crank, W, h->s2.off[0], h->s2.off[1], (T *)h->s2.N[0],
                                                       (T *)h->s2.N[1]));
    return cudaGetLastError();
}

template <class T, int GW>
cudaError_t s2_launch(hm_ctx *h, bool fwd, const T *W, const T *x, T *y, int nrhs)
{
    const Plan &P = h->plan;
    typedef S2Smem<T, GW> SM;
    static DeviceOnce attr;
    cudaError_t e;
    if (attr.need()) {
        if ((e = cudaFuncSetAttribute(k_sweep2<T, GW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::BYTES)) ||
            (e = cudaFuncSetAttribute(k_sweep2<T, GW, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::BYTES)))
            return e;
        attr.done();
    }
    const int G = (nrhs + GW - 1) / GW;
    const size_t len = (size_t)P.n * G * GW;
    int *ticket = (int *)h->s2.buf;
    T *Y = (T *)((char *)h->s2.buf + 256), *Z = Y + len;
    // nothing published yet: every word, the ticket among them, all ones
    if ((e = cudaMemsetAsync(h->s2.buf, 0xff, 256 + 2 * sizeof(T) * len, h->stream))) return e;
    const unsigned grid = (unsigned)(P.nb * G);
    if (fwd)
        HM_LAUNCH(h, K_SWEEP_FWD,
                  (k_sweep2<T, GW, true><<<grid, 32 * S2_NW, SM::BYTES, h->stream>>>(
                      P.nb, h->s2.rows[0], h->s2.deps[0], W, (const T *)h->s2.N[0], x, y, P.n, nrhs, G, ticket, Y, Z,
                      h->d_err)));
    else
        HM_LAUNCH(h, K_SWEEP_BWD,
                  (k_sweep2<T, GW, false><<<grid, 32 * S2_NW, SM::BYTES, h->stream>>>(
                      P.nb, h->s2.rows[1], h->s2.deps[1], W, (const T *)h->s2.N[1], x, y, P.n, nrhs, G, ticket, Y, Z,
                      h->d_err)));
    return cudaGetLastError();
}

}  // namespace

void sweep2_release(hm_ctx *h)
{
    h->s2.on = false;
    for (int d = 0; d < 2; ++d) {
        h->arena.release(h->s2.rows[d], 0);
        h->arena.release(h->s2.off[d], 0);
        h->arena.release(h->s2.deps[d], 0);
        h->arena.release(h->s2.N[d], 0);
        h->s2.rows[d] = nullptr;
        h->s2.off[d] = nullptr;
        h->s2.deps[d] = nullptr;
        h->s2.N[d] = nullptr;
    }
    h->arena.release(h->s2.buf, 0);
    h->s2.buf = nullptr;
}

// After every setup: the plan entries and N_S of the coefficients the sweeps read.  Without room
// for them (hbm_budget) the sweeps stay with the kinds of ops.cu.
cudaError_t sweep2_setup(hm_ctx *h)
{
    h->s2.on = h->s2.given = false;
    const cudaError_t e = h->opts.precision == 1 ? s2_build<float2>(h, h->d_Wc32) : s2_build<double2>(h, h->d_Wc);
    if (e == cudaErrorMemoryAllocation) {
        sweep2_release(h);
        return cudaSuccess;
    }
    h->s2.on = e == cudaSuccess;
    return e;
}

// Where a solve or a batch made the handle give the data back and has returned its own memory: formed again.
void sweep2_restore(hm_ctx *h)
{
    if (!h->s2.given || !h->setup_done) return;
    const size_t tags = h->d_ytag && !h->sweep_fixed ? Arena::rounded(sizeof(uint4) * (size_t)h->plan.n * 64) : 0;
    if (h->arena.budget && h->arena.used - tags + h->s2.bytes > h->arena.budget) return;
    if (tags) {   // the other sweeps' words, which are no longer needed
        h->arena.release(h->d_ytag, 0);
        h->d_ytag = nullptr;
    }
    if (sweep2_setup(h)) cudaGetLastError();
    h->s2.given = !h->s2.on;
}

// Column groups: one column alone; 4 in FP64 and in complex FP32 up to 16 columns (on the 30,720-unknown
// sphere 16 columns took 1.03-1.26 ms a sweep in groups of 4, 1.24-1.51 in groups of 8: the chain binds);
// 8 in complex FP32 above (64 columns: 2.4-3.1 against 3.4-4.0 ms: the instructions bind).  Groups
// of 16 leave one CTA per SM (4.2 ms).
template <class T> cudaError_t sweep2_run(hm_ctx *h, bool fwd, const T *W, const T *x, T *y, int nrhs)
{
    if (nrhs == 1) return s2_launch<T, 1>(h, fwd, W, x, y, nrhs);
    if (sizeof(T) == 16 || nrhs <= 16) return s2_launch<T, 4>(h, fwd, W, x, y, nrhs);
    if constexpr (sizeof(T) == 8) return s2_launch<T, 8>(h, fwd, W, x, y, nrhs);
    return cudaErrorInvalidValue;
}
template cudaError_t sweep2_run<float2>(hm_ctx *, bool, const float2 *, const float2 *, float2 *, int);
template cudaError_t sweep2_run<double2>(hm_ctx *, bool, const double2 *, const double2 *, double2 *, int);

}  // namespace hm
