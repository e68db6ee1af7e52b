// Far-field product v = Z_F u (Sec. 2 Eq. 9 blocks, Eq. 11), complex FP64 or FP32.
//
// Z_F is stored once per admissible pair (rows r-range, columns c-range, r before c): a
// low-rank block U V^T or a dense block B; the mirrored block is its transpose.  u is given
// in cluster order with the right-hand sides interleaved (u[i * nrhs + r]); v is written
// in solve order, column-major.
//
// Phase 1 (k_far_t): the rank vectors t_b = V_b^T u[c-range] and s_b = U_b^T u[r-range].
// Factor columns that contract over the same index range are stacked (up to 64 per task),
// so one CTA stages each piece of u once for all of them (cp.async, double buffered) and
// runs a register-tiled product (tile.cuh; complex FP64: integer digits on the tensor cores); t and s are stored
// interleaved like u.
// Phase 2 (k_far_y): one CTA per leaf accumulates, in the order of the leaf's list of
// covering far blocks, U_b t_b (row side), V_b s_b (column side), B u (dense row side) and
// B^T u (dense column side) for the leaf's rows; the host plan cuts the list into
// contraction segments of at most 32, which are staged in shared memory in chunks.  Each
// leaf's list is split into FAR_PARTS consecutive parts of about equal length, one CTA each
// (so that the uneven leaves spread over all SMs); k_far_sum adds the parts in order.  Every output sums its terms in
// one fixed order, so results are deterministic and do not depend on how many right-hand
// sides share the launch.
#include <algorithm>
#include <cstdint>

#include "cplx.cuh"
#include "hm_internal.h"
#include "tc.cuh"
#include "tile.cuh"

namespace hm {

static inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

namespace {
constexpr int SEG = 64;   // longest staged contraction segment
}

// Phase 1: one CTA per task (a range [lo, hi) and up to 64 stacked factor columns).  The
// range is walked in pieces of FAR_T1 rows, each piece's factor rows and vector rows copied
// with cp.async into the two halves of shared memory in turn, so the copy of the next piece
// overlaps the product of the current; every output sums its rows in ascending order.
constexpr int FAR_T1 = 32;

template <class T> __device__ __forceinline__ void far_cp(T *dst, const T *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}

// The task's factor columns, in item order (at most 64 columns, so at most 64 items of rank >= 1): column R of
// item s_item[R], its l-th, at s_src[R]; returns their number.  One thread per column: a walk by one thread
// waited on memory twice per item, about 5 us per task.
template <class T>
__device__ __forceinline__ int far_items(int i0, int i1, const int64_t *item_off, const int *item_ld, const int *item_rank,
                                         const int *item_isv, const T *U, const T *V, int *s_item, int *s_l,
                                         const T **s_src)
{
    __shared__ int s_cum[65];
    const int ni = min(i1 - i0, 64), tid = threadIdx.x;
    if (tid < ni) s_cum[tid + 1] = item_rank[i0 + tid];
    __syncthreads();
    if (tid == 0) {
        s_cum[0] = 0;
        for (int q = 0; q < ni; ++q) s_cum[q + 1] += s_cum[q];
    }
    __syncthreads();
    const int R = min(s_cum[ni], 64);
    if (tid < R) {
        int q = 0;
        while (s_cum[q + 1] <= tid) ++q;
        const int it = i0 + q, l = tid - s_cum[q];
        s_item[tid] = it;
        s_l[tid] = l;
        s_src[tid] = (item_isv[it] ? V : U) + item_off[it] + (int64_t)l * item_ld[it];
    }
    __syncthreads();
    return R;
}

template <class T, int TR, int TC, int NT>
__global__ void __launch_bounds__(256) k_far_t(const int *task_lo, const int *task_hi, const int *task_ptr,
                                               const int64_t *item_off, const int *item_ld, const int *item_rank,
                                               const int *item_row, const int *item_isv, const T *U, const T *V,
                                               const T *u, int nrhs, T *t, T *s, int budget)
{
    extern __shared__ unsigned char smraw[];
    __shared__ int s_item[64], s_l[64];
    __shared__ const T *s_src[64];
    const int task = blockIdx.x;
    const int lo = task_lo[task], hi = task_hi[task], i0 = task_ptr[task], i1 = task_ptr[task + 1];
    const int R = far_items(i0, i1, item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src);
    const int nrt = (R + TR - 1) / TR, ntiles = nrt * ((nrhs + TC - 1) / TC);
    const int ldw = stage_ldw(R, TR), ldr = stage_ldr(nrhs, TC);
    T *const bufs[2] = {(T *)smraw, (T *)smraw + budget / 2};
    Tile<T, TR, TC, NT> acc;
    tile_load(acc, (const T *)nullptr, 0, 0, R, nrhs, nrt, ntiles);
    // copy piece [c0, c0 + ch) into bufs[which]: Ws[qq*ldw + rr] = factor rr at row c0 + qq,
    // Ys[qq*ldr + r] = u[(c0 + qq) * nrhs + r]
    auto stage = [&](int c0, int which) {
        const int ch = min(FAR_T1, hi - c0);
        T *Ws = bufs[which], *Ys = bufs[which] + ch * ldw;
        for (int e = threadIdx.x; e < ch * R; e += blockDim.x) {
            const int qq = e % ch, rr = e / ch;
            far_cp(Ws + qq * ldw + rr, s_src[rr] + (c0 - lo + qq));
        }
        const T *uc = u + (int64_t)c0 * nrhs;
        for (int e = threadIdx.x; e < ch * nrhs; e += blockDim.x) far_cp(Ys + (e / nrhs) * ldr + e % nrhs, uc + e);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (lo < hi) stage(lo, 0);
    for (int c0 = lo, it = 0; c0 < hi; c0 += FAR_T1, ++it) {
        const int ch = min(FAR_T1, hi - c0);
        if (c0 + FAR_T1 < hi) {
            stage(c0 + FAR_T1, (it + 1) & 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        T *Ws = bufs[it & 1];
        tile_mac<false>(acc, Ws, ldw, Ws + ch * ldw, ldr, 1, ch, nrt, ntiles);
        __syncthreads();
    }
#pragma unroll
    for (int tt = 0; tt < NT; ++tt) {
        const TileRC m = tile_rc<TR, TC>(threadIdx.x + tt * blockDim.x, nrt, ntiles);
        const int row0 = m.row0, r0 = m.c0;
#pragma unroll
        for (int a = 0; a < TR; ++a)
#pragma unroll
            for (int c = 0; c < TC; ++c)
                if (m.ok && row0 + a < R && r0 + c < nrhs) {
                    const int it = s_item[row0 + a];
                    T *dst = item_isv[it] ? t : s;
                    dst[(int64_t)(item_row[it] + s_l[row0 + a]) * nrhs + r0 + c] = acc.v[tt][a][c];
                }
    }
}

// ---- complex FP64 ---------------------------------------------------------------------------
// GB300 has two DFMA lanes per SM and clock, so the FP64 products run on the tensor cores, split into integer digits
// (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 2012).  With e the largest exponent of a coefficient row, and of
// a vector column, an entry x is the integer v = x 2^(1084 - e), |v| < 2^62, truncated below 1, in eight signed
// digits of 8 bits.  Products of digits i + j <= 7 are summed by mma.sync m16n8k16 (FP16 digits, FP32 sums): every sum of
// 64 entries stays within 2^24 and is exact, and goes into 64-bit integers.  So a result is the exact sum of
// truncated integers, in any order and at any width.  Its error per term, relative to 2^(sum of the two exponents), is
// 2^-58.8 at most (the digit products left out, at most 2^64.8 of 2^124, and the two truncations) and about 2^-62 as a rule,
// whatever the term's own size.
// That is FP64's accuracy or better where row and column do not both hold terms far below their largest entries.
// Two things see to that.  The exponents are local: a CTA takes them from the rows and the piece of the
// contraction that it sums, and what multiplies different vectors (t, s, u in the far field, u in the near field) is summed
// apart (FarPlan::zsegs), so that neither the scale of U against V nor that of one table against another matters.
// And a result below OZ_MIN of row maximum x column maximum is computed again with FP64 FMAs, a warp per output
// (OzAgain): for it the bound, 2 K 2^-58.8 for the K complex terms, may lie above that of FMAs, 2 K 2^-53 sum |a x|, for
// whose sum the result itself stands in.  At OZ_MIN = 2^-5.75 the two meet.  Of the outputs of a sphere and a plate, with
// random vectors, plane waves and solutions, that is 0.1% to 0.5%.
constexpr double OZ_MIN = 5.5e18;   // 2^62.25 of 2^68 units
constexpr int OZ_KC = 16, OZ_FOLD = 4;   // chunk = one step of the MMA; steps between foldings
constexpr int OZ_ROWS = 32;               // rows of a CTA

// |x| < 2^(e - 1022): bytes of the result less 128 are the signed digits of the modulus, the first in the highest byte
__device__ __forceinline__ uint2 oz_bytes(double x, int e)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t mh = hi & 0xfffff | 0x100000, a = __funnelshift_l(lo, mh, 9), b = lo << 9;
    const uint32_t r = (uint32_t)(e - (int)(hi >> 20 & 0x7ff));   // e >= 64: a zero is shifted out
    uint32_t l, h, l2;   // (a : b) >> r
    asm("shr.u32 %0, %1, %2;" : "=r"(h) : "r"(a), "r"(r));        // shifts of 32 and more give 0
    l = __funnelshift_rc(b, a, r);
    asm("shr.u32 %0, %1, %2;" : "=r"(l2) : "r"(l), "r"((uint32_t)max((int)r - 32, 0)));
    const uint64_t w = ((uint64_t)h << 32 | l2) + 0x8080808080808080ull;
    return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}
// digits i of two entries as a pair of FP16 numbers: 1024 + byte - 1152 with the entry's sign
__device__ __forceinline__ void oz_pair(double x0, double x1, int e, uint32_t (&d)[8])
{
    const uint2 w0 = oz_bytes(x0, e), w1 = oz_bytes(x1, e);
    const uint32_t sg = __byte_perm((uint32_t)__double2hiint(x0), (uint32_t)__double2hiint(x1), 0x7632) & 0x80008000u;
    const uint32_t one = sg | 0x3c003c00u, off = sg ^ 0xe480e480u;   // +-1, -+1152
#pragma unroll
    for (int i = 0; i < 8; i += 2) {   // bytes 3, 2 (1, 0) of both words, then each pair between bytes 0x64
        const uint32_t p = __byte_perm(i < 4 ? w0.y : w0.x, i < 4 ? w1.y : w1.x, i & 2 ? 0x4051 : 0x6273);
        const uint32_t q0 = __byte_perm(p, 0x64646464u, 0x4140), q1 = __byte_perm(p, 0x64646464u, 0x4342);
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d[i]) : "r"(q0), "r"(one), "r"(off));
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d[i + 1]) : "r"(q1), "r"(one), "r"(off));
    }
}
__device__ __forceinline__ void oz_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// A CTA takes 32 rows x NT column tiles of 8 right-hand sides, one warp per 16 x 8 outputs.  Per chunk of 16 contraction
// entries: the raw entries land in one of two buffers (cp.async), the warps turn them into digit fragments in
// shared memory, once for all warps that use them, and then each runs its 144 MMAs.  Up to four columns (NARROW) the real and
// the imaginary parts of the vectors share one tile, columns 0 .. 3 and 4 .. 7: 72 MMAs.  The integers of all forms are the
// same, so a column's bits do not depend on the width.
// Bound by latency and issue slots: 12 warps per SM issue in 40% of the cycles, the tensor pipe is a third busy, a pair of
// entries takes 47 instructions to split.  Z on 64 columns of the 30,720-unknown sphere, phases 1 + 2: DFMA 22.8 + 47.2 ms
// (its rate), with the digits in each warp's registers (225 of them, six warps per SM) 8.2 + 21.1, with one exponent
// for all of a row and a column, and so only for balanced factors, 4.6 + 13.1, now 5.0 + 15.6: four tables instead of two
// 1.3 ms, the columns' exponents 0.4, the outputs computed again 1.5.  One column: 0.46 + 1.43 by DFMA, 0.47 + 1.67 now; four:
// 1.53 + 3.44 and 0.51 + 1.79.  Error of Z x against products with 64-bit mantissas, of |Z| |x| per entry: 1.5e-16 to 3.6e-16;
// 2-norm, relative: 1.1e-16 to 1.3e-16, by FP64 FMAs 6e-16 to 1.1e-15.
template <bool NARROW> struct Oz {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int nct, ldr;                  // column tiles; row stride of the raw vector entries
    double2 *raw;                  // [2][OZ_KC * (ldw + ldr)]
    uint4 *ad;                     // [2 row tiles][2 parts][8 digits][32 lanes]
    uint4 *bd;                     // [nct][8][32]: real (two words), imaginary part
    int64_t *sum;                  // [nw][16][32]: of this lane, (part * 4 + output) * 2 + {high, low}
    float c[2][8][4];              // sums of digit products of weight i + j
    int steps = 0;
    static constexpr int ldw = OZ_ROWS | 1;
    static __host__ __device__ int tiles(int nrhs) { return NARROW ? 1 : (nrhs + 7) / 8; }
    static size_t smem(int nrhs)
    {
        const int nt = tiles(nrhs);
        return sizeof(double2) * 2 * OZ_KC * (size_t)(ldw + (nt * 8 | 1)) + (NARROW ? 8 * 32 * 8 : 16 * 32 * 8 * (size_t)(4 + nt)) + 8 * 16 * 32 * (size_t)(2 * nt);
    }
    __device__ __forceinline__ Oz(unsigned char *sm, int nrhs) : nct(tiles(nrhs)), ldr(nct * 8 | 1)
    {
        ad = (uint4 *)sm;
        bd = ad + (NARROW ? 0 : 4 * 8 * 32);
        sum = (int64_t *)(bd + nct * 8 * (NARROW ? 16 : 32));
        raw = (double2 *)(sum + nw * 16 * 32);
        sum += wp * 16 * 32 + lane;
        reset();
    }
    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int x = 0; x < 16; ++x) sum[32 * x] = 0;
        clear();
    }
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int z = 0; z < 2; ++z)
#pragma unroll
            for (int w = 0; w < 8; ++w)
#pragma unroll
                for (int x = 0; x < 4; ++x) c[z][w][x] = 0.f;
        steps = 0;
    }
    __device__ __forceinline__ double2 *ws(int ch) const { return raw + (ch & 1) * OZ_KC * (ldw + ldr); }
    __device__ __forceinline__ double2 *ys(int ch) const { return ws(ch) + OZ_KC * ldw; }
    __device__ __forceinline__ int row0() const { return NARROW ? 16 * wp : 16 * (wp / nct); }
    __device__ __forceinline__ int col0() const { return NARROW ? 0 : 8 * (wp % nct); }
    // digits of chunk ch: rows r < rows, exponents re(row) and ce(column)
    template <class RE, class CE> __device__ __forceinline__ void split(int ch, int rows, RE &&re, CE &&ce)
    {
        const int g = lane >> 2, k = 2 * (lane & 3);
        const double2 *Ws = ws(ch), *Ys = ys(ch);
        if constexpr (NARROW) {   // two warps, a word of the vector fragments (entries + 8 word) each; by column real or imaginary part
            uint32_t d[8];
            const double *y0 = (const double *)(Ys + (k + 8 * wp) * ldr + (g & 3)) + (g >> 2);
            oz_pair(y0[0], y0[2 * ldr], max(ce(g & 3), 64), d);
#pragma unroll
            for (int i = 0; i < 8; ++i) ((uint32_t *)bd)[(i * 32 + lane) * 2 + wp] = d[i];
        } else {   // 8 halves of coefficient fragments, then 2 of each column tile's, dealt out to the warps
            for (int x = wp; x < 8 + 2 * nct; x += nw) {
                uint32_t d[2][8];
                uint2 *dst;
                if (x < 8) {   // words q: rows + 8 q of entries + 8 (x & 1)
                    const int r = 16 * (x >> 2) + g;
                    if (r - g >= rows) continue;
                    const double *w0 = (const double *)(Ws + (k + 8 * (x & 1)) * ldw + r) + (x >> 1 & 1);
                    oz_pair(w0[0], w0[2 * ldw], max(re(r), 64), d[0]);
                    oz_pair(w0[16], w0[2 * ldw + 16], max(re(r + 8), 64), d[1]);
                    dst = (uint2 *)(ad + (x >> 1) * 8 * 32 + lane) + (x & 1);
                } else {   // words q: entries + 8 q of one part
                    const int t = x - 8 >> 1, part = x & 1, e = max(ce(8 * t + g), 64);
                    const double *y0 = (const double *)(Ys + k * ldr + 8 * t + g) + part;
                    oz_pair(y0[0], y0[2 * ldr], e, d[0]);
                    oz_pair(y0[16 * ldr], y0[18 * ldr], e, d[1]);
                    dst = (uint2 *)(bd + t * 8 * 32 + lane) + part;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) dst[64 * i] = make_uint2(d[0][i], d[1][i]);
            }
        }
    }
    // NARROW: a warp is alone with its rows and splits them into its registers
    template <class RE> __device__ __forceinline__ void multiply_own(int ch, RE &&re)
    {
        const int g = lane >> 2, k = 2 * (lane & 3);
        const uint2 *B = (const uint2 *)bd + lane;
        uint32_t b[8][2];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint2 v = B[32 * j];
            b[j][0] = v.x;
            b[j][1] = v.y;
        }
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            uint32_t d[4][8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = row0() + g + 8 * (q & 1);
                const double *w0 = (const double *)(ws(ch) + (k + 8 * (q >> 1)) * ldw + r) + part;
                oz_pair(w0[0], w0[2 * ldw], max(re(r), 64), d[q]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t a[4] = {d[0][i], d[1][i], d[2][i], d[3][i]};
#pragma unroll
                for (int j = 0; j < 8 - i; ++j) oz_mma(c[part][i + j], a, b[j][0], b[j][1]);
            }
        }
        if (++steps == OZ_FOLD) fold();
    }
    __device__ __forceinline__ void multiply()
    {
        const uint4 *B = bd + wp % nct * 8 * 32 + lane, *A = ad + (row0() >> 4) * 2 * 8 * 32 + lane;
        uint4 b[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) b[j] = B[32 * j];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 vr = A[32 * i], vi = A[32 * (8 + i)];
            const uint32_t ar[4] = {vr.x, vr.y, vr.z, vr.w}, ai[4] = {vi.x, vi.y, vi.z, vi.w};
            const uint32_t an[4] = {ai[0] ^ 0x80008000u, ai[1] ^ 0x80008000u, ai[2] ^ 0x80008000u, ai[3] ^ 0x80008000u};
#pragma unroll
            for (int j = 0; j < 8 - i; ++j) {
                oz_mma(c[0][i + j], ar, b[j].x, b[j].y);
                oz_mma(c[1][i + j], ar, b[j].z, b[j].w);
                oz_mma(c[0][i + j], an, b[j].z, b[j].w);
                oz_mma(c[1][i + j], ai, b[j].x, b[j].y);
            }
        }
        if (++steps == OZ_FOLD) fold();
    }
    __device__ __forceinline__ void fold()
    {
#pragma unroll
        for (int z = 0; z < 2; ++z)
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                int64_t h = sum[32 * (8 * z + 2 * x)], l = sum[32 * (8 * z + 2 * x + 1)];
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    h += (int64_t)__float2int_rn(c[z][w][x]) * (1 << 8 * (3 - w));
                    l += (int64_t)__float2int_rn(c[z][4 + w][x]) * (1 << 8 * (3 - w));
                }
                sum[32 * (8 * z + 2 * x)] = h;
                sum[32 * (8 * z + 2 * x + 1)] = l;
            }
        clear();
    }
    // the chunks 0 .. nch - 1 that stage(c) copies (one commit each, also past the end); every thread calls it
    template <class Stage, class RE, class CE>
    __device__ __forceinline__ void run(int nch, int rows, Stage &&stage, RE &&re, CE &&ce)
    {
        stage(0);
        stage(1);
        for (int ch = 0; ch < nch; ++ch) {
            if (NARROW && ch) asm volatile("cp.async.wait_group 0;\n" ::: "memory");   // its stage was the last one
            else asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            __syncthreads();   // chunk ch has landed, the digits of the one before are consumed
            split(ch, rows, re, ce);
            __syncthreads();   // its raw buffer is free, the digits are there
            if (NARROW) {   // the raw coefficients are still read: the next barrier frees them
                if (ch) stage(ch + 1);
                if (row0() < rows) multiply_own(ch, re);
            } else {
                stage(ch + 2);
                if (row0() < rows) multiply();
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
    }
    // put(row, column, value, again) for the outputs of the warp (rows, columns of the CTA); whole warps call it.  re, ce:
    // largest exponents of the row and the column, 0 with nothing but zeros; again: the value is to be computed by FP64 FMAs
    template <class RE, class CE, class Put>
    __device__ __forceinline__ void store(int rows, int nrhs, RE &&re, CE &&ce, Put &&put)
    {
        if (row0() >= rows) return;
        fold();
#pragma unroll 1
        for (int x = 0; x < 4; ++x) {
            const int row = row0() + (lane >> 2) + 8 * (x >> 1), col = col0() + 2 * (lane & 3) + (x & 1);
            int64_t v[2][2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                v[0][p] = sum[32 * (2 * x + p)];
                v[1][p] = sum[32 * (8 + 2 * x + p)];
                if (NARROW) {   // real x real, real x imaginary two lanes on; imaginary x the same
                    const int64_t r2 = __shfl_down_sync(0xffffffffu, v[0][p], 2), i2 = __shfl_down_sync(0xffffffffu, v[1][p], 2);
                    v[0][p] -= i2;
                    v[1][p] += r2;
                }
            }
            const bool ok = row < rows && col < nrhs && (!NARROW || (lane & 3) < 2);
            double2 y = make_double2(0.0, 0.0);
            bool again = false;
            if (ok) {
                const int ra = re(row), rb = ce(col), e = max(ra, 64) + max(rb, 64) - 2112, eh = e / 2;
                y.x = fma((double)v[0][0], 4294967296.0, (double)v[0][1]);
                y.y = fma((double)v[1][0], 4294967296.0, (double)v[1][1]);
                again = ra && rb && (fmax(fabs(y.x), fabs(y.y)) < OZ_MIN || ra == 0x7ff || rb == 0x7ff);
                // in two steps: 2^e alone may be below the smallest power of two
                const double s0 = __hiloint2double(eh + 1023 << 20, 0), s1 = __hiloint2double(e - eh + 1023 << 20, 0);
                y.x = y.x * s0 * s1;
                y.y = y.y * s0 * s1;
            }
            if (ok) put(row, col, y, again);
        }
    }
};
// the largest exponent of entries: 0 for zeros alone
__device__ __forceinline__ int oz_exp(double2 v)
{
    const int hx = __double2hiint(v.x) & 0x7fffffff, hy = __double2hiint(v.y) & 0x7fffffff;
    const int e = max(hx, hy) >> 20;
    return e ? e : (hx | hy | __double2loint(v.x) | __double2loint(v.y)) != 0;   // 1: nothing but subnormals
}
// A CTA's outputs to be computed again, row * 16 + column, dealt out to the warps at its end (a warp that
// did so at once held up the others: phase 2 of 64 columns of the 30,720-unknown sphere 17.3 ms for 16.5)
struct OzAgain {
    int n;
    uint16_t list[OZ_ROWS * 16];
    uint8_t tabs[OZ_ROWS * 16];   // phase 2: the tables concerned, a bit each
};
__device__ __forceinline__ double2 warp_sum(double2 v)
{
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// Column exponents of pieces of the vectors.  The kernels that write u, t and s also write their entries' exponents, 16 per
// row, so that a piece is 32 bytes a row to look at instead of 256: eight columns per thread (four when NARROW).
constexpr int VEXP = 16;
template <bool NARROW> struct OzCols {
    static constexpr int HV = NARROW ? 1 : 2;   // threads abreast over a row
    uint4 m = make_uint4(0, 0, 0, 0);           // pairs of columns
    __device__ __forceinline__ void row(const uint16_t *e)
    {
        if (NARROW) {
            const uint2 v = *(const uint2 *)e;
            m.x = __vmaxu2(m.x, v.x);
            m.y = __vmaxu2(m.y, v.y);
        } else {
            const uint4 v = *(const uint4 *)(e + 8 * (threadIdx.x & 1));
            m.x = __vmaxu2(m.x, v.x);
            m.y = __vmaxu2(m.y, v.y);
            m.z = __vmaxu2(m.z, v.z);
            m.w = __vmaxu2(m.w, v.w);
        }
    }
    __device__ __forceinline__ void max_into(int *s_ce)   // whole warps
    {
        uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
        for (int i = 0; i < (NARROW ? 2 : 4); ++i) {
#pragma unroll
            for (int o = HV; o < 32; o <<= 1) w[i] = __vmaxu2(w[i], __shfl_xor_sync(0xffffffffu, w[i], o));
            if ((threadIdx.x & 31) < HV) {
                atomicMax(&s_ce[8 * (threadIdx.x & 1) + 2 * i], (int)(w[i] & 0xffff));
                atomicMax(&s_ce[8 * (threadIdx.x & 1) + 2 * i + 1], (int)(w[i] >> 16));
            }
        }
    }
};

// a staged vector entry, zero past the contraction's end
__device__ __forceinline__ void oz_cp(double2 *dst, const double2 *src, bool ok)
{
    if (ok) far_cp(dst, src);
    else *dst = make_double2(0.0, 0.0);
}

// phase 1, tasks as in k_far_t, blockIdx.y: which 32 of its factor columns; rexp: exponents of the factor columns, of V
// (tlen), then of U; vexp: of the entries of t, s (written) and u (read)
template <bool NARROW>
__global__ void __launch_bounds__(NARROW ? 64 : 128, NARROW ? 6 : 3) k_far_t64(const int *task_lo, const int *task_hi, const int *task_ptr,
                                                    const int64_t *item_off, const int *item_ld, const int *item_rank,
                                                    const int *item_row, const int *item_isv, const double2 *U,
                                                    const double2 *V, const double2 *u, int nrhs, double2 *t, double2 *s,
                                                    const uint16_t *rexp, uint16_t *vexp, int64_t tlen)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_item[64], s_l[64], s_re[OZ_ROWS], s_ce[16];
    __shared__ const double2 *s_src[64];
    __shared__ OzAgain s_ag;
    const int task = blockIdx.x, f0 = OZ_ROWS * blockIdx.y;
    const int lo = task_lo[task], hi = task_hi[task], i0 = task_ptr[task], i1 = task_ptr[task + 1];
    const int R = far_items(i0, i1, item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src) - f0;
    if (R <= 0) return;
    const int rows = min(R, OZ_ROWS);
    auto dest = [&](int row) {
        const int it = s_item[f0 + row];
        return (item_isv[it] ? 0 : tlen) + item_row[it] + s_l[f0 + row];
    };
    if (threadIdx.x == 0) s_ag.n = 0;
    if (threadIdx.x < 16) s_ce[threadIdx.x] = 0;
    if (threadIdx.x < OZ_ROWS) s_re[threadIdx.x] = threadIdx.x < rows ? rexp[dest(threadIdx.x)] : 0;
    Oz<NARROW> oz(smraw, nrhs);
    __syncthreads();
    {   // the columns' exponents over the task's rows
        OzCols<NARROW> cm;
#pragma unroll 4
        for (int q = lo + threadIdx.x / cm.HV; q < hi; q += blockDim.x / cm.HV) cm.row(vexp + (2 * tlen + q) * VEXP);
        cm.max_into(s_ce);
    }
    const int nch = (hi - lo + OZ_KC - 1) / OZ_KC;
    auto stage = [&](int c) {   // factor column rr of row c0 + qq, half a warp each; then the vector rows
        if (c < nch) {
            const int c0 = lo + c * OZ_KC, ch = min(OZ_KC, hi - c0), qh = oz.lane & 15;
            double2 *Ws = oz.ws(c), *Ys = oz.ys(c);
            if (qh < ch)
                for (int rr = 2 * oz.wp + (oz.lane >> 4); rr < rows; rr += 2 * oz.nw)
                    far_cp(Ws + qh * oz.ldw + rr, s_src[f0 + rr] + (c0 - lo + qh));
            const double2 *uc = u + (int64_t)c0 * nrhs;
            if (NARROW) {
                const int qq = threadIdx.x >> 2, r = threadIdx.x & 3;   // 64 threads, 16 rows of at most 4
                if (r < nrhs) oz_cp(Ys + qq * oz.ldr + r, uc + qq * nrhs + r, qq < ch);
            } else
                for (int qq = oz.wp; qq < OZ_KC; qq += oz.nw)
                    if (oz.lane < nrhs) oz_cp(Ys + qq * oz.ldr + oz.lane, uc + qq * nrhs + oz.lane, qq < ch);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    auto re = [&](int row) { return s_re[row]; };
    auto ce = [&](int col) { return s_ce[col]; };
    oz.run(nch, rows, stage, re, ce);
    auto put = [&](int row, int col, double2 v) {
        const int64_t d = dest(row);
        (d < tlen ? t + d * nrhs : s + (d - tlen) * nrhs)[col] = v;
        vexp[d * VEXP + col] = (uint16_t)oz_exp(v);
    };
    oz.store(rows, nrhs, re, ce, [&](int row, int col, double2 v, bool again) {
        if (again) s_ag.list[atomicAdd(&s_ag.n, 1)] = (uint16_t)(row * 16 + col);
        else put(row, col, v);
    });
    __syncthreads();
    for (int x = oz.wp; x < s_ag.n; x += oz.nw) {   // a lane per row of the range, in turn
        const int row = s_ag.list[x] >> 4, col = s_ag.list[x] & 15;
        const double2 *f = s_src[f0 + row];
        double2 v = make_double2(0.0, 0.0);
#pragma unroll 8
        for (int q = oz.lane; q < hi - lo; q += 32) v = cfma(f[q], u[(int64_t)(lo + q) * nrhs + col], v);
        v = warp_sum(v);
        if (oz.lane == 0) put(row, col, v);
    }
}

// exponents of the factor columns (see k_far_t64): task as there, one warp per factor column
__global__ void k_far_rexp1(const int *task_lo, const int *task_hi, const int *task_ptr, const int64_t *item_off,
                            const int *item_ld, const int *item_rank, const int *item_row, const int *item_isv,
                            const double2 *U, const double2 *V, uint16_t *rexp, int64_t tlen)
{
    __shared__ int s_item[64], s_l[64];
    __shared__ const double2 *s_src[64];
    const int task = blockIdx.x, lane = threadIdx.x & 31;
    const int R = far_items(task_ptr[task], task_ptr[task + 1], item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src);
    for (int rr = threadIdx.x >> 5; rr < R; rr += blockDim.x >> 5) {
        int e = 0;
        for (int q = lane; q < task_hi[task] - task_lo[task]; q += 32) e = max(e, oz_exp(s_src[rr][q]));
        e = __reduce_max_sync(0xffffffffu, e);
        const int it = s_item[rr];
        if (lane == 0) rexp[(item_isv[it] ? 0 : tlen) + item_row[it] + s_l[rr]] = (uint16_t)e;
    }
}
// exponents of the coefficient rows of one part (blockIdx.x, see FarPlan::zpart) of a leaf in one table (blockIdx.y):
// rexp[(table * FAR_PARTS + part) * n + row]
__global__ void k_far_rexp2(int nl, int n, const int *leaf_ptr, const int *zpart, const FarSegD *segs, const double2 *U,
                            const double2 *V, const double2 *nearp, uint16_t *rexp)
{
    __shared__ int s_e[64];
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS, tab = blockIdx.y;
    const int a = leaf_ptr[l], ni = leaf_ptr[l + 1] - a, i = threadIdx.x & 63;
    const int *pt = zpart + tab * (nl * FAR_PARTS + 1) + blockIdx.x;
    if (threadIdx.x < 64) s_e[threadIdx.x] = 0;
    __syncthreads();
    int e = 0;
    for (int q = pt[0]; q < pt[1] && i < ni; ++q) {
        const FarSegD g = segs[q];
        const double2 *F = (tab == FAR_TABS - 1 ? nearp : (g.src & 1) ? V : U) + g.foff + (int64_t)i * g.fi;
        for (int kk = threadIdx.x >> 6; kk < g.len; kk += blockDim.x >> 6) e = max(e, oz_exp(F[(int64_t)kk * g.fk]));
    }
    atomicMax(&s_e[i], e);
    __syncthreads();
    if (threadIdx.x < ni) rexp[(int64_t)(tab * FAR_PARTS + pp) * n + a + threadIdx.x] = (uint16_t)s_e[threadIdx.x];
}
// u[i * nrhs + r] = x[idx[i] + r * n], its exponent; bit r of *bad (zero before): an infinity or a NaN in column r
__global__ void k_far_gather64(int n, int nrhs, const int *idx, const double2 *x, double2 *u, uint16_t *uexp, int *bad)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * nrhs) return;
    const int i = (int)(e / nrhs), r = (int)(e - (int64_t)i * nrhs);
    const double2 v = x[idx[i] + (int64_t)r * n];
    const int ex = oz_exp(v);
    u[e] = v;
    uexp[(int64_t)i * VEXP + r] = (uint16_t)ex;
    if (ex == 0x7ff) atomicOr(bad, 1 << r);
}

// Phase 2: one CTA per leaf over the leaf's segments (FarSegD, list order, len <= 32).
// Consecutive segments form a chunk while their summed length fits half the staging buffer;
// the chunk's coefficient rows and vector rows are stacked into one contraction, so a
// single tile product per chunk keeps every output's order (segment by segment, k
// ascending).  Chunks are copied with cp.async by one warp per segment into the two halves
// of the buffer in turn, so the copy of the next chunk overlaps the product of the current.
template <class T> __device__ __forceinline__ void cp_async_el(T *dst, const T *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

template <class T, int TR, int TC, int NT>
__global__ void __launch_bounds__(256) k_far_y(int nl, const int *leaf_ptr, const int *part_ptr, const int *kcum,
                                               const FarSegD *segs, const T *U, const T *V, const T *t, const T *s,
                                               const T *u, const int *cl2new, int n, int nrhs, T *part, int budget)
{
    extern __shared__ unsigned char smraw[];
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS;
    if (l >= nl) return;
    const int a = leaf_ptr[l], ni = leaf_ptr[l + 1] - a;
    const int nrt = (ni + TR - 1) / TR, ntiles = nrt * ((nrhs + TC - 1) / TC);
    const int ldw = stage_ldw(ni, TR), ldr = stage_ldr(nrhs, TC);
    const int half = budget / 2, kmax = half / (ldw + ldr);   // >= 32 for ni <= 64
    T *const bufs[2] = {(T *)smraw, (T *)smraw + half};
    Tile<T, TR, TC, NT> acc;
    tile_load(acc, (const T *)nullptr, 0, 0, ni, nrhs, nrt, ntiles);
    const int w1 = part_ptr[blockIdx.x + 1];
    // segments [p, p + count) of the chunk starting at p: those whose stacked length fits kmax
    auto chunk_count = [&](int p) {
        const int q = p + threadIdx.x;
        const bool fit = q < w1 && kcum[q + 1] - kcum[p] <= kmax;
        return __syncthreads_count(fit);
    };
    // the chunk's stacked contraction rows kk = 0 .. klen-1 (segment q's rows kcum[p+q] - k0 ..)
    // copied by all threads: entry e of the coefficient rows is (kk, i) = (e / ni, e % ni), of
    // the vector rows (e / nrhs, e % nrhs); a thread's kk only grows, so it follows the segments
    // in order and reloads a segment's descriptor when it moves to the next
    auto stage = [&](int p, int cnt, T *buf) {
        const int k0 = kcum[p], klen = kcum[p + cnt] - k0;
        T *Wst = buf, *Yst = buf + kmax * ldw;
        int q = -1, qlo = 0, qhi = 0;
        const T *F = nullptr;
        int64_t fi = 0, fk = 0;
        for (int e = threadIdx.x; e < klen * ni; e += blockDim.x) {
            const int kk = e / ni, i = e - kk * ni;
            while (kk >= qhi) {
                ++q;
                qlo = kcum[p + q] - k0;
                qhi = kcum[p + q + 1] - k0;
                const FarSegD g = segs[p + q];
                F = ((g.src & 1) ? V : U) + g.foff;
                fi = g.fi;
                fk = g.fk;
            }
            cp_async_el(Wst + kk * ldw + i, F + (int64_t)i * fi + (int64_t)(kk - qlo) * fk);
        }
        q = -1;
        qhi = 0;
        const T *Yb = nullptr;
        for (int e = threadIdx.x; e < klen * nrhs; e += blockDim.x) {
            const int kk = e / nrhs, r = e - kk * nrhs;
            while (kk >= qhi) {
                ++q;
                qlo = kcum[p + q] - k0;
                qhi = kcum[p + q + 1] - k0;
                const FarSegD g = segs[p + q];
                const int ys = g.src >> 1;
                Yb = (ys == 0 ? t : (ys == 1 ? s : u)) + g.yrow * nrhs;
            }
            cp_async_el(Yst + kk * ldr + r, Yb + (int64_t)(kk - qlo) * nrhs + r);
        }
        cp_async_commit();
        return klen;
    };
    int p = part_ptr[blockIdx.x];
    if (p < w1) {
        int cnt = chunk_count(p), klen = stage(p, cnt, bufs[0]);
        for (int it = 0;; ++it) {
            const int pn = p + cnt;
            int cntn = 0, klenn = 0;
            if (pn < w1) {
                cntn = chunk_count(pn);
                klenn = stage(pn, cntn, bufs[(it + 1) & 1]);
                cp_async_wait<1>();
            } else
                cp_async_wait<0>();
            __syncthreads();
            T *buf = bufs[it & 1];
            tile_mac<false>(acc, buf, ldw, buf + kmax * ldw, ldr, 1, klen, nrt, ntiles);
            __syncthreads();
            if (pn >= w1) break;
            p = pn;
            cnt = cntn;
            klen = klenn;
        }
    }
    tile_store(acc, part + (size_t)pp * n * nrhs + cl2new[a], 1, n, ni, nrhs, nrt, ntiles);
}

// ---- complex FP32, more than 16 columns ----------------------------------------------------
// The same two phases for wide batches.  A warp owns a patch of 16 rows x 32 columns, a lane 4 x 4 outputs of it: rows
// 2 (l % 4) + {0, 1, 8, 9} and columns 4 (l / 4) + {0 .. 3}, so that a contraction step is four conflict-free 16-byte
// shared-memory loads for 64 FMAs; the CTA has as many warps as the block has patches.  Staging goes one contraction row
// (or factor column) per warp turn, without divisions, the vector rows in 16-byte words when nrhs is even.
// Issue slots bound it: 2 x 4 outputs per lane of a 256-thread CTA with element-wise staging spent as many on addresses
// and loads as on FMAs (64 columns of the 30,720-unknown sphere: 1.04 + 1.98 ms, now
// 0.68 + 1.52; 23 columns of a 22,500-unknown plate: 0.25 + 0.42, now 0.24 + 0.29).  A ring of four chunks leaves fewer CTAs
// per SM (phase 2 of 23 columns 0.95 -> 1.11 ms), patches of 32 rows waste more of the 28-row leaves (1.64 for 1.52).
constexpr int F32_ROWS = 16, F32_COLS = 32;   // patch of a warp
constexpr int F32_KC = 16, F32_RING = 3;      // contraction entries of a chunk, chunks in shared memory
__host__ __device__ __forceinline__ int f32_np(int no) { return (no + F32_ROWS - 1) / F32_ROWS; }
__host__ __device__ __forceinline__ int f32_nc(int nrhs) { return (nrhs + F32_COLS - 1) / F32_COLS; }
// row strides of the staged blocks: whole patches; even, for 16-byte loads
__host__ __device__ __forceinline__ int f32_ldw(int np) { return np * F32_ROWS + 2; }

__device__ __forceinline__ void far_cp16(float2 *dst, const float2 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// one vector row of nrhs <= 64 entries; v16: nrhs is even and the vectors start on 16 bytes, so every row does
__device__ __forceinline__ void f32_row(float2 *dst, const float2 *src, int nrhs, bool v16)
{
    const int lane = threadIdx.x & 31;
    if (v16) {
        if (2 * lane < nrhs) far_cp16(dst + 2 * lane, src + 2 * lane);
    } else
        for (int r = lane; r < nrhs; r += 32) far_cp(dst + r, src + r);
}
// acc += the staged step, terms in ascending order (the order of tile_mac)
__device__ __forceinline__ void f32_mac(float2 (&acc)[4][4], const float2 *wp, int ldw, const float2 *yp, int ldr, int nc)
{
#pragma unroll 2
    for (int q = 0; q < nc; ++q, wp += ldw, yp += ldr) {
        const float4 w0 = *(const float4 *)wp, w1 = *(const float4 *)(wp + 8), y0 = *(const float4 *)yp,
                     y1 = *(const float4 *)(yp + 2);
        const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                             make_float2(w1.z, w1.w)};
        const float2 y[4] = {make_float2(y0.x, y0.y), make_float2(y0.z, y0.w), make_float2(y1.x, y1.y),
                             make_float2(y1.z, y1.w)};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] = cfma(w[a], y[c], acc[a][c]);
    }
}

__global__ void __launch_bounds__(256) k_far_t32(const int *task_lo, const int *task_hi, const int *task_ptr,
                                                 const int64_t *item_off, const int *item_ld, const int *item_rank,
                                                 const int *item_row, const int *item_isv, const float2 *U, const float2 *V,
                                                 const float2 *u, int nrhs, float2 *t, float2 *s, bool v16)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_item[64], s_l[64];
    __shared__ const float2 *s_src[64];
    const int task = blockIdx.x;
    const int lo = task_lo[task], hi = task_hi[task], i0 = task_ptr[task], i1 = task_ptr[task + 1];
    const int R = far_items(i0, i1, item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ncol = f32_nc(nrhs), ldw = f32_ldw(4), ldr = ncol * F32_COLS;
    const int prow = wp / ncol, row0 = prow * F32_ROWS + 2 * (lane & 3), col0 = wp % ncol * F32_COLS + 4 * (lane >> 2);
    float2 *const ring = (float2 *)smraw;
    float2 acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = make_float2(0.f, 0.f);
    const int nch = (hi - lo + F32_KC - 1) / F32_KC;
    // chunk c: Ws[qq * ldw + rr], then Ys[qq * ldr + r]; half a warp per factor column
    auto stage = [&](int c) {
        const int c0 = lo + c * F32_KC, ch = min(F32_KC, hi - c0), qh = lane & 15;
        float2 *Ws = ring + c % F32_RING * F32_KC * (ldw + ldr), *Ys = Ws + F32_KC * ldw;
        if (c < nch) {
            if (qh < ch)
                for (int rr = 2 * wp + (lane >> 4); rr < R; rr += 2 * nw) far_cp(Ws + qh * ldw + rr, s_src[rr] + (c0 - lo + qh));
            for (int qq = wp; qq < ch; qq += nw) f32_row(Ys + qq * ldr, u + (int64_t)(c0 + qq) * nrhs, nrhs, v16);
        }
        cp_async_commit();
    };
    stage(0);
    stage(1);
    for (int c = 0; c < nch; ++c) {
        cp_async_wait<1>();
        __syncthreads();   // chunk c has landed, chunk c - 1 is consumed
        stage(c + 2);
        const float2 *Ws = ring + c % F32_RING * F32_KC * (ldw + ldr);
        if (prow * F32_ROWS < R)
            f32_mac(acc, Ws + row0, ldw, Ws + F32_KC * ldw + col0, ldr, min(F32_KC, hi - lo - c * F32_KC));
    }
    cp_async_wait<0>();
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int row = row0 + (a & 1) + 8 * (a >> 1);
        if (row >= R) continue;
        const int it = s_item[row];
        float2 *dst = (item_isv[it] ? t : s) + (int64_t)(item_row[it] + s_l[row]) * nrhs;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (col0 + c < nrhs) dst[col0 + c] = acc[a][c];
    }
}

// phase 2 (see k_far_y); np: patches that cover the rows of the largest leaf
__global__ void __launch_bounds__(256) k_far_y32(int nl, const int *leaf_ptr, const int *part_ptr, const int *kcum,
                                                 const FarSegD *segs, const float2 *U, const float2 *V, const float2 *t,
                                                 const float2 *s, const float2 *u, const int *cl2new, int n, int nrhs,
                                                 float2 *part, int np, bool v16)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS;
    if (l >= nl) return;
    const int a0 = leaf_ptr[l], ni = leaf_ptr[l + 1] - a0;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ncol = f32_nc(nrhs), ldw = f32_ldw(np), ldr = ncol * F32_COLS;
    const int prow = wp / ncol, row0 = prow * F32_ROWS + 2 * (lane & 3), col0 = wp % ncol * F32_COLS + 4 * (lane >> 2);
    float2 *const ring = (float2 *)smraw;
    float2 acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = make_float2(0.f, 0.f);
    const int p0 = part_ptr[blockIdx.x], w1 = part_ptr[blockIdx.x + 1];
    const int k0 = p0 < w1 ? kcum[p0] : 0, K = p0 < w1 ? kcum[w1] - k0 : 0, nch = (K + F32_KC - 1) / F32_KC;
    // the part's stacked contraction entries, one per warp turn; a warp follows the segments in order, with the next
    // segment's descriptor on its way
    int q = p0, qlo = 0, qhi = 0;
    FarSegD g = {}, gn = {};
    int hn = 0;   // end of the next segment
    if (K > 0) {
        gn = segs[p0];
        hn = kcum[p0 + 1] - k0;
    }
    const float2 *F = nullptr, *Yb = nullptr;
    auto stage = [&](int c) {
        float2 *Ws = ring + c % F32_RING * F32_KC * (ldw + ldr), *Ys = Ws + F32_KC * ldw;
        const int ke = min(K, (c + 1) * F32_KC);
        for (int kk = c * F32_KC + wp; kk < ke; kk += nw) {
            while (kk >= qhi) {
                g = gn;
                qlo = qhi;
                qhi = hn;
                ++q;
                if (q < w1) {
                    gn = segs[q];
                    hn = kcum[q + 1] - k0;
                }
                F = ((g.src & 1) ? V : U) + g.foff;
                const int ys = g.src >> 1;
                Yb = (ys == 0 ? t : (ys == 1 ? s : u)) + g.yrow * nrhs;
            }
            const float2 *f = F + (int64_t)(kk - qlo) * g.fk;
            const int o = kk - c * F32_KC;
            for (int i = lane; i < ni; i += 32) far_cp(Ws + o * ldw + i, f + (int64_t)i * g.fi);
            f32_row(Ys + o * ldr, Yb + (int64_t)(kk - qlo) * nrhs, nrhs, v16);
        }
        cp_async_commit();
    };
    stage(0);
    stage(1);
    for (int c = 0; c < nch; ++c) {
        cp_async_wait<1>();
        __syncthreads();   // chunk c has landed, chunk c - 1 is consumed
        stage(c + 2);
        const float2 *Ws = ring + c % F32_RING * F32_KC * (ldw + ldr);
        if (prow * F32_ROWS < ni) f32_mac(acc, Ws + row0, ldw, Ws + F32_KC * ldw + col0, ldr, min(F32_KC, K - c * F32_KC));
    }
    cp_async_wait<0>();
    float2 *out = part + (size_t)pp * n * nrhs + cl2new[a0];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int row = row0 + (a & 1) + 8 * (a >> 1);
            if (row < ni && col0 + c < nrhs) out[row + (int64_t)(col0 + c) * n] = acc[a][c];
        }
}

// complex FP64, phase 2: the segments of the tables of the far field and, with nearp, those of the leaf's near-field
// blocks, which gives Z u in one pass, the tables added in their order; blockIdx.y: which 32 of the leaf's rows; rexp: see
// k_far_rexp2; vexp: see k_far_t64
template <bool NARROW>
__global__ void __launch_bounds__(NARROW ? 64 : 128, NARROW ? 6 : 3) k_far_y64(int nl, const int *leaf_ptr, const int *zpart,
                                                    const int *kc, const FarSegD *sg, const double2 *U, const double2 *V,
                                                    const double2 *nearp, const double2 *t, const double2 *s,
                                                    const double2 *u, const int *cl2new, int n, int nrhs, double2 *part,
                                                    const uint16_t *rexp, const uint16_t *vexp, int64_t tlen)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_re[OZ_ROWS], s_ce[16];
    __shared__ OzAgain s_ag;
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS;
    if (l >= nl) return;
    const int r0 = OZ_ROWS * blockIdx.y, a = leaf_ptr[l] + r0, rows = min(leaf_ptr[l + 1] - a, OZ_ROWS);
    if (rows <= 0) return;
    double2 *out = part + (size_t)pp * n * nrhs + cl2new[leaf_ptr[l]] + r0;
    Oz<NARROW> oz(smraw, nrhs);
    auto re = [&](int row) { return s_re[row]; };
    auto ce = [&](int col) { return s_ce[col]; };
    if (threadIdx.x == 0) s_ag.n = 0;
    for (int x = threadIdx.x; x < OZ_ROWS * 16; x += blockDim.x) s_ag.tabs[x] = 0;
    bool first = true;
    for (int tab = 0; tab < (nearp ? FAR_TABS : FAR_TABS - 1); ++tab) {
        const int *pt = zpart + tab * (nl * FAR_PARTS + 1) + blockIdx.x;
        const int p0 = pt[0], w1 = pt[1];
        if (p0 >= w1) continue;
        const int k0 = kc[p0], K = kc[w1] - k0, nch = (K + OZ_KC - 1) / OZ_KC;
        const double2 *F0 = tab == FAR_TABS - 1 ? nearp : U, *F1 = tab == FAR_TABS - 1 ? nearp : V;
        const double2 *Y = tab == 0 ? t : tab == 1 ? s : u;
        if (threadIdx.x < OZ_ROWS)
            s_re[threadIdx.x] = threadIdx.x < rows ? rexp[(int64_t)(tab * FAR_PARTS + pp) * n + a + threadIdx.x] : 0;
        if (threadIdx.x < 16) s_ce[threadIdx.x] = 0;
        __syncthreads();
        {   // the columns' exponents over the part, eight rows of a segment side by side
            const uint16_t *ve = vexp + (tab == 0 ? 0 : tab == 1 ? tlen : 2 * tlen) * VEXP;
            OzCols<NARROW> cm;
            for (int q = p0 + threadIdx.x / (8 * cm.HV); q < w1; q += blockDim.x / (8 * cm.HV)) {
                const int64_t y0 = sg[q].yrow;
                const int len = sg[q].len;
                for (int kk = threadIdx.x / cm.HV & 7; kk < len; kk += 8) cm.row(ve + (y0 + kk) * VEXP);
            }
            cm.max_into(s_ce);
        }
        // lane o and o + 16 of every warp follow contraction entry o of the chunks through the segments, with the next
        // segment's descriptor on its way
        int q = p0, qlo = 0, qhi = 0, hn = kc[p0 + 1] - k0;
        FarSegD gn = sg[p0];
        const double2 *F = nullptr, *Yb = nullptr;
        int fi = 0, fk = 0;
        auto stage = [&](int c) {
            if (c < nch) {
                double2 *Ws = oz.ws(c), *Ys = oz.ys(c);
                const int o = oz.lane & 15, kk = c * OZ_KC + o;
                while (kk < K && kk >= qhi) {
                    F = ((gn.src & 1) ? F1 : F0) + gn.foff + (int64_t)r0 * gn.fi;
                    Yb = Y + gn.yrow * nrhs;
                    fi = gn.fi;
                    fk = gn.fk;
                    qlo = qhi;
                    qhi = hn;
                    if (++q < w1) {
                        gn = sg[q];
                        hn = kc[q + 1] - k0;
                    }
                }
                const bool in = kk < K;
                const uint64_t f = in ? (uint64_t)(F + (int64_t)(kk - qlo) * fk) : 0, y = (uint64_t)(Yb + (int64_t)(kk - qlo) * nrhs);
#pragma unroll 4
                for (int x = oz.wp; x < OZ_KC; x += oz.nw) {
                    const double2 *fx = (const double2 *)__shfl_sync(0xffffffffu, f, x);
                    const int fix = __shfl_sync(0xffffffffu, fi, x);
                    if (fx && oz.lane < rows) far_cp(Ws + x * oz.ldw + oz.lane, fx + (int64_t)oz.lane * fix);
                }
                if (NARROW) {
                    for (int r = 2 * oz.wp + (oz.lane >> 4); r < nrhs; r += 2 * oz.nw)
                        oz_cp(Ys + o * oz.ldr + r, (const double2 *)y + r, in);
                } else
#pragma unroll 4
                    for (int x = oz.wp; x < OZ_KC; x += oz.nw) {
                        const double2 *yx = (const double2 *)__shfl_sync(0xffffffffu, y, x);
                        if (oz.lane < nrhs) oz_cp(Ys + x * oz.ldr + oz.lane, yx + oz.lane, c * OZ_KC + x < K);
                    }
            }
            cp_async_commit();
        };
        oz.run(nch, rows, stage, re, ce);
        oz.store(rows, nrhs, re, ce, [&](int row, int col, double2 v, bool again) {   // one lane's, in every table
            if (again) {
                uint8_t *b = s_ag.tabs + row * 16 + col;
                if (!*b) s_ag.list[atomicAdd(&s_ag.n, 1)] = (uint16_t)(row * 16 + col);
                *b |= (uint8_t)(1 << tab);
                v = make_double2(0.0, 0.0);
            }
            double2 *o = out + row + (int64_t)col * n;
            *o = first ? v : make_double2(o->x + v.x, o->y + v.y);
        });
        oz.reset();
        first = false;
        __syncthreads();   // the exponents are read
    }
    for (int x = oz.wp; x < s_ag.n; x += oz.nw) {
        const int row = s_ag.list[x] >> 4, col = s_ag.list[x] & 15;
        double2 *o = out + row + (int64_t)col * n, w = make_double2(0.0, 0.0);
        for (int tabs = s_ag.tabs[row * 16 + col]; tabs; tabs &= tabs - 1) {
            const int tab = __ffs(tabs) - 1;
            const int *pt = zpart + tab * (nl * FAR_PARTS + 1) + blockIdx.x;
            const double2 *F0 = tab == FAR_TABS - 1 ? nearp : U, *F1 = tab == FAR_TABS - 1 ? nearp : V;
            const double2 *Y = tab == 0 ? t : tab == 1 ? s : u;
            const int J = tab < 2 ? 1 : 4;   // a lane per (short) segment of rank vectors, four per segment of blocks
            double2 v = make_double2(0.0, 0.0);
            for (int q = pt[0] + oz.lane / J; q < pt[1]; q += 32 / J) {
                const FarSegD g = sg[q];
                const double2 *f = ((g.src & 1) ? F1 : F0) + g.foff + (int64_t)(r0 + row) * g.fi;
                const double2 *y = Y + g.yrow * nrhs + col;
#pragma unroll 4
                for (int kk = oz.lane % J; kk < g.len; kk += J) v = cfma(f[(int64_t)kk * g.fk], y[kk * nrhs], v);
            }
            v = warp_sum(v);
            w.x += v.x;
            w.y += v.y;
        }
        if (oz.lane == 0) *o = make_double2(o->x + w.x, o->y + w.y);
    }
    if (first)
        for (int e = threadIdx.x; e < rows * nrhs; e += blockDim.x)
            out[e % rows + (int64_t)(e / rows) * n] = make_double2(0.0, 0.0);
}

// ---- complex FP32 on the tensor cores ------------------------------------------------------
// The same two phases with the block products on the tensor-core micro-kernel of tc.cuh
// (TF32 operands split into a rounded part and a remainder, FP32 accumulation in tensor
// memory), streamed in chunks of tc::KC2 contraction entries through a three-deep pipeline:
// the raw coefficient and vector entries of chunk c+1 are copied with cp.async while chunk c is
// split into one stage of operand planes and the MMAs of chunk c-1 run on the other stage.
// Fixed chunk order, so every output sums its terms in one order whatever the number of
// right-hand sides.
constexpr int FTC_LD = 64;                                   // raw[kk * FTC_LD + row or column]
constexpr int FTC_RAW = tc::KC2 * FTC_LD * 8;                // one raw buffer (8 KB)
constexpr int FTC_REGION = 2 * tc::STAGE2 + 4 * FTC_RAW;     // planes, then raw A and B x 2
constexpr unsigned long long FTC_WAIT_NS = 2000000000ull;
constexpr size_t FTC_SMEM = (FTC_REGION > tc::REGION_BYTES ? FTC_REGION : tc::REGION_BYTES) + 1024;

// Phase 1: task -> up to 64 factor columns (rows of the product) contracted over [lo, hi)
__global__ void __launch_bounds__(256, 2) k_far_t_tc(const int *task_lo, const int *task_hi, const int *task_ptr,
                                                     const int64_t *item_off, const int *item_ld,
                                                     const int *item_rank, const int *item_row, const int *item_isv,
                                                     const float2 *U, const float2 *V, const float2 *u, int nrhs,
                                                     float2 *t, float2 *s, int *err)
{
    extern __shared__ unsigned char smraw[];
    __shared__ int s_item[64], s_l[64];
    __shared__ const float2 *s_src[64];
    __shared__ uint64_t s_mbar[2];
    __shared__ uint32_t s_tmem;
    const int task = blockIdx.x;
    const int lo = task_lo[task], hi = task_hi[task], i0 = task_ptr[task], i1 = task_ptr[task + 1];
    const int R = far_items(i0, i1, item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src);
    if (R == 0) return;
    unsigned char *region = tc::align1024(smraw);
    float2 *rawA = (float2 *)(region + 2 * tc::STAGE2), *rawB = rawA + 2 * tc::KC2 * FTC_LD;
    tc::Acc2 acc;
    acc.planes = region;
    acc.mbar = s_mbar;
    acc.tslot = &s_tmem;
    acc.open(R, nrhs);
    const int nch = (hi - lo + tc::KC2 - 1) / tc::KC2;
    auto fetch = [&](int c) {   // raw entries of chunk c into raw buffer c & 1
        const int c0 = lo + c * tc::KC2, kl = min(tc::KC2, hi - c0), b = c & 1;
        float2 *ra = rawA + b * tc::KC2 * FTC_LD, *rb = rawB + b * tc::KC2 * FTC_LD;
        for (int e = threadIdx.x; e < kl * R; e += blockDim.x) {
            const int kk = e % kl, rr = e / kl;
            cp_async_el(ra + kk * FTC_LD + rr, s_src[rr] + (c0 - lo + kk));
        }
        const float2 *uc = u + (int64_t)c0 * nrhs;
        for (int e = threadIdx.x; e < kl * nrhs; e += blockDim.x) cp_async_el(rb + (e / nrhs) * FTC_LD + e % nrhs, uc + e);
        cp_async_commit();
    };
    if (nch > 0) fetch(0);
    for (int c = 0; c < nch; ++c) {
        const int st = c & 1, kl = min(tc::KC2, hi - (lo + c * tc::KC2));
        if (c + 1 < nch) {
            fetch(c + 1);
            cp_async_wait<1>();
        } else
            cp_async_wait<0>();
        __syncthreads();                       // chunk c's raw entries are visible
        acc.wait(st, err, FTC_WAIT_NS);        // the MMAs of chunk c - 2 have left stage st
        const float2 *ra = rawA + st * tc::KC2 * FTC_LD, *rb = rawB + st * tc::KC2 * FTC_LD;
        for (int e = threadIdx.x; e < acc.m8 * kl; e += blockDim.x) {
            const int r = e % acc.m8, kk = e / acc.m8;
            acc.put_a(st, r, kk, r < R ? ra[kk * FTC_LD + r] : make_float2(0.f, 0.f));
        }
        for (int e = threadIdx.x; e < acc.p * kl; e += blockDim.x) {
            const int col = e % acc.p, kk = e / acc.p;
            acc.put_b(st, col, kk, col < nrhs ? rb[kk * FTC_LD + col] : make_float2(0.f, 0.f));
        }
        acc.zero_pad(st, kl);
        acc.issue(st, kl);
    }
    acc.wait(0, err, FTC_WAIT_NS);
    acc.wait(1, err, FTC_WAIT_NS);
    float *dsm = (float *)region;
    const bool any = acc.drain(dsm);
    for (int e = threadIdx.x; e < R * nrhs; e += blockDim.x) {
        const int rr = e / nrhs, r = e % nrhs, it = s_item[rr];
        float2 *dst = item_isv[it] ? t : s;
        dst[(int64_t)(item_row[it] + s_l[rr]) * nrhs + r] = any ? acc.entry(dsm, rr, r) : make_float2(0.f, 0.f);
    }
    acc.close();
}

// Phase 2: CTA = (leaf, part); the part's segments streamed in chunks of tc::KC2 entries (a
// segment may be split between chunks)
struct FarTcChunk {
    const float2 *f[tc::KC2];   // coefficient entry kk of row i: f[kk][i * fi[kk]]
    int fi[tc::KC2];
    const float2 *y[tc::KC2];   // vector entry kk of column r: y[kk][r]
    int kl;
};

struct FarTcWalk {
    int q, koff;   // next segment and its first entry not yet taken
};

// thread 0: the next chunk of the part's segments [w.q, w1)
__device__ __forceinline__ void far_tc_chunk(FarTcWalk &w, int w1, const FarSegD *segs, const float2 *U,
                                             const float2 *V, const float2 *t, const float2 *s, const float2 *u,
                                             int nrhs, FarTcChunk &c)
{
    int kl = 0;
    while (w.q < w1 && kl < tc::KC2) {
        const FarSegD g = segs[w.q];
        const float2 *F = ((g.src & 1) ? V : U) + g.foff;
        const int ys = g.src >> 1;
        const float2 *Yb = (ys == 0 ? t : (ys == 1 ? s : u)) + g.yrow * nrhs;
        const int take = min(g.len - w.koff, tc::KC2 - kl);
        for (int k = 0; k < take; ++k) {
            const int kk = w.koff + k;
            c.f[kl + k] = F + (int64_t)kk * g.fk;
            c.fi[kl + k] = g.fi;
            c.y[kl + k] = Yb + (int64_t)kk * nrhs;
        }
        kl += take;
        w.koff += take;
        if (w.koff == g.len) {
            ++w.q;
            w.koff = 0;
        }
    }
    c.kl = kl;
}

__global__ void __launch_bounds__(256, 2) k_far_y_tc(int nl, const int *leaf_ptr, const int *part_ptr,
                                                     const int *kcum, const FarSegD *segs, const float2 *U,
                                                     const float2 *V, const float2 *t, const float2 *s,
                                                     const float2 *u, const int *cl2new, int n, int nrhs,
                                                     float2 *part, int *err)
{
    extern __shared__ unsigned char smraw[];
    __shared__ FarTcChunk s_ch[3];
    __shared__ uint64_t s_mbar[2];
    __shared__ uint32_t s_tmem;
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS;
    if (l >= nl) return;
    const int a = leaf_ptr[l], ni = leaf_ptr[l + 1] - a;
    const int p0 = part_ptr[blockIdx.x], w1 = part_ptr[blockIdx.x + 1];
    float2 *out = part + (size_t)pp * n * nrhs + cl2new[a];
    if (p0 >= w1) {   // an empty part still contributes zeros to the sum
        for (int e = threadIdx.x; e < ni * nrhs; e += blockDim.x) out[e % ni + (int64_t)(e / ni) * n] = make_float2(0.f, 0.f);
        return;
    }
    unsigned char *region = tc::align1024(smraw);
    float2 *rawA = (float2 *)(region + 2 * tc::STAGE2), *rawB = rawA + 2 * tc::KC2 * FTC_LD;
    tc::Acc2 acc;
    acc.planes = region;
    acc.mbar = s_mbar;
    acc.tslot = &s_tmem;
    FarTcWalk w{p0, 0};
    if (threadIdx.x == 0) {
        far_tc_chunk(w, w1, segs, U, V, t, s, u, nrhs, s_ch[0]);
        far_tc_chunk(w, w1, segs, U, V, t, s, u, nrhs, s_ch[1]);
    }
    acc.open(ni, nrhs);   // synchronises: s_ch[0], s_ch[1] are visible
    (void)kcum;
    auto fetch = [&](int c) {
        const FarTcChunk &ch = s_ch[c % 3];
        const int b = c & 1;
        float2 *ra = rawA + b * tc::KC2 * FTC_LD, *rb = rawB + b * tc::KC2 * FTC_LD;
        for (int e = threadIdx.x; e < ch.kl * ni; e += blockDim.x) {
            const int i = e % ni, kk = e / ni;
            cp_async_el(ra + kk * FTC_LD + i, ch.f[kk] + (int64_t)i * ch.fi[kk]);
        }
        for (int e = threadIdx.x; e < ch.kl * nrhs; e += blockDim.x)
            cp_async_el(rb + (e / nrhs) * FTC_LD + e % nrhs, ch.y[e / nrhs] + e % nrhs);
        cp_async_commit();
    };
    fetch(0);
    for (int c = 0; s_ch[c % 3].kl > 0; ++c) {
        const int st = c & 1, kl = s_ch[c % 3].kl;
        const bool more = s_ch[(c + 1) % 3].kl > 0;
        if (more) {
            fetch(c + 1);
            cp_async_wait<1>();
        } else
            cp_async_wait<0>();
        __syncthreads();                       // chunk c's raw entries are visible
        // thread 0: the sources of chunk c + 2 (its buffer held chunk c - 1, no longer read)
        if (threadIdx.x == 0) far_tc_chunk(w, w1, segs, U, V, t, s, u, nrhs, s_ch[(c + 2) % 3]);
        acc.wait(st, err, FTC_WAIT_NS);        // the MMAs of chunk c - 2 have left stage st
        const float2 *ra = rawA + st * tc::KC2 * FTC_LD, *rb = rawB + st * tc::KC2 * FTC_LD;
        for (int e = threadIdx.x; e < acc.m8 * kl; e += blockDim.x) {
            const int r = e % acc.m8, kk = e / acc.m8;
            acc.put_a(st, r, kk, r < ni ? ra[kk * FTC_LD + r] : make_float2(0.f, 0.f));
        }
        for (int e = threadIdx.x; e < acc.p * kl; e += blockDim.x) {
            const int col = e % acc.p, kk = e / acc.p;
            acc.put_b(st, col, kk, col < nrhs ? rb[kk * FTC_LD + col] : make_float2(0.f, 0.f));
        }
        acc.zero_pad(st, kl);
        acc.issue(st, kl);                     // barrier inside: s_ch[(c + 2) % 3] is visible after it
    }
    acc.wait(0, err, FTC_WAIT_NS);
    acc.wait(1, err, FTC_WAIT_NS);
    float *dsm = (float *)region;
    const bool any = acc.drain(dsm);
    for (int e = threadIdx.x; e < ni * nrhs; e += blockDim.x) {
        const int i = e % ni, r = e / ni;
        out[i + (int64_t)r * n] = any ? acc.entry(dsm, i, r) : make_float2(0.f, 0.f);
    }
    acc.close();
}

// y = sum of the FAR_PARTS partial products, added in part order; bad: see k_far_gather64
template <class T> __global__ void k_far_sum(int n, int64_t len, const T *part, T *y, const int *bad = nullptr)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= len) return;
    T v = part[e];
    for (int p = 1; p < FAR_PARTS; ++p) {
        const T w = part[p * len + e];
        v.x += w.x;
        v.y += w.y;
    }
    if constexpr (sizeof(T) == 16) {
        const int b = bad ? *bad : 0;
        if (b && b >> (int)(e / n) & 1) v = make_double2(nan(""), nan(""));
    }
    y[e] = v;
}

namespace {
template <class T> struct FarLaunch {
    hm_ctx *h;
    const T *U, *V;
    T *t, *s;
    const T *ucl;
    T *y;
    int nrhs;
    template <int TR, int TC, int NT> cudaError_t run(int maxw)
    {
        const FarPlan &F = h->fplan;
        const int n = h->plan.n;
        const int budget = stage_need(64, SEG, nrhs, TR, TC);
        const size_t smem = sizeof(T) * (size_t)budget;
        static DeviceOnce attr;   // one per instantiation
        if (attr.need()) {
            const int smax = (int)(sizeof(T) * (size_t)stage_need(64, SEG, maxw, TR, TC));
            cudaError_t e;
            if ((e = cudaFuncSetAttribute(k_far_t<T, TR, TC, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)) ||
                (e = cudaFuncSetAttribute(k_far_y<T, TR, TC, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)))
                return e;
            attr.done();
        }
        const int ntask = (int)F.p1_lo.size();
        if (ntask > 0)
            HM_LAUNCH(h, K_FAR1,
                      (k_far_t<T, TR, TC, NT><<<ntask, 256, smem, h->stream>>>(
                          h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off, h->d_p1_ld, h->d_p1_rank, h->d_p1_row,
                          h->d_p1_isv, U, V, ucl, nrhs, t, s, budget)));
        T *part = (T *)h->d_farpart;
        HM_LAUNCH(h, K_FAR2,
                  (k_far_y<T, TR, TC, NT><<<h->nl * FAR_PARTS, 256, smem, h->stream>>>(
                      h->nl, h->d_leaf_ptr, h->d_part_ptr, h->d_seg_kcum, h->d_segs, U, V, t, s, ucl, h->d_cl2new,
                      n, nrhs, part, budget)));
        const int64_t len = (int64_t)n * nrhs;
        HM_LAUNCH(h, K_FAR2, k_far_sum<T><<<nblk(len, 256), 256, 0, h->stream>>>(n, len, part, y));
        return cudaGetLastError();
    }
};
}  // namespace

// complex FP32 on the tensor cores: phase 1, the phase-2 partial products, their sum
static cudaError_t far_tc_launch(hm_ctx *h, const float2 *U, const float2 *V, float2 *t, float2 *s,
                                 const float2 *ucl, float2 *y, int nrhs)
{
    const FarPlan &F = h->fplan;
    const int n = h->plan.n;
    static DeviceOnce attr;
    if (attr.need()) {
        cudaError_t e;
        if ((e = cudaFuncSetAttribute(k_far_t_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FTC_SMEM)) ||
            (e = cudaFuncSetAttribute(k_far_y_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FTC_SMEM)))
            return e;
        attr.done();
    }
    const int ntask = (int)F.p1_lo.size();
    if (ntask > 0)
        HM_LAUNCH(h, K_FAR1,
                  (k_far_t_tc<<<ntask, 256, FTC_SMEM, h->stream>>>(h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off,
                                                                   h->d_p1_ld, h->d_p1_rank, h->d_p1_row, h->d_p1_isv,
                                                                   U, V, ucl, nrhs, t, s, h->d_err)));
    float2 *part = (float2 *)h->d_farpart;
    HM_LAUNCH(h, K_FAR2,
              (k_far_y_tc<<<h->nl * FAR_PARTS, 256, FTC_SMEM, h->stream>>>(
                  h->nl, h->d_leaf_ptr, h->d_part_ptr, h->d_seg_kcum, h->d_segs, U, V, t, s, ucl, h->d_cl2new, n, nrhs,
                  part, h->d_err)));
    const int64_t len = (int64_t)n * nrhs;
    HM_LAUNCH(h, K_FAR2, k_far_sum<float2><<<nblk(len, 256), 256, 0, h->stream>>>(n, len, part, y));
    return cudaGetLastError();
}

// exponents of the coefficient rows for the FP64 products, once per handle (h->d_rexp: V columns, U columns, then the rows
// of the leaves by table and part)
cudaError_t far64_prepare(hm_ctx *h)
{
    const FarPlan &F = h->fplan;
    const int64_t tlen = F.tlen, n = h->n, len = 2 * tlen + FAR_TABS * FAR_PARTS * n;
    cudaError_t e;
    if ((e = h->arena.alloc((void **)&h->d_rexp, sizeof(uint16_t) * (size_t)len)) ||
        (e = h->arena.alloc((void **)&h->d_vexp, sizeof(uint16_t) * VEXP * (size_t)(2 * tlen + n))) ||
        (e = h->arena.alloc((void **)&h->d_colbad, sizeof(int))))
        return e;
    if ((e = cudaMemsetAsync(h->d_rexp, 0, sizeof(uint16_t) * (size_t)len, h->stream))) return e;
    const int ntask = (int)F.p1_lo.size();
    if (ntask > 0)
        k_far_rexp1<<<ntask, 256, 0, h->stream>>>(h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off, h->d_p1_ld, h->d_p1_rank,
                                                  h->d_p1_row, h->d_p1_isv, h->d_farU, h->d_farV, h->d_rexp, tlen);
    k_far_rexp2<<<dim3(h->nl * FAR_PARTS, FAR_TABS), 256, 0, h->stream>>>(h->nl, h->n, h->d_leaf_ptr, h->d_zpart, h->d_zsegs,
                                                                       h->d_farU, h->d_farV, h->d_near,
                                                                       h->d_rexp + 2 * tlen);
    return cudaGetLastError();
}

template <bool NARROW>
static cudaError_t far64_run(hm_ctx *h, const double2 *U, const double2 *V, double2 *t, double2 *s, const double2 *x,
                             double2 *u, double2 *y, int nrhs, bool near)
{
    const FarPlan &F = h->fplan;
    const int n = h->plan.n, threads = 64 * Oz<NARROW>::tiles(nrhs);
    const size_t smem = Oz<NARROW>::smem(nrhs);
    const int64_t len = (int64_t)n * nrhs;
    static DeviceOnce attr;
    cudaError_t e;
    if (attr.need()) {
        const int smax = (int)Oz<NARROW>::smem(16);
        if ((e = cudaFuncSetAttribute(k_far_t64<NARROW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)) ||
            (e = cudaFuncSetAttribute(k_far_y64<NARROW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)))
            return e;
        attr.done();
    }
    if ((e = cudaMemsetAsync(h->d_colbad, 0, sizeof(int), h->stream))) return e;
    HM_LAUNCH(h, K_PERMUTE, k_far_gather64<<<nblk(len, 256), 256, 0, h->stream>>>(n, nrhs, h->d_cl2new, x, u,
                                                                              h->d_vexp + 2 * F.tlen * VEXP, h->d_colbad));
    const int ntask = (int)F.p1_lo.size();
    if (ntask > 0)
        HM_LAUNCH(h, K_FAR1,
                  k_far_t64<NARROW><<<dim3(ntask, 64 / OZ_ROWS), threads, smem, h->stream>>>(
                      h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off, h->d_p1_ld, h->d_p1_rank, h->d_p1_row,
                      h->d_p1_isv, U, V, u, nrhs, t, s, h->d_rexp, h->d_vexp, F.tlen));
    double2 *part = (double2 *)h->d_farpart;
    HM_LAUNCH(h, K_FAR2,
              k_far_y64<NARROW><<<dim3(h->nl * FAR_PARTS, (h->max_leaf + OZ_ROWS - 1) / OZ_ROWS), threads, smem, h->stream>>>(
                  h->nl, h->d_leaf_ptr, h->d_zpart, h->d_zkcum, h->d_zsegs, U, V, near ? h->d_near : nullptr, t, s, u,
                  h->d_cl2new, n, nrhs, part, h->d_rexp + 2 * F.tlen, h->d_vexp, F.tlen));
    HM_LAUNCH(h, K_FAR2, k_far_sum<double2><<<nblk(len, 256), 256, 0, h->stream>>>(n, len, part, y, h->d_colbad));
    return cudaGetLastError();
}

// complex FP64: y = Z_F x, or Z x with the near-field segments, x and y in solve order; at most 16 columns; u: n x nrhs
// entries of scratch
cudaError_t far_product64(hm_ctx *h, const double2 *U, const double2 *V, double2 *t, double2 *s, const double2 *x,
                          double2 *u, double2 *y, int nrhs, bool near)
{
    h->prof.cols[K_FAR1] += nrhs;
    h->prof.cols[K_FAR2] += nrhs;
    return nrhs <= 4 ? far64_run<true>(h, U, V, t, s, x, u, y, nrhs, near) : far64_run<false>(h, U, V, t, s, x, u, y, nrhs, near);
}

// complex FP32, 17 to 64 columns
static cudaError_t far32_run(hm_ctx *h, const float2 *U, const float2 *V, float2 *t, float2 *s, const float2 *ucl,
                             float2 *y, int nrhs)
{
    const FarPlan &F = h->fplan;
    const int n = h->plan.n, np = f32_np(h->max_leaf), nc = f32_nc(nrhs), ldr = nc * F32_COLS;
    const size_t smt = sizeof(float2) * F32_RING * F32_KC * (size_t)(f32_ldw(4) + ldr);
    const size_t smy = sizeof(float2) * F32_RING * F32_KC * (size_t)(f32_ldw(np) + ldr);
    static DeviceOnce attr;
    if (attr.need()) {   // 64 rows and 64 columns
        const int smax = (int)(sizeof(float2) * F32_RING * F32_KC * (f32_ldw(4) + 64));
        cudaError_t e;
        if ((e = cudaFuncSetAttribute(k_far_t32, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)) ||
            (e = cudaFuncSetAttribute(k_far_y32, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)))
            return e;
        attr.done();
    }
    const bool v16 = nrhs % 2 == 0 && (((uintptr_t)t | (uintptr_t)s | (uintptr_t)ucl) & 15) == 0;
    const int ntask = (int)F.p1_lo.size();
    if (ntask > 0)
        HM_LAUNCH(h, K_FAR1,
                  k_far_t32<<<ntask, 32 * 4 * nc, smt, h->stream>>>(h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off,
                                                                    h->d_p1_ld, h->d_p1_rank, h->d_p1_row, h->d_p1_isv, U,
                                                                    V, ucl, nrhs, t, s, v16));
    float2 *part = (float2 *)h->d_farpart;
    HM_LAUNCH(h, K_FAR2,
              k_far_y32<<<h->nl * FAR_PARTS, 32 * np * nc, smy, h->stream>>>(
                  h->nl, h->d_leaf_ptr, h->d_part_ptr, h->d_seg_kcum, h->d_segs, U, V, t, s, ucl, h->d_cl2new, n, nrhs,
                  part, np, v16));
    const int64_t len = (int64_t)n * nrhs;
    HM_LAUNCH(h, K_FAR2, k_far_sum<float2><<<nblk(len, 256), 256, 0, h->stream>>>(n, len, part, y));
    return cudaGetLastError();
}

cudaError_t far_product32(hm_ctx *h, const float2 *U, const float2 *V, float2 *t, float2 *s, const float2 *ucl, float2 *y,
                          int nrhs)
{
    h->prof.cols[K_FAR1] += nrhs;
    h->prof.cols[K_FAR2] += nrhs;
    if (h->far_kind == 2) return far_tc_launch(h, U, V, t, s, ucl, y, nrhs);
    // the wide kernels from 17 columns on: their warps cover 32 (at 16 columns half of the lanes would be idle)
    if (nrhs > 16) return far32_run(h, U, V, t, s, ucl, y, nrhs);
    FarLaunch<float2> f{h, U, V, t, s, ucl, y, nrhs};
    return nrhs <= 4 ? f.run<1, 1, 1>(4) : f.run<2, 2, 1>(16);
}

}  // namespace hm
