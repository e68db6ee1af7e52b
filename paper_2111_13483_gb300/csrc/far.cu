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
// runs a register-tiled product (tile.cuh); t and s are stored interleaved like u.
// Phase 2 (k_far_y): one CTA per leaf accumulates, in the order of the leaf's list of
// covering far blocks, U_b t_b (row side), V_b s_b (column side), B u (dense row side) and
// B^T u (dense column side) for the leaf's rows; the host plan cuts the list into
// contraction segments of at most 32, which are staged in shared memory in chunks.  Each
// leaf's list is split into FAR_PARTS consecutive parts of about equal length, one CTA each
// (so that the uneven leaves spread over all SMs); k_far_sum adds the parts in order.  Every output sums its terms in
// one fixed order, so results are deterministic and do not depend on how many right-hand
// sides share the launch.
#include <algorithm>

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
// GB300 issues a DFMA for two lanes per SM and clock: one warp instruction holds its scheduler for 64
// cycles whatever its lanes do, and shared-memory loads are free beside it.  So the outputs are laid flat
// over the lanes (28 rows x 16 columns are 14 full warps; 2 x 2 register tiles left an eighth of the
// lanes idle), and the contraction is split F64_NK ways (entry kk of the whole contraction to
// way kk mod F64_NK, partial sums added in order), so that one column keeps all four schedulers busy
// too.  The split does not depend on the columns: a column's bits are the same in any batch.
// The near-field blocks of a leaf join its phase-2 segments where Z itself is applied.
// Measured at 64 columns on the 30,720-unknown sphere: phase 1 23.5 -> 22.8 ms, phase 2 38.6 and the near field
// 34.6 (a CTA of its own per leaf) -> 47.2 ms together; one column: 0.64 -> 0.46 and 1.37 + 0.80 -> 1.42 ms.
// Phase 2 runs at the DFMA rate (0.63 T/s measured by a chain of FMAs).
constexpr int F64_NK = 4, F64_NH = 2;   // ways the contraction and the outputs are split over the warps
constexpr int F64_T = 32 * F64_NK * F64_NH;

// acc[u] += sum over this warp's kk of Ws[kk * ldw + i] Ys[kk * ldr + c], output e = lane + 32 (F64_NH u + half) = c * no + i
template <int NU>
__device__ __forceinline__ void f64_mac(double2 (&acc)[NU], const double2 *Ws, int ldw, const double2 *Ys, int ldr, int k0,
                                        int klen, int no, int len)
{
    const int w = (threadIdx.x >> 5) - k0 & F64_NK - 1;   // the chunk starts at entry k0
    const int e0 = (threadIdx.x & 31) + 32 * (threadIdx.x >> 7), di = 32 * F64_NH % no, dc = 32 * F64_NH / no;
    for (int kk = w; kk < klen; kk += F64_NK) {
        const double2 *wp = Ws + kk * ldw, *yp = Ys + kk * ldr;
        int i = e0 % no, c = e0 / no;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int e = e0 + 32 * F64_NH * u;
            if (e - (int)(threadIdx.x & 31) >= len) break;
            if (e < len) acc[u] = cfma(wp[i], yp[c], acc[u]);
            i += di;
            c += dc;
            if (i >= no) i -= no, ++c;
        }
    }
}

// the warps' partial sums through shared memory: put(e, sum) for every output e < len
template <int NU, class Put> __device__ __forceinline__ void f64_reduce(const double2 (&acc)[NU], double2 *sm, int len, Put &&put)
{
    const int e0 = (threadIdx.x & 31) + 32 * (threadIdx.x >> 7), w = threadIdx.x >> 5 & F64_NK - 1;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        const int e = e0 + 32 * F64_NH * u;
        if (e < len) sm[w * len + e] = acc[u];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < len; e += F64_T) {
        double2 v = sm[e];
        for (int q = 1; q < F64_NK; ++q) {
            v.x += sm[q * len + e].x;
            v.y += sm[q * len + e].y;
        }
        put(e, v);
    }
}

// phase 1, tasks as in k_far_t
template <int NU>
__global__ void __launch_bounds__(F64_T) k_far_t64(const int *task_lo, const int *task_hi, const int *task_ptr,
                                                   const int64_t *item_off, const int *item_ld, const int *item_rank,
                                                   const int *item_row, const int *item_isv, const double2 *U,
                                                   const double2 *V, const double2 *u, int nrhs, double2 *t, double2 *s,
                                                   int half)
{
    extern __shared__ unsigned char smraw[];
    __shared__ int s_item[64], s_l[64];
    __shared__ const double2 *s_src[64];
    const int task = blockIdx.x;
    const int lo = task_lo[task], hi = task_hi[task], i0 = task_ptr[task], i1 = task_ptr[task + 1];
    const int R = far_items(i0, i1, item_off, item_ld, item_rank, item_isv, U, V, s_item, s_l, s_src), len = R * nrhs, ldw = R | 1;
    double2 *const bufs[2] = {(double2 *)smraw, (double2 *)smraw + half};
    double2 acc[NU];
#pragma unroll
    for (int q = 0; q < NU; ++q) acc[q] = make_double2(0.0, 0.0);
    auto stage = [&](int c0, int which) {   // as in k_far_t: Ws[qq * ldw + rr], then Ys[qq * nrhs + r]
        const int ch = min(FAR_T1, hi - c0);
        double2 *Ws = bufs[which], *Ys = Ws + ch * ldw;
        for (int rr = threadIdx.x / FAR_T1; rr < R; rr += F64_T / FAR_T1) {
            const int qq = threadIdx.x % FAR_T1;
            if (qq < ch) far_cp(Ws + qq * ldw + rr, s_src[rr] + (c0 - lo + qq));
        }
        const double2 *uc = u + (int64_t)c0 * nrhs;
        for (int e = threadIdx.x; e < ch * nrhs; e += F64_T) far_cp(Ys + e, uc + e);
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
        const double2 *Ws = bufs[it & 1];
        f64_mac<NU>(acc, Ws, ldw, Ws + ch * ldw, nrhs, c0 - lo, ch, R, len);
        __syncthreads();
    }
    f64_reduce<NU>(acc, (double2 *)smraw, len, [&](int e, double2 v) {
        const int rr = e % R, r = e / R, it = s_item[rr];
        (item_isv[it] ? t : s)[(int64_t)(item_row[it] + s_l[rr]) * nrhs + r] = v;
    });
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

// complex FP64, phase 2 (see f64_mac): the segments of the far list and, with nearp, those of the leaf's
// near-field blocks (zpart / zkcum / zsegs), which gives Z u in one pass
template <int NU>
__global__ void __launch_bounds__(F64_T) k_far_y64(int nl, const int *leaf_ptr, const int *part_ptr, const int *kcum,
                                                   const FarSegD *segs, const int *zpart, const int *zkcum,
                                                   const FarSegD *zsegs, const double2 *U, const double2 *V,
                                                   const double2 *nearp, const double2 *t, const double2 *s,
                                                   const double2 *u, const int *cl2new, int n, int nrhs, double2 *part,
                                                   int half)
{
    extern __shared__ unsigned char smraw[];
    const int l = blockIdx.x / FAR_PARTS, pp = blockIdx.x % FAR_PARTS;
    if (l >= nl) return;
    const int a = leaf_ptr[l], ni = leaf_ptr[l + 1] - a, len = ni * nrhs, ldw = ni | 1;
    const int kmax = half / (ldw + nrhs);   // >= 32
    double2 *const bufs[2] = {(double2 *)smraw, (double2 *)smraw + half};
    double2 acc[NU];
#pragma unroll
    for (int q = 0; q < NU; ++q) acc[q] = make_double2(0.0, 0.0);
    for (int tab = 0; tab < (nearp ? 2 : 1); ++tab) {
        const int *pt = tab ? zpart : part_ptr, *kc = tab ? zkcum : kcum;
        const FarSegD *sg = tab ? zsegs : segs;
        const double2 *F0 = tab ? nearp : U, *F1 = tab ? nearp : V;
        const int w1 = pt[blockIdx.x + 1];
        auto chunk_count = [&](int p) {   // segments from p on whose stacked length fits kmax
            const int q = p + threadIdx.x;
            return __syncthreads_count(q < w1 && kc[q + 1] - kc[p] <= kmax);
        };
        auto stage = [&](int p, int cnt, double2 *buf) {   // as in k_far_y
            const int k0 = kc[p], klen = kc[p + cnt] - k0;
            double2 *Wst = buf, *Yst = buf + kmax * ldw;
            int q = -1, qlo = 0, qhi = 0;
            const double2 *F = nullptr;
            int64_t fi = 0, fk = 0;
            for (int e = threadIdx.x; e < klen * ni; e += F64_T) {
                const int kk = e / ni, i = e - kk * ni;
                while (kk >= qhi) {
                    ++q;
                    qlo = kc[p + q] - k0;
                    qhi = kc[p + q + 1] - k0;
                    const FarSegD g = sg[p + q];
                    F = ((g.src & 1) ? F1 : F0) + g.foff;
                    fi = g.fi;
                    fk = g.fk;
                }
                cp_async_el(Wst + kk * ldw + i, F + (int64_t)i * fi + (int64_t)(kk - qlo) * fk);
            }
            q = -1;
            qhi = 0;
            const double2 *Yb = nullptr;
            for (int e = threadIdx.x; e < klen * nrhs; e += F64_T) {
                const int kk = e / nrhs, r = e - kk * nrhs;
                while (kk >= qhi) {
                    ++q;
                    qlo = kc[p + q] - k0;
                    qhi = kc[p + q + 1] - k0;
                    const FarSegD g = sg[p + q];
                    const int ys = g.src >> 1;
                    Yb = (ys == 0 ? t : (ys == 1 ? s : u)) + g.yrow * nrhs;
                }
                cp_async_el(Yst + e, Yb + (int64_t)(kk - qlo) * nrhs + r);
            }
            cp_async_commit();
            return klen;
        };
        const int p0 = pt[blockIdx.x];
        int p = p0;
        if (p >= w1) continue;
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
            const double2 *buf = bufs[it & 1];
            f64_mac<NU>(acc, buf, ldw, buf + kmax * ldw, nrhs, kc[p] - kc[p0], klen, ni, len);
            __syncthreads();
            if (pn >= w1) break;
            p = pn;
            cnt = cntn;
            klen = klenn;
        }
    }
    double2 *out = part + (size_t)pp * n * nrhs + cl2new[a];
    f64_reduce<NU>(acc, (double2 *)smraw, len, [&](int e, double2 v) { out[e % ni + (int64_t)(e / ni) * n] = v; });
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

// y = sum of the FAR_PARTS partial products, added in part order
template <class T> __global__ void k_far_sum(int64_t len, const T *part, T *y)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= len) return;
    T v = part[e];
    for (int p = 1; p < FAR_PARTS; ++p) {
        const T w = part[p * len + e];
        v.x += w.x;
        v.y += w.y;
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
        HM_LAUNCH(h, K_FAR2, k_far_sum<T><<<nblk(len, 256), 256, 0, h->stream>>>(len, part, y));
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
    HM_LAUNCH(h, K_FAR2, k_far_sum<float2><<<nblk(len, 256), 256, 0, h->stream>>>(len, part, y));
    return cudaGetLastError();
}

// complex FP64: y = Z_F u, or Z u with the near-field segments.  NU: outputs per lane of the largest block (64 rank
// rows in phase 1, the largest leaf in phase 2).
template <int NT, int NY>
static cudaError_t far64_run(hm_ctx *h, const double2 *U, const double2 *V, double2 *t, double2 *s, const double2 *ucl,
                             double2 *y, int nrhs, bool near)
{
    const FarPlan &F = h->fplan;
    const int n = h->plan.n, maxn = h->max_leaf;
    const int ht = std::max(FAR_T1 * (65 + nrhs), (F64_NK * 64 * nrhs + 1) / 2);
    const int hy = std::max(32 * ((maxn | 1) + nrhs), (F64_NK * maxn * nrhs + 1) / 2);
    static DeviceOnce attr;
    if (attr.need()) {   // nrhs <= 16, blocks of up to 64 rows
        const int smax = (int)(sizeof(double2) * 2 * 32 * (65 + 16));
        cudaError_t e;
        if ((e = cudaFuncSetAttribute(k_far_t64<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)) ||
            (e = cudaFuncSetAttribute(k_far_y64<NY>, cudaFuncAttributeMaxDynamicSharedMemorySize, smax)))
            return e;
        attr.done();
    }
    const int ntask = (int)F.p1_lo.size();
    if (ntask > 0)
        HM_LAUNCH(h, K_FAR1,
                  k_far_t64<NT><<<ntask, F64_T, sizeof(double2) * 2 * ht, h->stream>>>(
                      h->d_p1_lo, h->d_p1_hi, h->d_p1_ptr, h->d_p1_off, h->d_p1_ld, h->d_p1_rank, h->d_p1_row,
                      h->d_p1_isv, U, V, ucl, nrhs, t, s, ht));
    double2 *part = (double2 *)h->d_farpart;
    HM_LAUNCH(h, K_FAR2,
              k_far_y64<NY><<<h->nl * FAR_PARTS, F64_T, sizeof(double2) * 2 * hy, h->stream>>>(
                  h->nl, h->d_leaf_ptr, h->d_part_ptr, h->d_seg_kcum, h->d_segs, h->d_zpart, h->d_zkcum, h->d_zsegs, U, V,
                  near ? h->d_near : nullptr, t, s, ucl, h->d_cl2new, n, nrhs, part, hy));
    const int64_t len = (int64_t)n * nrhs;
    HM_LAUNCH(h, K_FAR2, k_far_sum<double2><<<nblk(len, 256), 256, 0, h->stream>>>(len, part, y));
    return cudaGetLastError();
}

cudaError_t far_product64(hm_ctx *h, const double2 *U, const double2 *V, double2 *t, double2 *s, const double2 *ucl,
                          double2 *y, int nrhs, bool near)
{
    h->prof.cols[K_FAR1] += nrhs;
    h->prof.cols[K_FAR2] += nrhs;
    if (nrhs <= 4) return far64_run<4, 4>(h, U, V, t, s, ucl, y, nrhs, near);
    if (h->max_leaf <= 32) return far64_run<16, 8>(h, U, V, t, s, ucl, y, nrhs, near);
    return far64_run<16, 16>(h, U, V, t, s, ucl, y, nrhs, near);
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
    HM_LAUNCH(h, K_FAR2, k_far_sum<float2><<<nblk(len, 256), 256, 0, h->stream>>>(len, part, y));
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
