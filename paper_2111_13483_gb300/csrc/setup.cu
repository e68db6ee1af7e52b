// Symmetric near-field Schur-complement setup (Sec. 3.1-3.2, Eqs. 12-21) on the GPU.
//
// Storage (solve order, blocks k = 0..nb-1 of n_k <= 64 unknowns):
//   Ad + doff[k]        A_kk, n_k x n_k; after the step it is D_k (Eq. 21);
//   A  + coff[k]        stacked column k: the blocks A_jk, j in S_k, one under the other,
//                       (M_k x n_k, ld M_k), the lower half of the symmetric near field
//                       plus its fill (scratch during setup);
//   W  + coff[k]        coefficient panel W_k = D_k^{-1} [A_kj]_{j in S_k} (n_k x M_k,
//                       ld n_k): W_kj = -alpha_kj of Eq. 14, the left coefficients being
//                       their transposes (Sec. 3.2);
//   Dinv + doff[k]      D_k^{-1} for the Eq. 28 preconditioner.
// Step k: pivot inverse, panel, Schur updates
// A_ij -= A_ik W_kj for i >= j in S_k (Eq. 19; diagonal blocks in full; one CTA per block
// pair in FP64, one CTA per row block and group of up to 16 column blocks in FP32).  Stream
// order and the two events of the look-ahead give the step dependencies.
//
// S is the storage and arithmetic type of A, the diagonal blocks and W: complex FP64, or
// complex FP32 in the mixed-precision setup, where the pivot blocks are still inverted in
// FP64 (their inverse is kept in FP64 and as an FP32 copy for the panels and the inner
// operator) and everything else stays FP32, so no step converts between the two.
#include <algorithm>
#include <cstdio>

#include "cluster.cuh"
#include "cplx.cuh"
#include "hm_internal.h"
#include "tc.cuh"
#include "tile.cuh"

namespace hm {

// row offset of block i inside stacked column j (binary search in S_j); -1 if absent
__device__ __forceinline__ int find_row(const int *sptr, const int *sidx, const int *srow, int j, int i)
{
    int lo = sptr[j], hi = sptr[j + 1];
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        int v = sidx[mid];
        if (v == i) return srow[mid];
        if (v < i) lo = mid + 1; else hi = mid;
    }
    return -1;
}

// Near-field blocks (cluster leaves t <= s) into the solve-order workspace.
template <class S>
__global__ void k_scatter_near(int n_near, const int *near_t, const int *near_s, const int64_t *near_off,
                               const double2 *near, const int *leaf_ptr, const int *pos, const int *sptr,
                               const int *sidx, const int *srow, const int *M, const int64_t *coff,
                               const int64_t *doff, S *A, S *Ad, int *err, bool diag_only = false)
{
    int b = blockIdx.x;
    if (b >= n_near) return;
    int t = near_t[b], s = near_s[b];
    if (diag_only && t != s) return;
    int m = leaf_ptr[t + 1] - leaf_ptr[t], n = leaf_ptr[s + 1] - leaf_ptr[s];
    const double2 *B = near + near_off[b];
    int i = pos[t], j = pos[s];
    S *dst;
    int ld;
    bool tr;
    if (i == j) {
        dst = Ad + doff[i];
        ld = m;
        tr = false;
    } else if (i > j) {
        int r = find_row(sptr, sidx, srow, j, i);
        if (r < 0) { atomicExch(err, 0x7fffffff); return; }
        dst = A + coff[j] + r;
        ld = M[j];
        tr = false;
    } else {
        int r = find_row(sptr, sidx, srow, i, j);
        if (r < 0) { atomicExch(err, 0x7fffffff); return; }
        dst = A + coff[i] + r;
        ld = M[i];
        tr = true;
    }
    for (int e = threadIdx.x; e < m * n; e += blockDim.x) {
        int rr = e % m, cc = e / m;
        const S v = cconv<S>(B[e]);
        if (!tr) dst[rr + (int64_t)cc * ld] = v;
        else dst[cc + (int64_t)rr * ld] = v;
    }
}

// the warp's largest key, the lowest row on ties; row n with no key
__device__ __forceinline__ void gj_pick(unsigned long long &best, int &bi, int n)
{
    const bool any = bi < n;
    const unsigned hi = any ? (unsigned)(best >> 32) : 0u;
    const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
    const bool c1 = any && hi == mhi;
    const unsigned mlo = __reduce_max_sync(0xffffffffu, c1 ? (unsigned)best : 0u);
    bi = (int)__reduce_min_sync(0xffffffffu, c1 && (unsigned)best == mlo ? (unsigned)bi : (unsigned)n);
    best = (unsigned long long)mhi << 32 | mlo;
}
// conj(p) / |p|^2, |p|^2 = pv: the two divisions run on two lanes at once (a division is some ten FP64 instructions of
// 64 cycles each)
__device__ __forceinline__ double2 gj_reciprocal(double2 p, double pv)
{
    const double q = ((threadIdx.x & 1) ? -p.y : p.x) / pv;
    return make_double2(__shfl_sync(0xffffffffu, q, 0), __shfl_sync(0xffffffffu, q, 1));
}

// Pivot search of Gauss-Jordan step c by one warp over rows r >= c of column `col` of a
// (row-major, leading dimension ld): the largest |a_rc|^2, the lowest row on ties.  The
// squares are compared as the integer bit patterns of non-negative doubles (same order as
// the values), which keeps the compares off the slow FP64 pipe.  Lane 0 returns the row p,
// 1 / pivot in *d, and whether the pivot is singular (|pivot|^2 <= 1e-300 or not finite).
__device__ __forceinline__ int gj_pivot(const double2 *a, int ld, int col, int c, int n, double2 *d, bool *bad)
{
    const int lane = threadIdx.x & 31;
    unsigned long long best = 0;
    int bi = n;
    for (int r = c + lane; r < n; r += 32) {
        double2 v = a[r * ld + col];
        unsigned long long key = (unsigned long long)__double_as_longlong(fma(v.x, v.x, v.y * v.y));
        if (key > best || (key == best && r < bi) || bi == n) { best = key; bi = r; }
    }
    gj_pick(best, bi, n);
    const double pv = __longlong_as_double((long long)best);
    *bad = !(pv > 1e-300) || best >= 0x7ff0000000000000ull;
    *d = gj_reciprocal(a[bi * ld + col], pv);
    return bi;
}

// Entry (r, j) of Gauss-Jordan step c: row c takes the scaled pivot row rc; column c becomes
// -f d; every other entry cur - f rc (f = entry r of the pivot column after the interchange,
// d = 1 / pivot).
__device__ __forceinline__ double2 gj_col(double2 f, double2 d)
{
    return make_double2(-(f.x * d.x - f.y * d.y), -(f.x * d.y + f.y * d.x));
}
__device__ __forceinline__ double2 gj_other(double2 rc, double2 f, double2 cur)
{
    return make_double2(fma(-f.x, rc.x, fma(f.y, rc.y, cur.x)), fma(-f.x, rc.y, fma(-f.y, rc.x, cur.y)));
}

// In-place Gauss-Jordan inverse with partial pivoting (largest modulus, lowest row on
// ties) of D_k = Ad[k], in FP64 whatever S is; result to Dinv[k] (and its FP32 copy when
// Dinv32 is given).  err <- k+1 on a singular pivot.  One block per CTA, or per cluster of CL CTAs of
// which CTA q keeps the columns j = q, q + CL, ....  Rows lie on the lanes, a warp takes a column at a
// time, and the columns are kept in two copies that the steps read and write in turn, so a step has no
// barrier inside.  Step c eliminates with the pivot row p, 1 / pivot and the interchanged column c found in the step
// before (two alternating buffers; in a cluster they are pushed to every CTA through distributed shared
// memory).  Warp 0 of the CTA that holds column c + 1 eliminates that column first, searches it for the next
// pivot and publishes it, while the other warps eliminate the rest; one barrier ends the step.  The
// results agree bit for bit whatever CL is: each entry goes through cmul, gj_col and gj_other alone.  The
// row interchanges are undone by writing column x of the result from the column they moved there.
//
// What binds it: an FP64 instruction holds its scheduler 64 cycles and so does the next one that needs its result
// (a division 565), so the chain to the next pivot -- a product, an elimination, two squares, a search, a
// division -- takes about 1 us beside the elimination itself (four instructions per column, 32 rows and
// scheduler) and, in a cluster, the pushes and a barrier (400 cycles).  Four warps, one per scheduler, leave
// the chain's scheduler to it.  Searching, scaling and eliminating one after the other with a barrier
// between took 3.5 us a pivot on eight CTAs: 104 ms per setup of the 30,720-unknown sphere, now 83.
template <int CL> __device__ __forceinline__ void pivot_sync()
{
    if (CL > 1) cluster_sync();
    else __syncthreads();
}

template <class S, int CL>
__global__ void __launch_bounds__(128) k_pivot_inverse(int kbase, const int *size, const int64_t *doff, const S *Ad,
                                                       double2 *Dinv, float2 *Dinv32, int *err)
{
    const int q = CL > 1 ? (int)cluster_rank() : 0, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int k = kbase + (int)(blockIdx.x / CL);
    extern __shared__ double2 sm[];
    const int n = size[k];
    const int nloc = (n - q + CL - 1) / CL;    // columns q, q + CL, ... below n
    double2 *a = sm;                           // 2 x nloc x n: a[(copy * nloc + jl) * n + r] = column jl * CL + q
    __shared__ double2 s_col[2][64];           // pivot column after the interchange
    __shared__ double2 s_d[2];                 // 1 / pivot
    __shared__ int s_p[2];                     // pivot row
    __shared__ int piv[64];
    __shared__ int at[64];
    const S *D = Ad + doff[k];
    for (int e = threadIdx.x; e < n * nloc; e += blockDim.x) {
        const int r = e % n, jl = e / n;
        a[e] = cwiden(D[r + (int64_t)(jl * CL + q) * n]);
    }
    // one warp: the pivot of column c in col (rows >= c), to every CTA's buffer c & 1 with the column
    auto publish = [&](const double2 *col, int c) {
        double2 d;
        bool bad;
        const int p = gj_pivot(col, 1, 0, c, n, &d, &bad), b = c & 1;
        if (lane == 0 && bad) atomicCAS(err, 0, k + 1);
        for (int dst = 0; CL > 1 && dst < CL; ++dst) {
            for (int r = lane; r < n; r += 32)
                st_remote_d2(cluster_map(smem_addr(&s_col[b][r]), (unsigned)dst), col[r == p ? c : r]);
            if (lane == dst) {
                st_remote_d2(cluster_map(smem_addr(&s_d[b]), (unsigned)dst), d);
                st_remote_s32(cluster_map(smem_addr(&s_p[b]), (unsigned)dst), p);
            }
        }
        if (CL == 1) {
            for (int r = lane; r < n; r += 32) s_col[b][r] = col[r == p ? c : r];
            if (lane == 0) {
                s_d[b] = d;
                s_p[b] = p;
            }
        }
    };
    pivot_sync<CL>();   // the columns are loaded; every CTA of the cluster is running before any remote store
    if (q == 0 && wp == 0) publish(a, 0);
    pivot_sync<CL>();
    for (int c = 0; c < n; ++c) {
        const int b = c & 1, p = s_p[b];
        const double2 d = s_d[b];
        const double2 *cur = a + b * nloc * n;
        double2 *nxt = a + (b ^ 1) * nloc * n;
        if (threadIdx.x == 0) piv[c] = p;
        auto eliminate = [&](int jl, double2 rc) {
            const double2 *x = cur + jl * n;
            double2 *y = nxt + jl * n;
            if (jl * CL + q == c)   // the warp's whole column: one branch, not both products for every entry
                for (int r = lane; r < n; r += 32) y[r] = r == c ? d : gj_col(s_col[b][r], d);
            else
                for (int r = lane; r < n; r += 32) {
                    const double2 v = gj_other(rc, s_col[b][r], x[r == p ? c : r]);
                    y[r] = r == c ? rc : v;
                }
        };
        const bool mine = c + 1 < n && (c + 1) % CL == q;   // the next pivot's column is here
        const int first = mine ? (c + 1) / CL : nloc;
        if (mine && wp == 0) {
            eliminate(first, cmul(cur[first * n + p], d));
            __syncwarp();
            publish(nxt + first * n, c + 1);
        }
        // the other columns [lo, hi) of this warp (the search takes warp 0 as long as six columns); lane l scales the
        // pivot row's entry of the l-th of them
        const int cols = mine ? nloc - 1 : nloc, c0 = mine ? max(cols - 18, 0) / 4 : (cols + 3) / 4;
        const int each = (cols - c0 + 2) / 3, lo = wp == 0 ? 0 : min(c0 + (wp - 1) * each, cols);
        const int hi = wp == 0 ? c0 : min(lo + each, cols);
        const int j0 = lo + lane < first ? lo + lane : lo + lane + 1;
        double2 rcl = make_double2(0.0, 0.0);
        if (lo + lane < hi) rcl = cmul(cur[j0 * n + p], d);
        for (int t = lo; t < hi; ++t) {
            const double2 rc = make_double2(__shfl_sync(0xffffffffu, rcl.x, t - lo), __shfl_sync(0xffffffffu, rcl.y, t - lo));
            eliminate(t < first ? t : t + 1, rc);
        }
        pivot_sync<CL>();
    }
    a += (n & 1) * nloc * n;   // the copy the last step wrote
    // at[x] = the column of the array that the interchanges (undone last first) move to x
    for (int x = threadIdx.x; x < n; x += blockDim.x) {   // position x followed back through them
        int pos = x;
        for (int c = 0; c < n; ++c) {
            const int p = piv[c];
            pos = pos == c ? p : pos == p ? c : pos;
        }
        at[x] = pos;
    }
    __syncthreads();
    double2 *out = Dinv + doff[k];
    float2 *out32 = Dinv32 ? Dinv32 + doff[k] : nullptr;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int r = e % n, x = e / n, src = at[x];
        if (src % CL != q) continue;
        const double2 v = a[src / CL * n + r];
        out[e] = v;
        if (out32) out32[e] = make_float2((float)v.x, (float)v.y);
    }
}

// W_k[:, c0 : c0 + PC] = D_k^{-1} (A_col_k[c0 : c0 + PC, :])^T in S arithmetic.  Few columns per CTA spread a step's panel
// over the SMs: 64 FP64 columns of an 18-unknown block held one SM's DFMA pipe for 20 us.
template <class S> constexpr int PANEL_COLS = sizeof(S) == 16 ? 16 : 32;
template <class S> size_t panel_smem(int nk) { return sizeof(S) * (size_t)nk * ((nk | 1) + (PANEL_COLS<S> | 1)); }
template <class S>
__global__ void __launch_bounds__(256) k_panel(int k, const int *size, const int *M, const int64_t *coff,
                                               const int64_t *doff, const S *Dinv, const S *A, S *W)
{
    constexpr int PC = PANEL_COLS<S>, LC = PC | 1;
    extern __shared__ unsigned char psraw[];
    const int n = size[k], Mk = M[k], ld = n | 1;
    S *dinv = (S *)psraw;             // dinv[r*ld + q] = D_k^{-1}[r, q]
    S *ac = dinv + n * ld;            // ac[q*LC + col] = A_col[c0+col, q]
    const int c0 = blockIdx.x * PC;
    const int nc = min(PC, Mk - c0);
    const S *Di = Dinv + doff[k];
    const S *Ac = A + coff[k];
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        int r = e % n, q = e / n;
        dinv[r * ld + q] = Di[e];
    }
    for (int e = threadIdx.x; e < nc * n; e += blockDim.x) {
        int col = e % nc, q = e / nc;
        ac[q * LC + col] = Ac[(c0 + col) + (int64_t)q * Mk];
    }
    __syncthreads();
    S *Wk = W + coff[k];
    for (int e = threadIdx.x; e < n * nc; e += blockDim.x) {
        int r = e % n, col = e / n;
        S acc = czero(S());
        for (int q = 0; q < n; ++q) acc = cfma(dinv[r * ld + q], ac[q * LC + col], acc);
        Wk[r + (int64_t)(c0 + col) * n] = acc;
    }
}

// Schur updates of step k (Eq. 19), FP64 setup: one CTA per pair (a >= b) of S_k, A_ij -= A_ik W_kj.  The
// outputs of the block lie flat over the threads: a DFMA warp instruction holds its scheduler for 64 cycles whatever its
// lanes do and shared-memory loads are free beside it, so full warps count, not register tiles (32 x 32 tiles
// padded the 18-unknown blocks of a 4,720-unknown plate threefold: 59 ms per setup).
// The updates of a step come in one launch (UPD_ALL), or in two: the blocks of the first column of S_k, which the next
// pivot block may be waiting for (UPD_FIRST, ns CTAs), and those of the other ns columns (UPD_REST, ns one less).
constexpr int UPD_ALL = 0, UPD_FIRST = 1, UPD_REST = 2;
constexpr int UPD64_T = 128;
__device__ __forceinline__ void upd64_cp(double2 *dst, const double2 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__global__ void __launch_bounds__(UPD64_T) k_update64(int k, int ns, int part, const int *size, const int *sptr, const int *sidx,
                                                      const int *srow, const int *M, const int64_t *coff,
                                                      const int64_t *doff, const double2 *W, double2 *A, double2 *Ad)
{
    extern __shared__ double2 upd64_sm[];
    // triangular index -> (a, b), a >= b (integer arithmetic only)
    const long t = blockIdx.x;
    int a = (int)sqrtf(2.0f * (float)t);
    while ((long)(a + 1) * (a + 2) / 2 <= t) ++a;
    while ((long)a * (a + 1) / 2 > t) --a;
    int b = (int)(t - (long)a * (a + 1) / 2);
    if (part == UPD_FIRST) {
        a = (int)t;
        b = 0;
    }
    if (a >= ns) return;
    const int e0 = sptr[k] + (part == UPD_REST);
    const int i = sidx[e0 + a], j = sidx[e0 + b];
    const int nk = size[k], ni = size[i], nj = size[j];
    const int Mk = M[k];
    const double2 *Aik = A + coff[k] + srow[e0 + a];                 // ld Mk
    const double2 *Wkj = W + coff[k] + (int64_t)srow[e0 + b] * nk;   // ld nk
    double2 *C;
    int ldc;
    if (i == j) {
        C = Ad + doff[i];
        ldc = ni;
    } else {
        int r = find_row(sptr, sidx, srow, j, i);
        if (r < 0) return;   // a dropped update of the elimination without fill (else i is in S_j)
        C = A + coff[j] + r;
        ldc = M[j];
    }
    double2 *As = upd64_sm, *Ws = As + ni * nk;                      // As[q * ni + r] = A_ik[r, q], Ws[c * nk + q] = W_kj[q, c]
    for (int e = threadIdx.x; e < ni * nk; e += UPD64_T) upd64_cp(As + e, Aik + e % ni + (int64_t)(e / ni) * Mk);
    for (int e = threadIdx.x; e < nk * nj; e += UPD64_T) upd64_cp(Ws + e, Wkj + e);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int e = threadIdx.x; e < ni * nj; e += UPD64_T) {
        const int r = e % ni, c = e / ni;
        double2 *p = C + r + (int64_t)c * ldc;
        const double2 old = *p;
        double2 acc = make_double2(0.0, 0.0);
        for (int q = 0; q < nk; ++q) acc = cfma(As[q * ni + r], Ws[c * nk + q], acc);
        *p = make_double2(old.x - acc.x, old.y - acc.y);
    }
}

// Grouped Schur updates of step k for the complex-FP32 setup.  CTA -> (a, g): row block a
// of S_k and the column blocks b = g*gb .. min(a, g*gb + gb - 1), one warp per column block.
// A_ik is staged once per CTA; each warp streams its W_kj, UPD_C columns at a time, through two buffers of its
// own and multiplies 32 x UPD_C pieces of the block, up to 4 x 4 outputs per lane (8 row lanes, 4 column lanes;
// the pieces of uneven blocks have fewer), so that 8 shared-memory loads feed 64 FMAs and nothing
// but A_ik is shared between warps.  The old values of a piece are loaded before its operands have landed.  Every output
// sums its n_k products in order and is then subtracted from the old value.
// What bounds it is latency: a block's product takes 2 us of a warp, the loads of its operands and old values (HBM: the
// 1.2 GB workspace does not fit L2) as long again, so many warps matter: 4 x 8 outputs per lane leave 8 warps
// per SM, 197 ms of updates per setup of the 30,720-unknown sphere.  The whole CTA on one block with 2 x 2 outputs per
// thread loaded 4 values for 16 FMAs and met at two barriers per block: 249 ms (217 with smaller buffers and
// three CTAs per SM); this is 158 (a 100 x 100 plate, 29,800 unknowns: 118 -> 62).
constexpr int UPD_NW = 4, UPD_C = 16, UPD_CTAS = 4;   // CTAs per SM: 3 / 4 / 5 give 156 / 158 / 182 ms (plate 64 / 62 / 70)

// CTAs of the rows a' < a: sum over m = 1..a of ceil(m / gb), gb = 2^lg
__host__ __device__ __forceinline__ long upd_first(int a, int lg)
{
    const long q = a >> lg, r = a & (1 << lg) - 1;
    return (q * (q + 1) / 2 << lg) + r * (q + 1);
}

__device__ __forceinline__ void upd_cp(float2 *dst, const float2 *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// row offset of block i inside stacked column j, found by one warp (-1 if absent): 32 probes, then the entries between two
__device__ __forceinline__ int find_row_warp(const int *sptr, const int *sidx, const int *srow, int j, int i)
{
    const int lane = threadIdx.x & 31, lo = sptr[j], len = sptr[j + 1] - lo, step = (len + 31) / 32;
    const int e = lane * step;
    const unsigned below = __ballot_sync(0xffffffffu, e < len && sidx[lo + e] <= i);
    if (!below) return -1;
    const int f = (31 - __clz(below)) * step;
    int found = -1;
    for (int g = f; g < f + step; g += 32) {   // one round for up to 1024 blocks
        const int x = g + lane;
        const unsigned hit = __ballot_sync(0xffffffffu, x < f + step && x < len && sidx[lo + x] == i);
        if (hit) found = g + 31 - __clz(hit);
    }
    return found < 0 ? -1 : srow[lo + found];
}

// C (nr x nc, nr <= 8 U, nc <= 4 V) -= A W: As[q * lda + r], Ws[c * nk + q], once landed() says they are there
template <int U, int V, class Landed>
__device__ __forceinline__ void upd_piece(const float2 *As, int lda, const float2 *Ws, int nk, int nr, int nc, float2 *C,
                                          int ldc, Landed &&landed)
{
    const int lr = threadIdx.x & 7, lc = (threadIdx.x & 31) >> 3;
    float2 old[U][V], acc[U][V];
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = lr + 8 * u, c = lc + 4 * v;
            old[u][v] = (r < nr && c < nc) ? C[r + (int64_t)c * ldc] : czero(float2());
            acc[u][v] = czero(float2());
        }
    landed();
    const float2 *ap = As + lr, *wp = Ws + lc * nk;
    for (int q = 0; q < nk; ++q) {
        float2 av[U], wv[V];
#pragma unroll
        for (int u = 0; u < U; ++u) av[u] = ap[q * lda + 8 * u];
#pragma unroll
        for (int v = 0; v < V; ++v) wv[v] = wp[4 * v * nk + q];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[u][v] = cfma(av[u], wv[v], acc[u][v]);
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = lr + 8 * u, c = lc + 4 * v;
            if (r < nr && c < nc) C[r + (int64_t)c * ldc] = make_float2(old[u][v].x - acc[u][v].x, old[u][v].y - acc[u][v].y);
        }
}

// entries of a warp's W buffer: UPD_C columns and the alignment of the first
__host__ __device__ __forceinline__ int upd_wcap(int nk) { return UPD_C * nk + 2; }
static size_t upd_smem(int nk, int lda) { return sizeof(float2) * ((size_t)nk * lda + 2 * UPD_NW * (size_t)upd_wcap(nk)); }

__global__ void __launch_bounds__(32 * UPD_NW, UPD_CTAS) k_update_grp(int k, int ns, int part, int lg, int lda, const int *size,
                                                                      const int *sptr, const int *sidx, const int *srow,
                                                                      const int *M, const int64_t *coff,
                                                                      const int64_t *doff, const float2 *W, float2 *A,
                                                                      float2 *Ad)
{
    extern __shared__ float2 upd_sm[];
    const long t = blockIdx.x;
    int lo = 0, hi = ns;   // largest a with upd_first(a) <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (upd_first(mid, lg) <= t) lo = mid;
        else hi = mid;
    }
    // UPD_FIRST: CTA = row, the warps share its block of column 0 (UPD_NW UPD_C = 64 columns at most)
    const bool one = part == UPD_FIRST;
    const int a = one ? (int)t : lo, b0 = one ? 0 : (int)(t - upd_first(a, lg)) << lg;
    const int b1 = one ? 1 : min(a + 1, b0 + (1 << lg));
    if (b0 > a || a >= ns) return;   // cannot happen: row a has ceil((a + 1) / gb) groups
    const int e0 = sptr[k] + (part == UPD_REST), i = sidx[e0 + a], nk = size[k], ni = size[i], Mk = M[k];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, cap = upd_wcap(nk);
    float2 *As = upd_sm;   // As[q * lda + r] = A_ik[r, q]
    float2 *const wb = upd_sm + nk * lda + 2 * wp * cap;
    const float2 *const Wk = W + coff[k];
    const float2 *Aik = A + coff[k] + srow[e0 + a];   // ld Mk; panel k is not written in this step
    for (int q = wp; q < nk; q += UPD_NW)
        for (int r = lane; r < ni; r += 32) upd_cp(As + q * lda + r, Aik + r + (int64_t)q * Mk);
    // this warp's pieces: columns [c0, c0 + UPD_C) of W_kj for b = b0 + wp, b0 + wp + UPD_NW, ...; the 16-byte words that
    // hold them (panel allocations end on 256 bytes)
    const int cstart = one ? wp * UPD_C : 0, cstep = one ? UPD_NW * UPD_C : UPD_C;
    int b = one ? (cstart < size[sidx[e0]] ? 0 : 1) : b0 + wp, c0 = cstart;
    auto stage = [&](int bb, int cc, int buf) {
        if (bb < b1) {
            const float2 *src = Wk + (srow[e0 + bb] + cc) * nk;
            const int rem = (int)((size_t)src >> 3 & 1), n16 = (rem + min(UPD_C, size[sidx[e0 + bb]] - cc) * nk + 1) / 2;
            const unsigned d = (unsigned)__cvta_generic_to_shared(wb + buf * cap);
            const char *g = (const char *)(src - rem);
#pragma unroll 4
            for (int x = lane; x < n16; x += 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16 * x), "l"(g + 16 * x) : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(b, c0, 0);   // one group with the A_ik copies
    float2 *C = nullptr;
    int ldc = 0;
    bool first = true;   // A_ik is still to be waited for, by the whole CTA
    for (int buf = 0; b < b1; buf ^= 1) {
        const int j = sidx[e0 + b], nj = size[j], nc = min(UPD_C, nj - c0);
        const bool last = c0 + cstep >= nj;
        const int bn = last ? b + UPD_NW : b, cn = last ? cstart : c0 + cstep;
        stage(bn, cn, buf ^ 1);
        if (c0 == cstart) {
            if (i == j) {
                C = Ad + doff[i];
                ldc = ni;
            } else {
                const int r = find_row_warp(sptr, sidx, srow, j, i);   // >= 0 when S is the symbolic fill
                C = r >= 0 ? A + coff[j] + r : nullptr;
                ldc = M[j];
            }
        }
        auto landed = [&]() {
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            if (first) __syncthreads();
            else __syncwarp();
            first = false;
        };
        const float2 *Ws = wb + buf * cap + ((size_t)(Wk + (srow[e0 + b] + c0) * nk) >> 3 & 1);
        for (int r0 = 0; r0 < ni; r0 += 32) {
            const int nr = C ? min(32, ni - r0) : 0;
            float2 *Cp = C + r0 + (int64_t)c0 * ldc;
            switch ((max(nr, 1) - 1 >> 3) * 4 + (nc - 1 >> 2)) {   // (U - 1) * 4 + (V - 1)
#define HM_UPD(U, V) \
    case (U - 1) * 4 + (V - 1): upd_piece<U, V>(As + r0, lda, Ws, nk, nr, nc, Cp, ldc, landed); break;
                HM_UPD(1, 1) HM_UPD(1, 2) HM_UPD(1, 3) HM_UPD(1, 4)
                HM_UPD(2, 1) HM_UPD(2, 2) HM_UPD(2, 3) HM_UPD(2, 4)
                HM_UPD(3, 1) HM_UPD(3, 2) HM_UPD(3, 3) HM_UPD(3, 4)
                HM_UPD(4, 1) HM_UPD(4, 2) HM_UPD(4, 3) HM_UPD(4, 4)
#undef HM_UPD
            default: break;   // pieces are 1..32 x 1..16
            }
        }
        __syncwarp();   // the buffer is restaged in the next turn
        b = bn;
        c0 = cn;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    if (first) __syncthreads();   // a warp without pieces
}

// Schur updates of step k on the tensor cores (complex-FP32 setup, update kind 2).  The step's
// products are one lower-triangular product of the stacked column [A_ik; i in S_k] (M_k x n_k)
// with the panel W_k (n_k x M_k): CTA t takes row block a of S_k (i = S_k[a], n_i rows) and 64
// consecutive columns of W_k among those of blocks b <= a (tasks of row a: ceil((srow_a + n_i) /
// 64), ucum[e0 + a] the tasks before row a).  C = A_ik W_k[:, c0 : c0 + nc] runs as tcgen05
// MMAs on 3xTF32 operands (tc::Acc, chunks of tc::KC along n_k); every output column is then
// subtracted from its block A_ij (j = the S_k block holding the column; the diagonal block in Ad
// when j = i).  Each output adds its n_k terms in one fixed order.
__global__ void __launch_bounds__(256) k_update_tc(int k, int ns, const int *ucum, const int *size, const int *sptr,
                                                   const int *sidx, const int *srow, const int *M, const int64_t *coff,
                                                   const int64_t *doff, const float2 *W, float2 *A, float2 *Ad,
                                                   int *err, unsigned long long bound)
{
    extern __shared__ unsigned char smraw[];
    __shared__ uint64_t s_mbar;
    __shared__ uint32_t s_tslot;
    __shared__ float2 *s_col[64];
    const int e0 = sptr[k], t = blockIdx.x;
    int lo = 0, hi = ns;   // row a: the largest with ucum[e0 + a] <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (ucum[e0 + mid] <= t) lo = mid;
        else hi = mid;
    }
    const int a = lo, i = sidx[e0 + a], ni = size[i], nk = size[k], Mk = M[k];
    const int c0 = (t - ucum[e0 + a]) * 64, nc = min(64, srow[e0 + a] + ni - c0);
    if (threadIdx.x < nc) {   // where output column c0 + x goes
        const int c = c0 + threadIdx.x;
        int l2 = 0, h2 = a + 1;   // block b holding column c: the largest with srow[e0 + b] <= c
        while (h2 - l2 > 1) {
            const int mid = (l2 + h2) >> 1;
            if (srow[e0 + mid] <= c) l2 = mid;
            else h2 = mid;
        }
        const int j = sidx[e0 + l2], cl = c - srow[e0 + l2];
        float2 *dst = nullptr;
        if (j == i) {
            dst = Ad + doff[i] + (int64_t)cl * ni;
        } else {
            const int r = find_row(sptr, sidx, srow, j, i);   // >= 0 when S is the symbolic fill
            if (r >= 0) dst = A + coff[j] + r + (int64_t)cl * M[j];
        }
        s_col[threadIdx.x] = dst;
    }
    tc::Acc acc;
    unsigned char *base = tc::align1024(smraw);
    acc.planes = base;
    acc.mbar = &s_mbar;
    acc.tslot = &s_tslot;
    acc.open(ni, nc);
    const float2 *Aik = A + coff[k] + srow[e0 + a];        // n_i x n_k, ld M_k (panel k is not written)
    const float2 *Wc = W + coff[k] + (int64_t)c0 * nk;     // n_k x nc, ld n_k
    for (int q0 = 0; q0 < nk; q0 += tc::KC) {
        const int kl = min(tc::KC, nk - q0);
        acc.wait(err, bound);   // the previous chunk's MMAs have read the planes
        for (int e = threadIdx.x; e < ni * kl; e += blockDim.x) {
            const int r = e % ni, q = e / ni;
            acc.put_a(r, q, Aik[r + (int64_t)(q0 + q) * Mk]);
        }
        for (int e = threadIdx.x; e < kl * nc; e += blockDim.x) {
            const int q = e % kl, c = e / kl;
            acc.put_b(c, q, Wc[(q0 + q) + (int64_t)c * nk]);
        }
        acc.zero_pad(kl);
        acc.issue(kl);
    }
    acc.wait(err, bound);
    float *dsm = (float *)base;
    if (acc.drain(dsm)) {
        for (int e = threadIdx.x; e < ni * nc; e += blockDim.x) {
            const int r = e % ni, c = e / ni;
            float2 *dst = s_col[c];
            if (dst) {
                const float2 v = acc.entry(dsm, r, c);
                float2 o = dst[r];
                o.x -= v.x;
                o.y -= v.y;
                dst[r] = o;
            }
        }
    }
    acc.close();
}

// Column blocks per CTA of the grouped update, as a power of two: as many as leave UPD_MIN CTAs per SM (A_ik is staged
// once for them), at least one and at most four per warp.  30,720-unknown sphere: 173, 166, 158, 158 ms for 3, 6, 12, 24.
constexpr int UPD_MIN = 12;
static int upd_group(int ns, int nsm)
{
    int lg = 4;
    while (lg > 2 && upd_first(ns, lg) < (long)UPD_MIN * nsm) --lg;
    return lg;
}

// count pivot blocks from k on, of at most nk unknowns, each on CL CTAs
template <class S, int CL>
static cudaError_t pivot_launch(hm_ctx *h, cudaStream_t st, int k, int count, int nk, const S *Ad, float2 *Dinv32)
{
    const size_t smem = sizeof(double2) * 2 * (size_t)nk * ((nk + CL - 1) / CL);
    static DeviceOnce attr;
    if (attr.need()) {
        const cudaError_t e = cudaFuncSetAttribute(k_pivot_inverse<S, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(double2) * 2 * 64 * (64 / CL)));
        if (e) return e;
        attr.done();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CL * count), 1, 1);
    cfg.blockDim = dim3(128, 1, 1);   // one warp per scheduler
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    cudaError_t e = cudaSuccess;
    HM_LAUNCH(h, K_PIVOT,
              e = cudaLaunchKernelEx(&cfg, k_pivot_inverse<S, CL>, k, (const int *)h->d_size, (const int64_t *)h->d_doff, Ad,
                                     h->d_Dinv, Dinv32, h->d_err));
    return e ? e : cudaGetLastError();
}

// One pivot block on h->pivot_cl CTAs.  By default on two up to 28 unknowns, where the pushes to more CTAs cost what
// their schedulers save (4,720-unknown plate, blocks of 18: 11.7 / 10.2 / 11.7 / 14.8 ms per setup on 1 / 2 /
// 4 / 8; 29,800-unknown plate, 29: 101 / 70 / 71 / 91), on four above (1,920-unknown sphere, 34: 11.5 / 7.2 /
// 5.1 / 6.6 ms; 30,720-unknown sphere: 175 / 113 / 83 / 105 ms).
template <class S>
static cudaError_t pivot_step(hm_ctx *h, cudaStream_t st, int k, int nk, const S *Ad, float2 *Dinv32)
{
    switch (h->pivot_cl ? h->pivot_cl : nk <= 28 ? 2 : 4) {
    case 2: return pivot_launch<S, 2>(h, st, k, 1, nk, Ad, Dinv32);
    case 4: return pivot_launch<S, 4>(h, st, k, 1, nk, Ad, Dinv32);
    case 8: return pivot_launch<S, 8>(h, st, k, 1, nk, Ad, Dinv32);
    default: return pivot_launch<S, 1>(h, st, k, 1, nk, Ad, Dinv32);
    }
}

// The stream of the pivots that run ahead.  Its work is over before the object is, on every way out.
struct Ahead {
    cudaStream_t st = nullptr;
    cudaEvent_t upd = nullptr, pan = nullptr;   // the next pivot's inputs are final; its panel is
    cudaError_t open()
    {
        int lo = 0, hi = 0;
        cudaError_t e;
        if ((e = cudaDeviceGetStreamPriorityRange(&lo, &hi)) ||
            (e = cudaStreamCreateWithPriority(&st, cudaStreamNonBlocking, hi)) ||
            (e = cudaEventCreateWithFlags(&upd, cudaEventDisableTiming)))
            return e;
        return cudaEventCreateWithFlags(&pan, cudaEventDisableTiming);
    }
    ~Ahead()
    {
        if (st) {
            cudaStreamSynchronize(st);
            cudaStreamDestroy(st);
        }
        if (upd) cudaEventDestroy(upd);
        if (pan) cudaEventDestroy(pan);
    }
};

template <class S>
static cudaError_t setup_typed(hm_ctx *h, S *A, S *Ad, S *W, S *DinvS, float2 *Dinv32, int *bad_block)
{
    Plan &P = h->plan;
    cudaStream_t st = h->stream;
    cudaError_t e;
    *bad_block = -1;
    if ((e = cudaMemsetAsync(A, 0, sizeof(S) * P.coef_entries, st))) return e;
    if ((e = cudaMemsetAsync(Ad, 0, sizeof(S) * P.diag_entries, st))) return e;
    if ((e = cudaMemsetAsync(h->d_err, 0, sizeof(int), st))) return e;
    HM_LAUNCH(h, K_SCATTER,
              k_scatter_near<S><<<(int)h->near_t.size(), 128, 0, st>>>(
                  (int)h->near_t.size(), h->d_near_t, h->d_near_s, h->d_near_off, h->d_near, h->d_leaf_ptr, h->d_pos,
                  h->d_sptr, h->d_sidx, h->d_srow, h->d_M, h->d_coff, h->d_doff, A, Ad, h->d_err));
    if ((e = cudaGetLastError())) return e;
    if ((e = cudaFuncSetAttribute(k_panel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)panel_smem<S>(64))))
        return e;
    if ((e = cudaFuncSetAttribute(k_update_grp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)upd_smem(64, 64)))) return e;
    int dev = 0, nsm = 0;
    if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev))) return e;
    const int maxn = *std::max_element(P.size.begin(), P.size.end()), lda = (maxn + 7) / 8 * 8;
    if ((e = cudaFuncSetAttribute(k_update64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(double2) * 2 * 64 * 64)))
        return e;
    if (sizeof(S) == 8 && h->update_kind == 2) {
        if (!h->d_ucum) {   // tensor-core update tasks: per row a of S_k, 64-column pieces of W_k
            std::vector<int> uc(std::max<size_t>(P.sidx.size(), 1));
            h->utot.assign(P.nb, 0);
            for (int k = 0; k < P.nb; ++k) {
                int c = 0;
                for (int x = P.sptr[k]; x < P.sptr[k + 1]; ++x) {
                    uc[x] = c;
                    c += (P.srow[x] + P.size[P.sidx[x]] + 63) / 64;
                }
                h->utot[k] = c;
            }
            if ((e = h->arena.alloc((void **)&h->d_ucum, sizeof(int) * uc.size())) ||
                (e = cudaMemcpyAsync(h->d_ucum, uc.data(), sizeof(int) * uc.size(), cudaMemcpyHostToDevice, st)) ||
                (e = cudaStreamSynchronize(st)))
                return e;
        }
        if ((e = cudaFuncSetAttribute(k_update_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::SMEM_BYTES)))
            return e;
    }
    // Look-ahead: the pivot and panel of block k + 1 run on a stream of their own once the first column of the updates
    // of step k is done, beside the others.  They occupy a few SMs for 85 us a step, the updates up to all of them:
    // 345 -> 302 ms per mixed setup of the 30,720-unknown sphere, 162 -> 130 of a 29,800-unknown plate, 35 -> 31 per FP64
    // setup of a 4,720-unknown plate.
    // Off where a launch is timed, where the panel is compressed before its updates and for the tensor-core updates.
    Ahead ahead;
    const bool on = P.nb > 1 && !h->prof.on && !h->opts.compress_in_setup && !(sizeof(S) == 8 && h->update_kind == 2);
    if (on && (e = ahead.open())) return e;
    const cudaStream_t ps = on ? ahead.st : st;
    auto factor = [&](int k) -> cudaError_t {   // pivot block k and its panel
        cudaError_t e2;
        if (on && ((e2 = cudaEventRecord(ahead.upd, st)) || (e2 = cudaStreamWaitEvent(ps, ahead.upd, 0)))) return e2;
        if ((e2 = pivot_step<S>(h, ps, k, P.size[k], Ad, Dinv32))) return e2;
        if (P.sptr[k + 1] > P.sptr[k])
            HM_LAUNCH(h, K_PANEL,
                      k_panel<S><<<(P.M[k] + PANEL_COLS<S> - 1) / PANEL_COLS<S>, 256, panel_smem<S>(P.size[k]), ps>>>(
                          k, h->d_size, h->d_M, h->d_coff, h->d_doff, DinvS, A, W));
        if ((e2 = cudaGetLastError())) return e2;
        return on ? cudaEventRecord(ahead.pan, ps) : cudaSuccess;
    };
    auto update = [&](int k, int ns, int part) -> cudaError_t {
        if (ns <= 0) return cudaSuccess;
        const int nk = P.size[k];
        if constexpr (sizeof(S) == 8) {
            const int lg = upd_group(ns, nsm);
            HM_LAUNCH(h, K_UPDATE,
                      k_update_grp<<<(unsigned)(part == UPD_FIRST ? ns : upd_first(ns, lg)), 32 * UPD_NW, upd_smem(nk, lda), st>>>(
                          k, ns, part, lg, lda, h->d_size, h->d_sptr, h->d_sidx, h->d_srow, h->d_M, h->d_coff, h->d_doff,
                          W, A, Ad));
        } else {
            const long nt = part == UPD_FIRST ? ns : (long)ns * (ns + 1) / 2;
            HM_LAUNCH(h, K_UPDATE,
                      k_update64<<<(unsigned)nt, UPD64_T, sizeof(double2) * 2 * maxn * nk, st>>>(
                          k, ns, part, h->d_size, h->d_sptr, h->d_sidx, h->d_srow, h->d_M, h->d_coff, h->d_doff, W, A, Ad));
        }
        return cudaGetLastError();
    };
    if ((e = factor(0))) return e;
    for (int k = 0; k < P.nb; ++k) {
        const int ns = P.sptr[k + 1] - P.sptr[k];
        if (on) {
            const bool next = ns > 0 && P.sidx[P.sptr[k]] == k + 1;
            if ((e = cudaStreamWaitEvent(st, ahead.pan, 0))) return e;
            if (next && (e = update(k, ns, UPD_FIRST))) return e;
            if (k + 1 < P.nb && (e = factor(k + 1))) return e;
            if ((e = next ? update(k, ns - 1, UPD_REST) : update(k, ns, UPD_ALL))) return e;
            continue;
        }
        if (ns > 0 && h->opts.compress_in_setup && (e = compress_step<S>(h, k, W))) return e;
        if constexpr (sizeof(S) == 8) {
            if (ns > 0 && h->update_kind == 2)
                HM_LAUNCH(h, K_UPDATE,
                          k_update_tc<<<(unsigned)h->utot[k], 256, tc::SMEM_BYTES, st>>>(
                              k, ns, h->d_ucum, h->d_size, h->d_sptr, h->d_sidx, h->d_srow, h->d_M, h->d_coff, h->d_doff,
                              W, A, Ad, h->d_err, WAIT_NS_DEFAULT));
        }
        if (!(sizeof(S) == 8 && h->update_kind == 2) && (e = update(k, ns, UPD_ALL))) return e;
        if (k + 1 < P.nb && (e = factor(k + 1))) return e;
    }
    int herr = 0;
    if ((e = cudaMemcpyAsync(&herr, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaStreamSynchronize(st))) return e;
    if (herr == 0x7fffffff) return cudaErrorInvalidValue;   // plan / pattern mismatch
    if (herr == ERR_TIMEOUT) return cudaErrorLaunchTimeout;   // a tensor-core wait gave up
    if (herr > 0) *bad_block = herr - 1;
    return cudaSuccess;
}

// Block Jacobi (Sec. 1's block diagonal preconditioner): D_k = Z_kk, all inverted at once.
cudaError_t block_jacobi_setup(hm_ctx *h, int *bad_block)
{
    Plan &P = h->plan;
    cudaStream_t st = h->stream;
    cudaError_t e;
    *bad_block = -1;
    if ((e = cudaMemsetAsync(h->d_Ad, 0, sizeof(double2) * P.diag_entries, st))) return e;
    if ((e = cudaMemsetAsync(h->d_err, 0, sizeof(int), st))) return e;
    HM_LAUNCH(h, K_SCATTER,
              k_scatter_near<double2><<<(int)h->near_t.size(), 128, 0, st>>>(
                  (int)h->near_t.size(), h->d_near_t, h->d_near_s, h->d_near_off, h->d_near, h->d_leaf_ptr, h->d_pos,
                  h->d_sptr, h->d_sidx, h->d_srow, h->d_M, h->d_coff, h->d_doff, (double2 *)nullptr, h->d_Ad, h->d_err,
                  true));
    if ((e = pivot_launch<double2, 1>(h, st, 0, P.nb, *std::max_element(P.size.begin(), P.size.end()), h->d_Ad, nullptr)))
        return e;
    if ((e = cudaGetLastError())) return e;
    int herr = 0;
    if ((e = cudaMemcpyAsync(&herr, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaStreamSynchronize(st))) return e;
    if (herr > 0 && herr != 0x7fffffff) *bad_block = herr - 1;
    return cudaSuccess;
}

cudaError_t setup_run(hm_ctx *h, int *bad_block)
{
    if (h->opts.precision == 1)
        return setup_typed<float2>(h, h->d_A32, h->d_Ad32, h->d_W32, h->d_Dinv32, h->d_Dinv32, bad_block);
    return setup_typed<double2>(h, h->d_A, h->d_Ad, h->d_W, h->d_Dinv, nullptr, bad_block);
}

}  // namespace hm
