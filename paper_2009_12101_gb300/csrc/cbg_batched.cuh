// cbg_batched.cuh -- batched GMRES(m): many independent systems in one persistent launch.
//
// Each system runs the same restarted Arnoldi process as the single-system path (Fig. 1
// with the explicit-residual recheck of Section 5.2), entirely on the device.  The
// launch uses thread-block clusters.  A cluster takes systems from a device work queue
// ordered by decreasing size.  Systems with at least `split_rows` rows are solved by the
// whole cluster (rows split across its blocks; sums through distributed shared memory
// and the hardware cluster barrier); once the queue reaches the small systems, every
// block takes its own systems and runs alone.  No block ever spins on a flag: all waits
// are __syncthreads or cluster barriers, which the hardware guarantees to complete.
//
// Per block, the block's rows of w live in shared memory as FP32 hi and lo planes; only
// the compressed basis, x and b are in HBM.
#pragma once
#include <cooperative_groups.h>

#include "cbg_kernels.cuh"

namespace cbg {

namespace cgx = cooperative_groups;

constexpr int BT_THREADS = 256;
constexpr int BT_MAXM = 64;          // largest restart length of the batched kernel
constexpr int BT_OK = 0, BT_NOT_CONVERGED = 1, BT_NONFINITE = -2;   // cbgmres.h status values

struct BatchSys {
    int n;                  // rows
    int ld;                 // padded rows of a basis column (multiple of 64)
    long long rp_off;       // offset of the system's n+1 row pointers
    long long nz_off;       // offset of its nonzeros (column indices are local)
    long long vec_off;      // offset of its b / x / dinv entries
    long long v_off;        // byte offset of its basis
    long long ch_off;       // offset of its sliced-ELL chunks (BatchArgs::sell_off)
    double pscale;          // 2^s normalising its per-step operator (largest |value| in [1, 2))
    double hscale;          // 2^-s: Hessenberg columns back to the unscaled operator
};

struct BatchOut {
    long long iters;
    long long restarts;
    double relres;
    int status;
    int pad0;
};

struct BatchArgs {
    const BatchSys* sys;
    const int* order;       // queue order (decreasing n)
    int nsys;
    int m;
    const int* rowptr;
    const int* col;
    const double* valp;     // A D^{-1} (Jacobi) or A
    const double* val;      // A
    const double* dinv;     // D^{-1} or null
    const float* valpdf;    // valp times each system's pscale as FP32 hi [nnz_all] then lo
                            // [nnz_all] planes for the per-step SpMV in double-float, or null
                            // (FP64 products)
    long long nnz_all;
    // the same planes in chunks of 32 rows (sliced ELL: entry k of the chunk's row l at
    // sell_off[chunk] + 32 k + l, shorter rows padded with zero values), or null.  Read with one
    // thread per row the CSR planes cost a cache line per lane and entry: most of the SM's
    // cache is shared memory here, so the lines did not survive to the row's next entry
    // (65,025 rows on 8 blocks, f32: 145,000 cycles per SpMV of 420,000 per step).
    const long long* sell_off;
    const int* sell_col;
    const float* sell_val;  // hi [entries], lo [entries]; f64 codes: null, sell_val64 instead
    const double* sell_val64;   // valp in the same order (FP64 products)
    long long sell_entries;
    double* const* io;      // io[0] = b (packed), io[1] = x (packed); device table
    unsigned char* V;
    BatchOut* out;
    unsigned int* queue;    // work-queue head (zeroed before every launch)
    double tol;
    long long maxit;
    double eps_bd;
    int split_rows;
    int max_rows_block;     // capacity of the shared-memory planes of w (rows, multiple of 16)
    int spmv_lanes;         // SpMV schedule: 1 = a thread per row (4 rows in flight), or 2, 4, 8
                            // lanes per row (the lanes split the row's nonzeros)
};

// shared-memory layout of one block (dynamic)
struct BtSmem {
    double H[(BT_MAXM + 1) * BT_MAXM];
    double g[BT_MAXM + 1], cs[BT_MAXM], sn[BT_MAXM], y[BT_MAXM + 1];
    double h[BT_MAXM + 1], u[BT_MAXM + 1], scale[BT_MAXM + 1];
    double red[BT_MAXM + 4];           // this block's partial sums (read by the cluster)
    double tot[BT_MAXM + 4];           // team totals
    alignas(16) double wred[BT_THREADS / 32][BT_MAXM + 4];   // (the dot: row splits' sums as float2; the
                                                             // axpy: the warps' norms)
    double inv, omega;                 // of the current step (formed by one thread: an FP64 instruction
    EncParams ep;                      // occupies the narrow pipe for a whole warp)
    int sys_idx;
    int stop;
    alignas(16) float w[1];            // w of this block's rows: hi plane, then lo plane
                                       // (max_rows_block entries each)
};

template <bool CLUSTER> struct Team {
    int rank, size;
    __device__ __forceinline__ void sync() const
    {
        if constexpr (CLUSTER) {
            __threadfence();
            cgx::this_cluster().sync();
        } else {
            __syncthreads();
        }
    }
    // tot[i] = sum over the team's blocks of red[i], i < k, in block order (identical in
    // every block).
    __device__ __forceinline__ void reduce(BtSmem* sm, int k) const
    {
        if constexpr (CLUSTER) {
            cgx::cluster_group cl = cgx::this_cluster();
            cl.sync();
            for (int i = threadIdx.x; i < k; i += BT_THREADS) {
                double t = 0.0;
                for (int r = 0; r < size; r++) t += cl.map_shared_rank(sm->red, r)[i];
                sm->tot[i] = t;
            }
            cl.sync();
        } else {
            __syncthreads();
            for (int i = threadIdx.x; i < k; i += BT_THREADS) sm->tot[i] = sm->red[i];
            __syncthreads();
        }
    }
};

// block-wide sum of per-thread values v[0..k) into sm->red[0..k) (fixed order)
template <int K>
__device__ __forceinline__ void block_sum(BtSmem* sm, const double (&v)[K], int k, int red_off)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < K; i++) {
        if (i >= k) break;
        double s = warp_sum(v[i]);
        if (lane == 0) sm->wred[warp][i] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += BT_THREADS) {
        double s = 0.0;
        for (int w = 0; w < BT_THREADS / 32; w++) s += sm->wred[w][i];
        sm->red[red_off + i] = s;
    }
    __syncthreads();
}

template <int FMT> struct BatchedSolver {
    static constexpr int BS = FmtInfo<FMT>::bytes;
    static constexpr int E = 16 / BS;
    static constexpr int NW = BT_THREADS / 32;
    static constexpr bool SCALED = FMT == I32 || FMT == I16 || FMT == BF16 || FMT == E4M3;   // encoding needs max |w|

    // ------------------------------------------------------------------ block kernels
    // w (own rows) = A_pc x  with x given by codes (column `col`, scaled) or FP64 array;
    // ws <- DF(w).  Returns the thread's sum of w^2.
    template <bool CODES>
    static __device__ double spmv(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                  const void* x, double xscale, const double* vals, bool residual)
    {
        const int* rp = a.rowptr + s.rp_off;
        const int* ci = a.col + s.nz_off;
        float* wl = sm->w + a.max_rows_block;
        const double* va = vals + s.nz_off;
        const double* bb = a.io[0] + s.vec_off;
        double ss = 0.0;
        constexpr int RW = 4;                              // rows per thread in flight
        for (int rb = r0 + threadIdx.x; rb < r1; rb += RW * BT_THREADS) {
            double t[RW];
            int p0[RW], p1[RW];
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = rb + q * BT_THREADS;
                t[q] = 0.0;
                p0[q] = r < r1 ? rp[r] : 0;
                p1[q] = r < r1 ? rp[r + 1] : 0;
            }
            int len = 0;
#pragma unroll
            for (int q = 0; q < RW; q++) len = max(len, p1[q] - p0[q]);
            for (int i = 0; i < len; i++) {
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const int p = p0[q] + i;
                    if (p < p1[q]) {
                        double xv;
                        if constexpr (CODES) xv = code_value<FMT>(x, ci[p]);
                        else xv = reinterpret_cast<const double*>(x)[ci[p]];
                        t[q] = __fma_rn(va[p], xv, t[q]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = rb + q * BT_THREADS;
                if (r < r1) {
                    double v = t[q];
                    if constexpr (CODES) v = __dmul_rn(v, xscale);
                    if (residual) v = __dsub_rn(bb[r], v);
                    float hi, lo;
                    split_f64(v, hi, lo);
                    sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                    ss = __fma_rn(v, v, ss);
                }
            }
        }
        return ss;
    }

    // The per-step w = A_pc v_j in double-float: every product val * code is formed as an
    // FP32 pair (TwoProd on the split values; exact for single-float codes up to the
    // rounding of the lo term) and summed with TwoSum; w goes to ws as its renormalised
    // pair and the sum of w^2 is accumulated in double-float, so no FP64 operation runs
    // per nonzero or per row (GB300's FP64 pipe is ~70x narrower than its FP32 pipe).
    // The planes hold the normalised operator 2^s A_pc.
    static __device__ double spmv_df(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                     const void* x, double xscale)
    {
        const int* rp = a.rowptr + s.rp_off;
        const int* ci = a.col + s.nz_off;
        float* wl = sm->w + a.max_rows_block;
        const float* vh = a.valpdf + s.nz_off;
        const float* vl = a.valpdf + a.nnz_all + s.nz_off;
        const bool xsplit = xscale != 1.0;                 // unit scale (float formats): no product
        float xsh = 1.f, xsl = 0.f;
        if (xsplit) split_f64(xscale, xsh, xsl);
        float ssS = 0.f, ssC = 0.f;
        constexpr int RW = 4;                              // rows per thread in flight
        for (int rb = r0 + threadIdx.x; rb < r1; rb += RW * BT_THREADS) {
            float S[RW], C[RW];
            int p0[RW], p1[RW];
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = rb + q * BT_THREADS;
                S[q] = 0.f;
                C[q] = 0.f;
                p0[q] = r < r1 ? rp[r] : 0;
                p1[q] = r < r1 ? rp[r + 1] : 0;
            }
            int len = 0;
#pragma unroll
            for (int q = 0; q < RW; q++) len = max(len, p1[q] - p0[q]);
            for (int i = 0; i < len; i++) {
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const int p = p0[q] + i;
                    if (p < p1[q]) {
                        float xh, xl;
                        xval_df<FMT>(x, ci[p], xh, xl);
                        if constexpr (SingleFloat<FMT>::value) df_mac(S[q], C[q], xh, vh[p], vl[p]);
                        else df_mac2(S[q], C[q], xh, xl, vh[p], vl[p]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = rb + q * BT_THREADS;
                if (r < r1) {
                    float hi, lo;
                    two_sum(S[q], C[q], hi, lo);             // renormalise
                    if (xsplit) {                            // (hi + lo) * (xsh + xsl)
                        const float p = __fmul_rn(hi, xsh);
                        float e = __fmaf_rn(hi, xsh, -p);
                        e = __fmaf_rn(hi, xsl, e);
                        e = __fmaf_rn(lo, xsh, e);
                        two_sum(p, e, hi, lo);
                    }
                    sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                    // w^2 = hi^2 + 2 hi lo to double-float accuracy
                    const float p = __fmul_rn(hi, hi);
                    float e = __fmaf_rn(hi, hi, -p);
                    e = __fmaf_rn(__fadd_rn(hi, hi), lo, e);
                    float t, te;
                    two_sum(ssS, p, t, te);
                    ssC = __fadd_rn(ssC, __fadd_rn(te, e));
                    ssS = t;
                }
            }
        }
        return df_to_double(ssS, ssC);
    }

    // End of the chunks r0 >> 5, ... of a block's rows [r0, r1).  A block's rows start at a multiple
    // of 32, except that a trailing rank of a cluster may own none (r0 = r1 = n): its r0 may lie
    // inside the last chunk, which belongs to another block.
    static __device__ __forceinline__ int sell_end(int r0, int r1) { return r1 > r0 ? (r1 + 31) >> 5 : r0 >> 5; }

    // spmv_df on the sliced-ELL planes: a warp takes four chunks of 32 rows at a time (a lane
    // per row), every load of columns and values is one contiguous 128-byte access, and the next
    // entries are loaded while the current ones' gathers are in flight.
    static __device__ double spmv_df_sell(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                          const void* x, double xscale)
    {
        constexpr int RW = 4;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        float* wl = sm->w + a.max_rows_block;
        const long long* off = a.sell_off + s.ch_off;
        const float* vhp = a.sell_val;
        const float* vlp = a.sell_val + a.sell_entries;
        const bool xsplit = xscale != 1.0;
        float xsh = 1.f, xsl = 0.f;
        if (xsplit) split_f64(xscale, xsh, xsl);
        float ssS = 0.f, ssC = 0.f;
        const int cb = r0 >> 5, ce = sell_end(r0, r1);
        for (int c0 = cb + warp * RW; c0 < ce; c0 += NW * RW) {
            float S[RW], C[RW], vh[RW], vl[RW];
            long long p[RW];
            int len[RW], c[RW], top = 0;
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const bool in = c0 + q < ce;
                const long long b = in ? __ldg(off + c0 + q) : 0, e = in ? __ldg(off + c0 + q + 1) : 0;
                p[q] = b + lane;
                len[q] = (int)((e - b) >> 5);
                top = max(top, len[q]);
                S[q] = C[q] = 0.f;
            }
            auto entries = [&](int i) {                            // column -1: no entry
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const bool in = i < len[q];
                    vh[q] = in ? __ldg(vhp + p[q]) : 0.f;
                    vl[q] = in ? __ldg(vlp + p[q]) : 0.f;
                    c[q] = in ? __ldg(a.sell_col + p[q]) : -1;
                    p[q] += 32;
                }
            };
            entries(0);
            for (int i = 0; i < top; i++) {
                float xh[RW], xl[RW], fh[RW], fl[RW];
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    xh[q] = xl[q] = 0.f;
                    fh[q] = vh[q];
                    fl[q] = vl[q];
                    if (c[q] >= 0) xval_df<FMT>(x, c[q], xh[q], xl[q]);
                }
                entries(i + 1);
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    if constexpr (SingleFloat<FMT>::value) df_mac(S[q], C[q], xh[q], fh[q], fl[q]);
                    else df_mac2(S[q], C[q], xh[q], xl[q], fh[q], fl[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = (c0 + q) * 32 + lane;
                if (r < r1 && c0 + q < ce) {
                    float hi, lo;
                    two_sum(S[q], C[q], hi, lo);                   // renormalise
                    if (xsplit) {
                        const float pr = __fmul_rn(hi, xsh);
                        float e = __fmaf_rn(hi, xsh, -pr);
                        e = __fmaf_rn(hi, xsl, e);
                        e = __fmaf_rn(lo, xsh, e);
                        two_sum(pr, e, hi, lo);
                    }
                    sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                    const float pr = __fmul_rn(hi, hi);
                    float e = __fmaf_rn(hi, hi, -pr);
                    e = __fmaf_rn(__fadd_rn(hi, hi), lo, e);
                    float t, te;
                    two_sum(ssS, pr, t, te);
                    ssC = __fadd_rn(ssC, __fadd_rn(te, e));
                    ssS = t;
                }
            }
        }
        return df_to_double(ssS, ssC);
    }

    // the same for f64 codes, which keep FP64 products
    static __device__ double spmv_sell64(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                         const double* x, double xscale)
    {
        constexpr int RW = 4;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        float* wl = sm->w + a.max_rows_block;
        const long long* off = a.sell_off + s.ch_off;
        double ss = 0.0;
        const int cb = r0 >> 5, ce = sell_end(r0, r1);
        for (int c0 = cb + warp * RW; c0 < ce; c0 += NW * RW) {
            double t[RW], v[RW];
            long long p[RW];
            int len[RW], c[RW], top = 0;
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const bool in = c0 + q < ce;
                const long long b = in ? __ldg(off + c0 + q) : 0, e = in ? __ldg(off + c0 + q + 1) : 0;
                p[q] = b + lane;
                len[q] = (int)((e - b) >> 5);
                top = max(top, len[q]);
                t[q] = 0.0;
            }
            auto entries = [&](int i) {
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const bool in = i < len[q];
                    v[q] = in ? __ldg(a.sell_val64 + p[q]) : 0.0;
                    c[q] = in ? __ldg(a.sell_col + p[q]) : -1;
                    p[q] += 32;
                }
            };
            entries(0);
            for (int i = 0; i < top; i++) {
                double xv[RW], f[RW];
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    f[q] = v[q];
                    xv[q] = c[q] >= 0 ? x[c[q]] : 0.0;
                }
                entries(i + 1);
#pragma unroll
                for (int q = 0; q < RW; q++) t[q] = __fma_rn(f[q], xv[q], t[q]);
            }
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = (c0 + q) * 32 + lane;
                if (r < r1 && c0 + q < ce) {
                    const double y = __dmul_rn(t[q], xscale);
                    float hi, lo;
                    split_f64(y, hi, lo);
                    sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                    ss = __fma_rn(y, y, ss);
                }
            }
        }
        return ss;
    }

    // The SpMVs above with L = a.spmv_lanes lanes per row (L = 2, 4, 8): the lanes of a
    // group take every L-th nonzero of the row and their partial sums meet in shuffles.
    // Groups walk the block's rows in warp-uniform passes, so every shuffle has the whole
    // warp.  Same results up to the order of each row's sum.
    template <bool CODES>
    static __device__ double spmv_lanes(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                        const void* x, double xscale, const double* vals, bool residual)
    {
        const int* rp = a.rowptr + s.rp_off;
        const int* ci = a.col + s.nz_off;
        float* wl = sm->w + a.max_rows_block;
        const double* va = vals + s.nz_off;
        const double* bb = a.io[0] + s.vec_off;
        const int L = a.spmv_lanes, lg = threadIdx.x & (L - 1), gpw = 32 / L;
        const int gw = (threadIdx.x & 31) / L, warp = threadIdx.x >> 5;
        double ss = 0.0;
        for (int base = r0 + warp * gpw; base < r1; base += (BT_THREADS / 32) * gpw) {
            const int r = base + gw;
            const bool valid = r < r1;
            double t = 0.0;
            if (valid) {
                const int p1 = rp[r + 1];
                for (int p = rp[r] + lg; p < p1; p += L) {
                    double xv;
                    if constexpr (CODES) xv = code_value<FMT>(x, ci[p]);
                    else xv = reinterpret_cast<const double*>(x)[ci[p]];
                    t = __fma_rn(va[p], xv, t);
                }
            }
            for (int o = L >> 1; o > 0; o >>= 1) t = __dadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
            if (valid && lg == 0) {
                double v = t;
                if constexpr (CODES) v = __dmul_rn(v, xscale);
                if (residual) v = __dsub_rn(bb[r], v);
                float hi, lo;
                split_f64(v, hi, lo);
                sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                ss = __fma_rn(v, v, ss);
            }
        }
        return ss;
    }

    static __device__ double spmv_df_lanes(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1,
                                           const void* x, double xscale)
    {
        const int* rp = a.rowptr + s.rp_off;
        const int* ci = a.col + s.nz_off;
        float* wl = sm->w + a.max_rows_block;
        const float* vh = a.valpdf + s.nz_off;
        const float* vl = a.valpdf + a.nnz_all + s.nz_off;
        const bool xsplit = xscale != 1.0;
        float xsh = 1.f, xsl = 0.f;
        if (xsplit) split_f64(xscale, xsh, xsl);
        const int L = a.spmv_lanes, lg = threadIdx.x & (L - 1), gpw = 32 / L;
        const int gw = (threadIdx.x & 31) / L, warp = threadIdx.x >> 5;
        float ssS = 0.f, ssC = 0.f;
        for (int base = r0 + warp * gpw; base < r1; base += (BT_THREADS / 32) * gpw) {
            const int r = base + gw;
            const bool valid = r < r1;
            float S = 0.f, C = 0.f;
            if (valid) {
                const int p1 = rp[r + 1];
                for (int p = rp[r] + lg; p < p1; p += L) {
                    float xh, xl;
                    xval_df<FMT>(x, ci[p], xh, xl);
                    if constexpr (SingleFloat<FMT>::value) df_mac(S, C, xh, vh[p], vl[p]);
                    else df_mac2(S, C, xh, xl, vh[p], vl[p]);
                }
            }
            for (int o = L >> 1; o > 0; o >>= 1) {
                const float S2 = __shfl_xor_sync(0xffffffffu, S, o), C2 = __shfl_xor_sync(0xffffffffu, C, o);
                df_add(S, C, S2, C2);
            }
            if (valid && lg == 0) {
                float hi, lo;
                two_sum(S, C, hi, lo);
                if (xsplit) {
                    const float p = __fmul_rn(hi, xsh);
                    float e = __fmaf_rn(hi, xsh, -p);
                    e = __fmaf_rn(hi, xsl, e);
                    e = __fmaf_rn(lo, xsh, e);
                    two_sum(p, e, hi, lo);
                }
                sm->w[r - r0] = hi;
                    wl[r - r0] = lo;
                const float p = __fmul_rn(hi, hi);
                float e = __fmaf_rn(hi, hi, -p);
                e = __fmaf_rn(__fadd_rn(hi, hi), lo, e);
                float t, te;
                two_sum(ssS, p, t, te);
                ssC = __fadd_rn(ssC, __fadd_rn(te, e));
                ssS = t;
            }
        }
        return df_to_double(ssS, ssC);
    }

    // 16 bytes of codes.  encode() writes the columns in this launch, and again in every cycle, so
    // the loads are coherent ones past L1 (ld.global.nc is for data that no one writes).
    static __device__ __forceinline__ uint4 codes16(const unsigned char* p)
    {
        return __ldcg(reinterpret_cast<const uint4*>(p));
    }

    // partial h_k = sum over own rows of dec(V_k) w, k < ncols, into sm->red[0..ncols) (scale
    // applied).  Warps are dealt out as row splits x groups of eight columns so that the
    // slowest has the fewest (group, segment of 32 chunks) items; a warp reads its rows of w
    // once for the eight columns (one column per warp read them from shared memory per
    // column, with bank conflicts, and left warps idle while the basis was short).  Halves of
    // a group are software-pipelined.
    static __device__ void dot(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1, int ncols)
    {
        constexpr int CG = 8, H = CG / 2;
        static_assert(NW == 8, "the deal below assumes eight warps");
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const long long vstride = (long long)s.ld * BS;
        const unsigned char* vs = a.V + s.v_off + (long long)r0 * BS;
        const int nch = (r1 - r0 + E - 1) / E, nseg = (nch + 31) >> 5, ngroups = (ncols + CG - 1) / CG;
        const float* wl = sm->w + a.max_rows_block;
        float2* red = reinterpret_cast<float2*>(&sm->wred[0][0]);
        constexpr int RS = BT_MAXM + 4;
        int lc = 0, best = 0x7fffffff;
#pragma unroll
        for (int c = 0; c <= 3; c++) {                         // 2^c column groups at a time
            const int items = ((ngroups + (1 << c) - 1) >> c) * ((nseg + (NW >> c) - 1) >> (3 - c));
            if (items <= best) {
                best = items;
                lc = c;
            }
        }
        const int wc = 1 << lc, lr = 3 - lc, wr = 1 << lr, mc = warp >> lr, mr = warp & (wr - 1);
        for (int g = mc; g < ngroups; g += wc) {
            const int c0 = g * CG, nc = ncols - c0 < CG ? ncols - c0 : CG;
            float2 S2[CG / 2], C2[CG / 2];
#pragma unroll
            for (int q = 0; q < CG / 2; q++) { S2[q] = make_float2(0.f, 0.f); C2[q] = make_float2(0.f, 0.f); }
            const unsigned char* vc = vs + (long long)c0 * vstride;
            auto fetch = [&](int ch, int q0, uint4 (&raw)[H]) {
                const unsigned char* p = vc + (long long)q0 * vstride + ch * 16;
#pragma unroll
                for (int q = 0; q < H; q++) {
                    raw[q] = ch < nch && q0 + q < nc ? codes16(p) : make_uint4(0u, 0u, 0u, 0u);
                    p += vstride;
                }
            };
            int ch = mr * 32 + lane;
            uint4 ra[H], rb[H];
            fetch(ch, 0, ra);
            for (int sg = mr; sg < nseg; sg += wr) {
                const int r = ch < nch ? ch * E : 0;
                fetch(ch, H, rb);
                float xh[E], xl[E];
#pragma unroll
                for (int e = 0; e < E; e += 2) {
                    const float2 h2 = *reinterpret_cast<const float2*>(sm->w + r + e);
                    const float2 l2 = *reinterpret_cast<const float2*>(wl + r + e);
                    xh[e] = h2.x; xh[e + 1] = h2.y; xl[e] = l2.x; xl[e + 1] = l2.y;
                }
                auto accumulate = [&](const uint4& u0, const uint4& u1, float2& S, float2& C) {
                    Chunk<FMT> k0, k1;
                    decode_chunk<FMT>(u0, k0);
                    decode_chunk<FMT>(u1, k1);
#pragma unroll
                    for (int e = 0; e < E; e++) {
                        const float2 w2 = make_float2(xh[e], xh[e]), nw2 = make_float2(-xh[e], -xh[e]);
                        const float2 l2 = make_float2(xl[e], xl[e]);
                        if constexpr (SingleFloat<FMT>::value)
                            df2_mac(S, C, make_float2(k0.vh[e], k1.vh[e]), w2, nw2, l2);
                        else
                            df2_mac2(S, C, make_float2(k0.vh[e], k1.vh[e]), make_float2(k0.vl[e], k1.vl[e]), w2, nw2, l2);
                    }
                    df2_renorm(S, C);
                };
#pragma unroll
                for (int q = 0; q < H; q += 2)
                    if (q < nc) accumulate(ra[q], ra[q + 1], S2[q / 2], C2[q / 2]);
                ch += wr * 32;
                fetch(ch, 0, ra);
#pragma unroll
                for (int q = 0; q < H; q += 2)
                    if (H + q < nc) accumulate(rb[q], rb[q + 1], S2[(H + q) / 2], C2[(H + q) / 2]);
            }
            float S[CG], C[CG];
#pragma unroll
            for (int q = 0; q < CG / 2; q++) {
                S[2 * q] = S2[q].x; S[2 * q + 1] = S2[q].y;
                C[2 * q] = C2[q].x; C[2 * q + 1] = C2[q].y;
            }
            const int col = df_warp_fold<CG>(S, C, lane);
            if ((lane & fold_low<CG>()) == 0 && col < nc) red[mr * RS + c0 + col] = make_float2(S[0], C[0]);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < ncols; c += BT_THREADS) {
            float2 t = red[c];
            for (int k = 1; k < wr; k++) df_add(t.x, t.y, red[k * RS + c].x, red[k * RS + c].y);
            sm->red[c] = __dmul_rn(df_to_double(t.x, t.y), sm->scale[c]);
        }
        __syncthreads();
    }

    // e with omega < 2^e, within the float exponents; 0 for zero and what is not finite
    static __device__ __forceinline__ int norm_exponent(double omega)
    {
        const int e = ((__double2hiint(omega) >> 20) & 0x7FF) - 1022;
        return e == -1022 || e == 1025 ? 0 : max(-126, min(126, e));
    }

    // w -= V coef over own rows; with NORMS, also the block's sum of squares (triples of floats,
    // tf_add, into sm->red[0]) and, for the formats whose scale needs it, the maximum of |w| (into
    // sm->red[1]).  Blocks with fewer row chunks than threads split the columns over the
    // lanes of a warp; the column loads are software-pipelined.
    template <bool NORMS>
    static __device__ void axpy(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1, int ncols,
                                const double* coef)
    {
        __shared__ float2 cdf[BT_MAXM + 1];
        float4* wsum = reinterpret_cast<float4*>(&sm->wred[0][0]);     // (shared memory bounds the systems' size)
        float2* wmax = reinterpret_cast<float2*>(wsum + NW);
        for (int k = threadIdx.x; k < ncols; k += BT_THREADS) {
            float hi, lo;
            split_f64(-coef[k] * sm->scale[k], hi, lo);
            cdf[k] = make_float2(hi, lo);
        }
        __syncthreads();
        constexpr int U = 4;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int nloc = r1 - r0, nch = (nloc + E - 1) / E;
        const long long vstride = (long long)s.ld * BS;
        const unsigned char* vs = a.V + s.v_off + (long long)r0 * BS;
        float* wl = sm->w + a.max_rows_block;
        int lk = 0;                                            // 2^lk column splits
        while (lk < 3 && (nch << (lk + 1)) <= BT_THREADS) lk++;
        const int ks = 1 << lk, cpw = 32 >> lk, mk = lane >> (5 - lk), mch = lane & (cpw - 1);
        float4 ss = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 mx = make_float2(0.f, 0.f);
        // the squares are taken of w 2^-e with omega < 2^e: an operator whose largest value is so small
        // that it could not be normalised would have them underflow in FP32
        const int e = NORMS ? norm_exponent(sm->omega) : 0;
        const float down = __int_as_float((127 - e) << 23);
        for (int base = warp * cpw; base < nch; base += NW * cpw) {
            const int ch = base + mch;
            const bool in = ch < nch;
            float2 S2[E / 2], C2[E / 2];
#pragma unroll
            for (int e = 0; e < E / 2; e++) { S2[e] = make_float2(0.f, 0.f); C2[e] = make_float2(0.f, 0.f); }
            const unsigned char* cp = vs + (long long)ch * 16;
            auto fetch = [&](int k0, uint4 (&raw)[U]) {
                const unsigned char* p = cp + (long long)k0 * vstride;
#pragma unroll
                for (int q = 0; q < U; q++) {
                    raw[q] = in && k0 + q * ks < ncols ? codes16(p) : make_uint4(0u, 0u, 0u, 0u);
                    p += ks * vstride;
                }
            };
            // (a column past the last has zero codes and adds exact zeros)
            auto accumulate = [&](int k0, const uint4 (&raw)[U]) {
#pragma unroll
                for (int q = 0; q < U; q++) {
                    Chunk<FMT> cd;
                    decode_chunk<FMT>(raw[q], cd);
                    const float2 c = k0 + q * ks < ncols ? cdf[k0 + q * ks] : make_float2(0.f, 0.f);
                    const float2 ch2 = make_float2(c.x, c.x), nch2 = make_float2(-c.x, -c.x), cl2 = make_float2(c.y, c.y);
#pragma unroll
                    for (int e = 0; e < E; e += 2) {
                        if constexpr (SingleFloat<FMT>::value)
                            df2_mac(S2[e / 2], C2[e / 2], make_float2(cd.vh[e], cd.vh[e + 1]), ch2, nch2, cl2);
                        else
                            df2_mac2(S2[e / 2], C2[e / 2], make_float2(cd.vh[e], cd.vh[e + 1]),
                                     make_float2(cd.vl[e], cd.vl[e + 1]), ch2, nch2, cl2);
                    }
                }
#pragma unroll
                for (int e = 0; e < E / 2; e++) df2_renorm(S2[e], C2[e]);
            };
            uint4 ra[U], rb[U];
            fetch(mk, ra);
            for (int k0 = mk; k0 - mk < ncols; k0 += 2 * U * ks) {   // (the same trips for every lane)
                fetch(k0 + U * ks, rb);
                accumulate(k0, ra);
                if (k0 - mk + U * ks >= ncols) break;
                fetch(k0 + 2 * U * ks, ra);
                accumulate(k0 + U * ks, rb);
            }
#pragma unroll
            for (int e = 0; e < E; e++) {
                float S = e & 1 ? S2[e / 2].y : S2[e / 2].x, C = e & 1 ? C2[e / 2].y : C2[e / 2].x;
                for (int o = cpw; o < 32; o <<= 1) {
                    const float oS = __shfl_xor_sync(0xffffffffu, S, o), oC = __shfl_xor_sync(0xffffffffu, C, o);
                    df_add(S, C, oS, oC);
                }
                const int r = ch * E + e;
                if (in && mk == 0 && r < nloc) {
                    df_add(S, C, sm->w[r], wl[r]);
                    float h, l;
                    two_sum(S, C, h, l);
                    sm->w[r] = h;
                    wl[r] = l;
                    if constexpr (NORMS) {
                        // h^2 = p + q and 2 h l = t + u exactly, l^2
                        const float hs = __fmul_rn(h, down), ls = __fmul_rn(l, down);
                        const float p = __fmul_rn(hs, hs), q = __fmaf_rn(hs, hs, -p);
                        const float h2 = __fadd_rn(hs, hs), t = __fmul_rn(h2, ls), u = __fmaf_rn(h2, ls, -t);
                        float y, z;
                        two_sum(t, q, y, z);
                        tf_add(ss, p, y, __fadd_rn(z, __fmaf_rn(ls, ls, u)));
                        if constexpr (SCALED) {
                            const float ah = fabsf(h), al = h < 0.f ? -l : l;
                            if (!(ah < mx.x || (ah == mx.x && al <= mx.y))) mx = make_float2(ah, al);
                        }
                    }
                }
            }
        }
        if constexpr (NORMS) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                tf_add(ss, tf_shfl_xor(ss, o));
                if constexpr (SCALED) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, mx.x, o), l2 = __shfl_xor_sync(0xffffffffu, mx.y, o);
                    if (!(h2 < mx.x || (h2 == mx.x && l2 <= mx.y))) mx = make_float2(h2, l2);
                }
            }
            if (lane == 0) {
                wsum[warp] = ss;
                wmax[warp] = mx;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                float4 t = wsum[0];
                float2 m = wmax[0];
                for (int w = 1; w < NW; w++) {
                    tf_add(t, wsum[w]);
                    if (!(wmax[w].x < m.x || (wmax[w].x == m.x && wmax[w].y <= m.y))) m = wmax[w];
                }
                sm->red[0] = __dmul_rn(tf_to_double<true>(t), pow2d(2 * e));
                sm->red[1] = df_to_double(m.x, m.y);
            }
        }
        __syncthreads();
    }

    // store v = w * inv (own rows) into basis column `col`
    static __device__ void encode(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int r0, int r1, int col,
                                  double inv, const EncParams& ep)
    {
        unsigned char* dst = a.V + s.v_off + (long long)col * s.ld * BS;
        const float* wl = sm->w + a.max_rows_block;
        for (int r = r0 + threadIdx.x; r < r1; r += BT_THREADS)
            encode_store<FMT>(dst, r, __dmul_rn(df_to_double(sm->w[r - r0], wl[r - r0]), inv), ep);
    }

    // Warp 0: column j of the Hessenberg matrix (scaled back from the normalised operator,
    // exactly), the previous rotations, the new one, g and the stopping tests.  The rotations
    // form a first-order recurrence in the carried entry, evaluated as a warp scan of affine maps
    // (as in the single-system store kernel) instead of a chain of j dependent steps.
    static __device__ void givens(const BatchArgs& a, const BatchSys& s, BtSmem* sm, int j, int kcap, double target)
    {
        const int lane = threadIdx.x & 31, m = a.m;
        double* Hc = sm->H + j * (m + 1);
        const double hn = sqrt(sm->tot[0]), hnt = __dmul_rn(hn, s.hscale);
        const int K = (j + 31) / 32, i0 = min(lane * K, j), i1 = min(i0 + K, j);   // K <= 2
        double hv[3], A = 1.0, B = 0.0;                        // entries i0 .. i1 of the raw column
#pragma unroll
        for (int q = 0; q < 3; q++)
            hv[q] = i0 + q <= j && q <= K ? __dmul_rn(__dadd_rn(sm->h[i0 + q], sm->u[i0 + q]), s.hscale) : 0.0;
        const double h0 = __shfl_sync(0xffffffffu, hv[0], 0);
        for (int i = i0; i < i1; i++) {
            const double ai = -sm->sn[i], bi = __dmul_rn(sm->cs[i], i == i0 ? hv[1] : hv[2]);
            B = __fma_rn(ai, B, bi);
            A = __dmul_rn(ai, A);
        }
        double PA = A, PB = B;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double qa = __shfl_up_sync(0xffffffffu, PA, o), qb = __shfl_up_sync(0xffffffffu, PB, o);
            if (lane >= o) {
                PB = __fma_rn(PA, qb, PB);
                PA = __dmul_rn(PA, qa);
            }
        }
        double EA = __shfl_up_sync(0xffffffffu, PA, 1), EB = __shfl_up_sync(0xffffffffu, PB, 1);
        if (lane == 0) { EA = 1.0; EB = 0.0; }
        double x = __fma_rn(EA, h0, EB);                       // carried entry entering this lane's rotations
        for (int i = i0; i < i1; i++) {
            const double c = sm->cs[i], sn = sm->sn[i], h1 = i == i0 ? hv[1] : hv[2];
            Hc[i] = __dadd_rn(__dmul_rn(c, x), __dmul_rn(sn, h1));
            x = __dadd_rn(__dmul_rn(-sn, x), __dmul_rn(c, h1));
        }
        const double xl = __shfl_sync(0xffffffffu, x, j > 0 ? (j - 1) / K : 0);
        if (lane == 0) {
            const double r0v = j > 0 ? xl : h0;
            const double rr = hypot(r0v, hnt);
            double c = 1.0, sn = 0.0;
            if (rr != 0.0) {
                const double ri = 1.0 / rr;
                c = __dmul_rn(r0v, ri);
                sn = __dmul_rn(hnt, ri);
                if (!isfinite(ri)) {                           // a subnormal rr
                    c = r0v / rr;
                    sn = hnt / rr;
                }
            }
            sm->cs[j] = c;
            sm->sn[j] = sn;
            Hc[j] = rr;
            Hc[j + 1] = 0.0;
            const double gj = sm->g[j];
            sm->g[j + 1] = __dmul_rn(-sn, gj);
            sm->g[j] = __dmul_rn(c, gj);
            const double est = fabs(sm->g[j + 1]);
            int stop = 0;
            if (!isfinite(hnt) || !isfinite(sm->omega) || !isfinite(est)) stop = 3;
            else if (!(hn > a.eps_bd * sm->omega)) stop = 2;   // both of the scaled operator
            else if (est <= target) stop = 1;
            else if (j + 1 >= kcap) stop = 4;
            sm->stop = stop;
        }
    }

    // --------------------------------------------------------------------- one system
    template <bool CLUSTER>
    static __device__ void solve(const BatchArgs& a, int si, BtSmem* sm, const Team<CLUSTER>& team)
    {
        const BatchSys s = a.sys[si];
        const int m = a.m;
        const int chunk = ((s.n + team.size - 1) / team.size + 31) / 32 * 32;   // whole sliced-ELL chunks
        const int r0 = min(s.n, team.rank * chunk);
        const int r1 = min(s.n, r0 + chunk);
        const int nloc = r1 - r0;
        float* wl = sm->w + a.max_rows_block;
        // zero the w rows, and those up to the next 16, which the chunked loops read
        for (int i = threadIdx.x; i < (nloc + 15) / 16 * 16; i += BT_THREADS) sm->w[i] = wl[i] = 0.f;
        double* x = a.io[1] + s.vec_off;
        const double* dinv = a.dinv ? a.dinv + s.vec_off : nullptr;

        // ||b||
        {
            double v[1] = {0.0};
            for (int r = r0 + threadIdx.x; r < r1; r += BT_THREADS) {
                const double bv = a.io[0][s.vec_off + r];
                v[0] = __fma_rn(bv, bv, v[0]);
            }
            block_sum<1>(sm, v, 1, 0);
            team.reduce(sm, 1);
        }
        const double bnorm = sqrt(sm->tot[0]);
        long long iters = 0, cycles = 0;
        int status = BT_NOT_CONVERGED;
        double beta = 0.0;
        if (bnorm == 0.0) {
            for (int r = r0 + threadIdx.x; r < r1; r += BT_THREADS) x[r] = 0.0;
            status = 0;
        } else {
            const double target = a.tol * bnorm;
            for (;;) {
                // residual r = b - A x into ws; beta, ||r||_inf
                team.sync();                                   // x of all blocks visible
                double v[2];
                v[0] = a.spmv_lanes > 1 ? spmv_lanes<false>(a, s, sm, r0, r1, x, 1.0, a.val, true)
                                        : spmv<false>(a, s, sm, r0, r1, x, 1.0, a.val, true);
                v[1] = 0.0;
                double mxl = 0.0;
                for (int r = r0 + threadIdx.x; r < r1; r += BT_THREADS) {
                    mxl = fmax(mxl, fabs(df_to_double(sm->w[r - r0], wl[r - r0])));
                }
                {
                    __syncthreads();
                    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
                    double s2 = warp_sum(v[0]), m2 = warp_max(mxl);
                    if (lane == 0) { sm->wred[warp][0] = s2; sm->wred[warp][1] = m2; }
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        double t = 0.0, mm = 0.0;
                        for (int w = 0; w < BT_THREADS / 32; w++) { t += sm->wred[w][0]; mm = fmax(mm, sm->wred[w][1]); }
                        sm->red[0] = t;
                        sm->red[1] = mm;
                    }
                }
                // the max is combined through the same fixed-order path (sum of block maxima
                // is not needed: take the max over blocks explicitly)
                team.reduce(sm, 1);
                beta = sqrt(sm->tot[0]);
                double rinf = sm->red[1];
                if constexpr (CLUSTER) {
                    cgx::cluster_group cl = cgx::this_cluster();
                    for (int r = 0; r < team.size; r++) rinf = fmax(rinf, cl.map_shared_rank(sm->red, r)[1]);
                    cl.sync();
                }
                if (!(beta > target)) { status = isfinite(beta) ? 0 : BT_NONFINITE; break; }
                if (iters >= a.maxit) { status = BT_NOT_CONVERGED; break; }
                cycles++;
                const long long left = a.maxit - iters;
                const int kcap = (int)(left < m ? left : m);
                // v_1 = r / beta
                {
                    const double inv = 1.0 / beta;
                    const EncParams ep = enc_params(FMT, __dmul_rn(rinf, inv));
                    if (threadIdx.x == 0) sm->scale[0] = ep.scale;
                    encode(a, s, sm, r0, r1, 0, inv, ep);
                }
                for (int i = threadIdx.x; i <= m; i += BT_THREADS) { sm->g[i] = 0.0; sm->y[i] = 0.0; }
                if (threadIdx.x == 0) sm->g[0] = beta;
                int k = 0;
                for (int j = 0; j < kcap; j++) {
                    team.sync();                               // column j of all blocks visible
                    // w = 2^s A D^{-1} v_j (the normalised operator; Jacobi folded into the
                    // values), omega = ||w||.  Double-float products unless the planes are
                    // absent; f64 codes keep FP64 products, which measured faster than
                    // splitting every gathered code.
                    double om[1];
                    const unsigned char* vj = a.V + s.v_off + (long long)j * s.ld * BS;
                    const double xs = __dmul_rn(sm->scale[j], s.pscale);
                    if (FMT != F64 && a.valpdf)                  // planes hold 2^s A_pc
                        om[0] = a.spmv_lanes > 1 ? spmv_df_lanes(a, s, sm, r0, r1, vj, sm->scale[j])
                                : a.sell_off ? spmv_df_sell(a, s, sm, r0, r1, vj, sm->scale[j])
                                             : spmv_df(a, s, sm, r0, r1, vj, sm->scale[j]);
                    else if (FMT == F64 && a.spmv_lanes == 1 && a.sell_val64)
                        om[0] = spmv_sell64(a, s, sm, r0, r1, reinterpret_cast<const double*>(vj), xs);
                    else
                        om[0] = a.spmv_lanes > 1 ? spmv_lanes<true>(a, s, sm, r0, r1, vj, xs, a.valp, false)
                                                 : spmv<true>(a, s, sm, r0, r1, vj, xs, a.valp, false);
                    __syncthreads();
                    block_sum<1>(sm, om, 1, j + 1);              // red[j+1] = omega^2 partial
                    dot(a, s, sm, r0, r1, j + 1);                // red[0..j]
                    team.reduce(sm, j + 2);
                    if (threadIdx.x == BT_THREADS - 1) sm->omega = sqrt(sm->tot[j + 1]);
                    for (int i = threadIdx.x; i <= j; i += BT_THREADS) sm->h[i] = sm->tot[i];
                    __syncthreads();
                    axpy<false>(a, s, sm, r0, r1, j + 1, sm->h);           // (norms of w1 unused)
                    dot(a, s, sm, r0, r1, j + 1);
                    team.reduce(sm, j + 1);
                    for (int i = threadIdx.x; i <= j; i += BT_THREADS) sm->u[i] = sm->tot[i];
                    __syncthreads();
                    axpy<true>(a, s, sm, r0, r1, j + 1, sm->u);
                    team.reduce(sm, 1);
                    if constexpr (CLUSTER && SCALED) {
                        cgx::cluster_group cl = cgx::this_cluster();
                        if (threadIdx.x == 0) {
                            double wmax = sm->red[1];
                            for (int r = 0; r < team.size; r++) wmax = fmax(wmax, cl.map_shared_rank(sm->red, r)[1]);
                            sm->tot[1] = wmax;
                        }
                        cl.sync();
                    }
                    // Hessenberg column, Givens rotations, stopping tests (warp 0) and what the
                    // encoding needs (warp 1), identical in every block
                    if (threadIdx.x < 32) {
                        givens(a, s, sm, j, kcap, target);
                    } else if (threadIdx.x == 32) {
                        const double inv = 1.0 / sqrt(sm->tot[0]);
                        sm->inv = inv;
                        sm->ep = enc_params(FMT, SCALED ? __dmul_rn(CLUSTER ? sm->tot[1] : sm->red[1], inv) : 1.0);
                    }
                    __syncthreads();
                    iters++;
                    k = j + 1;
                    if (sm->stop) break;
                    const double inv = sm->inv;
                    const EncParams ep = sm->ep;
                    if (threadIdx.x == 0) sm->scale[j + 1] = ep.scale;
                    encode(a, s, sm, r0, r1, j + 1, inv, ep);
                }
                if (sm->stop == 3) { status = BT_NONFINITE; break; }
                // y = R^{-1} g (Hessenberg columns hold R after the rotations)
                if (threadIdx.x == 0) {
                    for (int i = k - 1; i >= 0; i--) {
                        double t = sm->g[i];
                        for (int c2 = i + 1; c2 < k; c2++) t = __dsub_rn(t, __dmul_rn(sm->H[i + c2 * (m + 1)], sm->y[c2]));
                        sm->y[i] = t / sm->H[i + i * (m + 1)];
                    }
                }
                __syncthreads();
                // x += D^{-1} V y over own rows (the scales folded into y: one FP64 FMA per element)
                for (int i = threadIdx.x; i < k; i += BT_THREADS) sm->h[i] = __dmul_rn(sm->scale[i], sm->y[i]);
                __syncthreads();
                {
                    const unsigned char* Vs = a.V + s.v_off;
                    for (int r = r0 + threadIdx.x; r < r1; r += BT_THREADS) {
                        double t = 0.0;
                        for (int c2 = 0; c2 < k; c2++)
                            t = __fma_rn(code_value<FMT>(Vs + (long long)c2 * s.ld * BS, r), sm->h[c2], t);
                        if (dinv) t = __dmul_rn(dinv[r], t);
                        x[r] = __dadd_rn(x[r], t);
                    }
                }
            }
        }
        if (team.rank == 0 && threadIdx.x == 0) {
            a.out[si].iters = iters;
            a.out[si].restarts = cycles;
            a.out[si].relres = bnorm > 0.0 ? beta / bnorm : 0.0;
            a.out[si].status = status;
        }
        team.sync();
    }
};

template <int FMT>
__global__ void __launch_bounds__(BT_THREADS, 2) k_batched(BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char bt_smem_raw[];
    BtSmem* sm = reinterpret_cast<BtSmem*>(bt_smem_raw);
    cgx::cluster_group cl = cgx::this_cluster();
    const int crank = (int)cl.block_rank(), csize = (int)cl.num_blocks();
    int mine = -1;
    // cluster phase: large systems, one cluster each
    for (;;) {
        if (crank == 0 && threadIdx.x == 0) sm->sys_idx = (int)atomicAdd(a.queue, 1u);
        cl.sync();
        const int idx = *cl.map_shared_rank(&sm->sys_idx, 0);
        cl.sync();
        if (idx >= a.nsys) return;                           // every block of the cluster leaves together
        const int si = a.order[idx];
        if (csize > 1 && a.sys[si].n >= a.split_rows) {
            Team<true> t{crank, csize};
            BatchedSolver<FMT>::template solve<true>(a, si, sm, t);
            continue;
        }
        mine = crank == 0 ? si : -1;                         // small systems from here on
        break;
    }
    // block phase: small systems, one block each (no cluster-wide operation any more)
    for (;;) {
        if (mine < 0) {
            __syncthreads();
            if (threadIdx.x == 0) sm->sys_idx = (int)atomicAdd(a.queue, 1u);
            __syncthreads();
            const int idx = sm->sys_idx;
            if (idx >= a.nsys) return;
            mine = a.order[idx];
        }
        Team<false> t{0, 1};
        BatchedSolver<FMT>::template solve<false>(a, mine, sm, t);
        mine = -1;
    }
}

}  // namespace cbg
