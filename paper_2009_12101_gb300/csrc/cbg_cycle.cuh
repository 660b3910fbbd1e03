// cbg_cycle.cuh -- one restart cycle of the Arnoldi process (Fig. 1) in a single cooperative
// launch, for matrices whose steps are bound by launch and synchronisation latency rather
// than by HBM.
//
// The stepwise path issues five dependent kernels per Arnoldi step; each costs 7-17 us on
// GB300 however few rows there are (launch, ramp, one grid-wide sum, drain).  Here the
// blocks stay resident for the whole cycle: block b owns the rows [b R, (b + 1) R) and keeps
// them of w in shared memory as double-float planes.  A step is four phases, each ended by
// a barrier of all blocks (a counter in L2, bounded waits):
//   SpMV on the own rows; partials of h = V^T w
//   w1 = w - V h on the own rows; partials of u = V^T w1
//   w2 = w1 - V u on the own rows; partials of ||w2||, max |w2|
//   v_{j+1} = w2 / ||w2|| encoded for the own rows (the next SpMV gathers it)
// Every block forms the sums over the blocks itself, in the same order (a warp per four
// columns, its lanes over the blocks), so that all hold the same coefficients without a
// further exchange.  The Givens update (a serial FP64 chain of 5-7 us) runs on an extra warp
// of block 0 while the blocks go on with the next step; its decision to end the cycle is
// read after the next step's second barrier, so at most one SpMV and three basis products are
// computed in vain per cycle.
//
// With RES the own rows of the whole basis stay in shared memory as well, and only the
// SpMV's gather goes to L2.
//
// Arithmetic is that of the stepwise kernels: double-float products and sums, the same
// splits and epilogues; only the order of the sums differs, and the columns' sums over blocks are
// of double-float pairs (see collect).
//
// What bounds it: 64^2 f64, restart 100, takes 18.5 us per step (72 us as separate kernels): 11.5k
// of 37k cycles in the four barriers (about 1.4 us each: one release, one poll), 6k in the
// two sums over the blocks (an L2 round trip and a warp tree each), 11k in the basis
// products, 3.6k in the SpMV's chain of three loads, 3k in the FP64 root and division of
// the norm and the encoding.  Tagged exchange words in place of barriers were slower: every
// block polling every other's words queues at the few L2 slices that hold them (norm
// exchange 4.5 us, flags of the encoding 7 us).  From about 1000 rows per block on, the
// basis products take over, at 4.6 TB/s for f32 (loads in flight, limited by registers).
#pragma once
#include "cbg_kernels.cuh"
#include "cbg_stream.cuh"

namespace cbg {

constexpr int CY_WARPS = 16;                  // compute warps; one more runs the Givens update
constexpr int CY_CT = CY_WARPS * 32;
constexpr int CY_THREADS = CY_CT + 32;
constexpr int CY_ROWS = 16;                   // rows per block: a multiple of every format's chunk
constexpr int CY_MAXG = 160;                  // blocks (a lane adds up to five blocks' partials)

struct CycleArgs {
    DevArrays d;
    unsigned char* V;
    long long ldb;            // bytes per basis column
    long long n, nrows;       // rows, and padded rows of a column
    int rows;                 // rows per block (multiple of CY_ROWS)
    int mcols;                // columns the shared arrays are sized for (>= restart + 1)
    const int* rowptr;        // the per-step operator: CSR with double-float values
    const int* col;
    const float* valdf;       // hi[nnz], lo[nnz]
    long long nnz;
    const int* prow;          // two-stage preconditioner z = P v before A z (null: none)
    const int* pcol;
    const double* pvals;
    double* z;
    int lanes;                // SpMV lanes per row (power of two, at most 32)
    int hexp;                 // StoreArgs::hexp
    float2* part;             // [2][MAXCOLS][CY_MAXG] column partials: h, u
    float4* norm;             // [2][CY_MAXG] sums of squares: of w2, omega^2 (triples, see tf_add)
    float2* wmax;             // [CY_MAXG] maxima
    double* coef;             // [2][2][MAXCOLS] h and u of odd and even steps, for the Givens warp
    unsigned int* counter;    // arrivals; zero when the launch starts
    int* fault;               // set when a wait ran out
    long long limit;          // clock cycles a wait may take
    int withhold;             // test of the failure path: the last block does not arrive at this barrier (0: none)
};
// their sizes in float2 (8 bytes); norm starts on a 16-byte boundary
constexpr size_t CY_PART = (size_t)2 * MAXCOLS * CY_MAXG, CY_NORM = (size_t)4 * CY_MAXG, CY_WMAX = CY_MAXG, CY_COEF = (size_t)4 * MAXCOLS;

// shared memory of a block in bytes: planes of w, partial sums of the axpy, per-warp column
// sums, the resident basis
template <int FMT> struct CycleGeom {
    static constexpr int BS = FmtInfo<FMT>::bytes;
    static constexpr int E = 16 / BS;
    static constexpr int CG = 8;                 // columns (16-byte loads) in flight in the dot
    static constexpr size_t split_bytes = (size_t)CY_CT * E * sizeof(float2);
    static size_t smem(int rows, int mcols, int cols_resident)
    {
        return (size_t)rows * 8 + split_bytes + (size_t)CY_WARPS * mcols * sizeof(float2) +
               (size_t)rows * BS * cols_resident;
    }
};

struct CycleShared {
    double sR[MAXCOLS + 1], sRo[MAXCOLS + 1], scs[MAXCOLS], ssn[MAXCOLS];   // Givens warp
    double scale[MAXCOLS + 1];
    float2 cs[MAXCOLS];                        // axpy coefficients
    float4 wsum[CY_WARPS];                     // per warp sums of squares
    float2 wmax[CY_WARPS];                     // per warp maxima
    double hn, inv, omega[2];
    EncParams ep;
    int fail, quit;
};

__device__ __forceinline__ void cy_sync() { asm volatile("bar.sync 1, %0;" ::"r"(CY_CT) : "memory"); }
// barrier 2: compute warps hand a finished column to the Givens warp; barrier 3: it is done
__device__ __forceinline__ void cy_post(int id) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(CY_THREADS) : "memory"); }
__device__ __forceinline__ void cy_take(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(CY_THREADS) : "memory"); }

// Barrier of the compute warps of all blocks: thread 0 releases the block's writes into a
// counter that only grows within the launch and waits (bounded) until every block has
// arrived as often as this one.  Sets sm.fail when the wait ran out.  skip: the epoch at which the
// block does not arrive (a test; 0: it always does).
__device__ __forceinline__ void cy_grid_sync(const CycleArgs& a, CycleShared& sm, unsigned& epoch, unsigned skip)
{
    epoch += gridDim.x;
    cy_sync();
    if (threadIdx.x == 0) {
        unsigned now;
        if (epoch != skip)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.counter) : "memory");
        const long long t0 = clock64();
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(a.counter) : "memory");
            if (now >= epoch) break;
            if (clock64() - t0 > a.limit) {
                sm.fail = 1;
                break;
            }
        }
    }
    cy_sync();
}

__device__ __forceinline__ uint4 ld_cg16(const void* p)
{
    return __ldcg(reinterpret_cast<const uint4*>(p));
}

// (S, C) += y^2 for a renormalised pair y = h + l
__device__ __forceinline__ void cy_add_square(float& S, float& C, float h, float l)
{
    const float p = __fmul_rn(h, h);
    float q = __fmaf_rn(h, h, -p);
    q = __fmaf_rn(__fadd_rn(h, h), l, q);
    float s, e;
    two_sum(S, p, s, e);
    C = __fadd_rn(C, __fadd_rn(e, q));
    S = s;
}

template <int FMT, bool RES> struct Cycle {
    using G = CycleGeom<FMT>;
    static constexpr int BS = G::BS, E = G::E, CG = G::CG;
    static constexpr bool SCALED = FMT == I32 || FMT == I16 || FMT == BF16 || FMT == E4M3;

    // Resident f64 columns are kept as the float pairs the products use (hi, lo per row).
    static constexpr bool PAIRS = RES && FMT == F64;
    static __device__ __forceinline__ void decode(const uint4& raw, Chunk<FMT>& c)
    {
        if constexpr (PAIRS) {
            c.vh[0] = __uint_as_float(raw.x);
            c.vl[0] = __uint_as_float(raw.y);
            c.vh[1] = __uint_as_float(raw.z);
            c.vl[1] = __uint_as_float(raw.w);
        } else {
            decode_chunk<FMT>(raw, c);
        }
    }
    // v into row r of a resident column
    static __device__ __forceinline__ void keep(unsigned char* own, int r, double v, const EncParams& ep)
    {
        if constexpr (PAIRS) {
            float hi, lo;
            split_f64(v, hi, lo);
            reinterpret_cast<float2*>(own)[r] = make_float2(hi, lo);
        } else {
            encode_store<FMT>(own, r, v, ep);
        }
    }

    static __device__ __forceinline__ uint4 code16(const unsigned char* p)
    {
        if constexpr (RES) return *reinterpret_cast<const uint4*>(p);
        else return ld_cg16(p);
    }

    // w = A x on the own rows into the planes (x: the code column, or the FP64 vector z);
    // leaves the warps' sums of w^2 in sm.wsum.  L lanes share a row.
    template <int XFMT>
    static __device__ void spmv(const CycleArgs& a, CycleShared& sm, const void* x, double xs, long long r0, int R,
                                float* wh, float* wl)
    {
        const int L = a.lanes, lg = threadIdx.x & (L - 1), step = CY_CT / L;
        constexpr bool XEXACT = XFMT == F32 || XFMT == F16 || XFMT == BF16 || XFMT == E4M3 || XFMT == I16;
        const float* vlo = a.valdf + a.nnz;
        const bool xsplit = xs != 1.0;
        float xsh = 1.f, xsl = 0.f, ssS = 0.f, ssC = 0.f;
        if (xsplit) split_f64(xs, xsh, xsl);
        // RW rows of a lane group at a time, software-pipelined: the next entries' values and
        // columns are loaded while the current ones' gathers are in flight
        constexpr int RW = 4;
        for (int base = 0; base < R; base += RW * step) {
            float S[RW], C[RW], vh[RW], vl[RW];
            int p[RW], p1[RW], c[RW], len = 0;
#pragma unroll
            for (int q = 0; q < RW; q++) {
                const int r = base + q * step + threadIdx.x / L;
                const bool valid = r < R && r0 + r < a.n;
                p[q] = valid ? __ldg(a.rowptr + r0 + r) + lg : 0;
                p1[q] = valid ? __ldg(a.rowptr + r0 + r + 1) : 0;
                S[q] = C[q] = 0.f;
            }
            auto entries = [&]() {                             // column -1: no entry
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const bool in = p[q] < p1[q];
                    vh[q] = in ? __ldg(a.valdf + p[q]) : 0.f;
                    vl[q] = in ? __ldg(vlo + p[q]) : 0.f;
                    c[q] = in ? __ldg(a.col + p[q]) : -1;
                    p[q] += L;
                }
            };
#pragma unroll
            for (int q = 0; q < RW; q++) len = max(len, p1[q] - p[q]);
            entries();
            for (int i = 0; i < len; i += L) {
                float xh[RW], xl[RW], fh[RW], fl[RW];
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    xh[q] = xl[q] = 0.f;
                    fh[q] = vh[q];
                    fl[q] = vl[q];
                    if (c[q] >= 0 && col_ok(c[q], a.n, a.d.st)) xval_df<XFMT>(x, c[q], xh[q], xl[q]);
                    else fh[q] = fl[q] = 0.f;
                }
                entries();
#pragma unroll
                for (int q = 0; q < RW; q++) {
                    const float pr = __fmul_rn(fh[q], xh[q]);
                    float er = __fmaf_rn(fh[q], xh[q], -pr);
                    er = __fmaf_rn(fl[q], xh[q], er);
                    if constexpr (!XEXACT) er = __fmaf_rn(fh[q], xl[q], er);
                    float s, e;
                    two_sum(S[q], pr, s, e);
                    C[q] = __fadd_rn(C[q], __fadd_rn(e, er));
                    S[q] = s;
                }
            }
#pragma unroll
            for (int q = 0; q < RW; q++) {
                if (base + q * step >= R) break;               // (the same for all threads)
                for (int o = L >> 1; o > 0; o >>= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, S[q], o), c2 = __shfl_xor_sync(0xffffffffu, C[q], o);
                    float s, e;
                    two_sum(S[q], s2, s, e);
                    C[q] = __fadd_rn(__fadd_rn(C[q], c2), e);
                    S[q] = s;
                }
                const int r = base + q * step + threadIdx.x / L;
                if (r < R && lg == 0) {
                    float hi, lo;
                    two_sum(S[q], C[q], hi, lo);
                    if (xsplit) {
                        const float p = __fmul_rn(hi, xsh);
                        float e = __fmaf_rn(hi, xsh, -p);
                        e = __fmaf_rn(hi, xsl, e);
                        e = __fmaf_rn(lo, xsh, e);
                        two_sum(p, e, hi, lo);
                    }
                    wh[r] = hi;
                    wl[r] = lo;
                    cy_add_square(ssS, ssC, hi, lo);
                }
            }
        }
        float4 ss = make_float4(ssS, ssC, 0.f, 0.f);
        tf_warp_sum<true>(ss);
        if ((threadIdx.x & 31) == 0) sm.wsum[threadIdx.x >> 5] = ss;
    }

    // z = P v on the own rows (FP64, as the stepwise kernel)
    static __device__ void precondition(const CycleArgs& a, const void* x, double xs, long long r0, int R)
    {
        for (int r = threadIdx.x; r < R; r += CY_CT) {
            const long long row = r0 + r;
            if (row >= a.n) break;
            double s = 0.0;
            const int p1 = __ldg(a.prow + row + 1);
            for (int p = __ldg(a.prow + row); p < p1; p++) {
                const int c = __ldg(a.pcol + p);
                if (col_ok(c, a.n, a.d.st)) s = __fma_rn(__ldg(a.pvals + p), code_value<FMT>(x, c), s);
            }
            if (xs != 1.0) s = __dmul_rn(s, xs);
            a.z[row] = s;
        }
    }

    // The block's partial sums of V^T w over its rows, published as column partials.  The
    // warps are dealt out as wr row splits x wc column groups so that the slowest warp has
    // the fewest (group, segment) items.  omega: also the warps' sums of squares.
    static __device__ void dot(const CycleArgs& a, CycleShared& sm, float2* red, const unsigned char* vs,
                               long long vstride, int R, int ncols, const float* wh, const float* wl, float2* part,
                               bool omega)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, mcols = a.mcols;
        const int nch = R / E, nseg = (nch + 31) >> 5, ngroups = (ncols + CG - 1) / CG;
        int lc = 0, best = 0x7fffffff;
#pragma unroll
        for (int c = 0; c <= 4; c++) {                        // wc = 2^c
            const int items = ((ngroups + (1 << c) - 1) >> c) * ((nseg + (CY_WARPS >> c) - 1) >> (4 - c));
            if (items <= best) {
                best = items;
                lc = c;
            }
        }
        const int wc = 1 << lc, lr = 4 - lc, wr = 1 << lr, mc = warp >> lr, mr = warp & (wr - 1);
        for (int g = mc; g < ngroups; g += wc) {
            const int c0 = g * CG, nc = ncols - c0 < CG ? ncols - c0 : CG;
            float2 S2[CG / 2], C2[CG / 2];
#pragma unroll
            for (int q = 0; q < CG / 2; q++) { S2[q] = make_float2(0.f, 0.f); C2[q] = make_float2(0.f, 0.f); }
            // halves of the group, software-pipelined: one half's loads are in flight while the
            // other is accumulated
            constexpr int H = CG / 2;
            const unsigned char* vc = vs + (long long)c0 * vstride;
            auto fetch = [&](int ch, int q0, uint4 (&raw)[H]) {
                const unsigned char* p = vc + (long long)q0 * vstride + ch * 16;
#pragma unroll
                for (int q = 0; q < H; q++) {
                    raw[q] = ch < nch && q0 + q < nc ? code16(p) : make_uint4(0u, 0u, 0u, 0u);
                    p += vstride;
                }
            };
            int ch = mr * 32 + lane;
            uint4 ra[H], rb[H];
            fetch(ch, 0, ra);
            for (int s = mr; s < nseg; s += wr) {
                const int r = ch < nch ? ch * E : 0;
                fetch(ch, H, rb);
                float xh[E], xl[E];
#pragma unroll
                for (int e = 0; e < E; e += 2) {
                    const float2 h2 = *reinterpret_cast<const float2*>(wh + r + e);
                    const float2 l2 = *reinterpret_cast<const float2*>(wl + r + e);
                    xh[e] = h2.x; xh[e + 1] = h2.y; xl[e] = l2.x; xl[e + 1] = l2.y;
                }
                auto accumulate = [&](const uint4& u0, const uint4& u1, float2& S, float2& C) {
                    Chunk<FMT> k0, k1;
                    decode(u0, k0);
                    decode(u1, k1);
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
            if ((lane & fold_low<CG>()) == 0 && col < nc) red[mr * mcols + c0 + col] = make_float2(S[0], C[0]);
        }
        cy_sync();
        const int b = blockIdx.x;
        for (int c = threadIdx.x; c < ncols; c += CY_CT) {
            float2 t = red[c];
            for (int k = 1; k < wr; k++) df_add(t.x, t.y, red[k * mcols + c].x, red[k * mcols + c].y);
            part[c * CY_MAXG + b] = t;
        }
        if (omega && warp == CY_WARPS - 1) {
            const float4 t = fold_warps(sm.wsum, lane);
            if (lane == 0) a.norm[CY_MAXG + b] = t;
        }
    }

    // the sum of the warps' triples (one warp calls it; all its lanes hold the result)
    static __device__ float4 fold_warps(const float4* w, int lane)
    {
        float4 t = w[lane & (CY_WARPS - 1)];
#pragma unroll
        for (int o = CY_WARPS / 2; o > 0; o >>= 1) tf_add(t, tf_shfl_xor(t, o));
        return t;
    }
    // the sum of the blocks' triples (one warp; its lanes add the blocks lane, lane + 32, ...)
    static __device__ float4 sum_blocks(const float4* p, int lane)
    {
        float4 v[CY_MAXG / 32];                                // all of them in flight at once
#pragma unroll
        for (int u = 0; u < CY_MAXG / 32; u++)
            v[u] = lane + 32 * u < (int)gridDim.x ? __ldcg(p + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 1; u < CY_MAXG / 32; u++) tf_add(v[0], v[u]);
        tf_warp_sum<true>(v[0]);
        return v[0];
    }

    // After the barrier: the sums of all columns over the blocks (warp w takes the columns
    // 4 w .. 4 w + 3, then 64 further on; its lanes add the blocks lane, lane + 32, ...) and
    // from them the axpy's coefficients -scale h in sm.cs; block 0 also keeps h (hout).  These sums
    // are double-float: the second projection takes in what the first one missed, and h is recorded
    // as the pair that the subtraction uses, so that it is as close to 64 bits as from the
    // stepwise kernels, or closer (29,791 rows f32, rms of ||h||: 1.4e-16, stepwise 1.0e-15; triples
    // of floats gave 5e-16, a tenth slower).  The norms have no second pass, and double-float sums
    // doubled their error.
    static __device__ void collect(const CycleArgs& a, CycleShared& sm, const float2* part, int ncols, double* hout)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nb = gridDim.x;
        for (int c0 = 4 * warp; c0 < ncols; c0 += 4 * CY_WARPS) {
            float S[4], C[4];
#pragma unroll
            for (int q = 0; q < 4; q++) S[q] = C[q] = 0.f;
            float2 v[CY_MAXG / 32][4];                         // all of them in flight at once
#pragma unroll
            for (int u = 0; u < CY_MAXG / 32; u++)
#pragma unroll
                for (int q = 0; q < 4; q++)
                    v[u][q] = lane + 32 * u < nb && c0 + q < ncols ? __ldcg(part + (c0 + q) * CY_MAXG + lane + 32 * u)
                                                               : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < CY_MAXG / 32; u++) {
                if (32 * u >= nb) break;
#pragma unroll
                for (int q = 0; q < 4; q++) df_add(S[q], C[q], v[u][q].x, v[u][q].y);
            }
            const int c = c0 + df_warp_fold<4>(S, C, lane);
            if ((lane & 7) == 0 && c < ncols) {
                float h, l;                                    // -(the sum), renormalised
                two_sum(-S[0], -C[0], h, l);
                sm.cs[c] = make_float2(h, l);
            }
        }
        cy_sync();
        // FP64 only where it is needed (scaled formats; block 0 for the Givens update), and
        // there in as few warps as there are columns: an FP64 instruction occupies GB300's
        // narrow pipe for a whole warp however few lanes take part
        if (blockIdx.x == 0 || SCALED) {
            for (int c = threadIdx.x; c < ncols; c += CY_CT) {
                const float2 v = sm.cs[c];
                double h = -df_to_double(v.x, v.y);
                if constexpr (SCALED) {
                    const double sc = sm.scale[c];
                    h = __dmul_rn(h, sc);
                    float hi, lo;
                    split_f64(-__dmul_rn(sc, h), hi, lo);
                    sm.cs[c] = make_float2(hi, lo);
                }
                if (blockIdx.x == 0) hout[c] = h;
            }
            cy_sync();
        }
    }

    // w -= V c on the own rows; NORMS: the warps' sums of w^2 and maxima of |w| as well.
    // Blocks with fewer row chunks than threads split the columns over thread groups, whose
    // partial sums meet in shared memory (split).
    template <bool NORMS>
    static __device__ void axpy(const CycleArgs& a, CycleShared& sm, const unsigned char* vs, long long vstride,
                                long long r0, int R, int ncols, float* wh, float* wl, float2* split)
    {
        constexpr int U = 4;                                   // columns per half of the pipeline
        const int nch = R / E, ncp = (nch + 31) & ~31;
        const int width = ncp <= CY_CT ? ncp : CY_CT, ks = CY_CT / width;
        const int mk = threadIdx.x / width, mch = threadIdx.x - mk * width;
        const long long left = a.n - r0;
        const int nvalid = left < R ? (left > 0 ? (int)left : 0) : R;   // own rows below n
        float ssS = 0.f, ssC = 0.f;
        float2 mx = make_float2(0.f, 0.f);
        auto finish = [&](int r, float S, float C) {            // w[r] += S + C
            df_add(S, C, wh[r], wl[r]);
            float h, l;
            two_sum(S, C, h, l);
            wh[r] = h;
            wl[r] = l;
            if constexpr (NORMS) {
                if (r < nvalid) {
                    cy_add_square(ssS, ssC, h, l);
                    // the larger of two renormalised pairs in absolute value
                    const float ah = fabsf(h), al = h < 0.f ? -l : l;
                    if (!(ah < mx.x || (ah == mx.x && al <= mx.y))) mx = make_float2(ah, al);
                }
            }
        };
        for (int ch = mch; ch < ncp; ch += width) {
            const bool in = ch < nch && mk < ks;
            float2 S2[E / 2], C2[E / 2];
#pragma unroll
            for (int e = 0; e < E / 2; e++) { S2[e] = make_float2(0.f, 0.f); C2[e] = make_float2(0.f, 0.f); }
            if (in) {
                const unsigned char* base = vs + (long long)ch * 16;
                auto fetch = [&](int k0, uint4 (&raw)[U]) {
                    const unsigned char* p = base + (long long)k0 * vstride;
#pragma unroll
                    for (int q = 0; q < U; q++) {
                        raw[q] = k0 + q * ks < ncols ? code16(p) : make_uint4(0u, 0u, 0u, 0u);
                        p += ks * vstride;
                    }
                };
                // a column past the last has zero codes and adds exact zeros
                auto accumulate = [&](int k0, const uint4 (&raw)[U]) {
#pragma unroll
                    for (int q = 0; q < U; q++) {
                        Chunk<FMT> cd;
                        decode(raw[q], cd);
                        const float2 c = k0 + q * ks < ncols ? sm.cs[k0 + q * ks] : make_float2(0.f, 0.f);
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
                for (int k0 = mk; k0 < ncols; k0 += 2 * U * ks) {
                    fetch(k0 + U * ks, rb);
                    accumulate(k0, ra);
                    if (k0 + U * ks >= ncols) break;
                    fetch(k0 + 2 * U * ks, ra);
                    accumulate(k0 + U * ks, rb);
                }
            }
            if (ks == 1) {
                if (in) {
#pragma unroll
                    for (int e = 0; e < E; e++) {
                        const float S = e & 1 ? S2[e / 2].y : S2[e / 2].x, C = e & 1 ? C2[e / 2].y : C2[e / 2].x;
                        finish(ch * E + e, S, C);
                    }
                }
            } else if (in) {
#pragma unroll
                for (int e = 0; e < E; e++)
                    split[mk * R + e * nch + ch] = e & 1 ? make_float2(S2[e / 2].y, C2[e / 2].y)
                                                       : make_float2(S2[e / 2].x, C2[e / 2].x);
            }
        }
        if (ks > 1) {
            // 2^lg lanes per row add its ks partial sums (every lane of a warp stays in the loop)
            int lg = 0;
            while (lg < 3 && (2 << lg) <= ks && (long long)R << (lg + 1) <= CY_CT) lg++;
            const int part = threadIdx.x & ((1 << lg) - 1), rows = CY_CT >> lg;
            cy_sync();
            for (int base = 0; base < R; base += rows) {
                const int i = base + (threadIdx.x >> lg);      // the chunk i % nch, its row i / nch
                float2 t = make_float2(0.f, 0.f);
                if (i < R)
                    for (int k = part; k < ks; k += 1 << lg) df_add(t.x, t.y, split[k * R + i].x, split[k * R + i].y);
                for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, t.x, o), c2 = __shfl_xor_sync(0xffffffffu, t.y, o);
                    df_add(t.x, t.y, s2, c2);
                }
                if (i < R && part == 0) finish(i % nch * E + i / nch, t.x, t.y);
            }
        }
        if constexpr (NORMS) {
            float4 ss = make_float4(ssS, ssC, 0.f, 0.f);
            tf_warp_sum<true>(ss);
            fold_max(mx);
            if ((threadIdx.x & 31) == 0) {
                sm.wsum[threadIdx.x >> 5] = ss;
                sm.wmax[threadIdx.x >> 5] = mx;
            }
        }
        cy_sync();
    }

    static __device__ __forceinline__ void fold_max(float2& m)
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, m.x, o), l2 = __shfl_xor_sync(0xffffffffu, m.y, o);
            if (!(h2 < m.x || (h2 == m.x && l2 <= m.y))) m = make_float2(h2, l2);
        }
    }

    // ||w2||, max |w2| of the block to norm[]
    static __device__ void put_norms(const CycleArgs& a, CycleShared& sm)
    {
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            const float4 s = fold_warps(sm.wsum, lane);
            float2 m = sm.wmax[lane & (CY_WARPS - 1)];
            fold_max(m);
            if (lane == 0) {
                a.norm[blockIdx.x] = s;
                a.wmax[blockIdx.x] = m;
            }
        }
    }
    // after the barrier: those of all blocks, and what the encoding of column col needs; block 0
    // also sums omega^2 (*om), which only the Givens update reads
    static __device__ void collect_norms(const CycleArgs& a, CycleShared& sm, int col, double* om)
    {
        if (blockIdx.x == 0 && threadIdx.x >> 5 == 1) {
            const float4 s = sum_blocks(a.norm + CY_MAXG, threadIdx.x & 31);
            if (threadIdx.x == 32) *om = tf_to_double<true>(s);
        }
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x, nb = gridDim.x;
            float2 w[CY_MAXG / 32];
#pragma unroll
            for (int u = 0; u < CY_MAXG / 32; u++)
                w[u] = lane + 32 * u < nb ? __ldcg(a.wmax + lane + 32 * u) : make_float2(0.f, 0.f);
            const float4 s = sum_blocks(a.norm, lane);
            float2 m = w[0];
#pragma unroll
            for (int u = 1; u < CY_MAXG / 32; u++)
                if (!(w[u].x < m.x || (w[u].x == m.x && w[u].y <= m.y))) m = w[u];
            fold_max(m);
            if (lane == 0) {
                const double hn = sqrt(tf_to_double<true>(s)), inv = 1.0 / hn;
                sm.hn = hn;
                sm.inv = inv;
                sm.ep = enc_params(FMT, __dmul_rn(df_to_double(m.x, m.y), inv));
                sm.scale[col] = sm.ep.scale;
            }
        }
        cy_sync();
    }

    static __device__ void givens(const CycleArgs& a, CycleShared& sm, int kcap)
    {
        StoreArgs sa{};
        sa.d = a.d;
        sa.reorth = 1;
        sa.hexp = a.hexp;
        for (int j = 0; j < kcap; j++) {
            cy_take(2);
            if (*(volatile int*)&sm.quit) return;        // the compute warps gave up
            sa.j = j;
            sa.d.h = a.coef + (j & 1) * 2 * MAXCOLS;
            sa.d.u = sa.d.h + MAXCOLS;
            if ((threadIdx.x & 31) == 0) a.d.st->omega = sqrt(sm.omega[j & 1]);
            __syncwarp();
            arnoldi_finalize(sa, sm.hn, sm.sR, sm.sRo, sm.scs, sm.ssn);
            __threadfence();
            __syncwarp();
            const bool run = *(volatile int*)&a.d.st->active != 0;
            if (j + 1 < kcap) cy_post(3);                // (nobody waits for the last column)
            if (!run) return;
        }
    }

    static __device__ void compute(const CycleArgs& a, CycleShared& sm, int kcap, unsigned char* dyn)
    {
        const int b = blockIdx.x, t = threadIdx.x;
        const long long r0 = (long long)b * a.rows;
        const int R = a.nrows - r0 < a.rows ? (int)(a.nrows - r0) : a.rows;   // own rows (padding included)
        float* wh = reinterpret_cast<float*>(dyn);
        float* wl = wh + a.rows;
        float2* split = reinterpret_cast<float2*>(wl + a.rows);
        float2* red = split + G::split_bytes / sizeof(float2);
        unsigned char* res = reinterpret_cast<unsigned char*>(red + CY_WARPS * a.mcols);
        const unsigned char* vs = RES ? res : a.V + r0 * BS;          // own rows of column 0
        const long long vstride = RES ? (long long)a.rows * BS : a.ldb;
        float2* part2 = a.part + MAXCOLS * CY_MAXG;
        unsigned epoch = 0;
        const unsigned skip = blockIdx.x + 1 == gridDim.x ? a.withhold * gridDim.x : 0u;
        bool open = false;                        // block 0: the Givens warp will arrive at barrier 3
        volatile int* fail = &sm.fail;
        if (t == 0) sm.scale[0] = a.d.scales[0];
        for (int r = t; r < R; r += CY_CT) wh[r] = wl[r] = 0.f;
        if constexpr (PAIRS) {
            for (int r = t; r < R; r += CY_CT) keep(res, r, __ldcg(reinterpret_cast<const double*>(a.V) + r0 + r), EncParams{1.0, 1.0});
        } else if constexpr (RES) {
            for (int i = t; i < R * BS / 16; i += CY_CT)
                reinterpret_cast<uint4*>(res)[i] = ld_cg16(a.V + r0 * BS + 16ll * i);
        }
        cy_sync();
        for (int j = 0; j < kcap; j++) {
            const int ncols = j + 1;
            const unsigned char* vj = a.V + (long long)j * a.ldb;
            double* hj = a.coef + (j & 1) * 2 * MAXCOLS;
            // w = A M^{-1} v_j, omega
            if (a.prow) {
                precondition(a, vj, sm.scale[j], r0, R);
                cy_grid_sync(a, sm, epoch, skip);
                if (*fail) break;
                spmv<-1>(a, sm, a.z, 1.0, r0, R, wh, wl);
            } else {
                spmv<FMT>(a, sm, vj, sm.scale[j], r0, R, wh, wl);
            }
            cy_sync();
            // h = V^T w
            dot(a, sm, red, vs, vstride, R, ncols, wh, wl, a.part, true);
            cy_grid_sync(a, sm, epoch, skip);
            if (*fail) break;
            collect(a, sm, a.part, ncols, hj);
            // w1 = w - V h ; u = V^T w1
            axpy<false>(a, sm, vs, vstride, r0, R, ncols, wh, wl, split);
            dot(a, sm, red, vs, vstride, R, ncols, wh, wl, part2, false);
            if (b == 0 && j > 0) {
                cy_take(3);                                           // the Givens update of step j - 1
                open = false;
            }
            cy_grid_sync(a, sm, epoch, skip);
            if (*fail || (j > 0 && *(volatile int*)&a.d.st->active == 0)) break;
            collect(a, sm, part2, ncols, hj + MAXCOLS);
            // w2 = w1 - V u, its norms
            axpy<true>(a, sm, vs, vstride, r0, R, ncols, wh, wl, split);
            put_norms(a, sm);
            cy_grid_sync(a, sm, epoch, skip);
            if (*fail) break;
            collect_norms(a, sm, ncols, &sm.omega[j & 1]);
            if (b == 0) {
                if (t == 0) a.d.scales[ncols] = sm.ep.scale;
                cy_post(2);                                           // column j to the Givens warp
                open = j + 1 < kcap;
            }
            // v_{j+1}
            {
                const double inv = sm.inv;
                const EncParams ep = sm.ep;
                unsigned char* dst = a.V + (long long)ncols * a.ldb;
                unsigned char* own = RES ? res + (long long)ncols * vstride : nullptr;
                for (int r = t; r < R; r += CY_CT) {
                    if (r0 + r < a.n) {
                        const double v = __dmul_rn(df_to_double(wh[r], wl[r]), inv);
                        encode_store<FMT>(dst, r0 + r, v, ep);
                        if constexpr (RES) keep(own, r, v, ep);
                    } else if constexpr (RES) {
                        keep(own, r, 0.0, EncParams{1.0, 1.0});
                    }
                }
            }
            if (j + 1 < kcap) cy_grid_sync(a, sm, epoch, skip);
            if (*fail) break;
        }
        if (*fail) {
            if (t == 0) {
                record_fault(nullptr, a.fault);
                sm.quit = 1;
            }
            if (b == 0) {
                // release the Givens warp: once it has done with the column it was given (a second
                // arrival at barrier 2 before it took the first would be one too many) it waits
                // there for the next one, unless it has ended the cycle
                if (open) cy_take(3);
                cy_sync();
                if (*(volatile int*)&a.d.st->active != 0) cy_post(2);
            }
        }
    }
};

template <int FMT, bool RES>
__global__ void __launch_bounds__(CY_THREADS, 1) k_cycle(CycleArgs a)
{
    if (a.d.st->active == 0) return;
    extern __shared__ __align__(128) unsigned char cy_dyn[];
    __shared__ CycleShared sm;
    const int kcap = a.d.st->kcap;
    if (threadIdx.x == 0) sm.quit = sm.fail = 0;
    __syncthreads();
    if (threadIdx.x < CY_CT) Cycle<FMT, RES>::compute(a, sm, kcap, cy_dyn);
    else if (blockIdx.x == 0) Cycle<FMT, RES>::givens(a, sm, kcap);
}

}  // namespace cbg
