// multi.cu -- multi-RHS basis product H = V^T W for k vectors that share one compressed
// basis (the orthogonalisation of block Krylov methods; the paper has no counterpart:
// its GMRES has one right-hand side).
//
// Reading V once for all k vectors turns the k basis GEMVs into one split-K GEMM whose
// arithmetic (DF32, as in the single-vector kernels: 11 FP32 operations per product)
// dominates for k > 2.  W is split first into FP32 hi / lo planes, two vectors interleaved,
// in the order in which the lanes of a tile read them.  The product kernel runs one block
// per SM: sixteen consumer warps and a producer warp.  The work items are the (16 columns, row
// tile) pairs, column groups outermost, and a block owns a contiguous range of them.  The
// producer fills a ring in shared memory with bulk copies: 1 KiB of codes per column and the
// tile of W's planes (W stays in L2 between the column groups).  Consumer warp w takes row
// group w % 2 and columns 2 (w / 2), + 1: its lanes own E = 16 / bytes consecutive rows and
// keep 2 x 2 KP double-float accumulators (KP pairs of vectors on the packed FP32x2 pipe).
// After 32 rows a lane's sums are folded over the warp (transposing butterfly) and added to
// the warp's FP64 sums, so no double-float chain is longer than 32 products.  Blocks
// leave per-column partials, which a second kernel adds in block order.
//
// Measured per call, against one staged tile of W at a time, plain code loads and vectors
// padded to 8 (us): 999,983 x 67 f32, k = 5: 525 -> 220; 2^21 x 100, k = 8: f32 1141 -> 794,
// f64 1518 -> 1084; 2^20 x 120, k = 1: e4m3 272 -> 133.  The product kernel keeps the FMA pipe
// 74 % busy; the rest is the last, partly filled column group and the shared-memory reads
// of W's planes.  Eight warps of four columns each were 4 % faster for f32 and 19 % slower
// for f64.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "../../include/cbgmres.h"
#include "cbg_context.h"
#include "cbg_kernels.cuh"
#include "cbg_stream.cuh"

using namespace cbg;

void cbg_record_cuda_error(cudaError_t e);   // solver.cu
size_t cbg_tc_multi_workspace(int64_t ld);   // multi_tc.cu
int cbg_tc_multi(int64_t n, int ncols, const void* V, int64_t ld, const double* scales, int k, int ldh, const double* W,
                 int64_t ldw, double* H, void* workspace, cudaStream_t s, int** fault_out);

namespace {

constexpr int KMAX = 8;              // right-hand sides per launch
constexpr int KCALL = 64;            // right-hand sides per call (groups of KMAX)
constexpr int MU_RG = 2;             // row groups of a tile (32 lanes x E rows each)
constexpr int MU_CS = 8;             // column subsets of a stage
constexpr int MU_CW = MU_RG * MU_CS; // consumer warps
constexpr int MU_CPW = 2;            // columns per consumer warp
constexpr int MU_CG = MU_CS * MU_CPW;   // columns per stage
constexpr int MU_THREADS = (MU_CW + 1) * 32;
constexpr int MU_CHAIN = 32;         // rows a lane accumulates before its sums are folded (one pair of vectors: half)

template <int FMT, int KP> struct MultiGeom {
    static constexpr int BS = FmtInfo<FMT>::bytes;
    static constexpr int E = 16 / BS;                       // rows per lane
    static constexpr int TILE = MU_RG * 32 * E;             // rows per tile
    static constexpr int COLB = TILE * BS;                  // bytes of one column's tile (1024)
    static constexpr int PLANE = TILE * (int)sizeof(float2);   // one plane (hi or lo) of a pair of vectors
    static constexpr int STAGE = MU_CG * COLB + 2 * KP * PLANE;
};

struct MultiArgs {
    const unsigned char* V;
    long long ldb;            // bytes per basis column
    int ncols;
    const float2* wsplit;     // [KP][hi, lo][ld]: two vectors interleaved, tile order (k_split_multi)
    long long ld;             // rows per column (multiple of TILE_ROWS)
    double* part;             // [gridDim.x][ncols][2 KP]
    int* fault;
};

// W (n x k, column-major, leading dimension ldw) -> planes [pair][hi, lo][ld] of vector pairs
// (2p, 2p + 1), zero beyond n and beyond k.  Within a tile of 64 E rows, rows (2i, 2i + 1) of
// lane l (rows l E .. l E + E - 1) stand at 16-byte word 64 i + l: a consumer warp's 16-byte
// loads are then contiguous.  Clears the fault word.
__global__ void k_split_multi(const double* W, long long ldw, long long n, long long ld, int k, int KP, int E,
                              float2* out, int* fault)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *fault = 0;
    const long long half = ld / 2;                          // row pairs
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < (long long)KP * half;
         t += (long long)gridDim.x * blockDim.x) {
        const int p = (int)(t / half);
        const long long row = 2 * (t - p * half);
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
        const double* w0 = W + (long long)(2 * p) * ldw + row;
        if (row < n) {
            split_f64(w0[0], h.x, l.x);
            if (2 * p + 1 < k) split_f64(w0[ldw], h.y, l.y);
        }
        if (row + 1 < n) {
            split_f64(w0[1], h.z, l.z);
            if (2 * p + 1 < k) split_f64(w0[ldw + 1], h.w, l.w);
        }
        const int tile = MU_RG * 32 * E, in = (int)(row % tile);
        const long long at = (row - in) / 2 + (long long)(in % E / 2) * (MU_RG * 32) + in / E;   // 16-byte words
        float4* o = reinterpret_cast<float4*>(out) + (long long)(2 * p) * half;
        o[at] = h;
        o[half + at] = l;
    }
}

// Sixteen bytes of codes of BS bytes each, read one by one: a basis that starts between 16-byte
// boundaries, which neither the bulk copies nor 16-byte loads can take.
template <int BS> __device__ __forceinline__ uint4 load_codes(const unsigned char* p)
{
    using T = typename std::conditional<BS == 8, unsigned long long,
              typename std::conditional<BS == 4, unsigned int,
              typename std::conditional<BS == 2, unsigned short, unsigned char>::type>::type>::type;
    union { T c[16 / BS]; uint4 v; } u;
#pragma unroll
    for (int e = 0; e < 16 / BS; e++) u.c[e] = reinterpret_cast<const T*>(p)[e];
    return u.v;
}

__device__ __forceinline__ void multi_sync() { asm volatile("bar.sync 1, %0;" ::"r"(MU_CW * 32) : "memory"); }

// DIRECT: the basis is not on a 16-byte boundary, the consumers read its codes themselves
// (a branch at run time in place of the parameter made the aligned kernels spill)
template <int FMT, int KP, bool DIRECT>
__global__ void __launch_bounds__(MU_THREADS, 1) k_dot_multi(MultiArgs a, int stages)
{
    using G = MultiGeom<FMT, KP>;
    constexpr int E = G::E, KV = 2 * KP;
    constexpr int RENORM = KP == 1 ? 2 : (KP == 2 ? 4 : 8);   // rows between renormalisations
    extern __shared__ __align__(128) unsigned char mu_ring[];
    uint64_t* full = reinterpret_cast<uint64_t*>(mu_ring + (size_t)stages * G::STAGE);
    uint64_t* empty = full + stages;
    __shared__ double tot[MAXCOLS * KV];            // the block's totals [column][vector]
    __shared__ double red[MU_RG][MU_CG][KV];        // a column group's sums per row group
    __shared__ int failed;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long ntiles = a.ld / G::TILE;
    const int ngroups = (a.ncols + MU_CG - 1) / MU_CG;
    long long ib, ie;
    block_items(ntiles * ngroups, ib, ie);
    if (threadIdx.x == 0) {
        failed = 0;
        for (int s = 0; s < stages; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], MU_CW);
        }
        mbar_init_fence();
    }
    for (int i = threadIdx.x; i < a.ncols * KV; i += MU_THREADS) tot[i] = 0.0;
    __syncthreads();

    if (warp == MU_CW) {
        // producer: lane q < columns of the group copies column q's codes, lanes 16 .. 16 + 2 KP - 1
        // the planes of W; afterwards wait (bounded) until every issued copy has landed
        const uint64_t pol = l2_evict_first_policy();
        Ring rg;
        int g = (int)(ib / ntiles);
        long long t = ib - (long long)g * ntiles, it = 0;
        const long long nitems = ie - ib;
        for (; it < nitems; it++) {
            const int c0 = g * MU_CG, nc = a.ncols - c0 < MU_CG ? a.ncols - c0 : MU_CG;
            if (it >= stages && !warp_wait(&empty[rg.s], rg.ph ^ 1u)) { failed = 1; break; }
            unsigned char* st = mu_ring + (size_t)rg.s * G::STAGE;
            if (lane == 0) mbar_arrive_expect_tx(&full[rg.s], (unsigned)((DIRECT ? 0 : nc * G::COLB) + 2 * KP * G::PLANE));
            __syncwarp();
            if (!DIRECT && lane < nc)
                bulk_g2s_hint(st + lane * G::COLB, a.V + (long long)(c0 + lane) * a.ldb + t * G::COLB, G::COLB, &full[rg.s], pol);
            if (lane >= 16 && lane < 16 + 2 * KP)
                bulk_g2s(st + MU_CG * G::COLB + (lane - 16) * G::PLANE, a.wsplit + (lane - 16) * a.ld + t * G::TILE, G::PLANE,
                         &full[rg.s]);
            __syncwarp();
            rg.next(stages);
            if (++t == ntiles) { t = 0; g++; }
        }
        const long long nd = it < stages ? it : stages;
        for (long long j = 0; j < nd; j++) {
            if (--rg.s < 0) { rg.s = stages - 1; rg.ph ^= 1u; }
            if (!warp_wait(&full[rg.s], rg.ph)) { failed = 1; break; }
        }
    } else if (ie > ib) {
        const int rgp = warp % MU_RG, q0 = warp / MU_RG * MU_CPW;
        const int ln = rgp * 32 + lane;               // lane of the tile
        bool bad = false;
        Ring rg;
        const int gb = (int)(ib / ntiles), ge = (int)((ie - 1) / ntiles) + 1;
        for (int g = gb; g < ge; g++) {
            const int c0 = g * MU_CG, nc = a.ncols - c0 < MU_CG ? a.ncols - c0 : MU_CG;
            const long long tb = ib > (long long)g * ntiles ? ib - (long long)g * ntiles : 0;
            const long long te = ie < (long long)(g + 1) * ntiles ? ie - (long long)g * ntiles : ntiles;
            float2 S[MU_CPW][KP], C[MU_CPW][KP];
            double run[KP];                           // the warp's sums (one column and vector per lane)
#pragma unroll
            for (int p = 0; p < KP; p++) run[p] = 0.0;
            int rows = 0, at = 0;
            auto clear = [&]() {
#pragma unroll
                for (int q = 0; q < MU_CPW; q++)
#pragma unroll
                    for (int p = 0; p < KP; p++) { S[q][p] = make_float2(0.f, 0.f); C[q][p] = make_float2(0.f, 0.f); }
                rows = 0;
            };
            auto flush = [&]() {
#pragma unroll
                for (int p = 0; p < KP; p++) {
                    float fs[2 * MU_CPW], fc[2 * MU_CPW];
#pragma unroll
                    for (int q = 0; q < MU_CPW; q++) {
                        fs[2 * q] = S[q][p].x; fs[2 * q + 1] = S[q][p].y;
                        fc[2 * q] = C[q][p].x; fc[2 * q + 1] = C[q][p].y;
                    }
                    at = df_warp_fold<2 * MU_CPW>(fs, fc, lane);   // column at / 2, vector 2 p + at % 2
                    run[p] += df_to_double(fs[0], fc[0]);
                }
                clear();
            };
            clear();
            for (long long t = tb; t < te; t++) {
                if (!bad && !warp_wait(&full[rg.s], rg.ph)) {
                    bad = true;
                    failed = 1;
                }
                if (!bad) {
                    const unsigned char* st = mu_ring + (size_t)rg.s * G::STAGE;
                    if (q0 < nc) {                    // (a missing column's stale codes are never read back)
                        Chunk<FMT> ch[MU_CPW];
#pragma unroll
                        for (int q = 0; q < MU_CPW; q++) {
                            uint4 raw = make_uint4(0u, 0u, 0u, 0u);
                            if (!DIRECT) raw = *reinterpret_cast<const uint4*>(st + (q0 + q) * G::COLB + ln * 16);
                            else if (q0 + q < nc)
                                raw = load_codes<G::BS>(a.V + (long long)(c0 + q0 + q) * a.ldb + t * G::COLB + ln * 16);
                            decode_chunk<FMT>(raw, ch[q]);
                        }
                        const float4* wt = reinterpret_cast<const float4*>(st + MU_CG * G::COLB) + ln;
#pragma unroll
                        for (int e = 0; e < E; e += 2) {
                            float4 h4[KP], l4[KP];    // two rows of each pair of vectors
#pragma unroll
                            for (int p = 0; p < KP; p++) {
                                h4[p] = wt[(2 * p) * (G::PLANE / 16) + (e / 2) * (MU_RG * 32)];
                                l4[p] = wt[(2 * p + 1) * (G::PLANE / 16) + (e / 2) * (MU_RG * 32)];
                            }
#pragma unroll
                            for (int u = 0; u < 2; u++)
#pragma unroll
                                for (int p = 0; p < KP; p++) {
                                    const float2 wh = u ? make_float2(h4[p].z, h4[p].w) : make_float2(h4[p].x, h4[p].y);
                                    const float2 wl = u ? make_float2(l4[p].z, l4[p].w) : make_float2(l4[p].x, l4[p].y);
                                    const float2 nwh = make_float2(-wh.x, -wh.y);
#pragma unroll
                                    for (int q = 0; q < MU_CPW; q++) {
                                        const float v = ch[q].vh[e + u];
                                        if constexpr (SingleFloat<FMT>::value)
                                            df2_mac(S[q][p], C[q][p], make_float2(v, v), wh, nwh, wl);
                                        else
                                            df2_mac2(S[q][p], C[q][p], make_float2(v, v),
                                                     make_float2(ch[q].vl[e + u], ch[q].vl[e + u]), wh, nwh, wl);
                                    }
                                }
                            if (((e + 2) & (RENORM - 1)) == 0 || e + 2 == E) {
#pragma unroll
                                for (int q = 0; q < MU_CPW; q++)
#pragma unroll
                                    for (int p = 0; p < KP; p++) df2_renorm(S[q][p], C[q][p]);
                            }
                        }
                        rows += E;
                        if (rows >= (KP == 1 ? MU_CHAIN / 2 : MU_CHAIN)) flush();
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[rg.s]);
                }
                rg.next(stages);
            }
            flush();
            if ((lane & fold_low<2 * MU_CPW>()) == 0)
#pragma unroll
                for (int p = 0; p < KP; p++) red[rgp][q0 + at / 2][2 * p + at % 2] = run[p];
            multi_sync();
            for (int i = threadIdx.x; i < nc * KV; i += MU_CW * 32) {
                const int c = i / KV, v = i - c * KV;
                double s = red[0][c][v];
#pragma unroll
                for (int w = 1; w < MU_RG; w++) s += red[w][c][v];
                tot[(c0 + c) * KV + v] = s;
            }
            multi_sync();
        }
    }
    __syncthreads();
    if (failed && threadIdx.x == 0) atomicExch(a.fault, FAULT_TIMEOUT);
    for (int i = threadIdx.x; i < a.ncols * KV; i += MU_THREADS) a.part[(long long)blockIdx.x * a.ncols * KV + i] = tot[i];
}

// H[c][r] = scales[c] * sum over the blocks' partials in a fixed order: block x covers 32
// (column, vector) items, one per lane; its eight warps take the blocks w, w + 8, ... with
// their loads in flight, and the warps' sums are added in warp order.  NaN after a timeout.
__global__ void __launch_bounds__(256) k_multi_sum(const double* part, int nblk, int ncols, int KV, int k, int ldh,
                                                   const double* scales, const int* fault, double* H)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, items = ncols * KV, i = blockIdx.x * 32 + lane;
    double t = 0.0;
    if (i < items)
        for (int b0 = warp; b0 < nblk; b0 += 64) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = b0 + 8 * u < nblk ? part[(long long)(b0 + 8 * u) * items + i] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; u++) t += v[u];
        }
    sh[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && i < items) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < 8; w++) s += sh[w][lane];
        const int c = i / KV, r = i - c * KV;
        if (r < k) H[(long long)c * ldh + r] = *fault ? __longlong_as_double(0x7FF8000000000000ll) : s * scales[c];
    }
}

template <int FMT, int KP, bool DIRECT> void launch_multi(int grid, cudaStream_t s, const MultiArgs& a)
{
    using G = MultiGeom<FMT, KP>;
    static PerContext<int> plan;
    const int stages = plan.get([](int& st) {
        cudaFuncAttributes fa{};
        st = cudaFuncGetAttributes(&fa, k_dot_multi<FMT, KP, DIRECT>) == cudaSuccess
                           ? tma_stages(G::STAGE, (int)fa.sharedSizeBytes) : 0;
        if (st >= 2)
            cudaFuncSetAttribute(k_dot_multi<FMT, KP, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)tma_smem_bytes(st, G::STAGE));
        return true;
    });
    k_dot_multi<FMT, KP, DIRECT><<<grid, MU_THREADS, tma_smem_bytes(stages, G::STAGE), s>>>(a, stages);
}

template <int FMT, int KP> void launch_multi(int grid, cudaStream_t s, const MultiArgs& a)
{
    if (aligned(a.V, 16)) launch_multi<FMT, KP, false>(grid, s, a);
    else launch_multi<FMT, KP, true>(grid, s, a);
}

template <int KP> void launch_fmt(int fmt, int grid, cudaStream_t s, const MultiArgs& a)
{
    switch (fmt) {
    case CBG_F64: launch_multi<F64, KP>(grid, s, a); break;
    case CBG_F32: launch_multi<F32, KP>(grid, s, a); break;
    case CBG_F16: launch_multi<F16, KP>(grid, s, a); break;
    case CBG_BF16: launch_multi<BF16, KP>(grid, s, a); break;
    case CBG_E4M3: launch_multi<E4M3, KP>(grid, s, a); break;
    case CBG_I32: launch_multi<I32, KP>(grid, s, a); break;
    default: launch_multi<I16, KP>(grid, s, a); break;
    }
}

int multi_grid()
{
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, sms);
}

// one group of k <= KMAX vectors: H[c * ldh + r]
int dot_multi_group(int fmt, int64_t n, int ncols, const void* V, int64_t ld, const double* scales, int k,
                    const double* W, int64_t ldw, double* H, int ldh, void* workspace, cudaStream_t s, bool tc)
{
    if (tc) {
        int rc = cbg_tc_multi(n, ncols, V, ld, scales, k, ldh, W, ldw, H, workspace, s, nullptr);
        if (rc) { cbg_record_cuda_error(cudaGetLastError()); return rc; }
        return CBG_OK;
    }
    const int KP = (k + 1) / 2, grid = multi_grid();
    // [fault word | planes of W | partials], the planes on the last 16-byte boundary of the first 256
    // bytes' end (the workspace itself may lie anywhere)
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    ws += 256 - (reinterpret_cast<size_t>(ws) & 15);
    int* fault = reinterpret_cast<int*>(ws - 16);
    float2* wsplit = reinterpret_cast<float2*>(ws);
    const size_t split = (size_t)2 * KP * ld * sizeof(float2);
    double* part = reinterpret_cast<double*>(ws + (split + 255) / 256 * 256);
    const int E = 16 / cbgmres_format_bytes(fmt);
    k_split_multi<<<(int)std::min<long long>(((long long)KP * ld / 2 + 255) / 256, 4096), 256, 0, s>>>(
        W, ldw, n, ld, k, KP, E, wsplit, fault);
    MultiArgs a{};
    a.V = static_cast<const unsigned char*>(V);
    a.ldb = ld * cbgmres_format_bytes(fmt);
    a.ncols = ncols;
    a.wsplit = wsplit;
    a.ld = ld;
    a.part = part;
    a.fault = fault;
    if (KP == 1) launch_fmt<1>(fmt, grid, s, a);
    else if (KP == 2) launch_fmt<2>(fmt, grid, s, a);
    else if (KP == 3) launch_fmt<3>(fmt, grid, s, a);
    else launch_fmt<4>(fmt, grid, s, a);
    k_multi_sum<<<(ncols * 2 * KP + 31) / 32, 256, 0, s>>>(part, grid, ncols, 2 * KP, k, ldh, scales, fault, H);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { cbg_record_cuda_error(e); return CBG_ERR_CUDA; }
    return CBG_OK;
}

}  // namespace

extern "C" {

size_t cbg_basis_dot_multi_workspace(int64_t ld, int ncols, int k)
{
    if (ld < 1 || ncols < 1 || ncols > MAXCOLS || k < 1 || k > KCALL) return 0;
    const int KP = (std::min(k, KMAX) + 1) / 2;
    const size_t split = (size_t)2 * KP * ld * sizeof(float2);
    const size_t part = (size_t)multi_grid() * ncols * 2 * KP * sizeof(double);
    const size_t cuda_core = 256 + (split + 255) / 256 * 256 + (part + 255) / 256 * 256;
    return std::max(cuda_core, cbg_tc_multi_workspace(ld));
}

int cbg_basis_dot_multi_path(int fmt, int64_t n, int ncols, const void* V, int64_t ld, const double* scales, int k,
                             const double* W, int64_t ldw, double* H, void* workspace, size_t ws_bytes, void* stream,
                             int path)
{
    if (cbgmres_format_bytes(fmt) == 0 || n < 1 || ncols < 1 || ncols > MAXCOLS || k < 1 || k > KCALL || !V ||
        ld < n || ld % TILE_ROWS || !scales || !W || ldw < n || !H || !workspace ||
        ws_bytes < cbg_basis_dot_multi_workspace(ld, ncols, k) || path < 0 || path > 2)
        return CBG_ERR_ARG;
    if (!aligned(V, cbgmres_format_bytes(fmt)) || !aligned(W, 8) || !aligned(scales, 8) || !aligned(H, 8))
        return CBG_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const bool tc_ok = fmt == CBG_F16 && ncols <= 128 && aligned(V, 16);   // (it reads 16 bytes at a time)
    if (path == 2 && !tc_ok) return CBG_ERR_UNSUPPORTED;
    const bool tc = path == 2 || (path == 0 && tc_ok);
    // groups of up to KMAX vectors, one after the other on the stream (the workspace is reused)
    for (int r0 = 0; r0 < k; r0 += KMAX) {
        const int kg = std::min(KMAX, k - r0);
        int rc = dot_multi_group(fmt, n, ncols, V, ld, scales, kg, W + (long long)r0 * ldw, ldw, H + r0, k, workspace,
                                 s, tc);
        if (rc) return rc;
    }
    return CBG_OK;
}

int cbg_basis_dot_multi(int fmt, int64_t n, int ncols, const void* V, int64_t ld, const double* scales, int k,
                        const double* W, int64_t ldw, double* H, void* workspace, size_t ws_bytes, void* stream)
{
    return cbg_basis_dot_multi_path(fmt, n, ncols, V, ld, scales, k, W, ldw, H, workspace, ws_bytes, stream, 0);
}

}  // extern "C"
