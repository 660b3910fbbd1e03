// cbg_stream.cuh -- the basis dot product h = V^T w (the CGS projection and its re-orthogonalisation, Fig. 1) with the
// compressed basis staged in shared memory by bulk copies (TMA).
//
// One block per SM: sixteen consumer warps and one producer warp.  The work items are
// the (column group, row tile) pairs, numbered group-major (TILE = 8 row groups x 32
// lanes x E rows, E = 16 / bytes per code, so one tile of one column is 4 KiB of codes),
// and a block owns a contiguous range of items, so the blocks' shares differ by at most
// one item (a block may start or end inside a column group).  The producer walks the
// block's items and for each one fills a
// stage of a ring in shared memory with one bulk copy per column (4 KiB each, L2
// evict-first) plus the tile of w as FP32 hi and lo planes; completion is counted in
// bytes on the stage's "full" mbarrier.  Consumer warp w takes row group w % 8 and half
// w / 8 of the stage's columns; its lanes own E consecutive rows, read their 16-byte code
// chunks from shared memory (a warp reads 512 contiguous bytes: no bank conflicts), and
// accumulate in double-float on the packed FP32x2 pipe; each warp releases the stage on
// its "empty" mbarrier.  Loads in flight are bounded by the ring (about 200 KiB per SM),
// not by registers, and the arithmetic never waits on a global load.  Every wait is
// bounded (cbg_tma.cuh): a pipeline that stops making progress records FAULT_TIMEOUT and
// the kernel returns after draining its own copies.
#pragma once
#include <algorithm>
#include <type_traits>

#include "cbg_kernels.cuh"
#include "cbg_tma.cuh"

namespace cbg {

constexpr int TMA_CW = 8;                            // row groups of a tile
constexpr int DOT_CW = 2 * TMA_CW;                   // consumer warps: two per row group
constexpr int DOT_THREADS = (DOT_CW + 1) * 32;       // + one producer warp
constexpr int TMA_SMEM_OPTIN = 232448;               // shared memory per block (227 KiB)
constexpr int TMA_MAX_STAGES = 4;

template <int FMT> struct TmaGeom {
    static constexpr int BS = FmtInfo<FMT>::bytes;
    static constexpr int E = 16 / BS;                // rows per lane (a 16-byte code chunk)
    static constexpr int TILE = TMA_CW * 32 * E;     // rows per tile
    static constexpr int COLB = TILE * BS;           // bytes of one column's tile (4096)
    static constexpr int CG_DOT = E >= 8 ? 8 : 16;   // columns per stage (register accumulators)
    static constexpr int WB = TILE * 8;              // w tile: FP32 hi plane then lo plane
    static constexpr int STAGE_DOT = CG_DOT * COLB + WB;
};

// Dynamic shared memory of the pipelined dot: `stages` ring stages and 2 x stages
// mbarriers.  The ring gets whatever the kernel's static shared memory leaves.
inline int tma_stages(int stage_bytes, int static_bytes)
{
    const int s = (TMA_SMEM_OPTIN - static_bytes - 2 * TMA_MAX_STAGES * 8) / stage_bytes;
    return s < TMA_MAX_STAGES ? s : TMA_MAX_STAGES;
}
inline size_t tma_smem_bytes(int stages, int stage_bytes) { return (size_t)stages * stage_bytes + 2 * (size_t)stages * 8; }

// the block's contiguous range [ib, ie) of nitems work items
__device__ __forceinline__ void block_items(long long nitems, long long& ib, long long& ie)
{
    ib = (long long)blockIdx.x * nitems / gridDim.x;
    ie = ((long long)blockIdx.x + 1) * nitems / gridDim.x;
}

__device__ __forceinline__ void record_fault(DevState* st, int* fault)
{
    if (fault) atomicExch(fault, FAULT_TIMEOUT);
    else if (st) atomicExch(&st->fault, FAULT_TIMEOUT);
}

// Barrier of all blocks of a cooperative launch on one counter word: bits 0..30 count the
// arrivals, bit 31 is the sense, flipped by the last arrival (which also zeroes the
// count), so the word is ready for the next launch as it is left.  Thread 0 of each
// block arrives (releasing the block's writes) and polls (acquiring the others'; bounded:
// false when the wait gave up).
__device__ __forceinline__ bool grid_barrier(unsigned int* cnt, long long limit)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned sense, old, now;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(sense) : "l"(cnt) : "memory");
        sense &= 0x80000000u;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(cnt) : "memory");
        int good = 1;
        if ((old & 0x7FFFFFFFu) == gridDim.x - 1) {
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(cnt), "r"(sense ^ 0x80000000u) : "memory");
        } else {
            const long long t0 = clock64();
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(cnt) : "memory");
                if ((now & 0x80000000u) != sense) break;
                if (clock64() - t0 > limit) {
                    good = 0;
                    break;
                }
            }
        }
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// position in the ring: stage index and the parity of its current use
struct Ring {
    int s = 0;
    unsigned ph = 0;
    __device__ __forceinline__ void next(int stages)
    {
        if (++s == stages) { s = 0; ph ^= 1u; }
    }
};

// E consecutive floats (E a power of two, 4*E-byte aligned) with vector loads
template <int E> __device__ __forceinline__ void load_floats(const float* p, float* out)
{
    if constexpr (E == 2) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        out[0] = v.x;
        out[1] = v.y;
    } else {
#pragma unroll
        for (int e = 0; e < E; e += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + e);
            out[e] = v.x;
            out[e + 1] = v.y;
            out[e + 2] = v.z;
            out[e + 3] = v.w;
        }
    }
}

// Producer side of the ring: for every work item (group-major), wait until the consumers
// released the stage, announce the bytes, and issue the copies (lane q < nc copies column
// c0 + q; lanes 30 and 31 copy the hi and lo planes of w's tile).  Afterwards wait
// (bounded) until every issued copy has landed, so no copy outlives the block.
template <int COLB>
__device__ __forceinline__ void tma_produce(unsigned char* ring, int stage_bytes, int stages, uint64_t* full,
                                            uint64_t* empty, long long ib, long long ie, long long ntiles, int ncols,
                                            int cg, const unsigned char* V, long long ldb, const float* wsrc,
                                            long long wld, int tile_rows, int* failed, long long limit, bool withhold)
{
    const int lane = threadIdx.x & 31;
    const long long nitems = ie - ib;
    const uint64_t pol = l2_evict_first_policy();
    const unsigned wplane = (unsigned)tile_rows * 4u;
    Ring rg;
    int g = ntiles > 0 ? (int)(ib / ntiles) : 0;
    long long t = ib - (long long)g * ntiles, it = 0;
    for (; it < nitems; it++) {
        const int c0 = g * cg;
        const int nc = ncols - c0 < cg ? ncols - c0 : cg;
        if (it >= stages && !warp_wait(&empty[rg.s], rg.ph ^ 1u, limit)) { *failed = 1; break; }
        unsigned char* st = ring + (size_t)rg.s * stage_bytes;
        if (!(withhold && it == 0)) {
            if (lane == 0) mbar_arrive_expect_tx(&full[rg.s], (unsigned)(nc * COLB) + 2u * wplane);
            __syncwarp();
            if (lane < nc)
                bulk_g2s_hint(st + lane * COLB, V + (long long)(c0 + lane) * ldb + t * COLB, COLB, &full[rg.s], pol);
            if (lane >= 30) {
                const float* src = wsrc + (lane == 31 ? wld : 0) + t * tile_rows;
                bulk_g2s(st + cg * COLB + (lane == 31 ? wplane : 0u), src, wplane, &full[rg.s]);
            }
        }
        __syncwarp();
        rg.next(stages);
        if (++t == ntiles) { t = 0; g++; }
    }
    // drain: walk back over the last min(it, stages) items, the newest use of each stage
    const long long nd = it < stages ? it : stages;
    for (long long j = 0; j < nd; j++) {
        if (--rg.s < 0) { rg.s = stages - 1; rg.ph ^= 1u; }
        if (!warp_wait(&full[rg.s], rg.ph, limit)) { *failed = 1; break; }
    }
}

// ============================================================== h = V^T w  (CGS)
// Consumer warp of the dot: rows r .. r+E-1 of the tile and the CGW = CG/2 columns
// starting at q0 within the stage.  The packed FP32x2 operations take two neighbouring rows
// of one column: codes and w both lie so in registers as they are loaded (pairs of columns
// need every code moved next to its partner's and w duplicated: a third more instructions, on
// the pipes the products run on).  Component x of S2[q], C2[q] sums the even rows, y the odd
// ones.  A missing column (>= nc) holds stale codes; its sums are never read back.
template <int FMT, bool FULL>
__device__ __forceinline__ void dot_consume(const unsigned char* st, int r, int q0, int nc, float2* S2, float2* C2)
{
    using G = TmaGeom<FMT>;
    constexpr int E = G::E, CG = G::CG_DOT, CGW = CG / 2, BS = G::BS;
    float wh[E], wl[E];
    const float* wt = reinterpret_cast<const float*>(st + CG * G::COLB);
    load_floats<E>(wt + r, wh);
    load_floats<E>(wt + G::TILE + r, wl);
    float2 w2[E / 2], nw2[E / 2], l2[E / 2];
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        w2[e / 2] = make_float2(wh[e], wh[e + 1]);
        nw2[e / 2] = make_float2(-wh[e], -wh[e + 1]);
        l2[e / 2] = make_float2(wl[e], wl[e + 1]);
    }
#pragma unroll
    for (int q = 0; q < CGW; q++) {
        if (!FULL && q0 + q >= nc) break;
        Chunk<FMT> ch;
        decode_chunk<FMT>(*reinterpret_cast<const uint4*>(st + (q0 + q) * G::COLB + r * BS), ch);
        df2_mac_chunk<FMT>(S2[q], C2[q], ch, w2, nw2, l2);
    }
}

// barrier among the dot's consumer warps only (the producer never takes part)
__device__ __forceinline__ void consumers_sync()
{
    asm volatile("bar.sync 1, %0;" ::"r"(DOT_CW * 32) : "memory");
}

// The blocks' column totals (a.part[block][MAXCOLS], written by the block's threads before) to
// a.out = scales .* total.  Grid barrier (the kernels are launched cooperatively: every block
// is resident), then block b adds the partials of the columns b, b + gridDim.x, ..., a warp per
// column: its lanes add the blocks lane, lane + 32, ... (five loads in flight) and fold.  The
// cross-block sum is in FP64 and spread over all SMs: an FP64 instruction occupies GB300's pipe for
// 20 cycles per SM, so a few columns per block cost little, where 152 partials of every
// column added by one block took 2 to 4 us of a launch.  Mean over a restart cycle of 100 at
// 112^3, against double-float sums: f32 52.4 us (52.6), i16 45.4 (45.0), f64 98.4 (98.8); of
// one-signed data those were 1e-15 off, these are 1e-16.
__device__ __forceinline__ void dot_finish(const DotArgs& a, int ncols, long long limit, int* fault)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (!grid_barrier(a.counter, limit)) {
        if (threadIdx.x == 0) record_fault(nullptr, fault);
        return;
    }
    const int nb = gridDim.x;
    for (int col = blockIdx.x + warp * nb; col < ncols; col += nw * nb) {
        double s = 0.0;
        for (int t0 = 0; t0 < nb; t0 += 160) {
            double v[5];
#pragma unroll
            for (int u = 0; u < 5; u++) {
                const int t = t0 + lane + 32 * u;
                v[u] = t < nb ? __ldcg(a.part + (long long)t * MAXCOLS + col) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 5; u++) s = __dadd_rn(s, v[u]);
        }
        s = warp_sum(s);
        if (lane == 0) a.out[col] = s * a.scales[col];
    }
}

// DF32 arithmetic; a.wdf (w split into FP32 hi and lo planes) is required.  Sixteen
// consumer warps: warp w takes rows group (w % 8) of every tile and half (w / 8) of every
// stage's columns.  At the end of every column group the consumer warps meet once (a
// hardware barrier) and the group's per-warp sums are added in a fixed order, so the
// block's column totals need only MAXCOLS doubles of shared memory.  A warp whose wait
// timed out stops computing and stops releasing stages but still takes every group
// barrier, so the other warps never wait on it forever.
template <int FMT>
__global__ void __launch_bounds__(DOT_THREADS, 1) k_basis_dot_tma(DotArgs a, int stages, int* fault)
{
    if (a.active && *a.active == 0) return;
    using G = TmaGeom<FMT>;
    constexpr int CG = G::CG_DOT, CGW = CG / 2, E = G::E;
    constexpr int LOW = fold_low<CGW>();
    extern __shared__ __align__(128) unsigned char tma_smem[];
    unsigned char* ring = tma_smem;
    uint64_t* full = reinterpret_cast<uint64_t*>(tma_smem + (size_t)stages * G::STAGE_DOT);
    uint64_t* empty = full + stages;
    __shared__ float2 red_g[2][TMA_CW][CG];   // per row group sums of the current group (double-buffered)
    __shared__ double red_tot[MAXCOLS];       // the block's column totals
    __shared__ int failed;
    const int ncols = a.ncols_dev ? *a.ncols_dev : a.ncols;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long limit = a.wait_limit > 0 ? a.wait_limit : WAIT_LIMIT_CYCLES;
    const long long ntiles = a.nrows / G::TILE;
    const int ngroups = (ncols + CG - 1) / CG;
    long long ib, ie;
    block_items(ntiles * ngroups, ib, ie);

    if (threadIdx.x == 0) {
        failed = 0;
        for (int s = 0; s < stages; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], DOT_CW);
        }
        mbar_init_fence();
    }
    for (int i = threadIdx.x; i < MAXCOLS; i += DOT_THREADS) red_tot[i] = 0.0;
    __syncthreads();

    if (warp == DOT_CW) {
        int f = 0;
        tma_produce<G::COLB>(ring, G::STAGE_DOT, stages, full, empty, ib, ie, ntiles, ncols, CG, a.V, a.ldb, a.wdf,
                             a.nrows, G::TILE, &f, limit, a.withhold != 0);
        if (f) failed = 1;
    } else if (ie > ib) {
        const int rgp = warp % TMA_CW, q0 = (warp / TMA_CW) * CGW;
        const int r = (rgp * 32 + lane) * E;      // first row of this lane within a tile
        bool bad = false;
        Ring rg;
        const int gb = (int)(ib / ntiles), ge = (int)((ie - 1) / ntiles) + 1;   // the block's column groups
        for (int g = gb; g < ge; g++) {
            const int c0 = g * CG;
            const int nc = ncols - c0 < CG ? ncols - c0 : CG;
            // this block's tiles of group g
            const long long tb = ib > (long long)g * ntiles ? ib - (long long)g * ntiles : 0;
            const long long te = ie < (long long)(g + 1) * ntiles ? ie - (long long)g * ntiles : ntiles;
            float2 S2[CGW], C2[CGW];
#pragma unroll
            for (int q = 0; q < CGW; q++) { S2[q] = make_float2(0.f, 0.f); C2[q] = make_float2(0.f, 0.f); }
            for (long long t = tb; t < te; t++) {
                if (!bad && !warp_wait(&full[rg.s], rg.ph, limit)) {
                    bad = true;
                    failed = 1;
                }
                if (!bad) {
                    const unsigned char* st = ring + (size_t)rg.s * G::STAGE_DOT;
                    if (nc == CG) dot_consume<FMT, true>(st, r, q0, nc, S2, C2);
                    else dot_consume<FMT, false>(st, r, q0, nc, S2, C2);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[rg.s]);
                }
                rg.next(stages);
            }
            float S[CGW], C[CGW];
#pragma unroll
            for (int q = 0; q < CGW; q++) {
                S[q] = S2[q].x;
                C[q] = C2[q].x;
                df_add(S[q], C[q], S2[q].y, C2[q].y);
            }
            const int col = df_warp_fold<CGW>(S, C, lane);
            if ((lane & LOW) == 0) red_g[g & 1][rgp][q0 + col] = make_float2(S[0], C[0]);
            consumers_sync();
            // red_g[g & 1] is rewritten two groups later, after the next barrier
            // (the row groups added in FP64, a lane each)
            const int tid = warp * 32 + lane;
            if (tid < CG * TMA_CW) {
                const int c = tid / TMA_CW;
                const float2 v = c < nc ? red_g[g & 1][tid % TMA_CW][c] : make_float2(0.f, 0.f);
                double s = df_to_double(v.x, v.y);
#pragma unroll
                for (int o = TMA_CW / 2; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
                if (tid % TMA_CW == 0 && c < nc) red_tot[c0 + c] = s;
            }
        }
    }
    __syncthreads();
    if (failed && threadIdx.x == 0) record_fault(nullptr, fault);
    for (int col = threadIdx.x; col < ncols; col += DOT_THREADS) a.part[(long long)blockIdx.x * MAXCOLS + col] = red_tot[col];
    dot_finish(a, ncols, limit, fault);
}

// =============================================== w -= V h, u = V^T w in one pass over V
// The subtraction of the first CGS pass and the projection of the second one: each row of
// w - V h needs only that row of V, so a tile of rows that holds all columns in shared memory
// serves both products, and a step reads the basis three times instead of four.
//
// What bounds it: the double-float products, 2 x 11 FP32 operations an element and the
// decoding (twice; FP64 codes are split once and kept as pairs in place); ncu at 96^3, 96
// columns: f32 89 us, FMA pipe 66 %, f64 160 us, issue 62 %, a tile's barriers 15 to 10 % of the
// stalls.  Mean over a restart cycle of 100, this pass against the axpy and the dot that it
// replaces: f32 128^3 150 -> 117 us, 96^3 76 -> 58; f64 276 -> 206, 132 -> 95; f16 131 -> 120,
// 67 -> 62; i16 137 -> 124; i32 164 -> 148; e4m3 133 -> 128; never slower from 27,000 rows (f32 25 -> 15)
// to 2,097,152 and from 16 to 112 columns.  (With double-float block totals; the FP64 ones since
// then take 0 to 1 us more, f32 of 57 columns and more 3 %: 112^3 116.6 -> 119.9.)
//
// Sixteen warps in two groups of eight; a group works on its own tile, so one group's
// products cover the other's barriers.  A tile is `rs` spans of 512 bytes of codes per
// column (32 lanes x 16 bytes), all columns; warp w of a group takes the span w / sets and
// the columns w % sets, w % sets + sets, ... (sets = 8 / rs).  Few columns take more spans: the
// tile stays large and the warps' partial rows few.  rs is a template parameter: with it
// at run time the divisions and strides took a third of the instructions (f32 128^3 150 us,
// no gain).  Every thread copies (cp.async) exactly the codes that it reads, into slots of
// its warp, so the copies need no barrier; bulk copies of 512 bytes a column took 80 cycles
// each to issue.
// Phase A: the lane's rows of V h over its columns; the sets' partial rows meet in shared
// memory, where w is updated, and in memory.  Phase B: the same codes times the new w,
// accumulated per column in registers over all tiles of the block; a slot read here
// takes its next column at once.
constexpr int PS_GROUPS = 2, PS_GW = 8;          // groups, warps of a group
constexpr int PS_WARPS = PS_GROUPS * PS_GW, PS_THREADS = PS_WARPS * 32;   // 128 registers a thread
constexpr int PS_NCW = 14;                       // columns of a warp (register accumulators: 56 of 128)
constexpr int PS_MAXC = PS_GW * PS_NCW;          // columns the pass can hold

// Shared memory: slots [warps][slots][512 B] | per group: partial rows, sets x (rows + pad)
// floats for S, again for C, then the new w's planes | coefficients.
template <int FMT> struct PassGeom {
    static constexpr int BS = FmtInfo<FMT>::bytes;
    static constexpr int E = 16 / BS;
    static constexpr int SPAN = 32 * E;                            // rows of a span
    static constexpr int HE = E > 8 ? 8 : E;                       // rows a lane works on at a time
    static constexpr int COEF = PS_MAXC * 24;
    static constexpr int STATIC = PS_WARPS * 16 * 8 + 128;
    // threads that add one row's sets
    static constexpr __host__ __device__ int lanes(int rs)
    {
        const int sets = PS_GW / rs, t = PS_GW * 32 / (rs * SPAN);
        return t < 1 ? 1 : (t < sets ? t : sets);
    }
    static constexpr __host__ __device__ int exld(int rs) { return rs * SPAN + 32 / lanes(rs); }
    static constexpr __host__ __device__ int exch_floats(int rs)
    {
        const int sets = PS_GW / rs;
        return (sets > 1 ? 2 * sets * exld(rs) : 0) + 2 * rs * SPAN;
    }
    static int warp_cols(int ncols, int rs) { return (ncols + PS_GW / rs - 1) / (PS_GW / rs); }
    static size_t fixed(int rs) { return (size_t)PS_GROUPS * exch_floats(rs) * 4 + COEF; }
    static int room(int rs) { return (int)((TMA_SMEM_OPTIN - STATIC - fixed(rs)) / (PS_WARPS * 512)); }
    // slots of a warp: the tile at work and (part of) the next one
    static int slots(int ncols, int rs) { return std::min(room(rs), 2 * warp_cols(ncols, rs)); }
    // whether `rs` spans hold all columns, with at least two slots for the next tile
    static bool holds(int ncols, int rs) { return warp_cols(ncols, rs) <= PS_NCW && warp_cols(ncols, rs) + 2 <= room(rs); }
    // the widest tile that leaves every block five of them (two groups): 16 of them was slower
    // (16 columns, 96^3: f16 31 -> 24 us, f32 28 -> 23), and as a rule on columns alone the last
    // tiles would leave half of the chip idle
    static int spans(int ncols, long long nrows, int grid)
    {
        int rs = 8;
        while (rs > 1 && (!holds(ncols, rs) || nrows / ((long long)rs * SPAN) < 5LL * grid)) rs >>= 1;
        return rs;
    }
};

struct PassArgs {
    DotArgs d;                // V, ldb, ncols, scales, nrows, part, active, counter; out = u
    const double* coef;       // h of the first pass
    float* wdf;               // w's planes, read and overwritten with w - V h
};

__device__ __forceinline__ void group_sync(int g)
{
    asm volatile("bar.sync %0, %1;" ::"r"(2 + g), "r"(PS_GW * 32) : "memory");
}

__device__ __forceinline__ void async_copy16(unsigned dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// P float pairs to p (8*P-byte aligned) with vector stores
template <int P> __device__ __forceinline__ void store_pairs(float* p, const float2* v)
{
    if constexpr (P == 1) *reinterpret_cast<float2*>(p) = v[0];
    else {
#pragma unroll
        for (int e = 0; e < P; e += 2)
            *reinterpret_cast<float4*>(p + 2 * e) = make_float4(v[e].x, v[e].y, v[e + 1].x, v[e + 1].y);
    }
}

// HE rows of one column as float pairs (1-byte codes: 8 of a chunk's 16 rows).  SPLIT: FP64
// codes were replaced by their pairs
template <int FMT> __device__ __forceinline__ uint4 pass_load(unsigned p)
{
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (PassGeom<FMT>::E > PassGeom<FMT>::HE)
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(p) : "memory");
    else
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p) : "memory");
    return v;
}
template <int FMT, bool SPLIT> __device__ __forceinline__ void pass_decode(const uint4& raw, float2* vh, float2* vl)
{
    constexpr int E = PassGeom<FMT>::E, HE = PassGeom<FMT>::HE;
    if constexpr (FMT == F64 && SPLIT) {
        vh[0] = make_float2(__uint_as_float(raw.x), __uint_as_float(raw.y));
        vl[0] = make_float2(__uint_as_float(raw.z), __uint_as_float(raw.w));
    } else if constexpr (E > HE) {
        const unsigned w[2] = {raw.x, raw.y};
#pragma unroll
        for (int k = 0; k < 2; k++) {
            dec_e4m3x2(w[k] & 0xFFFFu, vh[2 * k].x, vh[2 * k].y);
            dec_e4m3x2(w[k] >> 16, vh[2 * k + 1].x, vh[2 * k + 1].y);
        }
    } else {
        Chunk<FMT> ch;
        decode_chunk<FMT>(raw, ch);
#pragma unroll
        for (int e = 0; e < E; e += 2) {
            vh[e / 2] = make_float2(ch.vh[e], ch.vh[e + 1]);
            if constexpr (!SingleFloat<FMT>::value) vl[e / 2] = make_float2(ch.vl[e], ch.vl[e + 1]);
        }
    }
}

template <int FMT, int rs>
__global__ void __launch_bounds__(PS_THREADS, 1) k_basis_pass(PassArgs a, int slots, int* fault)
{
    if (a.d.active && *a.d.active == 0) return;
    using G = PassGeom<FMT>;
    constexpr int E = G::E, HE = G::HE, SPAN = G::SPAN;
    constexpr bool SF = SingleFloat<FMT>::value;
    extern __shared__ __align__(128) unsigned char tma_smem[];
    constexpr int rows = rs * SPAN, sets = PS_GW / rs, tpr = G::lanes(rs), exld = G::exld(rs);
    const int ncols = a.d.ncols;
    // (the shuffle tells the compiler that everything derived from the warp index is uniform)
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int g = warp / PS_GW, gw = warp % PS_GW, set = gw % sets, span = gw / sets;
    const int nq = ncols > set ? (ncols - set + sets - 1) / sets : 0;     // this warp's columns
    const int gt = threadIdx.x & (PS_GW * 32 - 1);                        // thread of the group
    const int r0 = (span * 32 + lane) * E;                                // first row of this lane in the tile
    float* exS = reinterpret_cast<float*>(tma_smem + (size_t)PS_WARPS * slots * 512) + g * G::exch_floats(rs);
    float* exC = exS + sets * exld;
    float* wt = exS + (sets > 1 ? 2 * sets * exld : 0);                   // the new w's planes
    float4* ca = reinterpret_cast<float4*>(tma_smem + (size_t)PS_WARPS * slots * 512 +
                                           PS_GROUPS * G::exch_floats(rs) * 4);      // (c, c, -c, -c)
    float2* cb = reinterpret_cast<float2*>(ca + PS_MAXC);                            // (c low, c low)
    __shared__ float2 red_w[PS_WARPS][16];
    const long long limit = a.d.wait_limit > 0 ? a.d.wait_limit : WAIT_LIMIT_CYCLES;
    long long tb, te;
    block_items(a.d.nrows / rows, tb, te);

    // The warp's slots.  Column q of a tile lies in slot q; the first `ahead` columns (a multiple
    // of four, or all) alternate with the slots nq + q from tile to tile, so that they can be
    // copied a tile earlier.  A slot read for the last time takes its next column at once.
    const unsigned slot0 = smem_addr(tma_smem) + (unsigned)(warp * slots * 512 + lane * 16);
    int ahead = slots - nq;
    ahead = ahead >= nq ? nq : ahead & ~3;
    const long long cstep = (long long)sets * a.d.ldb, tstep = (long long)PS_GROUPS * rs * 512;
    const unsigned char* src = a.d.V + set * a.d.ldb + (span * 32 + lane) * 16 + (tb + g) * (rs * 512);
    // copies are committed as: a tile's first columns, its others, the next tile's first columns
    if (tb + g < te)
        for (int i = 0; i < ahead; i++) async_copy16(slot0 + i * 512, src + i * cstep);
    async_commit();
    if (tb + g < te)
        for (int i = ahead; i < nq; i++) async_copy16(slot0 + i * 512, src + i * cstep);
    async_commit();
    if (tb + g + PS_GROUPS < te)
        for (int i = 0; i < ahead; i++) async_copy16(slot0 + (nq + i) * 512, src + tstep + i * cstep);
    async_commit();
    // coefficients in the order of use: [set][q]
    for (int k = threadIdx.x; k < PS_MAXC; k += PS_THREADS) {
        float h = 0.f, l = 0.f;
        if (k < ncols) split_f64(-a.d.scales[k] * a.coef[k], h, l);
        const int at = (k % sets) * PS_NCW * rs + k / sets;
        ca[at] = make_float4(h, h, -h, -h);
        cb[at] = make_float2(l, l);
    }
    __syncthreads();

    float2 S2[PS_NCW], C2[PS_NCW];
#pragma unroll
    for (int q = 0; q < PS_NCW; q++) { S2[q] = make_float2(0.f, 0.f); C2[q] = make_float2(0.f, 0.f); }
    const float4* const wca = ca + set * PS_NCW * rs;
    const float2* const wcb = cb + set * PS_NCW * rs;
    unsigned first = slot0;                       // slots of the first columns: slot0 or slot0 + nq * 512
    float* wg = a.wdf + (tb + g) * rows;
    for (int left = (int)((te - tb - g + PS_GROUPS - 1) / PS_GROUPS); left > 0; left--, wg += PS_GROUPS * rows) {
        // the row that this thread will update, ahead of its use
        float w0h = 0.f, w0l = 0.f;
        if (sets > 1 && gt % tpr == 0) {
            w0h = __ldcg(wg + gt / tpr);
            w0l = __ldcg(wg + a.d.nrows + gt / tpr);
        }
        // ---- phase A: rows of V c over this warp's columns
        async_wait<2>();
#pragma unroll
        for (int hf = 0; hf < E / HE; hf++) {
            constexpr int P = HE / 2, NA = P == 1 ? 2 : 1;   // FP64: two chains of sums
            float2 A2[NA * P], B2[NA * P];
#pragma unroll
            for (int e = 0; e < NA * P; e++) { A2[e] = make_float2(0.f, 0.f); B2[e] = make_float2(0.f, 0.f); }
            auto columns = [&](int q0, auto count) {              // the codes of a few columns, then their products
                constexpr int N = decltype(count)::value;
                const unsigned p = (q0 < ahead ? first : slot0) + (unsigned)q0 * 512u;
                uint4 raw[N];
                float4 c4[N];
                float2 cl[N];
#pragma unroll
                for (int u = 0; u < N; u++) {
                    raw[u] = pass_load<FMT>(p + u * 512 + hf * 8);
                    c4[u] = wca[q0 + u];
                    cl[u] = wcb[q0 + u];
                }
                float2 vh[N][P], vl[N][SF ? 1 : P];
#pragma unroll
                for (int u = 0; u < N; u++) {
                    pass_decode<FMT, false>(raw[u], vh[u], vl[u]);
                    const float2 ch = make_float2(c4[u].x, c4[u].y), nch = make_float2(c4[u].z, c4[u].w);
#pragma unroll
                    for (int e = 0; e < P; e++) {
                        const int x = (u % NA) * P + e;
                        if constexpr (SF) df2_mac(A2[x], B2[x], vh[u][e], ch, nch, cl[u]);
                        else df2_mac2(A2[x], B2[x], vh[u][e], vl[u][e], ch, nch, cl[u]);
                    }
                }
                if constexpr (FMT == F64) {
#pragma unroll
                    for (int u = 0; u < N; u++)
                        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p + u * 512), "f"(vh[u][0].x),
                                     "f"(vh[u][0].y), "f"(vl[u][0].x), "f"(vl[u][0].y)
                                     : "memory");
                }
            };
            auto renorm = [&] {
#pragma unroll
                for (int e = 0; e < NA * P; e++) df2_renorm(A2[e], B2[e]);
            };
            int q = 0;
            for (; q + 4 <= nq; q += 4) {
                if (q + 4 > ahead) async_wait<1>();
                if constexpr (SF) {
                    columns(q, std::integral_constant<int, 4>{});
                } else {                     // (pairs of floats: registers for two columns at a time)
                    columns(q, std::integral_constant<int, 2>{});
                    columns(q + 2, std::integral_constant<int, 2>{});
                }
                renorm();
            }
            async_wait<1>();
            for (; q < nq; q++) columns(q, std::integral_constant<int, 1>{});
            renorm();
            if constexpr (NA == 2) {
                df_add(A2[0].x, B2[0].x, A2[1].x, B2[1].x);
                df_add(A2[0].y, B2[0].y, A2[1].y, B2[1].y);
            }
            const int r = r0 + hf * HE;
            if (sets > 1) {
                store_pairs<HE / 2>(exS + set * exld + r, A2);
                store_pairs<HE / 2>(exC + set * exld + r, B2);
            } else {                    // all columns are this lane's own
#pragma unroll
                for (int e = 0; e < HE / 2; e++) {
                    const float2 wh = *reinterpret_cast<const float2*>(wg + r + 2 * e);
                    const float2 wl = *reinterpret_cast<const float2*>(wg + a.d.nrows + r + 2 * e);
                    df_add(A2[e].x, B2[e].x, wh.x, wl.x);
                    df_add(A2[e].y, B2[e].y, wh.y, wl.y);
                    df2_renorm(A2[e], B2[e]);
                }
                store_pairs<HE / 2>(wt + r, A2);
                store_pairs<HE / 2>(wt + rows + r, B2);
                store_pairs<HE / 2>(wg + r, A2);
                store_pairs<HE / 2>(wg + a.d.nrows + r, B2);
            }
        }
        if (sets > 1) {
            group_sync(g);
            const int part = gt % tpr;
#pragma unroll
            for (int i = 0; i < rows / (PS_GW * 32 / tpr); i++) {
                const int r = gt / tpr + i * (PS_GW * 32 / tpr);
                const float* e = exS + part * exld + r;
                float s = e[0], c = e[sets * exld];
#pragma unroll
                for (int k = tpr; k < sets; k += tpr) df_add(s, c, e[k * exld], e[(sets + k) * exld]);
#pragma unroll
                for (int o = 1; o < tpr; o <<= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
                    df_add(s, c, s2, c2);
                }
                if (part == 0) {
                    if (i > 0) {
                        w0h = __ldcg(wg + r);
                        w0l = __ldcg(wg + a.d.nrows + r);
                    }
                    df_add(s, c, w0h, w0l);
                    float h, l;
                    two_sum(s, c, h, l);
                    wt[r] = h;
                    wt[rows + r] = l;
                    wg[r] = h;
                    wg[a.d.nrows + r] = l;
                }
            }
            group_sync(g);
        }
        // ---- phase B: the warp's columns times the new w, last column first; their slots take
        // the next tile's columns, those of the first columns the tile's after that
        const bool more1 = left > 1, more2 = left > 2;
        if (ahead >= nq) async_commit();
#pragma unroll
        for (int hf = 0; hf < E / HE; hf++) {
            constexpr int U = HE > 4 ? 2 : 4;
            const int r = r0 + hf * HE;
            float2 w2[HE / 2], nw2[HE / 2], l2[HE / 2];
            load_floats<HE>(wt + r, reinterpret_cast<float*>(w2));
            load_floats<HE>(wt + rows + r, reinterpret_cast<float*>(l2));
#pragma unroll
            for (int e = 0; e < HE / 2; e++) nw2[e] = make_float2(-w2[e].x, -w2[e].y);
#pragma unroll
            for (int q0 = (PS_NCW - 1) / U * U; q0 >= 0; q0 -= U) {
                if (q0 < nq) {
                    const bool fst = q0 < ahead, more = fst ? more2 : more1;
                    const unsigned p = (fst ? first : slot0) + (unsigned)q0 * 512u;
                    const unsigned char* np = src + (fst ? 2 * tstep : tstep) + q0 * cstep;
                    auto group = [&](auto whole) {
                        constexpr bool W = decltype(whole)::value;       // all U columns exist
                        uint4 raw[U];
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (q0 + u < PS_NCW && (W || q0 + u < nq)) raw[u] = pass_load<FMT>(p + u * 512 + hf * 8);
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            if (q0 + u < PS_NCW && (W || q0 + u < nq)) {
                                const int q = q0 + u;
                                float2 vh[HE / 2], vl[SF ? 1 : HE / 2];
                                pass_decode<FMT, true>(raw[u], vh, vl);
#pragma unroll
                                for (int e = 0; e < HE / 2; e++) {
                                    if constexpr (SF) df2_mac(S2[q], C2[q], vh[e], w2[e], nw2[e], l2[e]);
                                    else df2_mac2(S2[q], C2[q], vh[e], vl[e], w2[e], nw2[e], l2[e]);
                                }
                                df2_renorm(S2[q], C2[q]);
                                if (!W && hf == E / HE - 1 && more) async_copy16(p + u * 512, np + u * cstep);
                            }
                        }
                        if (W && hf == E / HE - 1 && more) {
#pragma unroll
                            for (int u = 0; u < U; u++)
                                if (q0 + u < PS_NCW) async_copy16(p + u * 512, np + u * cstep);
                        }
                    };
                    if (q0 + U <= nq) group(std::true_type{});
                    else group(std::false_type{});
                    if (hf == E / HE - 1 && q0 == ahead) async_commit();
                }
            }
        }
        async_commit();
        src += tstep;
        first = first == slot0 ? slot0 + (unsigned)nq * 512u : slot0;
    }
    async_wait<0>();
    float S[16], C[16];
#pragma unroll
    for (int q = 0; q < 16; q++) {
        S[q] = q < PS_NCW ? S2[q < PS_NCW ? q : 0].x : 0.f;
        C[q] = q < PS_NCW ? C2[q < PS_NCW ? q : 0].x : 0.f;
        if (q < PS_NCW) df_add(S[q], C[q], S2[q].y, C2[q].y);
    }
    const int q = df_warp_fold<16>(S, C, lane);
    if ((lane & fold_low<16>()) == 0) red_w[warp][q] = make_float2(S[0], C[0]);
    __syncthreads();
    for (int c = threadIdx.x; c < ncols; c += PS_THREADS) {
        float4 tot = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int w = c % sets; w < PS_WARPS; w += sets) tf_add(tot, red_w[w][c / sets].x, red_w[w][c / sets].y);
        a.d.part[(long long)blockIdx.x * MAXCOLS + c] = tf_to_double(tot);
    }
    if (a.d.withhold && blockIdx.x + 1 == gridDim.x) return;     // (a test: the others' waits run out)
    dot_finish(a.d, ncols, limit, fault);
}

}  // namespace cbg
