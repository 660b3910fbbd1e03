// mlp_tc.cu -- the learned preconditioner's per-row network on the 5th-generation tensor
// cores: forward pass, backward pass, and one fused training pass (forward, loss from the
// per-row pair statistics, backward, weight gradients).
//
// Precision contract: every tensor-core operand is BF16 and every product sum accumulates
// in FP32 in tensor memory (the weight gradients over all of a CTA's rows).  The inputs
// of layers 1 and 2 (features, H1) and the output gradient enter as split pairs
// hi + lo of BF16 values (about 16 significant bits; the lo half is a second K block
// against a copy of the same weights), so the ReLU decisions are taken on FP32-accurate
// pre-activations; H2 and the backward's dZ2, dZ1 and the gradient products' operands
// are single BF16 values.  Biases, ReLU, the loss and its gradient are FP32 on the CUDA
// cores; the cross-CTA gradient sum is FP64 (k_grad_reduce).
//
// One CTA per SM, three warpgroups of 128 threads that work on tiles of their own (while one
// waits for the tensor core or for a barrier, the others compute): thread t of a warpgroup
// owns row t of a 128-row tile and tensor-memory lane t.  The weights are shared; a
// warpgroup has 64 KiB of activations, 160 columns of tensor memory and its own mbarrier.
// Per tile, with D = A B^T and activations as tiles of 128-byte rows (64 BF16 values, 128-byte
// swizzle, cbg_tc.cuh):
//   layer 1  Z1 = F  W1^T       M 128, N 64, K 16 (7 features hi, a one, 7 lo)
//   layer 2  Z2 = H1 W2^T       M 128, N 64, K 2 x 64    H1 = relu(Z1 + b1), hi and lo
//   layer 3  Y  = H2 W3^T       M 128, N 16, K 64        H2 = relu(Z2 + b2), out = Y + b3
//   dH2 = Gout W3               M 128, N 64, K 16        Gout = dL/dout, hi and lo
//   gW3^T += H2^T Gout          M 128, N 16, K = rows
//   dH1 = dZ2 W2                M 128, N 64, K 64        dZ2 = dH2 * [Z2 + b2 > 0]
//   [gW2 ; .] += [dZ2 | dZ1]^T H1                        M 128, N 64, K = rows
//   [. gb2 ; gW1 gb1] += [dZ2 | dZ1]^T [F | 1]           M 128, N 16, K = rows
// (dZ1 = dH1 * [Z1 + b1 > 0].)  The products over the rows read the row-major activations as
// MN-major operands, so no transposed copy is written (those took some 270 two-byte shared
// stores per row and 72 KiB per tile); the one behind the features (against a zero weight in
// layer 1) turns the bias gradients into output columns.  Rows 64-127 of the first and 0-63
// of the second product that are not named are not read.  Buffers are reused as they fall
// free: dZ2 takes the place of H1's lo part, dZ1 that of H2.  The weight-gradient sums stay in
// tensor memory across the warpgroup's tiles and are written once.  The inputs of a row go
// straight to registers, a phase ahead (the pair statistics lie one array per entry:
// coalesced, and the symmetric 7 x 7 matrix as its 28 entries).  Every wait on the tensor core
// is bounded: a wait that runs out sets *fault and the warpgroup leaves its tile loop.
//
// What bounds it: six dependent phases per tile (tensor-memory load, epilogue, operand stores,
// fence, barrier, MMA), the tensor pipe 14 % busy.  One training pass of 262,144 rows: 112 us
// with one warpgroup and transposed copies, 62 with two warpgroups reading MN-major operands,
// 54 with the weights copied from an image, about 48 with three; a training step with the
// gradient sum and Adam in one kernel 125 -> 61 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "cbg_device.cuh"
#include "cbg_mlp.h"
#include "cbg_tc.cuh"

namespace cbg {
namespace {

constexpr int WG = 128;                        // threads of a warpgroup: one per row of a tile
constexpr int NWG = MLP_PARTS;                 // warpgroups of a CTA
constexpr int MT = NWG * WG;
constexpr int ROWS = MLP_ROWS;
constexpr int TM_WG = 160;                     // tensor-memory columns of a warpgroup
constexpr int TM_COLS = 512;                   // allocated
// (one area for Z1, Z2, Y, dH2 and dH1: each is read before the next is issued)
constexpr int C_Z = 0, C_G2 = 64, C_GF = 128, C_G3 = 144;
constexpr int TILE_B = ROWS * TC_ROWB;         // bytes of an activation tile (16 KiB)
// shared memory, bytes from the 1024-aligned base: the weight image (cbg_mlp.h), the
// warpgroups' activations, and in their place at the end the gradient sums
constexpr int S_ACT = MLP_IMAGE_OPS;           // the warpgroups' activations
constexpr int A_H1 = 0;                        // [128 r][64] H1 hi
constexpr int A_HX = A_H1 + TILE_B;            // [128 r][64] H1 lo, then dZ2
constexpr int A_H2 = A_HX + TILE_B;            // [128 r][64] H2, then dZ1 (behind dZ2: one operand)
constexpr int A_FG = A_H2 + TILE_B;            // [128 r][F hi, 1, F lo, 0: 0-15 | Gout hi, 0, lo, 0: 16-31]
constexpr int ACT_BYTES = A_FG + TILE_B;       // (the tile behind A_H2 exists: an M of 128 reads it)
constexpr int S_BIAS = S_ACT + NWG * ACT_BYTES;   // b1[64], b2[64], b3[7] floats
constexpr int S_END = S_BIAS + MLP_IMAGE - MLP_IMAGE_OPS;
// gradient sums of a warpgroup, floats: gW2 with rows of 65 (conflict-free), then the rest
constexpr int GS_W2 = 65, GS_END = NH * GS_W2 + NPARAM - NH * NH;
constexpr int MLP_SMEM = S_END + 1024;         // + alignment slack
static_assert(S_ACT % 1024 == 0 && ACT_BYTES % 1024 == 0, "operand tiles start on 1024-byte swizzle atoms");
static_assert(MLP_SMEM <= 232448, "fits the opt-in shared memory of one CTA");
static_assert(NWG * TM_WG <= TM_COLS, "fits tensor memory");
static_assert(GS_END * 4 <= ACT_BYTES, "gradient sums fit the warpgroup's activations");

__device__ __forceinline__ unsigned int bf2(float lo, float hi)
{
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned int*>(&b);
}
__device__ __forceinline__ float bf_lo(unsigned int u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(unsigned int u) { return __uint_as_float(u & 0xFFFF0000u); }
// the rounding residuals of a packed pair: (x0, x1) - (hi pair), again as a BF16 pair
// (the differences are exact in FP32)
__device__ __forceinline__ unsigned int bf2_rest(float x0, float x1, unsigned int hi)
{
    return bf2(x0 - bf_lo(hi), x1 - bf_hi(hi));
}

// a parameter's place in the gradient sums
__device__ __forceinline__ int grad_slot(int idx)
{
    const int q = idx - OFF_W2;
    if (q >= 0 && q < NH * NH) return (q >> 6) * GS_W2 + (q & 63);
    return NH * GS_W2 + (q < 0 ? idx : idx - NH * NH);
}

// Eight BF16 values of this thread's row (four packed pairs) into chunk `chunk` of an
// activation row
__device__ __forceinline__ void put_row8(unsigned char* base, int row, int chunk, const unsigned int* pk)
{
    *reinterpret_cast<uint4*>(base + tc_swz(row, chunk)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

// barrier of one warpgroup
__device__ __forceinline__ void wg_sync(int wg) { asm volatile("bar.sync %0, %1;" ::"r"(1 + wg), "r"(WG) : "memory"); }
__device__ __forceinline__ bool wg_all(int wg, bool mine)
{
    unsigned all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.red.and.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(all)
        : "r"((unsigned)mine), "r"(1 + wg), "r"(WG)
        : "memory");
    return all != 0;
}

template <int MODE>
__global__ void __launch_bounds__(MT, 1) k_mlp_tc(MlpArgs a)
{
    extern __shared__ unsigned char mlp_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(((size_t)mlp_raw + 1023) & ~(size_t)1023);
    __shared__ __align__(8) uint64_t mbar[NWG];
    __shared__ uint32_t tbase;
    __shared__ float red_b3[MT / 32][8];
    __shared__ double red_l[MT / 32];
    const int wg = threadIdx.x / WG, t = threadIdx.x % WG, warp = threadIdx.x >> 5, lane = t & 31;
    const long long ntiles = (a.n + ROWS - 1) / ROWS;
    constexpr bool BACK = MODE != MLP_FWD;

    // the weight operands and biases as they lie in the image (activations are written before
    // they are read; what an MMA reads beyond them only reaches outputs that are not read)
    const uint4* img = reinterpret_cast<const uint4*>(a.image);
    for (int i = threadIdx.x; i < MLP_IMAGE / 16; i += MT)
        reinterpret_cast<uint4*>(sm + (i < MLP_IMAGE_OPS / 16 ? 0 : S_BIAS - MLP_IMAGE_OPS))[i] = __ldg(img + i);
    if (warp == 0) tc_alloc(&tbase, TM_COLS);
    if (threadIdx.x == 0) {
        for (int w = 0; w < NWG; w++) mbar_init(&mbar[w], 1);
        mbar_init_fence();
    }
    const float* sb = reinterpret_cast<const float*>(sm + S_BIAS);
    tc_fence_proxy();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    unsigned char* act = sm + S_ACT + wg * ACT_BYTES;
    const uint32_t tmem = tbase + (uint32_t)(wg * TM_WG);
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);   // this warp's lanes
    const uint32_t wbase = smem_addr(sm), abase = smem_addr(act);
    const float* b1 = sb;
    const float* b2 = sb + NH;
    const float* b3 = sb + 2 * NH;

    unsigned phase = 0;
    bool ok = true;
    // the warpgroup: the MMAs committed last have completed (bounded), agreed by all its threads
    auto mma_wait = [&]() -> bool {
        const bool mine = mbar_wait(&mbar[wg], phase & 1u);
        phase++;
        const bool all = wg_all(wg, mine);
        tc_fence_after();
        return all;
    };
    // the operand stores of the warpgroup are visible to the tensor core, and its
    // tensor-memory loads are complete, before thread 0 issues the next MMAs
    auto to_tensor_core = [&]() {
        tc_fence_proxy();
        tc_fence_before();
        wg_sync(wg);
    };
    // K-major operands: ksteps of 16 values
    auto mma = [&](int col, uint32_t a_at, uint32_t b_at, int N, int ksteps, int acc0) {
        const uint32_t id = tc_idesc(128, N, true);
        for (int kk = 0; kk < ksteps; kk++)
            tc_mma(tmem + (uint32_t)col, tc_desc(a_at + kk * 32), tc_desc(b_at + kk * 32), id,
                   (kk == 0 && !acc0) ? 0 : 1);
    };
    // products over the 128 rows: both operands MN-major, A the 64 columns at a_at and the 64 of
    // the next tile behind it
    auto mma_rows = [&](int col, uint32_t a_at, uint32_t b_at, int N, bool acc0) {
        const uint32_t id = tc_idesc(128, N, true) | TC_A_MN | TC_B_MN;
        for (int kk = 0; kk < ROWS / 16; kk++)
            tc_mma(tmem + (uint32_t)col, tc_desc_mn(a_at + kk * 16 * TC_ROWB, TILE_B),
                   tc_desc_mn(b_at + kk * 16 * TC_ROWB, TILE_B), id, (kk == 0 && !acc0) ? 0 : 1);
    };

    float gb3[NOUT];
#pragma unroll
    for (int k = 0; k < NOUT; k++) gb3[k] = 0.f;
    double loss = 0.0;
    bool first = true;
    const long long tile0 = (long long)blockIdx.x * NWG + wg, tstep = (long long)gridDim.x * NWG;
    float feat[NIN];
    auto load_features = [&](long long tile) {
        const long long i = tile * ROWS + t;
        const bool in = tile < ntiles && i < a.n;
#pragma unroll
        for (int k = 0; k < NIN; k++) feat[k] = in ? __ldg(a.feat + i * NIN + k) : 0.f;
    };
    load_features(tile0);
    bool pending = false;                                 // the last gradient products still run
    for (long long tile = tile0; tile < ntiles; tile += tstep) {
        const long long i = tile * ROWS + t;
        const bool valid = i < a.n;
        // ---- features: F hi, the one, F lo (after the previous tile's gradient products)
        if (pending && !(ok = mma_wait())) break;
        pending = false;
        {
            unsigned int pk[4] = {bf2(feat[0], feat[1]), bf2(feat[2], feat[3]), bf2(feat[4], feat[5]), bf2(feat[6], 1.f)};
            unsigned int pl[4] = {bf2_rest(feat[0], feat[1], pk[0]), bf2_rest(feat[2], feat[3], pk[1]),
                                  bf2_rest(feat[4], feat[5], pk[2]), bf2_rest(feat[6], 1.f, pk[3])};
            put_row8(act + A_FG, t, 0, pk);
            put_row8(act + A_FG, t, 1, pl);
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma(C_Z, abase + A_FG, wbase + IMG_W1, 64, 1, 0);
            tc_commit(&mbar[wg]);
        }
        load_features(tile + tstep);
        if (!(ok = mma_wait())) break;
        // ---- layer 1 epilogue: H1 = relu(Z1 + b1)
        unsigned long long m1 = 0ull, m2 = 0ull;
#pragma unroll
        for (int c1 = 0; c1 < NH; c1 += 32) {
          uint32_t vv[32];
          tc_ld16(tl + C_Z + c1, vv);
          tc_ld16(tl + C_Z + c1 + 16, vv + 16);
          tc_wait_ld();
#pragma unroll
          for (int c0 = c1; c0 < c1 + 32; c0 += 16) {
            const uint32_t* v = vv + (c0 - c1);
            unsigned int pk[8], pl[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const float z0 = __uint_as_float(v[e]) + b1[c0 + e], z1 = __uint_as_float(v[e + 1]) + b1[c0 + e + 1];
                m1 |= (z0 > 0.f ? 1ull : 0ull) << (c0 + e);
                m1 |= (z1 > 0.f ? 1ull : 0ull) << (c0 + e + 1);
                const float h0 = fmaxf(z0, 0.f), h1 = fmaxf(z1, 0.f);
                pk[e >> 1] = bf2(h0, h1);
                pl[e >> 1] = bf2_rest(h0, h1, pk[e >> 1]);
            }
            put_row8(act + A_H1, t, c0 >> 3, pk);
            put_row8(act + A_H1, t, (c0 >> 3) + 1, pk + 4);
            put_row8(act + A_HX, t, c0 >> 3, pl);
            put_row8(act + A_HX, t, (c0 >> 3) + 1, pl + 4);
          }
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma(C_Z, abase + A_H1, wbase + IMG_W2, 64, 4, 0);
            mma(C_Z, abase + A_HX, wbase + IMG_W2, 64, 4, 1);
            tc_commit(&mbar[wg]);
        }
        if (!(ok = mma_wait())) break;
        // ---- layer 2 epilogue: H2 = relu(Z2 + b2)
#pragma unroll
        for (int c1 = 0; c1 < NH; c1 += 32) {
          uint32_t vv[32];
          tc_ld16(tl + C_Z + c1, vv);
          tc_ld16(tl + C_Z + c1 + 16, vv + 16);
          tc_wait_ld();
#pragma unroll
          for (int c0 = c1; c0 < c1 + 32; c0 += 16) {
            const uint32_t* v = vv + (c0 - c1);
            unsigned int pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const float z0 = __uint_as_float(v[e]) + b2[c0 + e], z1 = __uint_as_float(v[e + 1]) + b2[c0 + e + 1];
                m2 |= (z0 > 0.f ? 1ull : 0ull) << (c0 + e);
                m2 |= (z1 > 0.f ? 1ull : 0ull) << (c0 + e + 1);
                pk[e >> 1] = bf2(fmaxf(z0, 0.f), fmaxf(z1, 0.f));
            }
            put_row8(act + A_H2, t, c0 >> 3, pk);
            put_row8(act + A_H2, t, (c0 >> 3) + 1, pk + 4);
          }
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma(C_Z, abase + A_H2, wbase + IMG_W3, 16, 4, 0);
            tc_commit(&mbar[wg]);
        }
        // ---- inputs of the loss or the given output gradient, in flight during layer 3
        float gin[NOUT], G[28], cc[NOUT], dd = 0.f, id = 0.f;
        unsigned int mk = 0u;
        if (MODE == MLP_TRAIN) {
#pragma unroll
            for (int k = 0; k < 28; k++) G[k] = valid ? __ldg(a.G + (long long)k * a.stride + i) : 0.f;
#pragma unroll
            for (int k = 0; k < NOUT; k++) cc[k] = valid ? __ldg(a.c + (long long)k * a.stride + i) : 0.f;
            dd = valid ? __ldg(a.d + i) : 0.f;
            id = valid ? __ldg(a.idiag + i) : 0.f;
            mk = valid ? (unsigned)__ldg(a.mask + i) : 0u;
        }
        if (MODE == MLP_BWD) {
#pragma unroll
            for (int k = 0; k < NOUT; k++) gin[k] = valid ? __ldg(a.gout + i * NOUT + k) : 0.f;
        }
        if (!(ok = mma_wait())) break;
        // ---- layer 3 epilogue: out = Y + b3
        float y[NOUT];
        {
            uint32_t v[16];
            tc_ld16(tl + C_Z, v);
            tc_wait_ld();
#pragma unroll
            for (int k = 0; k < NOUT; k++) y[k] = __uint_as_float(v[k]) + b3[k];
        }
        if (MODE == MLP_FWD) {
            if (valid) {
#pragma unroll
                for (int k = 0; k < NOUT; k++) a.out[i * NOUT + k] = y[k];
            }
            tc_fence_before();
            wg_sync(wg);                                  // every row's loads done before the next tile's MMAs
            continue;
        }
        if (MODE == MLP_TRAIN) {
            // loss and dL/dout from the per-row statistics (quadratic in the seven P values)
            float p[NOUT];
#pragma unroll
            for (int k = 0; k < NOUT; k++) p[k] = (mk >> k) & 1u ? y[k] * id : 0.f;
            float li = dd;
#pragma unroll
            for (int k = 0; k < NOUT; k++) {
                float gp = 0.f;
#pragma unroll
                for (int l = 0; l < NOUT; l++) gp = fmaf(G[k < l ? spai_sym(k, l) : spai_sym(l, k)], p[l], gp);
                li = fmaf(p[k], gp - 2.f * cc[k], li);
                gin[k] = (mk >> k) & 1u ? 2.f * (gp - cc[k]) * id * (float)a.inv_npairs : 0.f;
            }
            if (valid) loss += (double)li;
        }
        if (!valid) {
#pragma unroll
            for (int k = 0; k < NOUT; k++) gin[k] = 0.f;
        }
        // ---- Gout hi and lo
        {
            unsigned int pk[4] = {bf2(gin[0], gin[1]), bf2(gin[2], gin[3]), bf2(gin[4], gin[5]), bf2(gin[6], 0.f)};
            unsigned int pl[4] = {bf2_rest(gin[0], gin[1], pk[0]), bf2_rest(gin[2], gin[3], pk[1]),
                                  bf2_rest(gin[4], gin[5], pk[2]), bf2_rest(gin[6], 0.f, pk[3])};
            put_row8(act + A_FG, t, 2, pk);
            put_row8(act + A_FG, t, 3, pl);
#pragma unroll
            for (int k = 0; k < NOUT; k++) gb3[k] += gin[k];
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma(C_Z, abase + A_FG + 32, wbase + IMG_W3T + 32, 64, 1, 0);            // dH2 = Gout W3 (values 16-31)
            mma_rows(C_G3, abase + A_H2, abase + A_FG + 32, 16, !first);       // gW3^T += H2^T Gout
            tc_commit(&mbar[wg]);
        }
        if (!(ok = mma_wait())) break;
        // ---- dZ2 = dH2 * relu'(layer 2), in place of H1's lo part
#pragma unroll
        for (int c1 = 0; c1 < NH; c1 += 32) {
          uint32_t vv[32];
          tc_ld16(tl + C_Z + c1, vv);
          tc_ld16(tl + C_Z + c1 + 16, vv + 16);
          tc_wait_ld();
#pragma unroll
          for (int c0 = c1; c0 < c1 + 32; c0 += 16) {
            const uint32_t* v = vv + (c0 - c1);
            unsigned int pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const float d0 = (m2 >> (c0 + e)) & 1ull ? __uint_as_float(v[e]) : 0.f;
                const float d1 = (m2 >> (c0 + e + 1)) & 1ull ? __uint_as_float(v[e + 1]) : 0.f;
                pk[e >> 1] = bf2(d0, d1);
            }
            put_row8(act + A_HX, t, c0 >> 3, pk);
            put_row8(act + A_HX, t, (c0 >> 3) + 1, pk + 4);
          }
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma(C_Z, abase + A_HX, wbase + IMG_W2T, 64, 4, 0);                 // dH1 = dZ2 W2
            tc_commit(&mbar[wg]);
        }
        if (!(ok = mma_wait())) break;
        // ---- dZ1 = dH1 * relu'(layer 1), in place of H2
#pragma unroll
        for (int c1 = 0; c1 < NH; c1 += 32) {
          uint32_t vv[32];
          tc_ld16(tl + C_Z + c1, vv);
          tc_ld16(tl + C_Z + c1 + 16, vv + 16);
          tc_wait_ld();
#pragma unroll
          for (int c0 = c1; c0 < c1 + 32; c0 += 16) {
            const uint32_t* v = vv + (c0 - c1);
            unsigned int pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const float d0 = (m1 >> (c0 + e)) & 1ull ? __uint_as_float(v[e]) : 0.f;
                const float d1 = (m1 >> (c0 + e + 1)) & 1ull ? __uint_as_float(v[e + 1]) : 0.f;
                pk[e >> 1] = bf2(d0, d1);
            }
            put_row8(act + A_H2, t, c0 >> 3, pk);
            put_row8(act + A_H2, t, (c0 >> 3) + 1, pk + 4);
          }
        }
        to_tensor_core();
        if (t == 0) {
            tc_fence_after();
            mma_rows(C_G2, abase + A_HX, abase + A_H1, 64, !first);
            mma_rows(C_GF, abase + A_HX, abase + A_FG, 16, !first);
            tc_commit(&mbar[wg]);
        }
        pending = true;
        first = false;
    }
    if (ok && pending) ok = mma_wait();
    if (!ok) {
        if (t == 0 && a.fault) atomicExch(a.fault, 1);
        mbar_wait(&mbar[wg], (phase - 1u) & 1u);          // bounded: let a late MMA finish before freeing
    }
    if (BACK) {
        // gradient sums to shared memory (the activations are no longer read): gW2, gb2 (lanes
        // 0-63), gW1, gb1 (lanes 64-127), gW3; then all warpgroups' together, coalesced
        float* gs = reinterpret_cast<float*>(act);
        const bool any = ok && tile0 < ntiles;
        uint32_t v[16];
        if (t < 64) {
            const int o = t;
            for (int c0 = 0; c0 < 64; c0 += 16) {
                if (any) { tc_ld16(tl + C_G2 + c0, v); tc_wait_ld(); }
#pragma unroll
                for (int e = 0; e < 16; e++) gs[grad_slot(OFF_W2 + o * NH + c0 + e)] = any ? __uint_as_float(v[e]) : 0.f;
            }
            if (any) { tc_ld16(tl + C_GF, v); tc_wait_ld(); }
            gs[grad_slot(OFF_B2 + o)] = any ? __uint_as_float(v[NIN]) : 0.f;
            if (any) { tc_ld16(tl + C_G3, v); tc_wait_ld(); }
#pragma unroll
            for (int k = 0; k < NOUT; k++) gs[grad_slot(OFF_W3 + k * NH + o)] = any ? __uint_as_float(v[k]) : 0.f;
        } else {
            const int o = t - 64;
            if (any) { tc_ld16(tl + C_GF, v); tc_wait_ld(); }
#pragma unroll
            for (int k = 0; k < NIN; k++) gs[grad_slot(OFF_W1 + o * NIN + k)] = any ? __uint_as_float(v[k]) : 0.f;
            gs[grad_slot(OFF_B1 + o)] = any ? __uint_as_float(v[NIN]) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < NOUT; k++) {
            float s = gb3[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) red_b3[warp][k] = s;
        }
        const double ls = warp_sum(loss);
        if (lane == 0) red_l[warp] = ls;
        wg_sync(wg);
        if (t < NOUT) {
            const int w0 = wg * (WG / 32);
            float s = 0.f;
            for (int w = 0; w < WG / 32; w++) s += red_b3[w0 + w][t];
            gs[grad_slot(OFF_B3 + t)] = s;
        }
        __syncthreads();
        float* gp = a.gpart + (long long)blockIdx.x * NPARAM;
        for (int i = threadIdx.x; i < NPARAM; i += MT) {
            const int q = grad_slot(i);
            float s = reinterpret_cast<const float*>(sm + S_ACT)[q];
            for (int w = 1; w < NWG; w++) s += reinterpret_cast<const float*>(sm + S_ACT + w * ACT_BYTES)[q];
            gp[i] = s;
        }
        if (MODE == MLP_TRAIN && threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < MT / 32; w++) s += red_l[w];
            a.lpart[blockIdx.x] = s * a.inv_npairs;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tbase, TM_COLS);
}

}  // namespace

int mlp_tc_grid(long long n)
{
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (n + MLP_ROWS - 1) / MLP_ROWS;
    return (int)std::max<long long>(1, std::min<long long>((tiles + MLP_PARTS - 1) / MLP_PARTS, sms));
}

cudaError_t mlp_tc_launch(int mode, int grid, cudaStream_t s, const MlpArgs& a)
{
    static bool attr[3] = {false, false, false};
    cudaError_t e = cudaSuccess;
    switch (mode) {
    case MLP_FWD:
        if (!attr[0]) { e = cudaFuncSetAttribute(k_mlp_tc<MLP_FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM); attr[0] = e == cudaSuccess; }
        if (e == cudaSuccess) k_mlp_tc<MLP_FWD><<<grid, MT, MLP_SMEM, s>>>(a);
        break;
    case MLP_BWD:
        if (!attr[1]) { e = cudaFuncSetAttribute(k_mlp_tc<MLP_BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM); attr[1] = e == cudaSuccess; }
        if (e == cudaSuccess) k_mlp_tc<MLP_BWD><<<grid, MT, MLP_SMEM, s>>>(a);
        break;
    default:
        if (!attr[2]) { e = cudaFuncSetAttribute(k_mlp_tc<MLP_TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM); attr[2] = e == cudaSuccess; }
        if (e == cudaSuccess) k_mlp_tc<MLP_TRAIN><<<grid, MT, MLP_SMEM, s>>>(a);
        break;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace cbg
