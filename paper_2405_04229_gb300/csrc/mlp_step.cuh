// One training step of the surrogate network in two kernels.
//
// step_kernel: a block takes 256 rows of the batch as two slices of 128 (256
// threads each, two per row, 32 units a thread) through forward, loss and
// backward without leaving the SM, and writes its slices' weight-gradient
// products and its partial sums; reduce_kernel adds them in a fixed order and
// applies Adam.  As 27 launches through global memory (GEMMs that re-stage
// their operands, elementwise passes between them) a step of 32,768 rows took
// 260 us; in this form 31 + 11 us.  What bounds it: latency -- 16 warps per SM
// (23 % of issue slots) evaluate 192 tanh a row twice and store the operands
// between seven MMA round trips and their barriers.  (1,024 threads, four per
// row, took the same time.)
//
// Arithmetic and its order are the unfused path's: the same BF16 hi + lo
// splits, the same K = 16 products in the same order, partial sums over the
// same rows.  Loss and gradients of 256, 512, 4,352, 32,768, 33,024 and
// 131,072 rows were equal bit for bit to those of the library from before
// this step, which took these sizes through global memory.
//
// Operand tiles: an activation tile of 128 rows x 64 units is stored once, in
// the no-swizzle core-matrix layout with the units contiguous.  As the A
// operand of the forward and input-gradient products its K are the units
// (K-major); as an operand of the weight gradients, whose K are the rows, the
// same bytes are the MN-major layout (8 x 8 core matrices of 16-byte rows,
// 2048 bytes apart along the units, 128 along the rows) -- the transpose bits
// of the instruction descriptor, no second copy.  The weights likewise serve
// W x and W^T dz from one tile.  M is 128 always: a weight gradient has 64 (or
// 8) valid accumulator lanes, the others come from whatever follows the tile
// in shared memory (within the block's allocation) and are never read.
//
// FP32 activations are not kept: the accumulators of layers 2 and 3 stay in
// tensor memory and the backward pass evaluates their tanh again.  Tensor
// memory per slice: layer 2, layer 3, output / input gradients, weight
// gradients, 64 columns each; two slices fill the SM's 512.
#pragma once

#include "mlp_tc.cuh"

namespace cs {
namespace {

constexpr int kStepRows = 256, kStepThreads = 512;
constexpr int kStepMaxB = 131072;   // above it a weight-gradient slice is longer than 128 rows

constexpr uint32_t kTransA = 1u << 15, kTransB = 1u << 16;   // MN-major operands

struct StepSlice {
    __align__(128) unsigned char z[2][kTcATile];    // H3, then dZ3 and dZ2: hi, lo (not last: see M above)
    __align__(128) unsigned char h1[2][kTcATile];   // later FP32 scratch of layer 1's dZ
    __align__(128) unsigned char h2[2][kTcATile];   // later FP32 scratch of layer 2's dZ
};
struct StepSmem {
    __align__(128) unsigned char w2[kHid * kHid * 2], w3[kHid * kHid * 2], w4[kTcN4 * kHid * 2];
    __align__(128) unsigned char dy[2][2][2048];    // per slice: dY hi, lo (128 rows x 8); later reduction scratch
    __align__(128) unsigned char zero[2048];        // K = 8 .. 15 of dY
    StepSlice s[2];
    float x[kStepRows][kNIn];
    float w1[kHid * kNIn], b1[kHid], b2[kHid], b3[kHid], b4[kNOutP];
    float loss[kStepRows / 32][4];
    unsigned long long mbar[2];
    unsigned int tmem_base;
    int abort[2];
};
static_assert(sizeof(StepSmem) <= 227 * 1024, "one block per SM");

struct StepArgs {
    const float *X, *T, *Wt;        // samples (Wt may be null: weights one)
    unsigned long long n;           // samples drawn from; 0: row i is sample i
    int B;
    uint32_t key0, key1;
    unsigned int *step, *step_red;  // step counters of this kernel and of the reduction (null: none)
    const float* p;                 // FP32 master parameters
    float *g2, *g3, *g4;            // weight-gradient products per slice
    float *bias1, *bias2, *bias3;   // bias-gradient sums per 64 rows
    float *loss, *w1;               // {loss, db4[3]} and layer-1 weight gradient per 256 rows
};

__device__ __forceinline__ void group_barrier(int g) { asm volatile("bar.sync %0, 256;" ::"r"(g + 1) : "memory"); }

// Element (unit, row) of the FP32 scratch tile: conflict-free for a warp of rows and for a warp of units.
__device__ __forceinline__ int scratch_at(int unit, int row) { return unit * 128 + (row ^ (unit & 31)); }

__global__ void __launch_bounds__(kStepThreads, 1) step_kernel(const StepArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    StepSmem& S = *reinterpret_cast<StepSmem*>(smem_raw);
    const int t = threadIdx.x, grp = t >> 8, tg = t & 255, row = tg & 127, half = tg >> 7;
    if (t < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        for (int g = 0; g < 2; ++g) {
            mbar_init(smem_u32(&S.mbar[g]), 1);
            S.abort[g] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // this row's sample
    const int i = blockIdx.x * kStepRows + grp * 128 + row;
    size_t j = (size_t)i;
    if (a.n) {
        const uint4 r = philox((uint32_t)i, *a.step + 1u, 0xB47Cu, 0u, a.key0, a.key1);   // steps count from 1
        j = (size_t)(((unsigned long long)r.x * a.n) >> 32);
        if (blockIdx.x == 0 && t == 0) *a.step_red = *a.step;
    }
    float x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = __ldg(a.X + j * 3 + k);
    if (half == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) S.x[grp * 128 + row][k] = x[k];
    }
    // weights, rounded to BF16, in the core-matrix layout: rows of eight inputs
    for (int u = t; u < (2 * kHid + kTcN4) * (kHid / 8); u += kStepThreads) {
        const int r = u >> 3, g = u & 7;
        float v[8];
        unsigned char* dst;
        const float* src = nullptr;
        if (r < kHid) {
            src = a.p + kOffW2 + r * kHid;
            dst = S.w2 + tc_off(r, 8 * g, kHid);
        } else if (r < 2 * kHid) {
            src = a.p + kOffW3 + (r - kHid) * kHid;
            dst = S.w3 + tc_off(r - kHid, 8 * g, kHid);
        } else {
            const int o = r - 2 * kHid;
            if (o < kNOutP) src = a.p + kOffW4 + o * kHid;
            dst = S.w4 + tc_off(o, 8 * g, kTcN4);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = src ? __ldg(src + 8 * g + k) : 0.0f;
        *reinterpret_cast<uint4*>(dst) = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                                                    pack_bf16x2(v[6], v[7]));
    }
    if (t < kHid * kNIn) S.w1[t] = a.p[kOffW1 + t];
    if (t < kHid) {
        S.b1[t] = a.p[kOffB1 + t];
        S.b2[t] = a.p[kOffB2 + t];
        S.b3[t] = a.p[kOffB3 + t];
    }
    if (t < kNOutP) S.b4[t] = a.p[kOffB4 + t];
    if (t < 128) reinterpret_cast<uint4*>(S.zero)[t] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    StepSlice& L = S.s[grp];
    const uint32_t tm = S.tmem_base + (uint32_t)(grp * 256);
    const uint32_t D2 = tm, D3 = tm + 64, Dx = tm + 128, Dg = tm + 192;
    const uint32_t lane = (uint32_t)(((t >> 5) & 3) * 32) << 16, col0 = (uint32_t)(32 * half);
    const uint32_t mbar = smem_u32(&S.mbar[grp]);
    uint32_t ph = 0;
    const int c0 = 32 * half;   // first unit of this thread
    const auto h1_at = [&](int u) {
        const float* w = S.w1 + u * kNIn;
        return tanh_act(fmaf(w[2], x[2], fmaf(w[1], x[1], fmaf(w[0], x[0], S.b1[u]))));
    };
    // the operand tiles are complete and earlier accumulator reads are done: one thread issues, all wait
    const auto run = [&](auto&& issue) {
        fence_async_smem();
        tc_fence_before();
        group_barrier(grp);
        if (tg == 0) {
            tc_fence_after();
            issue();
            tc_commit(mbar);
        }
        if (!mbar_wait_bounded(mbar, ph)) S.abort[grp] = 1;
        group_barrier(grp);   // every thread has seen the completion, or the give-up
        if (S.abort[grp]) return false;
        ph ^= 1u;
        tc_fence_after();
        return true;
    };
    // D = A W^T over 64 units: A hi and lo, K-major
    const auto forward = [&](uint32_t D, unsigned char (*A)[kTcATile], const unsigned char* W, int rows_w) {
        const uint32_t ah = smem_u32(A[0]), al = smem_u32(A[1]), w = smem_u32(W), lbo = (uint32_t)rows_w * 16;
#pragma unroll
        for (int s = 0; s < kHid / 16; ++s) {
            const uint64_t bd = tc_desc(w + (uint32_t)s * 2 * lbo, lbo, 128);
            tc_mma(D, tc_desc(ah + (uint32_t)s * 4096, 2048, 128), bd, tc_idesc(rows_w), s > 0);
            tc_mma(D, tc_desc(al + (uint32_t)s * 4096, 2048, 128), bd, tc_idesc(rows_w), 1);
        }
    };
    // Dx = dZ W: K the 64 output units; W as stored (its rows are K), MN-major
    const auto input_grad = [&](unsigned char (*A)[kTcATile], const unsigned char* W) {
        const uint32_t ah = smem_u32(A[0]), al = smem_u32(A[1]), w = smem_u32(W);
#pragma unroll
        for (int s = 0; s < kHid / 16; ++s) {
            const uint64_t bd = tc_desc(w + (uint32_t)s * 256, 128, 1024);
            tc_mma(Dx, tc_desc(ah + (uint32_t)s * 4096, 2048, 128), bd, tc_idesc(kHid) | kTransB, s > 0);
            tc_mma(Dx, tc_desc(al + (uint32_t)s * 4096, 2048, 128), bd, tc_idesc(kHid) | kTransB, 1);
        }
    };
    // Dg = dZ^T H over the slice's 128 rows, both MN-major: hi hi + lo hi + hi lo
    const auto weight_grad = [&](const unsigned char* Ah, const unsigned char* Al, unsigned char (*H)[kTcATile]) {
        const uint32_t ah = smem_u32(Ah), al = smem_u32(Al), bh = smem_u32(H[0]), bl = smem_u32(H[1]);
        constexpr uint32_t id = tc_idesc(kHid) | kTransA | kTransB;
#pragma unroll 1
        for (int s = 0; s < 8; ++s) {
            const uint32_t o = (uint32_t)s * 256;
            const uint64_t da = tc_desc(ah + o, 128, 2048), db = tc_desc(bh + o, 128, 2048);
            tc_mma(Dg, da, db, id, s > 0);
            tc_mma(Dg, tc_desc(al + o, 128, 2048), db, id, 1);
            tc_mma(Dg, da, tc_desc(bl + o, 128, 2048), id, 1);
        }
    };
    const auto hidden = [&](uint32_t D, const float* bias, unsigned char (*H)[kTcATile]) {   // H = tanh(D + b)
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            float v[16];
            tc_ld16(D + lane + col0 + 16 * c, v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float h[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) h[k] = tanh_act(v[8 * q + k] + bias[c0 + 16 * c + 8 * q + k]);
                tc_store8<true>(H[0], H[1], row, c0 / 8 + 2 * c + q, h);
            }
        }
    };
    // the slice's weight-gradient product, one accumulator lane per output unit
    const auto store_grad = [&](float* part, int n_out) {
        const int m = tg & 127;
        if ((m & ~31) >= n_out) return;
        float* dst = part + (size_t)(blockIdx.x * 2 + grp) * n_out * kHid + (size_t)m * kHid + c0;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            float v[16];
            tc_ld16(Dg + lane + col0 + 16 * c, v);
            if (m < n_out) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    reinterpret_cast<float4*>(dst)[4 * c + q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        }
    };
    // column sums of the FP32 scratch per 64 rows (four phases of every fourth row)
    const auto bias_sums = [&](const float* z, float* out) {
        float* red = reinterpret_cast<float*>(S.dy[grp]);   // [2][4][64]
        const int u = tg & 63, q = tg >> 6;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            float s = 0.0f;
#pragma unroll
            for (int k = 0; k < 16; ++k) s += z[scratch_at(u, 64 * b + q + 4 * k)];
            red[(b * 4 + q) * 64 + u] = s;
        }
        group_barrier(grp);
        if (tg < 128) {
            const float* r = red + (tg >> 6) * 256 + (tg & 63);
            out[(size_t)((blockIdx.x * 2 + grp) * 2 + (tg >> 6)) * 64 + (tg & 63)] = (r[0] + r[64]) + (r[128] + r[192]);
        }
    };
    const auto pass = [&]() {
        // ---- forward
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            float h[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) h[k] = h1_at(c0 + 8 * g + k);
            tc_store8<true>(L.h1[0], L.h1[1], row, c0 / 8 + g, h);
        }
        if (!run([&]() { forward(D2, L.h1, S.w2, kHid); })) return;
        hidden(D2, S.b2, L.h2);
        if (!run([&]() { forward(D3, L.h2, S.w3, kHid); })) return;
        hidden(D3, S.b3, L.z);
        if (!run([&]() { forward(Dx, L.z, S.w4, kTcN4); })) return;
        // ---- loss: dY = 2 w (Y - T) / B, and the warp's sums
        if (half == 0) {
            float y[4], v4[4] = {0.0f, 0.0f, 0.0f, 0.0f}, d[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            tc_ld4(Dx + lane, y);
#pragma unroll
            for (int o = 0; o < kNOut; ++o) {
                const float e = (y[o] + S.b4[o]) - __ldg(a.T + j * kNOut + o);
                const float wt = a.Wt ? __ldg(a.Wt + j * kNOut + o) : 1.0f;
                v4[0] += wt * e * e / a.B;
                d[o] = 2.0f * wt * e / a.B;
                v4[1 + o] = d[o];
            }
            tc_store8<true>(S.dy[grp][0], S.dy[grp][1], row, 0, d);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < 4; ++c) v4[c] += __shfl_xor_sync(0xffffffffu, v4[c], o);
            if ((t & 31) == 0)
#pragma unroll
                for (int c = 0; c < 4; ++c) S.loss[grp * 4 + (row >> 5)][c] = v4[c];
        }
        // ---- layer 4: dW4 = dY^T H3, dH3 = dY W4 (K = 8 outputs and 8 zeros)
        if (!run([&]() {
                weight_grad(S.dy[grp][0], S.dy[grp][1], L.z);
                const uint32_t yh = smem_u32(S.dy[grp][0]), yl = smem_u32(S.dy[grp][1]), z = smem_u32(S.zero);
                const uint64_t bd = tc_desc(smem_u32(S.w4), 128, 256);
                tc_mma(Dx, tc_desc(yh, z - yh, 128), bd, tc_idesc(kHid) | kTransB, 0);
                tc_mma(Dx, tc_desc(yl, z - yl, 128), bd, tc_idesc(kHid) | kTransB, 1);
            }))
            return;
        store_grad(a.g4, kNOutP);
        // ---- layers 3, 2: dZ = dH (1 - H^2); FP32 copy for the bias sums, then the operand tile
        float z[32];
#pragma unroll 1
        for (int l = 3; l >= 2; --l) {
            const uint32_t D = l == 3 ? D3 : D2;
            const float* bias = l == 3 ? S.b3 : S.b2;
            float* scratch = reinterpret_cast<float*>(l == 3 ? L.z[0] : L.h2[0]);   // H3 and H2 are used up
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float v[16], d[16];
                tc_ld16(D + lane + col0 + 16 * c, v);
                tc_ld16(Dx + lane + col0 + 16 * c, d);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const float h = tanh_act(v[k] + bias[c0 + 16 * c + k]);
                    z[16 * c + k] = d[k] * fmaf(-h, h, 1.0f);
                    scratch[scratch_at(c0 + 16 * c + k, row)] = z[16 * c + k];
                }
            }
            group_barrier(grp);
            bias_sums(scratch, l == 3 ? a.bias3 : a.bias2);   // (its barrier: the tile below may overwrite the scratch)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float h[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) h[k] = z[8 * g + k];
                tc_store8<true>(L.z[0], L.z[1], row, c0 / 8 + g, h);
            }
            if (!run([&]() {
                    weight_grad(L.z[0], L.z[1], l == 3 ? L.h2 : L.h1);
                    input_grad(L.z, l == 3 ? S.w3 : S.w2);
                }))
                return;
            store_grad(l == 3 ? a.g3 : a.g2, kHid);
        }
        // ---- layer 1: dZ1 into the scratch, bias sums
        float* scratch = reinterpret_cast<float*>(L.h1[0]);
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            float d[16];
            tc_ld16(Dx + lane + col0 + 16 * c, d);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float h = h1_at(c0 + 16 * c + k);
                scratch[scratch_at(c0 + 16 * c + k, row)] = d[k] * fmaf(-h, h, 1.0f);
            }
        }
        group_barrier(grp);
        bias_sums(scratch, a.bias1);
    };
    pass();
    tc_fence_before();
    __syncthreads();
    if (!S.abort[0] && !S.abort[1]) {
        // layer-1 weight gradient of the 256 rows (four phases of every fourth row), loss and db4
        float* red = reinterpret_cast<float*>(S.dy);   // [4][192]
        if (t < 256) {
            const int u = t & 63, q = t >> 6;
            float acc[kNIn] = {0.0f, 0.0f, 0.0f};
#pragma unroll 4
            for (int r = q; r < kStepRows; r += 4) {
                const float z = reinterpret_cast<const float*>(S.s[r >> 7].h1[0])[scratch_at(u, r & 127)];
#pragma unroll
                for (int c = 0; c < kNIn; ++c) acc[c] = fmaf(z, S.x[r][c], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < kNIn; ++c) red[q * (kHid * kNIn) + u * kNIn + c] = acc[c];
        } else if (t < 260) {
            const int c = t - 256;
            float s = 0.0f;
            for (int w = 0; w < kStepRows / 32; ++w) s += S.loss[w][c];
            a.loss[blockIdx.x * 4 + c] = s;
        }
        __syncthreads();
        if (t < kHid * kNIn)
            a.w1[(size_t)blockIdx.x * (kHid * kNIn) + t] = (red[t] + red[192 + t]) + (red[384 + t] + red[576 + t]);
    } else {
        if (tg == 0 && S.abort[grp]) {   // let the MMAs in flight finish (bounded)
            mbar_wait_bounded(mbar, ph);
            atomicOr(&g_tc_timeout, 1u);
        }
        __syncthreads();
    }
    if (t < 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(S.tmem_base), "r"(512) : "memory");
    }
}

// Adam (bias-corrected) on one FP32 master parameter.
__device__ __forceinline__ void adam_update(int i, float gi, float* __restrict__ p, float* __restrict__ m,
                                            float* __restrict__ v, float4 sc) {
    const float lr = sc.x, c1 = sc.y, c2 = sc.z;
    if ((i >= kOffW4 + kNOut * kHid && i < kOffB4) || i >= kOffB4 + kNOut) return;   // padding
    const float mi = 0.9f * m[i] + 0.1f * gi, vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

struct ReduceArgs {
    const float *g2, *g3, *g4, *bias1, *bias2, *bias3, *loss, *w1;
    int B;
    float *p, *m, *v;               // Adam's state, or p null: gradients only
    const float4* sched;            // {lr, 1 - 0.9^step, 1 - 0.999^step} per step
    unsigned int *step, *step_red;
    float *g, *loss_out;            // gradients (may be null when p is given), loss
};

// Sums in the unfused path's order: a weight element over the slices one after the other, a column
// of the other partial sums by 128 threads and a pairwise tree; one block per 32 weight elements,
// then one per column.  The 9 MB of slices of a 32,768-row batch come from L2 through shared memory,
// 256 slices at a time by all threads, so that the loads and not the serial sum set the pace
// (one thread per element loading its own slices took 24 us, this form 11 us with the slices in L2).
constexpr int kRedThreads = 128, kRedW = 2 * kHid * kHid + kNOutP * kHid, kRedWPer = 32;
constexpr int kRedCols = 3 * kHid + kHid * kNIn + 1 + kNOut;
constexpr int kRedBlocks = kRedW / kRedWPer + kRedCols;
__global__ void __launch_bounds__(kRedThreads) reduce_kernel(const ReduceArgs a) {
    __shared__ float red[kRedThreads];
    __shared__ float tile[256][kRedWPer];
    const int t = threadIdx.x, slices = a.B / 128;
    float4 sc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (a.p) {
        const unsigned int step = *a.step_red;
        sc = a.sched[step];
        if (blockIdx.x == 0 && t == 0) *a.step = step + 1u;
    }
    int i;
    float s = 0.0f;
    if ((int)blockIdx.x < kRedW / kRedWPer) {
        const int e = blockIdx.x * kRedWPer + (t & 31);
        const float* part;
        int width;
        if (e < kHid * kHid) {
            part = a.g2 + e;
            width = kHid * kHid;
            i = kOffW2 + e;
        } else if (e < 2 * kHid * kHid) {
            part = a.g3 + (e - kHid * kHid);
            width = kHid * kHid;
            i = kOffW3 + (e - kHid * kHid);
        } else {
            part = a.g4 + (e - 2 * kHid * kHid);
            width = kNOutP * kHid;
            i = kOffW4 + (e - 2 * kHid * kHid);
        }
        for (int z0 = 0; z0 < slices; z0 += 256) {
            const int n = min(256, slices - z0);
            if (z0) __syncthreads();
#pragma unroll 16
            for (int z = t >> 5; z < n; z += kRedThreads / 32) tile[z][t & 31] = __ldcg(part + (size_t)(z0 + z) * width);
            __syncthreads();
            if (t < 32) {
#pragma unroll 16
                for (int z = 0; z < n; ++z) s += tile[z][t];
            }
        }
        if (t >= 32) return;
    } else {
        int c = blockIdx.x - kRedW / kRedWPer, rows, stride;
        const float* part;
        if (c < 3 * kHid) {
            const int l = c / kHid, u = c % kHid;
            part = (l == 0 ? a.bias1 : l == 1 ? a.bias2 : a.bias3) + u;
            i = (l == 0 ? kOffB1 : l == 1 ? kOffB2 : kOffB3) + u;
            rows = a.B / 64;
            stride = kHid;
        } else if (c < 3 * kHid + kHid * kNIn) {
            c -= 3 * kHid;
            part = a.w1 + c;
            i = kOffW1 + c;
            rows = a.B / kStepRows;
            stride = kHid * kNIn;
        } else {
            c -= 3 * kHid + kHid * kNIn;
            part = a.loss + c;
            i = c ? kOffB4 + c - 1 : -1;
            rows = a.B / kStepRows;
            stride = 4;
        }
        for (int r = t; r < rows; r += kRedThreads) s += __ldcg(part + (size_t)r * stride);
        red[t] = s;
        __syncthreads();
#pragma unroll
        for (int h = kRedThreads / 2; h > 0; h >>= 1) {
            if (t < h) red[t] += red[t + h];
            __syncthreads();
        }
        if (t) return;
        s = red[0];
        if (i < 0) {
            *a.loss_out = s;
            return;
        }
    }
    if (a.g) a.g[i] = s;
    if (a.p) adam_update(i, s, a.p, a.m, a.v, sc);
}

// Batches that the fused step takes: whole blocks, and weight-gradient slices of 128 rows.
bool step_fused(int B) { return B % kStepRows == 0 && B <= kStepMaxB; }

size_t step_part_floats(int B) {
    return (size_t)(B / 128) * kRedW + (size_t)(B / 64) * 3 * kHid + (size_t)(B / kStepRows) * (4 + kHid * kNIn);
}

// Lays the partial sums out in `part` (step_part_floats(B)) for both kernels.
void step_layout(float* part, int B, StepArgs& s, ReduceArgs& r) {
    const size_t slices = (size_t)B / 128;
    s.g2 = part;
    s.g3 = s.g2 + slices * kHid * kHid;
    s.g4 = s.g3 + slices * kHid * kHid;
    s.bias1 = s.g4 + slices * kNOutP * kHid;
    s.bias2 = s.bias1 + (size_t)(B / 64) * kHid;
    s.bias3 = s.bias2 + (size_t)(B / 64) * kHid;
    s.loss = s.bias3 + (size_t)(B / 64) * kHid;
    s.w1 = s.loss + (size_t)(B / kStepRows) * 4;
    s.B = r.B = B;
    r.g2 = s.g2; r.g3 = s.g3; r.g4 = s.g4;
    r.bias1 = s.bias1; r.bias2 = s.bias2; r.bias3 = s.bias3;
    r.loss = s.loss; r.w1 = s.w1;
}

cudaError_t step_attributes() {   // on the current device, outside stream capture
    return cudaFuncSetAttribute(step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StepSmem));
}

void step_launch(const StepArgs& s, const ReduceArgs& r, cudaStream_t stream) {
    step_kernel<<<s.B / kStepRows, kStepThreads, sizeof(StepSmem), stream>>>(s);
    reduce_kernel<<<kRedBlocks, kRedThreads, 0, stream>>>(r);
}

}  // namespace
}  // namespace cs
