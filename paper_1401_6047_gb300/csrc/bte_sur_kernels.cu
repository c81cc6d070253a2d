/*
 * bte_sur_kernels.cu -- CUDA kernels of the MLP surrogate (sm_103a).
 *
 * The two 256 x 256 hidden layers and their backward products run on the
 * fifth-generation BF16 tensor cores (tcgen05.mma, FP32 accumulators in
 * tensor memory) in two GEMM kernels: one for the products along the hidden
 * units (forward, and back through a layer), whose epilogue fuses the bias,
 * the SiLU activation and its derivative, and one for the weight gradients
 * (along the batch) beside the reductions over it.  The thin layers (5 inputs, 2 outputs) are FP32 FMA
 * kernels; batch reductions are two-pass and deterministic; Adam keeps FP32
 * master weights and refreshes the BF16 operand copies in the same pass.
 *
 * A training step of 8 members on 1024 points each moves about 90 MB through
 * L2 and 6.5 GFLOP through the tensor cores, 10 to 15 us of work; it is bound
 * by the latency of its kernels, each a few microseconds long and waiting on
 * the one before, so each is cut to fill the SMs once and to have its loads
 * in flight together.
 */
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "bte_device.cuh"
#include "bte_sur_internal.h"
#include "bte_tc.cuh"

namespace bte {
namespace sur {
namespace {

/* GEMMs of 128 x 128 outputs per CTA (MMAs of M = N = 128 per 16 of K), K in
 * stages of 64, four of them in shared memory: along the hidden units (K =
 * 256) all of both operands, every load in flight at once.  What bounds them
 * is that fill: asynchronous copies bring about 19 bytes per clock to an SM
 * (128 KB: 7000 cycles, the same in several orders of the copies), the MMAs
 * take 2500 and the epilogue 8000.  Core matrices (8 x 8, 128 bytes) sit 144
 * bytes apart, so that eight threads that fill the same row of eight of them
 * meet no bank twice and a warp reads whole 128-byte lines. */
constexpr int GM = 128, GN = 128, GK = 64, kGStages = 4;
constexpr int kGThreads = 256; /* 8 warps: two per tensor-memory lane quadrant */
constexpr uint32_t kGCore = 144;
constexpr uint32_t kGGroup = (GK / 8) * kGCore;        /* K-major: next 8-row group */
constexpr uint32_t kGTileBytes = (GM / 8) * kGGroup;   /* 18 KB per operand and stage */
constexpr uint32_t kGGroupMN = (GM / 8) * kGCore;      /* MN-major: next 8 k */
constexpr size_t kGSmem = 2 * kGStages * (size_t)kGTileBytes + 64 + 1024; /* A, B, barriers, align */

__device__ __forceinline__ float sigmoid_f(float z) { return tc::sigmoid_fast(z); }
__device__ __forceinline__ float silu_f(float z) { return z * sigmoid_f(z); }
__device__ __forceinline__ float silu_grad_f(float z) {
    const float s = sigmoid_f(z);
    return s * (1.0f + z * (1.0f - s));
}

/* The 128 rows of a K-major operand ([row][k], leading dimension ld), all
 * 256 k, into its four stage tiles by asynchronous copies: a warp takes a row
 * at a time, lane l its l-th chunk of 8 k. */
__device__ __forceinline__ void load_rows(unsigned char* s, const __nv_bfloat16* g, long long ld, int row0) {
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    const uint32_t d = dev::smem_u32(s) + (l >> 3) * kGTileBytes + (l & 7) * kGCore;
#pragma unroll
    for (int q = 0; q < GM / 8; ++q) {
        const int r = q * 8 + warp;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + (r >> 3) * kGGroup + (r & 7) * 16),
                     "l"(g + (long long)(row0 + r) * ld + l * 8)
                     : "memory");
    }
}
__device__ __forceinline__ void commit_stage() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void wait_stage() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

/* One stage (64 k x 128 rows) of an MN-major operand ([k][row]): eight rows
 * of one k are 16 contiguous bytes in the source and in a core matrix, which
 * holds 8 k of 8 rows; a warp takes two k at a time. */
__device__ __forceinline__ void load_stage_mn(unsigned char* s, const __nv_bfloat16* g, long long ld,
                                              int row0, int k0) {
    const uint32_t d = dev::smem_u32(s);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = threadIdx.x + q * kGThreads;
        const int rb = c & 15, k = c >> 4; /* 16 row blocks x 64 k */
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + (k >> 3) * kGGroupMN + rb * kGCore +
                                                                        (k & 7) * 16),
                     "l"(g + (long long)(k0 + k) * ld + row0 + rb * 8)
                     : "memory");
    }
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <int COLS>
__device__ __forceinline__ uint32_t tmem_begin(uint32_t* slot, int warp) {
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         dev::smem_u32(slot)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    return *slot;
}
template <int COLS>
__device__ __forceinline__ void tmem_end(uint32_t tmem, int warp) {
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS)
                     : "memory");
}

/* The four K = 16 MMAs of one stage.  The descriptor's two offsets: K-major,
 * the next core matrix along k and along the rows; MN-major, the next along k
 * and along the rows as well. */
template <bool MN>
__device__ __forceinline__ void stage_mma(uint32_t tmem, uint32_t aA, uint32_t aB, bool first) {
    constexpr uint32_t idesc = tc::instr_desc(GM, GN) | (MN ? 3u << 15 : 0u); /* both operands MN-major */
    constexpr uint32_t along_k = MN ? kGGroupMN : kGCore, along_rows = MN ? kGCore : kGGroup;
#pragma unroll
    for (int ks = 0; ks < GK / 16; ++ks) {
        const uint64_t ad = tc::smem_desc(aA + ks * 2 * along_k, along_k, along_rows);
        const uint64_t bd = tc::smem_desc(aB + ks * 2 * along_k, along_k, along_rows);
        tc::tc_mma(tmem, ad, bd, idesc, (!first || ks > 0) ? 1u : 0u);
    }
}

/* C = A B^T along the hidden units (see GemmArgs), both operands K-major.
 * One CTA per 128 x 128 output tile of one member (blockIdx.z).  Once both
 * operands have landed, one thread issues the MMAs into 128 columns of tensor
 * memory.  The epilogue reads the accumulators back with tcgen05.ld (warp
 * w: lanes 32 (w mod 4) .., columns 64 (w / 4) ..).  The wait is bounded; if
 * it gives up the error word is set, and the CTA still frees its tensor
 * memory before it exits.  Measured (8 members, 1024 rows, GB300): 19 us
 * with two stages filled through registers, 12 us so. */
template <int EPI>
__global__ void __launch_bounds__(kGThreads) gemm_tc_kernel(GemmArgs a) {
    extern __shared__ unsigned char gsm_raw[];
    unsigned char* gsm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~(uintptr_t)1023);
    /* the stages of A, those of B, the barrier */
    uint64_t* bars = reinterpret_cast<uint64_t*>(gsm + 2 * kGStages * kGTileBytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);
    const uint32_t bar = dev::smem_u32(bars);

    const int mem = blockIdx.z;
    const __nv_bfloat16* A = a.A + mem * a.sA;
    const __nv_bfloat16* B = a.B + mem * a.sB;
    const int m0 = blockIdx.y * GM, n0 = blockIdx.x * GN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) {
        dev::mbar_init(bar, 1);
        dev::fence_proxy_async_smem();
    }
    const uint32_t tmem = tmem_begin<GN>(tmem_slot, warp);
    pdl_wait();
    pdl_trigger();
    load_rows(gsm, A, a.lda, m0);
    load_rows(gsm + kGStages * kGTileBytes, B, a.ldb, n0);
    commit_stage();
    wait_stage<0>();
    /* generic-proxy writes -> visible to the tensor cores */
    dev::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
        tc::tc_fence_after();
#pragma unroll
        for (int st = 0; st < kGStages; ++st)
            stage_mma<false>(tmem, dev::smem_u32(gsm + st * kGTileBytes),
                             dev::smem_u32(gsm + (kGStages + st) * kGTileBytes), st == 0);
        tc::tc_commit(bar);
    }
    const bool ok = dev::mbar_wait(bar, 0u);
    tc::tc_fence_after();

    if (ok) {
        const int sub = warp & 3, half = warp >> 2;
        const int row = m0 + sub * 32 + lane;
#pragma unroll 1
        for (int cb = 0; cb < GN / 2; cb += 32) {
            const int cl = half * (GN / 2) + cb; /* column within the tile */
            float v[32];
            tc::tc_ld32(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)cl, v);
            const int col = n0 + cl;
            const long long o = mem * a.sZ + (long long)row * a.ldz + col;
            if (EPI == EPI_FWD) {
                const float* bias = a.bias + mem * a.sBias + col;
#pragma unroll
                for (int c8 = 0; c8 < 32; c8 += 8) {
                    float z[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) z[e] = v[c8 + e] + bias[c8 + e];
                    if (a.Z) {
                        *reinterpret_cast<float4*>(a.Z + o + c8) = make_float4(z[0], z[1], z[2], z[3]);
                        *reinterpret_cast<float4*>(a.Z + o + c8 + 4) = make_float4(z[4], z[5], z[6], z[7]);
                    }
                    __nv_bfloat162 pk[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        pk[e] = __floats2bfloat162_rn(silu_f(z[2 * e]), silu_f(z[2 * e + 1]));
                    *reinterpret_cast<uint4*>(a.Hout + o + c8) = *reinterpret_cast<const uint4*>(pk);
                }
            } else {
#pragma unroll
                for (int c8 = 0; c8 < 32; c8 += 8) {
                    const float4 z0 = *reinterpret_cast<const float4*>(a.Zin + o + c8);
                    const float4 z1 = *reinterpret_cast<const float4*>(a.Zin + o + c8 + 4);
                    const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
                    __nv_bfloat162 pk[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        pk[e] = __floats2bfloat162_rn(v[c8 + 2 * e] * silu_grad_f(z[2 * e]),
                                                      v[c8 + 2 * e + 1] * silu_grad_f(z[2 * e + 1]));
                    *reinterpret_cast<uint4*>(a.Dout + o + c8) = *reinterpret_cast<const uint4*>(pk);
                }
            }
        }
    }
    if (!ok && tid == 0 && a.err) atomicExch(a.err, 1);
    tmem_end<GN>(tmem, warp);
}

/* Weight gradients dW = dZ^T H of both hidden layers (see WgradArgs): 128 x
 * 128 outputs per CTA, K the batch.  Both
 * operands are stored [sample][unit], so they go to shared memory as they
 * are and the tensor cores take them MN-major; stages of 64 samples, three
 * in flight while one is multiplied.  The tile is square because the loads
 * bound it (34 MB through L2 for 8 members x 1024, 25 us; 128 x 32 tiles,
 * which fill more SMs, move 84 MB: 29 us), and K stays whole to keep the
 * order of the sum.  Every wait is bounded, as above. */
__device__ __forceinline__ void weight_gradients(const WgradArgs& a, int tile) {
    extern __shared__ unsigned char gsm_raw[];
    unsigned char* gsm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gsm + 2 * kGStages * kGTileBytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kGStages);
    const uint32_t bar0 = dev::smem_u32(bars);

    const int across = a.H0 / GN, per = across * (a.H0 / GM); /* tiles of one layer of one member */
    const int layer = tile / per & 1, mem = tile / per >> 1;
    const __nv_bfloat16* A = (layer ? a.dZ[1] : a.dZ[0]) + mem * a.sAct;
    const __nv_bfloat16* B = (layer ? a.H[1] : a.H[0]) + mem * a.sAct;
    const int m0 = tile % per / across * GM, n0 = tile % across * GN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int st = 0; st < kGStages; ++st) dev::mbar_init(bar0 + 8 * st, 1);
        dev::fence_proxy_async_smem();
    }
    const uint32_t tmem = tmem_begin<GN>(tmem_slot, warp);
    pdl_wait();
    pdl_trigger();

    const int nk = a.K / GK;
    auto load = [&](int kt) { /* one group per stage, empty past the end */
        if (kt < nk) {
            load_stage_mn(gsm + (kt % kGStages) * kGTileBytes, A, a.ld, m0, kt * GK);
            load_stage_mn(gsm + (kGStages + kt % kGStages) * kGTileBytes, B, a.ld, n0, kt * GK);
        }
        commit_stage();
    };
    bool ok = true;
    for (int kt = 0; kt < kGStages - 1; ++kt) load(kt);
    for (int kt = 0; kt < nk; ++kt) {
        const int st = kt % kGStages;
        wait_stage<kGStages - 2>();
        /* generic-proxy writes -> visible to the tensor cores */
        dev::fence_proxy_async_smem();
        if (__syncthreads_or(!ok)) break;
        if (tid == 0) {
            tc::tc_fence_after();
            stage_mma<true>(tmem, dev::smem_u32(gsm + st * kGTileBytes),
                            dev::smem_u32(gsm + (kGStages + st) * kGTileBytes), kt == 0);
            tc::tc_commit(bar0 + 8 * st);
        }
        /* the stage before this one is free once its MMAs are complete */
        if (kt >= 1 && !dev::mbar_wait(bar0 + 8 * ((kt - 1) % kGStages), (uint32_t)(((kt - 1) / kGStages) & 1)))
            ok = false;
        if (ok) load(kt + kGStages - 1);
        else commit_stage();
    }
    /* the last commit covers every MMA issued before it */
    if (ok && !dev::mbar_wait(bar0 + 8 * ((nk - 1) % kGStages), (uint32_t)(((nk - 1) / kGStages) & 1))) ok = false;
    wait_stage<0>();
    tc::tc_fence_after();
    if (ok) {
        const int sub = warp & 3, half = warp >> 2;
        float* o = a.grad + mem * a.pstride + (layer ? a.oW[1] : a.oW[0]) + (long long)(m0 + sub * 32 + lane) * a.ld + n0;
#pragma unroll 1
        for (int cb = 0; cb < GN / 2; cb += 32) {
            const int cl = half * (GN / 2) + cb;
            float v[32];
            tc::tc_ld32(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)cl, v);
#pragma unroll
            for (int c4 = 0; c4 < 32; c4 += 4)
                *reinterpret_cast<float4*>(o + cl + c4) = make_float4(v[c4], v[c4 + 1], v[c4 + 2], v[c4 + 3]);
        }
    }
    if (!ok && tid == 0 && a.err) atomicExch(a.err, 1);
    tmem_end<GN>(tmem, warp);
}

__device__ __forceinline__ void load_xh(const float* x, const int* idx, long long row0, int r,
                                        int nvalid, const Scale& sc, float (&xh)[kIn]) {
    if (r < nvalid) {
        const long long s = idx ? (long long)idx[r] : row0 + r;
#pragma unroll
        for (int i = 0; i < kIn; ++i) xh[i] = 2.0f * (x[s * kIn + i] - sc.x_lo[i]) * sc.x_inv[i] - 1.0f;
    } else {
#pragma unroll
        for (int i = 0; i < kIn; ++i) xh[i] = 0.0f;
    }
}

/* 16 rows of one member per CTA: thread o holds hidden unit o's weights,
 * the rows' inputs sit in shared memory (8 members x 1024 rows: 14 us with
 * one output per thread, 5 us so) */
constexpr int kL1Rows = 16;
__global__ void l1_kernel(L1Args a) {
    const int mem = blockIdx.y, r0 = blockIdx.x * kL1Rows, o = threadIdx.x;
    __shared__ float sxh[kL1Rows][kIn];
    pdl_wait();
    pdl_trigger();
    const int* idx = a.idx ? a.idx + (long long)mem * a.Bp : nullptr;
    if (o < kL1Rows) {
        float xh[kIn];
        load_xh(a.x, idx, a.row0, r0 + o, a.nvalid, a.sc, xh);
#pragma unroll
        for (int i = 0; i < kIn; ++i) sxh[o][i] = xh[i];
    }
    const float* P = a.params + mem * a.pstride;
    const float b = P[a.ob1 + o];
    float w[kIn];
#pragma unroll
    for (int i = 0; i < kIn; ++i) w[i] = P[a.oW1 + (long long)o * kIn + i];
    __syncthreads();
    const long long out = ((long long)mem * a.Bp + r0) * a.H + o;
#pragma unroll
    for (int r = 0; r < kL1Rows; ++r) {
        float z = b;
#pragma unroll
        for (int i = 0; i < kIn; ++i) z = fmaf(w[i], sxh[r][i], z);
        if (a.Z1) a.Z1[out + (long long)r * a.H] = z;
        a.H1[out + (long long)r * a.H] = __float2bfloat16_rn(silu_f(z));
    }
}

/* 8 consecutive floats at a 16-byte aligned address */
__device__ __forceinline__ void ld8(const float* p, float (&x)[8]) {
    const float4 u = reinterpret_cast<const float4*>(p)[0], v = reinterpret_cast<const float4*>(p)[1];
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
    x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
}

/* one warp per sample; lane l covers hidden units 8l .. 8l+7 (H = 256); the
 * loss of the CTA's 8 samples is formed by eight lanes of one warp (FP64
 * instructions cost a warp the same however few lanes they serve) and added
 * with one atomic */
__global__ void head_kernel(HeadArgs a) {
    const int mem = blockIdx.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * (blockDim.x >> 5) + warp; /* < Bp: a multiple of 128 */
    __shared__ float s_e[8][2];
    pdl_wait();
    pdl_trigger();
    const float* P = a.params + mem * a.pstride;
    const long long base = ((long long)mem * a.Bp + r) * a.H;
    float y0 = 0.0f, y1 = 0.0f;
    const int c0 = lane * 8;
    float hv[8], w0[8], w1[8];
    ld8(P + a.oW4 + c0, w0);
    ld8(P + a.oW4 + a.H + c0, w1);
    const uint4 raw = *reinterpret_cast<const uint4*>(a.H3 + base + c0);
    const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(hp[i]);
        hv[2 * i] = f.x;
        hv[2 * i + 1] = f.y;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        y0 = fmaf(w0[i], hv[i], y0);
        y1 = fmaf(w1[i], hv[i], y1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        y0 += __shfl_xor_sync(0xffffffffu, y0, o);
        y1 += __shfl_xor_sync(0xffffffffu, y1, o);
    }
    y0 += P[a.ob4];
    y1 += P[a.ob4 + 1];
    const long long yo = ((long long)mem * a.Bp + r) * kOut;
    if (lane == 0 && a.Yh) {
        a.Yh[yo] = y0;
        a.Yh[yo + 1] = y1;
    }
    if (!a.y) return;
    /* training: loss gradient and the output layer's backward product */
    float d0 = 0.0f, d1 = 0.0f;
    float e0 = 0.0f, e1 = 0.0f;
    if (r < a.nvalid) {
        const int* idx = a.idx ? a.idx + (long long)mem * a.Bp : nullptr;
        const long long s = idx ? (long long)idx[r] : a.row0 + r;
        const float t0 = (a.y[s * kOut] - a.sc.y_mean[0]) / a.sc.y_std[0];
        const float t1 = (a.y[s * kOut + 1] - a.sc.y_mean[1]) / a.sc.y_std[1];
        e0 = y0 - t0;
        e1 = y1 - t1;
        d0 = e0 * a.inv_n;
        d1 = e1 * a.inv_n;
    }
    if (lane == 0) {
        s_e[warp][0] = e0;
        s_e[warp][1] = e1;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double l = 0.0;
        if (lane < 8) l = 0.5 * ((double)s_e[lane][0] * s_e[lane][0] + (double)s_e[lane][1] * s_e[lane][1]) * a.inv_n;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
        if (lane == 0) atomicAdd(a.loss + mem, l);
    }
    if (lane == 0) {
        a.DY[yo] = d0;
        a.DY[yo + 1] = d1;
    }
    float z[8];
    ld8(a.Z3 + base + c0, z);
    __nv_bfloat162 outv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float dh = fmaf(d0, w0[2 * i + u], d1 * w1[2 * i + u]);
            v[u] = dh * silu_grad_f(z[2 * i + u]);
        }
        outv[i] = __floats2bfloat162_rn(v[0], v[1]);
    }
    *reinterpret_cast<uint4*>(a.DZ3 + base + c0) = *reinterpret_cast<const uint4*>(outv);
}

/* values per 128-sample block: b1, W1 (5 per unit), b2, b3, W4 (2 per unit), b4 */
__host__ __device__ inline int red_count(int H) { return H * (1 + kIn + 1 + 1 + kOut) + kOut; }

/* Partial sums over 128 samples of one member; `part` 0: b1 and W1 (from DZ1
 * and the inputs), 1: b2, 2: b3, 3: W4 and b4 (from H3 and DY).  One hidden
 * unit per thread, the samples added in order, 32 loads in flight (one CTA per
 * 128 samples that did all four arrays: 107 us for 8 members x 1024, one load
 * of each array in flight; so: 10 us). */
constexpr int kRedFly = 32;
template <class F>
__device__ __forceinline__ void over_samples(const __nv_bfloat16* p, int H, F f) {
    for (int r0 = 0; r0 < 128; r0 += kRedFly) {
        __nv_bfloat16 v[kRedFly];
#pragma unroll
        for (int q = 0; q < kRedFly; ++q) v[q] = p[(long long)(r0 + q) * H];
#pragma unroll
        for (int q = 0; q < kRedFly; ++q) f(r0 + q, __bfloat162float(v[q]));
    }
}
__device__ __forceinline__ void reduce_partial(const RedArgs& a, int chunk, int mem, int part) {
    const int r0 = chunk * 128, o = threadIdx.x;
    __shared__ float sx[128][kIn];
    const int H = a.H, nred = red_count(H);
    float* out = a.partial + ((long long)mem * (a.Bp / 128) + chunk) * nred;
    const long long e = ((long long)mem * a.Bp + r0) * H + o;
    pdl_wait();
    pdl_trigger();
    if (part == 0) {
        const int* idx = a.idx ? a.idx + (long long)mem * a.Bp : nullptr;
        for (int r = threadIdx.x; r < 128; r += blockDim.x) {
            float xh[kIn];
            load_xh(a.x, idx, a.row0, r0 + r, a.nvalid, a.sc, xh);
#pragma unroll
            for (int i = 0; i < kIn; ++i) sx[r][i] = xh[i];
        }
        __syncthreads();
        float gb = 0, gw[kIn] = {0, 0, 0, 0, 0};
        over_samples(a.DZ1 + e, H, [&](int r, float d) {
            gb += d;
#pragma unroll
            for (int i = 0; i < kIn; ++i) gw[i] = fmaf(d, sx[r][i], gw[i]);
        });
        out[o] = gb;
#pragma unroll
        for (int i = 0; i < kIn; ++i) out[H + o * kIn + i] = gw[i];
    } else if (part < 3) {
        float gb = 0;
        over_samples((part == 1 ? a.DZ2 : a.DZ3) + e, H, [&](int, float d) { gb += d; });
        out[H * (kIn + part) + o] = gb;
    } else {
        for (int r = threadIdx.x; r < 128; r += blockDim.x) {
            const long long yo = ((long long)mem * a.Bp + r0 + r) * kOut;
            sx[r][0] = a.DY[yo];
            sx[r][1] = a.DY[yo + 1];
        }
        __syncthreads();
        float gw[kOut] = {0, 0};
        over_samples(a.H3 + e, H, [&](int r, float h3) {
            gw[0] = fmaf(sx[r][0], h3, gw[0]);
            gw[1] = fmaf(sx[r][1], h3, gw[1]);
        });
        out[H * (3 + kIn) + o] = gw[0];
        out[H * (4 + kIn) + o] = gw[1];
        if (o < kOut) {
            float s = 0;
            for (int r = 0; r < 128; ++r) s += sx[r][o];
            out[H * (3 + kIn + kOut) + o] = s;
        }
    }
}

/* The gradients of a step in one launch: CTAs of weight-gradient tiles first,
 * then those of the reductions (member, 128 samples, part), which run on the
 * SMs that the tiles leave and are over before them.  Both read what the
 * backward products wrote, so every CTA waits for the launch before it (32
 * steps of 8 members on 1024 points, upload and read-back included: 3.49 ms
 * with the reductions in a launch of their own, 3.41 so). */
__global__ void __launch_bounds__(kGThreads) grad_kernel(WgradArgs w, RedArgs r, int tiles) {
    const int b = (int)blockIdx.x - tiles;
    if (b < 0) {
        weight_gradients(w, blockIdx.x);
    } else {
        const int chunks = r.Bp / 128;
        reduce_partial(r, b / 4 % chunks, b / (4 * chunks), b % 4);
    }
}

/* value q of a member's packed reductions: its sum over the 128-sample
 * blocks, and its place among the member's parameters */
__device__ __forceinline__ float reduced(const float* partial, int mem, int nch, int nred, int q) {
    const float* part = partial + (long long)mem * nch * nred;
    float s = 0;
    for (int c = 0; c < nch; ++c) s += part[(long long)c * nred + q];
    return s;
}
__device__ __forceinline__ long long reduced_place(const ParamOffsets& off, int H, int q) {
    if (q < H) return off.b1 + q;
    if (q < H * (1 + kIn)) return off.W1 + (q - H);
    if (q < H * (2 + kIn)) return off.b2 + (q - H * (1 + kIn));
    if (q < H * (3 + kIn)) return off.b3 + (q - H * (2 + kIn));
    if (q < H * (4 + kIn)) return off.W4 + (q - H * (3 + kIn));
    if (q < H * (5 + kIn)) return off.W4 + H + (q - H * (4 + kIn));
    return off.b4 + (q - H * (5 + kIn));
}

__global__ void reduce_final_kernel(RedArgs a) {
    const int mem = blockIdx.y;
    const int nred = red_count(a.H);
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nred) return;
    a.grad[mem * a.pstride + reduced_place(a.off, a.H, q)] = reduced(a.partial, mem, a.Bp / 128, nred, q);
}

/* one Adam update of parameter e with gradient g; the new value */
__device__ __forceinline__ float adam_one(const AdamArgs& a, long long e, float g) {
    const float m = fmaf(1.0f - a.beta1, g, a.beta1 * a.m[e]);
    const float v = fmaf((1.0f - a.beta2) * g, g, a.beta2 * a.v[e]);
    a.m[e] = m;
    a.v[e] = v;
    const float p = a.p[e] - a.lr * (m * a.c1) / (sqrtf(v * a.c2) + a.eps);
    a.p[e] = p;
    return p;
}

/* a 32 x 32 tile (blockIdx.x of 2 x 64) of a hidden layer's weights: f(e)
 * gives the value of parameter e, which goes as BF16 to W [out][in] and,
 * through shared memory, to its transpose [in][out] (the operands of the
 * forward and the backward products, both K-major) */
template <class F>
__device__ __forceinline__ void weight_tile(const AdamArgs& a, int mem, int tile, F f) {
    __shared__ __nv_bfloat16 t[32][34];
    const int layer = tile >> 6, o0 = ((tile >> 3) & 7) * 32, i0 = (tile & 7) * 32;
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
    const long long base = mem * a.pstride + (layer ? a.oW3 : a.oW2);
    const long long wo = ((long long)mem * 2 + layer) * a.H * a.H;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int o = o0 + r0 + 8 * j;
        const __nv_bfloat16 p = __float2bfloat16_rn(f(base + (long long)o * a.H + i0 + c));
        a.wb[wo + (long long)o * a.H + i0 + c] = p;
        t[r0 + 8 * j][c] = p;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = r0 + 8 * j;
        a.wbt[wo + (long long)(i0 + i) * a.H + o0 + c] = t[c][i];
    }
}

/* Adam of every member (blockIdx.y): 128 tiles of W2 and W3, then the other
 * parameters, whose gradients are still partial sums over 128-sample blocks */
__global__ void __launch_bounds__(256) adam_kernel(AdamArgs a) {
    const int mem = blockIdx.y;
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x < 128) {
        weight_tile(a, mem, blockIdx.x, [&](long long e) { return adam_one(a, e, a.g[e]); });
        return;
    }
    const int nred = red_count(a.H), q = (blockIdx.x - 128) * 256 + threadIdx.x;
    if (q < nred)
        adam_one(a, mem * a.pstride + reduced_place(a.off, a.H, q), reduced(a.partial, mem, a.nch, nred, q));
}

__global__ void __launch_bounds__(256) refresh_kernel(AdamArgs a) {
    weight_tile(a, blockIdx.y, blockIdx.x, [&](long long e) { return a.p[e]; });
}

__global__ void ensemble_kernel(EnsArgs a) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.n) return;
    float mean[kOut] = {0, 0}, sq[kOut] = {0, 0};
    for (int m = 0; m < a.members; ++m)
#pragma unroll
        for (int o = 0; o < kOut; ++o)
            mean[o] += a.Yh[((long long)m * a.Bp + r) * kOut + o] * a.sc.y_std[o] + a.sc.y_mean[o];
#pragma unroll
    for (int o = 0; o < kOut; ++o) mean[o] /= (float)a.members;
    for (int m = 0; m < a.members; ++m)
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
            const float d =
                a.Yh[((long long)m * a.Bp + r) * kOut + o] * a.sc.y_std[o] + a.sc.y_mean[o] - mean[o];
            sq[o] += d * d;
        }
    float worst = 0.0f;
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const float s = sqrtf(sq[o] / (float)a.members);
        a.mean[(long long)r * kOut + o] = mean[o];
        a.stdv[(long long)r * kOut + o] = s;
        worst = fmaxf(worst, s);
    }
    /* NaN anywhere also sends the point to the solver */
    if (a.mask) a.mask[r] = !(worst <= a.threshold);
}

int ok_or(cudaError_t e) { return e == cudaSuccess ? 0 : (int)e; }

}  // namespace

int reduce_count(int H) { return red_count(H); }

/* A launch that may begin while the one before it drains: the kernel reads
 * and writes nothing of it before its griddepcontrol.wait. */
template <class... P, class... A>
static int launch_pdl(void (*kernel)(P...), dim3 grid, int threads, size_t smem, void* stream, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return ok_or(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}

template <int EPI>
static int launch_tc(const GemmArgs& a, int members, cudaStream_t s) {
    const void* fn = reinterpret_cast<const void*>(&gemm_tc_kernel<EPI>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGSmem);
    if (e != cudaSuccess) return (int)e;
    return launch_pdl(gemm_tc_kernel<EPI>, dim3(a.N / GN, a.M / GM, members), kGThreads, kGSmem, s, a);
}

int launch_gemm(const GemmArgs& a, int epi, int members, void* stream) {
    if (a.M % GM || a.N % GN || a.K != kGStages * GK || a.M <= 0 || a.N <= 0) return (int)cudaErrorInvalidValue;
    cudaStream_t s = (cudaStream_t)stream;
    if (epi == EPI_FWD) return launch_tc<EPI_FWD>(a, members, s);
    if (epi == EPI_BWD) return launch_tc<EPI_BWD>(a, members, s);
    return (int)cudaErrorInvalidValue;
}

int launch_grad(const WgradArgs& w, const RedArgs& r, int members, void* stream) {
    if (w.H0 % GM || w.K % GK || w.K <= 0 || r.H != kGThreads || r.Bp % 128) return (int)cudaErrorInvalidValue;
    const cudaError_t e =
        cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGSmem);
    if (e != cudaSuccess) return (int)e;
    const int tiles = 2 * members * (w.H0 / GN) * (w.H0 / GM);
    return launch_pdl(grad_kernel, dim3(tiles + 4 * members * (r.Bp / 128)), kGThreads, kGSmem, stream, w, r, tiles);
}

int launch_l1(const L1Args& a, int members, void* stream) {
    return launch_pdl(l1_kernel, dim3(a.Bp / kL1Rows, members), a.H, 0, stream, a);
}

int launch_head(const HeadArgs& a, int members, void* stream) {
    return launch_pdl(head_kernel, dim3(a.Bp / 8, members), 256, 0, stream, a);
}

int launch_reduce_final(const RedArgs& a, int members, void* stream) {
    const int nred = red_count(a.H);
    reduce_final_kernel<<<dim3((nred + 255) / 256, members), 256, 0, (cudaStream_t)stream>>>(a);
    return ok_or(cudaGetLastError());
}

int launch_adam(const AdamArgs& a, void* stream) {
    return launch_pdl(adam_kernel, dim3(128 + (red_count(a.H) + 255) / 256, a.members), 256, 0, stream, a);
}

int launch_refresh_bf16(const AdamArgs& a, void* stream) {
    refresh_kernel<<<dim3(128, a.members), 256, 0, (cudaStream_t)stream>>>(a);
    return ok_or(cudaGetLastError());
}

int launch_ensemble(const EnsArgs& a, void* stream) {
    ensemble_kernel<<<(a.n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(a);
    return ok_or(cudaGetLastError());
}

}  // namespace sur
}  // namespace bte
