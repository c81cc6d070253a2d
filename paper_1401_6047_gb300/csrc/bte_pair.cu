/*
 * bte_pair.cu -- two leap-frog steps per pass over memory, FP32.
 *
 * A grid that does not fit on chip (2049 x 8193 FP32: 268 MB) is bound by
 * memory in the one launch per step kernel: every step reads the state and
 * writes it (85 % of the copy rate).  Here a launch advances two steps (Eqs.
 * leap_frog_1, leap_frog_2 twice) on each row while it passes, so a step
 * moves half the bytes.
 *
 * One warp is one work item: 128 columns (four per lane) of a chunk of rows,
 * walked row by row.  It needs no other warp: the central differences of a
 * new row come from the adjacent lanes (shuffles), and the four half-steps
 * follow one another one row apart,
 *     row j:   W1 = new whole grid after one step,   from old rows F0[j -+ 1]
 *     row j-1: F1 = new fractional grid,             from W1[j-2], W1[j]
 *     row j-2: W2 = whole grid after two steps,      from F1[j-3], F1[j-1]
 *     row j-3: F2 = fractional grid after two steps, from W2[j-4], W2[j-2]
 * each window of two rows of differences in registers (three sets that
 * change roles, so that nothing is moved).  A half-step needs its source one column
 * further on each side, four half-steps four columns: exactly the first and
 * the last lane, so a warp keeps 120 of its 128 columns, and three (source:
 * four) rows on each side of its chunk.
 *
 * Rows arrive by asynchronous 16-byte copies, each lane into its own places
 * of its warp's ring (kRing rows of four arrays) and back out by that lane
 * alone, so there is no barrier anywhere; an old row's place takes the new
 * row that is made from it until the next half-step has read it.
 *
 * What bounds it now: 385 warp instructions per row of 128 columns and two
 * steps (about 320 are the update, the differences and the traffic), issued
 * in 49 % of the slots with three warps per quarter of an SM (160 registers);
 * DRAM is at 56 %.  A row of a chunk's interior takes the fast form of the
 * iteration, with no test of its own; the rows at a chunk's ends take the
 * general one, which costs twice as much.
 *
 * Measured (GB300, us per step, one launch per step / here): 2049 x 8193
 * 93.2 / 58.8; 701 x 5000 27.3 / 15.3; 1024 x 2400 21.6 / 11.8; 1000 x 2503
 * 20.9 / 13.0; 20 x 120001 56.3 / 18.1; few rows, nearly all of whose
 * iterations are general: 16 x 200000 62 / 20, 8 x 350000 77 / 29, 4 x 390000
 * 78 / 25.
 *
 * Where the state is larger than L2, launches walk the rows upward and
 * downward in turn, as in bte_step.cu (DOWN, the mirror image).  The cells'
 * arithmetic is cn_row's, the same bits as one launch per step; rows 0 (a)
 * and 1 (b) of both new whole grids are kept for fold_rows_kernel, which
 * adds them in that kernel's order.
 */
#include <cuda_runtime.h>

#include "bte_device.cuh"
#include "bte_internal.h"

namespace bte {
namespace {

using namespace dev;

constexpr int kRing = 8;            /* rows of a warp's ring                    */
constexpr int kAhead = kRing - 4;   /* rows requested ahead: a place is read for
                                       the last time four rows after it arrived */
constexpr int kPairWarps = 4;       /* warps per CTA                            */
constexpr uint32_t kRowBytes = 4 * 512; /* a, b of the fractional grid, a, b of the whole one */

__host__ __device__ constexpr uint32_t warp_bytes(int rows) {
    return kRing * kRowBytes + 3 * 512 + ((uint32_t)(rows + 8) * 4 + 15) / 16 * 16;
}

__device__ __forceinline__ void cp16(uint32_t dst, const float* src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void lds4(uint32_t p, float (&x)[4]) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
                 : "r"(p)
                 : "memory");
}
__device__ __forceinline__ void sts4(uint32_t p, const float (&x)[4]) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3])
                 : "memory");
}

/* central differences of a row, the outer neighbours from the adjacent lanes
 * (the first and the last lane's outermost ones are not used) */
__device__ __forceinline__ void row_diffs(const float (&x)[4], float (&d)[4]) {
    const float l = __shfl_up_sync(0xffffffffu, x[3], 1), r = __shfl_down_sync(0xffffffffu, x[0], 1);
    d[0] = x[1] - l;
    d[1] = x[2] - x[0];
    d[2] = x[3] - x[1];
    d[3] = r - x[2];
}

__device__ __forceinline__ void zero4(float (&x)[4]) { x[0] = x[1] = x[2] = x[3] = 0.0f; }

/* differences of one row of each source: old fractional, new whole, new
 * fractional and second whole grid */
struct Diffs {
    float a[4], b[4];
};
struct Rows {
    Diffs F0, W1, F1, W2;
};
__device__ __forceinline__ void zero_rows(Rows& r) {
    for (Diffs* d : {&r.F0, &r.W1, &r.F1, &r.W2}) {
        zero4(d->a);
        zero4(d->b);
    }
}
template <bool B>
struct Const {
    static constexpr bool value = B;
};

template <bool DOWN>
__global__ void __launch_bounds__(kPairWarps * 32, 3) pair_kernel(PairArgs A, int launch_i, int parity) {
    constexpr int G = Cols<float>::G;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    /* a warp's shared memory: the ring, each lane's rotation factors of the
     * fractional grid, h times the row factors of rows n0-4 .. n1+3 */
    const uint32_t mine = smem_u32(smem) + (uint32_t)warp * warp_bytes(A.rows);
    const uint32_t ring = mine + lane * 16, rot_f = ring + kRing * kRowBytes;
    const uint32_t hrow = mine + kRing * kRowBytes + 3 * 512;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long kb = __ldcg(A.base) + 2 * launch_i; /* see step_counter in bte_step.cu */
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int item = (int)blockIdx.x * kPairWarps + warp;
    if (item >= A.ntile * A.nchunk) return;
    const int chunk = item / A.ntile, tile = item - chunk * A.ntile;
    const int N = A.N, M = A.M;
    const int n0 = chunk * A.rows, n1 = min(n0 + A.rows, N + 1);
    const int cur = (parity + launch_i) & 1;
    const int m = kPairCols * tile - 4 + 4 * lane; /* first of the lane's columns */
    const bool in_row = G + m + 3 < A.pitch;       /* else zeros (columns past M) */
    const bool own = lane >= 1 && lane <= 30 && m <= M;
    const bool all_ok = m >= 0 && m + 3 <= M;
    const bool warp_ok = __all_sync(0xffffffffu, all_ok);
    /* index of the lane's columns in row 0; rows `pitch` apart (the host
     * keeps an array below 2^32 elements) */
    const uint32_t col = (uint32_t)(G + m), pitch = (uint32_t)A.pitch;
    const float *const Fa = A.a_f[cur], *const Fb = A.b_f[cur], *const Wa = A.a_w[cur], *const Wb = A.b_w[cur];
    float *const oFa = A.a_f[cur ^ 1], *const oFb = A.b_f[cur ^ 1], *const oWa = A.a_w[cur ^ 1],
                *const oWb = A.b_w[cur ^ 1];

    /* drive of the two steps; the rotation factors at the end of a half-step
     * and the start of the grid's next one come from the same table entry,
     * except where the table starts over: there from its first entry and the
     * one after its last, which are the same bits for most drives and always
     * for a constant one (a table of period 1, which starts over every step:
     * 2049 x 8193 81 us per step in the general form of the iteration) */
    const int kk = (int)(kb % A.P), k1 = kk + 1 == A.P ? 0 : kk + 1;
    const Half<float> Dw = half_drive<float>(A.e_whole, A.dstride, kk), Df = half_drive<float>(A.e_frac, A.dstride, kk);
    const Half<float> Ew = half_drive<float>(A.e_whole, A.dstride, k1), Ef = half_drive<float>(A.e_frac, A.dstride, k1);
    const auto differ = [](float x, float y) { return __float_as_uint(x) != __float_as_uint(y); };
    const bool wrap = differ(Ew.E0, Dw.E1) || differ(Ew.B0, Dw.B1) || differ(Ef.E0, Df.E1) || differ(Ef.B0, Df.B1);
    const CnK<float> K = cn_constants<float>(A.h, A.nu, A.xi);
    float g[4], w0[4], w1[4], w2[4];
    {
    float f0[4], f1[4], f2[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool ok = m + e >= 0 && m + e <= M;
        const float ph = ok ? A.col_phi[G + m + e] : 0.0f;
        g[e] = ok ? A.col_g[G + m + e] : 0.0f;
        w0[e] = rot_factor<float>(Dw.E0, Dw.B0, ph, A.hh);
        w1[e] = rot_factor<float>(Dw.E1, Dw.B1, ph, A.hh);
        w2[e] = rot_factor<float>(Ew.E1, Ew.B1, ph, A.hh);
        f0[e] = rot_factor<float>(Df.E0, Df.B0, ph, A.hh);
        f1[e] = rot_factor<float>(Df.E1, Df.B1, ph, A.hh);
        f2[e] = rot_factor<float>(Ef.E1, Ef.B1, ph, A.hh);
    }
    sts4(rot_f, f0);
    sts4(rot_f + 512, f1);
    sts4(rot_f + 1024, f2);
    }
    for (int i = lane; i < n1 - n0 + 8; i += 32) {
        const int r = n0 - 4 + i;
        const float v = r >= 0 && r <= N ? Rn<float>::mul(A.h, A.row_a0[r]) : 0.0f;
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(hrow + i * 4), "f"(v) : "memory");
    }
    __syncwarp();
    /* the start factors of the second step where they differ */
    auto start_of = [&](const Half<float>& E, float (&x)[4]) {
        if (wrap) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                x[e] = rot_factor<float>(E.E0, E.B0, (m + e >= 0 && m + e <= M) ? A.col_phi[G + m + e] : 0.0f, A.hh);
        }
    };

    const int Q = n1 - n0 + 6; /* iterations q = 0 .. Q-1; q = -2, -1 only read a row */
    auto row_of = [&](int q) { return DOWN ? n1 + 2 - q : n0 - 3 + q; }; /* row j of iteration q */
    constexpr int dj = DOWN ? -1 : 1;
    auto place = [&](int q) { return ring + (uint32_t)((q + 2) & (kRing - 1)) * kRowBytes; };
    auto valid = [&](int r) { return r >= 0 && r <= N; };
    /* request old fractional row j + 1 and old whole row j of iteration q */
    auto request = [&](int q) {
        if (q < Q) {
            const int j = row_of(q), jf = j + dj;
            const uint32_t p = place(q);
            if (valid(jf)) {
                const uint32_t o = in_row ? (uint32_t)jf * pitch + col : 0u;
                cp16(p, Fa + o, in_row);
                cp16(p + 512, Fb + o, in_row);
            }
            if (q >= 0 && valid(j)) {
                const uint32_t o = in_row ? (uint32_t)j * pitch + col : 0u;
                cp16(p + 1024, Wa + o, in_row);
                cp16(p + 1536, Wb + o, in_row);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int q = -2; q < -2 + kAhead; ++q) request(q);

    auto row_factor = [&](int r) {
        float v;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(hrow + (r - n0 + 4) * 4) : "memory");
        return v;
    };

    /* One half-step of a row: own values at `src`, the source's row just made
     * or read (nw) and its row two back (od). */
    auto half = [&](uint32_t src, const Diffs& nw, const Diffs& od, float cc, int r, const float (&t0)[4],
                    const float (&t1)[4], float (&xa)[4], float (&xb)[4], auto fast) {
        constexpr bool F = decltype(fast)::value;
        const float hr = row_factor(r);
        float a[4], b[4];
        lds4(src, a);
        lds4(src + 512, b);
        const float chi = !F && r == 1 ? 2.0f : 1.0f;
        if constexpr (!DOWN)
            cn_row<float, 4, F>(a, b, nw.b, od.b, od.a, nw.a, cc, chi, hr, g, (float)r, t0, t1, K, xa, xb);
        else
            cn_row<float, 4, F>(a, b, od.b, nw.b, nw.a, od.a, cc, chi, hr, g, (float)r, t0, t1, K, xa, xb);
        if (!warp_ok) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool ok = m + e >= 0 && m + e <= M;
                xa[e] = ok ? xa[e] : 0.0f;
                xb[e] = ok ? xb[e] : 0.0f;
            }
        }
        if (!F && r == 0) zero4(xb);
    };
    auto store = [&](float* pa, float* pb, int r, const float (&xa)[4], const float (&xb)[4]) {
        if (!own) return;
        const uint32_t o = (uint32_t)r * pitch + col;
        if (warp_ok || all_ok) {
            *reinterpret_cast<float4*>(pa + o) = make_float4(xa[0], xa[1], xa[2], xa[3]);
            *reinterpret_cast<float4*>(pb + o) = make_float4(xb[0], xb[1], xb[2], xb[3]);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (m + e <= M) {
                    pa[o + e] = xa[e];
                    pb[o + e] = xb[e];
                }
        }
    };
    /* rows 0 (a) and 1 (b) of the whole grid after step s (0, 1) of this launch */
    auto keep = [&](int s, int r, const float (&xa)[4], const float (&xb)[4]) {
        if (r > 1 || n0 != 0 || !own) return;
        float* out = A.kept + ((size_t)(2 * launch_i + s) * 2 + r) * A.mpad + m;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (m + e <= M) out[e] = r == 0 ? xa[e] : xb[e];
    };

    /* iteration q: `od` holds the differences of the rows two back of each
     * source, `nw` takes those of the rows it makes.  FAST: every row it
     * touches exists and is none of rows 0 and 1, every output is this
     * chunk's, and the two steps share their rotation factors. */
    auto iteration = [&](int q, const Rows& od, Rows& nw, auto fast) {
        constexpr bool F = decltype(fast)::value;
        const int j = row_of(q);
        const uint32_t here = place(q), two = place(q - 2), four = place(q - 4);
        asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
        float xa[4], xb[4], t0[4];
        if (F || valid(j + dj)) {
            lds4(here, xa);
            lds4(here + 512, xb);
            row_diffs(xa, nw.F0.a);
            row_diffs(xb, nw.F0.b);
        } else {
            zero4(nw.F0.a);
            zero4(nw.F0.b);
        }
        /* W1, row j */
        if (F || (q >= 0 && valid(j))) {
            half(here + 1024, nw.F0, od.F0, Dw.cc, j, w0, w1, xa, xb, fast);
            sts4(here + 1024, xa);
            sts4(here + 1536, xb);
            if (!F) keep(0, j, xa, xb);
            row_diffs(xa, nw.W1.a);
            row_diffs(xb, nw.W1.b);
        } else {
            zero4(nw.W1.a);
            zero4(nw.W1.b);
        }
        /* F1, row j - 1 */
        const int r1 = j - dj, r2 = j - 2 * dj, r3 = j - 3 * dj;
        if (F || (q >= 2 && valid(r1))) {
            float t1[4];
            lds4(rot_f, t0);
            lds4(rot_f + 512, t1);
            half(two, nw.W1, od.W1, Df.cc, r1, t0, t1, xa, xb, fast);
            sts4(two, xa);
            sts4(two + 512, xb);
            row_diffs(xa, nw.F1.a);
            row_diffs(xb, nw.F1.b);
        } else {
            zero4(nw.F1.a);
            zero4(nw.F1.b);
        }
        /* W2, row j - 2 */
        if (F || (q >= 4 && valid(r2))) {
            if (F) {
                half(two + 1024, nw.F1, od.F1, Ew.cc, r2, w1, w2, xa, xb, fast);
                store(oWa, oWb, r2, xa, xb);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) t0[e] = w1[e];
                start_of(Ew, t0);
                half(two + 1024, nw.F1, od.F1, Ew.cc, r2, t0, w2, xa, xb, fast);
                if (r2 >= n0 && r2 < n1) {
                    store(oWa, oWb, r2, xa, xb);
                    keep(1, r2, xa, xb);
                }
            }
            row_diffs(xa, nw.W2.a);
            row_diffs(xb, nw.W2.b);
        } else {
            zero4(nw.W2.a);
            zero4(nw.W2.b);
        }
        /* F2, row j - 3 */
        if (F || (q >= 6 && valid(r3))) {
            float t1[4];
            lds4(rot_f + 512, t0);
            lds4(rot_f + 1024, t1);
            if (!F) start_of(Ef, t0);
            half(four, nw.W2, od.W2, Ef.cc, r3, t0, t1, xa, xb, fast);
            store(oFa, oFb, r3, xa, xb);
        }
        request(q + kAhead);
    };

    Rows R0, R1, R2; /* R0: two rows back, R1: the row between */
    zero_rows(R0);
    zero_rows(R1);
    /* fast iterations q0 .. q1 - 1: rows j + 1 to j - 3 exist and are none of
     * rows 0 and 1, the outputs r2 and r3 lie in the chunk */
    int q0 = 6, q1 = Q - 1;
    if (!DOWN) {
        q0 = max(q0, 8 - n0);     /* r3 = n0 - 6 + q >= 2 */
        q1 = min(q1, N + 3 - n0); /* j + 1 = n0 - 2 + q <= N */
    } else {
        q0 = max(q0, n1 + 5 - N); /* r3 = n1 + 5 - q <= N */
        q1 = min(q1, n1 + 1);     /* j = n1 + 2 - q >= 2 */
    }
    if (wrap) q1 = q0;
    int q = -2;
    for (; q < min(q0, Q); ++q) {
        iteration(q, R0, R2, Const<false>{});
        R0 = R1;
        R1 = R2;
    }
    for (; q + 3 <= q1; q += 3) {
        iteration(q, R0, R2, Const<true>{});
        iteration(q + 1, R1, R0, Const<true>{});
        iteration(q + 2, R2, R1, Const<true>{});
    }
    for (; q < Q; ++q) {
        iteration(q, R0, R2, Const<false>{});
        R0 = R1;
        R1 = R2;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

}  // namespace

int pair_configure(int rows, int* warps_per_sm) {
    for (const void* fn : {reinterpret_cast<const void*>(&pair_kernel<false>), reinterpret_cast<const void*>(&pair_kernel<true>)}) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        if (e != cudaSuccess) return (int)e;
    }
    int blocks = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, pair_kernel<false>, kPairWarps * 32,
                                                                        (size_t)kPairWarps * warp_bytes(rows));
    *warps_per_sm = blocks * kPairWarps;
    return (int)e;
}

int launch_pair(const PairArgs& a, int i, int parity, bool pdl, void* stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.ntile * a.nchunk + kPairWarps - 1) / kPairWarps);
    cfg.blockDim = dim3(kPairWarps * 32);
    cfg.dynamicSmemBytes = (size_t)kPairWarps * warp_bytes(a.rows);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = a.alt && (i & 1) ? cudaLaunchKernelEx(&cfg, pair_kernel<true>, a, i, parity)
                                           : cudaLaunchKernelEx(&cfg, pair_kernel<false>, a, i, parity);
    return (int)e;
}

}  // namespace bte
