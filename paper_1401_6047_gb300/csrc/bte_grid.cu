/*
 * bte_grid.cu -- single-instance solver with the whole grid on chip, one
 * block of it per SM.
 *
 * The four arrays (a and b of the whole and of the fractional grid, Sec. 3)
 * of a grid of up to about two million FP32 cells fit the shared memory of
 * the 152 SMs together (401 x 4001: 25.7 MB of 34).  The grid is cut into
 * GR x GC blocks of R harmonic rows x W phi_y columns, one CTA each, all
 * resident at once (a cooperative launch); a CTA keeps its block, with one
 * halo row and column on each side, in shared memory for the whole launch
 * and advances it in place: a half-step of the leap-frog scheme (Eqs.
 * leap_frog_1, leap_frog_2) updates one grid from the other one's rows n-1,
 * n+1 at columns m-1, m+1 and from the cell's own values.
 *
 * What bounds it: one launch per step moves the state through L2 twice and
 * walks its rows behind a block barrier each (401 x 4001 FP32: 17.4 us per
 * step); here a step moves only the blocks' edges, and what remains is the
 * arithmetic of the update (147 warp instructions per 128 cells of a
 * half-step; the issue slots are 40 % busy at 401 x 4001) and one
 * exchange of edges per half-step, about 0.5 us through L2.
 *
 * Measured (GB300, us per step, one launch per step / here): 31 x 201 FP64
 * 22.7 / 2.6, FP32 9.6 / 2.0; 65 x 1000 FP64 43 / 8.1; 138 x 1533 FP32 14.5 /
 * 3.2; 120 x 4000 FP32 13.9 / 3.8; 401 x 4001 FP32 17.0 / 7.2.  (With the
 * compute threads polling: 3.9, 2.5, 9.4, 3.6, 4.5 and 7.5.)
 *
 * A half-step of a CTA (its last 128 threads only poll, keep rows 0 and 1 and
 * make the next half-step's rotation factors; a poll is an L2 round trip, 700
 * to 1000 cycles, even when the word is there, so it runs beside 1.):
 *   1. cells that read no halo (all but the block's first and last rows and
 *      column groups), and in FP64 the part of the boundary cells that needs
 *      none, while the neighbours' edges are still under way;
 *   2. the halo cells of the grid that is read, polled from exchange words;
 *   3. the remaining cells; the outermost ones are published as exchange
 *      words as they are made.
 * An exchange word is 8 bytes, written and read as a whole: 32 bits of a
 * value under the number of the half-step that made it, so a value and its
 * flag arrive together and no fence or second load is needed (FP32: the a
 * and b of a cell are two words in one 16-byte access; FP64: four words in
 * two).  Words come in two buffers by the parity of the producing grid's
 * update count.  A word is rewritten four half-steps after it was written;
 * by then its writer has read words that each of its readers published
 * after reading it (blocks read each other's edges in both directions, the
 * corners included), so no reader can find it gone.
 *
 * FP32 cells are updated in column pairs (cn_row), whose last sums are
 * multiply-adds where the one-column form rounds twice; grid_kernel<float, 1>
 * has the latter's bits, those of bte_wide.cu, for the mode that gives them.
 *
 * Every wait is bounded by %globaltimer.  A wait that gives up sets the
 * launch's quit word, at which every other waiting CTA gives up too, and the
 * error word that the host reports as BTE_ETIMEOUT.
 *
 * Rows 0 (a) and 1 (b) of each new whole grid are copied to a buffer, and
 * fold_rows_kernel (wide rows: fold_tiles_kernel and fold_tail_kernel) adds
 * them afterwards in exactly the order of the one
 * launch per step kernel (V columns per lane, a 32-lane tree, the warps of a
 * tile in order, tiles in order), so the drift velocity and norm (Eqs.
 * v_dr_generic, norm_in_phi) of a step are the same bits whichever kernel
 * made it and wherever the blocks' borders lie.
 */
#include <cuda_runtime.h>

#include "bte_device.cuh"
#include "bte_internal.h"

namespace bte {
namespace {

using namespace dev;

/* groups of 32 lanes' columns that one CTA of the row sums takes: the whole
 * row where it has no more than kFoldGroups (16384 FP32 columns), else
 * kFoldTileGroups per CTA */
constexpr int kFoldGroups = 128, kFoldTileGroups = 64;

template <typename T, int V>
__device__ __forceinline__ void ldv(const T* p, T (&x)[V]) {
    if constexpr (sizeof(T) * V == 16 && sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        x[0] = v.x;
        x[1] = v.y;
        x[2] = v.z;
        x[3] = v.w;
    } else if constexpr (sizeof(T) * V == 16) {
        const double2 v = *reinterpret_cast<const double2*>(p);
        x[0] = v.x;
        x[1] = v.y;
    } else if constexpr (sizeof(T) * V == 8 && V == 2) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        x[0] = v.x;
        x[1] = v.y;
    } else {
#pragma unroll
        for (int e = 0; e < V; ++e) x[e] = p[e];
    }
}

template <typename T, int V>
__device__ __forceinline__ void stv(T* p, const T (&x)[V]) {
    if constexpr (sizeof(T) * V == 16 && sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    } else if constexpr (sizeof(T) * V == 16) {
        *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
    } else if constexpr (sizeof(T) * V == 8 && V == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
    } else {
#pragma unroll
        for (int e = 0; e < V; ++e) p[e] = x[e];
    }
}

/* central differences of a group from its values and outer neighbours */
template <typename T, int V>
__device__ __forceinline__ void diffs_of(const T (&own)[V], T left, T right, T (&d)[V]) {
    if constexpr (V == 1) {
        d[0] = right - left;
    } else {
        d[0] = own[1] - left;
#pragma unroll
        for (int e = 1; e < V - 1; ++e) d[e] = own[e + 1] - own[e - 1];
        d[V - 1] = right - own[V - 2];
    }
}

/* the same with the outer neighbours loaded */
template <typename T, int V>
__device__ __forceinline__ void diff_load(const T* p, T (&d)[V]) {
    T own[V];
    if constexpr (V > 1) ldv<T, V>(p, own);
    diffs_of<T, V>(own, p[-1], p[V], d);
}

/* the same with the outer neighbours taken from the adjacent lanes where
 * those hold the adjacent columns; every lane of the warp calls it */
template <typename T, int V>
__device__ __forceinline__ void diff_lanes(const T* p, bool l_adj, bool r_adj, T (&d)[V]) {
    if constexpr (V == 1) {
        d[0] = p[1] - p[-1];
    } else {
        T own[V];
        ldv<T, V>(p, own);
        T left = __shfl_up_sync(0xffffffffu, own[V - 1], 1);
        T right = __shfl_down_sync(0xffffffffu, own[0], 1);
        if (!l_adj) left = p[-1];
        if (!r_adj) right = p[V];
        diffs_of<T, V>(own, left, right, d);
    }
}

__device__ __forceinline__ int round_warp(int n) { return (n + 31) / 32 * 32; }

struct Words2 {
    unsigned long long x, y;
};
__device__ __forceinline__ Words2 ld_words(const Words2* p) {
    Words2 w;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void st_words(Words2* p, unsigned tag, unsigned lo, unsigned hi) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | lo), "l"(t | hi) : "memory");
}

/* the exchange entry of one cell: sizeof(T) / 4 pairs of words */
template <typename T>
__device__ __forceinline__ void publish(Words2* e, unsigned tag, T a, T b) {
    if constexpr (sizeof(T) == 4) {
        st_words(e, tag, __float_as_uint(a), __float_as_uint(b));
    } else {
        st_words(e, tag, (unsigned)__double2loint(a), (unsigned)__double2hiint(a));
        st_words(e + 1, tag, (unsigned)__double2loint(b), (unsigned)__double2hiint(b));
    }
}

/* shared memory: arrays and factors, then the poll and boundary tables */
template <typename T>
__host__ __device__ inline size_t poll_offset(int R, int W, int V) {
    const size_t b = ((4 * (size_t)(R + 2) + 6) * (W + 2 * V) + 2 * (R + 2)) * sizeof(T);
    return (b + 15) / 16 * 16;
}

template <typename T, int V>
__global__ void __launch_bounds__(kGridThreads, 1) grid_kernel(GridArgs<T> A) {
    static_assert(sizeof(T) == 4 || V == 1, "FP64 takes one column per thread");
    constexpr int GG = Cols<T>::G;            /* global ghost columns before m = 0 */
    constexpr int E = sizeof(T) / 4;          /* word pairs per exchange entry */
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int N = A.N, M = A.M, N1 = N + 1, M1 = M + 1, W = A.W;
    const int bi = (int)blockIdx.x / A.GC, bj = (int)blockIdx.x - bi * A.GC;
    const int r0 = bi * A.R, R = min(A.R, N1 - r0);
    const int c0 = bj * W, Wb = min(W, M1 - c0);
    const int ncg = (Wb + V - 1) / V;
    /* local columns: V ghosts (the last one the left halo), W own, V ghosts
     * (the first one the right halo) */
    const int P = W + 2 * V;
    const int arr = (A.R + 2) * P;
    T* s = reinterpret_cast<T*>(smem); /* [4][R + 2][P]: a_w, b_w, a_f, b_f */
    T* sG = s + 4 * arr;               /* [P] column factor of a0 */
    T* sPh = sG + P;                   /* [P] phi_m */
    T* sT = sPh + P;                   /* [2][2][P] rotation factors of this and the next half-step */
    T* sR = sT + 4 * P;                /* [R + 2] h times the row factor of a0 */
    T* sN = sR + A.R + 2;              /* [R + 2] n */
    /* the block's polls: {entry within one (buffer, grid) of the words,
     * place in an a array | column entry << 31}, and its boundary groups:
     * local row << 16 | group */
    uint2* sPoll = reinterpret_cast<uint2*>(smem + poll_offset<T>(A.R, W, V));
    uint32_t* sBnd = reinterpret_cast<uint32_t*>(sPoll + 2 * (W + 2 + A.R));
    T* const gs[4] = {A.a_w, A.b_w, A.a_f, A.b_f};

    /* ---- load: zero everything, then the block and its halo cells ---- */
    for (int q = tid; q < 4 * arr + 6 * P + 2 * (A.R + 2); q += nthr) s[q] = (T)0;
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const T* g = gs[a] + GG + c0;
        T* d = s + a * arr + V;
        for (int q = tid; q < (R + 2) * ncg; q += nthr) {
            const int li = q / ncg, gq = q - li * ncg, n = r0 - 1 + li;
            if (n < 0 || n > N) continue;
            T v[V];
            ldv<T, V>(g + (size_t)n * A.pitch + gq * V, v); /* ghost columns hold zeros */
            stv<T, V>(d + li * P + gq * V, v);
        }
        for (int q = tid; q < 2 * (R + 2); q += nthr) {
            const int li = q >> 1, n = r0 - 1 + li, m = (q & 1) ? W : -1;
            if (n < 0 || n > N || c0 + m < 0 || c0 + m > M) continue;
            d[li * P + m] = g[(size_t)n * A.pitch + m];
        }
    }
    for (int q = tid; q < Wb; q += nthr) {
        sG[V + q] = A.col_g[GG + c0 + q];
        sPh[V + q] = A.col_phi[GG + c0 + q];
    }
    for (int q = tid; q < R; q += nthr) {
        sR[q + 1] = Rn<T>::mul(A.h, A.row_a0[r0 + q]);
        sN[q + 1] = (T)(r0 + q);
    }
    const CnK<T> cn = cn_constants<T>(A.h, A.nu, A.xi);
    const T hh = A.hh;
    Words2* const rowx = reinterpret_cast<Words2*>(A.rowx);
    Words2* const colx = reinterpret_cast<Words2*>(A.colx);
    /* words of one (buffer, grid): [GR][first, last row][M+1] row entries, and
     * [GC][first, last column][N+1] column entries */
    const uint32_t row_set = (uint32_t)A.GR * 2 * M1 * E, col_set = (uint32_t)A.GC * 2 * N1 * E;

    /* interior cells: rows 1 .. R-2 of column groups 1 .. ncg-2; thread ->
     * (column group, block of consecutive rows), walked as two chains of
     * stride 2, so that the other grid's differences of row i+1 serve rows i
     * and i+2 */
    const int nci = max(ncg - 2, 0), nri = max(R - 2, 0);
    /* boundary cells: rows 0 and R-1, then groups 0 and ncg-1 of the rows between */
    const int nrb = R >= 2 ? 2 : 1, ncb = ncg >= 2 ? 2 : 1;
    const int nb_rows = nrb * ncg, nb = nb_rows + ncb * nri;
    for (int u = tid; u < nb; u += nthr) {
        int il, g;
        if (u < nb_rows) {
            il = u < ncg ? 0 : R - 1;
            g = u < ncg ? u : u - ncg;
        } else {
            const int v = u - nb_rows;
            il = 1 + v / ncb;
            g = (v - (il - 1) * ncb) ? ncg - 1 : 0;
        }
        sBnd[u] = (uint32_t)il << 16 | (uint32_t)g;
    }
    /* halo cells polled: top and bottom rows (corners included), left and right columns */
    const int nq = 2 * (Wb + 2) + 2 * R;
    for (int q = tid; q < nq; q += nthr) {
        uint32_t e = 0xffffffffu, col = 0;
        int li, lc;
        if (q < 2 * (Wb + 2)) {
            const bool bot = q >= Wb + 2;
            lc = (bot ? q - (Wb + 2) : q) - 1;
            li = bot ? R : -1;
            if (r0 + li >= 0 && r0 + li <= N && c0 + lc >= 0 && c0 + lc <= M)
                e = ((uint32_t)((bot ? bi + 1 : bi - 1) * 2 + (bot ? 0 : 1)) * M1 + (c0 + lc)) * E;
        } else {
            const int q2 = q - 2 * (Wb + 2);
            const bool rgt = q2 >= R;
            li = rgt ? q2 - R : q2;
            lc = rgt ? Wb : -1;
            if (c0 + lc >= 0 && c0 + lc <= M)
                e = ((uint32_t)((rgt ? bj + 1 : bj - 1) * 2 + (rgt ? 0 : 1)) * N1 + (r0 + li)) * E;
            col = 0x80000000u;
        }
        sPoll[q] = make_uint2(e, (uint32_t)((li + 1) * P + V + lc) | col);
    }
    /* this block's own entries, without the (buffer, grid) offset */
    Words2* const top = rowx + (size_t)((bi * 2) * M1 + c0) * E;
    Words2* const bottom = top + (size_t)M1 * E;
    Words2* const left = colx + (size_t)((bj * 2) * N1 + r0) * E;
    Words2* const right = left + (size_t)N1 * E;

    /* The last A.help threads poll.  Interior work starts at the threads that have
     * no boundary group, so that in a small block different warps do the two. */
    const int nc = nthr - A.help;
    const bool comp = tid < nc;
    const int ptid = tid - nc, pthr = A.help; /* polling threads: ptid >= 0 */
    const int cpp = max(min(nci, nc), 1);
    const int rsplit = nc / cpp;
    const int ntid = nb < nc ? tid - round_warp(nb) + (tid < round_warp(nb) ? nc : 0) : tid;
    const int gl = ntid % cpp, rpart = ntid / cpp;
    const int nrow = (nri + rsplit - 1) / rsplit;
    const int lo = 1 + rpart * nrow;
    const bool has_int = nci > 0 && nri > 0 && comp;

    const long long k0 = *A.base;
    int kk = (int)(k0 % A.P);
    Half<T> D = half_drive<T>(A.e_whole, A.dstride, kk);
    __syncthreads();
    /* rotation factors of the block's columns for a half-step */
    auto rotations = [&](T* t, const Half<T>& H, int q0, int step) {
        for (int q = q0; q < Wb; q += step) {
            const T ph = sPh[V + q];
            t[V + q] = rot_factor<T>(H.E0, H.B0, ph, hh);
            t[P + V + q] = rot_factor<T>(H.E1, H.B1, ph, hh);
        }
    };
    rotations(sT, D, tid, nthr);
    __syncthreads();

    /* FP64, where twice the boundary cells find threads: two adjacent lanes per
     * cell, one for a and one for b (the two halves of an update are the same
     * operations, so a warp's instruction serves both; it costs the same
     * however few of its lanes hold a cell) */
    const bool two = sizeof(T) == 8 && 2 * nb <= nc;
    const bool two_on = two && comp && (tid >> 1) < nb;
    const int ab = tid & 1;
    const int il2 = two_on ? (int)(sBnd[tid >> 1] >> 16) : 0, m2 = two_on ? (int)(sBnd[tid >> 1] & 0xffffu) : 0;

    const long long nhs = 2ll * A.K;
    for (long long hs = 0; hs < nhs; ++hs) {
        /* even: whole grid z_w^{k+1} = T(z_w^k; S(z_f^{k+1/2})); odd:
         * fractional grid z_f^{k+3/2} = T(z_f^{k+1/2}; S(z_w^{k+1})) */
        const int hf = (int)(hs & 1);
        T* const so = s + (hf ? 2 * arr : 0) + V;       /* own grid, column c0 */
        const T* const sx = s + (hf ? 0 : 2 * arr) + V; /* grid that is read */
        const unsigned tag = (unsigned)hs;
        const T* const rot = sT + (hs & 1) * 2 * P;
        /* the drive of the next half-step, long before it is needed */
        if (hf) kk = kk + 1 == A.P ? 0 : kk + 1;
        const Half<T> Dn = half_drive<T>(hf ? A.e_whole : A.e_frac, A.dstride, kk);

        if (has_int) {
            for (int g0 = 0; g0 < nci; g0 += cpp) {
                const int g = g0 + gl;
                const bool g_on = rpart < rsplit && g < nci;
                const int m = (g_on ? g + 1 : 1) * V;
                const bool l_adj = lane > 0 && gl > 0;
                const bool r_adj = lane < 31 && gl + 1 < cpp && g + 1 < nci;
                T gc[V], t0[V], t1[V];
                ldv<T, V>(sG + V + m, gc);
                ldv<T, V>(rot + V + m, t0);
                ldv<T, V>(rot + P + V + m, t1);
#pragma unroll 1
                for (int ch = 0; ch < 2; ++ch) {
                    const int len = (nrow + 1 - ch) / 2; /* same for every thread */
                    if (len == 0) continue;
                    const int i0 = lo + ch;
                    T da_u[V], db_u[V];
                    {
                        const T* p = sx + min(i0, R - 2) * P + m;
                        diff_lanes<T, V>(p, l_adj, r_adj, da_u);
                        diff_lanes<T, V>(p + arr, l_adj, r_adj, db_u);
                    }
#pragma unroll 2
                    for (int ii = 0; ii < len; ++ii) {
                        const int i = i0 + 2 * ii;
                        const bool on = g_on && i < R - 1;
                        const int il = min(i, R - 2);
                        const int n = r0 + il;
                        const T* p = sx + (il + 2) * P + m;
                        T da_d[V], db_d[V], oa[V], ob[V], an[V], bn[V];
                        diff_lanes<T, V>(p, l_adj, r_adj, da_d);
                        diff_lanes<T, V>(p + arr, l_adj, r_adj, db_d);
                        T* const po = so + (il + 1) * P + m;
                        ldv<T, V>(po, oa);
                        ldv<T, V>(po + arr, ob);
                        cn_row<T, V>(oa, ob, db_d, db_u, da_u, da_d, D.cc, n == 1 ? (T)2 : (T)1, sR[il + 1], gc,
                                     sN[il + 1], t0, t1, cn, an, bn);
                        if (on) {
                            stv<T, V>(po, an);
                            stv<T, V>(po + arr, bn);
                        }
#pragma unroll
                        for (int e = 0; e < V; ++e) {
                            da_u[e] = da_d[e];
                            db_u[e] = db_d[e];
                        }
                    }
                }
            }
        }
        /* rows 0 (a) and 1 (b) of the new whole grid, which this half-step
         * leaves unchanged, for the step's sums */
        if (hf && r0 <= 1) {
            T* out = A.rows + (size_t)(hs >> 1) * 2 * A.mpad + c0;
            for (int q = ptid; q >= 0 && q < Wb; q += pthr) {
                if (r0 == 0) out[q] = s[P + V + q];
                const int l1 = 1 - r0; /* local row of harmonic 1 */
                if (l1 < R) out[A.mpad + q] = s[arr + (l1 + 1) * P + V + q];
            }
        }
        /* FP64: the part of the first boundary cell's update that needs no
         * halo, while the edges are under way (11 of its 23 operations) */
        CnCoef<T> pre{};
        T preG = (T)0, preH = (T)0;
        auto own_part = [&](int il, int m, CnCoef<T>& c, T& G0, T& H0) {
            if constexpr (sizeof(T) == 8) {
                const T nf = sN[il + 1];
                c = cn_coef<T>(Rn<T>::mul(nf, rot[V + m]), Rn<T>::mul(nf, rot[P + V + m]), cn);
                const T* const po = so + (il + 1) * P + m;
                cn_own(po[0], po[arr], sR[il + 1], sG[V + m], c, cn, G0, H0);
            }
        };
        T own = (T)0, own0 = (T)0, sth1 = (T)0; /* two lanes: a and G0, or b and H0 */
        if constexpr (sizeof(T) == 8) {
            if (two_on) {
                const T nf = sN[il2 + 1];
                pre = cn_coef<T>(Rn<T>::mul(nf, rot[V + m2]), Rn<T>::mul(nf, rot[P + V + m2]), cn);
                const T* const po = so + (il2 + 1) * P + m2;
                own = po[ab ? arr : 0];
                const T p = Rn<T>::mul(pre.ca, po[ab ? 0 : arr]);
                own0 = Rn<T>::fma(ab ? (T)0 : sR[il2 + 1], sG[V + m2], Rn<T>::fma(-cn.h, own, ab ? p : -p));
                sth1 = ab ? pre.th1 : -pre.th1;
            }
        }
        if (sizeof(T) == 8 && !two && comp && tid < nb) own_part((int)(sBnd[tid] >> 16), (int)(sBnd[tid] & 0xffffu), pre, preG, preH);
        /* the halo cells of the grid that is read (loaded with the block for
         * the first half-step) */
        bool ok = true;
        if (hs > 0) {
            const uint32_t set = ((uint32_t)(hs - 1) >> 1 & 1) * 2 + (hf ? 0 : 1);
            const Words2* const rx = rowx + (size_t)set * row_set;
            const Words2* const cx = colx + (size_t)set * col_set;
            for (int q = ptid; q >= 0 && q < nq; q += pthr) {
                const uint2 pe = sPoll[q];
                if (pe.x == 0xffffffffu) continue;
                const Words2* const e = ((pe.y >> 31) ? cx : rx) + pe.x;
                Words2 w[E];
                auto fetch = [&]() {
                    bool fresh = true;
#pragma unroll
                    for (int u = 0; u < E; ++u) {
                        w[u] = ld_words(e + u);
                        fresh = fresh && (unsigned)(w[u].x >> 32) == tag && (unsigned)(w[u].y >> 32) == tag;
                    }
                    return fresh;
                };
                if (ok && !fetch()) {
                    const uint64_t t_start = global_timer();
                    for (int spin = 1; !fetch(); ++spin) {
                        if ((spin & 63) == 0 && (*reinterpret_cast<const volatile int*>(A.quit) != 0 ||
                                                 global_timer() - t_start > kWaitLimitNs)) {
                            ok = false;
                            break;
                        }
                    }
                }
                T* const d = const_cast<T*>(sx) - V + (pe.y & 0x7fffffffu);
                if constexpr (sizeof(T) == 4) {
                    d[0] = __uint_as_float((unsigned)w[0].x);
                    d[arr] = __uint_as_float((unsigned)w[0].y);
                } else {
                    d[0] = __hiloint2double((int)(unsigned)w[0].y, (int)(unsigned)w[0].x);
                    d[arr] = __hiloint2double((int)(unsigned)w[E - 1].y, (int)(unsigned)w[E - 1].x);
                }
            }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicExch(A.quit, 1);
                atomicExch(A.err, kErrTimeout);
            }
            return;
        }
        /* the next half-step's rotation factors */
        if (!comp) rotations(sT + ((hs + 1) & 1) * 2 * P, Dn, ptid, pthr);
        if (comp) {
            const uint32_t set = ((uint32_t)hs >> 1 & 1) * 2 + hf;
            const size_t rs = (size_t)set * row_set, cs = (size_t)set * col_set;
            if constexpr (sizeof(T) == 8) {
                if (two) { /* cn_finish, one half per lane */
                    const int n = r0 + il2;
                    T gh = (T)0;
                    if (two_on) {
                        const T* x = sx + (ab ? 0 : arr) + il2 * P + m2; /* row n - 1 of b (a's lane) or a */
                        const T d_prev = x[1] - x[-1], d_next = x[2 * P + 1] - x[2 * P - 1];
                        gh = Rn<T>::fma(D.cc, Rn<T>::fma(ab && n == 1 ? (T)2 : (T)1, ab ? d_prev : d_next,
                                                         ab ? -d_next : -d_prev),
                                        own0);
                    }
                    const T other = __shfl_xor_sync(0xffffffffu, gh, 1);
                    if (two_on) {
                        T v = Rn<T>::fma(Rn<T>::fma(sth1, other, gh), pre.inv, own);
                        if (ab && n == 0) v = (T)0;
                        so[(ab ? arr : 0) + (il2 + 1) * P + m2] = v;
                        const unsigned vl = (unsigned)__double2loint(v), vh = (unsigned)__double2hiint(v);
                        if (il2 == 0 && bi > 0) st_words(top + rs + m2 * E + ab, tag + 1, vl, vh);
                        if (il2 == R - 1 && bi + 1 < A.GR) st_words(bottom + rs + m2 * E + ab, tag + 1, vl, vh);
                        if (m2 == 0 && bj > 0) st_words(left + cs + il2 * E + ab, tag + 1, vl, vh);
                        if (m2 == ncg - 1 && bj + 1 < A.GC) st_words(right + cs + il2 * E + ab, tag + 1, vl, vh);
                    }
                }
            }
            for (int u = two ? nb : tid; u < nb; u += nc) {
                const uint32_t be = sBnd[u];
                const int il = (int)(be >> 16), g = (int)(be & 0xffffu);
                const int m = g * V, n = r0 + il;
                const T* pu = sx + il * P + m;
                const T* pd = pu + 2 * P;
                T da_u[V], da_d[V], db_u[V], db_d[V], oa[V], ob[V], an[V], bn[V];
                diff_load<T, V>(pu, da_u);
                diff_load<T, V>(pd, da_d);
                diff_load<T, V>(pu + arr, db_u);
                diff_load<T, V>(pd + arr, db_d);
                T* const po = so + (il + 1) * P + m;
                ldv<T, V>(po, oa);
                ldv<T, V>(po + arr, ob);
                if constexpr (sizeof(T) == 8) {
                    if (u != tid) own_part(il, m, pre, preG, preH);
                    cn_finish(oa[0], ob[0], stencil_a<T>(db_d[0], db_u[0]),
                              stencil_b<T>(n == 1 ? (T)2 : (T)1, da_u[0], da_d[0]), D.cc, preG, preH, pre, an[0], bn[0]);
                } else {
                    T gc[V], t0[V], t1[V];
                    ldv<T, V>(sG + V + m, gc);
                    ldv<T, V>(rot + V + m, t0);
                    ldv<T, V>(rot + P + V + m, t1);
                    cn_row<T, V>(oa, ob, db_d, db_u, da_u, da_d, D.cc, n == 1 ? (T)2 : (T)1, sR[il + 1], gc,
                                 sN[il + 1], t0, t1, cn, an, bn);
                }
                /* b_0 = 0 (Eq. b_boundary); columns past m = M stay zero */
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const bool in = m + e < Wb;
                    an[e] = in ? an[e] : (T)0;
                    bn[e] = (in && n > 0) ? bn[e] : (T)0;
                }
                stv<T, V>(po, an);
                stv<T, V>(po + arr, bn);
                /* what the neighbouring blocks read in the next half-step */
                if (il == 0 && bi > 0) {
#pragma unroll
                    for (int q = 0; q < V; ++q)
                        if (m + q < Wb) publish<T>(top + rs + (m + q) * E, tag + 1, an[q], bn[q]);
                }
                if (il == R - 1 && bi + 1 < A.GR) {
#pragma unroll
                    for (int q = 0; q < V; ++q)
                        if (m + q < Wb) publish<T>(bottom + rs + (m + q) * E, tag + 1, an[q], bn[q]);
                }
                if (g == 0 && bj > 0) publish<T>(left + cs + il * E, tag + 1, an[0], bn[0]);
                if (g == ncg - 1 && bj + 1 < A.GC) publish<T>(right + cs + il * E, tag + 1, an[V - 1], bn[V - 1]);
            }
        }
        D = Dn;
        __syncthreads();
    }

    /* ---- the block's final state (ghost columns of the arrays stay zero) ---- */
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        T* g = gs[a] + GG + c0;
        const T* d = s + a * arr + V;
        for (int q = tid; q < R * ncg; q += nthr) {
            const int li = q / ncg, gq = q - li * ncg;
            T v[V];
            ldv<T, V>(d + (li + 1) * P + gq * V, v);
            stv<T, V>(g + (size_t)(r0 + li) * A.pitch + gq * V, v);
        }
    }
}

/* sum of group gq (32 V columns from gq * 32 V) of a row, in every lane */
template <typename T, int V>
__device__ __forceinline__ double group_sum(const T* r, int gq, int M, int lane) {
    const long long m = ((long long)gq * 32 + lane) * V;
    double v = 0.0;
#pragma unroll
    for (int e = 0; e < V; ++e)
        if (m + e <= M) v += (double)r[m + e];
    return warp_sum(v);
}

/* Drift velocity and norm of steps base+1 .. base+K from the rows kept by
 * grid_kernel (CTA i: step base+1+i), added in the order of the one launch
 * per step kernel: lane l of a warp takes V consecutive columns in turn, the
 * warp's lanes a shuffle tree, then the warps of a tile_m tile, then the
 * tiles.  Warps here take the 32 V-column groups round robin; at most
 * kFoldGroups groups (wider rows: the two kernels below). */
template <typename T, int V>
__global__ void fold_rows_kernel(const T* rows, int mpad, int M, int tile_m, double vscale, double nscale,
                                 const long long* base, double* trace_v, double* trace_n) {
    __shared__ double part[2 * kFoldGroups];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int per_tile = tile_m / (32 * V), ntx = (M + tile_m) / tile_m, ng = ntx * per_tile;
    for (int q = warp; q < 2 * ng; q += nwarp) {
        const int which = q >= ng, gq = which ? q - ng : q;
        const double v = group_sum<T, V>(rows + ((size_t)blockIdx.x * 2 + which) * mpad, gq, M, lane);
        if (lane == 0) part[q] = v;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const double* p = part + threadIdx.x * ng;
        double sum = 0.0;
        for (int t = 0; t < ntx; ++t) {
            double st = 0.0;
            for (int w = 0; w < per_tile; ++w) st += p[t * per_tile + w];
            sum += st;
        }
        const long long slot = *base + 1 + blockIdx.x;
        if (threadIdx.x == 0) trace_n[slot] = nscale * sum;
        else trace_v[slot] = vscale * sum;
    }
}

/* The same for rows of any width: the sums of the tiles, kFoldTileGroups
 * groups per CTA (blockIdx.y: step), then the tiles of a step in order (one
 * warp per row, 32 tiles loaded at a time).  A row that one CTA walks takes
 * as long as the row is wide, however few steps there are to share the SMs
 * (us per step with one CTA per step / so: 2 x 60001 FP32 44 / 15, 2 x 160001
 * FP32 106 / 20, FP64 173 / 49; two steps per launch, 8 x 350000: 247 / 29). */
template <typename T, int V>
__global__ void __launch_bounds__(256) fold_tiles_kernel(const T* rows, int mpad, int M, int tile_m, double* tsum) {
    __shared__ double part[2 * kFoldTileGroups];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int per_tile = tile_m / (32 * V), ntx = (M + tile_m) / tile_m;
    const int tpb = kFoldTileGroups / per_tile, t0 = (int)blockIdx.x * tpb, nt = min(tpb, ntx - t0);
    const int ng = nt * per_tile;
    for (int q = warp; q < 2 * ng; q += nwarp) {
        const int which = q >= ng, gq = which ? q - ng : q;
        const double v =
            group_sum<T, V>(rows + ((size_t)blockIdx.y * 2 + which) * mpad, t0 * per_tile + gq, M, lane);
        if (lane == 0) part[q] = v;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * nt; q += blockDim.x) {
        const int which = q >= nt, t = which ? q - nt : q;
        const double* p = part + which * ng + t * per_tile;
        double st = 0.0;
        for (int w = 0; w < per_tile; ++w) st += p[w];
        tsum[((size_t)blockIdx.y * 2 + which) * ntx + t0 + t] = st;
    }
}

__global__ void __launch_bounds__(64) fold_tail_kernel(const double* tsum, int ntx, double vscale, double nscale,
                                                       const long long* base, double* trace_v, double* trace_n) {
    const int lane = threadIdx.x & 31, which = threadIdx.x >> 5;
    const double* p = tsum + ((size_t)blockIdx.x * 2 + which) * ntx;
    double sum = 0.0, next = lane < ntx ? p[lane] : 0.0;
    for (int t = 0; t < ntx; t += 32) {
        const double v = next;
        next = t + 32 + lane < ntx ? p[t + 32 + lane] : 0.0;
        const int n = min(32, ntx - t);
        for (int i = 0; i < n; ++i) sum += __shfl_sync(0xffffffffu, v, i);
    }
    if (lane != 0) return;
    const long long slot = *base + 1 + blockIdx.x;
    if (which == 0) trace_n[slot] = nscale * sum;
    else trace_v[slot] = vscale * sum;
}

template <typename T>
const void* grid_fn(int vec) {
    if constexpr (sizeof(T) == 4)
        return vec == 4   ? reinterpret_cast<const void*>(&grid_kernel<float, 4>)
               : vec == 2 ? reinterpret_cast<const void*>(&grid_kernel<float, 2>)
                          : reinterpret_cast<const void*>(&grid_kernel<float, 1>);
    else
        return reinterpret_cast<const void*>(&grid_kernel<double, 1>);
}

}  // namespace

template <typename T>
size_t grid_smem_bytes(int R, int W, int vec) {
    const size_t groups = (size_t)(W + vec - 1) / vec;
    return poll_offset<T>(R, W, vec) + 2 * (size_t)(W + 2 + R) * 8 + 2 * (groups + R) * 4;
}

template <typename T>
int grid_configure(int vec, size_t smem, int threads, int* blocks_per_sm) {
    const void* fn = grid_fn<T>(vec);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, threads, smem);
}

template <typename T>
int launch_grid(const GridArgs<T>& a, int vec, int threads, size_t smem, void* stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.GR * a.GC);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative; /* all CTAs resident at once */
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[1] = {const_cast<GridArgs<T>*>(&a)};
    return (int)cudaLaunchKernelExC(&cfg, grid_fn<T>(vec), args);
}

size_t fold_scratch_bytes(int M, int tile_m, int vec, int K) {
    const size_t ntx = ((size_t)M + tile_m) / tile_m;
    return ntx * (tile_m / (32 * vec)) > (size_t)kFoldGroups ? (size_t)K * 2 * ntx * sizeof(double) : 0;
}

template <typename T>
int launch_fold_rows(const T* rows, int mpad, int M, int tile_m, int vec, int K, double vscale, double nscale,
                     const long long* base, double* trace_v, double* trace_n, double* tsum, void* stream) {
    constexpr int V = sizeof(T) == 4 ? 4 : 2;
    cudaStream_t st = (cudaStream_t)stream;
    if (vec != V || tile_m % (32 * V) || tile_m / (32 * V) > kFoldTileGroups) return (int)cudaErrorInvalidValue;
    if (fold_scratch_bytes(M, tile_m, vec, K) == 0) {
        fold_rows_kernel<T, V><<<K, 256, 0, st>>>(rows, mpad, M, tile_m, vscale, nscale, base, trace_v, trace_n);
    } else {
        const int ntx = (int)(((long long)M + tile_m) / tile_m), tpb = kFoldTileGroups / (tile_m / (32 * V));
        fold_tiles_kernel<T, V><<<dim3((ntx + tpb - 1) / tpb, K), 256, 0, st>>>(rows, mpad, M, tile_m, tsum);
        fold_tail_kernel<<<K, 64, 0, st>>>(tsum, ntx, vscale, nscale, base, trace_v, trace_n);
    }
    return (int)cudaGetLastError();
}

#define BTE_GRID_INSTANTIATE(T)                                                                          \
    template size_t grid_smem_bytes<T>(int, int, int);                                                   \
    template int grid_configure<T>(int, size_t, int, int*);                                              \
    template int launch_grid<T>(const GridArgs<T>&, int, int, size_t, void*);                            \
    template int launch_fold_rows<T>(const T*, int, int, int, int, int, double, double, const long long*, \
                                     double*, double*, double*, void*);
BTE_GRID_INSTANTIATE(float)
BTE_GRID_INSTANTIATE(double)

}  // namespace bte
