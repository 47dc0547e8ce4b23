// Unified initialization (Algorithm 2) with the clipping strategies of
// App. E.2 and the general alternating update of Algorithm 3: one lane per
// group for g <= 256 (init_lane_kernel), one warp per group for larger groups
// and few groups of 256 (init_kernel, see run_init); the group's transformed
// weights x kept in shared memory.  Runs once before training; not on the
// per-step path.  A round of the alternating update that moves no code (and not
// z_B) is a fixed point: the remaining rounds are skipped, which changes nothing.
//
// Sums that feed alpha and z_B are those of fp64 (the group's fp32 values are
// summed exactly in practice; the lanes' fast path forms the same bits from
// integers); the normal equations C^T C alpha = C^T (x - z_B) have an integer
// matrix, so singularity is decided exactly by an integer determinant and the
// system is solved in fp64 by Gaussian elimination with partial pivoting.
#pragma once

#include "uq_common.cuh"
#include "uq_launch.h"

namespace uq {

constexpr int kInitMaxWarps = 8;

template <int Q>
struct InitTab {
    static constexpr int L = 1 << Q;
    float lv[L];
    float srt[L];
    uint8_t cor[L];
};

// Sorted levels of (a, zb) into registers of every lane (via the warp's table).
template <int Q>
__device__ __forceinline__ void sorted_levels(InitTab<Q>& tb, int lane, const float a[Q], float zb,
                                              float srt[1 << Q]) {
    constexpr int L = 1 << Q;
    __syncwarp();
    if (lane < L) tb.lv[lane] = level_of<Q>(lane, a, zb);
    __syncwarp();
    if (lane < L) {
        const float v = tb.lv[lane];
        int r = 0;
#pragma unroll
        for (int c2 = 0; c2 < L; ++c2) {
            const float v2 = tb.lv[c2];
            r += (v2 < v) || (v2 == v && c2 < lane);
        }
        tb.srt[r] = v;
        tb.cor[r] = static_cast<uint8_t>(lane);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < L; ++r) srt[r] = tb.srt[r];
}

// Exact singularity test of the integer matrix C^T C.  C^T C is a Gram
// matrix of +-1 columns, so |det| <= g^q <= 2^60 (Hadamard); the cofactor
// expansion below is evaluated with wrapping 64-bit unsigned arithmetic,
// which is exact modulo 2^64 and hence exact.
template <int Q>
__device__ __forceinline__ bool int_singular(const long long Min[Q][Q]) {
    using u64 = unsigned long long;
    u64 M[Q][Q];
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int j = 0; j < Q; ++j) M[i][j] = (u64)Min[i][j];
    auto det3 = [&](int r0, int r1, int r2, int c0, int c1, int c2) -> u64 {
        return M[r0][c0] * (M[r1][c1] * M[r2][c2] - M[r1][c2] * M[r2][c1])
             - M[r0][c1] * (M[r1][c0] * M[r2][c2] - M[r1][c2] * M[r2][c0])
             + M[r0][c2] * (M[r1][c0] * M[r2][c1] - M[r1][c1] * M[r2][c0]);
    };
    u64 det;
    if constexpr (Q == 1) {
        det = M[0][0];
    } else if constexpr (Q == 2) {
        det = M[0][0] * M[1][1] - M[0][1] * M[1][0];
    } else if constexpr (Q == 3) {
        det = det3(0, 1, 2, 0, 1, 2);
    } else {
        det = M[0][0] * det3(1, 2, 3, 1, 2, 3) - M[0][1] * det3(1, 2, 3, 0, 2, 3)
            + M[0][2] * det3(1, 2, 3, 0, 1, 3) - M[0][3] * det3(1, 2, 3, 0, 1, 2);
    }
    return det == 0ull;
}

// Solves A x = b in fp64: Gaussian elimination with partial pivoting (first
// largest |pivot| wins) and back substitution, every product and difference
// rounded separately (no FMA contraction).  The exact solution is often an
// fp32 rounding tie (short dyadic values), so the rounding order is fixed.
template <int Q>
__device__ __forceinline__ void solve_fp64(const long long Ain[Q][Q], const double bin[Q], double x[Q]) {
    double A[Q][Q], b[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        b[i] = bin[i];
#pragma unroll
        for (int j = 0; j < Q; ++j) A[i][j] = (double)Ain[i][j];
    }
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        int p = k;
        double piv = fabs(A[k][k]);
#pragma unroll
        for (int i = k + 1; i < Q; ++i)
            if (fabs(A[i][k]) > piv) { piv = fabs(A[i][k]); p = i; }
#pragma unroll
        for (int i = k + 1; i < Q; ++i) {
            if (i == p) {
#pragma unroll
                for (int j = 0; j < Q; ++j) { const double tmp = A[k][j]; A[k][j] = A[i][j]; A[i][j] = tmp; }
                const double tb = b[k]; b[k] = b[i]; b[i] = tb;
            }
        }
#pragma unroll
        for (int i = k + 1; i < Q; ++i) {
            const double f = __ddiv_rn(A[i][k], A[k][k]);
#pragma unroll
            for (int j = k; j < Q; ++j) A[i][j] = __dsub_rn(A[i][j], __dmul_rn(f, A[k][j]));
            b[i] = __dsub_rn(b[i], __dmul_rn(f, b[k]));
        }
    }
#pragma unroll
    for (int i = Q - 1; i >= 0; --i) {
        double s = b[i];
#pragma unroll
        for (int j = i + 1; j < Q; ++j) s = __dsub_rn(s, __dmul_rn(A[i][j], x[j]));
        x[i] = __ddiv_rn(s, A[i][i]);
    }
}

template <int Q, typename WT>
__global__ void init_kernel(const void* __restrict__ W, int64_t n_groups, int n_in, int g, int G, int T, int clip,
                            float* __restrict__ DELTA, float* __restrict__ ZU, float* __restrict__ S,
                            float* __restrict__ SR, float* __restrict__ ALPHA, float* __restrict__ ZB,
                            uint8_t* __restrict__ CODES) {
    constexpr int L = 1 << Q;
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpc = blockDim.x >> 5;
    __shared__ InitTab<Q> tabs[kInitMaxWarps];
    InitTab<Q>& tb = tabs[warp];
    float* xs = reinterpret_cast<float*>(smem) + (size_t)warp * g;
    uint8_t* cs = smem + (size_t)wpc * g * sizeof(float) + (size_t)warp * g;

    const int64_t grp = (int64_t)blockIdx.x * wpc + warp;
    if (grp >= n_groups) return;                       // whole warp; no block barrier follows
    const int Gr = n_in / g;
    const int64_t row = grp / Gr;
    const int64_t eoff = row * (int64_t)n_in + (grp % Gr) * (int64_t)g;
    auto wval = [&](int i) -> float {
        if constexpr (sizeof(typename WT::raw) == sizeof(float4))
            return __ldg(static_cast<const float*>(W) + eoff + i);
        else
            return __uint_as_float(uint32_t(__ldg(static_cast<const unsigned short*>(W) + eoff + i)) << 16);
    };

    float wmin = INFINITY, wmax = -INFINITY;
    for (int i = lane; i < g; i += 32) {
        const float w = wval(i);
        wmin = fminf(wmin, w);
        wmax = fmaxf(wmax, w);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        wmin = fminf(wmin, __shfl_xor_sync(kFull, wmin, off));
        wmax = fmaxf(wmax, __shfl_xor_sync(kFull, wmax, off));
    }
    const float top = (float)(L - 1);
    const float rng = fmaxf(__fsub_rn(wmax, wmin), 1e-12f);

    double e_best = INFINITY;
    float bd = 0.f, bz = 0.f, bzb = top * 0.5f, ba[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) ba[j] = 0.f;

    for (int gi = 1; gi <= G; ++gi) {
        const float gamma = __fdiv_rn((float)gi, (float)G);
        const float dc = __fdiv_rn(__fmul_rn(gamma, rng), top);
        float zc;
        if (clip == UQ_CLIP_FIXED_MIN) zc = __fdiv_rn(-wmin, dc);
        else if (clip == UQ_CLIP_FIXED_MAX) zc = __fsub_rn(top, __fdiv_rn(wmax, dc));
        else zc = __fdiv_rn(-__fmul_rn(gamma, wmin), dc);
        __syncwarp();
        for (int i = lane; i < g; i += 32) {
            float u;
            xs[i] = transform_x(wval(i), 1.f, dc, 1.f, zc, u);
            cs[i] = 0;
        }
        __syncwarp();

        // --- Algorithm 3: greedy start (one bit at a time) ---
        float a[Q], zb = bzb;
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            double sabs = 0.0;
            for (int i = lane; i < g; i += 32) {
                float r = __fsub_rn(xs[i], zb);
                const int c = cs[i];
#pragma unroll
                for (int jj = 0; jj < j; ++jj) r = __fsub_rn(r, ((c >> jj) & 1) ? a[jj] : -a[jj]);
                sabs += (double)fabsf(r);
                if (r >= 0.f) cs[i] = (uint8_t)(c | (1 << j));
            }
            sabs = warp_sum_d(sabs);
            a[j] = (float)(sabs / (double)g);
        }
        __syncwarp();

        // --- T rounds of alpha, C (and z_B when G == 1) ---
        for (int it = 0; it < T; ++it) {
            long long ctc[Q][Q];
            double cty[Q];
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                cty[j] = 0.0;
#pragma unroll
                for (int k = 0; k < Q; ++k) ctc[j][k] = 0;
            }
            const double zbd = (double)zb;
            for (int i = lane; i < g; i += 32) {
                const int c = cs[i];
                const double y = (double)xs[i] - zbd;
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    const int sj = ((c >> j) & 1) ? 1 : -1;
                    cty[j] += sj > 0 ? y : -y;
#pragma unroll
                    for (int k = j; k < Q; ++k) ctc[j][k] += (((c >> k) & 1) ? 1 : -1) * sj;
                }
            }
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                cty[j] = warp_sum_d(cty[j]);
#pragma unroll
                for (int k = j; k < Q; ++k) {
                    long long v = ctc[j][k];
#pragma unroll
                    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
                    ctc[j][k] = v;
                    ctc[k][j] = v;
                }
            }
            if (!int_singular<Q>(ctc)) {
                double sol[Q];
                solve_fp64<Q>(ctc, cty, sol);
#pragma unroll
                for (int j = 0; j < Q; ++j) a[j] = (float)sol[j];
            }
            float srt[L];
            sorted_levels<Q>(tb, lane, a, zb, srt);
            bool moved = false;
            for (int i = lane; i < g; i += 32) {
                float m;
                const int r = nearest_rank<L>(xs[i], srt, m);
                moved |= cs[i] != tb.cor[r];
                cs[i] = tb.cor[r];
            }
            moved = __any_sync(kFull, moved);
            __syncwarp();
            const float zb_prev = zb;
            if (G == 1) {
                double sres = 0.0;
                for (int i = lane; i < g; i += 32) {
                    const int c = cs[i];
                    double ca = 0.0;
#pragma unroll
                    for (int j = 0; j < Q; ++j) ca += ((c >> j) & 1) ? (double)a[j] : -(double)a[j];
                    sres += (double)xs[i] - ca;
                }
                sres = warp_sum_d(sres);
                zb = (float)(sres / (double)g);
            }
            // a fixed point (no code and not z_B moved): the remaining rounds
            // would repeat it bit for bit (warp-uniform: zb and moved are)
            if (!moved && __float_as_uint(zb) == __float_as_uint(zb_prev)) break;
        }

        // --- candidate error with the full mapping (Eq. 2), s = s_r = 1 ---
        float srt[L];
        sorted_levels<Q>(tb, lane, a, zb, srt);
        double e = 0.0;
        for (int i = lane; i < g; i += 32) {
            float m;
            nearest_rank<L>(xs[i], srt, m);
            const float what = __fmul_rn(dc, __fsub_rn(m, zc));
            const double df = (double)wval(i) - (double)what;
            e += df * df;
        }
        e = warp_sum_d(e);
        if (e < e_best) {
            e_best = e;
            bd = dc;
            bz = zc;
            bzb = zb;
#pragma unroll
            for (int j = 0; j < Q; ++j) ba[j] = a[j];
        }
    }

    if (lane == 0) {
        DELTA[grp] = bd;
        ZU[grp] = bz;
        ZB[grp] = bzb;
#pragma unroll
        for (int j = 0; j < Q; ++j) ALPHA[grp * Q + j] = ba[j];
        if (grp % Gr == 0) SR[row] = 1.f;
    }
    float srt[L];
    sorted_levels<Q>(tb, lane, ba, bzb, srt);
    for (int i = lane; i < g; i += 32) {
        float u, m;
        const float x = transform_x(wval(i), 1.f, bd, 1.f, bz, u);
        const int r = nearest_rank<L>(x, srt, m);
        CODES[eoff + i] = tb.cor[r];
        S[eoff + i] = 1.f;
    }
}

// ---------------------------------------------------------------------------
// One lane per group (g <= 256)
// ---------------------------------------------------------------------------
//
// The same computation as init_kernel, laid out for a GPU whose fp64 rate is
// a small fraction of its fp32 rate (1.8 fused operations per clock and SM
// measured): lane l of a warp owns group 32 w + l whole, so no sum needs a
// shuffle and each group's normal equations are solved once.  During the T
// rounds x is fixed and only the code words move, so C^T (x - z_B) and C^T C
// are formed from per-code-word sums of x and counts (fp64 path: kept over the
// rounds, an element whose code moves goes from one sum to the other).  Shared
// memory per warp, element-major so that the 32 lanes touch consecutive words
// (init_lane_warp_bytes).
//
// The fast path of a candidate works on the group's weights in ascending order
// (sorted once, kept in the group's part of the output S until the end): x is
// then ascending too, so the codes of a round are intervals of positions
// between L - 1 boundaries, a round finds the boundaries by binary search and
// forms its sums from prefix sums of x, and no element is touched.  Its values
// are those of the fp64 path:
//  * sums of |r| and x: with all values multiples of 2^-k below 2^44 2^-k
//    (k per group and candidate; every value is checked), the fp64 sums are
//    exact in any order, and so are 64-bit integer sums;
//  * the normal equations: the exact solution N_j / D from integers (Cramer's
//    rule), rounded to fp32 only where it lies further from a tie of that
//    rounding than the fp64 elimination can be off (see below), else the
//    elimination;
//  * the nearest level: with X the largest |x|, M the largest |level| and every
//    gap of distinct levels above 2^-21 (X + M), the test fl|x - l_{r+1}| <
//    fl|x - l_r| of neighbouring levels is false below the two, true above
//    them (the gap survives the rounding) and monotonic between them, since
//    rounding is; so it is monotonic in x and decides between ranks up to r
//    and above exactly as the scan does.  Equal levels: the scan takes the
//    lowest of their ranks, the others get no element;
//  * the candidate's error: an fp32 sum, and the fp64 sums of the candidate
//    and the kept one only where the two fp32 sums are within their bound.
// Where a value is no such multiple, levels are too close, or z_B moves (G =
// 1), the warp takes the fp64 path for the candidate.  So every output is bit
// for bit what fp64 gives.  1024 x 4096, q = 3, g = 128, G = 30, T = 15:
// 15.8 -> 3.5 ms, with the same shape at q = 2 2.0, q = 4 10.2 and g = 64 5.6
// ms.  (Rounds that moved element by element instead of boundaries: 8.8 ms,
// 5.6, 16.3 and 7.1; without the sort network of lane_sorted_levels and with g
// at run time 3.9 ms.)  Bound by issue and latency: 7 warps per SM, as many
// as this matrix has groups for and nearly as many as fit in shared memory.
constexpr int kLaneInitMaxG = 256;
// Warps of a block: with the fast path 12 (170 registers a thread), without (G = 1) 16.
constexpr int lane_init_max_warps(bool fast) { return fast ? 12 : 16; }

// Shared memory of one warp: x [g][32], then the prefix sums of x before every
// fourth element [g / 4][32] (64 bits) or, on the fp64 path, the per-code sums
// of x [L][32] (fp64) and the code words [g][32].
__host__ __device__ constexpr size_t init_lane_aux_bytes(int q, int g, bool fast) {
    const size_t slow = (size_t)g * 32 + ((size_t)256 << q);
    return fast && (size_t)g * 64 > slow ? (size_t)g * 64 : slow;
}
__host__ __device__ constexpr size_t init_lane_warp_bytes(int q, int g, bool fast) {
    return (size_t)g * 128 + init_lane_aux_bytes(q, g, fast);
}

// Counts of the L code words of one group, 16 bits per code word packed in
// 64-bit registers; c is a compile-time index wherever get() is used, add()
// takes any c.
template <int L>
struct CodeHist {
    static constexpr int BITS = 16, PER = 64 / BITS, NW = (L + PER - 1) / PER;
    uint64_t h[NW];
    __device__ __forceinline__ CodeHist() {
#pragma unroll
        for (int i = 0; i < NW; ++i) h[i] = 0;
    }
    __device__ __forceinline__ void add(int c, int d) {
        const uint64_t v = (uint64_t)(int64_t)d << (BITS * (c % PER));
#pragma unroll
        for (int i = 0; i < NW; ++i) h[i] += (NW == 1 || c / PER == i) ? v : 0ull;
    }
    __device__ __forceinline__ int get(int c) const {
        return (int)((h[c / PER] >> (BITS * (c % PER))) & ((1ull << BITS) - 1));
    }
};

// Levels of (a, zb), sorted ascending (ties by code word); cor holds the code word of rank r in bits 4 r .. 4 r + 3, that of
// the lowest rank among equal levels (the one nearest_rank takes).
template <int Q>
__device__ __forceinline__ void lane_sorted_levels(const float a[Q], float zb, float srt[1 << Q], uint64_t& cor) {
    constexpr int L = 1 << Q;
    int code[L];
#pragma unroll
    for (int c = 0; c < L; ++c) {
        srt[c] = level_of<Q>(c, a, zb);
        code[c] = c;
    }
    // Batcher's odd-even merge sort (19 exchanges of eight levels, 63 of sixteen)
#pragma unroll
    for (int p = 1; p < L; p *= 2)
#pragma unroll
        for (int k = p; k >= 1; k /= 2)
#pragma unroll
            for (int i = 0; i < L; ++i)
                if (i >= k % p && (i - k % p) % (2 * k) < k && i + k < L && i / (2 * p) == (i + k) / (2 * p)) {
                    const float u = srt[i], v = srt[i + k];
                    const int cu = code[i], cv = code[i + k];
                    const bool swap = v < u || (v == u && cv < cu);
                    srt[i] = swap ? v : u;
                    srt[i + k] = swap ? u : v;
                    code[i] = swap ? cv : cu;
                    code[i + k] = swap ? cu : cv;
                }
    cor = (uint64_t)code[0];
    int first = code[0];
#pragma unroll
    for (int r = 1; r < L; ++r) {
        first = srt[r] == srt[r - 1] ? first : code[r];
        cor |= (uint64_t)first << (4 * r);
    }
}

// Exact solution of C^T C alpha = b as integers: N_j / D (D = det, N = adj b),
// N_j rounded to fp64 once.  n[i][j] (|n| <= g <= 128) and D fit 32 bits, adj
// 24; |b| < 2^53, so N_j is formed from two parts of b.
template <int Q>
__device__ __forceinline__ int cramer(const int n[Q][Q], const long long b[Q], double N[Q]) {
    auto det2 = [&](int r0, int r1, int c0, int c1) { return n[r0][c0] * n[r1][c1] - n[r0][c1] * n[r1][c0]; };
    auto det3 = [&](int r0, int r1, int r2, int c0, int c1, int c2) {
        return n[r0][c0] * det2(r1, r2, c1, c2) - n[r0][c1] * det2(r1, r2, c0, c2) + n[r0][c2] * det2(r1, r2, c0, c1);
    };
    int adj[Q][Q];                                          // symmetric, as n is
    if constexpr (Q == 1) {
        adj[0][0] = 1;
    } else if constexpr (Q == 2) {
        adj[0][0] = n[1][1]; adj[1][1] = n[0][0]; adj[0][1] = adj[1][0] = -n[0][1];
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i)
#pragma unroll
            for (int j = i; j < Q; ++j) {
                int rr[Q - 1], cc[Q - 1];
#pragma unroll
                for (int k = 0; k < Q - 1; ++k) { rr[k] = k < i ? k : k + 1; cc[k] = k < j ? k : k + 1; }
                int d;
                if constexpr (Q == 3) d = det2(rr[0], rr[1], cc[0], cc[1]);
                else d = det3(rr[0], rr[1], rr[2], cc[0], cc[1], cc[2]);
                adj[i][j] = adj[j][i] = ((i + j) & 1) ? -d : d;
            }
    }
    int D = 0;
#pragma unroll
    for (int j = 0; j < Q; ++j) D += n[0][j] * adj[0][j];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        long long lo = 0, hi = 0;
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            lo += (long long)adj[i][j] * (b[j] & 0x3ffffff);
            hi += (long long)adj[i][j] * (b[j] >> 26);
        }
        hi += lo >> 26;                                     // |hi| < 2^53
        N[i] = fma((double)hi, 0x1p26, (double)(lo & 0x3ffffff));
    }
    return D;
}

// FAST: the fast path is compiled in (G > 1).
template <int Q, typename WT, int G_, bool FAST>
__global__ void __launch_bounds__(lane_init_max_warps(FAST) * 32, 1)
    init_lane_kernel(const void* __restrict__ W, int64_t n_groups, int n_in, int G, int T, int clip,
                     float* __restrict__ DELTA, float* __restrict__ ZU, float* S, float* __restrict__ SR,
                     float* __restrict__ ALPHA, float* __restrict__ ZB, uint8_t* __restrict__ CODES) {
    constexpr int g = G_, L = 1 << Q;
    constexpr size_t WARP_BYTES = init_lane_warp_bytes(Q, g, FAST);
    constexpr bool CRAMER = g <= 128;                                   // where the 32-bit determinant holds
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* base = smem + (size_t)warp * WARP_BYTES;
    float* xs = reinterpret_cast<float*>(base);                         // [g][32]
    unsigned char* aux = base + (size_t)g * 128;
    long long* pf = reinterpret_cast<long long*>(aux);                  // [g / 4][32]
    double* bx = reinterpret_cast<double*>(aux);                        // [L][32]
    uint8_t* cs = aux + (size_t)L * 256;                                // [g][32]

    const int64_t grp0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 32;
    if (grp0 >= n_groups) return;                      // whole warp; no block barrier in this kernel
    const int64_t grp_raw = grp0 + lane;
    const bool live = grp_raw < n_groups;
    const int64_t grp = live ? grp_raw : n_groups - 1; // absent lanes repeat the last group, store nothing of their own
    const int Gr = n_in / g;
    const int64_t row = grp / Gr;
    const int64_t eoff = row * (int64_t)n_in + (grp % Gr) * (int64_t)g;
    float* ws = S + eoff;                              // the sorted weights until the end
    auto w4 = [&](int i, float (&w)[4]) { WT::unpack(WT::load(W, eoff + i), w); };
    auto X = [&](int i) -> float& { return xs[i * 32 + lane]; };
    auto C = [&](int i) -> uint8_t& { return cs[i * 32 + lane]; };
    auto BX = [&](int c) -> double& { return bx[c * 32 + lane]; };
    const float inf = __int_as_float(0x7f800000), rg = 1.f / (float)g;    // exact: g is a power of two

    float wmin = INFINITY, wmax = -INFINITY;
    bool finite = true;
    for (int i = 0; i < g; i += 4) {
        float w[4];
        w4(i, w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            wmin = fminf(wmin, w[k]);
            wmax = fmaxf(wmax, w[k]);
            finite &= fabsf(w[k]) < inf;
            X(i + k) = w[k];
        }
    }
    const float top = (float)(L - 1);
    const float rng = fmaxf(__fsub_rn(wmax, wmin), 1e-12f);
    // the group's weights in ascending order (bitonic network), into ws, where the fast path may be taken
    const bool sorted = FAST && __all_sync(kFull, finite);
#pragma unroll 1
    for (int k = sorted ? 2 : 2 * g; k <= g; k *= 2)
#pragma unroll 1
        for (int j = k / 2; j >= 1; j /= 2)
#pragma unroll 4
            for (int p = 0; p < g / 2; ++p) {
                const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                const float u = X(i), v = X(i + j);
                const bool swap = (u > v) == ((i & k) == 0);
                X(i) = swap ? v : u;
                X(i + j) = swap ? u : v;
            }
#pragma unroll 4
    for (int i = sorted ? 0 : g; i < g; i += 4)
        *reinterpret_cast<float4*>(ws + i) = make_float4(X(i), X(i + 1), X(i + 2), X(i + 3));
    auto ws4 = [&](int i, float (&w)[4]) { f4_to(*reinterpret_cast<const float4*>(ws + i), w); };

    // The kept candidate, its fp32 error (ef) and its fp64 error (ed, where
    // have_ed); before the first one ed = infinity.
    double ed = INFINITY;
    float ef = inf;
    bool have_ed = true;
    float bd = 0.f, bz = 0.f, bzb = top * 0.5f, ba[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) ba[j] = 0.f;
    float srt[L];
    uint64_t cor;

    // fp64 error of a candidate from its own parameters (the values of init_kernel, in the same order)
    auto error64 = [&](float dc, float zc, const float (&a)[Q], float zb) {
        float sv[L];
        uint64_t unused;
        lane_sorted_levels<Q>(a, zb, sv, unused);
        double e = 0.0;
#pragma unroll 1
        for (int i = 0; i < g; i += 4) {
            float w[4];
            w4(i, w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float u, m;
                nearest_rank<L>(transform_x(w[k], 1.f, dc, 1.f, zc, u), sv, m);
                const double df = (double)w[k] - (double)__fmul_rn(dc, __fsub_rn(m, zc));
                e += df * df;
            }
        }
        return e;
    };

    // The fp64 elimination (alpha stays where C^T C is singular).
    auto solve64 = [&](const int (&ctc)[Q][Q], const double (&cty)[Q], float (&a)[Q]) {
        long long n64[Q][Q];
#pragma unroll
        for (int j = 0; j < Q; ++j)
#pragma unroll
            for (int k = 0; k < Q; ++k) n64[j][k] = ctc[j][k];
        if (!int_singular<Q>(n64)) {
            double sol[Q];
            solve_fp64<Q>(n64, cty, sol);
#pragma unroll
            for (int j = 0; j < Q; ++j) a[j] = (float)sol[j];
        }
    };

    // A candidate's alpha and fp32 error on the fast path.  Whole warp; false
    // (for every lane) where some lane's group cannot take it.
    auto fast = [&](float dc, float zc, float zb, float (&a)[Q], float& err) -> bool {
        float u;
        const float x0 = transform_x(wmin, 1.f, dc, 1.f, zc, u), x1 = transform_x(wmax, 1.f, dc, 1.f, zc, u);
        const float xmax = fmaxf(fabsf(x0), fabsf(x1));
        // Fixed point: values below 2^e in units of 2^-k, k = 44 - e (sums of 256 stay below 2^53;
        // with 30 bits groups with outliers fail, and the fp64 path of a few makes the kernel last
        // 9.6 ms where it takes 3.5).
        const float bound = xmax + fabsf(zb);
        const int ebits = (int)((__float_as_uint(bound) >> 23) & 0xffu) - 126;      // bound < 2^ebits
        const int kfix = 44 - ebits;
        bool ok = x0 == x0 && x1 == x1 && bound < 0x1p60f && bound > 0x1p-60f;
        const float up = ok ? __int_as_float((127 + kfix) << 23) : 1.f, down = ok ? __int_as_float((127 - kfix) << 23) : 1.f;
        // v in units of 2^-k, ok left set only where it is a multiple of it: the
        // leading 20 bits and the rest, both exact.  (The 64-bit conversions run
        // at the fp64 rate.)
        const float up_hi = up * 0x1p-24f, down_hi = down * -0x1p24f;
        auto to_fixed = [&](float v) -> long long {
            const int hi = __float2int_rn(v * up_hi);
            const float rest = fmaf((float)hi, down_hi, v) * up;
            const int lo = __float2int_rn(rest);
            ok &= (float)lo == rest && (unsigned)(hi + (1 << 20)) <= 1u << 21;
            return ((long long)hi << 24) + lo;
        };
        const long long zbi = to_fixed(zb);
        if (!__all_sync(kFull, ok)) return false;

        long long total = 0;
#pragma unroll 2
        for (int i = 0; i < g; i += 4) {
            float w[4];
            ws4(i, w);
            pf[(i >> 2) * 32 + lane] = total;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float x = transform_x(w[k], 1.f, dc, 1.f, zc, u);
                X(i + k) = x;
                total += to_fixed(x);
            }
        }
        // --- Algorithm 3: greedy start (one bit at a time); with the last bit the sums of the first round ---
        long long b[Q];                                     // C^T (x - z_B) in units of 2^-k
        int ctc[Q][Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) b[j] = 0;
        uint32_t diff[2] = {0u, 0u};                        // elements whose bits j < k differ: 10 bits per pair
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            long long sum = 0;
#pragma unroll 4
            for (int i = 0; i < g; ++i) {
                const float x = X(i);
                float r = __fsub_rn(x, zb);
                int c = 0;
#pragma unroll
                for (int jj = 0; jj < j; ++jj) {
                    const bool s1 = r >= 0.f;
                    c |= s1 ? 1 << jj : 0;
                    r = __fsub_rn(r, s1 ? a[jj] : -a[jj]);
                }
                sum += to_fixed(fabsf(r));
                if (j == Q - 1) {
                    c |= r >= 0.f ? 1 << j : 0;
                    const long long y = to_fixed(x) - zbi;
#pragma unroll
                    for (int jj = 0; jj < Q; ++jj) b[jj] += ((c >> jj) & 1) ? y : -y;
                    int pair = 0;
#pragma unroll
                    for (int jj = 0; jj < Q; ++jj)
#pragma unroll
                        for (int kk = jj + 1; kk < Q; ++kk, ++pair)
                            diff[pair / 3] += (uint32_t)(((c >> jj) ^ (c >> kk)) & 1) << (10 * (pair % 3));
                }
            }
            a[j] = __ll2float_rn(sum) * (down * rg);             // powers of two: exact
        }
        {
            int pair = 0;
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                ctc[j][j] = g;
#pragma unroll
                for (int k = j + 1; k < Q; ++k, ++pair)
                    ctc[j][k] = ctc[k][j] = g - 2 * (int)((diff[pair / 3] >> (10 * (pair % 3))) & 1023u);
            }
        }
        if (!__all_sync(kFull, ok)) return false;

        // Boundaries of the ranks in the sorted x: rank r holds the positions [B[r - 1], B[r]).
        int B[L];
        auto boundaries = [&]() {
            lane_sorted_levels<Q>(a, zb, srt, cor);
            const float M = fmaxf(fabsf(srt[0]), fabsf(srt[L - 1]));
            const float m = (xmax + M) * 0x1p-21f;
            ok &= M < 0x1p100f;                             // false also for NaN
#pragma unroll
            for (int r = 0; r + 1 < L; ++r) {
                const float gap = srt[r + 1] - srt[r];
                ok &= gap == 0.f || gap > m;
                B[r] = 0;
            }
#pragma unroll
            for (int step = g / 2; step >= 1; step /= 2)
#pragma unroll
                for (int r = 0; r + 1 < L; ++r) {
                    const float x = X(B[r] + step - 1);
                    if (!(fabsf(__fsub_rn(x, srt[r + 1])) < fabsf(__fsub_rn(x, srt[r])))) B[r] += step;
                }
#pragma unroll
            for (int r = 0; r + 1 < L; ++r) {
                const float x = X(B[r]);                    // at most g - 1 here
                if (!(fabsf(__fsub_rn(x, srt[r + 1])) < fabsf(__fsub_rn(x, srt[r])))) B[r] += 1;
            }
            B[L - 1] = g;
#pragma unroll
            for (int r = L - 2; r >= 0; --r)
                if (srt[r + 1] == srt[r]) B[r] = B[r + 1];  // the lower of two equal ranks takes all
        };
        // Sum of x before position p.
        auto before = [&](int p) {
            if (p == g) return total;
            long long v = pf[(p >> 2) * 32 + lane];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k < (p & 3)) v += to_fixed(X((p & ~3) + k));
            return v;
        };

        // --- T rounds of alpha and C ---
        bool done = false;
        uint64_t cor_prev = ~uint64_t(0);
        for (int it = 0; it < T; ++it) {
            if (!done) {
                bool solved = false;
                if constexpr (CRAMER) {
                    double N[Q];
                    const int D = cramer<Q>(ctc, b, N);
                    if (D == 0) {
                        solved = true;                      // singular: alpha stays
                    } else {
                        // The elimination's forward error is at most 2^11 u kappa max|alpha| (n <= 4,
                        // growth <= 8; kappa, the condition of the positive definite matrix, from its
                        // trace Q g and determinant), N_j / D as formed here within 2^-51 of itself.
                        const double rd = (double)down / (double)D;
                        double sol[Q];
                        float amax = 0.f, av[Q];
#pragma unroll
                        for (int j = 0; j < Q; ++j) {
                            sol[j] = N[j] * rd;
                            av[j] = (float)sol[j];
                            amax = fmaxf(amax, fabsf(av[j]));
                        }
                        float kappa = (float)(Q * g);
#pragma unroll
                        for (int j = 1; j < Q; ++j) kappa *= (float)(Q * g) / (float)(Q > 1 ? Q - 1 : 1);
                        kappa = __fdividef(kappa, fabsf((float)D));
                        bool sure = amax < 0x1p90f;
#pragma unroll
                        for (int j = 0; j < Q; ++j) {
                            const int off = (int)((uint32_t)__double2loint(sol[j]) & 0x1fffffffu) - (1 << 28);   // from a tie
                            const float need = 2048.f * kappa * __fdividef(amax, fabsf(av[j])) + 16.f;
                            sure &= fabsf(av[j]) > 0x1p-90f && (float)(off < 0 ? -off : off) > need;
                        }
                        if (sure) {
#pragma unroll
                            for (int j = 0; j < Q; ++j) a[j] = av[j];
                            solved = true;
                        }
                    }
                }
                if (!solved) {
                    double cty[Q];
#pragma unroll
                    for (int j = 0; j < Q; ++j) cty[j] = (double)b[j] * (double)down;      // exact
                    solve64(ctc, cty, a);
                }
                int P[L];
#pragma unroll
                for (int r = 0; r < L; ++r) P[r] = it == 0 ? -1 : B[r];
                boundaries();
                // the same intervals and codes as in the round before: a fixed point (every
                // later round would repeat it); a difference in empty ranks only costs a round
                done = cor == cor_prev;
                cor_prev = cor;
#pragma unroll
                for (int r = 0; r < L; ++r) done &= P[r] == B[r];
                if (!done) {
                    long long lo = 0;
                    int n_lo = 0;
#pragma unroll
                    for (int j = 0; j < Q; ++j) {
                        b[j] = 0;
#pragma unroll
                        for (int k = j + 1; k < Q; ++k) ctc[j][k] = 0;
                    }
#pragma unroll
                    for (int r = 0; r < L; ++r) {
                        const long long hi = r == L - 1 ? total : before(B[r]);
                        const int n = B[r] - n_lo, c = (int)((cor >> (4 * r)) & 15u);
                        const long long y = hi - lo - (long long)n * zbi;
                        lo = hi;
                        n_lo = B[r];
#pragma unroll
                        for (int j = 0; j < Q; ++j) {
                            b[j] += ((c >> j) & 1) ? y : -y;
#pragma unroll
                            for (int k = j + 1; k < Q; ++k) ctc[j][k] += (((c >> j) ^ (c >> k)) & 1) ? -n : n;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < Q; ++j)
#pragma unroll
                        for (int k = 0; k < j; ++k) ctc[j][k] = ctc[k][j];
                }
            }
            if (!__all_sync(kFull, ok)) return false;
            if (__all_sync(kFull, done)) break;
        }
        if (T == 0) boundaries();
        if (!__all_sync(kFull, ok)) return false;

        // --- candidate error with the full mapping (Eq. 2), s = s_r = 1: the last round's intervals ---
        float wh[L];
#pragma unroll
        for (int r = 0; r < L; ++r) wh[r] = __fmul_rn(dc, __fsub_rn(srt[r], zc));
        float e4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int i = 0; i < g; i += 4) {
            float w[4];
            ws4(i, w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float h = wh[0];
#pragma unroll
                for (int r = 0; r + 1 < L; ++r) h = i + k >= B[r] ? wh[r + 1] : h;
                const float df = w[k] - h;
                e4[k] = fmaf(df, df, e4[k]);
            }
        }
        err = (e4[0] + e4[1]) + (e4[2] + e4[3]);
        return true;
    };

    // A candidate's alpha and z_B with fp64 sums, element by element in the order of W.
    auto slow = [&](float dc, float zc, float (&a)[Q], float& zb) {
#pragma unroll 1
        for (int i = 0; i < g; i += 4) {
            float w[4];
            w4(i, w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float u;
                X(i + k) = transform_x(w[k], 1.f, dc, 1.f, zc, u);
                C(i + k) = 0;
            }
        }
        // --- Algorithm 3: greedy start (one bit at a time) ---
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            double sabs = 0.0;
#pragma unroll 1
            for (int i = 0; i < g; ++i) {
                float r = __fsub_rn(X(i), zb);
                const int c = C(i);
#pragma unroll
                for (int jj = 0; jj < j; ++jj) r = __fsub_rn(r, ((c >> jj) & 1) ? a[jj] : -a[jj]);
                sabs += (double)fabsf(r);
                if (r >= 0.f) C(i) = (uint8_t)(c | (1 << j));
            }
            a[j] = (float)(sabs / (double)g);
        }
        // Per code word c: the sum of x over the group's elements with code c
        // and their count (hist).  Then C^T (x - z_B) = sum_c s(c) (bx_c - n_c
        // z_B) and C^T C = sum_c n_c s(c) s(c)^T, where s(c) is the sign vector
        // of c; a round only moves the elements whose code changed from one sum
        // to the other.
        CodeHist<L> hist;
#pragma unroll
        for (int c = 0; c < L; ++c) BX(c) = 0.0;
#pragma unroll 1
        for (int i = 0; i < g; ++i) {
            const int c = C(i);
            BX(c) += (double)X(i);
            hist.add(c, 1);
        }
        // --- T rounds of alpha, C (and z_B when G == 1) ---
        for (int it = 0; it < T; ++it) {
            int ctc[Q][Q];
            double cty[Q];
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                cty[j] = 0.0;
#pragma unroll
                for (int k = j; k < Q; ++k) {
                    int v = 0;
#pragma unroll
                    for (int c = 0; c < L; ++c) v += (((c >> j) ^ (c >> k)) & 1) ? -hist.get(c) : hist.get(c);
                    ctc[j][k] = ctc[k][j] = v;
                }
            }
#pragma unroll
            for (int c = 0; c < L; ++c) {
                const double yc = BX(c) - (double)hist.get(c) * (double)zb;
#pragma unroll
                for (int j = 0; j < Q; ++j) cty[j] += ((c >> j) & 1) ? yc : -yc;
            }
            solve64(ctc, cty, a);
            lane_sorted_levels<Q>(a, zb, srt, cor);
            bool moved = false;
#pragma unroll 1
            for (int i = 0; i < g; ++i) {
                float m;
                const float x = X(i);
                const int r = nearest_rank<L>(x, srt, m);
                const int c = (int)((cor >> (4 * r)) & 15u);
                const int old = C(i);
                if (c != old) {
                    moved = true;
                    const double xd = (double)x;
                    BX(old) -= xd;
                    BX(c) += xd;
                    hist.add(old, -1);
                    hist.add(c, 1);
                    C(i) = (uint8_t)c;
                }
            }
            const float zb_prev = zb;
            if (G == 1) {
                // z_B = mean of x - C alpha = sum_c (bx_c - n_c (s(c) . alpha)) / g
                double sres = 0.0;
#pragma unroll
                for (int c = 0; c < L; ++c) {
                    double ca = 0.0;
#pragma unroll
                    for (int j = 0; j < Q; ++j) ca += ((c >> j) & 1) ? (double)a[j] : -(double)a[j];
                    sres += BX(c) - (double)hist.get(c) * ca;
                }
                zb = (float)(sres / (double)g);
            }
            // No code moved (and z_B did not either): the next round would
            // solve the same system, get the same alpha and the same codes, so
            // every remaining round repeats this state bit for bit.
            if (!moved && __float_as_uint(zb) == __float_as_uint(zb_prev)) break;
        }
    };

    for (int gi = 1; gi <= G; ++gi) {
        const float gamma = __fdiv_rn((float)gi, (float)G);
        const float dc = __fdiv_rn(__fmul_rn(gamma, rng), top);
        float zc;
        if (clip == UQ_CLIP_FIXED_MIN) zc = __fdiv_rn(-wmin, dc);
        else if (clip == UQ_CLIP_FIXED_MAX) zc = __fsub_rn(top, __fdiv_rn(wmax, dc));
        else zc = __fdiv_rn(-__fmul_rn(gamma, wmin), dc);
        float a[Q], zb = bzb, e = inf;
        __syncwarp();
        bool found = false;
        if constexpr (FAST) found = sorted && fast(dc, zc, zb, a, e);
        __syncwarp();
        if (!found) {
            e = inf;
            slow(dc, zc, a, zb);                       // (its code words share the prefix sums' memory)
        }
        // The fp32 error is within 2^-23 per square and 2^-24 per addition of
        // the exact sum (at most 66 of them): 5e-6; a square below 2^-126 may be
        // lost, so the sum has to be well above 256 of those.
        const bool usable = e > 0x1p-90f && e < inf;
        bool take;
        if (usable && (e * 1.00001f < ef * 0.99999f) && (ef < inf || !(ed < INFINITY))) {
            take = true;
            have_ed = false;
        } else if (usable && ef < inf && e * 0.99999f > ef * 1.00001f) {
            take = false;
        } else {
            if (!have_ed) {
                ed = error64(bd, bz, ba, bzb);
                have_ed = true;
            }
            const double en = error64(dc, zc, a, zb);
            take = en < ed;
            if (take) ed = en;
        }
        if (take) {
            ef = usable ? e : inf;
            bd = dc;
            bz = zc;
            bzb = zb;
#pragma unroll
            for (int j = 0; j < Q; ++j) ba[j] = a[j];
        }
    }

    lane_sorted_levels<Q>(ba, bzb, srt, cor);
    __syncwarp();                                      // absent lanes read the last group's sorted weights until here
    if (!live) return;                                 // no warp-wide operation follows
    DELTA[grp] = bd;
    ZU[grp] = bz;
    ZB[grp] = bzb;
#pragma unroll
    for (int j = 0; j < Q; ++j) ALPHA[grp * Q + j] = ba[j];
    if (grp % Gr == 0) SR[row] = 1.f;
#pragma unroll 2
    for (int i = 0; i < g; i += 4) {
        float w[4];
        w4(i, w);
        uint32_t c4 = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float u, m;
            const int r = nearest_rank<L>(transform_x(w[k], 1.f, bd, 1.f, bz, u), srt, m);
            c4 |= (uint32_t)((cor >> (4 * r)) & 15u) << (8 * k);
        }
        *reinterpret_cast<uint32_t*>(CODES + eoff + i) = c4;
        *reinterpret_cast<float4*>(S + eoff + i) = make_float4(1.f, 1.f, 1.f, 1.f);
    }
}

template <int Q, typename WT, int G_, bool FAST>
static cudaError_t run_init_lane(const Shape& sh, const void* W, int G, int T, int clip, uq_params p,
                                 uint8_t* codes, cudaStream_t st) {
    constexpr size_t warp_bytes = init_lane_warp_bytes(Q, G_, FAST);
    // as many warps as fit in the 227 KB a block may opt in to
    constexpr int fit = (int)((227 * 1024) / warp_bytes);
    static_assert(fit >= 1, "one warp's tables must fit");
    constexpr int most = fit > lane_init_max_warps(FAST) ? lane_init_max_warps(FAST) : fit;
    const int64_t n_groups = sh.out * (int64_t)(sh.n_in / G_);
    // ... but no more than spreads a small matrix over every SM
    const int64_t spread = ((n_groups + 31) / 32 + sm_count() - 1) / sm_count();
    const int wpb = spread < most ? (int)spread : most;
    const size_t dyn = warp_bytes * wpb;
    auto kern = init_lane_kernel<Q, WT, G_, FAST>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(warp_bytes * most));
    if (e != cudaSuccess) return e;
    const int64_t per_block = (int64_t)wpb * 32;
    const int64_t blocks = (n_groups + per_block - 1) / per_block;
    kern<<<dim3((unsigned)blocks), wpb * 32, dyn, st>>>(W, n_groups, sh.n_in, G, T, clip, p.delta, p.zu, p.s,
                                                       p.sr, p.alpha, p.zb, codes);
    return cudaGetLastError();
}

template <int Q, typename WT, int G_>
static cudaError_t run_init_lanes(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                                  cudaStream_t st) {
    return G > 1 ? run_init_lane<Q, WT, G_, true>(sh, W, G, T, clip, p, codes, st)
                 : run_init_lane<Q, WT, G_, false>(sh, W, G, T, clip, p, codes, st);
}

template <int Q, typename WT>
static cudaError_t run_init(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                            cudaStream_t st) {
    if (sh.g == 32) return run_init_lanes<Q, WT, 32>(sh, W, G, T, clip, p, codes, st);
    if (sh.g == 64) return run_init_lanes<Q, WT, 64>(sh, W, G, T, clip, p, codes, st);
    if (sh.g == 128) return run_init_lanes<Q, WT, 128>(sh, W, G, T, clip, p, codes, st);
    const int64_t n_groups = sh.out * (int64_t)(sh.n_in / sh.g);
    // A warp each for few groups of 256, by waves of eight warps per SM (1216
    // groups); warp vs lane, T = 15.  G = 30: q = 2 one wave 2.09 vs 2.40 ms (two:
    // 3.2 vs 2.4), q = 3 4.5 vs 4.7 to 5.2 (8.5 vs 5.2), q = 4 7.9 vs 9.1 to 10.0
    // (15.5 vs 10.0); q = 1 four waves 1.04 vs 1.25 (seven: 1.8 vs 1.5).  G = 1, q = 2,
    // 3, 4, three waves: 0.51, 1.00, 1.09 vs 0.62, 0.89, 1.25, four: 0.67, 1.01, 1.45 vs
    // 0.62, 0.89, 1.25.  No rounds and one candidate: 0.02 to 0.20 vs 0.13 to 0.25 up
    // to 16384 groups.
    const int waves = Q == 1 ? 4 : G == 1 ? (Q == 3 ? 2 : 3) : 1;
    const bool few = (G == 1 && T == 0) || n_groups <= (int64_t)waves * 8 * sm_count();
    if (sh.g == kLaneInitMaxG && !few) return run_init_lanes<Q, WT, kLaneInitMaxG>(sh, W, G, T, clip, p, codes, st);
    const size_t per_warp = (size_t)sh.g * (sizeof(float) + 1);
    int wpc = (int)((96 * 1024) / per_warp);
    wpc = wpc < 1 ? 1 : (wpc > kInitMaxWarps ? kInitMaxWarps : wpc);
    const size_t dyn = per_warp * wpc;
    auto kern = init_kernel<Q, WT>;
    if (dyn > 32 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    const int64_t blocks = (n_groups + wpc - 1) / wpc;
    kern<<<dim3((unsigned)blocks), wpc * 32, dyn, st>>>(W, n_groups, sh.n_in, sh.g, G, T, clip, p.delta, p.zu,
                                                          p.s, p.sr, p.alpha, p.zb, codes);
    return cudaGetLastError();
}

template <int Q>
cudaError_t launch_init_q(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                          cudaStream_t st) {
    if (sh.wdtype == UQ_W_BF16) return run_init<Q, WBF16>(sh, W, G, T, clip, p, codes, st);
    return run_init<Q, WF32>(sh, W, G, T, clip, p, codes, st);
}

}  // namespace uq
