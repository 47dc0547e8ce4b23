// Unified initialization (Algorithm 2) with the clipping strategies of
// App. E.2 and the general alternating update of Algorithm 3: one lane per
// group for g <= 256 (init_lane_kernel), one warp per group for larger
// groups (init_kernel); the group's transformed weights x and code words
// kept in shared memory.  Runs once before training; not on the per-step
// path.  A round of the alternating update that moves no code (and not z_B)
// is a fixed point: the remaining rounds are skipped, which changes nothing.
//
// Sums that feed alpha and z_B are taken in fp64 (the group's fp32 values
// are summed exactly in practice); the normal equations C^T C alpha =
// C^T (x - z_B) have an integer matrix, so singularity is decided exactly
// by an integer determinant and the system is solved in fp64 by Gaussian
// elimination with partial pivoting.
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
// are formed from per-code-word sums of x and counts; a round touches only
// the elements whose code moved.  Shared memory per warp, element-major so
// that the 32 lanes touch consecutive words (init_lane_warp_bytes).
//
// Where init_kernel sums in fp64 this kernel takes the same values without
// fp64, and goes back to fp64 wherever it cannot show that they are the same:
//  * sums of |r| and x: with all values multiples of 2^-k below 2^30 2^-k
//    (k per group and candidate; every value is checked), the fp64 sums are
//    exact in any order, and so are 64-bit integer sums;
//  * the normal equations: the exact solution N_j / D from integers (Cramer's
//    rule), rounded to fp32 only where it lies further from a tie of that
//    rounding than the fp64 elimination can be off (see below);
//  * the nearest level: a binary search over the midpoints of the sorted
//    levels where x is further from each of them than the fp32 distances can
//    be off, else the scan of nearest_rank;
//  * the candidate's error: an fp32 sum, and the fp64 sums of the candidate
//    and the kept one only where the two fp32 sums are within their bound.
// So every output is bit for bit what fp64 gave.  1024 x 4096, q = 3, g = 128,
// G = 30, T = 15: 15.8 -> 9.2 ms (fp64 pipe 76 % -> 7 % busy; now bound by
// issue at 1.7 warps per scheduler, half of the lanes idle in the late rounds).
constexpr int kLaneInitMaxG = 256;

// Shared memory of one warp: the per-code sums of x [L][32] (64 bits), x
// [g][32], the sorted levels [L][32], W^ of the sorted levels [L][32] and the
// code words [g][32]; rounded up to 16 bytes.
__host__ __device__ constexpr size_t init_lane_warp_bytes(int q, int g) {
    return (((size_t)(1 << q) * 32 * (8 + 4 + 4) + (size_t)g * 32 * (4 + 1)) + 15) & ~size_t(15);
}

// Counts of the L code words of one group, BITS bits per code word packed in
// 64-bit registers; c is a compile-time index wherever get() is used, add()
// takes any c.
template <int L, int BITS>
struct CodeHist {
    static constexpr int PER = 64 / BITS, NW = (L + PER - 1) / PER;
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

// Levels of (a, zb), sorted ascending (ties by code word) into srt_s and
// registers; cor holds the code word of rank r in bits 4 r .. 4 r + 3, that of
// the lowest rank among equal levels (the one nearest_rank takes).
template <int Q>
__device__ __forceinline__ void lane_sorted_levels(const float a[Q], float zb, float* srt_s, int lane,
                                                   float srt[1 << Q], uint64_t& cor) {
    constexpr int L = 1 << Q;
    float lv[L];
#pragma unroll
    for (int c = 0; c < L; ++c) lv[c] = level_of<Q>(c, a, zb);
    cor = 0;
#pragma unroll
    for (int c = 0; c < L; ++c) {
        int r = 0, first = 0;
#pragma unroll
        for (int c2 = 0; c2 < L; ++c2) {
            r += (lv[c2] < lv[c]) || (lv[c2] == lv[c] && c2 < c);
            if (c2 < c && lv[c2] == lv[c] && !(first & 16)) first = 16 | c2;     // lowest equal code word
        }
        srt_s[r * 32 + lane] = lv[c];
        cor |= uint64_t((first & 16) ? (first & 15) : c) << (4 * r);
    }
#pragma unroll
    for (int r = 0; r < L; ++r) srt[r] = srt_s[r * 32 + lane];
}

// The search for the nearest level: thresholds t (midpoints of neighbouring
// sorted levels) and the margin around them inside which the scan decides.
//
// With M the largest |level| and X the largest |x| of the group, x further
// than m = 2^-21 (X + M) from t_r lies on the same side of the exact midpoint
// (t_r is off by at most 2^-24 M), and where it lies between the two levels
// the exact distances differ by more than 2 m - 2^-23 M > 2^-23 M, their
// roundings by at most 2^-24 of their sum (at most 2^-23 M): the rounded
// distances keep the order.  Beyond both levels they differ by the gap of the
// levels, and rounding could make them equal only if the gap is below 2^-23
// (X + M): then no x is sure (m = infinity).  Equal levels have equal
// distances, and cor names the lowest of their ranks.
template <int L>
struct LevelSearch {
    float t[L - 1], m;
    __device__ __forceinline__ void set(const float srt[L], float xmax) {
        const float M = fmaxf(fabsf(srt[0]), fabsf(srt[L - 1]));
        m = (xmax + M) * 0x1p-21f;
        bool ok = M < 0x1p100f && xmax < 0x1p100f;          // false also for NaN
#pragma unroll
        for (int r = 0; r + 1 < L; ++r) {
            t[r] = 0.5f * (srt[r] + srt[r + 1]);
            const float gap = srt[r + 1] - srt[r];
            ok &= gap == 0.f || gap > m;
        }
        if (!ok) m = __int_as_float(0x7f800000);
    }
    // Rank of the nearest level; srt_s: the lane's sorted levels in shared memory (for the scan).
    __device__ __forceinline__ int rank(float x, const float* srt_s) const {
        float c[L - 1];
#pragma unroll
        for (int i = 0; i < L - 1; ++i) c[i] = t[i];
        int r = 0;
        float near = __int_as_float(0x7f800000);
#pragma unroll
        for (int n = L / 2; n >= 1; n /= 2) {                // 2 n - 1 candidates left, the middle one c[n - 1]
            const float d = x - c[n - 1];
            const bool up = d > 0.f;
            near = fminf(near, fabsf(d));
            r = 2 * r + (up ? 1 : 0);
#pragma unroll
            for (int i = 0; i < n - 1; ++i) c[i] = up ? c[n + i] : c[i];
        }
        if (!(near > m)) {
            float best = fabsf(__fsub_rn(x, srt_s[0]));
            r = 0;
#pragma unroll 1
            for (int k = 1; k < L; ++k) {
                const float d = fabsf(__fsub_rn(x, srt_s[k * 32]));
                if (d < best) { best = d; r = k; }
            }
        }
        return r;
    }
};

// Exact solution of C^T C alpha = b as integers: N_j / D (D = det, N = adj b).
// n[i][j] (|n| <= g <= 128) and D fit 32 bits, N 64 bits for |b| < 2^38.
template <int Q>
__device__ __forceinline__ int cramer(const int n[Q][Q], const long long b[Q], long long N[Q]) {
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
        N[i] = 0;
#pragma unroll
        for (int j = 0; j < Q; ++j) N[i] += (long long)adj[i][j] * b[j];
    }
    return D;
}

template <int Q, typename WT, int G_>
__global__ void init_lane_kernel(const void* __restrict__ W, int64_t n_groups, int n_in, int G, int T, int clip,
                                 float* __restrict__ DELTA, float* __restrict__ ZU, float* __restrict__ S,
                                 float* __restrict__ SR, float* __restrict__ ALPHA, float* __restrict__ ZB,
                                 uint8_t* __restrict__ CODES) {
    constexpr int L = 1 << Q;
    constexpr size_t WARP_BYTES = init_lane_warp_bytes(Q, G_);
    constexpr bool CRAMER = G_ <= 128;                      // the 32-bit determinant and the 64-bit N_j hold
    using Hist = CodeHist<L, G_ <= 128 ? 8 : 16>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* base = smem + (size_t)warp * WARP_BYTES;
    double* bx = reinterpret_cast<double*>(base);                       // [L][32]; integers where they are exact
    long long* bi = reinterpret_cast<long long*>(base);
    float* xs = reinterpret_cast<float*>(bx + L * 32);                  // [G_][32]
    float* srt_s = xs + G_ * 32;                                        // [L][32]
    float* wh_s = srt_s + L * 32;                                       // [L][32]
    uint8_t* cs = reinterpret_cast<uint8_t*>(wh_s + L * 32);            // [G_][32]

    const int64_t grp0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 32;
    if (grp0 >= n_groups) return;                      // whole warp; no block barrier in this kernel
    const int64_t grp_raw = grp0 + lane;
    const bool live = grp_raw < n_groups;
    const int64_t grp = live ? grp_raw : n_groups - 1; // absent lanes repeat the last group, store nothing
    const int Gr = n_in / G_;
    const int64_t row = grp / Gr;
    const int64_t eoff = row * (int64_t)n_in + (grp % Gr) * (int64_t)G_;
    auto w4 = [&](int i, float (&w)[4]) { WT::unpack(WT::load(W, eoff + i), w); };
    auto X = [&](int i) -> float& { return xs[i * 32 + lane]; };
    auto C = [&](int i) -> uint8_t& { return cs[i * 32 + lane]; };
    auto BX = [&](int c) -> double& { return bx[c * 32 + lane]; };
    auto BI = [&](int c) -> long long& { return bi[c * 32 + lane]; };
    const float inf = __int_as_float(0x7f800000);

    float wmin = INFINITY, wmax = -INFINITY;
    for (int i = 0; i < G_; i += 4) {
        float w[4];
        w4(i, w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            wmin = fminf(wmin, w[k]);
            wmax = fmaxf(wmax, w[k]);
        }
    }
    const float top = (float)(L - 1);
    const float rng = fmaxf(__fsub_rn(wmax, wmin), 1e-12f);

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
    LevelSearch<L> ls;

    // fp64 error of a candidate from its own parameters (the values of init_kernel, in the same order)
    auto error64 = [&](float dc, float zc, const float (&a)[Q], float zb) {
        float sv[L];
        uint64_t unused;
        lane_sorted_levels<Q>(a, zb, wh_s, lane, sv, unused);
        double e = 0.0;
#pragma unroll 1
        for (int i = 0; i < G_; i += 4) {
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

    for (int gi = 1; gi <= G; ++gi) {
        const float gamma = __fdiv_rn((float)gi, (float)G);
        const float dc = __fdiv_rn(__fmul_rn(gamma, rng), top);
        float zc;
        if (clip == UQ_CLIP_FIXED_MIN) zc = __fdiv_rn(-wmin, dc);
        else if (clip == UQ_CLIP_FIXED_MAX) zc = __fsub_rn(top, __fdiv_rn(wmax, dc));
        else zc = __fdiv_rn(-__fmul_rn(gamma, wmin), dc);
        float a[Q], zb = bzb;
        float xmax = 0.f;
        bool nan = false;
#pragma unroll 2
        for (int i = 0; i < G_; i += 4) {
            float w[4];
            w4(i, w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float u;
                const float x = transform_x(w[k], 1.f, dc, 1.f, zc, u);
                X(i + k) = x;
                C(i + k) = 0;
                xmax = fmaxf(xmax, fabsf(x));
                nan |= x != x;
            }
        }
        // Fixed point: values below 2^e in units of 2^-k, k = 30 - e.
        const float bound = xmax + fabsf(zb);
        const int ebits = (int)((__float_as_uint(bound) >> 23) & 0xffu) - 126;      // bound < 2^ebits
        const int kfix = 30 - ebits;
        bool fixed = !nan && bound < 0x1p60f && bound > 0x1p-60f;
        const float up = fixed ? __int_as_float((127 + kfix) << 23) : 1.f, down = fixed ? __int_as_float((127 - kfix) << 23) : 1.f;
        auto to_fixed = [&](float v) { return __float2int_rn(v * up); };
        auto is_fixed = [&](float v, int n) { return (float)n == v * up; };

        // --- Algorithm 3: greedy start (one bit at a time) ---
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            auto residual = [&](int i, int c) {
                float r = __fsub_rn(X(i), zb);
#pragma unroll
                for (int jj = 0; jj < j; ++jj) r = __fsub_rn(r, ((c >> jj) & 1) ? a[jj] : -a[jj]);
                return r;
            };
            long long sum = 0;
            bool exact = fixed;
#pragma unroll 4
            for (int i = 0; i < G_; ++i) {
                const int c = C(i);
                const float r = residual(i, c);
                const int n = to_fixed(fabsf(r));
                exact &= is_fixed(fabsf(r), n);
                sum += n;
                if (r >= 0.f) C(i) = (uint8_t)(c | (1 << j));
            }
            if (exact) {
                a[j] = __ll2float_rn(sum) * (down * (1.f / (float)G_));     // powers of two: exact
            } else {
                double sabs = 0.0;
#pragma unroll 1
                for (int i = 0; i < G_; ++i) sabs += (double)fabsf(residual(i, C(i) & ((1 << j) - 1)));
                a[j] = (float)(sabs / (double)G_);
            }
        }
        // Per code word c: the sum of x over the group's elements with code c
        // and their count (hist).  Then C^T (x - z_B) = sum_c s(c) (bx_c - n_c
        // z_B) and C^T C = sum_c n_c s(c) s(c)^T, where s(c) is the sign vector
        // of c; a round only moves the elements whose code changed from one sum
        // to the other.
        Hist hist;
#pragma unroll
        for (int c = 0; c < L; ++c) BI(c) = 0;
        const int zbi = to_fixed(zb);
        fixed &= is_fixed(zb, zbi) && G > 1;               // z_B moves when G == 1
#pragma unroll 2
        for (int i = 0; i < G_; ++i) {
            const int c = C(i);
            const float x = X(i);
            const int n = to_fixed(x);
            fixed &= is_fixed(x, n);
            BI(c) += n;
            hist.add(c, 1);
        }
        fixed = __all_sync(kFull, fixed);                   // one form of the sums for the warp
        if (!fixed) {
#pragma unroll
            for (int c = 0; c < L; ++c) BX(c) = 0.0;
#pragma unroll 1
            for (int i = 0; i < G_; ++i) BX(C(i)) += (double)X(i);
        }

        // --- T rounds of alpha, C (and z_B when G == 1) ---
        bool more = true;
        for (int it = 0; it < T; ++it) {
            int ctc[Q][Q];
#pragma unroll
            for (int j = 0; j < Q; ++j)
#pragma unroll
                for (int k = j; k < Q; ++k) {
                    int v = 0;
#pragma unroll
                    for (int c = 0; c < L; ++c) v += (((c >> j) ^ (c >> k)) & 1) ? -hist.get(c) : hist.get(c);
                    ctc[j][k] = ctc[k][j] = v;
                }
            bool solved = false;
            if (CRAMER && fixed) {
                long long b[Q], N[Q];
#pragma unroll
                for (int j = 0; j < Q; ++j) b[j] = 0;
#pragma unroll
                for (int c = 0; c < L; ++c) {
                    const long long y = BI(c) - (long long)hist.get(c) * zbi;
#pragma unroll
                    for (int j = 0; j < Q; ++j) b[j] += ((c >> j) & 1) ? y : -y;
                }
                const int D = cramer<Q>(ctc, b, N);
                if (D == 0) {
                    solved = true;                          // singular: alpha stays
                } else {
                    // The elimination's forward error is at most 2^11 u kappa max|alpha| (n <= 4,
                    // growth <= 8; kappa, the condition of the positive definite matrix, from its
                    // trace Q G_ and determinant), N_j / D as formed here within 2^-51 of itself.
                    const double rd = (double)down / (double)D;
                    double sol[Q];
                    float amax = 0.f, av[Q];
#pragma unroll
                    for (int j = 0; j < Q; ++j) {
                        sol[j] = (double)N[j] * rd;
                        av[j] = (float)sol[j];
                        amax = fmaxf(amax, fabsf(av[j]));
                    }
                    float kappa = (float)(Q * G_);
#pragma unroll
                    for (int j = 1; j < Q; ++j) kappa *= (float)(Q * G_) / (float)(Q > 1 ? Q - 1 : 1);
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
                long long n64[Q][Q];
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    cty[j] = 0.0;
#pragma unroll
                    for (int k = 0; k < Q; ++k) n64[j][k] = ctc[j][k];
                }
#pragma unroll 1
                for (int c = 0; c < L; ++c) {
                    int n = 0;
#pragma unroll
                    for (int c2 = 0; c2 < L; ++c2) n = c2 == c ? hist.get(c2) : n;
                    const double sx = fixed ? (double)BI(c) * (double)down : BX(c);
                    const double yc = sx - (double)n * (double)zb;
#pragma unroll
                    for (int j = 0; j < Q; ++j) cty[j] += ((c >> j) & 1) ? yc : -yc;
                }
                if (!int_singular<Q>(n64)) {
                    double sol[Q];
                    solve_fp64<Q>(n64, cty, sol);
#pragma unroll
                    for (int j = 0; j < Q; ++j) a[j] = (float)sol[j];
                }
            }
            lane_sorted_levels<Q>(a, zb, srt_s, lane, srt, cor);
            ls.set(srt, xmax);
            bool moved = false;
#pragma unroll 4
            for (int i = 0; i < G_; ++i) {
                const float x = X(i);
                const int r = ls.rank(x, srt_s + lane);
                const int c = (int)((cor >> (4 * r)) & 15u);
                const int old = C(i);
                if (c != old) {
                    moved = true;
                    if (fixed) {
                        const int n = to_fixed(x);
                        BI(old) -= n;
                        BI(c) += n;
                    } else {
                        const double xd = (double)x;
                        BX(old) -= xd;
                        BX(c) += xd;
                    }
                    hist.add(old, -1);
                    hist.add(c, 1);
                    C(i) = (uint8_t)c;
                }
            }
            const float zb_prev = zb;
            if (G == 1) {
                // z_B = mean of x - C alpha = sum_c (bx_c - n_c (s(c) . alpha)) / g (fp64 sums: not fixed)
                double sres = 0.0;
#pragma unroll
                for (int c = 0; c < L; ++c) {
                    double ca = 0.0;
#pragma unroll
                    for (int j = 0; j < Q; ++j) ca += ((c >> j) & 1) ? (double)a[j] : -(double)a[j];
                    sres += BX(c) - (double)hist.get(c) * ca;
                }
                zb = (float)(sres / (double)G_);
            }
            // No code moved (and z_B did not either): the next round would
            // solve the same system, get the same alpha and the same codes, so
            // every remaining round repeats this state bit for bit.
            more = moved || __float_as_uint(zb) != __float_as_uint(zb_prev);
            if (!more) break;
        }

        // --- candidate error with the full mapping (Eq. 2), s = s_r = 1 ---
        lane_sorted_levels<Q>(a, zb, srt_s, lane, srt, cor);
        ls.set(srt, xmax);
#pragma unroll
        for (int r = 0; r < L; ++r) wh_s[r * 32 + lane] = __fmul_rn(dc, __fsub_rn(srt[r], zc));
        float e4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int i = 0; i < G_; i += 4) {
            float w[4];
            w4(i, w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float df = w[k] - wh_s[ls.rank(X(i + k), srt_s + lane) * 32 + lane];
                e4[k] = fmaf(df, df, e4[k]);
            }
        }
        // Within 2^-23 per square and 2^-24 per addition of the exact sum (at
        // most 66 of them): 5e-6; a square below 2^-126 may be lost, so the sum
        // has to be well above 256 of those.
        const float e = (e4[0] + e4[1]) + (e4[2] + e4[3]);
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

    lane_sorted_levels<Q>(ba, bzb, srt_s, lane, srt, cor);
    if (!live) return;                                 // no warp-wide operation follows
    DELTA[grp] = bd;
    ZU[grp] = bz;
    ZB[grp] = bzb;
#pragma unroll
    for (int j = 0; j < Q; ++j) ALPHA[grp * Q + j] = ba[j];
    if (grp % Gr == 0) SR[row] = 1.f;
#pragma unroll 2
    for (int i = 0; i < G_; i += 4) {
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

template <int Q, typename WT, int G_>
static cudaError_t run_init_lane(const Shape& sh, const void* W, int G, int T, int clip, uq_params p,
                                 uint8_t* codes, cudaStream_t st) {
    constexpr size_t warp_bytes = init_lane_warp_bytes(Q, G_);
    // as many warps as fit in the 227 KB a block may opt in to, at most 16
    constexpr int most = (int)((227 * 1024) / warp_bytes) > 16 ? 16 : (int)((227 * 1024) / warp_bytes);
    static_assert(most >= 1, "one warp's tables must fit");
    const int64_t n_groups = sh.out * (int64_t)(sh.n_in / G_);
    // ... but no more than spreads a small matrix over every SM
    const int64_t spread = ((n_groups + 31) / 32 + sm_count() - 1) / sm_count();
    const int wpb = spread < most ? (int)spread : most;
    const size_t dyn = warp_bytes * wpb;
    auto kern = init_lane_kernel<Q, WT, G_>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(warp_bytes * most));
    if (e != cudaSuccess) return e;
    const int64_t per_block = (int64_t)wpb * 32;
    const int64_t blocks = (n_groups + per_block - 1) / per_block;
    kern<<<dim3((unsigned)blocks), wpb * 32, dyn, st>>>(W, n_groups, sh.n_in, G, T, clip, p.delta, p.zu, p.s, p.sr,
                                                       p.alpha, p.zb, codes);
    return cudaGetLastError();
}

template <int Q, typename WT>
static cudaError_t run_init(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                            cudaStream_t st) {
    if (sh.g == 32) return run_init_lane<Q, WT, 32>(sh, W, G, T, clip, p, codes, st);
    if (sh.g == 64) return run_init_lane<Q, WT, 64>(sh, W, G, T, clip, p, codes, st);
    if (sh.g == 128) return run_init_lane<Q, WT, 128>(sh, W, G, T, clip, p, codes, st);
    if (sh.g == kLaneInitMaxG) return run_init_lane<Q, WT, 256>(sh, W, G, T, clip, p, codes, st);
    const int64_t n_groups = sh.out * (int64_t)(sh.n_in / sh.g);
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
static cudaError_t init_w(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                          cudaStream_t st) {
    if (sh.wdtype == UQ_W_BF16) return run_init<Q, WBF16>(sh, W, G, T, clip, p, codes, st);
    return run_init<Q, WF32>(sh, W, G, T, clip, p, codes, st);
}

cudaError_t launch_init(const Shape& sh, const void* W, int G, int T, int clip, uq_params p, uint8_t* codes,
                        cudaStream_t st) {
    switch (sh.q) {
        case 1: return init_w<1>(sh, W, G, T, clip, p, codes, st);
        case 2: return init_w<2>(sh, W, G, T, clip, p, codes, st);
        case 3: return init_w<3>(sh, W, G, T, clip, p, codes, st);
        default: return init_w<4>(sh, W, G, T, clip, p, codes, st);
    }
}

}  // namespace uq
