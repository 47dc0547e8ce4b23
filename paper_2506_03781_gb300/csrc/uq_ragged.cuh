// Stages and copies of the pipelined kernels for rows that are no whole number
// of work units (uq_ragged_fwd.cu, uq_ragged_bwd.cu): g in {32, 64, 128} with
// a last unit of fewer groups, and g = 256 and 512, whose units hold two
// groups and one.
//
// A unit's weights, s, code words and dL/dW^ start and end on 16-byte
// boundaries whatever the row (32 columns are 32 bytes of codes), but its
// group parameters need not: the groups of a row start at any multiple of 4
// bytes.  So the parameter copies move whole 16-byte pieces -- a window from
// the boundary below the unit's first value to the one above its last -- and
// the kernels index from the remainder.  A window that would end beyond the
// array (the last groups of the last row) is not copied: the warp loads those
// values itself.
#pragma once

#include <atomic>

#include "uq_common.cuh"
#include "uq_launch.h"
#include "uq_pipe.cuh"

namespace uq {

// Stage of one unit.  HAS_X: weights and s; HAS_G: dL/dW^; HAS_C: code words.
template <int Q, typename WT, int G_, bool HAS_X, bool HAS_G, bool HAS_C, int BUDGET>
struct RaggedStage {
    static constexpr int LPG = G_ <= 64 ? 4 : G_ <= 256 ? G_ / 16 : 32;
    static constexpr int NG = 32 / LPG;                  // groups per unit
    static constexpr int NV = G_ / (4 * LPG);            // vectors per lane
    static constexpr int UE = NG * G_;                   // elements per unit
    static constexpr int WBYTES = sizeof(typename WT::raw) / 4;
    static constexpr int WIN_P = align_up(NG + 3, 4) * 4, WIN_A = align_up(NG * Q + 3, 4) * 4;   // bytes of a window
    static constexpr int OFF_W = 0;
    static constexpr int OFF_S = align_up(HAS_X ? UE * WBYTES : 0, 16);
    static constexpr int OFF_G = OFF_S + (HAS_X ? UE * 4 : 0);
    static constexpr int OFF_C = OFF_G + (HAS_G ? UE * 4 : 0);
    static constexpr int OFF_D = align_up(OFF_C + (HAS_C ? UE : 0), 16);
    static constexpr int OFF_Z = OFF_D + WIN_P;
    static constexpr int OFF_B = OFF_Z + WIN_P;
    static constexpr int OFF_A = OFF_B + WIN_P;
    static constexpr int BYTES = align_up(OFF_A + WIN_A, 128);
    static constexpr int FIT = BUDGET / BYTES;
    static constexpr int NST = FIT < 2 ? 2 : (FIT > kMaxStages ? kMaxStages : FIT);
    static constexpr int WARP_BYTES = NST * BYTES;
    static constexpr bool X = HAS_X, G = HAS_G, C = HAS_C;
};

struct RaggedSrc {
    const unsigned char *W, *S, *GUP, *CODES;
    const float *DELTA, *ZU, *ZB, *ALPHA;
};

// The eight copies of a unit, one per lane 0..7, from a per-block table:
// source, bytes per element (per group for the parameters) and stage offset;
// per = 0 where the kernel has no such stream.
struct RaggedCopy {
    const unsigned char* base;
    uint32_t per, to;
};
template <int Q, typename St>
__device__ __forceinline__ void ragged_copies(RaggedCopy* cps, const RaggedSrc& src) {
    if (threadIdx.x < 8) {
        const unsigned char* b[8] = {src.W, src.S, src.GUP, src.CODES, reinterpret_cast<const unsigned char*>(src.DELTA),
                                     reinterpret_cast<const unsigned char*>(src.ZU),
                                     reinterpret_cast<const unsigned char*>(src.ZB),
                                     reinterpret_cast<const unsigned char*>(src.ALPHA)};
        const uint32_t per[8] = {St::X ? (uint32_t)St::WBYTES : 0u, St::X ? 4u : 0u, St::G ? 4u : 0u, St::C ? 1u : 0u,
                                 4u, 4u, 4u, 4u * Q};
        const uint32_t to[8] = {St::OFF_W, St::OFF_S, St::OFF_G, St::OFF_C, St::OFF_D, St::OFF_Z, St::OFF_B, St::OFF_A};
        cps[threadIdx.x] = RaggedCopy{b[threadIdx.x], per[threadIdx.x], to[threadIdx.x]};
    }
}

// Where a unit's values are: its first group, the groups it holds (ng <= NG),
// the remainders of its parameter windows and whether the windows are copied
// (whole: the groups that whole 16-byte pieces of every parameter array cover).
template <int Q, int NG>
struct RaggedUnit {
    int64_t g0;
    int ng, po, ao;
    bool copied;
    __device__ __forceinline__ RaggedUnit(int64_t row, int unit, int Gr, int64_t whole) {
        g0 = row * Gr + unit * NG;
        ng = Gr - unit * NG < NG ? Gr - unit * NG : NG;
        po = (int)g0 & 3;
        ao = ((int)g0 * Q) & 3;
        copied = g0 + ng <= whole;
    }
};
template <int Q>
__device__ __forceinline__ int64_t ragged_whole(int64_t groups) {
    const int64_t p = groups & ~int64_t(3), a = (groups * Q & ~int64_t(3)) / Q;
    return p < a ? p : a;
}

// Starts the copies of one unit into the stage at st (shared-memory address);
// lanes 0..7 each arrive on bar (of 8 arrivals) with their bytes.  Every
// range is widened to 16-byte boundaries, which changes the windows only.
template <int Q, int G_, typename St>
__device__ __forceinline__ void ragged_issue(const RaggedUnit<Q, St::NG>& u, int64_t row, int unit, int n_in,
                                             const RaggedCopy* cps, uint32_t st, uint32_t bar, int lane) {
    if (lane >= 8) return;
    const RaggedCopy cp = cps[lane];
    const bool grp = lane >= 4;
    const int64_t lo = (grp ? u.g0 : row * n_in + unit * St::UE) * cp.per;
    const int64_t hi = lo + (int64_t)((grp ? u.ng : u.ng * G_) * cp.per);
    const int64_t from = lo & ~int64_t(15);
    const uint32_t bytes = (grp && !u.copied) ? 0u : (uint32_t)(((hi + 15) & ~int64_t(15)) - from);
    if (bytes != 0) {
        tma::bar_arrive_tx(bar, bytes);
        tma::fence_async_smem();                          // the warp's reads of this stage come first
        tma::copy_g2s(st + cp.to, cp.base + from, bytes, bar);
    } else {
        tma::bar_arrive(bar);
    }
}

// The parameters of a unit whose windows were not copied, by the warp itself.
template <int Q, typename St>
__device__ __forceinline__ void ragged_params(const RaggedUnit<Q, St::NG>& u, const RaggedSrc& src, unsigned char* st,
                                              int lane) {
    if (u.copied) return;
    float* d = reinterpret_cast<float*>(st + St::OFF_D) + u.po;
    float* z = reinterpret_cast<float*>(st + St::OFF_Z) + u.po;
    float* b = reinterpret_cast<float*>(st + St::OFF_B) + u.po;
    float* a = reinterpret_cast<float*>(st + St::OFF_A) + u.ao;
    for (int i = lane; i < u.ng; i += 32) {
        d[i] = __ldg(src.DELTA + u.g0 + i);
        z[i] = __ldg(src.ZU + u.g0 + i);
        b[i] = __ldg(src.ZB + u.g0 + i);
    }
    for (int i = lane; i < u.ng * Q; i += 32) a[i] = __ldg(src.ALPHA + u.g0 * Q + i);
    __syncwarp();
}

}  // namespace uq
