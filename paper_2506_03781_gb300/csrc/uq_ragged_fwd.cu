// Pipelined forward for rows that are no whole number of work units (see
// uq_ragged.cuh): the per-warp pipeline of uq_stream.cu, one unit per item,
// the last unit of a row with the groups that are left.  The remap step
// decides from the reciprocal inside a proven interval (remap_vec4), the full
// mapping from a search over the midpoints and such an interval (full_vec4);
// every decision is the IEEE one.
//
// Bound by issue: 50 to 80 instructions per element of which the tables of a
// unit (levels, order, intervals) are a third.  4096 x 11008, q = 4, g = 128,
// bf16, full mapping: 229 -> 144 us (the scan of 16 levels and the IEEE
// quotient before); 4096 x 4096, q = 2, g = 256: remap 42.7 -> 35.0 us, keep
// 21.2 -> 16.3 us (loads straight into registers before).
#include "uq_ragged.cuh"

namespace uq {

static __device__ unsigned int g_ragged_err = 0;

template <int Q, typename WT, int G_, int MODE>
using RaggedFwdStage =
    RaggedStage<Q, WT, G_, MODE != FWD_KEEP, false, MODE != FWD_FULL, MODE == FWD_KEEP ? 4096 : 7680>;

template <int Q, typename WT, int G_, int MODE>
__global__ void __launch_bounds__(kThreads, MODE == FWD_KEEP ? 4 : 3)
ragged_fwd_kernel(const RaggedSrc src, const float* __restrict__ SR, uint8_t* __restrict__ CODES,
                  float* __restrict__ WHAT, int64_t out, int n_in, int R, int n_rb) {
    using St = RaggedFwdStage<Q, WT, G_, MODE>;
    constexpr int L = 1 << Q, LPG = St::LPG, NG = St::NG, NV = St::NV, UE = St::UE, NST = St::NST;
    let_next_start((n_in / G_ + NG - 1) / NG, R, n_rb, kManyRounds);
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[kWarps][NST];
    __shared__ SortTab<Q, NG> tabs[kWarps];
    __shared__ float4 ivs[kWarps][MODE == FWD_KEEP ? 1 : NG][L];
    __shared__ __align__(16) float ths[kWarps][MODE == FWD_FULL ? NG : 1][L];      // midpoints of the full mapping
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / LPG, li = lane % LPG;
    const int Gr = n_in / G_, U = (Gr + NG - 1) / NG;
    const Items it(U, R, n_rb, warp);
    unsigned char* wsm = smem + (size_t)warp * St::WARP_BYTES;
    SortTab<Q, NG>& t = tabs[warp];

    if (lane == 0) {
        for (int s = 0; s < NST; ++s) tma::bar_init(tma::smem_addr(&bars[warp][s]), 8);
        tma::bar_init_fence();
    }
    __shared__ RaggedCopy cps[8];
    ragged_copies<Q, St>(cps, src);
    __syncthreads();
    const int64_t whole = ragged_whole<Q>(out * Gr);
    inputs_ready();
    auto issue = [&](const Cursor& c, int s) {           // the whole warp
        const uint32_t bar = tma::smem_addr(&bars[warp][s]);
        const int64_t row = it.row(c.k);
        if (row >= out) {
            if (lane < 8) tma::bar_arrive(bar);
            return;
        }
        const RaggedUnit<Q, NG> u(row, it.unit(c.j), Gr, whole);
        ragged_issue<Q, G_, St>(u, row, it.unit(c.j), n_in, cps, tma::smem_addr(wsm + (size_t)s * St::BYTES), bar, lane);
    };
    Cursor ic;
    long long issued = 0;
    for (int s = 0; s < NST && issued < it.total; ++s, ++issued) {
        issue(ic, s);
        ic.next(it.n_w);
    }
    Ring<NST> ring;
    Cursor cc;
    for (long long i = 0; i < it.total; ++i) {
        const int s = ring.s;
        if (!__all_sync(kFull, tma::bar_wait(tma::smem_addr(&bars[warp][s]), ring.parity))) {
            if (lane == 0) {
                atomicOr(&g_ragged_err, 1u);
                if (!drain(bars[warp], i, issued)) atomicOr(&g_ragged_err, kDrainTimeoutBit);
            }
            return;                                      // no block barrier in this kernel
        }
        const int64_t row = it.row(cc.k);
        if (row < out) {
            const int unit = it.unit(cc.j);
            const RaggedUnit<Q, NG> u(row, unit, Gr, whole);
            unsigned char* st = wsm + (size_t)s * St::BYTES;
            ragged_params<Q, St>(u, src, st, lane);
            const float* pd = reinterpret_cast<const float*>(st + St::OFF_D) + u.po;
            const float* pz = reinterpret_cast<const float*>(st + St::OFF_Z) + u.po;
            const float* pb = reinterpret_cast<const float*>(st + St::OFF_B) + u.po;
            const float* pa = reinterpret_cast<const float*>(st + St::OFF_A) + u.ao;
#pragma unroll
            for (int e = lane; e < NG * L; e += 32) {
                const int kk = e / L, c = e % L;
                float a[Q];
#pragma unroll
                for (int jj = 0; jj < Q; ++jj) a[jj] = kk < u.ng ? pa[kk * Q + jj] : 0.f;
                t.lv[kk][c] = level_of<Q>(c, a, kk < u.ng ? pb[kk] : 0.f);
            }
            __syncwarp();
            const bool ok = sub < u.ng;
            const int gs = ok ? sub : 0;                 // lanes of absent groups repeat the first one, store nothing
            const float dl = pd[gs], zu = pz[gs];
            const int64_t ebase = row * n_in + (int64_t)unit * UE;
            FullKeys<L> keys;
            float sr = 0.f;
            if constexpr (MODE != FWD_KEEP) {
                sr = __ldg(SR + row);
                unit_sort<Q, NG, false>(t, lane);
                if constexpr (MODE == FWD_REMAP) unit_remap_iv<Q, NG>(t, ivs[warp], lane, pd, pz);
                else unit_full_iv<Q, NG>(t, ivs[warp], ths[warp], lane, pd, pz, u.ng);
                if constexpr (MODE == FWD_FULL) keys.load(ths[warp][gs]);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int el = gs * G_ + 4 * li + 4 * LPG * v;
                float o[4];
                uint32_t nc = 0;
                if constexpr (MODE == FWD_KEEP) {
                    const uint32_t cv = *reinterpret_cast<const uint32_t*>(st + St::OFF_C + el);
#pragma unroll
                    for (int k = 0; k < 4; ++k) o[k] = __fmul_rn(dl, __fsub_rn(t.lv[gs][(cv >> (8 * k)) & (L - 1)], zu));
                } else {
                    float w[4], s4[4];
                    WT::unpack(*reinterpret_cast<const typename WT::raw*>(st + St::OFF_W + el * St::WBYTES), w);
                    f4_to(*reinterpret_cast<const float4*>(st + St::OFF_S + el * 4), s4);
                    if constexpr (MODE == FWD_REMAP) {
                        const uint32_t cv = *reinterpret_cast<const uint32_t*>(st + St::OFF_C + el);
                        nc = remap_vec4<Q, NG>(w, s4, cv, t, ivs[warp], gs, dl, sr, zu, o);
                    } else {
                        nc = full_vec4<Q, NG>(w, s4, t, ivs[warp], ths[warp], keys, gs, dl, sr, zu, o);
                    }
                }
                if (ok) {
                    if constexpr (MODE != FWD_KEEP) *reinterpret_cast<uint32_t*>(CODES + ebase + el) = nc;
                    *reinterpret_cast<float4*>(WHAT + ebase + el) = make_float4(o[0], o[1], o[2], o[3]);
                }
            }
        }
        __syncwarp();                                    // the stage and the tables are free again
        if (issued < it.total) {
            issue(ic, s);
            ic.next(it.n_w);
            ++issued;
        }
        ring.next();
        cc.next(it.n_w);
    }
}

template <typename St, int MODE>
struct RaggedFwdTag {};

template <int Q, typename WT, int G_, int MODE>
static cudaError_t run_ragged_fwd(const Shape& sh, const void* W, uq_params p, uint8_t* codes, float* what,
                                  cudaStream_t st) {
    using St = RaggedFwdStage<Q, WT, G_, MODE>;
    const int U = (sh.n_in / G_ + St::NG - 1) / St::NG;
    const int R = rows_per_block(U);
    const int n_rb = (int)((sh.out + R - 1) / R);
    const size_t dyn = (size_t)kWarps * St::WARP_BYTES;
    auto kern = ragged_fwd_kernel<Q, WT, G_, MODE>;
    int grid = 0;
    cudaError_t e = grid_for<RaggedFwdTag<St, MODE>>(kern, dyn, n_rb, grid);
    if (e != cudaSuccess) return e;
    const RaggedSrc src{static_cast<const unsigned char*>(W), reinterpret_cast<const unsigned char*>(p.s), nullptr,
                        codes, p.delta, p.zu, p.zb, p.alpha};
    return launch_dependent(kern, grid, kThreads, dyn, st, src, p.sr, codes, what, sh.out, sh.n_in, R, n_rb);
}

template <int Q, int G_>
static cudaError_t ragged_fwd_g(const Shape& sh, const void* W, uq_params p, uint8_t* codes, int mode, float* what,
                                cudaStream_t st) {
    if (mode == FWD_KEEP) return run_ragged_fwd<Q, WBF16, G_, FWD_KEEP>(sh, W, p, codes, what, st);
    const bool bf16 = sh.wdtype == UQ_W_BF16;
    if (mode == FWD_REMAP)
        return bf16 ? run_ragged_fwd<Q, WBF16, G_, FWD_REMAP>(sh, W, p, codes, what, st)
                    : run_ragged_fwd<Q, WF32, G_, FWD_REMAP>(sh, W, p, codes, what, st);
    if constexpr (ragged_full_has(Q, G_))
        return bf16 ? run_ragged_fwd<Q, WBF16, G_, FWD_FULL>(sh, W, p, codes, what, st)
                    : run_ragged_fwd<Q, WF32, G_, FWD_FULL>(sh, W, p, codes, what, st);
    return cudaErrorInvalidValue;                        // ragged_fwd_ok refuses the rest
}

template <int Q>
static cudaError_t ragged_fwd_q(const Shape& sh, const void* W, uq_params p, uint8_t* codes, int mode, float* what,
                                cudaStream_t st) {
    switch (sh.g) {
        case 32: return ragged_fwd_g<Q, 32>(sh, W, p, codes, mode, what, st);
        case 64: return ragged_fwd_g<Q, 64>(sh, W, p, codes, mode, what, st);
        case 128: return ragged_fwd_g<Q, 128>(sh, W, p, codes, mode, what, st);
        case 256: return ragged_fwd_g<Q, 256>(sh, W, p, codes, mode, what, st);
        default: return ragged_fwd_g<Q, 512>(sh, W, p, codes, mode, what, st);
    }
}

cudaError_t launch_fwd_ragged(const Shape& sh, const void* W, uq_params p, uint8_t* codes, int mode, float* what,
                              cudaStream_t st) {
    switch (sh.q) {
        case 1: return ragged_fwd_q<1>(sh, W, p, codes, mode, what, st);
        case 2: return ragged_fwd_q<2>(sh, W, p, codes, mode, what, st);
        case 3: return ragged_fwd_q<3>(sh, W, p, codes, mode, what, st);
        default: return ragged_fwd_q<4>(sh, W, p, codes, mode, what, st);
    }
}

cudaError_t ragged_fwd_error(bool clear, unsigned int* flag) {
    unsigned int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_ragged_err, sizeof(v));
    if (e != cudaSuccess) return e;
    *flag = v;
    if (clear && v) {
        const unsigned int z = 0;
        e = cudaMemcpyToSymbol(g_ragged_err, &z, sizeof(z));
    }
    return e;
}

}  // namespace uq
