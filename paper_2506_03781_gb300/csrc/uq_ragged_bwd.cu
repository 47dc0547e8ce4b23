// Pipelined backward for rows that are no whole number of work units (see
// uq_ragged.cuh): the per-warp pipeline and the ring of ds_r partials of
// uq_stream.cu, one unit per item, the last unit of a row with the groups that
// are left.  The arithmetic keeps the accuracy of the general kernel
// (uq_bwd.cu): signed sums for alpha, ds from the quotient by s, and w / den
// from the hardware reciprocal with one residual correction (Markstein: q' =
// q + r (w - q den), the residual exact in one fused operation), which is
// within 2^-23 of the quotient; the filter is taken from it where the margin
// of bwd_vec4 proves the IEEE decision, else from the IEEE quotient.
//
// Bound by issue and HBM together (64 % of the issue slots, 44 % of DRAM under
// ncu).  4096 x 11008, q = 4, g = 128, bf16: 178 -> 128 us (685 MB: 0.80 of
// the measured copy rate); 4096 x 4096, q = 2, g = 256: 62.0 -> 47.6 us.
#include "uq_ragged.cuh"

namespace uq {

static __device__ unsigned int g_ragged_err = 0;

constexpr int kRaggedRing = 32;          // row blocks whose ds_r partials wait in shared memory

template <int Q, typename WT, int G_>
using RaggedBwdStage = RaggedStage<Q, WT, G_, true, true, true, 12032>;

// Backward of 4 consecutive elements of one group; see bwd_vec4 for the sums
// (here acc[4 + j] += +-G) and the margin eg = 2^-19 (|z_U| + sum |alpha_j| +
// |z_B|) + 2^-126.
template <int Q, bool ELEM>
__device__ __forceinline__ void ragged_bwd_vec4(const float w[4], const float s4[4], const float G[4], uint32_t cv,
                                                const float2* __restrict__ tab, float dl, float sr, float zu, float tau,
                                                float eg, float ds[4], float acc[8]) {
    constexpr int L = 1 << Q;
    float2 mm[4];
    float u[4], d[4];
    bool sure = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        mm[k] = tab[(cv >> (8 * k)) & (L - 1)];
        const float den = __fmul_rn(__fmul_rn(dl, s4[k]), sr);
        const float r = rcp_approx(den);
        const float q0 = __fmul_rn(w[k], r);
        u[k] = __fmaf_rn(__fmaf_rn(-q0, den, w[k]), r, q0);
        const float x = __fadd_rn(u[k], zu);
        d[k] = __fsub_rn(x, mm[k].x);
        const float E = __fmaf_rn(fabsf(x), 0x1p-18f, eg);
        sure = sure & (fabsf(__fsub_rn(fabsf(d[k]), tau)) > E) & (fabsf(den) < 0x1p125f);
    }
    if (!sure) {
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = __fsub_rn(transform_x(w[k], s4[k], dl, sr, zu, u[k]), mm[k].x);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = (cv >> (8 * k)) & (L - 1);
        const bool f = fabsf(d[k]) <= tau;
        const float fu = f ? u[k] : 0.f;
        const float gk = (ELEM && !f) ? 0.f : G[k];
        const float gfu = gk * fu;
        ds[k] = -__fdividef(dl * gfu, s4[k]);
        acc[0] += gk * (mm[k].y - fu);
        acc[1] += f ? 0.f : gk;
        acc[2] += gk;
        acc[3] += gfu;
#pragma unroll
        for (int j = 0; j < Q; ++j) acc[4 + j] += ((c >> j) & 1) ? gk : -gk;
    }
}

template <int Q, typename WT, int G_, bool ELEM>
__global__ void __launch_bounds__(kThreads, 2)
ragged_bwd_kernel(const RaggedSrc src, const float* __restrict__ SR, float* __restrict__ DS, float* __restrict__ DSR,
                  float* __restrict__ DDELTA, float* __restrict__ DZU, float* __restrict__ DZB,
                  float* __restrict__ DALPHA, int64_t out, int n_in, int R, int n_rb) {
    using St = RaggedBwdStage<Q, WT, G_>;
    constexpr int L = 1 << Q, LPG = St::LPG, NG = St::NG, NV = St::NV, UE = St::UE, NST = St::NST;
    let_next_start((n_in / G_ + NG - 1) / NG, R, n_rb, kManyRoundsBwd);
    using SR8 = SegReduce<LPG>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[kWarps][NST];
    __shared__ float2 tabs[kWarps][NG][L];              // (l(c), l(c) - z_U) per group slot and code word
    __shared__ float red[kRaggedRing][kWarps];          // per row block and warp: sum of Delta S3
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / LPG, li = lane % LPG;
    const int Gr = n_in / G_, U = (Gr + NG - 1) / NG;
    const Items it(U, R, n_rb, warp);
    unsigned char* wsm = smem + (size_t)warp * St::WARP_BYTES;
    float2 (*t)[L] = tabs[warp];

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
    long long issued = 0, waited = 0;
    for (int s = 0; s < NST && issued < it.total; ++s, ++issued) {
        issue(ic, s);
        ic.next(it.n_w);
    }
    bool alive = true;
    Ring<NST> ring;
    const int n_mine = it.n_blocks;
    for (int k = 0; k < n_mine; ++k) {
        const int64_t row = it.row(k);
        const bool row_ok = row < out;
        const float sr = row_ok ? __ldg(SR + row) : 1.f;
        float prow = 0.f;
        for (int j = 0; j < it.n_w; ++j) {
            const int s = ring.s;
            if (alive) {
                // one verdict for the whole warp (lanes poll the mbarrier separately)
                if (__all_sync(kFull, tma::bar_wait(tma::smem_addr(&bars[warp][s]), ring.parity))) {
                    ++waited;
                } else {
                    alive = false;
                    if (lane == 0) atomicOr(&g_ragged_err, 1u);
                }
            }
            if (alive && row_ok) {
                const int unit = it.unit(j);
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
                    if (kk < u.ng) {
                        float a[Q];
#pragma unroll
                        for (int jj = 0; jj < Q; ++jj) a[jj] = pa[kk * Q + jj];
                        const float lvc = level_of<Q>(c, a, pb[kk]);
                        t[kk][c] = make_float2(lvc, lvc - pz[kk]);
                    }
                }
                __syncwarp();
                const bool ok = sub < u.ng;
                const int gs = ok ? sub : 0;             // lanes of absent groups repeat the first one, store nothing
                const float dl = pd[gs], zu = pz[gs];
                float tau = fabsf(pa[gs * Q]), mag = __fadd_rn(fabsf(zu), fabsf(pb[gs]));
#pragma unroll
                for (int jj = 0; jj < Q; ++jj) {
                    const float aj = fabsf(pa[gs * Q + jj]);
                    tau = fminf(tau, aj);
                    mag = __fadd_rn(mag, aj);
                }
                const float eg = __fmaf_rn(mag, 0x1p-19f, 0x1p-126f);
                const int64_t ebase = row * n_in + (int64_t)unit * UE;
                float acc[8];
#pragma unroll
                for (int q8 = 0; q8 < 8; ++q8) acc[q8] = 0.f;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int el = gs * G_ + 4 * li + 4 * LPG * v;
                    float w[4], s4[4], G[4], ds[4];
                    WT::unpack(*reinterpret_cast<const typename WT::raw*>(st + St::OFF_W + el * St::WBYTES), w);
                    f4_to(*reinterpret_cast<const float4*>(st + St::OFF_S + el * 4), s4);
                    f4_to(*reinterpret_cast<const float4*>(st + St::OFF_G + el * 4), G);
                    const uint32_t cv = *reinterpret_cast<const uint32_t*>(st + St::OFF_C + el);
                    ragged_bwd_vec4<Q, ELEM>(w, s4, G, cv, t[gs], dl, sr, zu, tau, eg, ds, acc);
                    if (ok) *reinterpret_cast<float4*>(DS + ebase + el) = make_float4(ds[0], ds[1], ds[2], ds[3]);
                }
                const int slot0 = SR8::run(acc, lane);
                if (ok && SR8::writer(lane)) {
                    const int64_t grp = u.g0 + sub;
#pragma unroll
                    for (int q8 = 0; q8 < SR8::NOUT; ++q8) {
                        const int slot = slot0 + q8;
                        const float tot = acc[q8];
                        const float dt = dl * tot;
                        const float val = slot == 0 ? tot : slot == 1 ? -dt : dt;
                        float* dst = slot == 0 ? DDELTA + grp
                                     : slot == 1 ? DZU + grp
                                     : slot == 2 ? DZB + grp
                                     : DALPHA + grp * Q + (slot >= 4 ? slot - 4 : 0);
                        prow = slot == 3 ? prow + dt : prow;
                        if (slot != 3 && slot < 4 + Q) *dst = val;
                    }
                }
            }
            __syncwarp();                                // stage s and the tables are free again
            if (alive && issued < it.total) {
                issue(ic, s);
                ic.next(it.n_w);
                ++issued;
            }
            ring.next();
        }
        prow = warp_sum(prow);
        if (lane == 0) red[k % kRaggedRing][warp] = prow;
        // ds_r of the last kRaggedRing row blocks, once the ring is full or at the end
        if (k % kRaggedRing == kRaggedRing - 1 || k == n_mine - 1) {
            __syncthreads();
            const int k0 = k - k % kRaggedRing;
            const int WPR = kWarps / R;
            for (int idx = threadIdx.x; idx < (k - k0 + 1) * R; idx += kThreads) {
                const int kk = k0 + idx / R, rsub = idx % R;
                const int64_t r = ((int64_t)blockIdx.x + (int64_t)kk * gridDim.x) * R + rsub;
                if (r < out) {
                    const float* rr = red[kk % kRaggedRing];
                    float s = rr[rsub * WPR];
                    for (int w = 1; w < WPR; ++w) s += rr[rsub * WPR + w];
                    DSR[r] = -s / __ldg(SR + r);
                }
            }
            __syncthreads();
        }
    }
    if (!alive && lane == 0 && !drain(bars[warp], waited, issued)) atomicOr(&g_ragged_err, kDrainTimeoutBit);
}

template <typename St, bool ELEM>
struct RaggedBwdTag {};

template <int Q, typename WT, int G_, bool ELEM>
static cudaError_t run_ragged_bwd(const Shape& sh, const void* W, uq_params p, const uint8_t* codes, const float* gup,
                                  uq_grads gr, cudaStream_t st) {
    using St = RaggedBwdStage<Q, WT, G_>;
    const int U = (sh.n_in / G_ + St::NG - 1) / St::NG;
    const int R = rows_per_block(U);
    const int n_rb = (int)((sh.out + R - 1) / R);
    const size_t dyn = (size_t)kWarps * St::WARP_BYTES;
    auto kern = ragged_bwd_kernel<Q, WT, G_, ELEM>;
    int grid = 0;
    cudaError_t e = grid_for<RaggedBwdTag<St, ELEM>>(kern, dyn, n_rb, grid);
    if (e != cudaSuccess) return e;
    const RaggedSrc src{static_cast<const unsigned char*>(W), reinterpret_cast<const unsigned char*>(p.s),
                        reinterpret_cast<const unsigned char*>(gup), codes, p.delta, p.zu, p.zb, p.alpha};
    return launch_dependent(kern, grid, kThreads, dyn, st, src, p.sr, gr.ds, gr.dsr, gr.ddelta, gr.dzu, gr.dzb,
                            gr.dalpha, sh.out, sh.n_in, R, n_rb);
}

template <int Q, int G_>
static cudaError_t ragged_bwd_g(const Shape& sh, const void* W, uq_params p, const uint8_t* codes, const float* gup,
                                uq_grads gr, int filter, cudaStream_t st) {
    const bool elem = filter == UQ_FILTER_ELEMENT;
    if (sh.wdtype == UQ_W_BF16)
        return elem ? run_ragged_bwd<Q, WBF16, G_, true>(sh, W, p, codes, gup, gr, st)
                    : run_ragged_bwd<Q, WBF16, G_, false>(sh, W, p, codes, gup, gr, st);
    return elem ? run_ragged_bwd<Q, WF32, G_, true>(sh, W, p, codes, gup, gr, st)
                : run_ragged_bwd<Q, WF32, G_, false>(sh, W, p, codes, gup, gr, st);
}

template <int Q>
static cudaError_t ragged_bwd_q(const Shape& sh, const void* W, uq_params p, const uint8_t* codes, const float* gup,
                                uq_grads gr, int filter, cudaStream_t st) {
    switch (sh.g) {
        case 32: return ragged_bwd_g<Q, 32>(sh, W, p, codes, gup, gr, filter, st);
        case 64: return ragged_bwd_g<Q, 64>(sh, W, p, codes, gup, gr, filter, st);
        case 128: return ragged_bwd_g<Q, 128>(sh, W, p, codes, gup, gr, filter, st);
        case 256: return ragged_bwd_g<Q, 256>(sh, W, p, codes, gup, gr, filter, st);
        default: return ragged_bwd_g<Q, 512>(sh, W, p, codes, gup, gr, filter, st);
    }
}

cudaError_t launch_bwd_ragged(const Shape& sh, const void* W, uq_params p, const uint8_t* codes, const float* gup,
                              uq_grads gr, cudaStream_t st, int filter) {
    switch (sh.q) {
        case 1: return ragged_bwd_q<1>(sh, W, p, codes, gup, gr, filter, st);
        case 2: return ragged_bwd_q<2>(sh, W, p, codes, gup, gr, filter, st);
        case 3: return ragged_bwd_q<3>(sh, W, p, codes, gup, gr, filter, st);
        default: return ragged_bwd_q<4>(sh, W, p, codes, gup, gr, filter, st);
    }
}

cudaError_t ragged_bwd_error(bool clear, unsigned int* flag) {
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
