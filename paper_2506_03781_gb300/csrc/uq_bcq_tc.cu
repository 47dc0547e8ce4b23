// BCQ product on the tensor cores: y = W~ x with
// W~[r, i] = sum_j alpha*_{r,k,j} c_{j,r,i} + z*_{r,k} (k = i / g) from the
// exported bit-planes, as one +-1 matrix product per plane and block of GB
// columns of one group (GB = 32, 64, or 128 for larger groups):
//   y_r += sum_j alpha*_j (C_j x)_r + z* S,   S = sum of x over the block.
//
// The entries are exact in bf16 and so are the activations: a bf16 token
// is one column of the right-hand matrix, an fp32 token three (its value cut
// into three bf16 pieces that add up to it), so every product is exact and the
// sums D_j are taken in fp32 (tcgen05.mma kind::f16, 128 rows by
// N columns, fp32 accumulators in tensor memory).  With 64 columns, or with
// several blocks to a pass, the entries are +-1 themselves, made by two
// operations per pair.  Else, where making them is the longest part of the chain
// (450 of 750 clocks), they are of four kinds, one operation
// each wherever the bit lies (see expand16): +-0.5; 2 or 0, against half the
// activation; 1 or 2^-64; 1 or 2^-32.  With S0 the sum of x over the columns
// of the first kind, (C_j x)_r = 2 D_j + S0 - S then, but for the 2^-64 and
// 2^-32 of the clear bits, at most 2^-33 of sum |x|.
//
// Pieces, halves and sums leave the range of bf16 or fp32 where activations
// are near its ends.  So a token whose largest activation in a slice is below
// 2^-64 is multiplied by 2^64 there, one of 2^110 or more by 2^-32, and its
// sums are multiplied back.  Of the others, what lies below the smallest bf16
// number, 2^-133, is lost: less than 2^-69 of the largest.  The operands are
// built without a look at this first, and again in the blocks that meet such a
// number (64 tokens of 14336 x 4096: 39.8 us without the look, 40.2 with it;
// with a scale for each pass, applied in the loop over the passes, 43.2).
//
// A warpgroup owns 128 rows, one per thread.  For every plane and 128
// columns a thread expands the row's four plane words in registers and stores
// them to tensor memory, which is the left operand; element k = 2 (16 word +
// p) + h of a row is bit p + 16 h of the word, so a register holds the bits p
// and p + 16.  The block keeps the activations of
// its column slice in shared memory in the same column order (K-major core
// matrices of 8 tokens x 16 bytes, no swizzle).  The sums come back one row per thread and are scaled
// by that row's alpha* in registers.  Operand and sums have two buffers each:
// a plane is expanded while the products of the one before run.  One to three
// warpgroups per block, each with its own rows and its own part of tensor
// memory, cover each other's waits.  The products and copies of a warpgroup
// are issued by one more warp of its own, so none of the four ever waits for
// another one (one such warp for all warpgroups issued a plane every 500
// clocks: its fence waits for the products that it issued before).
//
// The plane words come through a ring of shared-memory stages per warpgroup,
// filled by tensor copies (box: 16 kTcSbs bytes of 128 rows of all planes,
// swizzled so that one row per thread reads without bank conflicts); where
// rows are not whole 128-column passes every thread loads its row's words.
//
// Split: block (slice, row block) keeps one column slice of all tokens of its
// chunk and walks its 128-row tiles.  With one slice the result is y itself,
// else the slices go to the caller's workspace [slice][token][row] and are
// summed in order by a second kernel.  Every wait on a barrier is bounded; the
// wait for the work ahead on the stream and the allocation of tensor memory are
// the hardware's, and the order of the two (see the kernel) lets no block hold
// tensor memory that a kernel it waits for needs.  Deterministic; no atomics on
// outputs.
//
// What bounds it: latency.  A warpgroup takes each plane through one chain
// (expand, store, wait for the products of the plane before, read the sums,
// scale them: 1270 clocks with 64 columns, 750 with 16), and two or three share
// an SM, which takes 1180 and 520 clocks a plane of 128 x 128 where the tensor
// cores need 272 and 197.  Counters of 64 tokens of 14336 x 4096 and 4 fp32 tokens
// of 8192 x 28672: tensor pipe 27 and 16 %, logic pipe 22 and 42 %, issue 0.47 and
// 0.52, the largest stall the reads of tensor memory.  q = 3, g = 128, six sets of
// inputs in turn: 64 bf16 tokens of 14336 x 4096 40.2 us (per-token lookup tables
// 447), 16 tokens 21.4 (114), 4 tokens 20.5 (30); 8192 x 28672, 4 fp32 tokens 69.8
// (99.8).  The same product with mma.sync and fragments in registers took 72.5 us
// for 64 tokens and 108 for the 4: every lane of a quad repeats the loads and the
// scaling, and 64 columns are bound by that pipe (38 us).
// Error against 64 bits: 0.6e-7 to 1.3e-7, the lookup tables' 0.7e-7 to 1.7e-7.
#include <cuda.h>   // CUtensorMap
#include <cuda_bf16.h>

#include <atomic>

#include "uq_common.cuh"
#include "uq_launch.h"
#include "uq_pipe.cuh"

namespace uq {

static __device__ unsigned int g_tc_err = 0;

// Tensor map of the bit-planes (uq_gemv.cu); false if the driver cannot encode it.
bool bcq_planes_map(const uint32_t* planes, int64_t out, int n_in, int q, int box_words, int box_rows, CUtensorMap* map);

constexpr int kTcCols = 128;                      // columns of one pass
constexpr int kTcRows = 128;                      // rows of a tile: one per thread of a warpgroup
constexpr int kTcMaxGroups = 3;                   // warpgroups per block
constexpr int kTcSmem = 226 * 1024;               // dynamic shared memory a block may use
constexpr int kTcMinSmem = 116 * 1024;            // more than half an SM: one block, one user of tensor memory, per SM

// Passes of a stage, and stages of a warpgroup's ring.
__host__ __device__ constexpr int tc_sbs(int n) { return n == 64 ? 2 : 4; }
constexpr int kTcStages = 2;
__host__ __device__ constexpr int tc_stage_bytes(int q, int n) { return q * kTcRows * 16 * tc_sbs(n); }
// Tensor-memory columns of one warpgroup: two expanded planes (64 each) and
// two buffers of the sums of a pass's blocks.
__host__ __device__ constexpr int tc_tmem_cols(int gb, int n) { return 2 * (64 + kTcCols / gb * n); }
__host__ __device__ constexpr int tc_groups(int gb, int n) {
    return 512 / tc_tmem_cols(gb, n) < kTcMaxGroups ? 512 / tc_tmem_cols(gb, n) : kTcMaxGroups;
}
// Entries of four kinds instead of +-1, and the sums kept per block and column: S, and S0 - S for the kinds.
__host__ __device__ constexpr bool tc_kinds(int gb, int n) { return gb == 128 && n < 64; }
__host__ __device__ constexpr int tc_pass_bytes(int gb, int n) {
    return kTcCols * n * 2 + kTcCols / gb * n * (tc_kinds(gb, n) ? 8 : 4);
}

namespace tc {

__device__ __forceinline__ void alloc(uint32_t dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void dealloc(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// One lane of a converged warp.
__device__ __forceinline__ uint32_t elect() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(p));
    return p;
}
// d (128 x N, fp32) = a (128 x 16, tensor memory) b (16 x N, shared memory) + d if acc,
// issued by the elected lane.  Called by the whole warp with uniform
// arguments: inside a branch of one thread the operands cannot be uniform
// registers, and an issue took 85 to 195 clocks instead of 25 (16 columns).
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc, uint32_t elected) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(acc), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void load_box(uint32_t dst, const CUtensorMap* m, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 words per thread: lane i of the warp holds row i of its 32 rows
__device__ __forceinline__ void load(uint32_t addr, float (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(addr)
        : "memory");
}

__device__ __forceinline__ void store(uint32_t addr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::
            "r"(addr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// Instruction descriptor: fp32 sums, bf16 operands, both K-major, M = 128.
__host__ __device__ constexpr uint32_t idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcRows >> 4) << 24);
}
// Shared-memory descriptor without swizzle: core matrices of 8 rows x 16
// bytes, 128 bytes apart over the rows and n * 16 bytes apart over K.
__device__ __forceinline__ uint64_t desc(uint32_t addr, int n) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)(n) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

}  // namespace tc

// Bits p and p + 16 of w as two bf16 values.  Shifted left by 12 - 4 (p / 4)
// the two lie at positions 12 + p % 4 of the halves, where one three-input
// logic operation turns them into numbers:
//   15: sign of 0.5                        (t & 8000) ^ bf00: set 0.5, clear -0.5
//   14: top bit of the exponent            t & 4000: 2 or 0
//   13: second bit, the rest as in 1.0     (t & 2000) | 1f80: 1 or 2^-64
//   12: third bit, likewise                (t & 1000) | 2f80: 1 or 2^-32
// so a word takes 3 shifts and 16 logic operations (15 and 16 with one
// position for all).  The constants come from the kernel's arguments: a second
// immediate would cost a second operation.
struct Expand {
    uint32_t mask[4], fill[4];                              // positions 12, 13, 14, 15
    uint32_t mul[16];                                       // 2^(15 - p), for pm1
};
__device__ __forceinline__ void expand16(uint32_t w, const uint32_t (&mask)[4], const uint32_t (&fill)[4], uint32_t (&a)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t t = i == 3 ? w : w << (12 - 4 * i);
        asm("lop3.b32 %0, %1, %2, %3, 0xea;" : "=r"(a[4 * i]) : "r"(t), "r"(mask[0]), "r"(fill[0]));
        asm("lop3.b32 %0, %1, %2, %3, 0xea;" : "=r"(a[4 * i + 1]) : "r"(t), "r"(mask[1]), "r"(fill[1]));
        a[4 * i + 2] = t & mask[2];
        asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(a[4 * i + 3]) : "r"(t), "r"(mask[3]), "r"(fill[3]));
    }
}
// The same pairs as +-1: moved to the sign positions by a product (it runs
// beside the logic operations) and one logic operation.
__device__ __forceinline__ void expand16_pm1(uint32_t w, const uint32_t (&mul)[16], uint32_t mask, uint32_t one, uint32_t (&a)[16]) {
#pragma unroll
    for (int p = 0; p < 16; ++p)
        asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(a[p]) : "r"(p == 15 ? w : w * mul[p]), "r"(mask), "r"(one));
}
// Half of both bf16 values of a pair (but for subnormal results exact: see tc_scale).
__device__ __forceinline__ uint32_t half_pair(uint32_t v) {
    const __nv_bfloat162 h = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&v), __floats2bfloat162_rn(0.5f, 0.5f));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Piece 0, 1 or 2 of an fp32 value: three bf16 numbers that add up to it (8
// significant bits each, cut and not rounded, so none overflows; exactly from
// 2^-109 on).  Infinities and NaN stay in piece 0.
__device__ __forceinline__ uint32_t bf16_piece(float x, int piece) {
    const uint32_t b = __float_as_uint(x);
    if ((b & 0x7f800000u) == 0x7f800000u) return piece ? 0u : (b & 0x007fffffu) ? 0x7fc0u : b >> 16;
    const uint32_t h0 = b & 0xffff0000u;
    const float r = __fsub_rn(x, __uint_as_float(h0));
    const uint32_t h1 = __float_as_uint(r) & 0xffff0000u;
    if (piece == 0) return h0 >> 16;
    if (piece == 1) return h1 >> 16;
    return __float_as_uint(__fsub_rn(r, __uint_as_float(h1))) >> 16;
}

// What a token is multiplied by in a slice, from the bits of its largest |x| there,
// and what its sums are multiplied by.
constexpr uint32_t kTcTiny = (127u - 64u) << 23, kTcHuge = (127u + 110u) << 23;
__device__ __forceinline__ float tc_scale(uint32_t top) {
    return top >= kTcHuge ? 0x1p-32f : top < kTcTiny ? 0x1p64f : 1.f;
}
__device__ __forceinline__ float tc_unscale(uint32_t top) {
    return top >= kTcHuge ? 0x1p32f : top < kTcTiny ? 0x1p-64f : 1.f;
}

// The activations of a slice in operand order, into xs [sb][16][N], and their
// block sums; true where the thread met one that asks for scaling.  SCALED:
// with tops, the largest |x| of each token in the slice.
template <int GB, int N, bool SCALED>
__device__ __forceinline__ bool tc_operands(uint4* xs, float* sums, const uint32_t* tops, const void* __restrict__ X, int x_bf16,
                                            int n_in, int tok0, int toks, int sb0, int sbn, int warp, int nw, int lane) {
    constexpr int NB = kTcCols / GB;
    constexpr bool KINDS = tc_kinds(GB, N);
    constexpr int NSUM = KINDS ? 2 : 1;
    const int words = n_in / 32;
    bool odd = false;
    for (int it = warp; it < sbn * (N / 8); it += nw) {
        const int sb = it / (N / 8), n8 = it - sb * (N / 8);
        const int tig = lane & 3, col = n8 * 8 + (lane >> 2);
        const int tok = x_bf16 ? col : col / 3, piece = x_bf16 ? 0 : col - tok * 3;
        const int word = (sb0 + sb) * 4 + tig;
        uint32_t pr[16];                                   // columns p and p + 16 of the word
        uint32_t any = 0;                                  // bits of all of them (fp32)
        float sum = 0.f, sum0 = 0.f;                       // S, and its columns of the first kind (bits 3, 7, 11, 15)
        if (tok < toks && word < words) {
            const int64_t x0 = (int64_t)(tok0 + tok) * n_in + (int64_t)word * 32;
            const float scale = SCALED ? tc_scale(tops[tok]) : 1.f;
            if (x_bf16) {
                const uint4* p = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(X) + x0);
                uint32_t u[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = __ldg(p + i);
                    u[4 * i] = v.x; u[4 * i + 1] = v.y; u[4 * i + 2] = v.z; u[4 * i + 3] = v.w;
                }
                if (SCALED) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        u[i] = __byte_perm(__float_as_uint(__uint_as_float(u[i] << 16) * scale),
                                           __float_as_uint(__uint_as_float(u[i] & 0xffff0000u) * scale), 0x7632);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    pr[2 * i] = __byte_perm(u[i], u[i + 8], 0x5410);
                    pr[2 * i + 1] = __byte_perm(u[i], u[i + 8], 0x7632);
                }
            } else {
                const float4* p = reinterpret_cast<const float4*>(static_cast<const float*>(X) + x0);
                // x less its upper 16 bits once for piece 1 and twice for piece 2, then cut
                const uint32_t m1 = piece >= 1 ? 0xffff0000u : 0u, m2 = piece == 2 ? 0xffff0000u : 0u;
                auto cut = [&](float v) {
                    v = __fsub_rn(v, __uint_as_float(__float_as_uint(v) & m1));
                    v = __fsub_rn(v, __uint_as_float(__float_as_uint(v) & m2));
                    return __float_as_uint(v);
                };
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float lo[4], hi[4];
                    f4_to(__ldg(p + i), lo);
                    f4_to(__ldg(p + i + 4), hi);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (SCALED) {
                            pr[4 * i + k] = bf16_piece(lo[k] * scale, piece) | (bf16_piece(hi[k] * scale, piece) << 16);
                        } else {
                            any |= __float_as_uint(lo[k]) | __float_as_uint(hi[k]);
                            pr[4 * i + k] = __byte_perm(cut(lo[k]), cut(hi[k]), 0x7632);
                        }
                    }
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) pr[i] = 0u;
        }
        if (!SCALED && piece == 0) {                       // (the other pieces see the same activations)
            uint32_t top = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) top = __vmaxu2(top, pr[i] & 0x7fff7fffu);
            top = max(top & 0xffffu, top >> 16);
            odd |= top >= kTcHuge >> 16 || (top < kTcTiny >> 16 && ((top | any) & 0x7fffffffu) != 0u);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float v = __uint_as_float(pr[i] << 16) + __uint_as_float(pr[i] & 0xffff0000u);
            if (i % 4 == 3) sum0 += v;
            else sum += v;
            if (KINDS && i % 4 == 2) pr[i] = half_pair(pr[i]);
        }
        // sum: the columns of the other kinds, S - S0
        if (GB >= 64) {
            sum += __shfl_xor_sync(kFull, sum, 1);
            sum0 += __shfl_xor_sync(kFull, sum0, 1);
        }
        if (GB >= 128) {
            sum += __shfl_xor_sync(kFull, sum, 2);
            sum0 += __shfl_xor_sync(kFull, sum0, 2);
        }
        if (tig % (4 / NB) == 0) {
            float* d = sums + ((sb * NB + tig / (4 / NB)) * N + col) * NSUM;
            d[0] = sum + sum0;
            if (KINDS) d[NSUM - 1] = -sum;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v)
            xs[(sb * 16 + tig * 4 + v) * N + col] = make_uint4(pr[4 * v], pr[4 * v + 1], pr[4 * v + 2], pr[4 * v + 3]);
    }
    return odd;
}

// ... once more for a slice with tiny or huge activations: first the largest of each token.  Whole block.
template <int GB, int N>
__device__ __noinline__ void tc_scaled_operands(uint4* xs, float* sums, uint32_t* tops, const void* __restrict__ X, int x_bf16,
                                                int n_in, int tok0, int toks, int sb0, int sbn, int warp, int nw, int lane) {
    const int c0 = sb0 * kTcCols, c1 = min(n_in, c0 + sbn * kTcCols);
    for (int t = warp; t < toks; t += nw) {
        uint32_t top = 0;
        for (int c = c0 + lane; c < c1; c += 32) {
            const int64_t i = (int64_t)(tok0 + t) * n_in + c;
            const uint32_t b = x_bf16 ? (uint32_t)__ldg(static_cast<const unsigned short*>(X) + i) << 16
                                      : __float_as_uint(__ldg(static_cast<const float*>(X) + i));
            top = max(top, b & 0x7fffffffu);
        }
        top = __reduce_max_sync(kFull, top);
        if (lane == 0) tops[t] = top;
    }
    __syncthreads();
    tc_operands<GB, N, true>(xs, sums, tops, X, x_bf16, n_in, tok0, toks, sb0, sbn, warp, nw, lane);
}

// Waits (bounded) for a warpgroup's last stages of the ring, of `copies` in all,
// and for the last product of each buffer: ph has the parities of the next ones,
// so of a phase before the first where there was none.
__device__ __noinline__ void tc_drain(unsigned long long (&full)[kTcStages], int copies, unsigned long long (&done)[2], uint32_t ph) {
    bool landed = drain(full, copies > kTcStages ? copies - kTcStages : 0, copies);
    for (int k = 0; k < 2; ++k) landed &= tma::bar_wait(tma::smem_addr(&done[k]), ((ph >> k) & 1u) ^ 1u);
    if (!landed) atomicOr(&g_tc_err, kDrainTimeoutBit);
}

template <int Q, int GB, int N>
__global__ void __launch_bounds__(tc_groups(GB, N) * 160, 1)
bcq_tc_kernel(const __grid_constant__ CUtensorMap tm_planes, const uint32_t* __restrict__ PLANES,
              const float* __restrict__ ASTAR, const float* __restrict__ ZSTAR, const void* __restrict__ X, int x_bf16,
              float* __restrict__ DST, int64_t out, int n_in, int g, int batch, int n_ks, int sb_per, int tiles,
              int tmem_cols, int staged, const __grid_constant__ Expand ex) {
    constexpr int NB = kTcCols / GB;                       // scaling blocks of one pass
    constexpr int SBS = tc_sbs(N), SB = tc_stage_bytes(Q, N);
    constexpr bool KINDS = tc_kinds(GB, N);
    constexpr int NSUM = KINDS ? 2 : 1;
    extern __shared__ __align__(128) unsigned char tsm[];
    // per warpgroup and buffer: plane expanded (its four warps), products done; per stage: copies landed
    __shared__ __align__(8) unsigned long long ready[kTcMaxGroups][2], done[kTcMaxGroups][2], full[kTcMaxGroups][kTcStages];
    __shared__ uint32_t tm_addr;
    __shared__ volatile int dead;                          // a wait ran out: every warp stops
    __shared__ int started[kTcMaxGroups][2];               // by a warpgroup's issuing warp: stages, products (parities)
    __shared__ volatile int scaled;                        // some token of the slice is
    __shared__ uint32_t tops[N];                           // largest |x| of each token there
    const int warp = __shfl_sync(kFull, threadIdx.x >> 5, 0), lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    // warps 0 .. 4 n_wg - 1: four of each warpgroup; then the issuing warp of each
    const int n_wg = blockDim.x / 160, wt = threadIdx.x & 127;
    const bool issuer = warp >= 4 * n_wg;
    const int wg = issuer ? warp - 4 * n_wg : warp >> 2;
    const int slice = (int)(blockIdx.x % n_ks);
    const int64_t tile0 = (int64_t)(blockIdx.x / n_ks) * tiles;
    const int words = n_in / 32, Gr = n_in / g;
    const int n_sb = (n_in + kTcCols - 1) / kTcCols;
    const int sb0 = slice * sb_per, sbn = n_sb - sb0 < sb_per ? n_sb - sb0 : sb_per;
    const int tpc = x_bf16 ? N : N / 3;                    // tokens of a chunk
    const int tok0 = (int)blockIdx.y * tpc, toks = batch - tok0 < tpc ? batch - tok0 : tpc;
    // stages first (on a 1024-byte boundary), then the activations and the block sums
    unsigned char* base = tsm + ((1024u - (tma::smem_addr(tsm) & 1023u)) & 1023u);
    uint4* xs = reinterpret_cast<uint4*>(base + (staged ? (size_t)n_wg * kTcStages * SB : 0));      // [sb][16][N]
    float* sums = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(xs) + (size_t)sb_per * kTcCols * N * 2);

    if (threadIdx.x < kTcMaxGroups) {
        const int i = threadIdx.x;
        for (int k = 0; k < 2; ++k) {
            tma::bar_init(tma::smem_addr(&ready[i][k]), 4);
            tma::bar_init(tma::smem_addr(&done[i][k]), 1);
        }
        for (int k = 0; k < kTcStages; ++k) tma::bar_init(tma::smem_addr(&full[i][k]), 1);
        dead = scaled = 0;
        tma::bar_init_fence();
    }
    // Launched as a programmatic dependent: nothing global is touched before the work ahead has
    // completed, and no tensor memory is taken.  A block of the kernel ahead may need what is left of
    // it on this SM, and a block that held some while it waited for that kernel would never end.
    inputs_ready();
    if (warp == 0) tc::alloc(tma::smem_addr(&tm_addr), (uint32_t)tmem_cols);
    __syncthreads();
    // The next kernel (the slice sum first of all) may be scheduled only now, for the same reason: one
    // that takes tensor memory before it waits for this grid finds that every block here has its own.
    dependents_may_start();

    // stages of a warpgroup: tile-major, spt per tile
    const int spt = (sbn + SBS - 1) / SBS;
    const int64_t row_tiles = (out + kTcRows - 1) / kTcRows;
    const int n_tiles = (int)(row_tiles - tile0 < tiles ? row_tiles - tile0 : tiles);
    auto tiles_of = [&](int w) { return n_tiles > w ? (n_tiles - w + n_wg - 1) / n_wg : 0; };
    auto copy = [&](int w, int i) {                        // stage i of warpgroup w
        const int s = i & (kTcStages - 1), t = i / spt;
        const uint32_t fb = tma::smem_addr(&full[w][s]);
        tma::fence_async_smem();                           // the warpgroup's reads of this stage come first
        tma::bar_arrive_tx(fb, (uint32_t)SB);
        tc::load_box(tma::smem_addr(base + ((size_t)w * kTcStages + s) * SB), &tm_planes, (sb0 + (i - t * spt) * SBS) * 4,
                     (int)((tile0 + w + (int64_t)t * n_wg) * kTcRows), 0, fb);
    };
    const int my_tiles = tiles_of(wg);
    if (staged && issuer && lane == 0)
        for (int i = 0; i < kTcStages && i < my_tiles * spt; ++i) copy(wg, i);

    // --- the slice's activations in operand order, and their block sums ---
    if (tc_operands<GB, N, false>(xs, sums, nullptr, X, x_bf16, n_in, tok0, toks, sb0, sbn, warp, nw, lane)) scaled = 1;
    __syncthreads();
    if (scaled) tc_scaled_operands<GB, N>(xs, sums, tops, X, x_bf16, n_in, tok0, toks, sb0, sbn, warp, nw, lane);
    tma::fence_async_smem();                               // the products read shared memory through the async proxy
    tc::fence_before();
    __syncthreads();
    tc::fence_after();

    const uint32_t xbase = tma::smem_addr(xs);
    if (issuer) {
        // --- products and copies of the warpgroup: the whole warp, uniformly; one lane issues ---
        const uint32_t e = tc::elect();
        const uint32_t tm = __shfl_sync(kFull, tm_addr, 0) + (uint32_t)(wg * tc_tmem_cols(GB, N));
        const uint64_t xdesc = tc::desc(xbase, N);
        uint32_t b = 0, ph = 0;                             // next buffer, parities of its barriers
        int stage = 0;
        bool go = true;
        for (int t = 0; t < my_tiles && go; ++t)
            for (int sb = 0; sb < sbn && go; ++sb) {
                const uint64_t xd = xdesc + (uint32_t)(sb * 16 * N);               // 16-byte units
#pragma unroll 1
                for (int j = 0; j < Q; ++j) {
                    if (!__all_sync(kFull, tma::bar_wait(tma::smem_addr(&ready[wg][b]), (ph >> b) & 1u))) {
                        if (lane == 0) atomicOr(&g_tc_err, 4u);
                        dead = 1;
                    }
                    if (__any_sync(kFull, dead)) { go = false; break; }
                    tc::fence_after();
#pragma unroll
                    for (int k = 0; k < 8; ++k)             // 16 columns a step, 8 / NB steps a block
                        tc::mma(tm + 128 + (b * NB + k / (8 / NB)) * N, tm + 64 * b + 8 * k, xd + 2 * k * N, tc::idesc(N),
                                k % (8 / NB) ? 1u : 0u, e);
                    if (e) tc::commit(tma::smem_addr(&done[wg][b]));
                    __syncwarp();
                    ph ^= 1u << b;
                    b ^= 1u;
                }
                // the last plane of a stage has been read: its slot is free
                if (staged && go && (sb == sbn - 1 || sb % SBS == SBS - 1)) {
                    if (e && stage + kTcStages < my_tiles * spt) copy(wg, stage + kTcStages);
                    __syncwarp();
                    ++stage;
                }
            }
        // what this warp has started, for the wait at the end (kept in shared memory, and waited for by one
        // warp: in this branch it cost the whole kernel registers and 2.4 of 40.2 us)
        const int total = staged ? my_tiles * spt : 0, copies = stage + kTcStages < total ? stage + kTcStages : total;
        if (lane == 0) {
            started[wg][0] = copies;
            started[wg][1] = (int)ph;
        }
    }
    const uint32_t tmem = tm_addr + (uint32_t)(wg * tc_tmem_cols(GB, N));
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);         // this warp's 32 rows
    const unsigned char* ring = base + (size_t)wg * kTcStages * SB;
    const int64_t pstride = out * words;
    const int gdiv = g > kTcCols ? g / kTcCols : 1;        // passes per group
    const bool vec = g <= kTcCols && (Gr & 3) == 0;        // four groups of a row are 16-byte aligned
    const bool vec2 = gdiv == 2 && (Gr & 1) == 0;          // two groups of two passes each, 8-byte aligned
    uint32_t phase = 0;                                    // bit b: parity of buffer b's next completion
    int buf = 0, waited = 0;                               // buffer of the next plane; stages waited for
    bool alive = true;
    uint32_t mask[4], fill[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { mask[i] = ex.mask[i]; fill[i] = ex.fill[i]; }

    for (int mt = 0; mt < my_tiles && alive && !issuer; ++mt) {
        const int64_t row_raw = (tile0 + wg + (int64_t)mt * n_wg) * kTcRows + wt;
        const int64_t row = row_raw < out ? row_raw : out - 1;     // rows past the last one are not stored
        float acc[N], v[N];
#pragma unroll
        for (int n = 0; n < N; ++n) acc[n] = 0.f;

        // alpha* and z* of four blocks of the row at a time
        float pa[4][Q], pz[4];
        auto params = [&](int b0) {                        // blocks b0 .. b0 + 3 of the row
            if (vec) {
                if (b0 < Gr) {
                    const float4* a4 = reinterpret_cast<const float4*>(ASTAR + (row * Gr + b0) * Q);
                    float f[4 * Q];
#pragma unroll
                    for (int i = 0; i < Q; ++i) f4_to(__ldg(a4 + i), f + 4 * i);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int j = 0; j < Q; ++j) pa[k][j] = f[k * Q + j];
                    f4_to(__ldg(reinterpret_cast<const float4*>(ZSTAR + row * Gr + b0)), pz);
                }
            } else if (vec2) {                             // (value by value: 8192 x 8192, 4 tokens 32.5 vs 23.7 us)
                const int grp = b0 >> 1;
                if (grp < Gr) {
                    const float2* a2 = reinterpret_cast<const float2*>(ASTAR + (row * Gr + grp) * Q);
                    float f[2 * Q];
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const float2 t2 = __ldg(a2 + i);
                        f[2 * i] = t2.x;
                        f[2 * i + 1] = t2.y;
                    }
                    const float2 z2 = __ldg(reinterpret_cast<const float2*>(ZSTAR + row * Gr + grp));
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        pz[k] = k < 2 ? z2.x : z2.y;
#pragma unroll
                        for (int j = 0; j < Q; ++j) pa[k][j] = f[(k >> 1) * Q + j];
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int grp = (b0 + k) / gdiv;
                    const bool in = grp < Gr;
                    pz[k] = in ? __ldg(ZSTAR + row * Gr + grp) : 0.f;
#pragma unroll
                    for (int j = 0; j < Q; ++j) pa[k][j] = in ? __ldg(ASTAR + (row * Gr + grp) * Q + j) : 0.f;
                }
            }
        };
        // expands the warp's rows of plane j of pass sb into operand buffer b
        auto expand = [&](int sb, int j, int b) {
            if (staged && j == 0 && sb % SBS == 0) {
                const int s = waited & (kTcStages - 1);
                if (!tma::bar_wait(tma::smem_addr(&full[wg][s]), (uint32_t)(waited / kTcStages) & 1u)) {
                    atomicOr(&g_tc_err, 2u);
                    dead = 1;
                }
                ++waited;
                __syncwarp();
            }
            uint4 w4;
            if (staged) {
                const unsigned char* st = ring + ((waited - 1) & (kTcStages - 1)) * SB + j * (kTcRows * 16 * SBS);
                const int c = sb % SBS, x = SBS == 4 ? (wt >> 1) & 3 : (wt >> 2) & 1;      // the copy's swizzle
                w4 = *reinterpret_cast<const uint4*>(st + wt * 16 * SBS + ((c ^ x) << 4));
            } else {
                const int word = (sb0 + sb) * 4;
                const uint32_t* p = PLANES + row * words + j * pstride + word;
                w4.x = __ldg(p);
                w4.y = word + 1 < words ? __ldg(p + 1) : 0u;
                w4.z = word + 2 < words ? __ldg(p + 2) : 0u;
                w4.w = word + 3 < words ? __ldg(p + 3) : 0u;
            }
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t a[16];
                if constexpr (KINDS) expand16(w[i], mask, fill, a);
                else expand16_pm1(w[i], ex.mul, mask[3], fill[3], a);
                tc::store(tlane + 64 * b + 16 * i, a);
            }
            tc::wait_store();
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tma::bar_arrive(tma::smem_addr(&ready[wg][b]));
        };
        expand(0, 0, buf);
        int left = 0;                                      // blocks of pa, pz not yet used
        for (int sb = 0; sb < sbn && alive; ++sb) {
            if (left == 0) {
                const int b0 = ((sb0 + sb) * NB) & ~3, skip = (sb0 + sb) * NB - b0;
                params(b0);
                left = 4 - skip;
                for (int i = 0; i < skip; i += NB) {        // the slice begins inside the four
#pragma unroll
                    for (int k = 0; k + NB < 4; ++k) {
                        pz[k] = pz[k + NB];
#pragma unroll
                        for (int j = 0; j < Q; ++j) pa[k][j] = pa[k + NB][j];
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                if (j + 1 < Q) expand(sb, j + 1, buf ^ 1);
                else if (sb + 1 < sbn) expand(sb + 1, 0, buf ^ 1);
                if (!tma::bar_wait(tma::smem_addr(&done[wg][buf]), (phase >> buf) & 1u)) {
                    atomicOr(&g_tc_err, 1u);
                    dead = 1;
                }
                phase ^= 1u << buf;
                __syncwarp();
                tc::fence_after();
#pragma unroll
                for (int h = 0; h < NB; ++h) {
                    const float* S = sums + (sb * NB + h) * N * NSUM;
#pragma unroll
                    for (int n0 = 0; n0 < N; n0 += 16) {
                        float d[16];
                        tc::load(tlane + 128 + (buf * NB + h) * N + n0, d);
#pragma unroll
                        for (int n = 0; n < 16; ++n) {
                            // the block's terms first, then the running sum: one rounding per pass at its size
                            const float* s2 = S + (n0 + n) * NSUM;
                            if (j == 0) v[n0 + n] = h == 0 ? __fmul_rn(pz[h], s2[0]) : fmaf(pz[h], s2[0], v[n0 + n]);
                            const float cx = KINDS ? fmaf(2.f, d[n], s2[NSUM - 1]) : d[n];
                            v[n0 + n] = fmaf(pa[h][j], cx, v[n0 + n]);
                            if (j == Q - 1 && h == NB - 1) acc[n0 + n] += v[n0 + n];
                        }
                    }
                }
                buf ^= 1;
            }
            if (__any_sync(kFull, dead)) alive = false;
            left -= NB;
            if (NB < 4) {
#pragma unroll
                for (int k = 0; k + NB < 4; ++k) {
                    pz[k] = pz[k + NB];
#pragma unroll
                    for (int j = 0; j < Q; ++j) pa[k][j] = pa[k + NB][j];
                }
            }
        }
        if (alive && row_raw < out) {
            float* dst = DST + ((int64_t)slice * batch + tok0) * out + row;
            if (x_bf16) {
#pragma unroll
                for (int n = 0; n < N; ++n)
                    if (n < toks) dst[(int64_t)n * out] = acc[n];
            } else {
#pragma unroll
                for (int t = 0; t < N / 3; ++t)
                    if (t < toks) dst[(int64_t)t * out] = (acc[3 * t] + acc[3 * t + 1]) + acc[3 * t + 2];
            }
            if (scaled) {                                  // (from memory, for the registers' sake)
#pragma unroll 1
                for (int t = 0; t < toks; ++t) dst[(int64_t)t * out] *= tc_unscale(tops[t]);
            }
        }
    }
    // where a wait ran out, products and copies may still be in flight: they land before the block leaves
    __syncthreads();
    if (dead && warp == 0 && lane < n_wg) tc_drain(full[lane], started[lane][0], done[lane], (uint32_t)started[lane][1]);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::dealloc(tm_addr, (uint32_t)tmem_cols);
}

cudaError_t bcq_tc_error(bool clear, unsigned int* flag) {
    unsigned int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_err, sizeof(v));
    if (e != cudaSuccess) return e;
    *flag = v;
    if (clear && v) {
        const unsigned int z = 0;
        e = cudaMemcpyToSymbol(g_tc_err, &z, sizeof(z));
    }
    return e;
}

namespace {

struct TcPlan {
    int n_ks, sb_per, n_rb, tiles, groups;
};

// Slices, tiles per block and warpgroups for the least estimated time (in SM
// clocks): the waves of blocks, each with the operands it builds and its
// rounds of tiles, and the slice sum where there is more than one slice.  The
// constants order the plans and do not predict the time: a pass takes about
// twice as long (64 tokens of 14336 x 4096 19 us estimated, 40.2 taken; 4 fp32
// tokens of 8192 x 28672 34 and 69.8).
template <int Q, int GB, int N>
TcPlan tc_plan(int64_t out, int n_in, int chunks, bool staged) {
    const int sms = sm_count();
    const int n_sb = (n_in + kTcCols - 1) / kTcCols;
    const int64_t all = (out + kTcRows - 1) / kTcRows;
    const int most_ks = (n_in + 511) / 512;                // the workspace holds this many partials of every output
    // a pass of one plane: alone, and what it takes of the SM among others
    const double alone = 450.0 + 7.0 * N, busy = 4.5 * N > 200.0 ? 4.5 * N : 200.0;
    TcPlan best{};
    double best_cost = -1.0;
    for (int w = 1; w <= tc_groups(GB, N); ++w) {
        const int fit = (kTcSmem - 1024 - (staged ? w * kTcStages * tc_stage_bytes(Q, N) : 0)) / tc_pass_bytes(GB, N);
        const int least = (n_sb + fit - 1) / fit;
        for (int ks = least; ks <= most_ks && ks < least + 16; ++ks) {
            const int per = (n_sb + ks - 1) / ks, n_ks = (n_sb + per - 1) / per;
            for (int waves = 1; waves <= 2; ++waves) {
                int64_t n_rb = (int64_t)sms * waves / ((int64_t)n_ks * chunks);
                n_rb = n_rb < 1 ? 1 : n_rb > all ? all : n_rb;
                const int64_t tiles = (all + n_rb - 1) / n_rb;
                n_rb = (all + tiles - 1) / tiles;
                const int64_t wv = (n_rb * n_ks * chunks + sms - 1) / sms;
                const int ww = tiles < w ? (int)tiles : w;
                const int64_t rounds = (tiles + ww - 1) / ww;
                const double pass = alone > ww * busy ? alone : ww * busy;
                const double cost = (double)wv * (2500.0 + per * N * 12.0 / ww + (double)rounds * per * Q * pass) +
                                    (n_ks > 1 ? 3000.0 : 0.0);
                if (best_cost < 0.0 || cost < best_cost) {
                    best_cost = cost;
                    best = TcPlan{n_ks, per, (int)n_rb, (int)tiles, ww};
                }
            }
        }
    }
    return best;
}

template <int Q, int GB, int N>
cudaError_t run_tc(const uint32_t* planes, const float* astar, const float* zstar, int64_t out, int n_in, int g,
                   const void* x, int x_bf16, int batch, float* y, float* work, cudaStream_t st) {
    const int tpc = x_bf16 ? N : N / 3, chunks = (batch + tpc - 1) / tpc;
    // whole passes: the planes come through tensor copies
    CUtensorMap map = {};
    const bool staged = n_in % kTcCols == 0 && bcq_planes_map(planes, out, n_in, Q, 4 * tc_sbs(N), kTcRows, &map);
    const TcPlan p = tc_plan<Q, GB, N>(out, n_in, chunks, staged);
    Expand ex{{0x10001000u, 0x20002000u, 0x40004000u, 0x80008000u},
              {0x2f802f80u, 0x1f801f80u, 0u, tc_kinds(GB, N) ? 0xbf00bf00u : 0xbf80bf80u}, {}};
    for (int i = 0; i < 16; ++i) ex.mul[i] = 1u << (15 - i);
    auto kern = bcq_tc_kernel<Q, GB, N>;
    static std::atomic<int> ready[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices || ready[dev].load(std::memory_order_relaxed) == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDevices) ready[dev].store(1, std::memory_order_relaxed);
    }
    int cols = 32;
    while (cols < p.groups * tc_tmem_cols(GB, N)) cols *= 2;
    int smem = 1024 + p.sb_per * tc_pass_bytes(GB, N) + (staged ? p.groups * kTcStages * tc_stage_bytes(Q, N) : 0);
    if (smem < kTcMinSmem) smem = kTcMinSmem;
    e = launch_dependent(kern, dim3((unsigned)(p.n_ks * p.n_rb), (unsigned)chunks), dim3(p.groups * 160),
                         (size_t)smem, st, map, planes, astar, zstar, x, x_bf16,
                         p.n_ks > 1 ? work : y, out, n_in, g, batch, p.n_ks, p.sb_per, p.tiles, cols, staged ? 1 : 0, ex);
    if (e != cudaSuccess || p.n_ks == 1) return e;
    return gemv_reduce(work, y, (int64_t)batch * out, p.n_ks, st);
}

template <int Q, int GB>
cudaError_t tc_n(const uint32_t* planes, const float* astar, const float* zstar, int64_t out, int n_in, int g,
                 const void* x, int x_bf16, int batch, float* y, float* work, cudaStream_t st) {
    // columns of one pass; more go in chunks of tokens, each reading the planes
    // again.  64 columns only where a pass is one block: the sums of more
    // blocks leave tensor memory for one warpgroup alone.
    const int cols = batch * (x_bf16 ? 1 : 3);
    if (cols <= 16) return run_tc<Q, GB, 16>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
    if constexpr (GB == 128)
        if (cols > 32) return run_tc<Q, GB, 64>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
    return run_tc<Q, GB, 32>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
}

template <int Q>
cudaError_t tc_g(const uint32_t* planes, const float* astar, const float* zstar, int64_t out, int n_in, int g,
                 const void* x, int x_bf16, int batch, float* y, float* work, cudaStream_t st) {
    if (g == 32) return tc_n<Q, 32>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
    if (g == 64) return tc_n<Q, 64>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
    return tc_n<Q, 128>(planes, astar, zstar, out, n_in, g, x, x_bf16, batch, y, work, st);
}

}  // namespace

cudaError_t launch_bcq_tc(const uint32_t* planes, const float* astar, const float* zstar, int64_t out, int n_in, int q,
                          int g, const void* x, int xdtype, int batch, float* y, float* work, cudaStream_t st) {
    const int b16 = xdtype == UQ_W_BF16 ? 1 : 0;
    switch (q) {
        case 1: return tc_g<1>(planes, astar, zstar, out, n_in, g, x, b16, batch, y, work, st);
        case 2: return tc_g<2>(planes, astar, zstar, out, n_in, g, x, b16, batch, y, work, st);
        case 3: return tc_g<3>(planes, astar, zstar, out, n_in, g, x, b16, batch, y, work, st);
        default: return tc_g<4>(planes, astar, zstar, out, n_in, g, x, b16, batch, y, work, st);
    }
}

}  // namespace uq
