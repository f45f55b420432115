// Both passes of an iteration on the tensor cores (tcgen05, sm_103a).
//
// The lens-and-prism phase (Eq. 2) is separable, e^{i phi_n(x', y')} =
// C_n(x') R_n(y'), so over a tile of 128 rows x 64 columns both passes are
// dense complex matrix products with the spots as the contracted index:
//   back-propagation (Eq. 1):   S(y, x) = sum_n R'_n(y) C_n(x),
//                               R'_n = w_n a_n e^{i theta_n} R_n          [GEMM 1]
//   forward projection (Eq. 3): Z(n, y) = sum_x conj(C_n(x)) u(y, x),
//                               u = A e^{i Phi} = A S / |S|               [GEMM 2]
//                               V_n  = sum_y conj(R_n(y)) Z(n, y)         [per spot, CUDA cores]
// A compressed iteration is the same computation with u zero outside the
// subset S_j, so the sums run over S_j as Eqs. 1 and 3 ask.
// The accumulators (FP32) live in tensor memory.
// GEMM 1 sets each pixel's phase: its FP32 operands are split into two BF16
// halves, v = hi + lo, and each real product is kept as hi hi + hi lo + lo hi
// (2^-16 relative per product, FP32-class phases).  It runs its complex
// product as two real ones stacked along N (M = 128 rows, N = 128, K = 16
// spots):
//   [S_re | S_im] = R'_re [C_re | C_im] + R'_im [-C_im | C_re],
// with the two B operands as two 128-row windows of one 192-row tile
// [-C_im | C_re | C_im]: 6 instructions per spot chunk.
// GEMM 2 (the forward projection) is M = 128 spots x N = 128 rows x K = 16
// columns per instruction (N = 256 where real and imaginary parts share an A
// operand), with split BF16 operands too (9 instructions per K-step).  The
// half-precision option (compressed launches only) takes single FP16 operands
// instead (|u|, |C| <= 1; 3 instructions per K-step): the sums run over many
// pixels whose rounding errors (2^-12 relative) do not add up coherently.
//
// The operands are factor tables in global memory, laid out block by block
// exactly as the MMAs read them from shared memory (no-swizzle K-major core
// matrices, 8 rows x 16 bytes): C (per 64 columns and 16 spots) and C for
// GEMM 2 (per 16 columns, one K-step, and 128 spots) depend on the spots only
// and are made once per hologram; R' (per 128 rows and 16 spots) carries w and
// theta and is remade before every launch.  A tile streams its blocks into shared memory
// with bulk copies (cp.async.bulk, completion counted on an mbarrier) through
// a ring; a producer warp issues GEMM 1's copies, two issuing warps (GEMM 1,
// GEMM 2) issue the MMAs and commit them to mbarriers, and 12 or 16 epilogue
// warps run the CUDA-core stages: one or two groups of four turn S into u
// (epilogue 1), eight reduce Z to the spot fields (epilogue 2) once per strip of
// tiles along a row block and, in the final pass, write the phase map from S.
// The shared-memory pipe bounds a long launch of N <= 128: a tile's operand
// reads, copies and stores of u take 8.0 k of its ~8.6 k cycles (N = 100).  Every wait is bounded
// and a timeout is recorded in the launch's status word instead of hanging.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <functional>
#include <vector>
#include <type_traits>

#include "tile.cuh"

namespace cswgs {
namespace tc {

constexpr int kRows = 128;          // tile rows (GEMM 1 M, GEMM 2 N)
constexpr int kCols = 64;           // tile columns (GEMM 2 K; GEMM 1 N is re and im of them)
constexpr int kChunk = 16;          // spots per GEMM 1 instruction (K)
constexpr int kSpotBlock = 128;     // spots per GEMM 2 instruction (M)
constexpr uint32_t kWaitPolls = 1u << 20;   // polls of a bounded wait, unless a launch asks for fewer

// The launch's poll limit (set by thread 0 before the first block barrier).
__shared__ uint32_t s_wait_polls;

// component tiles (bytes): GEMM 1 operands per stage, GEMM 2 operands
constexpr uint32_t kA1 = kRows * kChunk * 2;        // R' component [128 rows][16 spots]
constexpr uint32_t kB1 = 3 * kCols * kChunk * 2;    // stacked C half [-C_im | C_re | C_im][16 spots]
constexpr uint32_t kB1Win = kCols * kChunk * 2;     // byte offset of the [C_re | C_im] window
constexpr uint32_t kStage = 4 * kA1 + 2 * kB1;      // one GEMM 1 stage: R' (4 components), C (hi, lo)
constexpr uint32_t kUc = kRows * 16 * 2;            // u component of one GEMM 2 K-step [128 rows][16 columns]
constexpr uint32_t kUSlot = 4 * kUc;                // u of one K-step (4 components)
constexpr uint32_t kCs = kSpotBlock * kCols * 2;    // C component [128 spots][64 columns]
constexpr uint32_t kCk = kSpotBlock * 16 * 2;       // C component of one GEMM 2 K-step [128 spots][16 columns]

__host__ __device__ inline int tiles(int P) { return ((P + kRows - 1) / kRows) * ((P + kCols - 1) / kCols); }

// Factor tables of one hologram (bytes): R' blocks (row block, spot chunk), C
// blocks (column block, spot chunk), GEMM 2 C blocks (column block, spot block).
__host__ __device__ inline int nchunks(int N) { return (N + kChunk - 1) / kChunk; }
__host__ __device__ inline int nspotblocks(int N) { return (N + kSpotBlock - 1) / kSpotBlock; }
__host__ __device__ inline size_t rw_table_bytes(int P, int N) { return (size_t)((P + kRows - 1) / kRows) * nchunks(N) * 4 * kA1; }
__host__ __device__ inline size_t c_table_bytes(int P, int N) { return (size_t)((P + kCols - 1) / kCols) * nchunks(N) * 2 * kB1; }
__host__ __device__ inline size_t cs_table_bytes(int P, int N)
{
    return (size_t)((P + kCols - 1) / kCols) * nspotblocks(N) * 4 * kCs;
}

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Byte offset of element (row, k) of a [rows][K] 16-bit tile in the no-swizzle
// K-major layout: core matrices of 8 rows x 8 elements (16 bytes a row, 128
// bytes each), the K / 8 cores of a row group side by side.
__device__ __forceinline__ uint32_t core_off(int row, int k, int K)
{
    return (uint32_t)((row >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Shared-memory matrix descriptor of a K-major no-swizzle tile: start address,
// leading byte offset (next core matrix along K), stride byte offset (next
// 8-row group), version 1, no swizzle.
__device__ __forceinline__ uint64_t desc(uint32_t start, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((start & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor, kind::f16: D FP32, A and B both BF16 (bf16 = 1) or
// both FP16 (bf16 = 0), both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc(int M, int N, int neg_a, int bf16 = 1)
{
    return (1u << 4) | ((uint32_t)bf16 << 7) | ((uint32_t)bf16 << 10) | ((uint32_t)neg_a << 13) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                 :: "r"(d_tmem), "l"(a), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ bool try_wait(uint32_t mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    return ok != 0u;
}

// Bounded wait for phase `parity` of an mbarrier; false when it ran out.  The
// first poll does not wait for the poll limit's shared-memory load.
__device__ __forceinline__ bool wait(uint32_t mbar, uint32_t parity)
{
    if (try_wait(mbar, parity)) return true;
    const uint32_t polls = s_wait_polls;
    for (uint32_t it = 1; it < polls; ++it)
        if (try_wait(mbar, parity)) return true;
    return false;
}

// One bulk copy global -> shared, counted on an mbarrier (16-byte aligned
// addresses, size a multiple of 16).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}

// The arrival of the issuing thread, announcing `bytes` of copies to come.
__device__ __forceinline__ void expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 16 consecutive FP32 columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t h2_bits(__half2 h)
{
    return (uint32_t)__half_as_ushort(__low2half(h)) | ((uint32_t)__half_as_ushort(__high2half(h)) << 16);
}

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat162 h)
{
    return (uint32_t)__bfloat16_as_ushort(h.x) | ((uint32_t)__bfloat16_as_ushort(h.y) << 16);
}

// The BF16 halves of a pair of values, converted together (round to nearest):
// hi = bf16(v), lo = bf16(v - hi).
struct Split2 {
    __nv_bfloat162 hi, lo;
};

__device__ __forceinline__ Split2 split2(float a, float b)
{
    Split2 r;
    r.hi = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(r.hi);
    r.lo = __floats2bfloat162_rn(a - f.x, b - f.y);
    return r;
}

// Eight complex values -> the four BF16 component rows (re hi, re lo, im hi,
// im lo), one 16-byte store each, at byte offset `off` of four tiles `stride`
// bytes apart.
__device__ __forceinline__ void put8(unsigned char *base, uint32_t stride, uint32_t off, const float2 *v)
{
    uint32_t w[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Split2 re = split2(v[2 * q].x, v[2 * q + 1].x), im = split2(v[2 * q].y, v[2 * q + 1].y);
        w[0][q] = bf16x2_bits(re.hi);
        w[1][q] = bf16x2_bits(re.lo);
        w[2][q] = bf16x2_bits(im.hi);
        w[3][q] = bf16x2_bits(im.lo);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4 *>(base + c * stride + off) = make_uint4(w[c][0], w[c][1], w[c][2], w[c][3]);
}

// Eight complex values -> FP16 rows of the re and im component tiles
// (`stride` bytes apart), one 16-byte store each (round to nearest).
__device__ __forceinline__ void put8h(unsigned char *base, uint32_t stride, uint32_t off, const float2 *v)
{
    uint32_t wr[4], wi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        wr[q] = h2_bits(__floats2half2_rn(v[2 * q].x, v[2 * q + 1].x));
        wi[q] = h2_bits(__floats2half2_rn(v[2 * q].y, v[2 * q + 1].y));
    }
    *reinterpret_cast<uint4 *>(base + off) = make_uint4(wr[0], wr[1], wr[2], wr[3]);
    *reinterpret_cast<uint4 *>(base + stride + off) = make_uint4(wi[0], wi[1], wi[2], wi[3]);
}

// Two FP32 values worked on by one instruction (fma.rn.f32x2 and its kin; each
// half is rounded like the scalar instruction's result).
__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Eight complex values of u, split for GEMM 2 and packed (the four BF16
// component rows, or the two FP16 ones), to be stored once their slot is free.
struct Packed8 {
    uint32_t w[4][4];
};

// The two values of a BF16 pair as an FP32 pair (a BF16 is an FP32's upper half).
__device__ __forceinline__ uint64_t bf16x2_floats(uint32_t h)
{
    return pack2(__uint_as_float(h << 16), __uint_as_float(h & 0xFFFF0000u));
}

// |S|^2 of 16 pixels, two by two, and whether every one is a normal FP32
// number (false for a NaN: min.NaN keeps it).
__device__ __forceinline__ bool norms16(const float *sr, const float *si, uint64_t *n2)
{
    float lo = 1.f, hi = 1.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint64_t a = pack2(sr[2 * q], sr[2 * q + 1]), b = pack2(si[2 * q], si[2 * q + 1]);
        n2[q] = fma2(a, a, mul2(b, b));
        const float2 n = unpack2(n2[q]);
        asm("min.NaN.f32 %0, %0, %1;" : "+f"(lo) : "f"(n.x));
        asm("min.NaN.f32 %0, %0, %1;" : "+f"(lo) : "f"(n.y));
        hi = fmaxf(hi, fmaxf(n.x, n.y));
    }
    return lo >= 1.17549435e-38f && hi <= 3.0e38f;
}

// Pixels whose |S|^2 is no normal FP32 number: S is scaled by a power of two so
// that it becomes one (u = S / |S| needs S up to a factor only).  S = 0 has
// phase 0, and so has an S that is no finite number.
__device__ __forceinline__ void rescale16(float *sr, float *si, uint64_t *n2)
{
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const float2 n = unpack2(n2[e >> 1]);
        float v = (e & 1) ? n.y : n.x, a = sr[e], b = si[e];
        if (!(v >= 1.17549435e-38f && v <= 3.0e38f)) {
            const float f = fmaxf(fabsf(a), fabsf(b)) < 1.f ? 0x1p100f : 0x1p-100f;
            a *= f;
            b *= f;
            v = fmaf(a, a, b * b);
            if (!(v > 0.f && v <= 3.0e38f)) {
                a = 1.f;
                b = 0.f;
                v = 1.f;
            }
        }
        sr[e] = a;
        si[e] = b;
        n2[e >> 1] = (e & 1) ? pack2(n.x, v) : pack2(v, n.y);
    }
}

// ur, ui: four pairs each, columns 2q and 2q + 1.
template <bool F16>
__device__ __forceinline__ Packed8 pack8(const uint64_t *ur, const uint64_t *ui)
{
    Packed8 p;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 a = unpack2(ur[q]), b = unpack2(ui[q]);
        if (F16) {
            p.w[0][q] = h2_bits(__floats2half2_rn(a.x, a.y));
            p.w[1][q] = h2_bits(__floats2half2_rn(b.x, b.y));
            p.w[2][q] = p.w[3][q] = 0u;
        } else {
            const uint32_t rh = bf16x2_bits(__floats2bfloat162_rn(a.x, a.y));
            const uint32_t ih = bf16x2_bits(__floats2bfloat162_rn(b.x, b.y));
            const float2 rl = unpack2(sub2(ur[q], bf16x2_floats(rh))), il = unpack2(sub2(ui[q], bf16x2_floats(ih)));
            p.w[0][q] = rh;
            p.w[1][q] = bf16x2_bits(__floats2bfloat162_rn(rl.x, rl.y));
            p.w[2][q] = ih;
            p.w[3][q] = bf16x2_bits(__floats2bfloat162_rn(il.x, il.y));
        }
    }
    return p;
}

// The rows of a Packed8 at byte offset `off` of the component tiles `stride`
// bytes apart: split BF16 re hi, im hi, re lo, im lo; FP16 re, im.
template <bool F16>
__device__ __forceinline__ void store8(unsigned char *base, uint32_t stride, uint32_t off, const Packed8 &p)
{
    constexpr int at[4] = {0, F16 ? 1 : 2, 1, 3};   // tile of p.w[c]
#pragma unroll
    for (int c = 0; c < (F16 ? 2 : 4); ++c)
        *reinterpret_cast<uint4 *>(base + at[c] * stride + off) =
            make_uint4(p.w[c][0], p.w[c][1], p.w[c][2], p.w[c][3]);
}

// ------------------------------------------------------------- factor tables --
// Items of eight phasors; consecutive threads take consecutive rows of one
// core matrix, so a warp's 16-byte stores fill whole 128-byte lines.

// Eight values -> rows of the two BF16 halves (hi, lo) of a stacked C block:
// hi at base, lo at base + kB1, row offsets re_off, im_off (C_im) and
// neg_off (-C_im); each a 16-byte store.
__device__ __forceinline__ void put8_stacked(unsigned char *base, uint32_t re_off, uint32_t im_off,
                                             uint32_t neg_off, const float2 *v)
{
    uint32_t w[6][4];   // re hi, re lo, im hi, im lo, -im hi, -im lo
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Split2 re = split2(v[2 * q].x, v[2 * q + 1].x), im = split2(v[2 * q].y, v[2 * q + 1].y);
        w[0][q] = bf16x2_bits(re.hi);
        w[1][q] = bf16x2_bits(re.lo);
        w[2][q] = bf16x2_bits(im.hi);
        w[3][q] = bf16x2_bits(im.lo);
        w[4][q] = bf16x2_bits(__hneg2(im.hi));   // the split of -v is -(hi), -(lo): exact
        w[5][q] = bf16x2_bits(__hneg2(im.lo));
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        unsigned char *t = base + h * kB1;
        *reinterpret_cast<uint4 *>(t + re_off) = make_uint4(w[h][0], w[h][1], w[h][2], w[h][3]);
        *reinterpret_cast<uint4 *>(t + im_off) = make_uint4(w[2 + h][0], w[2 + h][1], w[2 + h][2], w[2 + h][3]);
        *reinterpret_cast<uint4 *>(t + neg_off) = make_uint4(w[4 + h][0], w[4 + h][1], w[4 + h][2], w[4 + h][3]);
    }
}

// C (GEMM 1's B: per block of 64 columns and 16 spots, each half a 192-row
// tile [-C_im | C_re | C_im] with row = column within each third) and C for
// GEMM 2 (128 spots x 64 columns per block, stored K-step by K-step: 4 x [the
// components of 128 spots x 16 columns]; split BF16, and for the
// half-precision option also FP16 re and im) of hologram blockIdx.y, from its
// spot coefficients.
__global__ void __launch_bounds__(256) const_tables_kernel(const HoloDev *__restrict__ holos, int count)
{
    const HoloDev H = holos[blockIdx.y];
    if (!H.ctab) return;
    const int P = H.P, N = H.N, half = P >> 1, nc = nchunks(N), nsb = nspotblocks(N);
    const int ncb = (P + kCols - 1) / kCols;
    const int items_c = ncb * nc * 128;                 // (block, 64 columns x 2 groups)
    const int items_cs = ncb * nsb * 1024;              // (block, 128 spots x 8 groups)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < items_c + items_cs; i += gridDim.x * blockDim.x) {
        float2 v[8];
        if (i < items_c) {
            const int blk = i >> 7, j = i & 127;
            const int cb = blk / nc, c = blk % nc;
            const int col = (j & 7) + 8 * (j >> 4), g = (j >> 3) & 1;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int n = c * kChunk + 8 * g + e;
                if (n < N) {
                    const int4 cf = H.coef[n];
                    v[e] = spot_factor(cf.x, cf.z, __int_as_float(cf.w), cb * kCols + col - half, kFixRound, 1.f);
                } else {
                    v[e] = make_float2(0.f, 0.f);
                }
            }
            put8_stacked(H.ctab + (size_t)blk * (2 * kB1), core_off(kCols + col, 8 * g, kChunk),
                         core_off(2 * kCols + col, 8 * g, kChunk), core_off(col, 8 * g, kChunk), v);
        } else {
            const int k = i - items_c, blk = k >> 10, j = k & 1023;
            const int cb = blk / nsb, sb = blk % nsb;
            const int nl = (j & 7) + 8 * (j >> 6), g = (j >> 3) & 7, n = sb * kSpotBlock + nl;
            if (n < N) {
                const int4 cf = H.coef[n];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    v[e] = spot_factor(cf.x, cf.z, __int_as_float(cf.w), cb * kCols + 8 * g + e - half, kFixRound, 1.f);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = make_float2(0.f, 0.f);
            }
            // K-step g / 2 of the block, column group g % 2 of the K-step
            const int ks = g >> 1;
            put8(H.cstab + (size_t)blk * (4 * kCs) + (size_t)ks * (4 * kCk), kCk, core_off(nl, 8 * (g & 1), 16), v);
            if (H.cstab16)
                put8h(H.cstab16 + (size_t)blk * (2 * kCs) + (size_t)ks * (2 * kCk), kCk, core_off(nl, 8 * (g & 1), 16),
                      v);
        }
    }
}

// The Mp draws of S_j (Section 3) of the slot's hologram, each setting its
// pixel's bit in the iteration's mask, which is clear before (the tails of the
// last launch that used it cleared it).  Grid: blocks x slots.
__device__ __forceinline__ void scatter_subset(const HoloDev &H, const LaunchSlot &sl)
{
    uint32_t *mask = subset_mask(H, sl.j);
    const SubsetDraw d = subset_draw(H, sl.j);
    const UDiv dP = udiv_of((uint32_t)H.P);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < H.Mp; k += gridDim.x * blockDim.x) {
        const uint32_t m = subset_pixel(H, d, (uint32_t)k);
        uint32_t c;
        const uint32_t r = udiv(m, dP, c);
        atomicOr(mask + (size_t)r * H.mask_words + (c >> 5), 1u << (c & 31));
    }
}

__global__ void __launch_bounds__(256) mask_scatter_kernel(const HoloDev *__restrict__ holos,
                                                           const LaunchSlot *__restrict__ slots)
{
    const LaunchSlot sl = slots[blockIdx.y];
    const HoloDev H = holos[sl.holo];
    if (sl.pass == kPassSubset && H.mask) scatter_subset(H, sl);
}

// The same masks drawn in shared memory: a cluster of G CTAs per slot (grid G x
// slots), each holding the slot's whole mask and taking 1 / G of the Mp draws,
// each draw an OR in shared memory; then each CTA ORs its 1 / G of the words
// over the cluster (distributed shared memory) and stores them, zero words
// included.  P^2 / 8 bytes of shared memory: up to P of about 1280.
// A Feistel round adds F(R), a function of one half only, and a half takes at
// most P values: the four rounds' F are tabled first (4 P hashes instead of
// 4 Mp / G; 16 bits an entry, halves and entries carried doubled so that they
// are byte offsets), and a draw is four table loads, four additions modulo a
// half's range and the OR.  Bound by the latency of these dependent loads (32
// warps an SM wait for them most of the time; random, three to four lanes to a
// bank, they take half of the shared-memory pipe): 33 us for 64 masks of P =
// 1152, c = 1/8.  With the hashes made per draw it was bound by the ALU, and
// with G > 1 it ended in an OR of every word in global memory: 47 us.  (A
// 64-hologram batch of 31 launches: 11.70 ms with that form, 11.09 with this.)
constexpr int kLocalThreads = 1024;

// (L + F(R)) mod p with everything doubled: byte offsets into the round tables.
__device__ __forceinline__ void table_round(uint32_t &L, uint32_t &R, const unsigned char *tab, uint32_t p2)
{
    const uint32_t s = L + *reinterpret_cast<const uint16_t *>(tab + R);
    L = R;
    R = min(s, s - p2);   // s < 2 p2: the difference wraps past every p2 when s < p2
}

__global__ void __launch_bounds__(kLocalThreads) mask_local_kernel(const HoloDev *__restrict__ holos,
                                                                   const LaunchSlot *__restrict__ slots)
{
    extern __shared__ __align__(16) uint32_t s_words[];
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const LaunchSlot sl = slots[blockIdx.y];
    const HoloDev &H = holos[sl.holo];
    if (sl.pass != kPassSubset || !H.mask) return;   // the same in every CTA of the cluster
    const uint32_t G = gridDim.x, x = blockIdx.x;
    const int P = H.P, mw = H.mask_words, words = P * mw;
    const int tid = threadIdx.x;
    const uint32_t a = H.fa, b = H.fb, D = (uint32_t)H.D;   // the permutation's rectangle, D <= a b
    unsigned char *tab = reinterpret_cast<unsigned char *>(s_words + ((words + 3) & ~3));
    unsigned char *t0 = tab, *t1 = t0 + 2 * b, *t2 = t1 + 2 * a, *t3 = t2 + 2 * b;   // entries: b, a, b, a
    const SubsetDraw d = subset_draw(H, sl.j);
    for (int i = tid; i < words; i += kLocalThreads) s_words[i] = 0u;
    for (uint32_t v = tid; v < max(a, b); v += kLocalThreads) {
        if (v < b) {
            reinterpret_cast<uint16_t *>(t0)[v] = (uint16_t)(2u * __umulhi(fmix32(v ^ d.K.k0), a));
            reinterpret_cast<uint16_t *>(t2)[v] = (uint16_t)(2u * __umulhi(fmix32(v ^ d.K.k2), a));
        }
        if (v < a) {
            reinterpret_cast<uint16_t *>(t1)[v] = (uint16_t)(2u * __umulhi(fmix32(v ^ d.K.k1), b));
            reinterpret_cast<uint16_t *>(t3)[v] = (uint16_t)(2u * __umulhi(fmix32(v ^ d.K.k3), b));
        }
    }
    __syncthreads();
    const uint32_t k0 = (uint32_t)((uint64_t)H.Mp * x / G), k1 = (uint32_t)((uint64_t)H.Mp * (x + 1) / G);
    const bool grid = H.aperture == 0 && a == (uint32_t)P && b == (uint32_t)P && D == (uint32_t)P * (uint32_t)P;
    // this thread's draws, kLocalThreads apart: the halves of each kk = (k + off)
    // mod D step by a fixed pair (the square grid's D is a multiple of b: the
    // wrap around D leaves R as it is)
    if (grid) {
        const uint32_t p2 = 2u * (uint32_t)P;
        uint32_t kk = k0 + tid + d.off, r0;
        kk = kk >= D ? kk - D : kk;
        uint32_t l0 = 2u * udiv(kk, d.fb, r0);
        r0 *= 2u;
        const uint32_t dl = 2u * (kLocalThreads / (uint32_t)P % (uint32_t)P), dr = 2u * (kLocalThreads % (uint32_t)P);
#pragma unroll 4
        for (uint32_t k = k0 + tid; k < k1; k += kLocalThreads) {
            uint32_t L = l0, R = r0;
            table_round(L, R, t0, p2);
            table_round(L, R, t1, p2);
            table_round(L, R, t2, p2);
            table_round(L, R, t3, p2);
            atomicOr(s_words + (L >> 1) * (uint32_t)mw + (R >> 6), 1u << ((R >> 1) & 31));
            r0 += dr;
            l0 += dl;
            if (r0 >= p2) {
                r0 -= p2;
                l0 += 2u;
            }
            l0 = l0 >= p2 ? l0 - p2 : l0;
        }
    } else {
        const UDiv dP = udiv_of((uint32_t)P);
        const uint32_t a2 = 2u * a, b2 = 2u * b, extra = a * b - D;
        auto permute_tab = [&](uint32_t y) {
            uint32_t R;
            uint32_t L = 2u * udiv(y, d.fb, R);
            R *= 2u;
            table_round(L, R, t0, a2);
            table_round(L, R, t1, b2);
            table_round(L, R, t2, a2);
            table_round(L, R, t3, b2);
            return (L >> 1) * b + (R >> 1);
        };
        for (uint32_t k = k0 + tid; k < k1; k += kLocalThreads) {
            uint32_t y = k + d.off;
            y = permute_tab(y >= D ? y - D : y);
            for (uint32_t w = 0; y >= D && w < extra; ++w) y = permute_tab(y);   // cycle walk (permute_domain)
            const uint32_t m = pupil_pixel(H, y < D ? y : 0u);
            uint32_t c;
            const uint32_t r = udiv(m, dP, c);
            atomicOr(s_words + r * (uint32_t)mw + (c >> 5), 1u << (c & 31));
        }
    }
    uint32_t *g = subset_mask(H, sl.j);
    if (G == 1) {
        __syncthreads();
        for (int i = tid; i < words; i += kLocalThreads) g[i] = s_words[i];
    } else {
        cluster.sync();
        const int i1 = (int)((int64_t)words * (x + 1) / G);
        for (int i = (int)((int64_t)words * x / G) + tid; i < i1; i += kLocalThreads) {
            uint32_t v = 0u;
            for (uint32_t q = 0; q < G; ++q) v |= cluster.map_shared_rank(s_words, q)[i];
            g[i] = v;
        }
        cluster.sync();   // every CTA's words are read before it leaves
    }
}

// R' = w a e^{i theta} R (GEMM 1's A: 128 rows x 16 spots per block) of the
// hologram of each slot, from its current spot state.
__global__ void __launch_bounds__(256) rw_tables_kernel(const HoloDev *__restrict__ holos,
                                                        const LaunchSlot *__restrict__ slots)
{
    // one block (128 rows x 16 spots) per pass of the loop: its 16 spots' row
    // coefficients and state are read once into shared memory
    __shared__ int4 s_cf[kChunk];      // {B, Gh, gl, theta + rounding}
    __shared__ float s_wa[kChunk];     // w a
    chain_start();
    const LaunchSlot sl = slots[blockIdx.y];
    const HoloDev H = holos[sl.holo];
    chain_wait();
    if (!H.rwtab) return;
    const int P = H.P, N = H.N, half = P >> 1, nc = nchunks(N);
    const int blocks = ((P + kRows - 1) / kRows) * nc;   // (128 rows, 16 spots) blocks, 256 threads each
    const int j = threadIdx.x;
    const int row = (j & 7) + 8 * (j >> 4), g = (j >> 3) & 1;
    for (int blk = blockIdx.x; blk < blocks; blk += gridDim.x) {
        const int rb = blk / nc, c = blk % nc;
        __syncthreads();   // the previous block's spots are read
        if (j < kChunk) {
            const int n = c * kChunk + j;
            int4 v = make_int4(0, 0, 0, 0);
            float wa = 0.f;
            if (n < N) {
                const int4 cf = H.coef[n];
                const SpotState st = H.state[n];
                v = make_int4(cf.y, cf.z, cf.w, (int)(st.theta + kFixRound));
                wa = st.w * st.a0;
            }
            s_cf[j] = v;
            s_wa[j] = wa;
        }
        __syncthreads();
        float2 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int4 cf = s_cf[8 * g + e];
            v[e] = spot_factor(cf.x, cf.y, __int_as_float(cf.z), rb * kRows + row - half, (uint32_t)cf.w,
                               s_wa[8 * g + e]);
        }
        put8(H.rwtab + (size_t)blk * (4 * kA1), kA1, core_off(row, 8 * g, kChunk), v);
    }
}


// ----------------------------------------------------------- warp roles --
// Tiles are pipelined by warp roles: a producer warp (takes the work items and
// loads GEMM 1's operand stages), a GEMM 1 warp, a GEMM 2 warp (one elected
// lane of each issues its bulk copies and MMAs), 4 or 8 u warps (epilogue 1)
// and 8 V warps (epilogue 2).  The producer runs ahead of the GEMM 1 warp by the
// ring's depth: a tcgen05.mma issue waits for the tensor pipe, so copies
// issued from the MMA warp would start one stage late.
// A work item is a strip: LaunchSlot::strip consecutive tiles of one row block
// of a hologram.  Since V_n = sum_y conj(R_n(y)) Z(n, y) takes the same R_n(y)
// for every tile of a row block, GEMM 2 accumulates Z(n, y) over the strip's
// tiles and the V warps reduce it once per strip; a hologram with more than
// one GEMM 2 spot block (Z holds one) takes strips of one tile.
// Tensor memory holds two S buffers (columns 256..383 and 384..511; tile k
// uses buffer k & 1) and Z (columns 0..255).  GEMM 1 runs ahead into the next
// tile's back-propagation while the u warps turn S into u; the GEMM 2 warp
// streams the tile's C block in meanwhile and follows the u warps K-step by
// K-step; the u warps write a K-step's columns of u as soon as GEMM 2 of the
// previous tile has read them.  The per-hologram tails (Eqs. 4-6, or the
// metrics) run in a small kernel right after the launch, so tiles neither
// fence nor count arrivals.
// Hand-overs, all mbarriers:
//   ready[2]          producer -> GEMM 1, GEMM 2, u and V warps: tile k in info slot k & 1
//   full[r], empty[r] GEMM 1 operand ring: copies landed / MMAs done
//   s_full[2]         GEMM 1 of the tile in that S buffer is done
//   s_empty[2]        the tile's u warps have read that S buffer and info slot, the
//                     V and GEMM warps that info slot
//   u_step[4]         the u warps have written u's columns of one K-step of GEMM 2
//   u_free[2][4]      GEMM 2 has read them, by the parity of the tile's number
//                     among those with products
//   cs_full           GEMM 2's C block has landed
//   cs_free           the MMAs that read it are done (its buffer is free)
//   z_full            a Z accumulation is done: a strip, or one spot block of a tile
//   z_empty           the V warps have read Z
//   dot[2]            the second V warps' half of a dot is in shared memory
//   drain             both issuing warps' last commits, before tensor memory is freed
// Every wait is bounded; a timeout ends the loop of the side that saw it and
// sets the status word, and the other side's waits then run out in turn.
namespace ws {

constexpr int kRingMax = 4;
constexpr uint32_t kS0 = 256;       // S buffers at columns 256 and 384, Z at 0
constexpr int kTmemColsWs = 512;
constexpr int kKSteps = kCols / 16; // GEMM 2 K-steps per tile

enum Bar {
    kReady0 = 0,
    kFull0 = 2,
    kEmpty0 = kFull0 + kRingMax,
    kSFull0 = kEmpty0 + kRingMax,
    kSEmpty0 = kSFull0 + 2,
    kUStep0 = kSEmpty0 + 2,       // u's columns of GEMM 2's K-step 0 .. 3 are written
    kUFree0 = kUStep0 + kKSteps,  // ... and GEMM 2 has read them, by the parity of the product tile's number
    kCsFull = kUFree0 + 2 * kKSteps,  // GEMM 2's C block has landed
    kCsFree,                      // the MMAs that read it are done
    kZFull,                       // a Z accumulation is done
    kZEmpty,
    kDot0,      // the second V warps' half sums are in shared memory, by parity of the accumulation
    kDrain = kDot0 + 2,     // both issuing warps' last commits (2 arrivals)
    kBarsWs
};

// The GEMM 2 warp's work item: a published tile with products.
struct G2Info {
    const unsigned char *cstab;   // GEMM 2's C blocks in the launch's format
    int nsb, cb;
    int first, last;              // the tile opens / closes its strip's Z accumulation
};

// A published tile: its work item (strip), its tile index in the hologram's
// pass, its place in the strip, and copies of its launch slot and its
// hologram's descriptor (staged by the producer warp so that the other warps
// read them from shared memory).
struct Info {
    int item, empty, done, tile;
    int first, last;   // the first / last tile with products of the strip
    int zero;          // the strip's last tile, and the strip has no products
    uint32_t before;   // tiles with products published before this one
    LaunchSlot sl;
    HoloDev H;
};


// The epilogue warps: UG groups of 4 u warps (epilogue 1), one warp per TMEM
// lane quadrant, and 8 V warps (epilogue 2), two per quadrant: each takes half
// the rows of a strip's dot and half the columns of the final pass's phase map.
// GEMM 2 of the next strip (N > 128: of the next spot block) waits for the dot
// to have read Z, a latency-bound chain: with 4 V warps a batch of N = 100 spent
// 5 % and one of N up to 300 14 % of its time on it.
// With UG = 2, group g takes the tiles of S buffer g, and one tile's mask loads,
// tensor-memory latency and waits pass while the other group works; the kernel
// then has 96 registers a thread instead of 127.  At more than one spot block
// and in launches of few holograms that is worth it (64 holograms of N up to
// 300: 12.51 -> 12.29 ms; 16 of N = 100: 4.15 -> 4.07), at N <= 128, where the
// shared-memory pipe bounds a long launch, it is not (64 of N = 100: 10.73 ->
// 10.88, FP16 9.14 -> 9.25).
constexpr int kVWarps = 8;

template <int UG>
struct Cfg {
    static constexpr int kU = 4 * UG, kEpi = kU + kVWarps;   // u warps, epilogue warps
    static constexpr int kThreads = 32 * (kEpi + 3);         // and the producer, GEMM 1 and GEMM 2 warps
};

// Shared-memory layout of the kernel with US slots of u (one K-step each;
// GEMM 2 of more than one spot block re-reads all of a tile's u, so US = 4):
// the GEMM 1 ring, GEMM 2's C block and u (and 128 bytes to align the base;
// the no-swizzle layouts and the bulk copies need 16).  (Two u slots and a
// fourth ring stage were measured: the epilogue then waits for GEMM 2 to free
// a slot, 7 % slower at N = 100.)
template <int US>
struct Lay {
    static_assert(US == kKSteps, "u slots");
    static constexpr int kRing = 3;
    static constexpr size_t kSmem = 128 + (size_t)kRing * kStage + 4 * (size_t)kCs + (size_t)US * kUSlot;
};

struct SmemWs {
    unsigned char *ring, *cs, *u;
};

template <int US>
__device__ __forceinline__ SmemWs carve_ws(unsigned char *raw)
{
    unsigned char *b = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(raw) + 127) & ~(uintptr_t)127);
    SmemWs m;
    m.ring = b;
    m.cs = m.ring + Lay<US>::kRing * kStage;
    m.u = m.cs + 4 * kCs;
    return m;
}

__device__ __forceinline__ void arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mbar) : "memory");
}

__device__ __forceinline__ bool wait_newest(uint32_t mbar, uint32_t given) { return wait(mbar, (given - 1u) & 1u); }

// A warp's vote: true when every lane's p is.  The epilogue warps wait each
// on its own; the hand-over barriers keep them within a tile of each other,
// and a wait that runs out in one warp runs out in the others too, since the
// pipeline behind it has stopped.
__device__ __forceinline__ bool warp_and(bool p) { return __all_sync(0xffffffffu, p) != 0; }

// Tile t of hologram H lies wholly outside the round pupil.
__device__ __forceinline__ bool tile_outside(const HoloDev &H, int t)
{
    if (H.aperture == 0) return false;
    const int P = H.P, half = P >> 1, col_tiles = (P + kCols - 1) / kCols;
    const int y0 = (t / col_tiles) * kRows, x0 = (t % col_tiles) * kCols;
    const int ylo = y0 - half, yhi = min(y0 + kRows, P) - 1 - half;
    const int xlo = x0 - half, xhi = min(x0 + kCols, P) - 1 - half;
    const int64_t dy = ylo > 0 ? ylo : (yhi < 0 ? yhi : 0);
    const int64_t dx = xlo > 0 ? xlo : (xhi < 0 ? xhi : 0);
    return dx * dx + dy * dy > (int64_t)half * half;
}

// Barrier i of the block's array, by shared-memory address.
__device__ __forceinline__ uint32_t mbar_at(uint32_t base, int i) { return base + 8u * (uint32_t)i; }

// One elected lane of a converged warp (the issuing lane of a producer or MMA warp).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n selp.u32 %0, 1, 0, e;\n}\n" : "=r"(p));
    return p != 0;
}

// Every lane's bounded wait for phase `parity`, voted across the warp.
__device__ __forceinline__ bool warp_wait(uint32_t mbar, uint32_t parity)
{
    return __all_sync(0xffffffffu, wait(mbar, parity & 1u)) != 0;
}

// An issuing warp's pipeline state, the same in every lane and all scalars.
// GEMM 1 chunks go round the ring in order, so chunk q (counted over the
// block's tiles) is stage q % R's (q / R)-th use (R the ring's depth) and both ring waits
// take their parity from q; the other barriers count their phases.  The whole
// warp runs the loop and waits; one elected lane issues the copies, MMAs,
// commits and arrivals.
struct Ctl {
    uint32_t mb;      // barrier 0
    uint32_t tmem;
    uint32_t ring, cs, u;   // shared addresses of the ring, GEMM 2's C block and u
    uint32_t ql;      // GEMM 1 chunks loaded
    uint32_t qm;      // GEMM 1 chunks multiplied
    uint32_t nz;      // Z accumulations closed
    uint32_t ncs;     // GEMM 2 C blocks loaded
    uint32_t nu;      // u hand-overs taken
};

// GEMM 1's operands of one tile, issued by the producer warp: for each chunk of
// 16 spots, R' of row block rb and the stacked C of column block cb into the
// next ring stage once the GEMM 1 warp's products have released it.
template <int R>
__device__ __forceinline__ bool load_gemm1(Ctl &C, const HoloDev &H, int rb, int cb)
{
    const int nc = nchunks(H.N);
    for (int c = 0; c < nc; ++c) {
        const uint32_t s = C.ql % R;
        if (C.ql >= (uint32_t)R && !warp_wait(mbar_at(C.mb, kEmpty0 + s), C.ql / R - 1u)) return false;
        if (elect_one()) {
            const uint32_t stg = C.ring + s * kStage, full = mbar_at(C.mb, kFull0 + s);
            expect_tx(full, kStage);
            bulk_load(stg, H.rwtab + ((size_t)rb * nc + c) * (4 * kA1), 4 * kA1, full);
            bulk_load(stg + 4 * kA1, H.ctab + ((size_t)cb * nc + c) * (2 * kB1), 2 * kB1, full);
        }
        __syncwarp();
        C.ql++;
    }
    return true;
}

// GEMM 1 of one tile into S buffer j, [S_re | S_im] = R' [C_re | C_im] with
// the complex product stacked along N: per chunk six M128 N128 K16 MMAs (the
// split operands' hi hi, hi lo and lo hi terms of R'_re [C_re | C_im] and
// R'_im [-C_im | C_re]), issued as each ring stage lands.  The stage goes back
// to the producer when its MMAs complete.
template <int R>
__device__ __forceinline__ bool gemm1(Ctl &C, int nc, int j)
{
    const uint32_t id = idesc(kRows, 2 * kCols, 0);
    const uint32_t s_acc = C.tmem + kS0 + 2 * kCols * j;   // [S_re | S_im]
    const uint64_t ring0 = desc(C.ring, 128, 256);
    for (int c = 0; c < nc; ++c) {
        const uint32_t s = C.qm % R;
        if (!warp_wait(mbar_at(C.mb, kFull0 + s), C.qm / R)) return false;
        // A: R' re hi, re lo, im hi, im lo; B: [C_re | C_im] and [-C_im | C_re] windows, hi and lo
        const uint64_t st = ring0 + ((uint64_t)(s * kStage) >> 4);
        const uint64_t arh = st, arl = st + (kA1 >> 4), aih = st + (2 * kA1 >> 4), ail = st + (3 * kA1 >> 4);
        const uint64_t bh = st + (4 * kA1 >> 4), bl = bh + (kB1 >> 4);
        const uint64_t b1h = bh + (kB1Win >> 4), b1l = bl + (kB1Win >> 4);
        if (elect_one()) {
            mma(s_acc, arh, b1h, id, c > 0 ? 1u : 0u);
            mma(s_acc, arh, b1l, id, 1u);
            mma(s_acc, arl, b1h, id, 1u);
            mma(s_acc, aih, bh, id, 1u);
            mma(s_acc, aih, bl, id, 1u);
            mma(s_acc, ail, bh, id, 1u);
            commit(mbar_at(C.mb, kEmpty0 + s));
        }
        __syncwarp();
        C.qm++;
    }
    if (elect_one()) commit(mbar_at(C.mb, kSFull0 + j));   // covers this GEMM 1 and every MMA before it
    __syncwarp();
    return true;
}

// GEMM 2 of one tile: Z = conj(C)^T u, one block of 128 spots at a time, into
// columns 0..255; each block's C (its four K-steps one after the other)
// streams in once the MMAs that read the previous one are done (block 0 while
// u is still being written).  Split BF16 operands (4 components each), or FP16
// re and im for the half-precision option.  The first tile of a strip (and
// each spot block past the first) opens a Z accumulation, once the epilogue
// has read the last one; the last tile of a strip (and each spot block but the
// last) closes it.  After each K-step of the last spot block, u's columns of
// that K-step go back to the epilogue warps.
template <bool F16, int US>
__device__ __forceinline__ bool gemm2(Ctl &C, const G2Info &g)
{
    const uint32_t comps = F16 ? 2u : 4u, kbytes = comps * kCk;
    constexpr int kBf16 = F16 ? 0 : 1;
    const uint32_t id2 = idesc(kSpotBlock, 2 * kRows, 0, kBf16), id = idesc(kSpotBlock, kRows, 0, kBf16),
                   idn = idesc(kSpotBlock, kRows, 1, kBf16);
    const uint32_t z_re = C.tmem, z_im = C.tmem + kRows;
    const uint64_t cs0 = desc(C.cs, 128, 256);                       // [128 spots][16 columns] per component
    const uint64_t u0 = desc(C.u, 128, 256);                         // [128 rows][16 columns] per component
    const int ufree = kUFree0 + kKSteps * (int)(C.nu & 1u);          // this tile's releases of u
    for (int sb = 0; sb < g.nsb; ++sb) {
        if (C.ncs > 0 && !warp_wait(mbar_at(C.mb, kCsFree), C.ncs - 1u)) return false;
        if (elect_one()) {
            const uint32_t full = mbar_at(C.mb, kCsFull);
            expect_tx(full, kKSteps * kbytes);
            bulk_load(C.cs, g.cstab + ((size_t)g.cb * g.nsb + sb) * (kKSteps * kbytes), kKSteps * kbytes, full);
        }
        __syncwarp();
        C.ncs++;
        const bool opens = sb > 0 || g.first, closes = sb < g.nsb - 1 || g.last;
        // a new accumulation overwrites Z: the epilogue has read the last one
        if (opens && C.nz > 0 && !warp_wait(mbar_at(C.mb, kZEmpty), C.nz - 1u)) return false;
        if (!warp_wait(mbar_at(C.mb, kCsFull), C.ncs - 1u)) return false;
        fence_after();
        for (int ks = 0; ks < kKSteps; ++ks) {
            // on a tile's first spot block, each K-step waits for its columns of u
            if (sb == 0) {
                if (!warp_wait(mbar_at(C.mb, kUStep0 + ks), C.nu)) return false;
                fence_after();
            }
            const uint32_t acc = (opens && ks == 0) ? 0u : 1u;
            const uint64_t cs = cs0 + ((uint64_t)(ks * kbytes) >> 4);
            const uint64_t us = u0 + ((uint64_t)((ks % US) * kUSlot) >> 4);   // u's slot of this K-step
            // conj(C) u: [Z_re | Z_im] += C_re [u_re | u_im], both halves of u as one
            // operand of N = 256 (12 KB of shared memory read for its 128 cycles;
            // two of N = 128 read 16 KB); Z_re += C_im u_im, Z_im -= C_im u_re
            const uint64_t crh = cs, cih = cs + ((uint64_t)((F16 ? 1 : 2) * kCk) >> 4);
            const uint64_t crl = cs + ((uint64_t)kCk >> 4), cil = cs + ((uint64_t)(3 * kCk) >> 4);
            const uint64_t urh = us, uih = us + ((uint64_t)kUc >> 4);
            const uint64_t url = us + ((uint64_t)(2 * kUc) >> 4), uil = us + ((uint64_t)(3 * kUc) >> 4);
            if (elect_one()) {
                mma(z_re, crh, urh, id2, acc);
                mma(z_re, cih, uih, id, 1u);
                mma(z_im, cih, urh, idn, 1u);
                if (!F16) {
                    mma(z_re, crh, url, id2, 1u);
                    mma(z_re, crl, urh, id2, 1u);
                    mma(z_re, cih, uil, id, 1u);
                    mma(z_re, cil, uih, id, 1u);
                    mma(z_im, cih, url, idn, 1u);
                    mma(z_im, cil, urh, idn, 1u);
                }
                if (sb == g.nsb - 1) commit(mbar_at(C.mb, ufree + ks));
            }
            __syncwarp();
        }
        if (sb == 0) C.nu++;
        if (elect_one()) {
            commit(mbar_at(C.mb, kCsFree));
            if (closes) commit(mbar_at(C.mb, kZFull));
        }
        __syncwarp();
        if (closes) C.nz++;
    }
    return true;
}

// Every MMA of an issuing warp done before tensor memory is freed, and every
// copy of a warp landed before shared memory is; true when all ended in time.
template <int R>
__device__ __forceinline__ bool drain(const Ctl &C, bool mmas)
{
    bool drained = true;
    if (mmas) {
        if (elect_one()) commit(mbar_at(C.mb, kDrain));
        __syncwarp();
        drained = warp_wait(mbar_at(C.mb, kDrain), 0u);
    }
    for (uint32_t s = 0; s < (uint32_t)R; ++s) {
        const uint32_t loads = (C.ql + R - 1u - s) / R;   // chunks q < ql with q % R == s
        if (loads) drained &= warp_wait(mbar_at(C.mb, kFull0 + s), loads - 1u);
    }
    if (C.ncs) drained &= warp_wait(mbar_at(C.mb, kCsFull), C.ncs - 1u);
    return drained;
}

__device__ __forceinline__ Ctl ctl_init(const SmemWs &m, uint32_t mb, uint32_t tmem)
{
    Ctl C;
    C.mb = mb;
    C.tmem = tmem;
    C.ring = saddr(m.ring);
    C.cs = saddr(m.cs);
    C.u = saddr(m.u);
    C.ql = C.qm = C.nz = C.ncs = C.nu = 0u;
    return C;
}

// The GEMM 2 warp: per published tile with products, GEMM 2 as u's K-steps
// come in; the info slot goes back as soon as it is read.
template <bool F16, int US>
__device__ __noinline__ void control_gemm2(const SmemWs &m, const Info *info, uint32_t mb, uint32_t tmem,
                                           unsigned *status)
{
    Ctl C = ctl_init(m, mb, tmem);
    bool ok = true;
    for (uint32_t k = 0;; ++k) {
        const int j = k & 1;
        ok = warp_wait(mbar_at(mb, kReady0 + j), (k >> 1) & 1u);
        if (!ok || info[j].done) break;
        const int empty = info[j].empty, P = info[j].H.P;
        G2Info g;
        g.cstab = F16 ? info[j].H.cstab16 : info[j].H.cstab;
        g.nsb = nspotblocks(info[j].H.N);
        g.cb = info[j].tile % ((P + kCols - 1) / kCols);
        g.first = info[j].first;
        g.last = info[j].last;
        __syncwarp();
        if ((threadIdx.x & 31) == 0) arrive(mbar_at(mb, kSEmpty0 + j));
        if (empty) continue;
        ok = gemm2<F16, US>(C, g);
        if (!ok) break;
    }
    const bool drained = drain<Lay<US>::kRing>(C, true);
    if ((!ok || !drained) && (threadIdx.x & 31) == 0) atomicOr(status, 1u);
}

// The GEMM 1 warp: per published tile with products, GEMM 1 into S buffer j
// as the producer's stages land; then it gives info slot j back.
template <int R>
__device__ __noinline__ void control_gemm1(const SmemWs &m, const Info *info, uint32_t mb, uint32_t tmem,
                                           unsigned *status)
{
    Ctl C = ctl_init(m, mb, tmem);
    bool ok = true;
    for (uint32_t k = 0;; ++k) {
        const int j = k & 1;
        ok = warp_wait(mbar_at(mb, kReady0 + j), (k >> 1) & 1u);
        if (!ok) break;
        const int done = info[j].done, empty = info[j].empty, N = info[j].H.N;
        if (done) break;
        if (!empty) {
            fence_after();
            ok = gemm1<R>(C, nchunks(N), j);
        }
        __syncwarp();
        if ((threadIdx.x & 31) == 0) arrive(mbar_at(mb, kSEmpty0 + j));
        if (!ok) break;
    }
    const bool drained = drain<R>(C, true);
    if ((!ok || !drained) && (threadIdx.x & 31) == 0) atomicOr(status, 1u);
}

// The slot of work item `item`, at or after `slot` (tile_begin rises with the
// slot): 32 slots looked at per step by the whole warp.
__device__ __forceinline__ int find_slot(const LaunchSlot *__restrict__ slots, int nslots, int slot, int item)
{
    for (;;) {
        const int i = slot + 1 + (int)(threadIdx.x & 31);
        const unsigned m = __ballot_sync(0xffffffffu, i < nslots && slots[min(i, nslots - 1)].tile_begin <= item);
        slot += __popc(m);
        if (m != 0xffffffffu) return slot;
    }
}

// The producer warp: takes work items (strips), publishes their tiles one by
// one, and loads GEMM 1's operand stages of each (running up to the ring's
// depth ahead of the MMAs).  The pop of the next item and the global loads of
// the item's slot and descriptor are issued ahead of the waits they would
// otherwise follow.
template <int R>
__device__ __noinline__ void control_load(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots,
                                           int nslots, int total_tiles, unsigned *queue, const SmemWs &m,
                                           Info *info, uint32_t mb, uint32_t tmem, unsigned *status)
{
    constexpr int kHWords = (int)(sizeof(HoloDev) / 4), kHPer = (kHWords + 31) / 32;
    static_assert(sizeof(HoloDev) % 4 == 0, "word copies");
    Ctl C = ctl_init(m, mb, tmem);
    const int lane = threadIdx.x & 31;
    const bool lane0 = lane == 0;
    bool ok = true;
    int slot = 0;   // a block's items only rise, so their slots are found by scanning forward
    int item = blockIdx.x;   // the first items go to the blocks in order, the rest through the queue
    uint32_t k = 0;        // tiles published
    uint32_t before = 0;   // those with products
    for (bool stop = false; !stop;) {
        const bool fin = item >= total_tiles || !ok;
        // the next item's pop is in flight while this one is published and multiplied
        int next = total_tiles;
        if (lane0 && !fin) next = (int)(gridDim.x + atomicAdd(queue, 1u));
        const HoloDev *Hp = nullptr;
        LaunchSlot sl{};
        uint32_t hw[kHPer];
        // the strip: row block rb, column tiles c0 .. c1 - 1, the ones with
        // products cf .. cl (a round pupil is convex: they are contiguous)
        int rb = 0, c0 = 0, c1 = 1, col_tiles = 1, cf = -1, cl = -1;
        if (!fin) {
            slot = find_slot(slots, nslots, slot, item);
            sl = slots[slot];
            Hp = &holos[sl.holo];
            const uint32_t *src = reinterpret_cast<const uint32_t *>(Hp);
#pragma unroll
            for (int i = 0; i < kHPer; ++i) {
                const int w = lane + 32 * i;
                hw[i] = w < kHWords ? __ldg(src + w) : 0u;
            }
            col_tiles = (Hp->P + kCols - 1) / kCols;
            const int S = max(1, sl.strip), per_row = (col_tiles + S - 1) / S;
            const int s_loc = item - sl.tile_begin;
            rb = s_loc / per_row;
            c0 = (s_loc % per_row) * S;
            c1 = min(c0 + S, col_tiles);
            for (int c = c0; c < c1; ++c)
                if (!tile_outside(*Hp, rb * col_tiles + c)) {
                    if (cf < 0) cf = c;
                    cl = c;
                }
        }
        for (int c = c0; c < c1; ++c) {
            const int j = k & 1;
            // S buffer j and info slot j are free once the epilogue and the GEMM 1
            // warp are done with tile k - 2
            if (k >= 2 && ok) ok = warp_wait(mbar_at(mb, kSEmpty0 + j), (k >> 1) - 1u);
            stop = fin || !ok;
            const bool empty = stop || cf < 0 || c < cf || c > cl;
            if (stop) {
                if (lane0) info[j].done = 1;
            } else {
                if (lane0) {
                    info[j].item = item;
                    info[j].tile = rb * col_tiles + c;
                    info[j].empty = empty ? 1 : 0;
                    info[j].done = 0;
                    info[j].first = c == cf ? 1 : 0;
                    info[j].last = c == cl ? 1 : 0;
                    info[j].zero = (cf < 0 && c == c1 - 1) ? 1 : 0;
                    info[j].before = before;
                    info[j].sl = sl;
                }
                uint32_t *dst = reinterpret_cast<uint32_t *>(&info[j].H);
#pragma unroll
                for (int i = 0; i < kHPer; ++i) {
                    const int w = lane + 32 * i;
                    if (w < kHWords) dst[w] = hw[i];
                }
            }
            __syncwarp();
            if (lane0) arrive(mbar_at(mb, kReady0 + j));
            ++k;
            if (stop) {
                // the end goes to both u groups: into the other slot too
                if (k >= 2 && ok) ok = warp_wait(mbar_at(mb, kSEmpty0 + (j ^ 1)), (k >> 1) - 1u);
                if (lane0) {
                    info[j ^ 1].done = 1;
                    arrive(mbar_at(mb, kReady0 + (j ^ 1)));
                }
                break;
            }
            if (!empty) before++;
            if (!empty) ok = load_gemm1<R>(C, *Hp, rb, c);
        }
        item = __shfl_sync(0xffffffffu, next, 0);
    }
    // this block pops no more; the last one to say so clears the queue
    if (lane0 && atomicAdd(queue + 1, 1u) == gridDim.x - 1) {
        queue[0] = 0u;
        queue[1] = 0u;
        __threadfence();
    }
    __syncwarp();
    const bool drained = drain<R>(C, false);
    if ((!ok || !drained) && lane0) atomicOr(status, 1u);
}

// a b for complex a, b.
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// sin and cos of 2 pi T / 2^32 + corr to FP32 rounding (corr small): the top 24
// bits of T through sincospi, the rest and corr to first order.
__device__ __forceinline__ float2 phasor_exact(int32_t T, float corr)
{
    const int32_t hi = T & ~0xFF;
    float s, c;
    sincospif((float)hi * 0x1p-31f, &s, &c);   // hi has 24 significant bits: exact
    const float r = fmaf((float)(T & 0xFF), kTwoPiF * 0x1p-32f, corr);
    return make_float2(fmaf(-s, r, c), fmaf(c, r, s));
}

// The partial V_n = sum_y conj(R_n(y)) Z(n, y) of spot n of a closed Z
// accumulation (a strip at row block y0) over the tile's rows ys0 .. ys1 - 1.  R_n(y)
// along the rows by recurrence: its phase is quadratic in y, so R(y + 1) =
// R(y) D(y) and D(y + 1) = D(y) E with the constant E = e^{i (2 pi 2 Gh / 2^32
// + 2 gl)}; R and D are evaluated directly every 8 rows (the product's
// rounding grows with the run length).  Within a run the even and the odd rows
// go side by side in packed FP32 pairs, which the rows' Z are in as loaded:
// R(y + 2) = R(y) D2(y) and D2(y + 2) = D2(y) E^4 from D2(y) = D(y) D(y + 1).
// Every lane computes (a lane past N uses spot N - 1's factors and stores
// nothing): no divergent branch in the row loop.  A latency-bound chain: for
// holograms of more than 128 spots GEMM 2 waits for it, once per spot block.
// (Two runs in a pair instead, rows y and y + 8: seven steps one after the other
// and Z's rows moved into pairs; 64 holograms of N up to 300 12.34 ms against
// 11.93.)
// An error of E is the same way round in every run: with the hardware's sine and
// cosine every theta_n is off by 2e-6 rad rms per iteration.  With EXACT, E^4 is
// right to FP32 rounding and R and D2 are evaluated for even and odd rows each:
// 2e-7 to 3e-7, as much as phasors of each pixel's own.  Serving takes it where a
// request would otherwise run on those: u of 32 requests of N up to 1000 ends
// 6e-7 from exact (1.6e-6 on FP32 phasors, 2.8e-6 without), in the same time.
template <bool EXACT>
__device__ __forceinline__ float2 strip_dot(uint32_t z_re, uint32_t z_im, const int4 *coef, int n, int N, int y0,
                                            int half, int ys0, int ys1)
{
    const int4 cf = coef[min(n, N - 1)];
    const int32_t tilt = cf.y, Gh = cf.z;
    const float gl = __int_as_float(cf.w);
    float2 E, E3, E4;
    if constexpr (EXACT) {
        E4 = phasor_exact((int32_t)(8u * (uint32_t)Gh), 8.f * gl);
        E = E3 = E4;   // not used
    } else {
        sincos_fix(kFixRound + 2u * (uint32_t)Gh, fmaf(2.f, gl, -kTwoPiF), E.y, E.x);
        const float2 E2 = cmul(E, E);
        E3 = cmul(E2, E);
        E4 = cmul(E2, E2);
    }
    const uint64_t F_c = pack2(E.x, E3.x), F_s = pack2(E.y, E3.y), nF_s = pack2(-E.y, -E3.y);
    const uint64_t E_c = pack2(E4.x, E4.x), E_s = pack2(E4.y, E4.y), nE_s = pack2(-E4.y, -E4.y);
    uint64_t vr = 0ull, vi = 0ull;   // even and odd rows; vi is the sum's negative imaginary part
#pragma unroll 1
    for (int ys = ys0; ys < ys1; ys += 16) {
        float zr[16], zi[16];
        ld16(z_re + ys, zr);
        ld16(z_im + ys, zi);
        uint64_t Rc[8], Rs[8];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            // R at the run's first rows u0 and u0 + 1, and D2 there
            const int u0 = y0 + ys + 8 * b - half;
            const float2 r = spot_factor(tilt, Gh, gl, u0, kFixRound, 1.f);
            float2 r1;
            uint64_t Dc, Ds;
            if constexpr (EXACT) {
                // phase of R(u + 2) / R(u): tilt 2 + Gh (4 u + 4)
                float2 d0, d1;
                r1 = spot_factor(tilt, Gh, gl, u0 + 1, kFixRound, 1.f);
                sincos_fix(kFixRound + 2u * (uint32_t)tilt + (uint32_t)Gh * (uint32_t)(4 * u0 + 4),
                           fmaf(gl, (float)(4 * u0 + 4), -kTwoPiF), d0.y, d0.x);
                sincos_fix(kFixRound + 2u * (uint32_t)tilt + (uint32_t)Gh * (uint32_t)(4 * u0 + 8),
                           fmaf(gl, (float)(4 * u0 + 8), -kTwoPiF), d1.y, d1.x);
                Dc = pack2(d0.x, d1.x);
                Ds = pack2(d0.y, d1.y);
            } else {
                // D, the phase of R(u + 1) / R(u): tilt + Gh (2 u + 1); D2 = D^2 E and D^2 E^3
                const int du = 2 * u0 + 1;
                float2 d;
                sincos_fix(kFixRound + (uint32_t)tilt + (uint32_t)Gh * (uint32_t)du, fmaf(gl, (float)du, -kTwoPiF), d.y,
                           d.x);
                r1 = cmul(r, d);
                const float2 dd = cmul(d, d);
                const uint64_t dc = pack2(dd.x, dd.x), ds = pack2(dd.y, dd.y);
                Dc = fma2(dc, F_c, mul2(ds, nF_s));
                Ds = fma2(dc, F_s, mul2(ds, F_c));
            }
            Rc[4 * b] = pack2(r.x, r1.x);
            Rs[4 * b] = pack2(r.y, r1.y);
#pragma unroll
            for (int q = 4 * b; q < 4 * b + 3; ++q) {
                const uint64_t nDs = Ds ^ 0x8000000080000000ull;
                Rc[q + 1] = fma2(Rc[q], Dc, mul2(Rs[q], nDs));
                Rs[q + 1] = fma2(Rc[q], Ds, mul2(Rs[q], Dc));
                if (q < 4 * b + 2) {
                    const uint64_t t = fma2(Dc, E_c, mul2(Ds, nE_s));
                    Ds = fma2(Dc, E_s, mul2(Ds, E_c));
                    Dc = t;
                }
            }
        }
        ld_wait();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint64_t a = pack2(zr[2 * q], zr[2 * q + 1]), b = pack2(zi[2 * q], zi[2 * q + 1]);
            vr = fma2(Rc[q], a, fma2(Rs[q], b, vr));
            vi = fma2(Rs[q], a, fma2(Rc[q] ^ 0x8000000080000000ull, b, vi));
        }
    }
    const float2 r = unpack2(vr), i = unpack2(vi);
    return make_float2(r.x + r.y, -(i.x + i.y));
}

// The columns xl .. xr of grid row gy that lie in the pupil: the grid's, within
// the round pupil (|x - half|^2 + (gy - half)^2 <= half^2) unless the aperture
// is square; xr < xl for a row outside.
__device__ __forceinline__ void row_span(int P, int aperture, int gy, int &xl, int &xr)
{
    const int half = P >> 1, yq = gy - half;
    const int R2 = half * half, yq2 = yq * yq;   // P <= 32768: squares stay below 2^30
    xl = 0;
    xr = gy < P ? P - 1 : -1;
    if (aperture != 0) {
        const int D = R2 - yq2;
        int wr = -1;
        if (D >= 0) {
            wr = (int)sqrtf((float)D);   // within 1 of floor(sqrt(D))
            if ((wr + 1) * (wr + 1) <= D) ++wr;
            if (wr * wr > D) --wr;
        }
        xl = max(xl, half - wr);
        xr = min(xr, half + wr);
    }
}

// arg(x + i y) in [0, 2 pi] for x, y not both 0 and of ordinary size: atan of
// the smaller over the larger side (a division by reciprocal and one residual
// step) by an odd polynomial of degree 17 (least relative error on [0, 1],
// 1.5e-8, found by reweighted least squares), then the octant, with pi / 2 in
// two parts.  Error 3.5e-7 rad at most and 1e-7 rms (atan2f and the turn added
// below 0: 5e-7, 1.4e-7), in ~30 instructions without a branch: the final
// pass's maps on 4 warps bound a tile through atan2f (10 k cycles against 8.8 k
// for the tile's products).
__device__ __forceinline__ float arg_turn(float y, float x)
{
    const float ax = fabsf(x), ay = fabsf(y), mx = fmaxf(ax, ay), mn = fminf(ax, ay);
    float rc;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(mx));
    float q = mn * rc;
    q = fmaf(fmaf(-q, mx, mn), rc, q);
    const float z = q * q;
    float p = 0.0028498878236860037f;
    p = fmaf(p, z, -0.016068624332547188f);
    p = fmaf(p, z, 0.04269151762127876f);
    p = fmaf(p, z, -0.07504294812679291f);
    p = fmaf(p, z, 0.10640934109687805f);
    p = fmaf(p, z, -0.14203645288944244f);
    p = fmaf(p, z, 0.1999261975288391f);
    p = fmaf(p, z, -0.3333307206630707f);
    p = fmaf(p, z, 1.0f);
    const float t = q * p;
    const bool swap = ay > ax;
    const uint32_t sx = __float_as_uint(x), sy = __float_as_uint(y);
    const bool xn = (int)sx < 0, yn = (int)sy < 0;
    const float k = swap ? (yn ? 3.f : 1.f) : (xn ? 2.f : (yn ? 4.f : 0.f));   // quarter turns
    const uint32_t flip = (sx ^ sy ^ (swap ? 0x80000000u : 0u)) & 0x80000000u;
    const float st = __uint_as_float(__float_as_uint(t) ^ flip);
    return fmaf(k, 1.57079637f, fmaf(k, -4.37113883e-8f, st));
}

// The final pass's phase map Phi = arg S (Eq. 1) and SLM gray levels of one
// tile row (grid row gy, K-steps ks0 .. ks1 - 1 of the 64 columns from x0 on), from
// S in tensor memory, K-step by K-step: 0 outside the pupil.  Every lane of the warp runs the tensor-memory
// loads (they are warp-collective); a row past the grid stores nothing.
__device__ __forceinline__ void final_phases(const HoloDev &H, uint32_t s_re, uint32_t s_im, int gy, int x0, int ks0,
                                             int ks1)
{
    const int P = H.P;
    int xl, xr;
    row_span(P, H.aperture, gy, xl, xr);
#pragma unroll 1
    for (int ks = ks0; ks < ks1; ++ks) {
        const int gx0 = x0 + 16 * ks;
        float sr[16], si[16], o[16];
        __syncwarp();   // converged for the warp-collective loads
        ld16(s_re + 16 * ks, sr);
        ld16(s_im + 16 * ks, si);
        ld_wait();
        uint64_t n2[8];
        const bool normal = norms16(sr, si, n2);
        if (!__all_sync(0xffffffffu, normal)) rescale16(sr, si, n2);
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
            const int x = gx0 + jj;
            const float ph = arg_turn(si[jj], sr[jj]);
            o[jj] = (ph >= kTwoPiF || x < xl || x > xr) ? 0.f : ph;
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int col = gx0 + 4 * g;
            if (gy >= P || col >= P) break;
            if (H.phase_out) {
                float *dst = H.phase_out + (size_t)gy * P + col;
                if (col + 3 < P && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
                    *reinterpret_cast<float4 *>(dst) = make_float4(o[4 * g], o[4 * g + 1], o[4 * g + 2], o[4 * g + 3]);
                } else {
                    for (int e = 0; e < 4; ++e)
                        if (col + e < P) dst[e] = o[4 * g + e];
                }
            }
            if (H.slm) write_gray4(H, gy, col, o + 4 * g);
        }
    }
}

// A group of u warps (epilogue 1): per tile (UG = 2: of its S buffer), u = A S / |S| into
// GEMM 2's B operand, K-step by K-step: K-step ks goes to u's slot ks once
// GEMM 2 has read the slot's last K-step, the previous tile's (computed first,
// stored after the wait).  A tile outside the pupil gets, in the final pass,
// phase 0 and gray lut[0] here, and a strip with no tile inside the pupil its
// zero partials.
template <int UG, bool F16, int US>
__device__ __forceinline__ void epilogue_u(const SmemWs &m, const Info *info, uint32_t mb, uint32_t tmem,
                                           unsigned *status)
{
    static_assert(US == kKSteps, "a slot per K-step");
    constexpr int kT = 128;
    const int tid = threadIdx.x & (kT - 1), lane = tid & 31, q = tid >> 5;   // TMEM lane quadrant q
    const uint32_t lanes = (uint32_t)(32 * q) << 16;
    uint32_t n_seen = 0u;   // this group's tiles with products, per S buffer (low half: j = 0, high half: j = 1)
    bool ok = true;
    for (uint32_t k = threadIdx.x / kT;; k += UG) {
        const int j = k & 1;   // S buffer and info slot
        ok = warp_and(wait(mbar_at(mb, kReady0 + j), (k >> 1) & 1u));
        if (!ok || info[j].done) break;
        const int item = info[j].item, empty = info[j].empty, t = info[j].tile, zero = info[j].zero;
        const uint32_t before = info[j].before;
        const LaunchSlot sl = info[j].sl;
        const HoloDev H = info[j].H;   // by value: global stores below cannot alias it
        const int P = H.P, N = H.N, half = P >> 1, pass = sl.pass;
        const int col_tiles = (P + kCols - 1) / kCols;
        const int y0 = (t / col_tiles) * kRows, x0 = (t % col_tiles) * kCols;
        if (empty) {
            // wholly outside the round pupil: in the final pass phase 0 (gray
            // lut[0]) over its grid pixels; a strip without products has zero
            // partials
            __syncwarp();
            if (lane == 0) arrive(mbar_at(mb, kSEmpty0 + j));
            if (zero) {
                const size_t s_loc = (size_t)(item - sl.tile_begin);
                for (int n = tid; n < N; n += kT) {
                    if (pass == kPassFinal) H.part64[s_loc * N + n] = make_double2(0.0, 0.0);
                    else H.part[s_loc * N + n] = make_float2(0.f, 0.f);
                }
            }
            if (pass == kPassFinal) {
                const int rows = min(kRows, P - y0), cols = min(kCols, P - x0);
                const uint8_t g0 = H.slm ? __ldg(H.lut) : 0;
                for (int f = tid; f < rows * cols; f += kT) {
                    const int r = y0 + f / cols, c = x0 + f % cols;
                    if (H.phase_out) H.phase_out[(size_t)r * P + c] = 0.f;
                    if (H.slm) H.slm[(size_t)r * H.slm_pitch + c] = g0;
                }
            }
            continue;
        }

        // A compressed pass reads the subset mask bits of the tile's columns
        // first (two words: x0 is a multiple of 64), before the waits.
        const int row = 32 * q + lane, gy = y0 + row;
        uint64_t mword = ~0ull;
        if (pass == kPassSubset) {
            const int w0 = x0 >> 5;
            if (gy < P) {
                const uint32_t *mrow = subset_mask(H, sl.j) + (size_t)gy * H.mask_words;
                mword = (uint64_t)__ldg(mrow + w0) | (w0 + 1 < H.mask_words ? (uint64_t)__ldg(mrow + w0 + 1) << 32 : 0ull);
            } else {
                mword = 0ull;
            }
        }
        // tiles with products on this S buffer up to this one (s_full[j] completes
        // once per such tile)
        n_seen += 1u << (16 * j);
        ok = warp_and(wait_newest(mbar_at(mb, kSFull0 + j), (n_seen >> (16 * j)) & 0xFFFFu));
        if (!ok) break;
        fence_after();
        {
            const uint32_t s_re = tmem + kS0 + 2 * kCols * j, s_im = s_re + kCols;
            const int yq = gy - half, yq2 = yq * yq;
            int xl, xr;
            row_span(P, H.aperture, gy, xl, xr);
            const float kA = H.kA;
            // the row's 16 columns of each K-step, with the Gaussian beam's
            // amplitude or the uniform one (a uniform branch outside the loop)
            auto ksteps = [&](auto gauss_tag) {
                constexpr bool kGauss = decltype(gauss_tag)::value;
#pragma unroll 1
                for (int ks = 0; ks < kKSteps; ++ks) {
                    const int xs = 16 * ks, gx0 = x0 + xs;
                    // the pixels that carry u: in the row's span and, in a
                    // compressed pass, in S_j (the rest add nothing to Eq. 3's sum)
                    const int lo = max(xl - gx0, 0), hi = min(xr - gx0, 15);
                    uint32_t bits = 0u;
                    if (lo <= hi) bits = (0xFFFFu >> (15 - hi + lo)) << lo;
                    bits &= (uint32_t)(mword >> xs);
                    float sr[16], si[16];
                    ld16(s_re + lanes + xs, sr);
                    ld16(s_im + lanes + xs, si);
                    ld_wait();
                    uint64_t n2[8];
                    const bool normal = norms16(sr, si, n2);
                    if (!warp_and(normal)) rescale16(sr, si, n2);
                    Packed8 pk[2];
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        uint64_t ur[4], ui[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            // branch-free: the lanes are rows, so a per-pixel branch
                            // (subset membership, the pupil edge) would diverge; a
                            // pixel without u takes the factor 0
                            const int jj = 8 * g + 2 * e;
                            const float2 n = unpack2(n2[jj >> 1]);
                            float r0 = rsqrt_approx(n.x), r1 = rsqrt_approx(n.y);
                            if constexpr (kGauss) {   // Eq. 3's A
                                const int xq = gx0 + jj - half;
                                r0 *= exp2f(-kA * (float)(xq * xq + yq2));
                                r1 *= exp2f(-kA * (float)((xq + 1) * (xq + 1) + yq2));
                            }
                            r0 = ((bits >> jj) & 1u) ? r0 : 0.f;
                            r1 = ((bits >> (jj + 1)) & 1u) ? r1 : 0.f;
                            const uint64_t rs = pack2(r0, r1);
                            ur[e] = mul2(pack2(sr[jj], sr[jj + 1]), rs);
                            ui[e] = mul2(pack2(si[jj], si[jj + 1]), rs);
                        }
                        pk[g] = pack8<F16>(ur, ui);
                    }
                    // u's slot of this K-step is free once GEMM 2 has read the last u
                    // in it, that of the last tile with products (number before - 1).
                    // A wait by parity has to find its phase current or just over:
                    // GEMM 2 can't be past that tile, since it waits for this one's u;
                    // and the phase before on that barrier, of tile before - 3, was over
                    // for tile before - 2's u, which this group wrote, or GEMM 2 took in
                    // before this tile was published.  (Phases counted per S buffer
                    // left the two groups without either bound: a group that looked
                    // late, at an empty tile, found the other's barrier a phase too
                    // far, and the block stood until its waits ran out.)
                    if (before > 0u && !warp_and(wait_newest(mbar_at(mb, kUFree0 + kKSteps * (int)((before - 1u) & 1u) + ks),
                                                             ((before - 1u) >> 1) + 1u)))
                        return false;
                    unsigned char *slot = m.u + (ks % US) * kUSlot;
                    store8<F16>(slot, kUc, core_off(row, 0, 16), pk[0]);
                    store8<F16>(slot, kUc, core_off(row, 8, 16), pk[1]);
                    // this K-step's columns of u are in place
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) arrive(mbar_at(mb, kUStep0 + ks));
                }
                return true;
            };
            ok = kA != 0.f ? ksteps(std::true_type{}) : ksteps(std::false_type{});
            if (!ok) break;
        }
        fence_before();
        __syncwarp();
        if (lane == 0) arrive(mbar_at(mb, kSEmpty0 + j));
    }
    if (!ok && lane == 0) atomicOr(status, 1u);
}

// The V warps (epilogue 2): per strip (after the GEMM 2 of its last tile with
// products) and spot block, the strip's partial V_n = sum_y conj(R_n(y))
// Z(n, y), one spot per thread over half the 128 rows, while the u warps go on with
// the next tiles.  In the final pass they also write each tile's phase map
// (and gray levels) from S, beside the u warps' work on u.
template <int UG, bool EXACT>
__device__ __forceinline__ void epilogue_v(const Info *info, float2 (*s_half)[kSpotBlock], uint32_t mb, uint32_t tmem,
                                           unsigned *status)
{
    const int tid = threadIdx.x - 128 * UG, lane = tid & 31, q = (tid >> 5) & 3;       // TMEM lane quadrant q
    const int hv = tid >> 7;                                                           // half of the rows
    const uint32_t lanes = (uint32_t)(32 * q) << 16;
    uint32_t n_z = 0u;   // Z accumulations reduced
    uint32_t n_s = 0u;   // tiles with products seen, per S buffer (low half: j = 0, high half: j = 1)
    bool ok = true;
    for (uint32_t k = 0;; ++k) {
        const int j = k & 1;
        ok = warp_and(wait(mbar_at(mb, kReady0 + j), (k >> 1) & 1u));
        if (!ok) break;
        if (info[j].done) break;
        const int item = info[j].item, empty = info[j].empty, t = info[j].tile, last = info[j].last;
        const int tile_begin = info[j].sl.tile_begin, pass = info[j].sl.pass;
        const int P = info[j].H.P, N = info[j].H.N;
        const int4 *coef = info[j].H.coef;
        float2 *part = info[j].H.part;
        double2 *part64 = info[j].H.part64;
        const int y0 = (t / ((P + kCols - 1) / kCols)) * kRows;
        if (!empty) n_s += 1u << (16 * j);
        if (!empty && pass == kPassFinal) {
            // the final pass's phase map, from S beside the u warps (S buffer j
            // goes back once both groups have read it)
            const HoloDev H = info[j].H;
            ok = warp_and(wait_newest(mbar_at(mb, kSFull0 + j), (n_s >> (16 * j)) & 0xFFFFu));
            if (!ok) break;
            fence_after();
            const uint32_t s_re = tmem + kS0 + 2 * kCols * j + lanes;
            final_phases(H, s_re, s_re + kCols, y0 + 32 * q + lane, (t % ((P + kCols - 1) / kCols)) * kCols,
                         hv * (kKSteps / 2), (hv + 1) * (kKSteps / 2));
            fence_before();
        }
        // the info slot (and S buffer) is read: it goes back with this group's arrival
        __syncwarp();
        if (lane == 0) arrive(mbar_at(mb, kSEmpty0 + j));
        if (empty || !last) continue;
        const int s_loc = item - tile_begin, half = P >> 1;
        for (int sb = 0; sb * kSpotBlock < N; ++sb) {
            n_z++;
            ok = warp_and(wait_newest(mbar_at(mb, kZFull), n_z));
            if (!ok) break;
            fence_after();
            const int n = sb * kSpotBlock + 32 * q + lane;
            float2 v = strip_dot<EXACT>(tmem + lanes, tmem + kRows + lanes, coef, n, N, y0, half, hv * (kRows / 2),
                                        (hv + 1) * (kRows / 2));
            fence_before();
            const uint32_t buf = n_z & 1u;
            if (hv) s_half[buf][32 * q + lane] = v;
            __syncwarp();
            if (lane == 0) {
                arrive(mbar_at(mb, kZEmpty));
                if (hv) arrive(mbar_at(mb, kDot0 + buf));
            }
            if (hv) continue;
            // the first V warps add the second ones' halves (the second ones write
            // a buffer again only after Z has been released twice more)
            ok = warp_and(wait_newest(mbar_at(mb, kDot0 + buf), (n_z + 1u) >> 1));
            if (!ok) break;
            const float2 w = s_half[buf][32 * q + lane];
            v.x += w.x;
            v.y += w.y;
            if (n < N) {
                const size_t off = (size_t)s_loc * N + n;
                if (pass == kPassFinal) part64[off] = make_double2((double)v.x, (double)v.y);
                else part[off] = make_float2(v.x, v.y);
            }
        }
        if (!ok) break;
    }
    if (!ok && lane == 0) atomicOr(status, 1u);
}

}  // namespace ws

}  // namespace tc

template <int UG, bool F16, int US, bool EXACT>
__global__ void __launch_bounds__(tc::ws::Cfg<UG>::kThreads, 1)
iter_full_tcws_kernel(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots, int nslots,
                      int total_tiles, unsigned *queue)
{
    using namespace tc::ws;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_mbar[kBarsWs];
    __shared__ Info s_info[2];
    __shared__ float2 s_half[2][tc::kSpotBlock];
    __shared__ uint32_t s_tmem;
    constexpr int W = Cfg<UG>::kEpi;   // the producer's warp
    const int tid = threadIdx.x, warp = tid >> 5;
    // queue[3] != 0 (a test of the bounded waits): the producer publishes no
    // work item, so every other role's first wait runs out, before any copy
    // or MMA is issued; queue[4] != 0: the poll limit of every wait
    chain_start();
    const bool withhold = queue[3] != 0u;
    if (tid == 0) {
        tc::s_wait_polls = queue[4] != 0u ? queue[4] : tc::kWaitPolls;
        for (int b = 0; b < kBarsWs; ++b) {
            // the epilogue's releases arrive once per warp
            // S buffers and info slots go back from a u group, the V warps and both GEMM warps
            const uint32_t cnt = (b == kSEmpty0 || b == kSEmpty0 + 1) ? 4 + kVWarps + 2
                                 : b == kZEmpty                               ? kVWarps
                                 : (b == kDot0 || b == kDot0 + 1)             ? kVWarps / 2
                                 : (b >= kUStep0 && b < kUStep0 + kKSteps)    ? 4
                                 : b == kDrain                                ? 2
                                                                              : 1;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(tc::saddr(&s_mbar[b])), "r"(cnt));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W) {
        // the first item's slot and descriptor on their way into L1 while the
        // block sets up (the producer's chain of loads, a memory latency each,
        // took 2.8 k cycles of a one-hologram launch's 30 k)
        const int slot = find_slot(slots, nslots, 0, (int)blockIdx.x);
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&holos[slots[slot].holo]);
        for (int i = 8 * (tid & 31); i < (int)(sizeof(HoloDev) / 4); i += 8 * 32)
            asm volatile("prefetch.global.L1 [%0];" :: "l"(src + i));
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tc::saddr(&s_tmem)), "r"(kTmemColsWs));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    chain_wait();   // the R' tables, the masks, and the last launch's queue
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t mb = tc::saddr(&s_mbar[0]);
    const SmemWs m = carve_ws<US>(smem);
    constexpr int R = Lay<US>::kRing;
    unsigned *status = queue + 2;
    if (warp == W) {
        if (!withhold) control_load<R>(holos, slots, nslots, total_tiles, queue, m, s_info, mb, s_tmem, status);
    } else if (warp == W + 1) {
        control_gemm1<R>(m, s_info, mb, s_tmem, status);
    } else if (warp == W + 2) {
        control_gemm2<F16, US>(m, s_info, mb, s_tmem, status);
    } else if (warp < Cfg<UG>::kU) {
        epilogue_u<UG, F16, US>(m, s_info, mb, s_tmem, status);
    } else {
        epilogue_v<UG, EXACT>(s_info, s_half, mb, s_tmem, status);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(s_tmem), "r"(kTmemColsWs));
}

// The per-hologram tails of a launch whose kernel writes tile partials: the
// weighted update (Eqs. 4-6) or the metrics (Eq. 7), a cluster of CL blocks per
// slot.  Bound by latency: a hologram's partials (27 to 162 items x N) are few
// bytes, and on one SM their loads and FP64 additions queue behind each other,
// so a launch of few holograms spreads each over up to 8 SMs.  Spots are dealt
// out in fours (a 32-byte sector of an item's partials), a block taking every
// CL-th; the lanes of a warp are 4 spots x 8 groups of items, and where a block
// has warps to spare 2 to 16 of them share four spots.  The blocks' sums of
// |V_n| (or e and the extremes of I_n) meet in distributed shared memory.
// The blocks with blockIdx.y > 0 (compressed launches) clear the slot's subset
// mask for the next draw.  On one block of 1024 threads a lone hologram's update
// took 7 us (N = 100) and its metrics 38 us (N = 300: 63 us), most of it FP64
// additions; a whole final pass at N = 300 fell from 240 to 184 us per call.
constexpr int kTailThreads = 512;
constexpr int kTailMaxN = 6144;
constexpr int kTailClear = 8;               // blocks per slot that clear its mask

// Shared memory of a block whose share is nq fours: the warps' sums (16 bytes
// per spot and warp sharing it) and V_n.
__host__ __device__ constexpr size_t tail_smem(int nq)
{
    return (size_t)4 * 16 * (nq > kTailThreads / 32 ? nq : kTailThreads / 32) + (size_t)4 * 8 * nq;
}

// Sum of spot n's partials over the items t = g, g + G, ..., combined over the
// 8 lane groups of the warp (lanes that differ in bits 2 to 4).
__device__ __forceinline__ float4 tail_warp_sum(const HoloDev &H, int n, int g, int G, int tiles)
{
    const float4 q = tile_sum(H, n, g, G, tiles);
    float sr = q.x, cr = q.y, si = q.z, ci = q.w;   // the sum is s - c
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        add_comp(sr, cr, __shfl_xor_sync(0xffffffffu, sr, o), __shfl_xor_sync(0xffffffffu, cr, o));
        add_comp(si, ci, __shfl_xor_sync(0xffffffffu, si, o), __shfl_xor_sync(0xffffffffu, ci, o));
    }
    return make_float4(sr, cr, si, ci);
}

__device__ __forceinline__ double2 tail_warp_sum64(const HoloDev &H, int n, int g, int G, int tiles)
{
    const double2 v = tile_sum64(H.part64 + n, H.N, g, G, tiles);
    double vr = v.x, vi = v.y;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        vr += __shfl_xor_sync(0xffffffffu, vr, o);
        vi += __shfl_xor_sync(0xffffffffu, vi, o);
    }
    return make_double2(vr, vi);
}

template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kTailThreads)
tcws_tails_kernel(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots)
{
    constexpr int W = kTailThreads / 32;
    extern __shared__ __align__(16) double2 s_part[];   // per spot and warp: float4 {s_re, c_re, s_im, c_im} or FP64
    __shared__ double s_red[W];
    __shared__ double s_out[3];                  // this block's sum (and extremes), read by the cluster
    __shared__ double s_mean;
    const LaunchSlot sl = slots[blockIdx.x / CL];
    const HoloDev &H = holos[sl.holo];
    const int rank = blockIdx.x % CL, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_start();
    if (8 * tid < (int)sizeof(HoloDev))
        asm volatile("prefetch.global.L1 [%0];" :: "l"(reinterpret_cast<const char *>(&H) + 8 * tid));
    chain_wait();
    if (blockIdx.y > 0) {   // a whole cluster of its own
        if (sl.pass == kPassSubset && H.mask) {
            uint32_t *mask = subset_mask(H, sl.j);
            const size_t words = (size_t)H.P * H.mask_words;
            const size_t part = (blockIdx.y - 1) * CL + rank;
            for (size_t i = part * kTailThreads + tid; i < words; i += (size_t)kTailClear * kTailThreads) mask[i] = 0u;
        }
        return;
    }
    const int N = H.N, quads = (N + 3) / 4;
    const int nq = (quads - rank + CL - 1) / CL;   // this block's fours: rank, rank + CL, ...
    int wq = W;                                                        // warps per four spots: a power of two
    while (wq > 1 && wq * nq > W) wq >>= 1;
    const bool metrics = sl.pass == kPassFinal;
    float4 *s_part32 = reinterpret_cast<float4 *>(s_part);
    float2 *s_v = reinterpret_cast<float2 *>(s_part + 4 * max(nq, W));
    for (int i = warp / wq; i < nq; i += W / wq) {
        const int n = min(4 * (rank + CL * i) + (lane & 3), N - 1);   // past the last spot: not stored
        const int g = (lane >> 2) + 8 * (warp % wq), at = (i * wq + warp % wq) * 4 + lane;
        if (metrics) {
            const double2 v = tail_warp_sum64(H, n, g, 8 * wq, sl.tiles);
            if (lane < 4) s_part[at] = v;
        } else {
            const float4 v = tail_warp_sum(H, n, g, 8 * wq, sl.tiles);
            if (lane < 4) s_part32[at] = v;
        }
    }
    __syncthreads();
    // one thread per spot of this block
    const float inv = 1.0f / (float)sl.count;
    const double inv64 = 1.0 / H.norm;   // sum of A over the pupil (P^2 for the square uniform grid)
    double sum = 0.0, imax = -1.0, imin = 1e300;
    for (int k = tid; k < 4 * nq; k += kTailThreads) {
        const int i = k >> 2, n = 4 * (rank + CL * i) + (k & 3);
        if (n >= N) continue;
        if (metrics) {
            double vr = 0.0, vi = 0.0;
            for (int g = 0; g < wq; ++g) {
                const double2 p = s_part[(i * wq + g) * 4 + (k & 3)];
                vr += p.x;
                vi += p.y;
            }
            vr *= inv64;
            vi *= inv64;
            const double in = vr * vr + vi * vi;
            H.metrics[2 + n] = in;
            sum += in;
            imax = fmax(imax, in);
            imin = fmin(imin, in);
        } else {
            float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
            for (int g = 0; g < wq; ++g) {
                const float4 p = s_part32[(i * wq + g) * 4 + (k & 3)];
                add_comp(sr, cr, p.x, p.y);
                add_comp(si, ci, p.z, p.w);
            }
            const float2 v = make_float2((sr - cr) * inv, (si - ci) * inv);
            s_v[k] = v;
            sum += (double)hypotf(v.x, v.y);
        }
    }
    sum = block_sum_f64<kTailThreads>(sum, s_red);
    if (metrics) {
        imax = block_max_f64<kTailThreads>(imax, s_red);
        imin = block_min_f64<kTailThreads>(imin, s_red);
    }
    if (tid == 0) {
        s_out[0] = sum;
        s_out[1] = imax;
        s_out[2] = imin;
    }
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    cluster.sync();
    if (metrics) {
        if (rank == 0 && tid == 0) {
            double e = 0.0;
            imax = -1.0;
            imin = 1e300;
            for (int r = 0; r < CL; ++r) {
                const double *o = cluster.map_shared_rank(s_out, r);
                e += o[0];
                imax = fmax(imax, o[1]);
                imin = fmin(imin, o[2]);
            }
            H.metrics[0] = e;
            H.metrics[1] = (imax + imin) > 0.0 ? 1.0 - (imax - imin) / (imax + imin) : 0.0;
        }
    } else {
        if (warp == 0) {
            double m = lane < CL ? cluster.map_shared_rank(s_out, lane)[0] : 0.0;
            for (int o = CL / 2; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
            if (lane == 0) s_mean = m / (double)N;
        }
        __syncthreads();
        const double mean = s_mean;
        for (int k = tid; k < 4 * nq; k += kTailThreads) {
            const int n = 4 * (rank + CL * (k >> 2)) + (k & 3);
            if (n < N) update_spot(H, n, s_v[k], mean);
        }
    }
    cluster.sync();   // s_out is read before any block of the cluster leaves
}

template <int UG, bool F16, bool EXACT>
static int tcws_max_grid_of(int maxN, int sm_count)
{
    const auto kernel = iter_full_tcws_kernel<UG, F16, tc::ws::kKSteps, EXACT>;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return 0;
    const size_t limit = 227 * 1024 - fa.sharedSizeBytes;
    const size_t smem = tc::ws::Lay<tc::ws::kKSteps>::kSmem;
    if (smem > limit || maxN > kTailMaxN) return 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, tc::ws::Cfg<UG>::kThreads, smem) != cudaSuccess)
        return 0;
    return std::min(per_sm, 1) * sm_count;   // a block holds all 512 tensor-memory columns
}

// Resident blocks of the kernel (all forms; sets their shared-memory limits).
static int tcws_max_grid(int maxN, int sm_count)
{
    return std::min({tcws_max_grid_of<1, false, false>(maxN, sm_count), tcws_max_grid_of<1, true, false>(maxN, sm_count),
                     tcws_max_grid_of<2, false, false>(maxN, sm_count), tcws_max_grid_of<2, true, false>(maxN, sm_count),
                     tcws_max_grid_of<1, false, true>(maxN, sm_count), tcws_max_grid_of<2, false, true>(maxN, sm_count)});
}

template <int UG, bool F16, bool EXACT>
static cudaError_t tcws_launch_one(const HoloDev *holos, const LaunchSlot *slots, int nslots, int total_tiles,
                                   unsigned *queue, int grid, bool chain, cudaStream_t s)
{
    constexpr int K4 = tc::ws::kKSteps;
    return launch_chained(iter_full_tcws_kernel<UG, F16, K4, EXACT>, dim3(grid), dim3(tc::ws::Cfg<UG>::kThreads),
                          tc::ws::Lay<K4>::kSmem, chain, s, holos, slots, nslots, total_tiles, queue);
}

// The tails of a launch of `items` work items: clusters of as many blocks (up to
// 8) as leave every slot's on an SM of its own, one where a hologram's partials
// are a few loads per thread (the cluster's launch and barriers would cost more
// than they spread); and (compressed launches) the blocks that clear the masks.
cudaError_t launch_tc_tails(const HoloDev *holos, const LaunchSlot *slots, int nslots, int items, int maxN,
                            bool subset, int sm_count, cudaStream_t s)
{
    if (maxN > kTailMaxN) return cudaErrorInvalidValue;
    int cl = 8;
    while (cl > 1 && (cl * nslots > sm_count || (int64_t)items * maxN < (int64_t)2048 * nslots)) cl >>= 1;
    const dim3 grid((unsigned)(cl * nslots), 1u + (subset ? (unsigned)(kTailClear / cl) : 0u));
    const size_t smem = tail_smem((maxN + 4 * cl - 1) / (4 * cl));
    auto go = [&](auto kernel) {
        if (smem > 48 * 1024) {   // a limit for every launch, not this one's need: other threads launch it too
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)tail_smem(kTailMaxN / 4));
            if (e != cudaSuccess) return e;
        }
        return launch_chained(kernel, grid, dim3(kTailThreads), smem, chain_launch(nslots, sm_count), s, holos, slots);
    };
    switch (cl) {
    case 8: return go(tcws_tails_kernel<8>);
    case 4: return go(tcws_tails_kernel<4>);
    case 2: return go(tcws_tails_kernel<2>);
    default: return go(tcws_tails_kernel<1>);
    }
}

static cudaError_t tcws_launch(const HoloDev *holos, const LaunchSlot *slots, int nslots, int total_tiles, int maxN,
                               unsigned *queue, int grid, bool subset, int f16, int exact, int sm_count,
                               cudaStream_t s)
{
    (void)cudaGetLastError();
    // two groups of u warps where they pay (kVWarps' comment): more than one
    // spot block, or less than about 20 holograms' worth of work items (a
    // block's few tiles, where latency counts)
    const bool ug2 = tc::nspotblocks(maxN) > 1 || total_tiles < 8 * grid;
    const bool chain = chain_launch(nslots, sm_count);
    const auto one = f16     ? (ug2 ? tcws_launch_one<2, true, false> : tcws_launch_one<1, true, false>)
                     : exact ? (ug2 ? tcws_launch_one<2, false, true> : tcws_launch_one<1, false, true>)
                             : (ug2 ? tcws_launch_one<2, false, false> : tcws_launch_one<1, false, false>);
    const cudaError_t e = one(holos, slots, nslots, total_tiles, queue, grid, chain, s);
    if (e != cudaSuccess) return e;
    return launch_tc_tails(holos, slots, nslots, total_tiles, maxN, subset, sm_count, s);
}

int full_tc_tiles(int P) { return tc::tiles(P); }

int full_tc_spot_blocks(int N) { return tc::nspotblocks(N); }

// Strip length of a launch: the one that minimises an estimate of its time in
// tile times, (tiles + f items) / grid + S / 2: the work spread over the
// resident blocks, a flush per work item (epilogue 2 and the hand-over of Z,
// f = 1/2 a tile), and the tail left by the last strips (half a strip); or the
// forced length.  A hologram with more than one spot block per GEMM 2 takes
// strips of one tile.
int full_tc_assign_strips(LaunchSlot *slots, int nslots, const int *P, const int *N, int grid, int forced,
                          int *chosen)
{
    using namespace tc;
    grid = std::max(1, grid);
    auto cols = [&](int i) { return (P[i] + kCols - 1) / kCols; };
    auto rows = [&](int i) { return (P[i] + kRows - 1) / kRows; };
    auto strip_of = [&](int i, int S) { return nspotblocks(N[i]) == 1 ? std::min(S, cols(i)) : 1; };
    int smax = 1;
    for (int i = 0; i < nslots; ++i)
        if (nspotblocks(N[i]) == 1) smax = std::max(smax, cols(i));
    // The launch's finish time for strip length S, in tiles: the persistent
    // blocks take the work items in queue order, each the next free block
    // (simulated with a heap of the blocks' finish times); an item costs its
    // tiles plus a hand-over of ~0.15 tile, and 0.1 tile per unit of S stands
    // for the wider spread of holograms (and of their tables in L2) that long
    // strips keep in flight (fitted to strips of 1, 2, 3, 4, 6, 9, 12 and 18 at
    // 64 holograms of P = 1152, where 3 is fastest).
    constexpr double kItemCost = 0.15, kStripCost = 0.1;
    std::vector<double> heap;
    auto finish = [&](int S) {
        heap.assign((size_t)grid, 0.0);   // all zero: a valid min-heap
        auto take = [&](double w) {
            std::pop_heap(heap.begin(), heap.end(), std::greater<double>());
            heap.back() += w + kItemCost;
            std::push_heap(heap.begin(), heap.end(), std::greater<double>());
        };
        for (int i = 0; i < nslots; ++i) {
            const int st = strip_of(i, S), c = cols(i);
            for (int r = 0; r < rows(i); ++r)
                for (int c0 = 0; c0 < c; c0 += st) take((double)std::min(st, c - c0));
        }
        return *std::max_element(heap.begin(), heap.end());
    };
    // no launch ends before its work's share per block: lengths whose share is
    // already worse than the best time need no simulation (of a mixed launch's
    // 18 lengths, most; the simulation takes milliseconds of host time)
    auto share = [&](int S) {
        double w = 0.0;
        for (int i = 0; i < nslots; ++i) {
            const int st = strip_of(i, S), c = cols(i);
            w += rows(i) * (c + kItemCost * ((c + st - 1) / st));
        }
        return w / grid;
    };
    int best = forced > 0 ? forced : 1;
    double best_cost = 1e300;
    for (int S = 1; S <= smax && forced <= 0; ++S) {
        if (share(S) + kStripCost * S >= best_cost) continue;
        const double cost = finish(S) + kStripCost * S;
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = S;
        }
    }
    if (chosen) *chosen = best;
    int begin = 0;
    for (int i = 0; i < nslots; ++i) {
        const int st = strip_of(i, best);
        slots[i].strip = st;
        slots[i].tiles = rows(i) * ((cols(i) + st - 1) / st);
        slots[i].tile_begin = begin;
        begin += slots[i].tiles;
    }
    return begin;
}

int full_tc_max_grid(int variant, int maxN, int sm_count)
{
    return variant == kFullTcWs ? tcws_max_grid(maxN, sm_count) : 0;
}

void full_tc_table_bytes(int P, int N, size_t *rw, size_t *c, size_t *cs)
{
    *rw = tc::rw_table_bytes(P, N);
    *c = tc::c_table_bytes(P, N);
    *cs = tc::cs_table_bytes(P, N);
}

cudaError_t launch_tc_const_tables(const HoloDev *holos, int count, int sm_count, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    (void)cudaGetLastError();
    dim3 grid((unsigned)std::max(1, 2 * sm_count / std::max(1, count)), (unsigned)count);
    tc::const_tables_kernel<<<grid, 256, 0, s>>>(holos, count);
    return cudaGetLastError();
}

cudaError_t launch_tc_rw_tables(const HoloDev *holos, const LaunchSlot *slots, int nslots, int maxP, int maxN,
                                int sm_count, cudaStream_t s)
{
    if (nslots <= 0) return cudaSuccess;
    (void)cudaGetLastError();
    // at most a block of threads per table block of the largest hologram
    const int need = ((maxP + tc::kRows - 1) / tc::kRows) * tc::nchunks(maxN);
    dim3 grid((unsigned)std::max(1, std::min(need, 16 * sm_count / nslots)), (unsigned)nslots);
    return launch_chained(tc::rw_tables_kernel, grid, dim3(256), 0, chain_launch(nslots, sm_count), s, holos, slots);
}

// The shared-memory form of the mask draw for a launch whose holograms are
// at most maxP pixels a side: the CTAs per slot (a cluster: 1, 2, 4 or 8, about
// one wave over the SMs), or 0 when the mask and the round tables do not fit a
// CTA's shared memory or the launch has too few holograms for it: every CTA
// clears a whole mask, and 8 of them per hologram must still fill half the
// SMs; below that the global bit sets of mask_scatter_kernel (a few hundred
// thousand draws spread over every SM) cost less.
static int mask_local_shape(int maxP, int nslots, int sm_count, size_t *smem)
{
    if (16 * nslots < sm_count) return 0;
    int G = 8;
    while (G > 1 && G * nslots > sm_count) G >>= 1;
    // the mask, and four tables of at most maxP 16-bit entries (doubled: below 2^16)
    *smem = (((size_t)maxP * (size_t)mask_words_of(maxP) + 3) & ~(size_t)3) * 4 + 4 * 2 * (size_t)(maxP + 1);
    constexpr size_t kMaxSmem = 220 * 1024;   // the function's limit, which other threads' launches share
    if (*smem > kMaxSmem) return 0;
    if (cudaFuncSetAttribute(tc::mask_local_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return G;
}

cudaError_t launch_tc_mask_scatter(const HoloDev *holos, const LaunchSlot *slots, int nslots, int maxP, int sm_count,
                                   cudaStream_t s)
{
    if (nslots <= 0) return cudaSuccess;
    (void)cudaGetLastError();
    size_t smem = 0;
    if (const int G = mask_local_shape(maxP, nslots, sm_count, &smem)) {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)G;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)G, (unsigned)nslots);
        cfg.blockDim = dim3(tc::kLocalThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, tc::mask_local_kernel, holos, slots);
    }
    // a launch of few holograms (or holograms too large for the shared-memory
    // form): four blocks per SM over the launch, the draws' latency spread wide
    dim3 grid((unsigned)std::max(1, 4 * sm_count / std::max(1, nslots)), (unsigned)nslots);
    tc::mask_scatter_kernel<<<grid, 256, 0, s>>>(holos, slots);
    return cudaGetLastError();
}

cudaError_t launch_subset_tc(const HoloDev *holos, const LaunchSlot *slots, int nslots, int total_tiles, int maxN,
                             unsigned *queue, int grid, int f16, int exact, int sm_count, cudaStream_t s)
{
    return tcws_launch(holos, slots, nslots, total_tiles, maxN, queue, grid, true, f16, exact, sm_count, s);
}

cudaError_t launch_full_tc(int variant, const HoloDev *holos, const LaunchSlot *slots, int nslots, int total_tiles,
                           int maxN, unsigned *queue, int grid, int sm_count, cudaStream_t s)
{
    if (variant != kFullTcWs) return cudaErrorInvalidValue;
    return tcws_launch(holos, slots, nslots, total_tiles, maxN, queue, grid, false, 0, 0, sm_count, s);
}

}  // namespace cswgs
