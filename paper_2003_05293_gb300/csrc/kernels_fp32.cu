// FP32 CS-WGS kernels for sm_103a.
//
// One fused, persistent kernel runs one iteration (or the final pass) for
// every hologram of a launch.  A work item is a tile of THREADS * PPT pixels
// of one hologram; blocks take items from a queue.  Per tile:
//   back-propagation (Eq. 1) of the N spot fields at each pixel, with the
//   lens-and-prism phase (Eq. 2) generated on the fly in 32-bit fixed point
//   (exact range reduction) and FP32 sine/cosine;
//   Phi_m = arg of the sum, kept as a fixed-point turn;
//   forward projection (Eq. 3) of e^{i Phi_m} onto every spot, reduced over
//   the tile by warp shuffles and a shared-memory tree into one partial
//   field per spot (FP32 for iterations, FP64 for the metrics pass);
//   the last tile of a hologram (arrival counter) sums the partials and
//   applies the weighted update of Eqs. 4-6, or computes e and u (Eq. 7).
// The pixel set of a compressed iteration is the image of [0, Mp) under the
// keyed permutation of the iteration (Section 2, CS-WGS; Section 3,
// "Compressed sensing"), computed in registers: no index array.
#include "tile.cuh"

namespace cswgs {

// The persistent loop both iteration kernels share: blocks take work items
// (tiles) from the launch's queue until it is empty; the last block out resets
// the queue for the next launch on the stream.
template <class TileFn>
__device__ __forceinline__ void persistent_tiles(const HoloDev *__restrict__ holos,
                                                 const LaunchSlot *__restrict__ slots, int nslots,
                                                 int total_tiles, unsigned *queue, TileFn tile)
{
    __shared__ int s_item, s_slot;
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) {
            int item = (int)atomicAdd(queue, 1u);
            s_item = item;
            if (item < total_tiles) {
                int lo = 0, hi = nslots - 1;
                while (lo < hi) {
                    int mid = (lo + hi + 1) >> 1;
                    if (slots[mid].tile_begin <= item) lo = mid;
                    else hi = mid - 1;
                }
                s_slot = lo;
            }
        }
        __syncthreads();
        const int item = s_item;
        if (item >= total_tiles) break;
        const LaunchSlot sl = slots[s_slot];
        const HoloDev H = holos[sl.holo];
        tile(H, sl, item - sl.tile_begin);   // ends with __syncthreads()
    }
    if (tid == 0) {
        unsigned done = atomicAdd(queue + 1, 1u);
        if (done == gridDim.x - 1) {
            queue[0] = 0u;
            queue[1] = 0u;
            __threadfence();
        }
    }
}

// Minimum resident blocks per SM each register budget must allow (without a
// minimum, ptxas settles on 64 registers and spills): 32 warps per SM for
// compressed tiles of up to 4 pixels per thread, 24 warps otherwise.
template <int THREADS, int PPT>
constexpr int subset_min_blocks() { return (PPT <= 4 ? 1024 : 768) / THREADS; }
template <int THREADS>
constexpr int full_min_blocks() { return 768 / THREADS > 0 ? 768 / THREADS : 1; }

// Compressed iterations: tiles of THREADS * PPT pixels of the subsets S_j.
template <int THREADS, int PPT>
__global__ void __launch_bounds__(THREADS, (subset_min_blocks<THREADS, PPT>()))
iter_subset_kernel(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots, int nslots,
                   int total_tiles, int maxN, unsigned *queue)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_red[THREADS / 32];
    __shared__ int s_last;
    // the next iteration's blocks only once this one's work begins: started before
    // the wait, the blocks of eight iterations to come filled the SMs and left each
    // iteration's where room happened to be, several on one SM (30 iterations of
    // the paper's optics on this kernel, 512 threads x 4 pixels, 944 us; 769 so)
    chain_wait();
    chain_start();
    persistent_tiles(holos, slots, nslots, total_tiles, queue, [&](const HoloDev &H, const LaunchSlot &sl, int t) {
        process_tile<THREADS, PPT>(H, sl, t, maxN, smem, s_red, &s_last);
    });
}

// Compressed iterations with the half-precision sincos option.
template <int THREADS, int PPT>
__global__ void __launch_bounds__(THREADS, (subset_min_blocks<THREADS, PPT>()))
iter_subset_h2_kernel(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots, int nslots,
                      int total_tiles, int maxN, unsigned *queue)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_red[THREADS / 32];
    __shared__ int s_last;
    persistent_tiles(holos, slots, nslots, total_tiles, queue, [&](const HoloDev &H, const LaunchSlot &sl, int t) {
        process_tile_h2<THREADS, PPT>(H, sl, t, maxN, smem, s_red, &s_last);
    });
}

// Full iterations and the final pass: separable tiles of THREADS / 4 rows x 64 columns.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, (full_min_blocks<THREADS>()))
iter_full_kernel(const HoloDev *__restrict__ holos, const LaunchSlot *__restrict__ slots, int nslots,
                 int total_tiles, int maxN, unsigned *queue)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_red[THREADS / 32];
    __shared__ int s_last;
    persistent_tiles(holos, slots, nslots, total_tiles, queue, [&](const HoloDev &H, const LaunchSlot &sl, int t) {
        process_full_tile<THREADS>(H, sl, t, maxN, smem, s_red, &s_last);
    });
}

// Spot preparation (step 1 of the path): fixed-point coefficients of Eq. 2,
// theta^0 drawn from the seed (or the caller's start state), w = 1.
__global__ void prep_kernel(const HoloDev *__restrict__ holos)
{
    const HoloDev H = holos[blockIdx.y];
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < H.N; n += gridDim.x * blockDim.x) {
        prep_spot(H, n);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *H.counter = 0u;
}

__global__ void subset_kernel(int P, int64_t Mp, uint64_t seed, int j, int32_t *out)
{
    const SubsetKeys K = subset_keys(seed, j);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < Mp;
         k += (int64_t)gridDim.x * blockDim.x)
        out[k] = (int32_t)permute((uint32_t)k, (uint32_t)P, K);
}

// S_j under a pupil and subset reading: the solver's own pixel mapping.
__global__ void subset_ex_kernel(HoloDev H, int j, int32_t *out)
{
    const SubsetDraw d = subset_draw(H, j);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < H.Mp;
         k += (int64_t)gridDim.x * blockDim.x)
        out[k] = (int32_t)subset_pixel(H, d, (uint32_t)k);
}

// Throughput probe: eight independent sine/cosine chains per thread.
__global__ void sincos_probe_kernel(float *sink, long long *cycles, int iters)
{
    float a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = 0.1f * (float)(threadIdx.x + q);
    long long t0 = clock64();
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = __sinf(a[q]) + __cosf(a[q]);
    }
    long long t1 = clock64();
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc += a[q];
    if (acc == 12345.678f) sink[0] = acc;   // keeps the chains alive
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long *>(cycles),
                                    (unsigned long long)(t1 - t0));
}

// ------------------------------------------------------------- launchers --

#define CSWGS_SUBSET_SHAPES(X) \
    X(128, 2) X(128, 4) X(128, 8) X(256, 2) X(256, 4) X(256, 8) X(512, 1) X(512, 2) X(512, 4)
#define CSWGS_SUBSET_H2_SHAPES(X) \
    X(128, 2) X(128, 4) X(128, 8) X(256, 2) X(256, 4) X(256, 8) X(512, 2) X(512, 4)
#define CSWGS_FULL_SHAPES(X) X(128) X(256) X(512)

size_t iter_fp32_smem(TileShape shape, int kind, int maxN)
{
    return kind == kLaunchSubset ? tile_smem_bytes(shape.threads, maxN, false)
                                 : tile_smem_bytes(shape.full_threads, maxN, true);
}

bool tile_shape_supported(TileShape shape)
{
    bool sub = false, full = false;
    if (shape.fp16) {
#define X(T, K) sub |= shape.threads == T && shape.ppt == K;
        CSWGS_SUBSET_H2_SHAPES(X)
#undef X
    } else {
#define X(T, K) sub |= shape.threads == T && shape.ppt == K;
        CSWGS_SUBSET_SHAPES(X)
#undef X
    }
#define X(T) full |= shape.full_threads == T;
    CSWGS_FULL_SHAPES(X)
#undef X
    return sub && full;
}

// Dynamic shared memory the iteration kernels are allowed: enough for
// N = 4096 spots with any supported tile shape.
constexpr int kMaxDynSmem = 200 * 1024;

template <class K>
static int max_grid_of(K kernel, int threads, size_t smem, int sm_count)
{
    if (smem > (size_t)kMaxDynSmem) return 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem) != cudaSuccess)
        return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess) return 0;
    return per_sm * sm_count;
}

int iter_fp32_max_grid(TileShape shape, int kind, int maxN, int sm_count)
{
    const size_t smem = iter_fp32_smem(shape, kind, maxN);
    if (kind == kLaunchSubset && shape.fp16) {
#define X(T, K) if (shape.threads == T && shape.ppt == K) return max_grid_of(iter_subset_h2_kernel<T, K>, T, smem, sm_count);
        CSWGS_SUBSET_H2_SHAPES(X)
#undef X
    } else if (kind == kLaunchSubset) {
#define X(T, K) if (shape.threads == T && shape.ppt == K) return max_grid_of(iter_subset_kernel<T, K>, T, smem, sm_count);
        CSWGS_SUBSET_SHAPES(X)
#undef X
    } else {
#define X(T) if (shape.full_threads == T) return max_grid_of(iter_full_kernel<T>, T, smem, sm_count);
        CSWGS_FULL_SHAPES(X)
#undef X
    }
    return 0;
}

cudaError_t launch_iter_fp32(TileShape shape, int kind, const HoloDev *holos, const LaunchSlot *slots,
                             int nslots, int total_tiles, int maxN, unsigned *queue, int grid,
                             int sm_count, cudaStream_t s)
{
    // the smem attribute is set by iter_fp32_max_grid, which every batch calls first
    const size_t smem = iter_fp32_smem(shape, kind, maxN);
    (void)cudaGetLastError();   // report this launch, not an earlier call's error
    if (kind == kLaunchSubset && shape.fp16) {
#define X(T, K) if (shape.threads == T && shape.ppt == K) { \
            iter_subset_h2_kernel<T, K><<<grid, T, smem, s>>>(holos, slots, nslots, total_tiles, maxN, queue); \
            return cudaGetLastError(); }
        CSWGS_SUBSET_H2_SHAPES(X)
#undef X
    } else if (kind == kLaunchSubset) {
#define X(T, K) if (shape.threads == T && shape.ppt == K) { \
            return launch_chained(iter_subset_kernel<T, K>, dim3(grid), dim3(T), smem, chain_launch(nslots, sm_count), s, \
                                  holos, slots, nslots, total_tiles, maxN, queue); }
        CSWGS_SUBSET_SHAPES(X)
#undef X
    } else {
#define X(T) if (shape.full_threads == T) { \
            iter_full_kernel<T><<<grid, T, smem, s>>>(holos, slots, nslots, total_tiles, maxN, queue); \
            return cudaGetLastError(); }
        CSWGS_FULL_SHAPES(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_prep_fp32(const HoloDev *holos, int count, int maxN, cudaStream_t s)
{
    dim3 grid((unsigned)((maxN + 127) / 128), (unsigned)count);
    (void)cudaGetLastError();
    prep_kernel<<<grid, 128, 0, s>>>(holos);
    return cudaGetLastError();
}

cudaError_t launch_subset_kernel(int P, int64_t Mp, uint64_t seed, int j, int32_t *out, cudaStream_t s)
{
    int64_t blocks = (Mp + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    if (blocks < 1) blocks = 1;
    (void)cudaGetLastError();
    subset_kernel<<<(unsigned)blocks, 256, 0, s>>>(P, Mp, seed, j, out);
    return cudaGetLastError();
}

cudaError_t launch_subset_ex_kernel(const HoloDev &H, int j, int32_t *out, cudaStream_t s)
{
    int64_t blocks = ((int64_t)H.Mp + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    if (blocks < 1) blocks = 1;
    (void)cudaGetLastError();
    subset_ex_kernel<<<(unsigned)blocks, 256, 0, s>>>(H, j, out);
    return cudaGetLastError();
}

cudaError_t launch_sincos_probe(float *sink, long long *cycles, int iters, int blocks, int threads,
                                cudaStream_t s)
{
    (void)cudaGetLastError();
    sincos_probe_kernel<<<blocks, threads, 0, s>>>(sink, cycles, iters);
    return cudaGetLastError();
}

}  // namespace cswgs
