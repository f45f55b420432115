// Double-precision CS-WGS on the GPU: the baseline solver, one hologram at a
// time.
//
// The lens-and-prism phase (Eq. 2) is separable, e^{i phi_n(x', y')} =
// C_n(x') R_n(y'), so both passes are complex multiply-adds of factors made
// once per solve, and no phasor is evaluated per pixel-spot pair:
//   prep     per spot: w = 1, theta^0 drawn from the seed (Eq. 1, random
//            superposition), W_n = w_n a_n e^{i theta_n};
//   factors  C_n(x'), R_n(y'): one sine and cosine per (spot, coordinate);
//   mask     compressed iterations: a bit per pixel of S_j;
//   pass     per grid row of the pass: u = S / |S| with S(x) = sum_n W_n
//            R_n(y) C_n(x) (Eq. 1), then V_n += conj(R_n(y)) sum_x
//            conj(C_n(x)) u(x) over the row's pixels (Eq. 3);
//   tail     w_n <- w_n <|V|>/|V_n|, theta_n <- arg V_n (Eqs. 4-6), or I_n =
//            |V_n|^2, e = sum I_n, u (Eq. 7).
// Bound by the FP64 pipe (about 2 lanes a clock and SM): 4 FP64 multiply-adds
// per pair and pass, against ~45 for a phasor of its own.  A 10-iteration
// solve at P = 512, N = 100, c = 1/8 took 15.4 ms with one sincos per pair and
// pass and takes 2.32 ms in this form.
// Phases are evaluated in FP64 with the range reduction done in turns
// (t - rint(t)) before the double-precision sincospi.
#include <cooperative_groups.h>

#include <algorithm>

#include "cswgs_device.cuh"
#include "cswgs_internal.h"

namespace cswgs {

// Threads of a row block.  A row's forward sums take G = threads / N groups of
// threads per spot; 512 leaves few of them idle at the usual spot counts
// (N = 100: 500 of 512 at work; 256 threads would leave 56 idle).
constexpr int kF64Threads = 512;
constexpr int kF64Seg = 1024;       // listed pixels of a row held in shared memory at a time
constexpr int kF64MaskSeg = 1024;   // columns listed at a time (32 mask words: one warp scan)
static_assert(kF64MaskSeg <= kF64Seg, "a column segment's pixels fit the list");
// The pass's limit of dynamic shared memory, the same at every launch: it belongs
// to the function, so a solve that set it to its own need would take it from
// another thread's solve in the middle of its launches.  (N = 4096 needs 156 KB.)
constexpr size_t kF64MaxSmem = 200 * 1024;

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

__device__ __forceinline__ double2 spot_weight(double w, double amp, double theta)
{
    double s, c;
    sincos(theta, &s, &c);
    return make_double2(w * amp * c, w * amp * s);
}

__global__ void fp64_prep(const double *init_w, const double *init_th, const double *amp, int N, uint64_t seed,
                          double *w, double *theta, double2 *weight)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    w[n] = init_w ? init_w[n] : 1.0;
    theta[n] = init_th ? init_th[n] : kTwoPi * theta0_turns(seed, n);
    weight[n] = spot_weight(w[n], amp ? amp[n] : 1.0, theta[n]);
}

// e^{i 2 pi (tilt u + g u^2)} of spot n at coordinate u = i - P / 2: C (tilt
// alpha, blockIdx.z = 0) and R (tilt beta, blockIdx.z = 1), [N][P] each.
__global__ void fp64_factors(const double *xyz, int N, int P, double2 *C, double2 *R)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = blockIdx.y;
    if (i >= P) return;
    const double half = 0.5 * (double)P, u = (double)i - half;
    const double tilt = xyz[3 * n + blockIdx.z] / (double)P, g = xyz[3 * n + 2] / (half * half);
    const double t = fma(tilt, u, g * (u * u));
    double s, c;
    sincospi(2.0 * (t - rint(t)), &s, &c);
    (blockIdx.z ? R : C)[(size_t)n * P + i] = make_double2(c, s);
}

__global__ void fp64_mask(int P, int words, int Mp, uint64_t seed, int j, uint32_t *mask)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Mp) return;
    const SubsetKeys K = subset_keys(seed, j);
    const uint32_t m = permute((uint32_t)k, (uint32_t)P, K), r = m / (uint32_t)P, c = m - r * (uint32_t)P;
    atomicOr(mask + (size_t)r * words + (c >> 5), 1u << (c & 31));
}

// u = S / |S| (1 where S = 0), with S scaled by a power of two first so that
// |S|^2 neither overflows nor underflows.
__device__ __forceinline__ double2 unit64(double2 s)
{
    const double m = fmax(fabs(s.x), fabs(s.y));
    if (!(m > 0.0)) return make_double2(1.0, 0.0);
    const int e = ilogb(m);
    const double a = scalbn(s.x, -e), b = scalbn(s.y, -e);
    const double r = rsqrt(fma(a, a, b * b));
    return make_double2(a * r, b * r);
}

// One pass over the rows y = blockIdx.x rows_per .. of the grid (every pixel, or
// the mask's), partial V_n of the block's rows to part[blockIdx.x][n].
//   back: one thread per listed pixel and slice of the spots (a sparse row
//     lists few pixels: the spots are split over the threads left, so that
//     every warp has work for the FP64 pipe), the slices summed in order;
//   forward: one thread per spot and slice of the row's pixels.
__global__ void __launch_bounds__(kF64Threads) fp64_pass(int P, int N, int rows_per, const double2 *__restrict__ C,
                                                         const double2 *__restrict__ R,
                                                         const double2 *__restrict__ weight,
                                                         const uint32_t *__restrict__ mask, int words,
                                                         float *__restrict__ phase_out, double2 *__restrict__ part)
{
    extern __shared__ double2 s_dyn[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int G = N < kF64Threads ? kF64Threads / N : 1;   // forward: threads per spot
    double2 *s_w = s_dyn;                      // [N] W_n R_n(y)
    double2 *s_v = s_w + N;                    // [G N] forward sums of the block's rows
    double2 *s_u = s_v + (size_t)G * N;        // [kF64Seg] u of the listed pixels
    double2 *s_p = s_u + kF64Seg;              // [kF64Threads] back: the slices' sums
    int *s_x = reinterpret_cast<int *>(s_p + kF64Threads);   // [kF64Seg] their columns
    __shared__ int s_cnt;
    for (int k = tid; k < G * N; k += kF64Threads) s_v[k] = make_double2(0.0, 0.0);
    const int y1 = min(P, (int)(blockIdx.x + 1) * rows_per);
    for (int y = blockIdx.x * rows_per; y < y1; ++y) {
        __syncthreads();   // the previous row is done with s_w
        for (int n = tid; n < N; n += kF64Threads) s_w[n] = cmul(weight[n], R[(size_t)n * P + y]);
        for (int x0 = 0; x0 < P; x0 += kF64MaskSeg) {
            // the segment's pixels, in column order
            if (tid < 32) {
                if (mask) {
                    const int wd = (x0 >> 5) + lane;
                    uint32_t bits = wd < words ? mask[(size_t)y * words + wd] : 0u;
                    int at = __popc(bits);
                    for (int o = 1; o < 32; o <<= 1) {
                        const int t = __shfl_up_sync(0xffffffffu, at, o);
                        if (lane >= o) at += t;
                    }
                    if (lane == 31) s_cnt = at;
                    at -= __popc(bits);
                    for (; bits; bits &= bits - 1) s_x[at++] = 32 * wd + __ffs(bits) - 1;
                } else {
                    if (lane == 0) s_cnt = min(kF64MaskSeg, P - x0);
                }
            }
            if (!mask)
                for (int i = tid; i < min(kF64MaskSeg, P - x0); i += kF64Threads) s_x[i] = x0 + i;
            __syncthreads();
            const int cnt = s_cnt;
            const int pix = min(kF64Threads, ((cnt + 31) / 32) * 32);   // back: pixels per round, whole warps
            const int H = pix > 0 ? kF64Threads / pix : 1;             // slices of the spots
            for (int i0 = 0; i0 < cnt; i0 += pix) {
                const int h = tid / pix, i = i0 + tid % pix;
                double2 s = make_double2(0.0, 0.0);
                if (h < H && i < cnt) {
                    const double2 *c = C + s_x[i];
#pragma unroll 4
                    for (int n = h; n < N; n += H) {
                        const double2 a = s_w[n], b = __ldg(c + (size_t)n * P);
                        s.x = fma(a.x, b.x, fma(-a.y, b.y, s.x));
                        s.y = fma(a.x, b.y, fma(a.y, b.x, s.y));
                    }
                }
                if (H > 1) {
                    s_p[tid] = s;
                    __syncthreads();
                    if (h == 0 && i < cnt)
                        for (int q = 1; q < H; ++q) {
                            s.x += s_p[q * pix + tid].x;
                            s.y += s_p[q * pix + tid].y;
                        }
                }
                if (h == 0 && i < cnt) {
                    s_u[i] = unit64(s);
                    if (phase_out) {
                        double ph = atan2(s.y, s.x);
                        if (ph < 0.0) ph += kTwoPi;
                        const float o = (float)ph;
                        phase_out[(size_t)y * P + s_x[i]] = o >= kTwoPiF ? 0.f : o;
                    }
                }
                __syncthreads();   // u is in place, and s_p read
            }
            for (int k = tid; k < G * N; k += kF64Threads) {
                const int n = k % N, g = k / N;
                const double2 *c = C + (size_t)n * P;
                double2 z = make_double2(0.0, 0.0);
#pragma unroll 4
                for (int i = g; i < cnt; i += G) {
                    const double2 u = s_u[i], b = __ldg(c + s_x[i]);   // conj(C) u
                    z.x = fma(b.x, u.x, fma(b.y, u.y, z.x));
                    z.y = fma(b.x, u.y, fma(-b.y, u.x, z.y));
                }
                const double2 r = R[(size_t)n * P + y];
                double2 v = s_v[k];
                v.x = fma(r.x, z.x, fma(r.y, z.y, v.x));
                v.y = fma(r.x, z.y, fma(-r.y, z.x, v.y));
                s_v[k] = v;
            }
            __syncthreads();   // the list and u are read
        }
    }
    __syncthreads();
    for (int n = tid; n < N; n += kF64Threads) {
        double2 v = s_v[n];
        for (int g = 1; g < G; ++g) {
            v.x += s_v[g * N + n].x;
            v.y += s_v[g * N + n].y;
        }
        part[(size_t)blockIdx.x * N + n] = v;
    }
}

// V_n = (1 / count) sum of the items' partials, then the update or the
// metrics, by one cluster of 8 blocks (the items' sums are FP64 additions,
// which 8 SMs' pipes take 8 times as fast as one's).  Spots are dealt out to
// the blocks in fours: lanes are 4 spots x 8 groups of items, and where a block
// has warps to spare 2 to 16 of them share four spots (one warp each took 23 us
// a pass at N = 100, 512 items, waiting for 16 loads one after another).
constexpr int kF64Cluster = 8;
constexpr int kF64TailThreads = 512;

__global__ void __cluster_dims__(kF64Cluster, 1, 1) __launch_bounds__(kF64TailThreads)
fp64_tail(int N, int items, int64_t count, const double2 *__restrict__ part, const double *__restrict__ amp,
          double *w, double *theta, double2 *weight, double *metrics, int final_pass)
{
    constexpr int W = kF64TailThreads / 32;
    __shared__ double s_red[3][W];
    __shared__ double s_out[3];
    extern __shared__ double2 s_field[];   // this block's spots: V_n, four by four; then the warps' sums
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int quads = (N + 3) / 4, nq = (quads - rank + kF64Cluster - 1) / kF64Cluster;
    int wq = W;   // warps per four spots: a power of two
    while (wq > 1 && wq * nq > W) wq >>= 1;
    double2 *s_sum = s_field + 4 * nq;   // [nq wq][4]
    for (int i = warp / wq; i < nq; i += W / wq) {
        const int n = 4 * (rank + kF64Cluster * i) + (lane & 3);
        double vr = 0.0, vi = 0.0;
        if (n < N) {
#pragma unroll 8
            for (int t = (lane >> 2) + 8 * (warp % wq); t < items; t += 8 * wq) {
                const double2 p = part[(size_t)t * N + n];
                vr += p.x;
                vi += p.y;
            }
        }
        for (int o = 4; o < 32; o <<= 1) {
            vr += __shfl_xor_sync(0xffffffffu, vr, o);
            vi += __shfl_xor_sync(0xffffffffu, vi, o);
        }
        if (lane < 4) s_sum[(i * wq + warp % wq) * 4 + lane] = make_double2(vr, vi);
    }
    __syncthreads();
    double sum = 0.0, imax = -1.0, imin = 1e300;
    for (int k = tid; k < 4 * nq; k += kF64TailThreads) {   // a thread per spot
        const int n = 4 * (rank + kF64Cluster * (k >> 2)) + (k & 3);
        if (n >= N) continue;
        double vr = 0.0, vi = 0.0;
        for (int g = 0; g < wq; ++g) {
            const double2 p = s_sum[((k >> 2) * wq + g) * 4 + (k & 3)];
            vr += p.x;
            vi += p.y;
        }
        vr /= (double)count;
        vi /= (double)count;
        s_field[k] = make_double2(vr, vi);
        if (final_pass) {
            const double in = vr * vr + vi * vi;
            metrics[2 + n] = in;
            sum += in;
            imax = fmax(imax, in);
            imin = fmin(imin, in);
        } else {
            sum += hypot(vr, vi);
        }
    }
    if (32 * warp < 4 * nq)   // the other warps hold no spot
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
            imax = fmax(imax, __shfl_xor_sync(0xffffffffu, imax, o));
            imin = fmin(imin, __shfl_xor_sync(0xffffffffu, imin, o));
        }
    if (lane == 0) {
        s_red[0][warp] = sum;
        s_red[1][warp] = imax;
        s_red[2][warp] = imin;
    }
    __syncthreads();
    if (tid == 0) {
        for (int q = 1; q < W && 32 * q < 4 * nq; ++q) {
            sum += s_red[0][q];
            imax = fmax(imax, s_red[1][q]);
            imin = fmin(imin, s_red[2][q]);
        }
        s_out[0] = sum;
        s_out[1] = imax;
        s_out[2] = imin;
    }
    cluster.sync();
    double total = 0.0;
    if (final_pass ? rank == 0 && tid == 0 : tid < 4 * nq) {
        for (int r = 0; r < kF64Cluster; ++r) {
            const double *o = cluster.map_shared_rank(s_out, r);
            total += o[0];
            imax = fmax(imax, o[1]);
            imin = fmin(imin, o[2]);
        }
    }
    if (final_pass) {
        if (rank == 0 && tid == 0) {
            metrics[0] = total;
            metrics[1] = (imax + imin) > 0.0 ? 1.0 - (imax - imin) / (imax + imin) : 0.0;
        }
    } else {
        const double mean = total / (double)N;
        for (int k = tid; k < 4 * nq; k += kF64TailThreads) {
            const int n = 4 * (rank + kF64Cluster * (k >> 2)) + (k & 3);
            if (n >= N) continue;
            const double2 v = s_field[k];
            const double mag = hypot(v.x, v.y);
            w[n] = w[n] * mean / (mag > 1e-30 ? mag : 1e-30);
            if (mag > 0.0) theta[n] = atan2(v.y, v.x);
            weight[n] = spot_weight(w[n], amp ? amp[n] : 1.0, theta[n]);
        }
    }
    cluster.sync();   // s_out is read before any block leaves
}

static unsigned blocks_for(int64_t n, int threads)
{
    return (unsigned)((n + threads - 1) / threads);
}

// Rows per block of a pass: four blocks per SM are resident (their phases
// overlap), so a grid of more rows than that gives each block several and
// the tails fewer partials to sum.
int fp64_rows_per(int P, int sm_count) { return std::max(1, (P + 4 * sm_count - 1) / (4 * std::max(1, sm_count))); }

int fp64_items(int P, int sm_count)
{
    const int r = fp64_rows_per(P, sm_count);
    return (P + r - 1) / r;
}

cudaError_t fp64_solve(const Fp64Work &wk, int P, int N, int Mp, int iterations, int n_full,
                       int first_j, uint64_t seed, int final_pass, float *phase_out, int sm_count, cudaStream_t s)
{
    const int64_t M = (int64_t)P * P;
    const int words = (P + 31) / 32, rows_per = fp64_rows_per(P, sm_count), items = fp64_items(P, sm_count);
    (void)cudaGetLastError();   // report these launches, not an earlier call's error
    fp64_prep<<<blocks_for(N, 128), 128, 0, s>>>(wk.init_w, wk.init_th, wk.amp, N, seed, wk.w, wk.theta, wk.weight);
    fp64_factors<<<dim3(blocks_for(P, 128), (unsigned)N, 2), 128, 0, s>>>(wk.xyz, N, P, wk.C, wk.R);
    const int G = N < kF64Threads ? kF64Threads / N : 1;
    const size_t smem = sizeof(double2) * ((size_t)N + (size_t)G * N + kF64Seg + kF64Threads) + sizeof(int) * kF64Seg;
    // V_n of a block's fours, and the warps' sums (at least W entries of four, or one per four)
    const size_t nq = (size_t)((N + 31) / 32);
    const size_t tail_smem = sizeof(double2) * 4 * (nq + std::max<size_t>(nq, kF64TailThreads / 32));
    if (smem > kF64MaxSmem) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fp64_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF64MaxSmem);
    if (e != cudaSuccess) return e;
    auto tail = [&](int64_t count, int fin) {
        fp64_tail<<<kF64Cluster, kF64TailThreads, tail_smem, s>>>(N, items, count, wk.part, wk.amp, wk.w, wk.theta,
                                                                  wk.weight, wk.metrics, fin);
    };
    for (int it = 0; it < iterations; ++it) {
        const bool full = it >= iterations - n_full;
        if (!full) {
            e = cudaMemsetAsync(wk.mask, 0, sizeof(uint32_t) * (size_t)P * words, s);
            if (e != cudaSuccess) return e;
            fp64_mask<<<blocks_for(Mp, 256), 256, 0, s>>>(P, words, Mp, seed, first_j + it, wk.mask);
        }
        fp64_pass<<<items, kF64Threads, smem, s>>>(P, N, rows_per, wk.C, wk.R, wk.weight, full ? nullptr : wk.mask,
                                                   words, nullptr, wk.part);
        tail(full ? M : (int64_t)Mp, 0);
    }
    if (final_pass) {
        fp64_pass<<<items, kF64Threads, smem, s>>>(P, N, rows_per, wk.C, wk.R, wk.weight, nullptr, words, phase_out,
                                                   wk.part);
        tail(M, 1);
    }
    return cudaGetLastError();
}

}  // namespace cswgs
