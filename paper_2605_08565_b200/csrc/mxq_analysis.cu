// Analysis kernels around the quantizer (Results, numerical study; Appendix: clipping-only MSE,
// entry and scale histograms): the clipping part of the block SSE, histograms of the FP4 codes and
// of the scale codes, and the MSE of equal-length segments of a tensor (one sigma of the
// numerical study per segment).  None of them is on the bandwidth-critical path; they are written
// for exactness and determinism first.
#include <atomic>
#include <type_traits>

#include "mxq_device.cuh"
#include "mxq_internal.h"

namespace mxq {

// ------------------------------------------------------------------------------------------------
// Clipping part of the block SSE: elements with |fl32(v / D)| > 6 are all mapped to +-6; their
// error is accumulated exactly like the block SSE (e = fma(-q, D, v); s = fma(e, e, s), element
// order), the other elements are skipped.  A zero decode scale clips nothing.  One thread per block,
// two blocks in flight for the short ones.
//
// No division for decode scales within [2^-100, 2^100]: floats are 2^-21 apart above 6, and half way to the next one a tie
// rounds to 6, so fl32(v / D) > 6  <=>  v / D > 6 + 2^-22  <=>  |v| - 6 D > 2^-22 D.  The difference is formed by one FMA: near
// the limit it is a multiple of 2^(e - 22) below 2^(e - 20), D in [2^e, 2^(e+1)), and therefore exact, as is 2^-22 D; away
// from the limit its rounding cannot change the outcome.  It is also the residual.  Bound by the reads of x: fp32,
// B = 8, from memory, 16.8 M elements (77 MB) 16.8 -> 13.2 us against a division per element and one block at a time; 60.4 M 45 us.  The
// last block of a thread goes alone: a second load that is not needed (the tensor's last block, for every thread of a small
// tensor) cost bf16, B = 2 1.05 -> 1.28 us at 4096 elements.
// ------------------------------------------------------------------------------------------------
template <int B>
__device__ __forceinline__ float clip_sse(const float (&v)[B], int c, int fmt, float gs) {
    if (c >= num_codes(fmt)) return __uint_as_float(0x7FC00000u);   // not a code of the format
    const float D = __fmul_rn(scale_value(fmt, c), gs);
    float s = 0.0f;
    if (D >= 7.888609052210118e-31f && D <= 1.2676506002282294e30f) {   // 2^-100, 2^100
        const float limit = __fmul_rn(D, 2.384185791015625e-07f);       // 2^-22
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float e = __fmaf_rn(-6.0f, D, fabsf(v[i]));
            if (e > limit) s = __fmaf_rn(e, e, s);
        }
    } else if (D != 0.0f) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float t = __fdiv_rn(v[i], D);
            if (fabsf(t) > 6.0f) {
                const float q = copysignf(6.0f, v[i]);
                const float e = __fmaf_rn(-q, D, v[i]);
                s = __fmaf_rn(e, e, s);
            }
        }
    }
    return s;
}

template <int DT, int B>
__global__ void __launch_bounds__(kThreads) k_block_clip_sse(const void* x, size_t n_blocks, int fmt, float g,
                                                             const float* d_g, const uint8_t* scales, float* out) {
    wait_for_prior_grid();
    release_dependents();
    const float gs = d_g ? *d_g : g;
    const size_t stride = (size_t)gridDim.x * kThreads;
    // From the end of the tensor to its beginning: the pass that quantized it has left the end of it in L2 (scoring of 60.4 M fp32 elements,
    // B = 8, quantization included: 129.2 -> 127.0 us).  Blocks of 2 and 4 forwards: the backward indices take them past 32 registers, eight resident
    // CTAs to six (67 M bf16 elements, B = 4, us: backwards 58.4, forwards 44.0; 16.8 M fp32, B = 4, 23 % apart).
    const size_t last = n_blocks - 1;
    auto at = [last](size_t i) {
        if constexpr (B <= 4) return i;
        else return last - i;
    };
    auto do_blocks = [&](auto count, size_t b) {   // blocks at(b), at(b + stride), ...: all loads first
        constexpr int U = decltype(count)::value;
        float v[U][B];
        int c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            load_elems<DT, B>(x, at(b + u * stride) * B, v[u]);      // vector loads: a block is 4 .. 256 contiguous bytes
            c[u] = scales[at(b + u * stride)];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) out[at(b + u * stride)] = clip_sse<B>(v[u], c[u], fmt, gs);
    };
    size_t b = (size_t)blockIdx.x * kThreads + threadIdx.x;
    if constexpr (B <= 16) {
        for (; b + stride < n_blocks; b += 2 * stride) do_blocks(std::integral_constant<int, 2>{}, b);
    }
    for (; b < n_blocks; b += stride) do_blocks(std::integral_constant<int, 1>{}, b);
}

template <int DT>
static cudaError_t launch_clip_dt(const void* x, size_t n_blocks, int B, int fmt, float g, const float* d_g,
                                  const uint8_t* scales, float* out, unsigned grid, cudaStream_t s) {
    switch (B) {
    case 2: return launch_pdl(k_block_clip_sse<DT, 2>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    case 4: return launch_pdl(k_block_clip_sse<DT, 4>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    case 8: return launch_pdl(k_block_clip_sse<DT, 8>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    case 16: return launch_pdl(k_block_clip_sse<DT, 16>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    case 32: return launch_pdl(k_block_clip_sse<DT, 32>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    default: return launch_pdl(k_block_clip_sse<DT, 64>, grid, kThreads, 0, s, x, n_blocks, fmt, g, d_g, scales, out);
    }
}

cudaError_t launch_block_clip_sse(const void* x, int dtype, size_t n, int B, int fmt, float g, const float* d_g,
                                  const uint8_t* scales, float* out, cudaStream_t s) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const size_t n_blocks = n / (size_t)B;
    size_t want = (n_blocks + kThreads - 1) / kThreads;
    const size_t cap = (size_t)sm_count(dev) * 8;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    err = (dtype == kF32) ? launch_clip_dt<kF32>(x, n_blocks, B, fmt, g, d_g, scales, out, grid, s)
                          : launch_clip_dt<kBF16>(x, n_blocks, B, fmt, g, d_g, scales, out, grid, s);
    count_launch();
    return err;
}

// ------------------------------------------------------------------------------------------------
// Histograms: 16 bins of the 4-bit codes, 256 bins of the scale codes, ADDED to the caller's
// 64-bit counters.  The pass is a byte histogram: a code byte holds two codes, so the kernel counts
// the 256 byte values (one shared-memory integer atomic per TWO codes) and folds them into the 16 code
// bins at the end; scale bytes are counted the same way.  A table holds every byte value 32 times, once
// per lane and bank, so that no two lanes of a warp meet at an address or in a bank (one table per warp
// with all lanes in it: three to five lanes a bank, and every repeated value the same address).  16-byte loads, no per-code
// compares.  Per-CTA counts are 32-bit (a CTA sees far fewer than 2^32 bytes), flushed with 64-bit integer atomics --
// integer sums are order-free, so the result is deterministic.  60.4 M codes and 7.5 M scales 29 -> 23 us with the launch; bound by the
// latency of the one load that a thread has in flight in front of sixteen atomics, then by the atomics (LSU pipe 46 %).
// ------------------------------------------------------------------------------------------------
constexpr int kHistThreads = 512;
constexpr size_t kHistBytes = 2 * 256 * 32 * sizeof(unsigned int);

__device__ __forceinline__ void count_bytes_of_word(unsigned int* lane_tab, uint32_t w) {
    atomicAdd(lane_tab + 32 * (w & 0xFFu), 1u);
    atomicAdd(lane_tab + 32 * ((w >> 8) & 0xFFu), 1u);
    atomicAdd(lane_tab + 32 * ((w >> 16) & 0xFFu), 1u);
    atomicAdd(lane_tab + 32 * (w >> 24), 1u);
}

// Adds the byte histogram of p[0 .. n_bytes) to the lane's column of a table: bytes up to the first 16-byte
// boundary and past the last one singly (by the first threads of the grid), the rest as 16-byte loads.
__device__ __forceinline__ void count_byte_range(unsigned int* lane_tab, const uint8_t* p, size_t n_bytes, size_t tid, size_t stride) {
    size_t head = (16u - (size_t)(reinterpret_cast<uintptr_t>(p) & 15u)) & 15u;
    if (head > n_bytes) head = n_bytes;
    const size_t n_vec = (n_bytes - head) / 16;
    const size_t tail0 = head + n_vec * 16;
    const uint4* v = reinterpret_cast<const uint4*>(p + head);
    for (size_t i = tid; i < n_vec; i += stride) {
        const uint4 w = __ldcs(v + i);
        count_bytes_of_word(lane_tab, w.x);
        count_bytes_of_word(lane_tab, w.y);
        count_bytes_of_word(lane_tab, w.z);
        count_bytes_of_word(lane_tab, w.w);
    }
    if (tid < head) atomicAdd(lane_tab + 32 * p[tid], 1u);
    if (tid < n_bytes - tail0) atomicAdd(lane_tab + 32 * p[tail0 + tid], 1u);
}

__global__ void __launch_bounds__(kHistThreads) k_histograms(const uint8_t* codes, const uint8_t* scales, size_t n, size_t n_blocks,
                                                             unsigned long long* code_hist, unsigned long long* scale_hist) {
    extern __shared__ uint4 hist_dyn[];
    unsigned int* const tab = reinterpret_cast<unsigned int*>(hist_dyn);   // [code bytes, scale bytes][value][lane]
    __shared__ unsigned long long sh_code[16];
    for (int i = threadIdx.x; i < (int)(kHistBytes / 16); i += kHistThreads) hist_dyn[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < 16) sh_code[threadIdx.x] = 0;
    __syncthreads();
    wait_for_prior_grid();
    release_dependents();
    const size_t stride = (size_t)gridDim.x * kHistThreads;
    const size_t tid = (size_t)blockIdx.x * kHistThreads + threadIdx.x;
    const int lane = threadIdx.x & 31;
    count_byte_range(tab + lane, codes, n / 2, tid, stride);
    count_byte_range(tab + 256 * 32 + lane, scales, n_blocks, tid, stride);
    __syncthreads();
    // thread t owns byte value t % 256 of one table; columns are read starting at the thread's own lane: one per bank
    unsigned long long sum = 0;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) sum += tab[threadIdx.x * 32 + ((j + lane) & 31)];
    const int value = threadIdx.x & 255;
    if (sum) {
        if (threadIdx.x < 256) {
            atomicAdd(&sh_code[value & 15], sum);    // element 2j sits in the low nibble
            atomicAdd(&sh_code[value >> 4], sum);
        } else {
            atomicAdd(&scale_hist[value], sum);
        }
    }
    __syncthreads();
    if (threadIdx.x < 16 && sh_code[threadIdx.x]) atomicAdd(&code_hist[threadIdx.x], sh_code[threadIdx.x]);
}

cudaError_t launch_histograms(const uint8_t* codes, const uint8_t* scales, size_t n, int B, unsigned long long* code_hist,
                              unsigned long long* scale_hist, cudaStream_t s) {
    static_assert(kHistThreads == 512, "one thread per byte value and table in the fold");
    static std::atomic<int> cache[kMaxDevices];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    size_t resident = 0;
    err = resident_ctas(reinterpret_cast<const void*>(k_histograms), kHistBytes, dev, cache, resident, kHistThreads);
    if (err != cudaSuccess) return err;
    size_t want = (n / 32 + kHistThreads - 1) / kHistThreads;     // 32 codes per 16-byte load
    if (want == 0) want = 1;
    // a CTA must stay below 2^32 counts per table entry: n / 2 / grid bytes each -- true for any n < 2^40 here
    // Clearing and folding the tables costs a CTA 2 us, and three on one SM six: up to 24 loads per thread (29 MB) one CTA per SM is the
    // faster (4.2 M codes, B = 2, 256 CTAs 7.5 us, 148 5.1; 16.8 M 9.6, 8.1; 33.6 M 12.8, 13.6; 60.4 M 18.4, 22.4).
    const size_t sms = (size_t)sm_count(dev);
    const bool one_per_sm = n / 2 + n / (size_t)B <= sms * kHistThreads * 16 * 24;
    const size_t cap = one_per_sm ? sms : sms * resident;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    err = launch_pdl(k_histograms, grid, (unsigned)kHistThreads, kHistBytes, s, codes, scales, n, n / (size_t)B, code_hist, scale_hist);
    count_launch();
    return err;
}

// ------------------------------------------------------------------------------------------------
// Segment MSE: out[s] = (sum of the block SSEs of segment s) / elems_per_segment.  One CTA per segment (grid-stride over
// segments), binary64 sums whose shape depends on the length of the segment alone: L lanes (256 below 4096 blocks, 512 below 8192, else 1024),
// lane i adds elements i, i + L, ..., four at a time as (a + b) + (c + d) with zeros past the end, then a shuffle tree over 32
// lanes and one over their sums.  The same values give the same bits wherever the segment lies and however many threads share the
// lanes.  Single floats are read, not vectors of four: a warp's reads are whole lines at any alignment.  What a segment needs is
// loads in flight, sixteen a thread (with full occupancy at 32 registers).
// ------------------------------------------------------------------------------------------------
template <int T, int L>
__global__ void __launch_bounds__(T, 2048 / T) k_segment_mse(const float* sse, size_t n_segments, size_t blocks_per_segment,
                                                             double elems_per_segment, double* out) {
    constexpr int A = L / T;             // lanes per thread: t, t + T, ...
    static_assert(A == 1 || A == 2 || A == 4, "sixteen elements of a thread are whole groups of four of its lanes");
    __shared__ double sh[L / 32];
    wait_for_prior_grid();
    release_dependents();
    for (size_t seg = blockIdx.x; seg < n_segments; seg += gridDim.x) {
        const float* p = sse + seg * blocks_per_segment;
        double acc[A];
#pragma unroll
        for (int a = 0; a < A; ++a) acc[a] = 0.0;
        // element m * T + t belongs to lane m % A of the thread: group r of a lane is m = (4 r + 0 .. 3) A + a
        auto add_four = [&](const float* w, int r, int a) {
            const float* const x = w + 4 * r * A + a;
            acc[a] = __dadd_rn(acc[a], __dadd_rn(__dadd_rn((double)x[0], (double)x[A]), __dadd_rn((double)x[2 * A], (double)x[3 * A])));
        };
        size_t i = threadIdx.x;
        for (; i + 15 * T < blocks_per_segment; i += 16 * T) {
            float w[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) w[m] = p[i + m * T];
#pragma unroll
            for (int k = 0; k < 4; ++k) add_four(w, k / A, k % A);
        }
        const int rest = (int)(blocks_per_segment - (i - threadIdx.x));   // negative or below 16 T
        const float* const q = p + (i - threadIdx.x);
        if (rest > 4 * T) {
            float w[16];
#pragma unroll
            for (int m = 0; m < 16; ++m) w[m] = (int)threadIdx.x + m * T < rest ? q[m * T + threadIdx.x] : 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (4 * (k / A) * L < rest) add_four(w, k / A, k % A);
        } else if (rest > 0) {
            float w[4 * A];
#pragma unroll
            for (int m = 0; m < 4 * A; ++m) w[m] = m < 4 && (int)threadIdx.x + m * T < rest ? q[m * T + threadIdx.x] : 0.0f;
#pragma unroll
            for (int a = 0; a < A; ++a) add_four(w, 0, a);
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[a] = __dadd_rn(acc[a], __shfl_down_sync(0xFFFFFFFFu, acc[a], o));
            if ((threadIdx.x & 31) == 0) sh[a * (T / 32) + (threadIdx.x >> 5)] = acc[a];
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            double t = threadIdx.x < L / 32 ? sh[threadIdx.x] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t = __dadd_rn(t, __shfl_down_sync(0xFFFFFFFFu, t, o));
            if (threadIdx.x == 0) out[seg] = __ddiv_rn(t, elems_per_segment);
        }
        __syncthreads();
    }
}

cudaError_t launch_segment_mse(const float* sse, size_t n_segments, size_t blocks_per_segment, size_t elems_per_segment,
                               double* out, cudaStream_t s) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const size_t sms = (size_t)sm_count(dev);
    // Few segments need wide CTAs, many of them small ones; what counts is the pass right after the one that wrote the SSEs, which
    // finds part of them in L2 only.  us added to that pass, T = 256 / 512 / 1024: 151 segments of 6000 blocks 4.5 / 3.2 / 3.1, 10,000 6.2 /
    // 3.9 / 3.4, 50,000 25 / 15 / 10; 500 of 4096 3.9 / 2.7 / 4.4, of 20,000 22 / 15 / 18; 10,000 of 64, from L2, 9.8 / 19 / 37.
    int threads = 256;
    auto* kernel = k_segment_mse<256, 256>;
    if (blocks_per_segment >= 8192) {
        threads = n_segments <= 3 * sms ? 1024 : 512;
        kernel = threads == 1024 ? k_segment_mse<1024, 1024> : k_segment_mse<512, 1024>;
    } else if (blocks_per_segment >= 4096) {
        threads = n_segments <= 4 * sms ? 512 : 256;
        kernel = threads == 512 ? k_segment_mse<512, 512> : k_segment_mse<256, 512>;
    }
    const size_t cap = sms * (2048 / threads);
    const unsigned grid = (unsigned)(n_segments < cap ? n_segments : cap);
    err = launch_pdl(kernel, grid, (unsigned)threads, 0, s, sse, n_segments, blocks_per_segment, (double)elems_per_segment, out);
    count_launch();
    return err;
}

// ------------------------------------------------------------------------------------------------
// Magnitude-interval masking (Appendix, unquantized ablation): entries with lo <= |x| < hi become
// +0, all others pass unchanged.  Elementwise, 16 bytes per thread and trip.
// ------------------------------------------------------------------------------------------------
template <int DT>
__global__ void __launch_bounds__(kThreads) k_mask_interval(const void* x, size_t n, float lo, float hi, void* out) {
    constexpr int VEC = 16 / elem_bytes(DT);
    const size_t n_vec = n / VEC;
    const size_t stride = (size_t)gridDim.x * kThreads;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < n_vec; i += stride) {
        uint4 w = __ldcs(static_cast<const uint4*>(x) + i);
        uint32_t* p = reinterpret_cast<uint32_t*>(&w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (DT == kF32) {
                const float a = fabsf(__uint_as_float(p[k]));
                if (a >= lo && a < hi) p[k] = 0u;
            } else {
                const float a0 = fabsf(__uint_as_float(p[k] << 16)), a1 = fabsf(__uint_as_float(p[k] & 0xFFFF0000u));
                if (a0 >= lo && a0 < hi) p[k] &= 0xFFFF0000u;
                if (a1 >= lo && a1 < hi) p[k] &= 0x0000FFFFu;
            }
        }
        __stcs(static_cast<uint4*>(out) + i, w);
    }
    if (blockIdx.x == 0 && threadIdx.x < (unsigned)(n - n_vec * VEC)) {   // ragged end, scalar
        const size_t e = n_vec * VEC + threadIdx.x;
        if constexpr (DT == kF32) {
            const float v = static_cast<const float*>(x)[e];
            static_cast<float*>(out)[e] = (fabsf(v) >= lo && fabsf(v) < hi) ? 0.0f : v;
        } else {
            const uint16_t h = static_cast<const uint16_t*>(x)[e];
            const float a = fabsf(__uint_as_float((uint32_t)h << 16));
            static_cast<uint16_t*>(out)[e] = (a >= lo && a < hi) ? (uint16_t)0 : h;
        }
    }
}

cudaError_t launch_mask_interval(const void* x, int dtype, size_t n, float lo, float hi, void* out, cudaStream_t s) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    size_t want = (n / (16 / elem_bytes(dtype)) + kThreads - 1) / kThreads;
    if (want == 0) want = 1;
    const size_t cap = (size_t)sm_count(dev) * 8;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    if (dtype == kF32) k_mask_interval<kF32><<<grid, kThreads, 0, s>>>(x, n, lo, hi, out);
    else k_mask_interval<kBF16><<<grid, kThreads, 0, s>>>(x, n, lo, hi, out);
    count_launch();
    return cudaGetLastError();
}

}  // namespace mxq
