// Small kernels around the quantization pass: per-tensor abs-max (first stage of hierarchical
// scaling), deterministic tensor MSE and de-quantization.
#include <cuda_bf16.h>

#include <atomic>
#include <mutex>

#include "mxq_device.cuh"
#include "mxq_internal.h"

namespace mxq {

// ------------------------------------------------------------------------------------------------
// Slots in which the CTAs of a launch leave their maximum and count themselves, so that no kernel has to initialise those words: zero
// between launches, the last CTA puts them back.  A ring of them per device, 2 MB that every GPU which loads the library holds until
// exit, handed out in turn: a slot comes round again 2^18 calls later, where a stream holds about a thousand launches in flight.
// ------------------------------------------------------------------------------------------------
struct DoneSlot {
    unsigned arrived, max_bits;
};
constexpr unsigned kDoneSlots = 1u << 18;
static __device__ DoneSlot g_done_slots[kDoneSlots];

// The number of a slot for one launch (a number and not an address: the kernel finds the array of the context that it runs in, whichever
// device that is and however often its context was made anew), or -1 while the stream is being captured (a graph replays with the
// same slot at any later time, beside launches that were given it meanwhile): the launch then takes the route with the initialising kernel.
static int done_slot(cudaStream_t s) {
    static std::atomic<unsigned> next{0};
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) return -1;
    return (int)(next.fetch_add(1, std::memory_order_relaxed) % kDoneSlots);
}

// ------------------------------------------------------------------------------------------------
// Tensor abs-max: max is exact and order-independent, so the cross-CTA step is an integer
// atomicMax on the bit pattern of the non-negative result (deterministic).
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_max(float m) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    return m;
}

// Without a slot (under capture): zeroes the running maximum and, when a tensor scale is wanted, the word that first counts the
// CTAs that have finished and then receives the scale.
__global__ void k_amax_init(uint32_t* amax_bits, uint32_t* g_word) {
    wait_for_prior_grid();
    release_dependents();
    *amax_bits = 0u;
    if (g_word) *g_word = 0u;
}

__device__ __forceinline__ float scale_of_amax(float a) { return (a > 0.0f && a <= 3.402823466e38f) ? __fdiv_rn(a, 2688.0f) : 1.0f; }

// One CTA reads tiles of U x 256 sixteen-byte vectors (U independent loads per thread in flight).  The running maximum and the
// count of CTAs that have finished lie in the launch's slot, or, without one, in out_bits and g_word.  The
// last CTA to finish turns the maximum into g = amax / (6 * 448), the tensor
// maximum mapped to the top of FP4 times the top of E4M3, and stores both.  Loads are
// streaming (evict-first): reading with the default policy, so that the quantize pass that follows finds
// the tensor in L2, was measured on 33 to 117 MB tensors and gains nothing (that pass is not DRAM-bound
// enough at those sizes), while it slows this kernel by 5 %.
template <int DT>
__global__ void __launch_bounds__(kThreads) k_tensor_amax(const void* x, size_t n, uint32_t* out_bits, uint32_t* g_word, int slot) {
    constexpr int VEC = 16 / elem_bytes(DT);
    constexpr int U = 4;
    const size_t n_vec = n / VEC;
    const size_t tile = (size_t)U * kThreads;
    const uint4* p = static_cast<const uint4*>(x);
    {   // while the kernel before this one drains: ask L2 for this thread's first vector (no architectural effect)
        const size_t first = (size_t)blockIdx.x * tile + threadIdx.x;
        if (first < n_vec) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + first));
    }
    wait_for_prior_grid();
    release_dependents();
    float m = 0.0f;
    uint32_t a16 = 0;   // bf16: magnitudes order like their 15-bit patterns, packed unsigned 16-bit max
    for (size_t base = (size_t)blockIdx.x * tile; base < n_vec; base += (size_t)gridDim.x * tile) {
        uint4 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t i = base + (size_t)u * kThreads + threadIdx.x;
            w[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i < n_vec) w[u] = __ldcs(p + i);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (DT == kF32) {
                m = fmaxf(fmaxf(m, fabsf(__uint_as_float(w[u].x))), fabsf(__uint_as_float(w[u].y)));
                m = fmaxf(fmaxf(m, fabsf(__uint_as_float(w[u].z))), fabsf(__uint_as_float(w[u].w)));
            } else {
                a16 = __vmaxu2(a16, __vmaxu2(w[u].x & 0x7FFF7FFFu, w[u].y & 0x7FFF7FFFu));
                a16 = __vmaxu2(a16, __vmaxu2(w[u].z & 0x7FFF7FFFu, w[u].w & 0x7FFF7FFFu));
            }
        }
    }
    if constexpr (DT == kBF16) m = fmaxf(__uint_as_float(a16 << 16), __uint_as_float(a16 & 0xFFFF0000u));
    if (blockIdx.x == 0 && threadIdx.x < (unsigned)(n - n_vec * VEC)) {  // ragged end, scalar
        const size_t i = n_vec * VEC + threadIdx.x;
        float v;
        if constexpr (DT == kF32) v = static_cast<const float*>(x)[i];
        else v = __uint_as_float((uint32_t) static_cast<const uint16_t*>(x)[i] << 16);
        m = fmaxf(m, fabsf(v));
    }
    __shared__ float warp_m[kThreads / 32];
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) warp_m[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < kThreads / 32 ? warp_m[threadIdx.x] : 0.0f;
        m = warp_max(m);
        if (threadIdx.x == 0) {
            DoneSlot* const done = slot >= 0 ? &g_done_slots[slot] : nullptr;
            unsigned* const run = done ? &done->max_bits : out_bits;
            unsigned* const count = done ? &done->arrived : g_word;
            atomicMax(run, __float_as_uint(m));
            if (count) {
                __threadfence();
                if (atomicAdd(count, 1u) == gridDim.x - 1) {   // every CTA's maximum is in
                    __threadfence();
                    const uint32_t bits = done ? atomicExch(run, 0u) : atomicMax(run, 0u);
                    if (done) {
                        done->arrived = 0;
                        *out_bits = bits;
                    }
                    if (g_word) *reinterpret_cast<float*>(g_word) = scale_of_amax(__uint_as_float(bits));
                }
            }
        }
    }
}

// The same for up to kOneCtaBytes of input (the activations of a few tokens) in one launch of one CTA: nothing to
// initialise, nothing to count.  32 KB: 7.6 -> 4.7 us of host time per call, which is what such calls cost (with the
// quantization that follows, replayed from a graph: 6.4 -> 4.5 us).  The limit keeps one SM's reads, about 100 GB/s, below
// the launch that is saved.
constexpr size_t kOneCtaBytes = 256 * 1024;
constexpr int kOneCtaThreads = 1024;
template <int DT>
__global__ void __launch_bounds__(kOneCtaThreads) k_tensor_amax_one(const void* x, size_t n, float* out, float* out_g) {
    constexpr int VEC = 16 / elem_bytes(DT);
    constexpr int U = 4;
    const int n_vec = (int)(n / VEC);
    const uint4* p = static_cast<const uint4*>(x);
    wait_for_prior_grid();
    release_dependents();
    float m = 0.0f;
    [[maybe_unused]] uint32_t a16 = 0;   // bf16: magnitudes order like their 15-bit patterns
    for (int base = threadIdx.x; base < n_vec; base += U * kOneCtaThreads) {
        uint4 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            w[u] = make_uint4(0u, 0u, 0u, 0u);
            if (base + u * kOneCtaThreads < n_vec) w[u] = p[base + u * kOneCtaThreads];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (DT == kF32) {
                m = fmaxf(fmaxf(m, fabsf(__uint_as_float(w[u].x))), fabsf(__uint_as_float(w[u].y)));
                m = fmaxf(fmaxf(m, fabsf(__uint_as_float(w[u].z))), fabsf(__uint_as_float(w[u].w)));
            } else {
                const uint32_t a = __vmaxu2(__vmaxu2(w[u].x & 0x7FFF7FFFu, w[u].y & 0x7FFF7FFFu), __vmaxu2(w[u].z & 0x7FFF7FFFu, w[u].w & 0x7FFF7FFFu));
                a16 = __vmaxu2(a16, a);
            }
        }
    }
    if constexpr (DT == kBF16) m = fmaxf(__uint_as_float(a16 << 16), __uint_as_float(a16 & 0xFFFF0000u));
    if (threadIdx.x < (unsigned)(n - (size_t)n_vec * VEC)) {  // ragged end, scalar
        const size_t i = (size_t)n_vec * VEC + threadIdx.x;
        float v;
        if constexpr (DT == kF32) v = static_cast<const float*>(x)[i];
        else v = __uint_as_float((uint32_t) static_cast<const uint16_t*>(x)[i] << 16);
        m = fmaxf(m, fabsf(v));
    }
    __shared__ float warp_m[kOneCtaThreads / 32];
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) warp_m[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = warp_max(warp_m[threadIdx.x]);
        if (threadIdx.x == 0) {
            *out = m;
            if (out_g) *out_g = scale_of_amax(m);
        }
    }
}

cudaError_t launch_tensor_amax(const void* x, int dtype, size_t n, float* d_amax, float* d_g, cudaStream_t s) {
    if (n * elem_bytes(dtype) <= kOneCtaBytes) {
        const cudaError_t e = dtype == kF32 ? launch_pdl(k_tensor_amax_one<kF32>, 1u, (unsigned)kOneCtaThreads, 0, s, x, n, d_amax, d_g)
                                            : launch_pdl(k_tensor_amax_one<kBF16>, 1u, (unsigned)kOneCtaThreads, 0, s, x, n, d_amax, d_g);
        count_launch();
        return e;
    }
    uint32_t* amax_bits = reinterpret_cast<uint32_t*>(d_amax);
    uint32_t* g_word = reinterpret_cast<uint32_t*>(d_g);
    const int slot = done_slot(s);
    cudaError_t err = cudaSuccess;
    if (slot < 0) {
        err = launch_pdl(k_amax_init, 1u, 1u, 0, s, amax_bits, g_word);
        count_launch();
        if (err != cudaSuccess) return err;
    }
    int dev = 0;
    err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const size_t n_vec = n / (16 / elem_bytes(dtype));
    size_t want = (n_vec + 4 * kThreads - 1) / (4 * kThreads);
    if (want == 0) want = 1;
    const size_t cap = (size_t)sm_count(dev) * 8;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    if (dtype == kF32) err = launch_pdl(k_tensor_amax<kF32>, grid, (unsigned)kThreads, 0, s, x, n, amax_bits, g_word, slot);
    else err = launch_pdl(k_tensor_amax<kBF16>, grid, (unsigned)kThreads, 0, s, x, n, amax_bits, g_word, slot);
    count_launch();
    return err;
}

// ------------------------------------------------------------------------------------------------
// Tensor MSE: two levels of fixed shape in binary64.  Level 1: P = min(1024, ceil(nb/256))
// CTAs, CTA p sums the contiguous slice [p*L, (p+1)*L), L = ceil(nb/P): thread t adds elements
// t, t+256, ... in order, then cta_sum_fixed_order().  Level 2: one CTA of 256 threads, sum_partials() over the P partials, divided by
// n (1024 threads and a halving tree of ten barriers: 0.5 us more; the last CTA of the first level in its place: 0.8 us more).
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_mse_partial(const float* sse, size_t nb, size_t slice, double* partials) {
    __shared__ double scratch[kThreads / 32];
    wait_for_prior_grid();
    release_dependents();
    const size_t lo = (size_t)blockIdx.x * slice;
    const size_t hi = (lo + slice < nb) ? lo + slice : nb;
    double acc = 0.0;
    for (size_t i = lo + threadIdx.x; i < hi; i += kThreads) acc = __dadd_rn(acc, (double)__ldcs(sse + i));
    const double total = cta_sum_fixed_order(acc, scratch);
    if (threadIdx.x == 0) partials[blockIdx.x] = total;
}

// The second level of a tensor MSE: sum of n partials over a CTA of kThreads threads in a fixed order (thread t those at t, t + 256,
// ..., then cta_sum_fixed_order()), valid in thread 0.  Read from L2: other CTAs have just written them.
__device__ __forceinline__ double sum_partials(const double* partials, int n, double* scratch) {
    static_assert(kMsePartials == 4 * kThreads, "four partials per thread");
    double w[4];   // all reads at once: one after the other they cost a large tensor 0.2 us
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = threadIdx.x + k * kThreads;
        w[k] = i < n ? __ldcg(partials + i) : 0.0;
    }
    return cta_sum_fixed_order(__dadd_rn(__dadd_rn(__dadd_rn(w[0], w[1]), w[2]), w[3]), scratch);
}

__global__ void __launch_bounds__(kThreads) k_mse_final(const double* partials, int n_partials, double n, double* out) {
    __shared__ double scratch[kThreads / 32];
    wait_for_prior_grid();
    release_dependents();
    const double total = sum_partials(partials, n_partials, scratch);
    if (threadIdx.x == 0) *out = __ddiv_rn(total, n);
}

cudaError_t launch_tensor_mse(const float* d_sse, size_t n_blocks, size_t n, double* d_out, double* d_partials,
                              cudaStream_t s) {
    size_t P = (n_blocks + kThreads - 1) / kThreads;
    if (P > (size_t)kMsePartials) P = kMsePartials;
    const size_t slice = (n_blocks + P - 1) / P;
    // staged launches: the launch latency of these two small kernels comes off the critical path
    cudaError_t err = launch_pdl(k_mse_partial, (unsigned)P, kThreads, 0, s, d_sse, n_blocks, slice, d_partials);
    count_launch();
    if (err != cudaSuccess) return err;
    return launch_mse_final(d_partials, (int)P, n, d_out, s);
}

cudaError_t launch_mse_final(const double* d_partials, int n_partials, size_t n, double* d_out, cudaStream_t s) {
    cudaError_t err = launch_pdl(k_mse_final, 1u, (unsigned)kThreads, 0, s, d_partials, n_partials, (double)n, d_out);
    count_launch();
    return err;
}

// ------------------------------------------------------------------------------------------------
// De-quantization: x_hat = fl32(grid(code) * D), D = fl32(S * g).  One thread per 8 elements.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float decode_scale(int fmt, int c, float g) {
    if (c >= num_codes(fmt)) return __uint_as_float(0x7FC00000u);
    return __fmul_rn(scale_value(fmt, c), g);
}

// A unit is the run of elements whose results one thread writes with ONE 16-byte store, so that a
// warp's store covers 512 contiguous bytes: 8 elements for bf16 output, 4 for fp32 output.  Four
// units per thread and trip, and the loads of the next trip issued before this trip's stores, keep
// eight independent loads in flight.  Measured on 134 M elements: 110 to 115 us for fp32 output (5.4 TB/s of
// codes + scales + output; a plain fill of the same output alone takes 82 us) whatever was tried -- plain
// instead of streaming stores, grids of 4, 8 or 16 CTAs per SM (five are resident with fp32 output, four with bf16), grid-stride or
// CTA-contiguous tiles, with
// or without the table and the early loads; those two shorten B = 2 by about 5 % and were kept.
// EARLY: the first loads are issued before the table is built, else between the table and its barrier.  Early is right from the third trip of a
// CTA on, behind it up to the second (launch_dequantize() counts them; B = 16, us, early / behind: bf16 out 2.1 M elements 2.65 / 2.39, 8.4 M
// 5.6 / 5.0, 67 M 32.7 / 33.8 or more; fp32 out 4.2 M 5.0 / 4.4, 67 M 56.3 / 57.4).
template <int ODT, bool EARLY>
__global__ void __launch_bounds__(kThreads) k_dequantize(const uint8_t* codes, const uint8_t* scales, size_t n,
                                                         int log2B, int fmt, float g_host, const float* d_g, void* out) {
    wait_for_prior_grid();
    release_dependents();
    // decode scales of all 256 codes, one per thread: a table read replaces a dozen instructions per unit
    __shared__ float Dtab[256];
    auto build_table = [&] {
        const float g = d_g ? *d_g : g_host;   // device-resident tensor scale (written by an earlier kernel of the stream)
        Dtab[threadIdx.x] = decode_scale(fmt, (int)threadIdx.x, g);
    };
    if constexpr (!EARLY) build_table();
    constexpr int E = (ODT == kF32) ? 4 : 8;      // elements per unit
    constexpr int LOG2E = (ODT == kF32) ? 2 : 3;
    constexpr int U = 4;
    const size_t n_units = n / E;
    const size_t stride = (size_t)gridDim.x * kThreads;
    // the loads of the next trip are issued before the arithmetic and the stores of this one
    auto load_trip = [&](size_t first, uint32_t (&w)[U], uint32_t (&sc)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t i = first + (size_t)u * kThreads;
            w[u] = 0;
            sc[u] = 0;
            if (i < n_units) {
                if constexpr (E == 8) w[u] = __ldcs(reinterpret_cast<const uint32_t*>(codes) + i);
                else w[u] = __ldcs(reinterpret_cast<const uint16_t*>(codes) + i);
                // the scale codes of the unit's blocks (one byte when a block holds the whole unit)
                if (log2B >= LOG2E) sc[u] = scales[(i << LOG2E) >> log2B];
                else if (E >> log2B == 2) sc[u] = reinterpret_cast<const uint16_t*>(scales)[i];
                else sc[u] = reinterpret_cast<const uint32_t*>(scales)[i];
            }
        }
    };
    // a CTA works on tiles of U x 256 consecutive units (16 KB of fp32 output), tiles b, b + grid, ...
    size_t base = (size_t)blockIdx.x * (U * kThreads) + threadIdx.x;
    uint32_t w[U], sc[U];
    load_trip(base, w, sc);
    if constexpr (EARLY) build_table();
    __syncthreads();
    for (; base < n_units; base += stride * U) {
        uint32_t wn[U], scn[U];
        load_trip(base + stride * U, wn, scn);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t i = base + (size_t)u * kThreads;
            if (i >= n_units) continue;
            float q[8];
            unpack_e2m1x8(w[u], q);
            float xh[E];
            if (log2B >= LOG2E) {
                const float D = Dtab[sc[u]];
#pragma unroll
                for (int k = 0; k < E; ++k) xh[k] = __fmul_rn(q[k], D);
            } else {
#pragma unroll
                for (int k = 0; k < E; ++k)
                    xh[k] = __fmul_rn(q[k], Dtab[(sc[u] >> (8 * (k >> log2B))) & 0xFFu]);
            }
            if constexpr (ODT == kF32) {
                __stcs(static_cast<float4*>(out) + i, make_float4(xh[0], xh[1], xh[2], xh[3]));
            } else {
                uint32_t h[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __nv_bfloat162 b = __floats2bfloat162_rn(xh[2 * k], xh[2 * k + 1]);
                    h[k] = *reinterpret_cast<const uint32_t*>(&b);
                }
                __stcs(static_cast<uint4*>(out) + i, make_uint4(h[0], h[1], h[2], h[3]));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            w[u] = wn[u];
            sc[u] = scn[u];
        }
    }
    // ragged end (n not a multiple of the unit; only possible for block sizes 2 and 4)
    if (blockIdx.x == 0 && threadIdx.x < (unsigned)(n - n_units * E)) {
        const size_t e = n_units * E + threadIdx.x;
        const uint32_t c4 = (codes[e >> 1] >> ((e & 1) ? 4 : 0)) & 15u;
        float q[8];
        unpack_e2m1x8(c4, q);
        const float xh = __fmul_rn(q[0], Dtab[scales[e >> log2B]]);
        if constexpr (ODT == kF32) static_cast<float*>(out)[e] = xh;
        else static_cast<__nv_bfloat16*>(out)[e] = __float2bfloat16_rn(xh);
    }
}

cudaError_t launch_dequantize(const uint8_t* codes, const uint8_t* scales, size_t n, int B, int fmt, float g,
                              const float* d_g, void* out, int out_dtype, cudaStream_t s) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    int log2B = 0;
    while ((1 << log2B) < B) ++log2B;
    size_t want = ((n >> (out_dtype == kF32 ? 2 : 3)) / 4 + kThreads - 1) / kThreads;   // four units per thread
    if (want == 0) want = 1;
    const size_t cap = (size_t)sm_count(dev) * 8;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    const bool early = want > 2 * cap;
    auto* const kernel = out_dtype == kF32 ? (early ? k_dequantize<kF32, true> : k_dequantize<kF32, false>)
                                           : (early ? k_dequantize<kBF16, true> : k_dequantize<kBF16, false>);
    err = launch_pdl(kernel, grid, (unsigned)kThreads, 0, s, codes, scales, n, log2B, fmt, g, d_g, out);
    count_launch();
    return err;
}

}  // namespace mxq

// ------------------------------------------------------------------------------------------------
// Tensor MSE for callers that cannot provide scratch memory: the first-level partial sums live in
// a file-scope device array instead of a caller workspace.  Every GPU that loads the library
// carries these 8 KiB until the process exits.  In host code the array's name is only a handle
// for the runtime, so its device address is looked up once per device (with that device current)
// and handed to the same two kernels as the workspace variant.  Nothing in the array has to start
// at zero: the first kernel writes every partial the second one reads.
// ------------------------------------------------------------------------------------------------
namespace mxq {

static __device__ __align__(256) double g_mse_static_partials[kMsePartials];

cudaError_t launch_tensor_mse_static(const float* d_sse, size_t n_blocks, size_t n, double* d_out, cudaStream_t s) {
    static std::mutex mu;
    static double* scratch_of_device[kMaxDevices] = {nullptr};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    double* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        scratch = scratch_of_device[dev];
        if (scratch == nullptr) {  // first call on this device: resolve the symbol to a device address
            void* p = nullptr;
            err = cudaGetSymbolAddress(&p, g_mse_static_partials);
            if (err != cudaSuccess) return err;
            if (p == nullptr) return cudaErrorInvalidSymbol;
            scratch = static_cast<double*>(p);
            scratch_of_device[dev] = scratch;
        }
    }
    return launch_tensor_mse(d_sse, n_blocks, n, d_out, scratch, s);
}

}  // namespace mxq
