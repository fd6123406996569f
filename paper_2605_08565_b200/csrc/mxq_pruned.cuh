// Pruned scale search (MXQ_OPT_BRUTE_PRUNE): the brute-force recipes with the codes left out that provably cannot change
// an output, decided BLOCK BY BLOCK.  Outputs are those of the full sweep (mxq_brute.cuh), bit for bit.
//
// A block tries two codes first (the ones nearest to a / 6 and a / 4, a = max |v|); the better SSE, U, bounds the rest.
// With e = fma(q, -D, v), s = fma(e, e, s) in element order and round-to-nearest, which is monotone, an SSE never
// decreases when a term is added or grows, so every rule below compares in the very arithmetic of the SSE, or with a
// slack far above its rounding:
//   zero rule    D >= 4 a: every quotient is at most 1/4 and rounds to 0 (the tie goes to the even index).  All such codes
//                have the SSE of the all-zero quantization, which is entered once with the smallest of them (a zero decode
//                scale counts as one).
//   high rule    D >= 4 theta, theta = a / 8 or a / 4: the elements with |v| <= theta go to zero; if their sum of squares (same
//                order) exceeds U, no such code can win or tie.
//   low rule     6 D <= a: the largest element saturates and leaves fl(a - 6 D); every D below a D' with fl(fl(a - 6 D')^2) >
//                U is out.
//   windows      (FP8 formats, B <= 16) the largest element alone costs (a - q D)^2 for SOME grid value q, so with
//                r = sqrt(U) the code is out unless a - r <= q D <= a + r for one q of {1/2, 1, 3/2, 2, 3, 4, 6} (q = 0 is
//                out when r < a).  Codes of these formats are eight per binade, so the windows of q = 6, 3, 3/2 are one
//                bit pattern shifted by 8, and so are those of q = 4, 2, 1, 1/2: two windows are computed, seven covered.
// What is left is a bit mask of codes per block: on average 9 (B = 4) to 17 (B = 64) of 127 or 255 for Laplace and
// Student-t data.
//
// Work layout (FP8 formats).  A CTA takes a tile of consecutive blocks.  Phase 1: one thread per block loads it (to
// registers and to a shared tile), tries the two codes and forms the mask.  A counting sort on the number of candidate
// pairs then brings blocks with equally long lists together, so that the lanes of a warp finish together.  Phase 2: one
// thread per block, in sorted order, two candidates per trip (the two lanes of the packed SSE accumulation); decode scales
// are read from shared tables at per-lane codes.  Phase 3: encode with the winner and store, in the original order.  A
// block's result does not depend on where it was evaluated, so the (unordered) ranks inside a bin change nothing.  The
// power-of-two format leaves two to four codes per block and has a kernel of its own without tile and sort.
//
// Bound by issue slots (FP4 pack and unpack, quotients, residuals, and for small blocks the bookkeeping of the lists), like
// the full sweep; the gain is the shorter list.  Measured against a sweep whose warps cut their code ranges by the extreme
// maxima of all the blocks they hold (sorted by magnitude), 16.8 M elements, us before -> now:
//   fp32 Laplace, tensor scale, UE4M3   B = 2 336 -> 196   4 259 -> 133   8 191 -> 115   16 167 -> 116   32 161 -> 131   64 167 -> 154
//   bf16 Student-t, UE5M3               B = 2 330 -> 212   4 258 -> 134   8 209 -> 106   16 185 -> 97    32 181 -> 113   64 197 -> 132
//   bf16 Student-t, UE8M0               B = 2 185 -> 76    4 107 -> 59    8 88 -> 47     16 84 -> 37     32 59 -> 31     64 72 -> 34
#pragma once

#include <atomic>

#include "mxq_brute.cuh"
#include "mxq_quantize.cuh"

namespace mxq {

// Shared-memory layout of a tile.  The blocks' elements are kept as binary32; a block of B >= 4 elements is B / 4 pieces of 16
// bytes whose order is rotated by the block index (swizzle()), so that consecutive threads reading piece k of consecutive
// blocks spread over all banks.
template <int B>
struct PrunedTile {
    static constexpr int NB = B >= 32 ? 256 : (B == 16 ? 512 : 4096 / B);   // blocks per tile (one or more per thread)
    static constexpr int CH = B >= 4 ? B / 4 : 1;           // 16-byte pieces per block (B = 2: one of 8 bytes)
    static constexpr int BINS = 1024;
    static constexpr size_t KEY_OFF = (size_t)NB * B * 4;   // best (SSE bits, code) so far
    static constexpr size_t MASK_OFF = KEY_OFF + (size_t)NB * 8;
    static constexpr size_t HIST_OFF = MASK_OFF + (size_t)NB * 8;
    static constexpr size_t INFO_OFF = HIST_OFF + (size_t)BINS * 4;   // first code of the mask, evaluation mode
    static constexpr size_t PERM_OFF = INFO_OFF + (size_t)NB * 2;
    static constexpr size_t BYTES = PERM_OFF + (size_t)NB * 2;
    static __device__ __forceinline__ int swizzle(int blk) {
        return CH == 1 ? 0 : CH == 2 ? (blk >> 2) & 1 : CH == 4 ? (blk >> 1) & 3 : blk & 7;
    }
    static __device__ __forceinline__ int piece(int blk, int k) { return (blk * CH + (k ^ swizzle(blk))) * 4; }   // in floats
};

// Elements first .. first + N - 1 of block blk as pairs.
template <int B, int N>
__device__ __forceinline__ void tile_pairs(const float* tile, int blk, int first, float2 (&v2)[N / 2]) {
    if constexpr (B == 2) {
        v2[0] = *reinterpret_cast<const float2*>(tile + blk * 2);
    } else {
#pragma unroll
        for (int k = 0; k < N / 4; ++k) {
            const float4 w = *reinterpret_cast<const float4*>(tile + PrunedTile<B>::piece(blk, first / 4 + k));
            v2[2 * k] = make_float2(w.x, w.y);
            v2[2 * k + 1] = make_float2(w.z, w.w);
        }
    }
}

// A block in the form the evaluation takes it: each element twice (B <= 8), or pairs of neighbours.
__host__ __device__ constexpr int pruned_values(int B) { return B <= 8 ? B : B / 2; }
template <int B>
__device__ __forceinline__ void hold(const float2 (&v2)[B / 2], float2 (&v)[pruned_values(B)]) {
    if constexpr (B <= 8) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float x = (i & 1) ? v2[i / 2].y : v2[i / 2].x;
            v[i] = make_float2(x, x);
            asm volatile("" : "+f"(v[i].x), "+f"(v[i].y));   // two registers, not two names of one that every use has to copy
        }
    } else {
#pragma unroll
        for (int i = 0; i < B / 2; ++i) v[i] = v2[i];
    }
}
template <int B>
__device__ __forceinline__ float element(const float2 (&v)[pruned_values(B)], int i) {
    if constexpr (B <= 8) return v[i].x;
    else return (i & 1) ? v[i / 2].y : v[i / 2].x;
}

// How candidates are evaluated; table entries at the candidate's code.  kModeExact: corrected quotient, binary32 residual
// (-D, RN(1 / D)); holds for every decode scale in [2^-60, 2^60].  kModeHalf: -D is exact in f16 (and for bf16 input D
// has at most four significant bits, so that the quotient is one multiply rounded toward zero): z holds f16(-D).
// kModeChecked (bf16): the one-multiply quotient with the reciprocal that build_quant_tables() checked, which z holds.
// kModeSlow: search_by_division().
enum { kModeExact = 0, kModeHalf = 1, kModeChecked = 2, kModeSlow = 3 };
struct PrunedTables {
    float nD[256], R[256], z[256];
};

// The grid values that two quotients round to, widened by mixed-precision adds of -0 (exact).
__device__ __forceinline__ float2 round_widen_pair(float2 t) {
    float2 q;
    asm("{\n"
        " .reg .b8 b0;\n"
        " .reg .b32 h;\n"
        " .reg .b16 lo, hi;\n"
        " cvt.rn.satfinite.e2m1x2.f32 b0, %3, %2;\n"
        " cvt.rn.f16x2.e2m1x2 h, b0;\n"
        " mov.b32 {lo, hi}, h;\n"
        " add.rn.f32.f16 %0, lo, %4;\n"
        " add.rn.f32.f16 %1, hi, %4;\n"
        "}"
        : "=f"(q.x), "=f"(q.y)
        : "f"(t.x), "f"(t.y), "f"(-0.0f));
    return q;
}

// What an evaluation needs of two candidates (.x, .y).
template <int DT, int MODE>
struct Candidates {
    static constexpr bool ONE_MULTIPLY = (DT == kBF16) && MODE != kModeExact;
    float2 nD, R;
    uint32_t nD16;   // kModeHalf: f16(-D) of the two
    __device__ __forceinline__ void read(const PrunedTables& T, int cA, int cB) {
        const float* const recip = MODE == kModeChecked ? T.z : T.R;
        R = make_float2(recip[cA], recip[cB]);
        if constexpr (MODE != kModeHalf || !ONE_MULTIPLY) nD = make_float2(T.nD[cA], T.nD[cB]);
        else nD = make_float2(0.0f, 0.0f);
        if constexpr (MODE == kModeHalf) nD16 = __byte_perm(__float_as_uint(T.z[cA]), __float_as_uint(T.z[cB]), 0x5410);
        else nD16 = 0;
    }
};

// SSEs of one block under two candidates.
template <int DT, int B, int MODE>
__device__ __forceinline__ float2 sse_two_candidates(const float2 (&v2)[pruned_values(B)], const Candidates<DT, MODE>& c) {
    constexpr bool HALF = (MODE == kModeHalf);
    constexpr bool ONE_MULTIPLY = Candidates<DT, MODE>::ONE_MULTIPLY;
    const float2 nD = c.nD, R = c.R;
    const uint32_t nD16 = c.nD16;
    float2 s = make_float2(0.0f, 0.0f);
    if constexpr (B <= 8) {
        // the lanes of every packed instruction are the two candidates, the elements held twice
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float2 vv = v2[i];
            const float v = vv.x;
            const float2 t = ONE_MULTIPLY ? __fmul2_rz(vv, R) : quotient_pair(vv, nD, R);
            float2 e;
            if constexpr (HALF) {
                e = residual_two_candidates<true>(t.x, t.y, v, 0.0f, 0.0f, nD16);
            } else {
                e = __ffma2_rn(round_widen_pair(t), nD, vv);
            }
            s = __ffma2_rn(e, e, s);
        }
    } else {
        // quotients of two elements per instruction: longer blocks would need too many registers held twice
        const float2 RA2 = make_float2(R.x, R.x), RB2 = make_float2(R.y, R.y);
        const float2 DA2 = make_float2(nD.x, nD.x), DB2 = make_float2(nD.y, nD.y);
#pragma unroll
        for (int i = 0; i < B / 2; ++i) {
            float2 tA, tB;
            if constexpr (ONE_MULTIPLY) {
                tA = __fmul2_rz(v2[i], RA2);
                tB = __fmul2_rz(v2[i], RB2);
            } else {
                tA = quotient_pair(v2[i], DA2, RA2);
                tB = quotient_pair(v2[i], DB2, RB2);
            }
            const float2 e0 = residual_two_candidates<HALF>(tA.x, tB.x, v2[i].x, nD.x, nD.y, nD16);
            s = __ffma2_rn(e0, e0, s);
            const float2 e1 = residual_two_candidates<HALF>(tA.y, tB.y, v2[i].y, nD.x, nD.y, nD16);
            s = __ffma2_rn(e1, e1, s);
        }
    }
    return s;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ unsigned long long shr64(unsigned long long x, int n) {
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}

__device__ __forceinline__ void keep_smaller_or_equal(uint32_t& best_bits, int& best_code, uint32_t bits, int code) {
    best_code = bits <= best_bits ? code : best_code;
    best_bits = min(best_bits, bits);
}

// Shift left by n; 0 for n outside 0 .. 63 (the instruction clamps).
__device__ __forceinline__ unsigned long long shl64(unsigned long long x, int n) {
    unsigned long long r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}

// A block outside the ranges of the shortcuts, with IEEE division: the best (SSE bits, code) among codes first .. n_codes - 1.
// decode(c): the decode scale, nondecreasing in c; pair(i): elements i and i + 1; a: the largest magnitude.  Codes are taken upwards from
// the first with 6 D >= a, then downwards from there, until
//   upwards     D >= 4 a: this and every larger D has the SSE of the all-zero quantization (ties go to the smaller code); or the
//               elements that D sends to zero (4 |v| <= D) alone cost more than the best SSE so far: they do under every larger D;
//   downwards   what the saturated elements leave, fl(|v| - 6 D) each, alone costs more: it does so under every smaller D.
// The sums compared are taken in the order and arithmetic of the SSE.  Magnitudes of 1e-20 under their tensor scale, 4.2 M elements:
// every code 1108 us for UE4M3 at B = 16 (fp32) and 1261 for UE5M3 at B = 2 (bf16), here 191 and 332.
template <int B, int UNROLL, typename Decode, typename Pair>
__device__ __forceinline__ unsigned long long search_by_division(Decode decode, Pair pair, float a, int first, int n_codes) {
    int c0 = first, end = n_codes;
    while (c0 < end) {
        const int mid = (c0 + end) >> 1;
        if (__fmul_rn(6.0f, decode(mid)) < a) c0 = mid + 1;
        else end = mid;
    }
    unsigned long long best = sse_key(__uint_as_float(0xFFFFFFFFu), first);
    bool up = true;
    int c = c0;
    while (up || c >= first) {
        const float D = c < n_codes ? decode(c) : __uint_as_float(0x7F800000u);
        if (!(fabsf(D) <= 3.402823466e38f)) {   // overflowed: not usable, nor is any larger code
            c = up ? c0 - 1 : c - 1;
            up = false;
            continue;
        }
        float s = 0.0f, z = 0.0f;
#pragma unroll UNROLL
        for (int i = 0; i < B; i += 2) {
            const float2 v = pair(i);
            const float2 q = round_e2m1x2(quotient_general(v.x, D), quotient_general(v.y, D));
            const float e0 = __fmaf_rn(-q.x, D, v.x), e1 = __fmaf_rn(-q.y, D, v.y);
            s = __fmaf_rn(e0, e0, s);
            s = __fmaf_rn(e1, e1, s);
            const float a0 = fabsf(v.x), a1 = fabsf(v.y);
            const float z0 = up ? (__fmul_rn(4.0f, a0) <= D ? a0 : 0.0f) : fmaxf(__fmaf_rn(-6.0f, D, a0), 0.0f);
            const float z1 = up ? (__fmul_rn(4.0f, a1) <= D ? a1 : 0.0f) : fmaxf(__fmaf_rn(-6.0f, D, a1), 0.0f);
            z = __fmaf_rn(z0, z0, z);
            z = __fmaf_rn(z1, z1, z);
        }
        best = min(best, sse_key(s, c));
        const bool rest_is_out = __float_as_uint(z) > (uint32_t)(best >> 32) || (up && D >= __fmul_rn(4.0f, a));
        if (!rest_is_out) {
            c += up ? 1 : -1;
        } else if (up) {
            up = false;
            c = c0 - 1;
        } else {
            break;
        }
    }
    return best;
}

// The same for block b of a tile; out of line, to leave the registers of the search proper alone.
template <int B>
__device__ __noinline__ unsigned long long search_tile_block(const float* tile, int b, const float* nD, int first, int n_codes) {
    auto pair = [&](int i) {
        if constexpr (B == 2) return *reinterpret_cast<const float2*>(tile + b * 2);
        else return *reinterpret_cast<const float2*>(tile + PrunedTile<B>::piece(b, i / 4) + (i & 3));
    };
    float a = 0.0f;
#pragma unroll 1
    for (int i = 0; i < B; i += 2) a = fmaxf(a, fmaxf(fabsf(pair(i).x), fabsf(pair(i).y)));
    return search_by_division<B, 1>([&](int c) { return -nD[c]; }, pair, a, first, n_codes);
}

// The first n blocks of a unit of eight elements (B = 2 or 4), from block blk on.
template <int B, int UB>
__device__ __forceinline__ void store_whole_blocks(const QuantArgs& p, size_t blk, size_t n, uint32_t packed, uint32_t sc, const uint32_t (&sw)[UB]) {
    if constexpr (B < 8) {
#pragma unroll
        for (int j = 0; j < UB; ++j) {
            if ((size_t)j >= n) break;
            const uint32_t codes = packed >> (4 * B * j);
            store_bytes<B / 2>(p.codes + (blk + j) * (B / 2), &codes);
            p.scales[blk + j] = (uint8_t)(sc >> (8 * j));
            if (p.block_sse) p.block_sse[blk + j] = __uint_as_float(sw[j]);
        }
    }
}

// Resident CTAs per SM asked of the register allocator: a block is held in registers through the search, up to 32 elements
// beside two or three CTAs of 256 threads; B = 64 runs one (parts of 16 or 32 elements read from the tile on every trip
// leave room for two or three and lose 20 to 45 %).
__host__ __device__ constexpr int pruned_min_ctas(int B) { return B <= 16 ? 3 : B == 32 ? 2 : 1; }

template <int DT, int B, int FMT>
__global__ void __launch_bounds__(kThreads, pruned_min_ctas(B)) k_pruned(QuantArgs p, int tile_blocks) {
    using Tile = PrunedTile<B>;
    constexpr int NV = pruned_values(B);
    constexpr bool AHEAD = B <= 16;   // the next block's elements are loaded while one is worked on
    constexpr int NC = num_codes(FMT);
    static_assert(FMT != kUE8M0, "the power-of-two format has its own kernel");
    constexpr bool WINDOWS = B <= 16;
    constexpr float kUp = 1.00000095367431640625f, kDown = 0.99999904632568359375f;   // 1 +- 2^-20: above the rounding of a / g
    extern __shared__ uint4 pruned_dyn[];
    unsigned char* const dyn = reinterpret_cast<unsigned char*>(pruned_dyn);
    float* const tile = reinterpret_cast<float*>(dyn);
    unsigned long long* const key = reinterpret_cast<unsigned long long*>(dyn + Tile::KEY_OFF);
    unsigned long long* const mask = reinterpret_cast<unsigned long long*>(dyn + Tile::MASK_OFF);
    uint32_t* const hist = reinterpret_cast<uint32_t*>(dyn + Tile::HIST_OFF);
    uint16_t* const info = reinterpret_cast<uint16_t*>(dyn + Tile::INFO_OFF);
    uint16_t* const perm = reinterpret_cast<uint16_t*>(dyn + Tile::PERM_OFF);
    __shared__ QuantTables T;
    __shared__ PrunedTables tab;
    __shared__ uint32_t warp_total[kThreads / 32];
    __shared__ int short_end;   // f32: first code whose -D is not exact in f16

    wait_for_prior_grid();
    release_dependents();
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const int first = p.prevent_zero ? 1 : 0;
    if (threadIdx.x == 0) short_end = NC;
    int first_bad;
    const bool checked = build_quant_tables<FMT, DT == kBF16>(T, g, first_bad);   // barriers inside
    {
        const int c = threadIdx.x;
        const float4 E = T.E[c];
        tab.nD[c] = -E.x;
        tab.R[c] = E.y;
        tab.z[c] = E.z;   // a reciprocal when checked, else f16(-D) in the low half
        if (DT == kF32 && c < NC && E.w < 2.0f) atomicMin(&short_end, c);
    }
    __syncthreads();
    const int fast_mode = checked ? kModeChecked : kModeHalf;
    const int fast_end = checked ? NC : (DT == kF32 ? short_end : first_bad);   // codes below it may be evaluated in fast_mode
    // The shortcuts need decode scales in [2^-60, 2^60].  For g within kMaxG of 1 every nonzero code has one.  Beyond, the codes from a / 12
    // to 4 a do (a within [2^-55, 2^57], codes are at most a factor of two apart), which are all that a block with r < a / 2 looks at
    // (magnitudes of 1e-12 under their tensor scale, UE5M3, B = 8, 4.2 M elements: 2166 -> 36 us).
    constexpr float kMaxG = FMT == kUE4M3 ? 2.251799813685248e15f /* 2^51 */ : 8.796093022208e12f /* 2^43 */;
    const bool g_ok = g >= kFastMin && g <= kFastMax;
    const bool all_in_range = g >= 1.0f / kMaxG && g <= kMaxG;
    const float Rg = g_ok ? __frcp_rn(g) : 1.0f;
    // fast_mode for the blocks all of whose codes, up to the first with D >= 4 a, lie below fast_end
    const float fast_below = fast_end == NC ? 3.402823466e38f : (fast_end >= 8 ? __fmul_rn(-0.25f, tab.nD[fast_end - 1]) : 0.0f);

    const size_t n_blocks = p.n_items;
    double sse_sum = 0.0;
    for (size_t tile0 = (size_t)blockIdx.x * tile_blocks; tile0 < n_blocks; tile0 += (size_t)gridDim.x * tile_blocks) {
        const int nb = (int)min((size_t)tile_blocks, n_blocks - tile0);
        [[maybe_unused]] float ahead[B];
        if constexpr (AHEAD) {
            if ((int)threadIdx.x < nb) load_elems<DT, B>(p.x, (tile0 + threadIdx.x) * B, ahead);
        }
        reinterpret_cast<uint4*>(hist)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();   // also: the previous tile has been read
        uint32_t place[Tile::NB / kThreads];   // bin << 16 | rank
        // ---- phase 1: load, two candidates, bounds -> mask of the codes that are left
#pragma unroll 1
        for (int kb = 0; kb < Tile::NB / kThreads; ++kb) {
            const int b = kb * kThreads + threadIdx.x;
            if (b >= nb) break;
            float a = 0.0f;
            float2 v2[NV];
            {
                float w[B];
                if constexpr (AHEAD) {
#pragma unroll
                    for (int i = 0; i < B; ++i) w[i] = ahead[i];
                    if (b + kThreads < nb) load_elems<DT, B>(p.x, (tile0 + b + kThreads) * B, ahead);   // this thread's next block
                } else {
                    load_elems<DT, B>(p.x, (tile0 + b) * B, w);
                }
#pragma unroll
                for (int i = 0; i < B; ++i) a = fmaxf(a, fabsf(w[i]));
                if constexpr (B == 2) {
                    *reinterpret_cast<float2*>(tile + b * 2) = make_float2(w[0], w[1]);
                } else {
#pragma unroll
                    for (int k = 0; k < B / 4; ++k)
                        *reinterpret_cast<float4*>(tile + Tile::piece(b, k)) = make_float4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
                }
                float2 w2[B / 2];
#pragma unroll
                for (int i = 0; i < B / 2; ++i) w2[i] = make_float2(w[2 * i], w[2 * i + 1]);
                hold<B>(w2, v2);
            }
            // a sum of squares over the elements f(v) keeps, in element order
            auto sum_of_squares = [&](auto f) {
                float s = 0.0f;
#pragma unroll
                for (int i = 0; i < B; ++i) {
                    const float x = f(element<B>(v2, i));
                    s = __fmaf_rn(x, x, s);
                }
                return s;
            };

            unsigned long long best = sse_key(__uint_as_float(0xFFFFFFFFu), first), m = 0;
            int base = 0, mode = kModeExact;
            if (a == 0.0f) {
                best = sse_key(0.0f, first);   // every code reproduces the zeros
            } else if (!(g_ok && a <= 1.44115188075855872e17f /* 2^57 */ && a >= 2.77555756156289135e-17f /* 2^-55 */)) {
                mode = kModeSlow;
            } else {
                const float u = __fmul_rn(a, Rg);
                const int c6 = max(round_scale<FMT>(__fmul_rn(u, 0.16666667f)), 1);
                const int c4 = max(round_scale<FMT>(__fmul_rn(u, 0.25f)), 1);
                if (a < fast_below) mode = fast_mode;
                float2 s;
                auto evaluate = [&](auto mode_tag) {
                    Candidates<DT, decltype(mode_tag)::value> c;
                    c.read(tab, c6, c4);
                    return sse_two_candidates<DT, B, decltype(mode_tag)::value>(v2, c);
                };
                if (mode == kModeExact) s = evaluate(std::integral_constant<int, kModeExact>{});
                else if (mode == kModeHalf) s = evaluate(std::integral_constant<int, kModeHalf>{});
                else if constexpr (DT == kBF16) s = evaluate(std::integral_constant<int, kModeChecked>{});
                best = min(sse_key(s.x, c6), sse_key(s.y, c4));
                uint32_t ubits = (uint32_t)(best >> 32);
                // r: sqrt(U) rounded up by more than every rounding below
                float r = __fmaf_rn(sqrt_approx(__uint_as_float(ubits)), 1.0009765625f, 2.168404344971009e-19f /* 2^-62 */);
                // zero rule; with r < a / 2 the all-zero quantization (at least a^2) cannot be the best
                if (!(r < 0.5f * a)) {
                    if (!all_in_range) mode = kModeSlow;
                    const int zc = first == 0 ? 0 : floor_code<FMT>(__fmul_rn(4.0f * kUp, u)) + 1;
                    if (zc < NC) best = min(best, sse_key(sum_of_squares([](float v) { return v; }), zc));
                    ubits = (uint32_t)(best >> 32);
                    r = __fmaf_rn(sqrt_approx(__uint_as_float(ubits)), 1.0009765625f, 2.168404344971009e-19f);
                }
                // low rule: D < (a - r) * 0.1665 leaves a - 6 D > r + (a - r) / 1000
                int lo = max(1, floor_code<FMT>(__fmul_rn(__fmul_rn(fmaxf(__fsub_rn(a, r), 0.0f), 0.1665f * kDown), Rg)));
                // high rule, with a second theta twice as large (both sums side by side)
                float limit = 4.0f * kUp;
                if constexpr (B >= 4) {
                    const float th8 = __fmul_rn(a, 0.125f), th4 = __fmul_rn(a, 0.25f);
                    float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int i = 0; i < B; ++i) {
                        const float v = element<B>(v2, i);
                        const float2 w = make_float2(fabsf(v) <= th8 ? v : 0.0f, fabsf(v) <= th4 ? v : 0.0f);
                        z = __ffma2_rn(w, w, z);
                    }
                    limit = __float_as_uint(z.x) > ubits ? 0.5f * kUp : (__float_as_uint(z.y) > ubits ? kUp : 4.0f * kUp);
                }
                const int hi = floor_code<FMT>(__fmul_rn(limit, u));
                bool windows = WINDOWS && r < 0.5f * a;
                if (hi - lo >= 64) {
                    // the low rule with all elements: those above 6 D' leave fl(|v| - 6 D') each
                    float d = __fmul_rn(-0.5f, tab.nD[hi]);
                    for (int k = 0; k < 32; ++k, d = __fmul_rn(d, 0.5f)) {
                        const float z = sum_of_squares([d](float v) { return fmaxf(__fmaf_rn(-6.0f, d, fabsf(v)), 0.0f); });
                        if (__float_as_uint(z) > ubits) {
                            lo = max(lo, floor_code<FMT>(__fmul_rn(__fmul_rn(d, Rg), kDown)));
                            break;
                        }
                    }
                    windows = false;
                }
                if (hi >= lo) {
                    if (hi - lo >= 64) {
                        mode = kModeSlow;
                    } else {
                        base = lo;
                        m = ~0ull >> (63 - (hi - lo));
                        if constexpr (WINDOWS) {
                            if (windows) {
                                // Counted in eighths of a binade from the code of 2^0 on, as the codes of the normal scales are.
                                constexpr int kOff = (127 - (FMT == kUE4M3 ? 7 : 15)) << 3;
                                const float rs = __fmul_rn(r, Rg), ul = __fsub_rn(u, rs), uh = __fadd_rn(u, rs);
                                // first and last code of the windows of q = 6 and q = 4, 2^-18 wider on either side
                                auto first_code = [&](float x) { return (int)((__float_as_uint(x) + 0xFFFFFu) >> 20) - kOff; };
                                auto last_code = [&](float x) { return (int)(__float_as_uint(x) >> 20) - kOff; };
                                constexpr float kW = 1.0f / 262144.0f;
                                const int l6 = first_code(__fmul_rn(ul, (1.0f - kW) / 6.0f)), h6 = last_code(__fmul_rn(uh, (1.0f + kW) / 6.0f));
                                const int l4 = first_code(__fmul_rn(ul, (1.0f - kW) / 4.0f)), h4 = last_code(__fmul_rn(uh, (1.0f + kW) / 4.0f));
                                // r < a / 2: a window reaches from u - r to u + r, a factor of at most 3 (1.6 binades), 14 codes
                                const uint32_t w6 = (1u << (h6 - l6 + 1)) - 1u, w4 = (1u << (h4 - l4 + 1)) - 1u;
                                const uint32_t p6 = w6 | (w6 << 8) | (w6 << 16);                       // q = 6, 3, 3/2
                                const unsigned long long p4 = (unsigned long long)(w4 >> 8) << 32 |    // q = 4, 2, 1, 1/2
                                                              (w4 | (w4 << 8) | (w4 << 16) | (w4 << 24));
                                const int v0 = lo >= 8 ? lo : l6;
                                unsigned long long w = shl64(p6, l6 - v0) | shl64(p4, l4 - v0);
                                if (lo < 8) {
                                    // the subnormal codes 1 .. 7 have the values of the eighths -16, -8, -4, 0, 2, 4, 6
                                    unsigned long long t = v0 <= 8 ? shr64(w, 8 - v0) << 8 : shl64(w, v0);
                                    t |= (shr64(w, -16 - v0) & 1ull) << 1 | (shr64(w, -8 - v0) & 1ull) << 2 | (shr64(w, -4 - v0) & 1ull) << 3;
                                    t |= (shr64(w, 0 - v0) & 1ull) << 4 | (shr64(w, 2 - v0) & 1ull) << 5;
                                    t |= (shr64(w, 4 - v0) & 1ull) << 6 | (shr64(w, 6 - v0) & 1ull) << 7;
                                    w = t >> lo;
                                }
                                m &= w;
                            }
                        }
                        // the two codes tried above
                        m &= ~(shl64(1ull, c6 - lo) | shl64(1ull, c4 - lo));
                    }
                }
            }
            key[b] = best;
            mask[b] = m;
            info[b] = (uint16_t)(base | (mode << 8));
            const uint32_t trips = mode == kModeSlow ? 127u : (uint32_t)(__popcll(m) + 1) / 2u;
            // eight bins per length keep the lanes' counter updates apart
            const uint32_t bin = trips * 8u + (threadIdx.x & 7u);
            place[kb] = bin << 16 | atomicAdd(&hist[bin], 1u);
        }
        __syncthreads();
        // ---- counting sort by list length: four bins per thread, a scan over the warps' totals
        {
            const uint4 h = reinterpret_cast<const uint4*>(hist)[threadIdx.x];
            const uint32_t mine = h.x + h.y + h.z + h.w;
            uint32_t incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if ((threadIdx.x & 31) >= o) incl += up;
            }
            if ((threadIdx.x & 31) == 31) warp_total[threadIdx.x >> 5] = incl;
            __syncthreads();
            uint32_t before = incl - mine;
            for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += warp_total[w];
            reinterpret_cast<uint4*>(hist)[threadIdx.x] = make_uint4(before, before + h.x, before + h.x + h.y, before + h.x + h.y + h.z);
        }
        __syncthreads();
#pragma unroll
        for (int kb = 0; kb < Tile::NB / kThreads; ++kb) {
            const int b = kb * kThreads + threadIdx.x;
            if (b < nb) perm[hist[place[kb] >> 16] + (place[kb] & 0xFFFFu)] = (uint16_t)b;
        }
        __syncthreads();
        {   // ask L2 for the next tile, one 128-byte line per thread and step
            const size_t next = tile0 + (size_t)gridDim.x * tile_blocks;
            if (next < n_blocks) {
                const char* const from = static_cast<const char*>(p.x) + next * B * elem_bytes(DT);
                const size_t bytes = min((size_t)tile_blocks, n_blocks - next) * B * elem_bytes(DT);
                for (size_t o = (size_t)threadIdx.x * 128; o < bytes; o += kThreads * 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(from + o));
            }
        }
        // ---- phase 2: the codes that are left, blocks in sorted order (every other round backwards, so that the rounds'
        // long lists do not all fall to the same warps)
#pragma unroll 1
        for (int kb = 0; kb < Tile::NB / kThreads; ++kb) {
            const int at = kb * kThreads + ((kb & 1) ? kThreads - 1 - (int)threadIdx.x : (int)threadIdx.x);
            if (at >= nb) continue;
            const int b = perm[at];
            const int mode = info[b] >> 8;
            if (mode == kModeSlow) {
                key[b] = search_tile_block<B>(tile, b, tab.nD, first, NC);
                continue;
            }
            const unsigned long long m64 = mask[b];
            if (m64 == 0) continue;
            float2 v2[NV];
            {
                float2 w2[B / 2];
                tile_pairs<B, B>(tile, b, 0, w2);
                hold<B>(w2, v2);
            }
            uint32_t best_bits = 0xFFFFFFFFu;
            int best_code = 0;
            // codes in descending order, an equal SSE replaces: the smallest code of a tie stays
            auto search = [&](auto mode_tag) {
                constexpr int MODE = decltype(mode_tag)::value;
                uint32_t m = (uint32_t)(m64 >> 32), next = (uint32_t)m64;
                int base = (info[b] & 0xFF) + 32;
                if (m == 0) { m = next; next = 0; base -= 32; }
                // the table entries of a trip are read one trip ahead
                int cA, cB;
                Candidates<DT, MODE> now;
                auto take_two = [&]() {
                    const int iA = 31 - __clz(m);
                    m ^= 1u << iA;
                    const int iB = m ? 31 - __clz(m) : iA;
                    m &= ~(1u << iB);
                    cA = base + iA;
                    cB = base + iB;
                    now.read(tab, cA, cB);
                };
                take_two();
                bool more;
                do {
                    const int kA = cA, kB = cB;
                    const Candidates<DT, MODE> use = now;
                    if (m == 0) { m = next; next = 0; base -= 32; }
                    more = m != 0;
                    if (more) take_two();
                    const float2 s = sse_two_candidates<DT, B, MODE>(v2, use);
                    keep_smaller_or_equal(best_bits, best_code, __float_as_uint(s.x), kA);
                    keep_smaller_or_equal(best_bits, best_code, __float_as_uint(s.y), kB);
                } while (more);
            };
            if (mode == kModeExact) search(std::integral_constant<int, kModeExact>{});
            else if (mode == kModeHalf) search(std::integral_constant<int, kModeHalf>{});
            else if constexpr (DT == kBF16) search(std::integral_constant<int, kModeChecked>{});
            key[b] = min(key[b], ((unsigned long long)best_bits << 32) | (unsigned)best_code);
        }
        __syncthreads();
        // ---- phase 3: encode with the winners; a unit is eight elements (8 / B blocks, or part of one)
        constexpr int UB = B < 8 ? 8 / B : 1;      // blocks per unit
        constexpr int PU = B < 8 ? 1 : B / 8;      // units per block
        const int units = (nb + UB - 1) / UB * PU;
        for (int un = threadIdx.x; un < units; un += kThreads) {
            const int blk0 = un / PU * UB;
            constexpr int N = B < 8 ? B : 8;           // elements of the unit in one block
            float v[8], D[UB], R[UB], R1[UB], t[8];
            uint32_t sc = 0;
            uint32_t sw[UB];
            bool fast = true, one_multiply = DT == kBF16;
#pragma unroll
            for (int j = 0; j < UB; ++j) {
                const int b = min(blk0 + j, nb - 1);
                const unsigned long long k = key[b];
                const int code = (int)(k & 0xFFu);
                D[j] = -tab.nD[code];
                R[j] = tab.R[code];
                const int mode = info[b] >> 8;
                fast &= R[j] != 0.0f && mode != kModeSlow;
                one_multiply &= mode == fast_mode && code < fast_end;
                if (DT == kBF16 && fast_mode == kModeChecked) R1[j] = tab.z[code];
                else R1[j] = R[j];
                sc |= (uint32_t)code << (8 * j);
                sw[j] = (uint32_t)(k >> 32);
                float2 v2[N / 2];
                tile_pairs<B, N>(tile, b, (un % PU) * 8, v2);
#pragma unroll
                for (int i = 0; i < N / 2; ++i) {
                    v[j * N + 2 * i] = v2[i].x;
                    v[j * N + 2 * i + 1] = v2[i].y;
                }
            }
            if (one_multiply) {
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = __fmul_rz(v[i], R1[i / N]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = quotient_corrected(v[i], D[i / N], R[i / N]);
            }
            if (!fast) {
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = quotient_general(v[i], D[i / N]);
            }
            const uint32_t packed = pack_e2m1x8(t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7]);
            const size_t gb = tile0 + blk0;
            if (blk0 + UB <= nb) {
                store_bytes<4>(p.codes + gb * (B / 2) + (un % PU) * 4, &packed);
                if (un % PU == 0) {
                    store_bytes<UB>(p.scales + gb, &sc);
                    if (p.block_sse) store_bytes<4 * UB>(p.block_sse + gb, sw);
                }
            } else {   // the tensor ends inside the unit (B = 2 and 4)
                store_whole_blocks<B>(p, gb, nb - blk0, packed, sc, sw);
            }
            if (un % PU == 0) {
#pragma unroll
                for (int j = 0; j < UB; ++j)
                    if (blk0 + j < nb) sse_sum = __dadd_rn(sse_sum, (double)__uint_as_float(sw[j]));
            }
        }
    }
    if (p.mse_partials != nullptr) {   // launch-uniform: fused tensor-MSE partial sum of this CTA
        __syncthreads();               // the tables are no longer read: their memory serves as scratch
        const double total = cta_sum_fixed_order(sse_sum, reinterpret_cast<double*>(&T));
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

// ------------------------------------------------------------------------------------------------
// The power-of-two format.  Codes are a factor of two apart, so the bounds leave two to four of them and there is nothing
// to sort: one thread searches its block in registers, from the two codes around a / 6 outwards.  Upwards to the
// limit of the high rule; downwards until the low rule holds (first for the largest element alone, then for all).
// Decode scales are formed from the code, D = g * 2^(c - 127) and 1 / D by the exponent, so there is no table to build.
// POW2: g is a power of two, so that a quotient is one exact multiply.
// ------------------------------------------------------------------------------------------------
template <int B, bool POW2>
__device__ __forceinline__ float2 pow2_sse_two(const float2 (&v2)[B / 2], float nDA, float RA, float nDB, float RB) {
    const float2 RA2 = make_float2(RA, RA), RB2 = make_float2(RB, RB);
    const float2 DA2 = make_float2(nDA, nDA), DB2 = make_float2(nDB, nDB);
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < B / 2; ++i) {
        const float2 tA = POW2 ? __fmul2_rn(v2[i], RA2) : quotient_pair(v2[i], DA2, RA2);
        const float2 tB = POW2 ? __fmul2_rn(v2[i], RB2) : quotient_pair(v2[i], DB2, RB2);
        const float2 e0 = residual_two_candidates<false>(tA.x, tB.x, v2[i].x, nDA, nDB, 0);
        s = __ffma2_rn(e0, e0, s);
        const float2 e1 = residual_two_candidates<false>(tA.y, tB.y, v2[i].y, nDA, nDB, 0);
        s = __ffma2_rn(e1, e1, s);
    }
    return s;
}

// value * 2^k for a normal value and a normal result
__device__ __forceinline__ float shifted(float value, int k) { return __uint_as_float(__float_as_uint(value) + ((uint32_t)k << 23)); }

// One block: its code, SSE bits and whether the shortcuts hold for it.
template <int B, bool POW2>
__device__ __forceinline__ unsigned long long pow2_search(const float2 (&v2)[B / 2], float g, float Rg, bool g_ok, bool& fast) {
    constexpr float kUp = 1.00000095367431640625f;   // 1 + 2^-20: above the rounding of a / g
    float a = 0.0f;
#pragma unroll
    for (int i = 0; i < B / 2; ++i) a = fmaxf(a, fmaxf(fabsf(v2[i].x), fabsf(v2[i].y)));
    fast = g_ok && a <= 1.44115188075855872e17f /* 2^57 */ && a >= 2.77555756156289135e-17f /* 2^-55 */;
    if (a == 0.0f) return sse_key(0.0f, 0);   // every code reproduces the zeros
    if (!fast) return search_by_division<B, B / 2>([g](int c) { return __fmul_rn(scale_value(kUE8M0, c), g); }, [&](int i) { return v2[i / 2]; }, a, 0, num_codes(kUE8M0));
    unsigned long long best = sse_key(__uint_as_float(0xFFFFFFFFu), 0);
    // a / g lies within [2^-98, 2^100]: every code below is far from either end of the format, and every D and 1 / D
    // within [2^-60, 2^60]
    const float u = __fmul_rn(a, Rg);
    const int c0 = (int)(__float_as_uint(__fmul_rn(u, 0.16666667f)) >> 23);
    const float nD0 = shifted(-g, c0 - 127), R0 = shifted(Rg, 127 - c0);
    auto try_two = [&](int k) {   // codes c0 + k, c0 + k + 1
        const float2 s = pow2_sse_two<B, POW2>(v2, shifted(nD0, k), shifted(R0, -k), shifted(nD0, k + 1), shifted(R0, -k - 1));
        best = min(best, min(sse_key(s.x, c0 + k), sse_key(s.y, c0 + k + 1)));
    };
    try_two(0);
    uint32_t ubits = (uint32_t)(best >> 32);
    float limit = 4.0f * kUp;
    if constexpr (B >= 4) {
        const float th8 = __fmul_rn(a, 0.125f), th4 = __fmul_rn(a, 0.25f);
        float2 z = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float v = (i & 1) ? v2[i / 2].y : v2[i / 2].x;
            const float2 w = make_float2(fabsf(v) <= th8 ? v : 0.0f, fabsf(v) <= th4 ? v : 0.0f);
            z = __ffma2_rn(w, w, z);
        }
        limit = __float_as_uint(z.x) > ubits ? 0.5f * kUp : (__float_as_uint(z.y) > ubits ? kUp : 4.0f * kUp);
    }
    const int hi = (int)(__float_as_uint(__fmul_rn(limit, u)) >> 23) - c0;   // every code above it is out
    for (int k = 2; k <= hi; k += 2) try_two(k);
    // zero rule: the smallest code with D >= 4 a; its SSE is at least a^2
    ubits = (uint32_t)(best >> 32);
    if (!(__float_as_uint(__fmul_rn(a, a)) > ubits)) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < B / 2; ++i) {
            s = __fmaf_rn(v2[i].x, v2[i].x, s);
            s = __fmaf_rn(v2[i].y, v2[i].y, s);
        }
        best = min(best, sse_key(s, (int)(__float_as_uint(__fmul_rn(4.0f * kUp, u)) >> 23) + 1));
    }
    for (int k = -1; c0 + k >= 0; --k) {
        const float nD = shifted(nD0, k), R = shifted(R0, -k);
        const float e = __fmaf_rn(6.0f, nD, a);
        if (e > 0.0f && __float_as_uint(__fmul_rn(e, e)) > ubits) break;
        float z = 0.0f;
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float x = fmaxf(__fmaf_rn(6.0f, nD, fabsf((i & 1) ? v2[i / 2].y : v2[i / 2].x)), 0.0f);
            z = __fmaf_rn(x, x, z);
        }
        if (__float_as_uint(z) > ubits) break;
        best = min(best, sse_key(pow2_sse_two<B, POW2>(v2, nD, R, nD, R).x, c0 + k));
    }
    return best;
}

template <int DT, int B>
__global__ void __launch_bounds__(kThreads) k_pruned_pow2(QuantArgs p) {
    constexpr int UE = B < 8 ? 8 : B;         // elements per thread and trip: one 32-bit word of codes at least
    constexpr int UB = UE / B;
    wait_for_prior_grid();
    release_dependents();
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const bool g_ok = g >= 2.2737367544323206e-13f /* 2^-42 */ && g <= 4.398046511104e12f /* 2^42 */;
    const float Rg = g_ok ? __frcp_rn(g) : 1.0f;
    const bool pow2 = (__float_as_uint(g) & 0x007FFFFFu) == 0u;
    const size_t n_units = (p.n_items + UB - 1) / UB;
    double sse_sum = 0.0;
    for (size_t un = (size_t)blockIdx.x * kThreads + threadIdx.x; un < n_units; un += (size_t)gridDim.x * kThreads) {
        const size_t blk = un * UB;
        const bool whole = blk + UB <= p.n_items;   // else the tensor ends inside the unit (B = 2 and 4)
        float v[UE];
        if (whole) {
            load_elems<DT, UE>(p.x, un * UE, v);
        } else {
#pragma unroll
            for (int i = 0; i < UE; ++i) v[i] = 0.0f;
#pragma unroll
            for (int j = 0; j < UB; ++j) {
                if (blk + j < p.n_items) {
                    float w[B];
                    load_elems<DT, B>(p.x, (blk + j) * B, w);
#pragma unroll
                    for (int i = 0; i < B; ++i) v[j * B + i] = w[i];
                }
            }
        }
        uint32_t packed[UE / 8];
        uint32_t sw[UB], sc = 0;
        float t[UE];
#pragma unroll
        for (int j = 0; j < UB; ++j) {
            float2 v2[B / 2];
#pragma unroll
            for (int i = 0; i < B / 2; ++i) v2[i] = make_float2(v[j * B + 2 * i], v[j * B + 2 * i + 1]);
            bool fast;
            const unsigned long long k = pow2 ? pow2_search<B, true>(v2, g, Rg, g_ok, fast) : pow2_search<B, false>(v2, g, Rg, g_ok, fast);
            const int code = (int)(k & 0xFFu);
            sw[j] = (uint32_t)(k >> 32);
            sc |= (uint32_t)code << (8 * j);
            if (fast) {
                const float D = shifted(g, code - 127), R = shifted(Rg, 127 - code);
#pragma unroll
                for (int i = 0; i < B; ++i) t[j * B + i] = quotient_corrected(v[j * B + i], D, R);
            } else {
                const float D = __fmul_rn(scale_value(kUE8M0, code), g);
#pragma unroll
                for (int i = 0; i < B; ++i) t[j * B + i] = quotient_general(v[j * B + i], D);
            }
        }
#pragma unroll
        for (int k = 0; k < UE / 8; ++k)
            packed[k] = pack_e2m1x8(t[8 * k], t[8 * k + 1], t[8 * k + 2], t[8 * k + 3], t[8 * k + 4], t[8 * k + 5], t[8 * k + 6], t[8 * k + 7]);
        if (whole) {
            store_bytes<UE / 2>(p.codes + un * (UE / 2), packed);
            store_bytes<UB>(p.scales + blk, &sc);
            if (p.block_sse) store_bytes<4 * UB>(p.block_sse + blk, sw);
        } else {
            store_whole_blocks<B>(p, blk, p.n_items - blk, packed[0], sc, sw);
        }
#pragma unroll
        for (int j = 0; j < UB; ++j)
            if (whole || blk + j < p.n_items) sse_sum = __dadd_rn(sse_sum, (double)__uint_as_float(sw[j]));
    }
    if (p.mse_partials != nullptr) {   // launch-uniform: fused tensor-MSE partial sum of this CTA
        __shared__ double scratch[kThreads / 32];
        const double total = cta_sum_fixed_order(sse_sum, scratch);
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

template <int DT, int B, int FMT>
static cudaError_t launch_pruned_inst(const QuantArgs& a, cudaStream_t stream) {
    static std::atomic<int> cache[kMaxDevices];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    size_t cap = 0;
    if constexpr (FMT == kUE8M0) {
        err = resident_ctas(reinterpret_cast<const void*>(k_pruned_pow2<DT, B>), 0, dev, cache, cap);
        if (err != cudaSuccess) return err;
        cap *= (size_t)sm_count(dev);
        if (a.mse_partials && cap > (size_t)kMsePartials) cap = kMsePartials;
        constexpr size_t UB = B < 8 ? 8 / B : 1;
        const size_t want = ((a.n_items + UB - 1) / UB + kThreads - 1) / kThreads;
        const unsigned grid = (unsigned)(want < cap ? want : cap);
        err = launch_pdl(k_pruned_pow2<DT, B>, grid, kThreads, 0, stream, a);
        count_launch();
        if (err == cudaSuccess && a.mse_n_partials) *a.mse_n_partials = (int)grid;
        return err;
    } else {
        using Tile = PrunedTile<B>;
        err = resident_ctas(reinterpret_cast<const void*>(k_pruned<DT, B, FMT>), Tile::BYTES, dev, cache, cap);
        if (err != cudaSuccess) return err;
        cap *= (size_t)sm_count(dev);
        if (a.mse_partials && cap > (size_t)kMsePartials) cap = kMsePartials;
        // Tensors too small to give every resident CTA a full tile are cut into smaller ones (a multiple of 32 blocks,
        // so that every tile starts on a 16-byte boundary of each output).
        size_t tile = (a.n_items + cap - 1) / cap;
        tile = (tile + 31) / 32 * 32;
        if (tile > (size_t)Tile::NB) tile = Tile::NB;
        const size_t want = (a.n_items + tile - 1) / tile;
        const unsigned grid = (unsigned)(want < cap ? want : cap);
        err = launch_pdl(k_pruned<DT, B, FMT>, grid, kThreads, Tile::BYTES, stream, a, (int)tile);
        count_launch();
        if (err == cudaSuccess && a.mse_n_partials) *a.mse_n_partials = (int)grid;
        return err;
    }
}

template <int DT, int B>
static cudaError_t launch_pruned_fmt(const QuantArgs& a, int fmt, cudaStream_t s) {
    switch (fmt) {
    case kUE8M0: return launch_pruned_inst<DT, B, kUE8M0>(a, s);
    case kUE4M3: return launch_pruned_inst<DT, B, kUE4M3>(a, s);
    default: return launch_pruned_inst<DT, B, kUE5M3>(a, s);
    }
}

template <int DT>
static cudaError_t launch_pruned_dt(const QuantArgs& a, int B, int fmt, cudaStream_t s) {
    switch (B) {
    case 2: return launch_pruned_fmt<DT, 2>(a, fmt, s);
    case 4: return launch_pruned_fmt<DT, 4>(a, fmt, s);
    case 8: return launch_pruned_fmt<DT, 8>(a, fmt, s);
    case 16: return launch_pruned_fmt<DT, 16>(a, fmt, s);
    case 32: return launch_pruned_fmt<DT, 32>(a, fmt, s);
    default: return launch_pruned_fmt<DT, 64>(a, fmt, s);
    }
}

}  // namespace mxq
