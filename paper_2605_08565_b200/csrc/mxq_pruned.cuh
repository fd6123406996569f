// Pruned scale search (MXQ_OPT_BRUTE_PRUNE): the brute-force recipes with the codes left out that provably cannot change
// an output, decided BLOCK BY BLOCK.  Outputs are those of the full sweep (mxq_brute.cuh), bit for bit.
//
// With e = fma(q, -D, v), s = fma(e, e, s) in element order and round-to-nearest, which is monotone, an SSE never
// decreases when the magnitude of an error grows, so the rules below hold in the very arithmetic of the SSE.  a = max |v|.
//   halving rule 7 D > a: the code with 2 D (eight codes up in the FP8 formats, one in UE8M0) is never better.  The FP4 grid times 2 D
//                is part of the grid times D but for 8 D and 12 D, which are nearest only to magnitudes above 7 D, so every
//                element's error under 2 D is at least its error under D; and a tie goes to the smaller code, D.  In binary32: 2 D is exact, so
//                fl(v / 2D) = fl(v / D) / 2; a quotient rounded onto the midpoint of two grid values goes to the even one of
//                the FP4 grid under D and under 2 D to the same point (1.25, 1.75, 2.5, 3.5, 5 go to 1, 2, 2, 4, 4), so that the point
//                under 2 D is never the nearer one.  What is left lies below 2 a / 7, whatever the block holds.
//                Codes below 16 of the FP8 formats are the multiples 1 .. 15 of the smallest scale: the even ones have a
//                half among them, the odd ones have none.
//   low rule     6 D <= a: the largest element saturates and leaves fl(a - 6 D); once that alone (or what all saturated
//                elements leave) costs more than the best SSE so far, this and every smaller D is out.
//   high rule    (odd codes below 16) the elements with 4 |v| <= D go to zero; once they alone cost more, every larger D is out.
// The search runs downwards from the largest code with D <= 2 a / 7: eight codes reach a / 6.4, and few blocks need a ninth (B <= 8: one
// in a hundred; B = 64: two more on average), so the lanes of a warp finish together with a block each in registers, no lists
// and no tables of codes left.  Bound by issue slots: FP4 pack and unpack, quotients, residuals.
//
// Measured against lists of the codes that bounds from the best of two probes left (9 to 17 a block), evaluated in the order of their
// length after a sort in shared memory; 16.8 M elements, us before -> now:
//   fp32 Laplace, tensor scale, UE4M3   B = 2 186 -> 62    4 124 -> 52   8 107 -> 48   16 109 -> 53   32 123 -> 54   64 145 -> 60
//   bf16 Student-t, UE5M3               B = 2 205 -> 60    4 128 -> 43   8 99 -> 37    16 92 -> 36    32 92 -> 34    64 106 -> 38
//   bf16 Student-t, UE4M3 (scale codes below 16)
//                                       B = 2 218 -> 118   4 127 -> 84   8 91 -> 68    16 79 -> 52    32 80 -> 48    64 97 -> 51
//   bf16 Student-t, UE8M0               B = 2 64 -> 36     4 51 -> 28    8 40 -> 21    16 31 -> 16    32 25 -> 15    64 27 -> 18
// 65 K elements, B = 16, 8.0 -> 4.8.
#pragma once

#include <atomic>

#include "mxq_brute.cuh"
#include "mxq_quantize.cuh"

namespace mxq {

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

// How candidates are evaluated.  kModeExact: corrected quotient, binary32 residual; holds for every decode scale in [2^-60,
// 2^60].  kModeHalf: -D is exact in f16 (and for bf16 input D has at most four significant bits, so that the quotient is one
// multiply rounded toward zero).  kModeChecked (bf16): the one-multiply quotient with the reciprocal that
// build_quant_tables() checked.
// kModeAny: a loop whose blocks choose.
enum { kModeExact = 0, kModeHalf = 1, kModeChecked = 2, kModeAny = 3 };

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

// What an evaluation needs of two candidates (.x, .y).  The table holds for code c what the pair c, c - 1 takes: -D of
// the two, then their reciprocals (RN(1 / D), or the checked one of the launch), in the register pairs of the packed
// instructions: one 128-bit read.  Codes below 1 stand for code 1, down to the last that the eight codes from any first one on reach.
constexpr int kLeadIn = 8;   // entries before that of code 0
template <int DT, int MODE>
struct Candidates {
    static constexpr bool ONE_MULTIPLY = (DT == kBF16) && MODE != kModeExact;
    float2 nD, R;
    uint32_t nD16;   // kModeHalf: f16(-D) of the two
    __device__ __forceinline__ void set(float nDA, float nDB, float RA, float RB) {
        nD = make_float2(nDA, nDB);
        R = make_float2(RA, RB);
        nD16 = 0;
        if constexpr (MODE == kModeHalf) {
            const __half2 h = __floats2half2_rn(nDA, nDB);
            nD16 = *reinterpret_cast<const uint32_t*>(&h);
        }
    }
    __device__ __forceinline__ void read_down(const float4* tab, int c) {   // c, c - 1
        const float4 P = tab[c];
        set(P.x, P.y, P.z, P.w);
    }
    __device__ __forceinline__ void read(const float4* tab, int cA, int cB) { set(tab[cA].x, tab[cB].x, tab[cA].z, tab[cB].z); }
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

__device__ __forceinline__ void keep_smaller_or_equal(uint32_t& best_bits, int& best_code, uint32_t bits, int code) {
    best_code = bits <= best_bits ? code : best_code;
    best_bits = min(best_bits, bits);
}

// The first code of a format that is twice another one, and how many codes lie between the two.
__host__ __device__ constexpr int first_halved(int fmt) { return fmt == kUE8M0 ? 1 : 16; }
__host__ __device__ constexpr int halving_step(int fmt) { return fmt == kUE8M0 ? 1 : 8; }

// A block outside the ranges of the shortcuts, with IEEE division: the best (SSE bits, code) among codes first .. num_codes - 1.
// decode(c): the decode scale, nondecreasing in c; pair(i): elements i and i + 1; a: the largest magnitude.  Codes are taken upwards from
// the first with 6 D >= a, then downwards from there, until
//   upwards     the halving rule covers the next code (its half a normal number: the double is exact); or D >= 4 a: this and
//               every larger D has the SSE of the all-zero quantization (ties go to the smaller code); or the high rule holds;
//   downwards   the low rule holds for all saturated elements together.
// The sums compared are taken in the order and arithmetic of the SSE.  Magnitudes of 1e-20 under their tensor scale, 4.2 M elements:
// the codes that bounds left 192 us for UE4M3 at B = 16 (fp32) and 334 for UE5M3 at B = 2 (bf16), here 69 and 113.
template <int FMT, int B, typename Decode, typename Pair>
__device__ __forceinline__ unsigned long long search_by_division(Decode decode, Pair pair, float a, int first) {
    constexpr int n_codes = num_codes(FMT);
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
#pragma unroll 1
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
        bool rest_is_out = __float_as_uint(z) > (uint32_t)(best >> 32);
        if (up) {
            rest_is_out |= D >= __fmul_rn(4.0f, a);
            if (c + 1 >= first_halved(FMT)) {
                const float half = decode(c + 1 - halving_step(FMT));
                rest_is_out |= half >= 1.17549435e-38f && __fmul_rn(7.0f, half) > __fmul_rn(a, 1.00000095367431640625f);
            }
        }
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

// The same for block blk of the tensor, read again; out of line, to leave the registers of the search proper alone.
template <int DT, int B, int FMT>
__device__ __noinline__ unsigned long long search_block_by_division(const void* x, size_t blk, float a, float g, int first) {
    auto pair = [&](int i) {
        float v[2];
        load_elems<DT, 2>(x, blk * B + i, v);
        return make_float2(v[0], v[1]);
    };
    return search_by_division<FMT, B>([g](int c) { return __fmul_rn(scale_value(FMT, c), g); }, pair, a, first);
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

// Where a thread starts: sets of 32 units go round the CTAs before they go round a CTA's warps, so that a small tensor is spread over
// all SMs.
__device__ __forceinline__ size_t pruned_first_unit() {
    return ((size_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
}

// What a CTA knows before it searches.
struct PrunedConsts {
    float g, Rg;          // tensor scale and RN(1 / g)
    int first;            // smallest admissible code
    float a_lo, a_hi;     // largest magnitudes for which the shortcuts hold
};

// One block under the codes that the rules leave: the largest code with D <= 2 a / 7, `top` (0: none), and the seven below it, further down
// while the low rule allows; where top is below 15, the odd codes above it up to 15 that the high rule and the largest element leave
// (some grid value has to bring q D as near to it as the best SSE so far).  u = a / g.  False: a decode scale is out of range, the block
// has to be divided.
template <int DT, int B, int FMT, int MODE>
__device__ __forceinline__ bool search_codes(const float4* tab, const float2 (&v)[pruned_values(B)], float a, float u, int top,
                                             const PrunedConsts& k, uint32_t& best_bits, int& best_code) {
    constexpr int kMain = 4;   // pairs of codes that are always tried: the seventh code below top is the first with D < a / 6
    constexpr float kUp = 1.00000095367431640625f;
    best_bits = 0xFFFFFFFFu;
    auto sum_of_squares = [&](auto f) {   // over the elements f(|v|) keeps, in element order
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float x = f(fabsf(element<B>(v, i)));
            s = __fmaf_rn(x, x, s);
        }
        return s;
    };
    Candidates<DT, MODE> c2;
    {
        int at = 0;   // the best code is `at` below top; in descending order an equal SSE replaces: the smallest code of a tie stays
#pragma unroll (B <= 16 ? kMain : 1)
        for (int i = 0; i < kMain; ++i) {
            c2.read_down(tab, top - 2 * i);
            const float2 s = sse_two_candidates<DT, B, MODE>(v, c2);
            keep_smaller_or_equal(best_bits, at, __float_as_uint(s.x), 2 * i);
            keep_smaller_or_equal(best_bits, at, __float_as_uint(s.y), 2 * i + 1);
        }
        best_code = max(top - at, 1);   // code 1 again and again at the end
    }
    {   // nearly every block ends here: no code below can be better, and there is none above
        const float e = __fmaf_rn(6.0f, tab[top - 2 * kMain].x, a);
        if (top >= 16 && e > 0.0f && __float_as_uint(__fmul_rn(e, e)) > best_bits) return true;
    }
    bool in_range = true, stopped = false;
#pragma unroll 1
    for (int c = top - 2 * kMain; c >= 1 && !stopped; c -= 2) {
        c2.read_down(tab, c);
        const float nD = c2.nD.x;
        const float e = __fmaf_rn(6.0f, nD, a);
        stopped = e > 0.0f && __float_as_uint(__fmul_rn(e, e)) > best_bits;
        if (!stopped) {
            const float z = sum_of_squares([nD](float m) { return fmaxf(__fmaf_rn(6.0f, nD, m), 0.0f); });
            in_range = c2.R.x != 0.0f && c2.R.y != 0.0f;
            stopped = __float_as_uint(z) > best_bits || !in_range;
        }
        if (!stopped) {
            const float2 s = sse_two_candidates<DT, B, MODE>(v, c2);
            keep_smaller_or_equal(best_bits, best_code, __float_as_uint(s.x), c);
            keep_smaller_or_equal(best_bits, best_code, __float_as_uint(s.y), max(c - 1, 1));
        }
    }
    if (k.first == 0 && !(__float_as_uint(__fmul_rn(a, a)) > best_bits))   // code 0: all elements to zero
        keep_smaller_or_equal(best_bits, best_code, __float_as_uint(sum_of_squares([](float m) { return m; })), 0);
    if (top < 15) {
        // the odd codes up to the first with D >= 4 a (4 kUp u), under which every element goes to zero; less where the elements up to
        // a / 4 or a / 8 alone cost too much
        float limit = 4.0f * kUp;
        if constexpr (B >= 4) {
            const float th8 = __fmul_rn(a, 0.125f), th4 = __fmul_rn(a, 0.25f);
            const float z8 = sum_of_squares([th8](float m) { return m <= th8 ? m : 0.0f; });
            const float z4 = sum_of_squares([th4](float m) { return m <= th4 ? m : 0.0f; });
            limit = __float_as_uint(z8) > best_bits ? 0.5f * kUp : (__float_as_uint(z4) > best_bits ? kUp : 4.0f * kUp);
        }
        const int end = min(15, floor_code<FMT>(__fmul_rn(u, limit)) + (limit > 2.0f ? 1 : 0));
        in_range &= tab[1].z != 0.0f;
        uint32_t left = 0;
        const int begin = (max(top, 1) + 1) | 1;
        if constexpr (B <= 4) {   // so few elements are evaluated in less than the largest takes to be looked at
            left = (0xAAAAu >> begin << begin) & ((2u << max(end, 0)) - 1u);
        } else {
#pragma unroll 1
            for (int c = begin; c <= end; c += 2) {
                const float nD = tab[c].x;   // a rounded product: next to a midpoint of the grid the error of either side is the same to 2^-16
                const float e = __fmaf_rn(round_widen_pair(make_float2(__fmul_rn(a, tab[c].z), 0.0f)).x, nD, a);
                if (!(__float_as_uint(__fmul_rn(__fmul_rn(e, 0.999f), e)) > best_bits)) left |= 1u << c;
            }
        }
#pragma unroll 1
        while (left != 0) {
            const int cA = __ffs(left) - 1;
            left &= left - 1;
            const int cB = left != 0 ? __ffs(left) - 1 : cA;
            left &= left - 1;
            c2.read(tab, cA, cB);
            const float2 s = sse_two_candidates<DT, B, MODE>(v, c2);
            keep_smaller(best_bits, best_code, __float_as_uint(s.x), cA);
            keep_smaller(best_bits, best_code, __float_as_uint(s.y), cB);
        }
    }
    return in_range;
}

// Resident CTAs per SM asked of the register allocator (a block is held in registers through the search).
__host__ __device__ constexpr int pruned_min_ctas(int B) { return B <= 16 ? 4 : B == 32 ? 3 : 2; }

// One thread searches a unit of eight elements (B < 8: two or four blocks) or one block.
template <int DT, int B, int FMT>
__global__ void __launch_bounds__(kThreads, pruned_min_ctas(B)) k_pruned(QuantArgs p) {
    static_assert(FMT != kUE8M0, "the power-of-two format has its own kernel");
    constexpr int UE = B < 8 ? 8 : B;
    constexpr int UB = UE / B;
    constexpr int NC = num_codes(FMT);
    constexpr float kUp = 1.00000095367431640625f;   // 1 + 2^-20: above the rounding of a / g
    __shared__ QuantTables T;
    __shared__ float4 pair_table[kLeadIn + 256];
    const float4* const tab = pair_table + kLeadIn;
    __shared__ int short_end;   // f32: first code whose -D is not exact in f16

    wait_for_prior_grid();
    release_dependents();
    PrunedConsts k;
    k.g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    k.first = p.prevent_zero ? 1 : 0;
    if (threadIdx.x == 0) short_end = NC;
    int first_bad;
    const bool checked = build_quant_tables<FMT, DT == kBF16>(T, k.g, first_bad);   // barriers inside
    for (int c = (int)threadIdx.x - kLeadIn; c < 256; c += kThreads) {
        const float4 E = T.E[max(c, 1)], F = T.E[max(c - 1, 1)];
        pair_table[c + kLeadIn] = make_float4(-E.x, -F.x, checked ? E.z : E.y, checked ? F.z : F.y);
        if (DT == kF32 && c >= 0 && c < NC && T.E[c].w < 2.0f) atomicMin(&short_end, c);
    }
    __syncthreads();
    const int fast_mode = checked ? kModeChecked : kModeHalf;
    const int fast_end = checked ? NC : (DT == kF32 ? short_end : first_bad);   // codes below it may be evaluated in fast_mode
    const bool g_ok = k.g >= kFastMin && k.g <= kFastMax;
    k.Rg = g_ok ? __frcp_rn(k.g) : 1.0f;
    k.a_lo = g_ok ? 2.77555756156289135e-17f /* 2^-55 */ : 1.0f;
    k.a_hi = g_ok ? 1.44115188075855872e17f /* 2^57 */ : 0.0f;   // no block at all
    // the launch's mode; a block whose codes reach beyond its end is evaluated exactly
    const int main_mode = fast_end >= 64 ? fast_mode : kModeExact;
    const int top_end = main_mode == kModeExact ? NC : fast_end;

    const size_t n_units = (p.n_items + UB - 1) / UB;
    double sse_sum = 0.0;
    auto unit_loop = [&](auto mode_tag) {
        constexpr int MODE = decltype(mode_tag)::value;
        for (size_t un = pruned_first_unit(); un < n_units; un += (size_t)gridDim.x * kThreads) {
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
                float a = 0.0f;
#pragma unroll
                for (int i = 0; i < B; ++i) a = fmaxf(a, fabsf(v[j * B + i]));
                uint32_t bits = 0;
                int code = k.first;   // a block of zeros: every code reproduces it
                bool divide = false, one_multiply = false;
                if (a >= k.a_lo && a <= k.a_hi) {
                    float2 vh[pruned_values(B)];
                    {
                        float2 w2[B / 2];
#pragma unroll
                        for (int i = 0; i < B / 2; ++i) w2[i] = make_float2(v[j * B + 2 * i], v[j * B + 2 * i + 1]);
                        hold<B>(w2, vh);
                    }
                    const float u = __fmul_rn(a, k.Rg);
                    const int top = floor_code<FMT>(__fmul_rn(u, 0.2857142857f * kUp));
                    auto search = [&](auto tag) {
                        constexpr int M = decltype(tag)::value;
                        divide = !search_codes<DT, B, FMT, M>(tab, vh, a, u, top, k, bits, code);
                        one_multiply = DT == kBF16 && M != kModeExact;
                    };
                    const int mode = top < top_end ? (MODE == kModeAny ? main_mode : MODE) : kModeExact;
                    if (mode == kModeExact) search(std::integral_constant<int, kModeExact>{});
                    else if (MODE == kModeHalf || (MODE == kModeAny && mode == kModeHalf)) search(std::integral_constant<int, kModeHalf>{});
                    else if constexpr (DT == kBF16 && (MODE == kModeChecked || MODE == kModeAny)) search(std::integral_constant<int, kModeChecked>{});
                } else {
                    divide = a != 0.0f;
                }
                if (divide) {
                    const unsigned long long key = search_block_by_division<DT, B, FMT>(p.x, blk + j, a, k.g, k.first);
                    bits = (uint32_t)(key >> 32);
                    code = (int)(key & 0xFFu);
                }
                sw[j] = bits;
                sc |= (uint32_t)code << (8 * j);
                // encode with the winner
                const float4 E = T.E[code];
                if (divide || E.y == 0.0f) {
#pragma unroll
                    for (int i = 0; i < B; ++i) t[j * B + i] = quotient_general(v[j * B + i], E.x);
                } else if (one_multiply) {
                    const float R = tab[code].z;
#pragma unroll
                    for (int i = 0; i < B; ++i) t[j * B + i] = __fmul_rz(v[j * B + i], R);
                } else {
#pragma unroll
                    for (int i = 0; i < B; ++i) t[j * B + i] = quotient_corrected(v[j * B + i], E.x, E.y);
                }
            }
#pragma unroll
            for (int w = 0; w < UE / 8; ++w)
                packed[w] = pack_e2m1x8(t[8 * w], t[8 * w + 1], t[8 * w + 2], t[8 * w + 3], t[8 * w + 4], t[8 * w + 5], t[8 * w + 6], t[8 * w + 7]);
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
    };
    // a loop for the launch's mode pays for short blocks, whose tests and branches weigh (16.8 M elements, us: fp32, tensor scale, B = 2 76 -> 62, 4 57 ->
    // 52, 8 50 -> 48; bf16, UE5M3, 72 -> 60, 49 -> 43, 38 -> 37); B = 32 lost 1 % on small tensors
    if constexpr (B > 8) unit_loop(std::integral_constant<int, kModeAny>{});
    else if (main_mode == kModeExact) unit_loop(std::integral_constant<int, kModeExact>{});
    else if (main_mode == kModeHalf) unit_loop(std::integral_constant<int, kModeHalf>{});
    else if constexpr (DT == kBF16) unit_loop(std::integral_constant<int, kModeChecked>{});
    if (p.mse_partials != nullptr) {   // launch-uniform: fused tensor-MSE partial sum of this CTA
        __syncthreads();               // the tables are no longer read: their memory serves as scratch
        const double total = cta_sum_fixed_order(sse_sum, reinterpret_cast<double*>(&T));
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

// ------------------------------------------------------------------------------------------------
// The power-of-two format.  Codes are a factor of two apart: the halving rule leaves the two codes around a / 6, and downwards the
// low rule (first for the largest element alone, then for all) nearly always holds at once.  Decode scales are formed from
// the code, D = g * 2^(c - 127) and 1 / D by the exponent, so there is no table to build.
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
template <int DT, int B, bool POW2>
__device__ __forceinline__ unsigned long long pow2_search(const float2 (&v2)[B / 2], const void* x, size_t blk, float g, float Rg, bool g_ok, bool& fast) {
    float a = 0.0f;
#pragma unroll
    for (int i = 0; i < B / 2; ++i) a = fmaxf(a, fmaxf(fabsf(v2[i].x), fabsf(v2[i].y)));
    fast = g_ok && a <= 1.44115188075855872e17f /* 2^57 */ && a >= 2.77555756156289135e-17f /* 2^-55 */;
    if (a == 0.0f) return sse_key(0.0f, 0);   // every code reproduces the zeros
    if (!fast) return search_block_by_division<DT, B, kUE8M0>(x, blk, a, g, 0);
    unsigned long long best = sse_key(__uint_as_float(0xFFFFFFFFu), 0);
    // a / g lies within [2^-116, 2^118]: every code below is far from either end of the format.  So are D and 1 / D, which lie about a / 6
    // whatever g is: the low rule holds for all elements together before D falls to a / 2^11 (B = 64).
    const float u = __fmul_rn(a, Rg);
    const int c0 = (int)(__float_as_uint(__fmul_rn(u, 0.16666667f)) >> 23);
    const float nD0 = shifted(-g, c0 - 127), R0 = shifted(Rg, 127 - c0);
    auto try_two = [&](int k) {   // codes c0 + k, c0 + k + 1
        const float2 s = pow2_sse_two<B, POW2>(v2, shifted(nD0, k), shifted(R0, -k), shifted(nD0, k + 1), shifted(R0, -k - 1));
        best = min(best, min(sse_key(s.x, c0 + k), sse_key(s.y, c0 + k + 1)));
    };
    // 2^c0 <= a / 6g < 2^(c0 + 1), to within the rounding: code c0 + 2 and all above it are beyond 2 a / 7
    try_two(0);
    const uint32_t ubits = (uint32_t)(best >> 32);
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
        if (ubits > 0x7F800000u) {   // a NaN element: so is every SSE, no rule ends the search, and the codes it would end at are out of the shortcuts' range
            fast = false;
            return sse_key(__uint_as_float(ubits), 0);
        }
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
    const bool g_ok = g >= kFastMin && g <= kFastMax;
    const float Rg = g_ok ? __frcp_rn(g) : 1.0f;
    const bool pow2 = (__float_as_uint(g) & 0x007FFFFFu) == 0u;
    const size_t n_units = (p.n_items + UB - 1) / UB;
    double sse_sum = 0.0;
    for (size_t un = pruned_first_unit(); un < n_units; un += (size_t)gridDim.x * kThreads) {
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
            const unsigned long long k = pow2 ? pow2_search<DT, B, true>(v2, p.x, blk + j, g, Rg, g_ok, fast) : pow2_search<DT, B, false>(v2, p.x, blk + j, g, Rg, g_ok, fast);
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
        // full CTAs, but one on every SM as long as there are warps for it (bf16, B = 8, us, full CTAs -> spread over one per SM -> one
        // warp a CTA: 65 K elements 3.6 -> 3.4 -> 3.4, 262 K 3.2 -> 3.2 -> 3.6)
        const size_t sets = ((a.n_items + UB - 1) / UB + 31) / 32, full = (sets + kThreads / 32 - 1) / (kThreads / 32), sms = (size_t)sm_count(dev);
        const size_t want = full > sms ? full : (sets < sms ? sets : sms);
        const unsigned grid = (unsigned)(want < cap ? want : cap);
        err = launch_pdl(k_pruned_pow2<DT, B>, grid, kThreads, 0, stream, a);
        count_launch();
        if (err == cudaSuccess && a.mse_n_partials) *a.mse_n_partials = (int)grid;
        return err;
    } else {
        err = resident_ctas(reinterpret_cast<const void*>(k_pruned<DT, B, FMT>), 0, dev, cache, cap);
        if (err != cudaSuccess) return err;
        cap *= (size_t)sm_count(dev);
        if (a.mse_partials && cap > (size_t)kMsePartials) cap = kMsePartials;
        constexpr size_t UB = B < 8 ? 8 / B : 1;
        const size_t want = ((a.n_items + UB - 1) / UB + 31) / 32;   // one set of 32 units each before a CTA takes a second
        const unsigned grid = (unsigned)(want < cap ? want : cap);
        err = launch_pdl(k_pruned<DT, B, FMT>, grid, kThreads, 0, stream, a);
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
