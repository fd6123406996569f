// Brute-force scale search (Experimental Setup: the optimal baseline, found by trying the possible
// scale values and keeping the one with the least error): every finite scale code of the format
// is tried on every block and the code with the smallest SSE is kept (equal SSE: the smaller code).
//
// Work layout.  A thread keeps its elements in registers as float pairs and the candidate loop
// works on float pairs with the packed binary32 instructions of sm_100 (fma.rn.f32x2 /
// mul.rn.f32x2, FP4 pack and unpack two at a time):
//   B <= 16   the thread owns G = 32 consecutive elements (16 for B = 2), pair i = (element i,
//             element G/2 + i): the two halves of a pair belong to different blocks, so one instruction serves two
//             elements of one candidate and the two SSE chains are independent.  Two candidates
//             per trip.
//   B >= 32   the thread owns one block, pair i = (element 2i, element 2i + 1).  Its SSE is one
//             sequential chain over all elements, so the two lanes of the SSE pair are two
//             CANDIDATES: the scaling multiplies run on element pairs, the FP4 rounding and the
//             residuals on candidate pairs of one element, and the elements are walked in order.
// The candidate loop is uniform across the CTA: decode scales come from shared memory as
// broadcasts.
//
// One exact quotient per mantissa, not per candidate.  The decode scale of code c is
// D_c = fl(S_c * g).  All codes whose S_c share a mantissa (eight classes for the FP8 scale
// formats, one for the power-of-two format) have decode scales that differ by exact powers of two,
// D_c = Dref * 2^k, as long as D_c is a normal number.  Hence fl(v / D_c) = fl(v / Dref) * 2^-k
// exactly: the correctly rounded quotient is formed once per class and element, and a candidate
// costs one multiply by a power of two, the FP4 rounding, and the two FMAs of the SSE.  Codes
// whose decode scale is zero, subnormal or above 2^126 need no quotient at all (every element
// rounds to zero, or saturates) and form one more list.  Threads holding a magnitude above 2^60
// or a nonzero one below 2^-62 take the general path (IEEE division), candidate by candidate.
//
// Inside a class the members are visited in ascending code order and the smallest SSE bit pattern
// is kept with a strict compare (SSE >= 0, so integer order is float order and the first of equals
// is the smaller code); class winners are merged as 64-bit keys (SSE bits << 32 | code).
#pragma once

#include <atomic>

#include "mxq_device.cuh"
#include "mxq_internal.h"

namespace mxq {

constexpr int kMaxMembers = 36;  // codes per mantissa class, FP8 formats (31 normal + 3 subnormal at most)

// Mantissa class of a scale code: index of the 3-bit mantissa of its value.
template <int FMT>
__device__ __forceinline__ int code_class(int c) {
    if constexpr (FMT == kUE8M0) return 0;
    if (c >= 8) return c & 7;
    // subnormal codes m * 2^(1-bias-3): 1, 2, 4 -> 1.0; 3, 6 -> 1.5; 5 -> 1.25; 7 -> 1.75
    return (int)((0x64204000u >> (4 * c)) & 7u);
}

// Per-CTA tables of the search.  Every code with a finite decode scale D sits in one candidate list:
//   * D normal with a biased exponent of at most 253 ("paired": D = Dref * 2^k and 2^-k are both
//     representable): list 2 * class + kind, where kind 1 holds the codes whose -D is exactly
//     representable in f16 (their residual is one mixed-precision FMA from the unpacked f16 grid
//     value) and kind 0 the others (f16 -> f32 convert, then an FFMA);
//   * the "flat" list kFlatList for the rest.  D = 0 or D >= 2^127: every quotient of a magnitude
//     <= 2^60 rounds to FP4 zero, so the candidate is entered with the multiplier 0.  D subnormal:
//     every nonzero magnitude >= 2^-62 divided by it exceeds 2^64 and saturates at 6, so it is
//     entered with the multiplier 2^126.  The flat list is evaluated on the elements themselves
//     (Dref = 1), which needs no quotient.
constexpr int kLists = 17;
constexpr int kFlatList = 16;
constexpr int kCandSlots = 16 * kMaxMembers + 256;
struct BruteTables {
    float D[256];            // decode scale of the code; NaN for codes that do not exist
    float R[256];            // RN(1 / D) when 2^-60 <= D <= 2^60, else 0 (used by the final encode)
    float4 cand[kCandSlots];    // per list, ascending code order: (-D, multiplier, f16(-D) twice as bits, 0)
    uint8_t member[kCandSlots]; // the code of each slot of cand[]
    uint8_t kind[256];       // 0, 1 paired as above; 3 = flat list; 2 = not a candidate
    float clsD[8];           // Dref of the class, in [1, 2)
    float clsR[8];           // RN(1 / Dref)
    int cnt[kLists];         // members per list
    uint32_t kind_mask[3][8];
};

template <int FMT>
__device__ __forceinline__ int members_base(int list) {
    if (list == kFlatList) return 16 * kMaxMembers;
    // the power-of-two format has one class: its two lists get half of the class area each
    return FMT == kUE8M0 ? list * (16 * kMaxMembers / 2) : list * kMaxMembers;
}

// first: smallest admissible code (1 under prevent-zero for the FP8 formats, else 0).
template <int FMT>
__device__ __forceinline__ void build_brute_tables(BruteTables& T, float g, int first) {
    static_assert(kThreads == 256, "one thread per table entry");
    build_scale_tables<FMT>(T.D, T.R, g);
    const int c = threadIdx.x;
    const float D = T.D[c];
    const uint32_t b = __float_as_uint(D);
    const uint32_t e = (b >> 23) & 0xFFu;
    const bool usable = c >= first && c < num_codes(FMT) && (b >> 31) == 0 && e != 255;
    const bool is_paired = usable && e >= 1 && e <= 253;
    const __half hD = __float2half_rn(-D);
    const int kind = !usable ? 2 : (!is_paired ? 3 : (__half2float(hD) == -D ? 1 : 0));
    T.kind[c] = (uint8_t)kind;
    if (c < kLists) T.cnt[c] = 0;
    const uint32_t ballot0 = __ballot_sync(0xFFFFFFFFu, kind == 0);
    const uint32_t ballot1 = __ballot_sync(0xFFFFFFFFu, kind == 1);
    const uint32_t ballot3 = __ballot_sync(0xFFFFFFFFu, kind == 3);
    if ((c & 31) == 0) {
        T.kind_mask[0][c >> 5] = ballot0;
        T.kind_mask[1][c >> 5] = ballot1;
        T.kind_mask[2][c >> 5] = ballot3;
    }
    __syncthreads();
    const uint32_t below = (1u << (c & 31)) - 1u;
    if (kind == 3) {
        int rank = __popc(ballot3 & below);
        for (int w = 0; w < (c >> 5); ++w) rank += __popc(T.kind_mask[2][w]);
        // multiplier 0 -> every quotient is zero; 2^126 -> every nonzero quotient saturates
        const float P = (e == 0 && D != 0.0f) ? __uint_as_float(0x7E800000u) : 0.0f;
        const int slot = members_base<FMT>(kFlatList) + rank;
        T.cand[slot] = make_float4(-D, P, 0.0f, 0.0f);
        T.member[slot] = (uint8_t)c;
        atomicAdd(&T.cnt[kFlatList], 1);
    }
    if (is_paired) {
        const int cls = code_class<FMT>(c);
        int rank = 0;
        if constexpr (FMT == kUE8M0) {
            for (int w = 0; w < (c >> 5); ++w) rank += __popc(T.kind_mask[kind][w]);
            rank += __popc((kind ? ballot1 : ballot0) & below);
        } else {
            for (int o = 1; o < 8 && o < c; ++o) rank += (T.kind[o] == kind && code_class<FMT>(o) == cls) ? 1 : 0;
            for (int o = 8 + cls; o < c; o += 8) rank += (T.kind[o] == kind) ? 1 : 0;
        }
        const float P = __uint_as_float((254u - e) << 23);
        const uint32_t h16 = (uint32_t)__half_as_ushort(hD);
        const int list = 2 * cls + kind;
        const int slot = members_base<FMT>(list) + rank;
        T.cand[slot] = make_float4(-D, P, __uint_as_float(h16 | (h16 << 16)), 0.0f);
        T.member[slot] = (uint8_t)c;
        atomicAdd(&T.cnt[list], 1);
        if (rank == 0) {   // both kinds of a class write the same values
            const float Dref = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
            T.clsD[cls] = Dref;
            T.clsR[cls] = __frcp_rn(Dref);
        }
    }
    __syncthreads();
    // the search takes two members per trip: a range that ends with the list may read one slot
    // past it, which repeats the last member
    if (c < kLists && T.cnt[c] > 0) {
        const int last = members_base<FMT>(c) + T.cnt[c] - 1;
        T.cand[last + 1] = T.cand[last];
        T.member[last + 1] = T.member[last];
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------------------
// packed helpers
// ------------------------------------------------------------------------------------------------
// Residuals of one pair for one candidate: t = tb * 2^-k, q = t rounded onto the FP4 grid
// (round-to-nearest-even, saturating at +-6), e = fma(q, -D, v).  HALF: -D is given in f16
// (low half of nD16 for .x, high half for .y) and the FMA takes q straight from the unpacked f16
// pair (fma.rn.f32.f16: exact product, one rounding to binary32); otherwise q is widened first.
template <bool HALF>
__device__ __forceinline__ float2 residual_pair(float2 tb, float2 P2, float2 v, float2 nD2, uint32_t nD16) {
    const float2 t = __fmul2_rn(tb, P2);
    uint32_t h;
    asm("{\n"
        " .reg .b8 b0;\n"
        " cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n"
        " cvt.rn.f16x2.e2m1x2 %0, b0;\n"
        "}"
        : "=r"(h)
        : "f"(t.x), "f"(t.y));
    if constexpr (HALF) {
        float2 e;
        asm("{\n"
            " .reg .b16 qlo, qhi, dlo, dhi;\n"
            " mov.b32 {qlo, qhi}, %2;\n"
            " mov.b32 {dlo, dhi}, %3;\n"
            " fma.rn.f32.f16 %0, qlo, dlo, %4;\n"
            " fma.rn.f32.f16 %1, qhi, dhi, %5;\n"
            "}"
            : "=f"(e.x), "=f"(e.y)
            : "r"(h), "r"(nD16), "f"(v.x), "f"(v.y));
        return e;
    } else {
        // f16 -> binary32 as a mixed-precision add of -0 (exact, keeps the sign of zero): unlike a
        // plain convert it takes its half straight out of the 32-bit register
        float2 q;
        asm("{\n"
            " .reg .b16 qlo, qhi;\n"
            " mov.b32 {qlo, qhi}, %2;\n"
            " add.rn.f32.f16 %0, qlo, %3;\n"
            " add.rn.f32.f16 %1, qhi, %3;\n"
            "}"
            : "=f"(q.x), "=f"(q.y)
            : "r"(h), "f"(-0.0f));
        return make_float2(__fmaf_rn(q.x, nD2.x, v.x), __fmaf_rn(q.y, nD2.y, v.y));
    }
}

// Residuals of ONE element for TWO candidates A, B, given its scaled quotients tA = tb * 2^-kA and
// tB: q = FP4 rounding of t, e = fma(q, -D, v) for either candidate (.x = A, .y = B).  HALF: nD16
// holds f16(-D_A) in the low half and f16(-D_B) in the high half.
template <bool HALF>
__device__ __forceinline__ float2 residual_two_candidates(float tA, float tB, float v, float nDA, float nDB,
                                                          uint32_t nD16) {
    uint32_t h;
    asm("{\n"
        " .reg .b8 b0;\n"
        " cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n"
        " cvt.rn.f16x2.e2m1x2 %0, b0;\n"
        "}"
        : "=r"(h)
        : "f"(tA), "f"(tB));
    float2 e;
    if constexpr (HALF) {
        asm("{\n"
            " .reg .b16 qlo, qhi, dlo, dhi;\n"
            " mov.b32 {qlo, qhi}, %2;\n"
            " mov.b32 {dlo, dhi}, %3;\n"
            " fma.rn.f32.f16 %0, qlo, dlo, %4;\n"
            " fma.rn.f32.f16 %1, qhi, dhi, %4;\n"
            "}"
            : "=f"(e.x), "=f"(e.y)
            : "r"(h), "r"(nD16), "f"(v));
    } else {
        float2 q;   // f16 -> binary32 as in residual_pair()
        asm("{\n"
            " .reg .b16 qlo, qhi;\n"
            " mov.b32 {qlo, qhi}, %2;\n"
            " add.rn.f32.f16 %0, qlo, %3;\n"
            " add.rn.f32.f16 %1, qhi, %3;\n"
            "}"
            : "=f"(q.x), "=f"(q.y)
            : "r"(h), "f"(-0.0f));
        e.x = __fmaf_rn(q.x, nDA, v);
        e.y = __fmaf_rn(q.y, nDB, v);
    }
    return e;
}

// fl32(v / Dref) for both halves; nD = -Dref, R = RN(1 / Dref), Dref in [1, 2), |v| <= 2^60: the
// reciprocal multiply with one residual correction of quotient_short() (see there why one
// correction gives the IEEE quotient for every divisor), except for the sign of a zero quotient,
// which the search does not use.
__device__ __forceinline__ float2 quotient_pair(float2 v, float2 nD, float2 R) {
    const float2 q = __fmul2_rn(v, R);
    const float2 r = __ffma2_rn(q, nD, v);
    return __ffma2_rn(r, R, q);
}

__device__ __forceinline__ unsigned long long sse_key(float s, int c) {
    return ((unsigned long long)__float_as_uint(s) << 32) | (unsigned long long)(unsigned)c;
}

// General path for one block held in `lane` (0 = .x, 1 = .y) of pairs first .. first + B - 1.
template <int B, int NP>
__device__ __forceinline__ float general_sse(const float2 (&v2)[NP], int first, int lane, float D) {
    float s = 0.0f;
#pragma unroll
    for (int i = 0; i < B; i += 2) {
        const float a = lane ? v2[first + i].y : v2[first + i].x;
        const float b = lane ? v2[first + i + 1].y : v2[first + i + 1].x;
        const float2 q = round_e2m1x2(quotient_general(a, D), quotient_general(b, D));
        const float e0 = __fmaf_rn(-q.x, D, a);
        s = __fmaf_rn(e0, e0, s);
        const float e1 = __fmaf_rn(-q.y, D, b);
        s = __fmaf_rn(e1, e1, s);
    }
    return s;
}

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
// Fold the winner of one class (smallest SSE bits; first, i.e. smallest, code among equals) into
// the running (SSE, code) key.
__device__ __forceinline__ void merge_class_winner(unsigned long long& best, uint32_t bits, int code) {
    const unsigned long long k = ((unsigned long long)bits << 32) | (unsigned long long)(unsigned)code;
    if (k < best) best = k;
}

// Strict "smaller SSE bits wins", without a branch.
__device__ __forceinline__ void keep_smaller(uint32_t& best_bits, int& best_slot, uint32_t bits, int slot) {
    best_slot = bits < best_bits ? slot : best_slot;
    best_bits = min(best_bits, bits);
}

// All members of one range of one list (one mantissa class, one residual kind) against the
// thread's elements; the winner of every block is folded into best[].
// Members first .. first + cnt_raw - 1 of the list are evaluated.
template <int B, int FMT, bool HALF, int NP, int NBT>
__device__ __forceinline__ void search_list(const BruteTables& T, int list, int first, int cnt_raw,
                                            const float2 (&v2)[NP], const float2 (&tb)[NP],
                                            unsigned long long (&best)[NBT]) {
    constexpr bool ONEBLK = (B >= 32);
    constexpr int BL = ONEBLK ? NP : B;
    constexpr int NBL = NP / BL;
    if (cnt_raw <= 0) return;
    [[maybe_unused]] const int cnt = cnt_raw;
    const int base = members_base<FMT>(list) + first;
    const float4* cand = T.cand + base;
    uint32_t cbest[NBT];
    int cslot[NBT];
#pragma unroll
    for (int k = 0; k < NBT; ++k) { cbest[k] = 0xFFFFFFFFu; cslot[k] = 0; }

    if constexpr (!ONEBLK) {
        // two members per trip: two independent SSE chains keep the FMA pipe fed
        const int pairs_end = cnt & ~1;
        for (int m = 0; m < pairs_end; m += 2) {
            const float4 dpA = cand[m], dpB = cand[m + 1];
            const float2 nDA = make_float2(dpA.x, dpA.x), PA = make_float2(dpA.y, dpA.y);
            const float2 nDB = make_float2(dpB.x, dpB.x), PB = make_float2(dpB.y, dpB.y);
            const uint32_t hA = __float_as_uint(dpA.z), hB = __float_as_uint(dpB.z);
            float2 sA[NBL], sB[NBL];
#pragma unroll
            for (int k = 0; k < NBL; ++k) sA[k] = sB[k] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 eA = residual_pair<HALF>(tb[i], PA, v2[i], nDA, hA);
                const float2 eB = residual_pair<HALF>(tb[i], PB, v2[i], nDB, hB);
                sA[i / BL] = __ffma2_rn(eA, eA, sA[i / BL]);
                sB[i / BL] = __ffma2_rn(eB, eB, sB[i / BL]);
            }
#pragma unroll
            for (int k = 0; k < NBL; ++k) {
                keep_smaller(cbest[k], cslot[k], __float_as_uint(sA[k].x), m);
                keep_smaller(cbest[NBL + k], cslot[NBL + k], __float_as_uint(sA[k].y), m);
                keep_smaller(cbest[k], cslot[k], __float_as_uint(sB[k].x), m + 1);
                keep_smaller(cbest[NBL + k], cslot[NBL + k], __float_as_uint(sB[k].y), m + 1);
            }
        }
        if (cnt & 1) {   // the odd member on its own
            const int m = cnt - 1;
            const float4 dpA = cand[m];
            const float2 nDA = make_float2(dpA.x, dpA.x), PA = make_float2(dpA.y, dpA.y);
            const uint32_t hA = __float_as_uint(dpA.z);
            float2 sA[NBL];
#pragma unroll
            for (int k = 0; k < NBL; ++k) sA[k] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 eA = residual_pair<HALF>(tb[i], PA, v2[i], nDA, hA);
                sA[i / BL] = __ffma2_rn(eA, eA, sA[i / BL]);
            }
#pragma unroll
            for (int k = 0; k < NBL; ++k) {
                keep_smaller(cbest[k], cslot[k], __float_as_uint(sA[k].x), m);
                keep_smaller(cbest[NBL + k], cslot[NBL + k], __float_as_uint(sA[k].y), m);
            }
        }
    } else {
        // one block per thread: lane .x of the SSE pair is member m, lane .y member m + 1 (the
        // slot behind an odd range holds a real member or the copy of the last one: harmless)
        for (int m = 0; m < cnt; m += 2) {
            const float4 dpA = cand[m], dpB = cand[m + 1];
            const float2 PA = make_float2(dpA.y, dpA.y), PB = make_float2(dpB.y, dpB.y);
            const uint32_t nD16 = (__float_as_uint(dpA.z) & 0xFFFFu) | (__float_as_uint(dpB.z) << 16);
            float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 tA = __fmul2_rn(tb[i], PA), tB = __fmul2_rn(tb[i], PB);   // elements 2i, 2i + 1
                const float2 e0 = residual_two_candidates<HALF>(tA.x, tB.x, v2[i].x, dpA.x, dpB.x, nD16);
                s = __ffma2_rn(e0, e0, s);
                const float2 e1 = residual_two_candidates<HALF>(tA.y, tB.y, v2[i].y, dpA.x, dpB.x, nD16);
                s = __ffma2_rn(e1, e1, s);
            }
            keep_smaller(cbest[0], cslot[0], __float_as_uint(s.x), m);
            keep_smaller(cbest[0], cslot[0], __float_as_uint(s.y), m + 1);
        }
    }
#pragma unroll
    for (int k = 0; k < NBT; ++k)
        if (cbest[k] != 0xFFFFFFFFu) merge_class_winner(best[k], cbest[k], T.member[base + cslot[k]]);
}

// Resident CTAs per SM asked of the register allocator: two (at most 128 registers) for every block
// size up to 32 -- the kernels sit within a few registers of that limit, and falling to one
// resident CTA costs far more (measured: 8 % at B = 16) than the allocator's squeeze; B = 64 needs
// about 170 registers and runs one CTA per SM.
// Elements a thread of k_brute owns: one block for B >= 32, else 32; 16 for B = 2, whose 16
// running minima per 32 elements otherwise leave room for one CTA per SM only (measured: 496 -> 452 us;
// B = 4 and B = 8 lose with 16).
__host__ __device__ constexpr int brute_group_elems(int B) { return B >= 32 ? B : (B == 2 ? 16 : 32); }

constexpr int brute_min_ctas(int B) { return B <= 32 ? 2 : 1; }

template <int DT, int B, int FMT>
__global__ void __launch_bounds__(kThreads, brute_min_ctas(B)) k_brute(QuantArgs p) {
    constexpr bool ONEBLK = (B >= 32);        // the thread owns exactly one block
    constexpr int G = brute_group_elems(B);     // elements per thread
    constexpr int NP = G / 2;                 // pairs per thread
    constexpr int BL = ONEBLK ? NP : B;         // elements of one block inside one half
    constexpr int NBL = NP / BL;              // blocks per half (1 when ONEBLK)
    constexpr int NBT = ONEBLK ? 1 : 2 * NBL;   // blocks per thread
    constexpr int NCLS = (FMT == kUE8M0) ? 1 : 8;
    constexpr float kTiny = 2.168404344971009e-19f;  // 2^-62

    __shared__ BruteTables T;
    wait_for_prior_grid();
    release_dependents();
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const int first = (p.prevent_zero && FMT != kUE8M0) ? 1 : 0;
    build_brute_tables<FMT>(T, g, first);

    const size_t stride = (size_t)gridDim.x * kThreads;
    double sse_sum = 0.0;                  // binary64 sum of the SSEs of this thread's blocks, in the order it stored them
    for (size_t grp = (size_t)blockIdx.x * kThreads + threadIdx.x; grp < p.n_items; grp += stride) {
        float2 v2[NP];
        float amax = 0.0f;
        bool tiny = false;   // a nonzero magnitude below 2^-62: its quotient by Dref may be inexact
        {
            float v[G];
            load_elems<DT, G>(p.x, grp * G, v);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                // one block per thread: adjacent elements; else element i of either half
                const float x0 = ONEBLK ? v[2 * i] : v[i], x1 = ONEBLK ? v[2 * i + 1] : v[NP + i];
                v2[i] = make_float2(x0, x1);
                const float a0 = fabsf(x0), a1 = fabsf(x1);
                amax = fmaxf(amax, fmaxf(a0, a1));
                tiny |= (a0 < kTiny && a0 != 0.0f) || (a1 < kTiny && a1 != 0.0f);
            }
        }
        const bool fast_ok = (amax <= kFastMax) && !tiny;

        // best[k]: k < NBL -> block k of the low half, else block k - NBL of the high half
        unsigned long long best[NBT];
#pragma unroll
        for (int k = 0; k < NBT; ++k) best[k] = sse_key(__uint_as_float(0xFFFFFFFFu), first);

        auto class_quotients = [&](int cls, float2 (&tb)[NP]) {
            const float Dr = T.clsD[cls], Rr = T.clsR[cls];
            const float2 nDr2 = make_float2(-Dr, -Dr), Rr2 = make_float2(Rr, Rr);
#pragma unroll
            for (int i = 0; i < NP; ++i)
                tb[i] = quotient_pair(v2[i], nDr2, Rr2);
        };

        if (fast_ok) {
            for (int cls = 0; cls < NCLS; ++cls) {
                const int n0 = T.cnt[2 * cls], n1 = T.cnt[2 * cls + 1];
                if (n0 + n1 == 0) continue;
                float2 tb[NP];
                class_quotients(cls, tb);
                search_list<B, FMT, false>(T, 2 * cls, 0, n0, v2, tb, best);
                search_list<B, FMT, true>(T, 2 * cls + 1, 0, n1, v2, tb, best);
            }
            // Dref = 1: the elements are their own quotients
            search_list<B, FMT, false>(T, kFlatList, 0, T.cnt[kFlatList], v2, v2, best);
        }

        // general path (IEEE division), candidate by candidate: threads that hold a magnitude above
        // 2^60 or a nonzero one below 2^-62
        const int n_general = fast_ok ? 0 : num_codes(FMT);
        for (int c = first; c < n_general; ++c) {
            const float D = T.D[c];
            if (!(fabsf(D) <= 3.402823466e38f)) continue;  // decode scale overflowed: not usable
            if constexpr (!ONEBLK) {
#pragma unroll
                for (int k = 0; k < NBL; ++k) {
                    const unsigned long long k0 = sse_key(general_sse<B, NP>(v2, k * BL, 0, D), c);
                    const unsigned long long k1 = sse_key(general_sse<B, NP>(v2, k * BL, 1, D), c);
                    if (k0 < best[k]) best[k] = k0;
                    if (k1 < best[NBL + k]) best[NBL + k] = k1;
                }
            } else {
                float s = 0.0f;
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const float a = v2[i].x, b = v2[i].y;
                    const float2 q = round_e2m1x2(quotient_general(a, D), quotient_general(b, D));
                    const float e0 = __fmaf_rn(-q.x, D, a);
                    s = __fmaf_rn(e0, e0, s);
                    const float e1 = __fmaf_rn(-q.y, D, b);
                    s = __fmaf_rn(e1, e1, s);
                }
                const unsigned long long k0 = sse_key(s, c);
                if (k0 < best[0]) best[0] = k0;
            }
        }

        // final encode with the winners
        uint32_t packed[G / 8];
        uint32_t sc[(NBT + 3) / 4];
        uint32_t sw[NBT];
#pragma unroll
        for (int k = 0; k < (NBT + 3) / 4; ++k) sc[k] = 0;
        if constexpr (ONEBLK) {
            const int code = (int)(best[0] & 0xFFu);
            const float D = T.D[code];
            const float R = T.R[code];
            const bool fast = (R != 0.0f) && (amax <= kFastMax);
            sc[0] = (uint32_t)code;
            sw[0] = (uint32_t)(best[0] >> 32);
#pragma unroll
            for (int k = 0; k < G / 8; ++k) {
                float t[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 a = v2[4 * k + i];
                    t[2 * i] = fast ? quotient_corrected(a.x, D, R) : quotient_general(a.x, D);
                    t[2 * i + 1] = fast ? quotient_corrected(a.y, D, R) : quotient_general(a.y, D);
                }
                packed[k] = pack_e2m1x8(t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7]);
            }
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float t[NP];
#pragma unroll
                for (int k = 0; k < NBL; ++k) {
                    const int kb = h * NBL + k;   // block index inside the thread
                    const int code = (int)(best[kb] & 0xFFu);
                    const float D = T.D[code];
                    const float R = T.R[code];
                    const bool fast = (R != 0.0f) && (amax <= kFastMax);
#pragma unroll
                    for (int i = 0; i < BL; ++i) {
                        const float a = h ? v2[k * BL + i].y : v2[k * BL + i].x;
                        t[k * BL + i] = fast ? quotient_corrected(a, D, R) : quotient_general(a, D);
                    }
                    sc[kb / 4] |= (uint32_t)code << (8 * (kb % 4));
                    sw[kb] = (uint32_t)(best[kb] >> 32);
                }
#pragma unroll
                for (int k = 0; k < NP / 8; ++k)
                    packed[h * (NP / 8) + k] = pack_e2m1x8(t[8 * k], t[8 * k + 1], t[8 * k + 2], t[8 * k + 3], t[8 * k + 4],
                                                           t[8 * k + 5], t[8 * k + 6], t[8 * k + 7]);
            }
        }
        store_bytes<G / 2>(p.codes + grp * (G / 2), packed);
        store_bytes<NBT>(p.scales + grp * NBT, sc);
        if (p.block_sse) store_bytes<4 * NBT>(p.block_sse + grp * NBT, sw);
#pragma unroll
        for (int k = 0; k < NBT; ++k) sse_sum = __dadd_rn(sse_sum, (double)__uint_as_float(sw[k]));
    }
    if (p.mse_partials != nullptr) {   // launch-uniform: fused tensor-MSE partial sum of this CTA
        __syncthreads();               // the tables are no longer read: their memory serves as scratch
        const double total = cta_sum_fixed_order(sse_sum, reinterpret_cast<double*>(&T));
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

// ------------------------------------------------------------------------------------------------
// The blocks past the last whole per-thread group (block sizes up to 16 only): one block per
// thread, general path.
// ------------------------------------------------------------------------------------------------
template <int DT, int B, int FMT>
__global__ void k_brute_tail(QuantArgs p) {
    const size_t b = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    float my_sse = 0.0f;
    if (b < p.n_items) {
    const size_t blk = p.first_item + b;
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const int first = (p.prevent_zero && FMT != kUE8M0) ? 1 : 0;
    float v[B];
    load_elems<DT, B>(p.x, blk * B, v);
    unsigned long long best = sse_key(__uint_as_float(0xFFFFFFFFu), first);
    for (int c = first; c < num_codes(FMT); ++c) {
        const float D = __fmul_rn(scale_value(FMT, c), g);
        if (!(fabsf(D) <= 3.402823466e38f)) continue;
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < B; i += 2) {
            const float2 q = round_e2m1x2(quotient_general(v[i], D), quotient_general(v[i + 1], D));
            const float e0 = __fmaf_rn(-q.x, D, v[i]);
            s = __fmaf_rn(e0, e0, s);
            const float e1 = __fmaf_rn(-q.y, D, v[i + 1]);
            s = __fmaf_rn(e1, e1, s);
        }
        const unsigned long long k = sse_key(s, c);
        if (k < best) best = k;
    }
    const int code = (int)(best & 0xFFu);
    const float D = __fmul_rn(scale_value(FMT, code), g);
    uint32_t packed[(B + 7) / 8];
#pragma unroll
    for (int k = 0; k < (B + 7) / 8; ++k) packed[k] = 0;
#pragma unroll
    for (int k = 0; k < B / 2; ++k)
        packed[k / 4] |= pack_e2m1x2(quotient_general(v[2 * k], D), quotient_general(v[2 * k + 1], D)) << (8 * (k % 4));
    store_bytes<B / 2>(p.codes + blk * (B / 2), packed);
    p.scales[blk] = (uint8_t)code;
    if (p.block_sse) p.block_sse[blk] = __uint_as_float((uint32_t)(best >> 32));
    my_sse = __uint_as_float((uint32_t)(best >> 32));
    }
    // fused tensor-MSE partial sum: the kernel is one warp, every lane takes part (idle lanes add 0)
    if (p.mse_partials != nullptr) warp_sum_to_partial(p, my_sse);
}

template <int DT, int B, int FMT>
static cudaError_t launch_brute_inst(const QuantArgs& a, cudaStream_t stream) {
    static std::atomic<int> ctas_per_sm[kMaxDevices];   // first-use cache; racing threads store the same value
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    int resident = ctas_per_sm[dev].load(std::memory_order_relaxed);
    if (resident == 0) {
        int n = 0;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_brute<DT, B, FMT>, kThreads, 0);
        if (err != cudaSuccess) return err;
        resident = n > 0 ? n : 1;
        ctas_per_sm[dev].store(resident, std::memory_order_relaxed);
    }
    constexpr size_t G = brute_group_elems(B);    // elements per thread of k_brute
    const size_t n_blocks = a.n_items;
    const size_t n_groups = n_blocks * B / G;
    const size_t done = n_groups * G / B;
    // The blocks past the last whole group go to the one-warp tail kernel.  With fused MSE partial sums it
    // runs first and owns partial 0; the CTAs of the main kernel own the partials from 1 on.
    auto launch_tail = [&]() -> cudaError_t {
        if constexpr (B < 32) {
            if (done < n_blocks) {
                QuantArgs t = a;
                t.first_item = done;
                t.n_items = n_blocks - done;
                t.mse_first = 0;
                k_brute_tail<DT, B, FMT><<<1, 32, 0, stream>>>(t);
                count_launch();
                return cudaGetLastError();
            }
        }
        return cudaSuccess;
    };
    if (a.mse_partials) {
        err = launch_tail();
        if (err != cudaSuccess) return err;
    }
    if (n_groups > 0) {
        QuantArgs m = a;
        m.n_items = n_groups;
        m.mse_first = (done < n_blocks) ? 1 : 0;
        const size_t want = (n_groups + kThreads - 1) / kThreads;
        size_t cap = (size_t)sm_count(dev) * (size_t)resident;
        if (a.mse_partials && cap > (size_t)kMsePartials - 1) cap = kMsePartials - 1;
        const unsigned grid = (unsigned)(want < cap ? want : cap);
        err = launch_pdl(k_brute<DT, B, FMT>, grid, kThreads, 0, stream, m);
        count_launch();
        if (err != cudaSuccess) return err;
        if (a.mse_n_partials) *a.mse_n_partials = (int)grid + m.mse_first;
    } else if (a.mse_n_partials) {
        *a.mse_n_partials = (done < n_blocks) ? 1 : 0;
    }
    if (!a.mse_partials) err = launch_tail();
    return err;
}

template <int DT, int B>
static cudaError_t launch_brute_fmt(const QuantArgs& a, int fmt, cudaStream_t s) {
    switch (fmt) {
    case kUE8M0: return launch_brute_inst<DT, B, kUE8M0>(a, s);
    case kUE4M3: return launch_brute_inst<DT, B, kUE4M3>(a, s);
    default: return launch_brute_inst<DT, B, kUE5M3>(a, s);
    }
}

template <int DT>
static cudaError_t launch_brute_dt(const QuantArgs& a, int B, int fmt, cudaStream_t s) {
    switch (B) {
    case 2: return launch_brute_fmt<DT, 2>(a, fmt, s);
    case 4: return launch_brute_fmt<DT, 4>(a, fmt, s);
    case 8: return launch_brute_fmt<DT, 8>(a, fmt, s);
    case 16: return launch_brute_fmt<DT, 16>(a, fmt, s);
    case 32: return launch_brute_fmt<DT, 32>(a, fmt, s);
    default: return launch_brute_fmt<DT, 64>(a, fmt, s);
    }
}

}  // namespace mxq
