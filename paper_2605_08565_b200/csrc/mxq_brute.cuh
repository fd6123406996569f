// Brute-force scale search (Experimental Setup: the optimal baseline, found by trying the possible
// scale values and keeping the one with the least error): every finite scale code of the format
// is tried on every block and the code with the smallest SSE is kept (equal SSE: the smaller code).
//
// Work layout.  A thread owns a group of G consecutive elements, whole blocks: G = B for B >= 32; 16 for B = 2 and 4; 32 for B = 8 and
// 16, or 16 where the tensor is too small to fill the chip with groups of 32 (launch_brute_inst()).  They stay in registers as float
// pairs and the candidate loop works on pairs with the packed binary32 instructions of sm_100 (fma.rn.f32x2 /
// mul.rn.f32x2, FP4 pack and unpack two at a time):
//   G > B     pair i = (element i, element G/2 + i): the two halves of a pair belong to different blocks, so one
//             instruction serves two elements of one candidate and the two SSE chains are independent.  Two candidates
//             per trip.
//   G = B     the thread owns one block, pair i = (element 2i, element 2i + 1).  Its SSE is one
//             sequential chain over all elements, so the two lanes of the SSE pair are two
//             CANDIDATES: the scaling multiplies run on element pairs, the FP4 rounding and the
//             residuals on candidate pairs of one element, and the elements are walked in order.
// The candidate loop is uniform across a warp (not across the CTA: a warp's ranges depend on its elements, its slice of the codes on
// its place): decode scales come from shared memory as broadcasts, and no barrier may stand inside.
//
// Three kernels: k_brute leaves the cheap stretches of the codes out of the full evaluation, any number of blocks; k_brute_plain
// evaluates every code in full, whole groups only (k_brute_split takes the blocks behind them); k_brute_split shares a group
// between 2, 4 or 8 warps, any number of blocks.
//
// One exact quotient per mantissa, not per candidate.  The decode scale of code c is
// D_c = fl(S_c * g).  All codes whose S_c share a mantissa (eight classes for the FP8 scale
// formats, one for the power-of-two format) have decode scales that differ by exact powers of two,
// D_c = Dref * 2^k, as long as D_c is a normal number.  Hence fl(v / D_c) = fl(v / Dref) * 2^-k
// exactly: the correctly rounded quotient is formed once per class and element, and a candidate
// costs one multiply by a power of two, the FP4 rounding, and the two FMAs of the SSE.  Codes under
// which every element of the warp rounds to zero or saturates cost less (search_group()).  Threads holding a magnitude above
// 2^60 or a nonzero one below 2^-62 take the general path (IEEE division), candidate by candidate.
//
// Inside a class the members are visited in ascending code order and the smallest SSE bit pattern
// is kept with a strict compare (SSE >= 0, so integer order is float order and the first of equals
// is the smaller code); class winners are merged as 64-bit keys (SSE bits << 32 | code).
#pragma once

#include <atomic>
#include <type_traits>

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

// Per-CTA tables of the search.  Every code whose decode scale D is normal with a biased exponent of at most 253 (D = Dref *
// 2^k and 2^-k are both representable) sits in the candidate list 2 * class + kind, where kind 1 holds the codes whose -D is
// exactly representable in f16 (their residual is one mixed-precision FMA from the unpacked f16 grid value) and kind 0
// the others (f16 -> f32 convert, then an FFMA).  Codes with D zero, subnormal or at least 2^127 never need the full
// evaluation (see search_group()).
constexpr int kLists = 16;
constexpr int kCandSlots = kLists * kMaxMembers;
struct BruteTables {
    float D[256];            // decode scale of the code; NaN for codes that do not exist
    float R[256];            // RN(1 / D) when 2^-60 <= D <= 2^60, else 0 (used by the final encode)
    float4 cand[kCandSlots];    // per list, ascending code order: (-D, multiplier, f16(-D) twice as bits, 0)
    uint8_t member[kCandSlots]; // the code of each slot of cand[]
    float clsD[8];           // Dref of the class, in [1, 2)
    float clsR[8];           // RN(1 / Dref)
    int cnt[kLists];         // members per list
    int flat_min;            // smallest code with D zero, subnormal or at least 2^127; 256 if there is none
    uint8_t below[kLists][256];   // members of the list whose code is smaller
    uint8_t in_warp[kThreads / 32][kLists];   // members of the list among the 32 codes of a warp (scratch of the build)
};

template <int FMT>
__device__ __forceinline__ int members_base(int list) {
    // the power-of-two format has one class: its two lists get half of the class area each
    return FMT == kUE8M0 ? list * (kCandSlots / 2) : list * kMaxMembers;
}

// first: smallest admissible code (1 under prevent-zero for the FP8 formats, else 0).  BELOW: with the index by code.
template <int FMT, bool BELOW>
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
    const int my_list = !is_paired ? -1 : 2 * code_class<FMT>(c) + (__half2float(hD) == -D ? 1 : 0);
    if (c == 0) T.flat_min = 256;
    constexpr int NL = FMT == kUE8M0 ? 2 : kLists;
    const int warp = c >> 5, lane = c & 31;
    uint32_t members[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        members[l] = __ballot_sync(0xFFFFFFFFu, my_list == l);
        if (lane == l) T.in_warp[warp][l] = (uint8_t)__popc(members[l]);
    }
    __syncthreads();
    if (c < NL) {   // exclusive prefix sums over the warps, and the total
        int n = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            const int here = T.in_warp[w][c];
            T.in_warp[w][c] = (uint8_t)n;
            n += here;
        }
        T.cnt[c] = n;
    }
    __syncthreads();
    int rank = 0;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const int n = T.in_warp[warp][l] + __popc(members[l] & ((1u << lane) - 1u));
        if constexpr (BELOW) T.below[l][c] = (uint8_t)n;
        if (l == my_list) rank = n;
    }
    if (usable && !is_paired) atomicMin(&T.flat_min, c);
    if (is_paired) {
        const float P = __uint_as_float((254u - e) << 23);
        const uint32_t h16 = (uint32_t)__half_as_ushort(hD);
        const int slot = members_base<FMT>(my_list) + rank;
        T.cand[slot] = make_float4(-D, P, __uint_as_float(h16 | (h16 << 16)), 0.0f);
        T.member[slot] = (uint8_t)c;
        if (rank == 0) {   // both kinds of a class write the same values
            const float Dref = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
            T.clsD[my_list >> 1] = Dref;
            T.clsR[my_list >> 1] = __frcp_rn(Dref);
        }
    }
    __syncthreads();
    // the search takes two members per trip: a range that ends with the list may read one slot
    // past it, which repeats the last member
    if (c < NL && T.cnt[c] > 0) {
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

// Largest code whose value is at most S (0 if there is none), S >= 0.
template <int FMT>
__device__ __forceinline__ int floor_code(float S) {
    const uint32_t b = __float_as_uint(S);
    if constexpr (FMT == kUE8M0) return (int)min(b >> 23, 254u);
    constexpr int bias = (FMT == kUE4M3) ? 7 : 15;
    const int normal = (int)(b >> 20) - ((127 - bias) << 3);
    const int sub = __float2int_rz(__fmul_rn(S, (float)(1 << (bias + 2))));
    return min(normal < 8 ? sub : normal, num_codes(FMT) - 1);
}

// All members of one range of one list (one mantissa class, one residual kind) against the
// thread's elements; the winner of every block is folded into best[].
// Members first .. first + cnt_raw - 1 of the list are evaluated.
template <int B, int FMT, bool HALF, bool ONEBLK, int NP, typename Best>
__device__ __forceinline__ void search_list(const BruteTables& T, int list, int first, int cnt_raw,
                                            const float2 (&v2)[NP], const float2 (&tb)[NP], Best& best) {
    constexpr int BL = ONEBLK ? NP : B;
    constexpr int NBL = NP / BL;
    constexpr int NBT = ONEBLK ? 1 : 2 * NBL;
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
// Elements a thread owns: one block for B >= 32, else 32; 16 for B = 2 and 4, whose 16 or 8 running minima per 32 elements
// otherwise leave room for one CTA per SM only, or spill (16.8 M elements: B = 2 496 -> 452 us, B = 4 662 -> 632).
__host__ __device__ constexpr int brute_group_elems(int B) { return B >= 32 ? B : (B <= 4 ? 16 : 32); }

constexpr int brute_min_ctas(int B) { return B <= 32 ? 2 : 1; }

// Where k_brute keeps the best (SSE bits, code) key of each of a thread's blocks: in registers, except at B = 32, B = 8 in groups of 32
// and UE8M0 at B = 64, which pay for the registers (16.8 M fp32 elements, shared memory -> registers, us: unscaled UE4M3 of N(0, 300),
// B = 2 476 -> 451, 64 349 -> 337, but 8 336 -> 343; UE5M3 under a tensor scale, B = 16 539 -> 532, 64 589 -> 578, but 32 527 -> 559; UE8M0,
// B = 2 171 -> 168, but 64 144 -> 145).
__host__ __device__ constexpr bool brute_keys_in_registers(int B, int G, int fmt) {
    return B != 32 && !(B == 8 && G == 32) && !(B == 64 && fmt == kUE8M0);
}

// Keys in shared memory, 32 lanes apart.
struct SharedBest {
    unsigned long long* p;
    __device__ __forceinline__ unsigned long long& operator[](int k) const { return p[32 * k]; }
};

// Keys in registers.
template <int N>
struct RegisterBest {
    unsigned long long k[N];
    __device__ __forceinline__ unsigned long long& operator[](int i) { return k[i]; }
};

// G: elements per thread.
template <int B, int G_>
struct BruteShape {
    static constexpr int G = G_;
    static constexpr bool ONEBLK = (G == B);        // the thread owns exactly one block
    static constexpr int NP = G / 2;                // pairs per thread
    static constexpr int BL = ONEBLK ? NP : B;      // elements of one block inside one half
    static constexpr int NBL = NP / BL;             // blocks per half (1 when ONEBLK)
    static constexpr int NBT = G / B;               // blocks per thread
};

// What a thread knows of its elements beside their magnitudes.
struct GroupRange {
    float amax, amin;      // largest magnitude; smallest nonzero one (+inf if there is none)
    bool has_zero;
    bool fast;             // no magnitude above 2^60, no nonzero one below 2^-62 (its quotient by Dref may be inexact)
};

// A thread's elements.  n_here: elements of the tensor in this group (a multiple of B, at most G); what is missing is taken
// as zero.
template <int DT, int B, int G>
__device__ __forceinline__ void load_group(float (&v)[BruteShape<B, G>::G], const void* x, size_t e0, int n_here) {
    using S = BruteShape<B, G>;
    if (n_here >= S::G) {
        load_elems<DT, S::G>(x, e0, v);
        return;
    }
#pragma unroll
    for (int k = 0; k < S::NBT; ++k) {
        float w[B];
        if (k * B < n_here) {
            load_elems<DT, B>(x, e0 + k * B, w);
        } else {
#pragma unroll
            for (int i = 0; i < B; ++i) w[i] = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < B; ++i) v[k * B + i] = w[i];
    }
}

// Where a warp starts.  Sets of 32 groups go round the CTAs before they go round a CTA's warps, so that a tensor, or
// its last trip, that does not occupy every warp is spread over all SMs (2^20.5 elements, B = 16: 64 -> 50 us).  Not for
// B = 32, where a CTA's warps then run apart and 16.8 M elements take 565 us instead of 538.
__host__ __device__ constexpr bool brute_spread(int B) { return B != 32; }
template <int B>
__device__ __forceinline__ size_t first_set() {   // of the warp, in groups
    if constexpr (!brute_spread(B)) return (size_t)blockIdx.x * kThreads + (threadIdx.x & ~31u);
    return ((size_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32;
}

// Stores a thread's results; blocks: how many of them the tensor has (fewer than NBT in its last group).
template <int B, int G>
__device__ __forceinline__ void store_group(const QuantArgs& p, size_t grp, int blocks, const uint32_t (&packed)[BruteShape<B, G>::G / 8],
                                            const uint32_t (&sc)[(BruteShape<B, G>::NBT + 3) / 4], const uint32_t (&sw)[BruteShape<B, G>::NBT]) {
    using S = BruteShape<B, G>;
    if (blocks == S::NBT) {
        store_bytes<S::G / 2>(p.codes + grp * (S::G / 2), packed);
        store_bytes<S::NBT>(p.scales + grp * S::NBT, sc);
        if (p.block_sse) store_bytes<4 * S::NBT>(p.block_sse + grp * S::NBT, sw);
    } else {
#pragma unroll
        for (int k = 0; k < S::NBT; ++k) {
            if (k >= blocks) break;
            const size_t b = grp * S::NBT + k;
            uint32_t w[(B + 7) / 8];
            if constexpr (B < 8) {
                w[0] = packed[k * B / 8] >> (4 * (k * B % 8));
            } else {
#pragma unroll
                for (int i = 0; i < B / 8; ++i) w[i] = packed[k * B / 8 + i];
            }
            store_bytes<B / 2>(p.codes + b * (B / 2), w);
            p.scales[b] = (uint8_t)(sc[k / 4] >> (8 * (k % 4)));
            if (p.block_sse) p.block_sse[b] = __uint_as_float(sw[k]);
        }
    }
}

// Their magnitudes (an SSE does not depend on signs): pair i = adjacent elements (one block per thread) or element i of
// either half.
template <int B, int G>
__device__ __forceinline__ GroupRange take_magnitudes(float2 (&v2)[BruteShape<B, G>::NP], float (&v)[BruteShape<B, G>::G]) {
    using S = BruteShape<B, G>;
    constexpr float kTiny = 2.168404344971009e-19f;  // 2^-62
    GroupRange r;
    r.amax = 0.0f;
    r.amin = __uint_as_float(0x7F800000u);
    r.has_zero = false;
#pragma unroll
    for (int i = 0; i < S::G; ++i) {
        v[i] = fabsf(v[i]);
        r.amax = fmaxf(r.amax, v[i]);
        r.amin = fminf(r.amin, v[i] == 0.0f ? __uint_as_float(0x7F800000u) : v[i]);
        r.has_zero |= v[i] == 0.0f;
    }
#pragma unroll
    for (int i = 0; i < S::NP; ++i) v2[i] = S::ONEBLK ? make_float2(v[2 * i], v[2 * i + 1]) : make_float2(v[i], v[S::NP + i]);
    r.fast = r.amax <= kFastMax && r.amin >= kTiny;
    return r;
}

// SSEs of all blocks of a thread when every element saturates, for the codes lo .. hi - 1: q = 6 and e = fma(6, -D, |v|).
template <int B, int G, typename Best>
__device__ __forceinline__ void search_saturated(const BruteTables& T, int lo, int hi, const float2 (&v2)[BruteShape<B, G>::NP],
                                                 Best& best) {
    using S = BruteShape<B, G>;
    if (lo >= hi) return;
    uint32_t cbest[S::NBT];
    int ccode[S::NBT];
#pragma unroll
    for (int k = 0; k < S::NBT; ++k) { cbest[k] = 0xFFFFFFFFu; ccode[k] = 0; }
    for (int c = lo; c < hi; c += 2) {
        const int cB = min(c + 1, hi - 1);   // an odd code out is evaluated twice
        const float nDA = -T.D[c], nDB = -T.D[cB];
        if constexpr (!S::ONEBLK) {
            const float2 six = make_float2(6.0f, 6.0f), A2 = make_float2(nDA, nDA), B2 = make_float2(nDB, nDB);
            float2 sA[S::NBL], sB[S::NBL];
#pragma unroll
            for (int k = 0; k < S::NBL; ++k) sA[k] = sB[k] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < S::NP; ++i) {
                const float2 eA = __ffma2_rn(six, A2, v2[i]), eB = __ffma2_rn(six, B2, v2[i]);
                sA[i / S::BL] = __ffma2_rn(eA, eA, sA[i / S::BL]);
                sB[i / S::BL] = __ffma2_rn(eB, eB, sB[i / S::BL]);
            }
#pragma unroll
            for (int k = 0; k < S::NBL; ++k) {
                keep_smaller(cbest[k], ccode[k], __float_as_uint(sA[k].x), c);
                keep_smaller(cbest[S::NBL + k], ccode[S::NBL + k], __float_as_uint(sA[k].y), c);
                keep_smaller(cbest[k], ccode[k], __float_as_uint(sB[k].x), cB);
                keep_smaller(cbest[S::NBL + k], ccode[S::NBL + k], __float_as_uint(sB[k].y), cB);
            }
        } else {
            float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < S::NP; ++i) {
                const float2 e0 = make_float2(__fmaf_rn(6.0f, nDA, v2[i].x), __fmaf_rn(6.0f, nDB, v2[i].x));
                s = __ffma2_rn(e0, e0, s);
                const float2 e1 = make_float2(__fmaf_rn(6.0f, nDA, v2[i].y), __fmaf_rn(6.0f, nDB, v2[i].y));
                s = __ffma2_rn(e1, e1, s);
            }
            keep_smaller(cbest[0], ccode[0], __float_as_uint(s.x), c);
            keep_smaller(cbest[0], ccode[0], __float_as_uint(s.y), cB);
        }
    }
#pragma unroll
    for (int k = 0; k < S::NBT; ++k) merge_class_winner(best[k], cbest[k], ccode[k]);
}

// The SSE of every code on every block of the warp's threads; best[k] receives the smallest of block k, ties to the smaller
// code.  Rg = RN(1 / g), or 0 for g beyond 2^+-60.
// Called by whole warps; `live` lanes take part.  Slice `slice` of `slices` covers its share of the codes.
//
// Three stretches of the codes need less than the full evaluation, and are the same for the whole warp (decode scales rise
// with the code; lo and hi are the warp's smallest nonzero and largest magnitude):
//   D <  lo * 2^-30   fl(|v| - 6 D) = |v|: the SSE is the sum of squares of the elements, and
//   D >= 4 hi         every quotient is at most 1/4 and rounds to 0: the same sum.  It is formed once and entered with the
//                     smallest of these codes, which is how the full evaluation of each would end.
//   D <= lo / 6       (no zero among the elements) every element saturates: the error is fl(|v| - 6 D), two packed FMAs
//                     per pair of elements and code instead of quotient, rounding, widening and two FMAs.
template <int B, int G, int FMT, typename Best>
__device__ __forceinline__ void search_group(const BruteTables& T, const float2 (&v2)[BruteShape<B, G>::NP], const GroupRange& gr, bool live,
                                             float Rg, int first, int slice, int slices, Best& best) {
    using S = BruteShape<B, G>;
    constexpr int NCLS = (FMT == kUE8M0) ? 1 : 8;
    constexpr int NC = num_codes(FMT);
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    const bool fast = live && gr.fast;
    const float hi = __uint_as_float(__reduce_max_sync(kFull, fast ? __float_as_uint(gr.amax) : 0u));
    const float lo = __uint_as_float(__reduce_min_sync(kFull, fast ? __float_as_uint(gr.amin) : 0x7F800000u));
    const bool zeros = __any_sync(kFull, fast && gr.has_zero);
    const float same_below = __fmul_rn(lo, 9.31322574615478515625e-10f /* 2^-30 */);
    const float sat_below = zeros ? 0.0f : __fmul_rn(lo, 0.1666f);
    const float zero_from = __fmul_rn(4.0f, hi);
    int c_same = 0, c_sat = 0, c_zero = 0;    // every code below c_same (c_sat) has its D below the limit, every one from c_zero on D >= 4 hi
    if (Rg != 0.0f && lo <= hi) {
        // from the limits' quotients by g, 2^-20 (far more than their rounding) to the safe side; code 0 of the FP8 formats is 0
        constexpr float kUp = 1.00000095367431640625f, kDown = 0.99999904632568359375f;
        constexpr int kZero = FMT == kUE8M0 ? 0 : 1;
        c_same = floor_code<FMT>(__fmul_rn(__fmul_rn(same_below, Rg), kDown)) + kZero;
        c_sat = floor_code<FMT>(__fmul_rn(__fmul_rn(sat_below, Rg), kDown));
        c_zero = floor_code<FMT>(__fmul_rn(__fmul_rn(zero_from, Rg), kUp)) + 1;
    } else {   // tensor scales beyond 2^+-60, or no nonzero element at all: by the table
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {
            const float D = T.D[32 * k + (threadIdx.x & 31)];   // NaN past the last code
            c_same += __popc(__ballot_sync(kFull, D < same_below));
            c_sat += __popc(__ballot_sync(kFull, D < sat_below));
            c_zero += __popc(__ballot_sync(kFull, D < zero_from));
        }
    }
    c_same = max(c_same, first);
    c_sat = max(c_sat, c_same);
    c_zero = max(c_zero, c_sat);
    if (fast) {
        const int zc = first < c_same ? first : c_zero;
        if (slice == 0 && zc < NC && fabsf(T.D[zc]) <= 3.402823466e38f) {
            if constexpr (!S::ONEBLK) {
                float2 s[S::NBL];
#pragma unroll
                for (int k = 0; k < S::NBL; ++k) s[k] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int i = 0; i < S::NP; ++i) s[i / S::BL] = __ffma2_rn(v2[i], v2[i], s[i / S::BL]);
#pragma unroll
                for (int k = 0; k < S::NBL; ++k) {
                    merge_class_winner(best[k], __float_as_uint(s[k].x), zc);
                    merge_class_winner(best[S::NBL + k], __float_as_uint(s[k].y), zc);
                }
            } else {
                float s = 0.0f;
#pragma unroll
                for (int i = 0; i < S::NP; ++i) {
                    s = __fmaf_rn(v2[i].x, v2[i].x, s);
                    s = __fmaf_rn(v2[i].y, v2[i].y, s);
                }
                merge_class_winner(best[0], __float_as_uint(s), zc);
            }
        }
        const int n = c_sat - c_same;
        search_saturated<B, G>(T, c_same + n * slice / slices, c_same + n * (slice + 1) / slices, v2, best);
        // the rest, one mantissa class after the other (slices share the classes, or the one class of the power-of-two format)
        for (int cls = NCLS == 1 ? 0 : slice; cls < NCLS; cls += NCLS == 1 ? 1 : slices) {
            int f0 = T.below[2 * cls][c_sat], n0 = T.below[2 * cls][c_zero] - f0;
            int f1 = T.below[2 * cls + 1][c_sat], n1 = T.below[2 * cls + 1][c_zero] - f1;
            if (NCLS == 1) {
                const int a0 = n0 * slice / slices, a1 = n1 * slice / slices;
                n0 = n0 * (slice + 1) / slices - a0;
                n1 = n1 * (slice + 1) / slices - a1;
                f0 += a0;
                f1 += a1;
            }
            if (n0 + n1 == 0) continue;
            const float Dr = T.clsD[cls], Rr = T.clsR[cls];
            const float2 nDr2 = make_float2(-Dr, -Dr), Rr2 = make_float2(Rr, Rr);
            float2 tb[S::NP];
#pragma unroll
            for (int i = 0; i < S::NP; ++i) tb[i] = quotient_pair(v2[i], nDr2, Rr2);
            search_list<B, FMT, false, S::ONEBLK>(T, 2 * cls, f0, n0, v2, tb, best);
            search_list<B, FMT, true, S::ONEBLK>(T, 2 * cls + 1, f1, n1, v2, tb, best);
        }
    }
    // general path (IEEE division), candidate by candidate
    const int n_general = live && !gr.fast ? NC - first : 0;
    const int c_end = first + n_general * (slice + 1) / slices;
    for (int c = first + n_general * slice / slices; c < c_end; ++c) {
        const float D = T.D[c];
        if (!(fabsf(D) <= 3.402823466e38f)) continue;  // decode scale overflowed: not usable
        if constexpr (!S::ONEBLK) {
#pragma unroll
            for (int k = 0; k < S::NBL; ++k) {
                merge_class_winner(best[k], __float_as_uint(general_sse<B, S::NP>(v2, k * S::BL, 0, D)), c);
                merge_class_winner(best[S::NBL + k], __float_as_uint(general_sse<B, S::NP>(v2, k * S::BL, 1, D)), c);
            }
        } else {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < S::NP; ++i) {
                const float a = v2[i].x, b = v2[i].y;
                const float2 q = round_e2m1x2(quotient_general(a, D), quotient_general(b, D));
                const float e0 = __fmaf_rn(-q.x, D, a);
                s = __fmaf_rn(e0, e0, s);
                const float e1 = __fmaf_rn(-q.y, D, b);
                s = __fmaf_rn(e1, e1, s);
            }
            merge_class_winner(best[0], __float_as_uint(s), c);
        }
    }
}

// One thread searches its elements under every code, all of them evaluated in full; whole groups only (n_items counts
// groups here).
template <int DT, int B, int G, int FMT>
__global__ void __launch_bounds__(kThreads, brute_min_ctas(B)) k_brute_plain(QuantArgs p) {
    constexpr bool ONEBLK = (G == B);         // the thread owns exactly one block
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
    build_brute_tables<FMT, false>(T, g, first);

    const size_t stride = (size_t)gridDim.x * kThreads;
    double sse_sum = 0.0;                  // binary64 sum of the SSEs of this thread's blocks, in the order it stored them
    for (size_t grp = first_set<B>() + (threadIdx.x & 31); grp < p.n_items; grp += stride) {
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
                search_list<B, FMT, false, ONEBLK>(T, 2 * cls, 0, n0, v2, tb, best);
                search_list<B, FMT, true, ONEBLK>(T, 2 * cls + 1, 0, n1, v2, tb, best);
            }
            if (T.flat_min < 256) {   // codes outside the lists: the sum of squares of the elements, see search_group()
                float2 s[NBL];
                float s1 = 0.0f;
#pragma unroll
                for (int k = 0; k < NBL; ++k) s[k] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    if constexpr (ONEBLK) {
                        s1 = __fmaf_rn(v2[i].x, v2[i].x, s1);
                        s1 = __fmaf_rn(v2[i].y, v2[i].y, s1);
                    } else {
                        s[i / BL] = __ffma2_rn(v2[i], v2[i], s[i / BL]);
                    }
                }
#pragma unroll
                for (int k = 0; k < NBL; ++k) {
                    merge_class_winner(best[k], __float_as_uint(ONEBLK ? s1 : s[k].x), T.flat_min);
                    if constexpr (!ONEBLK) merge_class_winner(best[NBL + k], __float_as_uint(s[k].y), T.flat_min);
                }
            }
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

// One thread searches its elements under all codes; the warp stays together, lanes past the end idle.
template <int DT, int B, int G, int FMT>
__global__ void __launch_bounds__(kThreads, brute_min_ctas(B)) k_brute(QuantArgs p) {
    using S = BruteShape<B, G>;
    __shared__ BruteTables T;
    constexpr bool kKeysInRegisters = brute_keys_in_registers(B, G, FMT);
    __shared__ unsigned long long key[kKeysInRegisters ? 1 : kThreads / 32][kKeysInRegisters ? 1 : 32 * S::NBT];   // per warp: block k of lane l at k * 32 + l
    wait_for_prior_grid();
    release_dependents();
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const int first = (p.prevent_zero && FMT != kUE8M0) ? 1 : 0;
    build_brute_tables<FMT, true>(T, g, first);
    const float Rg = g >= kFastMin && g <= kFastMax ? __frcp_rn(g) : 0.0f;

    const size_t n_groups = (p.n_items + S::NBT - 1) / S::NBT;
    const size_t stride = (size_t)gridDim.x * kThreads;
    const int lane = threadIdx.x & 31;
    typename std::conditional<kKeysInRegisters, RegisterBest<S::NBT>, const SharedBest>::type best = [&] {
        if constexpr (kKeysInRegisters) return RegisterBest<S::NBT>{};
        else return SharedBest{&key[threadIdx.x >> 5][lane]};
    }();
    double sse_sum = 0.0;                  // binary64 sum of the SSEs of this thread's blocks, in the order it stored them
    for (size_t wbase = first_set<B>(); wbase < n_groups; wbase += stride) {
        const size_t grp = wbase + lane;
        const bool active = grp < n_groups;
        const int blocks = active ? (int)min((size_t)S::NBT, p.n_items - grp * S::NBT) : 0;   // fewer in the last group
#pragma unroll
        for (int k = 0; k < S::NBT; ++k) best[k] = sse_key(__uint_as_float(0xFFFFFFFFu), first);
        float v[S::G];
        {
            float2 v2[S::NP];
            load_group<DT, B, G>(v, p.x, grp * S::G, blocks * B);
            const GroupRange gr = take_magnitudes<B, G>(v2, v);
            search_group<B, G, FMT>(T, v2, gr, active, Rg, first, 0, 1, best);
        }

        // final encode with the winners; the elements are read again (from L2) rather than kept with their signs
        load_group<DT, B, G>(v, p.x, grp * S::G, blocks * B);
        float amax = 0.0f;
#pragma unroll
        for (int i = 0; i < S::G; ++i) amax = fmaxf(amax, fabsf(v[i]));
        uint32_t packed[S::G / 8];
        uint32_t sc[(S::NBT + 3) / 4];
        uint32_t sw[S::NBT];
#pragma unroll
        for (int k = 0; k < (S::NBT + 3) / 4; ++k) sc[k] = 0;
        float t[S::G];
#pragma unroll
        for (int kb = 0; kb < S::NBT; ++kb) {
            const unsigned long long winner = best[kb];
            const int code = (int)(winner & 0xFFu);
            const float D = T.D[code];
            const float R = T.R[code];
            const bool fast = (R != 0.0f) && (amax <= kFastMax);
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int e = kb * B + i;
                t[e] = fast ? quotient_corrected(v[e], D, R) : quotient_general(v[e], D);
            }
            sc[kb / 4] |= (uint32_t)code << (8 * (kb % 4));
            sw[kb] = (uint32_t)(winner >> 32);
        }
#pragma unroll
        for (int k = 0; k < S::G / 8; ++k)
            packed[k] = pack_e2m1x8(t[8 * k], t[8 * k + 1], t[8 * k + 2], t[8 * k + 3], t[8 * k + 4], t[8 * k + 5], t[8 * k + 6], t[8 * k + 7]);
        store_group<B, G>(p, grp, blocks, packed, sc, sw);
#pragma unroll
        for (int k = 0; k < S::NBT; ++k)
            if (k < blocks) sse_sum = __dadd_rn(sse_sum, (double)__uint_as_float(sw[k]));
    }
    if (p.mse_partials != nullptr) {   // launch-uniform: fused tensor-MSE partial sum of this CTA
        __syncthreads();               // the tables are no longer read: their memory serves as scratch
        const double total = cta_sum_fixed_order(sse_sum, reinterpret_cast<double*>(&T));
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

// The same search for tensors that do not fill the chip with one thread per group: `slices` warps (2, 4 or 8) of a CTA share
// 32 groups and take their part of the codes each (mantissa classes of the FP8 formats); the winners meet in shared
// memory and the CTA encodes the elements together.
template <int DT, int B, int G, int FMT>
__global__ void __launch_bounds__(kThreads, brute_min_ctas(B)) k_brute_split(QuantArgs p, int slices) {
    using S = BruteShape<B, G>;
    constexpr int W = kThreads / 32;
    constexpr int EPT = 32 * S::G / kThreads;      // elements of 32 groups that a thread encodes: at most one block
    constexpr int NBW = 32 * S::NBT;               // blocks of 32 groups
    __shared__ BruteTables T;
    __shared__ unsigned long long key[W][NBW];     // per warp: best of block k of lane l at k * 32 + l
    wait_for_prior_grid();
    release_dependents();
    const float g = p.d_global_scale ? *p.d_global_scale : p.global_scale;
    const int first = (p.prevent_zero && FMT != kUE8M0) ? 1 : 0;
    build_brute_tables<FMT, true>(T, g, first);
    const float Rg = g >= kFastMin && g <= kFastMax ? __frcp_rn(g) : 0.0f;

    const size_t n_groups = (p.n_items + S::NBT - 1) / S::NBT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sets = W / slices;                   // sets of 32 groups the CTA works on
    double sse_sum = 0.0;
    for (size_t base = (size_t)blockIdx.x * (sets * 32); base < n_groups; base += (size_t)gridDim.x * (sets * 32)) {
        {
            const size_t grp = base + warp / slices * 32 + lane;
            const int blocks = grp < n_groups ? (int)min((size_t)S::NBT, p.n_items - grp * S::NBT) : 0;
            float v[S::G];
            float2 v2[S::NP];
            load_group<DT, B, G>(v, p.x, grp * S::G, blocks * B);
            const GroupRange gr = take_magnitudes<B, G>(v2, v);
            const SharedBest best = {&key[warp][lane]};
#pragma unroll
            for (int k = 0; k < S::NBT; ++k) best[k] = sse_key(__uint_as_float(0xFFFFFFFFu), first);
            search_group<B, G, FMT>(T, v2, gr, grp < n_groups, Rg, first, warp % slices, slices, best);
        }
        __syncthreads();
        for (int set = 0; set < sets; ++set) {
            const size_t e0 = (base + set * 32) * S::G + threadIdx.x * EPT;
            const int b = threadIdx.x * EPT / B;   // block of the set, in memory order
            const size_t blk = e0 / B;
            if (blk < p.n_items) {
                const int at = (b % S::NBT) * 32 + b / S::NBT;
                unsigned long long k = key[set * slices][at];
                for (int w = 1; w < slices; ++w) k = min(k, key[set * slices + w][at]);
                const int code = (int)(k & 0xFFu);
                const float D = T.D[code], R = T.R[code];
                float v[EPT];
                load_elems<DT, EPT>(p.x, e0, v);
                uint32_t packed = 0;
#pragma unroll
                for (int i = 0; i < EPT; i += 2) {
                    const bool fast = R != 0.0f && fmaxf(fabsf(v[i]), fabsf(v[i + 1])) <= kFastMax;
                    const float t0 = fast ? quotient_corrected(v[i], D, R) : quotient_general(v[i], D);
                    const float t1 = fast ? quotient_corrected(v[i + 1], D, R) : quotient_general(v[i + 1], D);
                    packed |= pack_e2m1x2(t0, t1) << (4 * i);
                }
                store_bytes<EPT / 2>(p.codes + e0 / 2, &packed);
                if (e0 % B == 0) {
                    const float sse = __uint_as_float((uint32_t)(k >> 32));
                    p.scales[blk] = (uint8_t)code;
                    if (p.block_sse) p.block_sse[blk] = sse;
                    sse_sum = __dadd_rn(sse_sum, (double)sse);
                }
            }
        }
        __syncthreads();   // the keys have been read
    }
    if (p.mse_partials != nullptr) {
        const double total = cta_sum_fixed_order(sse_sum, reinterpret_cast<double*>(&T));
        if (threadIdx.x == 0) p.mse_partials[p.mse_first + blockIdx.x] = total;
    }
}

template <int DT, int B, int FMT, int G>
static cudaError_t launch_brute_size(const QuantArgs& a, int slices, cudaStream_t stream) {
    using S = BruteShape<B, G>;
    static std::atomic<int> cache[3][kMaxDevices];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const size_t n_groups = (a.n_items + S::NBT - 1) / S::NBT;
    const size_t sms = (size_t)sm_count(dev);
    // Under a tensor scale the codes of UE4M3 reach from the top of the tensor down by 17 binades only: next to none lies in
    // the cheap stretches of search_group(), and the kernel without them is faster by the registers they take (16.8 M fp32
    // Laplace elements, with -> without, us: B = 2 534 -> 499, 4 458 -> 440, 8 393 -> 371, 16 385 -> 367, 64 427 -> 420; B = 32
    // 385 -> 391).  The other formats gain (all codes in full -> with, B = 16): UE5M3 678 -> 532, UE8M0 650 -> 115.  So does unscaled
    // UE4M3 of weights (322 -> 167) and of N(0, 1) (322 -> 242).  Where its elements lie at the top of the codes or all over them
    // there is little to skip, which only the kernel can see: N(0, 300) 322 -> 318, activations with outlier columns 322 -> 323; bf16
    // loses most, outlier columns at B = 8 and 16 3 % (317 -> 326, 302 -> 311), exponents drawn from 22 binades 5 %.
    constexpr bool kHasPlain = FMT == kUE4M3 && B != 32;
    const bool plain = kHasPlain && slices == 1 && (a.d_global_scale != nullptr || a.global_scale != 1.0f);
    const void* kernel = reinterpret_cast<const void*>(k_brute<DT, B, G, FMT>);
    if (slices > 1) kernel = reinterpret_cast<const void*>(k_brute_split<DT, B, G, FMT>);
    if constexpr (kHasPlain) {
        if (plain) kernel = reinterpret_cast<const void*>(k_brute_plain<DT, B, G, FMT>);
    }
    size_t cap = 0;
    err = resident_ctas(kernel, 0, dev, cache[slices > 1 ? 1 : plain ? 2 : 0], cap);
    if (err != cudaSuccess) return err;
    cap *= sms;
    if (a.mse_partials && cap > (size_t)kMsePartials) cap = kMsePartials;
    const unsigned per_cta = slices > 1 ? (unsigned)(kThreads / slices) : brute_spread(B) ? 32u : (unsigned)kThreads;
    auto ctas = [&](size_t groups) {
        const size_t want = (groups + per_cta - 1) / per_cta;
        return (unsigned)(want < cap ? want : cap);
    };
    unsigned grid = ctas(n_groups), rest = 0;
    if (slices > 1) {
        err = launch_pdl(k_brute_split<DT, B, G, FMT>, grid, kThreads, 0, stream, a, slices);
    } else if (!plain) {
        err = launch_pdl(k_brute<DT, B, G, FMT>, grid, kThreads, 0, stream, a);
    } else if constexpr (kHasPlain) {
        // whole groups; the blocks past the last one go to the split kernel (one CTA, partial sum 0)
        QuantArgs m = a;
        m.n_items = a.n_items / S::NBT;
        const size_t done = m.n_items * S::NBT;
        if (done < a.n_items) {
            QuantArgs t = a;
            t.x = static_cast<const char*>(a.x) + done * B * elem_bytes(DT);
            t.codes = a.codes + done * B / 2;
            t.scales = a.scales + done;
            if (a.block_sse) t.block_sse = a.block_sse + done;
            t.n_items = a.n_items - done;
            rest = 1;
            err = launch_pdl(k_brute_split<DT, B, G, FMT>, 1u, kThreads, 0, stream, t, 8);
            count_launch();
            if (err != cudaSuccess) return err;
        }
        m.mse_first = (int)rest;
        if (a.mse_partials && cap > (size_t)kMsePartials - rest) cap = kMsePartials - rest;
        grid = ctas(m.n_items);
        err = launch_pdl(k_brute_plain<DT, B, G, FMT>, grid, kThreads, 0, stream, m);
    }
    count_launch();
    if (err == cudaSuccess && a.mse_n_partials) *a.mse_n_partials = (int)(grid + rest);
    return err;
}

template <int DT, int B, int FMT>
static cudaError_t launch_brute_inst(const QuantArgs& a, cudaStream_t stream) {
    int dev = 0;
    const cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    constexpr int G = brute_group_elems(B);
    const size_t n_groups = (a.n_items * B + G - 1) / G;
    const size_t sms = (size_t)sm_count(dev);
    const size_t per_sm = (n_groups + sms - 1) / sms;
    // A tensor with fewer groups than threads that fit leaves SMs idle or with too few warps.  Up to 32, 64, 128 groups per
    // SM its groups are split over 8, 4, 2 warps.  Beside and beyond that groups of 16 help B = 8 up to four million elements,
    // and B = 16 in a short stretch (a pair of lanes then holds two codes instead of two blocks; UE8M0, with few full
    // evaluations, does not mind).  fp32 Laplace under a tensor scale, UE4M3, us, groups of 32 not split -> as chosen here: 2^16
    // elements, B = 8 42 -> 19, B = 16 41 -> 18; 2^18 40 -> 23, 39 -> 23; 2^19 40 -> 28, 39 -> 28; 2^19.5 40 -> 32, 40 ->
    // 33; 2^21.5 88 -> 81 (B = 8).
    if constexpr (B == 8 || B == 16) {
        const bool small = B == 8 ? (per_sm > 64 && per_sm <= 1024) : (per_sm > 128 && (per_sm <= 200 || FMT == kUE8M0));
        if (small) return launch_brute_size<DT, B, FMT, 16>(a, 1, stream);
    }
    // (256, 384] at B = 32: without the spreading some SMs would get a second CTA of 256 groups and the others one (68 -> 58 us)
    const int slices = per_sm <= 32 ? 8 : per_sm <= 64 ? 4 : (per_sm <= 128 || (!brute_spread(B) && per_sm > 256 && per_sm <= 384)) ? 2 : 1;
    return launch_brute_size<DT, B, FMT, G>(a, slices, stream);
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
