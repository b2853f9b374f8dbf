// Bit-sliced decode of narrow widths.
//
// A thread's share of a 1024-value block is 32 codes in B words (one lane's
// stream).  Instead of extracting the codes one by one, the B words are
// rearranged into B slices: slice i holds bit i of all 32 codes, one code per
// bit position.  COUNT and SUM do not care which position holds which code, so
// the rearrangement only has to use the same order in every slice, and it needs
// no extraction at all for the odd part of the width:
//   write B = m * 2^k, m odd, and cut the stream into 2^k segments of m words,
//   each holding D = 32 / 2^k whole codes of m digits of 2^k bits.  At digit
//   position p, word w of a segment holds digit (D*w + p) mod m of some code: over
//   the m words every digit occurs once, in the order of a rotation by p.  A
//   barrel shifter whose rotation depends on the bit position (a bit select per
//   word and binary digit of m, one constant mask per stage) therefore collects
//   digit j of every code into one word, and a rotation by j digits brings code c
//   to position m*c mod D for every j.  k butterfly stages over the 2^k segments
//   then split the digits into bits (a shift and a select per word and stage).
// Per 32 codes that is 8 ALU operations at B = 3, 19 at 5, 25 at 6, 27 at 7, 36 at 8,
// 44 at 9, 53 at 10, 68 at 12 and 75 at 14, with the left one of the two shifts per pair
// of words and butterfly stage as a multiplication on the FMA pipe beside them.
//
// The range test then runs on all 32 codes at once: u >= lo and u > hi are
// carry chains of B majorities (one LOP3 each) from the lowest bit up, the count
// is one POPC of the match mask, and the sum is the B weighted POPCs of the
// masked slices.
#pragma once
#include <cstdint>

namespace gb {

__host__ __device__ constexpr int slice_segments(int b) { return b & -b; }        // 2^k
__host__ __device__ constexpr int slice_odd(int b) { return b / slice_segments(b); }  // m

// Constant masks, folded by the compiler into immediates.
template <int B>
struct SliceMasks {
    uint32_t turn[5];  // [e]: digit positions p with bit e of p mod m set
    uint32_t low[5];   // [e]: bit positions p with bit e clear
    __host__ __device__ constexpr SliceMasks() : turn{}, low{}
    {
        constexpr int s = slice_segments(B), m = slice_odd(B), d = 32 / s;
        for (int e = 0; e < 5; ++e) {
            for (int p = 0; p < d; ++p)
                if (((p % m) >> e) & 1) turn[e] |= (s == 32 ? 0xffffffffu : ((1u << (s & 31)) - 1u)) << (p * s);
            for (int p = 0; p < 32; ++p)
                if (((p >> e) & 1) == 0) low[e] |= 1u << p;
        }
    }
};

// Left shifts as multiplications by 2^t, opaque to the compiler: the integer ALU
// is the busy pipe here (bit selects, rotations, majorities), the FMA pipe has room.
// (A right shift as a high-word product takes that pipe four cycles; with those
// too the scan was 1-3% slower at B = 8, 10 and 12.)
struct SliceShifts {
    uint32_t mul[5];  // 2^(1 << e)
};

// (a & mask) | (b & ~mask).  On the device spelled out as one LOP3: written as the
// expression the scans took up to 1.28 times as long (2^28 values, us, expression / spelled
// out: 34.8 / 30.8 at b = 5, 51.3 / 43.8 at 8, 77.9 / 63.7 at 12, branchy 101.3 / 81.9 at 16).
#ifdef __CUDA_ARCH__
__device__ __forceinline__ uint32_t bit_select(uint32_t a, uint32_t b, uint32_t mask)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xE4;" : "=r"(d) : "r"(a), "r"(b), "r"(mask));
    return d;
}
__device__ __forceinline__ uint32_t slice_shl(uint32_t x, int e, const SliceShifts& P)
{
    uint32_t d;
    asm("mul.lo.u32 %0, %1, %2;" : "=r"(d) : "r"(x), "r"(P.mul[e]));
    return d;
}
#else
inline uint32_t bit_select(uint32_t a, uint32_t b, uint32_t mask) { return (a & mask) | (b & ~mask); }
inline uint32_t slice_shl(uint32_t x, int e, const SliceShifts&) { return x << (1 << e); }
#endif

// W: the 32 codes of one lane, stream order.  X[i]: bit i of every code.
template <int B>
__host__ __device__ __forceinline__ void to_slices(const uint32_t (&W)[B], uint32_t (&X)[B], const SliceShifts& P)
{
    constexpr int kS = slice_segments(B), kM = slice_odd(B);
    constexpr SliceMasks<B> kMask{};
#pragma unroll
    for (int g = 0; g < kS; ++g) {
        uint32_t R[kM];
#pragma unroll
        for (int w = 0; w < kM; ++w) R[32 / kS * w % kM] = W[g * kM + w];
#pragma unroll
        for (int e = 0; (1 << e) < kM; ++e) {
            uint32_t T[kM];
#pragma unroll
            for (int j = 0; j < kM; ++j) T[j] = bit_select(R[(j + kM - (1 << e)) % kM], R[j], kMask.turn[e]);
#pragma unroll
            for (int j = 0; j < kM; ++j) R[j] = T[j];
        }
#pragma unroll
        for (int j = 0; j < kM; ++j) {
            const int r = j * kS;
            X[j * kS + g] = r ? (R[j] >> r) | (R[j] << (32 - r)) : R[j];
        }
    }
#pragma unroll
    for (int e = 4; e >= 0; --e) {
        const int t = 1 << e;
        if (t >= kS) continue;
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if ((i % kS) & t) continue;
            const uint32_t a = X[i], c = X[i + t];
#ifdef __CUDA_ARCH__
            if (e == 3) {  // whole bytes: one permute for a shift and a select
                X[i] = __byte_perm(a, c, 0x6240);
                X[i + t] = __byte_perm(a, c, 0x7351);
                continue;
            }
#endif
            X[i] = bit_select(a, slice_shl(c, e, P), kMask.low[e]);
            X[i + t] = bit_select(a >> t, c, kMask.low[e]);
        }
    }
}

// Bit position of code r (row r of a lane) in the slices.
template <int B>
__host__ __device__ constexpr int slice_position(int r)
{
    constexpr int s = slice_segments(B), d = 32 / s;
    return slice_odd(B) * (r % d) % d * s + r / d;
}

// Block layouts.  A word of a power-of-two width holds whole codes in both, so there
// the lane decode reads a row-major block too.
enum Layout : int { kLayLanes = 0, kLayRow = 1 };
__host__ __device__ constexpr int row_decode(int b) { return slice_odd(b) == 1 ? kLayLanes : kLayRow; }

// The widths decoded this way.  The sliced decode costs less the narrower the
// width; the direct one (an extraction, a compare and an add per code, and a vote
// in the branchy flavour) about the same at every width, so it stays where the
// bandwidth binds it anyway.  Direct against sliced, 2^28 values, us per scan:
//   lane layout, branch-free: 57 / 13.5 at b = 1, 56.7 / 30.9 at 5, 56.8 / 44.4 at 8,
//     57.4 / 54.4 at 10, 62.5 / 64.5 at 12 (67.8 / 64.5 with the built-in shapes),
//     66.7 / 68.1 at 13;
//   lane layout, branchy: 90 / 14.4 at b = 1, 94 / 65.4 at 12, 102.6 / 77.4 at 15,
//     108.6 / 82.2 at 16, 86.0 / 91.8 at 17 (best shapes);
//   row-major: 61 / 13.4 at b = 1, 79.5 / 70.3 at 13, 80 / 76.6 at 15 branch-free.
__host__ __device__ constexpr bool sliced(int b, bool branchy, int lay = kLayLanes)
{
    return b <= (branchy ? 16 : (lay == kLayRow ? 15 : 12));
}

// Bounds of the range test in slice form: a code bit's majority with the running
// carry and an all-ones word where the bound's bit is 0, all zeros where it is 1.
template <int B>
struct SliceKeys {
    uint32_t lo[B], hi[B];  // lo' and hi' - 1
    SliceShifts shift;      // shift.mul[0] = 2 also weighs the sum
};

#ifdef __CUDACC__
template <int B>
__device__ __forceinline__ SliceKeys<B> make_slice_keys(uint32_t lo, uint32_t wm1, uint32_t one)
{
    SliceKeys<B> K;
    const uint32_t last = lo + wm1;  // the largest matching code
#pragma unroll
    for (int i = 0; i < B; ++i) {
        K.lo[i] = ((lo >> i) & 1u) - 1u;
        K.hi[i] = ((last >> i) & 1u) - 1u;
    }
#pragma unroll
    for (int e = 0; e < 5; ++e) K.shift.mul[e] = one << (1 << e);
    return K;
}

__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Match mask of 32 codes: lo <= u (ge) and not u > last (gt).
template <int B>
__device__ __forceinline__ uint32_t slice_match(const uint32_t (&X)[B], const SliceKeys<B>& K)
{
    uint32_t ge = 0xffffffffu, gt = 0u;
#pragma unroll
    for (int i = 0; i < B; ++i) {
        ge = majority(X[i], ge, K.lo[i]);
        gt = majority(X[i], gt, K.hi[i]);
    }
    return ge & ~gt;
}

// Sum of the codes under the mask m: Horner's rule over the slices' POPCs.
template <int B>
__device__ __forceinline__ uint32_t slice_sum(const uint32_t (&X)[B], uint32_t m, const SliceKeys<B>& K)
{
    uint32_t s = 0u;
#pragma unroll
    for (int i = B - 1; i >= 0; --i) {
        const uint32_t c = static_cast<uint32_t>(__popc(X[i] & m));
        asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(s) : "r"(s), "r"(K.shift.mul[0]), "r"(c));
    }
    return s;
}
#endif

}  // namespace gb
