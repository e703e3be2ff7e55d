// Shared pieces of the coset-split kernels (split_linear.cu, split_bwd_weight.cu): what the split is, and its register form.
//
// Let z be the central involution of a cyclic group of even order, the rotation by half a turn.  It splits the layer into two
// independent ones on half as many features,
//     x+[j] = x[j] + x[zj],   x-[j] = x[j] - x[zj]          j over one representative of every pair {j, zj}
//     y[g]  = y+[g] + y-[g],  y[zg] = y+[g] - y-[g],        y+- = x+- . W+-,   W+- = (w[h^-1 g] +- w[h^-1 z g]) / 2
// -- the first butterfly of the group DFT and nothing more.  The two products are dense matrix products of half the
// width each, i.e. half of the unrolled layer's multiplications.  That is more arithmetic than the full DFT's
// (T^2 / 2 products per channel pair against 2T - 2), but it comes as two long GEMMs the tensor cores run at their full
// rate, while the per-frequency products are bound by the shared-memory traffic of their many small operand tiles and
// the full transform by its instructions.
//
// Of 16-bit data x+ and x- are rounded to the 16-bit type, as the spectra of the full transform are, and a half-precision sum of
// two can pass its range.  So the split is for the orders whose 16-bit plans round a transform of their operands anyway (4, 8, 16,
// 32; the linear passes of 2).  The other groups -- odd orders, 6, 12, the dihedral groups, the weight gradient of order 2 -- run
// the same kernels unsplit: one dense product on the inputs as they are, operands straight from TMA.
//
// Features are viewed as [..., 2, D]: element e and its partner e + D, D = half the number of rotations.
#pragma once

#include "eql_internal.h"
#include "ptx_sm100.cuh"
#include "umma_common.cuh"

namespace eql {

// ---- tcgen05 operand descriptors with 128-byte swizzle ------------------------------------------------------------
// K-major tile: rows of 128 bytes (64 halves along K), 8-row groups 1024 bytes apart, 16-byte chunk c of row r at
// c ^ (r & 7).  A K step of 16 halves advances the start address by 32 bytes.  Tile base 1024-byte aligned.
__device__ __forceinline__ uint64_t desc_k_sw128(uint32_t smem_addr) {
    return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// MN-major tile: a block is 64 elements along M / N (128 bytes) x the K rows, rows 128 bytes apart, 16-byte chunk c of
// row k at c ^ (k & 7); 8-row groups along K 1024 bytes apart, blocks `mn_block_bytes` apart.
__device__ __forceinline__ uint64_t desc_mn_sw128(uint32_t smem_addr, uint32_t mn_block_bytes) {
    return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | ((uint64_t)((mn_block_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// ---- 16 bytes of representatives and their partners --------------------------------------------------------------
// A raw row piece of 128 bytes (64 elements, one TMA box row with 128-byte swizzle: 16-byte chunk j of row r at j ^ (r & 7))
// holds four "granules" of 8 representatives and their 8 partners, each two chunks:
//   D <= 8: chunks 2g and 2g + 1;   D = 16: a chunk of a 64-byte tuple's first half and the one two behind it.
// A warp takes 8 rows x 4 granules at a time.  The 8 lanes of a shared-memory wavefront hold two rows; the kernels choose which
// two, so that they never meet in a bank.
template <int D>
__device__ __forceinline__ int granule_chunk(int g) { return D == 16 ? (g >> 1) * 4 + (g & 1) : 2 * g; }
template <int D>
constexpr int kPartnerChunk = D == 16 ? 2 : 1;                 // chunks from a to b

__device__ __forceinline__ uint4 lds128(const uint8_t* p) { return *reinterpret_cast<const uint4*>(p); }

template <typename IO>
__device__ __forceinline__ uint32_t add2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr (H16<IO>::kIsHalf) asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
template <typename IO>
__device__ __forceinline__ uint32_t sub2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr (H16<IO>::kIsHalf) asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// The butterfly on packed 16-bit pairs: a sum or difference of two 16-bit numbers, rounded once -- the same value as
// adding in float and rounding.
template <int D, typename IO>
__device__ __forceinline__ void split_granule(const uint4& a, const uint4& b, uint4& p, uint4& m) {
    if constexpr (D >= 8) {
        p = make_uint4(add2<IO>(a.x, b.x), add2<IO>(a.y, b.y), add2<IO>(a.z, b.z), add2<IO>(a.w, b.w));
        m = make_uint4(sub2<IO>(a.x, b.x), sub2<IO>(a.y, b.y), sub2<IO>(a.z, b.z), sub2<IO>(a.w, b.w));
    } else if constexpr (D == 4) {
        p = make_uint4(add2<IO>(a.x, a.z), add2<IO>(a.y, a.w), add2<IO>(b.x, b.z), add2<IO>(b.y, b.w));
        m = make_uint4(sub2<IO>(a.x, a.z), sub2<IO>(a.y, a.w), sub2<IO>(b.x, b.z), sub2<IO>(b.y, b.w));
    } else if constexpr (D == 2) {
        p = make_uint4(add2<IO>(a.x, a.y), add2<IO>(a.z, a.w), add2<IO>(b.x, b.y), add2<IO>(b.z, b.w));
        m = make_uint4(sub2<IO>(a.x, a.y), sub2<IO>(a.z, a.w), sub2<IO>(b.x, b.y), sub2<IO>(b.z, b.w));
    } else {
        static_assert(D == 1, "pair distance");
        const uint32_t l0 = __byte_perm(a.x, a.y, 0x5410), h0 = __byte_perm(a.x, a.y, 0x7632);
        const uint32_t l1 = __byte_perm(a.z, a.w, 0x5410), h1 = __byte_perm(a.z, a.w, 0x7632);
        const uint32_t l2 = __byte_perm(b.x, b.y, 0x5410), h2 = __byte_perm(b.x, b.y, 0x7632);
        const uint32_t l3 = __byte_perm(b.z, b.w, 0x5410), h3 = __byte_perm(b.z, b.w, 0x7632);
        p = make_uint4(add2<IO>(l0, h0), add2<IO>(l1, h1), add2<IO>(l2, h2), add2<IO>(l3, h3));
        m = make_uint4(sub2<IO>(l0, h0), sub2<IO>(l1, h1), sub2<IO>(l2, h2), sub2<IO>(l3, h3));
    }
}

// ---- group arithmetic on representatives ---------------------------------------------------------------------------
// Element r^t s^f as (f, t), t in [0, R) with R rotations; cyclic groups have f = 0 only.  With a split, representatives
// are t in [0, R/2), numbered f * R/2 + t, and a product may come out as z times a representative.
// REPS representatives per channel, DIH dihedral, S products (2: split): everything below folds when h or q is a constant.
template <int REPS, bool DIH, int S>
struct Reps {
    static constexpr int kHalf = DIH ? REPS / 2 : REPS;        // rotations a representative set holds
    static constexpr int kRot = kHalf * S, kTuple = REPS * S;
    static __device__ __forceinline__ int element(int rep) { return (rep / kHalf) * kRot + rep % kHalf; }   // position in a tuple
    // h q (PRODUCT) or h^-1 q -> representative; `z` says whether it came out times z
    template <bool PRODUCT>
    static __device__ __forceinline__ int combine(int h, int q, bool& z) {
        const int f1 = h / kHalf, a = h % kHalf, f2 = q / kHalf, b = q % kHalf;
        // (r^a s^f1)(r^b s^f2) = r^(a +- b) s^(f1+f2);  (r^a s^f1)^-1 (r^b s^f2) = s^f1 r^(b-a) s^f2 = r^(+-(b-a)) s^(f1+f2)
        int t = PRODUCT ? (f1 ? a - b : a + b) : (f1 ? a - b : b - a);
        if (t < 0) t += kRot;
        if (t >= kRot) t -= kRot;
        z = S == 2 && t >= kHalf;
        return (f1 ^ f2) * kHalf + (z ? t - kHalf : t);
    }
};

// Calls f(Reps<...>{}) for the group of a shape; S is a constant of the kernel.
template <int S, typename F>
__host__ __device__ __forceinline__ bool with_reps(int reps, bool dih, F&& f) {
    if constexpr (S == 2) {
        switch (reps) {
            case 1: f(Reps<1, false, 2>{}); return true;
            case 2: f(Reps<2, false, 2>{}); return true;
            case 4: f(Reps<4, false, 2>{}); return true;
            case 8: f(Reps<8, false, 2>{}); return true;
            case 16: f(Reps<16, false, 2>{}); return true;
            default: return false;
        }
    } else {
        if (dih) switch (reps) {
            case 4: f(Reps<4, true, 1>{}); return true;
            case 6: f(Reps<6, true, 1>{}); return true;
            case 8: f(Reps<8, true, 1>{}); return true;
            case 10: f(Reps<10, true, 1>{}); return true;
            case 12: f(Reps<12, true, 1>{}); return true;
            case 16: f(Reps<16, true, 1>{}); return true;
            default: return false;
        }
        switch (reps) {
            case 1: f(Reps<1, false, 1>{}); return true;
            case 2: f(Reps<2, false, 1>{}); return true;
            case 3: f(Reps<3, false, 1>{}); return true;
            case 5: f(Reps<5, false, 1>{}); return true;
            case 6: f(Reps<6, false, 1>{}); return true;
            case 7: f(Reps<7, false, 1>{}); return true;
            case 12: f(Reps<12, false, 1>{}); return true;
            default: return false;
        }
    }
}

// The same for the groups of pair distance D (0: unsplit): D representatives of a cyclic group.
template <int D, typename F>
__device__ __forceinline__ void with_reps_of(int reps, bool dih, F&& f) {
    if constexpr (D == 0) with_reps<1>(reps, dih, f);
    else f(Reps<D, false, 2>{});
}

}  // namespace eql
