// Weight gradient of the coset-split dense products (16-bit inputs, or float as 3xTF32; FP32 accumulation; see split_common.cuh):
//   D+-[(i,h), (o,g)] = sum_n x+-[n, (i,h)] dy+-[n, (o,g)]            two products over all tokens (unsplit: one)
//   dw[o, i, q] = 1/2 sum_h (D+[h, hq] + sgn D-[h, hq]),  dw[o, i, zq] = 1/2 sum_h (D+[h, hq] - sgn D-[h, hq])
// by CTA pairs with tcgen05.mma.cta_group::2.  A pair owns a tile of 256 x nb entries of both products for one range of
// tokens; M and N may be either of x and dy, whichever fills the tiles better.
//
//   2 threads  TMA: raw rows of x and of dy, 32 tokens x 256 columns per stage, into one ring slot; operand tiles where no
//              arithmetic is needed (unsplit layers: both sides, 64 tokens; the halves of x that the forward pass saved)
//   16 warps   in place, two raw slabs [32 tokens x 64 elements] -> the MN-major operand blocks [32 tokens x 64 columns] of x+
//              and x-, 128-byte swizzle: a token's columns stay contiguous, so no transposition happens anywhere; db from the
//              unrounded rows
//   1 warp     tcgen05.mma, K = 16 tokens per step
//   16 warps   (after the loop) accumulators -> shared memory, the sum over h, partial dw
//
// The sum over h happens before anything is written, so the partial sums of a token range are the size of dw.
//
// Bounds: shared memory.  A stage of 32 tokens at nb = 256 is 32 KB each written by TMA, read and written by the transform and read
// by the MMAs, ~930 cycles, of which the MMAs take 512.  Behind the loop, the sums of db cost 1.3 K cycles (11 K when 64 rows of
// partial sums went through shared memory: the tokens of a warp are added by shuffles first) and dw ~7 K.  T = 16, 64 -> 64 channels,
// 65536 tokens: 109 us on the frequency-domain kernels, 83 here; dihedral group of order 8, 48 -> 96 channels, 12608 tokens: 22.
//
// Unsplit layers: the groups whose products are of exact inputs, so that the additions decide the error.  Two accumulators take two
// stages in turn; the warps behind the ring add each to float registers while the other fills.  Relative error of dw, 12608 tokens,
// order 3, 128 -> 256 channels: 1.7e-6 with one accumulator per range, 2.1e-7 so; 4.5e-7 on the CUDA cores.  p6, 92 -> 60 channels,
// 10007 tokens: 18.7 / 19.6 us.  (The copy thread answers for the stages whose db another pair sums: with all 16 warps at every stage
// their ~150 instructions per warp bound the loop, 1100 cycles per stage against 700.)
//
// Float: two passes over the tokens, the small products first, as in the linear kernel, which has the reason.  Tokens are the K
// dimension of a K-major TF32 operand (an MN-major one is not available at 32 bits), so the transform also transposes, four tokens
// by four representatives in registers.  T = 4, 256 -> 256 channels, 32768 tokens: 441 us in ten blocks of tokens on the
// frequency-domain kernels, 238 here; the error is half of theirs (9.8e-7 against 2.2e-6 of the largest |dw|).
#include <cuda_fp16.h>

#include <atomic>

#include "split_common.cuh"
#include "tensor_map.h"

namespace eql {
namespace {

constexpr int kThreadsSbw = 640;
constexpr int kWarpTmaM = 0, kWarpMma = 1, kWarpTmaN = 2, kWarpX0 = 4, kXWarps = 16, kXThreads = kXWarps * 32;
constexpr int kMaxStages = 8;
constexpr int sbw_tokens(int S, int elem) { return elem == 4 ? 16 : S == 2 ? 32 : 64; }      // tokens per stage
constexpr int kDrainStages = 2;                // unsplit: stages per accumulator
constexpr int kRoleRegs = 56, kXRegs = 104;    // unsplit: registers of the four role warps and of the sixteen behind the ring

struct SbwParams {
    float* part;                 // [splits][out channels][in channels][tuple] of this launch's tiles
    float* db_part;              // [splits * shares][Co]
    int* status;
    int64_t N, total_stages, stages_per_split;
    int m_slabs, n_slabs;        // raw tensor maps bring whole slabs of 128 bytes of a row in one copy
    int wM, wN;                  // valid columns of a CTA's 128 x nb/2 block of each product
    int nb, mTiles, nTiles, mt0, nt0;        // tiles of this launch, the first of either side
    int o0, i0, iCount;          // first channels of the launch's tiles, input channels they cover
    int64_t part_stride;         // entries of a token range's partial sums
    int m_is_y, shares;          // dy on M; pairs that share a dy tile (each sums db over its share of the stages)
    int stages, stage_bytes;     // ring slots
    int Ci, Co, tuple, corr, reps, dihedral;
};

struct SbwBarriers {
    uint64_t full[kMaxStages], empty[kMaxStages], raw_full[kMaxStages];
    uint64_t full_d[2], empty_d[2], mma_done;      // (split: full_d[0] alone; unsplit: an accumulator each)
    uint32_t tmem_base;
    int abort_flag, go;
};

// Adds the 16 raw elements of a granule to one sum per group of min(8, D) representatives and their partners.
template <int D, typename IO>
__device__ __forceinline__ void add_granule(const uint4& a, const uint4& b, float* acc) {
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    constexpr int PER = D >= 8 ? 8 : D;                          // words per sum: min(8, D) pairs = 2 min(8, D) elements
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 f = H16<IO>::unpack(w[i]);
        acc[i / PER] += f.x + f.y;
    }
}

__device__ __forceinline__ void x_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kXThreads) : "memory"); }

// D: pair distance (0 = unsplit).  SAVED: x comes as its saved halves [2][N][K] by TMA.
template <int D, typename IO, bool SAVED>
__global__ void __launch_bounds__(kThreadsSbw, 1)
split_bwd_weight_kernel(const __grid_constant__ CUtensorMap tmap_m, const __grid_constant__ CUtensorMap tmap_n, const SbwParams prm) {
    constexpr int S = D == 0 ? 1 : 2;
    constexpr bool F32 = sizeof(IO) == 4;
    static_assert(!F32 || (S == 2 && !SAVED), "float layers are split, their halves not saved");
    constexpr int kTok = sbw_tokens(S, sizeof(IO));
    constexpr int kBlock = kTok * 128;                           // an operand block: kTok tokens x 64 columns; a raw slab
    extern __shared__ uint8_t smem_raw_base[];
    uint8_t* smem = ptx::align_smem_1024(smem_raw_base);
    const int stages = prm.stages, stage_bytes = prm.stage_bytes, nb = prm.nb, nbh = nb / 2;
    SbwBarriers* bar = reinterpret_cast<SbwBarriers*>(smem + stages * stage_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &bar->abort_flag;
    int* status = prm.status;
    const uint32_t rank = ptx::cluster_ctarank();

    // Copies that end on barriers of this CTA (all but the saved halves): their warps set the barriers up and go ahead, without waiting
    // for the CTA and the pair.  (Order 6, 92 -> 60 channels, 10007 tokens, step 43.6 -> 43.2 us; dihedral group of order 8, 48 -> 96, 12608 tokens
    // 49.6 -> 48.9.  The same for the rows of x in the linear kernel gained nothing: its weights, which end on the leader's barriers, come later.)
    // They do not let the next kernel start: it could take the tensor memory that this CTA has still to allocate, and then wait for this
    // kernel.  The warps that the CTA's barrier holds back do, behind it.
    const bool early = warp == kWarpTmaM || warp == kWarpTmaN;
    if (warp == kWarpTmaM) {
        // split: only the leader's "full" is used, by both CTAs' warps and (saved halves) its TMA thread, which announces
        // the bytes of both CTAs.  unsplit: each CTA's own (its db warps wait for it too), and the peer's word to the leader.
        const uint32_t full_count = S == 2 ? kXWarps + (SAVED ? 1 : 0) : 2 + (rank == 0 ? 1 : 0);
        // unsplit: the warps that sum db read some of the stages too; the M side's copy thread answers for them at the others
        // float: the transform warps that leave a stage to the other group say that they have seen it
        const uint32_t empty_count = 1 + (S == 1 ? kXWarps : F32 ? kXWarps / 2 : 0);
        // (a lane for each barrier: the instructions of a chain of them have to be fetched first)
        static_assert(offsetof(SbwBarriers, tmem_base) == 8 * (3 * kMaxStages + 5) && kMaxStages == 8, "a lane for each barrier");
        if (lane < 3 * kMaxStages + 5)
            ptx::mbar_init(&bar->full[0] + lane, lane < 8 ? full_count : lane < 16 ? empty_count : lane < 24 ? (SAVED ? 1 : 2) : lane == 26 || lane == 27 ? 2 * kXWarps : 1);
        if (lane == 0) {
            bar->abort_flag = 0;
            ptx::prefetch_tensormap(&tmap_m);
            ptx::prefetch_tensormap(&tmap_n);
        }
        ptx::fence_mbar_init();
    }
    if (warp == kWarpMma) { ptx::tmem_alloc_pair(&bar->tmem_base, 512); ptx::tmem_relinquish_pair(); }
    __syncwarp();
    if (early) ptx::bar_sync(3, 64);
    ptx::tc_fence_before_sync();
    if (early) ptx::bar_arrive(2, kThreadsSbw);
    else ptx::bar_sync(2, kThreadsSbw);
    ptx::cluster_arrive();
    if (!early) ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bar->tmem_base;
    // (the roles wait for the kernel before themselves, see ptx::grid_dependency_wait)

    const int pair = blockIdx.x >> 1;
    const int nt = prm.nt0 + pair % prm.nTiles, mt = prm.mt0 + (pair / prm.nTiles) % prm.mTiles, split = pair / (prm.nTiles * prm.mTiles);
    const int64_t stage0 = (int64_t)split * prm.stages_per_split;
    int64_t nst = prm.total_stages - stage0;
    if (nst > prm.stages_per_split) nst = prm.stages_per_split;
    const int m_bytes = F32 ? 128 * 128 : 2 * S * kBlock;                          // M operand of a stage; the N operand follows it
    const int m0 = (2 * mt + (int)rank) * prm.wM, n0 = (2 * nt + (int)rank) * prm.wN;   // first columns of this CTA's operands
    const bool m_is_y = prm.m_is_y != 0;
    const int my_share = m_is_y ? nt : mt;
    const uint32_t leader_full = ptx::map_to_cta(ptx::smem_u32(&bar->full[0]), 0u);

    // The pair's last meeting: no CTA may leave, or free its tensor memory, while the other can still signal it or read its own.  Unsplit:
    // the warps behind the ring arrive once they have read the accumulators, as behind the stores of dw they would wait for those, ~1000
    // cycles.  (Split layers read the second half behind the stores of the first: arriving there costs what it saves.)
    bool met = false;

    // Registers (unsplit: the totals): 20 warps launch with 96 each = 1920 per lane; 4 warps at 56 and 16 at 104 make 1888.
    if (warp < kWarpX0) {
    if constexpr (S == 1) ptx::reg_dealloc<kRoleRegs>();
    if (warp == kWarpTmaM || warp == kWarpTmaN) {
        // ---------------------------------------------------------------- one thread for either side
        const bool side_m = warp == kWarpTmaM;
        const bool side_y = side_m == m_is_y;
        const CUtensorMap* map = side_m ? &tmap_m : &tmap_n;
        const int c0 = side_m ? m0 : n0, blocks = side_m ? 2 : nbh / 64;      // first column, 64-column operand blocks
        const int off = side_m ? 0 : m_bytes;
        const bool saved_side = SAVED && !side_y;
        if (saved_side) ptx::cluster_wait();
        if (lane == 0) {
            const bool direct = S == 1 || saved_side;    // operand tiles, no arithmetic
            uint64_t* const fullb = direct ? bar->full : bar->raw_full;
            const uint32_t bytes = (uint32_t)(blocks * S * kBlock);            // raw rows are as many bytes as their halves
            const int slabs = side_m ? prm.m_slabs : prm.n_slabs;
            int st = 0, share_at = 0;
            uint32_t ph = 1, issued = 0;
            if constexpr (F32) {
                // first pass: a stage's raw rows into the first of two slots, which the transform fills; second pass: one slot
                const uint32_t raw = (uint32_t)(side_m ? 128 * 128 : nbh * 128);
                for (int64_t q = 0; q < 3 * nst; ++q, ++issued) {
                    if (!ptx::mbar_wait(&bar->empty[st], ph, abort_flag, status, side_m ? 501 : 506, true, 64)) break;
                    if (q == 0) ptx::grid_dependency_wait();
                    if (q < 2 * nst && (q & 1)) {
                        ptx::mbar_arrive(&bar->raw_full[st]);
                    } else {
                        const int row = (int)((stage0 + (q < 2 * nst ? q >> 1 : q - 2 * nst)) * kTok);
                        uint8_t* dst = smem + st * stage_bytes + off;
                        ptx::mbar_arrive_expect_tx(&bar->raw_full[st], raw);
                        if (slabs) ptx::tma_load_3d(dst, map, 0, row, c0 / 16, &bar->raw_full[st]);
                        else
                            for (int b = 0; b < (int)raw / kBlock; ++b) ptx::tma_load_2d(dst + b * kBlock, map, c0 * 2 + b * 32, row, &bar->raw_full[st]);
                    }
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
            } else {
                // ODD: raw rows that are not whole slabs.  Their up to eight copies per stage, one after the other, bound such layers, and the
                // test in the loop slows them: order 16, 8 -> 119 channels, 99903 tokens 104 us with it, 98 without; 110 -> 198, 1118 tokens 25.4,
                // 24.4.  (The others are the faster for it, see ptx::grid_dependency_wait: order 4, 128 -> 128 channels, 25000 tokens 22.2, 21.8.)
                auto copies = [&](auto odd) {
                    constexpr bool ODD = decltype(odd)::value;
                    if (ODD) ptx::grid_dependency_wait();
                    for (int64_t q = 0; q < nst; ++q, ++issued) {
                        if (!ptx::mbar_wait(&bar->empty[st], ph, abort_flag, status, side_m ? 501 : 506, true, 64)) break;
                        if (!ODD && q == 0) ptx::grid_dependency_wait();
                        const int row = (int)((stage0 + q) * kTok);
                        uint8_t* dst = smem + st * stage_bytes + off;
                        if (ODD) {
                            ptx::mbar_arrive_expect_tx(&fullb[st], bytes);
                            for (int b = 0; b < 2 * blocks; ++b) ptx::tma_load_2d(dst + b * kBlock, map, c0 * 2 + b * 64, row, &fullb[st]);
                        } else if (!direct) {
                            ptx::mbar_arrive_expect_tx(&fullb[st], bytes);
                            ptx::tma_load_3d(dst, map, 0, row, c0 / 32, &fullb[st]);
                        } else if constexpr (S == 2) {           // saved halves: counted on the leader's barrier, for both CTAs
                            if (rank == 0) ptx::mbar_arrive_expect_tx(&fullb[st], 2 * bytes);
                            ptx::tma_load_4d_pair(dst, map, 0, row, 0, c0 / 64, leader_full + st * 8u);
                        } else {
                            ptx::mbar_arrive_expect_tx(&fullb[st], bytes);
                            for (int b = 0; b < blocks; ++b)
                                ptx::tma_load_2d(dst + b * kBlock, map, c0 + b * 64, row, &fullb[st]);
                            if (side_m && share_at != my_share) ptx::mbar_arrive(&bar->empty[st], (uint32_t)kXWarps);
                            if (++share_at == prm.shares) share_at = 0;
                        }
                        if (++st == stages) { st = 0; ph ^= 1u; }
                    }
                };
                if constexpr (S == 2) {
                    if (!direct && !slabs) copies(std::true_type{});
                    else copies(std::false_type{});
                } else {
                    copies(std::false_type{});
                }
            }
            // the copies issued last must have landed before the CTA may exit: their stages have been released
            for (uint32_t c = issued > (uint32_t)stages ? issued - stages : 0; c < issued; ++c)
                ptx::mbar_wait(&bar->empty[c % stages], (c / stages) & 1, abort_flag, status, 511, false);
        }
        __syncwarp();
        if (!saved_side) ptx::cluster_wait();                    // (of the first meeting)
    } else if (warp == kWarpMma) {
        ptx::grid_handover();
        if (rank == 0) {
            int st = 0;
            uint32_t ph = 0;
            bool ok = true;
            const uint32_t idesc = F32 ? ptx::umma_idesc_tf32_f32(256, nb) : ptx::umma_idesc_f16_f32_mn_major(256, nb, H16<IO>::kUmmaFormat);
            const uint64_t a_ring = F32 ? desc_k_sw128(ptx::smem_u32(smem)) : desc_mn_sw128(ptx::smem_u32(smem), S * kBlock);
            const uint64_t b_ring = F32 ? desc_k_sw128(ptx::smem_u32(smem + m_bytes)) : desc_mn_sw128(ptx::smem_u32(smem + m_bytes), S * kBlock);
            if constexpr (F32) {
                // first pass: rows of [+hi 8 tokens | -hi 8 | +lo 8 | -lo 8], the two small products of either half; second pass:
                // rows of [+hi 16 tokens | -hi 16]
                for (int64_t q = 0; q < 3 * nst; ++q) {
                    ok = ptx::mbar_wait_warp(&bar->full[st], ph, abort_flag, status, 502, true, 256);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t a0 = a_ring + (uint64_t)((st * stage_bytes) >> 4), b0 = b_ring + (uint64_t)((st * stage_bytes) >> 4);
                    const bool first = q < 2 * nst;
                    // operands of the two MMAs of a half, in 16-byte units; the second half's come 2 (first pass) or 4 behind
                    const int half = first ? 2 : 4, a1 = first ? 4 : 2, b1 = first ? 0 : 2, b00 = first ? 4 : 0;
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            ptx::umma_tf32_pair(tmem_base + (uint32_t)(s * nb), a0 + s * half, b0 + s * half + b00, idesc, q > 0 ? 1u : 0u);
                            ptx::umma_tf32_pair(tmem_base + (uint32_t)(s * nb), a0 + s * half + a1, b0 + s * half + b1, idesc, 1u);
                        }
                        ptx::umma_commit_pair_both(&bar->empty[st]);
                        if (q + 1 == 3 * nst) ptx::umma_commit_pair_both(&bar->full_d[0]);
                    }
                    __syncwarp();
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
            } else
            for (int64_t q = 0; q < nst; ++q) {
                // (unsplit: two accumulators take kDrainStages stages in turn)
                const uint32_t acc = S == 1 ? (uint32_t)(q / kDrainStages) & 1u : 0u;
                const bool fresh = S == 1 ? q % kDrainStages == 0 : q == 0;
                if (S == 1 && fresh) ok = ptx::mbar_wait_warp(&bar->empty_d[acc], (uint32_t)(q / (2 * kDrainStages) & 1) ^ 1u, abort_flag, status, 507, true, 256);
                ok = ok && ptx::mbar_wait_warp(&bar->full[st], ph, abort_flag, status, 502, true, 256);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint64_t a0 = a_ring + (uint64_t)((st * stage_bytes) >> 4), b0 = b_ring + (uint64_t)((st * stage_bytes) >> 4);
                if (ptx::elect_one()) {
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int k = 0; k < kTok / 16; ++k)      // 16 tokens = two 8-row groups
                            ptx::umma_f16_pair(tmem_base + acc * 256u + (uint32_t)(s * nb), a0 + ((s * kBlock + k * 2048) >> 4),
                                               b0 + ((s * kBlock + k * 2048) >> 4), idesc, (!fresh || k > 0) ? 1u : 0u);
                    ptx::umma_commit_pair_both(&bar->empty[st]);
                    if (q + 1 == nst || (S == 1 && q % kDrainStages == kDrainStages - 1)) ptx::umma_commit_pair_both(&bar->full_d[acc]);
                }
                __syncwarp();
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
            if (ptx::elect_one()) ptx::umma_commit_pair(&bar->mma_done);
            __syncwarp();
            ptx::mbar_wait_warp(&bar->mma_done, 0, abort_flag, status, 513, false);
        } else if (S == 1 && lane == 0) {
            int st = 0;
            uint32_t ph = 0;
            for (int64_t q = 0; q < nst; ++q) {
                if (!ptx::mbar_wait(&bar->full[st], ph, abort_flag, status, 504, true, 256)) break;
                ptx::mbar_arrive_remote(leader_full + st * 8u);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
        }
    }
    } else {
        if constexpr (S == 1) ptx::reg_alloc<kXRegs>();
        ptx::grid_handover();
        const int xt = threadIdx.x - kWarpX0 * 32;               // 0 .. 511
        constexpr int NSUM = F32 ? 4 / D : D == 0 ? 2 : D >= 8 ? 1 : 8 / (D ? D : 1);       // sums per granule
        constexpr int NACC = !F32 && S == 2 ? 2 * NSUM : NSUM;   // (16-bit, split: two granules per thread)
        float acc[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0.f;
        const int quad = warp & 3, part4 = (warp - kWarpX0) >> 2;              // this warp's share of the accumulators: lanes, columns
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        // unsplit: this thread's entries of the accumulators, in either half nb / 8 columns of its lane
        float total[S == 1 ? 64 : 1];
        if constexpr (S == 1) {
#pragma unroll
            for (int i = 0; i < 64; ++i) total[i] = 0.f;
        }
        bool ok = true;
        int share_at = 0;                                        // stage number modulo shares
        int st = 0;
        uint32_t ph = 0;
        if constexpr (F32) {
            // Two groups of eight warps take alternate stages, a warp two raw slabs [16 tokens x 32 columns] of one side, a lane four
            // tokens x two chunks (four representatives and their partners): transposed in registers, four tokens of a
            // representative are one 16-byte chunk of its K-major row.  hi is cut off and lo rounded as in the linear kernel, but
            // hi of the N side is rounded, so that the product of the lo parts, which is left out, has no preferred sign.
            // The order of a lane's accesses is chosen so that the eight lanes of a wavefront never meet in a bank: tokens are
            // read in the order j ^ t4 -- a permutation of the four tokens of a chunk, the same on both sides --, the upper two
            // representatives first where g is odd, and the upper eight tokens write the difference before the sum.
            const int group = (warp - kWarpX0) >> 3, wx = (warp - kWarpX0) & 7;
            const bool side_n = wx >= 4;
            const int t4 = lane & 3, g = (lane >> 2) & 3, gl = g & 1, up = t4 >> 1;
            const int slab = 2 * (wx & 3) + (lane >> 4);
            // slabs behind the layer's last column: their rows reach only entries that nobody reads
            const int c0 = (side_n ? n0 : m0) + (wx & 3) * 32, cols = (side_n != m_is_y ? prm.Co : prm.Ci) * prm.reps;
            const bool mine = c0 < cols && (!side_n || wx - 4 < nbh / 32);
            const int base = (side_n ? m_bytes : 0) + slab * 2048;
            const float sgn = up ? -1.f : 1.f;
            const bool sums = (side_n != m_is_y) && my_share < prm.shares;
            share_at = 0;
            int64_t done = 0;
            for (int64_t q = 0; q < 3 * nst; ++done) {
                const bool first = q < 2 * nst;
                // (every warp waits for every slot, in order, and says which of the other group's it has seen: as in the linear kernel)
                ok = ptx::mbar_wait(&bar->raw_full[st], ph, abort_flag, status, 508, true, 4);
                if (!ok) break;
                const int cur = st;
                int next = st;
                if (++st == stages) { st = 0; ph ^= 1u; }
                if (first) {
                    next = st;
                    ok = ptx::mbar_wait(&bar->raw_full[next], ph, abort_flag, status, 509, true, 4);
                    if (!ok) break;
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
                q += first ? 2 : 1;
                const bool sum = sums && !first && share_at == my_share;
                if (!first && ++share_at == prm.shares) share_at = 0;
                if ((done & 1) != group) {
                    __syncwarp();
                    if (lane == 0) {
                        ptx::mbar_arrive(&bar->empty[cur]);
                        if (first) ptx::mbar_arrive(&bar->empty[next]);
                    }
                    continue;
                }
                if (mine) {
                    const uint8_t* src = smem + cur * stage_bytes + base;
                    uint4 a[4], b[4];                            // a: chunk 2g + gl, b: the other one
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int t = j ^ t4, row = 4 * t4 + t;
                        a[j] = lds128(src + row * 128 + (((2 * g + gl) ^ (row & 7)) << 4));
                        b[j] = lds128(src + row * 128 + (((2 * g + 1 - gl) ^ (row & 7)) << 4));
                    }
                    __syncwarp();                                // both slabs have been read before any lane writes into them
                    if (sum) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float sa = (__uint_as_float(a[j].x) + __uint_as_float(a[j].y)) + (__uint_as_float(a[j].z) + __uint_as_float(a[j].w));
                            const float sb = (__uint_as_float(b[j].x) + __uint_as_float(b[j].y)) + (__uint_as_float(b[j].z) + __uint_as_float(b[j].w));
                            if constexpr (NSUM == 1) acc[0] += sa + sb;
                            else { acc[0] += sa; acc[NSUM - 1] += sb; }
                        }
                    }
                    uint8_t* dst = smem + (first && up ? next : cur) * stage_bytes + base;
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        // D = 4: representative r and its partner are words r of the two chunks (in either order: with gl the
                        // difference comes out negated, see the epilogue).  D = 2: two representatives and partners per chunk.
                        const int row = D == 4 ? 4 * g + r : 4 * g + (r ^ (2 * gl));
                        uint8_t* line = dst + row * 128;
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            uint32_t hi[4], lo[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t wa[4] = {a[j].x, a[j].y, a[j].z, a[j].w}, wb[4] = {b[j].x, b[j].y, b[j].z, b[j].w};
                                const float e = __uint_as_float(D == 4 ? wa[r] : r < 2 ? wa[r & 1] : wb[r & 1]);
                                const float z = __uint_as_float(D == 4 ? wb[r] : r < 2 ? wa[2 + (r & 1)] : wb[2 + (r & 1)]);
                                const float v = fmaf(t ? -sgn : sgn, z, e);
                                hi[j] = side_n ? round_tf32(v) : __float_as_uint(v) & 0xFFFFE000u;
                                lo[j] = __float_as_uint(v - __uint_as_float(hi[j])) + 0x1000u;
                            }
                            const int hf = t ^ up;               // 0: sum, 1: difference
                            if (first) {
                                *reinterpret_cast<uint4*>(line + (((2 * hf + (t4 & 1)) ^ (row & 7)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                                *reinterpret_cast<uint4*>(line + (((4 + 2 * hf + (t4 & 1)) ^ (row & 7)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                            } else {
                                *reinterpret_cast<uint4*>(line + (((4 * hf + t4) ^ (row & 7)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                            }
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive_remote(leader_full + cur * 8u);
                    if (first) ptx::mbar_arrive_remote(leader_full + next * 8u);
                }
            }
        } else if constexpr (S == 2) {
            // Two groups of eight warps take alternate stages (an even number of slots, so that a group sees every phase of its
            // slots).  Work items are 8 tokens of a pair of raw slabs, 4 granules of either: a warp has one of the M side and (nb =
            // 128: every second warp) one of the N side.  Which two tokens share a shared-memory wavefront: the chunks read are
            // disjoint when they differ in parity (D = 16: in the second bit), the chunks written when they differ in the third bit.
            constexpr int kTokPair = D == 16 ? 6 : 5;
            const int group = (warp - kWarpX0) >> 3, wx = (warp - kWarpX0) & 7;
            const int g = lane & 3, t8 = (lane >> 3) ^ (((lane >> 2) & 1) ? kTokPair : 0);      // granule of the slab, token of eight
            const int ca = granule_chunk<D>(g), cb = ca + kPartnerChunk<D>;
            const bool do_m = !SAVED || m_is_y;
            const bool do_n = (!SAVED || !m_is_y) && (nbh == 128 || wx < 4);
            const int item = (wx & 3) * 1024 + t8 * 128;         // 8 tokens
            const int m_off = item + (wx >> 2) * 2 * kBlock, n_off = m_bytes + item + (nbh == 128 ? (wx >> 2) * 2 * kBlock : 0);
            const int a_off = (ca ^ t8) << 4, b_off = (cb ^ t8) << 4, lo = (g ^ t8) << 4, hi = ((4 | g) ^ t8) << 4;
            struct Item { uint4 a0, b0, a1, b1; };               // t: this thread's row in the first slab
            auto load = [&](const uint8_t* t) {
                return Item{lds128(t + a_off), lds128(t + b_off), lds128(t + kBlock + a_off), lds128(t + kBlock + b_off)};
            };
            auto halves = [&](uint8_t* t, const Item& v) {
                uint4 p0, m0, p1, m1;
                split_granule<D, IO>(v.a0, v.b0, p0, m0);
                split_granule<D, IO>(v.a1, v.b1, p1, m1);
                *reinterpret_cast<uint4*>(t + lo) = p0;
                *reinterpret_cast<uint4*>(t + hi) = p1;
                *reinterpret_cast<uint4*>(t + kBlock + lo) = m0;
                *reinterpret_cast<uint4*>(t + kBlock + hi) = m1;
            };
            share_at = group % prm.shares;                       // (one share: only pairs of the first tile sum, see the launcher)
            st = group;
            for (uint32_t q = group; q < (uint32_t)nst; q += 2) {
                ok = ptx::mbar_wait(&bar->raw_full[st], ph, abort_flag, status, 508, true, 4);
                if (!ok) break;
                uint8_t* slot = smem + st * stage_bytes;
                const bool sum = share_at == my_share;           // this pair's share of the column sums of dy (tokens past N are zero)
                Item vm{}, vn{};
                if (do_m) vm = load(slot + m_off);
                if (do_n) vn = load(slot + n_off);
                __syncwarp();                                    // the rows have been read before any lane writes into them
                if (do_m) halves(slot + m_off, vm);
                if (do_n) halves(slot + n_off, vn);
                if (sum) {
                    const Item& y = m_is_y ? vm : vn;
                    add_granule<D, IO>(y.a0, y.b0, acc);
                    add_granule<D, IO>(y.a1, y.b1, acc + NSUM);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(leader_full + st * 8u);
                st += 2;
                if (st >= stages) { st -= stages; ph ^= 1u; }
                share_at += 2;
                while (share_at >= prm.shares) share_at -= prm.shares;
            }
        } else {
            // unsplit: the operands come by TMA; these warps only sum the columns of dy
            const int words = m_is_y ? 64 : nbh / 2;             // 32-bit words (column pairs) of this CTA's dy operand
            const int wd = xt % words, tg = xt / words, tgs = kXThreads / words;
            // (tgs is 8 or 16: the tokens of a thread are alike modulo 8, and with it the place of its chunk)
            const int off = (m_is_y ? 0 : m_bytes) + (wd >> 5) * kBlock + (wd & 3) * 4 + tg * 128 + ((((wd & 31) >> 2) ^ (tg & 7)) << 4);
            const bool sums = 2 * wd < prm.Co * prm.reps - (m_is_y ? m0 : n0);
            const uint32_t empty_leader = ptx::map_to_cta(ptx::smem_u32(&bar->empty_d[0]), 0u);
            // Lanes and columns of the accumulators that hold something of the layer (the others stay zero).
            const int mcols = (m_is_y ? prm.Co : prm.Ci) * prm.reps - m0, ncols = (m_is_y ? prm.Ci : prm.Co) * prm.reps - 2 * nt * prm.wN;
            const bool lanes = quad * 32 < (mcols < prm.wM ? mcols : prm.wM);
            const int valid0 = !lanes ? 0 : ncols < prm.wN ? ncols : prm.wN, valid1 = !lanes ? 0 : ncols - prm.wN < prm.wN ? ncols - prm.wN : prm.wN;
            // Adds an accumulator to the totals.  (The tensor core adds with truncation, 1.9e-8 of relative error per step of 16 tokens;
            // eight steps and a rounded addition are as good as the CUDA cores' sums of the same tokens.)
            auto drain = [&](uint32_t block) {
                const uint32_t b = block & 1u;
                ok = ptx::mbar_wait(&bar->full_d[b], (block >> 1) & 1u, abort_flag, status, 505, true, 256);
                if (!ok) return;
                ptx::tc_fence_after_sync();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int half = i >> 1, c = (i & 1) * 16;
                    if (c < nbh / 4 && part4 * (nbh / 4) + c < (half ? valid1 : valid0)) {
                        uint32_t v[16];
                        ptx::tmem_ld<16>(lane_base + b * 256u + (uint32_t)(half * nbh + part4 * (nbh / 4) + c), v);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) total[16 * i + j] += __uint_as_float(v[j]);
                    }
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(empty_leader + b * 8u);
            };
            uint32_t drained = 0;
            const uint32_t n = (uint32_t)nst;
            for (uint32_t q = 0; q < n && ok; ++q) {
                // (a stage is looked at only after the MMAs of those two before it: no old phase of its barrier can be taken for its own)
                if (share_at == my_share) {
                    ok = ptx::mbar_wait(&bar->full[st], ph, abort_flag, status, 503, true, 16);
                    if (!ok) break;
                    const uint8_t* src = smem + st * stage_bytes + off;
                    float2 sum = make_float2(0.f, 0.f);          // of the stage, then of all: short chains
                    if (sums) {
#pragma unroll
                        for (int i = 0; i < kTok / 8; ++i) {
                            if (i * tgs < kTok) {
                                const float2 f = H16<IO>::unpack(*reinterpret_cast<const uint32_t*>(src + i * tgs * 128));
                                sum.x += f.x; sum.y += f.y;
                            }
                        }
                    }
                    acc[0] += sum.x; acc[1] += sum.y;
                    ptx::fence_proxy_async_smem();               // these reads before the TMA refill the release allows
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&bar->empty[st]);
                }
                if (++share_at == prm.shares) share_at = 0;
                if (++st == stages) { st = 0; ph ^= 1u; }
                // the accumulator before, while the MMAs of the next one run
                if (q % kDrainStages == 0 && q > 0) drain(drained++);
            }
            for (; ok && drained * kDrainStages < n; ++drained) drain(drained);
        }
        if (S == 2 && ok && nst > 0) ok = ptx::mbar_wait(&bar->full_d[0], 0, abort_flag, status, 505, true, 16);
        // all warps go on or none: the barriers below are for all of them (whoever gave up has raised the abort flag)
        x_barrier();
        if (xt == 0) bar->go = *abort_flag == 0 ? 1 : 0;
        x_barrier();
        if (bar->go != 0) {
            ptx::tc_fence_after_sync();
            const int h = prm.reps;
            const int pitch = (S == 1 ? nb : nbh) + 1;
            float* buf = reinterpret_cast<float*>(smem);         // entries of a product: [S][128][pitch], one half of the columns (unsplit: all)
            if constexpr (S == 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if ((i & 1) * 16 < nbh / 4) {
                        float* b = buf + (quad * 32 + lane) * pitch + (i >> 1) * nbh + part4 * (nbh / 4) + (i & 1) * 16;
#pragma unroll
                        for (int j = 0; j < 16; ++j) b[j] = total[16 * i + j];
                    }
                }
                if (my_share >= prm.shares) x_barrier();         // (else the ones below do)
                __syncwarp();
                ptx::cluster_arrive();
                met = true;
            }
            // ---- db: a row of sums per warp (split; tokens of a warp added by shuffles) or per token group of the threads, added
            // per channel in a fixed order (unsplit: up to 16 groups and 16 columns per channel; the groups of a column first, a thread
            // each, for the chain of 256 additions is ~2 K cycles)
            if (my_share < prm.shares) {
                float* red = buf + (S == 1 ? 128 * pitch : 0);
                // columns of the dy operand come in groups of GC representatives per accumulator
                constexpr int GC = D == 0 ? 1 : D >= 8 ? 8 : (D ? D : 1);
                int groups, valid;
                if constexpr (F32) {
                    // a row per group of warps, already one value per lane and channel (D = 4) or two (D = 2)
                    const int w8 = (xt >> 5) & 7, grp = xt >> 8;
                    const int col = (w8 & 3) * 32 + (lane >> 4) * 16 + ((lane >> 2) & 3) * 4, gl = (lane >> 2) & 1;
#pragma unroll
                    for (int i = 0; i < NACC; ++i) {
                        float v = acc[i];
                        v += __shfl_xor_sync(0xffffffffu, v, 1);
                        v += __shfl_xor_sync(0xffffffffu, v, 2);
                        if ((lane & 3) == 0 && (w8 >= 4) != m_is_y && (w8 & 3) < (m_is_y ? 4 : nbh / 32)) red[grp * 129 + col + (i ^ (NACC == 2 ? gl : 0)) * 2] = v;
                    }
                    groups = 2; valid = m_is_y ? 128 : nbh;
                } else if constexpr (S == 2) {
                    // thread = (stage parity, pair of slabs, four groups of eight tokens, granule of either slab)
                    const int pairs = m_is_y || nbh == 128 ? 2 : 1, w8 = (xt >> 5) & 7;
                    const int col = (pairs == 2 ? w8 >> 2 : 0) * 64 + (lane & 3) * 8, grp = (xt >> 8) * 4 + (w8 & 3);
#pragma unroll
                    for (int i = 0; i < NACC; ++i) {
                        float v = acc[i];
                        v += __shfl_xor_sync(0xffffffffu, v, 4);
                        v += __shfl_xor_sync(0xffffffffu, v, 8);
                        v += __shfl_xor_sync(0xffffffffu, v, 16);
                        if (lane < 4 && (pairs == 2 || w8 < 4)) red[grp * 129 + col + (i / NSUM) * 32 + (i % NSUM) * GC] = v;
                    }
                    groups = 8; valid = pairs * 64;
                } else {
                    const int words = m_is_y ? 64 : nbh / 2, col = (xt % words) * 2, grp = xt / words;
                    red[grp * 129 + col] = acc[0];
                    red[grp * 129 + col + 1] = acc[1];
                    groups = kXThreads / words; valid = m_is_y ? prm.wM : prm.wN;
                }
                x_barrier();
                if constexpr (S == 1) {
                    if (xt < valid) {
                        float v = 0.f;
#pragma unroll
                        for (int g = 0; g < 16; ++g)
                            if (g < groups) v += red[g * 129 + xt];
                        red[16 * 129 + xt] = v;
                    }
                    red += 16 * 129;
                    groups = 1;
                    x_barrier();
                }
                const int channels = valid / h;
                const int c0 = (m_is_y ? m0 : n0) / h;
                for (int c = xt; c < channels; c += kXThreads) {
                    if (c0 + c >= prm.Co) break;
                    float v = 0.f;
                    for (int k = 0; k < h; k += GC)
#pragma unroll 8
                        for (int g = 0; g < groups; ++g) v += red[g * 129 + c * h + k];
                    prm.db_part[(size_t)(split * prm.shares + my_share) * prm.Co + c0 + c] = v;
                }
                if constexpr (S == 2) x_barrier();               // (unsplit: dw's entries lie elsewhere)
            }
            // ---- dw: nb/2 columns of the accumulators at a time through shared memory; a thread adds the REPS products
            // D[h, h q] of its (output channel, input channel, q)
            float* out = prm.part + split * prm.part_stride;
            for (int half = 0; half < 2; ++half) {
                const int ncol = (2 * nt + half) * prm.wN;       // first column of this half on the N side
                if (m0 >= (m_is_y ? prm.Co : prm.Ci) * h || ncol >= (m_is_y ? prm.Ci : prm.Co) * h) continue;   // nothing of the layer
                const int mv = (m_is_y ? prm.Co : prm.Ci) * h - m0 - quad * 32, nv = (m_is_y ? prm.Ci : prm.Co) * h - ncol;     // entries there
                if constexpr (S == 2) {
                for (int c = part4 * (nbh / 4); c < (part4 + 1) * (nbh / 4) && c < nv && mv > 0; c += 16) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        uint32_t v[16];
                        ptx::tmem_ld<16>(lane_base + (uint32_t)(s * nb + half * nbh + c), v);
                        ptx::tmem_ld_wait();
                        float* b = buf + (s * 128 + quad * 32 + lane) * pitch + c;
#pragma unroll
                        for (int j = 0; j < 16; ++j) b[j] = __uint_as_float(v[j]);
                    }
                }
                x_barrier();
                }
                // (a copy the compiler cannot see through: it would work out every group's places before the main loop, and spill)
                int xo;
                asm volatile("mov.u32 %0, %1;" : "=r"(xo) : "r"(xt));
                with_reps_of<D>(prm.reps, prm.dihedral != 0, [&](auto rt) {
                    using R = decltype(rt);
                    constexpr int REPS = R::kTuple / S;
                    const int tM = (S == 2 ? 128 : prm.wM) / REPS, tN = (S == 2 ? nbh : prm.wN) / REPS;   // channels of the tile
                    const int mch = m0 / REPS, nch = ncol / REPS;                   // first channels
                    // input channels fastest: neighbouring threads write neighbouring tuples
                    const int tI = m_is_y ? tN : tM, tO = m_is_y ? tM : tN;
                    const int ibase = m_is_y ? nch : mch, obase = m_is_y ? mch : nch;
                    // D[(i, h), (o, g)] with x on M, D[(o, g), (i, h)] with dy on M
                    const int step_i = m_is_y ? REPS : REPS * pitch, step_o = m_is_y ? REPS * pitch : REPS;
                    auto place = [&](int q, int k, bool& z) {    // of product D[k, k q] in its channel pair's block
                        const int g = R::template combine<true>(k, q, z);
                        return m_is_y ? g * pitch + k : k * pitch + g;
                    };
                    // entries q and zq of this thread's tuples
                    auto places = [&](int q, int& p, int& pz) {
                        p = R::element(q), pz = p + R::kHalf;
                        if (prm.corr) { p = (R::kTuple - p) % R::kTuple; pz = (R::kTuple - pz) % R::kTuple; }
                    };
                    if constexpr (S == 2) {
                        // everything a power of two: a thread keeps its q, and with it the places and signs, and its ti for all its pairs
                        constexpr int GROUPS = kXThreads / REPS;
                        const int q = xt % REPS, shift = 31 - __clz(tI);
                        const int ti = xt / REPS & (tI - 1), to0 = xt / REPS >> shift, dto = GROUPS >> shift;
                        const int toEnd = ibase + ti >= prm.Ci ? 0 : prm.Co - obase < tO ? prm.Co - obase : tO;
                        int at[REPS], p, pz;
                        float sg[REPS];
#pragma unroll
                        for (int k = 0; k < REPS; ++k) {
                            bool z;
                            at[k] = place(q, k, z);
                            sg[k] = z ? -1.f : 1.f;
                        }
                        places(q, p, pz);
                        const float* b = buf + ti * step_i + to0 * step_o;
                        float* dst = out + ((size_t)(obase + to0 - prm.o0) * prm.iCount + (ibase + ti - prm.i0)) * R::kTuple;
#pragma unroll 2
                        for (int to = to0; to < toEnd; to += dto) {
                            const float* bm = b + 128 * pitch;
                            float cp = 0.f, cm = 0.f;
#pragma unroll
                            for (int k = 0; k < REPS; ++k) { cp += b[at[k]]; cm = fmaf(sg[k], bm[at[k]], cm); }
                            // (float, D = 4: the differences of every second channel are negated on either side)
                            if (F32 && D == 4 && ((ti ^ to) & 1)) cm = -cm;
                            dst[p] = 0.5f * (cp + cm);
                            dst[pz] = 0.5f * (cp - cm);
                            b += dto * step_o;
                            dst += (size_t)dto * prm.iCount * R::kTuple;
                        }
                    } else {
                        constexpr int GROUPS = kXThreads / REPS;             // (a thread keeps its q here too; a few may idle)
                        const int q = xo % REPS;
                        int at[REPS], p, pz;
#pragma unroll
                        for (int k = 0; k < REPS; ++k) { bool z; at[k] = place(q, k, z); }
                        places(q, p, pz);
                        const int dti = GROUPS % tI, dto = GROUPS / tI;      // (no division per pair: ~40 instructions beside REPS additions)
                        int ti = xo / REPS % tI, to = xo / REPS / tI;
                        const int toEnd = xo >= GROUPS * REPS ? 0 : prm.Co - obase < tO ? prm.Co - obase : tO;
#pragma unroll 2
                        while (to < toEnd) {
                            if (ibase + ti < prm.Ci) {
                                const float* b = buf + half * nbh + ti * step_i + to * step_o;
                                float cp = 0.f;
#pragma unroll
                                for (int k = 0; k < REPS; ++k) cp += b[at[k]];
                                out[((size_t)(obase + to - prm.o0) * prm.iCount + (ibase + ti - prm.i0)) * R::kTuple + p] = cp;
                            }
                            ti += dti;
                            to += dto;
                            if (ti >= tI) { ti -= tI; ++to; }
                        }
                    }
                });
                if (S == 2) x_barrier();
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncwarp();                               // (roles of one lane: the arrival is a whole warp's)
    if (!met) ptx::cluster_arrive();
    __syncthreads();
    ptx::cluster_wait();
    if (warp == kWarpMma) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512);
    }
}

// dw = sum over token ranges of part[range][e], rows of row4 float4 elements that are pitch4 apart in dw; db likewise over ranges and
// shares.  A block takes COLS float4 elements (and channels of db): CHAINS groups of threads add a share of the ranges each, in order, and
// the first adds the sums -- a fixed order, and a fraction of the latency chain (one chain: 7 us of a 30 us gradient at 74 ranges).
// Two forms, which form where: finalize_narrow() below.
template <int COLS, int CHAINS>
__global__ void __launch_bounds__(COLS * CHAINS)
split_finalize_kernel(const float* __restrict__ part, const float* __restrict__ db_part, int splits, int db_parts, int64_t nw4,
                      int row4, int pitch4, int Co, float* __restrict__ dw, float* __restrict__ db) {
    __shared__ float4 sum[CHAINS][COLS];
    __shared__ float dsum[CHAINS][COLS];
    const int chain = threadIdx.x / COLS, col = threadIdx.x % COLS;
    const int64_t e = (int64_t)blockIdx.x * COLS + col;
    const bool has_w = e < nw4, has_b = db != nullptr && e < Co;
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    float d = 0.f;
    if (has_w) {
        const float4* p = reinterpret_cast<const float4*>(part) + e;
        const int per = (splits + CHAINS - 1) / CHAINS, s0 = chain * per, s1 = s0 + per < splits ? s0 + per : splits;
#pragma unroll 8
        for (int s = s0; s < s1; ++s) {
            const float4 b = __ldcs(p + (int64_t)s * nw4);
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
        }
    }
    if (has_b) {
        const int per = (db_parts + CHAINS - 1) / CHAINS, s0 = chain * per, s1 = s0 + per < db_parts ? s0 + per : db_parts;
#pragma unroll 8
        for (int s = s0; s < s1; ++s) d += db_part[(int64_t)s * Co + e];
    }
    sum[chain][col] = a;
    dsum[chain][col] = d;
    __syncthreads();
    if (chain == 0) {
#pragma unroll
        for (int g = 1; g < CHAINS; ++g) {
            const float4 b = sum[g][col];
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            d += dsum[g][col];
        }
        if (has_w) reinterpret_cast<float4*>(dw)[row4 == pitch4 ? e : e / row4 * pitch4 + e % row4] = a;
        if (has_b) db[e] = d;
    }
}

constexpr size_t kSmemMax = 227 * 1024;
constexpr size_t kFixedSmem = 1024 + sizeof(SbwBarriers) + 64;
// A ring slot: the operand tiles, or raw rows, of either side; as many of them as there is room for, an even number for split layers
// (see the kernel's transform warps).  Nothing is asked for beyond the ring: order 4, 64 -> 64 channels, 32768 tokens 18.8 -> 18.2 us against
// all there is, float, order 8, 48 -> 48, 12608 tokens 33.4 -> 33.2, others the same.  (No other block fits beside one of these: their
// registers leave room for three warps.)
constexpr int sbw_stage_bytes(int S, int elem, int nb) {
    return elem == 4 ? (128 + nb / 2) * 128 : (2 + nb / 128) * S * sbw_tokens(S, elem) * 128;
}
constexpr int sbw_stages(int S, int elem, int nb) {
    const int fit = (int)(kSmemMax - kFixedSmem) / sbw_stage_bytes(S, elem, nb), stages = fit < kMaxStages ? fit : kMaxStages;
    return S == 2 ? stages & ~1 : stages;
}
// Behind the loop the ring holds a product's entries and the sums of db; the barriers lie at its end and are still in use.
constexpr bool sbw_sums_fit(int S, int elem, int nb) {
    return (128 * ((S == 1 ? nb : nb / 2) + 1) * S + 17 * 129) * (int)sizeof(float) <= sbw_stages(S, elem, nb) * sbw_stage_bytes(S, elem, nb);
}
static_assert(sbw_sums_fit(1, 2, 128) && sbw_sums_fit(1, 2, 256) && sbw_sums_fit(2, 2, 128) && sbw_sums_fit(2, 2, 256) &&
              sbw_sums_fit(2, 4, 128) && sbw_sums_fit(2, 4, 256), "the sums behind the loop would overwrite barriers");
// Float: the error of a partial sum grows with the accumulations onto the large products (measured: 2.7e-8 of the largest |dw| per
// stage of 16 tokens; the other kernel, which mixes small and large ones, is at the same error after 192 tokens).
constexpr int64_t kMaxStagesPerSplitF32 = 80;
constexpr size_t kMaxScratchF32 = (size_t)192 << 20;             // beyond, the other kernel, which runs in blocks of tokens
// What one tile's partial sums may take, so that every layer can run in blocks of tiles through the array of
// eqlinear_bwd_weight_static: bounds the token ranges.
constexpr int64_t kMaxTileScratch = EQL_STATIC_SCRATCH_BYTES;
constexpr int64_t kMaxTokensPerSplit = 32768;  // (split) 2048 accumulation steps of 16 tokens: the tensor core adds with truncation

// Finalize kernel: 8 x 16, or 32 x 8, whose reads are 512 bytes wide.  A thread of either loads eight ranges at a time and what is left one
// after the other, so up to 56 ranges the narrow form, with half the loads per thread and four times the blocks, has the shorter chain.  It
// pays while the wide one leaves the SMs with at most two blocks (9472 elements are 2 x 148 blocks of 32), from 17 ranges on, where its own
// threads have two loads and more, with at most one.  Weight gradient, us, narrow / wide, float4 elements x ranges: 8280 x 12 17.4 / 18.2, 7744 x
// 10 8.8 / 9.0, 2304 x 32 8.8 / 9.3, 4096 x 29 9.9 / 10.9, x 50 12.9 / 13.8, 720 x 47 8.9 / 10.2; 7680 x 24 10.8 / 10.3, 8192 x 21 14.6 / 14.1; 720
// x 57 9.4 / 8.7, 2304 x 71 12.4 / 11.5.  With few ranges the same or less (8192 x 8 11.6 / 11.3, in a step 47.1 / 47.3 at 9216 x 8; 7776 x 6 10.0 /
// 9.8); with more elements the small reads cost more (16384 x 9 14.7 / 13.9, 24576 x 4 18.7 / 17.0, 65536 x 9 23.0 / 17.6, 262144 x 4 61 / 36).
// The layer's elements, not a launch's: calls in blocks of tiles add in the same order.
bool finalize_narrow(int splits, int64_t elements) { return splits >= 8 && splits <= 56 && elements <= (splits <= 16 ? 9472 : 4736); }

int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }

// The form the weight gradient of a layer takes: that of its linear passes, but order 2 unsplit (see split_common.cuh).
SplitShape weight_gradient_form(SplitShape s) {
    if (s.D == 1) { s.S = 1; s.D = 0; s.half = s.T; s.reps = s.tuple; }
    return s;
}

template <typename F>
cudaError_t dispatch_split(int D, eql_dtype_t dtype, F&& f) {
    if (dtype == EQL_FP32) {
        if (D == 2) return f(std::integral_constant<int, 2>{}, float{});
        if (D == 4) return f(std::integral_constant<int, 4>{}, float{});
        return cudaErrorInvalidValue;
    }
    auto with = [&](auto io) -> cudaError_t {
        switch (D) {
            case 0: return f(std::integral_constant<int, 0>{}, io);
            case 2: return f(std::integral_constant<int, 2>{}, io);
            case 4: return f(std::integral_constant<int, 4>{}, io);
            case 8: return f(std::integral_constant<int, 8>{}, io);
            case 16: return f(std::integral_constant<int, 16>{}, io);
            default: return cudaErrorInvalidValue;
        }
    };
    return dtype == EQL_BF16 ? with(__nv_bfloat16{}) : with(__half{});
}

}  // namespace

// Tiles and token ranges.  Time of a launch in cycles: rounds of pairs x (stages of a range x max(tensor core, operand
// bytes) per product + the epilogue), plus the finalize kernel's traffic of one partial dw per range.
SplitBwdWeightShape split_bwd_weight_shape(const SplitShape& layer, int64_t N, int num_sms) {
    const SplitShape sp = weight_gradient_form(layer);
    SplitBwdWeightShape b{};
    const int lcm = sp.reps / gcd(sp.reps, 8) * 8;               // whole channels, and columns that start on 16 bytes
    const int pairs = num_sms / 2;
    const bool f32 = sp.dtype == EQL_FP32;
    const int tok = sbw_tokens(sp.S, f32 ? 4 : 2);
    b.total_stages = (N + tok - 1) / tok;
    double best = 1e30;
    const int cols_x = sp.Ci * sp.reps, cols_y = sp.Co * sp.reps;
    for (int y_on_m = 0; y_on_m < 2; ++y_on_m) {
        for (int nb = 128; nb <= 256; nb += 128) {
            const int wM = 128 / lcm * lcm, wN = nb / 2 / lcm * lcm;
            if (wN == 0) continue;
            const int mc = y_on_m ? cols_y : cols_x, nc = y_on_m ? cols_x : cols_y;
            const int mT = (mc + 2 * wM - 1) / (2 * wM), nT = (nc + 2 * wN - 1) / (2 * wN);
            const int64_t tiles = (int64_t)mT * nT;
            const double stage_c = f32 ? (nb == 256 ? 1800 : 1300) : sp.S == 2 ? (nb == 256 ? 1100 : 800) : (nb == 256 ? 800 : 600);
            const int64_t s_min = f32 ? (b.total_stages + kMaxStagesPerSplitF32 - 1) / kMaxStagesPerSplitF32
                                : sp.S == 1 ? 1 : (b.total_stages * tok + kMaxTokensPerSplit - 1) / kMaxTokensPerSplit;
            // a range's share of the smallest scratch: one tile's partial sums (with room for db's)
            const int64_t tile_o = (int64_t)(y_on_m ? wM : wN) * 2 / sp.reps, tile_i = (int64_t)(y_on_m ? wN : wM) * 2 / sp.reps;
            const int64_t tile_bytes = 4 * ((tile_o < sp.Co ? tile_o : sp.Co) * (tile_i < sp.Ci ? tile_i : sp.Ci) * sp.tuple + (int64_t)(y_on_m ? nT : mT) * sp.Co);
            const int64_t s_fit = kMaxTileScratch / (tile_bytes + 1);
            if (s_fit < 1 || (f32 && s_min > s_fit)) continue;
            auto consider = [&](int64_t s) {
                if (s > b.total_stages) s = b.total_stages;
                if (s < s_min) s = s_min;
                if (s > s_fit) s = s_fit;
                const int64_t per = (b.total_stages + s - 1) / s, used = (b.total_stages + per - 1) / per;
                const double rounds = (double)((tiles * used + pairs - 1) / pairs);
                const double bytes = used > 1 ? 2.0 * (double)used * sp.Co * sp.Ci * sp.tuple * 4 : 0.0;
                const double total = rounds * (per * stage_c + (f32 ? 12000.0 : 3000.0) + 12.0 * sp.S * nb) + bytes / 2000.0 + (used > 1 ? 5000.0 : 0.0);
                if (total < best * 0.999) {
                    best = total;
                    b.y_on_m = y_on_m != 0; b.nb = nb; b.wM = wM; b.wN = wN; b.mTiles = mT; b.nTiles = nT;
                    b.splits = (int)used; b.stages_per_split = per; b.min_scratch_bytes = used > 1 ? align_up(used * tile_bytes, kWsAlign) : 0;
                }
            };
            // as many ranges as fill one to four rounds of pairs, and halves of those (less to write and add up)
            for (int r = 1; r <= 4; ++r)
                for (int64_t s = r * pairs / tiles; s >= 1; s /= 2) consider(s);
            consider(1);
            for (int64_t r = 1; r <= 8 && f32; ++r) consider((s_min * tiles + pairs * r - 1) / (pairs * r) * pairs * r / tiles);     // whole rounds
        }
    }
    // One token range: dw and db leave the kernel directly; the pairs of the first tile sum db alone.
    b.shares = b.splits == 1 ? 1 : b.y_on_m ? b.nTiles : b.mTiles;
    const size_t nw = (size_t)sp.Co * sp.Ci * sp.tuple;
    b.scratch_bytes = align_up(((b.splits > 1 ? (size_t)b.splits * nw : 0) + (size_t)b.splits * b.shares * sp.Co) * sizeof(float), kWsAlign);
    if (b.min_scratch_bytes == 0 || b.min_scratch_bytes > b.scratch_bytes) b.min_scratch_bytes = b.scratch_bytes;
    // (float products of fewer entries: a tile of 256 x 128 is mostly padding; T = 4, 24 -> 24 channels, 100000 tokens: 115 against
    // 167 us, 64 -> 64 channels, 60000 tokens: 128 against 103)
    b.supported = b.splits > 0 && (!f32 || (b.scratch_bytes <= kMaxScratchF32 && (int64_t)cols_x * cols_y >= 8192));
    b.stash_bytes = align_up((size_t)2 * (N > 0 ? N : 1) * sp.stash_pitch * 2 + 128, kWsAlign);    // (the last row's last slab reads past it)
    return b;
}

cudaError_t launch_split_bwd_weight(const SplitShape& layer, const SplitBwdWeightShape& b, bool correlation, const void* x, bool x_saved,
                                    const void* dy, float* dw, float* db, int64_t N, float* scratch, size_t scratch_bytes, int* status,
                                    cudaStream_t stream) {
    const SplitShape sp = weight_gradient_form(layer);
    if (x_saved && (sp.S != 2 || sp.dtype == EQL_FP32)) return cudaErrorInvalidValue;
    SbwParams p{};
    // Tiles per launch.  All of them where the scratch holds every tile's partial sums; else as many rows of tiles along the output
    // channels as it holds, or as many tiles of one row.  The entries of dw are added in the same order either way.
    const int oTiles = b.y_on_m ? b.mTiles : b.nTiles, iTiles = b.y_on_m ? b.nTiles : b.mTiles;
    const int tile_o = (b.y_on_m ? b.wM : b.wN) * 2 / sp.reps, tile_i = (b.y_on_m ? b.wN : b.wM) * 2 / sp.reps;      // channels
    auto covered = [](int tile, int first, int count, int C) { const int e = (first + count) * tile; return (e < C ? e : C) - first * tile; };
    int oStep = oTiles, iStep = iTiles;
    const size_t db_bytes = (size_t)b.splits * b.shares * sp.Co * sizeof(float);
    auto part_bytes = [&] { return (size_t)b.splits * covered(tile_o, 0, oStep, sp.Co) * covered(tile_i, 0, iStep, sp.Ci) * sp.tuple * sizeof(float); };
    if (b.splits > 1) {
        while (oStep > 1 && part_bytes() + db_bytes > scratch_bytes) --oStep;
        while (iStep > 1 && part_bytes() + db_bytes > scratch_bytes) --iStep;
        if (part_bytes() + db_bytes > scratch_bytes) return cudaErrorInvalidValue;
    }
    p.db_part = b.splits > 1 ? scratch + part_bytes() / sizeof(float) : db != nullptr ? db : scratch;
    p.status = status; p.N = N; p.total_stages = b.total_stages; p.stages_per_split = b.stages_per_split;
    p.wM = b.wM; p.wN = b.wN; p.nb = b.nb;
    p.m_is_y = b.y_on_m ? 1 : 0; p.shares = b.shares;
    p.Ci = sp.Ci; p.Co = sp.Co; p.tuple = sp.tuple; p.corr = correlation ? 1 : 0;
    p.reps = sp.reps; p.dihedral = sp.dihedral ? 1 : 0;
    const bool f32 = sp.dtype == EQL_FP32;
    const int elem = f32 ? 4 : 2, line = 128 / elem;             // line: elements of 128 bytes
    const int tok = sbw_tokens(sp.S, elem);
    p.stage_bytes = sbw_stage_bytes(sp.S, elem, b.nb);
    p.stages = sbw_stages(sp.S, elem, b.nb);
    // raw rows in whole slabs of 128 bytes come as one copy per stage and side, others slab by slab
    const int64_t xcols = (int64_t)sp.Ci * sp.tuple, ycols = (int64_t)sp.Co * sp.tuple;
    const int xblocks = b.y_on_m ? b.nb / 128 : 2, yblocks = b.y_on_m ? 2 : b.nb / 128;       // 64-column operand blocks of a CTA
    CUtensorMap mx, my;
    bool ok;
    int xslabs = 0, yslabs = 0;
    auto raw_map = [&](CUtensorMap* m, const void* base, int64_t cols, int blocks, int* slabs) {
        *slabs = cols % line == 0 && b.wM % 32 == 0 && b.wN % 32 == 0 ? 1 : 0;   // (a tile's first column must start a slab)
        return *slabs ? encode_map_slabs(m, base, cols / line, N, cols, blocks * (f32 ? 4 : 2), tok, elem) : encode_map_2d(m, base, cols, N, cols, line, tok, elem);
    };
    if (sp.S == 1) {
        ok = encode_map_2d(&mx, x, xcols, N, xcols, 64, tok, 2) && encode_map_2d(&my, dy, ycols, N, ycols, 64, tok, 2);
    } else {
        ok = raw_map(&my, dy, ycols, yblocks, &yslabs);
        if (x_saved) ok = ok && encode_map_plane_slabs(&mx, x, (sp.Ci * sp.reps + 63) / 64, N, sp.stash_pitch, N * (int64_t)sp.stash_pitch, xblocks, tok, 2);
        else ok = ok && raw_map(&mx, x, xcols, xblocks, &xslabs);
    }
    if (!ok) return cudaErrorInvalidValue;
    p.m_slabs = b.y_on_m ? yslabs : xslabs; p.n_slabs = b.y_on_m ? xslabs : yslabs;
    const CUtensorMap mm = b.y_on_m ? my : mx, mn = b.y_on_m ? mx : my;
    for (int ot = 0; ot < oTiles; ot += oStep)
        for (int it = 0; it < iTiles; it += iStep) {
            const int oc = oTiles - ot < oStep ? oTiles - ot : oStep, ic = iTiles - it < iStep ? iTiles - it : iStep;
            p.mTiles = b.y_on_m ? oc : ic; p.nTiles = b.y_on_m ? ic : oc;
            p.mt0 = b.y_on_m ? ot : it; p.nt0 = b.y_on_m ? it : ot;
            p.o0 = ot * tile_o; p.i0 = it * tile_i; p.iCount = covered(tile_i, it, ic, sp.Ci);
            const int64_t entries = (int64_t)covered(tile_o, ot, oc, sp.Co) * p.iCount * sp.tuple;
            p.part_stride = entries;
            p.part = b.splits > 1 ? scratch : dw;
            cudaError_t e = dispatch_split(sp.D, sp.dtype, [&](auto dc, auto io) -> cudaError_t {
                constexpr int D = decltype(dc)::value;
                using IO = decltype(io);
                static SmemLimitOnce limit[2];
                auto kernel = split_bwd_weight_kernel<D, IO, false>;
                if constexpr (D != 0 && sizeof(IO) == 2) { if (x_saved) kernel = split_bwd_weight_kernel<D, IO, true>; }
                if (cudaError_t err = limit[x_saved ? 1 : 0].ensure(kernel, kSmemMax, kThreadsSbw, D == 0 ? kWarpX0 * 32 * kRoleRegs + kXThreads * kXRegs : 0); err != cudaSuccess) return err;
                cudaLaunchConfig_t cfg{};
                cudaLaunchAttribute attr[2];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
                attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see ptx::grid_dependency_wait
                attr[1].val.programmaticStreamSerializationAllowed = 1;
                cfg.gridDim = dim3(2 * p.mTiles * p.nTiles * b.splits);
                cfg.blockDim = dim3(kThreadsSbw); cfg.dynamicSmemBytes = kFixedSmem + p.stages * p.stage_bytes; cfg.stream = stream;
                cfg.attrs = attr; cfg.numAttrs = 2;
                return cudaLaunchKernelEx(&cfg, kernel, mm, mn, p);
            });
            if (e != cudaSuccess || b.splits == 1) return e;     // (one range: all tiles in one launch)
            const bool last = ot + oc == oTiles && it + ic == iTiles;                    // db: once every tile has left its share
            const int64_t nw4 = entries / 4, items = last && nw4 < sp.Co ? sp.Co : nw4;
            const int row4 = p.iCount * sp.tuple / 4, pitch4 = sp.Ci * sp.tuple / 4;
            auto finalize = [&](auto kernel, int cols, int chains) {
                return launch_overlapped(kernel, dim3((unsigned)((items + cols - 1) / cols)), dim3(cols * chains), 0, stream, p.part, p.db_part,
                                         b.splits, b.splits * b.shares, nw4, row4, pitch4, sp.Co,
                                         dw + ((size_t)p.o0 * sp.Ci + p.i0) * sp.tuple, last ? db : nullptr);
            };
            e = finalize_narrow(b.splits, (int64_t)sp.Co * sp.Ci * sp.tuple / 4) ? finalize(split_finalize_kernel<8, 16>, 8, 16) : finalize(split_finalize_kernel<32, 8>, 32, 8);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace eql
