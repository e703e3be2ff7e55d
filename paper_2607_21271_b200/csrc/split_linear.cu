// Coset-split forward / data-gradient kernel on the tensor cores (16-bit I/O, or float as 3xTF32; FP32 accumulation): the layer as one or two
// dense products (see split_common.cuh), run by CTA pairs with tcgen05.mma.cta_group::2.
//
//   1 thread     TMA: raw rows of x, [128 tokens x 64 elements] per K stage, into a ring slot
//   8 warps      in place, raw rows -> [x+ | x-] (one packed add and one subtract): the slot is then the K-major operand
//                [128 tokens x 2 x 32], 128-byte swizzle.  (Unsplit: the raw rows are the operand.)
//   1 thread     TMA: weight tiles [nb/2 rows x (W+ 32 | W- 32)]
//   1 warp       tcgen05.mma M = 256 (two CTAs' tokens), N = nb, into y+ and y- accumulators of nb TMEM columns each
//   8 warps      tcgen05.ld, y+ + y- and y+ - y-, bias, optional GELU, one rounding, packed; [32 tokens x 128 bytes] per warp
//                staged in shared memory and written by TMA stores, which run beside the next unit's MMAs
//
// A unit is (256 tokens, nb columns of each product); units are dealt round-robin to the pairs, column tile fastest, so
// the pairs that work on one token tile run together and x comes from DRAM once.
//
// Bounds, per SM: a stage's bytes from L2, 16 KB of x and 64 nb of weights at ~50 B per cycle with all SMs loading, i.e. 640
// cycles at nb = 256, 2 nb cycles of MMA, and for layers with few input channels the stores.  Six slots of x and four of
// weights cover most of the TMA latency (~2.5 K cycles from the release of a slot to its data under load).  Measured on the way
// (T = 32, 32 -> 32 channels, 65536 tokens): x loaded into registers, whose data was waited for where the loads stood, 125 us;
// separate rings for raw rows and operands, four slots each, 92; one ring 80.  Stores of 32 bytes per lane straight from
// registers took 113 us where TMA stores of whole lines take 68 (T = 4, 24 -> 96 channels, 401408 tokens), 103 against 47 where
// rows are not whole sectors (T = 8, 10 -> 117 channels, 96774 tokens).
//
// Eight epilogue warps (sixteen: the same times within 2 %, but their staging cost two weight slots, whose ring then bounded: T = 8,
// 96 -> 384 channels, 25216 tokens, 71.4 against 70.1 us).  Reading the accumulators ahead of the arithmetic gained nothing.
//
// Float.  A value is hi + lo, both TF32, and the products hi hi + hi lo + lo hi.  The tensor core adds into its accumulator with
// truncation, so the error grows with the number of additions to a large accumulator.  The kernel therefore goes over the
// reduction twice: first the two small products, while the accumulator is small, then hi hi alone -- a third of the additions
// that count.  Relative error at T = 4, 256 channels: 1.4e-6, against 3.2e-6 of the frequency-domain kernel.  An operand row of
// the first pass is [+hi 8 | -hi 8 | +lo 8 | -lo 8] (a block of 32 raw columns fills two slots), of the second [+hi 16 | -hi 16] (in
// place); four MMAs of 256 x nb x 8 per slot either way, 512 cycles at nb = 256.  x is read twice, the second time from L2.
// T = 4, 256 -> 256 channels, 32768 tokens: 229 us on the frequency-domain kernel, 162 here, of which the MMAs are ~105; the rest
// is the latency from a slot's release over the copy and the transform to its next MMAs.  sixteen transform warps and eight slots
// of x against eight and six: 162 / 171; conversions to TF32 (a quarter of the rate) instead of cutting hi off: 195.
//
// Every wait on an mbarrier is bounded, as in the other tensor-core kernels.  The leader's MMA warp waits at CTA scope for arrivals
// that stand for the peer's shared memory too: the peer's threads fence their writes towards the async proxy, which reads them, before
// they arrive, and a wait with acquire at cluster scope costs ~250 cycles per stage.
#include <cuda_fp16.h>

#include <atomic>

#include "split_common.cuh"
#include "tensor_map.h"

namespace eql {
namespace {

constexpr int kWarpTmaW = 0, kWarpMma = 1, kWarpTmaX = 2, kWarpEpi0 = 4, kWarpX0 = kWarpEpi0 + 8;
// Transform warps (two groups that take alternate stages), slots of x (an even number: a group of transform
// warps sees every phase of its slots).  Float data is twice the transform per slot and half the slots per byte of x.
constexpr int kEpiWarps = kWarpX0 - kWarpEpi0;
constexpr int x_warps(int elem) { return elem == 4 ? 16 : 8; }
constexpr int a_slots(int elem) { return elem == 4 ? 8 : 6; }
constexpr int split_threads(int S, int elem) { return 32 * (kWarpEpi0 + kEpiWarps + (S == 2 ? x_warps(elem) : 0)); }
constexpr int kMaxASlots = 8;
constexpr int kStageOut = 32 * 128;           // staged output block of an epilogue warp: 32 tokens x 128 bytes
constexpr int kTileA = 128 * 128;             // bytes of a slot of x
constexpr uint32_t kSpin = 256;
constexpr int kGeluStages = 16;               // main loops worth hiding a GELU behind, see choose_nb
constexpr int kGeluHidden = 24;               // main loops that hide an unrolled one, see launch_split_linear
constexpr int kRestRegs = 48, kEpiRegs = 120;  // float: registers of the epilogue warps and of the others

struct SplitParams {
    uint8_t* stash;              // optional: also write x+ | x- as [2][N][stash_pitch bytes] (weight gradient of the batch)
    const float* bias;           // per output column of one product, or nullptr
    int* status;
    int64_t N;
    int out_row;                 // bytes of a row of y
    int stash_pitch;             // bytes of a row of the saved halves
    int nb, nTiles, nK;          // columns per tile, column tiles, ring slots per unit
    int nRaw;                    // float: blocks of 32 raw columns (two slots each in the first pass, one in the second)
    int last_ksteps;             // K steps of 16 per product in the last stage
    int nbuf;                    // accumulators in flight
    int sb;                      // slots of the weight ring
    int num_units, step_tile, step_tt;       // from a pair's unit to its next one: column tiles and token tiles (pairs = step_tt * nTiles + step_tile)
};

struct SplitBarriers {
    uint64_t full[kMaxASlots];    // leader CTA, stage n on full[n % slots]: both CTAs' operands are there
    uint64_t done[kMaxASlots];    // both CTAs: the MMAs of stage n have read them (float: and the warps that leave the slot to the other group have seen it)
    uint64_t raw_full[kMaxASlots];    // this CTA's raw rows have landed
    uint64_t full_d[2], empty_d[2], mma_done;
    uint32_t tmem_base;
    int abort_flag;
    alignas(16) float bias[256];
};

// A pair's units: unit u is (token tile u / nTiles, column tile u % nTiles), a pair takes every pairs-th.
struct Units {
    int tile, tt, left;
    __device__ __forceinline__ explicit Units(const SplitParams& p) {
        const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
        tile = pair % p.nTiles;
        tt = pair / p.nTiles;
        left = (p.num_units - pair + pairs - 1) / pairs;
    }
    __device__ __forceinline__ void next(const SplitParams& p) {
        tile += p.step_tile;
        tt += p.step_tt;
        if (tile >= p.nTiles) { tile -= p.nTiles; ++tt; }
        --left;
    }
    __device__ __forceinline__ int row0(uint32_t rank) const { return (tt * 2 + (int)rank) * 128; }
};

// D: pair distance, 0 = unsplit
// ACT: 0 none, 1 GELU, 2 GELU behind a long main loop (16-bit data, see the epilogue)
template <int D, typename IO, int ACT>
__global__ void __launch_bounds__(split_threads(D == 0 ? 1 : 2, sizeof(IO)), 1)
split_linear_kernel(const __grid_constant__ CUtensorMap tmap_in, const __grid_constant__ CUtensorMap tmap_w,
                    const __grid_constant__ CUtensorMap tmap_out, const SplitParams prm) {
    constexpr int S = D == 0 ? 1 : 2;
    constexpr bool F32 = sizeof(IO) == 4;
    static_assert(!F32 || (S == 2 && ACT != 2), "float layers are split, their GELU in a loop");
    constexpr int kXWarps = x_warps(sizeof(IO));
    constexpr int kASlots = a_slots(sizeof(IO));
    constexpr int KSTEPS = S == 2 ? 2 : 4;                       // K steps of 32 bytes per product and slot
    constexpr int kBoxCols = 128 / (int)sizeof(IO);              // elements of 128 bytes
    extern __shared__ uint8_t smem_raw_base[];
    uint8_t* smem = ptx::align_smem_1024(smem_raw_base);
    const int sb = prm.sb, nb = prm.nb, nK = prm.nK;
    uint8_t* aring = smem;
    uint8_t* staging = aring + kASlots * kTileA;
    uint8_t* bring = staging + kEpiWarps * kStageOut;
    const int b_bytes = (nb / 2) * 128;                          // this CTA's weight rows of a stage
    SplitBarriers* bar = reinterpret_cast<SplitBarriers*>(bring + sb * b_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &bar->abort_flag;
    int* status = prm.status;
    const uint32_t rank = ptx::cluster_ctarank();

    if (threadIdx.x == 0) {
        // "full" (leader): its weight TMA thread, which announces the bytes of both CTAs, and both CTAs' transform warps
        for (int i = 0; i < kASlots; ++i) {
            ptx::mbar_init(&bar->full[i], 1 + (S == 2 ? kXWarps : 0));
            ptx::mbar_init(&bar->done[i], 1 + (F32 ? kXWarps / 2 : 0));
            ptx::mbar_init(&bar->raw_full[i], 1);
        }
        for (int i = 0; i < 2; ++i) { ptx::mbar_init(&bar->full_d[i], 1); ptx::mbar_init(&bar->empty_d[i], 2 * kEpiWarps); }
        ptx::mbar_init(&bar->mma_done, 1);
        bar->abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_in);
        ptx::prefetch_tensormap(&tmap_w);
    }
    if (warp == kWarpMma) { ptx::tmem_alloc_pair(&bar->tmem_base, 512); ptx::tmem_relinquish_pair(); }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();                      // the peer's barriers must be initialised before anything arrives on them
    ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bar->tmem_base;
    // (nothing above touches global memory that an earlier kernel writes; the roles wait for it themselves, see ptx::grid_dependency_wait)

    // The pair's last meeting: no CTA may leave, or free its tensor memory, while the other can still signal it or read its own.
    // 16-bit data: where every pair has one unit, the warps arrive as they get there, epilogue warps with a single block to store once they have read the
    // accumulators (T = 4, 64 -> 64 channels, 500 tokens 5.03 -> 4.72 us a pass); behind stores the arrival would wait for them.  With
    // more units they arrive together (order 6, 92 -> 60 channels, 10007 tokens, step 41.0 us, 41.4 the other way), as
    // do those of float layers (order 8, 48 -> 48 channels, 12608 tokens, step 76.7, 77.5).
    const bool once = !F32 && prm.num_units * 2 == (int)gridDim.x;
    bool met = false;
    const uint32_t leader_full = ptx::map_to_cta(ptx::smem_u32(&bar->full[0]), 0u);

    // Registers (float): 28 warps launch with 72 each = 2016 per lane; 20 warps at 48 and the 8 epilogue warps at 120 make 1920.
    if (warp < kWarpEpi0) {
        if constexpr (F32) ptx::reg_dealloc<kRestRegs>();
        if (warp == kWarpTmaW && lane == 0) {
            // ------------------------------------------------------------ weight tiles
            // Slot n % sb is free when the MMAs of stage n - sb are done (sb <= slots of x: a parity wait on that stage's barrier
            // is unambiguous, its next phase needs stage n itself).
            uint32_t n = 0, d = 0;                               // stage; stage whose completion frees its slot
            int slot = 0;
            bool ok = true;
            const uint32_t bytes = 2u * (uint32_t)(b_bytes + (S == 1 ? kTileA : 0));
            for (Units u(prm); u.left > 0 && ok; u.next(prm)) {
                const int wrow = u.tile * nb + (int)rank * (nb / 2);
                for (int kc = 0; kc < nK; ++kc, ++n) {
                    if (n >= (uint32_t)sb) {
                        ok = ptx::mbar_wait(&bar->done[d % kASlots], (d / kASlots) & 1, abort_flag, status, 401, true, kSpin);
                        if (!ok) break;
                        ++d;
                    }
                    if (n == 0) ptx::grid_handover();
                    if (rank == 0) ptx::mbar_arrive_expect_tx(&bar->full[n % kASlots], bytes);
                    ptx::tma_load_2d_pair(bring + slot * b_bytes, &tmap_w, kc * kBoxCols, wrow, leader_full + (n % kASlots) * 8u);
                    if (++slot == sb) slot = 0;
                }
            }
            for (; d < n; ++d)                                   // every copy must have landed before the CTA may exit
                ptx::mbar_wait(&bar->done[d % kASlots], (d / kASlots) & 1, abort_flag, status, 411, false);
        } else if (warp == kWarpTmaX && lane == 0) {
            // ------------------------------------------------------------ rows of x (a thread of its own: one thread gets a
            // copy accepted only every ~350 cycles)
            uint32_t n = 0;
            bool ok = true;
            for (Units u(prm); u.left > 0 && ok; u.next(prm)) {
                const int row0 = u.row0(rank);
                for (int kc = 0; kc < nK; ++kc, ++n) {
                    const uint32_t slot = n % kASlots;
                    if (n >= (uint32_t)kASlots) {
                        ok = ptx::mbar_wait(&bar->done[slot], ((n / kASlots) & 1) ^ 1, abort_flag, status, 407, true, kSpin);
                        if (!ok) break;
                    }
                    if (n == 0) ptx::grid_handover();
                    if constexpr (F32) {
                        if (kc < 2 * prm.nRaw && (kc & 1)) {     // the second slot of a pair is filled by the transform alone
                            ptx::mbar_arrive(&bar->raw_full[slot]);
                            continue;
                        }
                        const int block = kc < 2 * prm.nRaw ? kc >> 1 : kc - 2 * prm.nRaw;
                        ptx::mbar_arrive_expect_tx(&bar->raw_full[slot], kTileA);
                        ptx::tma_load_2d(aring + slot * kTileA, &tmap_in, block * kBoxCols, row0, &bar->raw_full[slot]);
                    } else if constexpr (S == 2) {
                        ptx::mbar_arrive_expect_tx(&bar->raw_full[slot], kTileA);
                        ptx::tma_load_2d(aring + slot * kTileA, &tmap_in, kc * 64, row0, &bar->raw_full[slot]);
                    } else {
                        ptx::tma_load_2d_pair(aring + slot * kTileA, &tmap_in, kc * 64, row0, leader_full + slot * 8u);
                    }
                }
            }
            for (uint32_t c = n > (uint32_t)kASlots ? n - kASlots : 0; c < n; ++c)
                ptx::mbar_wait(&bar->done[c % kASlots], (c / kASlots) & 1, abort_flag, status, 417, false);
        } else if (warp == kWarpMma && rank == 0) {
            // ------------------------------------------------------------ tensor-core issue (leader CTA, one elected lane)
            ptx::grid_handover();
            uint32_t n = 0, cu = 0;
            int bslot = 0;
            bool ok = true;
            const uint32_t idesc = F32 ? ptx::umma_idesc_tf32_f32(256, nb) : ptx::umma_idesc_f16_f32(256, nb, H16<IO>::kUmmaFormat);
            const uint64_t a_ring = desc_k_sw128(ptx::smem_u32(aring)), b_ring = desc_k_sw128(ptx::smem_u32(bring));
            const uint64_t b_slot = (uint64_t)b_bytes >> 4;
            for (Units u(prm); u.left > 0 && ok; u.next(prm), ++cu) {
                const uint32_t buf = prm.nbuf == 2 ? (cu & 1) : 0u, use = prm.nbuf == 2 ? (cu >> 1) : cu;
                const uint32_t d0 = tmem_base + buf * (uint32_t)(S * nb);
                ok = ptx::mbar_wait_warp(&bar->empty_d[buf], (use & 1) ^ 1, abort_flag, status, 402, true, kSpin);
                if (!ok) break;
                int kc = 0;
                if constexpr (F32) {
                    // first pass: [+hi 8 | -hi 8 | +lo 8 | -lo 8], the two small products of either half
                    for (; kc < 2 * prm.nRaw; ++kc, ++n) {
                        const uint32_t slot = n % kASlots;
                        ok = ptx::mbar_wait_warp(&bar->full[slot], (n / kASlots) & 1, abort_flag, status, 403, true, kSpin);
                        if (!ok) break;
                        ptx::tc_fence_after_sync();
                        const uint64_t a0 = a_ring + (uint64_t)(slot * (kTileA >> 4)), b0 = b_ring + (uint64_t)bslot * b_slot;
                        if (ptx::elect_one()) {
#pragma unroll
                            for (int s = 0; s < S; ++s) {
                                ptx::umma_tf32_pair(d0 + (uint32_t)(s * nb), a0 + 2 * s, b0 + 4 + 2 * s, idesc, kc ? 1u : 0u);
                                ptx::umma_tf32_pair(d0 + (uint32_t)(s * nb), a0 + 4 + 2 * s, b0 + 2 * s, idesc, 1u);
                            }
                            ptx::umma_commit_pair_both(&bar->done[slot]);
                        }
                        __syncwarp();
                        if (++bslot == sb) bslot = 0;
                    }
                }
                for (; kc < nK && ok; ++kc, ++n) {
                    const uint32_t slot = n % kASlots;
                    ok = ptx::mbar_wait_warp(&bar->full[slot], (n / kASlots) & 1, abort_flag, status, 403, true, kSpin);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t a0 = a_ring + (uint64_t)(slot * (kTileA >> 4)), b0 = b_ring + (uint64_t)bslot * b_slot;
                    const int ksteps = kc + 1 < nK ? KSTEPS : prm.last_ksteps;
                    if (ptx::elect_one()) {
                        // 32 bytes per K step; the second product's half of the 128-byte rows comes behind the first's
#pragma unroll
                        for (int s = 0; s < S; ++s)
#pragma unroll
                            for (int k = 0; k < KSTEPS; ++k)
                                if (k < ksteps) {
                                    if constexpr (F32)
                                        ptx::umma_tf32_pair(d0 + (uint32_t)(s * nb), a0 + 4 * s + 2 * k, b0 + 4 * s + 2 * k, idesc, 1u);
                                    else
                                        ptx::umma_f16_pair(d0 + (uint32_t)(s * nb), a0 + 4 * s + 2 * k, b0 + 4 * s + 2 * k, idesc,
                                                           (kc | k) ? 1u : 0u);
                                }
                        ptx::umma_commit_pair_both(&bar->done[slot]);
                        if (kc + 1 == nK) ptx::umma_commit_pair_both(&bar->full_d[buf]);
                    }
                    __syncwarp();
                    if (++bslot == sb) bslot = 0;
                }
            }
            if (ptx::elect_one()) ptx::umma_commit_pair(&bar->mma_done);
            __syncwarp();
            ptx::mbar_wait_warp(&bar->mma_done, 0, abort_flag, status, 413, false);
        }
    } else if (S == 2 && warp >= kWarpX0) {
        // ---------------------------------------------------------------- raw rows -> [x+ | x-], in place
        ptx::grid_handover();
        if constexpr (F32) {
            ptx::reg_dealloc<kRestRegs>();
            // Two groups of eight warps take alternate blocks of raw columns; a warp has 16 rows, a lane 4 representatives and their
            // partners of a row at a time.  First pass: hi and lo of both halves, 8 + 8 columns of each per slot, over two slots;
            // second pass: hi only, one slot.  Rows r and r ^ 5 share a shared-memory wavefront, as for 16-bit data; the lanes of
            // the upper columns (whose chunks would meet those of the lower ones) write the halves in the opposite order: they
            // compute the difference first.
            // hi is cut off, not rounded: one instruction instead of a conversion at a quarter of the rate.  Its lo part then has
            // the sign of the value, but the weights' are rounded, so that the product of the lo parts, which is left out, still
            // has no preferred sign.  lo is rounded by adding half a unit: the tensor core ignores the bits below.
            const int group = (warp - kWarpX0) >> 3, wx = (warp - kWarpX0) & 7;
            const int g = lane & 3, r8 = (lane >> 3) ^ (((lane >> 2) & 1) ? 5 : 0), up = g >> 1;
            const int row_off = (wx * 16 + r8) * 128;
            const int a_off = row_off + (((2 * g) ^ r8) << 4), b_off = row_off + (((2 * g + 1) ^ r8) << 4);
            // places of the half computed first: hi and lo of the first pass, hi of the second; the other half's differ by one bit
            const int hi_off = row_off + (((2 * up + (g & 1)) ^ r8) << 4), lo_off = hi_off ^ 64;
            const int hi2_off = row_off + (((4 * up + g) ^ r8) << 4);
            const float sgn = up ? -1.f : 1.f;
            Units u(prm);
            const uint32_t total = (uint32_t)u.left * (uint32_t)nK;
            int kc = 0;
            uint32_t slot = 0, ph = 0, item = 0;
            for (uint32_t n = 0; n < total; ++item) {
                const bool first = kc < 2 * prm.nRaw;
                // Every warp waits for every slot, in order: a group that skipped the other's could take an old phase for its own.  And
                // it says that it has seen the other's: else the other group's work, the MMAs and a new copy could go through the slot
                // twice over while a late warp still waits for the first copy, and its parity test would wait for one too many.
                if (!ptx::mbar_wait(&bar->raw_full[slot], ph, abort_flag, status, 408, true, 4)) break;
                const uint32_t cur = slot;
                uint32_t next = slot;
                if (++slot == (uint32_t)kASlots) { slot = 0; ph ^= 1u; }
                if (first) {                                     // the second slot must be free too
                    next = slot;
                    if (!ptx::mbar_wait(&bar->raw_full[next], ph, abort_flag, status, 409, true, 4)) break;
                    if (++slot == (uint32_t)kASlots) { slot = 0; ph ^= 1u; }
                }
                n += first ? 2 : 1;
                kc += first ? 2 : 1;
                if (kc == nK) kc = 0;
                if ((item & 1) != (uint32_t)group) {
                    __syncwarp();
                    if (lane == 0) {
                        ptx::mbar_arrive(&bar->done[cur]);
                        if (first) ptx::mbar_arrive(&bar->done[next]);
                    }
                    continue;
                }
                uint8_t* tile = aring + cur * kTileA;
                uint8_t* dst = up ? aring + next * kTileA : tile;
                {
                    uint4 a[2], b[2];
#pragma unroll
                    for (int i = 0; i < 2; ++i) { a[i] = lds128(tile + i * 1024 + a_off); b[i] = lds128(tile + i * 1024 + b_off); }
                    __syncwarp();                                // the rows have been read before any lane writes into them
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float x[8] = {__uint_as_float(a[i].x), __uint_as_float(a[i].y), __uint_as_float(a[i].z), __uint_as_float(a[i].w),
                                            __uint_as_float(b[i].x), __uint_as_float(b[i].y), __uint_as_float(b[i].z), __uint_as_float(b[i].w)};
#pragma unroll
                        for (int t = 0; t < 2; ++t) {            // (a product by 1 or -1: the sum or the difference, rounded once)
                            uint32_t hi[4], lo[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int e = (j / D) * 2 * D + j % D;
                                const float v = fmaf(t ? -sgn : sgn, x[e + D], x[e]);
                                hi[j] = __float_as_uint(v) & 0xFFFFE000u;
                                lo[j] = __float_as_uint(v - __uint_as_float(hi[j])) + 0x1000u;
                            }
                            if (first) {
                                *reinterpret_cast<uint4*>(dst + i * 1024 + (hi_off ^ (t << 5))) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                                *reinterpret_cast<uint4*>(dst + i * 1024 + (lo_off ^ (t << 5))) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                            } else {
                                *reinterpret_cast<uint4*>(tile + i * 1024 + (hi2_off ^ (t << 6))) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                            }
                        }
                    }
                }
                ptx::fence_proxy_async_smem();                   // generic-proxy writes -> visible to the MMA (async proxy)
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive_remote(leader_full + cur * 8u);
                    if (first) ptx::mbar_arrive_remote(leader_full + next * 8u);
                }
            }
        } else if constexpr (S == 2) {
            // A warp has 32 rows of a stage, 8 rows x 4 granules at a time.  Rows r and r ^ kRowPair share a shared-memory
            // wavefront: the chunks read are disjoint when the rows differ in parity (D = 16: in the second bit), the chunks
            // written (0..3 for x+, 4..7 for x-) when they differ in the third bit.
            constexpr int kRowPair = D == 16 ? 6 : 5;
            const int group = (warp - kWarpX0) >> 2, wx = (warp - kWarpX0) & 3;
            const int g = lane & 3, r8 = (lane >> 3) ^ (((lane >> 2) & 1) ? kRowPair : 0);
            const int ca = granule_chunk<D>(g), cb = ca + kPartnerChunk<D>;
            const int row_off = (wx * 32 + r8) * 128;
            const int a_off = row_off + ((ca ^ r8) << 4), b_off = row_off + ((cb ^ r8) << 4);
            const int p_off = row_off + ((g ^ r8) << 4), m_off = row_off + (((4 | g) ^ r8) << 4);
            Units u(prm);                                        // (position: for the saved halves only)
            const uint32_t total = (uint32_t)u.left * (uint32_t)nK;
            int pk = group;                                      // K stage inside the unit
            while (pk >= nK) { pk -= nK; u.next(prm); }
            for (uint32_t n = group; n < total; n += 2) {
                const uint32_t slot = n % kASlots;
                if (!ptx::mbar_wait(&bar->raw_full[slot], (n / kASlots) & 1, abort_flag, status, 408, true, 4)) break;
                uint8_t* tile = aring + slot * kTileA;
                const bool save = prm.stash != nullptr && pk % prm.nTiles == u.tile;   // the column tiles share the saving
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    uint8_t* t = tile + h * 2048;
                    const uint4 a0 = lds128(t + a_off), b0 = lds128(t + b_off), a1 = lds128(t + 1024 + a_off), b1 = lds128(t + 1024 + b_off);
                    uint4 p0, m0, p1, m1;
                    split_granule<D, IO>(a0, b0, p0, m0);
                    split_granule<D, IO>(a1, b1, p1, m1);
                    __syncwarp();                                // the eight rows have been read before any lane writes into them
                    *reinterpret_cast<uint4*>(t + p_off) = p0;
                    *reinterpret_cast<uint4*>(t + m_off) = m0;
                    *reinterpret_cast<uint4*>(t + 1024 + p_off) = p1;
                    *reinterpret_cast<uint4*>(t + 1024 + m_off) = m1;
                    if (save) {
                        const int c = pk * 64 + g * 16;
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int row = u.row0(rank) + wx * 32 + r8 + 16 * h + 8 * i;
                            if (row < prm.N && c < prm.stash_pitch) {
                                uint8_t* s = prm.stash + (size_t)row * prm.stash_pitch + c;
                                const uint4 p = i ? p1 : p0, m = i ? m1 : m0;
                                ptx::st_global_v4(s, p.x, p.y, p.z, p.w);
                                ptx::st_global_v4(s + (size_t)prm.N * prm.stash_pitch, m.x, m.y, m.z, m.w);
                            }
                        }
                    }
                }
                ptx::fence_proxy_async_smem();                   // generic-proxy writes -> visible to the MMA (async proxy)
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(leader_full + slot * 8u);
                if (prm.stash != nullptr) {
                    pk += 2;
                    while (pk >= nK) { pk -= nK; u.next(prm); }
                }
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue: a lane owns a token
        if constexpr (F32) ptx::reg_alloc<kEpiRegs>();
        ptx::grid_handover();
        const int ew = warp - kWarpEpi0, quad = warp & 3, share = ew >> 2;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t empty_leader = ptx::map_to_cta(ptx::smem_u32(&bar->empty_d[0]), 0u);
        constexpr int GC = 32 / S;                               // accumulator columns per 32 elements (64 bytes; float: 128) of a row
        constexpr int EW4 = kEpiWarps / 4, MAXG = 256 / GC / EW4;    // groups of a warp: its share of at most 256 columns
        constexpr int BLK = F32 ? 1 : 2;                         // groups per staged block of 128 bytes
        const int groups = nb / GC, per = ((groups + EW4 - 1) / EW4 + BLK - 1) & ~(BLK - 1);
        const int g0 = share * per, g1 = g0 + per < groups ? g0 + per : groups;      // this warp's groups, contiguous
        uint32_t cu = 0;
        int bias_tile = -1;
        uint8_t* stg = staging + ew * kStageOut;
        for (Units u(prm); u.left > 0; u.next(prm), ++cu) {
            const uint32_t buf = prm.nbuf == 2 ? (cu & 1) : 0u, use = prm.nbuf == 2 ? (cu >> 1) : cu;
            const int tile = u.tile, col0 = tile * nb;           // first column of the product
            if (prm.bias != nullptr && tile != bias_tile) {      // (columns past the row's end read the padding of the bias array)
                asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
                for (int c = ew * 32 + lane; c < nb; c += kEpiWarps * 32) bar->bias[c] = __ldg(prm.bias + col0 + c);
                asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
                bias_tile = tile;
            }
            // (the warps meet at the barriers above, so none leaves alone: after a time-out, which every warp sees through the
            // abort flag, they go on without touching the output)
            const bool ok = ptx::mbar_wait(&bar->full_d[buf], use & 1, abort_flag, status, 406, true, 16);
            ptx::tc_fence_after_sync();
            uint32_t o[32];                                      // a block
            auto stage_out = [&](int blk) {
                if (lane == 0) ptx::bulk_wait_group_read0();     // the block before has been read
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t* q = &o[4 * j];
                    *reinterpret_cast<uint4*>(stg + lane * 128 + ((j ^ (lane & 7)) << 4)) = make_uint4(q[0], q[1], q[2], q[3]);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    const int c = (col0 + (g0 + BLK * blk) * GC) * S;     // element column
                    // (rows past N and columns past the row's end are clipped by the hardware)
                    if (ok && c * (int)sizeof(IO) < prm.out_row) ptx::tma_store_2d(&tmap_out, c, u.row0(rank) + quad * 32, stg);
                    ptx::bulk_commit_group();
                }
            };
            auto release = [&] {                                 // this warp has read its share of the accumulator
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(empty_leader + buf * 8u);
            };
            // GELU: the same half group by half group through shared memory, in a loop whose code is used again -- unrolled, the GELU of a
            // unit's outputs is up to 180 KB of instructions, whose fetching took ~110 cycles per output of a lane (one image, T = 8, 96 ->
            // 384 channels, 11.0 -> 10.3 us; T = 4, 64 -> 256, 32768 tokens 65 -> 55).  Not where the next unit's main loop is long enough to
            // hide even that: the warps that wait for instructions leave it the issue slots (see launch_split_linear).
            constexpr bool loop = ACT == 1;
            if constexpr (loop) {
                constexpr int WORDS = F32 ? 16 : 8;              // of a half group
#pragma unroll 1
                for (int i = 0; i < 2 * (g1 - g0); ++i) {
                    const int gi = g0 + (i >> 1), h = i & 1;
                    constexpr int HC = GC / 2;
                    const uint32_t t0 = lane_base + buf * (uint32_t)(S * nb) + (uint32_t)(gi * GC + h * HC);
                    uint32_t v[16], wd[WORDS];
                    if constexpr (S == 2) {
                        ptx::tmem_ld<8>(t0, v);
                        ptx::tmem_ld<8>(t0 + (uint32_t)nb, v + 8);
                    } else {
                        ptx::tmem_ld<16>(t0, v);
                    }
                    ptx::tmem_ld_wait();
                    if (i + 1 == 2 * (g1 - g0)) release();
                    float f[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) f[j] = __uint_as_float(v[j]);
                    if (prm.bias != nullptr) {
#pragma unroll
                        for (int j = 0; j < HC; ++j) f[j] += bar->bias[gi * GC + h * HC + j];
                    }
                    if constexpr (S == 2) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float p = f[j], m = f[8 + j];
                            f[j] = p + m;
                            f[8 + j] = p - m;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) f[j] = gelu_erf(f[j]);
                    // words of the half group, 16-byte chunks of the row in order (D = 16: the partners' chunk lies two behind)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if constexpr (F32) {
                            const int e = (j / D) * 2 * D + j % D;
                            wd[e] = __float_as_uint(f[j]);
                            wd[e + D] = __float_as_uint(f[8 + j]);
                        } else if constexpr (S == 1) {
                            wd[j] = H16<IO>::pack(f[2 * j], f[2 * j + 1]);
                        } else if constexpr (D == 1) {
                            wd[j] = H16<IO>::pack(f[j], f[8 + j]);
                        } else if (j % 2 == 0) {
                            constexpr int DH = D >= 8 ? 8 : D;
                            const int w = ((j / DH) * 2 * DH + j % DH) / 2;
                            wd[w] = H16<IO>::pack(f[j], f[j + 1]);
                            wd[w + DH / 2] = H16<IO>::pack(f[8 + j], f[9 + j]);
                        }
                    }
                    if (i % (2 * BLK) == 0) {                    // a block begins: the one before has been read
                        if (lane == 0) ptx::bulk_wait_group_read0();
                        __syncwarp();
                    }
#pragma unroll
                    for (int k = 0; k < WORDS / 4; ++k) {
                        const int chunk = F32 ? 4 * h + k : (i >> 1) % BLK * 4 + (D == 16 ? 2 * k + h : 2 * h + k);
                        *reinterpret_cast<uint4*>(stg + lane * 128 + ((chunk ^ (lane & 7)) << 4)) = make_uint4(wd[4 * k], wd[4 * k + 1], wd[4 * k + 2], wd[4 * k + 3]);
                    }
                    if (i % (2 * BLK) == 2 * BLK - 1 || i + 1 == 2 * (g1 - g0)) {
                        ptx::fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const int c = (col0 + (g0 + (i >> 1) / BLK * BLK) * GC) * S;
                            if (ok && c * (int)sizeof(IO) < prm.out_row) ptx::tma_store_2d(&tmap_out, c, u.row0(rank) + quad * 32, stg);
                            ptx::bulk_commit_group();
                        }
                    }
                }
            } else {
#pragma unroll
            for (int i = 0; i < MAXG; ++i) {
                if (g0 + i < g1) {
                    if (i > 0 && i % BLK == 0) stage_out(i / BLK - 1);
                    uint32_t* const oi = o + (i % BLK) * 16;
                    const int gi = g0 + i;
                    const uint32_t t0 = lane_base + buf * (uint32_t)(S * nb) + (uint32_t)(gi * GC);
                    // two halves of 32 bytes' worth of columns; representative column c gives element (c / D) * 2D + c % D of the
                    // 32 and its partner D elements behind
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        constexpr int HC = GC / 2;
                        uint32_t v[16];
                        if constexpr (S == 2) {
                            ptx::tmem_ld<8>(t0 + (uint32_t)(h * HC), v);
                            ptx::tmem_ld<8>(t0 + (uint32_t)(nb + h * HC), v + 8);
                        } else {
                            ptx::tmem_ld<16>(t0 + (uint32_t)(h * HC), v);
                        }
                        ptx::tmem_ld_wait();
                        if (prm.bias != nullptr) {
#pragma unroll
                            for (int j = 0; j < HC; j += 4) {
                                const float4 bv = *reinterpret_cast<const float4*>(&bar->bias[gi * GC + h * HC + j]);
                                v[j] = __float_as_uint(__uint_as_float(v[j]) + bv.x);
                                v[j + 1] = __float_as_uint(__uint_as_float(v[j + 1]) + bv.y);
                                v[j + 2] = __float_as_uint(__uint_as_float(v[j + 2]) + bv.z);
                                v[j + 3] = __float_as_uint(__uint_as_float(v[j + 3]) + bv.w);
                            }
                        }
                        if constexpr (S == 2) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float p = __uint_as_float(v[j]), m = __uint_as_float(v[8 + j]);
                                v[j] = __float_as_uint(p + m);
                                v[8 + j] = __float_as_uint(p - m);
                            }
                        }
                        if constexpr (ACT != 0) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(gelu_erf(__uint_as_float(v[j])));
                        }
                        if constexpr (F32) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int c = h * 8 + j, e = (c / D) * 2 * D + c % D;
                                o[e] = v[j];
                                o[e + D] = v[8 + j];
                            }
                        } else {
                        auto word = [&](int x, int y) { return H16<IO>::pack(__uint_as_float(v[x]), __uint_as_float(v[y])); };
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if constexpr (S == 1) oi[h * 8 + j] = word(2 * j, 2 * j + 1);
                            else if constexpr (D == 1) oi[h * 8 + j] = word(j, 8 + j);
                            else if (j % 2 == 0) {
                                const int c = h * 8 + j, w = ((c / D) * 2 * D + c % D) / 2;
                                oi[w] = word(j, j + 1);
                                oi[w + D / 2] = word(8 + j, 9 + j);
                            }
                        }
                        }
                    }
                }
            }
            }
            if (!loop || g0 >= g1) release();
            if (ACT == 0 && once && g1 - g0 <= BLK) {
                __syncwarp();
                ptx::cluster_arrive();
                met = true;
            }
            if (!loop && g0 < g1) stage_out((g1 - g0 - 1) / BLK);
        }
        if (lane == 0) ptx::bulk_wait_group_read0();
    }

    ptx::tc_fence_before_sync();
    __syncwarp();                               // (roles of one lane: the arrival is a whole warp's)
    if (once && !met) ptx::cluster_arrive();
    __syncthreads();
    if (!once) ptx::cluster_arrive();
    ptx::cluster_wait();
    if (warp == kWarpMma) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------------
// Weight matrices of the dense products, both K-major, from w[Co][Ci][tuple]:
//   wf[(o, g)][(i, h)]  (rows of the forward product's columns)      pitch kf elements
//   wb[(i, h)][(o, g)]  (the data gradient's)                        pitch kb elements
// with entry (w[h^-1 g] + sigma_s w[h^-1 z g]) / 2 (unsplit: w[h^-1 g]), rounded once; the two products' matrices interleaved
// in blocks of 32 columns, [W+ 32 | W- 32], padded with zeros to whole blocks; and the bias expanded to one value per column
// of the forward product.  A block builds CH x CH channel pairs: about 32 x 32 entries, so that both matrices are written in
// 16-byte pieces of contiguous 64..128-byte runs.
// Float matrices hold what the kernel's two passes read: per 8 columns [W+ 8 | W- 8 | lo of W+ | lo of W-], hi and lo parts in
// TF32, and behind all of these, per 16 columns, [W+ 16 | W- 16], hi parts only.
struct WeightParams {
    int Ci, Co;
    int corr;                    // weight index h^-1 g replaced by its inverse
    int kf, kb;                  // pitches (elements)
    int first_f, first_b;        // float: elements of a row the first pass reads
};

// Channels per block side: about 32 entries, rows of whole 16 bytes.  (64 leave small layers to a handful of blocks: T = 8, 48 -> 48
// channels, float, 8.9 against 3.4 us, 24 -> 96 at T = 4 4.8 against 3.3; with 16 representatives, two channels per side, large
// layers take longer: 128 -> 128 at T = 32 14.1 against 11.3.)
constexpr int weight_block(int reps) {
    int ch = reps < 16 ? 32 / reps : 64 / reps;
    while ((ch * reps) % 8 != 0) ++ch;
    return ch;
}

template <typename R, int S, typename IO>
__global__ void __launch_bounds__(256)
split_weights_kernel(const IO* __restrict__ w, const IO* __restrict__ bias, IO* __restrict__ wf, IO* __restrict__ wb,
                     float* __restrict__ bias_cols, const WeightParams prm) {
    constexpr int TUPLE = R::kTuple, REPS = TUPLE / S, CH = weight_block(REPS), SIDE = CH * REPS;
    constexpr int PITCH = SIDE + 1;                              // floats per output channel: consecutive rows on distinct banks
    __shared__ float c[S][CH * PITCH];                           // [o][i * REPS + rep]
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int o0 = blockIdx.y * CH, i0 = blockIdx.x * CH;
    for (int e = threadIdx.x; e < CH * SIDE; e += 256) {
        const int o = e / SIDE, x = e % SIDE, i = x / REPS, rep = x % REPS;
        float a = 0.f, b = 0.f;
        if (o0 + o < prm.Co && i0 + i < prm.Ci) {
            const IO* wt = w + ((size_t)(o0 + o) * prm.Ci + i0 + i) * TUPLE;
            int q = R::element(rep), qz = S == 2 ? q + R::kHalf : q;
            if (prm.corr) { q = (TUPLE - q) % TUPLE; qz = (TUPLE - qz) % TUPLE; }    // cyclic groups only
            a = (float)wt[q];
            if (S == 2) b = (float)wt[qz];
        }
        if constexpr (S == 2) { c[0][o * PITCH + x] = 0.5f * (a + b); c[S - 1][o * PITCH + x] = 0.5f * (a - b); }
        else c[0][o * PITCH + x] = a;
    }
    __syncthreads();
    const int rows_f = prm.Co * REPS, rows_b = prm.Ci * REPS;    // rows of the matrices
    auto entry = [&](int s, int o, int i, int h, int g) {
        bool z;
        const int rep = R::template combine<false>(h, g, z);
        const float x = c[s][o * PITCH + i * REPS + rep];
        return (s == 1 && z) ? -x : x;
    };
    // 8 entries of a row per thread: forward matrix, rows (o, g), columns (i, h); data-gradient matrix, rows (i, h), columns (o, g)
    for (int e = threadIdx.x; e < 2 * S * SIDE * (SIDE / 8); e += 256) {
        const int ch = e % (SIDE / 8), r = (e / (SIDE / 8)) % SIDE, sm = e / (SIDE / 8 * SIDE);
        const int s = S == 2 ? sm & 1 : 0;
        const bool back = (S == 2 ? sm >> 1 : sm) != 0;
        const int rc = r / REPS, rr = r % REPS;
        const int col = (back ? o0 : i0) * REPS + ch * 8, row = (back ? i0 : o0) * REPS + r;
        if constexpr (sizeof(IO) == 4) {
            const int first = back ? prm.first_b : prm.first_f;
            if (row >= (back ? rows_b : rows_f) || col * 4 >= first) continue;
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int k = ch * 8 + j, kc = k / REPS, kh = k % REPS;
                split_tf32(back ? entry(s, kc, rc, rr, kh) : entry(s, rc, kc, kh, rr), hi[j], lo[j]);
            }
            IO* dst = back ? wb + (size_t)row * prm.kb : wf + (size_t)row * prm.kf;
            IO* d1 = dst + col * 4 + s * 8;
            IO* d2 = dst + first + (col >> 4) * 32 + s * 16 + (col & 8);
#pragma unroll
            for (int j = 0; j < 8; j += 4) {
                const uint4 h = make_uint4(hi[j], hi[j + 1], hi[j + 2], hi[j + 3]);
                *reinterpret_cast<uint4*>(d1 + j) = h;
                *reinterpret_cast<uint4*>(d1 + 16 + j) = make_uint4(lo[j], lo[j + 1], lo[j + 2], lo[j + 3]);
                *reinterpret_cast<uint4*>(d2 + j) = h;
            }
        } else {
        const int at = S == 2 ? (col >> 5) * 64 + s * 32 + (col & 31) : col;
        if (row >= (back ? rows_b : rows_f) || at >= (back ? prm.kb : prm.kf)) continue;
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = ch * 8 + 2 * j, c0 = k / REPS, h0 = k % REPS, c1 = (k + 1) / REPS, h1 = (k + 1) % REPS;
            v[j] = back ? H16<IO>::pack(entry(s, c0, rc, rr, h0), entry(s, c1, rc, rr, h1))
                        : H16<IO>::pack(entry(s, rc, c0, h0, rr), entry(s, rc, c1, h1, rr));
        }
        *reinterpret_cast<uint4*>((back ? wb + (size_t)row * prm.kb : wf + (size_t)row * prm.kf) + at) = make_uint4(v[0], v[1], v[2], v[3]);
        }
    }
    if (bias != nullptr && blockIdx.x == 0) {
        for (int r = threadIdx.x; r < SIDE; r += 256)
            if (o0 * REPS + r < rows_f) bias_cols[o0 * REPS + r] = (float)bias[o0 + r / REPS];
    }
}

// ------------------------------------------------------------------------------------------------ host side
constexpr size_t kSmemMax = 227 * 1024;
constexpr size_t kFixedSmem = 1024 + sizeof(SplitBarriers) + 64;

// Columns per tile, by a model of the launch in cycles.  A stage takes as long as its bytes from L2, 16 KB of x and 64 nb of
// weights at ~50 B per cycle and SM with all SMs loading (measured 350 / 390 / 475 / 640 cycles at nb = 32 / 64 / 128 / 256), or
// its MMAs (2 nb); of float layers, whose transform bounds it, ~560 + 0.9 nb (608 / 730 / 800 at nb = 96 / 192 / 256).  An epilogue
// reads and packs in ~300 + 4 nb cycles and stores at ~30 B per cycle.  Accumulators of up to 256 columns in all alternate, so that
// the epilogue overlaps the next unit's MMAs; of wider ones only the stores do.  A unit costs ~500 cycles beside these.  Units go
// to the pairs in whole rounds, which is what decides for small batches: the last one counts whole, those before as long as the next
// one waits for them.  (Without the 500, and with the epilogue counted in every round, short reductions were cut into many small
// tiles: float T = 4, 8 -> 192 channels, 5000 tokens 13.9 us at nb = 16, 8.2 at 128; bfloat16 T = 4, 4 -> 248, 4000 tokens 8.4 at 32, 6.4 at 128.)
//
// GELU costs ~100 cycles per column of a product: every round counts its epilogue (T = 8, 48 -> 192 channels, 25216 tokens: 78 us at
// five rounds of 256 columns, 88 at six of 192), and it is worth hiding behind a long main loop, i.e. two narrow accumulators in
// flight rather than a wide one, where a pair has several units.  Half precision, frequency-domain kernel before / one wide / two narrow, us
// (all with the unrolled epilogue; the loop of the short ones has since made T = 8, 48 -> 192 67, 64 -> 64 46, T = 4, 64 -> 256 55):
// T = 8, 192 -> 192, 40000 tokens 179 / 224 / 147; 512 -> 512, 8000 171 / 201 / 169; 384 -> 192, 25216 145 / 226 / 180; T = 4, 256 -> 256, 32768
// 96 / 125 / 77; T = 16, 64 -> 64, 65536 174 / 217 / 146.  With fewer than 16 stages the narrow ones lose: T = 8, 64 -> 64 (8 stages), 40000
// 49 / 53; T = 4, 64 -> 256 (4 stages), 32768 65 / 76.
int choose_nb(int S, bool f32, bool act, int rows, int nK, int64_t token_tiles, int pairs) {
    const int gran = (f32 ? 32 : 64) / S;                                     // tiles of whole 128-byte pieces of a row
    double best = 1e30;
    int best_nb = 256;
    int64_t best_rounds = 0;
    for (int tiles = (rows + 255) / 256; tiles <= (rows + gran - 1) / gran; ++tiles) {
        const int nb = ((rows + tiles - 1) / tiles + gran - 1) / gran * gran;
        if (nb > 256) continue;
        const int64_t units = token_tiles * ((rows + nb - 1) / nb);
        const int64_t rounds = (units + pairs - 1) / pairs;
        const double busy = units < pairs ? (double)units / pairs : 1.0;       // few pairs: L2 is not the limit
        const double load_c = f32 ? 560 + 0.9 * nb : busy * (16384 + 64.0 * nb) / 50, mma_c = 2.0 * nb + 50;
        const double main_c = nK * (load_c > mma_c ? load_c : mma_c);
        const double read_c = 300 + 4.0 * nb, store_c = (f32 ? 17 : 8.5) * S * nb;
        double unit_c = S * nb <= 256 ? (main_c > read_c ? main_c : read_c) : main_c + read_c + 300;
        const double extra_c = act ? 0 : 500;
        if (unit_c < read_c + store_c + extra_c) unit_c = read_c + store_c + extra_c;
        const double total = (rounds - 1) * unit_c + (act ? unit_c : main_c) + read_c + store_c;
        // A single round: nothing hides the GELU, narrower tiles share it out over more SMs (of 32 columns four of the eight epilogue warps have
        // all, one on each scheduler).  197 tokens, 64 and 32 columns: T = 8, 96 -> 384 channels 10.3 and 9.8 us, 192 -> 384 14.1 and 13.4.
        if (act && best_rounds == 1 && rounds == 1) { if (total + 45.0 * S * nb < best + 45.0 * S * best_nb) { best = total; best_nb = nb; } continue; }
        if (total < best * 0.999) { best = total; best_nb = nb; best_rounds = rounds; }
        if (rounds == 1 && nb <= gran) break;
    }
    if (act && S * best_nb > 256 && nK >= kGeluStages && best_rounds > 1) {
        const int cols = 256 / S, tiles = (rows + cols - 1) / cols;
        best_nb = ((rows + tiles - 1) / tiles + gran - 1) / gran * gran;
    }
    return best_nb;
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
            case 1: return f(std::integral_constant<int, 1>{}, io);
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

SplitShape split_shape(int T, bool dihedral, int Ci, int Co, eql_dtype_t dtype) {
    SplitShape s{};
    s.T = T; s.dihedral = dihedral; s.Ci = Ci; s.Co = Co;
    s.tuple = dihedral ? 2 * T : T;
    s.dtype = dtype;
    const int d = T / 2;
    const bool split = !dihedral && T % 2 == 0 && (d == 1 || d == 2 || d == 4 || d == 8 || d == 16);
    s.S = split ? 2 : 1;
    s.D = split ? d : 0;
    s.half = T / s.S;
    s.reps = s.tuple / s.S;
    const bool f32 = dtype == EQL_FP32;
    auto first_pass = [&](int C) { return (int)align_up((size_t)C * s.reps, 16) * 4; };
    if (f32) { s.kf = first_pass(Ci) * 3 / 2; s.kb = first_pass(Co) * 3 / 2; }
    else s.kf = split ? (int)align_up((size_t)Ci * s.reps, 32) * 2 : (int)align_up((size_t)Ci * s.reps, 8);
    if (!f32) s.kb = split ? (int)align_up((size_t)Co * s.reps, 32) * 2 : (int)align_up((size_t)Co * s.reps, 8);
    s.stash_pitch = (int)align_up((size_t)Ci * s.reps, 8);
    s.wf_bytes = align_up((size_t)Co * s.reps * s.kf * (f32 ? 4 : 2), kWsAlign);
    s.wb_bytes = align_up((size_t)Ci * s.reps * s.kb * (f32 ? 4 : 2), kWsAlign);
    s.bias_bytes = align_up(((size_t)Co * s.reps + 256) * sizeof(float), kWsAlign);
    // The matrices hold reps times the weight's own elements: layers whose matrix would pass 256 MB keep the other
    // kernels, whose operands grow with the weight only.
    // Float: T = 4 and 8, which use 3xTF32 in the other kernels too, up to 768 columns per product (the other kernels' error at
    // 256 channels, see above).  Layers of at most 32 columns are launch latency, of which the other kernels have less (T = 4, 8 -> 8
    // channels, 64 tokens: 6.0 against 6.7 us).
    const bool f32_ok = !dihedral && (T == 4 || T == 8) && (Ci > Co ? Ci : Co) * s.reps <= 768 && (Ci > Co ? Ci : Co) * s.reps > 32;
    s.supported = (!f32 || f32_ok) && s.wf_bytes <= (size_t)256 << 20 && s.wb_bytes <= (size_t)256 << 20;
    return s;
}

cudaError_t launch_split_weights(const SplitShape& s, bool correlation, const void* w, const void* bias, void* wf, void* wb,
                                 float* bias_cols, cudaStream_t stream) {
    WeightParams p{};
    p.Ci = s.Ci; p.Co = s.Co; p.corr = correlation ? 1 : 0;
    p.kf = s.kf; p.kb = s.kb;
    p.first_f = s.kf / 3 * 2; p.first_b = s.kb / 3 * 2;
    cudaError_t err = cudaErrorInvalidValue;
    auto launch = [&](auto r, auto sc, auto io) {
        using R = decltype(r);
        using IO = decltype(io);
        constexpr int S = decltype(sc)::value, CH = weight_block(R::kTuple / S);
        const dim3 grid((s.Ci + CH - 1) / CH, (s.Co + CH - 1) / CH);
        err = launch_overlapped(split_weights_kernel<R, S, IO>, grid, dim3(256), 0, stream, (const IO*)w, (const IO*)bias,
                                (IO*)wf, (IO*)wb, bias_cols, p);
    };
    auto typed = [&](auto r, auto sc) {
        using R = decltype(r);
        if (s.dtype == EQL_FP32) {
            if constexpr (R::kHalf == R::kTuple / 2 && (R::kTuple == 4 || R::kTuple == 8)) launch(r, sc, float{});
        } else if (s.dtype == EQL_BF16) launch(r, sc, __nv_bfloat16{});
        else launch(r, sc, __half{});
    };
    if (s.S == 2) with_reps<2>(s.reps, s.dihedral, [&](auto r) { typed(r, std::integral_constant<int, 2>{}); });
    else with_reps<1>(s.reps, s.dihedral, [&](auto r) { typed(r, std::integral_constant<int, 1>{}); });
    return err;
}

// forward: in = x, matrix = wf, C_in = Ci;  data gradient: in = dy, matrix = wb, C_in = Co
cudaError_t launch_split_linear(const SplitShape& s, bool backward, const void* in, void* out, int64_t N, const void* matrix,
                                const float* bias_cols, int* status, int num_sms, cudaStream_t stream, int act, void* stash) {
    const int Cin = backward ? s.Co : s.Ci, Cout = backward ? s.Ci : s.Co;
    const int in_cols = Cin * s.tuple, out_cols = Cout * s.tuple, K = Cin * s.reps, rows = Cout * s.reps;
    const int pitch = backward ? s.kb : s.kf;
    const int64_t token_tiles = (N + 255) / 256;
    SplitParams p{};
    const bool f32 = s.dtype == EQL_FP32;
    const int elem = f32 ? 4 : 2, kw = f32 ? 16 : s.S == 2 ? 32 : 64;      // K per slot and product (float: of the second pass)
    p.stash = (uint8_t*)stash; p.bias = bias_cols; p.status = status; p.N = N;
    p.out_row = out_cols * elem;
    p.stash_pitch = s.stash_pitch * 2;
    p.nRaw = (K + kw - 1) / kw;
    p.nK = f32 ? 3 * p.nRaw : p.nRaw;
    p.last_ksteps = (K - (p.nRaw - 1) * kw + 32 / elem - 1) / (32 / elem);
    return dispatch_split(s.D, s.dtype, [&](auto dc, auto io) -> cudaError_t {
        constexpr int D = decltype(dc)::value;
        constexpr int S = D == 0 ? 1 : 2;
        using IO = decltype(io);
        static SmemLimitOnce limit[3];
        static std::atomic<int> max_pairs{0};
        auto kernel = split_linear_kernel<D, IO, 0>;
        auto take = [&](auto form) {
            constexpr int threads = split_threads(S, sizeof(IO)), epi = kEpiWarps * 32, ACT = decltype(form)::value;
            kernel = split_linear_kernel<D, IO, ACT>;
            return limit[ACT].ensure(kernel, kSmemMax, threads, sizeof(IO) == 4 ? (threads - epi) * kRestRegs + epi * kEpiRegs : 0);
        };
        if (cudaError_t e = act ? take(std::integral_constant<int, 1>{}) : take(std::integral_constant<int, 0>{}); e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see ptx::grid_dependency_wait
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        constexpr int kASlots = a_slots(sizeof(IO));
        cfg.blockDim = dim3(split_threads(S, sizeof(IO))); cfg.dynamicSmemBytes = kSmemMax; cfg.stream = stream;
        cfg.attrs = attr; cfg.numAttrs = 2;
        int pairs = max_pairs.load(std::memory_order_relaxed);
        if (pairs == 0) {                                        // as many pairs as can be resident at once
            cfg.gridDim = dim3(2 * (num_sms / 2));
            if (cudaError_t e = cudaOccupancyMaxActiveClusters(&pairs, kernel, &cfg); e != cudaSuccess) return e;
            if (pairs <= 0) return cudaErrorInvalidConfiguration;
            if (pairs > num_sms / 2) pairs = num_sms / 2;
            max_pairs.store(pairs, std::memory_order_relaxed);
        }
        p.nb = choose_nb(S, f32, act != 0, rows, p.nK, token_tiles, pairs);
        p.nTiles = (rows + p.nb - 1) / p.nb;
        const int64_t units = token_tiles * p.nTiles;
        if (units > (1 << 30)) return cudaErrorInvalidConfiguration;
        p.num_units = (int)units;
        p.nbuf = 2 * S * p.nb <= 512 ? 2 : 1;
        // The unrolled GELU, where a pair's next unit runs beside it and its main loop hides it.  Half precision, loop / unrolled, us: 16 stages
        // T = 4, 256 -> 256, 32768 tokens 74 / 85, T = 2, 512 -> 512 78 / 86; 20, T = 8, 160 -> 160, 25216 82 / 88; 24, T = 4, 384 -> 256, 32768
        // 97 / 98, T = 2, 768 -> 512 99 / 97; 32, T = 4, 512 -> 256 124 / 119, T = 8, 256 -> 256, 8000 65.4 / 63.5; 48, T = 8, 384 -> 192, 25216
        // 192 / 182; unsplit T = 6, 256 -> 128, 20000 (24) 58.5 / 57.8.  One unit per pair, 197 tokens: T = 8, 192 -> 384 (24) 13.4 / 14.9, 192 ->
        // 768 14.7 / 15.6, 256 -> 512 (32) 16.6 / 17.3.  Float stages wait for the transform, whose issue slots any GELU takes: T = 8, 32 -> 32,
        // 12608 tokens 18.0 / 19.2, 96 -> 96 81.2 / 82.8, T = 4, 256 -> 256, 32768 261 / 266.
        if constexpr (sizeof(IO) == 2) {
            if (act && p.nbuf == 2 && p.nK >= kGeluHidden && p.num_units > pairs)
                if (cudaError_t e = take(std::integral_constant<int, 2>{}); e != cudaSuccess) return e;
        }
        p.sb = (int)(kSmemMax - kFixedSmem - kASlots * kTileA - kEpiWarps * kStageOut) / (p.nb / 2 * 128);
        if (p.sb > kASlots) p.sb = kASlots;
        CUtensorMap min, mw, mout;
        if (!encode_map_2d(&min, in, in_cols, N, in_cols, 128 / elem, 128, elem)) return cudaErrorInvalidValue;
        if (!encode_map_2d(&mw, matrix, S == 2 ? pitch : K, rows, pitch, 128 / elem, p.nb / 2, elem)) return cudaErrorInvalidValue;
        if (!encode_map_2d(&mout, out, out_cols, N, out_cols, 128 / elem, 32, elem)) return cudaErrorInvalidValue;
        if (p.num_units < pairs) pairs = p.num_units;
        p.step_tile = pairs % p.nTiles; p.step_tt = pairs / p.nTiles;
        cfg.gridDim = dim3(2 * pairs);
        return cudaLaunchKernelEx(&cfg, kernel, min, mw, mout, p);
    });
}

}  // namespace eql
