// Coset-split forward / data-gradient kernel on the tensor cores (16-bit I/O, FP32 accumulation): the layer as one or two
// dense products (see split_common.cuh), run by CTA pairs with tcgen05.mma.cta_group::2.
//
//   16 warps     rows of x (global, 16-byte loads two stages ahead) -> x+ and x- in registers (one packed add and one
//                subtract) -> K-major operand tiles [128 tokens x 64], 128-byte swizzle
//   1 thread     TMA: weight tiles [nb/2 rows x 64] of W+ and W- (and, unsplit, the tile of x itself)
//   1 thread     tcgen05.mma M = 256 (two CTAs' tokens), N = nb, into y+ and y- accumulators of nb TMEM columns each
//   4 (12) warps tcgen05.ld, y+ + y- and y+ - y-, bias, optional GELU, one rounding, 32-byte stores (a lane owns a token)
//
// A unit is (256 tokens, nb columns of each product); units are dealt round-robin to the pairs, column tile fastest, so
// the pairs that work on one token tile run together and x comes from DRAM once.
//
// Every wait on an mbarrier is bounded, as in the other tensor-core kernels.
#include <cuda_fp16.h>

#include <atomic>
#include <cstring>

#include "split_common.cuh"
#include "tensor_map.h"

namespace eql {
namespace {

constexpr int kWarpTma = 0, kWarpMma = 1, kWarpEpi0 = 4, kWarpX0 = 8;
constexpr int kXWarps = 16;
constexpr int split_threads(int S) { return S == 2 ? 32 * (kWarpX0 + kXWarps) : 512; }
constexpr int kMaxStages = 8;
constexpr int kTileA = 128 * 128;             // bytes of one operand tile of x: 128 tokens x 64 halves
constexpr uint32_t kSpin = 256;

struct SplitParams {
    const uint8_t* in;           // [N, in_row bytes]
    uint8_t* out;                // [N, out_row bytes]
    uint8_t* stash;              // optional: also write x+ | x- as [2][N][stash_pitch bytes] (weight gradient of the batch)
    const float* bias;           // per output column of one product, or nullptr
    int* status;
    int64_t N;
    int in_row, out_row;         // bytes of a row of x / y
    int stash_pitch;             // bytes of a row of the saved halves
    int nb, nTiles, nK, last_ksteps;      // columns per tile, column tiles, 64-wide K stages, K steps of the last stage
    int nbuf;                    // accumulators in flight
    int sa, sb;                  // slots of the operand rings of x and of the weights
    int64_t num_units;
};

struct SplitBarriers {
    uint64_t full[kMaxStages];   // leader CTA: stage q on full[q % ring] -- both CTAs' operands of the stage
    uint64_t done[kMaxStages];   // both CTAs: the MMAs of stage q have read them
    uint64_t full_d[2], empty_d[2], mma_done;
    uint32_t tmem_base;
    int abort_flag;
    alignas(16) float bias[256];
};

// D: pair distance, 0 = unsplit
template <int D, typename IO, bool ACT>
__global__ void __launch_bounds__(split_threads(D == 0 ? 1 : 2), 1)
split_linear_kernel(const __grid_constant__ CUtensorMap tmap_in, const __grid_constant__ CUtensorMap tmap_w, const SplitParams prm) {
    constexpr int S = D == 0 ? 1 : 2;
    constexpr int NEPI = S == 2 ? 4 : 12;                        // epilogue warps (unsplit: the transform warps' places too)
    extern __shared__ uint8_t smem_raw_base[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_base) + 1023) & ~(uintptr_t)1023);
    const int sa = prm.sa, sb = prm.sb, nb = prm.nb, nK = prm.nK;
    const int ring = sa > sb ? sa : sb;                          // barriers of a stage: one "full" and one "done" for both rings
    uint8_t* aring = smem;
    uint8_t* bring = aring + sa * S * kTileA;
    const int b_bytes = S * (nb / 2) * 128;                      // this CTA's weight rows of a stage
    SplitBarriers* bar = reinterpret_cast<SplitBarriers*>(bring + sb * b_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &bar->abort_flag;
    int* status = prm.status;
    const uint32_t rank = ptx::cluster_ctarank();

    if (threadIdx.x == 0) {
        // "full" (leader): its TMA thread, which announces the bytes of both CTAs, and both CTAs' transform warps
        for (int i = 0; i < kMaxStages; ++i) { ptx::mbar_init(&bar->full[i], 1 + (S == 2 ? 2 * kXWarps : 0)); ptx::mbar_init(&bar->done[i], 1); }
        for (int i = 0; i < 2; ++i) { ptx::mbar_init(&bar->full_d[i], 1); ptx::mbar_init(&bar->empty_d[i], 2 * NEPI); }
        ptx::mbar_init(&bar->mma_done, 1);
        bar->abort_flag = 0;
        ptx::fence_mbar_init();
        if (S == 1) ptx::prefetch_tensormap(&tmap_in);
        ptx::prefetch_tensormap(&tmap_w);
    }
    if (warp == kWarpMma) { ptx::tmem_alloc_pair(&bar->tmem_base, 512); ptx::tmem_relinquish_pair(); }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();                      // the peer's barriers must be initialised before anything arrives on them
    ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bar->tmem_base;
    ptx::grid_dependency_wait();                // nothing above touches global memory that an earlier kernel writes
    ptx::grid_launch_dependents();

    const int64_t first = blockIdx.x >> 1, stride = gridDim.x >> 1;
    const int nTiles = prm.nTiles;
    auto unit_row0 = [&](int64_t u) { return ((u / nTiles) * 2 + rank) * 128; };
    const uint32_t leader_full = ptx::map_to_cta(ptx::smem_u32(&bar->full[0]), 0u);

    // Slot q of a ring may be refilled when the MMAs of stage q - slots are done; that stage's barrier is ring - slots
    // positions ahead of stage q's own, and a parity wait on it is unambiguous: its next phase needs stage q itself.
    if (warp == kWarpTma) {
        // ---------------------------------------------------------------- weight tiles (unsplit: and tiles of x)
        if (lane == 0) {
            RingPos q, d;                                        // stage, and the stage whose completion frees its slot
            int slot = 0;
            uint32_t n = 0;
            bool ok = true;
            const uint32_t bytes = 2u * (uint32_t)(b_bytes + (S == 1 ? kTileA : 0));
            for (int64_t u = first; u < prm.num_units && ok; u += stride) {
                const int wrow = (int)(u % nTiles) * nb + (int)rank * (nb / 2);
                const int row0 = (int)unit_row0(u);
                for (int kc = 0; kc < nK; ++kc, ++n) {
                    if (n >= (uint32_t)sb) {
                        ok = ptx::mbar_wait(&bar->done[d.at], d.phase, abort_flag, status, 401, true, kSpin);
                        if (!ok) break;
                        d.next(ring);
                    }
                    const uint32_t full = leader_full + q.at * 8u;
                    if (rank == 0) ptx::mbar_arrive_expect_tx(&bar->full[q.at], bytes);
                    if constexpr (S == 1) ptx::tma_load_2d_pair(aring + slot * kTileA, &tmap_in, kc * 64, row0, full);
                    ptx::tma_load_3d_pair(bring + slot * b_bytes, &tmap_w, kc * 64, wrow, 0, full);
                    q.next(ring);
                    if (++slot == sb) slot = 0;
                }
            }
            // every copy issued must have landed before the CTA may exit: wait for the stages still in flight
            for (uint32_t c = n > (uint32_t)sb ? n - sb : 0; c < n; ++c) {
                ptx::mbar_wait(&bar->done[d.at], d.phase, abort_flag, status, 411, false);
                d.next(ring);
            }
        }
    } else if (warp == kWarpMma) {
        if (lane == 0 && rank == 0) {
            // ------------------------------------------------------------ tensor-core issue (leader CTA, one thread)
            RingPos q;
            int aslot = 0, bslot = 0;
            uint32_t cu = 0;
            bool ok = true;
            const uint32_t idesc = ptx::umma_idesc_f16_f32(256, nb, H16<IO>::kUmmaFormat);
            const uint64_t a_ring = desc_k_sw128(ptx::smem_u32(aring)), b_ring = desc_k_sw128(ptx::smem_u32(bring));
            const uint64_t b_block = (uint64_t)((nb / 2) * 128) >> 4, b_slot = (uint64_t)b_bytes >> 4;
            for (int64_t u = first; u < prm.num_units && ok; u += stride, ++cu) {
                const uint32_t buf = prm.nbuf == 2 ? (cu & 1) : 0u, use = prm.nbuf == 2 ? (cu >> 1) : cu;
                const uint32_t d0 = tmem_base + buf * (uint32_t)(S * nb);
                ok = ptx::mbar_wait(&bar->empty_d[buf], (use & 1) ^ 1, abort_flag, status, 402, true, kSpin);
                if (!ok) break;
                for (int kc = 0; kc < nK; ++kc) {
                    ok = ptx::mbar_wait(&bar->full[q.at], q.phase, abort_flag, status, 403, true, kSpin);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t a0 = a_ring + (uint64_t)(aslot * S) * (kTileA >> 4), b0 = b_ring + (uint64_t)bslot * b_slot;
                    const int ksteps = kc + 1 < nK ? 4 : prm.last_ksteps;
                    if (ksteps == 4) {
#pragma unroll
                        for (int s = 0; s < S; ++s)
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                ptx::umma_f16_pair(d0 + (uint32_t)(s * nb), a0 + s * (kTileA >> 4) + 2 * k, b0 + s * b_block + 2 * k,
                                                   idesc, (kc | k) ? 1u : 0u);
                    } else {
                        for (int s = 0; s < S; ++s)
                            for (int k = 0; k < ksteps; ++k)
                                ptx::umma_f16_pair(d0 + (uint32_t)(s * nb), a0 + s * (kTileA >> 4) + 2 * k, b0 + s * b_block + 2 * k,
                                                   idesc, (kc | k) ? 1u : 0u);
                    }
                    ptx::umma_commit_pair_both(&bar->done[q.at]);
                    q.next(ring);
                    if (++aslot == sa) aslot = 0;
                    if (++bslot == sb) bslot = 0;
                }
                if (ok) ptx::umma_commit_pair_both(&bar->full_d[buf]);
            }
            ptx::umma_commit_pair(&bar->mma_done);
            ptx::mbar_wait(&bar->mma_done, 0, abort_flag, status, 413, false);
        }
    } else if (S == 2 && warp >= kWarpX0) {
        // ---------------------------------------------------------------- x -> x+, x- operand tiles
        if constexpr (S == 2) {
            // Per stage a thread takes one granule (8 representatives and their partners) of two rows, 4 rows apart; 8
            // lanes cover the 256 bytes of a row, and a warp's 16-byte stores fill whole 128-byte rows of the swizzled tile
            // (no bank conflicts).  Sixteen warps with little each: a warp's chain of loads, adds, stores and the fence
            // takes ~1 K cycles whatever its width, and that has to stay below a stage's MMA time.
            constexpr int PD = 2;                                // stages of loads in flight
            const int g = lane & 7, r0 = (warp - kWarpX0) * 8 + (lane >> 3);
            const int goff = granule_offset<D>(g);
            const int64_t my_units = first < prm.num_units ? (prm.num_units - first + stride - 1) / stride : 0;
            const int64_t total = my_units * nK;                 // stages of this pair
            int64_t lu = first;                                  // position of the loads
            int lc = goff;                                       // byte column of word a
            const int last = prm.in_row - 16;
            const uint8_t* lrow[2];
            auto set_row = [&]() {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int64_t n = unit_row0(lu) + r0 + 4 * i;
                    lrow[i] = prm.in + (size_t)(n < prm.N ? n : prm.N - 1) * prm.in_row;
                }
            };
            if (total > 0) set_row();
            uint4 xa[PD][2], xb[PD][2];
            auto load = [&](uint4 (&a)[2], uint4 (&b)[2]) {
                const int ca = lc < last ? lc : last, cb = lc + kGranulePartner<D> < last ? lc + kGranulePartner<D> : last;
#pragma unroll
                for (int i = 0; i < 2; ++i) { a[i] = load_word(lrow[i] + ca); b[i] = load_word(lrow[i] + cb); }
                lc += 256;
                if (lc - goff >= nK * 256) {
                    lc = goff;
                    lu += stride;
                    if (lu < prm.num_units) set_row();           // (past the last unit: its rows again, nobody uses them)
                }
            };
            RingPos q, d;
            int slot = 0, pk = 0;
            uint32_t n = 0;
            int64_t pu = first, prow = 0;
            bool ok = true, save = false;
            auto set_save = [&]() {
                save = prm.stash != nullptr && pu < prm.num_units && pu % nTiles == 0;   // one column tile saves for all
                if (save) prow = unit_row0(pu) + r0;
            };
            set_save();
            const bool ragged = nK * 256 > prm.in_row;           // the last stage reaches past the row's end
            const int toff = r0 * 128;
            auto process = [&](uint4 (&a)[2], uint4 (&b)[2]) {
                if (n >= (uint32_t)sa) {
                    ok = ptx::mbar_wait(&bar->done[d.at], d.phase, abort_flag, status, 405, true, 16);
                    if (!ok) return;
                    d.next(ring);
                }
                uint8_t* dst = aring + slot * (2 * kTileA) + toff;
                const bool edge = ragged && pk == nK - 1;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (edge) {
                        mask_word(a[i], pk * 256 + goff < prm.in_row);
                        mask_word(b[i], pk * 256 + goff + kGranulePartner<D> < prm.in_row);
                    }
                    uint4 p, m;
                    split_granule<D, IO>(a[i], b[i], p, m);
                    uint8_t* t = dst + i * 512 + ((g ^ ((r0 + 4 * i) & 7)) << 4);
                    *reinterpret_cast<uint4*>(t) = p;
                    *reinterpret_cast<uint4*>(t + kTileA) = m;
                    if (save) {
                        const int64_t nr = prow + 4 * i;
                        const int c = pk * 128 + g * 16;
                        if (nr < prm.N && c < prm.stash_pitch) {
                            uint8_t* s = prm.stash + (size_t)nr * prm.stash_pitch + c;
                            ptx::st_global_v4(s, p.x, p.y, p.z, p.w);
                            ptx::st_global_v4(s + (size_t)prm.N * prm.stash_pitch, m.x, m.y, m.z, m.w);
                        }
                    }
                }
                ptx::fence_proxy_async_smem();                   // generic-proxy writes -> visible to the MMA (async proxy)
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(leader_full + q.at * 8u);
                q.next(ring);
                ++n;
                if (++slot == sa) slot = 0;
                if (++pk == nK) { pk = 0; pu += stride; set_save(); }
            };
            if (total > 0) {
#pragma unroll
                for (int i = 0; i < PD; ++i) load(xa[i], xb[i]);
            }
            for (int64_t t = 0; t < total && ok; t += PD) {
#pragma unroll
                for (int i = 0; i < PD; ++i) {
                    if (ok && t + i < total) process(xa[i], xb[i]);
                    load(xa[i], xb[i]);
                }
            }
        }
    } else if (warp >= kWarpEpi0 && warp < kWarpEpi0 + NEPI) {
        // ---------------------------------------------------------------- epilogue: a lane owns a token
        const int ew = warp - kWarpEpi0, quad = warp & 3, share = ew >> 2;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t empty_leader = ptx::map_to_cta(ptx::smem_u32(&bar->empty_d[0]), 0u);
        constexpr int GC = 32 / S;                               // accumulator columns per 32 elements (64 bytes) of a row
        const bool wide = prm.out_row % 32 == 0 && (reinterpret_cast<uintptr_t>(prm.out) & 31) == 0;   // 32-byte stores
        uint32_t cu = 0;
        int bias_tile = -1;
        for (int64_t u = first; u < prm.num_units; u += stride, ++cu) {
            const uint32_t buf = prm.nbuf == 2 ? (cu & 1) : 0u, use = prm.nbuf == 2 ? (cu >> 1) : cu;
            const int tile = (int)(u % nTiles), col0 = tile * nb;      // first column of the product
            if (prm.bias != nullptr && tile != bias_tile) {      // (columns past the row's end read the padding of the bias array)
                asm volatile("bar.sync 1, %0;" ::"n"(NEPI * 32) : "memory");
                for (int c = ew * 32 + lane; c < nb; c += NEPI * 32) bar->bias[c] = __ldg(prm.bias + col0 + c);
                asm volatile("bar.sync 1, %0;" ::"n"(NEPI * 32) : "memory");
                bias_tile = tile;
            }
            // (the warps meet at the barriers above, so none leaves alone: after a time-out, which every warp sees through the
            // abort flag, they go on without touching the output)
            const bool ok = ptx::mbar_wait(&bar->full_d[buf], use & 1, abort_flag, status, 406, true, 16);
            ptx::tc_fence_after_sync();
            const int64_t row = unit_row0(u) + quad * 32 + lane;
            uint8_t* out_row = prm.out + (size_t)row * prm.out_row;
            const int groups = nb / GC;
            for (int gi = share; gi < groups; gi += NEPI / 4) {
                const uint32_t t0 = lane_base + buf * (uint32_t)(S * nb) + (uint32_t)(gi * GC);
                uint32_t v[32];
                ptx::tmem_ld<16>(t0, v);
                ptx::tmem_ld<16>(t0 + (uint32_t)(S == 2 ? nb : 16), v + 16);
                ptx::tmem_ld_wait();
                if (gi + NEPI / 4 >= groups) {                   // this warp's last read of the accumulator
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive_remote(empty_leader + buf * 8u);
                }
                if (prm.bias != nullptr) {
#pragma unroll
                    for (int j = 0; j < GC; j += 4) {
                        const float4 bv = *reinterpret_cast<const float4*>(&bar->bias[gi * GC + j]);
                        v[j] = __float_as_uint(__uint_as_float(v[j]) + bv.x);
                        v[j + 1] = __float_as_uint(__uint_as_float(v[j + 1]) + bv.y);
                        v[j + 2] = __float_as_uint(__uint_as_float(v[j + 2]) + bv.z);
                        v[j + 3] = __float_as_uint(__uint_as_float(v[j + 3]) + bv.w);
                    }
                }
                if constexpr (S == 2) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float p = __uint_as_float(v[j]), m = __uint_as_float(v[16 + j]);
                        v[j] = __float_as_uint(p + m);
                        v[16 + j] = __float_as_uint(p - m);
                    }
                }
                if constexpr (ACT) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(gelu_erf(__uint_as_float(v[j])));
                }
                // element e of the 32: representative / partner of pair (e / 2D) * D + e % D
                auto elem = [&](int e) {
                    if constexpr (S == 1) return __uint_as_float(v[e]);
                    else return __uint_as_float(v[((e / (D ? D : 1)) & 1) * 16 + (e / (2 * (D ? D : 1))) * D + e % (D ? D : 1)]);
                };
                uint32_t o[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) o[j] = H16<IO>::pack(elem(2 * j), elem(2 * j + 1));
                const int c = (col0 + gi * GC) * S * 2;          // byte column
                if (ok && row < prm.N) {
                    if (wide && c + 64 <= prm.out_row) {
                        ptx::st_global_v8(out_row + c, o);
                        ptx::st_global_v8(out_row + c + 32, o + 8);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (c + 16 * j < prm.out_row)
                                ptx::st_global_v4(out_row + c + 16 * j, o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
                    }
                }
            }
            if (share >= groups) {                               // fewer column groups than shares: nothing to read
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(empty_leader + buf * 8u);
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();                      // neither CTA may leave while the other can still signal it or read its memory
    ptx::cluster_wait();
    if (warp == kWarpMma) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------------
// Weight matrices of the dense products, both K-major, from w[Co][Ci][tuple]:
//   wf[s][(o, g)][(i, h)]  (rows of the forward product's columns)      pitch kf elements
//   wb[s][(i, h)][(o, g)]  (the data gradient's)                        pitch kb elements
// with entry (w[h^-1 g] + sigma_s w[h^-1 z g]) / 2 (unsplit: w[h^-1 g]), rounded once; and the bias expanded to one
// value per column of the forward product.  A block builds OB x IB channel pairs: about 64 x 64 entries, so that both
// matrices are written in 16-byte pieces of contiguous 80..128-byte runs.
struct WeightParams {
    GroupRep grp;
    int Ci, Co, tuple, reps, S, OB, IB;
    int corr;                    // weight index h^-1 g replaced by its inverse
    int kf, kb;                  // pitches (elements): Ci * reps and Co * reps rounded up to 8
};

template <typename IO>
__global__ void __launch_bounds__(256)
split_weights_kernel(const IO* __restrict__ w, const IO* __restrict__ bias, IO* __restrict__ wf, IO* __restrict__ wb,
                     float* __restrict__ bias_cols, const WeightParams prm) {
    extern __shared__ float smem_w[];
    const int reps = prm.reps, S = prm.S, OB = prm.OB, IB = prm.IB, tuple = prm.tuple;
    float* c = smem_w;                                           // [s][o][i][rep]
    const int cs = OB * IB * reps;
    uint8_t* tab = reinterpret_cast<uint8_t*>(c + S * cs);       // [h][g] -> rep of h^-1 g, bit 7: times z
    for (int e = threadIdx.x; e < reps * reps; e += blockDim.x) {
        bool sign;
        const int rep = prm.grp.combine(e / reps, e % reps, false, sign);
        tab[e] = (uint8_t)(rep | (sign ? 0x80 : 0));
    }
    const int o0 = blockIdx.y * OB, i0 = blockIdx.x * IB;
    for (int e = threadIdx.x; e < cs; e += blockDim.x) {
        const int rep = e % reps, i = (e / reps) % IB, o = e / (reps * IB);
        float a = 0.f, b = 0.f;
        if (o0 + o < prm.Co && i0 + i < prm.Ci) {
            const IO* wt = w + ((size_t)(o0 + o) * prm.Ci + i0 + i) * tuple;
            int q = prm.grp.element(rep), qz = S == 2 ? q + prm.grp.half : q;
            if (prm.corr) { q = (tuple - q) % tuple; qz = (tuple - qz) % tuple; }    // cyclic groups only
            a = (float)wt[q];
            if (S == 2) b = (float)wt[qz];
        }
        if (S == 2) { c[e] = 0.5f * (a + b); c[cs + e] = 0.5f * (a - b); }
        else c[e] = a;
    }
    __syncthreads();
    const int rows_f = prm.Co * reps, rows_b = prm.Ci * reps;    // rows of one product's matrix
    auto entry = [&](int s, int o, int i, int h, int g) {
        const uint8_t t = tab[h * reps + g];
        const float x = c[s * cs + (o * IB + i) * reps + (t & 0x7F)];
        return (s == 1 && (t & 0x80)) ? -x : x;
    };
    // forward matrix: rows (o, g), 8 columns (i, h) per thread
    const int fr = OB * reps, fc = IB * reps / 8;
    for (int e = threadIdx.x; e < S * fr * fc; e += blockDim.x) {
        const int ch = e % fc, r = (e / fc) % fr, s = e / (fc * fr);
        const int o = r / reps, g = r % reps;
        const int col = i0 * reps + ch * 8, row = o0 * reps + r;
        if (row >= rows_f || col >= prm.kf) continue;
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = ch * 8 + 2 * j;
            v[j] = H16<IO>::pack(entry(s, o, k / reps, k % reps, g), entry(s, o, (k + 1) / reps, (k + 1) % reps, g));
        }
        *reinterpret_cast<uint4*>(wf + ((size_t)s * rows_f + row) * prm.kf + col) = make_uint4(v[0], v[1], v[2], v[3]);
    }
    // data-gradient matrix: rows (i, h), 8 columns (o, g) per thread
    const int br = IB * reps, bc = OB * reps / 8;
    for (int e = threadIdx.x; e < S * br * bc; e += blockDim.x) {
        const int ch = e % bc, r = (e / bc) % br, s = e / (bc * br);
        const int i = r / reps, h = r % reps;
        const int col = o0 * reps + ch * 8, row = i0 * reps + r;
        if (row >= rows_b || col >= prm.kb) continue;
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = ch * 8 + 2 * j;
            v[j] = H16<IO>::pack(entry(s, k / reps, i, h, k % reps), entry(s, (k + 1) / reps, i, h, (k + 1) % reps));
        }
        *reinterpret_cast<uint4*>(wb + ((size_t)s * rows_b + row) * prm.kb + col) = make_uint4(v[0], v[1], v[2], v[3]);
    }
    if (bias != nullptr && blockIdx.x == 0) {
        for (int r = threadIdx.x; r < fr; r += blockDim.x)
            if (o0 * reps + r < rows_f) bias_cols[o0 * reps + r] = (float)bias[o0 + r / reps];
    }
}

// ------------------------------------------------------------------------------------------------ host side
constexpr size_t kSmemMax = 227 * 1024;
constexpr size_t kFixedSmem = 1024 + sizeof(SplitBarriers) + 64;

// Columns per tile.  A unit's main loop takes, per 64-wide K stage and product, max(tensor core, operand bytes) cycles;
// its epilogue ~8.5 cycles per column and product (stores leave an SM at ~30 B per cycle).  Accumulators of up to 256
// columns in all alternate, so that the epilogue overlaps the next unit's main loop; wider ones do not.  Units go to the
// pairs in whole rounds, which is what decides for small batches.
int choose_nb(int S, int rows, int nK, int64_t token_tiles, int pairs) {
    const int gran = 64 / S;                                     // tiles of whole 128-byte pieces of a row
    double best = 1e30;
    int best_nb = 256;
    for (int tiles = (rows + 255) / 256; tiles <= (rows + gran - 1) / gran; ++tiles) {
        const int nb = ((rows + tiles - 1) / tiles + gran - 1) / gran * gran;
        if (nb > 256) continue;
        const int64_t units = token_tiles * ((rows + nb - 1) / nb);
        const int64_t rounds = (units + pairs - 1) / pairs;
        const double main_c = 600.0 + (double)nK * S * (2 * nb > 256 + nb ? 2 * nb : 256 + nb);
        const double epi_c = 1000.0 + 8.5 * S * nb;
        const double total = 2 * S * nb <= 512 ? rounds * (main_c > epi_c ? main_c : epi_c) + (main_c > epi_c ? epi_c : main_c)
                                               : rounds * (main_c + epi_c);
        if (total < best * 0.999) { best = total; best_nb = nb; }
        if (rounds == 1 && nb <= gran) break;
    }
    return best_nb;
}

template <typename F>
cudaError_t dispatch_split(int D, bool bf16, F&& f) {
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
    return bf16 ? with(__nv_bfloat16{}) : with(__half{});
}

}  // namespace

SplitShape split_shape(int T, bool dihedral, int Ci, int Co, eql_dtype_t dtype) {
    SplitShape s{};
    s.T = T; s.dihedral = dihedral; s.Ci = Ci; s.Co = Co;
    s.tuple = dihedral ? 2 * T : T;
    s.bf16 = dtype == EQL_BF16;
    const int d = T / 2;
    const bool split = T % 2 == 0 && (d == 1 || d == 2 || d == 4 || d == 8 || d == 16);
    s.S = split ? 2 : 1;
    s.D = split ? d : 0;
    s.half = T / s.S;
    s.reps = s.tuple / s.S;
    s.kf = (int)align_up((size_t)Ci * s.reps, 8);
    s.kb = (int)align_up((size_t)Co * s.reps, 8);
    s.wf_bytes = align_up((size_t)s.S * Co * s.reps * s.kf * 2, kWsAlign);
    s.wb_bytes = align_up((size_t)s.S * Ci * s.reps * s.kb * 2, kWsAlign);
    s.bias_bytes = align_up(((size_t)Co * s.reps + 256) * sizeof(float), kWsAlign);
    // The matrices hold reps times the weight's own elements: layers whose matrix would pass 256 MB keep the other
    // kernels, whose operands grow with the weight only.
    s.supported = dtype != EQL_FP32 && s.wf_bytes <= (size_t)256 << 20 && s.wb_bytes <= (size_t)256 << 20;
    return s;
}

cudaError_t launch_split_weights(const SplitShape& s, bool correlation, const void* w, const void* bias, void* wf, void* wb,
                                 float* bias_cols, cudaStream_t stream) {
    WeightParams p{};
    p.grp = GroupRep{s.T, s.reps, s.half};
    p.Ci = s.Ci; p.Co = s.Co; p.tuple = s.tuple; p.reps = s.reps; p.S = s.S; p.corr = correlation ? 1 : 0;
    p.kf = s.kf; p.kb = s.kb;
    int ch = 64 / s.reps;                                        // channels per block side: about 64 entries, rows of whole 16 bytes
    while (ch < 1 || (ch * s.reps) % 8 != 0) ++ch;
    p.OB = p.IB = ch;
    const size_t smem = (size_t)s.S * p.OB * p.IB * s.reps * sizeof(float) + (size_t)s.reps * s.reps;
    const dim3 grid((s.Ci + p.IB - 1) / p.IB, (s.Co + p.OB - 1) / p.OB);
    if (s.bf16)
        split_weights_kernel<__nv_bfloat16><<<grid, 256, smem, stream>>>((const __nv_bfloat16*)w, (const __nv_bfloat16*)bias,
                                                                        (__nv_bfloat16*)wf, (__nv_bfloat16*)wb, bias_cols, p);
    else
        split_weights_kernel<__half><<<grid, 256, smem, stream>>>((const __half*)w, (const __half*)bias, (__half*)wf, (__half*)wb,
                                                                  bias_cols, p);
    return cudaGetLastError();
}

// forward: in = x, matrix = wf [S][Co * reps][kf], C_in = Ci;  data gradient: in = dy, matrix = wb [S][Ci * reps][kb], C_in = Co
cudaError_t launch_split_linear(const SplitShape& s, bool backward, const void* in, void* out, int64_t N, const void* matrix,
                                const float* bias_cols, int* status, int num_sms, cudaStream_t stream, int act, void* stash) {
    const int Cin = backward ? s.Co : s.Ci, Cout = backward ? s.Ci : s.Co;
    const int in_cols = Cin * s.tuple, out_cols = Cout * s.tuple, K = Cin * s.reps, rows = Cout * s.reps;
    const int pitch = backward ? s.kb : s.kf;
    const int64_t token_tiles = (N + 255) / 256;
    SplitParams p{};
    p.in = (const uint8_t*)in; p.out = (uint8_t*)out; p.stash = (uint8_t*)stash; p.bias = bias_cols; p.status = status; p.N = N;
    p.in_row = in_cols * 2; p.out_row = out_cols * 2;
    p.stash_pitch = pitch * 2;
    p.nK = (K + 63) / 64;
    p.last_ksteps = (K - (p.nK - 1) * 64 + 15) / 16;
    return dispatch_split(s.D, s.bf16, [&](auto dc, auto io) -> cudaError_t {
        constexpr int D = decltype(dc)::value;
        constexpr int S = D == 0 ? 1 : 2;
        using IO = decltype(io);
        static SmemLimitOnce limit[2];
        static std::atomic<int> max_pairs{0};
        auto kernel = act ? split_linear_kernel<D, IO, true> : split_linear_kernel<D, IO, false>;
        if (cudaError_t e = limit[act ? 1 : 0].ensure(kernel, kSmemMax); e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see ptx::grid_dependency_wait
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.blockDim = dim3(split_threads(S)); cfg.dynamicSmemBytes = kSmemMax; cfg.stream = stream;
        cfg.attrs = attr; cfg.numAttrs = 2;
        int pairs = max_pairs.load(std::memory_order_relaxed);
        if (pairs == 0) {                                        // as many pairs as can be resident at once
            cfg.gridDim = dim3(2 * (num_sms / 2));
            if (cudaError_t e = cudaOccupancyMaxActiveClusters(&pairs, kernel, &cfg); e != cudaSuccess) return e;
            if (pairs <= 0) return cudaErrorInvalidConfiguration;
            if (pairs > num_sms / 2) pairs = num_sms / 2;
            max_pairs.store(pairs, std::memory_order_relaxed);
        }
        p.nb = choose_nb(S, rows, p.nK, token_tiles, pairs);
        p.nTiles = (rows + p.nb - 1) / p.nb;
        p.num_units = token_tiles * p.nTiles;
        p.nbuf = 2 * S * p.nb <= 512 ? 2 : 1;
        // Rings: x is prefetched in registers as well, so its slots only cover the transform and the MMA (3 will do); a
        // weight slot covers a TMA load, ~2.5 K cycles from release to data under load against ~1 K of MMA per stage.
        const int room = (int)(kSmemMax - kFixedSmem), a_bytes = S * kTileA, b_bytes = S * (p.nb / 2) * 128;
        if (S == 1) {
            p.sa = p.sb = room / (a_bytes + b_bytes) < kMaxStages ? room / (a_bytes + b_bytes) : kMaxStages;
        } else {
            for (p.sa = 5; p.sa > 2; --p.sa) {
                p.sb = (room - p.sa * a_bytes) / b_bytes;
                if (p.sb > kMaxStages) p.sb = kMaxStages;
                if (p.sb > p.sa) break;
            }
        }
        CUtensorMap min, mw;
        if (S == 2) std::memset(&min, 0, sizeof(min));           // (split: x is read with plain loads)
        else if (!encode_map_2d(&min, in, in_cols, N, in_cols, 64, 128, 2)) return cudaErrorInvalidValue;
        if (!encode_map_3d(&mw, matrix, K, rows, S, pitch, (int64_t)rows * pitch, 64, p.nb / 2, S, 2)) return cudaErrorInvalidValue;
        if (p.num_units < pairs) pairs = (int)p.num_units;
        cfg.gridDim = dim3(2 * pairs);
        return cudaLaunchKernelEx(&cfg, kernel, min, mw, p);
    });
}

}  // namespace eql
