// Weight gradient of the coset-split dense products (16-bit inputs, FP32 accumulation; see split_common.cuh):
//   D+-[(i,h), (o,g)] = sum_n x+-[n, (i,h)] dy+-[n, (o,g)]            two products over all tokens (unsplit: one)
//   dw[o, i, q] = 1/2 sum_h (D+[h, hq] + sgn D-[h, hq]),  dw[o, i, zq] = 1/2 sum_h (D+[h, hq] - sgn D-[h, hq])
// by CTA pairs with tcgen05.mma.cta_group::2.  A pair owns a tile of 256 x nb entries of both products for one range of
// tokens; M and N may be either of x and dy, whichever fills the tiles better.
//
//   16 warps   rows of x and dy (global, 16-byte loads one stage ahead) -> halves in registers -> MN-major operand tiles
//              [64 tokens x 64 columns], 128-byte swizzle: a token's columns stay contiguous, so a row of a tile is one
//              128-byte store row and no transposition happens anywhere; db from the unrounded rows
//   1 thread   TMA: operand tiles that need no arithmetic (unsplit layers: both; halves of x saved by the forward pass)
//   1 thread   tcgen05.mma, K = 16 tokens per step
//   16 warps   (after the loop) accumulators -> shared memory, the sum over h, partial dw
//
// The sum over h happens before anything is written, so the partial sums of a token range are the size of dw.
#include <cuda_fp16.h>

#include <atomic>
#include <cstring>

#include "split_common.cuh"
#include "tensor_map.h"

namespace eql {
namespace {

constexpr int kThreadsSbw = 640;
constexpr int kWarpTma = 0, kWarpMma = 1, kWarpX0 = 4, kXWarps = 16, kXThreads = kXWarps * 32;
constexpr int kMaxStages = 8;
constexpr int kTok = 64;                      // tokens per stage
constexpr int kBlock = kTok * 128;            // one operand block: 64 tokens x 64 columns

struct SbwParams {
    const uint8_t* m_in;         // the side on M: [N, m_row bytes]
    const uint8_t* n_in;
    float* part;                 // [splits][Co][Ci][tuple]
    float* db_part;              // [splits * shares][Co]
    int* status;
    int64_t N, total_stages, stages_per_split;
    int m_row, n_row;            // bytes of a row (raw)
    int wM, wN;                  // valid columns of a CTA's 128 x nb/2 block of each product
    int nb, mTiles, nTiles;
    int m_is_y, shares;          // dy on M; pairs that share a dy tile (each sums db over its share of the stages)
    int stages, stage_bytes;
    int Ci, Co, tuple, corr;
    GroupRep grp;
};

struct SbwBarriers {
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t full_d, mma_done;
    uint32_t tmem_base;
    int abort_flag, go;
    uint8_t tab[256];            // [h][q] -> rep of h q, bit 7: times z
};

// Adds the 16 raw elements of a granule to one sum per group of min(8, D) representatives and their partners.
template <int D, typename IO>
__device__ __forceinline__ void add_granule(const uint4& a, const uint4& b, float (&acc)[D >= 8 ? 1 : 8 / (D ? D : 1)]) {
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
    constexpr bool ANY_TMA = S == 1 || SAVED;
    extern __shared__ uint8_t smem_raw_base[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_base) + 1023) & ~(uintptr_t)1023);
    const int stages = prm.stages, stage_bytes = prm.stage_bytes, nb = prm.nb, nbh = nb / 2;
    SbwBarriers* bar = reinterpret_cast<SbwBarriers*>(smem + stages * stage_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &bar->abort_flag;
    int* status = prm.status;
    const uint32_t rank = ptx::cluster_ctarank();

    if (threadIdx.x == 0) {
        // split: only the leader's "full" is used, by both CTAs' warps and (saved halves) its TMA thread, which announces
        // the bytes of both CTAs.  unsplit: each CTA's own (its db warps wait for it too), and the peer's word to the leader.
        const uint32_t full_count = S == 2 ? 2 * kXWarps + (SAVED ? 1 : 0) : 1 + (rank == 0 ? 1 : 0);
        const uint32_t empty_count = 1 + (S == 1 ? kXWarps : 0);         // unsplit: the warps that sum db read the stage too
        for (int i = 0; i < kMaxStages; ++i) { ptx::mbar_init(&bar->full[i], full_count); ptx::mbar_init(&bar->empty[i], empty_count); }
        ptx::mbar_init(&bar->full_d, 1);
        ptx::mbar_init(&bar->mma_done, 1);
        bar->abort_flag = 0;
        ptx::fence_mbar_init();
        if (ANY_TMA) { ptx::prefetch_tensormap(&tmap_m); ptx::prefetch_tensormap(&tmap_n); }
    }
    for (int e = threadIdx.x; e < prm.grp.reps * prm.grp.reps; e += kThreadsSbw) {
        bool sign;
        const int rep = prm.grp.combine(e / prm.grp.reps, e % prm.grp.reps, true, sign);
        bar->tab[e] = (uint8_t)(rep | (sign ? 0x80 : 0));
    }
    if (warp == kWarpMma) { ptx::tmem_alloc_pair(&bar->tmem_base, 512); ptx::tmem_relinquish_pair(); }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();
    ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bar->tmem_base;
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();

    const int pair = blockIdx.x >> 1;
    const int nt = pair % prm.nTiles, mt = (pair / prm.nTiles) % prm.mTiles, split = pair / (prm.nTiles * prm.mTiles);
    const int64_t stage0 = (int64_t)split * prm.stages_per_split;
    int64_t nst = prm.total_stages - stage0;
    if (nst > prm.stages_per_split) nst = prm.stages_per_split;
    const int m_bytes = 2 * S * kBlock;                          // M operand of a stage; the N operand follows it
    const int m0 = (2 * mt + (int)rank) * prm.wM, n0 = (2 * nt + (int)rank) * prm.wN;   // first columns of this CTA's operands
    const bool m_is_y = prm.m_is_y != 0;
    const int my_share = m_is_y ? nt : mt;
    const uint32_t leader_full = ptx::map_to_cta(ptx::smem_u32(&bar->full[0]), 0u);

    if (warp == kWarpTma) {
        if (ANY_TMA && lane == 0) {
            int st = 0;
            uint32_t ph = 1, issued = 0;
            const bool do_m = S == 1 || !m_is_y, do_n = S == 1 || m_is_y;
            const uint32_t bytes = (do_m ? m_bytes : 0) + (do_n ? (nbh / 64) * S * kBlock : 0);
            for (int64_t q = 0; q < nst; ++q, ++issued) {
                if (!ptx::mbar_wait(&bar->empty[st], ph, abort_flag, status, 501, true, 64)) break;
                uint8_t* dst = smem + st * stage_bytes;
                const int row = (int)((stage0 + q) * kTok);
                if constexpr (S == 2) {
                    if (rank == 0) ptx::mbar_arrive_expect_tx(&bar->full[st], 2 * bytes);
                } else {
                    ptx::mbar_arrive_expect_tx(&bar->full[st], bytes);
                }
                const uint32_t full = S == 2 ? leader_full + st * 8u : ptx::smem_u32(&bar->full[st]);
                if (do_m)
                    for (int b = 0; b < 2; ++b) ptx::tma_load_3d_pair(dst + b * S * kBlock, &tmap_m, m0 + b * 64, row, 0, full);
                if (do_n)
                    for (int b = 0; b < nbh / 64; ++b)
                        ptx::tma_load_3d_pair(dst + m_bytes + b * S * kBlock, &tmap_n, n0 + b * 64, row, 0, full);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
            // the copies issued last must have landed before the CTA may exit: their stages have been released
            const uint32_t lo = issued > (uint32_t)stages ? issued - stages : 0;
            for (uint32_t c = lo; c < issued; ++c)
                ptx::mbar_wait(&bar->empty[c % stages], (c / stages) & 1, abort_flag, status, 511, false);
        }
    } else if (warp == kWarpMma) {
        if (lane == 0 && rank == 0) {
            int st = 0;
            uint32_t ph = 0;
            bool ok = true;
            const uint32_t idesc = ptx::umma_idesc_f16_f32_mn_major(256, nb, H16<IO>::kUmmaFormat);
            for (int64_t q = 0; q < nst; ++q) {
                ok = ptx::mbar_wait(&bar->full[st], ph, abort_flag, status, 502, true, 256);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint64_t a0 = desc_mn_sw128(ptx::smem_u32(smem + st * stage_bytes), S * kBlock);
                const uint64_t b0 = desc_mn_sw128(ptx::smem_u32(smem + st * stage_bytes + m_bytes), S * kBlock);
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int k = 0; k < kTok / 16; ++k)          // 16 tokens = two 8-row groups
                        ptx::umma_f16_pair(tmem_base + (uint32_t)(s * nb), a0 + ((s * kBlock + k * 2048) >> 4),
                                           b0 + ((s * kBlock + k * 2048) >> 4), idesc, (q > 0 || k > 0) ? 1u : 0u);
                ptx::umma_commit_pair_both(&bar->empty[st]);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
            if (ok) ptx::umma_commit_pair_both(&bar->full_d);
            ptx::umma_commit_pair(&bar->mma_done);
            ptx::mbar_wait(&bar->mma_done, 0, abort_flag, status, 513, false);
        } else if (S == 1 && lane == 0) {
            int st = 0;
            uint32_t ph = 0;
            for (int64_t q = 0; q < nst; ++q) {
                if (!ptx::mbar_wait(&bar->full[st], ph, abort_flag, status, 504, true, 256)) break;
                ptx::mbar_arrive_remote(leader_full + st * 8u);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
        }
    } else if (warp >= kWarpX0) {
        const int xt = threadIdx.x - kWarpX0 * 32;               // 0 .. 511
        constexpr int NACC = D == 0 ? 2 : D >= 8 ? 1 : 8 / (D ? D : 1);
        float acc[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0.f;
        bool ok = true;
        int share_at = 0;                                        // stage number modulo shares
        int st = 0;
        uint32_t ph = S == 2 ? 1 : 0;
        if constexpr (S == 2) {
            // M operand: 64 tokens x 16 granules, two per thread (tokens 32 apart); N operand the same, or 64 x 8 and one
            const int mg = xt & 15, mtok = xt >> 4;
            const int ng = nbh == 128 ? mg : xt & 7, ntok = nbh == 128 ? mtok : xt >> 3;
            const int nN = nbh == 128 ? 2 : 1;
            const int mc = m0 * 4 + granule_offset<D>(mg), nc = n0 * 4 + granule_offset<D>(ng);   // byte column of granule word a
            const bool do_m = !SAVED || m_is_y, do_n = !SAVED || !m_is_y;
            const int m_off = (mg >> 3) * 2 * kBlock + mtok * 128 + (((mg & 7) ^ (mtok & 7)) << 4);
            const int n_off = m_bytes + (ng >> 3) * 2 * kBlock + ntok * 128 + (((ng & 7) ^ (ntok & 7)) << 4);
            // (columns past a row's end: some other columns of it; what they give is never stored)
            const int mlast = prm.m_row - 16, nlast = prm.n_row - 16;
            const int mca = mc < mlast ? mc : mlast, mcb = mc + kGranulePartner<D> < mlast ? mc + kGranulePartner<D> : mlast;
            const int nca = nc < nlast ? nc : nlast, ncb = nc + kGranulePartner<D> < nlast ? nc + kGranulePartner<D> : nlast;
            const int64_t end = (stage0 + nst) * kTok < prm.N ? (stage0 + nst) * kTok : prm.N;   // of the token range
            int64_t l0 = stage0 * kTok;                          // first token of the stage being loaded
            uint4 ma[2], mb[2], na[2], nbv[2];
            auto row = [&](int tok) { const int64_t r = l0 + tok; return (size_t)(r < prm.N ? r : prm.N - 1); };
            auto load_m = [&]() {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const uint8_t* p = prm.m_in + row(mtok + 32 * i) * prm.m_row;
                    ma[i] = load_word(p + mca);
                    mb[i] = load_word(p + mcb);
                }
            };
            auto load_n = [&]() {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (i < nN) {
                        const uint8_t* p = prm.n_in + row(ntok + 32 * i) * prm.n_row;
                        na[i] = load_word(p + nca);
                        nbv[i] = load_word(p + ncb);
                    }
                }
            };
            auto put = [&](uint8_t* d, const uint4& a, const uint4& b) {
                uint4 p, m;
                split_granule<D, IO>(a, b, p, m);
                *reinterpret_cast<uint4*>(d) = p;
                *reinterpret_cast<uint4*>(d + kBlock) = m;
            };
            if (do_m) load_m();
            if (do_n) load_n();
            for (int64_t q = 0; q < nst; ++q) {
                ok = ptx::mbar_wait(&bar->empty[st], ph, abort_flag, status, 503, true, 16);
                if (!ok) break;
                uint8_t* dst = smem + st * stage_bytes;
                const bool sum_db = share_at == my_share;
                if (++share_at == prm.shares) share_at = 0;
                if (l0 + kTok > end) {                           // the last stage: tokens past the end count nothing
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const bool mk = l0 + mtok + 32 * i < end, nk = l0 + ntok + 32 * i < end;
                        mask_word(ma[i], mk); mask_word(mb[i], mk);
                        mask_word(na[i], nk); mask_word(nbv[i], nk);
                    }
                }
                l0 += kTok;                                      // (past the range: clamped rows, nobody uses them)
                if (do_m) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) put(dst + m_off + i * 32 * 128, ma[i], mb[i]);
                    if (sum_db && m_is_y) { add_granule<D, IO>(ma[0], mb[0], acc); add_granule<D, IO>(ma[1], mb[1], acc); }
                    load_m();
                }
                if (do_n) {
                    put(dst + n_off, na[0], nbv[0]);
                    if (nN == 2) put(dst + n_off + 32 * 128, na[1], nbv[1]);
                    if (sum_db && !m_is_y) {
                        add_granule<D, IO>(na[0], nbv[0], acc);
                        if (nN == 2) add_granule<D, IO>(na[1], nbv[1], acc);
                    }
                    load_n();
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_remote(leader_full + st * 8u);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
        } else {
            // unsplit: the operands come by TMA; these warps only sum the columns of dy
            const int words = m_is_y ? 64 : nbh / 2;             // 32-bit words (column pairs) of this CTA's dy operand
            const int wd = xt % words, tg = xt / words, tgs = kXThreads / words;
            const int off = (m_is_y ? 0 : m_bytes) + (wd >> 5) * kBlock + (wd & 3) * 4, chunk = (wd & 31) >> 2;
            for (int64_t q = 0; q < nst; ++q) {
                ok = ptx::mbar_wait(&bar->full[st], ph, abort_flag, status, 503, true, 16);
                if (!ok) break;
                if (share_at == my_share) {
                    const uint8_t* src = smem + st * stage_bytes + off;
                    for (int t = tg; t < kTok; t += tgs) {
                        const float2 f = H16<IO>::unpack(*reinterpret_cast<const uint32_t*>(src + t * 128 + ((chunk ^ (t & 7)) << 4)));
                        acc[0] += f.x; acc[1] += f.y;
                    }
                }
                if (++share_at == prm.shares) share_at = 0;
                ptx::fence_proxy_async_smem();                   // these reads before the TMA refill the release allows
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&bar->empty[st]);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
        }
        if (ok && nst > 0) ok = ptx::mbar_wait(&bar->full_d, 0, abort_flag, status, 505, true, 16);
        // all warps go on or none: the barriers below are for all of them (whoever gave up has raised the abort flag)
        x_barrier();
        if (xt == 0) bar->go = *abort_flag == 0 ? 1 : 0;
        x_barrier();
        if (bar->go != 0) {
            ptx::tc_fence_after_sync();
            const int h = prm.grp.reps;
            // ---- db: one row of sums per token group of the threads, added per channel in a fixed order
            {
                float* red = reinterpret_cast<float*>(smem);
                // columns of the dy operand come in groups of GC representatives per accumulator
                constexpr int GC = D == 0 ? 1 : D >= 8 ? 8 : (D ? D : 1);
                int col, grp, groups, valid;
                if constexpr (S == 2) {
                    const int gw = m_is_y || nbh == 128 ? 16 : 8;
                    col = (xt % gw) * 8; grp = xt / gw; groups = kXThreads / gw; valid = gw * 8;
                } else {
                    const int words = m_is_y ? 64 : nbh / 2;
                    col = (xt % words) * 2; grp = xt / words; groups = kXThreads / words; valid = m_is_y ? prm.wM : prm.wN;
                }
#pragma unroll
                for (int i = 0; i < NACC; ++i) red[grp * 129 + col + i * GC] = acc[i];
                x_barrier();
                const int channels = valid / h;
                const int c0 = (m_is_y ? m0 : n0) / h;
                for (int c = xt; c < channels; c += kXThreads) {
                    if (c0 + c >= prm.Co) break;
                    float v = 0.f;
                    for (int g = 0; g < groups; ++g)
                        for (int k = 0; k < h; k += GC) v += red[g * 129 + c * h + k];
                    prm.db_part[(size_t)(split * prm.shares + my_share) * prm.Co + c0 + c] = v;
                }
                x_barrier();
            }
            // ---- dw: 64 (unsplit: nb/2) columns of the accumulators at a time through shared memory
            const int CW = S == 2 ? 64 : nbh, pitch = CW + 1;
            float* buf = reinterpret_cast<float*>(smem);         // [S][128][pitch]
            const int quad = warp & 3, part4 = (warp - kWarpX0) >> 2;
            const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
            const int tM = prm.wM / h;
            float* out = prm.part + (size_t)split * prm.Co * prm.Ci * prm.tuple;
            for (int c0 = 0; c0 < nb; c0 += CW) {
                for (int c = part4 * (CW / 4); c < (part4 + 1) * (CW / 4); c += 16) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        uint32_t v[16];
                        ptx::tmem_ld<16>(lane_base + (uint32_t)(s * nb + c0 + c), v);
                        ptx::tmem_ld_wait();
                        float* b = buf + (s * 128 + quad * 32 + lane) * pitch + c;
#pragma unroll
                        for (int j = 0; j < 16; ++j) b[j] = __uint_as_float(v[j]);
                    }
                }
                x_barrier();
                const int half = c0 / nbh;
                const int ncol = (2 * nt + half) * prm.wN + (c0 - half * nbh);      // first column of this chunk on the N side
                const int tC = (S == 2 ? 64 : prm.wN) / h;
                const int total = tM * tC * h;
                const int mch = m0 / h, nch = ncol / h;          // first channels
                for (int e = xt; e < total; e += kXThreads) {
                    const int q = e % h, r = e / h;
                    const int tm = m_is_y ? r / tC : r % tM, tn = m_is_y ? r % tC : r / tM;
                    const int i = m_is_y ? nch + tn : mch + tm, o = m_is_y ? mch + tm : nch + tn;
                    if (i >= prm.Ci || o >= prm.Co) continue;
                    const float* b = buf + (tm * h) * pitch + tn * h;
                    float cp = 0.f, cm = 0.f;
                    for (int k = 0; k < h; ++k) {
                        const uint8_t t = bar->tab[k * h + q];
                        const int g = t & 0x7F;
                        const int at = m_is_y ? g * pitch + k : k * pitch + g;
                        cp += b[at];
                        if constexpr (S == 2) {
                            const float m = b[128 * pitch + at];
                            cm += (t & 0x80) ? -m : m;
                        }
                    }
                    int p = prm.grp.element(q), pz = p + prm.grp.half;
                    if (prm.corr) { p = (prm.tuple - p) % prm.tuple; pz = (prm.tuple - pz) % prm.tuple; }
                    float* dst = out + ((size_t)o * prm.Ci + i) * prm.tuple;
                    if constexpr (S == 2) {
                        dst[p] = 0.5f * (cp + cm);
                        dst[pz] = 0.5f * (cp - cm);
                    } else {
                        dst[p] = cp;
                    }
                }
                x_barrier();
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();
    ptx::cluster_wait();
    if (warp == kWarpMma) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 512);
    }
}

// dw[e] = sum over token ranges of part[range][e], in their order; db likewise over ranges and shares.
__global__ void __launch_bounds__(256)
split_finalize_kernel(const float* __restrict__ part, const float* __restrict__ db_part, int splits, int db_parts, int64_t nw4,
                      int Co, float* __restrict__ dw, float* __restrict__ db) {
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float4* p = reinterpret_cast<const float4*>(part);
    if (splits > 1 && e < nw4) {
        float4 a = p[e];
#pragma unroll 4
        for (int s = 1; s < splits; ++s) {
            const float4 b = p[(int64_t)s * nw4 + e];
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
        }
        reinterpret_cast<float4*>(dw)[e] = a;
    }
    if (db != nullptr && e < Co) {
        float a = 0.f;
        for (int s = 0; s < db_parts; ++s) a += db_part[(int64_t)s * Co + e];
        db[e] = a;
    }
}

constexpr size_t kSmemMax = 227 * 1024;
constexpr size_t kFixedSmem = 1024 + sizeof(SbwBarriers) + 64;
constexpr int64_t kMaxStagesPerSplit = 512;   // 2048 accumulation steps of 16 tokens: the tensor core adds with truncation

int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }

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

// Tiles and token ranges.  Time of a launch in cycles: rounds of pairs x (stages of a range x max(tensor core, operand
// bytes) per product + the epilogue), plus the finalize kernel's traffic of one partial dw per range.
SplitBwdWeightShape split_bwd_weight_shape(const SplitShape& sp, int64_t N, int num_sms) {
    SplitBwdWeightShape b{};
    const int lcm = sp.reps / gcd(sp.reps, 8) * 8;               // whole channels, and columns that start on 16 bytes
    const int pairs = num_sms / 2;
    b.total_stages = (N + kTok - 1) / kTok;
    double best = 1e30;
    const int cols_x = sp.Ci * sp.reps, cols_y = sp.Co * sp.reps;
    for (int y_on_m = 0; y_on_m < 2; ++y_on_m) {
        for (int nb = 128; nb <= 256; nb += 128) {
            const int wM = 128 / lcm * lcm, wN = nb / 2 / lcm * lcm;
            if (wN == 0) continue;
            const int mc = y_on_m ? cols_y : cols_x, nc = y_on_m ? cols_x : cols_y;
            const int mT = (mc + 2 * wM - 1) / (2 * wM), nT = (nc + 2 * wN - 1) / (2 * wN);
            const int64_t tiles = (int64_t)mT * nT;
            const double stage_c = sp.S * (double)(2 * nb > 256 + nb ? 2 * nb : 256 + nb);
            const int64_t s_min = (b.total_stages + kMaxStagesPerSplit - 1) / kMaxStagesPerSplit;
            auto consider = [&](int64_t s) {
                if (s > b.total_stages) s = b.total_stages;
                if (s < s_min) s = s_min;
                const int64_t per = (b.total_stages + s - 1) / s, used = (b.total_stages + per - 1) / per;
                const double rounds = (double)((tiles * used + pairs - 1) / pairs);
                const double bytes = used > 1 ? 2.0 * (double)used * sp.Co * sp.Ci * sp.tuple * 4 : 0.0;
                const double total = rounds * (per * stage_c + 3000.0 + 12.0 * sp.S * nb) + bytes / 2000.0 + (used > 1 ? 2000.0 : 0.0);
                if (total < best * 0.999) {
                    best = total;
                    b.y_on_m = y_on_m != 0; b.nb = nb; b.wM = wM; b.wN = wN; b.mTiles = mT; b.nTiles = nT;
                    b.splits = (int)used; b.stages_per_split = per;
                }
            };
            // as many ranges as fill one to four rounds of pairs, and halves of those (less to write and add up)
            for (int r = 1; r <= 4; ++r)
                for (int64_t s = r * pairs / tiles; s >= 1; s /= 2) consider(s);
            consider(1);
        }
    }
    b.shares = b.y_on_m ? b.nTiles : b.mTiles;
    const size_t nw = (size_t)sp.Co * sp.Ci * sp.tuple;
    b.scratch_bytes = align_up(((b.splits > 1 ? (size_t)b.splits * nw : 0) + (size_t)b.splits * b.shares * sp.Co) * sizeof(float), kWsAlign);
    b.stash_bytes = align_up((size_t)2 * (N > 0 ? N : 1) * sp.kf * 2, kWsAlign);
    return b;
}

cudaError_t launch_split_bwd_weight(const SplitShape& sp, const SplitBwdWeightShape& b, bool correlation, const void* x, bool x_saved,
                                    const void* dy, float* dw, float* db, int64_t N, float* scratch, int* status, cudaStream_t stream) {
    if (x_saved && sp.S != 2) return cudaErrorInvalidValue;
    SbwParams p{};
    const int xrow = sp.Ci * sp.tuple * 2, yrow = sp.Co * sp.tuple * 2;
    p.m_in = (const uint8_t*)(b.y_on_m ? dy : x); p.n_in = (const uint8_t*)(b.y_on_m ? x : dy);
    p.m_row = b.y_on_m ? yrow : xrow; p.n_row = b.y_on_m ? xrow : yrow;
    const size_t nw = (size_t)sp.Co * sp.Ci * sp.tuple;
    p.part = b.splits > 1 ? scratch : dw;
    p.db_part = b.splits > 1 ? scratch + (size_t)b.splits * nw : scratch;
    p.status = status; p.N = N; p.total_stages = b.total_stages; p.stages_per_split = b.stages_per_split;
    p.wM = b.wM; p.wN = b.wN; p.nb = b.nb; p.mTiles = b.mTiles; p.nTiles = b.nTiles;
    p.m_is_y = b.y_on_m ? 1 : 0; p.shares = b.shares;
    p.Ci = sp.Ci; p.Co = sp.Co; p.tuple = sp.tuple; p.corr = correlation ? 1 : 0;
    p.grp = GroupRep{sp.T, sp.reps, sp.half};
    p.stage_bytes = (2 + b.nb / 128) * sp.S * kBlock;
    p.stages = (int)((kSmemMax - kFixedSmem) / p.stage_bytes);
    if (p.stages > kMaxStages) p.stages = kMaxStages;
    // maps of the sides that come by TMA (the other one is a copy nobody uses)
    CUtensorMap mx, my;
    bool ok = true;
    if (sp.S == 1) {
        ok = encode_map_3d(&mx, x, sp.Ci * sp.tuple, N, 1, sp.Ci * sp.tuple, (int64_t)N * sp.Ci * sp.tuple, 64, kTok, 1, 2) &&
             encode_map_3d(&my, dy, sp.Co * sp.tuple, N, 1, sp.Co * sp.tuple, (int64_t)N * sp.Co * sp.tuple, 64, kTok, 1, 2);
    } else if (x_saved) {
        ok = encode_map_3d(&mx, x, sp.Ci * sp.reps, N, 2, sp.kf, (int64_t)N * sp.kf, 64, kTok, 2, 2);
        my = mx;
    } else {
        std::memset(&mx, 0, sizeof(mx));
        my = mx;
    }
    if (!ok) return cudaErrorInvalidValue;
    const CUtensorMap mm = b.y_on_m ? my : mx, mn = b.y_on_m ? mx : my;
    cudaError_t e = dispatch_split(sp.D, sp.bf16, [&](auto dc, auto io) -> cudaError_t {
        constexpr int D = decltype(dc)::value;
        using IO = decltype(io);
        static SmemLimitOnce limit[2];
        auto kernel = split_bwd_weight_kernel<D, IO, false>;
        if constexpr (D != 0) { if (x_saved) kernel = split_bwd_weight_kernel<D, IO, true>; }
        if (cudaError_t err = limit[x_saved ? 1 : 0].ensure(kernel, kSmemMax); err != cudaSuccess) return err;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see ptx::grid_dependency_wait
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3(2 * b.mTiles * b.nTiles * b.splits);
        cfg.blockDim = dim3(kThreadsSbw); cfg.dynamicSmemBytes = kSmemMax; cfg.stream = stream;
        cfg.attrs = attr; cfg.numAttrs = 2;
        return cudaLaunchKernelEx(&cfg, kernel, mm, mn, p);
    });
    if (e != cudaSuccess) return e;
    const int64_t nw4 = b.splits > 1 ? (int64_t)(nw / 4) : 0;
    const int64_t items = nw4 > sp.Co ? nw4 : sp.Co;
    if (b.splits > 1 || db != nullptr)
        e = launch_overlapped(split_finalize_kernel, dim3((unsigned)((items + 255) / 256)), dim3(256), 0, stream, p.part, p.db_part,
                              b.splits, b.splits * b.shares, nw4, sp.Co, dw, db);
    return e;
}

}  // namespace eql
