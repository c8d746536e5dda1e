// Pair kernel of the workspace mode: two CTAs of a cluster work on ONE output tile of 256 weight
// rows x up to 256 pixels with tcgen05.mma.cta_group::2.
//
// Why: a single CTA reads both MMA operands from its shared memory (12 KB per 128x256x32
// instruction, 96 B/clk at the pipe's full rate) while TMA refills the stages through the same
// 128 B/clk port, so it cannot keep the tensor pipe full.  In a pair each CTA holds its own 128
// weight rows and HALF of the pixels; the hardware feeds both tensor cores from both halves, so
// per instruction a CTA reads 8 KB and receives 8 KB.
//
// Roles per CTA (448 threads): warp 0 lane 0 fetches this CTA's half of the activation codes,
// warp 2 lane 0 its 128 expanded weight rows (both signal the LEADER's "full" barrier, rank 0;
// warps 3 and 4 are second producers taking the odd k-blocks),
// warp 1 of the leader issues the MMAs and commits to both CTAs' barriers, warps 6-13 are the
// epilogue of this CTA's 128 rows (tcgen05.ld, scale, staged bulk stores as in the single-CTA
// kernel).  Accumulators: tensor-memory columns [0, N) and [256, 256 + N), alternating by tile.
// A tile's pixels are two "halves" of up to 128 pixels each (whole images, or whole output rows of
// one image); half h occupies accumulator columns h * nh_pad ...
//
// Every mbarrier wait is bounded; when one runs out the CTA records RMSMP_ERR_TIMEOUT, its roles
// leave their loops and both CTAs still meet at the closing cluster barrier, free tensor memory
// and return.  No load uses cluster multicast.
#include <cuda.h>
#include <cstring>
#include <algorithm>
#include "common.cuh"
#include "ptx.cuh"
#include "tmap.cuh"

namespace rmsmp {

namespace {

constexpr int kThreads2 = 448;
constexpr int kStageA = 128 * 128;               // 16 KB: 128 rows x 128 B
constexpr int kStageB = 128 * 128;               // 16 KB: up to 128 pixels x 128 B
constexpr int kWarpStage2 = 32 * 32 * 4;         // per-warp output staging
constexpr int kEpiWarps2 = 8;
constexpr int kFirstEpi2 = 6;                   // warps 6-13, two per tensor-memory quarter
constexpr int kRing2 = 3;                       // stages; a stage holds TWO k-blocks of each operand (64 KB per CTA)
constexpr int kSub2 = 2;
constexpr int kPairSmem = 232448 - 1024;         // 227 KB per CTA less room for the static variables
constexpr int kPairRest = kEpiWarps2 * kWarpStage2 + 1024 + 64 * 2 * kRing2;      // all but the stages

struct PairCfg {
    int tb, th;              // images / output rows per half
    int npix_h;              // pixels per half
    int nh_pad;              // npix_h rounded up to 8: accumulator columns per half
    int halves_per_image;    // ceil(Ho/th) when tb == 1 and th < Ho, else 0 (the last half of an image ends at row Ho)
    int64_t nhalves;         // halves in the problem
    int64_t ntiles_n;        // pixel tiles = ceil(nhalves / 2)
    int nbt;                 // row-block pairs
    int64_t ntiles;          // ntiles_n * nbt
    int cpt;                 // 128-channel chunks per tap
    int nkb;                 // k-blocks per tile
    int shift;               // 1: column-shift stages (see plan_pair)
    int ring, b_stage;       // stages; bytes of a stage's activation operand
    int img_pix, img_cols;   // pixels stored as one run and the accumulator columns from one run to the next: all of a half,
                             // or (column shift) an image's
    int runs;                // of them in a half
    uint32_t idesc;
    uint32_t tx_b;           // bytes one activation box brings
    int tail_rows;           // img_pix % 32
    uint32_t smem_bytes;
};

struct PairMaps {
    CUtensorMap act[4], wexp, out_full, out_tail;      // act: one map, or one per parity sub-grid (stride 2)
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of `addr` (a shared::cta address of this CTA) in CTA `rank`
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// arrivals on a barrier given by its shared::cluster address (own or peer CTA)
__device__ __forceinline__ void bar_arrive_cluster(uint32_t cbar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cbar) : "memory");
}
// TMA loads of a CTA pair: data into this CTA's shared memory, completion on a barrier that may
// live in the peer CTA (cta_group::2 form; no multicast).
__device__ __forceinline__ void pair_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t cbar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(cbar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void pair_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t cbar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(cbar), "r"(c0), "r"(c1) : "memory");
}
// Arrive (once all MMAs issued so far have finished) on the barrier at this shared-memory offset in BOTH CTAs.
__device__ __forceinline__ void pair_commit(uint32_t bar)
{
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
                 "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}

// First pixel and geometry of half `hf` (global half index): image / row coordinates for the TMA
// box and the index of its first output pixel.
struct HalfPos { int b0, h0; int64_t n0; };
__device__ __forceinline__ HalfPos half_pos(const Problem& p, const PairCfg& cfg, int64_t hf)
{
    HalfPos r;
    if (cfg.halves_per_image) {
        r.b0 = (int)(hf / cfg.halves_per_image);
        r.h0 = min((int)(hf - (int64_t)r.b0 * cfg.halves_per_image) * cfg.th, p.Ho - cfg.th);
        r.n0 = ((int64_t)r.b0 * p.Ho + r.h0) * p.Wo;
    } else {
        r.b0 = (int)(hf * cfg.tb);
        r.h0 = 0;
        r.n0 = hf * (int64_t)cfg.npix_h;
    }
    return r;
}

// kShift: column-shift stages (PairCfg::shift).
template <bool kShift>
__global__ void __launch_bounds__(kThreads2, 1)
pair_kernel(const Problem p, const PairCfg cfg, const __grid_constant__ PairMaps maps)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = smem_base;
    const int ring = kShift ? cfg.ring : kRing2;
    const uint32_t a_stage = kShift ? 3 * kStageA : kSub2 * kStageA, b_stage = kShift ? (uint32_t)cfg.b_stage : kSub2 * kStageB;
    const uint32_t sB = sA + ring * a_stage;
    const uint32_t sOut = sB + ring * b_stage;
    const uint32_t sBar = sOut + kEpiWarps2 * kWarpStage2;
    const uint32_t bar_full = sBar, bar_empty = sBar + 8 * kRing2;
    const uint32_t bar_tfull = sBar + 16 * kRing2, bar_tempty = bar_tfull + 16;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();                 // 0 = leader: owns the "full" and "accumulator free" barriers

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing2; ++s) {               // (a ring has no more stages than that)
            mbar_init(bar_full + 8 * s, 1);       // the leader's activation producer announces all four copies' bytes; leader only
            mbar_init(bar_empty + 8 * s, 1);      // the leader's commit, delivered to both CTAs
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_tfull + 8 * b, 1);                    // the leader's commit, delivered to both CTAs
            mbar_init(bar_tempty + 8 * b, 2 * kEpiWarps2);      // every epilogue warp of both CTAs; used in the leader only
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        // one warp of EACH CTA of the pair takes part in the allocation
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                   // both CTAs' barriers exist before anyone signals the peer
    tc_fence_after();
    // Every role waits for the kernel in front by itself: before its first access to weights, activations or outputs, and before
    // its first wait for another role.  No trigger: see launch_dependent.
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    volatile int* abort_flag = &s_abort;

    const int64_t first = blockIdx.x >> 1, step = gridDim.x >> 1;      // cluster index, clusters in the grid
    const uint32_t lead_full = map_to_rank(bar_full, 0), lead_tempty = map_to_rank(bar_tempty, 0);

    if (kShift && (warp == 0 || (warp >= 2 && warp <= 4))) {
        // ---------------------------------------------------------- producers, column-shift stages
        // A stage is one kernel column j of one channel chunk: warp 0 fetches the th + 2 input rows at that shift, warps 2 to 4
        // the weights of the taps (0, j), (1, j), (2, j).
        if (lane == 0) {
            const int ti = warp - 2;
            tensormap_prefetch(warp == 0 ? &maps.act[0] : &maps.wexp);
            pdl_wait();
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (int64_t tile = first; tile < cfg.ntiles && ok; tile += step) {
                const int64_t nt = tile / cfg.nbt;
                const int blk = (int)(tile - nt * cfg.nbt) * 2 + (int)rank;
                const HalfPos hp = half_pos(p, cfg, 2 * nt + rank);
                int cc = 0, tj = 0;
                for (int st = 0; st < 3 * cfg.cpt; ++st) {
                    if (!mbar_wait(bar_empty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
                    const uint32_t fb = lead_full + 8 * s;
                    if (warp == 0) {
                        if (rank == 0)
                            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                         ::"r"(bar_full + 8 * s), "r"(2u * (cfg.tx_b + 3u * (uint32_t)kStageA)) : "memory");
                        pair_load_4d(sB + s * b_stage, &maps.act[0], fb, cc * 128, tj - 1, hp.h0 - 1, hp.b0);
                    } else {
                        pair_load_2d(sA + s * a_stage + ti * kStageA, &maps.wexp, fb, (3 * ti + tj) * p.Cp + cc * 128, blk * kBlockRows);
                    }
                    if (++s == (uint32_t)ring) { s = 0; ph ^= 1; }
                    if (++tj == 3) { tj = 0; ++cc; }
                }
            }
            if (!ok) {
                for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
            }
        }
    } else if (!kShift && (warp == 0 || warp == 2 || warp == 3 || warp == 4)) {
      if (lane == 0) {
        // ---------------------------------------------------------- producers (both CTAs)
        // One thread can start a bulk tensor copy only every ~300 ns, about the time four MMAs take,
        // so each operand has two producer threads taking alternate stages.
        const bool is_b = (warp == 0 || warp == 3);
        const uint32_t mine = (warp >= 3) ? 1u : 0u;
        pdl_wait();
        uint32_t s = 0, ph = 0, g = 0;
        bool ok = true;
        for (int64_t tile = first; tile < cfg.ntiles && ok; tile += step) {
            const int64_t nt = tile / cfg.nbt;
            const int blk = (int)(tile - nt * cfg.nbt) * 2 + (int)rank;        // this CTA's row block
            const HalfPos hp = half_pos(p, cfg, 2 * nt + rank);               // this CTA's half of the pixels
            int tap = 0, cc = 0, ti = 0, tj = 0;
            for (int kb = 0; kb < cfg.nkb; kb += kSub2, ++g) {
                const int nsub = min(kSub2, cfg.nkb - kb);
                const bool skip = (g & 1u) != mine;
                if (!skip) {
                    if (!mbar_wait(bar_empty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
                    // all copies of this stage (up to two k-blocks of two operands in two CTAs) complete on the leader's barrier
                    if (is_b && rank == 0)
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                     ::"r"(bar_full + 8 * s), "r"(2u * nsub * (cfg.tx_b + (uint32_t)kStageA)) : "memory");
                }
                const uint32_t fb = lead_full + 8 * s;
                for (int u = 0; u < nsub; ++u) {
                    if (!skip) {
                        if (is_b) {
                            const TapBox tb = tap_box(p, hp.h0, ti, tj);
                            pair_load_4d(sB + (s * kSub2 + u) * kStageB, &maps.act[tb.map], fb, cc * 128, tb.x, tb.y, hp.b0);
                        }
                        else pair_load_2d(sA + (s * kSub2 + u) * kStageA, &maps.wexp, fb, tap * p.Cp + cc * 128, blk * kBlockRows);
                    }
                    if (++cc == cfg.cpt) { cc = 0; ++tap; if (++tj == p.kw) { tj = 0; ++ti; } }
                }
                if (++s == kRing2) { s = 0; ph ^= 1; }
            }
        }
        if (!ok) {
            for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
        }
      }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer (leader CTA only)
        if (rank == 0) {
            uint32_t s = 0, ph = 0, it = 0;
            const uint32_t hi = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);     // SBO 1024 B, version 1, 128-byte swizzle
            const uint32_t a_lo0 = ((sA >> 4) & 0x3FFFu) | (1u << 16), b_lo0 = ((sB >> 4) & 0x3FFFu) | (1u << 16);
            const uint32_t a_step = a_stage >> 4, b_step = b_stage >> 4;
            const uint32_t row_step = (uint32_t)(p.W * 128) >> 4;                      // (column shift) a tap's rows lie W pixels further on
            uint32_t a_lo = a_lo0, b_lo = b_lo0;
            pdl_wait();                                                                // (a bounded wait begins when the kernel in front is over)
            for (int64_t tile = first; tile < cfg.ntiles; tile += step, ++it) {
                const uint32_t ab = it & 1;
                if (!mbar_wait_step(bar_tempty + 8 * ab, ((it >> 1) & 1) ^ 1, abort_flag)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + ab * 256;
                bool ok = true;
                for (int kb = 0; kb < cfg.nkb; kb += kShift ? 3 : kSub2) {
                    if (!mbar_wait_step(bar_full + 8 * s, ph, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    if (kShift) {
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const uint32_t a1 = a_lo + i * (kStageA >> 4), b1 = b_lo + i * row_step;
                            mma_i8_pair_step(d_tmem, a1, b1, hi, cfg.idesc, (kb | i) ? 1u : 0u);
                        }
                        pair_commit(bar_empty + 8 * s);
                    } else {
                        mma_i8_pair_step(d_tmem, a_lo, b_lo, hi, cfg.idesc, kb ? 1u : 0u);
                        if (kb + 1 < cfg.nkb) mma_i8_pair_step(d_tmem, a_lo + (kStageA >> 4), b_lo + (kStageB >> 4), hi, cfg.idesc, 1u);
                        pair_commit(bar_empty + 8 * s);
                    }
                    a_lo += a_step;
                    b_lo += b_step;
                    if (++s == (uint32_t)ring) { s = 0; ph ^= 1; a_lo = a_lo0; b_lo = b_lo0; }
                }
                if (!ok) break;
                pair_commit(bar_tfull + 8 * ab);
            }
        }
    } else if (warp >= kFirstEpi2) {
        // ---------------------------------------------------------- epilogue (both CTAs, own 128 rows)
        const int quarter = warp & 3;
        const int first_epi = kFirstEpi2;
        auto count_q = [&](int q) { const int f = first_epi + ((q - first_epi) & 3); return (kThreads2 / 32 - 1 - f) / 4 + 1; };
        const int my_rank = (warp - (first_epi + ((quarter - first_epi) & 3))) >> 2;
        const int cstride = count_q(quarter);
        const uint32_t my_stage = sOut + (uint32_t)(warp - first_epi) * kWarpStage2;
        const int nch = (cfg.img_pix + 31) >> 5;             // 32-pixel chunks per run of pixels
        uint32_t it = 0;
        bool alive = true;
        pdl_wait();
        for (int64_t tile = first; tile < cfg.ntiles && alive; tile += step, ++it) {
            const uint32_t ab = it & 1;
            const int64_t nt = tile / cfg.nbt;
            const int blk = (int)(tile - nt * cfg.nbt) * 2 + (int)rank;
            const int m = blk * kBlockRows + quarter * 32 + lane;
            const float scale = (m < p.M) ? __fmul_rn(__ldg(pdl_ordered(p.wstep) + m), p.act_step) : 0.f;
            int64_t n0h[2];
            int nvalid[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const HalfPos hp = half_pos(p, cfg, 2 * nt + h);
                n0h[h] = hp.n0;
                nvalid[h] = (int)max((int64_t)0, min((int64_t)cfg.npix_h, p.N - hp.n0));
            }
            if (!mbar_wait_warp(bar_tfull + 8 * ab, (it >> 1) & 1, abort_flag)) { alive = false; break; }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + ab * 256;
            const bool rows_ok = blk * kBlockRows + quarter * 32 < p.M;
            // chunk index i = (h * runs + e) * nch + c; this warp takes i = my_rank, my_rank + cstride, ...
            uint32_t v[32];
            const int per_half = kShift ? cfg.runs * nch : nch;
            for (int i = my_rank; i < 2 * per_half; i += cstride) {
                const int h = i >= per_half, u = i - h * per_half, e = kShift ? u / nch : 0, c = u - e * nch;
                const int at = e * cfg.img_pix + c * 32;                 // the chunk's first pixel in its half
                if (!rows_ok || at >= nvalid[h]) continue;
                tmem_ld_issue(taddr + h * cfg.nh_pad + e * cfg.img_cols + c * 32, v);
                tmem_ld_wait(v);
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
                const uint32_t a0 = my_stage + lane * 4;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const uint32_t w = __float_as_uint(__fmul_rn(__int2float_rn((int)v[j]), scale));
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a0 + j * 128), "r"(w) : "memory");
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    const bool tail = cfg.tail_rows && (c == (cfg.img_pix >> 5));
                    tma_store_2d(tail ? &maps.out_tail : &maps.out_full, my_stage, blk * kBlockRows + quarter * 32, (int)(n0h[h] + at));
                }
            }
            // accumulators of this tile are out of tensor memory: tell the leader
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive_cluster(lead_tempty + 8 * ab);
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                   // nobody signals a CTA that has left
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    if (threadIdx.x == 0 && s_abort) atomicMax(p.status, (uint32_t)RMSMP_ERR_TIMEOUT);
}

// ------------------------------------------------------------------ host side

// The pair kernel takes: expanded weights, an even number of row blocks, full 128-channel chunks,
// fp32 [N][M] output through bulk stores, no accumulator dump, no re-quantizing epilogue.
bool plan_pair(const Problem& p, PairCfg& c)
{
    if (!p.wexp || p.acc || p.rq_codes || p.out_mn) return false;
    if (p.nblocks < 2 || (p.nblocks & 1)) return false;
    if (p.Cin % 128 != 0 || p.pix_pitch % 16 != 0) return false;
    if ((reinterpret_cast<uintptr_t>(p.act) & 15) || (reinterpret_cast<uintptr_t>(p.wexp) & 15)) return false;
    if ((p.ld_out % 4) || (p.M % 4) || (reinterpret_cast<uintptr_t>(p.out) & 15)) return false;
    const int64_t hw = (int64_t)p.Ho * p.Wo;
    if (p.Wo > 128 || (int64_t)p.Wo * p.stride > 256) return false;
    if (hw <= 128) {
        c.th = p.Ho;
        c.tb = (int)std::min<int64_t>(128 / hw, p.B);
        // narrower halves where the widest ones leave SMs idle in the last round: a tile takes about a third of its time
        // for the weights and the rest in proportion to its pixels (768x3072 N=4096: 48 tiles for 74 pairs of SMs, or 72
        // with halves of 88 tokens: 14.1 against 12.6 us)
        {
            const int64_t pairs = p.sms / 2;
            auto cost = [&](int tb) {
                const int64_t tiles = (((int64_t)p.B + tb - 1) / tb + 1) / 2 * (p.nblocks / 2);
                return (double)((tiles + pairs - 1) / pairs) * (0.35 + 0.65 * (double)tb * (double)hw / 128.0);
            };
            double best = 0.9 * cost(c.tb);
            const int most = c.tb, step = hw == 1 ? 8 : 1;
            for (int tb = (most - 1) / step * step; tb >= 1 && tb * hw >= 64; tb -= step)
                if (cost(tb) < best) { best = cost(tb); c.tb = tb; }
        }
        c.halves_per_image = 0;
        c.nhalves = (p.B + c.tb - 1) / c.tb;
    } else {
        const int most = std::min(128 / p.Wo, 256 / p.stride);
        c.halves_per_image = (p.Ho + most - 1) / most;
        c.th = (p.Ho + c.halves_per_image - 1) / c.halves_per_image;
        c.tb = 1;
        c.nhalves = (int64_t)p.B * c.halves_per_image;
    }
    if ((int64_t)c.th * p.stride > 256) return false;
    c.npix_h = c.tb * c.th * p.Wo;
    c.cpt = p.Cin / 128;
    c.nkb = p.kh * p.kw * c.cpt;
    c.tx_b = (uint32_t)c.npix_h * 128u;
    c.shift = 0;
    c.ring = kRing2;
    c.b_stage = kSub2 * kStageB;
    c.runs = 1;
    c.img_pix = c.img_cols = c.npix_h;
    // Column-shift stages (3x3, step one): a stage holds, for one kernel column and channel chunk, the th + 2 input rows of the half
    // once and the weights of the three taps of that column, which read it at row offsets of W pixels (of several images, with the
    // staged rows between them as accumulator columns that nobody stores).  Where a pixel then costs fewer rows of copies
    // (weights: 128 rows of nine taps to a half) and two stages fit: 256x256 on 256 images of 14x14 30.6 us without, 29.0 so, 512x512
    // of 7x7 26.9 and 26.0, 256x256 on 64 of 29x29 32.0 and 31.7.
    if (p.kh == 3 && p.kw == 3 && p.stride == 1 && p.pad == 1) {
        const int hw1 = p.Ho * p.Wo, pitch = (c.th + 2) * p.W;           // staged pixels from one image to the next
        const int tb = c.halves_per_image || hw1 > 128 ? 1 : std::min(c.tb, (128 - hw1) / pitch + 1);
        const int rows = tb * pitch, pix = tb * c.th * p.Wo;
        const int64_t stage = 3 * kStageA + ((int64_t)rows * 128 + 1023) / 1024 * 1024;
        const int ring = (int)std::min<int64_t>(kRing2, (kPairSmem - kPairRest) / stage);
        if (ring >= 2 && c.th + 2 <= 256 && (1152.0 + 3 * rows) / pix < (1152.0 + 9 * c.npix_h) / c.npix_h) {
            c.shift = 1;
            c.ring = ring;
            c.b_stage = (int)stage - 3 * kStageA;
            if (tb != c.tb) { c.tb = tb; c.nhalves = (p.B + tb - 1) / tb; }
            c.npix_h = pix;
            c.tx_b = (uint32_t)rows * 128u;
            c.runs = tb;
            c.img_pix = c.th * p.Wo;
            c.img_cols = pitch;
        }
    }
    c.nh_pad = (c.shift ? (c.runs - 1) * c.img_cols + c.img_pix + 7 : c.npix_h + 7) / 8 * 8;
    c.ntiles_n = (c.nhalves + 1) / 2;
    c.nbt = p.nblocks / 2;
    c.ntiles = c.ntiles_n * c.nbt;
    c.tail_rows = c.img_pix & 31;
    // kind::i8, int32 accumulate, signed 8-bit A and B, K-major; N = both halves, M = 256 over the pair
    c.idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * c.nh_pad) >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
    c.smem_bytes = (uint32_t)(c.ring * ((c.shift ? 3 * kStageA : kSub2 * kStageA) + c.b_stage) + kPairRest);
    return true;
}

rmsmp_status launch_planned(const Problem& p, const PairCfg& c, cudaStream_t st)
{
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return RMSMP_ERR_CUDA;
    PairMaps mp;
    memset(&mp, 0, sizeof(mp));
    if (!encode_act_maps_4(p, 128, c.shift ? c.th + 2 : c.th, c.tb, mp.act)) return RMSMP_ERR_CUDA;
    {
        const cuuint64_t gd[2] = {(cuuint64_t)p.Kp, (cuuint64_t)p.M};
        const cuuint64_t gs[1] = {(cuuint64_t)p.Kp};
        const cuuint32_t bx[2] = {128u, (cuuint32_t)kBlockRows};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mp.wexp, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(p.wexp), gd, gs, bx, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return RMSMP_ERR_CUDA;
    }
    auto make_out = [&](CUtensorMap* m, int rows) -> bool {
        const cuuint32_t es[2] = {1, 1};
        const cuuint64_t gs[1] = {(cuuint64_t)p.ld_out * 4};
        const cuuint64_t gd[2] = {(cuuint64_t)p.M, (cuuint64_t)p.N};
        const cuuint32_t bx[2] = {32u, (cuuint32_t)rows};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, p.out, gd, gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (!make_out(&mp.out_full, 32)) return RMSMP_ERR_CUDA;
    if (c.tail_rows && !make_out(&mp.out_tail, c.tail_rows)) return RMSMP_ERR_CUDA;

    void (*const kernel)(const Problem, const PairCfg, const PairMaps) = c.shift ? pair_kernel<true> : pair_kernel<false>;
    static bool attr_set[2][kMaxDevices] = {};
    if (!ensure_smem_attr(reinterpret_cast<const void*>(kernel), kPairSmem, attr_set[c.shift])) return RMSMP_ERR_CUDA;
    const int clusters = (int)std::min<int64_t>(c.ntiles, p.sms / 2);
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    lc.gridDim = dim3((unsigned)(2 * clusters), 1, 1);
    lc.blockDim = dim3(kThreads2, 1, 1);
    lc.dynamicSmemBytes = c.smem_bytes;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // as launch_dependent
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 2;
    if (cudaLaunchKernelEx(&lc, kernel, p, c, mp) != cudaSuccess) {
        cudaGetLastError();
        return RMSMP_ERR_CUDA;
    }
    return RMSMP_OK;
}

}  // namespace

// Worth it when K is long (short reductions are dominated by the pair's start-up and by the
// epilogue: BERT-base FFN1 with 6 k-blocks is 40 % slower this way) and both halves are well filled.
bool launch_pair_if_better(const Problem& p, cudaStream_t st, rmsmp_status* s)
{
    PairCfg c;
    if (!plan_pair(p, c) || c.nkb < 16 || c.npix_h < 64 || !tensor_map_encoder()) return false;
    *s = launch_planned(p, c, st);
    return true;
}

}  // namespace rmsmp
