// Tensor-core contraction for problems that do not fill the chip: few pixels or tokens, a few row blocks, often a
// long reduction (a network's late layers for one image, a small linear layer).  The persistent kernel gives such a
// problem two to sixty tiles, one CTA each, and every CTA walks the whole reduction alone (18 k-blocks: 12 us, 36:
// 16.6 us, with 2 and 4 of 148 SMs busy).  Here the tiles are narrow (128 rows x 16 to 128 pixels) and the reduction
// of a tile is shared by the CTAs of a cluster (1, 2, 4 or 8): each multiplies its k-blocks into its own tensor
// memory, sends every eight columns of its int32 sums to the CTA that owns them through distributed shared memory,
// and the owner adds the parts and writes the output.  Integer sums: the order does not matter.
//
// Warp roles (448 threads): warp 0 fetches the activation boxes (TMA, filter taps as in the persistent kernel); warp 1
// allocates tensor memory and issues the MMAs; warps 2-13 make the A operand -- with a workspace, warp 2 fetches the
// expanded rows by TMA; without one, three groups of four warps take the k-blocks in turn, a thread per row, and
// expand the codes into the swizzled stage -- and are the
// epilogue afterwards, three warps per tensor-memory quarter.  The ring is as deep as the CTA's share of the
// reduction where that fits, so that all copies are in flight at once.
// Activations that the copy engine cannot address (a convolution whose channel count is not a multiple of 16) are
// gathered by the same groups of warps, a thread per pixel: a k-block is then 128 codes of the packed reduction order,
// whichever taps they belong to.  (A MobileNet-v2 block whose first layer is 24 -> 144 channels on 200,704 pixels: 16.5 ms
// with that layer on the CUDA cores, 0.15 ms so.)
// Every mbarrier wait is bounded; when one runs out RMSMP_ERR_TIMEOUT is recorded, the roles leave their loops, and
// the cluster barriers are still met by every thread.  No load uses cluster multicast.
#include <cuda.h>
#include <algorithm>
#include <cstring>
#include "common.cuh"
#include "decode.cuh"
#include "actq.cuh"
#include "ptx.cuh"
#include "tmap.cuh"

namespace rmsmp {

namespace {

constexpr int kSplitThreads = 448;
constexpr int kSplitFirst = 2;                   // first of the twelve working warps
constexpr int kSplitRing = 8;
constexpr int kSplitSmem = 200 * 1024;

struct SplitCfg {
    int tb, th, npix;        // images / output rows / pixels per tile (the last tile of an image or batch may have fewer)
    int n_pad;               // npix rounded up to 16: accumulator columns
    int tiles_per_image;     // > 0: a tile is th rows of one image
    int ntn;                 // pixel tiles
    int cpt, nkb;            // bk-channel chunks per tap, k-blocks
    int last_ksteps;         // 32-code steps in the last chunk of a tap
    int S;                   // CTAs that share a tile's reduction
    int bk, a_bytes, b_bytes, nst;
    int tmem_cols;
    int cpo;                 // groups of eight columns per owner
    int pre;                 // 1: the A operand comes expanded from a workspace
    int gather;              // 1: activations gathered by threads; their loads are this many bytes wide (1, 4 or 8)
    uint32_t idesc, tx_b, smem_bytes;
};

struct SplitMaps { CUtensorMap act[4], wexp; };

__device__ __forceinline__ uint32_t split_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t split_map(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void split_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void split_sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// kRQ: the epilogue writes the next layer's activation codes.  kPre: the A operand comes expanded from a workspace
// (registers for two CTAs per SM, so that the next launch's set-up fits beside this one).  kGather: see the top.
template <int kRQ, int kPre, int kGather>
__global__ void __launch_bounds__(kSplitThreads, kPre || kGather ? 2 : 1)
split_kernel(const Problem p, const SplitCfg cfg, const __grid_constant__ SplitMaps maps)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = smem_base, sB = sA + cfg.nst * cfg.a_bytes;
    const uint32_t sRed = sB + cfg.nst * cfg.b_bytes;            // S > 1: [source CTA][column][128 rows] int32
    __shared__ __align__(8) uint64_t s_full[kSplitRing], s_empty[kSplitRing], s_tfull;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;      // (a shuffle: the same for the warp to the compiler too)
    const uint32_t rank = cfg.S > 1 ? split_rank() : 0u;
    const uint32_t tile = blockIdx.x / (uint32_t)cfg.S;
    const int nt = (int)(tile / (uint32_t)p.nblocks), blk = (int)(tile - (uint32_t)nt * (uint32_t)p.nblocks);
    const int kb0 = (int)rank * cfg.nkb / cfg.S, n_kb = ((int)rank + 1) * cfg.nkb / cfg.S - kb0;      // this CTA's k-blocks

    if (threadIdx.x == 0) {
        for (int s = 0; s < cfg.nst; ++s) {
            mbar_init(smem_u32(&s_full[s]), kPre ? 2 : kGather ? 4 : 5);     // activation producer, and weight producer or the four warps of a group
            mbar_init(smem_u32(&s_empty[s]), 1);
        }
        mbar_init(smem_u32(&s_tfull), 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(cfg.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (cfg.S > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // this CTA runs: its shared memory may be written
    // Every role waits for the kernel in front by itself, behind what it can work out without memory: before its first access to
    // weights, activations or outputs, and before its first wait for another role.
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    volatile int* abort_flag = &s_abort;

    int b0, h0;
    if (cfg.tiles_per_image) { b0 = nt / cfg.tiles_per_image; h0 = (nt - b0 * cfg.tiles_per_image) * cfg.th; }
    else { b0 = nt * cfg.tb; h0 = 0; }
    auto full = [&](int s) { return smem_u32(&s_full[s]); };
    auto empty = [&](int s) { return smem_u32(&s_empty[s]); };

    if ((warp == 0 && !kGather) || (warp == kSplitFirst && kPre)) {
        // ---------------------------------------------------------- TMA producers
        if (lane == 0) {
            if (warp == 0) {
                tensormap_prefetch(&maps.act[0]);
                if (act_parity_split(p)) { tensormap_prefetch(&maps.act[1]); tensormap_prefetch(&maps.act[2]); tensormap_prefetch(&maps.act[3]); }
            } else {
                tensormap_prefetch(&maps.wexp);
            }
            int tap = kb0 / cfg.cpt, cc = kb0 - tap * cfg.cpt;
            int ti = tap / p.kw, tj = tap - ti * p.kw;
            pdl_wait();
            if (warp == 0) pdl_trigger();
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int i = 0; i < n_kb; ++i) {
                if (i >= cfg.nst && !mbar_wait(empty(s), ph ^ 1, abort_flag)) { ok = false; break; }
                if (warp == 0) {
                    mbar_arrive_expect_tx(full(s), cfg.tx_b);
                    const TapBox t = tap_box(p, h0, ti, tj);
                    tma_load_4d(sB + s * cfg.b_bytes, &maps.act[t.map], full(s), cc * cfg.bk, t.x, t.y, b0);
                } else {
                    mbar_arrive_expect_tx(full(s), (uint32_t)cfg.a_bytes);
                    tma_load_2d(sA + s * cfg.a_bytes, &maps.wexp, full(s), tap * p.Cp + cc * cfg.bk, blk * kBlockRows);
                }
                if (++s == cfg.nst) { s = 0; ph ^= 1; }
                if (++cc == cfg.cpt) { cc = 0; ++tap; if (++tj == p.kw) { tj = 0; ++ti; } }
            }
            if (!ok)
                for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer (the warp walks in step, the elected lane issues)
        const uint64_t da = smem_desc_kmajor(sA, cfg.bk), db = smem_desc_kmajor(sB, cfg.bk);
        const uint32_t hi = (uint32_t)(da >> 32), a_step = (uint32_t)cfg.a_bytes >> 4, b_step = (uint32_t)cfg.b_bytes >> 4;
        int s = 0, cc = kb0 % cfg.cpt;
        uint32_t ph = 0;
        bool ok = true;
        pdl_wait();                                       // (a bounded wait begins when the kernel in front is over)
        for (int i = 0; i < n_kb; ++i) {
            if (!mbar_wait_step(full(s), ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const int ksteps = (kGather ? kb0 + i == cfg.nkb - 1 : cc == cfg.cpt - 1) ? cfg.last_ksteps : cfg.bk >> 5;
            const uint32_t a_lo = (uint32_t)da + s * a_step, b_lo = (uint32_t)db + s * b_step;
            mma_i8_steps(ksteps, tmem_base, a_lo, b_lo, hi, cfg.idesc, i ? 1u : 0u);
            mma_commit_step(empty(s));
            if (++s == cfg.nst) { s = 0; ph ^= 1; }
            if (++cc == cfg.cpt) cc = 0;
        }
        if (ok) mma_commit_step(smem_u32(&s_tfull));
    } else if (!kPre && warp >= kSplitFirst) {
        // ---------------------------------------------------------- expanders
        const int grp = (warp - kSplitFirst) >> 2;
        // A thread expands one row, in original order: eight neighbouring lanes store to eight different swizzle phases.
        // (In packed order a warp decodes one kind only, but its lanes' rows collide in the banks; 2 % slower.  Against
        // the workspace form this costs about 2.3 us a launch, the way from the row's place to its first codes to the
        // first stage, and 0.1 to 0.2 us a k-block.)
        const int row = ((warp - kSplitFirst) & 3) * 32 + lane, m_row = blk * kBlockRows + row;
        int kind = -1;
        const uint8_t* src = p.q4;
        pdl_wait();
        if (kGather) pdl_trigger();
        if (m_row < p.M) {
            kind = __ldg(pdl_ordered(p.kind) + m_row);
            const int packed = __ldg(pdl_ordered(p.slot) + m_row);
            src = kind == kFixed8 ? p.q8 + (size_t)(packed - p.nP - p.nF4) * p.Kp : p.q4 + (size_t)packed * (p.Kp >> 1);
        }
        src = pdl_ordered(src);
        const uint32_t swz = cfg.bk == 128 ? (uint32_t)(row & 7) : (uint32_t)((row >> 1) & 3);
        const uint32_t row_off = (uint32_t)row * (uint32_t)cfg.bk;
        // The codes of a k-block are in registers before its turn comes: the next one's are loaded as soon as this one's
        // are expanded, so that the trip to L2 passes during the other groups' turns.
        const bool eight = kind == kFixed8;
        uint4 raw[8];
        auto fetch_pos = [&](int i, int& ksteps) -> const uint4* {
            const int kb = kb0 + i, tap = kGather ? 0 : kb / cfg.cpt, cc = kb - tap * cfg.cpt;
            const int koff = tap * p.Cp + cc * cfg.bk;
            ksteps = i >= n_kb ? 0 : ((kGather ? kb == cfg.nkb - 1 : cc == cfg.cpt - 1) ? cfg.last_ksteps : cfg.bk >> 5);
            return reinterpret_cast<const uint4*>(src + (eight ? koff : koff >> 1));
        };
        auto pieces_of = [&](int ksteps) { return kind < 0 ? 0 : (eight ? 2 * ksteps : ksteps); };      // 16-byte pieces of a row
        // this thread's pixel of the tile (kGather): its image, and the input position of its tap (0, 0)
        int px_y = 0, px_x = 0;
        const int8_t* px_img = pdl_ordered(p.act);
        const bool px_ok = kGather && row < cfg.npix && (int64_t)nt * cfg.npix + row < p.N;
        if (px_ok) {
            const uint32_t n = (uint32_t)((int64_t)nt * cfg.npix + row), t = n / (uint32_t)p.Wo, b = t / (uint32_t)p.Ho;
            px_x = (int)(n - t * (uint32_t)p.Wo) * p.stride - p.pad;
            px_y = (int)(t - b * (uint32_t)p.Ho) * p.stride - p.pad;
            px_img += (int64_t)b * p.H * p.W * p.pix_pitch;
        }
        int ksteps;
        {
            const uint4* q = fetch_pos(grp, ksteps);
            const int pieces = pieces_of(ksteps);
#pragma unroll
            for (int u = 0; u < 8; ++u) raw[u] = u < pieces ? __ldg(q + u) : make_uint4(0u, 0u, 0u, 0u);
        }
        for (int i = grp; i < n_kb; i += 3) {
            const int s = i % cfg.nst;
            int next_ksteps;
            const uint4* q = fetch_pos(i + 3, next_ksteps);
            const int next_pieces = pieces_of(next_ksteps);
            if (i >= cfg.nst && !mbar_wait_warp(empty(s), ((i / cfg.nst) & 1) ^ 1, abort_flag)) break;
            const uint32_t dst = sA + s * cfg.a_bytes + row_off;
            if (kGather) {
                // 32 codes of one tap at a time; a Cp is a multiple of 32, so a step never spans two taps
                const bool b_row = row < cfg.n_pad;                        // (the stage has no more rows than that)
                const uint32_t bdst = sB + s * cfg.b_bytes + (uint32_t)row * 128u;
#pragma unroll 1
                for (int u = 0; u < ksteps; ++u) {
                    const int k = (kb0 + i) * 128 + 32 * u, tap = k / p.Cp, c0 = k - tap * p.Cp;
                    const int ti = tap / p.kw, y = px_y + ti, x = px_x + tap - ti * p.kw;
                    const int n = px_ok && (unsigned)y < (unsigned)p.H && (unsigned)x < (unsigned)p.W ? p.Cin - c0 : 0;      // codes of this tap from c0
                    const int8_t* a = px_img + ((int64_t)y * p.W + x) * p.pix_pitch + c0;
                    uint32_t w[8];
                    if (cfg.gather == 8) {
#pragma unroll
                        for (int q8 = 0; q8 < 4; ++q8) {
                            const uint2 v = 8 * q8 < n ? __ldg(reinterpret_cast<const uint2*>(a) + q8) : make_uint2(0u, 0u);
                            w[2 * q8] = v.x; w[2 * q8 + 1] = v.y;
                        }
                    } else if (cfg.gather == 4) {
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4) w[q4] = 4 * q4 < n ? __ldg(reinterpret_cast<const uint32_t*>(a) + q4) : 0u;
                    } else {
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4) {
                            w[q4] = 0u;
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (4 * q4 + e < n) w[q4] |= (uint32_t)(uint8_t)__ldg(a + 4 * q4 + e) << (8 * e);
                        }
                    }
                    __syncwarp();
                    if (b_row) {
                        split_sts128(bdst + (((uint32_t)(2 * u) ^ (uint32_t)(row & 7)) << 4), w[0], w[1], w[2], w[3]);
                        split_sts128(bdst + (((uint32_t)(2 * u + 1) ^ (uint32_t)(row & 7)) << 4), w[4], w[5], w[6], w[7]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (u < ksteps) {
                    uint32_t w[8];
                    if (kind == kPoT4) {
                        expand_pot_chunk(raw[u], w);
                    } else if (kind == kFixed4) {
                        expand_fixed4_chunk_x16(raw[u], w);
                    } else {
                        w[0] = raw[2 * u].x; w[1] = raw[2 * u].y; w[2] = raw[2 * u].z; w[3] = raw[2 * u].w;
                        w[4] = raw[2 * u + 1].x; w[5] = raw[2 * u + 1].y; w[6] = raw[2 * u + 1].z; w[7] = raw[2 * u + 1].w;
                    }
                    __syncwarp();
                    split_sts128(dst + (((uint32_t)(2 * u) ^ swz) << 4), w[0], w[1], w[2], w[3]);
                    split_sts128(dst + (((uint32_t)(2 * u + 1) ^ swz) << 4), w[4], w[5], w[6], w[7]);
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (u < next_pieces) raw[u] = __ldg(q + u);
            ksteps = next_ksteps;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full(s));
        }
        __syncwarp();
    }

    // -------------------------------------------------------------- epilogue
    const int quarter = warp & 3, rank3 = (warp - kSplitFirst) >> 2;       // tensor-memory lanes; which of the quarter's three warps
    const int m = blk * kBlockRows + quarter * 32 + lane;
    const bool worker = warp >= kSplitFirst, row_ok = worker && m < p.M;
    int64_t n0;
    int nvalid;
    if (cfg.tiles_per_image) {
        n0 = ((int64_t)b0 * p.Ho + h0) * p.Wo;
        nvalid = min(cfg.th, p.Ho - h0) * p.Wo;
    } else {
        n0 = (int64_t)nt * cfg.npix;
        nvalid = (int)min((int64_t)cfg.npix, p.N - n0);
    }
    float scale = 0.0f;
    int shift = 0;
    pdl_wait();
    if (row_ok) {
        scale = __fmul_rn(__ldg(pdl_ordered(p.wstep) + m), p.act_step);
        shift = (!kPre && __ldg(pdl_ordered(p.kind) + m) == kFixed4) ? 4 : 0;         // expanded as 16 * value
    }
    const ActFast rq = act_fast_setup(kRQ ? p.rq_alpha : 1.0f, kRQ ? p.rq_kind : 0);
    const bool out_mn = !kRQ && p.out_mn != 0;
    // the finished sum of this lane's row at column j of the tile
    auto put = [&](int j, int sum) {
        const int a = sum >> shift;
        const float y = __fmul_rn(__int2float_rn(a), scale);
        const int64_t n = n0 + j;
        if (kRQ) {
            p.rq_codes[n * p.ld_codes + m] = (int8_t)act_code_exact(y, p.rq_alpha, p.rq_kind, rq);
        } else {
            const int64_t o = out_mn ? (int64_t)m * p.ld_out + n : n * p.ld_out + m;
            p.out[o] = y;
            if (p.acc) p.acc[o] = a;
        }
    };
    bool alive = true;
    const int groups = (nvalid + 7) >> 3;
    if (worker) {
        alive = mbar_wait_warp(smem_u32(&s_tfull), 0, abort_flag);
        tc_fence_after();
    }
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    if (cfg.S == 1) {
        if (worker && alive && blk * kBlockRows + quarter * 32 < p.M) {
            for (int g = rank3; g < groups; g += 3) {
                uint32_t v[8];
                split_ld8(taddr + 8 * g, v);
                if (out_mn) {
                    // [row][pixel]: a store straight from the lanes' rows would touch 32 sectors for 128 bytes; the group is
                    // turned in shared memory (the stages are free: every multiplication has finished) and leaves as
                    // four rows of 32 bytes a store
                    const int most = min(8, nvalid - 8 * g);
                    for (int sub = 0; sub < (p.acc ? 2 : 1); ++sub) {
                        const uint32_t scratch = sA + (uint32_t)(warp - kSplitFirst) * 1024u;
                        uint32_t w[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int a = (int)v[j] >> shift;
                            w[j] = sub ? (uint32_t)a : __float_as_uint(__fmul_rn(__int2float_rn(a), scale));
                        }
                        split_sts128(scratch + lane * 32, w[0], w[1], w[2], w[3]);
                        split_sts128(scratch + lane * 32 + 16, w[4], w[5], w[6], w[7]);
                        __syncwarp();
                        uint32_t* o = sub ? reinterpret_cast<uint32_t*>(p.acc) : reinterpret_cast<uint32_t*>(p.out);
                        const int row = blk * kBlockRows + quarter * 32 + (lane >> 3);
                        o += (int64_t)row * p.ld_out + n0 + 8 * g + (lane & 7);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            uint32_t x;
                            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(scratch + (uint32_t)(i * 128 + lane * 4)) : "memory");
                            if (row + 4 * i < p.M && (lane & 7) < most) o[(int64_t)(4 * i) * p.ld_out] = x;
                        }
                        __syncwarp();
                    }
                } else if (row_ok) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (8 * g + j < nvalid) put(8 * g + j, (int)v[j]);
                }
                __syncwarp();
            }
        }
    } else {
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");         // every CTA of the cluster runs
        if (worker && alive) {
            for (int g = rank3; g < groups; g += 3) {
                uint32_t v[8];
                split_ld8(taddr + 8 * g, v);
                const uint32_t owner = (uint32_t)(g / cfg.cpo), col = 8u * ((uint32_t)g - owner * (uint32_t)cfg.cpo);
                const uint32_t dst = split_map(sRed + ((rank * 8u * (uint32_t)cfg.cpo + col) * 128u + (uint32_t)(quarter * 32 + lane)) * 4u, owner);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(dst + (uint32_t)j * 512u), "r"(v[j]) : "memory");
            }
        }
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        if (row_ok && alive) {
            const int c0 = (int)rank * 8 * cfg.cpo, c1 = min(c0 + 8 * cfg.cpo, nvalid);
            for (int j = c0 + rank3; j < c1; j += 3) {
                const uint32_t src = sRed + ((uint32_t)(j - c0) * 128u + (uint32_t)(quarter * 32 + lane)) * 4u;
                int sum = 0;
                for (int s = 0; s < cfg.S; ++s) {
                    int v;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(src + (uint32_t)s * (uint32_t)cfg.cpo * 4096u) : "memory");
                    sum += v;
                }
                put(j, sum);
            }
        }
    }

    // -------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cfg.tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && s_abort) atomicMax(p.status, (uint32_t)RMSMP_ERR_TIMEOUT);
}

// ------------------------------------------------------------------ host side

bool split_tile(const Problem& p, int target, SplitCfg& c)
{
    if (c.gather) {                                       // any run of pixels
        const int64_t tiles = (p.N + target - 1) / target;
        if (tiles > (1 << 24)) return false;
        c.tb = c.th = 0;
        c.tiles_per_image = 0;
        c.npix = (int)((p.N + tiles - 1) / tiles);
        c.ntn = (int)((p.N + c.npix - 1) / c.npix);
        c.n_pad = (c.npix + 15) / 16 * 16;
        return true;
    }
    const int64_t hw = (int64_t)p.Ho * p.Wo;
    if (hw <= target) {
        c.tb = (int)std::min<int64_t>(target / hw, p.B);
        const int64_t tiles = ((int64_t)p.B + c.tb - 1) / c.tb;
        if (tiles > (1 << 24)) return false;
        c.tb = (int)((p.B + tiles - 1) / tiles);
        c.th = p.Ho;
        c.tiles_per_image = 0;
        c.ntn = (int)((p.B + c.tb - 1) / c.tb);
    } else {
        if (p.Wo > target) return false;
        c.th = std::min(p.Ho, target / p.Wo);
        const int tiles = (p.Ho + c.th - 1) / c.th;
        c.th = (p.Ho + tiles - 1) / tiles;
        c.tb = 1;
        c.tiles_per_image = (p.Ho + c.th - 1) / c.th;
        if ((int64_t)p.B * c.tiles_per_image > (1 << 24)) return false;
        c.ntn = p.B * c.tiles_per_image;
    }
    if ((int64_t)p.Wo * p.stride > 256 || (int64_t)c.th * p.stride > 256 || c.tb > 256) return false;
    c.npix = c.tb * c.th * p.Wo;
    c.n_pad = (c.npix + 15) / 16 * 16;
    return c.npix <= 128;
}

// Tile width and cluster size by a cost in SM cycles: start-up, the k-blocks of one CTA (rows of up to 128 bytes through
// the SM's copy path, or the expansion of the codes), sending and adding the parts, the output; times the rounds that
// the grid needs.  Against every width and cluster size measured for two dozen problems (256x512 to 4096x4096, 32 to
// 6272 pixels) its choice was within 5 % of the best; where channels are few it is off by more (7x7 step two 240x16 on 4 images of
// 50x50 19.4 us chosen, 17.0 possible).  *us: the time that the cost stands for, as fitted to the same two dozen (a
// workspace: 2.2 us + 1400 units per us; expansion: 1.75 of that - 2 us).  Over 86 convolutions the kernel that it decides for
// takes 1.02 of the better one's time on average, 1.46 at worst.
bool plan_split(const Problem& p, SplitCfg& best, double* us = nullptr, bool gather = false)
{
    if (!gather && (p.pix_pitch % 16 != 0 || (reinterpret_cast<uintptr_t>(p.act) & 15) != 0)) return false;
    if (gather && (p.wexp || p.rq_codes || p.N >= (int64_t)1 << 31)) return false;
    if (p.wexp && (reinterpret_cast<uintptr_t>(p.wexp) & 15) != 0) return false;
    const int64_t sms = p.sms;
    SplitCfg c;
    memset(&c, 0, sizeof(c));
    c.pre = p.wexp ? 1 : 0;
    c.bk = (p.Cin % 128 != 0 && p.Cin % 128 <= 64) ? 64 : 128;
    c.a_bytes = kBlockRows * c.bk;
    c.cpt = (p.Cin + c.bk - 1) / c.bk;
    if ((int64_t)p.kh * p.kw * c.cpt > (1 << 20)) return false;
    c.nkb = p.kh * p.kw * c.cpt;
    c.last_ksteps = (p.Cin - (c.cpt - 1) * c.bk + 31) / 32;
    if (gather) {
        auto fits = [&](int w) { return p.pix_pitch % w == 0 && p.Cin % w == 0 && (reinterpret_cast<uintptr_t>(p.act) & (w - 1)) == 0; };
        c.gather = fits(8) ? 8 : fits(4) ? 4 : 1;
        const int steps = p.kh * p.kw * p.Cp / 32;
        c.bk = 128;
        c.a_bytes = kBlockRows * 128;
        c.cpt = 1;
        c.nkb = (steps + 3) / 4;
        c.last_ksteps = steps - 4 * (c.nkb - 1);
    }
    double best_cost = 1e30;
    static const int targets[] = {16, 32, 48, 64, 96, 128};
    for (int target : targets) {
        if (!split_tile(p, target, c)) continue;
        c.b_bytes = (c.n_pad * c.bk + 1023) / 1024 * 1024;
        c.tx_b = (uint32_t)c.npix * (uint32_t)c.bk;
        for (int S = 1; S <= 8 && S <= c.nkb; S *= 2) {
            const int64_t ctas = (int64_t)p.nblocks * c.ntn * S;
            if (ctas > (1 << 30)) break;
            c.S = S;
            const int kpc = (c.nkb + S - 1) / S;
            c.cpo = S > 1 ? (c.n_pad / 8 + S - 1) / S : 0;
            const int red = S * c.cpo * 8 * 512;
            c.nst = std::min(std::min(kpc, kSplitRing), (kSplitSmem - 2048 - red) / (c.a_bytes + c.b_bytes));
            // fewer than three stages are not enough for the three expander groups: a group may run ahead of the others by
            // two of its own k-blocks, and a stage's barrier tells only neighbouring phases apart
            if (c.nst < 3 && c.nst < kpc) continue;
            c.smem_bytes = (uint32_t)std::max(c.nst * (c.a_bytes + c.b_bytes) + red, (kSplitThreads / 32 - kSplitFirst) * 1024) + 1024;
            // clusters do not tile the SMs of every processing cluster (of 148, 128 CTAs in clusters of four are placed at once but
            // not 136 -- 3x3 48x368 on 17 images of 15x11 17.6 us so, 11.0 in pairs --, 112 in clusters of eight but not 128)
            const double usable = (double)sms * (S == 1 ? 1.0 : S == 2 ? 0.97 : S == 4 ? 0.9 : 0.85);
            const double waves = std::max(1.0, std::ceil((double)ctas / usable));
            const double load = (c.pre ? kBlockRows + c.npix : c.npix) * 2.56, expand = c.pre ? 0.0 : (c.gather ? 900.0 : 420.0) * c.bk / 128.0;
            const double kblock = std::max(std::max(load, expand), 90.0 * (c.bk / 32));
            const double cost = waves * (1500.0 + kpc * kblock + (S > 1 ? 900.0 + 14.0 * c.n_pad : 0.0) + 14.0 * c.n_pad / S);
            if (cost < best_cost) { best_cost = cost; best = c; }
        }
    }
    if (best_cost >= 1e30) return false;
    if (us) {
        *us = 2.2 + best_cost / 1400.0;
        if (!best.pre) *us = (1.75 * *us - 2.0) * ((int64_t)p.nblocks * best.ntn * best.S > sms ? 1.15 : 1.0);
    }
    best.tmem_cols = 32;
    while (best.tmem_cols < best.n_pad) best.tmem_cols *= 2;
    // kind::i8: int32 accumulate, signed 8-bit A and B, both K-major, N/8 at bit 17, M/16 at bit 24
    best.idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(best.n_pad >> 3) << 17) | ((uint32_t)(kBlockRows >> 4) << 24);
    return true;
}

rmsmp_status launch_planned(const Problem& p, const SplitCfg& c, cudaStream_t st, bool gather)
{
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return RMSMP_ERR_CUDA;
    SplitMaps mp;
    memset(&mp, 0, sizeof(mp));
    if (!gather && !encode_act_maps_4(p, c.bk, c.th, c.tb, mp.act)) return RMSMP_ERR_CUDA;
    if (c.pre) {
        const cuuint64_t gd[2] = {(cuuint64_t)p.Kp, (cuuint64_t)p.M};
        const cuuint64_t gs[1] = {(cuuint64_t)p.Kp};
        const cuuint32_t bx[2] = {(cuuint32_t)c.bk, (cuuint32_t)kBlockRows};
        const cuuint32_t es[2] = {1, 1};
        if (enc(&mp.wexp, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(p.wexp), gd, gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                c.bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return RMSMP_ERR_CUDA;
    }
    auto fn = p.rq_codes ? split_kernel<1, 1, 0> : c.pre ? split_kernel<0, 1, 0> : gather ? split_kernel<0, 0, 1> : split_kernel<0, 0, 0>;      // (re-quantizing calls have a workspace)
    if (p.rq_codes && !c.pre) return RMSMP_ERR_VARIANT;
    static bool attr_set[4][kMaxDevices] = {};
    if (!ensure_smem_attr(reinterpret_cast<const void*>(fn), kSplitSmem, attr_set[p.rq_codes ? 2 : gather ? 3 : c.pre])) return RMSMP_ERR_CUDA;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // as launch_dependent
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)c.S; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((int64_t)p.nblocks * c.ntn * c.S)); lc.blockDim = dim3(kSplitThreads);
    lc.dynamicSmemBytes = c.smem_bytes; lc.stream = st; lc.attrs = at; lc.numAttrs = c.S > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&lc, fn, p, c, mp) != cudaSuccess) {
        cudaGetLastError();
        return RMSMP_ERR_CUDA;
    }
    return RMSMP_OK;
}

}  // namespace

// Which of the two kernels takes a problem.  With a workspace the persistent kernel takes whatever fills the chip;
// below that its time is one tile's: 3.4 us + 1.2 for the output of 256 pixels + 0.28 to 0.41 per k-block of 128 codes
// (measured: 256x512 N=64 4.8 us against 4.1 here, 256x2304 N=196 11.7 against 5.4, 512x4608 N=49 16 against 6,
// 768x3072 N=512 13.5 against 10.2, N=2048 13.7 against 14).  Without one it expands the weights first, 1.7 us + 0.7 a
// k-block, if they stay resident (128x512 N=2000 10.6 against 6.5, 1024x512 N=4096 10.9 against 17.4), and otherwise
// again for every tile, 0.59 us a k-block and round of tiles (768x3072 N=1024 21.5 against 14.7, N=4096 22.2 against 37.5;
// 3x3 256x256 on 6272 pixels 17.8 against 15.9, on 12,544 18.2 against 31.5).
bool launch_split_if_better(const Problem& p, cudaStream_t st, rmsmp_status* s)
{
    const double sms = p.sms, tiles = (double)((p.N + 255) / 256 * p.nblocks);
    const bool bk64 = p.Cin % 128 != 0 && p.Cin % 128 <= 64;
    const double nkb = (double)p.kh * p.kw * ((p.Cin + 127) / 128) * (bk64 && p.Cin < 128 ? 0.5 : 1.0);
    double other;
    if (p.wexp || tensor_resident(p)) {
        if (tiles >= sms) return false;
        const int64_t hw = (int64_t)p.Ho * p.Wo;          // (its tiles are whole images: 3x3 256x256 on 32 of 14x14 11.7 us there, 12.5 here)
        const double n = (double)std::min<int64_t>(p.N, hw <= 256 && !bk64 ? 256 / hw * hw : 256);
        other = 3.4 + 1.2 * n / 256 + nkb * (0.28 + 0.13 * n / 256) + (p.wexp ? 0.0 : 1.7 + 0.7 * nkb);
        if (p.out_mn && p.N < 32) other += 1.4;           // (no bulk stores: 64x64 N=8 5.2 us there, 3.3 here)
    } else {
        other = 7.4 + std::ceil(tiles / sms) * (0.8 + 0.59 * nkb);
    }
    SplitCfg c;
    double us = 0.0;
    if (!plan_split(p, c, &us) || us >= other || tensor_map_encoder() == nullptr) return false;
    *s = launch_planned(p, c, st, false);
    return true;
}

// Convolutions whose activations the copy engine cannot address.
rmsmp_status launch_gather(const Problem& p, cudaStream_t st)
{
    SplitCfg c;
    return plan_split(p, c, nullptr, true) ? launch_planned(p, c, st, true) : RMSMP_ERR_VARIANT;
}

}  // namespace rmsmp
