// Tensor-core variant of the contraction for sm_100a.
//
// One persistent CTA per SM walks over output tiles of 128 weight rows x up to 256 pixels; the
// reduction is cut into k-blocks of 128 codes.  Warp roles:
//   warp 0      TMA producer.  Per k-block it fetches the activation-code tile (the B operand): one 4-D box into
//               swizzled shared memory -- for a convolution the box is the window of input pixels one filter tap
//               needs, zero fill outside the image being the padding, so no im2col buffer exists anywhere.
//   warp 1      allocates tensor memory and issues tcgen05.mma (kind::i8, int32 accumulators in
//               tensor memory, two 256-column buffers: tile i+1 is computed while tile i is
//               written out).
//   expanders   (weights without a workspace that do not stay resident) groups of four warps that take alternate
//               k-blocks: a thread loads the packed codes of one row of the tile, expands them to int8 in registers and
//               stores them in the K-major swizzled layout the MMA reads (the A operand).  Rows lie in the packed
//               buffer group by group (PoT, Fixed-4, Fixed-8) but are written to the row of their ORIGINAL
//               index, so accumulator lanes are in original row order and the output needs no
//               scatter through the permutation.
//   last four   epilogue, one per tensor-memory quarter (in workspace mode the expander warps
//               have nothing to expand and join the epilogue, about three warps per quarter, five where codes leave; see
//               warps_of): tcgen05.ld (of fp32 outputs the next chunk is in flight while the current one is processed), undo the x16 of
//               Fixed-4 rows, convert, scale by wstep*act_step, stage 32 pixels x 32 rows in buffers of the warp's own and write them
//               with a bulk tensor store (codes: sixteen bytes a store).
// Every wait on an mbarrier is bounded; when one runs out the kernel records
// RMSMP_ERR_TIMEOUT in the packed buffer's status word, all roles leave their loops, tensor
// memory is freed and the kernel returns.
#include <cuda.h>
#include <cstring>
#include "common.cuh"
#include "decode.cuh"
#include "actq.cuh"
#include "ptx.cuh"
#include "tmap.cuh"

namespace rmsmp {

namespace {

constexpr int kTileN = 256;                      // pixels per tile (max) = TMEM columns per buffer
constexpr int kABytes = kBlockRows * 128;        // 16 KB: 128 rows x 128 B (one k-block)
constexpr int kNumEpiWarps = 4;
constexpr int kPreWarps = 2 + 8 + kNumEpiWarps;  // warps of the forms that have no expanders
constexpr int kGroups = 2;                       // expander groups taking alternate k-blocks
constexpr int kNumExpWarps = 4 * kGroups;
// Codes out: a chunk is some 250 instructions, most of them waiting for the one in front, and its bytes are few: many warps, with one
// set of registers each, where nothing else bounds the tile (plan(): tiles of one k-block on resident weights, four rounds of them and
// more: 192x32 on 200,704 pixels 23.8 us with twenty, 24.2 with twelve, 512x64 on 50,000 16.6 and 16.9) or where the codes have to leave one by one
// (332x384 3x3 on 234 images of 7x7 19.0 and 22.8).  Elsewhere warps that wait for a tile are in the way of its copies and products: 128x64 3x3 of
// step two on 256 of 56x56 26.7 with twenty, 23.5 with twelve, 288x288 1x1 of step two on 36 of 72x72 18.4 and 15.8, 64x64 1x1 on 2 of 96x96 4.9 and 4.5;
// through the rings 160x192 3x3 on 64 of 28x28 43.4 with nineteen, 36.7 with eleven, 768x3072 N=4096 13.3 and 11.8, 32x32 7x7 of step two on 145 of
// 11x11 19.5 and 16.1, 64x32 7x7 on 64 of 28x28 41.5 and 42.7.
constexpr int kRqWarps = 22;
__host__ __device__ constexpr int warps_of(int mode, bool many) { return mode ? (many ? kRqWarps : kPreWarps) : 2 + kNumExpWarps + kNumEpiWarps; }
constexpr int kWarpStage = 32 * 32 * 4;          // 4 KB: 32 pixels x 32 rows of fp32/int32
constexpr int kRqStage = 2 * 32 * 32;            // two buffers of 32 pixels x 32 codes
constexpr int kWideEpi = 8;                      // epilogue warps of the form with 144 KB of resident weights (codes out: twice as many)
constexpr int kMaxRing = 8;
constexpr int kResidentBlocks = 16;              // row blocks of a layer with resident weights (the grid is a multiple of them)
constexpr int kSmemLimit = 232448 - 1024;        // 227 KB per CTA less room for the static variables

struct TensorCfg {
    int tb, th;            // images / output rows per tile
    int npix;              // pixels per full tile = tb*th*Wo
    int n_mma;             // npix rounded up to 16
    int tiles_per_image;   // ceil(Ho/th) when tb == 1 and th < Ho, else 0; the last tile of an image ends at row Ho, so that it
                           // may repeat rows of the one before it (the same values to the same places)
    int64_t ntiles_n;
    int64_t ntiles;        // ntiles_n * nblocks
    int cpt;               // 128-channel chunks per tap
    int nkb;               // k-blocks per tile = taps * cpt
    int last_ksteps;       // 32-code steps in the last chunk of a tap
    uint32_t idesc;
    uint32_t tx_bytes;     // bytes one activation box brings
    int a_rows;            // rows of a box of expanded weights: a layer of one row block leaves the rows that it does not have as they are
                           // (nothing reads their sums; zeros from outside the matrix take as long as rows: 10x4096 N=20000 25.2 against 22.2 us)
    uint32_t a_tx;         // bytes of a weight stage's boxes
    int tma_store;         // 1: output chunks leave through shared memory and bulk tensor stores (codes: 16-byte stores)
    int tail_rows;         // npix % 32: height of the last chunk of a tile (0: none)
    int nA, nB;            // ring depths: expanded weights, activations
    int out_bufs;          // staging buffers per epilogue warp (1 or 2)
    int pre;               // 1: the A operand comes expanded (int8) from a workspace, no expander work
    int dup;               // 1 (pre mode, M <= 64, or resident weights whose last row block is at most half full): that block's
                           //    first 64 rows are loaded twice, into lanes 0..63 and 64..127, so that all
                           //    four tensor-memory quarters hold valid rows and every epilogue warp has work
    int cta_full;          // > 0: CTAs of every row block but the last, which gets the rest of the grid (its tiles take less)
    int trigger;           // 1: the grid leaves half of the SMs free, where the next launch's set-up and weights may go ahead (see launch_dependent)
    int epi_warps;         // epilogue warps: 4, or 12 in pre mode (the idle expander warps join)
    int bk;                // codes per k-block and bytes per operand row in shared memory: 128, or 64 (pre mode,
                           //    channel counts that would leave half of a 128-byte row empty)
    int a_bytes, b_bytes;  // one A / B stage
    int fill;              // 1 (resident weights, no workspace given): the CTA expands its row block from the packed codes
                           //    itself, once, instead of copying expanded weights in
    int ares;              // 1 (pre mode, small K): the expanded weights of all k-blocks are loaded once per CTA and stay in
                           //    shared memory; only activation boxes flow through a ring.  The grid is a multiple of the row
                           //    blocks, so that all tiles of a CTA are of one block
    int m2;                // 1 (pre mode, even number of row blocks): a tile covers TWO row blocks.  Both use the same
                           //    activation stage, so a k-block brings 64 KB for eight MMAs instead of 48 KB for four;
                           //    the two accumulators take the two halves of tensor memory
    int nbt;               // row-block groups per pixel tile: nblocks, or nblocks / 2
    int tps;               // k-blocks per activation stage: 1, or 3 (resident weights, 64-byte k-blocks, 3-wide kernels):
                           //    one barrier round trip then covers a whole kernel row instead of a single tap
    int b_sub;             // bytes of one k-block inside an activation stage
    int colshift;          // 1 (with tps == 3; 3x3, stride 1, tiles of whole output rows of one image): an activation
                           //    stage holds the th + 2 input rows the tile needs at ONE column shift j, fetched once; the
                           //    taps (0..2, j) read it at row offsets of W pixels (the swizzle goes by the address: rows may start
                           //    anywhere in its pattern; 3x3 64x48 on 60 images of 51x51 29.0 us without, 19.4 so).  The copy engine
                           //    then moves 3 (th + 2) rows per tile instead of 9 th
    uint32_t smem_bytes;
};

struct Maps {
    CUtensorMap act[4];                                // [B][H][W][Cin] activation codes; stride 2: one map per row/column parity
    CUtensorMap wexp;                                  // [M][Kp] int8 weights expanded beforehand (pre mode); 64-row box when all rows are dup
    CUtensorMap wexp_dup;                              // the same in 64-row boxes, where only the last of several row blocks is dup
    CUtensorMap out_full, out_tail, acc_full, acc_tail;   // bulk stores: 32-row and tail chunks
};

// Resident weights without a workspace: the threads of the CTA expand the row block from the packed codes (exact
// int8 values, as expand_kernel writes them) straight into the resident stages, at the place the bulk copy of an
// expanded [rows][bk] box would have put them: stage kb = (tap, channel chunk) holds codes
// [tap * Cp + chunk * bk, + bk) of every row, 16-byte units XOR-swizzled by the row (128-byte rows: unit ^ (row & 7);
// 64-byte rows: unit ^ ((row >> 1) & 3)), zeros beyond M and Kp; with duplicated rows (M <= 64) a second copy goes to
// lanes 64..127.  Nothing overlaps with it in a CTA's first tile, and it is a chain (slot, codes, expansion): a few
// threads share a row, and a thread has the loads of four pieces of 32 codes in flight at a time (512x512 N=4096, all in one tile per
// CTA: 14.7 us with a load at a time and half of each piece kept, 10.8 so; 128x512 N=2000 10.6).
__device__ __forceinline__ void fill_resident_weights(const Problem& p, const TensorCfg& cfg, uint32_t sA, int row_first, bool dup, int tid, int nthreads)
{
    const int rows = dup ? kBlockRows / 2 : kBlockRows;
    const int pshift = cfg.bk == 128 ? 2 : 1;            // 32-code pieces of a row and k-block: 4 or 2
    const int n4 = p.nP + p.nF4;
    const int tpr = nthreads / rows;
    const int r = tid / tpr, sub = tid - r * tpr;
    if (r < rows) {
        const int m = row_first + r;
        const bool have = m < p.M;
        const int kind = have ? (int)__ldg(pdl_ordered(p.kind) + m) : kFixed8;
        const int slot = have ? __ldg(pdl_ordered(p.slot) + m) : 0;
        const uint8_t* src = (kind == kFixed8) ? p.q8 + (size_t)(have ? slot - n4 : 0) * p.Kp : p.q4 + (size_t)slot * (p.Kp >> 1);
        src = pdl_ordered(src);
        const uint32_t phase = (cfg.bk == 128) ? (uint32_t)(r & 7) : (uint32_t)((r >> 1) & 3);
        const uint32_t row_base = sA + (uint32_t)r * (uint32_t)cfg.bk;
        const int pieces = cfg.nkb << pshift;
        auto code_of = [&](int i) {                      // first code of piece i in the packed row
            const int kb = i >> pshift;
            const int tap = cfg.cpt == 1 ? kb : kb / cfg.cpt;
            return tap * p.Cp + (kb - tap * cfg.cpt) * cfg.bk + 32 * (i - (kb << pshift));
        };
        for (int base = sub; base < pieces; base += 4 * tpr) {
            uint4 raw[4], raw2[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + u * tpr;
                raw[u] = raw2[u] = make_uint4(0u, 0u, 0u, 0u);
                if (have && i < pieces) {
                    const int k = code_of(i);
                    if (k < p.Kp) {
                        raw[u] = __ldg(reinterpret_cast<const uint4*>(src + (kind == kFixed8 ? k : k >> 1)));
                        if (kind == kFixed8) raw2[u] = __ldg(reinterpret_cast<const uint4*>(src + k + 16));
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + u * tpr;
                if (i >= pieces) continue;
                uint32_t w[8] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w, raw2[u].x, raw2[u].y, raw2[u].z, raw2[u].w};
                if (kind == kPoT4) {
                    expand_pot_chunk(raw[u], w);
                } else if (kind == kFixed4) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {        // nibbles to bytes; a set sign bit adds the 0xF0 above it
                        const uint32_t hi = (w[j] >> 4) & 0x0F0F0F0Fu, lo = w[j] & 0x0F0F0F0Fu;
                        w[j] = hi + (hi & 0x08080808u) * 0x1Eu;
                        w[j + 4] = lo + (lo & 0x08080808u) * 0x1Eu;
                    }
                }
                const int kb = i >> pshift;
                const uint32_t unit = (uint32_t)(i - (kb << pshift)) * 2u;
                const uint32_t dst = row_base + (uint32_t)kb * (uint32_t)cfg.a_bytes;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t at = dst + (((unit + (uint32_t)h) ^ phase) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(w[4 * h]), "r"(w[4 * h + 1]), "r"(w[4 * h + 2]), "r"(w[4 * h + 3]));
                    if (dup)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + (uint32_t)(cfg.a_bytes / 2)), "r"(w[4 * h]), "r"(w[4 * h + 1]), "r"(w[4 * h + 2]), "r"(w[4 * h + 3]));
                }
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the MMAs read these bytes through the async proxy
}

// ------------------------------------------------------------------ re-quantizing epilogue

constexpr float kRqMagic = 12582912.0f;          // 1.5 * 2^23: adding it rounds to an integer, half to even

// Two fp32 values per instruction.
__device__ __forceinline__ uint64_t f32x2(float a, float b)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void f32x2_split(uint64_t d, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d)); }
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// Four accumulator columns of the warp's 32 lanes.
__device__ __forceinline__ void tmem_ld_four(uint32_t taddr, uint32_t (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
}

// ------------------------------------------------------------------ the kernel

// kM2: a tile covers two row blocks (TensorCfg::m2), compiled separately so that the common form keeps its registers.
// kRQ: the epilogue writes the next layer's activation codes instead of fp32 (Problem::rq_codes).
// kMode: which of the kernel's forms this instantiation is (the host picks it from the plan): 0 codes expanded in
//        shared memory; 1 expanded weights from a workspace through the ring; 2 the same, weights resident in
//        shared memory; 3 resident weights and three taps per activation stage.  A compile-time constant so that
//        an instantiation carries only the code of its own form.
// kOut:  1 when the output is fp32 [N][M] through bulk stores without an accumulator dump (the common case), or codes through the
//        rings by 16-byte stores: the epilogue then carries only that path; 0 decides at run time.
template <int kM2, int kRQ, int kMode, int kOut>
__global__ void __launch_bounds__(32 * warps_of(kMode, kRQ && !kOut), 1)
tensor_kernel(const Problem p, const TensorCfg cfg, const __grid_constant__ Maps maps)
{
    constexpr int kThreads = 32 * warps_of(kMode, kRQ && !kOut);
    constexpr bool kPre = kMode != 0, kAres = kMode >= 2, kTps3 = kMode == 3;
    const bool use_tma_store = kOut ? true : (cfg.tma_store != 0);
    const bool out_mn = kOut ? false : (p.out_mn != 0);
    int32_t* const acc_out = kOut ? nullptr : p.acc;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = smem_base;
    const uint32_t sB = sA + cfg.nA * cfg.a_bytes;
    const uint32_t sOut = sB + cfg.nB * cfg.b_bytes;
    const uint32_t sBar = sOut + cfg.epi_warps * cfg.out_bufs * (kRQ ? kRqStage : kWarpStage);
    // barriers, 8 bytes each
    const uint32_t bar_fullA = sBar, bar_emptyA = sBar + 8 * kMaxRing;
    const uint32_t bar_fullB = sBar + 16 * kMaxRing, bar_emptyB = sBar + 24 * kMaxRing;
    const uint32_t bar_tfull = sBar + 32 * kMaxRing, bar_tempty = bar_tfull + 16;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;      // (a shuffle: the same for the warp to the compiler too)

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxRing; ++s) {
            mbar_init(bar_fullA + 8 * s, kPre ? 1 : 4);   // producer (+ bytes), or the four warps of one expander group
            mbar_init(bar_emptyA + 8 * s, 1);    // tcgen05.commit
            mbar_init(bar_fullB + 8 * s, 1);     // producer (+ transaction bytes)
            mbar_init(bar_emptyB + 8 * s, 1);    // tcgen05.commit
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_tfull + 8 * b, 1);                  // tcgen05.commit
            mbar_init(bar_tempty + 8 * b, cfg.epi_warps);     // one arrival per epilogue warp
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Every role waits for the kernel in front by itself, behind what it can work out without memory: before its first access to
    // weights, activations or outputs, and before its first wait for another role.
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    volatile int* abort_flag = &s_abort;

    // (tile indices fit 32 bits with a step to spare: checked on the host)
    const uint32_t ntiles = (uint32_t)cfg.ntiles;
    uint32_t first = blockIdx.x, step = gridDim.x;
    if (kAres && cfg.cta_full) {
        // (see TensorCfg::cta_full) the CTA's row block, and its place among that block's CTAs
        const uint32_t rest = (uint32_t)cfg.nbt - 1u, full = (uint32_t)cfg.cta_full * rest;
        const bool last = blockIdx.x >= full;
        const uint32_t mine = last ? rest : blockIdx.x % rest, at = last ? blockIdx.x - full : blockIdx.x / rest;
        first = at * (uint32_t)cfg.nbt + mine;
        step = (last ? gridDim.x - full : (uint32_t)cfg.cta_full) * (uint32_t)cfg.nbt;
    }
    const int my_blk = kAres ? (int)(first % (uint32_t)cfg.nbt) : 0;
    const bool dup = cfg.dup && (!kAres || my_blk == cfg.nbt - 1);
    const int64_t my_tiles = (ntiles > first) ? (ntiles - first + step - 1) / step : 0;

    if (kAres && cfg.fill && warp != 0) {
        pdl_wait();
        // every warp but the activation producer's (whose first copies go out meanwhile) expands the row block;
        // one of them then reports the resident weights to the MMA thread
        if (my_tiles > 0) fill_resident_weights(p, cfg, sA, my_blk * kBlockRows, dup, (int)threadIdx.x - 32, kThreads - 32);
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads - 32) : "memory");
        if (threadIdx.x == 32 && my_tiles > 0) mbar_arrive(bar_fullA);
    }

    // Workspace mode splits the producer: one thread can start a bulk tensor copy only every few
    // hundred cycles, so the activation boxes and the weight boxes are issued by two different warps.
    const bool pre_b_producer = warp == 0;
    const bool pre_a_producer = kPre && !kAres && warp == 2;
    if (pre_b_producer || pre_a_producer) {
        if (lane == 0) {
            if (pre_b_producer) tensormap_prefetch(&maps.act[0]);
            if (kPre && !cfg.fill && (kAres || pre_a_producer)) tensormap_prefetch(kAres && dup && cfg.nbt > 1 ? &maps.wexp_dup : &maps.wexp);
            pdl_wait();
            if (pre_b_producer && cfg.trigger) pdl_trigger();
            if (pre_b_producer && kAres && my_tiles > 0 && !cfg.fill) {
                // resident weights: every k-block's rows, once
                mbar_arrive_expect_tx(bar_fullA, (uint32_t)cfg.nkb * cfg.a_tx);
                int tap = 0, cc = 0;
                for (int kb = 0; kb < cfg.nkb; ++kb) {
                    const int koff = tap * p.Cp + cc * cfg.bk;
                    const uint32_t dst = sA + kb * cfg.a_bytes;
                    const CUtensorMap* map = dup && cfg.nbt > 1 ? &maps.wexp_dup : &maps.wexp;
                    tma_load_2d(dst, map, bar_fullA, koff, my_blk * kBlockRows);
                    if (dup) tma_load_2d(dst + cfg.a_bytes / 2, map, bar_fullA, koff, my_blk * kBlockRows);
                    if (++cc == cfg.cpt) { cc = 0; ++tap; }
                }
            }
            const uint32_t nring = pre_b_producer ? (uint32_t)cfg.nB : (uint32_t)cfg.nA;
            const uint32_t bar_e = pre_b_producer ? bar_emptyB : bar_emptyA;
            const uint32_t bar_f = pre_b_producer ? bar_fullB : bar_fullA;
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (uint32_t tile = first; tile < ntiles && ok; tile += step) {
                const uint32_t nt = tile / (uint32_t)cfg.nbt;
                const int blk = (int)(tile - nt * (uint32_t)cfg.nbt) << kM2;
                int b0, h0;
                if (cfg.tiles_per_image) {
                    b0 = (int)(nt / (uint32_t)cfg.tiles_per_image);
                    h0 = min((int)(nt - (uint32_t)b0 * (uint32_t)cfg.tiles_per_image) * cfg.th, p.Ho - cfg.th);
                } else {
                    b0 = (int)nt * cfg.tb;
                    h0 = 0;
                }
                const int row_a = blk * kBlockRows;
                int tap = 0, cc = 0, ti = 0, tj = 0;
                for (int kb = 0; kb < cfg.nkb; ++kb) {
                    if (!mbar_wait(bar_e + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
                    if (pre_b_producer && kTps3) {
                        if (cfg.colshift) {
                            // one stage = one column shift: the th + kh - 1 input rows the tile needs, fetched once
                            // and read by the kh taps of that column at row offsets (see TensorCfg::colshift)
                            mbar_arrive_expect_tx(bar_f + 8 * s, cfg.tx_bytes);
                            tma_load_4d(sB + s * cfg.b_bytes, &maps.act[0], bar_f + 8 * s, cc * cfg.bk, ti - p.pad, h0 - p.pad, b0);
                            if (++cc == cfg.cpt) { cc = 0; ++ti; }
                        } else {
                            // one stage = the taps of one kernel row (one channel chunk per tap in this mode)
                            mbar_arrive_expect_tx(bar_f + 8 * s, cfg.tps * cfg.tx_bytes);
                            for (int t = 0; t < cfg.tps; ++t) {
                                const TapBox tb = tap_box(p, h0, ti, tj + t);
                                tma_load_4d(sB + s * cfg.b_bytes + t * cfg.b_sub, &maps.act[tb.map], bar_f + 8 * s, 0, tb.x, tb.y, b0);
                            }
                            ++ti;
                        }
                        kb += cfg.tps - 1;
                        if (++s == nring) { s = 0; ph ^= 1; }
                        continue;
                    }
                    if (pre_b_producer) {
                        mbar_arrive_expect_tx(bar_f + 8 * s, cfg.tx_bytes);
                        const TapBox tb = tap_box(p, h0, ti, tj);
                        tma_load_4d(sB + s * cfg.b_bytes, &maps.act[tb.map], bar_f + 8 * s, cc * cfg.bk, tb.x, tb.y, b0);
                    } else {
                        const int koff = tap * p.Cp + cc * cfg.bk;
                        mbar_arrive_expect_tx(bar_f + 8 * s, cfg.a_tx);
                        tma_load_2d(sA + s * cfg.a_bytes, &maps.wexp, bar_f + 8 * s, koff, row_a);
                        if (dup) tma_load_2d(sA + s * cfg.a_bytes + cfg.a_bytes / 2, &maps.wexp, bar_f + 8 * s, koff, row_a);
                    }
                    if (++s == nring) { s = 0; ph ^= 1; }
                    if (++cc == cfg.cpt) { cc = 0; ++tap; if (++tj == p.kw) { tj = 0; ++ti; } }
                }
            }
            if (!ok) {
                for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        // The whole warp walks the loops in step, so that ring positions and descriptors are the same for all lanes and known to
        // be; the elected lane issues the MMAs and commits.
        {
            uint32_t sa = 0, phA = 0, sb = 0, phB = 0, it = 0;
            const uint64_t desc_a0 = smem_desc_kmajor(sA, cfg.bk), desc_b0 = smem_desc_kmajor(sB, cfg.bk);
            const uint32_t desc_lo0_a = (uint32_t)desc_a0, desc_lo0_b = (uint32_t)desc_b0, desc_hi = (uint32_t)(desc_a0 >> 32);
            pdl_wait();                                   // (a bounded wait begins when the kernel in front is over)
            bool have_a = !kAres || my_tiles == 0 || mbar_wait_step(bar_fullA, 0, abort_flag);
            for (uint32_t tile = first; tile < ntiles && have_a; tile += step, ++it) {
                // one accumulator per tile, alternating; or (two row blocks per tile) both, every tile
                const uint32_t ab = kM2 ? 0u : (it & 1);
                const uint32_t tpar = kM2 ? ((it & 1) ^ 1) : (((it >> 1) & 1) ^ 1);
                if (!mbar_wait_step(bar_tempty + 8 * ab, tpar, abort_flag)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + ab * kTileN;
                bool ok = true;
                int cc = 0;
                if (kTps3) {
                    // resident weights, three 64-byte k-blocks per activation stage (never with two row blocks):
                    // the taps of a kernel row in three sub-buffers, or (colshift) the taps of a kernel COLUMN
                    // reading one buffer at three row offsets
                    const uint32_t a_step = (uint32_t)cfg.a_bytes >> 4, b_step = (uint32_t)cfg.b_bytes >> 4;
                    const uint32_t t_step = cfg.colshift ? ((uint32_t)(p.W * cfg.bk) >> 4) : ((uint32_t)cfg.b_sub >> 4);
                    const uint32_t a_t = cfg.colshift ? 3 * a_step * (uint32_t)cfg.cpt : a_step;       // between the three taps of a stage
                    const uint32_t a_adv = cfg.colshift ? a_step : 3 * a_step;     // from stage to stage
                    uint32_t a_lo = desc_lo0_a, b_lo = desc_lo0_b + sb * b_step;
                    const bool two_last = (cfg.last_ksteps == 2);
                    bool two = two_last || cfg.cpt > 1;                            // (of two chunks the first is whole)
                    for (int kb = 0; kb < cfg.nkb; kb += 3) {
                        if (!mbar_wait_step(bar_fullB + 8 * sb, phB, abort_flag)) { ok = false; break; }
                        tc_fence_after();
                        if (two) {
                            mma_i8_step<2>(d_tmem, a_lo, b_lo, desc_hi, cfg.idesc, kb ? 1u : 0u);
                            mma_i8_step<2>(d_tmem, a_lo + a_t, b_lo + t_step, desc_hi, cfg.idesc, 1u);
                            mma_i8_step<2>(d_tmem, a_lo + 2 * a_t, b_lo + 2 * t_step, desc_hi, cfg.idesc, 1u);
                        } else {
                            mma_i8_step<1>(d_tmem, a_lo, b_lo, desc_hi, cfg.idesc, kb ? 1u : 0u);
                            mma_i8_step<1>(d_tmem, a_lo + a_t, b_lo + t_step, desc_hi, cfg.idesc, 1u);
                            mma_i8_step<1>(d_tmem, a_lo + 2 * a_t, b_lo + 2 * t_step, desc_hi, cfg.idesc, 1u);
                        }
                        mma_commit_step(bar_emptyB + 8 * sb);
                        a_lo += a_adv;
                        b_lo += b_step;
                        if (cfg.cpt > 1) two = !two || two_last;
                        if (++sb == (uint32_t)cfg.nB) { sb = 0; phB ^= 1; b_lo = desc_lo0_b; }
                    }
                } else if (!kAres && cfg.bk == 128 && cfg.last_ksteps == 4) {
                    // The common deep-K form, kept as short as it gets: every k-block is four MMAs (eight
                    // with two row blocks) on a full 128-byte stage of each ring.
                    const uint32_t a_step = (uint32_t)cfg.a_bytes >> 4, b_step = (uint32_t)cfg.b_bytes >> 4;
                    uint32_t a_lo = desc_lo0_a + sa * a_step, b_lo = desc_lo0_b + sb * b_step;
                    if (kM2) {
                        if (!mbar_wait_step(bar_tempty + 8, tpar, abort_flag)) break;
                        tc_fence_after();
                    }
                    for (int kb = 0; kb < cfg.nkb; ++kb) {
                        if (!mbar_wait_step(bar_fullB + 8 * sb, phB, abort_flag) || !mbar_wait_step(bar_fullA + 8 * sa, phA, abort_flag)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t acc = kb ? 1u : 0u;
                        mma_i8_step<4>(d_tmem, a_lo, b_lo, desc_hi, cfg.idesc, acc);
                        if (kM2) mma_i8_step<4>(d_tmem + kTileN, a_lo + (kABytes >> 4), b_lo, desc_hi, cfg.idesc, acc);
                        mma_commit_step(bar_emptyA + 8 * sa);
                        mma_commit_step(bar_emptyB + 8 * sb);
                        a_lo += a_step;
                        b_lo += b_step;
                        if (++sa == (uint32_t)cfg.nA) { sa = 0; phA ^= 1; a_lo = desc_lo0_a; }
                        if (++sb == (uint32_t)cfg.nB) { sb = 0; phB ^= 1; b_lo = desc_lo0_b; }
                    }
                } else {
                    const bool uniform = (cfg.last_ksteps == (cfg.bk >> 5));      // every k-block has the same depth
                    const uint32_t a_step = (uint32_t)cfg.a_bytes >> 4, b_step = (uint32_t)cfg.b_bytes >> 4;
                    uint32_t a_lo = kAres ? desc_lo0_a : desc_lo0_a + sa * a_step;
                    uint32_t b_lo = desc_lo0_b + sb * b_step;
                    for (int kb = 0; kb < cfg.nkb; ++kb) {
                        if (!mbar_wait_step(bar_fullB + 8 * sb, phB, abort_flag) ||
                            (!kAres && !mbar_wait_step(bar_fullA + 8 * sa, phA, abort_flag))) { ok = false; break; }
                        tc_fence_after();
                        const int ksteps = (uniform || cc != cfg.cpt - 1) ? (cfg.bk >> 5) : cfg.last_ksteps;
                        mma_i8_steps(ksteps, d_tmem, a_lo, b_lo, desc_hi, cfg.idesc, kb ? 1u : 0u);
                        if (kM2) {
                            // second row block: rows 128..255 of the weight stage, second accumulator
                            if (kb == 0) {
                                if (!mbar_wait_step(bar_tempty + 8, tpar, abort_flag)) { ok = false; break; }
                                tc_fence_after();
                            }
                            const uint32_t a1 = a_lo + (kABytes >> 4);
                            mma_i8_steps(ksteps, d_tmem + kTileN, a1, b_lo, desc_hi, cfg.idesc, kb ? 1u : 0u);
                        }
                        if (!kAres) mma_commit_step(bar_emptyA + 8 * sa);
                        mma_commit_step(bar_emptyB + 8 * sb);
                        a_lo += a_step;
                        b_lo += b_step;
                        if (++sa == (uint32_t)cfg.nA) { sa = 0; phA ^= 1; if (!kAres) a_lo = desc_lo0_a; }
                        if (++sb == (uint32_t)cfg.nB) { sb = 0; phB ^= 1; b_lo = desc_lo0_b; }
                        if (!uniform && ++cc == cfg.cpt) cc = 0;
                    }
                }
                if (!ok) break;
                mma_commit_step(bar_tfull + 8 * ab);
                if (kM2) mma_commit_step(bar_tfull + 8);
            }
        }
    } else if (!kPre && warp < 2 + kNumExpWarps) {
        // ---------------------------------------------------------- expanders
        // The packed codes of a k-block (a few KB, in L2) go to registers and from there, expanded, to the stage.  A warp
        // takes 32 rows in packed order, which are of one kind but where two kinds meet, and then runs without a branch;
        // the four (64-byte k-blocks: two) 32-code pieces of a row are neighbours, so that a load touches eight rows and not
        // 32, and of eight lanes' stores at most two meet in a bank.  What bounds it is one warp's chain of instructions
        // (four to eight cycles each), which is why everything that stays the same for a tile is worked out once for it,
        // a tile ahead, and a piece's registers are loaded again as soon as it is expanded.  With the
        // codes brought to shared memory in boxes of 16 rows and expanded from there: 3072x768 N=4096 36.9 us, now 21.6;
        // 3x3 512x512 on 12,544 pixels 84, now 51 to 59.
        const int grp = (warp - 2) >> 2;                 // which k-blocks: g % kGroups == grp
        const int ppr = cfg.bk >> 5;                     // pieces of a row, and rows of a thread, per k-block
        const int q = lane & (ppr - 1), r0 = ((warp - 2) & 3) * 32 + (ppr == 4 ? lane >> 2 : lane >> 1), r_step = 32 / ppr;
        // tile look-ahead: one tile, or kGroups tiles when every tile is a single k-block
        const int64_t look = (cfg.nkb == 1) ? kGroups : 1;
        const int64_t total = my_tiles * cfg.nkb;
        const bool rows_change = step % (uint32_t)p.nblocks != 0u;
        // a row block's rows in the packed buffer: first and number of each kind
        pdl_wait();
        const int32_t* const blocks = pdl_ordered(p.blocks), *const perm = pdl_ordered(p.perm);
        const uint4* const codes = reinterpret_cast<const uint4*>(pdl_ordered(p.q4));
        int4 blk_a;
        int2 blk_b;
        int blk_next = 0;
        auto load_block = [&](int64_t local) {
            blk_next = (int)((uint32_t)(first + (uint32_t)min(local, my_tiles - 1) * step) % (uint32_t)p.nblocks);
            blk_a = __ldg(reinterpret_cast<const int4*>(blocks + 8 * blk_next));
            blk_b = __ldg(reinterpret_cast<const int2*>(blocks + 8 * blk_next + 4));
        };
        const int n4 = p.nP + p.nF4;
        const uint32_t q8_first = (uint32_t)((p.q8 - p.q4) >> 4);
        // this thread's rows in tile f_tl (and, _next, in tile f_tl + look): first code / 16 bytes; place in a stage, two of 16 bits
        // each; a byte with the kind (3: no such row); the kind all rows of the warp have, or 4
        uint32_t off[4], off_next[4], place[2], kinds = 0, kinds_next = 0, uni = 3, uni_next = 3;
        int row_next[4], first_next = 0;
        auto look_up = [&]() {
            first_next = blk_next * kBlockRows;
            kinds_next = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + (i & (ppr - 1)) * r_step, f = r - blk_a.y, e = f - blk_a.w;
                const int kind = e >= blk_b.y ? 3 : f < 0 ? kPoT4 : e < 0 ? kFixed4 : kFixed8;
                const int packed = kind == kPoT4 ? blk_a.x + r : kind == kFixed4 ? p.nP + blk_a.z + f : n4 + blk_b.x + e;
                off_next[i] = kind == 3 ? 0u : kind == kFixed8 ? q8_first + (uint32_t)(packed - n4) * (uint32_t)(p.Kp >> 4) : (uint32_t)packed * (uint32_t)(p.Kp >> 5);
                row_next[i] = kind == 3 ? first_next : __ldg(perm + packed);
                kinds_next |= (uint32_t)kind << (8 * i);
            }
            const uint32_t k0 = __shfl_sync(0xffffffffu, kinds_next, 0) & 3u;      // (every lane takes part in both votes)
            const uint32_t same = __all_sync(0xffffffffu, kinds_next == k0 * 0x01010101u);
            uni_next = same ? k0 : 4u;
        };
        auto take_rows = [&]() {
            kinds = kinds_next;
            uni = uni_next;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                off[i] = off_next[i];
                const uint32_t r = (uint32_t)(row_next[i] - first_next), swz = ppr == 4 ? r & 7u : (r >> 1) & 3u;
                const uint32_t d = r * (uint32_t)cfg.bk + (((uint32_t)(2 * q) ^ swz) << 4);
                place[i >> 1] = i & 1 ? place[i >> 1] | (d << 16) : d;
            }
        };
        int64_t g = grp, f_tl = g / cfg.nkb;             // this CTA's k-block counter; tile and place of the k-block to be loaded next
        int f_kb = (int)(g - f_tl * cfg.nkb), f_tap = f_kb / cfg.cpt, f_cc = f_kb - f_tap * cfg.cpt;
        const int Cp32 = p.Cp >> 5;
        uint4 lo[4], hi[4];                              // (hi: the second half of 32 eight-bit codes)
        auto load = [&](int i, uint32_t piece) {
            const bool eight = ((kinds >> (8 * i)) & 3u) == kFixed8;
            const uint4* src = codes + (off[i] + (eight ? 2u * piece : piece));
            lo[i] = __ldg(src);
            if (eight) hi[i] = __ldg(src + 1);
        };
        auto has_piece = [&]() { return uni != 3u && q < (f_cc == cfg.cpt - 1 ? cfg.last_ksteps : ppr); };
        auto piece_of = [&]() { return (uint32_t)(f_tap * Cp32 + f_cc * ppr + q); };
        auto put = [&](uint32_t dst, const uint32_t (&w)[8]) {
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]));
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst ^ 16u), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]));
        };
        // (a piece is not touched before the one in front of it is stored: its own load may still be on its way.  Left to
        // itself the compiler interleaves the pieces and waits for all four loads at once)
        auto hold = [&](int i) { asm volatile("" : "+r"(lo[i].x), "+r"(lo[i].y), "+r"(lo[i].z), "+r"(lo[i].w)); };
        uint32_t sa = (uint32_t)(grp % cfg.nA), phA = (uint32_t)((grp / cfg.nA) & 1);
        if (g < total) {
            load_block(f_tl);
            look_up();
            take_rows();
            load_block(f_tl + look);
            look_up();
            load_block(f_tl + 2 * look);
            if (has_piece()) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < ppr) load(i, piece_of());
            }
        }
        while (g < total) {
            // what is in the registers now, and then the place of what follows it there
            const uint32_t c_kinds = kinds, c_uni = uni, c_place[2] = {place[0], place[1]};
            const bool c_on = has_piece();
            g += kGroups;
            f_kb += kGroups;
            f_cc += kGroups;
            while (f_cc >= cfg.cpt) { f_cc -= cfg.cpt; ++f_tap; }
            if (f_kb >= cfg.nkb) {
                int64_t adv = 0;
                while (f_kb >= cfg.nkb) { f_kb -= cfg.nkb; ++adv; }
                f_tap = f_kb / cfg.cpt;
                f_cc = f_kb - f_tap * cfg.cpt;
                f_tl += adv;
                if (rows_change) {
                    take_rows();                          // (the look-ahead's tile: with two groups adv is look, 2 for nkb == 1 and else 1)
                    look_up();
                    load_block(f_tl + 2 * look);
                }
            }
            const bool on = g < total && has_piece();
            const uint32_t piece = piece_of();
            if (!mbar_wait_warp(bar_emptyA + 8 * sa, phA ^ 1, abort_flag)) break;
            const uint32_t dst = sA + sa * cfg.a_bytes;
            auto at = [&](int i) { return dst + (i & 1 ? c_place[i >> 1] >> 16 : c_place[i >> 1] & 0xFFFFu); };
            if (c_uni == kPoT4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= ppr) break;
                    hold(i);
                    uint32_t w[8];
                    expand_pot_chunk(lo[i], w);
                    if (on) load(i, piece);
                    if (c_on) put(at(i), w);
                }
            } else if (c_uni == kFixed4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= ppr) break;
                    hold(i);
                    uint32_t w[8];
                    expand_fixed4_chunk_x16(lo[i], w);
                    if (on) load(i, piece);
                    if (c_on) put(at(i), w);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= ppr) break;
                    hold(i);
                    const uint32_t kind = (c_kinds >> (8 * i)) & 3u;
                    uint32_t w[8] = {lo[i].x, lo[i].y, lo[i].z, lo[i].w, hi[i].x, hi[i].y, hi[i].z, hi[i].w};
                    if (kind == kPoT4) expand_pot_chunk(lo[i], w);
                    else if (kind == kFixed4) expand_fixed4_chunk_x16(lo[i], w);
                    if (on) load(i, piece);
                    if (c_on && kind != 3u) put(at(i), w);
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_fullA + 8 * sa);
            sa += kGroups; while (sa >= (uint32_t)cfg.nA) { sa -= cfg.nA; phA ^= 1; }
        }
        __syncwarp();
    } else if (warp >= kThreads / 32 - cfg.epi_warps) {
        // ---------------------------------------------------------- epilogue
        // Warp w may read tensor-memory lanes 32*(w%4)..+31.  The warps that share a quarter (one, or
        // three in pre mode) take alternate 32-pixel chunks; with duplicated rows the two quarters
        // holding the same rows share the chunks as well.
        const int quarter = warp & 3;
        const int first_epi = kThreads / 32 - cfg.epi_warps;               // epilogue warps are the last epi_warps warps
        const int ew = warp - first_epi;                                   // 0 .. epi_warps-1
        // how many epilogue warps share a quarter, and this warp's rank among them
        auto count_q = [&](int q) { const int f = first_epi + ((q - first_epi) & 3); return (kThreads / 32 - 1 - f) / 4 + 1; };
        const int my_rank = (warp - (first_epi + ((quarter - first_epi) & 3))) >> 2;
        const int row0 = dup ? (quarter & 1) * 32 : quarter * 32;       // first row (within the block) of this warp
        const int cstride = dup ? count_q(quarter & 1) + count_q((quarter & 1) + 2) : count_q(quarter);
        const int cfirst = (dup && (quarter >> 1)) ? count_q(quarter & 1) + my_rank : my_rank;
        const uint32_t my_stage = sOut + (uint32_t)ew * (cfg.out_bufs * (kRQ ? kRqStage : kWarpStage));
        uint32_t it = 0, stg_count = 0;
        bool alive = true;
        int scale_blk = -1, shift = 0;
        float scale = 0.f;
        const ActFast rq_fast = act_fast_setup(kRQ ? p.rq_alpha : 1.0f, kRQ ? p.rq_kind : 0);
        pdl_wait();
        for (uint32_t tile = first; tile < ntiles && alive; tile += step, ++it) {
          // a tile is one row block (accumulators alternate between tiles), or two (one accumulator each)
          for (int half = 0; half <= kM2; ++half) {
            const uint32_t ab = kM2 ? (uint32_t)half : (it & 1);
            const uint32_t tpar = kM2 ? (it & 1) : ((it >> 1) & 1);
            // tile indices fit 32 bits (checked on the host): 32-bit divisions, a fraction of the 64-bit ones' cost,
            // which every epilogue warp would otherwise pay in front of each tile
            const uint32_t nt = tile / (uint32_t)cfg.nbt;
            const int blk = ((int)(tile - nt * (uint32_t)cfg.nbt) << kM2) + half;
            int64_t n0;
            if (cfg.tiles_per_image) {
                const uint32_t img = nt / (uint32_t)cfg.tiles_per_image, tin = nt - img * (uint32_t)cfg.tiles_per_image;
                n0 = ((int64_t)img * p.Ho + min((int)tin * cfg.th, p.Ho - cfg.th)) * (int64_t)p.Wo;
            } else {
                n0 = (int64_t)nt * cfg.npix;
            }
            const int nvalid = (int)min((int64_t)cfg.npix, p.N - n0);
            const int m = blk * kBlockRows + row0 + lane;
            const bool row_ok = m < p.M;
            if (blk != scale_blk) {
                // the row's scale: loaded when the row block changes (never again for layers of one row block)
                scale_blk = blk;
                scale = 0.f;
                shift = 0;
                if (row_ok) {
                    scale = __fmul_rn(__ldg(pdl_ordered(p.wstep) + m), p.act_step);
                    shift = (!kPre && __ldg(pdl_ordered(p.kind) + m) == kFixed4) ? 4 : 0;   // expanders store Fixed-4 codes as 16 * value
                }
            }
            if (!mbar_wait_warp(bar_tfull + 8 * ab, tpar, abort_flag)) { alive = false; break; }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + ab * kTileN;
            const int nchunks = (nvalid + 31) >> 5;
            auto release_tmem = [&]() {
                // all accumulators of this tile are in registers: hand the buffer back
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tempty + 8 * ab);
            };
            if (blk * kBlockRows + row0 >= p.M || cfirst >= nchunks) {      // no valid row, or no chunk, for this warp
                release_tmem();
                continue;
            }
            // Output one 32-pixel chunk held in registers.
            auto emit = [&](const uint32_t (&v)[32], int c) {
                const int jmax = min(32, nvalid - c * 32);
                if (kRQ) {
                    // y as in the fp32 epilogue, then the activation quantizer's arithmetic on it;
                    // one code byte per output, 32 pixels x 32 rows = 1 KB per chunk
                    if (use_tma_store) {
                        // (two buffers take turns: the barrier of the chunk in between is behind this one's last readers)
                        const uint32_t stg = my_stage + (stg_count & 1) * 1024u;
                        ++stg_count;
                        // t = the clipped value on 0..1 from one saturating fused operation, u = t * range + low; adding
                        // 1.5 * 2^23 in the same operation as that product rounds u, and the same product again with the
                        // rounded value taken off says how far u was from it.  The defining chain and this one are a
                        // handful of roundings of relative size 2^-24 of at most 15 apart (< 8e-6), so a value at least
                        // 1e-5 away from every boundary k + 1/2 has the same code.  The largest remainder of a lane's
                        // values decides about the second pass (one chunk of 32 x 32 in fifty has a value to decide again).
                        const float range = p.rq_kind == RMSMP_ACT_U4 ? 15.0f : 14.0f, low = p.rq_kind == RMSMP_ACT_U4 ? 0.0f : -7.0f;
                        const float bias = p.rq_kind == RMSMP_ACT_U4 ? 0.0f : 0.5f;
                        const float g = __fmul_rn(__fmul_rn(scale, rq_fast.r), p.rq_kind == RMSMP_ACT_U4 ? 1.0f : 0.5f);
                        const bool fast = rq_fast.ok && fabsf(g) <= 1e20f;
                        const uint64_t range2 = f32x2(range, range), magic2 = f32x2(kRqMagic + low, kRqMagic + low), minus2 = f32x2(-1.0f, -1.0f);
                        uint32_t again = fast ? 0u : 0xFFu;              // bit i: a value of columns 4i .. 4i + 3 has to be decided again
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float far = 0.0f;
#pragma unroll
                            for (int j = 4 * i; j < 4 * i + 4; j += 2) {
                                const uint64_t t2 = f32x2(__saturatef(__fmaf_rn(__int2float_rn((int)v[j] >> shift), g, bias)),
                                                          __saturatef(__fmaf_rn(__int2float_rn((int)v[j + 1] >> shift), g, bias)));
                                const uint64_t s2 = fma_f32x2(t2, range2, magic2);
                                const uint64_t d2 = fma_f32x2(t2, range2, fma_f32x2(s2, minus2, magic2));
                                float s0, s1, d0, d1;
                                f32x2_split(s2, s0, s1);
                                f32x2_split(d2, d0, d1);
                                asm("max.abs.f32 %0, %0, %1, %2;" : "+f"(far) : "f"(d0), "f"(d1));
                                asm volatile("st.shared.u8 [%0], %1;" ::"r"(stg + j * 32 + lane), "r"(__float_as_uint(s0)) : "memory");
                                asm volatile("st.shared.u8 [%0], %1;" ::"r"(stg + j * 32 + 32 + lane), "r"(__float_as_uint(s1)) : "memory");
                            }
                            again |= far > 0.49999f ? 1u << i : 0u;
                        }
                        // Those columns again by the definition, from tensor memory (the whole warp takes every step: the
                        // load is a warp-wide instruction).  This code is small and touches none of the registers above,
                        // so that its mere presence costs nothing.
                        again = __reduce_or_sync(0xffffffffu, again);
                        while (again) {
                            const int j0 = 4 * (__ffs(again) - 1);
                            again &= again - 1;
                            uint32_t w[4];
                            tmem_ld_four(taddr + c * 32 + j0, w);
#pragma unroll 1
                            for (int j = j0; j < j0 + 4; ++j) {
                                const float y = __fmul_rn(__int2float_rn((int)w[0] >> shift), scale);
                                asm volatile("st.shared.u8 [%0], %1;" ::"r"(stg + j * 32 + lane), "r"((uint32_t)act_code(y, p.rq_alpha, p.rq_kind)) : "memory");
                                w[0] = w[1]; w[1] = w[2]; w[2] = w[3];
                            }
                            __syncwarp();
                        }
                        __syncwarp();
                        // whole 32-byte sectors, two lanes a pixel.  (A bulk store of 32 rows of 32 bytes holds its thread, and the next
                        // chunk waits until it has been read out: 192x32 on 200,704 pixels 27.8 against 26.8 us, 128x128 3x3 above 30.4 and 29.4.)
                        const int m0 = blk * kBlockRows + row0 + 16 * (lane & 1);
                        int8_t* o = p.rq_codes + (n0 + c * 32 + (lane >> 1)) * p.ld_codes + m0;
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            uint32_t w[4];
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(stg + 512 * t + 16 * lane) : "memory");
                            if ((lane >> 1) + 16 * t < jmax && m0 < p.M) *reinterpret_cast<uint4*>(o) = make_uint4(w[0], w[1], w[2], w[3]);
                            o += 16 * p.ld_codes;
                        }
                    } else if (row_ok) {
                        int8_t* o = p.rq_codes + (n0 + c * 32) * p.ld_codes + m;
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            if (j < jmax) {
                                const float y = __fmul_rn(__int2float_rn((int)v[j] >> shift), scale);
                                o[(int64_t)j * p.ld_codes] = (int8_t)act_code_exact(y, p.rq_alpha, p.rq_kind, rq_fast);
                            }
                        }
                    }
                } else if (use_tma_store) {
                    const bool tail = cfg.tail_rows && (c == (cfg.npix >> 5));
                    const int nsub = acc_out ? 2 : 1;
                    for (int sub = 0; sub < nsub; ++sub) {
                        const uint32_t stg = my_stage + (cfg.out_bufs == 2 ? (stg_count & 1) * kWarpStage : 0);
                        ++stg_count;
                        if (lane == 0) {
                            if (cfg.out_bufs == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                            else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        }
                        __syncwarp();                    // the buffer's previous store has been read out
                        if (!out_mn) {
                            // [pixel][row]: the warp writes 128 contiguous bytes per pixel
                            const uint32_t a0 = stg + lane * 4;
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const int a = (int)v[j] >> shift;
                                const uint32_t w = sub ? (uint32_t)a : __float_as_uint(__fmul_rn(__int2float_rn(a), scale));
                                asm volatile("st.shared.b32 [%0], %1;" ::"r"(a0 + j * 128), "r"(w) : "memory");
                            }
                        } else {
                            // [row][pixel], 16-byte chunks swizzled by row (matches the 128-byte-swizzled store map)
                            const uint32_t a0 = stg + lane * 128;
#pragma unroll
                            for (int cch = 0; cch < 8; ++cch) {
                                uint32_t w[4];
#pragma unroll
                                for (int t = 0; t < 4; ++t) {
                                    const int a = (int)v[4 * cch + t] >> shift;
                                    w[t] = sub ? (uint32_t)a : __float_as_uint(__fmul_rn(__int2float_rn(a), scale));
                                }
                                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                                             ::"r"(a0 + ((cch ^ (lane & 7)) << 4)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
                            }
                        }
                        fence_proxy_async_smem();
                        __syncwarp();                    // chunk complete in shared memory
                        if (lane == 0) {
                            const CUtensorMap* map = sub ? (tail ? &maps.acc_tail : &maps.acc_full)
                                                         : (tail ? &maps.out_tail : &maps.out_full);
                            const int cm = blk * kBlockRows + row0, cn = (int)(n0 + c * 32);
                            if (!out_mn) tma_store_2d(map, stg, cm, cn); else tma_store_2d(map, stg, cn, cm);
                        }
                    }
                } else if (out_mn) {
                    // [row][pixel] that bulk stores cannot address (a row is no multiple of 16 bytes): turned in shared
                    // memory (word r * 32 + (j ^ r): no bank conflicts on either side), then 128 contiguous bytes a store.
                    // Straight from the lanes' rows a store touched 32 sectors (1088x64 N=515: 27.5 us)
                    const int rows = min(32, p.M - (blk * kBlockRows + row0));
#pragma unroll 1
                    for (int sub = 0; sub < (acc_out ? 2 : 1); ++sub) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int a = (int)v[j] >> shift;
                            const uint32_t w = sub ? (uint32_t)a : __float_as_uint(__fmul_rn(__int2float_rn(a), scale));
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(my_stage + (uint32_t)(lane * 32 + (j ^ lane)) * 4u), "r"(w) : "memory");
                        }
                        __syncwarp();
                        uint32_t* o = (sub ? reinterpret_cast<uint32_t*>(acc_out) : reinterpret_cast<uint32_t*>(p.out)) +
                                      (int64_t)(blk * kBlockRows + row0) * p.ld_out + n0 + c * 32 + lane;
#pragma unroll 4
                        for (int r = 0; r < rows; ++r) {
                            uint32_t x;
                            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(my_stage + (uint32_t)(r * 32 + (lane ^ r)) * 4u) : "memory");
                            if (lane < jmax) o[(int64_t)r * p.ld_out] = x;
                        }
                        __syncwarp();
                    }
                } else if (row_ok) {
                    // direct stores: outputs whose leading dimension or base rules out bulk stores
                    float* o = p.out + (n0 + c * 32) * p.ld_out + m;
                    int32_t* oa = acc_out ? acc_out + (n0 + c * 32) * p.ld_out + m : nullptr;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        if (j < jmax) {
                            const int a = (int)v[j] >> shift;
                            o[(int64_t)j * p.ld_out] = __fmul_rn(__int2float_rn(a), scale);
                            if (oa) oa[(int64_t)j * p.ld_out] = a;
                        }
                    }
                }
            };
            if (kRQ) {
                // (a re-quantizing chunk may read its accumulators again: the buffer is handed back after the last one)
                uint32_t v[32];
#pragma unroll 1
                for (int c = cfirst; c < nchunks; c += cstride) {
                    tmem_ld_issue(taddr + c * 32, v);
                    tmem_ld_wait(v);
                    emit(v, c);
                    __syncwarp();
                }
                release_tmem();
                continue;
            }
            // two register sets: the load of this warp's next chunk is in flight while the current one is emitted
            // (tensor-memory loads and their waits are warp-wide: every chunk ends with the warp together again)
            uint32_t va[32], vb[32];
            tmem_ld_issue(taddr + cfirst * 32, va);
            tmem_ld_wait(va);
            for (int c = cfirst; c < nchunks; c += 2 * cstride) {
                const int c1 = c + cstride, c2 = c + 2 * cstride;
                const bool more1 = c1 < nchunks;
                if (more1) tmem_ld_issue(taddr + c1 * 32, vb); else release_tmem();
                emit(va, c);
                __syncwarp();
                if (more1) {
                    tmem_ld_wait(vb);
                    const bool more2 = c2 < nchunks;
                    if (more2) tmem_ld_issue(taddr + c2 * 32, va); else release_tmem();
                    emit(vb, c1);
                    __syncwarp();
                    if (more2) tmem_ld_wait(va);
                }
            }
          }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    if (threadIdx.x == 0 && s_abort) atomicMax(p.status, (uint32_t)RMSMP_ERR_TIMEOUT);
}

// ------------------------------------------------------------------ host side

EncodeTiledFn encode_fn() { return tensor_map_encoder(); }

// Tensor maps of the activation codes for boxes of `bk` channels x th output rows x tb images
// (see act_parity_split: one map, or one per parity sub-grid of a stride-2 layer).
bool encode_act_maps(EncodeTiledFn enc, const Problem& p, int bk, int th, int tb, CUtensorMapSwizzle swz, CUtensorMap out[4])
{
    const cuuint64_t pitch = (cuuint64_t)p.pix_pitch;
    if (act_parity_split(p)) {
        for (int py = 0; py < 2; ++py)
            for (int px = 0; px < 2; ++px) {
                const cuuint64_t gdim[4] = {(cuuint64_t)p.Cin, (cuuint64_t)((p.W - px + 1) / 2), (cuuint64_t)((p.H - py + 1) / 2), (cuuint64_t)p.B};
                const cuuint64_t gstr[3] = {2 * pitch, 2 * pitch * p.W, pitch * p.W * p.H};
                const cuuint32_t box[4] = {(cuuint32_t)bk, (cuuint32_t)p.Wo, (cuuint32_t)th, (cuuint32_t)tb};
                const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
                const int8_t* base = p.act + ((int64_t)py * p.W + px) * p.pix_pitch;
                if (enc(&out[py * 2 + px], CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<int8_t*>(base), gdim, gstr, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                    return false;
            }
        return true;
    }
    const cuuint64_t gdim[4] = {(cuuint64_t)p.Cin, (cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.B};
    const cuuint64_t gstr[3] = {pitch, pitch * p.W, pitch * p.W * p.H};
    const cuuint32_t box[4] = {(cuuint32_t)bk, (cuuint32_t)(p.Wo * p.stride), (cuuint32_t)(th * p.stride), (cuuint32_t)tb};
    const cuuint32_t estr[4] = {1u, (cuuint32_t)p.stride, (cuuint32_t)p.stride, 1u};
    return enc(&out[0], CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<int8_t*>(p.act), gdim, gstr, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// One row block of a 3x3 convolution of step one with 65 to 128 channels, on expanded weights: they stay resident (144 KB, as two
// 64-channel k-blocks a tap) beside a ring of column-shift stages, from two tiles per CTA up.  Through the rings a tile brings 373 KB
// into the SM, so 97: 128x128 on 256 images of 28x28 36.0 against 34.8 us, codes out 35.0 and 29.4 (three stages, and
// eight epilogue warps, are what fits).
bool wide_shift(const Problem& p)
{
    const int most = p.Wo <= kTileN ? kTileN / p.Wo : 0;
    if (!p.wexp || p.nblocks != 1 || p.Cin <= 64 || p.Cin > 128 || p.kh != 3 || p.kw != 3 || p.stride != 1 || p.pad != 1 || most < 1) return false;
    if ((int64_t)p.Ho * p.Wo <= kTileN && 2 * (int64_t)p.Ho * p.Wo <= kTileN) return false;      // (several images a tile)
    const int per_image = (p.Ho + most - 1) / most, th = (p.Ho + per_image - 1) / per_image;
    return 3 * (((th + 2) * p.W * 64 + 1023) / 1024 * 1024) <= kSmemLimit - (1024 + 64 * kMaxRing) - 18 * kBlockRows * 64 - kWideEpi * kWarpStage &&
           (int64_t)p.B * per_image >= 2 * p.sms;
}

// Whether the copy engine can fetch the activations, one box a tap.
bool addressable(const Problem& p)
{
    if (p.pix_pitch % 16 != 0 || (p.Cin % 16 != 0 && !p.ragged_k)) return false;
    if ((reinterpret_cast<uintptr_t>(p.act) & 15) != 0) return false;
    if (p.wexp && (reinterpret_cast<uintptr_t>(p.wexp) & 15) != 0) return false;
    if (p.Wo > kTileN || (int64_t)p.Wo * p.stride > 256) return false;
    return (int64_t)p.Ho * p.Wo > kTileN || (int64_t)p.Ho * p.stride <= 256;      // (tiles of whole images, or of as many rows as a box has)
}

bool plan(const Problem& p, TensorCfg& c)
{
    if (!addressable(p)) return false;
    const int64_t hw = (int64_t)p.Ho * p.Wo;
    if (hw <= kTileN) {
        c.th = p.Ho;
        c.tb = (int)std::min<int64_t>(kTileN / hw, p.B);
        // Narrower tiles where the widest ones leave SMs idle in the last round: a k-block takes 0.28 us + 0.13 per 256
        // pixels, the output of 256 pixels 0.8 beside the next tile's k-blocks and 1.2 at the end (768x768 N=4096: 96 tiles
        // of 256 tokens, or 144 of 176: 7.7 against 7.2 us); not for gains
        // below a tenth, which measure as losses as often, nor where reading the activations takes as long (10x4096 N=20000:
        // 24.1 us with 256 tokens a tile, 28.3 with 144).  [row][pixel] outputs keep to whole chunks of 32 pixels, without
        // which they leave through direct stores (256x64 N=20000 16.5 us with tiles of 144 pixels).
        if (p.wexp) {
            const int64_t sms = p.sms;
            const double nkb = (double)p.kh * p.kw * ((p.Cin + 127) / 128);
            const double read = (double)p.N * p.Cin / 6.3e6;
            auto cost = [&](int tb) {
                const double n = (double)tb * hw / 256.0, waves = (double)((((int64_t)p.B + tb - 1) / tb * p.nblocks + sms - 1) / sms);
                return std::max(waves * std::max(nkb * (0.28 + 0.13 * n), 0.4 + 0.8 * n) + 1.2 * n, read);
            };
            double best = 0.9 * cost(c.tb);
            const int most = c.tb, step = hw == 1 ? 16 : 1;
            const bool whole = p.out_mn && p.ld_out % 4 == 0 && p.N % 4 == 0 && most * hw % 32 == 0;
            for (int tb = (most - 1) / step * step; tb >= 1 && 2 * tb >= most; tb -= step)
                if (!(whole && tb * hw % 32 != 0) && cost(tb) < best) { best = cost(tb); c.tb = tb; }
        }
        c.tiles_per_image = 0;
        c.ntiles_n = (p.B + c.tb - 1) / c.tb;
    } else {
        // As few tiles as cover an image's rows, all of the same height.  (Heights that divide the image's make tiles of
        // one row where that is a prime: 3x3 256x256 on 64 images of 29x29 133 us against 30 so.)
        const int most = std::min(kTileN / p.Wo, 256 / p.stride);
        c.tiles_per_image = (p.Ho + most - 1) / most;
        // Lower tiles where the tallest leave SMs idle (few images): a k-block takes 0.25 us (128-byte rows 0.33) + 0.04 per 256
        // pixels + 0.1 with every SM busy, the output of 256 pixels 1.7.  3x3 64x32 on 2 of 49x49, tiles of five rows 8.3 us,
        // of one 6.0.  Not for a few rows, whose boxes of weights lie mostly outside the matrix and then take longer than the
        // activations' (3x3 16x16 on 12 of 62x8 6.6 and 9.9).
        if (p.wexp && p.M > 32) {
            const double sms = p.sms, bk = p.Cin % 128 != 0 && p.Cin % 128 <= 64 ? 64 : 128;
            const double nkb = p.kh * p.kw * std::ceil(p.Cin / bk);
            auto cost = [&](int per_image) {
                const double n = (double)((p.Ho + per_image - 1) / per_image * p.Wo) / 256.0;
                return 3.8 + 1.7 * n + nkb * ((bk == 64 ? 0.25 : 0.33) + 0.04 * n + 0.1 * ((double)p.B * per_image * p.nblocks / sms));
            };
            double best = 0.9 * cost(c.tiles_per_image);
            for (int per_image = c.tiles_per_image + 1; per_image <= p.Ho && (double)p.B * per_image * p.nblocks <= sms; ++per_image)
                if (cost(per_image) < best) { best = cost(per_image); c.tiles_per_image = per_image; }
        }
        c.th = (p.Ho + c.tiles_per_image - 1) / c.tiles_per_image;
        c.tiles_per_image = (p.Ho + c.th - 1) / c.th;
        c.tb = 1;
        c.ntiles_n = (int64_t)p.B * c.tiles_per_image;
    }
    c.npix = c.tb * c.th * p.Wo;
    c.n_mma = (c.npix + 15) / 16 * 16;
    c.ntiles = c.ntiles_n * p.nblocks;
    if (c.ntiles >= (1ll << 31)) return false;       // (the kernel counts in 32 bits, a step beyond the last)
    c.m2 = 0;
    c.nbt = p.nblocks;
    c.tps = 1;
    c.b_sub = 0;
    c.colshift = 0;
    c.pre = p.wexp ? 1 : 0;
    c.fill = 0;
    const bool resident = tensor_resident(p);
    // no workspace, but a whole row block's expanded weights stay resident: the CTA expands them once itself and the
    // layer runs in the workspace form
    if (!p.wexp && resident) { c.pre = 1; c.fill = 1; }
    // 64-byte k-blocks when a 128-byte row would be at most half used by the (last) channel chunk
    const bool wide = wide_shift(p);
    c.bk = wide || (c.pre ? p.Cin % 128 != 0 && p.Cin % 128 <= 64 : p.Cin <= 64) ? 64 : 128;
    c.a_bytes = kBlockRows * c.bk;
    c.b_bytes = kTileN * c.bk;
    c.cpt = (p.Cin + c.bk - 1) / c.bk;
    c.nkb = p.kh * p.kw * c.cpt;
    c.last_ksteps = (p.Cin - (c.cpt - 1) * c.bk + 31) / 32;
    c.tx_bytes = (uint32_t)c.npix * (uint32_t)c.bk;
    // kind::i8: int32 accumulate (bits 4-5 = 2), signed 8-bit A and B (bits 7-9, 10-12 = 1),
    // both K-major, N/8 at bit 17, M/16 at bit 24
    c.idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(c.n_mma >> 3) << 17) | ((uint32_t)(kBlockRows >> 4) << 24);
    c.tail_rows = c.npix & 31;
    c.tma_store = 0;
    c.dup = 0;
    c.ares = 0;
    c.cta_full = 0;
    c.epi_warps = kNumEpiWarps;
    const int stage = p.rq_codes ? kRqStage : kWarpStage;
    // (a row count that is not a multiple of 16 would spill into the padding columns)
    if (p.rq_codes && p.M % 16 == 0 && p.ld_codes % 16 == 0 && (reinterpret_cast<uintptr_t>(p.rq_codes) & 15) == 0) c.tma_store = 1;
    if (c.pre) {
        c.nA = (c.bk == 64) ? 6 : 3; c.nB = (c.bk == 64) ? 8 : 4; c.out_bufs = 1;
        c.epi_warps = warps_of(1, p.rq_codes && !c.tma_store) - 3;   // warp 2 fetches the weights (unless they are resident)
        c.dup = (p.M <= 64) ? 1 : 0;
        if (resident) {
            c.ares = 1;
            const bool many = p.rq_codes && (!c.tma_store || (c.nkb == 1 && c.ntiles >= 4 * (int64_t)p.sms));
            c.epi_warps = wide ? (p.rq_codes ? 2 * kWideEpi : kWideEpi) : warps_of(2, many) - 2;
            c.nA = c.nkb;
            const int64_t left = kSmemLimit - (1024 + 64 * kMaxRing) - (int64_t)c.nkb * c.a_bytes -
                                 (int64_t)c.epi_warps * stage;
            c.nB = (int)std::min<int64_t>(kMaxRing, left / c.b_bytes);
        }
        c.tps = 1;
        c.b_sub = c.b_bytes;
        if (c.ares && c.bk == 64 && (c.cpt == 1 || wide) && p.kw == 3 && c.last_ksteps <= 2) {
            c.tps = 3;
            c.b_sub = (c.n_mma * c.bk + 1023) / 1024 * 1024;
            c.b_bytes = c.tps * c.b_sub;
            if (p.kh == 3 && p.stride == 1 && p.Wo == p.W && c.tb == 1 && c.npix == c.th * p.W) {
                c.colshift = 1;
                c.tx_bytes = (uint32_t)((c.th + 2) * p.W * c.bk);
                c.b_bytes = ((c.th + 2) * p.W * c.bk + 1023) / 1024 * 1024;
            }
            const int64_t left = kSmemLimit - (1024 + 64 * kMaxRing) - (int64_t)c.nkb * c.a_bytes -
                                 (int64_t)c.epi_warps * stage;
            c.nB = (int)std::min<int64_t>(kMaxRing, left / c.b_bytes);
            if (c.nB < 2) { c.tps = 1; c.colshift = 0; c.tx_bytes = (uint32_t)c.npix * (uint32_t)c.bk; c.b_bytes = kTileN * c.bk; c.b_sub = c.b_bytes; c.nB = (int)std::min<int64_t>(kMaxRing, left / c.b_bytes); }
        }
        // Two row blocks per tile pay when K is long (the two accumulators' epilogue is only half
        // hidden behind the next tile's MMAs) and when the halved tile count does not cost more in
        // idle SMs of the last wave than the ~20 % a double tile saves.
        const int64_t sms = p.sms;
        const int64_t waves1 = (c.ntiles + sms - 1) / sms, waves2 = (c.ntiles / 2 + sms - 1) / sms;
        if (!c.ares && !c.dup && c.bk == 128 && p.nblocks % 2 == 0 && c.nkb >= 16 && 16 * waves2 < 10 * waves1) {
            c.m2 = 1;
            c.nbt = p.nblocks / 2;
            c.ntiles = c.ntiles_n * c.nbt;
            c.a_bytes = 2 * kABytes;
            c.nA = 2; c.nB = 3;
        }
        c.a_rows = c.m2 ? 2 * kBlockRows : c.nbt > 1 ? kBlockRows : (std::min(p.M, c.dup ? kBlockRows / 2 : kBlockRows) + 7) / 8 * 8;
        c.a_tx = (uint32_t)(c.a_rows * c.bk * (c.dup && c.nbt == 1 ? 2 : 1));
        c.smem_bytes = (uint32_t)(c.nA * c.a_bytes + c.nB * c.b_bytes + c.epi_warps * c.out_bufs * stage + 1024 +
                                  64 * kMaxRing);
        return true;
    }
    // Four weight stages (a group expands into one while its last and the other group's two wait for their turn: three
    // are 20 to 30 % slower, six no faster), an output buffer a warp, and all the rest for activations.
    c.nA = 4;
    c.out_bufs = 1;
    c.b_bytes = (c.n_mma * c.bk + 1023) / 1024 * 1024;
    const int fixed = c.nA * c.a_bytes + kNumEpiWarps * c.out_bufs * kWarpStage + 1024 + 64 * kMaxRing;
    c.nB = std::min(kMaxRing, (kSmemLimit - fixed) / c.b_bytes);
    c.smem_bytes = (uint32_t)(fixed + c.nB * c.b_bytes);
    return true;
}

}  // namespace

static EncodeTiledFn driver_encoder()
{
    // (threads that come while another looks it up wait for it)
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(ptr);
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

// The driver's call needs a current context, which a thread has only after a runtime call that makes one: a thread whose first
// call comes here gets its device's.
static CUresult encode_tiled(CUtensorMap* map, CUtensorMapDataType type, cuuint32_t rank, void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                             const cuuint32_t* box, const cuuint32_t* steps, CUtensorMapInterleave interleave, CUtensorMapSwizzle swizzle,
                             CUtensorMapL2promotion promotion, CUtensorMapFloatOOBfill fill)
{
    const EncodeTiledFn fn = driver_encoder();
    CUresult r = fn(map, type, rank, base, dims, strides, box, steps, interleave, swizzle, promotion, fill);
    if (r == CUDA_ERROR_INVALID_CONTEXT || r == CUDA_ERROR_NOT_INITIALIZED) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) { cudaGetLastError(); return r; }
        r = fn(map, type, rank, base, dims, strides, box, steps, interleave, swizzle, promotion, fill);
    }
    return r;
}

EncodeTiledFn tensor_map_encoder() { return driver_encoder() ? encode_tiled : nullptr; }

bool encode_act_maps_4(const Problem& p, int bk, int th, int tb, void* maps4)
{
    EncodeTiledFn enc = encode_fn();
    return enc && encode_act_maps(enc, p, bk, th, tb, bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                                  static_cast<CUtensorMap*>(maps4));
}

// Whether the persistent kernel keeps a row block's expanded weights in shared memory: they fit beside the activation
// ring, and the grid can be a multiple of the row blocks without costing a round of tiles to speak of (a CTA then stays with
// one).  Without a workspace that is always
// the better form: the codes are expanded once per CTA, not per tile (144x160 on 740,050 pixels 355 against 131 us,
// 2048x512 N=4096 20.9 against 13.8).  With one, the weights of several row blocks are a stream that the activations of a
// first tile would wait behind (1024x512 N=4096, a tile per CTA: 8.1 us resident, 7.3 through the rings), and save
// shared-memory fills from two tiles per CTA up (144x32 on 200,704 pixels 39.7 against 36.1, 3x3 256x64 on 50,176 20.7
// against 17.7).  Beside 64 KB of them fewer than four activation stages of 128-byte rows are left, too few for a linear layer
// with fp32 outputs (192x512 on 200,000 tokens 56.3 us against 46.1, 512x512 on 50,176 28.6 against 26.3, 1024x512 on 20,000
// 23.2 against 21.5; codes out 37.0 against 38.1, 21.0 against 21.9, 19.1 against 19.6).
bool tensor_resident(const Problem& p)
{
    if (!p.wexp && p.rq_codes) return false;
    const int64_t sms = p.sms, tiles = (p.N + kTileN - 1) / kTileN * p.nblocks, whole = sms / p.nblocks * p.nblocks;
    if (whole == 0 || (p.nblocks > kResidentBlocks && (tiles + whole - 1) / whole > (tiles + sms - 1) / sms)) return false;
    if (wide_shift(p)) return true;
    const int bk = ((p.Cin % 128 != 0) && (p.Cin % 128 <= 64)) ? 64 : 128;
    const int64_t bytes = (int64_t)p.kh * p.kw * ((p.Cin + bk - 1) / bk) * kBlockRows * bk;
    if (bytes > 72 * 1024) return false;
    if (!p.wexp || p.nblocks == 1) return true;
    if (tiles < 2 * sms) return false;
    if (p.rq_codes) return true;
    // (two rounds of full tiles against three: 1872x160 on 4880 tokens, 20 tiles for the nine CTAs of a block, 14.4 us
    // resident, 11.7 through the rings)
    if ((p.N / kTileN * p.nblocks + sms - 1) / sms <= 2 && (tiles + whole - 1) / whole > 2) return false;
    return p.kh * p.kw > 1 || bk == 64 || bytes < 64 * 1024;
}

bool tensor_supported(const Problem& p)
{
    TensorCfg c;
    return plan(p, c) && encode_fn() != nullptr;
}

rmsmp_status launch_tensor(const Problem& p, cudaStream_t st)
{
    rmsmp_status s;
    if (!addressable(p) || !encode_fn()) return RMSMP_ERR_VARIANT;
    if (launch_split_if_better(p, st, &s) || launch_pair_if_better(p, st, &s)) return s;
    TensorCfg c;
    if (!plan(p, c)) return RMSMP_ERR_VARIANT;
    // All tiles of a CTA are of one row block where the grid is a multiple of them: required by resident weights, and with
    // expanders worth having when it costs no round of tiles (they look up a tile's rows only once then).
    int64_t grid = p.sms;
    const int64_t whole = grid / c.nbt * c.nbt;
    if (c.ares || (!c.pre && whole > 0 && (c.ntiles + whole - 1) / whole == (c.ntiles + grid - 1) / grid)) grid = whole;
    grid = std::min(grid, c.ntiles);
    if (c.ares && c.nbt > 1 && p.M % kBlockRows >= 1 && p.M % kBlockRows <= kBlockRows / 2) {
        // Shares of the grid by what a tile takes: the last block's output, done by all warps for half of the rows or less,
        // takes 0.5 to 0.7 of a full one's (256 pixels: 2.8 us; the products 0.17 to 0.41 a k-block).  Equal shares and a
        // half of the warps idle: 192x32 on 200,704 pixels 33.3 us against 31.7, codes out 30.5 and 27.8, 160x64 on 50,176
        // 10.5 and 8.9, 144x160 on 740,050 134 and 108.
        const double n = c.npix / 256.0, mma = c.nkb * (0.28 + 0.13 * n) * (c.bk == 64 ? 0.6 : 1.0), out = 2.8 * n;
        const double full_us = std::max(mma, out), last_us = std::max(mma, (p.rq_codes ? 0.72 : 0.45 + 0.15 * (p.M % kBlockRows) / 64.0) * out);
        const int64_t sms = p.sms, even = whole / c.nbt;
        double best = 0.95 * std::ceil((double)c.ntiles_n / even) * full_us;
        for (int64_t last = 1; last < even; ++last) {
            const int64_t full = (sms - last) / (c.nbt - 1);
            const double us = std::max(std::ceil((double)c.ntiles_n / full) * full_us, std::ceil((double)c.ntiles_n / last) * last_us);
            if (c.ntiles_n >= full && us < best) { best = us; c.cta_full = (int)full; c.dup = 1; grid = full * (c.nbt - 1) + last; }
        }
    }
    EncodeTiledFn enc = encode_fn();
    Maps mp;
    memset(&mp, 0, sizeof(mp));
    if (!encode_act_maps(enc, p, c.bk, c.colshift ? c.th + 2 : c.th, c.tb, c.bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, mp.act))
        return RMSMP_ERR_CUDA;
    if (p.wexp) {
        const cuuint64_t gd[2] = {(cuuint64_t)p.Kp, (cuuint64_t)p.M};
        const cuuint64_t gs[1] = {(cuuint64_t)p.Kp};
        const cuuint32_t es[2] = {1, 1};
        auto make = [&](CUtensorMap* m, int rows) -> bool {
            const cuuint32_t bx[2] = {(cuuint32_t)c.bk, (cuuint32_t)rows};
            return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t*>(p.wexp), gd, gs, bx, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, c.bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        };
        if (!make(&mp.wexp, c.a_rows) || (c.dup && c.nbt > 1 && !make(&mp.wexp_dup, kBlockRows / 2)))
            return RMSMP_ERR_CUDA;
    }

    const bool ld_ok = !p.rq_codes && (p.ld_out % 4 == 0) && (p.out_mn ? p.N % 4 == 0 : p.M % 4 == 0) && ((reinterpret_cast<uintptr_t>(p.out) & 15) == 0) &&
                       (!p.acc || (reinterpret_cast<uintptr_t>(p.acc) & 15) == 0);
    if (p.rq_codes) {
        // re-quantized output: [N][ld_codes] code bytes, sixteen rows of a pixel a store
        if (!c.pre || p.out_mn) return RMSMP_ERR_VARIANT;
    }
    // ([row][pixel]: a bulk store starts at a pixel that is a multiple of four)
    if (ld_ok && (!p.out_mn || (c.tail_rows == 0 && (c.tiles_per_image == 0 || p.Ho % c.th == 0)))) {
        auto make = [&](CUtensorMap* m, void* base, CUtensorMapDataType dt, int rows) -> bool {
            const cuuint32_t es[2] = {1, 1};
            const cuuint64_t gs[1] = {(cuuint64_t)p.ld_out * 4};
            if (!p.out_mn) {
                const cuuint64_t gd[2] = {(cuuint64_t)p.M, (cuuint64_t)p.N};
                const cuuint32_t bx[2] = {32u, (cuuint32_t)rows};
                return enc(m, dt, 2, base, gd, gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
            }
            const cuuint64_t gd[2] = {(cuuint64_t)p.N, (cuuint64_t)p.M};
            const cuuint32_t bx[2] = {32u, 32u};
            return enc(m, dt, 2, base, gd, gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        };
        bool ok = make(&mp.out_full, p.out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 32);
        if (ok && c.tail_rows) ok = make(&mp.out_tail, p.out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, c.tail_rows);
        if (ok && p.acc) ok = make(&mp.acc_full, p.acc, CU_TENSOR_MAP_DATA_TYPE_INT32, 32);
        if (ok && p.acc && c.tail_rows) ok = make(&mp.acc_tail, p.acc, CU_TENSOR_MAP_DATA_TYPE_INT32, c.tail_rows);
        c.tma_store = ok ? 1 : 0;
    }

    c.trigger = 2 * grid <= p.sms;

    // the kernel's form (see tensor_kernel): [mode][two row blocks][1: re-quantizing epilogue, 2: plain fp32 [N][M] bulk-store output,
    // 3: codes through the rings by 16-byte stores]
    typedef void (*KernelFn)(const Problem, const TensorCfg, const Maps);
    static const KernelFn table[4][2][4] = {
        {{tensor_kernel<0, 0, 0, 0>, nullptr, tensor_kernel<0, 0, 0, 1>}, {}},
        {{tensor_kernel<0, 0, 1, 0>, tensor_kernel<0, 1, 1, 0>, tensor_kernel<0, 0, 1, 1>, tensor_kernel<0, 1, 1, 1>},
         {tensor_kernel<1, 0, 1, 0>, tensor_kernel<1, 1, 1, 0>, tensor_kernel<1, 0, 1, 1>, tensor_kernel<1, 1, 1, 1>}},
        {{tensor_kernel<0, 0, 2, 0>, tensor_kernel<0, 1, 2, 0>, tensor_kernel<0, 0, 2, 1>}, {}},
        {{tensor_kernel<0, 0, 3, 0>, tensor_kernel<0, 1, 3, 0>, tensor_kernel<0, 0, 3, 1>}, {}},
    };
    const int mode = !c.pre ? 0 : (!c.ares ? 1 : (c.tps > 1 ? 3 : 2));
    const int i2 = c.m2 ? 1 : 0;
    const int io = p.rq_codes ? (mode == 1 && c.tma_store ? 3 : 1) : ((c.tma_store && !p.out_mn && !p.acc) ? 2 : 0);
    const KernelFn fn = table[mode][i2][io];
    if (!fn) return RMSMP_ERR_VARIANT;
    static bool attr_set[4][2][4][kMaxDevices] = {};
    if (!ensure_smem_attr(reinterpret_cast<const void*>(fn), kSmemLimit, attr_set[mode][i2][io])) return RMSMP_ERR_CUDA;
    if (launch_dependent(fn, (unsigned)grid, 32 * warps_of(mode, io == 1), c.smem_bytes, st, p, c, mp) != cudaSuccess) {
        cudaGetLastError();
        return RMSMP_ERR_CUDA;
    }
    return RMSMP_OK;
}

}  // namespace rmsmp
