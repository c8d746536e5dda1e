// Patch matrix of a convolution's activation codes, for layers whose channel count is too small for the
// implicit form (a network's first layer: 3 channels, 7 x 7 filters; Section 4.1, Table 6 quantizes it like
// the rest): cols[n][(i * kw + j) * C + c] = act[b][ho * s + i - p][wo * s + j - p][c] for output pixel
// n = (b, ho, wo), zero outside the image and in the columns beyond kh * kw * C.  The layer is then a linear
// layer over these rows (reduction order tap-major, channel fastest), which the GEMM entry points take.
// A filter tap of such a layer is 3 bytes, which no bulk tensor copy can start on (16-byte rule), so this is
// plain loads: the input is read many times, but it is small and stays in L1/L2; the kernel is bound by
// writing the matrix.  One thread per 16 output bytes, stepping through filter row, column and channel.
#include <algorithm>
#include "common.cuh"

namespace rmsmp {

namespace {

constexpr int kGatherThreads = 256;
constexpr size_t kRowsSmem = 100 * 1024;                  // im2col_rows_kernel's most

struct GatherArgs {
    const int8_t* act;
    int8_t* cols;
    int64_t pix_pitch, ld_cols, N;
    int B, H, W, C, kh, kw, stride, pad, Ho, Wo, K, units;      // units: 16-byte pieces per output row
};

__global__ void __launch_bounds__(kGatherThreads) im2col_kernel(GatherArgs a)
{
    // thread <-> (pixel of the block's current group, 16-byte piece of its row): fixed per thread; the pixel index
    // advances by whole groups; 32-bit index arithmetic (the host checks the counts)
    pdl_wait();
    pdl_trigger();
    a.act = pdl_ordered(a.act);
    const int upr = a.units;
    const int ppg = kGatherThreads / upr;                 // pixels per group (units <= kGatherThreads is checked by the host)
    const int my_p = threadIdx.x / upr, k0 = (threadIdx.x - my_p * upr) << 4;
    if (my_p >= ppg) return;
    const int tap0 = k0 / a.C, c0 = k0 - tap0 * a.C;
    const int i0 = tap0 / a.kw, j0 = tap0 - i0 * a.kw;
    const uint32_t N = (uint32_t)a.N;
    const int64_t row_pitch = (int64_t)a.W * a.pix_pitch;
    for (uint32_t n = blockIdx.x * (uint32_t)ppg + my_p; n < N; n += gridDim.x * (uint32_t)ppg) {
        const uint32_t t = n / (uint32_t)a.Wo;
        const int wo = (int)(n - t * (uint32_t)a.Wo);
        const uint32_t b = t / (uint32_t)a.Ho;
        const int ho = (int)(t - b * (uint32_t)a.Ho);
        const int y0 = ho * a.stride - a.pad, x0 = wo * a.stride - a.pad;
        int i = i0, j = j0, c = c0;
        const int8_t* ptr = a.act + (int64_t)b * a.H * row_pitch + (int64_t)(y0 + i) * row_pitch + (int64_t)(x0 + j) * a.pix_pitch + c;
        bool yok = (unsigned)(y0 + i) < (unsigned)a.H;
        uint32_t out[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (k0 + e < a.K) {
                if (yok && (unsigned)(x0 + j) < (unsigned)a.W) out[e >> 2] |= (uint32_t)(uint8_t)__ldg(ptr) << (8 * (e & 3));
                ++ptr;
                if (++c == a.C) {
                    c = 0;
                    ptr += a.pix_pitch - a.C;
                    if (++j == a.kw) {
                        j = 0; ++i;
                        ptr += row_pitch - (int64_t)a.kw * a.pix_pitch;
                        yok = (unsigned)(y0 + i) < (unsigned)a.H;
                    }
                }
            }
        }
        *reinterpret_cast<uint4*>(a.cols + (int64_t)n * a.ld_cols + k0) = make_uint4(out[0], out[1], out[2], out[3]);
    }
}

// The same through shared memory, one output row (b, ho) per block pass.  The kh input rows it touches are copied
// in first, channels packed, zeros around them (the padding).  A row of the patch matrix is then kh runs of kw * C
// consecutive bytes, one from each input row, so sixteen output bytes are one to three unaligned 16-byte pieces of
// shared memory: five words and four funnel shifts each.  A warp builds the same sixteen columns for 32 neighbouring
// pixels: which runs they come from is uniform, and lanes that are stride * C bytes apart hit the banks at most two
// deep (a byte at a time with the columns spread over the lanes, conflicts made the layer 96 us at 64 x 224 x 224 x 3,
// four times what writing the matrix takes; 53 us this way).  The finished rows are assembled in shared memory and
// leave as one bulk copy: they are consecutive in memory.
struct RowsArgs {
    int zero_left, rowb;      // bytes of zeros in front of a staged row (a multiple of 16, at least 16 + pad * C), bytes per staged row
    int tile;                 // pixels assembled at a time
    int wide;                 // padded pixels: bytes per copy into shared memory (16, 4 or 1), 0: a word a pixel
};
// One run's share of a unit (sixteen columns): which input row, the byte that would be the unit's column 0 relative to
// the pixel's first byte in that row, and the columns that are this run's.
struct alignas(32) Piece { uint32_t keep[4]; int row, off, last, pad; };      // last: 1 on a unit's last piece

// kDense: pixels follow one another without padding bytes.
template <bool kDense>
__global__ void __launch_bounds__(kGatherThreads) im2col_rows_kernel(GatherArgs a, const RowsArgs ra)
{
    extern __shared__ __align__(32) uint8_t s_mem[];
    uint8_t* const s_out = s_mem;                                          // [tile][ld_cols]
    uint8_t* const s_rows = s_mem + (size_t)ra.tile * a.ld_cols;           // [kh][rowb]
    Piece* const s_piece = reinterpret_cast<Piece*>(s_mem + ((size_t)ra.tile * a.ld_cols + (size_t)a.kh * ra.rowb + 31) / 32 * 32);      // in the order of the columns
    __shared__ int s_base[16];                                             // per input row: where its column -pad starts in s_rows
    __shared__ int s_first[kGatherThreads];                                // per unit: its first piece, -1 for zero columns
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = a.kw * a.C;
    const int row_bytes = a.W * a.C;                                       // a staged row's own bytes
    const int chunks = ra.rowb >> 4;
    const int rows_total = a.B * a.Ho;
    if (tid < a.units) {
        // a unit's pieces; in front of it lie as many pieces as whole units, and one more for every run that ended inside one
        int k = 16 * tid, i = k / run, o = k - i * run;
        int n = tid + min(i, a.kh - 1);
        for (int j = 1; j <= min(i, a.kh - 1); ++j) n -= (j * run) % 16 == 0 ? 1 : 0;
        s_first[tid] = i < a.kh ? n : -1;
        for (int e = 0; e < 16 && i < a.kh; ++i, o = 0, ++n) {
            const int len = min(run - o, 16 - e);
            for (int j = 0; j < 4; ++j) {
                const int lo = max(e - 4 * j, 0), hi = min(e + len - 4 * j, 4);
                s_piece[n].keep[j] = hi > lo ? (0xFFFFFFFFu >> (8 * (4 - hi + lo))) << (8 * lo) : 0u;
            }
            s_piece[n].row = i; s_piece[n].off = o - e;
            e += len;
            s_piece[n].last = (e == 16 || i + 1 == a.kh) ? 1 : 0;
        }
    }
    if (!kDense) {
        // padded pixels are copied one by one to the same place of every row: the zeros around them are written once
        for (int q = tid; q < a.kh * chunks; q += kGatherThreads) *reinterpret_cast<uint4*>(s_rows + 16 * q) = make_uint4(0u, 0u, 0u, 0u);
        if (tid < a.kh) s_base[tid] = tid * ra.rowb + ra.zero_left - a.pad * a.C;
    }
    pdl_wait();
    pdl_trigger();
    a.act = pdl_ordered(a.act);
    for (int r = blockIdx.x; r < rows_total; r += gridDim.x) {
        const int b = r / a.Ho, ho = r - b * a.Ho;
        const int y0 = ho * a.stride - a.pad;
        __syncthreads();                                                   // the previous row's readers are done
        if constexpr (kDense) {
            // rows of packed pixels: 16-byte granules of global memory to the same place inside a granule of shared memory
            for (int q = tid; q < a.kh * chunks; q += kGatherThreads) {
                const int i = q / chunks, j = q - i * chunks;
                const int y = y0 + i;
                const bool in_y = (unsigned)y < (unsigned)a.H;
                const int8_t* row = a.act + (int64_t)(b * a.H + (in_y ? y : 0)) * row_bytes;
                const int lead = (int)(reinterpret_cast<uintptr_t>(row) & 15);
                const int first = 16 * j - ra.zero_left - lead;            // the granule's first byte, relative to the row
                uint32_t v[4] = {0u, 0u, 0u, 0u};
                if (in_y && first > -16 && first < row_bytes) {
                    if (first >= 0 && first + 16 <= row_bytes) {
                        const uint4 w = __ldg(reinterpret_cast<const uint4*>(row + first));
                        v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
                    } else {
                        for (int e = 0; e < 16; ++e)
                            if ((unsigned)(first + e) < (unsigned)row_bytes)
                                v[e >> 2] |= (uint32_t)(uint8_t)__ldg(row + first + e) << (8 * (e & 3));
                    }
                }
                *reinterpret_cast<uint4*>(s_rows + i * ra.rowb + 16 * j) = make_uint4(v[0], v[1], v[2], v[3]);
                if (j == 0) s_base[i] = i * ra.rowb + ra.zero_left + lead - a.pad * a.C;
            }
        } else {
            const int pixels = a.kh * a.W;
            auto source = [&](int q, int& i, int& x) -> const int8_t* {        // pixel q of the kh rows; null outside the image
                i = q / a.W; x = q - i * a.W;
                const int y = y0 + i;
                return (unsigned)y < (unsigned)a.H ? a.act + ((int64_t)(b * a.H + y) * a.W + x) * a.pix_pitch : nullptr;
            };
            if (ra.wide == 0) {
                // up to four channels in pixels of whole words: eight words on their way at a time.  (The tensor's last
                // pixel byte by byte: what lies behind its channels need not be there.)
                const int8_t* last = a.act + ((int64_t)a.B * a.H * a.W - 1) * a.pix_pitch;
                for (int q0 = tid; q0 < pixels; q0 += 8 * kGatherThreads) {
                    uint32_t w[8];
                    uint8_t* dst[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int q = q0 + u * kGatherThreads;
                        int i = 0, x = 0;
                        const int8_t* src = q < pixels ? source(q, i, x) : nullptr;
                        dst[u] = s_rows + i * ra.rowb + ra.zero_left + x * a.C;
                        w[u] = 0u;
                        if (src != nullptr && src != last) w[u] = __ldg(reinterpret_cast<const uint32_t*>(src));
                        else if (src != nullptr) for (int c = 0; c < a.C; ++c) w[u] |= (uint32_t)(uint8_t)__ldg(src + c) << (8 * c);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (q0 + u * kGatherThreads < pixels)
                            for (int c = 0; c < a.C; ++c) dst[u][c] = (uint8_t)(w[u] >> (8 * c));
                }
            } else {
                for (int q = tid; q < pixels; q += kGatherThreads) {
                    int i, x;
                    const int8_t* src = source(q, i, x);
                    uint8_t* dst = s_rows + i * ra.rowb + ra.zero_left + x * a.C;
                    if (ra.wide == 16) {
                        for (int c = 0; c < a.C; c += 16)
                            *reinterpret_cast<uint4*>(dst + c) = src ? __ldg(reinterpret_cast<const uint4*>(src + c)) : make_uint4(0u, 0u, 0u, 0u);
                    } else if (ra.wide == 4) {
                        for (int c = 0; c < a.C; c += 4)
                            *reinterpret_cast<uint32_t*>(dst + c) = src ? __ldg(reinterpret_cast<const uint32_t*>(src + c)) : 0u;
                    } else {
                        for (int c = 0; c < a.C; ++c) dst[c] = src ? (uint8_t)__ldg(src + c) : (uint8_t)0;
                    }
                }
            }
        }
        for (int p0 = 0; p0 < a.Wo; p0 += ra.tile) {
            const int np = min(ra.tile, a.Wo - p0);
            const int groups = (np + 31) >> 5;
            if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");       // the previous tile has left
            __syncthreads();
            int u = warp, g = 0;                                           // unit, group of 32 pixels
            while (u >= a.units) { u -= a.units; ++g; }
            while (g < groups) {
                const int p = g * 32 + lane;
                const int xoff = (p0 + min(p, np - 1)) * a.stride * a.C;
                uint32_t out[4] = {0u, 0u, 0u, 0u};
                for (int i = s_first[u]; i >= 0;) {                        // the same pieces for the whole warp
                    const uint4 keep = *reinterpret_cast<const uint4*>(s_piece[i].keep);
                    const int4 d = *reinterpret_cast<const int4*>(&s_piece[i].row);
                    const int at = s_base[d.x] + d.y + xoff;
                    const uint32_t* w = reinterpret_cast<const uint32_t*>(s_rows + (at & ~3));
                    const uint32_t sh = (uint32_t)at * 8u;                 // (the shift counts modulo 32)
                    out[0] |= __funnelshift_r(w[0], w[1], sh) & keep.x;
                    out[1] |= __funnelshift_r(w[1], w[2], sh) & keep.y;
                    out[2] |= __funnelshift_r(w[2], w[3], sh) & keep.z;
                    out[3] |= __funnelshift_r(w[3], w[4], sh) & keep.w;
                    i = d.z ? -1 : i + 1;
                }
                if (p < np) *reinterpret_cast<uint4*>(s_out + (size_t)p * a.ld_cols + 16 * u) = make_uint4(out[0], out[1], out[2], out[3]);
                u += kGatherThreads / 32;
                while (u >= a.units) { u -= a.units; ++g; }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (tid == 0) {
                const int8_t* dst = a.cols + ((int64_t)r * a.Wo + p0) * a.ld_cols;
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(dst), "r"((uint32_t)__cvta_generic_to_shared(s_out)), "r"((uint32_t)(np * (int)a.ld_cols)) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Three channels, K x K filters, pixels without padding bytes and patch rows without spare units: the row of the patch
// matrix is built by ONE thread, in registers, a run of kw * C bytes after the other.  Every place in it is known when
// this is compiled, so a run is four 8-byte loads, a funnel shift a word (the source is moved so that it lies as the
// destination does) and one merge with the run in front; a warp's 32 pixels are 6 bytes apart, so that half a warp's
// 8-byte loads lie within 32 banks.  A block takes `rows` neighbouring output rows of an image at a time (about 256
// pixels), whose input rows overlap.  What is left is the shared-memory pipe: 56 of a group's 150 passes are these
// loads, 40 the finished rows' stores, 40 the bulk copy's reads.  7x7 on 64 images of 224x224 33.5 us, against 52 by
// im2col_rows_kernel (which keeps other channel counts, padded pixels and rows too wide for two of them beside the tile).
template <int K>
__global__ void __launch_bounds__(kGatherThreads) im2col_rgb_kernel(GatherArgs a, const int zero_left, const int rowb, const int rows)
{
    constexpr int kRun = 3 * K, kUnits = (3 * K * K + 15) / 16;
    extern __shared__ __align__(32) uint8_t s_mem[];
    uint8_t* const s_out = s_mem;                                          // [rows * Wo][16 * kUnits]
    uint8_t* const s_rows = s_mem + (size_t)rows * a.Wo * (16 * kUnits);   // [(rows - 1) * stride + K][rowb]
    __shared__ int s_base[64];                                             // per input row: where its column -pad starts in s_rows
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row_bytes = 3 * a.W, chunks = rowb >> 4, per_image = (a.Ho + rows - 1) / rows, items = a.B * per_image;
    pdl_wait();
    pdl_trigger();
    a.act = pdl_ordered(a.act);
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int b = item / per_image, ho = (item - b * per_image) * rows;
        const int nr = min(rows, a.Ho - ho), np = nr * a.Wo, in_rows = (nr - 1) * a.stride + K;
        const int y0 = ho * a.stride - a.pad;
        __syncthreads();                                                   // the previous pass's readers are done
        // 16-byte granules of global memory to the same place inside a granule of shared memory, zeros around them
        for (int q = tid; q < in_rows * chunks; q += kGatherThreads) {
            const int i = q / chunks, j = q - i * chunks;
            const int y = y0 + i;
            const bool in_y = (unsigned)y < (unsigned)a.H;
            const int8_t* row = a.act + (int64_t)(b * a.H + (in_y ? y : 0)) * row_bytes;
            const int lead = (int)(reinterpret_cast<uintptr_t>(row) & 15);
            const int first = 16 * j - zero_left - lead;                   // the granule's first byte, relative to the row
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (in_y && first > -16 && first < row_bytes) {
                if (first >= 0 && first + 16 <= row_bytes) {
                    v = __ldg(reinterpret_cast<const uint4*>(row + first));
                } else {
                    uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if ((unsigned)(first + e) < (unsigned)row_bytes) w[e >> 2] |= (uint32_t)(uint8_t)__ldg(row + first + e) << (8 * (e & 3));
                    v = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            *reinterpret_cast<uint4*>(s_rows + i * rowb + 16 * j) = v;
            if (j == 0) s_base[i] = i * rowb + zero_left + lead - 3 * a.pad;
        }
        if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");       // the previous rows have left
        __syncthreads();
        for (int q0 = 32 * warp; q0 < np; q0 += kGatherThreads) {
            const int q = q0 + lane, px = min(q, np - 1), r = px / a.Wo;
            const int x3 = 3 * a.stride * (px - r * a.Wo), i0 = r * a.stride;
            uint32_t out[4 * kUnits];
#pragma unroll
            for (int i = 0; i < K; ++i) {
                constexpr uint32_t kLow[4] = {0u, 0xFFu, 0xFFFFu, 0xFFFFFFu};
                const int pos = kRun * i, front = pos & 3, words = (front + kRun + 3) / 4, loads = (front + kRun + 14) / 8;      // (known when compiled)
                const int at = s_base[i0 + i] + x3 - front;
                const uint2* src = reinterpret_cast<const uint2*>(s_rows + (at & ~7));
                uint32_t w[2 * ((kRun + 17) / 8) + 2] = {};
#pragma unroll
                for (int j = 0; j < loads; ++j) { const uint2 v = src[j]; w[2 * j] = v.x; w[2 * j + 1] = v.y; }
                const bool odd = (at & 4) != 0;
#pragma unroll
                for (int j = 0; j <= words; ++j) w[j] = odd ? w[j + 1] : w[j];
#pragma unroll
                for (int j = 0; j < words; ++j) {
                    const uint32_t v = __funnelshift_r(w[j], w[j + 1], 8u * (uint32_t)at);      // (the shift counts modulo 32)
                    const int o = (pos >> 2) + j;
                    out[o] = j == 0 && front ? (out[o] & kLow[front]) | (v & ~kLow[front]) : v;
                }
                if (i + 1 == K) {
                    const int end = (pos + kRun) & 3;
                    if (end) out[(pos + kRun) >> 2] &= kLow[end];
#pragma unroll
                    for (int o = (pos + kRun + 3) >> 2; o < 4 * kUnits; ++o) out[o] = 0u;
                }
            }
            // Rows of 2 or 10 units put the first and the last four of eight neighbouring lanes into the same banks: of two units
            // the last four store the second one first.
            if (q < np) {
                uint4* const dst = reinterpret_cast<uint4*>(s_out + (size_t)q * (16 * kUnits));
                constexpr bool kSwap = kUnits % 4 == 2;
                const bool second = kSwap && (lane & 4) != 0;
#pragma unroll
                for (int u = 0; u < kUnits; u += 2) {
                    const uint32_t* o = out + 4 * u;
                    if (kSwap) {
                        dst[u + second] = second ? make_uint4(o[4], o[5], o[6], o[7]) : make_uint4(o[0], o[1], o[2], o[3]);
                        dst[u + !second] = second ? make_uint4(o[0], o[1], o[2], o[3]) : make_uint4(o[4], o[5], o[6], o[7]);
                    } else {
                        dst[u] = make_uint4(o[0], o[1], o[2], o[3]);
                        if (u + 1 < kUnits) dst[u + 1] = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            const int8_t* dst = a.cols + ((int64_t)b * a.Ho + ho) * a.Wo * (16 * kUnits);
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(dst), "r"((uint32_t)__cvta_generic_to_shared(s_out)), "r"((uint32_t)(np * 16 * kUnits)) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

}  // namespace

cudaError_t launch_im2col(const int8_t* act, int B, int H, int W, int C, int64_t pix_pitch, int kh, int kw, int stride, int pad,
                          int Ho, int Wo, int8_t* cols, int64_t ld_cols, cudaStream_t st)
{
    GatherArgs a;
    a.act = act; a.cols = cols; a.pix_pitch = pix_pitch; a.ld_cols = ld_cols;
    a.B = B; a.H = H; a.W = W; a.C = C; a.kh = kh; a.kw = kw; a.stride = stride; a.pad = pad; a.Ho = Ho; a.Wo = Wo;
    a.N = (int64_t)B * Ho * Wo;
    a.K = kh * kw * C;
    a.units = (int)(ld_cols >> 4);
    if (a.N == 0) return cudaSuccess;
    if (a.units > kGatherThreads) return cudaErrorInvalidValue;
    // input rows in shared memory when they fit, beside the tile that is assembled
    RowsArgs ra;
    auto up16 = [](int n) { return (n + 15) & ~15; };
    ra.zero_left = up16(pad * C) + 16;
    ra.rowb = ra.zero_left + 16 + up16(std::max(W, (Wo - 1) * stride + kw - pad) * C) + up16(pad * C) + 32;
    ra.tile = (int)std::min<int64_t>(Wo, std::max<int64_t>(1, 20 * 1024 / ld_cols));
    if (ra.tile < Wo && ra.tile >= 32) ra.tile &= ~31;
    const size_t smem = ((size_t)ra.tile * ld_cols + (size_t)kh * ra.rowb + 31) / 32 * 32 + 32 + sizeof(Piece) * (size_t)(a.units + kh);
    if (C == 3 && pix_pitch == 3 && kh == kw && (kw == 3 || kw == 5 || kw == 7) && ld_cols == (3 * kw * kw + 15) / 16 * 16 && stride <= 4) {
        // As many rows a pass as leave every SM one: im2col_rows_kernel, here with about 256 pixels a pass whatever their number, and so: 7x7 of step
        // two, one image of 112x112 2.7, 3.4 and 2.7 us, 25 of 37x77 4.1, 3.9 and 3.4; twice as many passes: 256 of 32x32 at step four 4.4, now 3.4.
        // Few passes of several rows are too few at step four (7x7, 8 of 224x224 4.0, 4.0 and 4.4; 64 of 64x64 4.0, 3.4 and 3.3).
        const int64_t per_sm = (int64_t)B * Ho / sm_count();
        const int rows = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)Ho, 256 / Wo, 8, per_sm}));
        const size_t bytes = (size_t)rows * Wo * ld_cols + ((size_t)(rows - 1) * stride + kh) * ra.rowb;
        const int64_t items = (int64_t)B * ((Ho + rows - 1) / rows);
        if (bytes <= 46 * 1024 && items < (1ll << 31) && (stride < 4 || rows == 1 || per_sm >= 6)) {
            // (five blocks an SM at most, as below)
            const size_t smem3 = std::max<size_t>(bytes, 40 * 1024);
            auto* const kernel = kw == 3 ? im2col_rgb_kernel<3> : kw == 5 ? im2col_rgb_kernel<5> : im2col_rgb_kernel<7>;
            return launch_dependent(kernel, (unsigned)std::min<int64_t>(items, (int64_t)sm_count() * (200 * 1024 / smem3)), kGatherThreads, smem3, st, a, ra.zero_left, ra.rowb, rows);
        }
    }
    auto whole = [&](int w) { return pix_pitch % w == 0 && (reinterpret_cast<uintptr_t>(act) & (w - 1)) == 0; };
    ra.wide = C <= 4 && whole(4) ? 0 : C % 16 == 0 && whole(16) ? 16 : C % 4 == 0 && whole(4) ? 4 : 1;
    // Rows too wide for the shared memory that needs no opting in (7 x 7 x 3 from about 1000 pixels): fewer blocks share an SM, which
    // is worth it for few channels and rows enough (7 x 7, two images of 1080 x 1920 x 3 237 us by the other kernel, 74 so, and 130
    // with a fourth byte a pixel; 3 x 3, two of 224 x 224 x 64 47 and 71; 32 rows of 2000 x 3 10.7 and 18.8).
    static bool attr_set[2][kMaxDevices] = {};
    const bool dense = pix_pitch == C;
    void (*const rows_kernel)(GatherArgs, const RowsArgs) = dense ? im2col_rows_kernel<true> : im2col_rows_kernel<false>;
    const bool small = smem <= 46 * 1024, large = smem <= kRowsSmem && C <= 16 && (int64_t)B * Ho >= sm_count();
    if (small || (large && ensure_smem_attr(reinterpret_cast<const void*>(rows_kernel), (int)kRowsSmem, attr_set[dense]))) {
        const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(8, 200 * 1024 / smem));
        const int64_t blocks = std::min<int64_t>((int64_t)B * Ho, (int64_t)sm_count() * per_sm);
        // Rows that are not small take at least 40 KB, five blocks an SM: a launch is placed while the one in front drains, and more of them crowd together where
        // that leaves first (8 x 56 x 56 x 64 20.4 us against 22.6 with as many as fit; 2 x 640 x 640 x 3 10.3, 12.9).
        return launch_dependent(rows_kernel, (unsigned)blocks, kGatherThreads, dense && smem > 16 * 1024 ? std::max<size_t>(smem, 40 * 1024) : smem, st, a, ra);
    }
    const int ppg = kGatherThreads / a.units;
    const int64_t blocks = std::min<int64_t>((a.N + ppg - 1) / ppg, (int64_t)sm_count() * 16);
    return launch_dependent(im2col_kernel, (unsigned)blocks, kGatherThreads, 0, st, a);
}

}  // namespace rmsmp
