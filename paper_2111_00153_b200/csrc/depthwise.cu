// Depthwise convolution (one input channel per filter, as in MobileNet-v2's 3x3 layers): every channel c
// has its own filter row with its own scheme and precision (Figure 2), y[b][ho][wo][c] = sum over the
// taps of value[c][i][j] * a[b][ho*s+i-p][wo*s+j-p][c].  There is no reduction over channels, hence no
// matrix product: the layer is bound by its output write, and the work is integer multiply-adds on the
// CUDA cores.  A block expands the layer's codes once into shared memory, one word per tap and channel
// quad (channel 4q+j in byte j).
//
// 3 x 3 filters of stride 1 or 2: what bounds a straightforward kernel is the integer pipe, because
// channels-last words put four CHANNELS into a word while the 4-way dot product wants four TAPS (splitting
// every word into one-channel words spent three of four products on zeros: 42 instructions per output,
// 74 us for 56 x 56 x 192 at batch 64).  So the words of four neighbouring columns are transposed (4 x 4
// bytes, eight permutes), which makes the three taps of a kernel row one dot product; a thread owns a
// channel quad and four neighbouring columns and walks down a strip of rows, so that every input row is
// loaded and transposed once for the three output rows that it touches, and the next row's loads are in flight
// meanwhile.  What is left is load latency at two blocks of 128-register threads per SM; down tall strips the next four input
// rows are on their way instead, into words of shared memory of the thread's own, where nobody waits for anybody (see launch_depthwise).
// Other filters: a word is split into four one-channel words, one output per work item.
#include <algorithm>
#include "common.cuh"

namespace rmsmp {

namespace {

constexpr int kDwThreads = 256;
constexpr int kDwCols = 4;                                 // output columns per thread (3 x 3 path)
constexpr size_t kDwSmem = 226 * 1024;
constexpr int kDwAhead = 4;                                // input rows on their way per thread (with a ring)
constexpr uint32_t kDwRingColumn = kDwThreads * 4;         // a column of a ring row: a word per thread
__host__ __device__ constexpr size_t dw_ring(int s) { return (kDwAhead + 1) * (3 * s + 3) * (size_t)kDwRingColumn; }
// Sums start from the bits of 1.5 * 2^23: a nine-tap sum of int8 products is below 2^18, so the finished word IS the
// float 1.5 * 2^23 + sum and one subtraction gives float(sum) exactly.
constexpr int kDwMagicBits = 0x4B400000;
constexpr float kDwMagic = 12582912.0f;

__device__ __forceinline__ uint32_t dw_prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// Byte c of the words w0..w3 (columns) to bytes 0..3 of t[c]: channels-last words to one word per channel.
__device__ __forceinline__ void dw_transpose(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t (&t)[4])
{
    const uint32_t a = dw_prmt(w0, w1, 0x5140u), b = dw_prmt(w2, w3, 0x5140u);      // channels 0 and 1
    const uint32_t c = dw_prmt(w0, w1, 0x7362u), d = dw_prmt(w2, w3, 0x7362u);      // channels 2 and 3
    t[0] = dw_prmt(a, b, 0x5410u); t[1] = dw_prmt(a, b, 0x7632u);
    t[2] = dw_prmt(c, d, 0x5410u); t[3] = dw_prmt(c, d, 0x7632u);
}

// One input row of a thread's strip, ready for the dot products.  Stride 1: for every channel the words whose bytes 0..2
// are the three columns under a kernel row.  Stride 2: the transposed columns, from which dw_word forms those words
// where they are used -- a row serves one or two output rows there, and its sixteen words took registers that the
// loads ahead need (56 x 56 x 192 at batch 64, launches back to back: 22.6 us with them, 18.4 so; stride 1, three output rows a row, 47.8 with them).
template <int kS> struct DwRow { uint32_t g[4], t[kS == 1 ? 12 : 5]; };

template <int kS>
__device__ __forceinline__ void dw_arrange(const uint32_t (&a)[3 * kS + 3], DwRow<kS>& r)
{
    dw_transpose(a[0], a[1], a[2], a[3], r.g);                                              // columns 0 1 2 (3)
    if constexpr (kS == 1) {
        const uint32_t lo = dw_prmt(a[4], a[5], 0x5140u), hi = dw_prmt(a[4], a[5], 0x7362u);      // columns 4, 5: channels 0, 1 / 2, 3
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            r.t[3 * c] = r.g[c] >> 8;                                                       // columns 1 2 3
            r.t[3 * c + 1] = dw_prmt(r.g[c], c < 2 ? lo : hi, (c & 1) ? 0x6632u : 0x4432u); // columns 2 3 4
            r.t[3 * c + 2] = dw_prmt(r.g[c], c < 2 ? lo : hi, (c & 1) ? 0x7763u : 0x5543u); // columns 3 4 5
        }
    } else {
        uint32_t h[4];
        dw_transpose(a[4], a[5], a[6], a[7], h);
#pragma unroll
        for (int c = 0; c < 4; ++c) r.t[c] = h[c];
        r.t[4] = a[8];
    }
}

// The columns under output column j of channel c, in bytes 0..2.
template <int kS>
__device__ __forceinline__ uint32_t dw_word(const DwRow<kS>& r, int c, int j)
{
    if (j == 0) return r.g[c];
    if constexpr (kS == 1) return r.t[3 * c + j - 1];
    else if (j == 1) return dw_prmt(r.g[c], r.t[c], 0x4432u);                                              // columns 2 3 4
    else return j == 2 ? r.t[c] : dw_prmt(r.t[c], r.t[4], 0x0032u | (uint32_t)(4 + c) << 8 | (uint32_t)(4 + c) << 12);      // 4 5 6, 6 7 8
}

// A word from global to shared memory without passing through a register; `bytes` 0: zeros, nothing is read.
__device__ __forceinline__ void dw_copy(uint32_t dst, const int8_t* src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void dw_store(const Problem& p, uint32_t n, int q, const int* acc)
{
    const float4 ws = __ldg(reinterpret_cast<const float4*>(p.wstep) + q);
    float4 o;
    o.x = __fmul_rn(__int2float_rn(acc[0]), __fmul_rn(ws.x, p.act_step));
    o.y = __fmul_rn(__int2float_rn(acc[1]), __fmul_rn(ws.y, p.act_step));
    o.z = __fmul_rn(__int2float_rn(acc[2]), __fmul_rn(ws.z, p.act_step));
    o.w = __fmul_rn(__int2float_rn(acc[3]), __fmul_rn(ws.w, p.act_step));
    reinterpret_cast<float4*>(p.out + (size_t)n * p.ld_out)[q] = o;
    if (p.acc) reinterpret_cast<int4*>(p.acc + (size_t)n * p.ld_out)[q] = make_int4(acc[0], acc[1], acc[2], acc[3]);
}

// kS = 1, 2: 3 x 3 filters of that stride, strips of `strip` output rows; kS = 0: any filter, one output per item.
// kAcc: the sums are wanted too (their addresses take registers that the strips need: 5 % of the time).  kRing: input rows through
// a ring of the thread's own words.
template <int kS, bool kAcc, bool kRing>
__global__ void __launch_bounds__(kDwThreads, kS ? 2 : 4) depthwise_kernel(const Problem given, const int strip)
{
    extern __shared__ uint32_t s_w[];                     // [tap][quad]: channel 4q+j in byte j
    pdl_wait();
    Problem p = given;
    p.act = pdl_ordered(p.act); p.wstep = pdl_ordered(p.wstep);
    const int taps = p.kh * p.kw, C = p.M;
    // (the other form's blocks stay for its whole time: placed early, the next launch's crowd together where these leave
    // first; 960 channels, 64 images of 28 x 28, stride 3 56.4 us with the trigger, 49.7 without)
    if (kS != 0) pdl_trigger();
    {
        uint8_t* s_b = reinterpret_cast<uint8_t*>(s_w);
        for (int c = threadIdx.x; c < C; c += kDwThreads) {
            const int kind = p.kind[c], slot = p.slot[c];
            const uint8_t* r8 = p.q8 + (kind == kFixed8 ? (size_t)(slot - p.nP - p.nF4) * p.Kp : 0);
            const uint8_t* r4 = p.q4 + (size_t)slot * (p.Kp >> 1);
            for (int tap = 0; tap < taps; ++tap)
                s_b[tap * C + c] = (uint8_t)(kind == kFixed8 ? (int)(int8_t)r8[tap * p.Cp] : decode4(r4, tap * p.Cp, kind));
        }
    }
    __syncthreads();
    const int quads = C >> 2;
    // thread <-> (item of the block's current group, channel quad): the split is fixed per thread, the item
    // index advances by whole groups, and all index arithmetic is 32-bit (the host checks the counts)
    const int qpt = (quads + kDwThreads - 1) / kDwThreads;             // quads per thread when an item has more quads than threads
    const int lanes_q = min(quads, kDwThreads);                        // threads that share an item
    const int ipg = kDwThreads / lanes_q;                              // items per group
    const int my_i = threadIdx.x / lanes_q, my_q0 = threadIdx.x - my_i * lanes_q;
    if (my_i >= ipg) return;
    if constexpr (kS != 0) {
        const uint32_t ncol = (uint32_t)(p.Wo + kDwCols - 1) / kDwCols, nstrip = (uint32_t)(p.Ho + strip - 1) / (uint32_t)strip;
        const uint32_t n_items = (uint32_t)p.B * nstrip * ncol;
        constexpr int kXW = 3 * kS + 3;                                // input columns under four outputs
        const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_w) + (uint32_t)((taps * C + 15) & ~15) + 4u * threadIdx.x;
        for (int qi = 0; qi < qpt; ++qi) {
            const int q = my_q0 + qi * lanes_q;
            if (q >= quads) break;
            uint32_t f[3][4];                                          // kernel row, channel: taps in bytes 0..2
#pragma unroll
            for (int i = 0; i < 3; ++i) dw_transpose(s_w[(3 * i) * quads + q], s_w[(3 * i + 1) * quads + q], s_w[(3 * i + 2) * quads + q], 0u, f[i]);
            const float4 ws = __ldg(reinterpret_cast<const float4*>(p.wstep) + q);
            const float sc[4] = {__fmul_rn(ws.x, p.act_step), __fmul_rn(ws.y, p.act_step), __fmul_rn(ws.z, p.act_step), __fmul_rn(ws.w, p.act_step)};
            for (uint32_t item = blockIdx.x * (uint32_t)ipg + my_i; item < n_items; item += gridDim.x * (uint32_t)ipg) {
                const uint32_t sb = item / ncol;                       // image * strips + strip
                const int wo0 = (int)(item - sb * ncol) * kDwCols;
                const uint32_t b = sb / nstrip;
                const int ho0 = (int)(sb - b * nstrip) * strip;
                const int rows = min(strip, p.Ho - ho0), cols = min(kDwCols, p.Wo - wo0);
                const int x0 = wo0 * kS - p.pad;
                const int8_t* src = p.act + (size_t)b * p.H * p.W * p.pix_pitch + (int64_t)x0 * p.pix_pitch + 4 * q;
                const uint32_t pitch = (uint32_t)p.pix_pitch;
                const int64_t row_pitch = (int64_t)p.W * p.pix_pitch;
                uint32_t in_x = 0;                                     // which of the columns lie inside the image
#pragma unroll
                for (int x = 0; x < kXW; ++x) in_x |= ((unsigned)(x0 + x) < (unsigned)p.W ? 1u : 0u) << x;
                // behind the last input row of the strip; 0 where the whole strip lies in the padding above the image, so
                // that the one unsigned comparison in load() and fetch() rules out rows in front of the image too
                const int y_end = max(0, min(p.H, (ho0 + rows - 1) * kS - p.pad + 3));
                auto load = [&](int y, uint32_t (&a)[kXW]) {           // rows and columns outside the image read as zero
                    const int8_t* r = src + (int64_t)y * row_pitch;
                    if ((unsigned)y >= (unsigned)y_end) {
#pragma unroll
                        for (int x = 0; x < kXW; ++x) a[x] = 0u;
                    } else if (in_x == (1u << kXW) - 1u) {             // the usual case, without a predicate per column
#pragma unroll
                        for (int x = 0; x < kXW; ++x) a[x] = __ldg(reinterpret_cast<const uint32_t*>(r + (uint32_t)x * pitch));
                    } else {
#pragma unroll
                        for (int x = 0; x < kXW; ++x) a[x] = ((in_x >> x) & 1u) ? __ldg(reinterpret_cast<const uint32_t*>(r + (uint32_t)x * pitch)) : 0u;
                    }
                };
                int y = ho0 * kS - p.pad;                              // the input row to load next
                // kRing: that row on its way to the thread's own words of the ring; rows and columns outside the image become zeros.
                uint32_t put = ring, got = ring;                       // where it goes, and where the next one to be used lies
                auto fetch = [&]() {
                    const int8_t* r = src + (int64_t)y * row_pitch;
                    if ((unsigned)y >= (unsigned)y_end) {
#pragma unroll
                        for (int x = 0; x < kXW; ++x) dw_copy(put + x * kDwRingColumn, p.act, 0u);
                    } else if (in_x == (1u << kXW) - 1u) {
#pragma unroll
                        for (int x = 0; x < kXW; ++x) dw_copy(put + x * kDwRingColumn, r + (uint32_t)x * pitch, 4u);
                    } else {
#pragma unroll
                        for (int x = 0; x < kXW; ++x) dw_copy(put + x * kDwRingColumn, (in_x >> x) & 1u ? r + (uint32_t)x * pitch : p.act, (in_x >> x) & 1u ? 4u : 0u);
                    }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                    ++y;
                    put = put == ring + (kDwAhead * kXW) * kDwRingColumn ? ring : put + kXW * kDwRingColumn;
                };
                // The row fetched kDwAhead rows ago; the place of the one used before it is free for the next.
                auto take = [&](uint32_t (&a)[kXW]) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(kDwAhead - 1) : "memory");
#pragma unroll
                    for (int x = 0; x < kXW; ++x) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(a[x]) : "r"(got + x * kDwRingColumn) : "memory");
                    got = got == ring + (kDwAhead * kXW) * kDwRingColumn ? ring : got + kXW * kDwRingColumn;
                    fetch();
                };
                float* out = p.out + ((size_t)b * p.Ho * p.Wo + (size_t)ho0 * p.Wo + wo0) * p.ld_out + 4 * q;
                int32_t* const acc_out = kAcc ? p.acc + (out - p.out) : nullptr;
                const uint32_t ld = (uint32_t)p.ld_out;
                const size_t row_out = (size_t)p.Wo * p.ld_out;
                // one output row from the three arranged input rows under it
                auto emit = [&](int h, const DwRow<kS>& r0, const DwRow<kS>& r1, const DwRow<kS>& r2) {
                    float* o = out + (size_t)h * row_out;
#pragma unroll
                    for (int j = 0; j < kDwCols; ++j) {
                        int acc[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            acc[c] = __dp4a((int)dw_word(r2, c, j), (int)f[2][c], __dp4a((int)dw_word(r1, c, j), (int)f[1][c], __dp4a((int)dw_word(r0, c, j), (int)f[0][c], kDwMagicBits)));
                        if (j < cols) {
                            *reinterpret_cast<float4*>(o + (uint32_t)j * ld) =
                                make_float4(__fmul_rn(__fsub_rn(__int_as_float(acc[0]), kDwMagic), sc[0]), __fmul_rn(__fsub_rn(__int_as_float(acc[1]), kDwMagic), sc[1]),
                                            __fmul_rn(__fsub_rn(__int_as_float(acc[2]), kDwMagic), sc[2]), __fmul_rn(__fsub_rn(__int_as_float(acc[3]), kDwMagic), sc[3]));
                            if (kAcc)
                                *reinterpret_cast<int4*>(acc_out + (size_t)h * row_out + (uint32_t)j * ld) =
                                    make_int4(acc[0] - kDwMagicBits, acc[1] - kDwMagicBits, acc[2] - kDwMagicBits, acc[3] - kDwMagicBits);
                        }
                    }
                };
                DwRow<kS> r[3];
                uint32_t a[kXW];
                if constexpr (kRing) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");           // (what the last item fetched behind its end: zeros)
#pragma unroll
                    for (int i = 0; i < kDwAhead; ++i) fetch();
                    take(a); dw_arrange<kS>(a, r[0]);
                    if constexpr (kS == 1) {
                        take(a); dw_arrange<kS>(a, r[1]);
                        for (int h = 0; h < rows; h += 3) {
                            // three output rows a turn, so that the rows' places in r[] are fixed
                            take(a); dw_arrange<kS>(a, r[2]); emit(h, r[0], r[1], r[2]);
                            if (h + 1 < rows) { take(a); dw_arrange<kS>(a, r[0]); emit(h + 1, r[1], r[2], r[0]); }
                            if (h + 2 < rows) { take(a); dw_arrange<kS>(a, r[1]); emit(h + 2, r[2], r[0], r[1]); }
                        }
                    } else {
                        for (int h = 0; h < rows; h += 2) {            // r[0] and r[2] take turns as the shared row
                            take(a); dw_arrange<kS>(a, r[1]); take(a); dw_arrange<kS>(a, r[2]); emit(h, r[0], r[1], r[2]);
                            if (h + 1 < rows) { take(a); dw_arrange<kS>(a, r[1]); take(a); dw_arrange<kS>(a, r[0]); emit(h + 1, r[2], r[1], r[0]); }
                        }
                    }
                } else if constexpr (kS == 1) {
                    uint32_t nx[kXW];
                    load(y, a);
                    load(y + 1, nx);
                    dw_arrange<1>(a, r[0]);
                    load(y + 2, a);
                    dw_arrange<1>(nx, r[1]);
                    y += 3;
                    for (int h = 0; h < rows; h += 3) {                // a row's words are loaded while the row in front of it is worked on
                        load(y, nx); dw_arrange<1>(a, r[2]); emit(h, r[0], r[1], r[2]);
                        if (h + 1 < rows) { load(y + 1, a); dw_arrange<1>(nx, r[0]); emit(h + 1, r[1], r[2], r[0]); }
                        if (h + 2 < rows) { load(y + 2, nx); dw_arrange<1>(a, r[1]); emit(h + 2, r[2], r[0], r[1]); }
#pragma unroll
                        for (int x = 0; x < kXW; ++x) a[x] = nx[x];
                        y += 3;
                    }
                } else {
                    uint32_t nx[kXW];
                    load(y, a);
                    load(y + 1, nx);
                    dw_arrange<2>(a, r[0]);
                    load(y + 2, a);
                    y += 3;
                    for (int h = 0; h < rows; h += 2) {                // r[0] and r[2] take turns as the shared row
                        dw_arrange<2>(nx, r[1]); load(y, nx); dw_arrange<2>(a, r[2]); load(y + 1, a); emit(h, r[0], r[1], r[2]);
                        if (h + 1 < rows) { dw_arrange<2>(nx, r[1]); load(y + 2, nx); dw_arrange<2>(a, r[0]); load(y + 3, a); emit(h + 1, r[2], r[1], r[0]); }
                        y += 4;
                    }
                }
            }
        }
        if constexpr (kRing) asm volatile("cp.async.wait_group 0;" ::: "memory");      // (the block's shared memory is its own until it ends)
        return;
    } else {
    const uint32_t N = (uint32_t)p.N, hw = (uint32_t)(p.Ho * p.Wo);
    for (uint32_t n = blockIdx.x * (uint32_t)ipg + my_i; n < N; n += gridDim.x * (uint32_t)ipg) {
        const uint32_t b = n / hw, r = n - b * hw;
        const int ho = (int)(r / (uint32_t)p.Wo), wo = (int)(r - (uint32_t)ho * p.Wo);
        const int8_t* img = p.act + (size_t)b * p.H * p.W * p.pix_pitch;
        for (int qi = 0; qi < qpt; ++qi) {
            const int q = my_q0 + qi * lanes_q;
            if (q >= quads) break;
            int acc[4] = {0, 0, 0, 0};
            for (int i = 0; i < p.kh; ++i) {
                const int y = ho * p.stride + i - p.pad;
                if (y < 0 || y >= p.H) continue;
                for (int j = 0; j < p.kw; ++j) {
                    const int x = wo * p.stride + j - p.pad;
                    if (x < 0 || x >= p.W) continue;
                    const uint32_t a4 = __ldg(reinterpret_cast<const uint32_t*>(img + (size_t)(y * p.W + x) * p.pix_pitch) + q);
                    const int w = (int)s_w[(i * p.kw + j) * quads + q];
                    acc[0] = __dp4a((int)(a4 & 0x000000FFu), w, acc[0]);
                    acc[1] = __dp4a((int)(a4 & 0x0000FF00u), w, acc[1]);
                    acc[2] = __dp4a((int)(a4 & 0x00FF0000u), w, acc[2]);
                    acc[3] = __dp4a((int)(a4 & 0xFF000000u), w, acc[3]);
                }
            }
            dw_store(p, n, q, acc);
        }
    }
    }
}

}  // namespace

// Channels a multiple of 4, the expanded filter table within shared memory, 32-bit pixel counts.
bool depthwise_supported(const Problem& p)
{
    return p.Cin == 1 && (p.M & 3) == 0 && (size_t)p.kh * p.kw * p.M <= 200 * 1024 && (p.pix_pitch & 3) == 0 && (p.ld_out & 3) == 0 &&
           p.N < (int64_t)1 << 31;
}

cudaError_t launch_depthwise(const Problem& p, cudaStream_t st)
{
    const size_t table = (size_t)p.kh * p.kw * p.M, with_ring = ((table + 15) & ~(size_t)15) + dw_ring(p.stride);
    const int variant = (p.kh == 3 && p.kw == 3 && (p.stride == 1 || p.stride == 2)) ? p.stride : 0;
    const bool acc = variant != 0 && p.acc;
    static bool attr_set[5][2][kMaxDevices] = {};
    typedef void (*Kernel)(const Problem, const int);
    Kernel kernel = variant == 1 ? (acc ? depthwise_kernel<1, true, false> : depthwise_kernel<1, false, false>)
                  : variant == 2 ? (acc ? depthwise_kernel<2, true, false> : depthwise_kernel<2, false, false>)
                                 : depthwise_kernel<0, false, false>;
    if (table > 48 * 1024 && !ensure_smem_attr(reinterpret_cast<const void*>(kernel), (int)kDwSmem, attr_set[variant][acc])) return cudaErrorUnknown;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, reinterpret_cast<const void*>(kernel), kDwThreads, table);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int quads = p.M >> 2;
    const int ipg = kDwThreads / std::min(quads, kDwThreads);          // items a block takes per pass
    const int64_t cap = (int64_t)sm_count() * per_sm;
    int strip = 1;
    int64_t blocks;
    if (variant) {
        // Height of a strip: a tall one arranges fewer input rows twice, a short one gives more strips to share out
        // (an item costs about its rows plus one row's worth of start-up and rows shared with its neighbours).
        const int64_t per_row = (int64_t)p.B * ((p.Wo + kDwCols - 1) / kDwCols);
        int64_t best = INT64_MAX;
        for (int n = 1; n <= p.Ho; n += 1 + n / 4) {
            const int s = (p.Ho + n - 1) / n;
            const int64_t groups = (per_row * ((p.Ho + s - 1) / s) + ipg - 1) / ipg;
            const int64_t cost = ((groups + cap - 1) / cap) * (2 * s + 3);
            if (cost < best) { best = cost; strip = s; }
        }
        blocks = (per_row * ((p.Ho + strip - 1) / strip) + ipg - 1) / ipg;
    } else {
        // at least four passes per block, so that expanding the filter table stays a small part of its work
        blocks = ((p.N + ipg - 1) / ipg + 3) / 4;
        // whole rounds of the SMs (5 x 5, 32 channels, 64 images of 28 x 28: 392 blocks 34 to 43 us, 444 30)
        const int64_t sms = sm_count();
        if (blocks > sms) blocks = (blocks + sms - 1) / sms * sms;
    }
    const int64_t rounds = (blocks + cap - 1) / cap;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    // Tall strips through the ring, where as many blocks fit beside each other with it; of stride two, whose rows are nine words, where a
    // quarter of a block's threads has no item and a thread with one walks seven rows and more.  (Launches back to back, registers against ring: 576 channels, 64 images of 14 x 14, strips of 14
    // rows 24.8 us and 21.2; 192, 64 of 56 x 56, 19 rows 48.4 and 44.9; 192, 64 of 28 x 28, 10 rows 17.0 and 16.6; 384, 64 of 14 x 14, 7 rows 14.8
    // and 14.7; 960, 64 of 7 x 7, 4 rows 20.2 and 20.7; 144, 8 of 56 x 56, 4 rows 9.4 and 10.2.  With sums 192, 64 of 56 x 56 72.7 and 76.2.  Stride two:
    // 576, 64 of 28 x 28, 14 rows, 144 threads 34.5 and 28.9; 384, 64 of 28 x 28, 7 rows, 192 threads 21.4 and 20.4; 576, 64 of 14 x 14, 4 rows 17.1 and 17.6,
    // 43 of 30 x 30, 5 rows twice 29.5 and 25.8; 516, 9 of 43 x 43, 6 rows 17.1 and 17.8; 192, 64 of 56 x 56, 10 rows, 240 threads 25.3 and 26.4.)
    const bool tall = variant == 1 ? strip >= 10 : variant == 2 && strip * rounds >= 7 && 4 * ipg * std::min(quads, kDwThreads) <= 3 * kDwThreads;
    if (tall && !acc && with_ring <= kDwSmem && (with_ring + 1024) * (size_t)per_sm <= 228 * 1024) {
        const Kernel ringed = variant == 1 ? depthwise_kernel<1, false, true> : depthwise_kernel<2, false, true>;
        if (with_ring > 48 * 1024 && !ensure_smem_attr(reinterpret_cast<const void*>(ringed), (int)kDwSmem, attr_set[2 + variant][0])) return cudaErrorUnknown;
        return launch_dependent(ringed, (unsigned)blocks, kDwThreads, with_ring, st, p, strip);
    }
    return launch_dependent(kernel, (unsigned)blocks, kDwThreads, table, st, p, strip);
}

}  // namespace rmsmp
