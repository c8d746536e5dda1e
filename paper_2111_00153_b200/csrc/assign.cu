// Row assignment on the device (Section 3.1: lower variance -> PoT; Section 3.3: ratio A:B:C; Algorithm 1's
// assignment block) and the packed buffer's metadata built from it, so that a layer can be quantized and
// packed from nothing but its fp32 weights and the ratio.
//
// The ranking key is (population variance in double, summed in reduction order; row index).  Adding in
// reduction order is one dependent chain of 2 K double additions per row (55 us at K = 576, 450 us at K = 4608
// when every row walked its own), but the assignment needs no more than who is below the two cuts of the
// ranking.  So:
//   row_stats_kernel   one block per row, one pass over the weights: the variance summed in parallel, a bound
//                      on how far it can be from the definition's value, and max |w|.
//   assign_kernel      one block (and some that help): finds the two cuts by a radix selection over the parallel
//                      variances; a row whose interval reaches across a cut (in practice: rows that are copies
//                      of one another) is undecided and gets the definition's chain of additions; a second
//                      selection finds the cuts among the undecided rows, and of those at a cut's very key the
//                      first by row index lie in front (all-zero rows: 70 % of 65,536 1.0 ms; every undecided
//                      row compared with every other was 268 ms).  Then the kind of every row, the stable
//                      grouping by prefix sums in original order, and every metadata section of the packed buffer.
//   assign_small_kernel  the same for up to 4096 rows that the parallel variances decide, up to eight rows a thread: each cut
//                      is a threshold found by bisection, one counting barrier a step, and nothing goes through
//                      memory between the statistics and the metadata (64 to 512 rows 9 us -> 4).  Otherwise it leaves the
//                      layer to assign_kernel's code.
// The result is the definition's in every case.
#include <type_traits>
#include "common.cuh"

namespace rmsmp {

namespace {

constexpr int kStatThreads = 128;
constexpr int kAssignThreads = 1024;
constexpr int kSmallThreads = 512;                        // assign_small_kernel's most
constexpr int kAssignMaxBlocks = 65536 / kBlockRows;      // the entry point takes at most 65536 rows
constexpr int kAssignSmemRows = 2048;                     // rows whose statistics are kept in shared memory

struct RowStats {             // scratch, 16 bytes per row
    double* var;              // parallel variance; the exact one once an undecided row has been resolved
    float* err;               // |var - definition's variance| <= err; 0: var is exact
    float* amax;              // max |w|, 1 for an all-zero row
};

// The definition's variance: two plain passes in reduction order, every operation rounded on its own.
__device__ __noinline__ double exact_variance(const float* __restrict__ w, int K)
{
    double mean = 0.0, acc = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        acc = 0.0;
        auto add = [&](float v) {
            if (pass == 0) {
                acc = __dadd_rn(acc, (double)v);
            } else {
                const double d = __dsub_rn((double)v, mean);
                acc = __dadd_rn(acc, __dmul_rn(d, d));
            }
        };
        if ((K & 3) == 0) {
            const float4* w4 = reinterpret_cast<const float4*>(w);
            float4 v = __ldg(w4);
            for (int i = 0; i < (K >> 2); ++i) {
                const float4 nx = __ldg(w4 + min(i + 1, (K >> 2) - 1));
                add(v.x); add(v.y); add(v.z); add(v.w);
                v = nx;
            }
        } else {
            for (int i = 0; i < K; ++i) add(__ldg(w + i));
        }
        if (pass == 0) mean = acc / (double)K;
    }
    return acc / (double)K;
}

// One pass with the row's first weight as the origin: x = w - c, s1 = sum x, s2 = sum x^2, variance
// (s2 - s1^2 / K) / K.  With u = 2^-53 and q = s2 / K, any order of additions leaves |error| <= 4 (K + 8) u q
// (|s1| sum|x| <= K s2), and the definition's own two passes are off by at most (K + 4) u var + 2 ((K + 1) u A)^2
// with A = mean |w|, A^2 <= 2 (c^2 + q); G = 2 (K + 16) u below leaves a factor of more than two.
// A row whose bound says nothing -- it leaves the range of fp32 (weights of 1e25 and more), or is as large as the variance
// (weights all the same: the definition's variance is rounding noise) -- gets the definition's chain here, where every SM
// has rows to work on.
__global__ void __launch_bounds__(kStatThreads) row_stats_kernel(const float* __restrict__ W, int K, RowStats out)
{
    pdl_wait();
    pdl_trigger();
    W = pdl_ordered(W);
    __shared__ double s_red[2][kStatThreads / 32];
    __shared__ float s_max[kStatThreads / 32];
    const int row = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* w = W + (size_t)row * K;
    const double c = (double)__ldg(w);
    double s1 = 0.0, s2 = 0.0;
    float mx = 0.0f;
    auto add = [&](float v) {
        const double x = (double)v - c;
        s1 += x;
        s2 = __fma_rn(x, x, s2);
        mx = fmaxf(mx, fabsf(v));
    };
    if ((K & 3) == 0) {
        const int n4 = K >> 2;
        for (int i = threadIdx.x; i < n4; i += 4 * kStatThreads) {
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i + j * kStatThreads < n4) v[j] = __ldg(reinterpret_cast<const float4*>(w) + i + j * kStatThreads);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i + j * kStatThreads < n4) { add(v[j].x); add(v[j].y); add(v[j].z); add(v[j].w); }
        }
    } else {
        for (int i = threadIdx.x; i < K; i += kStatThreads) add(__ldg(w + i));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) { s_red[0][warp] = s1; s_red[1][warp] = s2; s_max[warp] = mx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kStatThreads / 32; ++i) { s1 += s_red[0][i]; s2 += s_red[1][i]; mx = fmaxf(mx, s_max[i]); }
        const double q = s2 / (double)K, G = (double)(K + 16) * 2.220446049250313e-16;      // 2^-52
        double v = fabs(fmax((s2 - s1 * s1 / (double)K) / (double)K, 0.0));
        float e = __double2float_ru(6.0 * G * q + 4.0 * G * G * (c * c + q));
        if (mx == 0.0f) { v = 0.0; e = 0.0f; }                     // an all-zero row's variance is exactly zero
        if (!(e <= 3e38f) || (e > 0.0f && (double)e >= v)) { v = exact_variance(w, K); e = 0.0f; }
        if (!(v <= 1e300)) { v = __longlong_as_double(0x7FF0000000000000ll); e = 0.0f; }     // not finite: last, by row index
        out.var[row] = v;
        out.err[row] = e;
        out.amax[row] = (mx == 0.0f) ? 1.0f : mx;
    }
}

struct MetaArgs {
    const float* W;
    uint8_t* blob;
    RowStats st;
    const float* alpha;       // per row: the caller's, or the max |w| found by row_stats_kernel
    uint8_t* scheme_out;      // optional
    uint8_t* bits_out;        // optional
    uint64_t off_perm, off_slot, off_wstep, off_alpha, off_kind, off_blocks;
    int M, K, Cin, kh, kw, Cp, Kp, nP, nF4, n8, nblocks, pot_mode;
};

__device__ __forceinline__ void write_header(const MetaArgs& a)
{
    BlobHeader* H = reinterpret_cast<BlobHeader*>(a.blob);
    H->magic = kLayerMagic; H->version = kBlobVersion;
    H->M = a.M; H->Cin = a.Cin; H->kh = a.kh; H->kw = a.kw; H->Cp = a.Cp; H->Kp = a.Kp;
    H->nP = a.nP; H->nF4 = a.nF4; H->n8 = a.n8; H->nblocks = a.nblocks; H->pot_mode = a.pot_mode;
    H->pad0[0] = H->pad0[1] = H->pad0[2] = 0;
    H->status = 0;
}

// N values reduced over the block, for every thread (s: N * 32 entries; id: the operation's identity).
template <int N, typename T, typename Op>
__device__ __forceinline__ void block_reduce(T (&v)[N], Op op, T* s, T id)
{
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] = op(v[i], __shfl_xor_sync(0xffffffffu, v[i], o));
    __syncthreads();                                      // the previous use of `s` is over
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) s[32 * i + (threadIdx.x >> 5)] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = (threadIdx.x & 31) < (blockDim.x >> 5) ? s[32 * i + (threadIdx.x & 31)] : id;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] = op(v[i], __shfl_xor_sync(0xffffffffu, v[i], o));
    }
}

// Share `rank` of `ranks` of the listed rows' variances by the definition; neighbouring rows go to different blocks and warps.
__device__ __forceinline__ void exact_variances(const MetaArgs& a, const int32_t* list, int n, int rank, int ranks)
{
    const int nt = blockDim.x, u = (threadIdx.x & 31) * (nt >> 5) + (threadIdx.x >> 5);
    for (int i = u * ranks + rank; i < n; i += nt * ranks) {
        const int r = list[i];
        if (a.st.err[r] != 0.0f) a.st.var[r] = exact_variance(a.W + (size_t)r * a.K, a.K);
    }
}

// assign_kernel is a cluster of kHelpers blocks, of which the first assigns.  The others sleep at the cluster's barrier until it
// knows how many undecided rows need the definition's chain of additions, take their share and leave: copies of four rows,
// 65,536 of 1024 weights 9.6 ms on one SM, 2.1 ms so; random weights no slower.  For up to 4096 rows there are no helpers:
// the cluster costs random weights 1 us of 26 to 32, and copies of four rows take 118 to 745 us without them (226 with three).
constexpr int kHelpers = 8;
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// What a block other than the first does.  s_rows: its own word, which the first block fills.
__device__ __forceinline__ void help(const MetaArgs& a, int* s_rows)
{
    if (threadIdx.x == 0) *s_rows = 0;
    cluster_arrive();                                     // (1) this block runs and its word is clear
    cluster_wait();
    cluster_arrive();                                     // (2) the first block knows the number of rows
    cluster_wait();
    const int n = *reinterpret_cast<volatile int*>(s_rows);
    if (n > 0) {
        exact_variances(a, reinterpret_cast<const int32_t*>(a.blob + a.off_slot), n, (int)blockIdx.x, kHelpers);
        cluster_arrive();                                 // (3) this share is done
    }
}

// The first block's side: n listed rows' variances.
__device__ __forceinline__ void exact_variances_with_helpers(const MetaArgs& a, int* s_rows, const int32_t* list, int n)
{
    cluster_wait();                                       // (1)
    if (n > 0 && threadIdx.x > 0 && threadIdx.x < kHelpers) {
        uint32_t at;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(s_rows)), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(at), "r"(n) : "memory");
    }
    cluster_arrive();                                     // (2)
    if (n == 0) return;
    cluster_wait();
    exact_variances(a, list, n, 0, kHelpers);
    cluster_arrive();                                     // (3)
    cluster_wait();
}

// One block: everything here is latency (a few barriers per step), so the statistics are copied to shared memory
// first and the selection starts at the first bit in which the variances differ at all (their exponents mostly
// agree): two or three digits for random weights instead of eight.
// kBlocks: the blocks that share the chains of additions, s_rows the helpers' word (see help()).
template <int kBlocks>
__device__ __forceinline__ void assign_rows_block(const MetaArgs& a, int* s_rows)
{
    __shared__ int s_hist[2][256];
    __shared__ unsigned long long s_prefix[2];
    __shared__ int s_left[2], s_same[2];
    __shared__ double s_dbl[4 * 32];
    __shared__ unsigned long long s_u64[4 * 32];
    __shared__ int s_int[4 * 32];
    __shared__ int s_undecided;
    __shared__ int s_warp[3][32];
    __shared__ int s_start[3][kAssignMaxBlocks + 1];      // rows of each kind in front of every 128-row block
    __shared__ double s_var[kAssignSmemRows];
    __shared__ float s_err[kAssignSmemRows];
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5;      // (128 threads or more)
    const int M = a.M;
    const bool local = M <= kAssignSmemRows;
    double* const var = local ? s_var : a.st.var;
    float* const err = local ? s_err : a.st.err;
    uint8_t* kind = a.blob + a.off_kind;
    int32_t* perm = reinterpret_cast<int32_t*>(a.blob + a.off_perm);
    int32_t* slot = reinterpret_cast<int32_t*>(a.blob + a.off_slot);
    const int cut[2] = {a.nP, M - a.n8};                  // rows in front of each cut of the ranking
    bool need[2];
    for (int c = 0; c < 2; ++c) need[c] = cut[c] > 0 && cut[c] < M && (c == 0 || cut[1] != cut[0]);

    // ---- the statistics in shared memory
    if (local) {
        for (int r = t; r < M; r += nt) { s_var[r] = a.st.var[r]; s_err[r] = a.st.err[r]; }
    }
    if (t == 0) s_undecided = 0;
    __syncthreads();

    // For each cut c with open[c]: the key of the want[c]-th of the rows that in(c, r) names (s_prefix), how many of the rows
    // with that key are among those want[c] (s_left), and how many there are (s_same).  Radix selection, up to eight bits
    // at a time, from the first bit in which the keys differ at all: two or three digits for random weights (their
    // exponents mostly agree), none where all keys are the same.  (A non-negative double orders like its bits.)
    // all_rows: in() is true everywhere; one histogram does for both cuts while they are in the same bin then.  Otherwise the rows
    // are those at a cut, many of which tie: a warp counts the digit of the first of its rows in one addition (20,000 rows
    // of random weights 7 % slower so, copies of four rows twice as fast).
    auto select = [&](auto all_rows, auto in, const bool (&open)[2], const int (&want)[2]) {
        constexpr bool kAll = decltype(all_rows)::value;
        unsigned long long bits[4] = {0ull, 0ull, 0ull, 0ull};         // per cut: bits set in a key, bits clear in a key
        for (int r = t; r < M; r += nt) {
            const unsigned long long key = (unsigned long long)__double_as_longlong(var[r]);
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (open[c] && in(c, r)) { bits[2 * c] |= key; bits[2 * c + 1] |= ~key; }
        }
        for (int i = t; i < 256; i += nt) { s_hist[0][i] = 0; s_hist[1][i] = 0; }
        block_reduce<4>(bits, [](unsigned long long x, unsigned long long y) { return x | y; }, s_u64, 0ull);
        int top = 64 - __clzll((long long)((bits[0] & bits[1]) | (bits[2] & bits[3])));      // bits from `top` up are common to a cut's keys
        if (t < 2) {
            s_prefix[t] = top < 64 ? (t == 0 ? bits[0] : bits[2]) & (~0ull << top) : 0ull;
            s_left[t] = t == 0 ? want[0] : want[1];
            s_same[t] = M;                                // (counted below)
        }
        __syncthreads();
        if (top == 0) {                                   // one key a cut
            int n[2] = {0, 0};
            for (int r = t; r < M; r += nt) { n[0] += open[0] && in(0, r); n[1] += open[1] && in(1, r); }
            block_reduce<2>(n, [](int x, int y) { return x + y; }, s_int, 0);
            if (t < 2) s_same[t] = t == 0 ? n[0] : n[1];
            __syncthreads();
        }
        while (top > 0) {
            const int shift = max(top - 8, 0);
            const unsigned long long above = top < 64 ? ~0ull << top : 0ull;
            const unsigned long long pre[2] = {s_prefix[0], s_prefix[1]};
            const bool one = kAll && pre[0] == pre[1] && open[0] && open[1];
            if (kAll) {
                for (int r = t; r < M; r += nt) {
                    const unsigned long long key = (unsigned long long)__double_as_longlong(var[r]);
                    const int d = (int)((key & ~above) >> shift);
                    if (open[0] && (key & above) == pre[0]) atomicAdd(&s_hist[0][d], 1);
                    if (open[1] && !one && (key & above) == pre[1]) atomicAdd(&s_hist[1][d], 1);
                }
            }
            for (int r0 = kAll ? M : t - lane; r0 < M; r0 += nt) {
                const int r = r0 + lane;
                const unsigned long long key = r < M ? (unsigned long long)__double_as_longlong(var[r]) : 0ull;
                const int d = (int)((key & ~above) >> shift);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (!open[c]) continue;
                    // (rows that tie share their digits: the first row's digit is counted once for the warp)
                    const bool on = r < M && (key & above) == pre[c] && in(c, r);
                    const unsigned m = __ballot_sync(0xffffffffu, on);
                    if (m == 0u) continue;
                    const int lead = __ffs((int)m) - 1, d0 = __shfl_sync(0xffffffffu, d, lead);
                    const unsigned same = __ballot_sync(0xffffffffu, on && d == d0);
                    if (lane == lead) atomicAdd(&s_hist[c][d0], __popc(same));
                    else if (on && d != d0) atomicAdd(&s_hist[c][d], 1);
                }
            }
            __syncthreads();
            if (warp < 2 && (warp == 0 ? open[0] : open[1])) {
                // the digit in which the cut's last row lies: a warp scans the 256 counters, eight to a lane
                const int* h = s_hist[one ? 0 : warp];
                int n[8], sum = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) { n[j] = h[8 * lane + j]; sum += n[j]; }
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
                int before = incl - sum;
                const int left = s_left[warp];
                __syncwarp();
                if (before < left && left <= incl) {
                    int j = 0;
                    while (before + n[j] < left) before += n[j++];
                    s_left[warp] = left - before;
                    s_same[warp] = n[j];
                    s_prefix[warp] |= (unsigned long long)(8 * lane + j) << shift;
                }
            }
            __syncthreads();
            top = shift;
            if (top > 0 && (!open[0] || s_same[0] == 1) && (!open[1] || s_same[1] == 1)) {
                // one row left at each cut: its key is the rest of the digits
                const unsigned long long known = ~0ull << shift, k0 = s_prefix[0], k1 = s_prefix[1];
                __syncthreads();
                for (int r = t; r < M; r += nt) {
                    const unsigned long long key = (unsigned long long)__double_as_longlong(var[r]);
                    if (open[0] && (key & known) == k0 && in(0, r)) s_prefix[0] = key;
                    if (open[1] && (key & known) == k1 && in(1, r)) s_prefix[1] = key;
                }
                __syncthreads();
                break;
            }
            for (int i = t; i < 256; i += nt) { s_hist[0][i] = 0; s_hist[1][i] = 0; }
            __syncthreads();
        }
    };

    // ---- the largest key in front of each cut
    select(std::true_type{}, [](int, int) { return true; }, need, cut);
    if (cut[1] == cut[0] && t == 0) { s_prefix[1] = s_prefix[0]; s_left[1] = s_left[0]; s_same[1] = s_same[0]; }
    __syncthreads();

    // ---- which side of each cut: rows that may lie on either are listed (in the slot section, free until the end)
    double key_at[2], edge[4];
    bool tie[2];
    for (int c = 0; c < 2; ++c) {
        key_at[c] = __longlong_as_double((long long)s_prefix[c]);
        tie[c] = s_same[c] > s_left[c];                   // more rows share the last key than fit in front of the cut
        double lo = -1.0, hi = -__longlong_as_double(0x7FF0000000000000ll);
        if (cut[c] > 0 && cut[c] < M) {
            for (int r = t; r < M; r += nt) {
                const double v = var[r], e = (double)err[r];
                if (v <= key_at[c]) lo = fmax(lo, v + e);
                if (v > key_at[c] || (tie[c] && v == key_at[c])) hi = fmax(hi, e - v);
            }
        }
        edge[2 * c] = lo; edge[2 * c + 1] = hi;
    }
    block_reduce<4>(edge, [](double x, double y) { return fmax(x, y); }, s_dbl, -__longlong_as_double(0x7FF0000000000000ll));
    // 0: in front of the cut, 1: behind it, 2: undecided
    auto side = [&](int c, double v, double e) -> int {
        if (cut[c] <= 0) return 1;
        if (cut[c] >= M) return 0;
        const double hi_edge = edge[2 * c], lo_edge = -edge[2 * c + 1];      // the rows in front reach up to, the rows behind down to here
        const bool clear = !tie[c] && hi_edge < lo_edge;
        if (v <= key_at[c]) return (clear || (!(tie[c] && v == key_at[c]) && v + e < lo_edge)) ? 0 : 2;
        return (clear || v - e > hi_edge) ? 1 : 2;
    };
    int in_front[2] = {0, 0};
    for (int r = t; r < M; r += nt) {
        const double v = var[r], e = (double)err[r];
        const int s0 = side(0, v, e), s1 = side(1, v, e);
        in_front[0] += s0 == 0; in_front[1] += s1 == 0;
        kind[r] = (uint8_t)(s0 | s1 << 2);                // the two sides; turned into the kind below
        if (s0 == 2 || s1 == 2) slot[atomicAdd(&s_undecided, 1)] = r;
    }
    __syncthreads();
    const int nu = s_undecided;
    // Undecided rows by the exact key: in front of a cut are those below und_key and the first und_left (by row index) of
    // those at it.
    unsigned long long und_key[2] = {0ull, 0ull};
    int und_left[2] = {0, 0}, und_n[2] = {0, 0};
    if (kBlocks > 1) exact_variances_with_helpers(a, s_rows, slot, nu);
    if (nu > 0) {
        if (kBlocks == 1) {
            exact_variances(a, slot, nu, 0, 1);
            __syncthreads();
        }
        if (local) {
            for (int i = t; i < nu; i += nt) s_var[slot[i]] = __ldcg(a.st.var + slot[i]);
        }
        auto undecided = [&](int c, int r) { return ((kind[r] >> (2 * c)) & 3) == 2; };
        int n[4] = {in_front[0], in_front[1], 0, 0};
        for (int i = t; i < nu; i += nt) { n[2] += undecided(0, slot[i]); n[3] += undecided(1, slot[i]); }
        block_reduce<4>(n, [](int x, int y) { return x + y; }, s_int, 0);      // (and the exact variances are there)
        const int want[2] = {cut[0] - n[0], cut[1] - n[1]};
        const bool open[2] = {want[0] > 0 && want[0] < n[2], want[1] > 0 && want[1] < n[3]};
        select(std::false_type{}, undecided, open, want);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            und_n[c] = n[2 + c];
            und_key[c] = open[c] ? s_prefix[c] : (want[c] > 0 ? ~0ull : 0ull);
            und_left[c] = open[c] ? s_left[c] : 0;
        }
    }
    // the side of an undecided row; `at` counts the rows at a cut's key as they come
    auto decide = [&](int c, int s, int r, int (&at)[2]) -> int {
        if (s != 2) return s;
        const unsigned long long key = (unsigned long long)__double_as_longlong(var[r]);
        if (key != und_key[c]) return key < und_key[c] ? 0 : 1;
        return at[c]++ < und_left[c] ? 0 : 1;
    };

    // ---- stable grouping: consecutive rows per thread, prefix sums over the threads
    const int per = (M + nt - 1) / nt;
    const int r0 = min(M, t * per), r1 = min(M, r0 + per);
    int at[2] = {0, 0};                                   // undecided rows at each cut's key in front of this thread's
    if (nu > 0) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (und_n[c] == 0) continue;                  // (the same for every thread)
            int n = 0;
            for (int r = r0; r < r1; ++r)
                n += ((kind[r] >> (2 * c)) & 3) == 2 && (unsigned long long)__double_as_longlong(var[r]) == und_key[c];
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
            if (lane == 31) s_warp[c][warp] = incl;
            __syncthreads();
            int before = lane < warp ? s_warp[c][lane] : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
            at[c] = before + incl - n;
        }
        __syncthreads();
    }
    int cnt[3] = {0, 0, 0};
    for (int r = r0; r < r1; ++r) {
        const int s = kind[r];
        const int s0 = decide(0, s & 3, r, at), s1 = decide(1, (s >> 2) & 3, r, at);
        const int k = s0 == 0 ? kPoT4 : (s1 == 0 ? kFixed4 : kFixed8);
        kind[r] = (uint8_t)k;
        cnt[0] += k == 0; cnt[1] += k == 1; cnt[2] += k == 2;
    }
    int next[3];                                          // position inside each group
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int incl = cnt[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) s_warp[k][warp] = incl;
        next[k] = incl - cnt[k];
    }
    __syncthreads();
    if (warp < 3) {
        const int v = lane < (nt >> 5) ? s_warp[warp][lane] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += u; }
        s_warp[warp][lane] = incl - v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; ++k) next[k] += s_warp[k][warp];

    float* wstep = reinterpret_cast<float*>(a.blob + a.off_wstep);
    float* alpha = reinterpret_cast<float*>(a.blob + a.off_alpha);
    const int base[3] = {0, a.nP, a.nP + a.nF4};
    for (int r = r0; r < r1; ++r) {
        if ((r & (kBlockRows - 1)) == 0)
            for (int k = 0; k < 3; ++k) s_start[k][r / kBlockRows] = next[k];
        const int k = kind[r];
        const int p = (k == 0 ? base[0] + next[0]++ : (k == 1 ? base[1] + next[1]++ : base[2] + next[2]++));
        perm[p] = r;
        slot[r] = p;
        const float al = a.alpha[r];
        alpha[r] = al;
        wstep[r] = __fdiv_rn(al, k == kPoT4 ? 64.0f : (k == kFixed4 ? 7.0f : 127.0f));
        if (a.scheme_out) a.scheme_out[r] = (k == kPoT4) ? RMSMP_SCHEME_POT : RMSMP_SCHEME_FIXED;
        if (a.bits_out) a.bits_out[r] = (k == kFixed8) ? 8 : 4;
    }
    if (t == 0) { s_start[0][a.nblocks] = a.nP; s_start[1][a.nblocks] = a.nF4; s_start[2][a.nblocks] = a.n8; }
    __syncthreads();
    // block table: first position (inside its group) and count of each kind among the block's 128 rows
    int32_t* blocks = reinterpret_cast<int32_t*>(a.blob + a.off_blocks);
    for (int i = t; i < 8 * a.nblocks; i += nt) {
        const int b = i >> 3, j = i & 7, k = j >> 1;
        int v = 0;
        if (k < 3) {
            const int n = s_start[k][b + 1] - s_start[k][b];
            v = (j & 1) ? n : (n ? s_start[k][b] : 0);
        }
        blocks[i] = v;
    }
    if (t == 0) write_header(a);
}

__global__ void __launch_bounds__(kAssignThreads, 1) assign_kernel(MetaArgs a)
{
    __shared__ int s_rows;
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x > 0) { help(a, &s_rows); return; }
    cluster_arrive();                                     // (1)
    assign_rows_block<kHelpers>(a, &s_rows);
}

// Up to kSmallThreads * R rows, R of them per thread (row i * threads + t); 128 threads or more, so that the other form can take over.
template <int R>
__global__ void __launch_bounds__(kSmallThreads) assign_small_kernel(MetaArgs a)
{
    __shared__ uint32_t s_red[4][32];
    __shared__ uint32_t s_sum[3];
    __shared__ int s_cnt[3][16 * R + 1];                  // rows of each kind in every 32 rows, then in front of them
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5, warps = nt >> 5;
    const int M = a.M;
    const int cut[2] = {a.nP, M - a.n8};
    pdl_wait();
    pdl_trigger();
    bool row[R];
    double v[R];
    float err[R], al[R];
    unsigned long long key[R];                            // a non-negative double orders like its bits
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = i * nt + t;
        row[i] = r < M;
        v[i] = row[i] ? a.st.var[r] : 0.0;
        err[i] = row[i] ? a.st.err[r] : 0.0f;
        al[i] = row[i] ? a.alpha[r] : 1.0f;
        key[i] = row[i] ? (unsigned long long)__double_as_longlong(v[i]) : ~0ull;      // (never below a threshold)
    }
    // four values reduced over the block (maxima; a minimum is the maximum of the complement)
    auto block_max4 = [&](uint32_t (&x)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __reduce_max_sync(0xffffffffu, x[i]);
        __syncthreads();
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i) s_red[i][warp] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __reduce_max_sync(0xffffffffu, lane < warps ? s_red[i][lane] : 0u);
    };
    uint32_t range[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < R; ++i)
        if (row[i]) { range[0] = max(range[0], (uint32_t)(key[i] >> 32)); range[1] = max(range[1], ~(uint32_t)(key[i] >> 32)); }
    block_max4(range);
    const unsigned long long key_lo = (unsigned long long)(~range[1]) << 32, key_hi = ((unsigned long long)range[0] + 1ull) << 32;

    // ---- a threshold for each cut with exactly the rows in front of it below (rows of equal variance at a cut: none)
    unsigned long long lo[2], hi[2], th[2];
    bool found[2];
    for (int c = 0; c < 2; ++c) {
        lo[c] = key_lo; hi[c] = key_hi;
        th[c] = cut[c] <= 0 ? 0ull : key_hi;
        found[c] = cut[c] <= 0 || cut[c] >= M;
    }
    // One barrier a step for both cuts: the two counts travel in one word that the warps add to (ballots and a shared
    // atomic: a warp-wide sum instruction takes as long as the rest of the step).  Three words take turns: a step adds to
    // one, the one in front of it is being read, the one behind is cleared.
    if (t < 3) s_sum[t] = 0u;
    __syncthreads();
    for (int step = 0;; step = step == 2 ? 0 : step + 1) {
        bool open[2];
        unsigned long long mid[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            open[c] = !found[c] && hi[c] - lo[c] > 1;
            mid[c] = lo[c] + ((hi[c] - lo[c]) >> 1);
        }
        if (!open[0] && !open[1]) break;                  // (the same for every thread)
        uint32_t n = 0;
#pragma unroll
        for (int i = 0; i < R; ++i)
            n += (uint32_t)__popc(__ballot_sync(0xffffffffu, key[i] < mid[0])) + ((uint32_t)__popc(__ballot_sync(0xffffffffu, key[i] < mid[1])) << 16);
        if (lane == 0 && n) atomicAdd(&s_sum[step], n);
        if (t == 0) s_sum[step == 2 ? 0 : step + 1] = 0u;
        __syncthreads();
        n = *reinterpret_cast<volatile uint32_t*>(&s_sum[step]);
        const int below[2] = {(int)(n & 0xFFFFu), (int)(n >> 16)};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (!open[c]) continue;
            if (below[c] == cut[c]) { found[c] = true; th[c] = mid[c]; }
            else if (below[c] < cut[c]) lo[c] = mid[c];
            else hi[c] = mid[c];
        }
    }
    // ---- do the variances' error bounds leave both cuts clear?  (in fp32, rounded outwards)
    uint32_t edge[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < R; ++i) {
        if (!row[i]) continue;
        const uint32_t up = __float_as_uint(__double2float_ru(v[i] + (double)err[i]));
        const uint32_t down = ~__float_as_uint(__double2float_rd(fmax(v[i] - (double)err[i], 0.0)));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (key[i] < th[c]) edge[2 * c] = max(edge[2 * c], up); else edge[2 * c + 1] = max(edge[2 * c + 1], down);
        }
    }
    __syncwarp();
    block_max4(edge);
    const bool clear0 = cut[0] <= 0 || cut[0] >= M || (found[0] && edge[0] < ~edge[1]);
    const bool clear1 = cut[1] <= 0 || cut[1] >= M || (found[1] && edge[2] < ~edge[3]);
    if (!clear0 || !clear1) {
        assign_rows_block<1>(a, nullptr);
        return;
    }

    // ---- kinds, stable grouping, metadata
    int kind[R];
    uint32_t mask[R][3];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        kind[i] = key[i] < th[0] ? kPoT4 : (key[i] < th[1] ? kFixed4 : kFixed8);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mask[i][k] = __ballot_sync(0xffffffffu, row[i] && kind[i] == k);
            if (lane == 0) s_cnt[k][i * warps + warp] = __popc(mask[i][k]);
        }
    }
    __syncthreads();
    const int groups = (M + 31) >> 5;                     // of 32 rows
    if (warp < 3) {
        // counts to exclusive prefix sums: a warp per kind, R / 2 (or one) consecutive groups a lane
        constexpr int kPer = (16 * R + 31) / 32;
        int n[kPer], sum = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int g = lane * kPer + j;
            n[j] = g < groups ? s_cnt[warp][g] : 0;
            sum += n[j];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += u; }
        int before = incl - sum;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int g = lane * kPer + j;
            if (g <= groups && g <= 16 * R) s_cnt[warp][g] = before;
            before += n[j];
        }
        if (lane == 31 && groups == 32 * kPer) s_cnt[warp][groups] = before;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int g = i * warps + warp, r = i * nt + t, k = kind[i];
        if (!row[i]) continue;
        const int p = s_cnt[k][g] + (k == 0 ? 0 : (k == 1 ? a.nP : a.nP + a.nF4)) +
                      __popc((k == 0 ? mask[i][0] : (k == 1 ? mask[i][1] : mask[i][2])) & ((1u << lane) - 1u));
        reinterpret_cast<int32_t*>(a.blob + a.off_perm)[p] = r;
        reinterpret_cast<int32_t*>(a.blob + a.off_slot)[r] = p;
        (a.blob + a.off_kind)[r] = (uint8_t)k;
        reinterpret_cast<float*>(a.blob + a.off_alpha)[r] = al[i];
        reinterpret_cast<float*>(a.blob + a.off_wstep)[r] = __fdiv_rn(al[i], k == kPoT4 ? 64.0f : (k == kFixed4 ? 7.0f : 127.0f));
        if (a.scheme_out) a.scheme_out[r] = (k == kPoT4) ? RMSMP_SCHEME_POT : RMSMP_SCHEME_FIXED;
        if (a.bits_out) a.bits_out[r] = (k == kFixed8) ? 8 : 4;
    }
    // block table: first position (inside its group) and count of each kind among the block's 128 rows
    for (int i = t; i < 8 * a.nblocks; i += nt) {
        const int g = (i >> 3) * 4, j = i & 7, k = j >> 1;
        int out = 0;
        if (k < 3) {
            const int first = s_cnt[k][g], n = s_cnt[k][min(g + 4, groups)] - first;
            out = (j & 1) ? n : (n ? first : 0);
        }
        reinterpret_cast<int32_t*>(a.blob + a.off_blocks)[i] = out;
    }
    if (t == 0) write_header(a);
}

}  // namespace

size_t assign_scratch_bytes(int M) { return ((size_t)M * (8 + 4 + 4) + 255) / 256 * 256; }

cudaError_t launch_assign_meta(const float* dW, const rmsmp_layer& L, const float* d_alpha, int pot_mode, uint8_t* blob,
                               void* d_scratch, uint8_t* d_scheme, uint8_t* d_bits, cudaStream_t st)
{
    const int M = L.M, K = L.Cin * L.kh * L.kw;
    RowStats rs;
    rs.var = static_cast<double*>(d_scratch);
    rs.err = reinterpret_cast<float*>(rs.var + M);
    rs.amax = rs.err + M;
    cudaError_t e = launch_dependent(row_stats_kernel, (unsigned)M, kStatThreads, 0, st, dW, K, rs);
    if (e != cudaSuccess) return e;
    MetaArgs a;
    a.W = dW; a.K = K; a.st = rs;
    a.blob = blob; a.alpha = d_alpha ? d_alpha : rs.amax; a.scheme_out = d_scheme; a.bits_out = d_bits;
    a.off_perm = L.off_perm; a.off_slot = L.off_slot; a.off_wstep = L.off_wstep; a.off_alpha = L.off_alpha;
    a.off_kind = L.off_kind; a.off_blocks = L.off_blocks;
    a.M = M; a.Cin = L.Cin; a.kh = L.kh; a.kw = L.kw; a.Cp = L.Cp; a.Kp = L.Kp;
    a.nP = L.nP; a.nF4 = L.nF4; a.n8 = L.n8; a.nblocks = L.nblocks; a.pot_mode = pot_mode;
    // few warps: cheap barriers, and a block that finds room on an SM while the statistics still run
    if (M > 8 * kSmallThreads) return launch_dependent_cluster(assign_kernel, kHelpers, kHelpers, kAssignThreads, 0, st, a);
    if (M > 2 * kSmallThreads) return launch_dependent(assign_small_kernel<8>, 1, kSmallThreads, 0, st, a);
    if (M > kSmallThreads) return launch_dependent(assign_small_kernel<2>, 1, kSmallThreads, 0, st, a);
    return launch_dependent(assign_small_kernel<1>, 1, (unsigned)(M <= 128 ? 128 : (M + 31) / 32 * 32), 0, st, a);
}

}  // namespace rmsmp
