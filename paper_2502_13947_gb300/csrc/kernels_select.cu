// kernels_select.cu -- control parameters, subQUBO selection and the
// mutation operator (Section 3).
//
//  k_sizes   uneven subQUBO sizes m_k = m_min + (Philox(k, TAG_SIZE, p, iter) mod span)
//            and their exclusive prefix (group offsets), one CTA.
//  k_select  one CTA per replica: Delta (Eq. 7) from the Tabu toggle counts,
//            A = w1 eta + w2 gamma - w3 Delta (Algorithm 3, Q16, floor), a
//            stable radix sort of the variables by A descending in shared
//            memory (which leaves equal A in index order), the S' mask, and one
//            more stable pass over the variables in index order by their group,
//            so that every group comes out in ascending index order
//            (Algorithm 4's subset choice).  In the learned mode S' comes from
//            a second sort by the network's score; the selection hit counts H
//            are incremented for S'.
//  k_mutate  one CTA per replica: the first L = floor((n - |S'|) r) ranked
//            variables outside S' are candidates; candidate i flips iff its
//            Philox word is below floor((A_i - A_min)(2^32 - 1)/(A_max - A_min)).
//            Flips go to the replica's flip list for k_apply.
#include <climits>

#include "common.cuh"

namespace icd2s {

namespace {

__device__ __forceinline__ long long floor_div_65536(long long v)
{
    return v >= 0 ? v / 65536 : -((-v + 65535) / 65536);
}

// ---- stable block radix sort (1024 threads) ----
// Items are taken in order, warp w the w-th run of `per` (a multiple of 32).  A pass
// by a digit of up to 8 bits counts each warp's digits, turns the counts
// [warp][digit] into start positions (all of a smaller digit first, then the same
// digit of earlier warps), and places the items 32 at a time: lanes of one digit
// (match_any) take consecutive positions, which keeps the order of equal digits.
//
// Against the bitonic sort of 64-bit keys that this replaces (78 to 105 barrier-separated
// steps over the next power of two), a sort is two to four passes of three
// barriers: only the bits in which the keys differ are sorted by.  k_select, 32
// solutions of n = 10 000: 207 -> 42 us; 256 solutions of n = 7000: 299 -> 88 us.
constexpr int kSortThreads = 1024, kSortWarps = kSortThreads / 32, kBins = 256;

// Rank pass: item q (0 <= q < count) has the digit dig(q) < kBins; put(q, position) places it.
template <class Dig, class Put>
__device__ __forceinline__ void stable_pass(int count, int* hist, int* part, Dig dig, Put put)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = ((count + kSortWarps - 1) / kSortWarps + 31) & ~31;
    const int lo = min(count, warp * per), hi = min(count, lo + per);
    int* const mine = hist + warp * kBins;
    for (int b = tid; b < kSortWarps * kBins; b += kSortThreads) hist[b] = 0;
    __syncthreads();
    for (int q = lo + lane; q < hi; q += 32) atomicAdd(&mine[dig(q)], 1);
    __syncthreads();
    // start positions: thread b scans digit b over the warps, then the digits' totals are scanned
    int total = 0;
    if (tid < kBins) {
#pragma unroll 8
        for (int w = 0; w < kSortWarps; ++w) {
            const int v = hist[w * kBins + tid];
            hist[w * kBins + tid] = total;
            total += v;
        }
        int incl = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) part[warp] = incl;
        total = incl - total;   // exclusive within the warp
    }
    __syncthreads();
    if (tid < kBins) {
        for (int w = 0; w < warp; ++w) total += part[w];
        part[kSortWarps + tid] = total;
    }
    __syncthreads();
    const int* const first = part + kSortWarps;
    for (int q0 = lo; q0 < hi; q0 += 32) {
        const int q = q0 + lane;
        const bool on = q < hi;
        const int d = on ? dig(q) : kBins;   // idle lanes: a digit of their own
        const unsigned same = __match_any_sync(0xffffffffu, d);
        int base = 0;
        if (on) base = mine[d];
        __syncwarp();
        const unsigned before = same & ((1u << lane) - 1u);
        if (on && before == 0u) mine[d] = base + __popc(same);
        __syncwarp();
        if (on) put(q, first[d] + base + __popc(before));
    }
    __syncthreads();
}

// Sorts the variables 0 .. n - 1 by key ascending (equal keys in index order) into
// ord; tmp is scratch.  kmin, kmax: the keys' range.
__device__ __forceinline__ void radix_sort(const unsigned* key, unsigned kmin, unsigned kmax, int n, uint16_t* ord,
                                           uint16_t* tmp, int* hist, int* part)
{
    const int bits = kmax == kmin ? 0 : 32 - __clz(kmax - kmin);
    const int passes = (bits + 7) / 8;
    for (int j = threadIdx.x; j < n; j += kSortThreads) (passes & 1 ? tmp : ord)[j] = (uint16_t)j;
    __syncthreads();
    const int width = passes ? (bits + passes - 1) / passes : 0;
    for (int k = 0; k < passes; ++k) {
        const uint16_t* from = ((passes - k) & 1) ? tmp : ord;
        uint16_t* to = ((passes - k) & 1) ? ord : tmp;
        const int sh = k * width;
        const unsigned mask = (1u << width) - 1u;
        stable_pass(n, hist, part, [&](int q) { return (int)(((key[from[q]] - kmin) >> sh) & mask); },
                    [&](int q, int pos) { to[pos] = from[q]; });
    }
}

__device__ __forceinline__ int block_reduce_max(int v, int* red)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        int w = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : INT_MIN;
        w = __reduce_max_sync(0xffffffffu, w);
        if (threadIdx.x == 0) red[32] = w;
    }
    __syncthreads();
    const int r = red[32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ int block_reduce_min(int v, int* red)
{
    return -block_reduce_max(-v, red);  // |A| < 2^30, negation is safe
}

// exclusive prefix sum of v over the block's 1024 threads; *total receives the sum
__device__ __forceinline__ int block_scan(int v, int* red, int* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) red[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = red[lane];
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        red[lane] = wi - w;
        if (lane == 31) red[32] = wi;
    }
    __syncthreads();
    const int r = red[warp] + incl - v;
    *total = red[32];
    __syncthreads();
    return r;
}

}  // namespace

// ---------------------------------------------------------------------------
// Also writes, when `order` is given, the subQUBOs in largest-first order
// (a counting sort by size; the order among equal sizes is immaterial) for
// the persistent anneal kernels, and the parts of it that are their size
// classes (queue: next [kAnnealClasses], end [kAnnealClasses]).
__global__ __launch_bounds__(1024) void k_sizes(int R, int K, int m_min, int m_max, uint32_t k0, uint32_t k1,
                                                uint32_t iter_arg, const int32_t* iter_dev, int32_t* off,
                                                int32_t* order, int32_t* queue, int p0)
{
    __shared__ int red[33];
    __shared__ int start[1024];   // (kMaxM + 2 used)
    const uint32_t iter = iter_dev ? (uint32_t)*iter_dev : iter_arg;
    const int total = R * K;
    const int NT = blockDim.x, tid = threadIdx.x;
    const int chunk = (total + NT - 1) / NT;
    const int lo = tid * chunk, hi = min(total, lo + chunk);
    const uint32_t span = (uint32_t)(m_max - m_min + 1);
    auto size_of = [&](int s) -> int {
        if (m_max == m_min) return m_min;
        const int p = p0 + s / K, k = s % K;   // the global replica
        const u32x4 w = philox10((uint32_t)k, kTagSize << 24, (uint32_t)p, iter, k0, k1);
        return m_min + (int)(w.v[0] % span);
    };
    int sum = 0;
    for (int s = lo; s < hi; ++s) sum += size_of(s);
    int all = 0;
    int run = block_scan(sum, red, &all);
    for (int s = lo; s < hi; ++s) { off[s] = run; run += size_of(s); }
    if (hi == total && lo < hi) off[total] = run;
    if (total == 0 && tid == 0) off[0] = 0;
    if (!order) return;
    start[tid] = 0;
    __syncthreads();
    // sizes descending: slot kMaxM - m counts the size m, so that the scan gives the
    // number of larger subQUBOs
    for (int s = lo; s < hi; ++s) atomicAdd(&start[kMaxM - size_of(s)], 1);
    __syncthreads();
    const int first = block_scan(start[tid], red, &all);
    start[tid] = first;
    __syncthreads();
    // the classes' parts of the order: class c ends where sizes up to its lower bound begin
    if (tid < kAnnealClasses) {
        constexpr int kAbove[kAnnealClasses + 1] = {kMaxM, kAnnealBound[1], kAnnealBound[2], kAnnealBound[3], 0};
        int at[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int v = 0;
#pragma unroll
            for (int c = 0; c <= kAnnealClasses; ++c) v = c == tid + q ? kAbove[c] : v;
            at[q] = v == 0 ? total : start[kMaxM - v];   // subQUBOs larger than v
        }
        queue[tid] = at[0];
        queue[kAnnealClasses + tid] = at[1];
    }
    __syncthreads();
    for (int s = lo; s < hi; ++s) order[atomicAdd(&start[kMaxM - size_of(s)], 1)] = s;
}

cudaError_t launch_sizes(int R, int K, int m_min, int m_max, uint32_t k0, uint32_t k1, uint32_t iter,
                         const int32_t* iter_dev, int32_t* off, int32_t* order, int32_t* queue, cudaStream_t s,
                         int p0)
{
    k_sizes<<<1, 1024, 0, s>>>(R, K, m_min, m_max, k0, k1, iter, iter_dev, off, order, queue, p0);
    note_launch(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
__global__ __launch_bounds__(1024) void k_select(Dev d, int64_t w1, int64_t w2, int64_t w3, int K,
                                                 const int32_t* __restrict__ off, int32_t* __restrict__ idx, int mode,
                                                 int32_t* __restrict__ H, uint32_t iter_arg, const int32_t* iter_dev,
                                                 int ablation)
{
    const uint32_t iter = iter_dev ? (uint32_t)*iter_dev : iter_arg;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int red[33];
    __shared__ int goff[65];
    __shared__ int part[kSortWarps + kBins];
    const int p = blockIdx.x, tid = threadIdx.x, NT = blockDim.x;
    const int n = d.n, ld = d.ld;
    int* hist = reinterpret_cast<int*>(smem);                               // [kSortWarps][kBins]
    unsigned* keys = reinterpret_cast<unsigned*>(hist + kSortWarps * kBins);  // [ld], by variable
    uint16_t* ord = reinterpret_cast<uint16_t*>(keys + ld);                 // [ld]
    uint16_t* tmp = ord + ld;                                               // [ld]
    uint8_t* grp = reinterpret_cast<uint8_t*>(tmp);                         // [ld] groups (after the sorts)
    const int32_t* Trow = d.T + (size_t)p * ld;
    int32_t* Arow = d.A + (size_t)p * ld;
    int32_t* Drow = d.delta + (size_t)p * ld;

    int mt = 0;
    for (int j = tid; j < n; j += NT) mt = max(mt, Trow[j]);
    mt = block_reduce_max(mt, red);

    // ascending keys, and their range (as signed numbers: the top bit flipped)
    int kmin = INT_MAX, kmax = INT_MIN;
    for (int j = tid; j < ld; j += NT) {
        if (j < n) {
            const int t = Trow[j];
            const int dl = mt > 0 ? (int)(((long long)(mt - t) * 65536) / mt) : 0;
            const long long v = w1 * (long long)d.etahat[j] + w2 * (long long)d.gamma[j] - w3 * (long long)dl;
            const int a = ablation == 2   // No_SM: a random ranking key instead of A
                              ? (int)(philox10((uint32_t)(j >> 2), kTagRank << 24, (uint32_t)(d.p0 + p), iter, d.k0,
                                               d.k1).v[j & 3] >> 1)
                              : (int)floor_div_65536(v);
            Arow[j] = a;
            Drow[j] = dl;
            keys[j] = ~((unsigned)a ^ 0x80000000u);
            kmin = min(kmin, ~a);
            kmax = max(kmax, ~a);
        } else {
            Arow[j] = 0;
            Drow[j] = 0;
        }
    }
    auto range = [&](unsigned& lo, unsigned& hi) {   // of the block's keys, from the threads' kmin, kmax
        hi = (unsigned)block_reduce_max(kmax, red) ^ 0x80000000u;
        lo = (unsigned)~block_reduce_max(~kmin, red) ^ 0x80000000u;
    };
    unsigned klo, khi;
    range(klo, khi);
    radix_sort(keys, klo, khi, n, ord, tmp, hist, part);

    int32_t* orow = d.order + (size_t)p * ld;
    uint8_t* srow = d.sel + (size_t)p * ld;
    for (int r = tid; r < ld; r += NT) {
        orow[r] = r < n ? (int32_t)ord[r] : 0;
        srow[r] = 0;
    }
    // Learned selection: S' ranked by (score desc, index asc) instead; the A
    // ranking above still orders the mutation candidates.  The score's bit
    // pattern maps to a signed integer with the float's order (-0 below +0).
    if (mode == 1 || (mode == 2 && (p & 1) == 0)) {
        __syncthreads();
        const float* sc = d.score + (size_t)p * ld;
        kmin = INT_MAX;
        kmax = INT_MIN;
        for (int j = tid; j < n; j += NT) {
            const unsigned b = __float_as_uint(sc[j]);
            const int a = b < 0x80000000u ? (int)b : -(int)(b & 0x7fffffffu) - 1;
            keys[j] = ~((unsigned)a ^ 0x80000000u);
            kmin = min(kmin, ~a);
            kmax = max(kmax, ~a);
        }
        range(klo, khi);
        radix_sort(keys, klo, khi, n, ord, tmp, hist, part);
    }
    const int base = off[p * K];
    if (tid <= K) goff[tid] = off[p * K + tid] - base;
    __syncthreads();
    const int M = goff[K];
    // group of every variable (K: none), then the groups' lists in index order
    for (int j = tid; j < n; j += NT) grp[j] = (uint8_t)K;
    __syncthreads();
    for (int r = tid; r < M; r += NT) {
        const int i = ord[r];
        int g = 0;
        while (g + 1 < K && goff[g + 1] <= r) ++g;
        grp[i] = (uint8_t)g;
        srow[i] = 1;
        if (H) H[(size_t)p * ld + i] += 1;
    }
    __syncthreads();
    stable_pass(n, hist, part, [&](int q) { return (int)grp[q]; },
                [&](int q, int pos) { if (pos < M) idx[base + pos] = q; });
}

cudaError_t launch_select(const Dev& d, int64_t w1, int64_t w2, int64_t w3, int K, const int32_t* off,
                          int32_t* idx, int mode, bool count_hits, cudaStream_t s, uint32_t iter,
                          const int32_t* iter_dev, int ablation)
{
    const size_t sm = sizeof(int) * kSortWarps * kBins + 8 * (size_t)d.ld;   // 32 KiB + 8 bytes per variable
    cudaError_t e = cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_select<<<d.R, 1024, sm, s>>>(d, w1, w2, w3, K, off, idx, mode, count_hits ? d.H : nullptr, iter, iter_dev,
                                   ablation);
    note_launch(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
__global__ __launch_bounds__(1024) void k_mutate(Dev d, int K, const int32_t* __restrict__ off, double rate_arg,
                                                 uint32_t iter_arg, const int32_t* iter_dev, const double* rates,
                                                 uint8_t* mask, int ldm, int half)
{
    __shared__ int red[33];
    __shared__ int wsum[32];
    const uint32_t iter = iter_dev ? (uint32_t)*iter_dev : iter_arg;
    const double rate = iter_dev ? rates[iter] : rate_arg;
    const int p = blockIdx.x, tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int n = d.n, ld = d.ld;
    const int32_t* Arow = d.A + (size_t)p * ld;
    const int32_t* orow = d.order + (size_t)p * ld;
    const uint8_t* srow = d.sel + (size_t)p * ld;
    const uint8_t* xrow = d.X + (size_t)p * ld;
    const int M = off[(p + 1) * K] - off[p * K];
    const int L = (int)floor((double)(n - M) * rate);
    if (L <= 0) return;

    int amin = INT_MAX, amax = INT_MIN;
    for (int j = tid; j < n; j += NT) { const int a = Arow[j]; amin = min(amin, a); amax = max(amax, a); }
    amin = block_reduce_min(amin, red);
    amax = block_reduce_max(amax, red);

    int taken = 0;  // candidates found before this chunk (uniform)
    for (int r0 = 0; r0 < n && taken < L; r0 += NT) {
        const int r = r0 + tid;
        int i = -1;
        bool pred = false;
        if (r < n) { i = orow[r]; pred = srow[i] == 0; }
        const unsigned bal = __ballot_sync(0xffffffffu, pred);
        if (lane == 0) wsum[warp] = __popc(bal);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < (NT >> 5); ++w) { const int v = wsum[w]; before += w < warp ? v : 0; total += v; }
        const int rank = taken + before + __popc(bal & ((1u << lane) - 1u));
        if (pred && rank < L) {
            unsigned long long P;
            if (amax == amin || half) P = 2147483648ull;
            else P = ((unsigned long long)((long long)Arow[i] - amin) * 4294967295ull) /
                     (unsigned long long)((long long)amax - amin);
            const u32x4 w = philox10((uint32_t)(i >> 2), kTagMut << 24, (uint32_t)(d.p0 + p), iter, d.k0, d.k1);
            if ((unsigned long long)w.v[i & 3] < P) {
                const int slot = atomicAdd(&d.FCNT[p], 1);
                if (slot < ld) d.FL[(size_t)p * ld + slot] = i | (int)((unsigned)xrow[i] << 31);
                if (mask) mask[(size_t)p * ldm + i] = 1;
            }
        }
        taken += total;
        __syncthreads();
    }
}

cudaError_t launch_mutate(const Dev& d, int K, const int32_t* off, double rate, uint32_t iter,
                          const int32_t* iter_dev, const double* rates, uint8_t* mask, int ldm, cudaStream_t s,
                          bool half)
{
    k_mutate<<<d.R, 1024, 0, s>>>(d, K, off, rate, iter, iter_dev, rates, mask, ldm, half ? 1 : 0);
    note_launch(1);
    return cudaGetLastError();
}

}  // namespace icd2s
