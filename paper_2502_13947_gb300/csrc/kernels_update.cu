// kernels_update.cu -- write-back of accepted flips into the solutions,
// their exact int32 gains and int64 energies.
//
// For a set F of variables flipped together (old values x_i, d_i = 1 - 2 x_i):
//   h_j  <- h_j + sum_{i in F, i != j} Q_ij d_i         (off-diagonal field)
//   x_j  <- x_j xor [j in F]
//   g_j  <- (1 - 2 x_j)(Q_jj + 2 h_j)
//   E    <- E + (1/2) sum_{i in F} (g_i(old) - g_i(new))
// The last identity follows from applying the flips one after the other:
// the energy change is sum_{i in F} g_i + 2 sum_{pairs {i,i'} in F} Q_ii' d_i d_i',
// and g_i(new) = -g_i(old) - 2 sum_{i' in F, i' != i} Q_ii' d_i d_i'.
// h is recovered from the tracked gain as h_j = ((1 - 2 x_j) g_j - Q_jj) / 2.
//
// k_apply: grid (ld / 2048, R, S), 128 threads, the S CTAs of a tile a thread-block
// cluster.  Each thread owns 16 consecutive columns j of one replica (4 columns
// and 256 threads when the caller's buffers are only 4-byte aligned).  CTA z of a
// cluster takes its share of the replica's flip list (of a short list all, for its
// part of the columns: apply_short), staged in shared memory in
// chunks; for every listed row i the thread streams the 16 bytes Q[i][j..j+15]
// (coalesced 2 KiB per CTA and row -- Q is symmetric, so the row is the column),
// several rows in flight.  Four rows are added at a time: their words are
// transposed bytewise (8 permutations per 4 x 4 bytes), so that one dp4a with the
// four signs d_i adds four entries to a column.  The CTAs then leave their sums in
// shared memory, and after a cluster barrier CTA z finishes its part of the tile's
// columns from all S (distributed shared memory); no partial sums pass through
// global memory, so the caller-owned path splits its lists as well.  S (1, 2, 4,
// 8) is chosen so that about six CTAs per SM run.  Energy terms go to an int64
// accumulator; the last CTA of the replica (ticket counter) folds it into E and
// resets the list, the accumulator and the counters, so the next producer starts
// clean.
//
// What bounds it: HBM for long lists, latency for short ones.
// 16 replicas x 1024 disjoint flips at n = 16 384 (268 MB of rows): 54.7 us with one
// multiply-add and extraction per byte and partial sums in global planes, 50.5 us
// here (5376 GB/s); the whole caller-owned call at n = 15 999 (no splitting before)
// 179 -> 56 us.
#include "common.cuh"

namespace icd2s {

// Two shapes: 16 columns per thread (16-byte loads; rows 16-byte aligned,
// ld % 16 == 0 -- every state the library allocates) and 4 columns per thread
// (4-byte loads; ld % 4 == 0, for caller-owned buffers).
template <int COLS> struct ApplyShape {
    static constexpr int threads = COLS == 16 ? 128 : 256;
    static constexpr int tile = COLS * threads;  // columns per CTA
};
constexpr int kApplyChunk = 2048;  // list entries staged per pass
constexpr int kApplyMaxSplit = 8;  // CTAs per cluster: the portable limit
constexpr int kApplyShort = 64;    // lists up to here are not split (up to a quarter of it in clusters of one or two)

template <int COLS> struct RowLoad;
template <> struct RowLoad<16> {
    static __device__ __forceinline__ void get(const int8_t* p, unsigned (&w)[4])
    {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
};
template <> struct RowLoad<4> {
    static __device__ __forceinline__ void get(const int8_t* p, unsigned (&w)[1])
    {
        w[0] = __ldg(reinterpret_cast<const unsigned*>(p));
    }
};

// acc[c] += d_i Q[i][j0 + c] over the staged rows e0 .. e1 - 1 (both multiples of 4;
// padding entries have sign 0), 4 B rows in flight; the diagonal term Q_jj d_j that a
// flipped j adds to its own sum is taken out when the tile is finished.
template <int COLS, int B>
__device__ __forceinline__ void add_rows(const Dev& d, const int32_t* rows, const unsigned* signs, int j0, int (&acc)[COLS])
{
    constexpr int NW = COLS / 4;
    unsigned rv[4 * B][NW];
#pragma unroll
    for (int q = 0; q < B; ++q) {
        const int4 r4 = reinterpret_cast<const int4*>(rows)[q];
        const int r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) RowLoad<COLS>::get(d.Q + (size_t)r[u] * d.ld + j0, rv[4 * q + u]);
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
        const int sg = (int)signs[q];
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const unsigned t0 = __byte_perm(rv[4 * q][k], rv[4 * q + 1][k], 0x5140u),
                           t1 = __byte_perm(rv[4 * q + 2][k], rv[4 * q + 3][k], 0x5140u),
                           t2 = __byte_perm(rv[4 * q][k], rv[4 * q + 1][k], 0x7362u),
                           t3 = __byte_perm(rv[4 * q + 2][k], rv[4 * q + 3][k], 0x7362u);
            acc[4 * k] = __dp4a((int)__byte_perm(t0, t1, 0x5410u), sg, acc[4 * k]);
            acc[4 * k + 1] = __dp4a((int)__byte_perm(t0, t1, 0x7632u), sg, acc[4 * k + 1]);
            acc[4 * k + 2] = __dp4a((int)__byte_perm(t2, t3, 0x5410u), sg, acc[4 * k + 2]);
            acc[4 * k + 3] = __dp4a((int)__byte_perm(t2, t3, 0x7632u), sg, acc[4 * k + 3]);
        }
    }
}

__device__ __forceinline__ void apply_cluster_barrier()
{
    __syncwarp();   // .aligned: the warp arrives as one, whatever branches came before
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 16 bytes at this CTA's shared-memory address `addr`, read from cluster CTA `rank`
__device__ __forceinline__ int4 cluster_load(uint32_t addr, uint32_t rank)
{
    int4 v;
    asm volatile(
        "{\n\t.reg .u32 ra;\n\t"
        "mapa.shared::cluster.u32 ra, %4, %5;\n\t"
        "ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [ra];\n\t}"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "r"(addr), "r"(rank)
        : "memory");
    return v;
}

// Columns tile0 + c .. + 3 of replica p from their sums, words of X and gains; returns
// their share of 2 (old - new energy).
__device__ __forceinline__ long long finish_columns(const Dev& d, int p, int j, unsigned fbits, const int (&av)[4],
                                                    uint32_t xw, int4 g4)
{
    const int gin[4] = {g4.x, g4.y, g4.z, g4.w};
    int gout[4];
    uint32_t xo = 0u;
    long long dpart = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        int xj = (int)((xw >> (8 * b)) & 1u);
        if (j + b < d.n) {
            const int dj = d.diag[j + b];
            const int fl_j = (int)((fbits >> b) & 1u);
            const int h = ((1 - 2 * xj) * gin[b] - dj) / 2 + av[b] - (fl_j ? (1 - 2 * xj) * dj : 0);
            xj ^= fl_j;
            gout[b] = (1 - 2 * xj) * (dj + 2 * h);
            if (fl_j) dpart += (long long)gin[b] - gout[b];
        } else {  // columns past n: left as they are (padding of caller-owned rows)
            gout[b] = gin[b];
            xj = (int)((xw >> (8 * b)) & 0xffu);
        }
        xo |= (uint32_t)xj << (8 * b);
    }
    *reinterpret_cast<int4*>(d.G + (size_t)p * d.ld + j) = make_int4(gout[0], gout[1], gout[2], gout[3]);
    *reinterpret_cast<uint32_t*>(d.X + (size_t)p * d.ld + j) = xo;
    return dpart;
}

// The CTA's energy term; the last of the replica's `ctas` folds them all into E and clears
// the counters for the next producer.
template <int THREADS>
__device__ __forceinline__ void fold_energy(const Dev& d, int p, unsigned ctas, long long dpart, long long* red)
{
    const int tid = threadIdx.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dpart += __shfl_xor_sync(0xffffffffu, dpart, o);
    if ((tid & 31) == 0) red[tid >> 5] = dpart;
    __syncthreads();
    if (tid == 0) {
        long long tot = 0;
        for (int w = 0; w < THREADS / 32; ++w) tot += red[w];
        if (tot != 0) atomicAdd(&d.DEACC[p], (unsigned long long)tot);
        __threadfence();
        const unsigned ticket = atomicAdd(&d.DONE[p], 1u);
        if (ticket == ctas - 1) {   // (every CTA has read the list and its length)
            __threadfence();
            const long long sum = (long long)atomicExch(&d.DEACC[p], 0ull);
            d.E[p] += sum / 2;
            d.DONE[p] = 0;
            d.FCNT[p] = 0;
        }
    }
}

// The whole of a short list for columns c0 .. c_end - 1 of the tile, four columns per thread,
// from registers: the exchange between a cluster's CTAs, with its two barriers, costs a
// short list more than the split saves.  Compaction and write-back, launches in a graph,
// split against this: n = 300, 8 solutions 8.0 and 6.7 us with 1 flip, 8.6 and 8.1 with 33, 8.68 and 8.71
// with 64; n = 7000, 32 solutions 11.1 and 8.0, 12.8 and 10.4, 13.8 and 11.7.  In clusters of two
// (n = 1000, 512 solutions) 12.2 and 10.5 us with 1 flip, 13.5 and 12.9 with 16, 14.1 and 14.9 with 32.
template <int THREADS, int TILE>
__device__ __forceinline__ void apply_short(const Dev& d, int p, int cnt, int tile0, int c0, int c_end, unsigned ctas,
                                            int32_t* rows, uint8_t* signs, uint32_t* tileflip, long long* red)
{
    const int tid = threadIdx.x, cp = (cnt + 3) & ~3;
    const int32_t* fl = d.FL + (size_t)p * d.ld;
    for (int e = tid; e < cp; e += THREADS) {
        const int v = e < cnt ? fl[e] : 0, i = v & 0x7fffffff;
        rows[e] = i;
        signs[e] = e < cnt ? (v < 0 ? 0xff : 0x01) : 0x00;
        if (e < cnt && i >= tile0 && i < tile0 + TILE)
            atomicOr(&tileflip[(i - tile0) >> 5], 1u << ((i - tile0) & 31));
    }
    __syncthreads();
    const unsigned* sw = reinterpret_cast<const unsigned*>(signs);
    long long dpart = 0;
    for (int c = c0 + 4 * tid; c < c_end; c += 4 * THREADS) {
        const int j = tile0 + c;
        const uint32_t xw = *reinterpret_cast<const uint32_t*>(d.X + (size_t)p * d.ld + j);
        const int4 g4 = *reinterpret_cast<const int4*>(d.G + (size_t)p * d.ld + j);
        int av[4] = {0, 0, 0, 0};
        int e = 0;
        for (; e + 16 <= cp; e += 16) add_rows<4, 4>(d, rows + e, sw + e / 4, j, av);
        for (; e < cp; e += 4) add_rows<4, 1>(d, rows + e, sw + e / 4, j, av);
        dpart += finish_columns(d, p, j, (tileflip[c >> 5] >> (c & 31)) & 15u, av, xw, g4);
    }
    fold_energy<THREADS>(d, p, ctas, dpart, red);
}

// (six CTAs of the 4-column shape per SM: with 48 registers five fit, and 768 CTAs no longer run
// at once: n = 2500, 32 solutions, 300 flips 17.9 against 20.9 us)
template <int COLS>
__global__ __launch_bounds__(ApplyShape<COLS>::threads, COLS == 16 ? 0 : 6) void k_apply(Dev d)
{
    using Shape = ApplyShape<COLS>;
    constexpr int kThreads = Shape::threads, kTile = Shape::tile;
    __shared__ __align__(16) int32_t rows[kApplyChunk];
    __shared__ __align__(16) uint8_t signs[kApplyChunk];
    __shared__ __align__(16) int sums[kTile];
    __shared__ uint32_t tileflip[kTile / 32];
    __shared__ long long red[kThreads / 32];
    const int p = blockIdx.y, tid = threadIdx.x;
    const int ld = d.ld, n = d.n;
    const int S = gridDim.z, z = blockIdx.z;   // the cluster is the whole z extent
    const int cnt = min(d.FCNT[p], ld);  // a list never exceeds n entries
    if (cnt == 0) return;  // nothing to apply for this replica (counters are already clear)
    const int tile0 = blockIdx.x * kTile;
    const int j0 = tile0 + COLS * tid;  // ld % COLS == 0: j0 < ld implies j0 + COLS <= ld
    const int32_t* fl = d.FL + (size_t)p * ld;
    for (int w = tid; w < kTile / 32; w += kThreads) tileflip[w] = 0;
    __syncthreads();
    if (cnt <= (S >= 4 ? kApplyShort : kApplyShort / 4)) {   // (the same in all CTAs of the cluster)
        apply_short<kThreads, kTile>(d, p, cnt, tile0, z * (kTile / S), min((z + 1) * (kTile / S), ld - tile0),
                                     gridDim.x * (unsigned)S, rows, signs, tileflip, red);
        return;
    }
    // the flips that fall in this tile (the whole list)
    for (int e = tid; e < cnt; e += kThreads) {
        const int i = fl[e] & 0x7fffffff;
        if (i >= tile0 && i < tile0 + kTile) atomicOr(&tileflip[(i - tile0) >> 5], 1u << ((i - tile0) & 31));
    }
    int acc[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) acc[c] = 0;
    const int lo = (int)((long long)cnt * z / S), hi = (int)((long long)cnt * (z + 1) / S);
    for (int c0 = lo; c0 < hi; c0 += kApplyChunk) {
        const int cn = min(kApplyChunk, hi - c0), cp = (cn + 3) & ~3;
        __syncthreads();
        for (int e = tid; e < cp; e += kThreads) {
            const int v = e < cn ? fl[c0 + e] : 0;
            rows[e] = v & 0x7fffffff;
            signs[e] = e < cn ? (v < 0 ? 0xff : 0x01) : 0x00;
        }
        __syncthreads();
        if (j0 < ld) {
            constexpr int B = COLS == 16 ? 4 : 8;   // batches of 4 rows in flight
            const unsigned* sw = reinterpret_cast<const unsigned*>(signs);
            int e = 0;
            for (; e + 4 * B <= cp; e += 4 * B) add_rows<COLS, B>(d, rows + e, sw + e / 4, j0, acc);
            for (; e < cp; e += 4) add_rows<COLS, 1>(d, rows + e, sw + e / 4, j0, acc);
        }
    }
#pragma unroll
    for (int c4 = 0; c4 < COLS / 4; ++c4)
        reinterpret_cast<int4*>(sums + COLS * tid)[c4] =
            make_int4(acc[4 * c4], acc[4 * c4 + 1], acc[4 * c4 + 2], acc[4 * c4 + 3]);
    if (S > 1) apply_cluster_barrier();
    else __syncthreads();
    long long dpart = 0;
    const int part = kTile / S;
    for (int c = z * part + 4 * tid; c < (z + 1) * part && tile0 + c < ld; c += 4 * kThreads) {
        const int j = tile0 + c;
        int4 a4 = make_int4(0, 0, 0, 0);
        if (S == 1) {
            a4 = *reinterpret_cast<const int4*>(sums + c);
        } else {
            const uint32_t addr = (uint32_t)__cvta_generic_to_shared(sums + c);
#pragma unroll 4
            for (int q = 0; q < S; ++q) {
                const int4 b4 = cluster_load(addr, (uint32_t)q);
                a4.x += b4.x; a4.y += b4.y; a4.z += b4.z; a4.w += b4.w;
            }
        }
        const int av[4] = {a4.x, a4.y, a4.z, a4.w};
        uint32_t* xp = reinterpret_cast<uint32_t*>(d.X + (size_t)p * ld + j);
        int4* gp = reinterpret_cast<int4*>(d.G + (size_t)p * ld + j);
        const uint32_t xw = *xp;
        const int4 g4 = *gp;
        const int gin[4] = {g4.x, g4.y, g4.z, g4.w};
        int gout[4];
        uint32_t xo = 0u;
        const unsigned fbits = (tileflip[c >> 5] >> (c & 31)) & 15u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int xj = (int)((xw >> (8 * b)) & 1u);
            if (j + b < n) {
                const int dj = d.diag[j + b];
                const int fl_j = (int)((fbits >> b) & 1u);
                const int h = ((1 - 2 * xj) * gin[b] - dj) / 2 + av[b] - (fl_j ? (1 - 2 * xj) * dj : 0);
                xj ^= fl_j;
                gout[b] = (1 - 2 * xj) * (dj + 2 * h);
                if (fl_j) dpart += (long long)gin[b] - gout[b];
            } else {  // columns past n: left as they are (padding of caller-owned rows)
                gout[b] = gin[b];
                xj = (int)((xw >> (8 * b)) & 0xffu);
            }
            xo |= (uint32_t)xj << (8 * b);
        }
        *gp = make_int4(gout[0], gout[1], gout[2], gout[3]);
        *xp = xo;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dpart += __shfl_xor_sync(0xffffffffu, dpart, o);
    if ((tid & 31) == 0) red[tid >> 5] = dpart;
    __syncthreads();
    if (tid == 0) {
        long long tot = 0;
        for (int w = 0; w < kThreads / 32; ++w) tot += red[w];
        if (tot != 0) atomicAdd(&d.DEACC[p], (unsigned long long)tot);
        __threadfence();
        const unsigned ticket = atomicAdd(&d.DONE[p], 1u);
        if (ticket == gridDim.x * (unsigned)S - 1) {   // (every CTA has read the list and its length)
            __threadfence();
            const long long sum = (long long)atomicExch(&d.DEACC[p], 0ull);
            d.E[p] += sum / 2;
            d.DONE[p] = 0;
            d.FCNT[p] = 0;
        }
    }
    if (S > 1) apply_cluster_barrier();   // the sums have been read by the whole cluster
}

template <int COLS>
static cudaError_t launch_apply_cols(const Dev& d, cudaStream_t s)
{
    using Shape = ApplyShape<COLS>;
    const int tiles = (d.ld + Shape::tile - 1) / Shape::tile;
    // about six CTAs per SM when every replica has a long list
    const long long base = (long long)tiles * d.R, want = 6LL * device_sm_count();
    int S = 1;
    while (S < kApplyMaxSplit && base * S * 2 <= want + want / 4) S *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles, (unsigned)d.R, (unsigned)S);
    cfg.blockDim = dim3(Shape::threads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = (unsigned)S;
    cfg.attrs = at;
    cfg.numAttrs = S > 1 ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_apply<COLS>, d);
    if (e != cudaSuccess) return e;
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_apply(const Dev& d, cudaStream_t s)
{
    const bool wide = d.ld % 16 == 0 && ((uintptr_t)d.Q % 16) == 0;
    return wide ? launch_apply_cols<16>(d, s) : launch_apply_cols<4>(d, s);
}

// mask [R][ldm] (0/1) -> flip lists (index | old x << 31).  Grid
// (ceil(n / 4096), R): each thread tests 16 columns (coalesced byte loads),
// a block-wide scan orders the CTA's flips and one atomic per CTA reserves
// their slots in the replica's list (the order of a list is immaterial).
constexpr int kCompactThreads = 256, kCompactPer = 16;

__global__ __launch_bounds__(kCompactThreads) void k_compact_mask(Dev d, const uint8_t* __restrict__ mask, int ldm)
{
    __shared__ int wsum[kCompactThreads / 32];
    __shared__ int s_base;
    const int p = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base_j = blockIdx.x * kCompactThreads * kCompactPer;
    const uint8_t* mrow = mask + (size_t)p * ldm;
    const uint8_t* xrow = d.X + (size_t)p * d.ld;
    unsigned bits = 0;
#pragma unroll
    for (int k = 0; k < kCompactPer; ++k) {
        const int j = base_j + k * kCompactThreads + tid;
        bits |= (unsigned)(j < d.n && mrow[j] != 0) << k;
    }
    const int c = __popc(bits);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (tid == 0) {
        int tot = 0;
        for (int w = 0; w < kCompactThreads / 32; ++w) { const int v = wsum[w]; wsum[w] = tot; tot += v; }
        s_base = tot ? atomicAdd(&d.FCNT[p], tot) : 0;
    }
    __syncthreads();
    int pos = s_base + wsum[warp] + incl - c;
    int32_t* fl = d.FL + (size_t)p * d.ld;
#pragma unroll
    for (int k = 0; k < kCompactPer; ++k)
        if ((bits >> k) & 1u) {
            const int j = base_j + k * kCompactThreads + tid;
            if (pos < d.ld) fl[pos] = j | (int)((unsigned)xrow[j] << 31);
            ++pos;
        }
}

cudaError_t launch_compact_mask(const Dev& d, const uint8_t* mask, int ldm, cudaStream_t s)
{
    const int per = kCompactThreads * kCompactPer;
    dim3 grid((d.n + per - 1) / per, d.R);
    k_compact_mask<<<grid, kCompactThreads, 0, s>>>(d, mask, ldm);
    note_launch(1);
    return cudaGetLastError();
}

}  // namespace icd2s
