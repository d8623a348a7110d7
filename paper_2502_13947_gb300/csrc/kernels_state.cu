// kernels_state.cu -- initial solutions, exact gain/energy recompute,
// Deviation_Extraction (gamma, Eq. 8) and best-solution tracking.
#include <climits>

#include "common.cuh"

namespace icd2s {

// ---------------------------------------------------------------------------
// Generate_Initial_Solution_Set (Algorithm 2): x[p][j] is bit (j mod 32) of
// word ((j / 32) mod 4) of Philox(ctr = (j / 128, TAG_INIT << 24, p, 0)), p
// the global replica index (p0 + the local one).
// One thread per (replica, 128 variables); padding bytes are written as 0.
// ---------------------------------------------------------------------------
__global__ void k_init_x(uint8_t* X, int n, int ld, int R, int p0, uint32_t k0, uint32_t k1)
{
    const int blocks = ld / 128;
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= R * blocks) return;
    const int p = gid / blocks, b = gid % blocks;
    const u32x4 w = philox10((uint32_t)b, kTagInit << 24, (uint32_t)(p0 + p), 0u, k0, k1);
    uint8_t* row = X + (size_t)p * ld + (size_t)b * 128;
#pragma unroll
    for (int v = 0; v < 8; ++v) {   // 8 x 16 bytes
        uint32_t packed[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t word = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int jj = v * 16 + q * 4 + t;            // 0..127
                const int j = b * 128 + jj;
                const uint32_t bit = (w.v[(jj >> 5) & 3] >> (jj & 31)) & 1u;
                word |= (j < n ? bit : 0u) << (8 * t);
            }
            packed[q] = word;
        }
        *reinterpret_cast<uint4*>(row + v * 16) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    }
}

cudaError_t launch_init_x(const Dev& d, cudaStream_t s)
{
    const int total = d.R * (d.ld / 128);
    k_init_x<<<(total + 127) / 128, 128, 0, s>>>(d.X, d.n, d.ld, d.R, d.p0, d.k0, d.k1);
    note_launch(1);
    return cudaGetLastError();
}

constexpr int kEnergySmallN = 512;   // energies in one launch up to this n, on the tensor cores beyond

// ---------------------------------------------------------------------------
// H[p][j] = sum_k Q[j][k] x[p][k]  (int8 x {0,1}, exact int32) with dp4a on
// 64 x 64 output tiles; the k loop walks 64-byte chunks staged in shared
// memory.  Rows are padded with zeros to ld, so no tail handling in k.  With
// few tiles the k range is split over gridDim.z CTAs whose partial sums are
// added into H (zeroed first) with integer atomics: exact in any order.
// ---------------------------------------------------------------------------
constexpr int kGT = 64;          // tile edge (rows j and replicas p)
constexpr int kGK = 64;          // bytes of k per stage
constexpr int kGS = kGK / 4 + 1; // row stride in ints (padding against bank conflicts)

// only_if: when given, the product is taken only if the word it points at is set
// (the tensor-core path's fallback: a pipeline wait that timed out).
__global__ __launch_bounds__(256) void k_hgemm(const int8_t* __restrict__ Q, int n, int ld,
                                               const uint8_t* __restrict__ X, int ldx, int R,
                                               int32_t* __restrict__ H, int ldh, const int* only_if)
{
    if (only_if && *only_if == 0) return;
    __shared__ int Qs[kGT * kGS];
    __shared__ int Xs[kGT * kGS];
    const int t = threadIdx.x;
    const int j0 = blockIdx.x * kGT, p0 = blockIdx.y * kGT;
    const int tj = t % 16, tp = t / 16;
    int acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0;
    const int lr = t / 4, lseg = (t % 4) * 16;  // loader: row, byte offset within the chunk
    const int chunks = ld / kGK, ks = (int)gridDim.z;
    const int kb = (int)((long long)chunks * blockIdx.z / ks) * kGK, ke = (int)((long long)chunks * (blockIdx.z + 1) / ks) * kGK;
    for (int k0 = kb; k0 < ke; k0 += kGK) {
        uint4 qv = make_uint4(0, 0, 0, 0), xv = make_uint4(0, 0, 0, 0);
        if (j0 + lr < n) qv = __ldg(reinterpret_cast<const uint4*>(Q + (size_t)(j0 + lr) * ld + k0 + lseg));
        if (p0 + lr < R) xv = *reinterpret_cast<const uint4*>(X + (size_t)(p0 + lr) * ldx + k0 + lseg);
        __syncthreads();
        int* qd = Qs + lr * kGS + lseg / 4;
        int* xd = Xs + lr * kGS + lseg / 4;
        qd[0] = (int)qv.x; qd[1] = (int)qv.y; qd[2] = (int)qv.z; qd[3] = (int)qv.w;
        xd[0] = (int)xv.x; xd[1] = (int)xv.y; xd[2] = (int)xv.z; xd[3] = (int)xv.w;
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < kGK / 4; ++kk) {
            int qa[4], xb[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) qa[a] = Qs[(tj * 4 + a) * kGS + kk];
#pragma unroll
            for (int b = 0; b < 4; ++b) xb[b] = Xs[(tp * 4 + b) * kGS + kk];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = __dp4a(qa[a], xb[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int p = p0 + tp * 4 + b;
        if (p >= R) continue;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int j = j0 + tj * 4 + a;
            if (j < n) {
                if (ks == 1) H[(size_t)p * ldh + j] = acc[a][b];
                else atomicAdd(&H[(size_t)p * ldh + j], acc[a][b]);
            }
        }
    }
}

// In place: H (incl. diagonal) -> g, and E += sum_j x_j (Q_jj + h_j) (E zeroed
// by the caller; written when one CTA takes the row).  Four columns per thread and pass,
// grid (1 or ld / 1024, R).
__global__ __launch_bounds__(256) void k_finish_gains(const int32_t* __restrict__ diag, int n, int ld,
                                                      const uint8_t* __restrict__ X, int ldx,
                                                      int32_t* G, unsigned long long* E)
{
    const int p = blockIdx.y;
    long long e = 0;
    for (int j0 = (blockIdx.x * 256 + threadIdx.x) * 4; j0 < ld; j0 += gridDim.x * 1024) {
        const uint32_t xv = *reinterpret_cast<const uint32_t*>(X + (size_t)p * ldx + j0);
        int4* gp = reinterpret_cast<int4*>(G + (size_t)p * ld + j0);
        const int4 h4 = *gp, d4 = *reinterpret_cast<const int4*>(diag + j0);
        const int hv[4] = {h4.x, h4.y, h4.z, h4.w}, dv[4] = {d4.x, d4.y, d4.z, d4.w};
        int gv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int xj = (int)((xv >> (8 * b)) & 1u), dj = dv[b];
            const int h = hv[b] - dj * xj;                    // off-diagonal field
            gv[b] = j0 + b < n ? (1 - 2 * xj) * (dj + 2 * h) : 0;
            if (j0 + b < n) e += (long long)xj * (dj + h);
        }
        *gp = make_int4(gv[0], gv[1], gv[2], gv[3]);
    }
    __shared__ long long red[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) e += red[w];
        if (gridDim.x == 1) E[p] = (unsigned long long)e;
        else if (e != 0) atomicAdd(E + p, (unsigned long long)e);
    }
}

cudaError_t launch_finish_gains(const int32_t* diag, int n, int ld, const uint8_t* X, int32_t* G, int64_t* E, int R,
                                cudaStream_t s)
{
    // One CTA per row up to 8192 columns, which needs neither the zeroed E nor atomics: the recompute of
    // n = 1200, one row 15.1 -> 11.2 us, n = 2500, 128 rows 26.0 -> 22.8, n = 7000 49.9 -> 47.5;
    // n = 10 000, 32 rows 68.5 against 69.8.
    const bool one = ld <= 8192;
    cudaError_t e = !one ? cudaMemsetAsync(E, 0, sizeof(int64_t) * (size_t)R, s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    for (int r0 = 0; r0 < R; r0 += 65535) {   // (the grid's y limit)
        const int r = R - r0 < 65535 ? R - r0 : 65535;
        k_finish_gains<<<dim3(one ? 1 : (ld + 1023) / 1024, r), 256, 0, s>>>(
            diag, n, ld, X + (size_t)r0 * ld, ld, G + (size_t)r0 * ld,
            reinterpret_cast<unsigned long long*>(E) + r0);
        note_launch(1);
    }
    return cudaGetLastError();
}

// Gains need the whole product in memory, so the tensor-core path (operand expansion, zeroed
// sums, two launches more) pays from about 2500^2 products of 64 rows on.  Loads of R solutions,
// launches in a graph, dp4a against tensor cores: n = 513, R = 8 12.7 and 15.5 us; 1000, 512 24.9 and
// 25.2; 1000, 1024 39.5 and 29.3; 1200, 256 19.3 and 24.4; 1400, 200 24.7 and 23.8; 1600, 128 19.1 and 20.7; 1800,
// 128 22.9 and 21.0; 2304, 64 20.4 and 21.1; 2500, 1 19.0 and 18.7; 2500, 128 35.6 and 22.7.  Small n: 640,
// 1024 24.2 and 26.7, 800, 1024 30.4 and 28.5.
bool recompute_on_tensor_cores(int n, int R)
{
    const long long work = (long long)n * n * ((R + 63) / 64);
    return n > kEnergySmallN && work >= (n < 1024 ? 8000000 : 6250000);
}

cudaError_t launch_recompute(const Dev& d, const uint8_t* X, int ldx, int R, int32_t* G, int64_t* E,
                             cudaStream_t s, void* Xh, int* err, ProductWait wait)
{
    dim3 grid((d.n + kGT - 1) / kGT, (R + kGT - 1) / kGT);
    cudaError_t e;
    if (Xh && ldx == d.ld && recompute_on_tensor_cores(d.n, R)) {
        if ((e = cudaMemsetAsync(G, 0, sizeof(int32_t) * (size_t)R * d.ld, s)) != cudaSuccess ||
            (e = cudaMemsetAsync(err, 0, sizeof(int), s)) != cudaSuccess ||
            (e = launch_expand_x(X, d.n, ldx, R, d.ld, Xh, nullptr, s)) != cudaSuccess ||
            (e = launch_refresh_i8(d.Q, Xh, d.n, R, d.ld, G, err, 0, 0, wait.ns, wait.skip_loads, s)) != cudaSuccess)
            return e;
        k_hgemm<<<grid, 256, 0, s>>>(d.Q, d.n, d.ld, X, ldx, R, G, d.ld, err);
        note_launch(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        return launch_finish_gains(d.diag, d.n, d.ld, X, G, E, R, s);
    }
    // k splits so that about two CTAs per SM run, each over at least 4 chunks of k
    const int tiles = (int)(grid.x * grid.y), chunks = d.ld / kGK;
    int ks = (2 * device_sm_count() + tiles - 1) / tiles;
    if (ks > chunks / 4) ks = chunks / 4;
    if (ks < 1) ks = 1;
    grid.z = (unsigned)ks;
    if (ks > 1 && (e = cudaMemsetAsync(G, 0, sizeof(int32_t) * (size_t)R * d.ld, s)) != cudaSuccess) return e;
    k_hgemm<<<grid, 256, 0, s>>>(d.Q, d.n, d.ld, X, ldx, R, G, d.ld, nullptr);
    note_launch(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_finish_gains(d.diag, d.n, d.ld, X, G, E, R, s);
}

// E_p = sum_j x_j sum_k Q_jk x_k by plain loops, one CTA per row: the fallback of
// the tensor-core energies.
__global__ __launch_bounds__(256) void k_energy_plain(const int8_t* __restrict__ Q, int n, int ld,
                                                      const uint8_t* __restrict__ x, int64_t* E, const int* only_if)
{
    if (*only_if == 0) return;
    const uint8_t* xp = x + (size_t)blockIdx.x * n;
    long long e = 0;
    for (int j = 0; j < n; ++j)
        if (xp[j])
            for (int k = threadIdx.x; k < n; k += 256) e += xp[k] ? Q[(size_t)j * ld + k] : 0;
    __shared__ long long red[256];
    red[threadIdx.x] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int t = 1; t < 256; ++t) e += red[t];
        E[blockIdx.x] = e;
    }
}

// Energies for n <= 512 in one launch: a CTA takes a row of x, its warps the rows j of Q
// with x_j = 1 (four in flight), a lane every 32nd word.  Padding, product and finish as three
// launches that wait for each other took 14.3 us at n = 64, 8 rows, this 7.5 us, calls back
// to back.  From there on the tensor cores were faster than those three at every number
// of rows measured (n = 600 14-19 us against 19-23, n = 2500, 128 rows 19 against 46,
// n = 7000, 1 row 38 against 103 and 256 rows 49 against 289).
bool energy_in_one_launch(int n) { return n <= kEnergySmallN; }

__global__ __launch_bounds__(256) void k_energy_small(const int8_t* __restrict__ Q, int n, int ld,
                                                      const uint8_t* __restrict__ x, int64_t* E)
{
    __shared__ __align__(16) uint8_t xs[kEnergySmallN];
    __shared__ int red[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint8_t* xp = x + (size_t)blockIdx.x * n;
    for (int j = tid; j < kEnergySmallN; j += 256) xs[j] = j < n ? xp[j] : (uint8_t)0;
    __syncthreads();
    int xw[4];   // the lane's words of x: columns 4 (lane + 32 q) ..
#pragma unroll
    for (int q = 0; q < 4; ++q) xw[q] = *reinterpret_cast<const int*>(xs + 4 * (lane + 32 * q));
    int acc = 0;
    for (int j0 = warp; j0 < n; j0 += 32) {
        int v[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + 8 * u;
            const bool on = j < n && xs[j];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[u][q] = on && 4 * (lane + 32 * q) < ld
                              ? __ldg(reinterpret_cast<const int*>(Q + (size_t)j * ld + 4 * (lane + 32 * q)))
                              : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc = __dp4a(v[u][q], xw[q], acc);
    }
    acc = __reduce_add_sync(0xffffffffu, acc);   // |E| <= 128 n^2 = 2^25
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) acc += red[w];
        E[blockIdx.x] = acc;
    }
}

cudaError_t launch_energy_small(const Dev& d, const uint8_t* x, int R, int64_t* E, cudaStream_t s)
{
    k_energy_small<<<R, 256, 0, s>>>(d.Q, d.n, d.ld, x, E);
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_energy_tc(const Dev& d, const uint8_t* x, int R, int64_t* E, void* Xh, uint32_t* bits, int* err,
                             cudaStream_t s, ProductWait wait)
{
    cudaError_t e;
    if ((e = cudaMemsetAsync(E, 0, sizeof(int64_t) * (size_t)R, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(err, 0, sizeof(int), s)) != cudaSuccess ||
        (e = launch_expand_x(x, d.n, d.n, R, d.ld, Xh, bits, s)) != cudaSuccess ||
        (e = launch_refresh_i8(d.Q, Xh, d.n, R, d.ld, nullptr, err, 0, 0, wait.ns, wait.skip_loads, s,
                               reinterpret_cast<unsigned long long*>(E), bits)) != cudaSuccess)
        return e;
    k_energy_plain<<<R, 256, 0, s>>>(d.Q, d.n, d.ld, x, E, err);
    note_launch(1);
    return cudaGetLastError();
}

// dense [rows][n] -> padded [rows][ld] (zero padding)
__global__ void k_pad_rows(const uint8_t* __restrict__ src, int n, int rows, uint8_t* __restrict__ dst, int ld)
{
    const size_t total = (size_t)rows * ld;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / ld, c = i % ld;
        dst[i] = c < (size_t)n ? src[r * n + c] : (uint8_t)0;
    }
}

cudaError_t launch_pad_rows(const uint8_t* src, int n, int rows, uint8_t* dst, int ld, cudaStream_t s)
{
    const size_t total = (size_t)rows * ld;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_pad_rows<<<blocks, 256, 0, s>>>(src, n, rows, dst, ld);
    note_launch(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Deviation_Extraction (Eq. 8): gamma_j = 1 - |sum_p x_pj - z/2| / (z/2)
//                                       = (z - |2 sum_p x_pj - z|) / z, Q16 floor,
// the sum over all z replicas: this state's own (counts == null), or the
// column counts of every replica shard added up by the caller.
// ---------------------------------------------------------------------------
// Column sums: a warp covers 128 columns (4 per lane, one word), the CTA's eight
// warps every eighth row, four rows in flight; their sums meet in shared memory.
// (One thread per column over all rows kept 10 to 28 CTAs busy: 13 us at
// n = 7000, 256 rows.)
__global__ __launch_bounds__(256) void k_gamma(const uint8_t* __restrict__ X, int n, int ld, int R,
                                               const int32_t* __restrict__ counts, int z,
                                               int32_t* __restrict__ gamma, int32_t* __restrict__ sums)
{
    __shared__ int4 part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * 128 + 4 * lane;   // (ld is a multiple of 128)
    int c[4] = {0, 0, 0, 0};
    if (!counts) {
        for (int p0 = warp; p0 < R; p0 += 32) {
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + 8 * u;
                v[u] = p < R ? *reinterpret_cast<const uint32_t*>(X + (size_t)p * ld + j0) : 0u;
            }
            const uint32_t w = v[0] + v[1] + v[2] + v[3];   // bytes up to 4
#pragma unroll
            for (int b = 0; b < 4; ++b) c[b] += (int)((w >> (8 * b)) & 0xffu);
        }
    }
    part[warp][lane] = make_int4(c[0], c[1], c[2], c[3]);
    __syncthreads();
    if (threadIdx.x >= 128) return;
    const int j = blockIdx.x * 128 + threadIdx.x;
    int col = 0;
    if (counts) {
        col = j < n ? counts[j] : 0;
    } else {
#pragma unroll
        for (int w = 0; w < 8; ++w) col += reinterpret_cast<const int*>(part[w])[threadIdx.x];
    }
    if (sums) {
        if (j < n) sums[j] = col;
        return;
    }
    const int dev = abs(2 * col - z);
    gamma[j] = j < n ? (int32_t)(((long long)(z - dev) * 65536) / z) : 0;
}

cudaError_t launch_gamma(const Dev& d, const int32_t* counts, cudaStream_t s)
{
    k_gamma<<<d.ld / 128, 256, 0, s>>>(d.X, d.n, d.ld, d.R, counts, counts ? d.z_total : d.R, d.gamma, nullptr);
    note_launch(1);
    return cudaGetLastError();
}

// column counts of this state's replicas (the shard's part of Eq. 8's sum)
cudaError_t launch_colsum(const Dev& d, int32_t* counts, cudaStream_t s)
{
    k_gamma<<<d.ld / 128, 256, 0, s>>>(d.X, d.n, d.ld, d.R, nullptr, 1, nullptr, counts);
    note_launch(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Best solution over the replicas (strictly lower energy; lowest replica on
// ties), optional trace of all energies, and the per-iteration stale counter
// used by the termination rule (Section 3: stop after a number of
// consecutive iterations without a new best).
// flags[0] = improved during this iteration, flags[1] = stale iterations,
// flags[3] = replica last copied into best_x, flags[4] = flags[0] of the
// iteration just ended, flags[5] = its improvement-log slot.
// ---------------------------------------------------------------------------
__global__ __launch_bounds__(256) void k_best(const uint8_t* __restrict__ X, int ld, const int64_t* __restrict__ E,
                                              int R, uint8_t* best_x, int64_t* best_E, int32_t* flags,
                                              int64_t* trace_slot, int iter_end, int32_t* iter_dev,
                                              int32_t* log_ctl, int phase, int t_arg)
{
    __shared__ long long sE[8];
    __shared__ int sP[8];
    __shared__ int s_win;
    long long me = LLONG_MAX;
    int mp = 0x7fffffff;
    for (int p = threadIdx.x; p < R; p += blockDim.x) {
        const long long e = E[p];
        if (trace_slot) trace_slot[p] = e;
        if (e < me || (e == me && p < mp)) { me = e; mp = p; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long oe = __shfl_xor_sync(0xffffffffu, me, o);
        const int op = __shfl_xor_sync(0xffffffffu, mp, o);
        if (oe < me || (oe == me && op < mp)) { me = oe; mp = op; }
    }
    if ((threadIdx.x & 31) == 0) { sE[threadIdx.x >> 5] = me; sP[threadIdx.x >> 5] = mp; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            if (sE[w] < me || (sE[w] == me && sP[w] < mp)) { me = sE[w]; mp = sP[w]; }
        const long long cur = *best_E;
        s_win = (me < cur) ? mp : -1;
        if (s_win >= 0) {
            *best_E = me; flags[0] = 1; flags[3] = mp;
            flags[7] = phase < 0 ? 0 : 3 * (iter_dev ? *iter_dev : t_arg) + phase + 1;
        }
    }
    __syncthreads();
    const int win = s_win;
    if (win >= 0)
        for (int j = threadIdx.x * 16; j < ld; j += blockDim.x * 16)
            *reinterpret_cast<uint4*>(best_x + j) = *reinterpret_cast<const uint4*>(X + (size_t)win * ld + j);
    if (threadIdx.x == 0 && iter_end) {
        if (trace_slot) trace_slot[R] = *best_E;
        flags[1] = flags[0] ? 0 : flags[1] + 1;
        flags[4] = flags[0];
        if (log_ctl && flags[0]) {  // slot of the improvement-log entry (ring buffer)
            flags[5] = log_ctl[0] % log_ctl[1];
            log_ctl[0] += 1;
        }
        flags[0] = 0;
        if (iter_dev) *iter_dev += 1;  // the next replay of a captured iteration is t + 1
    }
}

cudaError_t launch_best(const Dev& d, int64_t* trace_slot, int iter_end, int32_t* iter_dev, cudaStream_t s,
                        int32_t* log_ctl, int phase, int t)
{
    k_best<<<1, 256, 0, s>>>(d.X, d.ld, d.E, d.R, d.best_x, d.best_E, d.flags, trace_slot, iter_end, iter_dev,
                             log_ctl, phase, t);
    note_launch(1);
    return cudaGetLastError();
}

__global__ void k_set_iter(int32_t* iter_dev, int t) { *iter_dev = t; }

cudaError_t launch_set_iter(int32_t* iter_dev, int t, cudaStream_t s)
{
    k_set_iter<<<1, 1, 0, s>>>(iter_dev, t);
    note_launch(1);
    return cudaGetLastError();
}

int device_sm_count()
{
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    if (!cached[dev]) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 152;
        cached[dev] = v;
    }
    return cached[dev];
}

// ---------------------------------------------------------------------------
// Per-instance preparation.  k_symcheck compares 32 x 32 tiles of Q with the
// transposed tiles (counts mismatches); k_eta forms eta_j = sum_i |Q_ij|
// (Eq. 6), the diagonal and the column's largest gain over all x (one thread
// per column, coalesced across j): with P_j / N_j the sums of the positive /
// negative off-diagonal entries' magnitudes, Q_jj + 2 sum_{i != j} Q_ij x_i
// ranges over [Q_jj - 2 N_j, Q_jj + 2 P_j], so max |g_j| = max(|Q_jj - 2 N_j|,
// |Q_jj + 2 P_j|), attained; k_etahat normalises eta by its maximum (Q16, floor).
// ---------------------------------------------------------------------------
__global__ void k_symcheck(const int8_t* __restrict__ Q, int n, int ld, int* mismatches)
{
    __shared__ int8_t A[32][33], B[32][33];
    const int bi = blockIdx.y * 32, bj = blockIdx.x * 32;
    if (bi > bj) return;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int c = threadIdx.x;
        A[r][c] = (bi + r < n && bj + c < n) ? Q[(size_t)(bi + r) * ld + bj + c] : 0;
        B[r][c] = (bj + r < n && bi + c < n) ? Q[(size_t)(bj + r) * ld + bi + c] : 0;
    }
    __syncthreads();
    int bad = 0;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) bad += A[r][threadIdx.x] != B[threadIdx.x][r];
    bad = __reduce_add_sync(0xffffffffu, (unsigned)bad);
    if (threadIdx.x == 0 && bad) atomicAdd(mismatches, bad);
}

__global__ void k_eta(const int8_t* __restrict__ Q, int n, int ld, int32_t* eta, int32_t* diag, int* n128,
                      int* gmax)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ld) return;
    if (j >= n) { eta[j] = 0; diag[j] = 0; return; }
    int s = 0, m = 0, pos = 0, neg = 0;
    for (int i = 0; i < n; ++i) {
        const int v = Q[(size_t)i * ld + j];
        s += abs(v);
        m += v == -128;
        if (i != j) {
            pos += v > 0 ? v : 0;
            neg += v < 0 ? -v : 0;
        }
    }
    eta[j] = s;
    const int qjj = Q[(size_t)j * ld + j];
    diag[j] = qjj;
    if (m) atomicAdd(n128, m);
    atomicMax(gmax, max(abs(qjj - 2 * neg), abs(qjj + 2 * pos)));
}

__global__ __launch_bounds__(1024) void k_etahat(const int32_t* __restrict__ eta, int n, int ld, int32_t* etahat,
                                                 int* eta_max)
{
    __shared__ int red[32];
    int mx = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) mx = max(mx, eta[j]);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, red[w]);
    if (threadIdx.x == 0) *eta_max = mx;
    for (int j = threadIdx.x; j < ld; j += blockDim.x)
        etahat[j] = (j < n && mx > 0) ? (int32_t)(((long long)eta[j] * 65536) / mx) : 0;
}

// Signed row pairs for the Tabu search: one thread per 16 bytes of a row of Q
// writes them to rows 2i and 2i + 1 (bytewise negation; no entry is -128).
__global__ void k_signed_rows(const int8_t* __restrict__ Q, int n, int ld, int8_t* __restrict__ Q2)
{
    const size_t chunks = (size_t)n * (ld / 16);
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= chunks) return;
    const size_t i = t / (ld / 16), c = t % (ld / 16);
    const uint4 v = *reinterpret_cast<const uint4*>(Q + i * ld + 16 * c);
    uint32_t w[4] = {v.x, v.y, v.z, v.w}, m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t r = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) r |= (uint32_t)(uint8_t)(-(int8_t)(w[k] >> (8 * b))) << (8 * b);
        m[k] = r;
    }
    *reinterpret_cast<uint4*>(Q2 + (2 * i) * ld + 16 * c) = v;
    *reinterpret_cast<uint4*>(Q2 + (2 * i + 1) * ld + 16 * c) = make_uint4(m[0], m[1], m[2], m[3]);
}

// One CTA per row of the relabeled matrix; the label table is read through L1.
__global__ void k_relabel(const int8_t* __restrict__ Q, const int32_t* __restrict__ perm, int n, int ld,
                          int8_t* __restrict__ Qpk)
{
    const int L = blockIdx.x;
    const int8_t* src = Q + (size_t)perm[L] * ld;
    int8_t* dst = Qpk + (size_t)L * ld;
    for (int M = threadIdx.x; M < ld; M += blockDim.x) dst[M] = M < n ? src[perm[M]] : (int8_t)0;
}

cudaError_t launch_relabel(const int8_t* Q, const int32_t* perm, int n, int ld, int8_t* Qpk, cudaStream_t s)
{
    k_relabel<<<n, 256, 0, s>>>(Q, perm, n, ld, Qpk);
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_signed_rows(const int8_t* Q, int n, int ld, int8_t* Q2, cudaStream_t s)
{
    const size_t chunks = (size_t)n * (ld / 16);
    k_signed_rows<<<(unsigned)((chunks + 255) / 256), 256, 0, s>>>(Q, n, ld, Q2);
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_prepare(const int8_t* Q, int n, int ld, int32_t* eta, int32_t* etahat, int32_t* diag,
                           int* mismatches, int* eta_max, int* gain_max, cudaStream_t s)
{
    const int tiles = (n + 31) / 32;
    k_symcheck<<<dim3(tiles, tiles), dim3(32, 8), 0, s>>>(Q, n, ld, mismatches);
    note_launch(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_eta<<<(ld + 255) / 256, 256, 0, s>>>(Q, n, ld, eta, diag, eta_max + 1, gain_max);
    note_launch(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_etahat<<<1, 1024, 0, s>>>(eta, n, ld, etahat, eta_max);
    note_launch(1);
    return cudaGetLastError();
}

}  // namespace icd2s
