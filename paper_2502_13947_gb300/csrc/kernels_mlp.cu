// kernels_mlp.cu -- the proposal network of the learned subQUBO selection
// (an addition to IC-D2S's Algorithm 4 subset choice): per-variable features,
// the 6-64-64-1 score network (BF16 weights, FP32 arithmetic), its training by
// backpropagation of a weighted binary cross-entropy with a deterministic
// gradient reduction, Adam, and the improvement log that supplies the labels.
//
//  k_gmax       one CTA per replica: max_j |g_j|.
//  k_features   one thread per (replica, variable): the six features
//               f = (x, g/(max|g|+1), T/alpha, C/c, H/(t+1), eta_hat/2^16).
//  k_score      the network in float with one fused multiply-add per product in
//               a fixed order (units and inputs ascending), so the selection
//               decision is reproducible; 16 to 128 rows per CTA, register tiles.
//  k_mlp_grad   64 rows per CTA: forward, then the gradient of the mean loss
//               summed over the CTA's rows in a fixed order; one partial
//               gradient per CTA.
//  k_mlp_reduce sums the partial gradients in a fixed order (deterministic) and
//               applies Adam to the float32 master weights, re-rounding the
//               BF16 copy.
//  k_log        appends an improvement-log entry (features of the replica
//               that produced the new best, label = best_x XOR previous best).
//
// Why CUDA cores and not the tensor cores: the network is 9 088 FLOPs per
// row; at 32 replicas x 10 000 variables a score pass is ~3 GFLOP (tens of
// microseconds on the FP32 pipes), and rounding the activations to BF16/TF32
// for tcgen05 would move the scores by ~1e-3 relative -- the tolerance the
// scores are held to -- and would change the ranking the selection takes.
#include <cuda_bf16.h>

#include "common.cuh"

namespace icd2s {

namespace {

constexpr int kGradRows = 64;     // rows per CTA of k_mlp_grad
constexpr int kGradCtas = 4096;   // CTAs of one launch: more rows go through the same partial sums again

__device__ __forceinline__ float softplus(float v) { return fmaxf(v, 0.f) + log1pf(expf(-fabsf(v))); }
__device__ __forceinline__ float sigmoid(float v) { return 1.f / (1.f + expf(-v)); }

// Register-tiled FP32 products over tiles in shared memory.  Every 64-wide
// tile has rows of kLS floats and W1 rows of kL1 (its six weights and b1; a
// feature row ends in 1 and 0 there): 16-byte loads of eight consecutive rows
// then fall into different banks.
constexpr int kLS = 68;
constexpr int kL1 = 12;
constexpr int kTS = 72;   // the same for BF16 rows

struct NetTile {                      // the network in shared memory
    float W2[64 * kLS];               // row o: weights into unit o
    float W1[64 * kL1];
    float b2[64], w3[64];
    float b3, pad[3];
};

// Wb carries no __restrict__ here: the training step before this one may still be
// writing it when the kernel starts (see pdl_wait below).
template <int NT, bool F32>
__device__ __forceinline__ void load_net(const __nv_bfloat16* Wb, NetTile& w)
{
    for (int q = threadIdx.x; q < 512; q += NT) {   // 8 weights of row q / 8 of W2
        const uint4 v = *reinterpret_cast<const uint4*>(Wb + kOffW2 + 8 * q);
        if constexpr (!F32) {   // W2 as BF16 rows of kTS
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(w.W2) + (q >> 3) * kTS + 8 * (q & 7)) = v;
            continue;
        }
        float4* dst = reinterpret_cast<float4*>(w.W2 + (q >> 3) * kLS + 8 * (q & 7));
        dst[0] = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                             __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
        dst[1] = make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xffff0000u),
                             __uint_as_float(v.w << 16), __uint_as_float(v.w & 0xffff0000u));
    }
    for (int q = threadIdx.x; q < 384; q += NT) w.W1[(q / 6) * kL1 + q % 6] = __bfloat162float(Wb[kOffW1 + q]);
    if (threadIdx.x < 64) {
        const int o = threadIdx.x;
        w.W1[o * kL1 + 6] = __bfloat162float(Wb[kOffB1 + o]);
        w.W1[o * kL1 + 7] = 0.f;
        w.b2[o] = __bfloat162float(Wb[kOffB2 + o]);
        w.w3[o] = __bfloat162float(Wb[kOffW3 + o]);
        if (o == 0) w.b3 = __bfloat162float(Wb[kOffB3]);
    }
}

// acc[i][j] = relu(b1 + W1 f) of rows r0 + rs i and units o0 + os j, inputs ascending
template <int RT, int OT>
__device__ __forceinline__ void layer1(float (&acc)[RT][OT], const float* Fs, const NetTile& w, int r0, int rs,
                                       int o0, int os)
{
    float f[RT][8];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const float4* p = reinterpret_cast<const float4*>(Fs + (r0 + rs * i) * kL1);
        const float4 a = p[0], b = p[1];
        f[i][0] = a.x; f[i][1] = a.y; f[i][2] = a.z; f[i][3] = a.w; f[i][4] = b.x; f[i][5] = b.y;
    }
#pragma unroll
    for (int j = 0; j < OT; ++j) {
        const float4* p = reinterpret_cast<const float4*>(w.W1 + (o0 + os * j) * kL1);
        const float4 a = p[0], b = p[1];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            float v = __fmaf_rn(a.x, f[i][0], b.z);
            v = __fmaf_rn(a.y, f[i][1], v);
            v = __fmaf_rn(a.z, f[i][2], v);
            v = __fmaf_rn(a.w, f[i][3], v);
            v = __fmaf_rn(b.x, f[i][4], v);
            v = __fmaf_rn(b.y, f[i][5], v);
            acc[i][j] = v > 0.f ? v : 0.f;
        }
    }
}

// acc[i][j] += sum_k A[r0 + rs i][k] B[o0 + os j][k], k ascending
template <int RT, int OT>
__device__ __forceinline__ void gemm_nt(float (&acc)[RT][OT], const float* A, const float* B, int r0, int rs, int o0,
                                        int os)
{
#pragma unroll 2
    for (int k = 0; k < 64; k += 4) {
        float4 a[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) a[i] = *reinterpret_cast<const float4*>(A + (r0 + rs * i) * kLS + k);
#pragma unroll
        for (int j = 0; j < OT; ++j) {
            const float4 b = *reinterpret_cast<const float4*>(B + (o0 + os * j) * kLS + k);
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[i][j] = __fmaf_rn(b.x, a[i].x, acc[i][j]);
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[i][j] = __fmaf_rn(b.y, a[i].y, acc[i][j]);
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[i][j] = __fmaf_rn(b.z, a[i].z, acc[i][j]);
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[i][j] = __fmaf_rn(b.w, a[i].w, acc[i][j]);
        }
    }
}

__device__ __forceinline__ int block_max_int(int v, int* red)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        int w = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : 0;
        w = __reduce_max_sync(0xffffffffu, w);
        if (threadIdx.x == 0) red[32] = w;
    }
    __syncthreads();
    return red[32];
}

}  // namespace

// ---------------------------------------------------------------------------
__global__ __launch_bounds__(256) void k_gmax(const int32_t* __restrict__ G, int n, int ld, int32_t* gmax)
{
    __shared__ int red[33];
    const int p = blockIdx.x;
    int m = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) m = max(m, abs(G[(size_t)p * ld + j]));
    m = block_max_int(m, red);
    if (threadIdx.x == 0) gmax[p] = m;
}

__global__ __launch_bounds__(256) void k_features(Dev d, int t_arg, const int32_t* iter_dev, int alpha, int c,
                                                  const int32_t* __restrict__ gmax)
{
    const int p = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d.ld) return;
    const int t = iter_dev ? *iter_dev : t_arg;
    const size_t e = (size_t)p * d.ld + j;
    float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (j < d.n) {
        f[0] = (float)d.X[e];
        f[1] = __fdiv_rn((float)d.G[e], (float)(gmax[p] + 1));
        f[2] = alpha > 0 ? __fdiv_rn((float)d.T[e], (float)alpha) : 0.f;
        f[3] = __fdiv_rn((float)d.C[e], (float)c);
        f[4] = __fdiv_rn((float)d.H[e], (float)(t + 1));
        f[5] = __fdiv_rn((float)d.etahat[j], 65536.f);
    }
    float2* out = reinterpret_cast<float2*>(d.F + e * 6);
    out[0] = make_float2(f[0], f[1]);
    out[1] = make_float2(f[2], f[3]);
    out[2] = make_float2(f[4], f[5]);
}

// Two FP32 multiply-adds in one instruction, each rounded as fmaf rounds it.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 dup2(float v)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
    return d;
}

__device__ __forceinline__ float4 relu4(f32x2 a, f32x2 b)
{
    float4 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.z), "=f"(v.w) : "l"(b));
    return make_float4(v.x > 0.f ? v.x : 0.f, v.y > 0.f ? v.y : 0.f, v.z > 0.f ? v.z : 0.f, v.w > 0.f ? v.w : 0.f);
}

struct ScoreNet {                     // the network in shared memory, by inputs
    float W2[64 * kLS];               // row k: weights of input k into the 64 units
    float W1[6 * 64];
    float b1[64], b2[64], w3[64];
    float b3, pad[3];
};

// Units 4 tx .. + 3 and 32 + 4 tx .. + 3 as four pairs
__device__ __forceinline__ void unit_pairs(f32x2 (&v)[4], const float* p)
{
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p), b = *reinterpret_cast<const ulonglong2*>(p + 32);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// Scores of 16 RT rows per CTA of 128 threads.  Thread (ty, tx) forms the RT
// rows ty + 16 i times 8 units of each layer in registers, two units per
// multiply-add instruction; the output unit's chain over the 64 hidden units runs one
// row per thread.  Every sum starts at the bias and takes its inputs in
// ascending order with one fused multiply-add each, so the scores do not
// depend on the tile.
// Bound by the FP32 pipes: 4544 multiply-adds per row.  (One row per thread
// with its weights read as broadcasts needs a 16-byte shared load per four
// multiply-adds; a tile of 8 x 8 needs one per 16: 320 000 rows 107 -> 60 us, a
// single row 19 -> 8 us.  One unit per instruction took 71 us.)  By shared memory
// three CTAs of 128 rows (59.3 KiB each) or five of 64 (39.3 KiB) fit an SM.
template <int RT>
__global__ __launch_bounds__(128, RT == 8 ? 3 : 5) void k_score(const float* __restrict__ F, long long rows,
                                                  const __nv_bfloat16* __restrict__ Wb, float* __restrict__ out)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int kRows = 16 * RT;
    ScoreNet& w = *reinterpret_cast<ScoreNet*>(sm);
    float* Fs = sm + sizeof(ScoreNet) / 4;  // [kRows][kL1]
    float* H = Fs + kRows * kL1;            // [kRows][kLS]
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long r = (long long)blockIdx.x * kRows + tid;
    if (tid < kRows) {
        float2 a = make_float2(0.f, 0.f), b = a, c = a;
        if (r < rows) {
            const float2* fr = reinterpret_cast<const float2*>(F + r * 6);
            a = fr[0]; b = fr[1]; c = fr[2];
        }
        float4* dst = reinterpret_cast<float4*>(Fs + tid * kL1);
        dst[0] = make_float4(a.x, a.y, b.x, b.y);
        dst[1] = make_float4(c.x, c.y, 0.f, 0.f);
    }
#pragma unroll
    for (int q = tid; q < 512; q += 128) {   // inputs 8 (q / 64) .. + 7 of unit q mod 64
        const int o = q & 63, k = 8 * (q >> 6);
        const uint4 v = *reinterpret_cast<const uint4*>(Wb + kOffW2 + 64 * o + k);
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            w.W2[(k + 2 * e) * kLS + o] = __uint_as_float(u[e] << 16);
            w.W2[(k + 2 * e + 1) * kLS + o] = __uint_as_float(u[e] & 0xffff0000u);
        }
    }
#pragma unroll
    for (int q = tid; q < 384; q += 128) w.W1[(q % 6) * 64 + q / 6] = __bfloat162float(Wb[kOffW1 + q]);
    if (tid < 64) {
        w.b1[tid] = __bfloat162float(Wb[kOffB1 + tid]);
        w.b2[tid] = __bfloat162float(Wb[kOffB2 + tid]);
        w.w3[tid] = __bfloat162float(Wb[kOffW3 + tid]);
        if (tid == 0) w.b3 = __bfloat162float(Wb[kOffB3]);
    }
    __syncthreads();
    f32x2 acc[RT][4], b[4];
    unit_pairs(b, w.b1 + 4 * tx);
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = b[j];
#pragma unroll
    for (int k = 0; k < 6; k += 2) {
        float2 f[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) f[i] = *reinterpret_cast<const float2*>(Fs + (ty + 16 * i) * kL1 + k);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            unit_pairs(b, w.W1 + (k + e) * 64 + 4 * tx);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const f32x2 a = dup2(e ? f[i].y : f[i].x);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(b[j], a, acc[i][j]);
            }
        }
    }
    auto store = [&]() {
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            float* h = H + (ty + 16 * i) * kLS + 4 * tx;
            *reinterpret_cast<float4*>(h) = relu4(acc[i][0], acc[i][1]);
            *reinterpret_cast<float4*>(h + 32) = relu4(acc[i][2], acc[i][3]);
        }
    };
    store();
    __syncthreads();
    unit_pairs(b, w.b2 + 4 * tx);
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = b[j];
#pragma unroll 2
    for (int k = 0; k < 64; k += 4) {
        float4 h[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) h[i] = *reinterpret_cast<const float4*>(H + (ty + 16 * i) * kLS + k);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            unit_pairs(b, w.W2 + (k + e) * kLS + 4 * tx);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const f32x2 a = dup2(e == 0 ? h[i].x : e == 1 ? h[i].y : e == 2 ? h[i].z : h[i].w);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(b[j], a, acc[i][j]);
            }
        }
    }
    __syncthreads();   // every thread has read the first hidden layer
    store();
    __syncthreads();
    if (tid < kRows && r < rows) {
        float s = w.b3;
#pragma unroll 4
        for (int o = 0; o < 64; o += 4) {
            const float4 h = *reinterpret_cast<const float4*>(H + tid * kLS + o);
            const float4 v = *reinterpret_cast<const float4*>(w.w3 + o);
            s = __fmaf_rn(v.x, h.x, s);
            s = __fmaf_rn(v.y, h.y, s);
            s = __fmaf_rn(v.z, h.z, s);
            s = __fmaf_rn(v.w, h.w, s);
        }
        out[r] = s;
    }
}

// ---------------------------------------------------------------------------
// Row r of the step's batch: all rows in order when the batch covers them,
// otherwise a Philox draw (counter (r, TAG_TRAIN << 24, step, 0)) modulo rows.
__device__ __forceinline__ long long batch_row(long long r, long long rows, long long batch, uint32_t step, uint32_t k0,
                                               uint32_t k1)
{
    if (batch >= rows) return r;
    const u32x4 v = philox10((uint32_t)r, kTagTrain << 24, step, 0u, k0, k1);
    const unsigned long long u = ((unsigned long long)v.v[1] << 32) | v.v[0];
    return (long long)(u % (unsigned long long)rows);
}

// ---- the 64-wide products on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32
// accumulation): one warp forms 16 rows x 32 columns.  Operands lie as BF16 rows of kTS in
// shared memory; ldmatrix transposes on the way where the sum runs along their rows.
namespace {

// D += A B: A 16 x 16 (row-major), B 16 x 8 (column-major), BF16 -> FP32
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8 x 8 blocks of BF16; block m of the lane's row address is lane / 8
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    if constexpr (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a)
                     : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a)
                     : "memory");
}

// acc = sum_k A(m, k) B(n, k) over k < 64 for m0 .. + 15, n0 .. + 31.  AT: A is stored [k][m],
// otherwise [m][k]; BT: B is stored [k][n], otherwise [n][k].
template <bool AT, bool BT>
__device__ __forceinline__ void warp_mma(float (&acc)[4][4], const __nv_bfloat16* A, int m0, const __nv_bfloat16* B,
                                         int n0)
{
    const int lane = threadIdx.x & 31, lo = lane & 7, b1 = ((lane >> 3) & 1) * 8, b2 = (lane >> 4) * 8;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[nt][e] = 0.f;
#pragma unroll
    for (int k = 0; k < 64; k += 16) {
        uint32_t a[4];
        ldsm4<AT>(a, AT ? A + (k + b2 + lo) * kTS + m0 + b1 : A + (m0 + b1 + lo) * kTS + k + b2);
#pragma unroll
        for (int np = 0; np < 2; ++np) {
            uint32_t b[4];
            const int n = n0 + 16 * np;
            ldsm4<BT>(b, BT ? B + (k + b1 + lo) * kTS + n + b2 : B + (n + b2 + lo) * kTS + k + b1);
            mma_bf16_16816(acc[2 * np], a, b[0], b[1]);
            mma_bf16_16816(acc[2 * np + 1], a, b[2], b[3]);
        }
    }
}

template <bool ADD>
__device__ __forceinline__ void put(float* p, float v)
{
    *p = ADD ? *p + v : v;
}

template <bool ADD>
__device__ __forceinline__ void put2(float* p, float a, float b)
{
    const float2 o = ADD ? *reinterpret_cast<const float2*>(p) : make_float2(0.f, 0.f);
    *reinterpret_cast<float2*>(p) = ADD ? make_float2(o.x + a, o.y + b) : make_float2(a, b);
}

template <bool ADD>
__device__ __forceinline__ void put4(float* p, const float (&v)[4])
{
    const float4 o = ADD ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(p) = ADD ? make_float4(o.x + v[0], o.y + v[1], o.z + v[2], o.w + v[3])
                                        : make_float4(v[0], v[1], v[2], v[3]);
}

// the warp's 16 x 32 accumulators into rows of ld floats (ADD: onto them)
template <bool ADD>
__device__ __forceinline__ void store_acc(const float (&acc)[4][4], float* dst, int ld, int m0, int n0)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        put2<ADD>(dst + (m0 + g) * ld + n0 + 8 * nt + 2 * t, acc[nt][0], acc[nt][1]);
        put2<ADD>(dst + (m0 + g + 8) * ld + n0 + 8 * nt + 2 * t, acc[nt][2], acc[nt][3]);
    }
}

}  // namespace

// Programmatic dependent launch: a kernel lets the next one of its stream start
// (pdl_trigger), and the next one waits for all of it before it touches what
// it wrote or reads (pdl_wait).  Without the launch attribute both do nothing.
// What the kernel before may still be writing is not __restrict__: a const __restrict__
// argument is read-only from the kernel's first instruction on, and its loads may
// go through the non-coherent path or above pdl_wait.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One partial gradient (and loss) per CTA of 64 rows, 256 threads, from row first_row of
// the batch on; ADD: added to what the CTA of an earlier launch left there.  Thread
// (ty, tx) owns a 4 x 4 tile of each of the three 64-wide products: rows
// ty + 16 i times units tx + 16 j of the second layer, units 4 ty.. times inputs
// 4 tx.. of its weight gradient, rows ty + 16 i times units 4 tx.. of the way
// back.  The column sums (w3, b2, W1, b1) are taken from the tiles in
// registers: four rows per thread, then lanes, then warps, in a fixed order.
// 128 CTAs at 8192 rows, so the rows fill the SMs (64 CTAs of four warps that
// formed one output after the other before: 74 -> 14.4 us with the reduction,
// at 32 768 rows 99 -> 37 us).
// TC: the three products on the tensor cores instead, h1 and dL/da2 rounded to
// BF16 for them (the weights already are BF16) and the results passed on through
// shared memory; layer 1, the losses and the column sums stay in FP32 (8192 rows
// 22.9 -> 9.8 us, 32 768 rows 43 -> 22 us).
template <bool TC, bool ADD>
__global__ __launch_bounds__(256) void k_mlp_grad(const float* __restrict__ F, const uint8_t* __restrict__ y,
                                                  long long rows, long long batch, uint32_t step, uint32_t k0,
                                                  uint32_t k1, const __nv_bfloat16* Wb, float pos_weight, float* partial,
                                                  long long first_row)
{
    extern __shared__ __align__(16) float sm[];
    NetTile& w = *reinterpret_cast<NetTile*>(sm);
    float* Fs = sm + sizeof(NetTile) / 4;        // [64][kL1]
    float* H1 = Fs + kGradRows * kL1;            // [64][kLS] h1
    float* D2 = H1 + kGradRows * kLS;            // [64][kLS] dL/da2
    float* red = D2 + kGradRows * kLS;           // [4][512]: sums of four warps
    float* DS = red + 4 * 512;                   // [64] dL/ds
    float* SP = DS + kGradRows;                  // [2][64] halves of the score
    float* X = SP + 2 * kGradRows;               // TC: [64][kLS] products passed between the tilings
    // TC: BF16 tiles [64][kTS] in the places of the FP32 ones
    __nv_bfloat16* W2h = reinterpret_cast<__nv_bfloat16*>(w.W2);
    __nv_bfloat16* H1h = reinterpret_cast<__nv_bfloat16*>(H1);
    __nv_bfloat16* D2h = reinterpret_cast<__nv_bfloat16*>(D2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
    const long long nb = batch < rows ? batch : rows;
    const long long r0 = first_row + (long long)blockIdx.x * kGradRows;
    {
        // four threads per row: its features, the label beside them
        const int rr = tid >> 2, q = tid & 3;
        const bool valid = r0 + rr < nb;
        float a = 0.f, b = 0.f;
        if (valid) {
            const long long row = batch_row(r0 + rr, rows, batch, step, k0, k1);
            a = F[row * 6 + q];
            if (q < 2) b = F[row * 6 + 4 + q];
            else if (q == 2) b = 1.f;
            if (q == 3) b = y[row] ? 1.f : 0.f;
        }
        Fs[rr * kL1 + q] = a;
        Fs[rr * kL1 + 4 + q] = b;    // [6]: 1 for a row of the batch, [7]: its label
    }
    // the rows above are not written by a training step; the weights and the partial sums are
    pdl_wait();
    pdl_trigger();
    load_net<256, !TC>(Wb, w);
    __syncthreads();
    const int m0 = 16 * (warp >> 1), n0 = 32 * (warp & 1);   // TC: the warp's tile
    float acc[4][4];
    layer1<4, 4>(acc, Fs, w, ty, 16, tx, 16);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if constexpr (TC) H1h[(ty + 16 * i) * kTS + tx + 16 * j] = __float2bfloat16_rn(acc[i][j]);
            else H1[(ty + 16 * i) * kLS + tx + 16 * j] = acc[i][j];
        }
    float w3[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w3[j] = w.w3[tx + 16 * j];
        const float b2 = w.b2[tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = b2;
    }
    __syncthreads();
    if constexpr (TC) {
        float t[4][4];
        warp_mma<false, false>(t, H1h, m0, W2h, n0);
        store_acc<false>(t, X, kLS, m0, n0);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += X[(ty + 16 * i) * kLS + tx + 16 * j];
    } else {
        gemm_nt<4, 4>(acc, H1, w.W2, ty, 16, tx, 16);
    }
    // the score: four units per thread, 8 lanes, two warps
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc[i][j] = acc[i][j] > 0.f ? acc[i][j] : 0.f;
            s = __fmaf_rn(w3[j], acc[i][j], s);
        }
#pragma unroll
        for (int m = 1; m < 8; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        if ((lane & 7) == 0) SP[(warp & 1) * kGradRows + ty + 16 * i] = s;
    }
    __syncthreads();
    float* out = partial + (size_t)blockIdx.x * kPartStride;
    float lsum = 0.f, dsum = 0.f;
    if (tid < kGradRows) {
        const float s = w.b3 + (SP[tid] + SP[kGradRows + tid]);
        const float yv = Fs[tid * kL1 + 7];
        const bool valid = r0 + tid < nb;
        const float sg = sigmoid(s);
        const float ds = valid ? (pos_weight * yv * (sg - 1.f) + (1.f - yv) * sg) / (float)nb : 0.f;
        const float ls = valid ? pos_weight * yv * softplus(-s) + (1.f - yv) * softplus(s) : 0.f;
        DS[tid] = ds;
        lsum = ls;
        dsum = ds;
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            lsum += __shfl_xor_sync(0xffffffffu, lsum, m);
            dsum += __shfl_xor_sync(0xffffffffu, dsum, m);
        }
    }
    __syncthreads();
    if (tid == 32) { SP[0] = lsum; SP[1] = dsum; }   // the second warp's sums, for thread 0 below
    // dL/da2 = ds w3 [h2 > 0]; its column sums (b2) and those of ds h2 (w3)
    {
        float gw[4] = {0.f, 0.f, 0.f, 0.f}, gb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float ds = DS[ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float d2 = acc[i][j] > 0.f ? ds * w3[j] : 0.f;
                gw[j] = __fmaf_rn(ds, acc[i][j], gw[j]);
                gb[j] += d2;
                if constexpr (TC) D2h[(ty + 16 * i) * kTS + tx + 16 * j] = __float2bfloat16_rn(d2);
                else D2[(ty + 16 * i) * kLS + tx + 16 * j] = d2;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int m = 8; m < 32; m <<= 1) {
                gw[j] += __shfl_xor_sync(0xffffffffu, gw[j], m);
                gb[j] += __shfl_xor_sync(0xffffffffu, gb[j], m);
            }
            if (lane < 8) {
                red[(warp >> 1) * 512 + tx + 16 * j] = gw[j];
                red[(warp >> 1) * 512 + 64 + tx + 16 * j] = gb[j];
            }
        }
    }
    __syncthreads();
    if (tid < 128) {
        const float g = (red[tid] + red[512 + tid]) + (red[1024 + tid] + red[1536 + tid]);
        put<ADD>(out + (tid < 64 ? kOffW3 : kOffB2 - 64) + tid, g);
        if (tid == 0) {
            put<ADD>(out + kNPar, (lsum + SP[0]) / (float)nb);
            put<ADD>(out + kOffB3, dsum + SP[1]);
        }
    }
    float da[4][4] = {};   // dL/da1 before its mask: rows ty + 16 i, units 4 tx .. + 3
    if constexpr (TC) {
        float t[4][4];
        warp_mma<true, true>(t, D2h, m0, H1h, n0);         // dW2 = dA2^T H1
        store_acc<ADD>(t, out + kOffW2, 64, m0, n0);
        warp_mma<false, true>(t, D2h, m0, W2h, n0);        // dA2 W2
        store_acc<false>(t, X, kLS, m0, n0);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = *reinterpret_cast<const float4*>(X + (ty + 16 * i) * kLS + 4 * tx);
            da[i][0] = v.x; da[i][1] = v.y; da[i][2] = v.z; da[i][3] = v.w;
        }
    } else {
        // dW2 = dA2^T H1: units 4 ty .. + 3, inputs 4 tx .. + 3, rows ascending
        {
            float g[4][4] = {};
#pragma unroll 4
            for (int r = 0; r < kGradRows; ++r) {
                const float4 a = *reinterpret_cast<const float4*>(D2 + r * kLS + 4 * ty);
                const float4 b = *reinterpret_cast<const float4*>(H1 + r * kLS + 4 * tx);
                const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) g[i][j] = __fmaf_rn(av[i], bv[j], g[i][j]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                put4<ADD>(out + kOffW2 + (4 * ty + i) * 64 + 4 * tx, g[i]);
        }
        // dA2 W2
#pragma unroll 2
        for (int o = 0; o < 64; o += 4) {
            float4 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(D2 + (ty + 16 * i) * kLS + o);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 b = *reinterpret_cast<const float4*>(w.W2 + (o + e) * kLS + 4 * tx);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float av = e == 0 ? a[i].x : e == 1 ? a[i].y : e == 2 ? a[i].z : a[i].w;
                    da[i][0] = __fmaf_rn(av, b.x, da[i][0]);
                    da[i][1] = __fmaf_rn(av, b.y, da[i][1]);
                    da[i][2] = __fmaf_rn(av, b.z, da[i][2]);
                    da[i][3] = __fmaf_rn(av, b.w, da[i][3]);
                }
            }
        }
    }
    // W1 and b1 (the feature row's seventh entry is 1): [unit][8] per group of four warps
    {
        float g[4][7] = {};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float4 h;
            if constexpr (TC) {
                const uint2 v = *reinterpret_cast<const uint2*>(H1h + (ty + 16 * i) * kTS + 4 * tx);
                h = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                                __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
            } else {
                h = *reinterpret_cast<const float4*>(H1 + (ty + 16 * i) * kLS + 4 * tx);
            }
            const float4* fp = reinterpret_cast<const float4*>(Fs + (ty + 16 * i) * kL1);
            const float4 fa = fp[0], fb = fp[1];
            const float hv[4] = {h.x, h.y, h.z, h.w}, f[7] = {fa.x, fa.y, fa.z, fa.w, fb.x, fb.y, fb.z};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float d1 = hv[j] > 0.f ? da[i][j] : 0.f;
#pragma unroll
                for (int k = 0; k < 7; ++k) g[j][k] = __fmaf_rn(d1, f[k], g[j][k]);
            }
        }
        __syncthreads();   // the sums above have been read
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                float v = g[j][k];
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (lane < 8) red[(warp >> 1) * 512 + k * 64 + 4 * tx + j] = v;
            }
    }
    __syncthreads();
    for (int q = tid; q < 448; q += 256) {
        const int k = q >> 6, o = q & 63;
        const float g = (red[q] + red[512 + q]) + (red[1024 + q] + red[1536 + q]);
        put<ADD>(out + (k < 6 ? kOffW1 + o * 6 + k : kOffB1 + o), g);
    }
}

// Sums the partial gradients (and losses) of `blocks` CTAs in a fixed order
// (warp w the CTAs w, w + 8, ..., then the eight warps; lane = parameter, eight
// loads in flight); then optionally Adam: m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2,
// w -= lr (m / bc1) / (sqrt(v / bc2) + eps), with bc1/bc2 the bias corrections.
__global__ __launch_bounds__(256) void k_mlp_reduce(const float* partial, int blocks, float* grad_out,
                                                    float* loss_out, float* master, float* mom, float* vel,
                                                    __nv_bfloat16* Wb, int adam, float lr, float b1, float b2,
                                                    float eps, float bc1, float bc2)
{
    __shared__ float sum[8][32];
    const int q = blockIdx.x * 32 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
    float g = 0.f;
    pdl_wait();
    pdl_trigger();
    if (q <= kNPar) {
#pragma unroll 8
        for (int b = warp; b < blocks; b += 8) g += partial[(size_t)b * kPartStride + q];
    }
    sum[warp][threadIdx.x & 31] = g;
    __syncthreads();
    if (warp || q > kNPar) return;
    g = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k += 2) g += sum[k][threadIdx.x] + sum[k + 1][threadIdx.x];
    if (q == kNPar) {
        if (loss_out) *loss_out = g;
        return;
    }
    if (grad_out) grad_out[q] = g;
    if (!adam) return;
    const float m = b1 * mom[q] + (1.f - b1) * g;
    const float v = b2 * vel[q] + (1.f - b2) * g * g;
    mom[q] = m;
    vel[q] = v;
    const float wq = master[q] - lr * (m / bc1) / (sqrtf(v / bc2) + eps);
    master[q] = wq;
    Wb[q] = __float2bfloat16_rn(wq);
}

__global__ void k_round_bf16(const float* __restrict__ master, __nv_bfloat16* Wb)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < kNPar) Wb[q] = __float2bfloat16_rn(master[q]);
}

// ---------------------------------------------------------------------------
// flags[4] = improved during the iteration just finished, flags[3] = replica
// whose row was last copied into best_x, flags[5] = log slot of this entry.
__global__ __launch_bounds__(256) void k_log(const float* __restrict__ F, int n, int ld, const uint8_t* __restrict__ best_x,
                                             uint8_t* prev_x, const int32_t* __restrict__ flags, float* LF,
                                             uint8_t* LY, int32_t* lrep)
{
    if (!flags[4]) return;
    const int p = flags[3], slot = flags[5];
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j == 0) lrep[slot] = p;
    if (j >= n) return;
    const float* src = F + ((size_t)p * ld + j) * 6;
    float* dst = LF + ((size_t)slot * n + j) * 6;
#pragma unroll
    for (int k = 0; k < 6; ++k) dst[k] = src[k];
    const uint8_t b = best_x[j];
    LY[(size_t)slot * n + j] = b ^ prev_x[j];
    prev_x[j] = b;
}

// ---------------------------------------------------------------------------
cudaError_t launch_features(const Dev& d, int t, const int32_t* iter_dev, int alpha, int c, int32_t* gmax,
                            cudaStream_t s)
{
    k_gmax<<<d.R, 256, 0, s>>>(d.G, d.n, d.ld, gmax);
    dim3 grid((d.ld + 255) / 256, d.R);
    k_features<<<grid, 256, 0, s>>>(d, t, iter_dev, alpha, c, gmax);
    note_launch(2);
    return cudaGetLastError();
}

template <int RT>
static cudaError_t launch_score_rt(const float* F, long long rows, const void* Wb, float* out, cudaStream_t s)
{
    const long long grid = (rows + 16 * RT - 1) / (16 * RT);
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    const int smem = (int)(sizeof(ScoreNet) + sizeof(float) * 16 * RT * (kL1 + kLS));
    cudaError_t e = cudaFuncSetAttribute(k_score<RT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_score<RT><<<(unsigned)grid, 128, smem, s>>>(F, rows, reinterpret_cast<const __nv_bfloat16*>(Wb), out);
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_score(const float* F, long long rows, const void* Wb, float* out, cudaStream_t s)
{
    if (rows <= 0) return cudaSuccess;
    // Every CTA loads all weights, so small tiles pay only while the SMs would idle otherwise.
    // us with 16, 32, 64, 128 rows per CTA (launches in a graph): 100 rows 3.15, 3.30, 3.75, 5.2;
    // 1000 3.44, 3.42, 3.80, 5.3; 2400 4.24, 3.88, 4.04, 5.5; 4000 5.5, 4.18, 4.21, 5.6; 5000 6.6,
    // 5.38, 4.32, 5.6; 25 000 19, 12.2, 8.4, 9.4 (9729 to 19 456 rows: 128 per CTA 5 % ahead of
    // 64).  Back to back 45 000 rows take 14.5 with 64 and 128, 50 000 16.5 and 14.6, 320 000 70
    // and 60: 64 rows as long as one wave of five CTAs per SM holds them all.
    const long long sms = device_sm_count();
    if (rows > 64 * 5 * sms) return launch_score_rt<8>(F, rows, Wb, out, s);
    if (rows > 32 * sms) return launch_score_rt<4>(F, rows, Wb, out, s);
    if (rows > 8 * sms) return launch_score_rt<2>(F, rows, Wb, out, s);
    return launch_score_rt<1>(F, rows, Wb, out, s);
}

size_t mlp_partial_floats(long long batch)
{
    const long long ctas = (batch + kGradRows - 1) / kGradRows;
    return (size_t)(ctas < kGradCtas ? ctas : kGradCtas) * kPartStride;   // 77 MB at most
}

cudaError_t launch_mlp_grad(const float* F, const uint8_t* y, long long rows, long long batch, uint32_t step,
                            uint32_t k0, uint32_t k1, const void* Wb, float pos_weight, float* partial,
                            float* grad_out, float* loss_out, float* master, float* mom, float* vel, void* Wb_out,
                            int adam, float lr, float b1, float b2, float eps, float bc1, float bc2, cudaStream_t s,
                            bool tensor_cores, bool chained)
{
    const long long nb = batch < rows ? batch : rows;
    const long long ctas = (nb + kGradRows - 1) / kGradRows;
    const int blocks = (int)(ctas < kGradCtas ? ctas : kGradCtas);
    const size_t smem = sizeof(NetTile) + sizeof(float) * (kGradRows * (kL1 + 2 * kLS) + 4 * 512 + 3 * kGradRows +
                                                           (tensor_cores ? kGradRows * kLS : 0));
    // The reduction is launched while the gradient still runs, and the gradient of the next
    // training step (`chained`) while the reduction does: one gradient of 8192 rows 16.5 -> 14.4 us,
    // ten training steps 268 -> 223 us with the copies around them (not while a graph is captured,
    // so that its nodes keep plain edges)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool plain = cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    // A launch of at most kGradCtas CTAs; the CTAs of the next one add to the same partial
    // sums, so that the scratch does not grow with the rows (at 40 M rows 11.7 GB without)
    cudaError_t e;
    for (long long c0 = 0; c0 < ctas; c0 += kGradCtas) {
        auto kern = c0 ? (tensor_cores ? k_mlp_grad<true, true> : k_mlp_grad<false, true>)
                       : (tensor_cores ? k_mlp_grad<true, false> : k_mlp_grad<false, false>);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        cfg.gridDim = dim3((unsigned)(ctas - c0 < kGradCtas ? ctas - c0 : kGradCtas));
        cfg.numAttrs = c0 == 0 && chained && !plain ? 1 : 0;
        e = cudaLaunchKernelEx(&cfg, kern, F, y, rows, batch, step, k0, k1,
                               reinterpret_cast<const __nv_bfloat16*>(Wb), pos_weight, partial, c0 * kGradRows);
        if (e != cudaSuccess) return e;
        note_launch(1);
    }
    cfg.gridDim = dim3((kNPar + 1 + 31) / 32);
    cfg.dynamicSmemBytes = 0;
    cfg.numAttrs = plain ? 0 : 1;
    e = cudaLaunchKernelEx(&cfg, k_mlp_reduce, (const float*)partial, blocks, grad_out, loss_out, master, mom, vel,
                           reinterpret_cast<__nv_bfloat16*>(Wb_out), adam, lr, b1, b2, eps, bc1, bc2);
    if (e != cudaSuccess) return e;
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_round_bf16(const float* master, void* Wb, cudaStream_t s)
{
    k_round_bf16<<<(kNPar + 255) / 256, 256, 0, s>>>(master, reinterpret_cast<__nv_bfloat16*>(Wb));
    note_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_log(const Dev& d, uint8_t* prev_x, float* LF, uint8_t* LY, int32_t* lrep, cudaStream_t s)
{
    k_log<<<(d.n + 255) / 256, 256, 0, s>>>(d.F, d.n, d.ld, d.best_x, prev_x, d.flags, LF, LY, lrep);
    note_launch(1);
    return cudaGetLastError();
}

}  // namespace icd2s
