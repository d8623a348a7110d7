// kernels_anneal.cu -- the emulated Ising machine (Eq. 4, Algorithm 4).
//
// One warp per subQUBO S (m <= 32 P variables, ascending indices).  Lane l
// owns the P positions b = l + 32 q (q = 0..P-1): a sweep visits the blocks of
// 32 consecutive positions one after the other, one position of a block per
// lane.
//
// Gather (Eq. 4): Q' = Q[S, S] is staged as int8 in shared memory, one row per
// position, 32 P + 16 bytes apart (16-byte loads of 8 consecutive rows then
// fall in different banks); the diagonal is stored as 0, so a flip leaves the
// flipped position's own field alone.  The boundary bias
// b_i = sum_{j not in S} 2 Q_ij x_j is never formed explicitly: the local gain
// of position a in the biased subQUBO,
// (1 - 2 x_a)(Q_aa + b_a + 2 sum_{c in S, c != a} Q_ac x_c), equals the global
// gain g_a, which the solution set already tracks exactly; so the gains of S
// are read straight from G.
//
// Anneal: sweeps k = 0..K-1 visit positions 0..m-1 in order; attempt (k, b)
// draws u = Philox(ctr = (k / 4, (TAG_ANNEAL << 24) | b, slot, iter)).word[k mod 4]
// and accepts iff l_b <= 0 or l_b * BETA[k] < NLOG[u >> 20].  For integer
// gains this is l_b <= LIM[k][u >> 20] with LIM[k][j] = floor((NLOG[j] - 1) /
// BETA[k]) (0 when NLOG[j] = 0, unbounded when BETA[k] = 0): a per-schedule
// table built once on the device (k_limtab), so an attempt costs one
// L1-resident load and one compare.  Each lane draws one Philox block per
// owned position every 4 sweeps, so no random words are wasted or exchanged.
//
// Lanes keep the sign-free field h_b = (1 - 2 x_b) l_b: a flip of a adds
// 2 Q'_ab (1 - 2 x_a) to every h_b and only negates the sign of a itself.
//
// A block of 32 positions is decided as a whole.  The decisions a_0 .. a_31 of
// the one-at-a-time sweep satisfy
//     a_L = [ sg_L (h_L + sum_{k < L} a_k f_k Q'_Lk) <= lim_L ],  f_k = 2 (1 - 2 x_k),
// and are the only solution, because a_L depends on the earlier ones alone.
// The warp starts from the decisions against the current fields and takes all
// 32 again, each against the last decisions of the positions before it, until
// none changes.  After i rounds the first i decisions are final, so this ends
// (in at most 33 rounds) with the sequential trajectory bit for bit; in
// practice a decision seldom hangs on an earlier one (its threshold lies
// thousands wide, a coupling moves it by about a hundred), and two or three
// rounds settle a block.  The sum over k is a row of Q' times the vector of
// factors f: the 32 factor bytes are exchanged through shared memory and each
// lane takes eight dp4a over its own row (Q' is symmetric, so the row is the
// column), the entries with k >= L masked out; the final factors then update
// every field the same way.
//
// What bounds it: the chain of a round -- ballot, factor bytes through shared
// memory, dp4a, compare, ballot -- with one warp per scheduler.  One position
// decided per ballot (a chain of about 46 cycles each) took 1.47 ms on the
// n = 2500, m = 64, 1024-sweep, 128-subQUBO launch; blocks of 32 take 0.40 ms (some
// 400 cycles per block, 1.5 rounds on average).  Above 64 positions the rows of Q' a
// block needs are loaded before its rounds, so that they arrive while the rounds
// run: m = 100, 32 subQUBOs, 1024 sweeps 1.13 -> 1.01 ms, m = 200, 256 sweeps 0.74 ->
// 0.63 ms (up to 64 positions the rows stay in registers and every sweep of four is
// unrolled).  A round of the uneven 32-256 batch of 4096 subQUBOs at n = 7000 (256
// sweeps, T 2000 -> 1) went from 8.3 ms to 2.6 ms, selection and write-back included.
//
// Output: the changed positions, either as a 0/1 mask [R][ldm] or appended
// to the replica's flip list (index | old x << 31) for k_apply; and the
// subQUBO energy change (from the start and end gains of the changed positions).
#include <climits>

#include "common.cuh"

namespace icd2s {

// Largest gain accepted by the test l * beta < thr (see above).
__device__ __forceinline__ int accept_limit(uint32_t thr, uint32_t beta)
{
    if (thr == 0u) return 0;        // no positive gain passes
    if (beta == 0u) return INT_MAX; // every gain passes
    return (int)((thr - 1u) / beta);
}

// Shared memory of one warp: two buffers of 32 factor bytes, then the rows of Q'.
template <int P>
struct AnnealTile {
    static constexpr int rows = 64;             // offset of row 0
    static constexpr int stride = 32 * P + 16;  // bytes from row to row
    static constexpr size_t bytes = rows + (size_t)(32 * P) * stride;
};

// sum over the 32 positions of a block of factor x entry: 32 signed bytes each
__device__ __forceinline__ int dot32(const int (&r)[8], const int (&f)[8])
{
    int a = 0, b = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        a = __dp4a(r[w], f[w], a);
        b = __dp4a(r[w + 4], f[w + 4], b);
    }
    return a + b;
}

__device__ __forceinline__ void load32(const unsigned char* p, int (&r)[8])
{
    const int4 u = reinterpret_cast<const int4*>(p)[0], v = reinterpret_cast<const int4*>(p)[1];
    r[0] = u.x; r[1] = u.y; r[2] = u.z; r[3] = u.w;
    r[4] = v.x; r[5] = v.y; r[6] = v.z; r[7] = v.w;
}

// Anneals subQUBO s with the calling warp; `tile` is the warp's shared memory
// (AnnealTile<P>).  Warp-synchronous: no block-level barriers.
template <int P>
__device__ __forceinline__ void anneal_one(const Dev& d, const AnnealArgs& a, int s, int lane, unsigned char* tile)
{
    constexpr int RS = AnnealTile<P>::stride;
    unsigned char* const Qs = tile + AnnealTile<P>::rows;
    uint32_t iter = a.iter_dev ? (uint32_t)*a.iter_dev : a.iter;

    const int p = s / a.per_replica;
    const int* S = nullptr;
    int m;
    int bbase = a.block_base;
    uint32_t slot = a.slot_base + (uint32_t)s;
    if (a.idx) {
        const int b0 = a.off[s];
        m = a.off[s + 1] - b0;
        S = a.idx + b0;
    } else {
        // contiguous blocks: block k = s mod per_replica of the launch's group for
        // replica p starts k blocks after block_base and counts as iteration iter + k
        // of Call_IM_Solution_Set; its random stream is the replica's (slot p)
        m = a.block_m;
        const int k = s - p * a.per_replica;
        bbase += k * a.block_m;
        iter += (uint32_t)k;
        slot = a.slot_base + (uint32_t)p;
    }
    const int ld = d.ld;

    int col[P];
    bool valid[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int b = lane + 32 * q;
        valid[q] = b < m;
        col[q] = valid[q] ? (S ? __ldg(S + b) : bbase + b) : 0;
    }
    // gather Q[S, S], diagonal and padding as 0 (rows up to the end of the last block)
    const int mr = (m + 31) & ~31;
#pragma unroll 4
    for (int r = 0; r < mr; ++r) {
        const int ir = r < m ? (S ? __ldg(S + r) : bbase + r) : 0;
        const int8_t* row = d.Q + (size_t)ir * ld;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const bool take = valid[q] && r < m && (lane + 32 * q != r);
            Qs[(size_t)r * RS + 32 * q + lane] = take ? (uint8_t)__ldg(row + col[q]) : (uint8_t)0;
        }
    }
    __syncwarp();

    // Owned positions keep the sign-free field h = (1 - 2x) l (l the gain) and
    // the sign sg = 1 - 2x, so l = sg h.  A flip of position a changes the
    // field of every other position b by 2 Q'_ab (1 - 2 x_a) -- one
    // multiply-add per owned position with a warp-uniform factor -- and leaves
    // its own field alone (Q'_aa is stored as 0); the flipped position only
    // changes its sign.
    int h[P], sg[P];
    unsigned X[P];         // warp-uniform: bit lane of X[q] = x at position lane + 32 q
    const int32_t* grow = d.G + (size_t)p * ld;
    const uint8_t* xrow = d.X + (size_t)p * ld;
    unsigned x0 = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int xv = valid[q] ? (int)xrow[col[q]] : 0;
        sg[q] = 1 - 2 * xv;
        h[q] = valid[q] ? sg[q] * grow[col[q]] : 0;
        x0 |= (unsigned)xv << q;
        X[q] = __ballot_sync(0xffffffffu, xv != 0);
    }
    // The anneal's energy change comes at the end from the gains alone: for the
    // set F of positions whose value changed, E(x') - E(x) = (1/2) sum_{i in F}
    // (g_i(x) - g_i(x')) (flip them one after the other), so no step of a sweep
    // tracks it.  g0 = the gains at the start.
    int g0[P];
#pragma unroll
    for (int q = 0; q < P; ++q) g0[q] = sg[q] * h[q];

    // bytes k < lane of the 32 bytes of a block (the positions decided before this lane's)
    int below[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int c = lane - 4 * w;
        below[w] = c <= 0 ? 0 : (c >= 4 ? -1 : (int)((1u << (8 * c)) - 1u));
    }
    // up to 64 positions the owned rows stay in registers
    constexpr bool kRegs = P <= 2;
    // (of the own block, [q][q], the entries with k >= L; those below apart)
    int rows[kRegs ? P : 1][kRegs ? P : 1][8], lows[kRegs ? P : 1][8];
    if constexpr (kRegs) {
#pragma unroll
        for (int q2 = 0; q2 < P; ++q2)
#pragma unroll
            for (int q = 0; q < P; ++q) {
                load32(Qs + (size_t)(lane + 32 * q2) * RS + 32 * q, rows[q2][q]);
                if (q2 == q) {
#pragma unroll
                    for (int w = 0; w < 8; ++w) {
                        lows[q][w] = rows[q][q][w] & below[w];
                        rows[q][q][w] &= ~below[w];
                    }
                }
            }
    }
    unsigned char* const fbuf = tile;
    int cur = 0;   // the factor buffer written next

    // One sweep: block by block (see above).
    auto sweep = [&](const int (&lim)[P]) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
            if (32 * q >= m) break;
            const int hq = h[q];
            unsigned A = __ballot_sync(0xffffffffu, sg[q] * hq <= lim[q]);
            if (A == 0u) continue;   // nothing accepted: no field changes
            int low[8], up[8], f[8], all;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                if constexpr (kRegs) {
                    low[w] = lows[q][w];
                    up[w] = rows[q][q][w];
                }
            }
            // rows of the other blocks, on their way while the rounds run (a load does not
            // move over the rounds' exchanges by itself)
            int rest[kRegs ? 1 : P][8];
            if constexpr (!kRegs) {
                load32(Qs + (size_t)(lane + 32 * q) * RS + 32 * q, up);
#pragma unroll
                for (int q2 = 0; q2 < P; ++q2)
                    if (q2 != q && 32 * q2 < m) load32(Qs + (size_t)(lane + 32 * q2) * RS + 32 * q, rest[q2]);
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                    low[w] = up[w] & below[w];
                    up[w] &= ~below[w];
                }
            }
            const int fs = 2 * sg[q];
            while (true) {
                // two buffers: a round's factors are read before the round after the next writes
                unsigned char* fb = fbuf + 32 * cur;
                cur ^= 1;
                fb[lane] = (uint8_t)(((A >> lane) & 1u) ? fs : 0);
                __syncwarp();
                load32(fb, f);
                const int sum = dot32(low, f);
                if constexpr (kRegs) all = sum + dot32(up, f);   // beside the vote, for the last round
                else all = sum;
                const unsigned B = __ballot_sync(0xffffffffu, sg[q] * (hq + sum) <= lim[q]);
                if (B == A) break;
                A = B;
            }
            h[q] = hq + all + (kRegs ? 0 : dot32(up, f));
#pragma unroll
            for (int q2 = 0; q2 < P; ++q2) {
                if (q2 == q) continue;
                if constexpr (kRegs) {
                    h[q2] += dot32(rows[q2][q], f);
                } else if (32 * q2 < m) {
                    h[q2] += dot32(rest[q2], f);
                }
            }
            sg[q] = ((A >> lane) & 1u) ? -sg[q] : sg[q];
            X[q] ^= A;
        }
    };

    // A Philox block of each owned position covers 4 sweeps; the limits of the next
    // 4 sweeps are looked up (the table lies in L2) while the present 4 run
    auto limits_of = [&](int k4, int (&out)[4][P]) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const u32x4 u = philox10((uint32_t)(k4 >> 2), (kTagAnneal << 24) | (uint32_t)(lane + 32 * q), slot, iter,
                                     d.k0, d.k1);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int k = min(k4 + r, a.sweeps - 1);
                out[r][q] = __ldg(a.limtab + (size_t)k * 4096 + (u.v[r] >> 20));
            }
        }
    };
    int ahead[4][P];
    limits_of(0, ahead);
#pragma unroll 1
    for (int k4 = 0; k4 < a.sweeps; k4 += 4) {
        int now[4][P];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < P; ++q) now[r][q] = valid[q] ? ahead[r][q] : INT_MIN;
        if (k4 + 4 < a.sweeps) limits_of(k4 + 4, ahead);
        const int kn = min(4, a.sweeps - k4);
        if (P <= 2 && kn == 4) {
#pragma unroll
            for (int r = 0; r < 4; ++r) sweep(now[r]);
            continue;
        }
#pragma unroll 1
        for (int r = 0; r < kn; ++r) {
            int lim[P];
#pragma unroll
            for (int q = 0; q < P; ++q) {
                lim[q] = now[0][q];
                now[0][q] = now[1][q];
                now[1][q] = now[2][q];
                now[2][q] = now[3][q];
            }
            sweep(lim);
        }
    }

    unsigned changed = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) changed |= (unsigned)(valid[q] && (((X[q] >> lane) & 1u) != ((x0 >> q) & 1u))) << q;
    if (a.mask) {
#pragma unroll
        for (int q = 0; q < P; ++q)
            if ((changed >> q) & 1u) a.mask[(size_t)p * a.ldm + col[q]] = 1;
    } else {
        const int cnt = __popc(changed);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        int base = 0;
        if (lane == 0 && total > 0) base = atomicAdd(&d.FCNT[p], total);
        base = __shfl_sync(0xffffffffu, base, 0);
        int pos = base + incl - cnt;
        int32_t* fl = d.FL + (size_t)p * ld;
#pragma unroll
        for (int q = 0; q < P; ++q)
            if ((changed >> q) & 1u) {
                if (pos < ld) fl[pos] = col[q] | (int)(((x0 >> q) & 1u) << 31);  // a list never exceeds n entries
                ++pos;
            }
    }
    long long dEl = 0;  // twice the energy change
#pragma unroll
    for (int q = 0; q < P; ++q)
        if ((changed >> q) & 1u) dEl += (long long)g0[q] - (long long)(sg[q] * h[q]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dEl += __shfl_xor_sync(0xffffffffu, dEl, o);
    if (lane == 0) {
        if (a.dE) a.dE[s] = dEl / 2;
        if (a.attempts_acc) atomicAdd(reinterpret_cast<unsigned long long*>(a.attempts_acc),
                                      (unsigned long long)a.sweeps * (unsigned long long)m);
    }
}

// One warp per subQUBO, subQUBO s = CTA * warps + warp (sizes up to 32 P).
template <int P>
__global__ __launch_bounds__(128) void k_anneal(Dev d, AnnealArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int s = blockIdx.x * wpb + wib;
    if (s >= a.count) return;  // whole warp leaves; no block-level barriers below
    const int se = a.group_stride > 0 ? s * a.group_stride + a.group_k : s;
    anneal_one<P>(d, a, se, lane, smem + (size_t)wib * AnnealTile<P>::bytes);
}

// Persistent batch of subQUBOs of uneven size: every warp takes the next
// subQUBO of its size class from a device queue in largest-first order (a.order,
// sizes descending, built by k_sizes) and anneals it with the narrowest lane
// layout that fits its size.  A class is a launch of its own with the shared memory
// its largest size needs, and the classes run side by side: with one tile size
// for all, three subQUBOs of up to 256 fitted an SM (and its four schedulers) even
// where most were half as large.  Each queue is one counter; no warp ever waits
// on another, and each subQUBO's result does not depend on which warp runs it.
template <int PMAX>
__global__ __launch_bounds__(128) void k_anneal_queue(Dev d, AnnealArgs a, int cls)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char* tile = smem + (size_t)wib * AnnealTile<PMAX>::bytes;
    const int end = a.queue[kAnnealClasses + cls];
    while (true) {
        int next = 0;
        if (lane == 0) next = atomicAdd(a.queue + cls, 1);
        next = __shfl_sync(0xffffffffu, next, 0);
        if (next >= end) break;
        const int s = a.order[next];
        const int m = a.off[s + 1] - a.off[s];
        if constexpr (PMAX == 2) {
            if (m <= 32) anneal_one<1>(d, a, s, lane, tile);
            else anneal_one<2>(d, a, s, lane, tile);
        } else {
            anneal_one<PMAX>(d, a, s, lane, tile);
        }
        __syncwarp();  // the tile is reused by the next subQUBO
    }
}

// LIM[k][j] for the whole schedule: the largest gain that attempt (k, j) accepts.
__global__ void k_limtab(const uint32_t* __restrict__ beta, int sweeps, const uint32_t* __restrict__ nlog,
                         int* __restrict__ lim)
{
    const size_t total = (size_t)sweeps * 4096;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x)
        lim[e] = accept_limit(nlog[e & 4095], beta[e >> 12]);
}

cudaError_t launch_limtab(const uint32_t* beta, int sweeps, const uint32_t* nlog, int* lim, cudaStream_t s)
{
    const size_t total = (size_t)sweeps * 4096;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_limtab<<<blocks, 256, 0, s>>>(beta, sweeps, nlog, lim);
    note_launch(1);
    return cudaGetLastError();
}

template <int P>
static cudaError_t launch_anneal_p(const Dev& d, const AnnealArgs& a, int wpb, cudaStream_t s)
{
    const size_t sm = (size_t)wpb * AnnealTile<P>::bytes;
    cudaError_t e = cudaFuncSetAttribute(k_anneal<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const int blocks = (a.count + wpb - 1) / wpb;
    k_anneal<P><<<blocks, 32 * wpb, sm, s>>>(d, a);
    note_launch(1);
    return cudaGetLastError();
}

// Persistent launch: as many warps as fit on the GPU at once (by shared
// memory), never more than there are subQUBOs.
template <int PMAX>
static cudaError_t launch_anneal_queue(const Dev& d, const AnnealArgs& a, int cls, int wpb, cudaStream_t s)
{
    const size_t sm = (size_t)wpb * AnnealTile<PMAX>::bytes;
    cudaError_t e = cudaFuncSetAttribute(k_anneal_queue<PMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int ctas_per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas_per_sm, k_anneal_queue<PMAX>, 32 * wpb, sm);
    if (e != cudaSuccess) return e;
    if (ctas_per_sm < 1) ctas_per_sm = 1;
    int blocks = device_sm_count() * ctas_per_sm;
    const int need = (a.count + wpb - 1) / wpb;
    if (blocks > need) blocks = need;
    k_anneal_queue<PMAX><<<blocks, 32 * wpb, sm, s>>>(d, a, cls);
    note_launch(1);
    return cudaGetLastError();
}

bool anneal_has_class(int cls, int m_min, int m_max)
{
    const int top = kAnnealBound[cls], bottom = cls + 1 < kAnnealClasses ? kAnnealBound[cls + 1] : 0;
    return m_max > bottom && m_min <= top;
}

cudaError_t launch_anneal_class(const Dev& d, const AnnealArgs& a, int cls, cudaStream_t s)
{
    if (a.count <= 0) return cudaSuccess;
    int wpb = a.warps_per_cta <= 0 ? 1 : (a.warps_per_cta > 4 ? 4 : a.warps_per_cta);
    if (cls == 0 && wpb > 3) wpb = 3;
    switch (cls) {
        case 0: return launch_anneal_queue<8>(d, a, cls, wpb, s);
        case 1: return launch_anneal_queue<6>(d, a, cls, wpb, s);
        case 2: return launch_anneal_queue<4>(d, a, cls, wpb, s);
        case 3: return launch_anneal_queue<2>(d, a, cls, wpb, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_anneal(const Dev& d, const AnnealArgs& a, cudaStream_t s)
{
    if (a.count <= 0) return cudaSuccess;
    const int m = a.m_max;
    // warps (subQUBOs) per CTA: shared memory is 1.6 / 5.1 / 18.1 / 39.1 / 68.1 KiB per warp
    int wpb = a.warps_per_cta;
    if (wpb <= 0) wpb = m <= 128 ? 2 : 1;
    if (m > 192 && wpb > 3) wpb = 3;
    if (wpb > 4) wpb = 4;
    if (m <= 32) return launch_anneal_p<1>(d, a, wpb, s);
    if (m <= 64) return launch_anneal_p<2>(d, a, wpb, s);
    if (m <= 128) return launch_anneal_p<4>(d, a, wpb, s);
    if (m <= 192) return launch_anneal_p<6>(d, a, wpb, s);
    if (m <= 256) return launch_anneal_p<8>(d, a, wpb, s);
    return cudaErrorInvalidValue;
}

}  // namespace icd2s
