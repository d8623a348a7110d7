// kernels_exact.cu -- exact Ising machine for small subQUBOs (m <= 24): the
// "precise solution" of a subQUBO (Section 3) by trying all 2^m assignments.
//
// One CTA of 256 threads per subQUBO.  With Q' = Q[S, S] (diagonal as 0) and
// the linear coefficients L_a, the objective of an assignment y (relative to
// y = 0) is f(y) = sum_a y_a L_a + 2 sum_{a<b} Q'_ab y_a y_b.  The positions
// are split in three: the lowest 5 (z), up to 11 that a thread walks in
// Gray-code order, and up to 8 that the thread index fixes.  A thread keeps,
// for its current upper assignment, E = f with z = 0 and the fields
// phi_a = L_a + 2 sum_b Q'_ab y_b of the low and the walked positions; a step of
// the walk flips one position (the same in every thread) and costs one 16-byte
// row and 16 dp4a.  Between two steps all 32 assignments z are tried:
//     T[z] = sum_a z_a phi_a + 2 sum_{a<b} Q'_ab z_a z_b,
// built by doubling, T[z + 2^a] = T[z] + phi_a + P_a[z] with P_a[z] =
// 2 sum_{b<a} Q'_ab z_b the same for the whole subQUBO (26 registers): one
// three-operand add per assignment and half a three-operand minimum.  The walk of
// one assignment at a time that this replaces spent 24 multiply-adds and as
// many byte extractions on each.
//
// Choice among equal objectives: the smallest y as the integer sum_a y_a 2^a.
// A thread keeps the best (f, upper assignment) in lexicographic order, the
// CTA takes the minimum, and one warp then finds the smallest z of that block.
// The gains of the current assignment are the global gains (Eq. 4's bias
// makes the subQUBO's local gain equal the global one), read from G.
//
// What bounds it: the integer ALU (about 2.2 instructions per assignment).
// 128 subQUBOs of m = 24 (the whole call): 4.46 -> 0.29 ms, 7.4 T assignments/s.
//
// Output as for the annealer: the positions that change, as a 0/1 mask or
// appended to the replica's flip list, and the objective change.
#include <climits>

#include "common.cuh"

namespace icd2s {

constexpr int kExactMaxM = 24;
constexpr int kExactRow = 32;       // bytes per staged row
constexpr int kExactThreads = 256;
constexpr int kExactLow = 5;        // positions tried together
constexpr int kExactTop = 8;        // positions fixed by the thread index (at most)
constexpr int kExactKeep = 16;      // fields a thread keeps: the low and the walked positions
constexpr int kExactPad = 1 << 26;  // linear coefficient of a missing position: never chosen

__global__ __launch_bounds__(kExactThreads) void k_exact(Dev d, AnnealArgs a)
{
    __shared__ __align__(16) int8_t qs[kExactMaxM * kExactRow];
    __shared__ int lin[kExactMaxM];                      // L_a
    __shared__ long long wbest[kExactThreads / 32];
    __shared__ unsigned s_x0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s = a.group_stride > 0 ? (int)blockIdx.x * a.group_stride + a.group_k : (int)blockIdx.x;
    const int p = s / a.per_replica;
    const int* S = nullptr;
    int m;
    int bbase = a.block_base;
    if (a.idx) {
        const int b0 = a.off[s];
        m = a.off[s + 1] - b0;
        S = a.idx + b0;
    } else {
        m = a.block_m;
        bbase += (s - p * a.per_replica) * a.block_m;  // block s mod per_replica of the group
    }
    const int ld = d.ld;
    auto var = [&](int r) { return S ? __ldg(S + r) : bbase + r; };

    // stage Q' with a zero diagonal and zero padding
    for (int e = tid; e < kExactMaxM * kExactRow; e += kExactThreads) {
        const int r = e / kExactRow, c = e % kExactRow;
        int8_t v = 0;
        if (r < m && c < m && r != c) v = d.Q[(size_t)var(r) * ld + var(c)];
        qs[e] = v;
    }
    __syncthreads();
    const int32_t* grow = d.G + (size_t)p * ld;
    const uint8_t* xrow = d.X + (size_t)p * ld;
    if (warp == 0) {   // x0, and L_a = (1 - 2 x_a) g_a - 2 sum_b Q'_ab x_b
        const int xv = lane < m ? (int)xrow[var(lane)] : 0;
        const unsigned x0 = __ballot_sync(0xffffffffu, xv != 0);
        if (lane < kExactMaxM) {
            int v = kExactPad;
            if (lane < m) {
                const int g = grow[var(lane)];
                v = xv ? -g : g;
                for (int b = 0; b < m; ++b)
                    if ((x0 >> b) & 1u) v -= 2 * (int)qs[lane * kExactRow + b];
            }
            lin[lane] = v;
        }
        if (lane == 0) s_x0 = x0;
    }
    __syncthreads();
    const unsigned x0 = s_x0;
    // f(y) from its definition
    auto objective = [&](unsigned y) -> int {
        int f = 0;
        for (int b = 0; b < m; ++b)
            if ((y >> b) & 1u) {
                f += lin[b];
                for (int c = 0; c < b; ++c)
                    if ((y >> c) & 1u) f += 2 * (int)qs[b * kExactRow + c];
            }
        return f;
    };

    const int up = m > kExactLow ? m - kExactLow : 0;       // positions above the low ones
    const int tb = up < kExactTop ? up : kExactTop;         // of which fixed per thread: the highest
    const int wb = up - tb;                                 // and walked: kExactLow .. kExactLow + wb - 1 (<= 11)
    const bool active = tid < (1 << tb);
    long long best = LLONG_MAX;                             // f << 32 | upper assignment
    if (active) {
        const unsigned top = (unsigned)tid << wb;           // upper assignment with the walked positions 0
        int E = objective(top << kExactLow);
        int phi[kExactKeep];
#pragma unroll
        for (int c = 0; c < kExactKeep; ++c) {
            phi[c] = c < kExactLow || c < kExactLow + wb ? lin[c] : 0;
            for (int b = kExactLow + wb; b < m; ++b)
                if ((top >> (b - kExactLow)) & 1u) phi[c] += 2 * (int)qs[b * kExactRow + c];
        }
        // P_a[z], z < 2^a
        int P1, P2[4], P3[8], P4[16];
        auto q2 = [&](int r, int c) { return 2 * (int)qs[r * kExactRow + c]; };
        P1 = q2(1, 0);
#pragma unroll
        for (int z = 0; z < 16; ++z) {
            int v2 = 0, v3 = 0, v4 = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if ((z >> b) & 1) {
                    if (b < 2) v2 += q2(2, b);
                    if (b < 3) v3 += q2(3, b);
                    v4 += q2(4, b);
                }
            if (z < 4) P2[z] = v2;
            if (z < 8) P3[z] = v3;
            P4[z] = v4;
        }
        int bf = INT_MAX;
        unsigned bu = 0u;
        // the best of the 32 assignments z of the upper assignment `u`
        auto block = [&](unsigned u) {
            int T[16];
            T[0] = 0;
            T[1] = phi[0];
            T[2] = phi[1];
            T[3] = phi[0] + phi[1] + P1;
#pragma unroll
            for (int z = 0; z < 4; ++z) T[4 + z] = T[z] + phi[2] + P2[z];
#pragma unroll
            for (int z = 0; z < 8; ++z) T[8 + z] = T[z] + phi[3] + P3[z];
            int lo = INT_MAX, hi = INT_MAX;
#pragma unroll
            for (int z = 0; z < 16; z += 2) {
                lo = min(lo, min(T[z], T[z + 1]));
                hi = min(hi, min(T[z] + phi[4] + P4[z], T[z + 1] + phi[4] + P4[z + 1]));
            }
            const int f = E + min(lo, hi);
            const bool better = f < bf || (f == bf && u < bu);
            bf = better ? f : bf;
            bu = better ? u : bu;
        };
        // flip walked position b (field fb): the same in every thread
        unsigned walk = 0u;
        auto flip = [&](int b, int fb) {
            const bool on = (walk >> b) & 1u;    // 1 -> 0 ?
            walk ^= 1u << b;
            E += on ? -fb : fb;
            const int4 r = *reinterpret_cast<const int4*>(qs + (kExactLow + b) * kExactRow);
            const int rw[4] = {r.x, r.y, r.z, r.w};
            const unsigned wt = on ? 0xfeu : 0x02u;
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
                for (int e = 0; e < 4; ++e) phi[4 * w + e] = __dp4a(rw[w], (int)(wt << (8 * e)), phi[4 * w + e]);
        };
        auto flip_any = [&](int b) {             // b not known at compile time
            int fb = 0;
#pragma unroll
            for (int c = kExactLow; c < kExactKeep; ++c) fb |= phi[c] & -(int)(c == kExactLow + b);
            flip(b, fb);
        };
        block(top);
        if (wb < 3) {
            for (unsigned u = 1; u < (1u << wb); ++u) {
                flip_any(__ffs(u) - 1);
                block(top | walk);
            }
        } else {
            // runs of 8 blocks: inside a run the flipped positions are 0 1 0 2 0 1 0
            // (known at compile time); between two runs it is ctz(u0) >= 3
#pragma unroll 1
            for (unsigned u0 = 0; u0 < (1u << wb); u0 += 8) {
                if (u0) {
                    flip_any(__ffs(u0) - 1);
                    block(top | walk);
                }
#pragma unroll
                for (int v = 1; v < 8; ++v) {
                    const int b = (v & 1) ? 0 : (v & 2) ? 1 : 2;
                    flip(b, phi[kExactLow + b]);
                    block(top | walk);
                }
            }
        }
        best = (long long)bf * 4294967296LL + (long long)bu;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other < best ? other : best;
    }
    if (lane == 0) wbest[warp] = best;
    __syncthreads();
    if (warp != 0) return;
#pragma unroll
    for (int w = 1; w < kExactThreads / 32; ++w) best = wbest[w] < best ? wbest[w] : best;
    // the block of 32 assignments with the smallest (f, upper assignment): lane = z
    const unsigned ubest = (unsigned)((unsigned long long)best & 0xffffffffull);
    const int fz = lane < (1 << (m < kExactLow ? m : kExactLow)) ? objective((ubest << kExactLow) | (unsigned)lane) : INT_MAX;
    const int fmin = __reduce_min_sync(0xffffffffu, fz);
    const unsigned zbest = (unsigned)__ffs(__ballot_sync(0xffffffffu, fz == fmin)) - 1u;
    const unsigned ybest = (ubest << kExactLow) | zbest;
    const int fbest = fmin - objective(x0);
    const unsigned changed = ybest ^ x0;

    // output: positions r with bit r of `changed`, lane r handles position r (m <= 24 < 32)
    const bool mine = lane < m && ((changed >> lane) & 1u);
    if (a.mask) {
        if (mine) a.mask[(size_t)p * a.ldm + var(lane)] = 1;
    } else {
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        const int total = __popc(bal);
        int base = 0;
        if (lane == 0 && total > 0) base = atomicAdd(&d.FCNT[p], total);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (mine) {
            const int pos = base + __popc(bal & ((1u << lane) - 1u));
            if (pos < ld) d.FL[(size_t)p * ld + pos] = var(lane) | (int)(((x0 >> lane) & 1u) << 31);
        }
    }
    if (lane == 0 && a.dE) a.dE[s] = fbest;
}

cudaError_t launch_exact(const Dev& d, const AnnealArgs& a, cudaStream_t s)
{
    if (a.count <= 0) return cudaSuccess;
    if (a.m_max > kExactMaxM) return cudaErrorInvalidValue;
    k_exact<<<a.count, kExactThreads, 0, s>>>(d, a);
    note_launch(1);
    return cudaGetLastError();
}

}  // namespace icd2s
