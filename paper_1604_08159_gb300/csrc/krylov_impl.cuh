#pragma once
// Device helpers shared by the kernels of the Krylov projection (Sec. 2.1):
// the grid barrier with bounded waits, sums of a warp's lanes in a fixed
// order, phi_1 of the projected system, and the end of a clustered launch.
// The kernels are in krylov_mma.cuh and krylov_stream.cuh (digit products:
// the vorticity form, and the velocity-Exner form while it fits), exner.cu
// (its kernel with FP64 dots) and rosenbrock.cu.
// On this part one warp issues at most one FP64 instruction per ~64 cycles
// (about one per 16 cycles per SM), so what uses them is organised around the
// count of FP64 instructions each warp issues.
#include <cooperative_groups.h>

#include <cstdlib>

#include <type_traits>

#include "kernels.h"
#include "operator.cuh"

namespace wrc {

namespace {

constexpr int kPT = 128;      // threads of the block that evaluates phi_1 for the Rosenbrock step
constexpr int kNV = 32;       // accumulator slots: basis vectors per pass (<= m + 1 <= 32)
constexpr int kOutP = 66;     // partial sums per block: two sets of (kNV dots + one product)
constexpr int kGhostLanes = 8;   // lanes per ghost value
constexpr int kGatherLane = 8;   // row terms per lane fetched ahead of their additions
static_assert(kGhostLanes * kGatherLane == kGhostRowMax, "one gather pass covers a whole interpolation row");

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Sum of x over the 32 lanes of a warp, returned to every lane, through 40
// doubles of shared memory ws in a fixed order: lane l < 8 adds lanes
// 4l..4l+3 pairwise, then every lane adds the eight sums pairwise.  Inside
// this kernel a shuffle tree on FP64 values was measured at ~600 cycles per
// level on this part; this takes 4 dependent FP64 additions and shared
// memory round trips.
__device__ __forceinline__ double warp_sum(double x, double* ws) {
    const int l = threadIdx.x & 31;
    ws[l] = x;
    __syncwarp();
    if (l < 8) ws[32 + l] = (ws[4 * l] + ws[4 * l + 1]) + (ws[4 * l + 2] + ws[4 * l + 3]);
    __syncwarp();
    const double* p = ws + 32;
    const double r = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
    __syncwarp();
    return r;
}

// Sums over each group of kGhostLanes (= 8) consecutive lanes of the NV
// values v[] of every lane, through NV * 32 doubles of shared memory ws: lane
// gl < NV of a group adds quantity gl of its group pairwise (7 FP64 additions
// for all quantities at once), and lane 0 of the group receives the sums in
// v[].  Same order in every block.
template <int NV>
__device__ __forceinline__ void group_sums(double (&v)[NV], double* ws) {
    static_assert(kGhostLanes == 8 && NV <= 8, "groups of eight lanes");
    const int lane = threadIdx.x & 31, gl = lane & 7, g8 = lane - gl;
#pragma unroll
    for (int q = 0; q < NV; ++q) ws[q * 32 + lane] = v[q];
    __syncwarp();
    double sum = 0.0;
    if (gl < NV) {
        const double* p = ws + gl * 32 + g8;
        sum = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
    }
    __syncwarp();
    if (gl < NV) ws[gl * 32 + g8] = sum;
    __syncwarp();
    if (gl == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = ws[q * 32 + lane];
    __syncwarp();
}

// Grid-wide barrier for a cooperative launch: one atomic per block on a
// counter whose top bit flips when the last block arrives (block 0 adds
// 2^31 - (G - 1), the others 1, so each barrier adds exactly 2^31).  The
// arrival is a release atomic and the wait polls with acquire loads (GPU
// scope; the barrier's __syncthreads extend both to the whole block), so the
// plain loads of the next phase see every block's writes; this measured
// ~0.2 us faster per barrier than __threadfence around a relaxed atomic.
// The wait of each block is bounded by limit_ns; a block that runs out sets
// bit 1 of *err, and every waiter leaves as soon as one of the stopping bits
// (kErrStop) of *err is set, so the kernel always returns.  Bit 4 (16) only
// reports an unclustered run of a clustered launch and stops nothing.
// The barrier spans the nb blocks of one problem (bid = block index within it).
// With a trace buffer, the arrival of each block and the release of block 0
// are stamped (phase index `ph`, counted by the caller).
constexpr int kErrStop = 2 | 4;   // a barrier wait ran out; a ghost row exceeded its capacity

__device__ bool grid_sync(unsigned* bar, int* err, unsigned long long limit_ns, int bid, int nb,
                          unsigned long long* trace = nullptr, int ph = 0) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (trace && ph < kTracePhases) trace[1 + (size_t)ph * (nb + 1) + bid] = gtimer();
        const unsigned inc = bid == 0 ? 0x80000000u - (unsigned)(nb - 1) : 1u;
        unsigned old;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(bar), "r"(inc) : "memory");
        volatile int* verr = err;
        const unsigned long long t0 = gtimer();
        while (true) {
            unsigned cur;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(bar) : "memory");
            if ((old ^ cur) & 0x80000000u) break;
            if (*verr & kErrStop) break;
            if (gtimer() - t0 > limit_ns) {
                atomicOr(err, 2);
                break;
            }
        }
        if (trace && ph < kTracePhases && bid == 0) trace[1 + (size_t)ph * (nb + 1) + nb] = gtimer();
    }
    __syncthreads();
    return (*(volatile int*)err & kErrStop) == 0;
}

// ---- phi_1 from the exponential of the augmented matrix ------------------
// y = phi_1(dt H_k) e_1 is the upper part of the last column of exp(M),
// M = [[dt H_k, e_1], [0, 0]] ((k+1) x (k+1)).  That column, exp(M) e_k, is
// computed as the action of the exponential by scaling and the truncated
// Taylor series: B = M / s, x <- sum_{i<=m} B^i x / i!  applied s times.
// With theta = |M|_inf / s (max row sum; the bound only needs a
// sub-multiplicative norm) the dropped tail is at most
// sum_{i>m} theta^i / i! of |x|, and (theta, m) is taken from
//   (1/4, 12), (1/2, 15), (1, 18), (2, 24), (4, 32),
// each pair keeping that tail below 1e-17, as the one with the fewest
// matrix-vector products s m (s = max(1, ceil(|M|_inf / theta))).  exp(B)
// shrinks no vector by more than e^-theta, so the relative truncation error
// is below 6e-16 per sub-step.  Each product is 32 x 32 in FP64 on one SM,
// so their count matters.  One warp, lane r holds row r.
constexpr int kPhiChoices = 5;
__constant__ double c_phi_theta[kPhiChoices] = {0.25, 0.5, 1.0, 2.0, 4.0};
__constant__ int c_phi_terms[kPhiChoices] = {12, 15, 18, 24, 32};
constexpr int kTaylorMax = 32;
__constant__ double c_inv[kTaylorMax + 1] = {
    0.0,       1.0 / 1,  1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,  1.0 / 6,  1.0 / 7,  1.0 / 8,
    1.0 / 9,   1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17,
    1.0 / 18,  1.0 / 19, 1.0 / 20, 1.0 / 21, 1.0 / 22, 1.0 / 23, 1.0 / 24, 1.0 / 25, 1.0 / 26,
    1.0 / 27,  1.0 / 28, 1.0 / 29, 1.0 / 30, 1.0 / 31, 1.0 / 32};

// Largest norm of the Taylor evaluation: a step with |dt H| above it (or not
// finite) has blown up; phi_1 is then not evaluated, y is set to NaN and the
// non-finite flag is raised, so that the step fails cleanly instead of
// looping over an unbounded number of sub-steps.
constexpr double kMaxPhiScale = 4096.0;

// phi_1 by one block of PT threads: lane r of warp w holds row r of M over
// the column group w (32 / (PT/32) columns); each product B x is summed per
// group, then over the groups by warp 0, which keeps x and the partial sum of
// the series (the four FP64 sub-pipes of the SM share the products).
// s_part: [PT/32][>= 32], s_x: [>= 32], s_int: [3]; y (m entries) in global memory.
template <int PT>
__device__ __forceinline__ void phi1_block(const double* __restrict__ H, int k, int m, double dt,
                                           double* __restrict__ y, int* __restrict__ flags,
                                           double (*s_part)[kNV + 1], double* s_x, int* s_int) {
    constexpr int G = PT / 32;
    constexpr int CPG = 32 / G;
    const int r = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c0 = w * CPG;
    double row[CPG];
    double rs = 0.0;
#pragma unroll
    for (int cc = 0; cc < CPG; ++cc) {
        const int c = c0 + cc;
        double v = 0.0;
        if (r < k && c < k) v = dt * H[(size_t)r * m + c];
        if (r == 0 && c == k) v = 1.0;
        row[cc] = v;
        rs += fabs(v);
    }
    s_part[w][r] = rs;
    __syncthreads();
    if (w == 0) {
        double t = 0.0;   // |row r|_1
        for (int q = 0; q < G; ++q) t += s_part[q][r];
        double nrm = t;   // |M|_inf
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nrm = fmax(nrm, __shfl_xor_sync(0xffffffffu, nrm, o));
        const bool blown = __any_sync(0xffffffffu, !(t == t)) || !(nrm <= kMaxPhiScale);
        if (r == 0) {
            int sb = 1, mb = kTaylorMax;
            if (!blown) {
                long best = 1L << 40;
                for (int q = 0; q < kPhiChoices; ++q) {
                    const int sq = nrm > c_phi_theta[q] ? (int)ceil(nrm / c_phi_theta[q]) : 1;
                    const long cost = (long)sq * c_phi_terms[q];
                    if (cost < best) {
                        best = cost;
                        sb = sq;
                        mb = c_phi_terms[q];
                    }
                }
            }
            s_int[0] = blown ? 1 : 0;
            s_int[1] = sb;
            s_int[2] = mb;
        }
    }
    __syncthreads();
    const int blown = s_int[0], s = s_int[1], mt = s_int[2];
    if (blown) {
        if (threadIdx.x == 0) atomicOr(flags, 1);
        for (int t = threadIdx.x; t < m; t += PT) y[t] = t < k ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
        return;
    }
    if (s > 1) {
        const double inv_s = 1.0 / s;
#pragma unroll
        for (int cc = 0; cc < CPG; ++cc) row[cc] *= inv_s;
    }
    double x = (w == 0 && r == k) ? 1.0 : 0.0;   // meaningful in warp 0
    for (int q = 0; q < s; ++q) {
        double acc = x;
        if (w == 0) s_x[r] = x;
        __syncthreads();
        for (int i = 1; i <= mt; ++i) {
            double pr = 0.0;
#pragma unroll
            for (int cc = 0; cc < CPG; ++cc) pr += row[cc] * s_x[c0 + cc];
            s_part[w][r] = pr;
            __syncthreads();
            if (w == 0) {
                double t = s_part[0][r];
                for (int g = 1; g < G; ++g) t += s_part[g][r];
                t *= c_inv[i];
                acc += t;
                s_x[r] = t;
            }
            __syncthreads();
        }
        x = acc;
    }
    if (w == 0 && r < m) y[r] = r < k ? x : 0.0;
}

// True for a finite double (exponent field not all ones), by integer
// operations on its high word (an FP64 comparison would take a warp's FP64
// issue slot for ~64 cycles).
__device__ __forceinline__ bool finite_bits(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }

// Exact float -> double by integer operations on the bits (sign, exponent
// rebiased by 1023 - 127, mantissa shifted by 29; infinities and NaNs keep
// the all-ones exponent): the conversion instruction runs on the FP64 pipe,
// the scarce one on this part, at two to three FP64 operations' cost.  A
// float subnormal (never met in practice) takes the conversion instruction.
__device__ __forceinline__ double f2d_exact(float x) {
    const unsigned f = __float_as_uint(x);
    const unsigned e8 = (f >> 23) & 0xffu;
    const unsigned m = f & 0x7fffffu;
    if (e8 == 0u && m != 0u) return (double)x;
    const unsigned e11 = e8 == 0xffu ? 0x7ffu : (e8 == 0u ? 0u : e8 + (1023u - 127u));
    const unsigned hi = (f & 0x80000000u) | (e11 << 20) | (m >> 3);
    return __hiloint2double((int)hi, (int)(m << 29));
}
__device__ __forceinline__ double dbl(double x) { return x; }
__device__ __forceinline__ double dbl(float x) { return f2d_exact(x); }

// End of a clustered launch of m Arnoldi steps' dots, `calls` of which this
// block has taken: wait for the second cluster barrier of the last of them
// (if there was one), then take part in the barriers of those it did not take
// (a breakdown, a failed grid barrier, a refusal), so that every block of a
// cluster passes exactly 2 m of them and none exits while a peer may still
// read its shared memory.
// (Only for a launch that formed its clusters.)
// Each of these waits ends: every block of the cluster reaches its own
// remaining barriers, all its grid-barrier waits being bounded.
__device__ __forceinline__ void cluster_finish(int calls, int m) {
    if (calls > 0) __cluster_barrier_wait();
    for (int c = calls; c < m; ++c) {
        __cluster_barrier_arrive();
        __cluster_barrier_wait();
        __cluster_barrier_arrive();
        __cluster_barrier_wait();
    }
}

}  // namespace

}  // namespace wrc
