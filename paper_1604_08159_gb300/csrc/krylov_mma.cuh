#pragma once
// The Krylov projection of the time step (Sec. 2.1) as one persistent
// cooperative kernel whose orthogonalisation runs on the tensor cores.
//
// Method: that of krylov_impl.cuh -- Arnoldi with classical Gram-Schmidt
// applied twice, the second pass delayed by one step -- with b itself (times
// a power of two, first_scale) taken as the first "u": step j applies A to u (z = A u), one reduction gives
// s = Q^T u, |u|^2, t = Q^T z and u.z, and
//   q_j = (u - Q s) / h,  h^2 = |u|^2 - |s|^2  (step 0: h = beta, q_0 = b / beta),
//   next u = (z - Q t - q_j qz) / h,  qz = (u.z - s.t) / h.
//
// What bounds it.  This part issues one FP64 warp instruction per ~65 cycles
// and SM sub-partition (measured: DFMA 64.7, DADD 64.6), an FP32 or integer
// one per cycle, and one mma.sync m16n8k16 (f16 in, f32 sums) per 8.8.  The
// dots and updates of the Gram-Schmidt passes were 60% of the FP64
// instructions; here they are exact integer sums on the tensor cores:
//  - every value is held as a 64-bit fixed-point number split into eight
//    signed base-256 digits, an f16 each (exact); the products of digit i
//    of one factor and digit k of the other, i + k = c, are summed in f32
//    accumulators that stay below 2^24, i.e. exactly, and the columns c are
//    joined in integers;
//  - basis vectors: |q| <= 1, so one fixed scale, 2^-61 per unit; u and z:
//    a scale per block (its largest value's exponent); s and t: one scale.
//    The digit products beyond the eighth column are left out: a sum over
//    n points is off by less than n 2^-58 of the largest product (2^-61 a
//    product, root mean square), finer in norm than the rounding of an FP64
//    running sum over the same points, though not for every single entry.
//    Sums across warps, blocks and the grid are integer additions, exact and
//    independent of their order; how the points are dealt over blocks, whose
//    scales differ, still shows in the last bits.
// Layout: a block owns grid points and its share of the ghosts as columns of
// a table [row of the basis][column] in shared memory, as digits (halves) or
// as 64-bit integers whose digits are unpacked while they are loaded, so
// the basis is read from shared memory in both passes and never written to
// global memory.  Ghost values of the basis are columns too: their history
// terms sum(t_q Gb_q) come out of the same products as the points' updates.
// Roles within a step: eleven warps apply the operator while one finishes the
// last column of H; eight do the products; the interpolation rows of z at
// the ghosts are gathered while the sums are read; one warp does the scalars
// (h, qz) while the products of the updates run.
//
// Measured on GB300: see krylov_plan() in krylov.cu.
#include "exner_op.cuh"
#include "krylov_impl.cuh"

namespace wrc {

namespace {

constexpr int kMW = 12;               // warps: 0-7 products, 8 scalars, 9-11 (and 2-7) ghosts, all but 8 the operator
constexpr int kMT = 32 * kMW;
constexpr int kPW = 8;                // product warps
constexpr int kScr = 2560;            // scratch bytes per product warp (digit tile, dot sums, update sums)
constexpr int kTP = 80;               // pitch (bytes) of the s, t digit tile: 32 rows of the basis + pad
constexpr int kUP = 48;               // pitch of a unit's u, z digit tile: 16 points + pad
constexpr int kCP = 18;               // ints per basis row of a warp's dot sums
constexpr int kCopies = 8;            // copies of the global sums
constexpr unsigned long long kBias = 0x8080808080808080ull;

// Forms of the basis table, by the columns of a block:
//  kNarrow  at most 128 columns: digits as halves (16 bytes a value), 16
//           columns a product warp
//  kHalves  digits as halves, 32 columns a warp and turn
//  kWords   64-bit integers (8 bytes a value), digits unpacked while loaded:
//           twice the columns fit, at 20 more instructions per digit pair of
//           products
constexpr int kNarrow = 0, kHalves = 1, kWords = 2;

// Shared memory of a block: `cols` columns (its points, then its ghosts;
// multiples of 16), m + 1 rows.  nrc: ghosts whose interpolation rows (up to
// kRowCache terms) are kept here too, as room allows; -1: no room for the
// FP32 copy of H either.
constexpr int kRowCache = 64;
struct MmaLayout {
    int cols;
    int pitch;                                    // words (= 4 mod 16) or halves (= 8 mod 16) per row
    size_t q, us, zs, rz, vv, meta, gpos, glen, scr, tile, sH, sHf, rw, ri, bytes;
};
__host__ __device__ inline MmaLayout mma_layout(int form, int m, int ppb, int gpb, int nrc) {
    MmaLayout L;
    L.cols = ppb + gpb;
    L.pitch = form == kWords ? L.cols + 4 : L.cols + 8;
    size_t o = 0;
    L.q = o;    o += (size_t)(m + 1) * L.pitch * (form == kWords ? 8 : 16);
    L.us = o;   o += (size_t)L.cols * 8;
    L.zs = o;   o += (size_t)L.cols * 8;
    L.rz = o;   o += (size_t)gpb * 8;
    L.sH = o;   o += sizeof(double) * 32 * 33;
    L.sHf = o;  o += nrc < 0 ? 0 : sizeof(float) * 32 * 33;
    L.scr = o;  o += (size_t)kPW * kScr;
    L.tile = o; o += (size_t)kTP * 32;
    L.meta = o; o += (size_t)ppb * 4;
    L.gpos = o; o += (size_t)gpb * 4;
    L.glen = o; o += (size_t)gpb * 4;
    L.vv = o;   o += form == kNarrow ? (size_t)L.cols * 16 : 0;
    L.rw = o;   o += (size_t)(nrc < 0 ? 0 : nrc) * kRowCache * 8;
    L.ri = o;   o += (size_t)(nrc < 0 ? 0 : nrc) * kRowCache * 4;
    L.bytes = (o + 15) / 16 * 16;
    return L;
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void hmma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two bytes b, b' placed as 0x64bb, 0x64b'b' are the halves 1024 + b,
// 1024 + b'; minus 1152 they are the signed digits b - 128 (exact).
__device__ __forceinline__ unsigned unbias2(unsigned h) {
    unsigned r;
    asm("add.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0xe480e480u));
    return r;
}
// Digits 2q and 2q + 1 (q = 0: the most significant pair of a word) of two
// words as half2 (digit of x, digit of y) each.
__device__ __forceinline__ void digits2(unsigned x, unsigned y, int q, unsigned& d0, unsigned& d1) {
    const unsigned p = __byte_perm(x, y, q == 0 ? 0x6273 : 0x4051);
    d0 = unbias2(__byte_perm(p, 0x64646464u, 0x4140));
    d1 = unbias2(__byte_perm(p, 0x64646464u, 0x4342));
}
// One 64-bit number's digits as halves into a tile: digit i at row i.
__device__ __forceinline__ void put_digits(char* at, int pitch, unsigned long long x) {
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const unsigned v = w == 0 ? (unsigned)(x >> 32) : (unsigned)x;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned d = unbias2(__byte_perm(v, 0x64646464u, q == 0 ? 0x4243 : 0x4041));
            *reinterpret_cast<unsigned short*>(at + (4 * w + 2 * q) * pitch) = (unsigned short)d;
            *reinterpret_cast<unsigned short*>(at + (4 * w + 2 * q + 1) * pitch) = (unsigned short)(d >> 16);
        }
    }
}

__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Fixed point: round(x 2^(62 - E)), |x| < 2^E, E = emax - 1022 (emax the
// biased exponent of the scale), as a two's complement number plus kBias, so
// that its bytes are the digits + 128.  In integer operations; a subnormal
// counts as zero.
__device__ __forceinline__ unsigned long long fix62(double x, int emax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    unsigned long long y = e ? ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9 : 0ull;
    const int r = emax - e;
    if (r > 0) y = r < 63 ? (y + ((1ull << r) >> 1)) >> r : 0ull;
    else if (r < 0) y <<= 1;   // up to 2^(E + 1): a ghost value above the largest basis value
    if ((long long)b < 0) y = 0ull - y;
    return y + kBias;
}

// Paths for extreme values are kept out of line: the body of the step loop
// should stay within the instruction caches.
__device__ __noinline__ double scale_slow(double x, int k) { return scalbn(x, k); }
__device__ __noinline__ float scale_slow(float x, int k) { return scalbnf(x, k); }
__device__ __noinline__ double rsqrt_slow(double q) { return 1.0 / sqrt(q); }
// FP32 value of a double rounded towards zero, by integer operations (the
// conversion instruction takes an FP64 issue slot); |x| below 2^100, 0 below
// 2^-100.
__device__ __forceinline__ float d2f_trunc(double x) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const unsigned f = ((unsigned)(e - 1023 + 127) << 23) | ((unsigned)(hi & 0xfffff) << 3) |
                       ((unsigned)__double2loint(x) >> 29);
    return e < 1023 - 100 ? 0.f : __uint_as_float((hi & 0x80000000u) | f);
}
// A double that holds an FP32 value, as that value.
__device__ __forceinline__ float d2f_same(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    return e >= 1023 - 100 && e <= 1023 + 100 ? d2f_trunc(x) : (float)x;
}
// 1/sqrt(q): an FP32 seed y and one step of third order in the residual
// r = 1 - q y^2, y (1 + r/2 + 3 r^2/8), |r| < 2^-20 (five dependent FP64
// operations); q outside [2^-99, 2^99], negative or not finite takes the
// library's functions.
__device__ __forceinline__ double rsqrt_fast(double q) {
    const int hi = __double2hiint(q);
    const int e = (hi >> 20) & 0x7ff;
    if (hi >= 0 && e > 1023 - 99 && e < 1023 + 99) {
        const double y = f2d_exact(rsqrtf(d2f_trunc(q)));
        const double r = fma(-q, y * y, 1.0);
        return fma(y, r * fma(0.375, r, 0.5), y);
    }
    return rsqrt_slow(q);
}

// Grid-wide barrier, as grid_sync (krylov_impl.cuh), with what it leaves off
// the path: the phase is tracked by each block, so the arrival returns
// nothing; the error word is read once per 16 polls, and after the barrier by
// nobody (a block that gave up never arrives at the next one,
// where the others then stop).  `phase` is the counter's top bit after the
// last barrier.
__device__ __noinline__ bool grid_wait(unsigned* bar, int* err, unsigned long long limit_ns, int bid, int nb,
                                       unsigned phase, int* s_ok, unsigned long long* trace, int ph) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (trace && ph < kTracePhases) trace[1 + (size_t)ph * (nb + 1) + bid] = gtimer();
        const unsigned inc = bid == 0 ? 0x80000000u - (unsigned)(nb - 1) : 1u;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(inc) : "memory");
        const unsigned long long t0 = gtimer();
        int ok = 1;
        for (int n = 0;; ++n) {
            unsigned cur;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(bar) : "memory");
            if ((cur ^ phase) & 0x80000000u) break;
            if ((n & 15) == 15 && (*(volatile int*)err & kErrStop)) {
                ok = 0;
                break;
            }
            if (gtimer() - t0 > limit_ns) {
                atomicOr(err, 2);
                ok = 0;
                break;
            }
        }
        if (trace && ph < kTracePhases && bid == 0) trace[1 + (size_t)ph * (nb + 1) + nb] = gtimer();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// The same for an FP32 value (emax still biased as a double's).
__device__ __forceinline__ unsigned long long fix62(float x, int emax) {
    const unsigned b = __float_as_uint(x);
    const int e = (int)(b >> 23) & 0xff;
    unsigned long long y = e ? (unsigned long long)((b & 0x7fffffu) | 0x800000u) << 38 : 0ull;
    const int r = emax - (e + 896);
    if (r > 0) y = r < 63 ? (y + ((1ull << r) >> 1)) >> r : 0ull;
    else if (r < 0) y <<= 1;
    if ((int)b < 0) y = 0ull - y;
    return y + kBias;
}
// Biased exponent (as a double's) of an FP32 value.
__device__ __forceinline__ int expo(float x) {
    const int e = (__float_as_int(x) >> 23) & 0xff;
    return e == 0 ? 0 : (e == 0xff ? 0x7ff : e + 896);
}

// x 2^k for any double (an exponent addition where the result stays normal).
__device__ __forceinline__ double scale2(double x, int k) {
    const int e = expo(x);
    if (e != 0 && e != 0x7ff && e + k > 0 && e + k < 0x7ff)
        return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
    if (__double_as_longlong(x) << 1 == 0) return x;
    return scale_slow(x, k);
}
// The exponent by which a first vector b of largest magnitude below 2^(e - 1022)
// (e biased) is scaled: with b itself as the first u, z = A u, in the bulk
// type, has the scale of |b| |A| and u.z that of |b|^2 |A|; 0 (mid-range) in
// all but unusual units.
template <typename T>
__device__ __forceinline__ int first_scale(int e) {
    const int E = e - 1022;
    return e == 0 || e == 0x7ff || abs(E) <= (sizeof(T) == 4 ? 30 : 200) ? 0 : E;
}
// 2^k as a double, 0 below the normal range.
__device__ __forceinline__ double pow2d(int k) {
    return k <= -1023 ? 0.0 : __hiloint2double((min(k, 1023) + 1023) << 20, 0);
}

// y = phi_1(dt H_k) e_1 from the H of the block in shared memory (as
// phi1_block in krylov_impl.cuh: the scaled Taylor action, the same choices
// of sub-steps and terms), by eight warps; every thread of the block calls
// it.  The products' column groups are added pairwise.  Returns false for a
// blown-up step (y is then NaN).
__device__ __noinline__ bool phi1_mma(const double* sH, int k, double dt, double* y, double (*s_part)[33],
                                         double* s_x, int* s_int) {
    constexpr int G = kPW, CPG = 32 / G;
    const int r = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool on = w < G;
    const int c0 = w * CPG;
    double row[CPG];
    if (on) {
        double rs = 0.0;
#pragma unroll
        for (int cc = 0; cc < CPG; ++cc) {
            const int c = c0 + cc;
            double v = 0.0;
            if (r < k && c < k && r <= c + 1) v = dt * sH[r * 33 + c];
            if (r == 0 && c == k) v = 1.0;
            row[cc] = v;
            rs += fabs(v);
        }
        s_part[w][r] = rs;
    }
    __syncthreads();
    if (w == 0) {
        double t = 0.0;
        for (int q = 0; q < G; ++q) t += s_part[q][r];
        double nrm = t;
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
        if (w == 0) y[r] = r < k ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
        __syncthreads();
        return false;
    }
    if (on && s > 1) {
        const double inv_s = 1.0 / s;
#pragma unroll
        for (int cc = 0; cc < CPG; ++cc) row[cc] *= inv_s;
    }
    double x = (w == 0 && r == k) ? 1.0 : 0.0;
    for (int q = 0; q < s; ++q) {
        double acc = x;
        if (w == 0) s_x[r] = x;
        __syncthreads();
        for (int i = 1; i <= mt; ++i) {
            if (on) {
                double pr = 0.0;
#pragma unroll
                for (int cc = 0; cc < CPG; ++cc) pr += row[cc] * s_x[c0 + cc];
                s_part[w][r] = pr;
            }
            __syncthreads();
            if (w == 0) {
                double t = ((s_part[0][r] + s_part[1][r]) + (s_part[2][r] + s_part[3][r])) +
                           ((s_part[4][r] + s_part[5][r]) + (s_part[6][r] + s_part[7][r]));
                t *= c_inv[i];
                acc += t;
                s_x[r] = t;
            }
            __syncthreads();
        }
        x = acc;
    }
    if (w == 0) y[r] = r < k ? x : 0.0;
    __syncthreads();
    return true;
}

// The interpolation rows of a ghost applied to x, NG ghosts by each group of
// eight lanes (lane gl of it) at once, so that their loads overlap; rl: the
// rows' lengths (0: none); rows from the cache in shared memory (rw, ri) or
// from global memory (ri null).  The sums are returned to every lane of the
// group.  Mixed mode: x is FP32, and so, exactly, are most weights (binary
// fractions of at most 24 digits): the products are then exact FP32 pairs
// and their sums carry ~46 digits, in place of eleven FP64 instructions per
// four ghosts (65 cycles each); rows with longer weights take the FP64 path.
template <typename T, int NG>
__device__ __noinline__ void ghost_rows(const KrylovStepArgs& A, const T* x, const long long (&t)[NG], const int (&rl)[NG],
                                        int gl, const double* const (&rw)[NG], const int* const (&ri)[NG],
                                        double (&out)[NG]) {
    int most = 0;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
        out[q] = 0.0;
        most = max(most, rl[q]);
    }
    most = (int)__reduce_max_sync(0xffffffffu, (unsigned)most);
    float fs[NG], fc[NG];
#pragma unroll
    for (int q = 0; q < NG; ++q) fs[q] = fc[q] = 0.f;
    for (int e0 = 0; e0 < most; e0 += 64) {
        const int nu = min(8, (most - e0 + 7) / 8);
        for (int u0 = 0; u0 < nu; u0 += 4) {
            int id[NG][4];
            double wt[NG][4];
            T xv[NG][4];
#pragma unroll
            for (int q = 0; q < NG; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = e0 + gl + 8 * (u0 + u);
                    const bool hit = ri[q] != nullptr && rl[q] <= 64;
                    const size_t base = (size_t)t[q] * A.rmax;
                    id[q][u] = e < rl[q] ? (hit ? ri[q][e] : A.row_idx[base + e]) : -1;
                    wt[q][u] = e < rl[q] ? (hit ? rw[q][e] : A.row_w[base + e]) : 0.0;
                }
#pragma unroll
            for (int q = 0; q < NG; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u) xv[q][u] = id[q][u] >= 0 ? x[id[q][u]] : T(0);
            bool fp32 = false;
            if constexpr (sizeof(T) == 4) {
                int rest = 0;
#pragma unroll
                for (int q = 0; q < NG; ++q)
#pragma unroll
                    for (int u = 0; u < 4; ++u) rest |= __double2loint(wt[q][u]) & 0x1fffffff;
                fp32 = !__any_sync(0xffffffffu, rest != 0);
                if (fp32) {
#pragma unroll
                    for (int q = 0; q < NG; ++q)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float w = d2f_trunc(wt[q][u]), z = (float)xv[q][u];
                            const float p = __fmul_rn(w, z), pe = __fmaf_rn(w, z, -p);
                            const float a = __fadd_rn(fs[q], p), b = __fsub_rn(a, fs[q]);
                            const float er = __fadd_rn(__fsub_rn(fs[q], __fsub_rn(a, b)), __fsub_rn(p, b));
                            fs[q] = a;
                            fc[q] = __fadd_rn(fc[q], __fadd_rn(er, pe));
                        }
                }
            }
            if (!fp32) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (u0 + u < nu)
#pragma unroll
                        for (int q = 0; q < NG; ++q) out[q] += wt[q][u] * dbl(xv[q][u]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NG; ++q) {
        if constexpr (sizeof(T) == 4) {
            const bool some = __any_sync(0xffffffffu, __double_as_longlong(out[q]) != 0);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const float s2 = __shfl_xor_sync(0xffffffffu, fs[q], o), c2 = __shfl_xor_sync(0xffffffffu, fc[q], o);
                const float a = __fadd_rn(fs[q], s2), b = __fsub_rn(a, fs[q]);
                const float er = __fadd_rn(__fsub_rn(fs[q], __fsub_rn(a, b)), __fsub_rn(s2, b));
                fs[q] = a;
                fc[q] = __fadd_rn(__fadd_rn(fc[q], c2), er);
            }
            if (!some) {
                out[q] = f2d_exact(fs[q]) + f2d_exact(fc[q]);
                continue;
            }
        }
        out[q] += __shfl_xor_sync(0xffffffffu, out[q], 1);
        out[q] += __shfl_xor_sync(0xffffffffu, out[q], 2);
        out[q] += __shfl_xor_sync(0xffffffffu, out[q], 4);
        if constexpr (sizeof(T) == 4) out[q] += f2d_exact(fs[q]) + f2d_exact(fc[q]);
    }
}
template <typename T>
__device__ __forceinline__ double ghost_row(const KrylovStepArgs& A, const T* x, long long t, int rl, int gl,
                                            const double* rw, const int* ri) {
    const long long tt[1] = {t};
    const int rr[1] = {rl};
    const double* const ww[1] = {rw};
    const int* const ii[1] = {ri};
    double out[1];
    ghost_rows<T, 1>(A, x, tt, rr, gl, ww, ii, out);
    return out[0];
}

// A_n q at a point.  Order 2P = 4: with the point's constants prepared (U and
// V over 12 h, nu over 12 h^2 at the point's stencil levels, and the lattice
// offsets of its eight neighbours), the differences feed fused multiply-adds:
// 18 FP64 instructions against 25, and the loads go out at once.  Other
// orders: apply_point.
template <typename T>
struct OpPoint {
    uint32_t mw;
    T ux, vy, nx, ny;
    int o[9];
};
template <typename T, int P>
__device__ __forceinline__ void op_prepare(OpPoint<T>& c, uint32_t mw, T U, T V, T nu, const Geom& g, T c1J, T c2J) {
    c.mw = mw;
    if constexpr (P != 2) {
        c.ux = U;
        c.vy = V;
        c.nx = nu;
    } else {
        const int p = meta_pos(mw);
        const int i = p & g.mask, k = p >> g.L;
        const int shx = g.J - meta_jx(mw), shy = g.J - meta_jy(mw);
        const int sx = 1 << shx, sy = 1 << shy;
        c.ux = -U * pow2_down(c1J, shx);
        c.vy = -V * pow2_down(c1J, shy);
        c.nx = nu * pow2_down(c2J, 2 * shx);
        c.ny = nu * pow2_down(c2J, 2 * shy);
        const int row = k << g.L;
        c.o[0] = row + i;
        c.o[1] = row + ((i + sx) & g.mask);
        c.o[2] = row + ((i - sx) & g.mask);
        c.o[3] = row + ((i + 2 * sx) & g.mask);
        c.o[4] = row + ((i - 2 * sx) & g.mask);
        c.o[5] = (((k + sy) & g.mask) << g.L) + i;
        c.o[6] = (((k - sy) & g.mask) << g.L) + i;
        c.o[7] = (((k + 2 * sy) & g.mask) << g.L) + i;
        c.o[8] = (((k - 2 * sy) & g.mask) << g.L) + i;
    }
}
template <typename T, int P>
__device__ __forceinline__ T op_apply(const T* F, const OpPoint<T>& c, T r, const Geom& g, T c1J, T c2J) {
    if constexpr (P != 2) {
        return apply_point<T, false, P>(F, c.mw, c.ux, c.vy, c.nx, r, g, c1J, c2J);
    } else {
        T v[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) v[q] = F[c.o[q]];
        const T gx = fma(T(8), v[1] - v[2], v[4] - v[3]), gy = fma(T(8), v[5] - v[6], v[8] - v[7]);
        const T lx = fma(T(-30), v[0], fma(T(16), v[1] + v[2], -(v[3] + v[4])));
        const T ly = fma(T(-30), v[0], fma(T(16), v[5] + v[6], -(v[7] + v[8])));
        T z = fma(c.nx, lx, c.ny * ly);
        z = fma(c.ux, gx, z);
        z = fma(c.vy, gy, z);
        if (r != T(0)) z = fma(-r, v[0], z);
        return z;
    }
}

// Absolute sum of the operator's row, without the friction r, at a point:
// |(A + r) q| <= it times max |q|.
template <typename T, int P>
__device__ __forceinline__ double row_bound(const KrylovStepArgs& A, uint32_t mw, T U, T V) {
    double d1 = 0.0, d2 = -dd_d2(P, 0);
#pragma unroll
    for (int o = 1; o <= dd_reach1(P); ++o) d1 += 2.0 * (dd_d1(P, o) < 0 ? -dd_d1(P, o) : dd_d1(P, o));
#pragma unroll
    for (int o = 1; o <= P; ++o) d2 += 2.0 * (dd_d2(P, o) < 0 ? -dd_d2(P, o) : dd_d2(P, o));
    const int shx = A.g.J - meta_jx(mw), shy = A.g.J - meta_jy(mw);
    return d1 * (fabs(dbl(U)) * pow2_down(A.c1J, shx) + fabs(dbl(V)) * pow2_down(A.c1J, shy)) +
           d2 * A.nu * (pow2_down(A.c2J, 2 * shx) + pow2_down(A.c2J, 2 * shy));
}
// Extra scale bits of a ghost's basis values: its interpolation row's
// absolute sum beyond 1.9, as powers of two (basis values hold up to 2).
__device__ __forceinline__ int ghost_scale(const KrylovStepArgs& A, long long t, int rl, int gl) {
    float ab = 0.f;
    for (int e = gl; e < rl; e += 8) ab += fabsf((float)A.row_w[(size_t)t * A.rmax + e]);
    ab += __shfl_xor_sync(0xffffffffu, ab, 1);
    ab += __shfl_xor_sync(0xffffffffu, ab, 2);
    ab += __shfl_xor_sync(0xffffffffu, ab, 4);
    int gs = 0;
    while (gs < 20 && ab > 1.9f) {
        ab *= 0.5f;
        ++gs;
    }
    return gs;
}

// Digit tile of s and t for the updates (32 rows of kTP bytes): t's digits at
// rows 7-14 (zero rows 0-6 above, 15-16 below), s's at rows 24-31 (zero rows
// 17-23 above; the six most significant ones are used).
constexpr int kTileT = 7, kTileS = 24;

// Sums over the rows of the basis, for NU * 8 columns from c0 (a multiple of
// 8): per lane (one column each) the sums with t (x) and with s (y), in
// units 2^(Et - 60) and 2^(Es - 60) for a column of scale 2^-61.  Columns
// c = 0..9 of the digit products with t, 0..5 with s.  Even and odd digits
// have accumulators of their own: shorter chains of dependent products.
template <int NU, bool HALF>
__device__ __noinline__ longlong2 update_sums(const char* Qb, int pitch, int dstride, int nrow, int c0,
                                              const char* tile, float* scr) {
    const int lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
    // ldmatrix row of this lane: matrices (M rows 0-7, k 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15)
    const int mr = (lane & 7) + ((lane >> 3) & 1) * 8;
    const int trow = mr < 10 ? kTileT + mr : kTileS + (mr - 10);
    const unsigned ta = smem_addr(tile) + trow * kTP + (lane >> 4) * 16;
    float c[NU][2][4];
#pragma unroll
    for (int n = 0; n < NU; ++n)
#pragma unroll
        for (int e = 0; e < 8; ++e) c[n][e >> 2][e & 3] = 0.f;
    const int top = nrow - 1;   // rows from nrow on have zero digits in the tile
    for (int ks = 0; ks * 16 < nrow; ++ks) {
        if constexpr (HALF) {
            // matrices (digit 2w, rows 0-7), (2w, 8-15), (2w + 1, 0-7), (2w + 1, 8-15)
            const unsigned qa = smem_addr(Qb) + min(16 * ks + mr, top) * (2 * pitch) + c0 * 2 + (lane >> 4) * dstride;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                unsigned a0[4], a1[4], b[NU][4];
                ldsm4(a0, ta + ks * 32 - (2 * w) * kTP);
                ldsm4(a1, ta + ks * 32 - (2 * w + 1) * kTP);
#pragma unroll
                for (int n = 0; n < NU; ++n) ldsm4t(b[n], qa + 2 * w * dstride + n * 16);
#pragma unroll
                for (int n = 0; n < NU; ++n) hmma(c[n][0], a0, b[n][0], b[n][1]);
#pragma unroll
                for (int n = 0; n < NU; ++n) hmma(c[n][1], a1, b[n][2], b[n][3]);
            }
        } else {
            const int r0 = 16 * ks + tg;
            const unsigned long long* Q = reinterpret_cast<const unsigned long long*>(Qb);
            const unsigned long long* qa = Q + (size_t)min(r0, top) * pitch + c0 + g;
            const unsigned long long* qb = Q + (size_t)min(r0 + 4, top) * pitch + c0 + g;
            const unsigned long long* qc = Q + (size_t)min(r0 + 8, top) * pitch + c0 + g;
            const unsigned long long* qd = Q + (size_t)min(r0 + 12, top) * pitch + c0 + g;
            unsigned long long xa[NU], xb[NU], xc[NU], xd[NU];
#pragma unroll
            for (int n = 0; n < NU; ++n) {
                xa[n] = qa[8 * n];
                xb[n] = qb[8 * n];
                xc[n] = qc[8 * n];
                xd[n] = qd[8 * n];
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) {   // digit pairs, most significant first
                unsigned a0[4], a1[4];
                ldsm4(a0, ta + ks * 32 - (2 * w) * kTP);
                ldsm4(a1, ta + ks * 32 - (2 * w + 1) * kTP);
                unsigned b[NU][4];
#pragma unroll
                for (int n = 0; n < NU; ++n) {
                    digits2(w < 2 ? (unsigned)(xa[n] >> 32) : (unsigned)xa[n],
                            w < 2 ? (unsigned)(xb[n] >> 32) : (unsigned)xb[n], w & 1, b[n][0], b[n][1]);
                    digits2(w < 2 ? (unsigned)(xc[n] >> 32) : (unsigned)xc[n],
                            w < 2 ? (unsigned)(xd[n] >> 32) : (unsigned)xd[n], w & 1, b[n][2], b[n][3]);
                }
#pragma unroll
                for (int n = 0; n < NU; ++n) hmma(c[n][0], a0, b[n][0], b[n][2]);
#pragma unroll
                for (int n = 0; n < NU; ++n) hmma(c[n][1], a1, b[n][1], b[n][3]);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < NU; ++n) {
        float* p = scr + (8 * n + 2 * tg) * 20 + g;
        p[0] = c[n][0][0] + c[n][1][0];
        p[20] = c[n][0][1] + c[n][1][1];
        p[8] = c[n][0][2] + c[n][1][2];
        p[28] = c[n][0][3] + c[n][1][3];
    }
    __syncwarp();
    int S[16];
    const float4* f = reinterpret_cast<const float4*>(scr + (lane & (8 * NU - 1)) * 20);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = f[q];
        S[4 * q] = __float2int_rn(v.x);
        S[4 * q + 1] = __float2int_rn(v.y);
        S[4 * q + 2] = __float2int_rn(v.z);
        S[4 * q + 3] = __float2int_rn(v.w);
    }
    __syncwarp();
    const auto join = [](int a, int b, int c2, int d) {
        return ((long long)a << 24) + ((long long)b << 16) + ((long long)c2 << 8) + (long long)d;
    };
    longlong2 v;
    v.x = (join(S[0], S[1], S[2], S[3]) << 25) +
          ((join(S[4], S[5], S[6], S[7]) + ((((long long)S[8] << 8) + S[9]) >> 16)) >> 7);
    v.y = (join(S[10], S[11], S[12], S[13]) << 25) + (join(S[14], S[15], 0, 0) >> 7);
    return v;
}

// Digit products of a unit of 16 points (u and z digits in the tile at ta)
// with the first 8 NT rows of the table (rows beyond `top` repeat it).
template <int NT, bool HALF>
__device__ __forceinline__ void dot_unit(float (&c)[NT][2][4], const char* Qb, int pitch, int dstride, int top, int p0,
                                         unsigned ta) {
    const int lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
    if constexpr (HALF) {
        // matrices (digit 2w, points 0-7), (2w, 8-15), (2w + 1, 0-7), (2w + 1, 8-15)
        unsigned qa[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t)
            qa[t] = smem_addr(Qb) + min(8 * t + (lane & 7), top) * (2 * pitch) + (p0 + ((lane >> 3) & 1) * 8) * 2 +
                    (lane >> 4) * dstride;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            unsigned a0[4], a1[4], b[NT][4];
            ldsm4(a0, ta - (2 * w) * kUP);
            ldsm4(a1, ta - (2 * w + 1) * kUP);
#pragma unroll
            for (int t = 0; t < NT; ++t) ldsm4(b[t], qa[t] + 2 * w * dstride);
#pragma unroll
            for (int t = 0; t < NT; ++t) hmma(c[t][0], a0, b[t][0], b[t][1]);
#pragma unroll
            for (int t = 0; t < NT; ++t) hmma(c[t][1], a1, b[t][2], b[t][3]);
        }
    } else {
        const unsigned long long* Q = reinterpret_cast<const unsigned long long*>(Qb);
        const int pr = (g & 3) * 2 + (g >> 2);        // basis row of mma column g: 0 2 4 6 1 3 5 7
        ulonglong2 x0[NT], x1[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const ulonglong2* q =
                reinterpret_cast<const ulonglong2*>(Q + (size_t)min(8 * t + pr, top) * pitch + p0 + 2 * tg);
            x0[t] = q[0];
            x1[t] = q[4];
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            unsigned a0[4], a1[4];
            ldsm4(a0, ta - (2 * w) * kUP);
            ldsm4(a1, ta - (2 * w + 1) * kUP);
            unsigned b[NT][4];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                digits2(w < 2 ? (unsigned)(x0[t].x >> 32) : (unsigned)x0[t].x,
                        w < 2 ? (unsigned)(x0[t].y >> 32) : (unsigned)x0[t].y, w & 1, b[t][0], b[t][1]);
                digits2(w < 2 ? (unsigned)(x1[t].x >> 32) : (unsigned)x1[t].x,
                        w < 2 ? (unsigned)(x1[t].y >> 32) : (unsigned)x1[t].y, w & 1, b[t][2], b[t][3]);
            }
#pragma unroll
            for (int t = 0; t < NT; ++t) hmma(c[t][0], a0, b[t][0], b[t][2]);
#pragma unroll
            for (int t = 0; t < NT; ++t) hmma(c[t][1], a1, b[t][1], b[t][3]);
        }
    }
}

// Position of basis row r in the k order of the update products of the words
// form (thread tg of an mma holds k = 2 tg, 2 tg + 1, 2 tg + 8, 2 tg + 9:
// rows tg, tg + 4, tg + 8, tg + 12, whose words a warp then reads without
// bank conflicts); in order for the halves.
template <bool HALF>
__device__ __forceinline__ int tile_col(int r) {
    if (HALF) return r;
    const int q = r & 15;
    return (r & 16) + 2 * (q & 3) + ((q >> 2) & 1) + (q & 8);
}

// A basis value (or u) into row `row`, column c of the table.
template <bool HALF>
__device__ __forceinline__ void put_value(char* Qb, int pitch, int dstride, int row, int c, unsigned long long x) {
    if constexpr (HALF) put_digits(Qb + ((size_t)row * pitch + c) * 2, dstride, x);
    else reinterpret_cast<unsigned long long*>(Qb)[(size_t)row * pitch + c] = x;
}

// ---- q_j and the next u at one column ------------------------------------------
// q_j = (u - ps) / h, next u = (z - pc - q_j qz) / h with ps = sum s_t q_t and
// pc = sum t_t q_t as exact integers (vs 2^es, vt 2^et).  FP64: one rounding
// per operation.  Mixed mode: ps and pc are rounded to FP32 (2^-24 of
// them, as coefficients and sums of this mode are), u - ps and the results
// are FP32, and z - pc - q_j qz is formed in FP32 pairs (exact products by fma,
// exact sums), so that its cancellation adds nothing of its own: FP64
// instructions would cost 65 cycles each here.
struct StepScalars {
    double hinv, qz;
    float hh, hl, qh, ql;   // the same two as FP32 pairs
};
__device__ __forceinline__ void next_values(double u, double z, long long vs, int es, long long vt, int et,
                                            const StepScalars& S, double& qj, double& un) {
    qj = fma(-(double)vs, pow2d(es), u) * S.hinv;
    un = fma(-qj, S.qz, fma(-(double)vt, pow2d(et), z)) * S.hinv;
}
__device__ __forceinline__ float scaled_float(long long v, int e) {
    const float f = __ll2float_rn(v);
    const int e1 = max(-126, min(e / 2, 127)), e2 = max(-126, min(e - e / 2, 127));
    return f * __int_as_float((e1 + 127) << 23) * __int_as_float((e2 + 127) << 23);
}
__device__ __forceinline__ void next_values_f(float u, float z, float ps, float pc, const StepScalars& S, float& qj,
                                              float& un) {
    const float a = __fsub_rn(u, ps);
    const float p0 = __fmul_rn(a, S.hh);
    qj = __fadd_rn(p0, __fmaf_rn(a, S.hl, __fmaf_rn(a, S.hh, -p0)));
    // s + e = z - pc exactly
    const float s = __fsub_rn(z, pc), bb = __fsub_rn(s, z);
    const float e = __fadd_rn(__fsub_rn(z, __fsub_rn(s, bb)), __fsub_rn(-pc, bb));
    // p + pe = qj qh exactly; d + de = s - p exactly
    const float p = __fmul_rn(qj, S.qh), pe = __fmaf_rn(qj, S.qh, -p);
    const float d = __fsub_rn(s, p), db = __fsub_rn(d, s);
    const float de = __fadd_rn(__fsub_rn(s, __fsub_rn(d, db)), __fsub_rn(-p, db));
    const float low = __fsub_rn(__fadd_rn(e, de), __fmaf_rn(qj, S.ql, pe));
    const float m = __fmul_rn(d, S.hh);
    un = __fadd_rn(m, __fmaf_rn(low, S.hh, __fmaf_rn(d, S.hl, __fmaf_rn(d, S.hh, -m))));
}
// FP32 pair of a double.
__device__ __forceinline__ void split2(double x, float& h, float& l) {
    h = (float)x;
    l = (float)(x - (double)h);
}

// The Krylov step of one problem by its nb blocks (bid = this block's index);
// ppb points and gpb ghosts per block (multiples of 16).  formed: the launch
// formed clusters of CL blocks, whose sums are added in distributed shared
// memory first.  Returns the number of steps whose dots were taken, for
// the cluster barriers at the end.
// EX: the velocity-Exner step.  The points are the 3 X->n entries of the
// stacked vector (A.n of them, field after field), the ghosts likewise, each
// field on its own lattice; b = F(U^n) is in A.w on entry.
template <typename T, int CL, int P, int FORM, bool EX = false>
__device__ __forceinline__ int krylov_mma_body(const KrylovStepArgs& A, const int bid, const int nb, const int ppb,
                                               const int gpb, const int nrc, const bool formed, char* sm,
                                               const ExArgs* X = nullptr) {
    constexpr bool wide = FORM != kNarrow, HALF = FORM != kWords;
    constexpr int NU = wide ? 4 : 2, cstep = 8 * NU;   // columns a product warp takes in a turn
    __shared__ double s_v[2][32];        // s (and |u|^2), t (and u.z) of a step
    __shared__ double s_part[kPW][33];
    __shared__ double s_y[32], s_x[32];
    __shared__ double s_sc[4];           // h^2, 1/h, qz, beta
    __shared__ StepScalars s_S;          // what the new vectors need of them
    __shared__ float s_fs[32];           // s 2^-(its exponent)
    __shared__ int s_e[8];               // exponents: 0 u (points), 1 u (with ghosts), 2 z, 3 global u, 4 s, 5 t, 6 |A|, 7 last column of H
    __shared__ int s_int[4], s_ok;
    __shared__ longlong2 s_bp[64];       // the block's dot sums (high and low parts)
    const MmaLayout Y = mma_layout(FORM, A.m, ppb, gpb, nrc);
    char* Q = sm + Y.q;
    double* us = reinterpret_cast<double*>(sm + Y.us);
    double* zs = reinterpret_cast<double*>(sm + Y.zs);
    double* rz = reinterpret_cast<double*>(sm + Y.rz);
    uint32_t* meta = reinterpret_cast<uint32_t*>(sm + Y.meta);
    int* gpos = reinterpret_cast<int*>(sm + Y.gpos);   // lattice index | extra scale bits << 24
    int* glen = reinterpret_cast<int*>(sm + Y.glen);   // row lengths
    double* sH = reinterpret_cast<double*>(sm + Y.sH);
    float* sHf = reinterpret_cast<float*>(sm + Y.sHf);
    double* rw = reinterpret_cast<double*>(sm + Y.rw);
    int* ri = reinterpret_cast<int*>(sm + Y.ri);
    longlong2* vv = reinterpret_cast<longlong2*>(sm + Y.vv);
    char* tile = sm + Y.tile;
    const int pitch = Y.pitch;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    char* scr = sm + Y.scr + (size_t)(wid < kPW ? wid : 0) * kScr;
    const int m = A.m;
    const int dstride = (m + 1) * pitch * 2;           // bytes between the digits of the halves forms
    const long long p0 = (long long)bid * ppb;
    const int gev = (int)(((long long)A.ng + nb - 1) / nb);                   // ghosts dealt out evenly
    const long long t0 = (long long)bid * gev;
    const int n = (int)max(0ll, min((long long)ppb, (long long)A.n - p0));     // points of this block
    const int ng = (int)max(0ll, min((long long)gev, (long long)A.ng - t0));   // ghosts of this block (<= gpb)
    const bool lead = bid == 0 && threadIdx.x == 0;
    const T* Ua = (const T*)A.Ua + p0;
    const T* Va = (const T*)A.Va + p0;
    T* Lq = (T*)A.Lq;
    T* zb = (T*)A.w;                   // z at every active point (read by the ghosts' rows)
    const T nu = (T)A.nu, r = (T)A.r, c1J = (T)A.c1J, c2J = (T)A.c2J;
    // The steps apply A + r I: the same vectors, H + r I.  The ghost values of u
    // follow from those of z by the points' recurrence, which carries a
    // rounding d_0 of theirs on as d_{j+1} = -sum_q H_qj d_q / h_{j+1}: with H
    // near -r I it grew by r / h a step (r = 50: 10 to 100), until the ghost
    // values left the range of their fixed point.
    const bool shift = !EX && A.r != 0.0;
    // field and point of stacked entry e, field and ghost of stacked ghost t; a field's lattice
    const int xn = EX ? X->n : 0, xg = EX ? X->ng : 0;
    const auto field = [&](long long e) { return EX ? (e >= 2LL * xn ? 2 : (e >= xn ? 1 : 0)) : 0; };
    const auto gfield = [&](long long t) { return EX ? (t >= 2LL * xg ? 2 : (t >= xg ? 1 : 0)) : 0; };
    const auto row_of = [&](long long t) { return EX ? t - (long long)gfield(t) * xg : t; };
    const auto z_of = [&](long long t) { return EX ? zb + (size_t)gfield(t) * xn : zb; };
    const auto lattice = [&](int f) {
        if constexpr (EX) return (T*)(f == 2 ? X->Lq[2] : (f == 1 ? X->Lq[1] : X->Lq[0]));
        else return Lq;
    };
    // global scratch: sums [2][kCopies][64][2] (block b adds to copy b mod kCopies: with one
    // copy the additions of 152 blocks to the same words took up to 2 us), then per step
    // parity the exponents of u and of z not finite, and |A|'s
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(A.part);
    unsigned* slot = reinterpret_cast<unsigned*>(acc + 2 * kCopies * 128);   // [2][2], then |A|
    int ph = 0, calls = 0;
    if (lead && A.trace) A.trace[0] = gtimer();
    if (*(volatile const int*)A.row_overflow) {
        if (lead) atomicOr(A.err, 4);
        return calls;
    }
    if (*(volatile int*)A.err & kErrStop) return calls;   // an earlier wait ran out
    unsigned phase = *(volatile unsigned*)A.bar & 0x80000000u;
    const auto meet = [&]() {
        const bool ok = grid_wait(A.bar, A.err, A.limit_ns, bid, nb, phase, &s_ok, A.trace, ph);
        ++ph;
        phase ^= 0x80000000u;
        return ok;
    };
    if (bid == 0) {
        for (int t = threadIdx.x; t < 2 * kCopies * 128; t += kMT) acc[t] = 0ull;
        if (threadIdx.x < 8) slot[threadIdx.x] = 0u;
        for (int t = threadIdx.x; t < (m + 1) * m; t += kMT) A.H[t] = 0.0;
    }
    for (int c = threadIdx.x; c < Y.cols; c += kMT) {
        us[c] = 0.0;
        zs[c] = 0.0;
    }
    for (int c = threadIdx.x; c < gpb; c += kMT) rz[c] = 0.0;
    for (int c = threadIdx.x; c < 32 * 33; c += kMT) {
        sH[c] = 0.0;
        if (nrc >= 0) sHf[c] = 0.f;
    }
    for (int c = threadIdx.x; c < kTP * 32 / 4; c += kMT) reinterpret_cast<unsigned*>(tile)[c] = 0u;
    if (HALF)
        for (int c = threadIdx.x; c < (m + 1) * pitch * 4; c += kMT) reinterpret_cast<unsigned*>(Q)[c] = 0u;
    else
        for (int c = threadIdx.x; c < (m + 1) * pitch; c += kMT) reinterpret_cast<unsigned long long*>(Q)[c] = kBias;
    for (int c = threadIdx.x; c < n; c += kMT) meta[c] = A.meta[p0 + c - (EX ? (long long)field(p0 + c) * xn : 0)];
    for (int e = threadIdx.x; e < min(nrc, ng) * kRowCache; e += kMT) {
        const int q = e / kRowCache, i = e - q * kRowCache;
        const long long t = row_of(t0 + q);
        const int rl = A.row_len[t];
        if (i < rl && rl <= kRowCache) {
            ri[e] = A.row_idx[(size_t)t * A.rmax + i];
            rw[e] = A.row_w[(size_t)t * A.rmax + i];
        }
    }
    if (threadIdx.x < 8) s_e[threadIdx.x] = 0;
    __syncthreads();

    // b = A_n omega + g (L holds R(omega), ghosts included), and the bound
    // |A|_inf <= max over the points of its row's absolute sum (as an exponent;
    // the ghost values it multiplies are bounded by their own maximum)
    for (int c = wid * 32; c < n; c += 32 * kMW) {
        const int p = c + lane;
        int ea = 0;
        if (p < n) {
            const uint32_t mw = meta[p];
            if constexpr (EX) {
                const int f = field(p0 + p);
                const T v = zb[p0 + p];
                us[p] = dbl(v);
                lattice(f)[meta_pos(mw)] = v;
                ea = expo(ex_row_bound<P>(*X, mw, f, (int)(p0 + p - (long long)f * xn)));
            } else {
            const T U = Ua[p], V = Va[p];
            T v = apply_point<T, false, P>((const T*)A.L, mw, U, V, nu, r, A.g, c1J, c2J);
            if (A.ga) v += ((const T*)A.ga)[p0 + p];
            us[p] = dbl(v);
            zb[p0 + p] = v;
            Lq[meta_pos(mw)] = v;
            ea = expo(row_bound<T, P>(A, mw, U, V));
            }
        }
        ea = (int)__reduce_max_sync(0xffffffffu, (unsigned)ea);
        if (lane == 0) atomicMax(&s_e[6], ea);
    }
    if (!meet()) return calls;
    // ghost values of b through the interpolation rows; a ghost whose row's
    // absolute sum exceeds 1.9 gets a coarser scale for its basis values
    for (int q = wid * 4; q < ng; q += 4 * kMW) {
        const int gi = q + (lane >> 3), gl = lane & 7;
        const bool valid = gi < ng;
        const long long t = row_of(t0 + gi);
        const int rl = valid ? A.row_len[t] : 0;
        const double v = ghost_row<T>(A, z_of(t0 + gi), t, rl, gl, nullptr, nullptr);
        const int gs = ghost_scale(A, t, rl, gl);
        if (valid && gl == 0) {
            const T gv = (T)v;
            const int pos = A.glist[t], f = gfield(t0 + gi);
            gpos[gi] = pos | (gs << 24) | (f << 29);
            glen[gi] = rl;
            us[ppb + gi] = dbl(gv);
            lattice(f)[pos] = gv;
        }
    }
    __syncthreads();
    for (int c = wid * 32; c < Y.cols; c += 32 * kMW) {
        const int e = c + lane < Y.cols ? expo(us[c + lane]) : 0;
        const int ea = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
        const int ep = (int)__reduce_max_sync(0xffffffffu, (unsigned)(c + lane < ppb ? e : 0));
        if (lane == 0) {
            atomicMax(&s_e[0], ep);
            atomicMax(&s_e[1], ea);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&slot[0], (unsigned)s_e[1]);
        atomicMax(&slot[4], (unsigned)s_e[6]);
    }
    if (!meet()) return calls;
    const int be = first_scale<T>((int)__ldcg(&slot[0]));   // the same for every block
    if (be != 0) {   // u = b 2^-be
        for (int c = threadIdx.x; c < Y.cols; c += kMT) {
            const bool gh = c >= ppb;
            if (gh ? c - ppb >= ng : c >= n) continue;
            const int gp = gh ? gpos[c - ppb] : 0;
            const T v = (T)scale2(us[c], -be);
            us[c] = dbl(v);
            lattice(gh ? (gp >> 29) & 3 : field(p0 + c))[gh ? gp & 0xffffff : meta_pos(meta[c])] = v;
        }
        if (threadIdx.x < 2 && s_e[threadIdx.x]) s_e[threadIdx.x] = max(0, s_e[threadIdx.x] - be);
        if (!meet()) return calls;
    }

    const int nunit = (n + 15) / 16;
    const int nact = min(kPW, nunit);                    // product warps with points
    // the operator's constants of this warp's first 32 points stay in registers
    const int opw = wid < 8 ? wid : wid - 1;             // warp 8 takes no points
    OpPoint<T> op0;
    op_prepare<T, P>(op0, 0, T(0), T(0), T(0), A.g, c1J, c2J);
    if (!EX && wid != 8 && opw * 32 + lane < n)
        op_prepare<T, P>(op0, meta[opw * 32 + lane], Ua[opw * 32 + lane], Va[opw * 32 + lane], nu, A.g, c1J, c2J);
    const int gw = wid >= 9 ? wid - 9 : wid - 2 + 3;     // first ghost pass of this warp
    int k = m;
    const int eA = (int)__ldcg(&slot[4]) - 1022 + 1;     // |A u|_inf < 2^eA |u|_inf, with slack for rounding
    for (int j = 0;; ++j) {
        const bool last = j == m;   // only the second pass of u is left
        unsigned long long* accj = acc + (j & 1) * kCopies * 128;
        if (wid >= 8 && j > 1 && s_int[1] < 3) {
            // g = H s of step j - 1 in FP64 (warp 8 uses it below): the columns dealt over four warps
            double gi = 0.0;
            for (int c = wid - 8; c < j - 1; c += 4)
                gi += (c == j - 2 && lane < j - 1 ? sH[lane * 33 + c] + s_v[0][lane] : sH[lane * 33 + c]) * s_v[0][c];
            s_part[wid - 8][lane] = gi;
            asm volatile("bar.sync 3, 128;" ::: "memory");
        }
        // ---- z = A u at the own points ------------------------------------
        if (wid == 8) {
            if (lane == 0) s_e[3] = (int)__ldcg(&slot[(j & 1) * 2]) - (j == 0 ? be : 0);
            // the other parity's sums and exponents (last read before the barrier just passed)
            for (int q = bid; q < kCopies; q += nb) {
                unsigned long long* z = acc + (((j + 1) & 1) * kCopies + q) * 128;
                for (int t = lane; t < 128; t += 32) z[t] = 0ull;
            }
            if (bid == 0 && lane < 2) slot[((j + 1) & 1) * 2 + lane] = 0u;
            // what is off the path of step j - 1: h, column j - 2 of H after its second pass,
            // and column j - 1, first pass: h1 = ([t; qz] - g) / h with g = H s
            if (j > 0) {
                const int q = j - 1;
                const double si = lane < q ? s_v[0][lane] : 0.0;
                const double hinv = s_sc[1], h = s_sc[0] * hinv, qz = s_sc[2];
                if (q > 0) {
                    if (lane < q) sH[lane * 33 + q - 1] += si;
                    if (lane == 0) sH[q * 33 + q - 1] = h;
                }
                __syncwarp();
                double gi = 0.0;
                if (s_int[1] == 3) {
                    float g0 = 0.f, g1 = 0.f;
                    if (nrc >= 0) {
                        const float* hr = sHf + lane * 33;
#pragma unroll 4
                        for (int c = 0; c + 1 < q; c += 2) {
                            g0 = fmaf(hr[c], s_fs[c], g0);
                            g1 = fmaf(hr[c + 1], s_fs[c + 1], g1);
                        }
                        if (q & 1) g0 = fmaf(hr[q - 1], s_fs[q - 1], g0);
                    } else {
                        for (int c = 0; c < q; ++c) g0 = fmaf(d2f_trunc(sH[lane * 33 + c]), s_fs[c], g0);
                    }
                    gi = scale2(f2d_exact(g0 + g1), s_e[4] - 1022);
                } else {
                    if (q > 0) gi = (s_part[0][lane] + s_part[1][lane]) + (s_part[2][lane] + s_part[3][lane]);
                }
                double v = 0.0;
                if (lane < q) v = (s_v[1][lane] - gi) * hinv;
                else if (lane == q) v = (qz - (q > 0 ? h * s_v[0][q - 1] : 0.0)) * hinv;
                if (lane <= q) {
                    sH[lane * 33 + q] = v;
                    if (nrc >= 0) sHf[lane * 33 + q] = d2f_trunc(v);
                }
                const int ev = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(expo(v), shift ? expo(A.r) : 0));
                if (lane == 0) s_e[7] = ev;
            }
        } else if (!last) {
            for (int c = opw * 32; c < n; c += 32 * (kMW - 1)) {
                const int p = c + lane;
                int e = 0;
                if (p < n) {
                    T z;
                    if constexpr (EX) {
                        const int f = field(p0 + p);
                        z = (T)ex_entry<P>(*X, meta[p], f, (int)(p0 + p - (long long)f * xn));
                    } else if (c == opw * 32) {
                        z = op_apply<T, P>(Lq, op0, T(0), A.g, c1J, c2J);
                    } else {
                        OpPoint<T> op;
                        op_prepare<T, P>(op, meta[p], Ua[p], Va[p], nu, A.g, c1J, c2J);
                        z = op_apply<T, P>(Lq, op, T(0), A.g, c1J, c2J);
                    }
                    zb[p0 + p] = z;
                    const double zd = dbl(z);
                    zs[p] = zd;
                    e = expo(zd);
                }
                e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
                if (lane == 0) atomicMax(&s_e[2], e);
            }
        }
        __syncthreads();
        // ---- dots: [u; z] digits x basis digits (row j of the table: u) ----
        const int eu = s_e[0], ez = s_e[2], egu = s_e[3];
        if (wid < nact) {
            char* tu = scr;                               // rows 0-6 zero, 7-14 u; 15-21 zero, 22-29 z
            for (int t = lane; t < 30 * kUP / 4; t += 32) reinterpret_cast<unsigned*>(tu)[t] = 0u;
            __syncwarp();
            const int g = lane >> 2, tg = lane & 3;
            const int mr = (lane & 7) + ((lane >> 3) & 1) * 15 + 7;
            const unsigned ta = smem_addr(tu) + mr * kUP + (lane >> 4) * 16;
            const auto dots = [&](auto ntc) {
                constexpr int NT = decltype(ntc)::value;
                float c[NT][2][4];
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int e = 0; e < 8; ++e) c[t][e >> 2][e & 3] = 0.f;
                for (int u = wid; u < nunit; u += kPW) {
                    const int p = 16 * u + (lane & 15);
                    const unsigned long long x = lane < 16 ? fix62(us[p], eu) : fix62(zs[p], ez);
                    put_digits(tu + (lane < 16 ? 7 : 22) * kUP + (lane & 15) * 2, kUP, x);
                    if (lane < 16) put_value<HALF>(Q, pitch, dstride, j, p, x);
                    __syncwarp();
                    dot_unit<NT, HALF>(c, Q, pitch, dstride, j, 16 * u, ta);
                    __syncwarp();
                }
                int* o = reinterpret_cast<int*>(scr);
                // mma columns 2 tg, 2 tg + 1 are basis rows
                const int n0 = 2 * tg, n1 = 2 * tg + 1;
                const int r0 = HALF ? n0 : (n0 & 3) * 2 + (n0 >> 2), r1 = HALF ? n1 : (n1 & 3) * 2 + (n1 >> 2);
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    o[(8 * t + r0) * kCP + g] = __float2int_rn(c[t][0][0]) + __float2int_rn(c[t][1][0]);
                    o[(8 * t + r1) * kCP + g] = __float2int_rn(c[t][0][1]) + __float2int_rn(c[t][1][1]);
                    o[(8 * t + r0) * kCP + 8 + g] = __float2int_rn(c[t][0][2]) + __float2int_rn(c[t][1][2]);
                    o[(8 * t + r1) * kCP + 8 + g] = __float2int_rn(c[t][0][3]) + __float2int_rn(c[t][1][3]);
                }
            };
            if (j < 16) dots(std::integral_constant<int, 2>{});
            else dots(std::integral_constant<int, 4>{});
        }
        __syncthreads();
        const int egz = egu + eA;   // biased exponent bounding every |z| (|z| < 2^(egz - 1022))
        const bool pre = CL > 1 && formed;   // sums of the cluster's blocks added before the grid's
        if constexpr (CL > 1) {
            // two cluster barriers a step: the first makes the blocks' sums visible to the
            // cluster's block 0, the second (arrived at once they are read, waited for
            // here or at the end) keeps a block from rewriting them, or leaving, before
            if (pre && j > 0) __cluster_barrier_wait();
        }
        if (wid < 8) {
            // output (row, u or z) by four threads, two digit columns each: the sums
            // over the warps, then one 128-bit integer in units common to all blocks
            const int out = threadIdx.x >> 2, cp = threadIdx.x & 3;
            const int row = out >> 1, v = out & 1;
            long long s = 0;
            const bool on = row <= j && !(last && v);
            if (on) {
                int a = 0, b = 0;
                const char* x0 = sm + Y.scr + (row * kCP + v * 8 + 2 * cp) * 4;
#pragma unroll
                for (int w = 0; w < kPW; ++w) {
                    if (w < nact) {
                        const int2 x = *reinterpret_cast<const int2*>(x0 + w * kScr);
                        a += x.x;
                        b += x.y;
                    }
                }
                s = (cp & 1) ? ((long long)a << 8) + b : ((long long)a << 24) + ((long long)b << 16);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            const long long lo = __shfl_xor_sync(0xffffffffu, s, 2);
            if (cp == 0 && on) {
                int sh = (v ? egz - ez : egu - eu) + (row == j ? egu - eu : 0);
                sh = max(0, min(sh, 126));
                const __int128 W = ((((__int128)s << 32) + lo) << 16) >> sh;
                const unsigned long long wl = (unsigned long long)W & 0xffffffffffffull;
                const long long wh = (long long)(W >> 48);
                s_bp[out] = make_longlong2(wh, (long long)wl);
            }
        }
        unsigned long long* mine = accj + (bid & (kCopies - 1)) * 128;
        if constexpr (CL > 1) {
            if (pre) {
                cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
                __cluster_barrier_arrive();
                __cluster_barrier_wait();
                if (cl.block_rank() == 0 && threadIdx.x < 64) {
                    const int out = threadIdx.x, row = out >> 1, v = out & 1;
                    if (row <= j && !(last && v)) {
                        longlong2 w = s_bp[out];
#pragma unroll
                        for (int q = 1; q < CL; ++q) {
                            const longlong2 x = cl.map_shared_rank(s_bp, q)[out];
                            w.x += x.x;
                            w.y += x.y;
                        }
                        atomicAdd(&mine[2 * out], (unsigned long long)w.x);
                        atomicAdd(&mine[2 * out + 1], (unsigned long long)w.y);
                    }
                }
                __cluster_barrier_arrive();
            }
        }
        if (!pre) {
            __syncthreads();
            const int out = threadIdx.x >> 1;
            if (threadIdx.x < 4 * (j + 1) && nact > 0 && !(last && (out & 1)))
                atomicAdd(&mine[threadIdx.x], reinterpret_cast<unsigned long long*>(s_bp)[threadIdx.x]);
        }
        calls = j + 1;
        if (threadIdx.x == 0 && (eu == 0x7ff || ez == 0x7ff)) atomicMax(&slot[(j & 1) * 2 + 1], 1u);
        if (!meet()) return calls;

        // ---- the sums; z at the ghosts ------------------------------------------
        if (wid < 2) {
            const int v = wid;
            const bool on = lane <= j && !(last && v);
            double val = 0.0;
            if (on) {
                longlong2 x[kCopies];
#pragma unroll
                for (int q = 0; q < kCopies; ++q)
                    x[q] = __ldcg(reinterpret_cast<const longlong2*>(accj + q * 128) + 2 * lane + v);
                long long hi = 0, lo = 0;
#pragma unroll
                for (int q = 0; q < kCopies; ++q) {
                    hi += x[q].x;
                    lo += x[q].y;
                }
                const double d = fma((double)hi, 281474976710656.0, (double)lo);
                const int Eu = egu - 1022, Ez = egz - 1022;
                val = scale2(d, lane < j ? (v ? Ez : Eu) - 83 : (v ? Eu + Ez : 2 * Eu) - 84);
            }
            s_v[v][lane] = val;
            const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)(lane < j ? expo(val) : 0));
            if (lane == 0) s_e[4 + v] = e;
            put_digits(tile + (v ? kTileT : kTileS) * kTP + tile_col<HALF>(lane) * 2, kTP,
                       lane < j ? fix62(val, e) : kBias);
            if (v == 0) {
                // how small s is beside u: 1 below 2^-12 (its six leading digit columns are
                // enough for the updates), 2 below 2^-16 (|s|^2 in FP32 is exact to FP64
                // rounding of |u|^2), 3 below 2^-32 (so are s.t and H s beside u.z and t);
                // usual: 3 in FP64, 2 in the mixed mode
                const int euu = __shfl_sync(0xffffffffu, expo(val), j & 31) - 1023;
                s_fs[lane] = lane < j ? d2f_trunc(scale2(val, 1022 - e)) : 0.f;
                const int gap = j == 0 || e == 0 ? 1000 : euu - 2 * (e - 1022);
                // (3 has H in FP32: its largest entries are near |A + r I|, which must be mid-range)
                const bool mid = eA >= -60 && eA <= 90;
                if (lane == 0) s_int[1] = gap >= 64 && mid ? 3 : gap >= 32 ? 2 : gap >= 24 ? 1 : 0;
            }
        } else if (wid == 8) {
            if (lane < 3) s_e[lane] = 0;
        } else if (!last) {
            // passes of four ghosts over warps 9-11, then 2-7 (which would otherwise wait for the sums)
            for (int x = gw; 4 * x < ng; x += 9) {
                const int gi = 4 * x + (lane >> 3);
                const double v = ghost_row<T>(A, z_of(t0 + gi), row_of(t0 + gi), gi < ng ? glen[gi] : 0, lane & 7, rw + gi * kRowCache,
                                              gi < nrc ? ri + gi * kRowCache : nullptr);
                if (gi < ng && (lane & 7) == 0) rz[gi] = v;
            }
        }
        if (wid <= 8) asm volatile("bar.sync 1, 288;" ::: "memory");
        if (wid == 8) {
            const int small = s_int[1];
            const bool in = lane < j;
            const double si = in ? s_v[0][lane] : 0.0, ti = in ? s_v[1][lane] : 0.0;
            const double uu = s_v[0][j & 31], uz = s_v[1][j & 31];
            const int nan = (int)__ldcg(&slot[(j & 1) * 2 + 1]);
            const int Es = s_e[4] - 1022, Et = s_e[5] - 1022;
            const float sf = s_fs[lane];
            float a = sf * sf, b = in ? sf * d2f_trunc(scale2(ti, -Et)) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
            }
            double ss = scale2(f2d_exact(a), 2 * Es), st = scale2(f2d_exact(b), Es + Et);
            if (small < 3) {
                st = si * ti;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) st += __shfl_xor_sync(0xffffffffu, st, o);
            }
            if (small < 2) {
                ss = si * si;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            }
            double q2 = uu - ss;   // h^2, clamped at +0
            if (__double_as_longlong(q2) < 0) q2 = 0.0;
            const double hinv = rsqrt_fast(q2);
            const double uzs = uz - st;
            int stop = nan == 0 && finite_bits(uzs) && finite_bits(uu) && finite_bits(q2) && (j == 0 || s_e[7] != 0x7ff)
                           ? 0 : 2;
            if (stop == 0) {
                // happy breakdown: h <= tol |A q_{j-1}|, |A q_{j-1}|^2 = |H[0..j-1, j-1]|^2 + |u|^2 with
                // the column before its second pass; by the exponents first (|H|^2 < 2^(2 (e + 1) + 5))
                const int eh = j > 0 ? 2 * (s_e[7] - 1022) + 5 : -4000;
                const int em = max(expo(uu) - 1022, eh) + 1 + 2 * (expo(A.tol) - 1022);
                if (expo(q2) == 0 || expo(q2) - 1023 <= em) {
                    double thr = 0.0;
                    if (j > 0) {
                        double hv = in ? sH[lane * 33 + j - 1] : 0.0;
                        if (shift && lane == j - 1) hv -= A.r;
                        double hh = hv * hv;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
                        thr = A.tol * A.tol * (hh + uu);
                    }
                    stop = __double_as_longlong(q2) <= __double_as_longlong(thr) ? 1 : 0;
                }
            }
            if (lane == 0) {
                s_int[0] = stop;
                s_sc[0] = q2;
                s_sc[1] = hinv;
                s_sc[2] = uzs * hinv;
                s_S.hinv = hinv;
                s_S.qz = uzs * hinv;
                if (sizeof(T) == 4) {
                    split2(s_S.hinv, s_S.hh, s_S.hl);
                    split2(s_S.qz, s_S.qh, s_S.ql);
                }
            }
        } else if (wid < 8 && !last) {
            // u - Q s and z - Q t (at a ghost: -Q t)
            const bool small = s_int[1] > 0;
            const int et = s_e[5] - 1022, es = s_e[4] - 1022;
            for (int pass = 0; pass < (small ? 1 : 2); ++pass) {
                if (pass == 1) {   // s in the place of t: ten of its digit columns for six
                    asm volatile("bar.sync 2, 256;" ::: "memory");
                    if (wid == 0)
                        put_digits(tile + kTileT * kTP + tile_col<HALF>(lane) * 2, kTP,
                                   lane < j ? fix62(s_v[0][lane], s_e[4]) : kBias);
                    asm volatile("bar.sync 2, 256;" ::: "memory");
                }
                for (int c0 = wid * cstep; c0 < Y.cols; c0 += kPW * cstep) {
                    const int c = c0 + lane;
                    longlong2 v = make_longlong2(0, 0);
                    if (j > 0) v = update_sums<NU, HALF>(Q, pitch, dstride, j, c0, tile, (float*)scr);
                    if (!wide) {
                        if (lane < 16) {
                            if (pass == 0) vv[c] = v;
                            else vv[c].y = v.x;
                        }
                    } else if (c < Y.cols) {   // (the last turn may read past the end of the rows)
                        // in place: FP64 and the ghosts, the differences; mixed points, FP32 pairs (u, ps), (z, pc)
                        const int gs = c >= ppb && c - ppb < ng ? (gpos[c - ppb] >> 24) & 31 : 0;
                        if (sizeof(T) == 4 && c < ppb) {
                            if (pass == 0) {
                                const float z = d2f_same(zs[c]), u = d2f_same(us[c]);
                                reinterpret_cast<float2*>(zs)[c] = make_float2(z, scaled_float(v.x, et - 60));
                                reinterpret_cast<float2*>(us)[c] = make_float2(u, scaled_float(v.y, es - 60));
                            } else {
                                reinterpret_cast<float2*>(us)[c].y = scaled_float(v.x, es - 60);
                            }
                        } else {
                            if (pass == 0) zs[c] = fma(-(double)v.x, pow2d(et - 60 + gs), c >= ppb ? 0.0 : zs[c]);
                            us[c] = fma(-(double)(pass == 0 ? v.y : v.x - v.y), pow2d(es - 60 + gs), us[c]);
                        }
                    }
                }
            }
        }
        __syncthreads();
        const int stop = s_int[0];
        if (j == 0 && threadIdx.x == 0) {
            const double b = scale2(s_sc[0] > 0.0 && finite_bits(s_sc[0]) ? s_sc[0] * s_sc[1] : s_sc[0], be);
            s_sc[3] = b;
            if (lead) *A.beta = b;
        }
        if (stop != 0 || last) {
            if (stop == 2 && lead) atomicOr(A.flags, 1);
            k = j;
            break;
        }
        // ---- q_j and the next u ---------------------------------------------------
        if (wid < 8) {
            const StepScalars S = s_S;
            const int et = s_e[5] - 1022, es = s_e[4] - 1022;
            for (int c0 = wid * 32; c0 < Y.cols; c0 += kPW * 32) {
                const int c = c0 + lane;
                int e = 0;
                const bool gh = c >= ppb;
                if (gh ? c - ppb < ng : c < n) {
                    const int gp = gh ? gpos[c - ppb] : 0;
                    T qj, un;
                    if (sizeof(T) == 4 && !gh) {
                        float2 a, b;
                        if (!wide) {
                            const longlong2 v = vv[c];
                            a = make_float2(d2f_same(us[c]), scaled_float(v.y, es - 60));
                            b = make_float2(d2f_same(zs[c]), scaled_float(v.x, et - 60));
                        } else {
                            a = reinterpret_cast<const float2*>(us)[c];
                            b = reinterpret_cast<const float2*>(zs)[c];
                        }
                        float q1, u1;
                        next_values_f(a.x, b.x, a.y, b.y, S, q1, u1);
                        qj = (T)q1;
                        un = (T)u1;
                    } else {
                        const longlong2 v = wide ? make_longlong2(0, 0) : vv[c];
                        double q1, u1;
                        const double z = gh ? (wide ? rz[c - ppb] + zs[c] : rz[c - ppb]) : zs[c];
                        next_values(us[c], z, v.y, es - 60 + ((gp >> 24) & 31), v.x, et - 60 + ((gp >> 24) & 31), S, q1, u1);
                        qj = (T)q1;
                        if (sizeof(T) == 4) u1 = fma(q1 - dbl(qj), S.qz * S.hinv, u1);   // with the rounded q_j
                        un = (T)u1;
                    }
                    us[c] = dbl(un);
                    lattice(gh ? (gp >> 29) & 3 : field(p0 + c))[gh ? gp & 0xffffff : meta_pos(meta[c])] = un;
                    e = expo(un);
                    put_value<HALF>(Q, pitch, dstride, j, c, fix62(qj, 1023 + ((gp >> 24) & 31)));
                }
                const int ea = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
                const int ep = (int)__reduce_max_sync(0xffffffffu, (unsigned)(gh ? 0 : e));
                if (lane == 0) {
                    atomicMax(&s_e[0], ep);
                    atomicMax(&s_e[1], ea);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(&slot[((j + 1) & 1) * 2], (unsigned)s_e[1]);
        if (!meet()) return calls;
    }
    // the last column's second pass; H to global memory; y = phi_1(dt H_k) e_1, by every block for itself
    if (wid == 8 && k > 0) {
        if (lane < k) sH[lane * 33 + k - 1] += s_v[0][lane];
        if (lane == 0) sH[k * 33 + k - 1] = s_sc[0] > 0.0 && finite_bits(s_sc[0]) ? s_sc[0] * s_sc[1] : s_sc[0];
        __syncwarp();
        if (shift && lane < k) sH[lane * 33 + lane] -= A.r;   // H of A
    }
    __syncthreads();
    if (bid == 0)
        for (int e = threadIdx.x; e < (k + 1) * k; e += kMT) {
            const int i = e / k, c = e - i * k;
            if (i <= c + 1) A.H[(size_t)i * m + c] = sH[i * 33 + c];
        }
    if (k == 0) {
        if (bid == 0)
            for (int t = threadIdx.x; t < m; t += kMT) A.y[t] = 0.0;
        if (lead) *A.kstop = 0;
        return calls;
    }
    const double beta = s_sc[3];
    const bool fine = phi1_mma(sH, k, A.dt, s_y, s_part, s_x, s_int);
    if (lead && !fine) atomicOr(A.flags, 1);
    if (bid == 0)
        for (int t = threadIdx.x; t < m; t += kMT) A.y[t] = s_y[t];
    // omega <- omega + dt beta V_k y at the own points, also into the lattice array L
    if (wid == 0) {
        const double cv = lane < k ? A.dt * beta * s_y[lane] : 0.0;
        const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)expo(cv));
        put_digits(tile + kTileT * kTP + tile_col<HALF>(lane) * 2, kTP, lane < k ? fix62(cv, e) : kBias);
        if (lane == 0) s_e[5] = e;
    }
    __syncthreads();
    if (wid < 8) {
        T* om = (T*)A.omega + p0;
        T* Lo = (T*)A.L;
        const double sc = s_e[5] == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : pow2d(s_e[5] - 1022 - 60);
        for (int c0 = wid * cstep; c0 < n; c0 += kPW * cstep) {
            const int c = c0 + lane;
            const longlong2 v = update_sums<NU, HALF>(Q, pitch, dstride, k, c0, tile, (float*)scr);
            if (lane < cstep && c < n) {
                if constexpr (EX) {
                    const int f = field(p0 + c), i = (int)(p0 + c - (long long)f * xn);
                    double* F = f == 2 ? X->f_out[2] : (f == 1 ? X->f_out[1] : X->f_out[0]);
                    const double x = fma((double)v.x, sc, F[i]);
                    F[i] = x;
                    (f == 2 ? X->Lb[2] : (f == 1 ? X->Lb[1] : X->Lb[0]))[meta_pos(meta[c])] = x;
                } else {
                    const T x = (T)fma((double)v.x, sc, dbl(om[c]));
                    om[c] = x;
                    Lo[meta_pos(meta[c])] = x;
                }
            }
        }
    }
    if (lead) *A.kstop = k;
    return calls;
}

template <typename T, int CL, int P, int FORM>
__global__ void __launch_bounds__(kMT, 1) k_krylov_mma(KrylovStepArgs A, int ppb, int gpb, int nrc) {
    extern __shared__ __align__(16) char k_sm[];
    bool formed = false;
    if constexpr (CL > 1) {
        // the pre-sums read peers' shared memory: a launch that did not form the clusters (some
        // profilers replay cooperative launches without them; the test switch A.refuse acts as
        // one) runs unclustered -- no peer access, no cluster barrier -- and says so in bit 4
        // (16) of *err
        formed = cooperative_groups::this_cluster().num_blocks() == (unsigned)CL && !A.refuse;
        if (!formed && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(A.err, 16);
    }
    const int calls = krylov_mma_body<T, CL, P, FORM>(A, blockIdx.x, gridDim.x, ppb, gpb, nrc, formed, k_sm);
    if constexpr (CL > 1) {
        if (formed) cluster_finish(calls, A.m + 1);
    }
    (void)calls;
}

template <int P, int FORM>
__global__ void __launch_bounds__(kMT, 1) k_ex_mma(KrylovStepArgs A, const __grid_constant__ ExArgs X, int ppb, int gpb,
                                                   int nrc) {
    extern __shared__ __align__(16) char k_sm[];
    krylov_mma_body<double, 1, P, FORM, true>(A, blockIdx.x, gridDim.x, ppb, gpb, nrc, false, k_sm, &X);
}

}  // namespace

template <typename T, int P>
const void* KrylovKernels<T, P>::ex_kernel(int form) {
    if constexpr (sizeof(T) == 8)
        return form == kNarrow ? (const void*)k_ex_mma<P, kNarrow>
                               : form == kHalves ? (const void*)k_ex_mma<P, kHalves> : (const void*)k_ex_mma<P, kWords>;
    else
        return nullptr;
}
template <typename T, int P>
const void* KrylovKernels<T, P>::mma_kernel(int cl, int form) {
    if (form == kNarrow) return cl == 4 ? (const void*)k_krylov_mma<T, 4, P, kNarrow> : (const void*)k_krylov_mma<T, 1, P, kNarrow>;
    return form == kHalves ? (const void*)k_krylov_mma<T, 1, P, kHalves> : (const void*)k_krylov_mma<T, 1, P, kWords>;
}
template <typename T, int P>
int KrylovKernels<T, P>::mma_threads() {
    return kMT;
}
template <typename T, int P>
size_t KrylovKernels<T, P>::mma_bytes(int form, int m, int ppb, int gpb, int nrc) {
    return mma_layout(form, m, ppb, gpb, nrc).bytes;
}

}  // namespace wrc
