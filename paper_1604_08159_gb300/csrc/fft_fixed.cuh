#pragma once
// The FP64 transforms of the streamfunction solve in 64-bit fixed point.
//
// An FP64 addition takes ~70 cycles per warp and SM sub-partition on this
// part, a 64-bit integer addition 2.3 and a 32 x 32 -> 64-bit multiply-add
// ~5 (measured), so the butterflies run on integers: a transform's values
// share one exponent (block floating point), renewed at every exchange
// between passes from the largest value present, so that components use 57
// bits and a radix-8 pass has its headroom (8 sqrt(2) 2^57 < 2^61).  Twiddles
// are two 30-bit halves; a complex product is twelve 32 x 32 -> 64
// multiply-adds, its low halves' product added from their leading 15 bits,
// rounded once.  Conversions from FP64 are integer work; conversions back and
// the division by the symbol (a table: a division is nine FP64 instructions)
// take the FP64 pipe, otherwise idle, beside.
//
// Accuracy: a pass adds errors of ~2^-57 of the transform's largest value.
// Against an 80-bit solve the right-hand side that psi reproduces is off by
// 0.5 to 0.7 of what the FP64 transforms left, on lattices of 8^2 to 2048^2, for
// vortices and for noise (2048^2: 4.4e-12 of 8.7e-12, 9.4e-14 of 1.3e-13,
// relative L2); psi itself by the same, the symbol's rounding.
//
// Bound: the integer multiply and ALU pipes from 1024^2 on (half of the issue
// slots taken), the chain of one warp's instructions below, hence 8 values
// per thread (16 take 104 us at 1024^2 and 31 solves 12% longer at 512^2) and
// 4 on lattices up to 512^2.  psi's solve takes, FP64 transforms before:
// 128^2 94 -> 29 us, 512^2 ~110 -> 38, 1024^2 176 -> 70.
// Included by fft.cu inside its namespace.

using I2 = longlong2;
constexpr int kFxThreads = 512;        // 4096 points, 8 per thread
constexpr int kFxBits = 57;            // components below 2^kFxBits when a pass starts
constexpr long long kQ30 = 1ll << 30;

constexpr long long kFxR2 = 815238614083298888ll;   // 2^60 sqrt(1/2)

__device__ __forceinline__ int fx_hi(long long a) { return (int)(a >> 30); }
__device__ __forceinline__ int fx_lo(long long a) { return (int)a & 0x3fffffff; }
// The 30-bit halves' low product, in units of 2^30 (from 15 bits of each).
__device__ __forceinline__ int fx_ll(int a, int b) { return (a >> 15) * (b >> 15); }

// a (c - i s), c = ch 2^30 + cl and s likewise, over 2^60.
__device__ __forceinline__ I2 fx_mul(I2 a, int4 w) {
    const int ch = w.x, cl = w.y, sh = w.z, sl = w.w;
    const int xh = fx_hi(a.x), xl = fx_lo(a.x), yh = fx_hi(a.y), yl = fx_lo(a.y);
    const long long half = 1ll << 29;
    const long long mr = (long long)xl * ch + (long long)xh * cl + (long long)yl * sh + (long long)yh * sl + half +
                         ((long long)fx_ll(xl, cl) + fx_ll(yl, sl));
    const long long mi = (long long)yl * ch + (long long)yh * cl - ((long long)xl * sh + (long long)xh * sl) + half +
                         (fx_ll(yl, cl) - fx_ll(xl, sl));
    I2 r;
    r.x = (long long)xh * ch + (long long)yh * sh + (mr >> 30);
    r.y = (long long)yh * ch - (long long)xh * sh + (mi >> 30);
    return r;
}
// a sqrt(1/2)
__device__ __forceinline__ long long fx_r2(long long a) {
    constexpr int rh = (int)(kFxR2 >> 30), rl = (int)(kFxR2 & (kQ30 - 1));
    const int ah = fx_hi(a), al = fx_lo(a);
    const long long mid = (long long)al * rh + (long long)ah * rl + (1ll << 29) + fx_ll(al, rl);
    return (long long)ah * rh + (mid >> 30);
}
__device__ __forceinline__ void fx_dft8(I2 (&a)[8]) {
    I2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6];
    I2 o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
    dft4<false>(e0, e1, e2, e3);
    dft4<false>(o0, o1, o2, o3);
    o1 = mk<I2>(fx_r2(o1.x + o1.y), fx_r2(o1.y - o1.x));   // times exp(-i pi/4)
    o2 = mul_mi<false>(o2);
    o3 = mk<I2>(fx_r2(o3.y - o3.x), -fx_r2(o3.x + o3.y));  // times exp(-3 i pi/4)
    a[0] = cadd(e0, o0);
    a[4] = csub(e0, o0);
    a[1] = cadd(e1, o1);
    a[5] = csub(e1, o1);
    a[2] = cadd(e2, o2);
    a[6] = csub(e2, o2);
    a[3] = cadd(e3, o3);
    a[7] = csub(e3, o3);
}
template <int R>
__device__ __forceinline__ void fx_dft(I2 (&u)[R]) {
    if constexpr (R == 2) dft2<false>(u[0], u[1]);
    else if constexpr (R == 4) dft4<false>(u[0], u[1], u[2], u[3]);
    else fx_dft8(u);
}

// What the threads of one transform share beyond their values: the largest
// magnitude of an exchange.  A transform of at most 32 threads (nt) combines
// it within its lanes; a wider one through word `ev` of slot[], zeroed at
// the start of the kernel, one word per exchange.
struct FxShare {
    unsigned* slot;    // [kFxEvents] of this transform
    unsigned mask;     // lanes of the transform (nt <= 32)
    int nt, ev;
};
constexpr int kFxEvents = 12;

template <bool MAX>
__device__ __forceinline__ void fx_gather(FxShare& h, unsigned& x) {
    x = MAX ? __reduce_max_sync(h.mask, x) : __reduce_or_sync(h.mask, x);
    if (h.nt > 32 && (threadIdx.x & 31) == 0) {
        if (MAX) atomicMax(h.slot + h.ev, x);
        else atomicOr(h.slot + h.ev, x);
    }
}
// After the block's barrier.
__device__ __forceinline__ unsigned fx_gathered(FxShare& h, unsigned x) {
    if (h.nt > 32) x = h.slot[h.ev];
    h.ev += 1;
    return x;
}
__device__ __forceinline__ unsigned fx_mag(I2 a) {   // bits of the high words' magnitudes
    const int x = (int)(a.x >> 32), y = (int)(a.y >> 32);
    return (unsigned)((x ^ (x >> 31)) | (y ^ (y >> 31)));
}
// v 2^s, rounded for s < 0.
__device__ __forceinline__ long long fx_shift(long long v, int s) {
    return s >= 0 ? v << s : (v + (1ll << (-s - 1))) >> -s;
}

// As radix_pass, on integers: after the exchange the values are scaled to
// kFxBits bits by the transform's largest one.  ptw: (ch, cl, sh, sl) of
// cos and sin.
template <int E, int R>
__device__ __forceinline__ void fx_pass(I2 (&v)[E], int& ex, I2* sm, int i, int nt, int p, const int4* __restrict__ ptw,
                                        bool last, FxShare& h) {
    constexpr int G = E / R;
    const int pi = pad(i);
    unsigned big = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const int b = i + nt * g;
        const int k = b & (p - 1);
        I2 u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = v[g + r * G];
        if (p > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                u[r] = fx_mul(u[r], __ldg(ptw + r * p + k));
            }
        }
        fx_dft<R>(u);
        if (last) {
#pragma unroll
            for (int r = 0; r < R; ++r) v[g + r * G] = u[r];
        } else {
            const int wb = pad((b - k) * R + k);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                sm[wb + pad(r * p)] = u[r];
                big |= fx_mag(u[r]);
            }
        }
    }
    if (!last) {
        fx_gather<false>(h, big);
        __syncthreads();
        big = fx_gathered(h, big);
        const int s = kFxBits - 64 + __clz((int)(big | 1u));   // the top bit to position kFxBits - 1
        ex -= s;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const I2 a = sm[pi + pad(e * nt)];
            v[e].x = fx_shift(a.x, s);
            v[e].y = fx_shift(a.y, s);
        }
        __syncthreads();
    }
}

template <int E, int R0>
__device__ __forceinline__ void fx_fft(I2 (&v)[E], int& ex, I2* sm, int i, int n, int logn, const int4* __restrict__ tw,
                                       FxShare& h) {
    const int nt = n / E;
    int p = 1, logp = 0;
    const int4* ptw = tw;
    if constexpr (R0 > 1) {
        fx_pass<E, R0>(v, ex, sm, i, nt, p, ptw, false, h);
        p *= R0;
        logp += Log2<R0>::v;
    }
    const int npass = (logn - logp) / Log2<E>::v;
#pragma unroll 1
    for (int q = 0; q < npass; ++q) {
        fx_pass<E, E>(v, ex, sm, i, nt, p, ptw, q == npass - 1, h);
        if (p > 1) ptw += E * p;
        p *= E;
        logp += Log2<E>::v;
    }
}

constexpr int kFxBad = 1 << 20;   // exponent of a transform with a non-finite input: its outputs are NaN

// d[] (FP64 components) -> v[] below 2^kFxBits with a common exponent.
template <int E>
__device__ __forceinline__ void fx_from(const double2 (&d)[E], I2 (&v)[E], int& ex, FxShare& h) {
    unsigned em = 0;
#pragma unroll
    for (int e = 0; e < E; ++e)
        em = max(em, max((unsigned)__double2hiint(d[e].x) & 0x7fffffffu, (unsigned)__double2hiint(d[e].y) & 0x7fffffffu));
    fx_gather<true>(h, em);
    __syncthreads();
    const int emax = (int)(fx_gathered(h, em) >> 20);
    ex = emax == 0x7ff ? kFxBad : emax - 1022 - kFxBits;
    const auto fix = [&](double x) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        const int e = (int)(b >> 52) & 0x7ff, r = emax - e;
        unsigned long long y = e ? ((b & 0xfffffffffffffull) | 0x10000000000000ull) << (kFxBits - 53) : 0ull;
        if (r > 0) y = r < 60 ? (y + ((1ull << r) >> 1)) >> r : 0ull;
        return (long long)b < 0 ? -(long long)y : (long long)y;
    };
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e].x = fix(d[e].x);
        v[e].y = fix(d[e].y);
    }
}
// Outside the exponents that an integer addition can serve.
__device__ __noinline__ double fx_far(double x, int ex) {
    return ex >= kFxBad / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(x, ex);
}
// a 2^ex in FP64 (rounded once).
__device__ __forceinline__ double fx_to(long long a, int ex) {
    const double x = (double)a;
    if (ex > -900 && ex < 900) {
        const int hi = __double2hiint(x);
        return __hiloint2double(hi ? hi + (ex << 20) : 0, __double2loint(x));
    }
    return fx_far(x, ex);
}

__device__ __forceinline__ FxShare fx_share(unsigned* slot, int nt) {
    FxShare h;
    h.slot = slot;
    const int lane = threadIdx.x & 31;
    h.mask = nt >= 32 ? 0xffffffffu : ((1u << nt) - 1u) << (lane / nt * nt);
    h.nt = nt;
    h.ev = 0;
    if (threadIdx.x < kFxEvents) slot[threadIdx.x] = 0u;
    __syncthreads();
    return h;
}

// The per-pass twiddle tables, as k_fft_pass_tables, split for fx_mul.
__global__ void k_fx_pass_tables(int4* __restrict__ ptw, int n, int logn, int logE) {
    pdl_wait();
    int p = 1, logp = 0, off = 0;
    auto table = [&](int R, int logR) {
        if (p > 1)
            for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < R * p; idx += gridDim.x * blockDim.x) {
                const int r = idx / p, k = idx - r * p;
                const int t = (r * k) << (logn - logp - logR);
                double sn, cs;
                sincospi(2.0 * t / n, &sn, &cs);
                const long long c = __double2ll_rn(cs * 0x1p60), s = __double2ll_rn(sn * 0x1p60);
                ptw[off + idx] = make_int4((int)(c >> 30), (int)(c & (kQ30 - 1)), (int)(s >> 30), (int)(s & (kQ30 - 1)));
            }
        if (p > 1) off += R * p;
        p *= R;
        logp += logR;
    };
    if (logn % logE) table(1 << logn % logE, logn % logE);
    while (logp < logn) table(1 << logE, logE);
    pdl_trigger();
}
// inv[kx][ky] = scale / (sigma(kx) + sigma(ky)), kx <= n/2, 0 at kx = ky = 0
// (a division is nine FP64 instructions).
__global__ void k_fx_symbol(double* __restrict__ inv, const double* sigma, int n) {
    pdl_wait();
    const long long N = (long long)(n / 2 + 1) * n;
    const double scale = 1.0 / ((double)n * (double)n);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < N; e += (long long)gridDim.x * blockDim.x)
        inv[e] = e == 0 ? 0.0 : scale / (sigma[e / n] + sigma[e % n]);
    pdl_trigger();
}

// Step 1 (see k_px_fwd).  In these kernels the wait for the predecessor comes
// before anything else and its data is read by coherent loads (see launch_pdl).
template <int E, int R0>
__global__ void __launch_bounds__(kFxThreads) k_px_fwd_fx(const double* Rf, double2* __restrict__ S, int n,
                                                   int logn, const int4* __restrict__ tw) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned s_slot[kFxEvents];
    const int nt = n / E, F = blockDim.x / nt;
    const int f = threadIdx.x / nt, i = threadIdx.x - f * nt;
    FxShare sh = fx_share(s_slot, nt);
    const int h = n / 2;
    const int q = blockIdx.x * F + f;
    const bool on = q < h;
    I2* sm = (I2*)smraw + (size_t)f * smlen_of(n);
    I2 v[E];
    int ex;
    {
        double2 d[E];
        const double* r0 = Rf + (size_t)(2 * q) * n;
        const double* r1 = r0 + n;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int x = i + e * nt;
            d[e] = on ? make_double2(__ldcg(r0 + x), __ldcg(r1 + x)) : make_double2(0.0, 0.0);
        }
        fx_from(d, v, ex, sh);
    }
    fx_fft<E, R0>(v, ex, sm, i, n, logn, tw, sh);
#pragma unroll
    for (int e = 0; e < E; ++e) sm[pad(i + e * nt)] = v[e];
    __syncthreads();
    double2* sa = S + (size_t)(2 * q) * h;
    double2* sb = sa + h;
#pragma unroll
    for (int e = 0; e < E / 2; ++e) {
        const int x = i + e * nt;   // < n/2
        if (!on) continue;
        const I2 z = v[e];
        if (x == 0) {
            const I2 zh = sm[pad(h)];
            sa[0] = make_double2(fx_to(z.x, ex), fx_to(zh.x, ex));
            sb[0] = make_double2(fx_to(z.y, ex), fx_to(zh.y, ex));
        } else {
            const I2 zm = cconj(sm[pad(n - x)]);
            const I2 s = cadd(z, zm), d = csub(z, zm);
            sa[x] = make_double2(fx_to(s.x, ex - 1), fx_to(s.y, ex - 1));
            sb[x] = make_double2(fx_to(d.y, ex - 1), fx_to(-d.x, ex - 1));
        }
    }
    pdl_trigger();
}

// Step 3 for psi (see k_py_solve).
template <int E, int R0>
__global__ void __launch_bounds__(kFxThreads) k_py_solve_fx(double2* __restrict__ ST, int n, int logn,
                                                     const int4* __restrict__ tw, const double* __restrict__ inv) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned s_slot[kFxEvents];
    const int nt = n / E, F = blockDim.x / nt;
    const int f = threadIdx.x / nt, i = threadIdx.x - f * nt;
    FxShare sh = fx_share(s_slot, nt);
    const int h = n / 2;
    const int kx = blockIdx.x * F + f;
    const bool on = kx < h;
    const int kxs = on ? kx : 0;
    I2* sm = (I2*)smraw + (size_t)f * smlen_of(n);
    double2* row = ST + (size_t)kxs * n;
    I2 v[E];
    int ex;
    double2 d[E];
#pragma unroll
    for (int e = 0; e < E; ++e) d[e] = on ? row[i + e * nt] : make_double2(0.0, 0.0);
#pragma unroll 1
    for (int inverse = 0;; ++inverse) {   // one copy of the transform's code: the inverse as conj FFT conj
        fx_from<E>(d, v, ex, sh);
        fx_fft<E, R0>(v, ex, sm, i, n, logn, tw, sh);
        if (inverse) break;
        if (blockIdx.x == 0) {   // holds the packed column kx = 0, which reads F(n - ky) too
#pragma unroll
            for (int e = 0; e < E; ++e) sm[pad(i + e * nt)] = v[e];
            __syncthreads();
        }
        if (kxs == 0) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int ky = i + e * nt;
                const I2 fk = v[e], fm = blockIdx.x == 0 ? cconj(sm[pad((n - ky) & (n - 1))]) : v[e];
                const I2 s = cadd(fk, fm), dd = csub(fk, fm);
                const double f0 = inv[ky], fn = inv[(size_t)h * n + ky];
                // conj(X1 + i X2), X1 = s f0 / 2, X2 = -i dd fn / 2
                d[e].x = fx_to(s.x, ex - 1) * f0 + fx_to(dd.x, ex - 1) * fn;
                d[e].y = -(fx_to(s.y, ex - 1) * f0 + fx_to(dd.y, ex - 1) * fn);
            }
        } else {
            const double* fr = inv + (size_t)kxs * n;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const double fc = fr[i + e * nt];
                d[e].x = fx_to(v[e].x, ex) * fc;
                d[e].y = fx_to(-v[e].y, ex) * fc;
            }
        }
        __syncthreads();   // sm becomes the exchange buffer again
    }
    if (on)
#pragma unroll
        for (int e = 0; e < E; ++e) row[i + e * nt] = make_double2(fx_to(v[e].x, ex), fx_to(-v[e].y, ex));
    pdl_trigger();
}

// Step 5 for psi (see k_px_inv_real).
template <int E, int R0>
__global__ void __launch_bounds__(kFxThreads) k_px_inv_fx(const double2* S, double* __restrict__ out, int n,
                                                   int logn, const int4* __restrict__ tw,
                                                   const int* rows) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned s_slot[kFxEvents];
    const int nt = n / E, F = blockDim.x / nt;
    const int f = threadIdx.x / nt, i = threadIdx.x - f * nt;
    FxShare sh = fx_share(s_slot, nt);
    const int h = n / 2;
    int q = blockIdx.x * F + f;
    if (rows) {
        const int cnt = rows[h];
        if ((int)blockIdx.x * F >= cnt) {
            pdl_trigger();
            return;
        }
        q = q < cnt ? rows[h + 1 + q] : h;   // h: no pair
    }
    const bool on = q < h;
    I2* sm = (I2*)smraw + (size_t)f * smlen_of(n);
    const double2* sa = S + (size_t)(2 * (on ? q : 0)) * h;
    const double2* sb = sa + h;
    I2 v[E];
    int ex;
    {
        double2 d[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int x = i + e * nt;
            double2 a, b;
            if (x == 0) {
                a = make_double2(__ldcg(sa).x, 0.0);
                b = make_double2(__ldcg(sb).x, 0.0);
            } else if (x == h) {
                a = make_double2(__ldcg(sa).y, 0.0);
                b = make_double2(__ldcg(sb).y, 0.0);
            } else if (x < h) {
                a = __ldcg(sa + x);
                b = __ldcg(sb + x);
            } else {
                a = cconj(__ldcg(sa + n - x));
                b = cconj(__ldcg(sb + n - x));
            }
            d[e] = on ? make_double2(a.x - b.y, -(a.y + b.x)) : make_double2(0.0, 0.0);   // conj(a + i b)
        }
        fx_from(d, v, ex, sh);
    }
    fx_fft<E, R0>(v, ex, sm, i, n, logn, tw, sh);
    if (!on) return;
    double* o0 = out + (size_t)(2 * q) * n;
    double* o1 = o0 + n;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        o0[i + e * nt] = fx_to(v[e].x, ex);
        o1[i + e * nt] = fx_to(-v[e].y, ex);
    }
    pdl_trigger();
}

// The shapes: radix-E passes, after one of radix 2 or 4 when log2 n is not a
// multiple of log2 E.  One transform per block where it has a warp, else a
// warp of transforms: the solves are short of blocks, not of warps per block.
template <int E, int R0>
struct FxShape {
    static int setup() {
        int bad = 0;
        bad |= cudaFuncSetAttribute(k_px_fwd_fx<E, R0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        bad |= cudaFuncSetAttribute(k_py_solve_fx<E, R0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        bad |= cudaFuncSetAttribute(k_px_inv_fx<E, R0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        return bad;
    }

    static void run(const PoissonPlan& p, const double* Rf, double* psi, double2* S, cudaStream_t s, const int* rows) {
        const int n = p.n, logn = p.logn, h = n / 2;
        const int nt = n / E, F = nt >= 32 ? 1 : 32 / nt, thr = F * nt, blocks = (h + F - 1) / F;
        const size_t smem = sizeof(I2) * (size_t)F * smlen_of(n);
        const int4* tw = (const int4*)p.ptw;
        const double* inv = (const double*)p.inv;
        double2* ST = S + (size_t)n * h;   // S: n x h half spectra; ST: h x n, transposed
        const dim3 tb(32, 8), g_nh((h + 31) / 32, (n + 31) / 32), g_hn((n + 31) / 32, (h + 31) / 32);
        { launch_pdl(k_px_fwd_fx<E, R0>, blocks, thr, smem, s, Rf, S, n, logn, tw); note_launch(); }
        { launch_pdl(k_transpose<double2>, g_nh, tb, 0, s, S, ST, n, h); note_launch(); }
        { launch_pdl(k_py_solve_fx<E, R0>, blocks, thr, smem, s, ST, n, logn, tw, inv); note_launch(); }
        { launch_pdl(k_transpose<double2>, g_hn, tb, 0, s, ST, S, h, n); note_launch(); }
        { launch_pdl(k_px_inv_fx<E, R0>, blocks, thr, smem, s, S, psi, n, logn, tw, rows); note_launch(); }
        if (rows && poison_rows()) { launch_pdl(k_poison_rows<double>, 1216, 256, 0, s, psi, (double*)nullptr, rows, n); note_launch(); }
    }
};

// log2 of the values per thread.  4 halve a thread's chain, 8 take fewer
// exchanges: 128^2 29 against 39 us, 512^2 37.5 / 38.8, 1024^2 77 / 70.
int fx_log_e(int logn) { return logn <= 9 ? 2 : 3; }
