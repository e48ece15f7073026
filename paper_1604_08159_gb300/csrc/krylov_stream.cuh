#pragma once
// The streaming form of the tensor-core Krylov step (krylov_mma.cuh has the
// method, the digit products and the exact sums): the basis as 64-bit
// integers in global memory, read once for the dots and once for the updates
// of a step, for problems whose table does not fit shared memory and for
// several problems in one cooperative launch (the members of an ensemble or
// of the server's batch, or omega and the passive scalar of one run).
//
// A problem is worked on by its nb blocks (one block of twelve warps per
// SM), which meet at its own grid barriers; a problem of one block needs
// none.  A block may take several problems in turn (batch_plan.h), so that
// any number of them runs in one launch.
//
// What bounds it: the products' conversions (digits unpacked from 64-bit
// integers while they are loaded) and their loads, ~300 bytes per point and
// Arnoldi step at m = 30; the updates follow the scalars of a step, so that
// each column is read once: its sums, q_j, the next u and its lattice entry.
// Measured on GB300: see krylov_plan() in krylov.cu and batch_plan.h.
#include "krylov_mma.cuh"

namespace wrc {

namespace {

constexpr int kSW = 12;                            // warps, all taking points, units and columns
constexpr int kSTile = 1440, kSX = 1280;           // per warp: u, z digit tile; exchange of the updates
constexpr int kSP = 20;                            // words per row of a stage: 16 columns + pad (= 4 mod 16)
constexpr int kSStage = 32 * kSP * 8;              // a stage: 16 columns of up to 32 rows

struct StreamLayout {
    size_t scr, xch, stage, tile, tile2, sH, bytes;
};
__host__ __device__ inline StreamLayout stream_layout() {
    StreamLayout L;
    size_t o = 0;
    L.scr = o;   o += (size_t)kSW * kSTile;
    L.xch = o;   o += (size_t)kSW * kSX;
    L.stage = o; o += (size_t)kSW * 2 * kSStage;
    L.tile = o;  o += (size_t)kTP * 32;
    L.tile2 = o; o += (size_t)kTP * 32;
    L.sH = o;    o += sizeof(double) * 32 * 33;
    L.bytes = (o + 15) / 16 * 16;
    return L;
}

// Rows 0 .. nrow - 1 of the 16 columns at `src` (16-byte aligned, ld words a
// row) into a stage, asynchronously (one commit group).
__device__ __forceinline__ void stage_load(char* stage, const unsigned long long* src, int ld, int nrow) {
    const int lane = threadIdx.x & 31;
    const unsigned to = smem_addr(stage);
    for (int e = lane; e < nrow * 8; e += 32) {
        const int row = e >> 3, seg = e & 7;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + row * (kSP * 8) + seg * 16),
                     "l"(src + (size_t)row * ld + seg * 2)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void stage_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}

template <typename T, int P>
__device__ __forceinline__ void krylov_stream_body(const KrylovStepArgs& A, const int bid, const int nb, char* sm) {
    __shared__ double s_v[2][32];        // s (and |u|^2), t (and u.z) of a step
    __shared__ double s_part[kPW][33];
    __shared__ double s_y[32], s_x[32];
    __shared__ double s_sc[4];           // h^2, 1/h, qz, beta
    __shared__ StepScalars s_S;
    __shared__ int s_e[8];               // exponents, as in krylov_mma_body
    __shared__ int s_int[4], s_ok, s_next;
    __shared__ longlong2 s_bp[64];
    const StreamLayout Y = stream_layout();
    double* sH = reinterpret_cast<double*>(sm + Y.sH);
    char* tile = sm + Y.tile;
    char* tile2 = sm + Y.tile2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    char* tu = sm + Y.scr + (size_t)wid * kSTile;
    float* xch = reinterpret_cast<float*>(sm + Y.xch + (size_t)wid * kSX);
    char* stage[2] = {sm + Y.stage + (size_t)(2 * wid) * kSStage, sm + Y.stage + (size_t)(2 * wid + 1) * kSStage};
    const int m = A.m;
    const long long ppb = ((A.n + nb - 1) / nb + 31) / 32 * 32, p0 = (long long)bid * ppb;
    const int n = (int)max(0ll, min(ppb, (long long)A.n - p0));               // points of this block
    const int gev = (int)((((long long)A.ng + nb - 1) / nb + 15) / 16 * 16);   // (stages start on 16 columns)
    const long long t0 = (long long)bid * gev;
    const int ng = (int)max(0ll, min((long long)gev, (long long)A.ng - t0));   // ghosts
    const bool lead = bid == 0 && threadIdx.x == 0;
    const uint32_t* meta = A.meta + p0;
    const T* Ua = (const T*)A.Ua + p0;
    const T* Va = (const T*)A.Va + p0;
    T* Lq = (T*)A.Lq;
    T* zb = (T*)A.w;                     // z at every active point
    T* us = (T*)A.us + p0;               // u at the own points
    // the basis: rows of points and rows of ghosts, then u, z and the scale bits of the ghosts
    unsigned long long* Q = (unsigned long long*)A.basis + p0;
    unsigned long long* G = (unsigned long long*)A.Gb + t0;
    const int ld = (int)A.ld, ldg = (int)A.ldg;
    double* ug = (double*)A.Gb + (size_t)m * ldg + t0;
    double* rz = ug + ldg;
    int* gsx = (int*)((double*)A.Gb + (size_t)(m + 2) * ldg) + t0;
    const T nu = (T)A.nu, r = (T)A.r, c1J = (T)A.c1J, c2J = (T)A.c2J;
    const bool shift = A.r != 0.0;       // the steps apply A + r I, as in krylov_mma_body
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(A.part);
    unsigned* slot = reinterpret_cast<unsigned*>(acc + 2 * kCopies * 128);
    const bool solo = nb == 1;           // no other block: no grid barrier
    int ph = 0;
    if (lead && A.trace) A.trace[0] = gtimer();
    if (*(volatile const int*)A.row_overflow) {
        if (lead) atomicOr(A.err, 4);
        return;
    }
    if (*(volatile int*)A.err & kErrStop) return;
    unsigned phase = *(volatile unsigned*)A.bar & 0x80000000u;
    const auto meet = [&]() {
        if (solo) {
            __syncthreads();
            if (lead && A.trace && ph < kTracePhases) {
                A.trace[1 + (size_t)ph * 2] = gtimer();
                A.trace[2 + (size_t)ph * 2] = gtimer();
            }
            ++ph;
            return true;
        }
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
    for (int c = threadIdx.x; c < 32 * 33; c += kMT) sH[c] = 0.0;
    for (int c = threadIdx.x; c < 2 * kTP * 32 / 4; c += kMT) reinterpret_cast<unsigned*>(tile)[c] = 0u;
    for (int t = lane; t < kSTile / 4; t += 32) reinterpret_cast<unsigned*>(tu)[t] = 0u;
    if (threadIdx.x < 8) s_e[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();

    // b = A_n omega + g and the bound of |A|_inf, as in krylov_mma_body
    for (int c = wid * 32; c < n; c += 32 * kSW) {
        const int p = c + lane;
        int ea = 0, e = 0;
        if (p < n) {
            const uint32_t mw = meta[p];
            const T U = Ua[p], V = Va[p];
            T v = apply_point<T, false, P>((const T*)A.L, mw, U, V, nu, r, A.g, c1J, c2J);
            if (A.ga) v += ((const T*)A.ga)[p0 + p];
            us[p] = v;
            zb[p0 + p] = v;
            Lq[meta_pos(mw)] = v;
            e = expo(v);
            ea = expo(row_bound<T, P>(A, mw, U, V));
        }
        ea = (int)__reduce_max_sync(0xffffffffu, (unsigned)ea);
        e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
        if (lane == 0) {
            atomicMax(&s_e[6], ea);
            atomicMax(&s_e[0], e);
            atomicMax(&s_e[1], e);
        }
    }
    if (!meet()) return;
    for (int q = wid * 4; q < ng; q += 4 * kSW) {
        const int gi = q + (lane >> 3), gl = lane & 7;
        const bool valid = gi < ng;
        const int rl = valid ? A.row_len[t0 + gi] : 0;
        const double v = ghost_row<T>(A, zb, t0 + gi, rl, gl, nullptr, nullptr);
        const int gs = ghost_scale(A, t0 + gi, rl, gl);
        int e = 0;
        if (valid && gl == 0) {
            const T gv = (T)v;
            gsx[gi] = gs;
            ug[gi] = dbl(gv);
            Lq[A.glist[t0 + gi]] = gv;
            e = expo(gv);
        }
        e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
        if (lane == 0) atomicMax(&s_e[1], e);
    }
    __syncthreads();
    if (threadIdx.x == 0 && !solo) {
        atomicMax(&slot[0], (unsigned)s_e[1]);
        atomicMax(&slot[4], (unsigned)s_e[6]);
    }
    if (!meet()) return;
    const int be = first_scale<T>(solo ? s_e[1] : (int)__ldcg(&slot[0]));
    if (be != 0) {   // as in krylov_mma_body
        for (int c = threadIdx.x; c < n; c += kMT) {
            const T v = (T)scale2(dbl(us[c]), -be);
            us[c] = v;
            Lq[meta_pos(meta[c])] = v;
        }
        for (int c = threadIdx.x; c < ng; c += kMT) {
            const T v = (T)scale2(ug[c], -be);
            ug[c] = dbl(v);
            Lq[A.glist[t0 + c]] = v;
        }
        __syncthreads();   // s_e[1] has been read
        if (threadIdx.x < 2 && s_e[threadIdx.x]) s_e[threadIdx.x] = max(0, s_e[threadIdx.x] - be);
        if (!meet()) return;
    }

    const int nunit = (n + 15) / 16;
    const int nact = min(kSW, nunit);
    int k = m;
    const int eA = (solo ? s_e[6] : (int)__ldcg(&slot[4])) - 1022 + 1;
    for (int j = 0;; ++j) {
        const bool last = j == m;
        unsigned long long* accj = acc + (j & 1) * kCopies * 128;
        // ---- column j - 1 of H (warp 8), z = A u at the own points ------------
        if (wid == 8) {
            if (lane == 0) s_e[3] = solo ? s_e[1] : (int)__ldcg(&slot[(j & 1) * 2]) - (j == 0 ? be : 0);
            for (int q = bid; q < kCopies && !solo; q += nb) {
                unsigned long long* z = acc + (((j + 1) & 1) * kCopies + q) * 128;
                for (int t = lane; t < 128; t += 32) z[t] = 0ull;
            }
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
                for (int c = 0; c < q; ++c) gi += sH[lane * 33 + c] * s_v[0][c];
                double v = 0.0;
                if (lane < q) v = (s_v[1][lane] - gi) * hinv;
                else if (lane == q) v = (qz - (q > 0 ? h * s_v[0][q - 1] : 0.0)) * hinv;
                if (lane <= q) sH[lane * 33 + q] = v;
                const int ev = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(expo(v), shift ? expo(A.r) : 0));
                if (lane == 0) s_e[7] = ev;
            }
        }
        if (bid == 0 && threadIdx.x < 2) slot[((j + 1) & 1) * 2 + threadIdx.x] = 0u;
        if (!last) {
            // two chunks of 32 points at a time, their constants fetched one turn ahead
            uint32_t mw[2];
            T U[2], V[2];
            const auto fetch = [&](int c) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int p = c + 32 * kSW * q + lane;
                    mw[q] = p < n ? meta[p] : 0u;
                    U[q] = p < n ? Ua[p] : T(0);
                    V[q] = p < n ? Va[p] : T(0);
                }
            };
            fetch(wid * 32);
            for (int c = wid * 32; c < n; c += 64 * kSW) {
                OpPoint<T> op[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) op_prepare<T, P>(op[q], mw[q], U[q], V[q], nu, A.g, c1J, c2J);
                fetch(c + 64 * kSW);
                T z[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) z[q] = op_apply<T, P>(Lq, op[q], T(0), A.g, c1J, c2J);
                int e = 0;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int p = c + 32 * kSW * q + lane;
                    if (p < n) {
                        zb[p0 + p] = z[q];
                        e = max(e, expo(z[q]));
                    }
                }
                e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
                if (lane == 0) atomicMax(&s_e[2], e);
            }
        }
        __syncthreads();
        // ---- dots -----------------------------------------------------------------
        const int eu = s_e[0], ez = s_e[2], egu = s_e[3];
        if (wid < nact) {
            const int g = lane >> 2, tg = lane & 3;
            const int mr = (lane & 7) + ((lane >> 3) & 1) * 15 + 7;
            const unsigned ta = smem_addr(tu) + mr * kUP + (lane >> 4) * 16;
            const auto dots = [&](auto ntc) {
                constexpr int NT = decltype(ntc)::value;
                float c[NT][2][4];
                long long sum[NT][4];
                const auto clear = [&]() {
#pragma unroll
                    for (int t = 0; t < NT; ++t)
#pragma unroll
                        for (int e = 0; e < 8; ++e) c[t][e >> 2][e & 3] = 0.f;
                };
                // every eight units (128 points: below 2^24) the exact sums move to 64-bit integers
                const auto flush = [&]() {
#pragma unroll
                    for (int t = 0; t < NT; ++t)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            sum[t][e] += __float2int_rn(c[t][0][e]) + __float2int_rn(c[t][1][e]);
                };
                clear();
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e) sum[t][e] = 0;
                const auto value = [&](int u) {
                    const int p = 16 * u + (lane & 15);
                    return p < n ? (lane < 16 ? us[p] : zb[p0 + p]) : T(0);
                };
                int held = 0, at = 0;
                stage_load(stage[0], Q + 16 * wid, ld, j);
                T next = value(wid);
                for (int u = wid; u < nunit; u += kSW, at ^= 1) {
                    const T val = next;
                    if (u + kSW < nunit) {
                        stage_load(stage[at ^ 1], Q + 16 * (u + kSW), ld, j);
                        next = value(u + kSW);
                    } else {
                        asm volatile("cp.async.commit_group;" ::: "memory");
                    }
                    const unsigned long long x = last && lane >= 16 ? kBias : fix62(val, lane < 16 ? eu : ez);
                    put_digits(tu + (lane < 16 ? 7 : 22) * kUP + (lane & 15) * 2, kUP, x);
                    unsigned long long* S = reinterpret_cast<unsigned long long*>(stage[at]);
                    if (lane < 16) S[j * kSP + lane] = x;
                    stage_wait<1>();
                    dot_unit<NT, false>(c, stage[at], kSP, 0, j, 0, ta);
                    __syncwarp();
                    if (++held == 8) {
                        flush();
                        clear();
                        held = 0;
                    }
                }
                flush();
                // the warp's sums into its (now free) stages: row, u or z, digit column
                long long* o = reinterpret_cast<long long*>(stage[0]);
                const int n0 = 2 * tg, n1 = 2 * tg + 1;
                const int r0 = (n0 & 3) * 2 + (n0 >> 2), r1 = (n1 & 3) * 2 + (n1 >> 2);
                stage_wait<0>();
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    o[(8 * t + r0) * 16 + g] = sum[t][0];
                    o[(8 * t + r1) * 16 + g] = sum[t][1];
                    o[(8 * t + r0) * 16 + 8 + g] = sum[t][2];
                    o[(8 * t + r1) * 16 + 8 + g] = sum[t][3];
                }
            };
            if (j < 8) dots(std::integral_constant<int, 1>{});
            else if (j < 16) dots(std::integral_constant<int, 2>{});
            else if (j < 24) dots(std::integral_constant<int, 3>{});
            else dots(std::integral_constant<int, 4>{});
        }
        __syncthreads();
        const int egz = egu + eA;
        if (wid < 8) {
            const int out = threadIdx.x >> 2, cp = threadIdx.x & 3;
            const int row = out >> 1, v = out & 1;
            long long s = 0;
            const bool on = row <= j && !(last && v);
            if (on) {
                long long a = 0, b = 0;
                for (int w = 0; w < nact; ++w) {
                    const longlong2 x = *reinterpret_cast<const longlong2*>(sm + Y.stage + (size_t)(2 * w) * kSStage +
                                                                            (row * 16 + v * 8 + 2 * cp) * 8);
                    a += x.x;
                    b += x.y;
                }
                s = (cp & 1) ? (a << 8) + b : (a << 24) + (b << 16);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            const long long lo = __shfl_xor_sync(0xffffffffu, s, 2);
            if (cp == 0 && on) {
                int sh = (v ? egz - ez : egu - eu) + (row == j ? egu - eu : 0);
                sh = max(0, min(sh, 126));
                const __int128 W = ((((__int128)s << 32) + lo) << 16) >> sh;
                s_bp[out] = make_longlong2((long long)(W >> 48), (long long)((unsigned long long)W & 0xffffffffffffull));
            }
        }
        __syncthreads();
        if (!solo) {
            unsigned long long* mine = accj + (bid & (kCopies - 1)) * 128;
            const int out = threadIdx.x >> 1;
            if (threadIdx.x < 4 * (j + 1) && nact > 0 && !(last && (out & 1)))
                atomicAdd(&mine[threadIdx.x], reinterpret_cast<unsigned long long*>(s_bp)[threadIdx.x]);
        }
        const bool bad = eu == 0x7ff || ez == 0x7ff;
        if (threadIdx.x == 0 && bad && !solo) atomicMax(&slot[(j & 1) * 2 + 1], 1u);
        if (!meet()) return;

        // ---- the sums and the scalars; z at the ghosts ----------------------------
        if (wid < 2) {
            const int v = wid;
            const bool on = lane <= j && !(last && v);
            double val = 0.0;
            if (on) {
                long long hi = 0, lo = 0;
                if (solo) {
                    hi = s_bp[2 * lane + v].x;
                    lo = s_bp[2 * lane + v].y;
                } else {
                    longlong2 x[kCopies];
#pragma unroll
                    for (int q = 0; q < kCopies; ++q)
                        x[q] = __ldcg(reinterpret_cast<const longlong2*>(accj + q * 128) + 2 * lane + v);
#pragma unroll
                    for (int q = 0; q < kCopies; ++q) {
                        hi += x[q].x;
                        lo += x[q].y;
                    }
                }
                const double d = fma((double)hi, 281474976710656.0, (double)lo);
                const int Eu = egu - 1022, Ez = egz - 1022;
                val = scale2(d, lane < j ? (v ? Ez : Eu) - 83 : (v ? Eu + Ez : 2 * Eu) - 84);
            }
            s_v[v][lane] = val;
            const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)(lane < j ? expo(val) : 0));
            if (lane == 0) s_e[4 + v] = e;
            const unsigned long long x = lane < j ? fix62(val, e) : kBias;
            put_digits(tile + (v ? kTileT : kTileS) * kTP + tile_col<false>(lane) * 2, kTP, x);
            if (v == 0) {
                // s below 2^-12 |u|: six of its digit columns are enough; else a second tile with s in t's place
                const int euu = __shfl_sync(0xffffffffu, expo(val), j & 31) - 1023;
                const bool small = j == 0 || e == 0 || euu - 2 * (e - 1022) >= 24;
                if (!small) put_digits(tile2 + kTileT * kTP + tile_col<false>(lane) * 2, kTP, x);
                if (lane == 0) s_int[1] = small;
            }
            asm volatile("bar.arrive 1, 96;" ::: "memory");
        } else if (wid == 8) {
            if (lane < 3) s_e[lane] = 0;
            asm volatile("bar.sync 1, 96;" ::: "memory");
            const bool in = lane < j;
            const double si = in ? s_v[0][lane] : 0.0, ti = in ? s_v[1][lane] : 0.0;
            const double uu = s_v[0][j & 31], uz = s_v[1][j & 31];
            const int nan = solo ? (int)bad : (int)__ldcg(&slot[(j & 1) * 2 + 1]);
            double ss = si * si, st = si * ti;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
                st += __shfl_xor_sync(0xffffffffu, st, o);
            }
            double q2 = uu - ss;
            if (__double_as_longlong(q2) < 0) q2 = 0.0;
            const double hinv = rsqrt_fast(q2);
            const double uzs = uz - st;
            int stop = nan == 0 && finite_bits(uzs) && finite_bits(uu) && finite_bits(q2) && (j == 0 || s_e[7] != 0x7ff)
                           ? 0 : 2;
            if (stop == 0) {
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
            if (lane == 0) {
                s_int[0] = stop;
                s_sc[0] = q2;
                s_sc[1] = hinv;
                s_sc[2] = uzs * hinv;
                s_S.hinv = hinv;
                s_S.qz = uzs * hinv;
                split2(s_S.hinv, s_S.hh, s_S.hl);
                split2(s_S.qz, s_S.qh, s_S.ql);
            }
        }
        if (!last) {   // sixteen ghosts at a time, taken in turn as warps come free
            for (;;) {
                int q = 0;
                if (lane == 0) q = atomicAdd(&s_next, 16);
                q = __shfl_sync(0xffffffffu, q, 0);
                if (q >= ng) break;
                long long tt[4];
                int rl[4];
                const double* const rw[4] = {nullptr, nullptr, nullptr, nullptr};
                const int* const ri[4] = {nullptr, nullptr, nullptr, nullptr};
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int gi = q + 4 * x + (lane >> 3);
                    tt[x] = t0 + gi;
                    rl[x] = gi < ng ? A.row_len[t0 + gi] : 0;
                }
                double v[4];
                ghost_rows<T, 4>(A, zb, tt, rl, lane & 7, rw, ri, v);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int gi = q + 4 * x + (lane >> 3);
                    if ((lane & 7) == 0 && gi < ng) rz[gi] = v[x];
                }
            }
        }
        __syncthreads();
        const int stop = s_int[0];
        if (threadIdx.x == 0) {
            s_next = 0;
            if (j == 0) {
                const double b = scale2(s_sc[0] > 0.0 && finite_bits(s_sc[0]) ? s_sc[0] * s_sc[1] : s_sc[0], be);
                s_sc[3] = b;
                if (lead) *A.beta = b;
            }
        }
        if (stop != 0 || last) {
            if (stop == 2 && lead) atomicOr(A.flags, 1);
            k = j;
            break;
        }
        // ---- the updates: q_j and the next u, 32 columns a warp and turn ------------
        {
            const StepScalars S = s_S;
            const bool small = s_int[1] != 0;
            const int et = s_e[5] - 1022, es = s_e[4] - 1022;
            const int npg = (n + 31) / 32, ngg = (ng + 31) / 32;
            // a group's 32 columns in two stages, each refilled for the next group once read
            const auto fill = [&](int x, int half) {
                if (j > 0 && x < npg + ngg) {
                    const bool gh = x >= npg;
                    stage_load(stage[half], (gh ? G + (x - npg) * 32 : Q + x * 32) + 16 * half, gh ? ldg : ld, j);
                } else {
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
            };
            fill(wid, 0);
            fill(wid, 1);
            // u, z and the lattice position of a column, fetched one turn ahead
            T un_u = T(0), un_z = T(0);
            uint32_t un_m = 0;
            const auto fetch = [&](int x) {
                const int c = (x < npg ? x : x - npg) * 32 + lane;
                if (x < npg && c < n) {
                    un_u = us[c];
                    un_z = zb[p0 + c];
                    un_m = meta[c];
                } else if (x >= npg && c < ng) {
                    un_m = (uint32_t)A.glist[t0 + c] | ((uint32_t)gsx[c] << 24);
                }
            };
            fetch(wid);
            for (int x = wid; x < npg + ngg; x += kSW) {
                const bool gh = x >= npg;
                const int c = (gh ? x - npg : x) * 32 + lane;
                const T u0 = un_u, z0 = un_z;
                const uint32_t mw = un_m;
                fetch(x + kSW);
                longlong2 v = make_longlong2(0, 0);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    stage_wait<1>();
                    if (j > 0) {
                        longlong2 w = update_sums<2, false>(stage[half], kSP, 0, j, 0, tile, xch);
                        if (!small) w.y = update_sums<2, false>(stage[half], kSP, 0, j, 0, tile2, xch).x;
                        if (half == 0 || lane >= 16) v = w;
                    }
                    __syncwarp();
                    fill(x + kSW, half);
                }
                int e = 0;
                if (gh ? c < ng : c < n) {
                    T qj, un;
                    int pos, gs = 0;
                    if (gh) {
                        gs = (int)(mw >> 24);
                        double q1, u1;
                        next_values(ug[c], rz[c], v.y, es - 60 + gs, v.x, et - 60 + gs, S, q1, u1);
                        qj = (T)q1;
                        if (sizeof(T) == 4) u1 = fma(q1 - dbl(qj), S.qz * S.hinv, u1);   // with the rounded q_j
                        un = (T)u1;
                        ug[c] = dbl(un);
                        pos = meta_pos(mw);
                    } else {
                        const T u = u0, z = z0;
                        if constexpr (sizeof(T) == 4) {
                            next_values_f(u, z, scaled_float(v.y, es - 60), scaled_float(v.x, et - 60), S, qj, un);
                        } else {
                            next_values(u, z, v.y, es - 60, v.x, et - 60, S, qj, un);
                        }
                        us[c] = un;
                        pos = meta_pos(mw);
                    }
                    Lq[pos] = un;
                    e = expo(un);
                    (gh ? G + (size_t)j * ldg : Q + (size_t)j * ld)[c] = fix62(qj, 1023 + gs);
                }
                e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
                if (lane == 0) {
                    if (!gh) atomicMax(&s_e[0], e);
                    atomicMax(&s_e[1], e);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && !solo) atomicMax(&slot[((j + 1) & 1) * 2], (unsigned)s_e[1]);
        if (!meet()) return;
    }
    // as in krylov_mma_body
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
        return;
    }
    const double beta = s_sc[3];
    const bool fine = phi1_mma(sH, k, A.dt, s_y, s_part, s_x, s_int);
    if (lead && !fine) atomicOr(A.flags, 1);
    if (bid == 0)
        for (int t = threadIdx.x; t < m; t += kMT) A.y[t] = s_y[t];
    if (wid == 0) {
        const double cv = lane < k ? A.dt * beta * s_y[lane] : 0.0;
        const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)expo(cv));
        put_digits(tile + kTileT * kTP + tile_col<false>(lane) * 2, kTP, lane < k ? fix62(cv, e) : kBias);
        if (lane == 0) s_e[5] = e;
    }
    __syncthreads();
    {
        T* om = (T*)A.omega + p0;
        T* Lo = (T*)A.L;
        const double sc = s_e[5] == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : pow2d(s_e[5] - 1022 - 60);
        const int npu = (n + 15) / 16;
        stage_wait<0>();
        if (wid < npu) stage_load(stage[0], Q + 16 * wid, ld, k);
        int at = 0;
        for (int x = wid; x < npu; x += kSW, at ^= 1) {
            const int c = x * 16 + lane;
            if (x + kSW < npu) stage_load(stage[at ^ 1], Q + 16 * (x + kSW), ld, k);
            else asm volatile("cp.async.commit_group;" ::: "memory");
            stage_wait<1>();
            const longlong2 v = update_sums<2, false>(stage[at], kSP, 0, k, 0, tile, xch);
            if (lane < 16 && c < n) {
                const T w = (T)fma((double)v.x, sc, dbl(om[c]));
                om[c] = w;
                Lo[meta_pos(meta[c])] = w;
            }
            __syncwarp();
        }
        stage_wait<0>();
    }
    if (lead) *A.kstop = k;
}

// Block b works on items off[b] .. off[b + 1] - 1 in turn: (problem, its
// block's index in it, its block count).
template <typename T, int P>
__global__ void __launch_bounds__(kMT, 1) k_krylov_stream(const KrylovStepArgs* __restrict__ args,
                                                          const int* __restrict__ items, const int* __restrict__ off) {
    extern __shared__ __align__(16) char k_sm[];
    __shared__ KrylovStepArgs A;
    for (int i = off[blockIdx.x]; i < off[blockIdx.x + 1]; ++i) {
        __syncthreads();
        const int* src = reinterpret_cast<const int*>(args + items[3 * i]);
        for (int t = threadIdx.x; t < (int)(sizeof(KrylovStepArgs) / 4); t += kMT) reinterpret_cast<int*>(&A)[t] = src[t];
        __syncthreads();
        krylov_stream_body<T, P>(A, items[3 * i + 1], items[3 * i + 2], k_sm);
    }
}

// One problem on the whole grid.
template <typename T, int P>
__global__ void __launch_bounds__(kMT, 1) k_krylov_stream_one(KrylovStepArgs A) {
    extern __shared__ __align__(16) char k_sm[];
    krylov_stream_body<T, P>(A, blockIdx.x, gridDim.x, k_sm);
}

}  // namespace

template <typename T, int P>
const void* KrylovKernels<T, P>::stream_kernel() {
    return (const void*)k_krylov_stream<T, P>;
}
template <typename T, int P>
const void* KrylovKernels<T, P>::stream_one_kernel() {
    return (const void*)k_krylov_stream_one<T, P>;
}
template <typename T, int P>
size_t KrylovKernels<T, P>::stream_bytes() {
    return stream_layout().bytes;
}
template <typename T, int P>
cudaError_t KrylovKernels<T, P>::launch(const KrylovStepArgs& args, const KrylovPlan& plan, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = plan.cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3(plan.blocks);
    cfg.blockDim = dim3(kMT);
    cfg.dynamicSmemBytes = plan.form == 3 ? stream_bytes() : plan.smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = plan.cluster > 1 ? 2 : 1;
    KrylovStepArgs a = args;
    int ppb = plan.ppb, gpb = plan.gpb, nrc = plan.nrc;
    void* params[] = {&a, &ppb, &gpb, &nrc};
    return cudaLaunchKernelExC(&cfg, plan.form == 3 ? stream_one_kernel() : mma_kernel(plan.cluster, plan.form), params);
}

}  // namespace wrc
