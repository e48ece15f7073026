// Kernels of the exponential Rosenbrock-Euler step (Sec. 1 and 2.1: the
// Krylov projection with the Jacobian of the discrete right-hand side,
//   omega^{n+1} = omega^n + dt phi_1(dt J_n) F(omega^n),
//   J_n q = A_n q - U[q] D_x omega^n - V[q] D_y omega^n,
// U[q], V[q] the velocity of q's own streamfunction: a reconstruction and a
// Poisson solve per Krylov vector, so the Arnoldi process runs as a sequence
// of launches driven by the host (api.cu) rather than inside the persistent
// kernel.  Gram-Schmidt is applied twice (classical), with FP64 inner
// products accumulated per block and added in a fixed order, each pass one
// launch with the operator or the update before it and the bookkeeping after
// it (k_rb_pass); the Krylov
// dimension used (a happy breakdown stops it) lives on the device, and every
// kernel of a later Arnoldi step returns at once.  phi_1 and the update as in
// the persistent kernel.
#include <algorithm>

#include "krylov_impl.cuh"

namespace wrc {

namespace {

constexpr int kRbThreads = 256;
constexpr int kRbPts = 128;            // threads, and points of a turn, of a k_rb_pass block
constexpr int kRbMaxVec = kNV + 1;   // basis vectors of a pass, and w itself
static_assert(kRbMaxVec == kRbPartWidth, "partial-sum rows");

// D_x omega, D_y omega at the active points (the operator's first
// derivatives at the stencil levels, ghost values from the lattice F).
template <typename T, int P>
__global__ void k_rb_grad(const T* __restrict__ F, const uint32_t* __restrict__ meta, int n, T* __restrict__ dwx,
                          T* __restrict__ dwy, Geom g, T c1J, T c2J) {
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < n; a += gridDim.x * blockDim.x) {
        // -U Dx - V Dy with (U, V) = (-1, 0) and (0, -1), no diffusion or damping
        dwx[a] = apply_point<T, false, P>(F, meta[a], T(-1), T(0), T(0), T(0), g, c1J, c2J);
        dwy[a] = apply_point<T, false, P>(F, meta[a], T(0), T(-1), T(0), T(0), g, c1J, c2J);
    }
}

// What precedes a reduction of step j, the reduction, and its bookkeeping:
//   mode 0 (first pass): w = A_n q_j - U[q_j] D_x omega - V[q_j] D_y omega
//          (Lq holds R(q_j) with its ghosts); c = Q^T w -> H[:, j] = c,
//          coef = c, and |A q_j|^2 = |w|^2 kept for the breakdown test;
//   mode 1 (second pass): w -= Q coef; c = Q^T w -> H[:, j] += c, coef = c;
//   mode 2 (norm): w -= Q coef; h = |w|, H[j + 1][j] = h; a happy breakdown
//          (h <= tol |A q_j|) or a non-finite h stops the process at
//          k = j + 1 (non-finite also raises flags bit 0), else scale = 1/h;
//   mode 3 (beta): beta = |w| (w = b); beta = 0 stops it at k = 0, else
//          scale = 1/beta.
// sc: [0] scale, [1] |A q_j|^2.
//
// Bound by FP64 issue (one warp instruction per ~65 cycles and SM
// sub-partition): a block takes 128 points, its points' products with vector
// v go to warp v mod 4, four to a lane, and the lanes' sums of eight vectors
// are joined in nine exchanges instead of 8 x 5.  The block that finishes
// last adds the blocks' sums in block order.  One launch for what took three
// (the operator or update, the dots with every vector's 32-lane sums, one
// block's serial sums): 16.9K points of 512^2, m = 31, a vector's launches
// beside its reconstruction and solve 100 -> 20 us, the 31 vectors 4.97 ->
// 2.50 ms.
template <typename T, int P>
__global__ void __launch_bounds__(kRbPts) k_rb_pass(RbArgs A, int mode, int j) {
    pdl_wait();
    if (mode != 3 && j >= *(const volatile int*)A.kstop) return;
    __shared__ double s_w[kRbPts];
    __shared__ double s_red[kRbPts / 32][32];
    __shared__ T s_c[kNV];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, n = A.n;
    const int nv = mode == 3 ? 0 : j + 1, ndot = mode <= 1 ? nv : 0;
    const T* basis = (const T*)A.basis;
    T* w = (T*)A.w;
    if (mode == 1 || mode == 2)
        for (int t = tid; t < nv; t += kRbPts) s_c[t] = (T)A.coef[t];
    __syncthreads();
    double acc[8], nrm = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.0;
    for (int base = blockIdx.x * kRbPts; base < n; base += gridDim.x * kRbPts) {
        const int i = base + tid;
        T x = T(0);
        if (i < n) {
            if (mode == 0) {
                x = apply_point<T, false, P>((const T*)A.Lq, A.meta[i], ((const T*)A.Ua)[i], ((const T*)A.Va)[i],
                                             (T)A.nu, (T)A.r, A.g, (T)A.c1J, (T)A.c2J) -
                    ((const T*)A.Uq)[i] * ((const T*)A.dwx)[i] - ((const T*)A.Vq)[i] * ((const T*)A.dwy)[i];
                w[i] = x;
            } else {
                x = w[i];
                if (mode != 3) {
                    T p[4] = {T(0), T(0), T(0), T(0)};
                    for (int v = 0; v < nv; v += 8) {
                        T b[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) b[u] = v + u < nv ? basis[(size_t)(v + u) * A.ld + i] : T(0);
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (v + u < nv) p[u & 3] += b[u] * s_c[v + u];
                    }
                    x -= (p[0] + p[1]) + (p[2] + p[3]);
                    w[i] = x;
                }
            }
        }
        const double xd = (double)x;
        if (mode != 1) nrm += xd * xd;
        if (mode <= 1) {
            s_w[tid] = xd;
            T b[8][4];
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int v = wid + 4 * q, c = base + 32 * u + lane;
                    b[q][u] = v < ndot && c < n ? basis[(size_t)v * A.ld + c] : T(0);
                }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (wid + 4 * q < ndot)
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[q] += (double)b[q][u] * s_w[32 * u + lane];
            __syncthreads();
        }
    }
    double* part = A.part + (size_t)blockIdx.x * kRbMaxVec;
    if (mode <= 1) {
        // lane bits 4, 3, 2 choose the vector, the other lanes are added
        double r4[4], r2[2], r1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool h = lane & 16;
            const double send = h ? acc[q] : acc[q + 4];
            r4[q] = (h ? acc[q + 4] : acc[q]) + __shfl_xor_sync(0xffffffffu, send, 16);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const bool h = lane & 8;
            const double send = h ? r4[q] : r4[q + 2];
            r2[q] = (h ? r4[q + 2] : r4[q]) + __shfl_xor_sync(0xffffffffu, send, 8);
        }
        {
            const bool h = lane & 4;
            const double send = h ? r2[0] : r2[1];
            r1 = (h ? r2[1] : r2[0]) + __shfl_xor_sync(0xffffffffu, send, 4);
        }
        r1 += __shfl_xor_sync(0xffffffffu, r1, 2);
        r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
        const int v = wid + 4 * ((lane >> 2) & 4 | (lane >> 2) & 2 | (lane >> 2) & 1);
        if ((lane & 3) == 0 && v < ndot) part[v] = r1;
    }
    if (mode != 1) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        if (lane == 0) s_red[0][wid] = nrm;
        __syncthreads();
        if (tid == 0) part[kRbMaxVec - 1] = (s_red[0][0] + s_red[0][1]) + (s_red[0][2] + s_red[0][3]);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        s_last = atomicAdd(A.count, 1u) == gridDim.x - 1 ? 1 : 0;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) {
        pdl_trigger();
        return;
    }
    // the last block: sums over the blocks (warp q takes blocks q, q + 4, ..), then the bookkeeping
    const int nb = gridDim.x;
    double sum = 0.0;
    if (mode >= 2) {
        for (int b = tid; b < nb; b += kRbPts) sum += __ldcg(A.part + (size_t)b * kRbMaxVec + kRbMaxVec - 1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    } else if (lane < ndot || (mode == 0 && lane == ndot)) {
        const double* p = A.part + (lane < ndot ? lane : kRbMaxVec - 1);
        for (int b = wid; b < nb; b += 4 * 8) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = b + 4 * u < nb ? __ldcg(p + (size_t)(b + 4 * u) * kRbMaxVec) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (b + 4 * u < nb) sum += x[u];
        }
    }
    s_red[wid][lane] = sum;
    __syncthreads();
    if (wid == 0) {
        const double c = (s_red[0][lane] + s_red[1][lane]) + (s_red[2][lane] + s_red[3][lane]);
        if (lane < ndot) {
            A.coef[lane] = c;
            double* h = A.H + (size_t)lane * A.m + j;
            *h = mode == 0 ? c : *h + c;
        }
        if (mode == 0 && lane == ndot) A.sc[1] = c;
        if (mode >= 2 && lane == 0) {
            const double h = sqrt(c);
            if (mode == 3) {
                *A.beta = h;
                if (!(h > 0.0) || !isfinite(h)) {
                    if (!isfinite(h)) atomicOr(A.flags, 1);
                    *A.kstop = 0;
                    A.sc[0] = 0.0;
                } else {
                    *A.kstop = A.m;
                    A.sc[0] = 1.0 / h;
                }
            } else {
                A.H[(size_t)(j + 1) * A.m + j] = h;
                const double q = A.sc[1];
                const bool bad = !isfinite(h) || !isfinite(q);
                if (bad) atomicOr(A.flags, 1);
                if (bad || h <= A.tol * sqrt(q)) *A.kstop = j + 1;
                else A.sc[0] = 1.0 / h;
            }
        }
        if (lane == 0) *A.count = 0u;   // for the next launch
    }
    pdl_trigger();
}

// basis_{j + 1} = w * scale, also into the lattice Lq, unless the process
// stopped at step j.
template <typename T>
__global__ void k_rb_scale(RbArgs A, int j) {
    pdl_wait();
    if (j >= 0 && *(const volatile int*)A.kstop <= j + 1) return;   // stopped at or before step j
    const double s = A.sc[0];
    const T* w = (const T*)A.w;
    T* dst = (T*)A.basis + (size_t)(j + 1) * A.ld;
    T* Lq = (T*)A.Lq;
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < A.n; a += gridDim.x * blockDim.x) {
        const T x = (T)((double)w[a] * s);
        dst[a] = x;
        Lq[meta_pos(A.meta[a])] = x;
    }
    pdl_trigger();
}

// y = phi_1(dt H_k) e_1 (k = *kstop; zero for k = 0), by one block.
__global__ void __launch_bounds__(kPT) k_rb_phi1(const double* __restrict__ H, const int* __restrict__ kstop, int m,
                                                 double dt, double* __restrict__ y, int* __restrict__ flags) {
    __shared__ double s_part[kPT / 32][kNV + 1];
    __shared__ double s_x[kNV + 1];
    __shared__ int s_int[3];
    const int k = *kstop;
    if (k == 0) {
        for (int t = threadIdx.x; t < m; t += kPT) y[t] = 0.0;
        return;
    }
    phi1_block<kPT>(H, k, m, dt, y, flags, s_part, s_x, s_int);
}

// omega <- omega + dt beta V_k y at the active points (accumulated in FP64),
// also written into the lattice array L.
template <typename T>
__global__ void k_rb_combine(const T* __restrict__ basis, long long ld, const double* __restrict__ y,
                             const double* __restrict__ beta, double dt, const int* __restrict__ kstop,
                             T* __restrict__ omega, T* __restrict__ L, const uint32_t* __restrict__ meta, int n) {
    __shared__ double s_c[kNV];
    const int k = *kstop;
    for (int t = threadIdx.x; t < k; t += blockDim.x) s_c[t] = dt * (*beta) * y[t];
    __syncthreads();
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < n; a += gridDim.x * blockDim.x) {
        double inc = 0.0;
        for (int t = 0; t < k; ++t) inc += s_c[t] * (double)basis[(size_t)t * ld + a];
        const T x = (T)((double)omega[a] + inc);
        omega[a] = x;
        L[meta_pos(meta[a])] = x;
    }
}

int rb_blocks(long long n) {
    long long b = (n + kRbThreads - 1) / kRbThreads;
    if (b < 1) b = 1;
    if (b > kRbPartBlocks) b = kRbPartBlocks;
    return (int)b;
}

template <typename F>
void rb_by_order(int P, F&& f) {
    if (P == 3) f(std::integral_constant<int, 3>{});
    else if (P == 4) f(std::integral_constant<int, 4>{});
    else f(std::integral_constant<int, 2>{});
}

}  // namespace

template <typename T>
cudaError_t rb_gradient(const RbArgs& a, cudaStream_t s) {
    rb_by_order(a.g.P, [&](auto PC) {
        constexpr int P = decltype(PC)::value;
        k_rb_grad<T, P><<<rb_blocks(a.n), kRbThreads, 0, s>>>((const T*)a.L, a.meta, a.n, (T*)a.dwx, (T*)a.dwy, a.g,
                                                               (T)a.c1J, (T)a.c2J);
    });
    note_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t rb_pass(const RbArgs& a, int mode, int j, cudaStream_t s) {
    // the last block adds this many sums, one at a time: two blocks a SM beyond 39K points
    const int nb = std::max(1, std::min((a.n + kRbPts - 1) / kRbPts, 304));
    rb_by_order(a.g.P, [&](auto PC) {
        constexpr int P = decltype(PC)::value;
        launch_pdl(k_rb_pass<T, P>, nb, kRbPts, 0, s, a, mode, j);
    });
    note_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t rb_scale(const RbArgs& a, int j, cudaStream_t s) {
    launch_pdl(k_rb_scale<T>, rb_blocks(a.n), kRbThreads, 0, s, a, j);
    note_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t rb_finish(const RbArgs& a, cudaStream_t s) {
    k_rb_phi1<<<1, kPT, 0, s>>>(a.H, a.kstop, a.m, a.dt, a.y, a.flags);
    note_launch();
    k_rb_combine<T><<<rb_blocks(a.n), kRbThreads, 0, s>>>((const T*)a.basis, a.ld, a.y, a.beta, a.dt, a.kstop,
                                                          (T*)a.omega, (T*)a.L, a.meta, a.n);
    note_launch();
    return cudaGetLastError();
}

#define WRC_INST(T)                                                                   \
    template cudaError_t rb_gradient<T>(const RbArgs&, cudaStream_t);                 \
    template cudaError_t rb_pass<T>(const RbArgs&, int, int, cudaStream_t);           \
    template cudaError_t rb_scale<T>(const RbArgs&, int, cudaStream_t);               \
    template cudaError_t rb_finish<T>(const RbArgs&, cudaStream_t);
WRC_INST(double)
WRC_INST(float)
#undef WRC_INST

}  // namespace wrc
