// Host side of the Krylov-projected step (Sec. 2.1): shared-memory opt-in,
// co-resident capacity and thread-block clusters per device, the probe and
// check of cluster formation, the plans of the single-run and batched
// launches, dispatched by bulk type and DD order (the kernels are compiled
// per DD order in krylov_p2.cu, krylov_p3.cu and krylov_p4.cu from
// krylov_mma.cuh and krylov_stream.cuh).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "kernels.h"

namespace wrc {

namespace {

// Cluster formation check: launched with the attributes of the clustered
// Krylov kernel (cooperative, clusters of CL blocks, grid of one cluster),
// block 0 records how many blocks its cluster holds.  Reads no peer memory.
__global__ void k_cluster_probe(int* out) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *out = (int)cooperative_groups::this_cluster().num_blocks();
}

// Calls f with the KrylovKernels<T, P> of DD half-order P (2, 3 or 4).
template <typename T, typename F>
auto by_order(int P, F&& f) {
    if (P == 3) return f(KrylovKernels<T, 3>{});
    if (P == 4) return f(KrylovKernels<T, 4>{});
    return f(KrylovKernels<T, 2>{});
}
}  // namespace

namespace {
constexpr int kMaxDevices = 64;
// Per device, bulk type and DD order: co-resident blocks (one per SM), in
// clusters of four (0: not formed), and the dynamic shared memory a block of
// the single-run kernel may take.
struct MmaCaps {
    bool ready = false;
    int cap1 = 0, cap4 = 0;
    size_t bytes = 0;
};
struct DeviceClusters {
    MmaCaps mma[2][kMaxP + 1];               // [fp32][P]
    bool probed = false;
    bool formed4 = false;                    // clusters of four form on the launch path
    bool checked = false;                    // a clustered launch has been checked
};
DeviceClusters g_dev[kMaxDevices];
std::mutex g_caps_mutex;
// Test switch (environment variable WRC_KRYLOV_TEST_REFUSE=1, read once per
// process): the first, checked clustered launch on a device behaves as if
// its clusters were not formed, so that the fallback path can be tested on
// a launch path that does form them.
int g_test_refuse = -1;

// Launch the probe as one cluster of CL blocks with the Krylov kernel's
// attributes and report whether the cluster formed (1), did not (0), or the
// launch failed (-1).  Runs on a short-lived stream of its own.
int probe_cluster(int CL) {
    int* d = nullptr;
    cudaStream_t ps = nullptr;
    if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    int r = -1;
    if (cudaStreamCreateWithFlags(&ps, cudaStreamNonBlocking) == cudaSuccess &&
        cudaMemsetAsync(d, 0, sizeof(int), ps) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim.x = CL;
        at[1].val.clusterDim.y = 1;
        at[1].val.clusterDim.z = 1;
        cfg.gridDim = dim3(CL);
        cfg.blockDim = dim3(32);
        cfg.stream = ps;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        int h = 0;
        if (cudaLaunchKernelEx(&cfg, k_cluster_probe, d) == cudaSuccess &&
            cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, ps) == cudaSuccess &&
            cudaStreamSynchronize(ps) == cudaSuccess) {
            note_launch();
            r = h == CL ? 1 : 0;
        }
    }
    if (r < 0) cudaGetLastError();
    if (ps) cudaStreamDestroy(ps);
    cudaFree(d);
    return r;
}

int clamp_order(int P) { return P == 3 || P == 4 ? P : 2; }

MmaCaps caps_of(int dev, bool fp32, int P) {
    std::lock_guard<std::mutex> lk(g_caps_mutex);
    return dev >= 0 && dev < kMaxDevices ? g_dev[dev].mma[fp32][clamp_order(P)] : MmaCaps{};
}

bool cluster_checked(int dev) {
    std::lock_guard<std::mutex> lk(g_caps_mutex);
    return dev >= 0 && dev < kMaxDevices && g_dev[dev].checked;
}
}  // namespace

namespace {
// Shared-memory opt-in and co-resident capacity of the tensor-core kernels.
template <typename K>
int mma_init(K kern, int dev, int sms, bool clusters, MmaCaps& c) {
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    size_t room = 0;
    for (int q = 0; q < 7; ++q) {   // the three forms, the narrow one in clusters, the velocity-Exner ones
        cudaFuncAttributes fa;
        const void* f = q < 4 ? kern.mma_kernel(q == 3 ? 4 : 1, q == 3 ? 0 : q) : kern.ex_kernel(q - 4);
        if (!f) continue;
        if (cudaFuncGetAttributes(&fa, f) != cudaSuccess) return -1;
        const size_t dyn = (size_t)optin - fa.sharedSizeBytes;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) != cudaSuccess) return -1;
        room = room == 0 || dyn < room ? dyn : room;
    }
    c.bytes = room;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern.mma_kernel(1, 2), kern.mma_threads(), room) !=
        cudaSuccess)
        return -1;
    c.cap1 = per > 0 ? sms : 0;
    c.cap4 = 0;
    if (clusters) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 4;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeCooperative;
        at[1].val.cooperative = 1;
        cfg.gridDim = dim3(4);
        cfg.blockDim = dim3(kern.mma_threads());
        cfg.dynamicSmemBytes = room;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, kern.mma_kernel(4, 0), &cfg) == cudaSuccess) c.cap4 = 4 * nc;
        else cudaGetLastError();
    }
    const void* f = kern.stream_kernel();
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kern.stream_bytes()) != cudaSuccess ||
        cudaFuncSetAttribute(kern.stream_one_kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kern.stream_bytes()) != cudaSuccess)
        return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, kern.mma_threads(), kern.stream_bytes()) != cudaSuccess ||
        per < 1)
        return -1;
    c.ready = true;
    return 0;
}
}  // namespace

int krylov_cluster_max() {
    // WRC_KRYLOV_CLUSTER = 1 or 2 keeps launches unclustered (clusters are of four blocks)
    int cmax = 4;
    if (const char* ev = getenv("WRC_KRYLOV_CLUSTER")) cmax = atoi(ev) >= 4 ? 4 : (atoi(ev) >= 2 ? 2 : 1);
    return cmax;
}

int krylov_step_init(int dev, bool fp32, int P, int* max_blocks) {
    if (dev < 0 || dev >= kMaxDevices) return -1;
    P = clamp_order(P);
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return -2;
    *max_blocks = sms;
    std::lock_guard<std::mutex> lk(g_caps_mutex);
    if (g_test_refuse < 0) {
        const char* ev = getenv("WRC_KRYLOV_TEST_REFUSE");
        g_test_refuse = (ev && atoi(ev) == 1) ? 1 : 0;
    }
    DeviceClusters& D = g_dev[dev];
    if (!D.probed) {
        // a launch path that does not form clusters (some profilers replay a
        // cooperative launch without them): launch without
        D.formed4 = probe_cluster(4) == 1;
        D.probed = true;
    }
    MmaCaps& c = D.mma[fp32][P];
    if (c.ready) return 0;
    const int r = fp32 ? by_order<float>(P, [&](auto K) { return mma_init(K, dev, sms, D.formed4, c); })
                       : by_order<double>(P, [&](auto K) { return mma_init(K, dev, sms, D.formed4, c); });
    return r != 0 ? -3 : 0;
}

// Launch rule.  The kernel with its table in shared memory takes every problem
// that fits one block per SM; beyond, the streaming one.  Points per
// block: spread over all SMs, but at least 32, and 48 for order-4 runs of up
// to 3072 points.  A block has its SM to itself, so runs stepped at the same
// time, each on a stream of its own, share the device only where their blocks
// leave SMs free.  Up to 3072 points 48 a block cost a run alone nothing in
// FP64, 2% of a step in the mixed mode, and let two work side by side (128^2, 2.8K
// points, us a step alone / each of four / each of eight at once: 603 / 166 /
// 90 with the FP64 dots, 337 / 213 / 212 from 32 points on, 335 / 115 / 112
// so, 345 / 100 / 82 from 64).  Above, 32 points make more blocks than
// clusters are formed for, 3-4% faster than 48 in clusters; at higher orders
// longer ghost rows queue for a block's few warps (64 points: 8-10% slower
// at 3-4K points).  Larger runs keep all SMs, as half of them cost a run
// alone 3-10% (256^2, 9.2K points: 754 / 241 / 189, 445 / 294 / 297, on half
// the SMs 472 / 181 / 180): alone they take 0.5 to 0.7 of the time with the
// FP64 dots, four or eight at once up to 1.9 times it; an ensemble's one
// launch for all its members is the form for many.
// The narrow form up to 128 columns (points and ghosts) a block, digits as
// halves while they fit (~370 columns at m = 30), else 64-bit integers
// (~720): halves and integers measure the same at 220 columns (393 and 394
// us), the integers being the only form beyond.  Clusters of four blocks,
// which add their sums in distributed shared memory before the grid's, for
// launches of at most 96 blocks: above, unclustered launches are faster (142
// blocks: 317 us against 333) and use all SMs.
// Measured on GB300, one launch, against the kernel with FP64 dots that was
// used before: 128^2 pair, m = 20, 2.8K points 352 -> 209 us; m = 30: 256^2
// mixed, 10.9K points 553 -> 337; 1024^2, 17.0K points 484 -> 322 and 72.6K
// 1065 -> 634; 4096^2 mixed, 30.0K points 754 -> 396; order 6, 7.4K points
// 624 -> 391.
KrylovPlan krylov_plan(long long n, long long ng, int m, bool fp32, int P, int dev, int cmax) {
    KrylovPlan K;
    const MmaCaps c = caps_of(dev, fp32, P);
    const auto up16 = [](long long x) { return (int)((x + 15) / 16 * 16); };
    {
        int ppb = up16((n + c.cap1 - 1) / std::max(1, c.cap1));
        ppb = std::max(ppb, P == 2 && n <= 3072 ? 48 : 32);
        int nb = (int)((n + ppb - 1) / ppb);
        nb = nb < 1 ? 1 : nb;
        int cl = 1;
        const int b4 = (nb + 3) / 4 * 4;
        if (cmax >= 4 && b4 <= 96 && b4 <= c.cap4) {
            cl = 4;
            nb = b4;
        }
        int gpb = up16((ng + nb - 1) / nb), form = 0;
        const auto bytes = [&](int nrc) {
            return fp32 ? by_order<float>(P, [&](auto kk) { return kk.mma_bytes(form, m, ppb, gpb, nrc); })
                        : by_order<double>(P, [&](auto kk) { return kk.mma_bytes(form, m, ppb, gpb, nrc); });
        };
        if (ppb + gpb > 128) {
            form = 1;
            if (bytes(-1) > c.bytes) form = 2;
            cl = 1;                    // clusters in the narrow form only
        }
        size_t need = bytes(-1);
        if (need <= c.bytes && ppb <= 1024) {
            K.form = form;
            K.nrc = -1;
            if (bytes(0) <= c.bytes) {
                // the ghosts' interpolation rows in shared memory too, as many as fit
                const size_t per = bytes(2) - bytes(0);
                K.nrc = (int)((c.bytes - bytes(0)) / per * 2);
                if (K.nrc > gpb) K.nrc = gpb;
                need = bytes(K.nrc);
            }
            K.blocks = nb;
            K.cluster = cl;
            K.ppb = ppb;
            K.gpb = gpb;
            K.smem = need;
            return K;
        }
    }
    K.form = 3;
    K.blocks = std::max(1, c.cap1);
    return K;
}

// The velocity-Exner step takes the same kernel while its 3 n entries fit
// (up to ~30K points at m = 30): with two barriers per Arnoldi step instead of
// the four and FP64 dots of k_ex_krylov, which runs what does not fit, a step
// of 8.6K points at 1024^2, m = 30, takes 486 us instead of 1318.
KrylovPlan krylov_ex_plan(long long n, long long ng, int m, int P, int dev) {
    return krylov_plan(3 * n, 3 * ng, m, false, P, dev, 1);
}

cudaError_t launch_krylov_ex(const KrylovStepArgs& args, const ExArgs& x, const KrylovPlan& plan, cudaStream_t s) {
    KrylovStepArgs a = args;
    ExArgs xa = x;
    int ppb = plan.ppb, gpb = plan.gpb, nrc = plan.nrc;
    void* params[] = {&a, &xa, &ppb, &gpb, &nrc};
    const cudaError_t e = by_order<double>(clamp_order(args.g.P), [&](auto K) {
        return cudaLaunchCooperativeKernel(K.ex_kernel(plan.form), dim3(plan.blocks), dim3(K.mma_threads()), params,
                                           plan.smem, s);
    });
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

void krylov_clusters_unformed(int dev) {
    if (dev < 0 || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lk(g_caps_mutex);
    DeviceClusters& D = g_dev[dev];
    D.checked = true;
    D.formed4 = false;
    for (auto& byp : D.mma)
        for (auto& cc : byp) cc.cap4 = 0;
}

// The first clustered launch on a device is checked: the stream is
// synchronised and, if the kernel found its clusters not formed (it then
// runs as the unclustered kernel and raises bit 4 of the error word),
// clusters are switched off for the device.  Later launches are not
// synchronised; a later launch without its clusters (e.g. under a profiler)
// runs unclustered all the same and is seen at the step's host
// synchronisation.
template <typename T>
cudaError_t launch_krylov_step(const KrylovStepArgs& args, const KrylovPlan& plan, cudaStream_t s, int dev) {
    const int P = clamp_order(args.g.P);
    const bool check = plan.cluster > 1 && !cluster_checked(dev);
    KrylovStepArgs a = args;
    a.refuse = (check && g_test_refuse == 1) ? 1 : 0;
    cudaError_t e = by_order<T>(P, [&](auto K) { return K.launch(a, plan, s); });
    if (e != cudaSuccess) return e;
    note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess || !check) return e;
    int err = 0;
    e = cudaMemcpyAsync(&err, args.err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (err & 16) {
        krylov_clusters_unformed(dev);
        if (err == 16) e = cudaMemsetAsync(args.err, 0, sizeof(int), s);   // informational only
    } else {
        std::lock_guard<std::mutex> lk(g_caps_mutex);
        g_dev[dev].checked = true;
    }
    return e;
}

template cudaError_t launch_krylov_step<double>(const KrylovStepArgs&, const KrylovPlan&, cudaStream_t, int);
template cudaError_t launch_krylov_step<float>(const KrylovStepArgs&, const KrylovPlan&, cudaStream_t, int);

size_t krylov_partials_doubles() { return 2 * 8 * 128 + 16; }   // krylov_mma.cuh: sums and exponent slots

int krylov_batch_max_runs(int pt) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    return sms * (pt == 64 ? 8 : 4);
}

template <typename T>
cudaError_t launch_krylov_batch(const KrylovStepArgs* d_args, const int* d_items, const int* d_off, int blocks, int P,
                                cudaStream_t s) {
    void* params[] = {(void*)&d_args, (void*)&d_items, (void*)&d_off};
    const cudaError_t e = by_order<T>(P, [&](auto K) {
        return cudaLaunchCooperativeKernel(K.stream_kernel(), dim3(blocks), dim3(K.mma_threads()), params,
                                           K.stream_bytes(), s);
    });
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

template cudaError_t launch_krylov_batch<double>(const KrylovStepArgs*, const int*, const int*, int, int, cudaStream_t);
template cudaError_t launch_krylov_batch<float>(const KrylovStepArgs*, const int*, const int*, int, int, cudaStream_t);

}  // namespace wrc
