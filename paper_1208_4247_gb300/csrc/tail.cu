// Persistent tail: the small levels of a V-cycle in one launch of one CTA.
//
// Levels l_tail .. L-1 (the ones with n <= the tail threshold) run entirely
// in shared memory: the CTA loads q of level l_tail (just restricted from the
// level above), runs the rest of the V-cycle -- smoothing, residual,
// full-weighting restriction, exact one-unknown solve (or red-black sweeps on
// a larger coarsest grid), prolongation, smoothing -- with __syncthreads
// between the steps, and writes u of level l_tail back.  It replaces about
// 15 launches per small level, each dominated by launch latency, with one
// launch.  No waits other than __syncthreads.  The arithmetic of every step
// is the level kernels' (level_kernels.cuh), node for node.
#include <algorithm>

#include "tail_steps.cuh"

namespace gmg {
namespace tail {
namespace {

constexpr int kMaxGridLevels = 12;  // grid tail
constexpr int kGridThreads = 512;

// Grid barrier: a monotonic arrival count (zeroed before the launch); the
// b-th barrier waits until b * gridDim.x CTAs have arrived.  Thread 0 of each
// CTA publishes the CTA's writes (fence after the CTA barrier), arrives and
// spins with a limit of kSpinCycles SM clocks; past it the barrier sets
// bar->fault and every later one returns at once, so the kernel always ends
// (the host then reports the fault).  The fence after the spin orders the
// CTA's later loads after the other CTAs' published writes.
struct GridBar {
    unsigned count;
    int fault;
};
constexpr long long kSpinCycles = 200000000LL;  // about 0.1 s
struct GridX {
    GridBar* bar;
    unsigned target = 0;
    __device__ int tid() const { return blockIdx.x * blockDim.x + threadIdx.x; }
    __device__ int nt() const { return gridDim.x * blockDim.x; }
    __device__ void sync() {
        __syncthreads();
        target += gridDim.x;
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&bar->count, 1u);
            volatile unsigned* c = &bar->count;
            volatile int* f = &bar->fault;
            const long long t0 = clock64();
            while (*c < target && *f == 0) {
                if (clock64() - t0 > kSpinCycles) {
                    *f = 1;
                    break;
                }
            }
            __threadfence();
        }
        __syncthreads();
    }
};

// The whole grid is one thread-block cluster: the hardware cluster barrier
// (release / acquire at cluster scope, which orders the CTAs' global
// memory accesses too) between the steps.  Every thread of every CTA
// reaches each barrier (the steps call sync() outside divergent code).
struct ClusterX {
    __device__ int tid() const { return blockIdx.x * blockDim.x + threadIdx.x; }
    __device__ int nt() const { return gridDim.x * blockDim.x; }
    __device__ void sync() {
        asm volatile(
            "barrier.cluster.arrive.release.aligned;\n\t"
            "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
};

// The V-cycle on levels with n = n_top, n_top/2, ..., n_top >> (levels-1).
template <int DIM, typename T>
__global__ void __launch_bounds__(1024) k_tail(T* __restrict__ u_top, const T* __restrict__ q_top,
                                               Lay top, int levels, Cycle cy, int exact0,
                                               int first_done) {
    const int n_top = top.n;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int off[kMaxLevels + 1];
    int total = 0;  // nodes of all levels
    for (int l = 0; l < levels; ++l) {
        if (threadIdx.x == 0) off[l] = total;
        total += nodes_of<DIM>(n_top >> l);
    }
    if (threadIdx.x == 0) off[levels] = total;
    T* base = reinterpret_cast<T*>(smem);
    const SmemLevels<T> lv{base, off, 31 - __clz(n_top), cy.smoother == GMG_WJACOBI ? 4 : 3};
    // zero everything (boundaries stay zero), then load u and q of the top level
    for (int p = threadIdx.x; p < total * lv.arrays; p += blockDim.x)
        base[p] = Num<T>::st(typename Num<T>::C(0));
    __syncthreads();
    // the top level's interior nodes (n slots per row: shifts, no divisions);
    // its boundary is zero and stays so
    const int lg = lv.lg0;
    auto gaddr = [&](int i, int j, int k) {
        return k * top.sz + j * top.sy + (top.he ? lk::xo<true>(top, i) : i);
    };
    T* u0 = lv.u(0, 0);
    T* q0 = lv.q(0);
    auto load = [&](const T* src, T* dst) {
        copy_in(
            interior_slots<DIM>(lg),
            [&](int e) {
                int i, j, k;
                return inode<DIM>(e, lg, i, j, k) ? src[gaddr(i, j, k)]
                                                  : Num<T>::st(typename Num<T>::C(0));
            },
            [&](int e, T v) {
                int i, j, k;
                if (inode<DIM>(e, lg, i, j, k)) dst[node_at<DIM>(lg, i, j, k)] = v;
            });
    };
    load(q_top, q0);
    load(u_top, u0);
    __syncthreads();
    CtaX x;
    const int cur = vcycle<DIM>(x, lv, 0, levels, cy, exact0 != 0, first_done != 0);
    const T* ur = lv.u(0, cur);
    for (int e = threadIdx.x; e < interior_slots<DIM>(lg); e += blockDim.x) {
        int i, j, k;
        if (inode<DIM>(e, lg, i, j, k)) u_top[gaddr(i, j, k)] = ur[node_at<DIM>(lg, i, j, k)];
    }
}

// The same V-cycle on the levels' own arrays in global memory (dense
// layout), run by every CTA of a cooperative launch with grid barriers
// between the steps, on the levels with n > cta_n; block 0 alone runs the
// levels with n <= cta_n (__syncthreads) while the others wait at the next
// grid barrier.  One launch replaces the grid kernels of the middle levels
// (launch latency bound there) and the single-CTA tail.
template <typename T>
struct GridLevel {
    int lg;
    T *u, *q, *r;
};
template <typename T>
struct GridArgs {
    GridLevel<T> lv[kMaxGridLevels];
    int levels, cta_n;
    Cycle cy;
    GridBar* bar;
};
template <typename T>
struct GridLevels {
    using Type = T;
    const GridArgs<T>& a;
    __device__ int lg(int l) const { return a.lv[l].lg; }
    __device__ T* u(int l, int) const { return a.lv[l].u; }
    __device__ T* q(int l) const { return a.lv[l].q; }
    __device__ T* r(int l) const { return a.lv[l].r; }
};

// red-black smoothing with full weighting only (launch_grid)
template <int DIM, typename T, class X>
__device__ void gtail_body(X& gx, const GridArgs<T>& a) {
    const GridLevels<T> lv{a};
    const Cycle& cy = a.cy;
    const bool red_only = cy.nu1 > 0;
    int lc = 0;  // first level that block 0 takes alone
    while (lc + 1 < a.levels && (1 << lv.lg(lc)) > a.cta_n) ++lc;
    int cur = 0;
    for (int l = 0; l < lc; ++l) {
        relax<DIM>(gx, lv, l, cy, cy.nu1, cur, false, false);
        residual<DIM>(gx, lv.lg(l), lv.u(l, 0), lv.q(l), lv.r(l), red_only, false);
        restrict_to<DIM>(gx, lv.lg(l + 1), lv.r(l), lv.q(l + 1), lv.u(l + 1, 0), red_only, false,
                         l + 2 < a.levels ? INIT_ZERO : lv.lg(l + 1) == 1 ? INIT_EXACT : INIT_ZERO,
                         0.0);
    }
    if (blockIdx.x == 0) {
        CtaX cx;
        vcycle<DIM>(cx, lv, lc, a.levels, cy, false, false);
    }
    gx.sync();
    for (int l = lc - 1; l >= 0; --l) {
        prolong_add<DIM>(gx, lv.lg(l + 1), lv.u(l + 1, 0), lv.u(l, 0), false, cy.nu2 > 0);
        relax<DIM>(gx, lv, l, cy, cy.nu2, cur, true, false);
    }
}

template <int DIM, typename T>
__global__ void __launch_bounds__(kGridThreads) k_gtail(GridArgs<T> a) {
    GridX gx{a.bar};
    gtail_body<DIM>(gx, a);
}

// The same as one thread-block cluster (the grid is the cluster).
template <int DIM, typename T>
__global__ void __launch_bounds__(kGridThreads) k_ctail(GridArgs<T> a) {
    ClusterX cx;
    gtail_body<DIM>(cx, a);
}

}  // namespace

size_t smem_bytes(int d, int n_top, int levels, int smoother, size_t elem) {
    size_t total = 0;
    for (int l = 0; l < levels; ++l) {
        const size_t m = n_top >> l;
        const size_t nodes = d == 3 ? (m + 1) * (m + 1) * (m + 1) : (m + 1) * (m + 1);
        total += nodes * (smoother == GMG_WJACOBI ? 4 : 3);
    }
    return total * elem;
}

template <typename T>
cudaError_t launch(int d, const Lay& top, int levels, T* u_top, const T* q_top, int smoother,
                   double omega, int nu1, int nu2, int coarse_sweeps, cudaStream_t s,
                   bool exact_top, bool paper, bool first_done) {
    if (levels < 1 || levels > kMaxLevels) return cudaErrorInvalidValue;
    const int exact0 = exact_top && std::is_same<T, double>::value && d == 3 ? 1 : 0;
    const size_t bytes = smem_bytes(d, top.n, levels, smoother, sizeof(T));
    const Cycle cy{smoother, nu1, nu2, coarse_sweeps, paper, omega};
    // one thread per slot of the top level's sweeps (128..1024): more warps
    // only lengthen the barriers
    const int64_t nodes = d == 3 ? (int64_t)top.n * top.n * top.n : (int64_t)top.n * top.n;
    const int64_t slots = smoother == GMG_WJACOBI ? nodes : nodes / 2;
    const int threads = (int)std::min<int64_t>(1024, std::max<int64_t>(128, slots));
    if (bytes > kSmemLimit) return cudaErrorInvalidValue;
    auto kern = d == 3 ? k_tail<3, T> : k_tail<2, T>;
    // the limit belongs to the kernel: one value whatever the launch takes, so
    // that no thread lowers it between another's limit and launch
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmemLimit);
    if (e != cudaSuccess) return e;
    kern<<<1, threads, bytes, s>>>(u_top, q_top, top, levels, cy, exact0,
                                  first_done ? 1 : 0);
    return cudaGetLastError();
}

template <typename T>
int grid_blocks(int d) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
        return 0;
    const cudaError_t e =
        d == 3 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gtail<3, T>,
                                                               kGridThreads, 0)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gtail<2, T>,
                                                               kGridThreads, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms * per_sm;
}

template <typename T>
cudaError_t launch_grid(int d, int levels, const int* n, T* const* u, T* const* q, T* const* r,
                        int smoother, double omega, int nu1, int nu2, int coarse_sweeps,
                        int cta_n, void* bar, int blocks, cudaStream_t s, int cluster) {
    if (levels < 1 || levels > kMaxGridLevels || smoother != GMG_RBGS ||
        (cluster <= 0 && blocks < 1) || cluster > 16)
        return cudaErrorInvalidValue;
    GridArgs<T> a{};
    for (int l = 0; l < levels; ++l) {
        int lg = 0;
        while ((1 << lg) < n[l]) ++lg;
        a.lv[l] = GridLevel<T>{lg, u[l], q[l], r[l]};
    }
    a.levels = levels;
    a.cta_n = cta_n;
    a.cy = Cycle{smoother, nu1, nu2, coarse_sweeps, false, omega};
    a.bar = static_cast<GridBar*>(bar);
    if (cluster > 0) {
        auto kern = d == 3 ? k_ctail<3, T> : k_ctail<2, T>;
        cudaError_t e = cudaSuccess;
        if (cluster > 8)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(cluster);
        cfg.blockDim = dim3(kGridThreads);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cluster;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, kern, a);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(&a.bar->count, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&a};
    e = d == 3 ? cudaLaunchCooperativeKernel((const void*)k_gtail<3, T>, dim3(blocks),
                                             dim3(kGridThreads), args, 0, s)
               : cudaLaunchCooperativeKernel((const void*)k_gtail<2, T>, dim3(blocks),
                                             dim3(kGridThreads), args, 0, s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

size_t grid_bar_bytes() { return sizeof(GridBar); }

int grid_fault(const void* bar) {
    int v = 0;
    if (cudaMemcpy(&v, &static_cast<const GridBar*>(bar)->fault, sizeof(int),
                   cudaMemcpyDeviceToHost) != cudaSuccess)
        return -1;
    return v;
}

#define GMG_GRID_INST(T)                                                                        \
    template int grid_blocks<T>(int);                                                           \
    template cudaError_t launch_grid<T>(int, int, const int*, T* const*, T* const*, T* const*,  \
                                        int, double, int, int, int, int, void*, int,            \
                                        cudaStream_t, int);
GMG_GRID_INST(double)
GMG_GRID_INST(float)
GMG_GRID_INST(__nv_bfloat16)
GMG_GRID_INST(df32)
#undef GMG_GRID_INST

template cudaError_t launch<double>(int, const Lay&, int, double*, const double*, int, double,
                                    int, int, int, cudaStream_t, bool, bool, bool);
template cudaError_t launch<float>(int, const Lay&, int, float*, const float*, int, double, int,
                                   int, int, cudaStream_t, bool, bool, bool);
template cudaError_t launch<__nv_bfloat16>(int, const Lay&, int, __nv_bfloat16*,
                                           const __nv_bfloat16*, int, double, int, int, int,
                                           cudaStream_t, bool, bool, bool);
template cudaError_t launch<df32>(int, const Lay&, int, df32*, const df32*, int, double, int, int,
                                  int, cudaStream_t, bool, bool, bool);

}  // namespace tail
}  // namespace gmg
