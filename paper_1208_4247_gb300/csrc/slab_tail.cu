// The V-cycle from a 33^3 or 17^3 level down, in one launch of one cluster
// of 16 CTAs with every array in (distributed) shared memory.
//
// On these levels a launch per step costs 2.5 to 3 us whatever its work
// (1.25 us of launch, the rest the latency of its L2 loads), 11 steps a level.
// Here CTA r keeps the planes k = r P + 1 .. r P + P of a level (P = 2 at n =
// 32, 1 at n = 16) and one plane of its neighbours on either side; a thread
// that writes a node of a CTA's first or last plane stores it into the
// neighbour's copy too (distributed shared memory).  So every load is local,
// and a step ends with the cluster's hardware barrier.  The levels from 9^3
// down run in CTA 0 (tail_steps.cuh) while the others wait at that barrier.
// Red-black smoothing with full weighting; the arithmetic of every step is
// the level kernels', node for node, so the results are theirs bit for bit.
//
// What bounds it: the cluster barrier with the remote stores it waits for
// (750 cycles of a step's 1200 to 2000) and, in FP64, the 16 SMs' pipes: a half
// sweep at n = 32 takes 1.9 us of them, so the FP64 form starts at 17^3 and
// leaves 33^3 to the grid kernels, which spread it over every SM.  One launch,
// from 33^3: FP32 27 us, double-float 42 us, against 11 grid launches a level
// and the single-CTA tail, about 70 and 85 us; FP64 from 17^3 26 us (45 us).
// Per solve, single-CTA tail from 9^3 -> this: 65^3 FP64 1187 -> 1075 us (978
// from 17^3 with CoarseInit; 1044 from 33^3), 257^3 BF16 9.44 -> 8.89 ms (8.81
// from 33^3, 8.94 from 17^3), 257^3 double-float 6.94 -> 6.80 ms.
#include <algorithm>

#include "tail_steps.cuh"

namespace gmg {
namespace tail {
namespace {

constexpr int kRanks = 16;
constexpr int kSlabThreads = 512;

__device__ inline int cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
// Every thread of every CTA reaches each barrier.
__device__ inline void cluster_sync() {
    __syncwarp();
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this CTA's shared variable p in the CTA of another rank.
template <typename T>
__device__ inline T* at_rank(T* p, int rank) {
    uint64_t a;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"(p), "r"(rank));
    return reinterpret_cast<T*>(a);
}

// One level's planes in this CTA: u and r hold P + 2 planes (the neighbours'
// first), q holds P.  down / up: the neighbours' arrays (NULL at the ends).
template <typename T>
struct Slab {
    int lg, P, rank;
    T *u, *q, *r;
    T *u_down, *u_up, *r_down, *r_up;
    __device__ int n() const { return 1 << lg; }
    __device__ int m() const { return (1 << lg) + 1; }
    __device__ int plane(int kl) const { return rank * P + 1 + kl; }  // global k of plane kl
    // value of node o of plane kl into array a and the neighbours' copies
    __device__ void put(T* a, T* a_down, T* a_up, int kl, int o, T v) const {
        const int m2 = m() * m();
        a[(kl + 1) * m2 + o] = v;
        if (kl == 0 && a_down) a_down[(P + 1) * m2 + o] = v;
        if (kl == P - 1 && a_up) a_up[o] = v;
    }
    __device__ void put_u(int kl, int o, T v) const { put(u, u_down, u_up, kl, o, v); }
    __device__ void put_r(int kl, int o, T v) const { put(r, r_down, r_up, kl, o, v); }
};

template <typename T>
__device__ Slab<T> make_slab(T*& base, int lg, int rank) {
    Slab<T> L;
    L.lg = lg;
    L.P = (1 << lg) / kRanks;
    L.rank = rank;
    const int m2 = L.m() * L.m();
    L.u = base;
    L.r = base + (L.P + 2) * m2;
    L.q = base + 2 * (L.P + 2) * m2;
    base += (3 * L.P + 4) * m2;
    L.u_down = rank > 0 ? at_rank(L.u, rank - 1) : nullptr;
    L.r_down = rank > 0 ? at_rank(L.r, rank - 1) : nullptr;
    L.u_up = rank + 1 < kRanks ? at_rank(L.u, rank + 1) : nullptr;
    L.r_up = rank + 1 < kRanks ? at_rank(L.r, rank + 1) : nullptr;
    return L;
}
__host__ __device__ constexpr int slab_elems(int n) {
    return (3 * (n / kRanks) + 4) * (n + 1) * (n + 1);
}
constexpr int kSmallNodes = 729 + 125 + 27;  // levels 8, 4, 2

// f(kl, j, i, o) for this CTA's nodes of one colour, or (color < 0) for all of them
template <typename T, class F>
__device__ inline void slab_nodes(const Slab<T>& L, int color, F&& f) {
    const int n = L.n(), lg = L.lg;
    const int row = color < 0 ? lg : lg - 1;  // log2 slots per row
    for (int idx = threadIdx.x; idx < L.P << (lg + row); idx += blockDim.x) {
        const int t = idx & ((1 << row) - 1);
        const int j = (idx >> row) & (n - 1), kl = idx >> (row + lg);
        const int k = L.plane(kl);
        const int i = color < 0 ? t : 2 * t + (((color + j + k) & 1) ? 1 : 2);
        if (i > 0 && i < n && j > 0 && k < n) f(kl, j * L.m() + i);
    }
}

template <typename T>
__device__ void slab_half(const Slab<T>& L, int color, bool ex) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = C(1.0 / 6.0);
    const int m = L.m(), m2 = m * m;
    slab_nodes(L, color, [&](int kl, int o) {
        const C s = lk::nbr_sum<3>(L.u, (kl + 1) * m2 + o, m, m2);
        const C q = N::ld(L.q[kl * m2 + o]);
        L.put_u(kl, o,
                N::st(ex ? lk::gs_value<3, true>(c, s, q) : lk::gs_value<3, false>(c, s, q)));
    });
    cluster_sync();
}

// first_done: the first red half sweep ran already
template <typename T>
__device__ void slab_relax(const Slab<T>& L, int sweeps, bool first_done, bool exact_last) {
    for (int s = 0; s < sweeps; ++s)
        for (int color = first_done && s == 0 ? 1 : 0; color < 2; ++color)
            slab_half(L, color, exact_last && color == 1 && s == sweeps - 1);
}

template <typename T>
__device__ void slab_residual(const Slab<T>& L, bool red_only, bool ex) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = C(1.0 / 6.0);
    const int m = L.m(), m2 = m * m;
    slab_nodes(L, red_only ? 0 : -1, [&](int kl, int o) {
        const int p = (kl + 1) * m2 + o;
        const C s = lk::nbr_sum<3>(L.u, p, m, m2);
        const C q = N::ld(L.q[kl * m2 + o]);
        const C v = ex ? lk::gs_value<3, true>(c, s, q) : lk::gs_value<3, false>(c, s, q);
        L.put_r(kl, o, N::st(v - N::ld(L.u[p])));
    });
    cluster_sync();
}

// Coarse nodes (I, J) under the fine plane at r (its neighbours in z one
// plane before and after): f(I, J, value).  lg: the coarse level.
template <typename T, class F>
__device__ void slab_restrict(const T* r, int lg, bool red_only, F&& f) {
    using N = Num<T>;
    using C = typename N::C;
    const int sy = (2 << lg) + 1, sz = sy * sy;
    for (int idx = threadIdx.x; idx < 1 << (2 * lg); idx += blockDim.x) {
        const int I = idx & ((1 << lg) - 1), J = idx >> lg;
        if (I == 0 || J == 0) continue;
        f(I, J, fw3<C>([&](int o) { return N::ld(r[2 * J * sy + 2 * I + o]); }, sy, sz, red_only));
    }
}

// u += P u_c on one fine plane (kl of L): A, B the coarse planes below and
// above it (odd: it lies halfway between them, else on A).  black: the black
// fine nodes only (a red half sweep follows).
template <typename T>
__device__ void slab_prolong(const Slab<T>& L, int kl, const T* A, const T* B, bool odd,
                             bool black) {
    using N = Num<T>;
    using C = typename N::C;
    const int lc = L.lg - 1, nc = 1 << lc, mc = nc + 1, m = L.m();
    const T* u = L.u + (kl + 1) * m * m;
    for (int cell = threadIdx.x; cell < nc * nc; cell += blockDim.x) {
        const int I = cell & (nc - 1), J = cell >> lc;
        const int P = J * mc + I, o = 2 * J * m + 2 * I;
        // fine node (2I + (v & 1), 2J + (v >> 1)): interior, and corrected here?
        auto on = [&](int v) {
            const bool black_node = ((v & 1) ^ (v >> 1)) != (odd ? 1 : 0);
            return ((v & 1) || I > 0) && ((v & 2) || J > 0) && (black_node || !black);
        };
        auto off = [&](int v) { return o + (v & 1) + (v >> 1) * m; };
        C f[4];
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (on(v)) f[v] = N::ld(u[off(v)]);
        auto add = [&](int v, C w, C s) {
            if (on(v)) L.put_u(kl, off(v), N::st(fma(w, s, f[v])));
        };
        const C c000 = N::ld(A[P]), c100 = N::ld(A[P + 1]), c010 = N::ld(A[P + mc]),
                c110 = N::ld(A[P + 1 + mc]);
        const C x00 = c000 + c100, y00 = c000 + c010;
        if (!odd) {
            if (on(0)) L.put_u(kl, o, N::st(f[0] + c000));
            add(1, C(0.5), x00);
            add(2, C(0.5), y00);
            if (!black) add(3, C(0.25), x00 + (c010 + c110));
        } else {
            const C c001 = N::ld(B[P]), c101 = N::ld(B[P + 1]), c011 = N::ld(B[P + mc]),
                    c111 = N::ld(B[P + 1 + mc]);
            const C x01 = c001 + c101;
            add(0, C(0.5), c000 + c001);
            if (!black) {
                add(1, C(0.25), x00 + x01);
                add(2, C(0.25), y00 + (c001 + c011));
            }
            add(3, C(0.125), (x00 + (c010 + c110)) + (x01 + (c011 + c111)));
        }
    }
}

// first_done: the top level's first red half sweep ran already (u_top holds it)
template <typename T>
__global__ void __launch_bounds__(kSlabThreads)
    k_slab_tail(T* __restrict__ u_top, const T* __restrict__ q_top, Lay top, int levels, Cycle cy,
                int exact0, int first_done) {
    using N = Num<T>;
    using C = typename N::C;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int off[kMaxLevels + 1];
    const int rank = cluster_rank(), n = top.n;
    const bool big = n == 32;
    // shared memory: the top slab, the 17^3 slab (if the top is 33^3), the
    // small levels (used by CTA 0), two of the 9^3 level's planes
    T* base = reinterpret_cast<T*>(smem);
    T* p = base;
    const Slab<T> L0 = make_slab<T>(p, big ? 5 : 4, rank);
    const Slab<T> L1 = big ? make_slab<T>(p, 4, rank) : L0;
    T* small = p;
    T* c8 = small + 3 * kSmallNodes;
    for (int e = threadIdx.x; e < (int)(c8 - base) + 2 * 81; e += blockDim.x) base[e] = N::st(C(0));
    if (threadIdx.x == 0) {
        off[0] = 0;
        for (int l = 0, nn = 8; l < 3; ++l, nn /= 2) off[l + 1] = off[l] + nodes_of<3>(nn);
    }
    cluster_sync();  // zeroed everywhere before a neighbour stores into it
    // interior nodes of planes kl0.. by slots of n per row (shifts only: a
    // division per node made this the longest part of the launch): array
    // element and offset in top's layout; -1 for the rest, which is zero
    const int m = n + 1, m2 = m * m, lg = L0.lg;
    auto element = [&](int idx, int kl0) {
        const int i = idx & (n - 1), j = (idx >> lg) & (n - 1), kl = kl0 + (idx >> (2 * lg));
        const int k = L0.plane(kl);
        return i > 0 && j > 0 && k > 0 && k < n ? (kl - kl0) * m2 + j * m + i : -1;
    };
    auto gaddr = [&](int idx, int kl0) {
        const int i = idx & (n - 1), j = (idx >> lg) & (n - 1);
        return L0.plane(kl0 + (idx >> (2 * lg))) * top.sz + j * top.sy +
               (top.he ? lk::xo<true>(top, i) : i);
    };
    copy_in((L0.P + 2) << (2 * lg),
            [&](int e) { return element(e, -1) >= 0 ? u_top[gaddr(e, -1)] : N::st(C(0)); },
            [&](int e, T v) { if (element(e, -1) >= 0) L0.u[element(e, -1)] = v; });
    copy_in(L0.P << (2 * lg),
            [&](int e) { return element(e, 0) >= 0 ? q_top[gaddr(e, 0)] : N::st(C(0)); },
            [&](int e, T v) { if (element(e, 0) >= 0) L0.q[element(e, 0)] = v; });
    __syncthreads();

    const bool red_only = cy.nu1 > 0;
    const int init = cy.nu1 > 0 ? INIT_RED : INIT_ZERO;
    slab_relax(L0, cy.nu1, first_done != 0, exact0 != 0);
    slab_residual(L0, red_only, exact0 != 0);
    if (big) {
        // coarse plane rank + 1 lies under fine plane 2 rank + 2, local plane 1;
        // its first red half sweep is done here
        if (rank + 1 < 16)
            slab_restrict(L0.r + 2 * m2, 4, red_only, [&](int I, int J, C v) {
                const int o = J * 17 + I;
                L1.q[o] = N::st(v);
                L1.put_u(0, o, lk::coarse_init<3>(init, 0.0, I, J, rank + 1, N::st(v)));
            });
        cluster_sync();
        slab_relax(L1, cy.nu1, init != INIT_ZERO, false);
        slab_residual(L1, red_only, false);
    }
    // 17^3 -> 9^3 in CTA 0: coarse plane (rank + 1)/2 of the odd ranks
    T* u8 = at_rank(small, 0);
    T* q8 = u8 + 729;
    if (rank & 1 && rank + 1 < 16)
        slab_restrict(L1.r + 289, 3, red_only, [&](int I, int J, C v) {
            const int P = ((rank + 1) / 2) * 81 + J * 9 + I;
            q8[P] = N::st(v);
            u8[P] = lk::coarse_init<3>(init, 0.0, I, J, (rank + 1) / 2, N::st(v));
        });
    cluster_sync();
    if (rank == 0) {
        CtaX x;
        const SmemLevels<T> lv{small, off, 3, 3};
        vcycle<3>(x, lv, 0, levels - (big ? 2 : 1), cy, false, init != INIT_ZERO);
    }
    cluster_sync();
    const bool black = cy.nu2 > 0;
    if (rank + 1 < 16) {  // plane k = rank + 1 of the 17^3 level
        const int k = rank + 1;
        for (int e = threadIdx.x; e < (k & 1 ? 162 : 81); e += blockDim.x)
            c8[e] = u8[(k / 2) * 81 + e];
        __syncthreads();
        slab_prolong(L1, 0, c8, c8 + 81, k & 1, black);
    }
    cluster_sync();
    slab_relax(L1, cy.nu2, false, false);
    if (big) {
        slab_prolong(L0, 0, L1.u, L1.u + 289, true, black);
        if (L0.plane(1) < n) slab_prolong(L0, 1, L1.u + 289, L1.u, false, black);
        cluster_sync();
        slab_relax(L0, cy.nu2, false, false);
    }
    // the last barrier above also keeps every CTA's memory alive for the others
    for (int e = threadIdx.x; e < L0.P << (2 * lg); e += blockDim.x)
        if (element(e, 0) >= 0) u_top[gaddr(e, 0)] = L0.u[m2 + element(e, 0)];
}

}  // namespace

// At least two of the small levels: the cycle CTA 0 runs on them takes a single
// one for a whole hierarchy.
bool slab_applies(int d, int n, int levels, int smoother, bool paper, bool fp64) {
    return d == 3 && (n == 16 || (n == 32 && !fp64)) && levels >= (n == 32 ? 4 : 3) &&
           levels <= (n == 32 ? 5 : 4) &&
           (smoother == GMG_RBGS || smoother == GMG_LEARNED) && !paper;
}

// bytes of a launch whose top level has n intervals
template <typename T>
constexpr size_t slab_bytes(int n) {
    return sizeof(T) * (slab_elems(n) + (n == 32 ? slab_elems(16) : 0) + 3 * kSmallNodes + 2 * 81);
}

// The launch of a cluster over a top level of n intervals: its attribute is at
// `at`, and the kernel's limits are set.  They belong to the kernel: the larger
// launch's for both sizes, so that no thread lowers them between another's limit
// and launch.
template <typename T>
cudaError_t slab_config(int n, cudaStream_t s, cudaLaunchAttribute* at, cudaLaunchConfig_t* cfg) {
    auto kern = k_slab_tail<T>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)slab_bytes<T>(32));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(kRanks);
    cfg->blockDim = dim3(kSlabThreads);
    cfg->dynamicSmemBytes = slab_bytes<T>(n);
    cfg->stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = kRanks;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return e;
}

// 16 CTAs are more than the portable 8: whether the current device has a place
// for them (16 free SMs in one GPC, or in a part of the device) is its answer.
template <typename T>
bool slab_fits(int n) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg;
    int clusters = 0;
    cudaError_t e = slab_config<T>(n, nullptr, at, &cfg);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, k_slab_tail<T>, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters > 0;
}

template <typename T>
cudaError_t launch_slab(const Lay& top, int levels, T* u_top, const T* q_top, int smoother,
                        int nu1, int nu2, int coarse_sweeps, cudaStream_t s, bool exact_top,
                        bool first_done) {
    const Cycle cy{smoother, nu1, nu2, coarse_sweeps, false, 0.0};
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg;
    cudaError_t e = slab_config<T>(top.n, s, at, &cfg);
    if (e != cudaSuccess) return e;
    const int ex = exact_top && std::is_same<T, double>::value ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, k_slab_tail<T>, u_top, q_top, top, levels, cy, ex,
                           first_done ? 1 : 0);
    return e != cudaSuccess ? e : cudaGetLastError();
}

#define GMG_SLAB_INST(T)                                                                     \
    template bool slab_fits<T>(int);                                                         \
    template cudaError_t launch_slab<T>(const Lay&, int, T*, const T*, int, int, int, int,   \
                                        cudaStream_t, bool, bool);
GMG_SLAB_INST(double)
GMG_SLAB_INST(float)
GMG_SLAB_INST(__nv_bfloat16)
GMG_SLAB_INST(df32)
#undef GMG_SLAB_INST

}  // namespace tail
}  // namespace gmg
