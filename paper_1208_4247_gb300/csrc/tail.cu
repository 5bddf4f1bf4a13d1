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

#include "level_kernels.cuh"

namespace gmg {
namespace tail {
namespace {

using lk::Num;

constexpr int kMaxLevels = 8;       // single-CTA tail
constexpr int kMaxGridLevels = 12;  // grid tail
constexpr int kGridThreads = 512;

template <int DIM>
__device__ inline int nodes_of(int n) {
    const int m = n + 1;
    return DIM == 3 ? m * m * m : m * m;
}

// The steps take the level size at run time (lg = log2 n) and split a slot
// number by shifts and masks: one copy of each step's code serves every
// level.  A launch runs each step once per level, so its instructions are
// fetched once instead of once per level size: with the size as a template
// argument the single CTA spent much of its time on instruction fetches
// (about 1 us a step at 9^3, whatever the arithmetic).  Measured per solve,
// template size -> run-time size: 2D 257^2 weighted Jacobi V(2,2) 1440 ->
// 1273 us (14 launches of the tail from 33^2), 3D 65^3 red-black 1242 ->
// 1187 us (9 from 9^3), 257^3 double-float 7.19 -> 6.94 ms (9 from 9^3).
// What is left is the FP64 pipe of one SM (one warp's add takes 64 of its
// cycles) and, below 9^3, the chains of dependent adds.  The slots of a
// level are padded to powers of two (row 0, and the one slot past the end
// of a colour's row, are idle).
//
// Slots of the interior nodes: n per row.  (i, j, k) of slot idx; false for
// the idle ones.
template <int DIM>
__device__ inline int interior_slots(int lg) { return 1 << (DIM * lg); }
template <int DIM>
__device__ inline bool inode(int idx, int lg, int& i, int& j, int& k) {
    const int mask = (1 << lg) - 1;
    i = idx & mask;
    j = (idx >> lg) & mask;
    k = DIM == 3 ? idx >> (2 * lg) : 0;
    return i > 0 && j > 0 && (DIM == 2 || k > 0);
}
template <int DIM>
__device__ inline int node_at(int lg, int i, int j, int k) {
    const int m = (1 << lg) + 1;
    return ((DIM == 3 ? k * m : 0) + j) * m + i;
}
// Slots of one colour ((i + j + k) & 1 == color): n/2 per row.
template <int DIM>
__device__ inline int color_slots(int lg) { return 1 << (DIM * lg - 1); }
template <int DIM>
__device__ inline bool cnode(int idx, int lg, int color, int& p) {
    const int n = 1 << lg;
    const int t = idx & (n / 2 - 1);
    const int row = idx >> (lg - 1);
    const int j = row & (n - 1), k = DIM == 3 ? row >> lg : 0;
    const int i = 2 * t + (((color + j + k) & 1) ? 1 : 2);
    p = node_at<DIM>(lg, i, j, k);
    return i < n && j > 0 && (DIM == 2 || k > 0);
}

// Who runs a step and how the steps are separated: one CTA (__syncthreads),
// or every CTA of a cooperative launch (a grid barrier).
struct CtaX {
    __device__ int tid() const { return threadIdx.x; }
    __device__ int nt() const { return blockDim.x; }
    __device__ void sync() { __syncthreads(); }
};

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

// ex: the unbiased FP64 3D value (lk::gs_value), as the grid kernels take
// it on level 0 of a plain FP64 hierarchy
template <int DIM, typename T, class X>
__device__ void rb_half(X& x, int lg, T* u, const T* q, int color, bool ex = false) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = DIM == 3 ? C(1.0 / 6.0) : C(0.25);
    const int sy = (1 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    for (int idx = x.tid(); idx < color_slots<DIM>(lg); idx += x.nt()) {
        int p;
        if (!cnode<DIM>(idx, lg, color, p)) continue;
        const C s = lk::nbr_sum<DIM>(u, p, sy, sz);
        u[p] = N::st(ex ? lk::gs_value<DIM, true>(c, s, N::ld(q[p]))
                        : lk::gs_value<DIM, false>(c, s, N::ld(q[p])));
    }
    x.sync();
}

// One colour (i&1) + 2(j&1) + 4(k&1) of the paper's Gauss-Seidel (FP64).
template <int DIM, typename T, class X>
__device__ void mc_color(X& x, int lg, T* u, const T* q, int color) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = DIM == 3 ? C(1.0 / 6.0) : C(0.25);
    const int n = 1 << lg, h = n / 2 - 1;
    const int sy = n + 1, sz = DIM == 3 ? sy * sy : 0;
    for (int idx = x.tid(); idx < 1 << (DIM * (lg - 1)); idx += x.nt()) {
        const int i = 2 * (idx & h) + ((color & 1) ? 1 : 2);
        const int j = 2 * ((idx >> (lg - 1)) & h) + ((color & 2) ? 1 : 2);
        const int k = DIM == 3 ? 2 * (idx >> (2 * (lg - 1))) + ((color & 4) ? 1 : 2) : 0;
        if (i >= n || j >= n || (DIM == 3 && k >= n)) continue;
        const int p = node_at<DIM>(lg, i, j, k);
        u[p] = N::st(fma(c, lk::nbr_sum<DIM>(u, p, sy, sz), N::ld(q[p])));
    }
    x.sync();
}

template <int DIM, typename T, class X>
__device__ void wj_sweep(X& x, int lg, const T* u, T* uo, const T* q, double omega_d) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = DIM == 3 ? C(1.0 / 6.0) : C(0.25);
    const C omega = C(omega_d);
    const int sy = (1 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    for (int idx = x.tid(); idx < interior_slots<DIM>(lg); idx += x.nt()) {
        int i, j, k;
        if (!inode<DIM>(idx, lg, i, j, k)) continue;
        const int p = node_at<DIM>(lg, i, j, k);
        const C up = N::ld(u[p]);
        const C sig =
            lk::gs_value<DIM, false>(c, lk::nbr_sum<DIM>(u, p, sy, sz), N::ld(q[p])) - up;
        uo[p] = N::st(fma(omega, sig, up));
    }
    x.sync();
}

// What the steps of one V-cycle share.
struct Cycle {
    int smoother, nu1, nu2, coarse_sweeps;
    bool paper;  // the paper's transfers
    double omega;
};

// `sweeps` sweeps on level l of lv; cur: which u buffer holds the iterate
// (weighted Jacobi alternates).
template <int DIM, class X, class LV>
__device__ void relax(X& x, const LV& lv, int l, const Cycle& cy, int sweeps, int& cur,
                      bool backward, bool exact_last) {
    const int lg = lv.lg(l);
    for (int s = 0; s < sweeps; ++s) {
        if (cy.smoother == GMG_WJACOBI) {
            wj_sweep<DIM>(x, lg, lv.u(l, cur), lv.u(l, cur ^ 1), lv.q(l), cy.omega);
            cur ^= 1;
            continue;
        }
        if constexpr (std::is_same<typename LV::Type, double>::value) {
            if (cy.smoother == GMG_MCGS) {
                constexpr int ncol = 1 << DIM;
                for (int t = 0; t < ncol; ++t)
                    mc_color<DIM>(x, lg, lv.u(l, cur), lv.q(l), backward ? ncol - 1 - t : t);
                continue;
            }
        }
        for (int color = 0; color < 2; ++color)
            rb_half<DIM>(x, lg, lv.u(l, cur), lv.q(l), color,
                         exact_last && color == 1 && s == sweeps - 1);
    }
}

template <int DIM, typename T, class X>
__device__ void residual(X& x, int lg, const T* u, const T* q, T* r, bool red_only, bool ex) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = DIM == 3 ? C(1.0 / 6.0) : C(0.25);
    const int sy = (1 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    const int slots = red_only ? color_slots<DIM>(lg) : interior_slots<DIM>(lg);
    for (int idx = x.tid(); idx < slots; idx += x.nt()) {
        int p;
        if (red_only) {
            if (!cnode<DIM>(idx, lg, 0, p)) continue;
        } else {
            int i, j, k;
            if (!inode<DIM>(idx, lg, i, j, k)) continue;
            p = node_at<DIM>(lg, i, j, k);
        }
        const C s = lk::nbr_sum<DIM>(u, p, sy, sz);
        const C v = ex ? lk::gs_value<DIM, true>(c, s, N::ld(q[p]))
                       : lk::gs_value<DIM, false>(c, s, N::ld(q[p]));
        r[p] = N::st(v - N::ld(u[p]));
    }
    x.sync();
}

// fine level lg + 1 -> coarse level lg
template <int DIM, typename T, class X>
__device__ void restrict_to(X& x, int lg, const T* r, T* qc, T* uc, bool red_only, bool paper) {
    using N = Num<T>;
    using C = typename N::C;
    const int sy = (2 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    const bool exact = lg == 1;
    for (int idx = x.tid(); idx < interior_slots<DIM>(lg); idx += x.nt()) {
        int I, J, K;
        if (!inode<DIM>(idx, lg, I, J, K)) continue;
        const int P = node_at<DIM>(lg, I, J, K);
        const int p = 2 * K * sz + 2 * J * sy + 2 * I;
        auto R = [&](int o) { return N::ld(r[p + o]); };
        C v;
        if (std::is_same<T, double>::value && paper) {
            C s = (R(-1) + R(1)) + (R(-sy) + R(sy));
            s += R(-1 - sy) + R(1 + sy);
            if (DIM == 3) {
                C t = (R(-sz) + R(sz)) + (R(-1 - sz) + R(1 + sz));
                t += (R(-sy - sz) + R(sy + sz)) + (R(-1 - sy - sz) + R(1 + sy + sz));
                v = fma(C(0.25), s + t, C(0.5) * R(0));
            } else {
                v = fma(C(0.5), s, R(0));
            }
        } else if (DIM == 3) {
            C e = R(-1 - sy) + R(1 - sy);
            e += R(-1 + sy);
            e += R(1 + sy);
            e += R(-1 - sz);
            e += R(1 - sz);
            e += R(-sy - sz);
            e += R(sy - sz);
            e += R(-1 + sz);
            e += R(1 + sz);
            e += R(-sy + sz);
            e += R(sy + sz);
            if (red_only) {
                v = fma(C(0.125), e, C(0.5) * R(0));
            } else {
                C fc = R(-1) + R(1);
                fc += R(-sy);
                fc += R(sy);
                fc += R(-sz);
                fc += R(sz);
                C co = R(-1 - sy - sz) + R(1 - sy - sz);
                co += R(-1 + sy - sz);
                co += R(1 + sy - sz);
                co += R(-1 - sy + sz);
                co += R(1 - sy + sz);
                co += R(-1 + sy + sz);
                co += R(1 + sy + sz);
                v = fma(C(0.0625), co, fma(C(0.125), e, fma(C(0.25), fc, C(0.5) * R(0))));
            }
        } else {
            C co = R(-1 - sy) + R(1 - sy);
            co += R(-1 + sy);
            co += R(1 + sy);
            if (red_only) {
                v = fma(C(0.25), co, R(0));
            } else {
                C fc = R(-1) + R(1);
                fc += R(-sy);
                fc += R(sy);
                v = fma(C(0.25), co, fma(C(0.5), fc, R(0)));
            }
        }
        qc[P] = N::st(v);
        uc[P] = exact ? N::st(v) : N::st(C(0));
    }
    x.sync();
}

// coarse level lg -> fine level lg + 1
template <int DIM, typename T, class X>
__device__ void prolong_add(X& x, int lg, const T* uc, T* u, bool paper) {
    using N = Num<T>;
    using C = typename N::C;
    const int nc = 1 << lg;
    const int sy = (2 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    const int cy = nc + 1, cz = DIM == 3 ? cy * cy : 0;
    for (int cell = x.tid(); cell < interior_slots<DIM>(lg); cell += x.nt()) {
        const int I = cell & (nc - 1), J = (cell >> lg) & (nc - 1), K = DIM == 3 ? cell >> (2 * lg) : 0;
        const int P = K * cz + J * cy + I;
        const int p = 2 * K * sz + 2 * J * sy + 2 * I;
        auto add = [&](int o, C w, C v) { u[o] = N::st(fma(w, v, N::ld(u[o]))); };
        const C c000 = N::ld(uc[P]), c100 = N::ld(uc[P + 1]), c010 = N::ld(uc[P + cy]),
                c110 = N::ld(uc[P + 1 + cy]);
        if (std::is_same<T, double>::value && paper) {
            if (DIM == 2 || K > 0) {
                if (I > 0 && J > 0) u[p] = N::st(N::ld(u[p]) + c000);
                if (J > 0) add(p + 1, C(0.5), c000 + c100);
                if (I > 0) add(p + sy, C(0.5), c000 + c010);
                add(p + 1 + sy, C(0.5), c000 + c110);
            }
            if (DIM == 3) {
                const C c001 = N::ld(uc[P + cz]), c101 = N::ld(uc[P + 1 + cz]),
                        c011 = N::ld(uc[P + cy + cz]), c111 = N::ld(uc[P + 1 + cy + cz]);
                const int pz = p + sz;
                if (I > 0 && J > 0) add(pz, C(0.5), c000 + c001);
                if (J > 0) add(pz + 1, C(0.5), c000 + c101);
                if (I > 0) add(pz + sy, C(0.5), c000 + c011);
                add(pz + 1 + sy, C(0.5), c000 + c111);
            }
            continue;
        }
        const C x00 = c000 + c100;
        const C x10 = c010 + c110;
        const C y00 = c000 + c010;
        const C qxy = x00 + x10;
        if (DIM == 2) {
            if (I > 0 && J > 0) u[p] = N::st(N::ld(u[p]) + c000);
            if (J > 0) add(p + 1, C(0.5), x00);
            if (I > 0) add(p + sy, C(0.5), y00);
            add(p + 1 + sy, C(0.25), qxy);
        } else {
            const C c001 = N::ld(uc[P + cz]), c101 = N::ld(uc[P + 1 + cz]),
                    c011 = N::ld(uc[P + cy + cz]), c111 = N::ld(uc[P + 1 + cy + cz]);
            const C x01 = c001 + c101;
            const C x11 = c011 + c111;
            const C y01 = c001 + c011;
            const C z00 = c000 + c001;
            const C qxz = x00 + x01;
            const C qyz = y00 + y01;
            const C oct = qxy + (x01 + x11);
            if (K > 0) {
                if (I > 0 && J > 0) u[p] = N::st(N::ld(u[p]) + c000);
                if (J > 0) add(p + 1, C(0.5), x00);
                if (I > 0) add(p + sy, C(0.5), y00);
                add(p + 1 + sy, C(0.25), qxy);
            }
            const int pz = p + sz;
            if (I > 0 && J > 0) add(pz, C(0.5), z00);
            if (J > 0) add(pz + 1, C(0.25), qxz);
            if (I > 0) add(pz + sy, C(0.25), qyz);
            add(pz + 1 + sy, C(0.125), oct);
        }
    }
    x.sync();
}

// The V-cycle on levels from .. levels-1 of lv (level `from` given: q set, u =
// 0 or a start), run by x: down (pre-smoothing, residual, restriction), the
// coarsest grid, up (prolongation with correction, post-smoothing).  Returns
// the u buffer of level `from` that holds the result.
// exact0: level `from` is level 0 of a plain FP64 3D hierarchy (unbiased value).
template <int DIM, class X, class LV>
__device__ int vcycle(X& x, const LV& lv, int from, int levels, const Cycle& cy, bool exact0) {
    // (a learned handle's tail levels smooth with red-black Gauss-Seidel)
    const bool red_black = cy.smoother == GMG_RBGS || cy.smoother == GMG_LEARNED;
    const bool red_only = red_black && cy.nu1 > 0 && !cy.paper;
    // weighted Jacobi: every level descends in buffer nu1 & 1
    int down = 0;
    for (int l = from; l + 1 < levels; ++l) {
        down = 0;
        relax<DIM>(x, lv, l, cy, cy.nu1, down, false, exact0 && l == from);
        residual<DIM>(x, lv.lg(l), lv.u(l, down), lv.q(l), lv.r(l), red_only, exact0 && l == from);
        restrict_to<DIM>(x, lv.lg(l + 1), lv.r(l), lv.q(l + 1), lv.u(l + 1, 0), red_only, cy.paper);
    }
    const int b = levels - 1;
    int cur = 0;
    if (levels - from == 1) {
        relax<DIM>(x, lv, b, cy, cy.nu1, cur, false, false);
    } else if (lv.lg(b) > 1) {
        for (int s = 0; s < cy.coarse_sweeps; ++s) {
            rb_half<DIM>(x, lv.lg(b), lv.u(b, 0), lv.q(b), 0);
            rb_half<DIM>(x, lv.lg(b), lv.u(b, 0), lv.q(b), 1);
        }
    }
    for (int l = levels - 2; l >= from; --l) {
        const int c = cur;
        cur = down;
        prolong_add<DIM>(x, lv.lg(l + 1), lv.u(l + 1, c), lv.u(l, cur), cy.paper);
        relax<DIM>(x, lv, l, cy, cy.nu2, cur, true, false);
    }
    return cur;
}

// The levels of the single-CTA tail in shared memory: u, (u2 for weighted
// Jacobi), q, r of each level one after the other.
template <typename T>
struct SmemLevels {
    using Type = T;
    T* base;
    const int* off;  // element offset of each level's arrays (shared memory)
    int lg0, arrays;
    __device__ int lg(int l) const { return lg0 - l; }
    __device__ int size(int l) const { return off[l + 1] - off[l]; }
    __device__ T* u(int l, int buf) const { return base + off[l] * arrays + buf * size(l); }
    __device__ T* q(int l) const { return base + off[l] * arrays + (arrays - 2) * size(l); }
    __device__ T* r(int l) const { return base + off[l] * arrays + (arrays - 1) * size(l); }
};

// The V-cycle on levels with n = n_top, n_top/2, ..., n_top >> (levels-1).
template <int DIM, typename T>
__global__ void __launch_bounds__(1024) k_tail(T* __restrict__ u_top, const T* __restrict__ q_top,
                                               Lay top, int levels, Cycle cy, int exact0) {
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
    // f(dense node, its offset in top's layout) over the top level's rows
    auto top_nodes = [&](auto&& f) {
        const int m = n_top + 1, rows = DIM == 3 ? m * m : m;
        for (int row = threadIdx.x >> 5; row < rows; row += blockDim.x >> 5) {
            const int k = DIM == 3 ? row / m : 0, j = row - k * m;
            const int64_t g = k * top.sz + j * top.sy;
            for (int i = threadIdx.x & 31; i < m; i += 32)
                f(row * m + i, g + (top.he ? lk::xo<true>(top, i) : i));
        }
    };
    T* u0 = lv.u(0, 0);
    T* q0 = lv.q(0);
    top_nodes([&](int p, int64_t g) {
        q0[p] = q_top[g];
        u0[p] = u_top[g];
    });
    __syncthreads();
    CtaX x;
    const int cur = vcycle<DIM>(x, lv, 0, levels, cy, exact0 != 0);
    const T* ur = lv.u(0, cur);
    top_nodes([&](int p, int64_t g) { u_top[g] = ur[p]; });
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
        restrict_to<DIM>(gx, lv.lg(l + 1), lv.r(l), lv.q(l + 1), lv.u(l + 1, 0), red_only, false);
    }
    if (blockIdx.x == 0) {
        CtaX cx;
        vcycle<DIM>(cx, lv, lc, a.levels, cy, false);
    }
    gx.sync();
    for (int l = lc - 1; l >= 0; --l) {
        prolong_add<DIM>(gx, lv.lg(l + 1), lv.u(l + 1, 0), lv.u(l, 0), false);
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
                   bool exact_top, bool paper) {
    if (levels < 1 || levels > kMaxLevels) return cudaErrorInvalidValue;
    const int exact0 = exact_top && std::is_same<T, double>::value && d == 3 ? 1 : 0;
    const size_t bytes = smem_bytes(d, top.n, levels, smoother, sizeof(T));
    const Cycle cy{smoother, nu1, nu2, coarse_sweeps, paper, omega};
    // one thread per slot of the top level's sweeps (128..1024): more warps
    // only lengthen the barriers
    const int64_t nodes = d == 3 ? (int64_t)top.n * top.n * top.n : (int64_t)top.n * top.n;
    const int64_t slots = smoother == GMG_WJACOBI ? nodes : nodes / 2;
    const int threads = (int)std::min<int64_t>(1024, std::max<int64_t>(128, slots));
    auto kern = d == 3 ? k_tail<3, T> : k_tail<2, T>;
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    kern<<<1, threads, bytes, s>>>(u_top, q_top, top, levels, cy, exact0);
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
                                    int, int, int, cudaStream_t, bool, bool);
template cudaError_t launch<float>(int, const Lay&, int, float*, const float*, int, double, int,
                                   int, int, cudaStream_t, bool, bool);
template cudaError_t launch<__nv_bfloat16>(int, const Lay&, int, __nv_bfloat16*,
                                           const __nv_bfloat16*, int, double, int, int, int,
                                           cudaStream_t, bool, bool);
template cudaError_t launch<df32>(int, const Lay&, int, df32*, const df32*, int, double, int, int,
                                  int, cudaStream_t, bool, bool);

}  // namespace tail
}  // namespace gmg
