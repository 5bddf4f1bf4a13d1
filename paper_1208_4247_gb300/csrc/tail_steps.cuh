// The steps of a V-cycle on small levels (sweeps, residual, restriction,
// prolongation, the cycle itself), shared by the tail kernels: the levels' node
// slots are dealt to the threads of an executor X, which also separates the
// steps.  The arithmetic of every step is the level kernels'
// (level_kernels.cuh), node for node.
#pragma once

#include "level_kernels.cuh"

namespace gmg {
namespace tail {

using lk::Num;

constexpr int kMaxLevels = 8;       // single-CTA tail

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

// The colours (i&1) + 2(j&1) + 4(k&1) with `bits` set bits of the paper's
// Gauss-Seidel (FP64; lk::k_mc_sweep), n/2 slots per row.
template <int DIM, typename T, class X>
__device__ void mc_colors(X& x, int lg, T* u, const T* q, int bits) {
    using N = Num<T>;
    using C = typename N::C;
    const C c = DIM == 3 ? C(1.0 / 6.0) : C(0.25);
    const int n = 1 << lg;
    const int sy = n + 1, sz = DIM == 3 ? sy * sy : 0;
    for (int idx = x.tid(); idx < color_slots<DIM>(lg); idx += x.nt()) {
        const int row = idx >> (lg - 1);
        const int j = row & (n - 1), k = DIM == 3 ? row >> lg : 0;
        const int odd = bits - (j & 1) - (k & 1);
        const int i = 2 * (idx & (n / 2 - 1)) + (odd ? 1 : 2);
        if (odd < 0 || odd > 1 || i >= n || j == 0 || (DIM == 3 && k == 0)) continue;
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

// dst(e, src(e)) for e = 0 .. total-1 over the CTA's threads, the loads of
// eight elements in flight before the first store (one dependent load per row
// of a level cost the tail kernels 4 to 8 us a launch).
template <class Src, class Dst>
__device__ inline void copy_in(int total, Src&& src, Dst&& dst) {
    constexpr int U = 8;
    for (int e0 = threadIdx.x; e0 < total; e0 += U * blockDim.x) {
        decltype(src(0)) v[U];
#pragma unroll
        for (int t = 0; t < U; ++t)
            if (e0 + t * (int)blockDim.x < total) v[t] = src(e0 + t * (int)blockDim.x);
#pragma unroll
        for (int t = 0; t < U; ++t)
            if (e0 + t * (int)blockDim.x < total) dst(e0 + t * (int)blockDim.x, v[t]);
    }
}

// What the steps of one V-cycle share.
struct Cycle {
    int smoother, nu1, nu2, coarse_sweeps;
    bool paper;  // the paper's transfers
    double omega;
};

// `sweeps` sweeps on level l of lv; cur: which u buffer holds the iterate
// (weighted Jacobi alternates).  first_done: the first step (CoarseInit) ran
// already.
template <int DIM, class X, class LV>
__device__ void relax(X& x, const LV& lv, int l, const Cycle& cy, int sweeps, int& cur,
                      bool backward, bool exact_last, bool first_done = false) {
    const int lg = lv.lg(l);
    for (int s = 0; s < sweeps; ++s) {
        const bool first = first_done && s == 0;
        if (cy.smoother == GMG_WJACOBI) {
            if (first) continue;
            wj_sweep<DIM>(x, lg, lv.u(l, cur), lv.u(l, cur ^ 1), lv.q(l), cy.omega);
            cur ^= 1;
            continue;
        }
        if constexpr (std::is_same<typename LV::Type, double>::value) {
            if (cy.smoother == GMG_MCGS) {
                for (int t = first ? 1 : 0; t <= DIM; ++t)
                    mc_colors<DIM>(x, lg, lv.u(l, cur), lv.q(l), backward ? DIM - t : t);
                continue;
            }
        }
        for (int color = first ? 1 : 0; color < 2; ++color)
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

// 4 FW of sigma in 3D at the fine node whose neighbour at offset o is R(o).
template <typename C, class RF>
__device__ inline C fw3(RF&& R, int sy, int sz, bool red_only) {
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
    if (red_only) return fma(C(0.125), e, C(0.5) * R(0));
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
    return fma(C(0.0625), co, fma(C(0.125), e, fma(C(0.25), fc, C(0.5) * R(0))));
}

// fine level lg + 1 -> coarse level lg
template <int DIM, typename T, class X>
__device__ void restrict_to(X& x, int lg, const T* r, T* qc, T* uc, bool red_only, bool paper,
                            int init, double omega) {
    using N = Num<T>;
    using C = typename N::C;
    const int sy = (2 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
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
            v = fw3<C>(R, sy, sz, red_only);
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
        uc[P] = lk::coarse_init<DIM>(init, omega, I, J, K, N::st(v));
    }
    x.sync();
}

// coarse level lg -> fine level lg + 1.  black: the black fine nodes only (a
// red half sweep follows).  Every fine operand is loaded before the first
// store.
template <int DIM, typename T, class X>
__device__ void prolong_add(X& x, int lg, const T* uc, T* u, bool paper, bool black) {
    using N = Num<T>;
    using C = typename N::C;
    const int nc = 1 << lg;
    const int sy = (2 << lg) + 1, sz = DIM == 3 ? sy * sy : 0;
    const int cy = nc + 1, cz = DIM == 3 ? cy * cy : 0;
    for (int cell = x.tid(); cell < interior_slots<DIM>(lg); cell += x.nt()) {
        const int I = cell & (nc - 1), J = (cell >> lg) & (nc - 1), K = DIM == 3 ? cell >> (2 * lg) : 0;
        const int P = K * cz + J * cy + I;
        const int p = 2 * K * sz + 2 * J * sy + 2 * I;
        constexpr int V = DIM == 3 ? 8 : 4;
        // fine node 2(I,J,K) + (v & 1, v >> 1 & 1, v >> 2): interior, and
        // corrected here?
        auto on = [&](int v) {
            const bool odd = (v & 1) ^ (v >> 1 & 1) ^ (v >> 2);
            return ((v & 1) || I > 0) && ((v & 2) || J > 0) && (DIM == 2 || (v & 4) || K > 0) &&
                   (odd || !black);
        };
        auto off = [&](int v) { return (v & 1) + ((v >> 1) & 1) * sy + (v >> 2) * sz; };
        C f[V];
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (on(v)) f[v] = N::ld(u[p + off(v)]);
        const C c000 = N::ld(uc[P]), c100 = N::ld(uc[P + 1]), c010 = N::ld(uc[P + cy]),
                c110 = N::ld(uc[P + 1 + cy]);
        auto add = [&](int v, C w, C s) {
            if (on(v)) u[p + off(v)] = N::st(fma(w, s, f[v]));
        };
        if (std::is_same<T, double>::value && paper) {
            if (on(0)) u[p] = N::st(f[0] + c000);
            add(1, C(0.5), c000 + c100);
            add(2, C(0.5), c000 + c010);
            add(3, C(0.5), c000 + c110);
            if constexpr (DIM == 3) {
                const C c001 = N::ld(uc[P + cz]), c101 = N::ld(uc[P + 1 + cz]),
                        c011 = N::ld(uc[P + cy + cz]), c111 = N::ld(uc[P + 1 + cy + cz]);
                add(4, C(0.5), c000 + c001);
                add(5, C(0.5), c000 + c101);
                add(6, C(0.5), c000 + c011);
                add(7, C(0.5), c000 + c111);
            }
            continue;
        }
        const C x00 = c000 + c100;
        const C y00 = c000 + c010;
        if (on(0)) u[p] = N::st(f[0] + c000);
        add(1, C(0.5), x00);
        add(2, C(0.5), y00);
        if constexpr (DIM == 2) {
            add(3, C(0.25), x00 + (c010 + c110));
        } else {
            const C qxy = x00 + (c010 + c110);
            const C c001 = N::ld(uc[P + cz]), c101 = N::ld(uc[P + 1 + cz]),
                    c011 = N::ld(uc[P + cy + cz]), c111 = N::ld(uc[P + 1 + cy + cz]);
            const C x01 = c001 + c101;
            add(3, C(0.25), qxy);
            add(4, C(0.5), c000 + c001);
            if (!black) {
                add(5, C(0.25), x00 + x01);
                add(6, C(0.25), y00 + (c001 + c011));
            }
            add(7, C(0.125), qxy + (x01 + (c011 + c111)));
        }
    }
    x.sync();
}

// The V-cycle on levels from .. levels-1 of lv (level `from` given: q set, u =
// 0 or a start), run by x: down (pre-smoothing, residual, restriction), the
// coarsest grid, up (prolongation with correction, post-smoothing).  Returns
// the u buffer of level `from` that holds the result.
// exact0: level `from` is level 0 of a plain FP64 3D hierarchy (unbiased value).
// first_done: the first smoothing step of level `from` ran already.
template <int DIM, class X, class LV>
__device__ int vcycle(X& x, const LV& lv, int from, int levels, const Cycle& cy, bool exact0,
                      bool first_done) {
    // (a learned handle's tail levels smooth with red-black Gauss-Seidel)
    const bool red_black = cy.smoother == GMG_RBGS || cy.smoother == GMG_LEARNED;
    const bool red_only = red_black && cy.nu1 > 0 && !cy.paper;
    // a red half sweep follows the prolongation
    const bool black = red_black && cy.nu2 > 0;
    // every level but the coarsest gets its first smoothing step from the
    // restriction
    const int init = cy.nu1 == 0                    ? INIT_ZERO
                     : cy.smoother == GMG_WJACOBI ? INIT_WJ
                     : cy.smoother == GMG_MCGS    ? INIT_COLOR0
                                                    : INIT_RED;
    // down: u buffer of each level after its pre-smoothing (bit l; weighted
    // Jacobi), which the correction goes into
    unsigned down = 0;
    for (int l = from; l + 1 < levels; ++l) {
        int c = 0;
        const bool first = l == from ? first_done : init != INIT_ZERO;
        relax<DIM>(x, lv, l, cy, cy.nu1, c, false, exact0 && l == from, first);
        down |= (unsigned)c << l;
        residual<DIM>(x, lv.lg(l), lv.u(l, c), lv.q(l), lv.r(l), red_only, exact0 && l == from);
        const int lgc = lv.lg(l + 1);
        restrict_to<DIM>(x, lgc, lv.r(l), lv.q(l + 1), lv.u(l + 1, 0), red_only, cy.paper,
                         l + 2 < levels ? init : lgc == 1 ? INIT_EXACT : INIT_ZERO, cy.omega);
    }
    const int b = levels - 1;
    int cur = 0;
    if (levels - from == 1) {
        relax<DIM>(x, lv, b, cy, cy.nu1, cur, false, false, first_done);
    } else if (lv.lg(b) > 1) {
        for (int s = 0; s < cy.coarse_sweeps; ++s) {
            rb_half<DIM>(x, lv.lg(b), lv.u(b, 0), lv.q(b), 0);
            rb_half<DIM>(x, lv.lg(b), lv.u(b, 0), lv.q(b), 1);
        }
    }
    for (int l = levels - 2; l >= from; --l) {
        const int c = cur;
        cur = (down >> l) & 1;
        prolong_add<DIM>(x, lv.lg(l + 1), lv.u(l + 1, c), lv.u(l, cur), cy.paper, black);
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

}  // namespace tail
}  // namespace gmg
