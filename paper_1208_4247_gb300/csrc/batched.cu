// Batched form: many independent Poisson solves of uneven sizes (2D and 3D
// mixed) advanced together, FP32 or BF16-storage cycles inside FP64
// iterative refinement.
//
// Levels are aligned at the coarsest 3^d grid: level step g processes, for
// every solve with at least g+1 grids, its level L_s - 1 - g, of n = 2^(g+1)
// intervals.  The small solves' fine levels thus share launches with the large
// solves' coarse levels.  A step of the weighted-Jacobi cycle is a leg down and
// a leg up over tiles of all its levels; the 2D and the 3D solves' launches are
// two branches of the graph.  The other operations take work items that are
// chunks of one solve's level grid (interior nodes or coarse cells), the CTAs
// striding over them.  Tiles and items of converged solves are skipped
// (per-solve active flags, written only by the step's final kernel).
// One refinement step of the whole batch is captured into one CUDA graph;
// the host reads one counter (solves still active) per step.
#include <algorithm>
#include <climits>
#include <cmath>
#include <string>
#include <vector>

#include "batch_tiles.h"
#include "gmg_internal.cuh"
#include "level_kernels.cuh"
#include "timing.cuh"

namespace gmg {
namespace batch {

using lk::fastdiv;
using lk::FastDiv;
using lk::fastdiv_make;

struct BLevel {
    int d, n;
    int64_t u0, u1, q;  // element offsets into the inner pool (-1: none)
    int64_t sy, sz;     // inner pool row / plane pitch
    int lgG;            // log2 of the 16-byte groups per row the vector kernels take
    FastDiv rows;       // division by n - 1 (interior nodes per row)
};
struct BSolve {
    int d, n, levels, lev0;  // lev0: index of level 0 in the level table
    int64_t q64;             // offset of the FP64 scaled right-hand side
    int item0, item1;        // its items in the level-0 item list
    const double* f;
    double* u;
};
struct Item {
    int solve, level;
    int64_t start;
    int count;
};

using lk::Num;

// Node (i, j, k) of interior index idx (x fastest over the (n-1)^d interior
// nodes of level L) and its offset in the level's inner-pool array; no
// integer division (interior counts stay below 2^32).
__device__ inline int64_t node_of(const BLevel& L, uint32_t idx, int& i, int& j, int& k) {
    const uint32_t m = L.rows.d;
    const uint32_t t = fastdiv(idx, L.rows);
    i = (int)(idx - t * m) + 1;
    if (L.d == 3) {
        const uint32_t kk = fastdiv(t, L.rows);
        j = (int)(t - kk * m) + 1;
        k = (int)kk + 1;
    } else {
        j = (int)t + 1;
        k = 0;
    }
    return (int64_t)k * L.sz + (int64_t)j * L.sy + i;
}
// offset of node (i, j, k) in the solve's dense FP64 arrays
__device__ inline int64_t dense_of(const BLevel& L, int i, int j, int k) {
    return ((int64_t)k * (L.n + 1) + j) * (L.n + 1) + i;
}
__device__ inline int64_t node_of(const BLevel& L, uint32_t idx) {
    int i, j, k;
    return node_of(L, idx, i, j, k);
}

__device__ inline int64_t off_u(const BLevel& L, int which) { return which ? L.u1 : L.u0; }

// V = 16 bytes of inner-pool values (4 FP32, 8 BF16) as floats, and back
template <typename T>
__device__ inline void ldv(const T* p, float* v);
template <>
__device__ inline void ldv<float>(const float* p, float* v) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
template <>
__device__ inline void ldv<__nv_bfloat16>(const __nv_bfloat16* p, float* v) {
    const uint4 a = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&w[h]);
        v[2 * h] = __low2float(b);
        v[2 * h + 1] = __high2float(b);
    }
}
template <typename T>
__device__ inline void stv(T* p, const float* v);
template <>
__device__ inline void stv<float>(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ inline void stv<__nv_bfloat16>(__nv_bfloat16* p, const float* v) {
    uint32_t w[4];
#pragma unroll
    for (int h = 0; h < 4; ++h)
        *reinterpret_cast<__nv_bfloat162*>(&w[h]) = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Vector items: index gid over (interior row) x (16-byte group of the row),
// 2^lgG groups per row (x = V g .. V g + V - 1 covers 0 .. n - 1); the group's
// offset in the level's inner-pool array and its first x.
template <int V>
__device__ inline int64_t group_of(const BLevel& L, uint32_t gid, int& x0, int& j, int& k) {
    const uint32_t row = gid >> L.lgG;
    x0 = V * (int)(gid & ((1u << L.lgG) - 1u));
    if (L.d == 3) {
        const uint32_t m = L.rows.d;
        const uint32_t kk = fastdiv(row, L.rows);
        j = (int)(row - kk * m) + 1;
        k = (int)kk + 1;
    } else {
        j = (int)row + 1;
        k = 0;
    }
    return (int64_t)k * L.sz + (int64_t)j * L.sy + x0;
}

// Smoothing sweep over the items' groups: weighted Jacobi (src -> dst) or one
// colour of red-black Gauss-Seidel (in place, src == dst; the group's other
// nodes are written back unchanged, and no other thread writes them).  Per
// group: one 16-byte load each of the row, its y and z neighbour rows and q,
// the two x neighbours beyond the group as single loads, one 16-byte store;
// nodes outside 1..n-1 are written as 0 (Jacobi) or left unchanged.  zero: bit
// 0 / 1: the source is zero on the solves' finest level / coarser levels and is
// not read (Jacobi).  The
// neighbour sum is ((x- + x+) + y- + y+) + z- + z+ in this order.  pool_in and pool_out are the
// same pool: what a launch reads through pool_in is never written during the
// launch (the Jacobi source, q; in red-black the other colour).
template <typename T>
__global__ void __launch_bounds__(256) k_smooth(const Item* __restrict__ items, int nitems,
                                                const BSolve* __restrict__ sv,
                                                const BLevel* __restrict__ lv,
                                                const T* __restrict__ pool_in,
                                                T* __restrict__ pool_out,
                                                const int* __restrict__ active, int src, int dst,
                                                int color, int zero, float omega2, float omega3) {
    constexpr int V = 16 / (int)sizeof(T);
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        if (!active[w.solve]) continue;
        const BLevel L = lv[sv[w.solve].lev0 + w.level];
        const bool three = L.d == 3;
        const float c = three ? 1.f / 6.f : 0.25f;
        const float omega = three ? omega3 : omega2;
        const bool zs = (zero >> (w.level > 0)) & 1;
        const T* u = pool_in + off_u(L, src);
        T* uo = pool_out + off_u(L, dst);
        const T* q = pool_in + L.q;
        for (int t = threadIdx.x; t < w.count; t += blockDim.x) {
            int x0, j, k;
            const int64_t p = group_of<V>(L, (uint32_t)(w.start + t), x0, j, k);
            float x[V] = {}, ym[V] = {}, yp[V] = {}, zm[V] = {}, zp[V] = {}, qv[V], out[V];
            float xl = 0.f, xr = 0.f;
            if (!zs) {
                ldv(u + p, x);
                xl = Num<T>::ld(u[p - 1]);
                xr = Num<T>::ld(u[p + V]);
                ldv(u + p - L.sy, ym);
                ldv(u + p + L.sy, yp);
                if (three) {
                    ldv(u + p - L.sz, zm);
                    ldv(u + p + L.sz, zp);
                }
            }
            ldv(q + p, qv);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float s = (v > 0 ? x[v - 1] : xl) + (v < V - 1 ? x[v + 1] : xr);
                s += ym[v];
                s += yp[v];
                if (three) {
                    s += zm[v];
                    s += zp[v];
                }
                const float g = fmaf(c, s, qv[v]);
                const int xi = x0 + v;
                const bool in = xi >= 1 && xi <= L.n - 1;
                if (color >= 0)
                    out[v] = in && ((xi + j + k) & 1) == color ? g : x[v];
                else
                    out[v] = in ? fmaf(omega, g - x[v], x[v]) : 0.f;
            }
            stv(uo + p, out);
        }
    }
}

// ----------------------------------------------------------------- legs
// One kernel takes a level down (last pre-smoothing sweep, residual, full
// weighting) and one takes it up (prolongation, first post-smoothing sweep):
// each reads u and q once and writes u once, 12.5 bytes per FP32 node and leg;
// a kernel per operation moved 29 down and 20.5 up.  The 512-solve batch's step
// g = 6 (70 solves of 129^3 among them) took 326 + 326 + 261 us down and 251 +
// 326 us up that way and takes 432 and 408 us now (both dimensions, one after
// the other), 60% of a copy's rate: at one CTA per SM a plane's loads are in flight
// for two steps (540 and 412 us with one step, 96 registers and 38 rows a tile; 32
// rows now, 126 registers).  g = 9 (59 of 1025^2) 141 + 140 + 100 and 142 + 141 us, now 146 and 147,
// 80% of a copy's rate; the batch 121.1 -> 70.0 ms.
//
// A thread owns 4 nodes of x (one vector) and, in 3D, two rows of y, and
// walks z (2D: y) with the planes it still needs in registers; x neighbours
// come from the neighbour lanes by shuffles, y neighbours inside the pair of
// rows from its own registers and across pairs from shared memory (5 vectors
// per thread and plane, double buffered, so one barrier per plane).  A row of
// up to 128 nodes is at most a warp wide; wider rows are cut into pieces of 30
// groups with one halo group on each side.  In 3D the CTA is as wide as the
// rows of a tile ask for; in 2D nothing is shared and every warp (n < 128:
// part of a warp) walks alone.
//
// Per node and direction the neighbour sum runs ahead of the sweep: P(s) =
// ((x- + x+) + y- + y+) + z- of plane s is formed when plane s arrives, z+ is
// added when the next one does, so that a plane is kept as P and its centre
// values only.  The order of the additions is that of k_smooth, and r and the
// prolonged u are rounded to the storage type, so each result has the bits the
// separate kernels gave.

constexpr int kHaloLanes = 30;  // groups a warp keeps of a row wider than 32 groups

struct Tile {
    int solve, level;
    int g0;      // first lane's group (-1 mod 30 for rows wider than a warp)
    int y0;      // 3D: first row of the tile; even
    int ja, jb;  // down: coarse rows; up: fine rows [ja, jb) written
    int ka, kb;  // 3D: the same in z (2D: unused)
};

template <typename T>
__device__ inline void ld4(const T* p, bool ok, float* v);
template <>
__device__ inline void ld4<float>(const float* p, bool ok, float* v) {
    const float4 a = ok ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
template <>
__device__ inline void ld4<__nv_bfloat16>(const __nv_bfloat16* p, bool ok, float* v) {
    const uint2 a = ok ? __ldg(reinterpret_cast<const uint2*>(p)) : make_uint2(0u, 0u);
    v[0] = __uint_as_float(a.x << 16);
    v[1] = __uint_as_float(a.x & 0xffff0000u);
    v[2] = __uint_as_float(a.y << 16);
    v[3] = __uint_as_float(a.y & 0xffff0000u);
}
__device__ inline void st4(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ inline void st4(__nv_bfloat16* p, const float* v) {
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) =
        make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}
__device__ inline void st2(float* p, float a, float b) {
    *reinterpret_cast<float2*>(p) = make_float2(a, b);
}
__device__ inline void st2(__nv_bfloat16* p, float a, float b) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
__device__ inline float2 ld2(const float* p, bool ok) {
    return ok ? __ldg(reinterpret_cast<const float2*>(p)) : make_float2(0.f, 0.f);
}
__device__ inline float2 ld2(const __nv_bfloat16* p, bool ok) {
    const uint32_t a = ok ? __ldg(reinterpret_cast<const uint32_t*>(p)) : 0u;
    return make_float2(__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u));
}
template <typename T>
__device__ inline float rnd(float v) {
    return Num<T>::ld(Num<T>::st(v));
}

// x- + x+ of the lane's 4 nodes (lanes: the width of a row in the warp); past
// the last lane lies the boundary, or a value no kept node uses
__device__ inline void xsum(const float* x, int lanes, bool last, float* s) {
    const float l = __shfl_up_sync(0xffffffffu, x[3], 1, lanes);
    float r = __shfl_down_sync(0xffffffffu, x[0], 1, lanes);
    if (last) r = 0.f;
    s[0] = l + x[1];
    s[1] = x[0] + x[2];
    s[2] = x[1] + x[3];
    s[3] = x[2] + r;
}

__device__ inline void get4(const float4* p, bool ok, float* v) {
    const float4 a = ok ? *p : make_float4(0.f, 0.f, 0.f, 0.f);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
__device__ inline void put4(float4* p, const float* v) { *p = make_float4(v[0], v[1], v[2], v[3]); }

// the coarse nodes 2g and 2g + 1 take row values r (l = the value left of the
// lane's first) with weight w at dx = 0
__device__ inline void fw_row(float* acc, float l, const float* r, float w) {
    const float h = 0.5f * w;
    acc[0] = fmaf(h, l, acc[0]);
    acc[0] = fmaf(w, r[0], acc[0]);
    acc[0] = fmaf(h, r[1], acc[0]);
    acc[1] = fmaf(h, r[1], acc[1]);
    acc[1] = fmaf(w, r[2], acc[1]);
    acc[1] = fmaf(h, r[3], acc[1]);
}

// SWEEP: u1 = weighted-Jacobi step of u0 (buffer src), written to buffer dst,
// then the residual of u1 and its restriction; otherwise the residual and
// restriction of u0 alone.  zero: bit 0 / 1: u0 is zero on the solve's finest
// level / on its coarser levels and is not read.  clear: write u_c = 0 (the
// coarse level reads it); the one unknown of an n = 2 grid gets u_c = q_c.
template <typename T, bool SWEEP>
__global__ void __launch_bounds__(kLegThreads, 1)
    k_down3(const Tile* __restrict__ tiles, int ntiles, const BSolve* __restrict__ sv,
            const BLevel* __restrict__ lv, const T* __restrict__ pool_in, T* __restrict__ pool_out,
            const int* __restrict__ active, int src, int dst, int zero, int clear, float omega) {
    extern __shared__ float4 edge[];  // [2][u0 row 0, u0 row 1, u1 row 0, u1 row 1, r row 1][thread]
    const int nt = blockDim.x, tid = threadIdx.x;
    const float c = 1.f / 6.f;
    int buf = 0;
    for (int it = blockIdx.x; it < ntiles; it += gridDim.x) {
        const Tile t = tiles[it];
        if (!active[t.solve]) continue;
        const BLevel F = lv[sv[t.solve].lev0 + t.level];
        const BLevel C = lv[sv[t.solve].lev0 + t.level + 1];
        const int n = F.n, G = n >> 2, lanes = min(G, 32), lg = __ffs(lanes) - 1;
        const int gx = tid & (lanes - 1), pair = tid >> lg, pairs = nt >> lg;
        const int g = t.g0 + gx, y = t.y0 + 2 * pair;
        const bool gok = g >= 0 && g < G, last = gx == lanes - 1;
        const bool core = gok && (G <= 32 || (gx >= 1 && gx <= kHaloLanes));
        const bool in0 = gok && y >= 1 && y < n, in1 = gok && y + 1 >= 1 && y + 1 < n;
        const bool zs = SWEEP && ((zero >> (t.level > 0)) & 1);
        const int jl = 2 * t.jb - 2 + (t.jb == n / 2);  // last fine row the tile writes
        const int kl = 2 * t.kb - 2 + (t.kb == n / 2);
        const bool w0 = core && in0 && y >= 2 * t.ja - 1 && y <= jl;
        const bool w1 = core && in1 && y + 1 >= 2 * t.ja - 1 && y + 1 <= jl;
        const bool wc = core && y >= 2 * t.ja && y < 2 * t.jb;
        const int64_t o = (int64_t)y * F.sy + 4 * g;
        const T* u = pool_in + off_u(F, src) + o;
        const T* q = pool_in + F.q + o;
        T* uo = pool_out + off_u(F, dst) + o;
        const int64_t oc = (int64_t)(y >> 1) * C.sy + 2 * g;
        float uc[2][4], un[2][4], vc[2][4] = {}, P0[2][4] = {}, P1[2][4] = {}, qo[2][4] = {},
                                               qc[2][4] = {}, acc[2] = {};
        auto load = [&](const T* a, int z, bool ok, float (*v)[4]) {
            ok = ok && z >= 1 && z < n;
            ld4(a + (int64_t)z * F.sz, ok && in0, v[0]);
            ld4(a + (int64_t)z * F.sz + F.sy, ok && in1, v[1]);
        };
        const int s0 = 2 * t.ka - (SWEEP ? 3 : 2), s1 = 2 * t.kb;
        float u2[2][4], qn[2][4];
        load(u, s0, !zs, uc);
        load(u, s0 + 1, !zs, un);
        load(u, s0 + 2, !zs, u2);
        if (!SWEEP) load(q, s0, true, qc);
        load(q, s0 + 1, true, qn);
        for (int s = s0; s <= s1; ++s) {
            // two steps ahead of their use
            float u3[2][4], q2[2][4], v[2][4], r[2][4];
            load(u, s + 3, !zs && s + 1 < s1, u3);
            load(q, s + 2, s + 1 < s1, q2);
            const bool zin = s >= 1 && s < n;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool in = zin && (h ? in1 : in0);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (SWEEP) {
                        const float gs = fmaf(c, P0[h][e] + un[h][e], qc[h][e]);
                        const float w = rnd<T>(fmaf(omega, gs - uc[h][e], uc[h][e]));
                        v[h][e] = in && !(e == 0 && g == 0) ? w : 0.f;
                    } else {
                        v[h][e] = uc[h][e];
                    }
                }
            }
            if (SWEEP && s >= 2 * t.ka - 1 && s <= kl) {
                if (w0) st4(uo + (int64_t)s * F.sz, v[0]);
                if (w1) st4(uo + (int64_t)s * F.sz + F.sy, v[1]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    r[h][e] = rnd<T>(fmaf(c, P1[h][e] + v[h][e], qo[h][e]) - vc[h][e]);
            float4* E = edge + buf * 5 * nt + tid;
            if (SWEEP && !zs) {
                put4(E, un[0]);
                put4(E + nt, un[1]);
            }
            put4(E + 2 * nt, v[0]);
            put4(E + 3 * nt, v[1]);
            put4(E + 4 * nt, r[1]);
            __syncthreads();
            const bool up = pair > 0, dn = pair + 1 < pairs;
            float a[4], b[4], x[4];
            if (SWEEP && !zs) {
                get4(E + nt - lanes, up, a);
                get4(E + lanes, dn, b);
                xsum(un[0], lanes, last, x);
#pragma unroll
                for (int e = 0; e < 4; ++e) P0[0][e] = ((x[e] + a[e]) + un[1][e]) + uc[0][e];
                xsum(un[1], lanes, last, x);
#pragma unroll
                for (int e = 0; e < 4; ++e) P0[1][e] = ((x[e] + un[0][e]) + b[e]) + uc[1][e];
            }
            get4(E + 3 * nt - lanes, up, a);
            get4(E + 2 * nt + lanes, dn, b);
            xsum(v[0], lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P1[0][e] = ((x[e] + a[e]) + v[1][e]) + vc[0][e];
            xsum(v[1], lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P1[1][e] = ((x[e] + v[0][e]) + b[e]) + vc[1][e];
            // plane s - 1 of r: dz = 0 of a coarse plane, or dz = +1 of one and -1 of the next
            get4(E + 4 * nt - lanes, up, a);
            const float la = __shfl_up_sync(0xffffffffu, a[3], 1, lanes),
                        l0 = __shfl_up_sync(0xffffffffu, r[0][3], 1, lanes),
                        l1 = __shfl_up_sync(0xffffffffu, r[1][3], 1, lanes);
            if (s & 1) {
                fw_row(acc, la, a, 0.25f);
                fw_row(acc, l0, r[0], 0.5f);
                fw_row(acc, l1, r[1], 0.25f);
            } else {
                fw_row(acc, la, a, 0.125f);
                fw_row(acc, l0, r[0], 0.25f);
                fw_row(acc, l1, r[1], 0.125f);
                const int K = (s >> 1) - 1;
                if (wc && K >= t.ka) {
                    const int64_t P = (int64_t)K * C.sz + oc;
                    if (g == 0) acc[0] = 0.f;
                    st2(pool_out + C.q + P, acc[0], acc[1]);
                    if (C.n == 2)
                        st2(pool_out + C.u0 + P, acc[0], acc[1]);
                    else if (clear)
                        st2(pool_out + C.u0 + P, 0.f, 0.f);
                }
                acc[0] = acc[1] = 0.f;
                fw_row(acc, la, a, 0.125f);
                fw_row(acc, l0, r[0], 0.25f);
                fw_row(acc, l1, r[1], 0.125f);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    uc[h][e] = un[h][e];
                    un[h][e] = u2[h][e];
                    u2[h][e] = u3[h][e];
                    vc[h][e] = v[h][e];
                    qo[h][e] = qc[h][e];
                    qc[h][e] = qn[h][e];
                    qn[h][e] = q2[h][e];
                }
            buf ^= 1;
        }
    }
}
// the same in 2D: a warp (or part of one) walks y by itself
template <typename T, bool SWEEP>
__global__ void __launch_bounds__(128)
    k_down2(const Tile* __restrict__ tiles, int ntiles, const BSolve* __restrict__ sv,
            const BLevel* __restrict__ lv, const T* __restrict__ pool_in, T* __restrict__ pool_out,
            const int* __restrict__ active, int src, int dst, int zero, int clear, float omega,
            int lanes) {
    const int lane = threadIdx.x & 31, gx = lane & (lanes - 1), per = 32 / lanes;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
              nw = (gridDim.x * blockDim.x) >> 5;
    const float c = 0.25f;
    const bool last = gx == lanes - 1;
    for (int first = wid * per; first < ntiles; first += nw * per) {
        const int it = first + lane / lanes;
        const Tile t = tiles[min(it, ntiles - 1)];
        const bool on = it < ntiles && active[t.solve] != 0;
        const BLevel F = lv[sv[t.solve].lev0 + t.level];
        const BLevel C = lv[sv[t.solve].lev0 + t.level + 1];
        const int n = F.n, G = n >> 2, g = t.g0 + gx;
        const bool gok = on && g >= 0 && g < G;
        const bool core = gok && (G <= 32 || (gx >= 1 && gx <= kHaloLanes));
        const bool uok = gok && !(SWEEP && ((zero >> (t.level > 0)) & 1));
        const int s0 = 2 * t.ja - (SWEEP ? 3 : 2), s1 = 2 * t.jb;
        const int jl = 2 * t.jb - 2 + (t.jb == n / 2);
        const int steps = __reduce_max_sync(0xffffffffu, on ? s1 - s0 + 1 : 0);
        const T* u = pool_in + off_u(F, src) + 4 * g;
        const T* q = pool_in + F.q + 4 * g;
        T* uo = pool_out + off_u(F, dst) + 4 * g;
        float uc[4], un[4], qc[4] = {}, qo[4] = {}, vc[4] = {}, P0[4] = {}, P1[4] = {}, acc[2] = {};
        auto load = [&](const T* a, int y, bool ok, float* v) {
            ld4(a + (int64_t)y * F.sy, ok && y >= 1 && y < n, v);
        };
        load(u, s0, uok, uc);
        load(u, s0 + 1, uok, un);
        if (!SWEEP) load(q, s0, gok, qc);
        for (int i = 0; i < steps; ++i) {
            const int s = s0 + i;
            float u2[4], qn[4], v[4], r[4], x[4];
            load(u, s + 2, uok && s < s1, u2);
            load(q, s + 1, gok && s < s1, qn);
            const bool in = gok && s >= 1 && s < n;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (SWEEP) {
                    const float gs = fmaf(c, P0[e] + un[e], qc[e]);
                    const float w = rnd<T>(fmaf(omega, gs - uc[e], uc[e]));
                    v[e] = in && !(e == 0 && g == 0) ? w : 0.f;
                } else {
                    v[e] = uc[e];
                }
                r[e] = rnd<T>(fmaf(c, P1[e] + v[e], qo[e]) - vc[e]);
            }
            if (SWEEP && core && s >= 2 * t.ja - 1 && s <= jl) st4(uo + (int64_t)s * F.sy, v);
            if (SWEEP) {
                xsum(un, lanes, last, x);
#pragma unroll
                for (int e = 0; e < 4; ++e) P0[e] = x[e] + uc[e];
            }
            xsum(v, lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P1[e] = x[e] + vc[e];
            const float l = __shfl_up_sync(0xffffffffu, r[3], 1, lanes);
            if (s & 1) {  // row s - 1 even: dy = 0
                fw_row(acc, l, r, 1.f);
            } else {
                fw_row(acc, l, r, 0.5f);
                const int J = (s >> 1) - 1;
                if (core && J >= t.ja && J < t.jb) {
                    const int64_t P = (int64_t)J * C.sy + 2 * g;
                    if (g == 0) acc[0] = 0.f;
                    st2(pool_out + C.q + P, acc[0], acc[1]);
                    if (C.n == 2)
                        st2(pool_out + C.u0 + P, acc[0], acc[1]);
                    else if (clear)
                        st2(pool_out + C.u0 + P, 0.f, 0.f);
                }
                acc[0] = acc[1] = 0.f;
                fw_row(acc, l, r, 0.5f);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uc[e] = un[e];
                un[e] = u2[e];
                vc[e] = v[e];
                qo[e] = qc[e];
                qc[e] = qn[e];
            }
        }
    }
}

// the three coarse values of a row between which a lane's 4 fine nodes lie
__device__ inline void widen3(float2 a, int lanes, bool last, float* c) {
    c[0] = a.x;
    c[1] = a.y;
    c[2] = __shfl_down_sync(0xffffffffu, a.x, 1, lanes);
    if (last) c[2] = 0.f;
}

// dst = weighted-Jacobi step of u + P u_c (u in buffer src, u_c in buffer
// ccur).  The corners a fine node lies between are added in k_prolong's order
// (x, then y, then z), so the plane above is added value by value.
template <typename T>
__global__ void __launch_bounds__(kLegThreads, 1)
    k_up3(const Tile* __restrict__ tiles, int ntiles, const BSolve* __restrict__ sv,
          const BLevel* __restrict__ lv, const T* __restrict__ pool_in, T* __restrict__ pool_out,
          const int* __restrict__ active, int src, int dst, int ccur, float omega) {
    extern __shared__ float4 edge[];  // [2][row 0, row 1][thread]
    const int nt = blockDim.x, tid = threadIdx.x;
    const float c = 1.f / 6.f;
    int buf = 0;
    for (int it = blockIdx.x; it < ntiles; it += gridDim.x) {
        const Tile t = tiles[it];
        if (!active[t.solve]) continue;
        const BLevel F = lv[sv[t.solve].lev0 + t.level];
        const BLevel C = lv[sv[t.solve].lev0 + t.level + 1];
        const int n = F.n, G = n >> 2, lanes = min(G, 32), lg = __ffs(lanes) - 1;
        const int gx = tid & (lanes - 1), pair = tid >> lg, pairs = nt >> lg;
        const int g = t.g0 + gx, y = t.y0 + 2 * pair;
        const bool gok = g >= 0 && g < G, last = gx == lanes - 1;
        const bool core = gok && (G <= 32 || (gx >= 1 && gx <= kHaloLanes));
        const bool in0 = gok && y >= 1 && y < n, in1 = gok && y + 1 < n;
        const bool w0 = core && in0 && y >= t.ja && y < t.jb;
        const bool w1 = core && in1 && y + 1 >= t.ja && y + 1 < t.jb;
        const int64_t o = (int64_t)y * F.sy + 4 * g;
        const T* u = pool_in + off_u(F, src) + o;
        const T* q = pool_in + F.q + o;
        T* uo = pool_out + off_u(F, dst) + o;
        const bool cok = gok && y < n;
        const T* uk = pool_in + off_u(C, ccur) + (int64_t)(y >> 1) * C.sy + 2 * g;
        auto load = [&](const T* a, int z, bool ok, float (*v)[4]) {
            ok = ok && z >= 1 && z < n;
            ld4(a + (int64_t)z * F.sz, ok && in0, v[0]);
            ld4(a + (int64_t)z * F.sz + F.sy, ok && in1, v[1]);
        };
        float2 raw[2];
        auto cload = [&](int K) {
            const bool ok = cok && K < C.n;
            raw[0] = ld2(uk + (int64_t)K * C.sz, ok);
            raw[1] = ld2(uk + (int64_t)K * C.sz + C.sy, ok);
        };
        float ca[2][3] = {}, un[2][4], wc[2][4], P[2][4] = {}, qc[2][4] = {};
        // w = u + P u_c on plane z (planes in order: ca = coarse plane z / 2)
        auto correct = [&](int z, float (*v)[4]) {
            float m[2][4];
            m[0][0] = ca[0][0];
            m[0][1] = ca[0][0] + ca[0][1];
            m[0][2] = ca[0][1];
            m[0][3] = ca[0][1] + ca[0][2];
            m[1][0] = ca[0][0] + ca[1][0];
            m[1][1] = (m[0][1] + ca[1][0]) + ca[1][1];
            m[1][2] = ca[0][1] + ca[1][1];
            m[1][3] = (m[0][3] + ca[1][1]) + ca[1][2];
            float w = 1.f;
            if (z & 1) {
                float cb[2][3];
                widen3(raw[0], lanes, last, cb[0]);
                widen3(raw[1], lanes, last, cb[1]);
                m[0][0] += cb[0][0];
                m[0][1] = (m[0][1] + cb[0][0]) + cb[0][1];
                m[0][2] += cb[0][1];
                m[0][3] = (m[0][3] + cb[0][1]) + cb[0][2];
                m[1][0] = (m[1][0] + cb[0][0]) + cb[1][0];
                m[1][1] = (((m[1][1] + cb[0][0]) + cb[0][1]) + cb[1][0]) + cb[1][1];
                m[1][2] = (m[1][2] + cb[0][1]) + cb[1][1];
                m[1][3] = (((m[1][3] + cb[0][1]) + cb[0][2]) + cb[1][1]) + cb[1][2];
                w = 0.5f;
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    ca[0][e] = cb[0][e];
                    ca[1][e] = cb[1][e];
                }
                cload((z >> 1) + 2);
            }
            const bool zin = z >= 1 && z < n;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float f = w * (h ? 0.5f : 1.f) * (e & 1 ? 0.5f : 1.f);
                    const bool in = zin && (h ? in1 : in0) && !(e == 0 && g == 0);
                    v[h][e] = in ? rnd<T>(v[h][e] + f * m[h][e]) : 0.f;
                }
        };
        const int s0 = t.ka - 1, s1 = t.kb - 1;
        cload(s0 >> 1);
        widen3(raw[0], lanes, last, ca[0]);
        widen3(raw[1], lanes, last, ca[1]);
        cload((s0 >> 1) + 1);
        load(u, s0, true, wc);
        load(u, s0 + 1, true, un);
        float u2[2][4], qn[2][4];
        load(u, s0 + 2, true, u2);
        load(q, s0 + 1, true, qn);
        correct(s0, wc);
        for (int s = s0; s <= s1; ++s) {
            // two steps ahead of their use
            float u3[2][4], q2[2][4], v[2][4], x[4], a[4], b[4];
            load(u, s + 3, s + 1 < s1, u3);
            load(q, s + 2, s + 1 < s1, q2);
            correct(s + 1, un);
            if (s >= t.ka) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float gs = fmaf(c, P[h][e] + un[h][e], qc[h][e]);
                        v[h][e] = e == 0 && g == 0 ? 0.f : fmaf(omega, gs - wc[h][e], wc[h][e]);
                    }
                if (w0) st4(uo + (int64_t)s * F.sz, v[0]);
                if (w1) st4(uo + (int64_t)s * F.sz + F.sy, v[1]);
            }
            float4* E = edge + buf * 2 * nt + tid;
            put4(E, un[0]);
            put4(E + nt, un[1]);
            __syncthreads();
            get4(E + nt - lanes, pair > 0, a);
            get4(E + lanes, pair + 1 < pairs, b);
            xsum(un[0], lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P[0][e] = ((x[e] + a[e]) + un[1][e]) + wc[0][e];
            xsum(un[1], lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P[1][e] = ((x[e] + un[0][e]) + b[e]) + wc[1][e];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    wc[h][e] = un[h][e];
                    un[h][e] = u2[h][e];
                    u2[h][e] = u3[h][e];
                    qc[h][e] = qn[h][e];
                    qn[h][e] = q2[h][e];
                }
            buf ^= 1;
        }
    }
}

// the same in 2D
template <typename T>
__global__ void __launch_bounds__(128)
    k_up2(const Tile* __restrict__ tiles, int ntiles, const BSolve* __restrict__ sv,
          const BLevel* __restrict__ lv, const T* __restrict__ pool_in, T* __restrict__ pool_out,
          const int* __restrict__ active, int src, int dst, int ccur, float omega, int lanes) {
    const int lane = threadIdx.x & 31, gx = lane & (lanes - 1), per = 32 / lanes;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
              nw = (gridDim.x * blockDim.x) >> 5;
    const float c = 0.25f;
    const bool last = gx == lanes - 1;
    for (int first = wid * per; first < ntiles; first += nw * per) {
        const int it = first + lane / lanes;
        const Tile t = tiles[min(it, ntiles - 1)];
        const bool on = it < ntiles && active[t.solve] != 0;
        const BLevel F = lv[sv[t.solve].lev0 + t.level];
        const BLevel C = lv[sv[t.solve].lev0 + t.level + 1];
        const int n = F.n, G = n >> 2, g = t.g0 + gx;
        const bool gok = on && g >= 0 && g < G;
        const bool core = gok && (G <= 32 || (gx >= 1 && gx <= kHaloLanes));
        const int s0 = t.ja - 1, s1 = t.jb - 1;
        const int steps = __reduce_max_sync(0xffffffffu, on ? s1 - s0 + 1 : 0);
        const T* u = pool_in + off_u(F, src) + 4 * g;
        const T* q = pool_in + F.q + 4 * g;
        T* uo = pool_out + off_u(F, dst) + 4 * g;
        const T* uk = pool_in + off_u(C, ccur) + 2 * g;
        auto load = [&](const T* a, int y, bool ok, float* v) {
            ld4(a + (int64_t)y * F.sy, gok && ok && y >= 1 && y < n, v);
        };
        float2 raw;
        auto cload = [&](int J) { raw = ld2(uk + (int64_t)J * C.sy, gok && J < C.n); };
        float ca[3] = {}, un[4], wc[4], P[4] = {}, qc[4] = {};
        // the lanes of a warp whose rows are of the other parity take the same
        // shuffles: odd is the lane's own
        auto correct = [&](int y, float* v) {
            const bool odd = y & 1;
            float cb[3], m[4];
            widen3(raw, lanes, last, cb);
            m[0] = ca[0];
            m[1] = ca[0] + ca[1];
            m[2] = ca[1];
            m[3] = ca[1] + ca[2];
            if (odd) {
                m[0] += cb[0];
                m[1] = (m[1] + cb[0]) + cb[1];
                m[2] += cb[1];
                m[3] = (m[3] + cb[1]) + cb[2];
#pragma unroll
                for (int e = 0; e < 3; ++e) ca[e] = cb[e];
                cload((y >> 1) + 2);
            }
            const bool yin = gok && y >= 1 && y < n;
            const float w = odd ? 0.5f : 1.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float f = e & 1 ? 0.5f * w : w;
                v[e] = yin && !(e == 0 && g == 0) ? rnd<T>(v[e] + f * m[e]) : 0.f;
            }
        };
        cload(s0 >> 1);
        widen3(raw, lanes, last, ca);
        cload((s0 >> 1) + 1);
        load(u, s0, true, wc);
        load(u, s0 + 1, true, un);
        correct(s0, wc);
        for (int i = 0; i < steps; ++i) {
            const int s = s0 + i;
            float u2[4], qn[4], v[4], x[4];
            load(u, s + 2, s < s1, u2);
            load(q, s + 1, s < s1, qn);
            correct(s + 1, un);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float gs = fmaf(c, P[e] + un[e], qc[e]);
                v[e] = e == 0 && g == 0 ? 0.f : fmaf(omega, gs - wc[e], wc[e]);
            }
            if (core && s >= t.ja && s < t.jb) st4(uo + (int64_t)s * F.sy, v);
            xsum(un, lanes, last, x);
#pragma unroll
            for (int e = 0; e < 4; ++e) P[e] = x[e] + wc[e];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                wc[e] = un[e];
                un[e] = u2[e];
                qc[e] = qn[e];
            }
        }
    }
}

// u_fine += P u_coarse, one thread per coarse cell (item level = fine level):
// the cell's 2^d corners are loaded once, the corrections of its 2^d fine
// nodes formed from them (weight 2^-(number of odd offsets) times the sum of
// the corners the fine node lies between), then every fine operand is
// loaded before the first store.
template <typename T>
__global__ void __launch_bounds__(256) k_prolong(const Item* __restrict__ items, int nitems,
                                                 const BSolve* __restrict__ sv,
                                                 const BLevel* __restrict__ lv, T* pool,
                                                 const int* __restrict__ active, int fcur,
                                                 int ccur) {
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        if (!active[w.solve]) continue;
        const BLevel F = lv[sv[w.solve].lev0 + w.level];
        const BLevel C = lv[sv[w.solve].lev0 + w.level + 1];
        const bool three = F.d == 3;
        const int nc = C.n;
        const int64_t sy = F.sy, sz = three ? F.sz : 0;
        const int64_t cy = C.sy, cz = three ? C.sz : 0;
        const T* uc = pool + off_u(C, ccur);
        T* u = pool + off_u(F, fcur);
        const int lg = __ffs(nc) - 1;  // nc is a power of two
        for (int t = threadIdx.x; t < w.count; t += blockDim.x) {
            const uint32_t cell = (uint32_t)(w.start + t);
            const int I = (int)(cell & (nc - 1)), J = (int)((cell >> lg) & (nc - 1)),
                      K = three ? (int)(cell >> (2 * lg)) : 0;
            const int64_t P = K * cz + J * cy + I;
            const int64_t p = (2 * K) * sz + (2 * J) * sy + 2 * I;
            // corners c[a + 2b + 4c'] = u_c(I + a, J + b, K + c')
            float cv[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                cv[e] = (three || e < 4)
                            ? Num<T>::ld(uc[P + ((e >> 2) & 1) * cz + ((e >> 1) & 1) * cy + (e & 1)])
                            : 0.f;
            // the fine node (2I + a, 2J + b, 2K + c') gets 2^-(a+b+c') times the
            // sum of the corners (I + a', J + b', K + c'') with a' <= a, ...
            float corr[8], fv[8];
            bool on[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int a = e & 1, b = (e >> 1) & 1, cc = (e >> 2) & 1;
                on[e] = (three || cc == 0) && !(a == 0 && I == 0) && !(b == 0 && J == 0) &&
                        !(three && cc == 0 && K == 0);
                float sum = 0.f;
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    if ((g & ~e) == 0) sum += cv[g];
                corr[e] = ldexpf(sum, -(a + b + cc));
            }
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (on[e]) fv[e] = Num<T>::ld(u[p + ((e >> 2) & 1) * sz + ((e >> 1) & 1) * sy + (e & 1)]);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (on[e])
                    u[p + ((e >> 2) & 1) * sz + ((e >> 1) & 1) * sy + (e & 1)] =
                        Num<T>::st(fv[e] + corr[e]);
        }
    }
}

// e = 0 on the items' interior nodes (level 0)
template <typename T>
__global__ void __launch_bounds__(256) k_zero(const Item* __restrict__ items, int nitems,
                                              const BSolve* __restrict__ sv,
                                              const BLevel* __restrict__ lv, T* pool,
                                              const int* __restrict__ active) {
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        if (!active[w.solve]) continue;
        const BLevel L = lv[sv[w.solve].lev0];
        T* e = pool + L.u0;
        for (int t = threadIdx.x; t < w.count; t += blockDim.x)
            e[node_of(L, (uint32_t)(w.start + t))] = Num<T>::st(0.f);
    }
}

// u += e in FP64 on the items' interior nodes (level 0)
template <typename T>
__global__ void __launch_bounds__(256) k_update(const Item* __restrict__ items, int nitems,
                                                const BSolve* __restrict__ sv,
                                                const BLevel* __restrict__ lv, const T* pool,
                                                const int* __restrict__ active) {
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        if (!active[w.solve]) continue;
        const BSolve S = sv[w.solve];
        const BLevel L = lv[S.lev0];
        const T* e = pool + L.u0;
        for (int t = threadIdx.x; t < w.count; t += blockDim.x) {
            int i, j, k;
            const int64_t p = node_of(L, (uint32_t)(w.start + t), i, j, k);
            S.u[dense_of(L, i, j, k)] += (double)Num<T>::ld(e[p]);
        }
    }
}

// FP64 scaled right-hand side q64 = h^2 f / (2d) on interior nodes; zero
// u's boundary is the caller's layout contract, enforced here on faces
template <typename T>
__global__ void __launch_bounds__(256) k_prepare(const Item* __restrict__ items, int nitems,
                                                 const BSolve* __restrict__ sv,
                                                 const BLevel* __restrict__ lv, double* pool64) {
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        const BSolve S = sv[w.solve];
        const BLevel L = lv[S.lev0];
        const double h = 1.0 / S.n;
        const double scale = h * h / (2.0 * S.d);
        double* q = pool64 + S.q64;
        for (int t = threadIdx.x; t < w.count; t += blockDim.x) {
            int i, j, k;
            node_of(L, (uint32_t)(w.start + t), i, j, k);
            const int64_t p = dense_of(L, i, j, k);
            q[p] = scale * S.f[p];
        }
    }
}

__global__ void k_fill_int(int* a, int count, int v) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        a[i] = v;
}

__global__ void k_zero_boundary(const BSolve* __restrict__ sv, int count) {
    for (int s = blockIdx.x; s < count; s += gridDim.x) {
        const BSolve S = sv[s];
        const int64_t m = S.n + 1;
        const int64_t nodes = S.d == 3 ? m * m * m : m * m;
        for (int64_t p = threadIdx.x; p < nodes; p += blockDim.x) {
            const int i = (int)(p % m), j = (int)((p / m) % m), k = S.d == 3 ? (int)(p / (m * m)) : 1;
            if (i == 0 || i == S.n || j == 0 || j == S.n || k == 0 || k == (S.d == 3 ? S.n : 2))
                S.u[p] = 0.0;
        }
    }
}

// sigma = q64 + c sum(u) - u in FP64 on the items' interior nodes, stored to
// the inner right-hand side; one partial sum of sigma^2 per item
template <typename T>
__global__ void __launch_bounds__(256) k_outer(const Item* __restrict__ items, int nitems,
                                               const BSolve* __restrict__ sv,
                                               const BLevel* __restrict__ lv, T* pool,
                                               const double* __restrict__ pool64,
                                               const int* __restrict__ active,
                                               double* __restrict__ partial) {
    __shared__ double warp_sums[8];
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item w = items[it];
        if (!active[w.solve]) continue;
        const BSolve S = sv[w.solve];
        const BLevel L = lv[S.lev0];
        const bool three = L.d == 3;
        const double c = three ? 1.0 / 6.0 : 0.25;
        const int64_t sy = L.n + 1, sz = three ? sy * sy : 0;
        const double* u = S.u;
        const double* q = pool64 + S.q64;
        T* qin = pool + L.q;
        double acc = 0.0;
        for (int t = threadIdx.x; t < w.count; t += blockDim.x) {
            int i, j, k;
            const int64_t pin = node_of(L, (uint32_t)(w.start + t), i, j, k);
            const int64_t p = dense_of(L, i, j, k);
            double s = u[p - 1] + u[p + 1];
            s += u[p - sy];
            s += u[p + sy];
            if (three) {
                s += u[p - sz];
                s += u[p + sz];
            }
            const double sig = fma(c, s, q[p]) - u[p];
            qin[pin] = Num<T>::st(cvt::narrow(sig));  // FP64 pipe: one slot less
            acc = fma(sig, sig, acc);
        }
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
        if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int k = 0; k < (int)(blockDim.x / 32); ++k) s += warp_sums[k];
            partial[it] = s;
        }
        __syncthreads();
    }
}

// per solve: sum its partials in order; start (first != 0): res0; otherwise
// count the step, record the relative residual and retire converged solves
__global__ void __launch_bounds__(1024) k_finalize(const BSolve* __restrict__ sv, int count,
                                                   const double* __restrict__ partial,
                                                   double* res0_2, int* active, int* iters,
                                                   double* relres, double rtol2, int maxit,
                                                   int first, int* num_active) {
    __shared__ int warp_cnt[32];
    int cnt = 0;
    for (int s = threadIdx.x; s < count; s += blockDim.x) {
        const BSolve S = sv[s];
        if (first || active[s]) {
            double sum = 0.0;
            for (int i = S.item0; i < S.item1; ++i) sum += partial[i];
            if (first) {
                res0_2[s] = sum;
                iters[s] = 0;
                relres[s] = sum > 0.0 ? 1.0 : 0.0;
                active[s] = (sum > 0.0 && maxit > 0) ? 1 : 0;
            } else {
                iters[s] += 1;
                relres[s] = sqrt(sum / res0_2[s]);
                if (!(sum > rtol2 * res0_2[s]) || iters[s] >= maxit) active[s] = 0;
            }
        }
        cnt += active[s];
    }
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    if ((threadIdx.x & 31) == 0) warp_cnt[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += warp_cnt[w];
        *num_active = t;
    }
}

}  // namespace batch
}  // namespace gmg

using namespace gmg;
using namespace gmg::batch;

namespace {

struct Range {
    int off = 0, count = 0;
    int64_t nodes = 0;  // the items' work
};
// a level step of the solves of one dimension: plain items (chunks) and legs'
// tiles with their launch shapes
struct Step {
    Range fine, cells, down, up;
    int down_threads = 0, up_threads = 0, lanes = 32;
};

}  // namespace

struct gmg_batch_s {
    gmg_config cfg{};
    int count = 0, chunk = 1024, ctas = 608, device = 0, G = 0, elem = 4;
    int leg_ctas = 0;  // the legs' grids: a CTA per tile, up to the caller's ctas if given
    int sms = 152;
    // stream2: the 2D solves' launches inside the captured step, which depend
    // on none of the 3D solves'
    cudaStream_t user_stream = nullptr, stream = nullptr, stream2 = nullptr;
    cudaEvent_t ev = nullptr, fork = nullptr, join = nullptr;
    std::vector<BSolve> hs;
    std::vector<BLevel> hl;
    std::vector<Item> items;
    std::vector<Tile> tiles;
    std::vector<Step> steps[2];  // per level step g: 2D, 3D
    int leg_warps[4] = {0, 0, 0, 0};
    bool has_d[2] = {false, false};
    Range level0;                // level-0 interior items (all solves)
    BSolve* ds = nullptr;
    BLevel* dl = nullptr;
    Item* di = nullptr;
    Tile* dt = nullptr;
    void* pool = nullptr;
    double* pool64 = nullptr;
    double* partial = nullptr;
    double* res0_2 = nullptr;
    double* relres = nullptr;
    int* active = nullptr;
    int* iters = nullptr;
    int* num_active = nullptr;
    int* h_active = nullptr;  // pinned
    cudaGraphExec_t graph = nullptr;
    double graph_rtol2 = -1.0;  // the stopping tolerance baked into the graph
    KernelTimer timer;
};

namespace {

template <typename T>
struct PrecName;
template <>
struct PrecName<float> {
    static constexpr const char* s = "_f32";
};
template <>
struct PrecName<__nv_bfloat16> {
    static constexpr const char* s = "_bf16";
};

template <typename T, class F>
void launch_op(gmg_batch b, cudaStream_t st, const char* name, int g, const Range& r,
               double bytes_per_node, double ops_per_node, F&& body) {
    if (r.count == 0) return;
    const int grid = std::min(r.count, b->ctas);
    b->timer.run(st, std::string(name) + PrecName<T>::s, g, ops_per_node * r.nodes,
                 bytes_per_node * r.nodes, 1, [&] { body(grid, b->di + r.off, r.count); });
}

// The inner cycles of the solves of dimension d on stream st.
template <typename T>
gmg_status enqueue_cycles(gmg_batch b, int d, cudaStream_t st) {
    const gmg_config& c = b->cfg;
    const std::vector<Step>& steps = b->steps[d - 2];
    T* pool = static_cast<T*>(b->pool);
    const double w = sizeof(T);
    const bool rbgs = c.smoother == GMG_RBGS;
    // weighted-Jacobi weight per dimension: the configured one, or with
    // omega = 0 the defaults 4/5 (2D) and 6/7 (3D)
    const float omega2 = c.omega > 0.0 ? (float)c.omega : 0.8f;
    const float omega3 = c.omega > 0.0 ? (float)c.omega : (float)(6.0 / 7.0);
    const float omega = d == 3 ? omega3 : omega2;
    // a weighted-Jacobi sweep next to the transfer goes into the leg; the first
    // one from zero does not read u, so that u_c = 0 need not be written
    const bool sweep_down = !rbgs && c.nu1 >= 1, sweep_up = !rbgs && c.nu2 >= 1;
    int G = 0;
    for (int g = 1; g <= b->G; ++g)
        if (steps[g].down.count) G = g;
    std::vector<int> cur(G + 1, 0);  // which u buffer holds each level step's iterate
    auto relax = [&](int g, int sweeps, int zero) {
        const Range& r = steps[g].fine;
        for (int s = 0; s < sweeps; ++s) {
            if (rbgs) {
                for (int color = 0; color < 2; ++color)
                    launch_op<T>(b, st, "b_rb_half", g, r, 1.5 * w, 3.0,
                                 [&](int grid, const Item* it, int ni) {
                                     k_smooth<T><<<grid, 256, 0, st>>>(
                                         it, ni, b->ds, b->dl, pool, pool, b->active, cur[g],
                                         cur[g], color, 0, omega2, omega3);
                                 });
            } else {
                launch_op<T>(b, st, "b_wj_sweep", g, r, 3 * w, 8.0,
                             [&](int grid, const Item* it, int ni) {
                                 k_smooth<T><<<grid, 256, 0, st>>>(
                                     it, ni, b->ds, b->dl, pool, pool, b->active, cur[g],
                                     cur[g] ^ 1, -1, s == 0 ? zero : 0, omega2, omega3);
                             });
                cur[g] ^= 1;
            }
        }
    };
    auto down = [&](int g, int zero) {
        const Step& S = steps[g];
        const Tile* t = b->dt + S.down.off;
        const int nt = S.down.count, clear = !sweep_down, th = S.down_threads;
        const int src = cur[g], dst = sweep_down ? cur[g] ^ 1 : cur[g];
        b->timer.run(st, std::string(sweep_down ? "b_down_leg" : "b_res_restrict") + PrecName<T>::s,
                     g, (sweep_down ? 18.0 : 10.0) * S.down.nodes,
                     (sweep_down ? 3.125 : 2.125) * w * S.down.nodes, 1, [&] {
                         if (d == 3) {
                             auto k = sweep_down ? k_down3<T, true> : k_down3<T, false>;
                             k<<<std::min(nt, b->leg_ctas), th, 160 * th, st>>>(
                                 t, nt, b->ds, b->dl, pool, pool, b->active, src, dst, zero, clear,
                                 omega);
                         } else {
                             const int ctas = (nt * S.lanes + 127) / 128;
                             auto k = sweep_down ? k_down2<T, true> : k_down2<T, false>;
                             k<<<std::min(ctas, b->leg_ctas), 128, 0, st>>>(
                                 t, nt, b->ds, b->dl, pool, pool, b->active, src, dst, zero, clear,
                                 omega, S.lanes);
                         }
                     });
        cur[g] = dst;
    };
    auto up = [&](int g) {
        const Step& S = steps[g];
        const Tile* t = b->dt + S.up.off;
        const int nt = S.up.count, th = S.up_threads, src = cur[g], cc = cur[g - 1];
        b->timer.run(st, std::string("b_up_leg") + PrecName<T>::s, g, 12.0 * S.up.nodes,
                     3.125 * w * S.up.nodes, 1, [&] {
                         if (d == 3)
                             k_up3<T><<<std::min(nt, b->leg_ctas), th, 64 * th, st>>>(
                                 t, nt, b->ds, b->dl, pool, pool, b->active, src, src ^ 1, cc,
                                 omega);
                         else
                             k_up2<T><<<std::min((nt * S.lanes + 127) / 128, b->leg_ctas), 128, 0, st>>>(
                                 t, nt, b->ds, b->dl, pool, pool, b->active, src, src ^ 1, cc,
                                 omega, S.lanes);
                     });
        cur[g] ^= 1;
    };
    for (int k = 0; k < c.inner_cycles; ++k) {
        std::fill(cur.begin(), cur.end(), 0);
        // which levels start from zero: the coarse ones, in the first cycle all
        const int zero = 2 | (k == 0 ? 1 : 0);
        // down: level steps g = G..1 (fine levels of the deepest solves first)
        for (int g = G; g >= 1; --g) {
            relax(g, sweep_down ? c.nu1 - 1 : c.nu1, zero);
            down(g, sweep_down && c.nu1 == 1 ? zero : 0);
            cur[g - 1] = 0;
        }
        // up: g = 1..G
        for (int g = 1; g <= G; ++g) {
            if (sweep_up) {
                up(g);
            } else {
                const int fc = cur[g], cc = cur[g - 1];
                launch_op<T>(b, st, "b_prolong_add", g, steps[g].cells, 17 * w, 20.0,
                             [&](int grid, const Item* it, int ni) {
                                 k_prolong<T><<<grid, 256, 0, st>>>(it, ni, b->ds, b->dl, pool,
                                                                    b->active, fc, cc);
                             });
            }
            relax(g, sweep_up ? c.nu2 - 1 : c.nu2, 0);
        }
        if (cur[G] != 0) {
            set_error("batched weighted Jacobi needs an even nu1 + nu2 on the finest levels");
            return GMG_ERR_UNSUPPORTED;
        }
    }
    return GMG_OK;
}

// One refinement step of the whole batch (captured): e = 0, k inner
// cycles, u += e, new sigma and per-solve norms, retire converged solves.
template <typename T>
gmg_status enqueue_step(gmg_batch b, double rtol2) {
    const gmg_config& c = b->cfg;
    T* pool = static_cast<T*>(b->pool);
    const double w = sizeof(T);
    b->timer.begin_capture();
    if (c.smoother == GMG_RBGS || c.nu1 == 0)
        launch_op<T>(b, b->stream, "b_zero", 0, b->level0, w, 0,
                     [&](int grid, const Item* it, int ni) {
                         k_zero<T><<<grid, 256, 0, b->stream>>>(it, ni, b->ds, b->dl, pool,
                                                                b->active);
                     });
    // The 2D and the 3D solves' launches are two branches of the graph: the
    // small levels of one fill the chip beside the other's.  While kernels are
    // timed they run one after the other.
    const bool both = b->has_d[0] && b->has_d[1] && !b->timer.enabled;
    cudaStream_t st2 = both ? b->stream2 : b->stream;
    gmg_status rc = GMG_OK;
    if (both) {
        GMG_CUDA_TRY(cudaEventRecord(b->fork, b->stream));
        GMG_CUDA_TRY(cudaStreamWaitEvent(st2, b->fork, 0));
    }
    if (b->has_d[1]) rc = enqueue_cycles<T>(b, 3, b->stream);
    if (rc == GMG_OK && b->has_d[0]) rc = enqueue_cycles<T>(b, 2, st2);
    if (both) {
        GMG_CUDA_TRY(cudaEventRecord(b->join, st2));
        GMG_CUDA_TRY(cudaStreamWaitEvent(b->stream, b->join, 0));
    }
    if (rc != GMG_OK) return rc;
    launch_op<T>(b, b->stream, "b_update", 0, b->level0, 16 + w, 1.0,
                 [&](int grid, const Item* it, int ni) {
                     k_update<T><<<grid, 256, 0, b->stream>>>(it, ni, b->ds, b->dl, pool,
                                                              b->active);
                 });
    launch_op<T>(b, b->stream, "b_outer_residual", 0, b->level0, 16 + w, 8.0,
                 [&](int grid, const Item* it, int ni) {
                     k_outer<T><<<grid, 256, 0, b->stream>>>(it, ni, b->ds, b->dl, pool,
                                                             b->pool64, b->active, b->partial);
                 });
    b->timer.run(b->stream, "b_finalize", 0, 0, 0, 1, [&] {
        k_finalize<<<1, 1024, 0, b->stream>>>(b->ds, b->count, b->partial, b->res0_2, b->active,
                                              b->iters, b->relres, rtol2, c.maxit, 0,
                                              b->num_active);
    });
    GMG_CUDA_TRY(cudaMemcpyAsync(b->h_active, b->num_active, sizeof(int), cudaMemcpyDeviceToHost,
                                 b->stream));
    GMG_CUDA_TRY(cudaGetLastError());
    return GMG_OK;
}

template <typename T>
void enqueue_start(gmg_batch b) {
    T* pool = static_cast<T*>(b->pool);
    const int grid0 = std::min(b->level0.count, b->ctas);
    const Item* it0 = b->di + b->level0.off;
    k_zero_boundary<<<std::min(b->count, 1024), 256, 0, b->stream>>>(b->ds, b->count);
    k_prepare<T><<<grid0, 256, 0, b->stream>>>(it0, b->level0.count, b->ds, b->dl, b->pool64);
    // every solve counts as active for the initial residual
    k_fill_int<<<(b->count + 255) / 256, 256, 0, b->stream>>>(b->active, b->count, 1);
    k_outer<T><<<grid0, 256, 0, b->stream>>>(it0, b->level0.count, b->ds, b->dl, pool, b->pool64,
                                             b->active, b->partial);
    k_finalize<<<1, 1024, 0, b->stream>>>(b->ds, b->count, b->partial, b->res0_2, b->active,
                                          b->iters, b->relres, 0.0, b->cfg.maxit, 1,
                                          b->num_active);
    b->timer.launches += 5;
}

bool dev_ptr_ok(const void* p) {
    if (!p || ((uintptr_t)p) % 8) return false;
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

namespace {

// warps of each leg kernel that fit on an SM: leg_warps[2D up, 2D down, 3D up,
// 3D down]; the 3D kernels' shared memory is opted into here
template <typename T>
cudaError_t leg_occupancy(gmg_batch b) {
    const bool rbgs = b->cfg.smoother == GMG_RBGS;
    const bool sweep = !rbgs && b->cfg.nu1 >= 1;
    auto d3 = sweep ? k_down3<T, true> : k_down3<T, false>;
    auto d2 = sweep ? k_down2<T, true> : k_down2<T, false>;
    cudaError_t e = cudaFuncSetAttribute(d3, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * kLegThreads);
    auto occ = [&](auto k, int threads, int smem, int& warps) {
        int n = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem);
        warps = std::max(1, n) * threads / 32;
    };
    occ(k_up2<T>, 128, 0, b->leg_warps[0]);
    occ(d2, 128, 0, b->leg_warps[1]);
    occ(k_up3<T>, 128, 64 * 128, b->leg_warps[2]);
    occ(d3, 128, 160 * 128, b->leg_warps[3]);
    return e;
}

}  // namespace

extern "C" {

gmg_status gmg_batch_destroy(gmg_batch b) {
    if (!b) return GMG_OK;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->timer.destroy();
    for (void* p : {(void*)b->ds, (void*)b->dl, (void*)b->di, b->pool, (void*)b->pool64,
                    (void*)b->partial, (void*)b->res0_2, (void*)b->relres, (void*)b->active,
                    (void*)b->iters, (void*)b->num_active})
        if (p) cudaFree(p);
    if (b->h_active) cudaFreeHost(b->h_active);
    for (cudaEvent_t ev : {b->ev, b->fork, b->join})
        if (ev) cudaEventDestroy(ev);
    for (cudaStream_t st : {b->stream, b->stream2})
        if (st) cudaStreamDestroy(st);
    delete b;
    if (prev >= 0) cudaSetDevice(prev);
    return GMG_OK;
}

gmg_status gmg_batch_create(int count, const int* d, const int* n, const gmg_config* common,
                            int chunk, int ctas, void* cuda_stream, gmg_batch* out) {
    if (!out || !common || !d || !n || count < 1 || count > (1 << 20)) {
        set_error("gmg_batch_create: bad arguments");
        return GMG_ERR_ARG;
    }
    *out = nullptr;
    if (common->precision != GMG_FP32_IR && common->precision != GMG_BF16_IR) {
        set_error("gmg_batch_create: precision must be GMG_FP32_IR or GMG_BF16_IR");
        return GMG_ERR_UNSUPPORTED;
    }
    if (common->smoother != GMG_WJACOBI && common->smoother != GMG_RBGS) {
        set_error("gmg_batch_create: smoother must be weighted Jacobi or red-black GS");
        return GMG_ERR_ARG;
    }
    if (common->transfer != GMG_TRANSFER_FW) {
        set_error("gmg_batch_create: the batch uses full-weighting transfers");
        return GMG_ERR_UNSUPPORTED;
    }
    if (common->smoother == GMG_WJACOBI && ((common->nu1 + common->nu2) % 2 != 0)) {
        set_error("gmg_batch_create: weighted Jacobi needs nu1 + nu2 even");
        return GMG_ERR_UNSUPPORTED;
    }
    if (common->nu1 < 0 || common->nu2 < 0 || common->nu1 > 16 || common->nu2 > 16 ||
        common->inner_cycles < 1 || common->inner_cycles > 64 || common->maxit < 0 ||
        !(common->omega >= 0.0 && common->omega < 2.0)) {
        set_error("gmg_batch_create: nu1, nu2, inner_cycles, maxit or omega out of range");
        return GMG_ERR_ARG;
    }
    if (chunk < 0 || chunk > (1 << 20) || ctas < 0 || ctas > (1 << 16)) {
        set_error("gmg_batch_create: chunk / ctas out of range");
        return GMG_ERR_ARG;
    }
    for (int s = 0; s < count; ++s) {
        const int nmax = d[s] == 2 ? 16384 : 1024;
        if ((d[s] != 2 && d[s] != 3) || n[s] < 2 || n[s] > nmax || (n[s] & (n[s] - 1))) {
            set_error("gmg_batch_create: solve " + std::to_string(s) +
                      ": d must be 2 or 3 and n a power of two within limits");
            return GMG_ERR_ARG;
        }
    }
    gmg_batch b = new gmg_batch_s();
    b->cfg = *common;
    b->count = count;
    b->chunk = chunk > 0 ? chunk : 1024;
    b->user_stream = (cudaStream_t)cuda_stream;
    b->elem = common->precision == GMG_FP32_IR ? 4 : 2;
    auto fail = [&](gmg_status st, const std::string& msg) {
        set_error("gmg_batch_create: " + msg);
        gmg_batch_destroy(b);
        return st;
    };
    if (cudaGetDevice(&b->device) != cudaSuccess) return fail(GMG_ERR_CUDA, "no device");
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    b->ctas = ctas > 0 ? ctas : 4 * b->sms;
    b->leg_ctas = ctas > 0 ? ctas : INT_MAX;
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&b->stream2, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->join, cudaEventDisableTiming) != cudaSuccess)
        return fail(GMG_ERR_CUDA, "stream/event creation failed");
    // layout: per solve, per level: u0 [u1] q in the inner pool (256-byte
    // aligned regions); FP64 q64 per solve
    const int64_t align = 256 / b->elem;
    auto up = [&](int64_t v, int64_t a) { return (v + a - 1) / a * a; };
    int64_t poff = 0, off64 = 0;
    for (int s = 0; s < count; ++s) {
        BSolve S{};
        S.d = d[s];
        S.n = n[s];
        int L = 0;
        while ((2 << L) <= n[s]) ++L;  // log2(n) grids: n, n/2, ..., 2
        S.levels = L;
        S.lev0 = (int)b->hl.size();
        const int64_t m0 = n[s] + 1;
        S.q64 = off64;
        off64 = up(off64 + (d[s] == 3 ? m0 * m0 * m0 : m0 * m0), 32);
        for (int l = 0; l < L; ++l) {
            BLevel lv{};
            lv.d = d[s];
            lv.n = n[s] >> l;
            lv.rows = fastdiv_make((uint32_t)(lv.n - 1));
            // rows padded to a multiple of 8 elements (16 bytes in BF16, 32 in FP32)
            const int64_t m = lv.n + 1;
            lv.sy = up(m, 8);
            lv.sz = d[s] == 3 ? lv.sy * m : 0;
            const int V = 16 / b->elem;
            int lg = 0;
            while ((V << (lg + 1)) <= lv.n) ++lg;  // 2^lg groups of V cover x = 0 .. n-1
            lv.lgG = lg;
            const int64_t nodes = d[s] == 3 ? lv.sz * m : lv.sy * m;
            lv.u0 = poff;
            poff = up(poff + nodes, align);
            lv.u1 = -1;
            if (common->smoother == GMG_WJACOBI) {
                lv.u1 = poff;
                poff = up(poff + nodes, align);
            }
            lv.q = poff;
            poff = up(poff + nodes, align);
            b->hl.push_back(lv);
        }
        b->G = std::max(b->G, L - 1);
        b->hs.push_back(S);
    }
    // work items
    auto add_items = [&](int s, int level, int64_t total, std::vector<Item>& dst) {
        for (int64_t st = 0; st < total; st += b->chunk)
            dst.push_back({s, level, st, (int)std::min<int64_t>(b->chunk, total - st)});
    };
    auto pw = [](int64_t v, int d_) { return d_ == 3 ? v * v * v : v * v; };
    {  // level 0 interior items, grouped by solve (the finalize sums them in order)
        b->level0.off = (int)b->items.size();
        for (int s = 0; s < count; ++s) {
            b->hs[s].item0 = (int)b->items.size() - b->level0.off;
            add_items(s, 0, pw(b->hs[s].n - 1, b->hs[s].d), b->items);
            b->hs[s].item1 = (int)b->items.size() - b->level0.off;
        }
        b->level0.count = (int)b->items.size() - b->level0.off;
        for (int i = 0; i < b->level0.count; ++i)
            b->level0.nodes += b->items[b->level0.off + i].count;
    }
    const bool rbgs = common->smoother == GMG_RBGS;
    const cudaError_t oe = b->elem == 4 ? leg_occupancy<float>(b) : leg_occupancy<__nv_bfloat16>(b);
    if (oe != cudaSuccess) return fail(GMG_ERR_CUDA, cudaGetErrorString(oe));
    // sweeps that no leg takes (relax)
    const bool plain = rbgs || common->nu1 > 1 || common->nu2 > 1;
    struct Leg {  // the tiles of a step: a solve's side by side
        Range* r;
        int dim, g, len, np;
        std::vector<Rows> rows;
        std::vector<int> cols;
    };
    std::vector<Leg> legs;
    std::vector<std::vector<int>> members(2 * (b->G + 1));
    size_t ntiles = 0;
    for (int dim = 2; dim <= 3; ++dim) {
        b->steps[dim - 2].resize(b->G + 1);
        for (int g = 1; g <= b->G; ++g) {
            Step& S = b->steps[dim - 2][g];
            const int n_g = 2 << g, nc = n_g / 2;  // the same size for every solve
            std::vector<int>& mem = members[2 * g + dim - 2];
            for (int s = 0; s < count; ++s)
                if (b->hs[s].d == dim && b->hs[s].levels - 1 >= g) mem.push_back(s);
            if (mem.empty()) continue;
            b->has_d[dim - 2] = true;
            auto level_of = [&](int s) { return b->hs[s].levels - 1 - g; };
            // (interior row, 16-byte group) pairs, chunk / V groups per item
            S.fine.off = (int)b->items.size();
            const int V = 16 / b->elem;
            for (int s : mem) {
                const int l = level_of(s);
                const int64_t groups = (int64_t)(dim == 3 ? (n_g - 1) * (n_g - 1) : n_g - 1)
                                       << b->hl[b->hs[s].lev0 + l].lgG;
                const int64_t gchunk = std::max<int64_t>(1, b->chunk / V);
                for (int64_t st = 0; plain && st < groups; st += gchunk)
                    b->items.push_back({s, l, st, (int)std::min<int64_t>(gchunk, groups - st)});
                S.fine.nodes += groups * V;
            }
            S.fine.count = (int)b->items.size() - S.fine.off;
            if (rbgs || common->nu2 == 0) {
                S.cells.off = (int)b->items.size();
                for (int s : mem) {
                    add_items(s, level_of(s), pw(nc, dim), b->items);
                    S.cells.nodes += pw(nc, dim);
                }
                S.cells.count = (int)b->items.size() - S.cells.off;
            }
            S.lanes = std::min(n_g / 4, 32);
            for (int down = 0; down < 2; ++down) {
                if (!down && (rbgs || common->nu2 == 0)) continue;
                Leg L{down ? &S.down : &S.up, dim, g, 0, 0, {Rows{0, 0, 0}},
                      leg_columns(n_g / 4, kHaloLanes)};
                // walk: coarse planes 1..nc-1 down (2 fine planes each), fine planes 1..n-1 up
                L.len = down ? nc - 1 : n_g - 1;
                const int unit = down ? 2 : 1, extra = down ? 4 : 2;
                int& th = down ? S.down_threads : S.up_threads;
                int64_t slots;
                if (dim == 3) {
                    th = leg_threads(n_g, down);
                    const int R = leg_rows(n_g, th);
                    L.rows = down ? rows_down(n_g, R) : rows_up(n_g, R);
                    slots = (int64_t)b->sms * std::max(1, b->leg_warps[2 + down] / (th / 32));
                } else {
                    slots = (int64_t)b->sms * b->leg_warps[down] * (32 / S.lanes);
                }
                const int64_t columns = (int64_t)(mem.size() * L.rows.size() * L.cols.size());
                L.np = leg_pieces(columns, slots, L.len, unit, extra);
                L.r->off = (int)ntiles;
                L.r->count = (int)(columns * L.np);
                L.r->nodes = (int64_t)mem.size() * pw(n_g - 1, dim);
                ntiles += L.r->count;
                legs.push_back(std::move(L));
            }
        }
    }
    b->tiles.reserve(ntiles);  // (grown step by step they took longer than all else here)
    std::vector<int> cut;
    for (const Leg& L : legs) {
        cut.resize(L.np + 1);
        for (int pc = 0; pc <= L.np; ++pc) cut[pc] = 1 + (int)((int64_t)L.len * pc / L.np);
        for (int s : members[2 * L.g + L.dim - 2]) {
            const int level = b->hs[s].levels - 1 - L.g;
            for (int pc = 0; pc < L.np; ++pc)
                for (const Rows& rw : L.rows)
                    for (int g0 : L.cols)
                        b->tiles.push_back(
                            L.dim == 3 ? Tile{s, level, g0, rw.y0, rw.ja, rw.jb, cut[pc], cut[pc + 1]}
                                       : Tile{s, level, g0, 0, cut[pc], cut[pc + 1], 0, 0});
        }
    }
    cudaError_t e = cudaSuccess;
    auto al = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, std::max<size_t>(bytes, 8));
        if (e == cudaSuccess) e = cudaMemsetAsync(*p, 0, std::max<size_t>(bytes, 8), b->stream);
    };
    al((void**)&b->ds, sizeof(BSolve) * count);
    al((void**)&b->dl, sizeof(BLevel) * b->hl.size());
    al((void**)&b->di, sizeof(Item) * b->items.size());
    // the tiles behind the pool (an allocation of their own took 45 us)
    const size_t pool_bytes = ((size_t)b->elem * poff + 255) / 256 * 256;
    al(&b->pool, pool_bytes + sizeof(Tile) * b->tiles.size());
    b->dt = reinterpret_cast<Tile*>(static_cast<char*>(b->pool) + pool_bytes);
    al((void**)&b->pool64, sizeof(double) * off64);
    al((void**)&b->partial, sizeof(double) * b->level0.count);
    al((void**)&b->res0_2, sizeof(double) * count);
    al((void**)&b->relres, sizeof(double) * count);
    al((void**)&b->active, sizeof(int) * count);
    al((void**)&b->iters, sizeof(int) * count);
    al((void**)&b->num_active, sizeof(int));
    if (e != cudaSuccess)
        return fail(e == cudaErrorMemoryAllocation ? GMG_ERR_ALLOC : GMG_ERR_CUDA,
                    cudaGetErrorString(e));
    if (cudaMallocHost((void**)&b->h_active, sizeof(int)) != cudaSuccess)
        return fail(GMG_ERR_ALLOC, "cudaMallocHost failed");
    e = cudaMemcpyAsync(b->dl, b->hl.data(), sizeof(BLevel) * b->hl.size(), cudaMemcpyHostToDevice,
                        b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->di, b->items.data(), sizeof(Item) * b->items.size(),
                            cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess && !b->tiles.empty())
        e = cudaMemcpyAsync(b->dt, b->tiles.data(), sizeof(Tile) * b->tiles.size(),
                            cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return fail(GMG_ERR_CUDA, cudaGetErrorString(e));
    *out = b;
    return GMG_OK;
}

gmg_status gmg_batch_solve(gmg_batch b, const double* const* f, double* const* u, double rtol,
                           int* iters_out, double* relres_out, int* steps_out) {
    if (!b || !f || !u || !(rtol >= 0.0) || !std::isfinite(rtol)) {
        set_error("gmg_batch_solve: bad arguments");
        return GMG_ERR_ARG;
    }
    for (int s = 0; s < b->count; ++s) {
        if (!dev_ptr_ok(f[s]) || !dev_ptr_ok(u[s])) {
            set_error("gmg_batch_solve: f/u of solve " + std::to_string(s) +
                      " is not an aligned device pointer");
            return GMG_ERR_LAYOUT;
        }
        b->hs[s].f = f[s];
        b->hs[s].u = u[s];
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b->device) cudaSetDevice(b->device);
    struct Restore {
        int p, d;
        ~Restore() {
            if (p >= 0 && p != d) cudaSetDevice(p);
        }
    } restore{prev, b->device};
    const double rtol2 = rtol * rtol;
    GMG_CUDA_TRY(cudaEventRecord(b->ev, b->user_stream));
    GMG_CUDA_TRY(cudaStreamWaitEvent(b->stream, b->ev, 0));
    GMG_CUDA_TRY(cudaMemcpyAsync(b->ds, b->hs.data(), sizeof(BSolve) * b->count,
                                 cudaMemcpyHostToDevice, b->stream));
    if (b->elem == 4)
        enqueue_start<float>(b);
    else
        enqueue_start<__nv_bfloat16>(b);
    GMG_CUDA_TRY(cudaGetLastError());
    if (b->graph && b->graph_rtol2 != rtol2) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    if (!b->graph) {
        cudaGraph_t g = nullptr;
        GMG_CUDA_TRY(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
        gmg_status st = b->elem == 4 ? enqueue_step<float>(b, rtol2)
                                     : enqueue_step<__nv_bfloat16>(b, rtol2);
        cudaError_t e = cudaStreamEndCapture(b->stream, &g);
        if (st != GMG_OK) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        GMG_CUDA_TRY(e);
        e = cudaGraphInstantiate(&b->graph, g, 0);
        cudaGraphDestroy(g);
        GMG_CUDA_TRY(e);
        b->graph_rtol2 = rtol2;
    }
    GMG_CUDA_TRY(cudaMemcpyAsync(b->h_active, b->num_active, sizeof(int), cudaMemcpyDeviceToHost,
                                 b->stream));
    GMG_CUDA_TRY(cudaStreamSynchronize(b->stream));
    int steps = 0;
    while (*b->h_active > 0 && steps < b->cfg.maxit) {
        GMG_CUDA_TRY(cudaGraphLaunch(b->graph, b->stream));
        GMG_CUDA_TRY(cudaStreamSynchronize(b->stream));
        b->timer.after_graph_run();
        ++steps;
    }
    if (steps_out) *steps_out = steps;
    std::vector<int> it(b->count);
    std::vector<double> rel(b->count);
    GMG_CUDA_TRY(cudaMemcpy(it.data(), b->iters, sizeof(int) * b->count, cudaMemcpyDeviceToHost));
    GMG_CUDA_TRY(cudaMemcpy(rel.data(), b->relres, sizeof(double) * b->count,
                            cudaMemcpyDeviceToHost));
    bool all = true;
    for (int s = 0; s < b->count; ++s) {
        if (iters_out) iters_out[s] = it[s];
        if (relres_out) relres_out[s] = rel[s];
        if (!std::isfinite(rel[s])) {
            set_error("gmg_batch_solve: non-finite residual in solve " + std::to_string(s));
            return GMG_ERR_NONFINITE;
        }
        if (rel[s] > rtol) all = false;
    }
    if (!all) {
        set_error("gmg_batch_solve: some solves reached maxit above rtol");
        return GMG_ERR_NOT_CONVERGED;
    }
    return GMG_OK;
}

gmg_status gmg_batch_set_timing(gmg_batch b, int enable) {
    if (!b) {
        set_error("batch is NULL");
        return GMG_ERR_ARG;
    }
    if ((enable != 0) != b->timer.enabled) {
        b->timer.enabled = enable != 0;
        if (b->graph) {
            GMG_CUDA_TRY(cudaStreamSynchronize(b->stream));
            cudaGraphExecDestroy(b->graph);
            b->graph = nullptr;
        }
    }
    b->timer.reset();
    return GMG_OK;
}

gmg_status gmg_batch_timing_report(gmg_batch b, gmg_kernel_stat* out, int cap, int* count,
                                   int64_t* launches_out) {
    if (!b || (!out && cap > 0)) {
        set_error("bad arguments");
        return GMG_ERR_ARG;
    }
    b->timer.report(out, cap, count, launches_out);
    return GMG_OK;
}

gmg_status gmg_create_batched(int count, const gmg_config* cfgs, void* cuda_stream,
                              gmg_batch* out) {
    if (!out || !cfgs || count < 1 || count > (1 << 20)) {
        set_error("gmg_create_batched: bad arguments");
        return GMG_ERR_ARG;
    }
    *out = nullptr;
    const gmg_config& c0 = cfgs[0];
    std::vector<int> d(count), n(count);
    for (int i = 0; i < count; ++i) {
        const gmg_config& c = cfgs[i];
        if (c.smoother != c0.smoother || c.omega != c0.omega || c.nu1 != c0.nu1 ||
            c.nu2 != c0.nu2 || c.precision != c0.precision || c.inner_cycles != c0.inner_cycles ||
            c.maxit != c0.maxit) {
            set_error("gmg_create_batched: solves differ in smoother, sweeps, precision, "
                      "inner_cycles or maxit");
            return GMG_ERR_ARG;
        }
        d[i] = c.d;
        n[i] = c.n;
    }
    return gmg_batch_create(count, d.data(), n.data(), &c0, 0, 0, cuda_stream, out);
}

gmg_status gmg_solve_batched(gmg_batch b, const double* const* f, double* const* u, double rtol,
                             int* iters_out) {
    return gmg_batch_solve(b, f, u, rtol, iters_out, nullptr, nullptr);
}

}  // extern "C"
