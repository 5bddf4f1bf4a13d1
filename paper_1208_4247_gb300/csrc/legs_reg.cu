// Fused leg kernels of the FP32 3D red-black inner hierarchies (colour-split
// layout), planes in registers:
//
//   down leg  S half sweeps (alternating colours, the last one black), the
//             red residual and its full weighting;
//   up leg    the black nodes' prolongation and correction, then S half sweeps
//             (red first).
//
// The wavefront of legs.cuh (at step t stage s works on plane t - s) with
// another division of the work.  A thread owns 8 nodes of x (one 4-vector of
// each half row) and two rows of y, an even and an odd one.  All stages of a
// step work on the same half row of a thread's row, and the two rows on
// opposite ones, so which half that is depends on the step's parity alone: the
// loop is unrolled by two and every index is a constant.  A stage's operands:
// x from its own stage before of the previous step (the other half row; the
// entry beyond the vector by one shuffle), z from that of two steps before and
// of this step, y inside the pair of rows from registers, and across pairs by
// two vectors of shared memory, the only exchange.  The newest value of a
// stage takes the registers of its oldest.  q goes by cp.async into a ring of
// the thread's own; the first colour's old values are never read, so half of u
// is.
//
// Node values are formed by the level kernels' expressions in their order
// (k_rb_half_vec, k_residual, k_restrict, k_prolong_add with red-only /
// black-only nodes): the same bits.
//
// Measured at n = 512 (four half sweeps a leg): 493 us down and 374 us up, 10.5
// bytes per node of traffic that a copy moves in 210 us.  The legs that keep
// every plane in shared memory (legs.cuh; FP32 took them before) took 910 and
// 824 us with 532 M and 461 M warp instructions, 268 M and 201 M here.  What
// bounds it: shared memory (36 16-byte accesses per thread and step) and
// latency at 9 to 12 warps per SM, which the registers and the rings allow, and
// a halo of S + 2 rows that is worked through twice (half of the lanes at S =
// 4).  Tried and slower: q through registers (spills; 658 us down), cp.async
// through L1 (576 us), prefetches into L2 (521 us), loads of a stage issued
// with it instead of a stage ahead (506 us).
#include <algorithm>
#include <cstdlib>

#include "legs_api.h"
#include "level_kernels.cuh"

namespace gmg {
namespace rlegs {
namespace {

constexpr int kDown = 0, kUp = 1;
constexpr int LX = 16;       // lanes (groups of 8 nodes) per row
constexpr int kCore = 14;    // of them kept where a row is wider than 16 groups
constexpr unsigned kAll = 0xffffffffu;

// per leg: stages whose values other threads read, shared memory per thread,
// and the threads 227 KB have room for (the more rows, the smaller the halo)
template <int MODE, int S>
struct Geo {
    static constexpr int NST = MODE == kDown ? S + 1 : S;
    static constexpr int LS = MODE == kDown ? S + 1 : S;  // last stage that reads q
    // planes of q held of stage 1's colour (odd stages) and of the other: the
    // oldest a stage reads, up to the one on its way
    static constexpr int Q0 = (LS & 1 ? LS : LS - 1) + 1, Q1 = (LS & 1 ? LS - 1 : LS) + 1;
    static constexpr int kEx = 2 * NST * 2, kR = MODE == kDown ? 4 * 2 : 0, kQ = 2 * (Q0 + Q1);
    static constexpr int kBytes = 16 * (kEx + kR) + 16 * kQ;
    static constexpr int kFit = (227 * 1024 - 2 * 16 * LX) / kBytes / 32 * 32;
    // 12 warps: three per scheduler, 168 registers each
    static constexpr int NT = kFit < 384 ? kFit : 384;
    static constexpr int R = 2 * (NT / LX);
};

// Tile i of the rows: held rows y0 .. y0 + R - 1 (y0 even), written [ja, jb)
// (down: coarse rows).  A stage is right on the held rows less its number on
// each side (a side at the boundary loses none; row n is held there, as zeros).
struct Rows {
    int y0, ja, jb;
};
template <int MODE, int S>
__host__ __device__ inline Rows row_tile(int i, int n) {
    constexpr int R = Geo<MODE, S>::R;
    Rows r;
    if (MODE == kDown) {
        constexpr int H = (S + 3) / 2 * 2;  // rows below 2 ja held: S + 2, even
        constexpr int first = (R - S - 3) / 2 + 1, m = (R - S - 3 - H) / 2 + 1;
        r.ja = i == 0 ? 1 : first + (i - 1) * m;
        r.y0 = i == 0 ? 0 : 2 * r.ja - H;
        r.jb = r.y0 + R > n ? n / 2 : i == 0 ? first : r.ja + m;
    } else {
        r.ja = i == 0 ? 1 : R - S + (i - 1) * (R - 2 * S);
        r.y0 = i == 0 ? 0 : r.ja - S;
        r.jb = r.y0 + R > n ? n : r.y0 + R - S;
    }
    return r;
}

struct Args {
    Lay F, C;
    int zseg;
    const float* u;
    float* uo;
    const float* q;
    const float* ec;
    float* qc;
    float* uc;
    int init;
};

__device__ inline void ld4(const float* p, float* v) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ inline float2 ld2(const float* p, bool ok) {
    return ok ? __ldg(reinterpret_cast<const float2*>(p)) : make_float2(0.f, 0.f);
}
__device__ inline void st4(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ inline void st2(float* p, float a, float b) {
    *reinterpret_cast<float2*>(p) = make_float2(a, b);
}
// 4 nodes of q: global to shared memory, and from there
__device__ inline void cp4(float* d, const float* s) {  // not through L1
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(d)),
                 "l"(s)
                 : "memory");
}
__device__ inline void zero4(float* d) {
    *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ inline void getq(const float* p, float* v) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ inline void get4(const float4* p, float* v) {
    const float4 a = *p;
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ inline void put4(float4* p, const float* v) { *p = make_float4(v[0], v[1], v[2], v[3]); }

// Gauss-Seidel values of the half row PAR: xr = the other half of the row
template <int PAR>
__device__ inline float edge_of(const float* xr, bool last) {
    const float e = PAR ? __shfl_down_sync(kAll, xr[0], 1, LX) : __shfl_up_sync(kAll, xr[3], 1, LX);
    return PAR && last ? 0.f : e;  // x = n
}
// (x- + x+) + (y- + z-) of the half row PAR (xr: the other half of the row)
template <int PAR>
__device__ inline void part4(const float* xr, float edge, const float* ym, const float* zm,
                             float* w) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float xm = PAR ? xr[t] : t > 0 ? xr[t > 0 ? t - 1 : 0] : edge;
        const float xp = PAR ? (t < 3 ? xr[t < 3 ? t + 1 : 3] : edge) : xr[t];
        w[t] = (xm + xp) + (ym[t] + zm[t]);
    }
}

template <int MODE, int S>
__global__ void __launch_bounds__(Geo<MODE, S>::NT, 1) k_rleg(const __grid_constant__ Args a) {
    using G = Geo<MODE, S>;
    constexpr bool DOWN = MODE == kDown;
    constexpr int NT = G::NT, NST = G::NST;
    constexpr int c1 = DOWN ? (S & 1) : 0;  // colour of stage 1 (the last is black)
    extern __shared__ float4 sm[];
    const int tid = threadIdx.x, gx = tid & (LX - 1), pair = tid / LX;
    // a row of lanes free on both sides: the first and the last pair of rows
    // read there (or in the next array) what no kept node depends on
    float4* ex = sm + LX + tid;            // [2][NST][row][NT]
    float4* rr = ex + G::kEx * NT;         // [4][row][NT]
    // q, the thread's own: [Q0][row][NT] of stage 1's colour, [Q1][row][NT]
    float* qr = reinterpret_cast<float*>(sm + (G::kEx + G::kR) * NT + 2 * LX) + 4 * tid;
    constexpr int QS = 2 * 4 * NT;  // a plane of one colour
    const int n = a.F.n, nc = a.C.n, NG = n / 8;
    const int g = (NG > LX ? kCore * (int)blockIdx.x - 1 : 0) + gx;
    const bool gok = g >= 0 && g < NG, last = gx == LX - 1;
    const bool core = gok && (NG <= LX || (gx >= 1 && gx <= kCore));
    const Rows rt = row_tile<MODE, S>(blockIdx.y, n);
    const int y = rt.y0 + 2 * pair;  // even; the pair's second row y + 1
    const bool in0 = gok && y >= 1 && y < n, in1 = gok && y + 1 < n;
    int K0 = 0, K1 = 0, wlo, whi;
    if (DOWN) {
        K0 = 1 + a.zseg * (int)blockIdx.z;
        K1 = min(K0 + a.zseg, nc);
        wlo = 2 * K0 - 1;
        whi = K1 == nc ? n : 2 * K1 - 1;
    } else {
        wlo = 1 + a.zseg * (int)blockIdx.z;
        whi = min(wlo + a.zseg, n);
    }
    const int zlo = max(DOWN ? 2 * K0 - 2 - S : wlo - S, 0);
    const int tend = DOWN ? 2 * K1 + S : whi - 1 + S;
    const int ylo = DOWN ? 2 * rt.ja - 1 : rt.ja;
    const int yhi = DOWN ? 2 * rt.jb - 1 + (rt.jb == nc) : rt.jb;
    const bool w0 = core && in0 && y >= ylo && y < yhi;
    const bool w1 = core && in1 && y + 1 >= ylo && y + 1 < yhi;
    const bool wc = DOWN && core && y >= 2 * rt.ja && y < 2 * rt.jb;
    const int oc = (y >> 1) * (int)a.C.sy + 2 * g;
    const bool cok = gok && y < n;
    // no lane of the warp holds a boundary node: values are kept as they come
    const bool easy = __all_sync(kAll, in0 && in1 && g != 0);

    // half row `par` of row h of plane z.  Rows, planes and groups beyond the
    // grid take the boundary's zeros from memory (the group past the last one
    // its entry x = n); what the other positions of such a group hold reaches
    // no kept node.
    const int gc = min(max(g, 0), NG);
    uint32_t off[2][2];  // [row][half], within a plane
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        off[h][0] = (uint32_t)(min(y + h, n) * (int)a.F.sy + 4 * gc);
        off[h][1] = (uint32_t)(min(y + h, n) * (int)a.F.sy + a.F.he + 4 * min(gc, NG - 1));
    }
    auto plane = [&](const float* p, int z) { return p + (int64_t)min(z, n) * a.F.sz; };
    // q of plane z into its slots (i0 = z mod Q0, i1 = z mod Q1); par: row y's
    // half of stage 1's colour when it gets there
    auto qload = [&](int z, int i0, int i1, int par) {
        const float* pz = plane(a.q, z);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            cp4(qr + i0 * QS + h * 4 * NT, pz + off[h][par ^ h]);
            cp4(qr + (G::Q0 + i1) * QS + h * 4 * NT, pz + off[h][par ^ h ^ 1]);
        }
        asm volatile("cp.async.commit_group;");
    };
    // the pair's coarse rows J, J + 1 of plane K as values I = 4g .. 4g + 3
    auto cload = [&](int K, float (*v)[4]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float* p = a.ec + (int64_t)K * a.C.sz + (oc + (h ? (int)a.C.sy : 0));
            const float2 e = ld2(p, cok && K <= nc), d = ld2(p + a.C.he, cok && K <= nc);
            v[h][0] = e.x, v[h][1] = d.x, v[h][2] = e.y, v[h][3] = d.y;
        }
    };
    auto next = [&](float v) {  // I = 4g + 4
        const float w = __shfl_down_sync(kAll, v, 1, LX);
        return last ? 0.f : w;
    };

    constexpr int par_even = (c1 + 1) & 1;  // half of row y at even steps
    float X[NST][2][2][4];  // [stage][step parity][row]
    float un[2][4];         // loaded u of the step's plane
    float ck[2][4], cn[2][4];
#pragma unroll
    for (int s = 0; s < NST; ++s)
#pragma unroll
        for (int i = 0; i < 16; ++i) (&X[s][0][0][0])[i] = 0.f;
    const int t0 = zlo & ~1;
    ld4(plane(a.u, t0) + off[0][par_even], un[0]);
    ld4(plane(a.u, t0) + off[1][par_even ^ 1], un[1]);
    if (!DOWN) {
        cload(t0 >> 1, ck);
        cload((t0 >> 1) + 1, cn);
    }
    // the neighbours' values "one step before the first" are zeros
#pragma unroll
    for (int i = 0; i < G::kEx; ++i) ex[i * NT] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (DOWN)
#pragma unroll
        for (int i = 0; i < G::kR; ++i) rr[i * NT] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < G::kQ; ++i) zero4(qr + i * 4 * NT);
    __syncthreads();
    int i0 = 0, i1 = 0;  // the slots of the step's plane (t0's are the first)

    auto step = [&](auto parity, int t) {
        constexpr int P = decltype(parity)::value;
        constexpr int par0 = (c1 + P + 1) & 1;
        float4* exw = ex + P * NST * 2 * NT;
        const float4* exr = ex + (P ^ 1) * NST * 2 * NT;
        float prev[2][4], old[2][4], C[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) prev[h][e] = un[h][e];
        if (!DOWN) {
            const bool zin = t >= 1 && t < n;
            float v[2][4], w0p, w1p;
            if (P == 0) {  // z = 2K: (2I+1, 2J) and (2I, 2J+1)
                const float c4 = next(ck[0][0]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[0][e] = ck[0][e] + (e < 3 ? ck[0][e < 3 ? e + 1 : 3] : c4);
                    v[1][e] = ck[0][e] + ck[1][e];
                }
                w0p = w1p = 0.5f;
            } else {  // z = 2K+1: (2I, 2J) and the octet (2I+1, 2J+1)
                const float a4 = next(ck[0][0]), b4 = next(ck[1][0]), d4 = next(cn[0][0]),
                            f4 = next(cn[1][0]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[0][e] = ck[0][e] + cn[0][e];
                    const float x00 = ck[0][e] + (e < 3 ? ck[0][e < 3 ? e + 1 : 3] : a4);
                    const float x10 = ck[1][e] + (e < 3 ? ck[1][e < 3 ? e + 1 : 3] : b4);
                    const float x01 = cn[0][e] + (e < 3 ? cn[0][e < 3 ? e + 1 : 3] : d4);
                    const float x11 = cn[1][e] + (e < 3 ? cn[1][e < 3 ? e + 1 : 3] : f4);
                    v[1][e] = (x00 + x10) + (x01 + x11);
                }
                w0p = 0.5f;
                w1p = 0.125f;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e) ck[h][e] = cn[h][e];
                cload((t >> 1) + 2, cn);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    prev[h][e] = (fmaf(h ? w1p : w0p, v[h][e], prev[h][e]));
            if (!(easy && zin))
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (!(zin && (h ? in1 : in0)) ||
                            ((h ? par0 ^ 1 : par0) == 0 && e == 0 && g == 0))
                            prev[h][e] = 0.f;
        }
        // plane t - 1 of q has come; the next plane of u, this plane's q (used
        // from the next step on)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        ld4(plane(a.u, t + 1) + off[0][par0 ^ 1], un[0]);
        ld4(plane(a.u, t + 1) + off[1][par0], un[1]);
        qload(t, i0, i1, par0 ^ 1);
        constexpr int LS = G::LS;
        // Stage s in two parts: what does not depend on this step (all but z+
        // and q) is formed before the stage ahead of it ends, so that its
        // loads and its sums fill that stage's waits, and z- is used up when
        // the stage ahead writes over it.
        float w[2][2][4], yp[2][4], q0[4], q1[4], ym[2][4], e0[2], e1[2];
        auto raw = [&](int s) {
            get4(exr + (2 * (s - 1) + 1) * NT - LX, ym[s & 1]);
            get4(exr + 2 * (s - 1) * NT + LX, yp[s & 1]);
            e0[s & 1] = edge_of<par0>(X[s - 1][P ^ 1][0], last);
            e1[s & 1] = edge_of<par0 ^ 1>(X[s - 1][P ^ 1][1], last);
        };
        auto ahead = [&](int s) {
            float(&A)[2][4] = X[s - 1][P ^ 1];
            float(&B)[2][4] = X[s - 1][P];
            part4<par0>(A[0], e0[s & 1], ym[s & 1], B[0], w[s & 1][0]);
            part4<par0 ^ 1>(A[1], e1[s & 1], A[0], B[1], w[s & 1][1]);
        };
        auto fetch_q = [&](int s) {
            const int i = s & 1 ? i0 - s + (i0 < s ? G::Q0 : 0) : i1 - s + (i1 < s ? G::Q1 : 0);
            const float* qs = qr + (s & 1 ? i : G::Q0 + i) * QS;
            getq(qs, q0);
            getq(qs + 4 * NT, q1);
        };
        raw(1);
        fetch_q(1);
        if (LS > 1) raw(2);
        ahead(1);
        put4(exw, prev[0]);
        put4(exw + NT, prev[1]);
#pragma unroll
        for (int s = 1; s <= LS; ++s) {
            const int p = t - s;
            float(&A)[2][4] = X[s - 1][P ^ 1];
            float(&B)[2][4] = X[s - 1][P];
            if (s < LS) ahead(s + 1);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                C[0][e] = fmaf(1.f / 6.f, w[s & 1][0][e] + (A[1][e] + prev[0][e]), q0[e]);
                C[1][e] = fmaf(1.f / 6.f, w[s & 1][1][e] + (yp[s & 1][e] + prev[1][e]), q1[e]);
            }
            if (s < LS) fetch_q(s + 1);
            if (s + 2 <= LS) raw(s + 2);
            if (DOWN && s == S + 1) {  // the red residual: red values of two steps ago
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e) C[h][e] = (C[h][e] - old[h][e]);
            } else {
                const bool zin = p >= 1 && p < n;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e) C[h][e] = (C[h][e]);
                if (!(easy && zin))
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (!(zin && (h ? in1 : in0)) ||
                                ((h ? par0 ^ 1 : par0) == 0 && e == 0 && g == 0))
                                C[h][e] = 0.f;
            }
            if (s == S && p >= wlo && p < whi) {  // both colours of plane t - S are final
                float* d = a.uo + (int64_t)p * a.F.sz;
                if (w0) {
                    st4(d + off[0][par0], C[0]);
                    st4(d + off[0][par0 ^ 1], A[0]);
                }
                if (w1) {
                    st4(d + off[1][par0 ^ 1], C[1]);
                    st4(d + off[1][par0], A[1]);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (s == S) old[h][e] = B[h][e];
                    B[h][e] = prev[h][e];
                    prev[h][e] = C[h][e];
                }
            if (s < NST) {
                put4(exw + 2 * s * NT, C[0]);
                put4(exw + (2 * s + 1) * NT, C[1]);
            }
        }
        const int pr = t - S - 1;
        if (DOWN) {
            put4(rr + (pr & 3) * 2 * NT, C[0]);
            put4(rr + ((pr & 3) * 2 + 1) * NT, C[1]);
        }
        i0 = i0 + 1 < G::Q0 ? i0 + 1 : 0;
        i1 = i1 + 1 < G::Q1 ? i1 + 1 : 0;
        __syncthreads();
        if (DOWN && ((P + S + 1) & 1)) {  // pr odd: coarse plane K = (pr - 1) / 2 is complete
            const int K = pr >> 1;
            if (K >= K0 && K < K1) {
                float c0[4], o1[4], b1[4], m0[4], om[4], bm[4], bp[4], v[4];
                const float4 *r1 = rr + ((pr - 1) & 3) * 2 * NT, *r2 = rr + ((pr - 2) & 3) * 2 * NT,
                             *r0 = rr + (pr & 3) * 2 * NT;
                get4(r1, c0);
                get4(r1 + NT, o1);
                get4(r1 + NT - LX, b1);
                get4(r2, m0);
                get4(r2 + NT, om);
                get4(r2 + NT - LX, bm);
                get4(r0 + NT - LX, bp);
                const float b1l = __shfl_up_sync(kAll, b1[3], 1, LX),
                            o1l = __shfl_up_sync(kAll, o1[3], 1, LX),
                            m0l = __shfl_up_sync(kAll, m0[3], 1, LX),
                            p0l = __shfl_up_sync(kAll, C[0][3], 1, LX);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x = (e ? b1[e ? e - 1 : 0] : b1l) + b1[e];
                    x += e ? o1[e ? e - 1 : 0] : o1l;
                    x += o1[e];
                    x += e ? m0[e ? e - 1 : 0] : m0l;
                    x += m0[e];
                    x += bm[e];
                    x += om[e];
                    x += e ? C[0][e ? e - 1 : 0] : p0l;
                    x += C[0][e];
                    x += bp[e];
                    x += C[1][e];
                    v[e] = (fmaf(0.125f, x, 0.5f * c0[e]));
                }
                if (g == 0) v[0] = 0.f;
                if (wc) {
                    const int64_t pc = (int64_t)K * a.C.sz + oc;
                    st2(a.qc + pc, v[0], v[2]);
                    st2(a.qc + pc + a.C.he, v[1], v[3]);
                    // I = 4g + e: red where e + J + K is even
                    const bool odd = ((y >> 1) + K) & 1, red = a.init == INIT_RED;
                    const float z = 1.f / 6.f * 0.f;
                    st2(a.uc + pc, red && !odd ? v[0] + z : 0.f, red && !odd ? v[2] + z : 0.f);
                    st2(a.uc + pc + a.C.he, red && odd ? v[1] + z : 0.f, red && odd ? v[3] + z : 0.f);
                }
            }
        }
    };
    for (int t = t0; t <= tend; t += 2) {
        step(std::integral_constant<int, 0>{}, t);
        step(std::integral_constant<int, 1>{}, t + 1);
    }
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 152;
}

template <int MODE, int S>
cudaError_t launch(Args a, cudaStream_t s) {
    using G = Geo<MODE, S>;
    constexpr int smem = G::kBytes * G::NT + 2 * 16 * LX;
    const cudaError_t e = cudaFuncSetAttribute(
        k_rleg<MODE, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int n = a.F.n, NG = n / 8;
    const int tx = NG > LX ? (NG + kCore - 1) / kCore : 1;
    int ty = 1;
    while (row_tile<MODE, S>(ty - 1, n).jb < (MODE == kDown ? n / 2 : n)) ++ty;
    // pieces of z: the fewest waves (one CTA per SM) times steps of a piece
    const int len = MODE == kDown ? n / 2 - 1 : n - 1, unit = MODE == kDown ? 2 : 1;
    const int extra = MODE == kDown ? 2 * S + 3 : 2 * S, sms = sm_count();
    int64_t best = INT64_MAX;
    for (int p = 1; p <= len; ++p) {
        const int seg = (len + p - 1) / p;
        const int64_t ctas = (int64_t)tx * ty * ((len + seg - 1) / seg);
        const int64_t cost = (ctas + sms - 1) / sms * (unit * seg + extra);
        if (cost < best) {
            best = cost;
            a.zseg = seg;
        }
    }
    if (const char* v = std::getenv("GMG_LEG_SEGS")) {
        const int p = std::atoi(v);
        if (p > 0) a.zseg = (len + std::min(p, len) - 1) / std::min(p, len);
    }
    const dim3 grid(tx, ty, (len + a.zseg - 1) / a.zseg);
    k_rleg<MODE, S><<<grid, G::NT, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t down(const Lay& F, const Lay& C, const float* u_in, float* u_out, const float* q,
                 float* qc, float* uc, int init, int S, cudaStream_t s) {
    const Args a{F, C, 0, u_in, u_out, q, nullptr, qc, uc, init};
    return S == 2   ? launch<kDown, 2>(a, s)
           : S == 3 ? launch<kDown, 3>(a, s)
           : S == 4 ? launch<kDown, 4>(a, s)
                    : cudaErrorInvalidValue;
}
cudaError_t up(const Lay& C, const Lay& F, const float* ec, const float* u_in, float* u_out,
               const float* q, int S, cudaStream_t s) {
    const Args a{F, C, 0, u_in, u_out, q, ec, nullptr, nullptr, INIT_ZERO};
    return S == 2 ? launch<kUp, 2>(a, s) : S == 4 ? launch<kUp, 4>(a, s) : cudaErrorInvalidValue;
}

}  // namespace rlegs
}  // namespace gmg
