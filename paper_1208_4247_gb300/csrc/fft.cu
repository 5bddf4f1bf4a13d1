// Direct solve of the FD system by sine transforms (the paper's comparison
// method, section 2.3).  A'u = h^2 f is diagonal in the sine basis along
// every axis; here the first d-1 axes are transformed (DST-I), which leaves
// one tridiagonal system per line of the last axis,
//     -v_{k-1} + (2 + lambda) v_k - v_{k+1} = h^2 fhat_k,
//     lambda = sum over the transformed axes of 4 sin^2(pi k_m / (2n)),
// solved by elimination, and the same transforms back: S^-1 = (2/n) S.
// (The paper divides by the continuous symbol k_x^2 + k_y^2; the discrete
// eigenvalues make the result the exact solution of the same FD system the
// multigrid solves.)  The work array holds nodes 0..n-1 of each transformed
// axis, row pitch n, so that a tile of 16 columns is one 128-byte segment.
//
// What bounds the solve on GB300 is the FP64 pipe (0.505 T adds/s measured,
// against 6.8 TB/s of HBM: at 16 bytes a node and pass, 6 instructions cost as
// much as the traffic).  So the transforms are built for few FP64 operations:
// two real lines share one complex line, and a DST-I of length n - 1 is folded
// into DST-IIIs of sizes n/2, n/4, .., 1, each a complex FFT of its own size
// (about 14 instructions per value at n = 256; a complex FFT of the odd
// extension, length 2n, takes about 35, the real one of length 2n that a
// library offers the same again in gathers and scatters).  The elimination
// along the last axis takes 3 (2D: 9) where the two transforms and the division by
// the eigenvalues would take about 30.
// 3D 257^3: 14.94 ms with length-2n library transforms of the odd extension
// on all three axes, 2.16 ms with these kernels (0.50 ms a
// transform of one axis at 84% of the FP64 pipe, 0.13 ms the eliminations).
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "gmg_internal.cuh"

namespace gmg {
namespace fft {
namespace {

// ------------------------------------------------------------ DST-I of lines
//
// Positions 1..n-1 of a line hold x_1..x_{n-1} (complex: two real lines).
// Folding x_j, x_{r-j} (r = n, n/2, .., 4) into the difference at j and the sum
// at r - j leaves at positions M .. 2M-1 (M = r/2) the input c_0 .. c_{M-1} of
// a DCT-III of size M whose values are, up to the sign (-1)^k, the
// coefficients y_{(n/2M)(2k+1)} (sin(pi (M-j)(2k+1)/2M) = (-1)^k cos(pi j
// (2k+1)/2M)).  The DCT-III by one complex FFT of size M (Makhoul 1980, "A
// fast cosine transform in one and two dimensions"):
//     V_j = e^{i pi j/2M} (c_j - i c_{M-j}) / 2,  V_0 = c_0,
//     v = sum_j V_j e^{2 pi i jm/M},  C_{2m} = v_m, C_{2m+1} = v_{M-1-m}.
// The kernels form 2 V_j, hence twice the DST: the powers of two go into the
// scale of the line solves, exactly.
// Everything stays in place in shared memory: the FFTs are
// decimation-in-frequency radix-8 stages (the last one 8, 4 or 2) that leave
// their output digit-reversed, which the final gather undoes.
//
// A CTA takes a tile of 2^lgP pairs of lines with n/8 threads per pair (one
// radix-8 butterfly each and stage; 32 to 512 threads in all).  The tasks of a
// step are numbered with the pair fastest and dealt to the threads one loop
// after the other, so that the small folds and blocks, which would leave most
// of a warp idle if every pair kept its own warp, fill warps across pairs: an
// FP64 instruction costs its 64 cycles of a sub-core whatever lanes are on
// (257^3, one pass over an axis: 697 -> 500 us).
// Position p of a line sits at entry p + p/8 and a line's entries are an odd
// number apart: neither butterflies whose legs are 8, 4 or 2 apart nor the
// pairs of a tile meet in a bank.
struct Plan {
    int lg, lgP, threads;
    __host__ __device__ constexpr int n() const { return 1 << lg; }
    __host__ __device__ constexpr int pairs() const { return 1 << lgP; }
    __host__ __device__ constexpr int stride() const { return ((1 << lg) + ((1 << lg) >> 3)) | 1; }
    constexpr size_t smem() const { return sizeof(double2) * (size_t)pairs() * stride(); }
};
// total: pairs of lines of a transform.  Tiles of 256 threads (512 from n =
// 512 up: 8 pairs of columns there are 128-byte segments along x) where there
// are enough of them for two per SM, smaller ones (one warp at least) else.
Plan plan_of(int n, int64_t total) {
    Plan p;
    p.lg = 0;
    while ((1 << p.lg) < n) ++p.lg;
    const int lgG = std::min(9, std::max(1, p.lg - 3));  // log2 threads per pair
    p.lgP = (n >= 512 ? 9 : 8) - lgG;
    p.threads = 1 << (lgG + p.lgP);
    while (p.lgP > 0 && lgG + p.lgP > 5 && total >> p.lgP < 2 * 152) {
        --p.lgP;
        p.threads = std::max(p.threads / 2, 128);
    }
    return p;
}

__device__ inline double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ inline double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ inline double2 times_i(double2 a) { return make_double2(-a.y, a.x); }
__device__ inline double2 cmul(double2 a, double2 w) {
    return make_double2(fma(a.x, w.x, -(a.y * w.y)), fma(a.x, w.y, a.y * w.x));
}
// r + s * v
__device__ inline double2 axpy(double s, double2 v, double2 r) {
    return make_double2(fma(s, v.x, r.x), fma(s, v.y, r.y));
}
__device__ inline int at(int p) { return p + (p >> 3); }

__device__ inline void dft4(double2& a, double2& b, double2& c, double2& d) {
    const double2 s = a + c, t = a - c, u = b + d, v = times_i(b - d);
    a = s + u;
    b = t + v;
    c = s - u;
    d = t - v;
}
// x[p] <- sum_q x[q] e^{2 pi i p q / 8}: 52 instructions (the rotations by pi/4
// are scaled in the last sums)
__device__ inline void dft8(double2 (&x)[8]) {
    const double h = 0.70710678118654752440;  // sqrt(1/2)
    double2 e0 = x[0] + x[4], e1 = x[1] + x[5], e2 = x[2] + x[6], e3 = x[3] + x[7];
    const double2 o0 = x[0] - x[4], o1 = x[1] - x[5], o2 = times_i(x[2] - x[6]), o3 = x[3] - x[7];
    dft4(e0, e1, e2, e3);
    // o1 e^{i pi/4} = h r1, o3 e^{3 i pi/4} = h r3
    const double2 r1 = make_double2(o1.x - o1.y, o1.x + o1.y);
    const double2 r3 = make_double2(-o3.x - o3.y, o3.x - o3.y);
    const double2 s = o0 + o2, t = o0 - o2, u = r1 + r3, v = times_i(r1 - r3);
    x[0] = e0;
    x[2] = e1;
    x[4] = e2;
    x[6] = e3;
    x[1] = axpy(h, u, s);
    x[3] = axpy(h, v, t);
    x[5] = axpy(-h, u, s);
    x[7] = axpy(-h, v, t);
}

// The transform of the tile's pairs of lines (positions 1..n-1 of pair v at
// entries at(p) of sm + v * stride, the first fold done and visible) by the
// whole CTA; ends with a barrier.  T[k] = e^{i pi k/n}, k < 2n.
__device__ void dst_tile(double2* __restrict__ sm, const Plan& P, const double2* __restrict__ T) {
    const int lg = P.lg, n = 1 << lg, nt = blockDim.x, stride = P.stride();
    int cursor = 0;  // the thread that takes the next loop's first task
    auto tasks = [&](int w0, int w1, auto&& f) {
        const int total = (w1 - w0) << P.lgP;
        for (int id = ((int)threadIdx.x - cursor) & (nt - 1); id < total; id += nt)
            f(sm + (id & (P.pairs() - 1)) * stride, w0 + (id >> P.lgP));
        cursor = (cursor + ((total + 31) & ~31)) & (nt - 1);
    };
    // folds r = n/2, n/4, .., 4, two at a time: the orbit of j under both
    for (int r = n / 2; r >= 4; r /= 4) {
        const int h = r / 2;
        tasks(1, r / 4 + 1, [&](double2* s, int j) {
            const double2 a = s[at(j)], b = s[at(r - j)];
            if (j == r / 4) {  // h - j = j: the inner fold leaves its middle
                s[at(j)] = a - b;
                s[at(r - j)] = a + b;
            } else {
                const double2 c = s[at(h - j)], d = s[at(h + j)];
                const double2 e = a - b, f = c - d;
                s[at(r - j)] = a + b;
                s[at(h + j)] = c + d;
                s[at(j)] = e - f;
                s[at(h - j)] = e + f;
            }
        });
        __syncthreads();
    }
    // 2 V_j, 2 V_{M-j} in each block M = 2 .. n/2; the pair index w = M/2 + j runs
    // over all blocks (j = 0 of block M: V_0 and the middle element, M/2)
    tasks(0, 1, [&](double2* s, int) {  // the block of size 1
        s[at(1)].x *= 2.0;
        s[at(1)].y *= 2.0;
    });
    tasks(1, n / 2, [&](double2* s, int w) {
        const int l2 = 31 - __clz(w), m2 = 1 << l2;  // M/2
        const int j = w - m2, M = 2 * m2;
        if (j == 0) {
            const int p = at(M + m2), p0 = at(M);
            s[p].x *= 1.41421356237309504880;
            s[p].y *= 1.41421356237309504880;
            s[p0].x *= 2.0;
            s[p0].y *= 2.0;
        } else {
            const int p = at(M + j), q = at(2 * M - j);
            const double2 a = s[p], b = times_i(s[q]);
            const double2 t = T[j << (lg - 2 - l2)];
            s[p] = cmul(a - b, t);
            s[q] = cmul(a + b, make_double2(t.x, -t.y));
        }
    });
    __syncthreads();
    // radix-8 stages: sub-block length L = M, M/8, ..; butterfly index w over
    // all blocks with L >= 8 (block M holds w = M/8 .. M/4 - 1)
    for (int sh = 0; (n / 2 >> sh) >= 2; sh += 3) {  // L = M >> sh
        if (1 << sh < n / 8)
            tasks(1 << sh, n / 8, [&](double2* s, int w) {
                const int lm = 31 - __clz(w);
                const int M = 8 << lm, t = w - (1 << lm);
                const int L = M >> sh, sub = L >> 3;
                const int k = t & (sub - 1);
                const int p0 = M + (t - k) * 8 + k;
                double2 x[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) x[q] = s[at(p0 + q * sub)];
                dft8(x);
                if (sub > 1) {
                    const int st = (2 * n / L) * k;  // e^{2 pi i k/L} = T[st]
#pragma unroll
                    for (int q = 1; q < 8; ++q) x[q] = cmul(x[q], T[st * q]);
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) s[at(p0 + q * sub)] = x[q];
            });
        // the blocks whose sub-block length is now 4 or 2
        const int M4 = 4 << sh, M2 = 2 << sh;
        if (M4 <= n / 2)
            tasks(0, M4 / 4, [&](double2* s, int t) {
                double2* x = s + at(M4 + 4 * t);  // four entries of one group of 8
                double2 a = x[0], b = x[1], c = x[2], d = x[3];
                dft4(a, b, c, d);
                x[0] = a;
                x[1] = b;
                x[2] = c;
                x[3] = d;
            });
        if (M2 <= n / 2)
            tasks(0, M2 / 2, [&](double2* s, int t) {
                double2* x = s + at(M2 + 2 * t);
                const double2 a = x[0], b = x[1];
                x[0] = a + b;
                x[1] = a - b;
            });
        __syncthreads();
    }
}

// Entry of coefficient K (1..n-1) of a transformed line, and its sign.
__device__ inline int coeff_at(int K, int lg, bool& minus) {
    const int r = __ffs(K) - 1;
    const int lm = lg - 1 - r;  // log2 M
    const int k = K >> (r + 1);
    minus = k & 1;
    int m = minus ? (1 << lm) - 1 - (k >> 1) : k >> 1;
    int pos = 0, left = lm;
    while (left > 0) {  // digits from the first stage on
        const int b = left >= 3 ? 3 : left;
        left -= b;
        pos += (m & ((1 << b) - 1)) << left;
        m >>= b;
    }
    return at((1 << lm) + pos);
}

// DST-I along x of every interior row of src into dst (element (i, j, k) at
// k*sz + j*sy + i).  whole_u: dst is u, whose boundary nodes are set to 0 too
// (the rows' ends here, the boundary rows dealt over the CTAs).
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_dst_x(const double* __restrict__ src, int64_t ssy,
                                                   int64_t ssz, double* __restrict__ dst,
                                                   int64_t dsy, int64_t dsz, int64_t lines, int d,
                                                   Plan P, int whole_u,
                                                   const double2* __restrict__ T) {
    extern __shared__ double2 sm[];
    const int lg = P.lg, n = P.n();
    // loading and storing: the threads of a pair along x
    const int lgG = 31 - __clz(blockDim.x) - P.lgP, G = 1 << lgG;
    const int g = threadIdx.x & (G - 1), pair = threadIdx.x >> lgG;
    double2* s = sm + pair * P.stride();
    const int64_t la = 2 * ((int64_t)blockIdx.x * P.pairs() + pair), lb = la + 1;
    auto row = [&](int64_t l, int64_t sy, int64_t sz) {
        const int64_t k = l / (n - 1);
        return (l - k * (n - 1) + 1) * sy + (k + 1) * sz;  // sz = 0 in 2D
    };
    const bool ina = la < lines, inb = lb < lines;
    const double* pa = src + (ina ? row(la, ssy, ssz) : 0);
    const double* pb = src + (inb ? row(lb, ssy, ssz) : 0);
#pragma unroll 4
    for (int j = 1 + g; j < n / 2; j += G) {
        const double2 a = make_double2(ina ? pa[j] : 0.0, inb ? pb[j] : 0.0);
        const double2 b = make_double2(ina ? pa[n - j] : 0.0, inb ? pb[n - j] : 0.0);
        s[at(j)] = a - b;
        s[at(n - j)] = a + b;
    }
    if (g == 0) s[at(n / 2)] = make_double2(ina ? pa[n / 2] : 0.0, inb ? pb[n / 2] : 0.0);
    __syncthreads();
    dst_tile(sm, P, T);
    double* qa = dst + (ina ? row(la, dsy, dsz) : 0);
    double* qb = dst + (inb ? row(lb, dsy, dsz) : 0);
    for (int K = 1 + g; K < n; K += G) {
        bool minus;
        const double2 v = s[coeff_at(K, lg, minus)];
        if (ina) qa[K] = minus ? -v.x : v.x;
        if (inb) qb[K] = minus ? -v.y : v.y;
    }
    if (!whole_u) return;
    if (g == 0) {
        if (ina) qa[0] = qa[n] = 0.0;
        if (inb) qb[0] = qb[n] = 0.0;
    }
    const int m = n + 1;
    for (int r = blockIdx.x; r < (d == 3 ? 4 * m : 2); r += gridDim.x) {
        // 2D: j = 0, n; 3D: (j = 0, n; every k), then (every j; k = 0, n)
        const int side = d == 3 ? r / m : r, t = d == 3 ? r % m : 0;
        const int j = side == 0 ? 0 : side == 1 ? n : t;
        const int k = side == 2 ? 0 : side == 3 ? n : t;
        double* p = dst + k * dsz + j * dsy;
        for (int i = threadIdx.x; i < m; i += blockDim.x) p[i] = 0.0;
    }
}

// DST-I along y of the work array, in place (row pitch n, plane n*n, planes
// 1..n-1): a CTA takes the tile's pairs of neighbouring columns, loaded and
// stored row by row.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_dst_y(double* __restrict__ w, int64_t pairs, Plan P,
                                                   const double2* __restrict__ T) {
    extern __shared__ double2 sm[];
    const int lg = P.lg, n = P.n();
    const int cols = 2 * P.pairs();
    const int col = threadIdx.x & (cols - 1), lp = col >> 1;
    const int j0 = threadIdx.x / cols, dj = blockDim.x / cols;
    const int64_t q = (int64_t)blockIdx.x * P.pairs() + lp;
    const int64_t plane = q >> (lg - 1);
    const int64_t x = 2 * (q & (n / 2 - 1)) + (col & 1);
    // column 0 is no line: its partner's rounding errors must not stay in it
    const bool in = q < pairs && x > 0;
    double* base = w + (in ? ((plane + 1) << (2 * lg)) + x : 0);
    double* sl = reinterpret_cast<double*>(sm + lp * P.stride()) + (col & 1);
#pragma unroll 4
    for (int j = 1 + j0; j < n / 2; j += dj) {
        const double a = in ? base[(int64_t)j << lg] : 0.0;
        const double b = in ? base[(int64_t)(n - j) << lg] : 0.0;
        sl[2 * at(j)] = a - b;
        sl[2 * at(n - j)] = a + b;
    }
    if (j0 == 0) sl[2 * at(n / 2)] = in ? base[(int64_t)(n / 2) << lg] : 0.0;
    __syncthreads();
    dst_tile(sm, P, T);
    if (!in) return;
    for (int K = 1 + j0; K < n; K += dj) {
        bool minus;
        const double v = sl[2 * coeff_at(K, lg, minus)];
        base[(int64_t)K << lg] = minus ? -v : v;
    }
}

// -------------------------------------------------- lines of the last axis
//
// Elimination from both ends to the middle k = n/2 (half the chain, half the
// coefficients): c_1 = 1/(2+lambda), c_k = 1/(2+lambda - c_{k-1}) serve both
// halves, v'_k = (s d_k + v'_{k-1}) c_k, the middle value takes 1/(2+lambda -
// 2 c_{n/2-1}), and each half substitutes back v_k = v'_k + c_k v_{k+1}.
// With r + 1/r = 2 + lambda, r < 1, in closed form
//     c_k = 1 - e_k,  e_k = (1-r)(1 + r^{2k+1}) / (1 - r^{2k+2}),
//     1 - r = sqrt(lambda + lambda^2/4) - lambda/2.
// (r and its powers in double-double), a table of the plan: one row per k =
// 1..n/2, the last one the middle's coefficient.
//
// An error that the c_k of a line share enters its solution 2/(1-r) times over,
// and where r^{2k} is below the last bit all of them share the rounding of r to
// double: 2D 8193^2 was solved to 8.6e-15 in some modes that way.  So in 2D from n =
// 512 up, where 1 - r is small and the chains long, the table holds e_k, of the
// size of 1 - r, and a step takes c_k v as v - e_k v.  Else it holds c_k, each
// rounded together with the error of those before it, which saves the back
// substitution an instruction (257^3: 125 us, 151 with e_k; 2D 257^2 12.0, 12.7)
// and is as accurate up to there, but not above (2D 513^2 5.5e-16 against 4.5,
// 2049^2 13.5e-16 against 7.0).  Error against the exact solution of the system, smooth f
// (uniform f): 2D 257^2 3.6e-16 (3.3e-16), with c_k just rounded 6.7e-16 (5.2e-16),
// by transforms of both axes 4.1e-16 (4.2e-16); 2049^2 4.6e-16 (7.0e-16), 11.6e-16
// (18.4e-16), 6.0e-16 (9.6e-16); 3D 257^3 3.8e-16 (5.4e-16), 3.9e-16 (5.2e-16),
// 5.8e-16 (5.5e-16); 129^3 3.8e-16 (4.1e-16), 4.3e-16 (4.3e-16), 3.3e-16 (4.4e-16).
// The recurrence of c_k or e_k in double is worse still (4097^2: 1e-14).
struct DD {
    double h, l;
};
__device__ inline DD dd_sum(double a, double b) {  // a + b, exactly
    const double s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
__device__ inline DD dd_add(DD a, DD b) {
    const DD s = dd_sum(a.h, b.h);
    return dd_sum(s.h, s.l + (a.l + b.l));
}
__device__ inline DD dd_mul(DD a, DD b) {
    const double p = a.h * b.h;
    return dd_sum(p, fma(a.h, b.h, -p) + fma(a.h, b.l, a.l * b.h));
}
// The table holds e_k (2D, long chains), else c_k.
__host__ __device__ inline bool table_of_e(int d, int n) { return d == 2 && n > 256; }
// One thread per line and kSeg coefficients.
constexpr int kSeg = 16;
__global__ void __launch_bounds__(128) k_coeffs(double* __restrict__ c, int d, int n) {
    const int64_t lines = d == 3 ? (int64_t)n * n : n;
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= lines) return;
    const int x = (int)(l % n), y = (int)(l / n);  // y = 0 in 2D
    const double sx = sinpi(x / (2.0 * n)), sy = sinpi(y / (2.0 * n));
    const double lambda = 4.0 * fma(sx, sx, sy * sy);
    const int k0 = 1 + kSeg * (int)blockIdx.y, k1 = min(k0 + kSeg, n / 2);
    if (lambda == 0.0) {  // row and column 0 of the transformed axes: no line
        for (int k = k0; k < k1; ++k) c[(int64_t)k * lines + l] = 0.0;
        if (k1 == n / 2) c[(int64_t)k1 * lines + l] = 0.0;
        return;
    }
    const DD w = dd_mul({lambda, 0.0}, dd_sum(1.0, 0.25 * lambda));
    const double q = sqrt(w.h);
    const DD e1 = dd_add(dd_sum(q, (fma(-q, q, w.h) + w.l) / (2.0 * q)), {-0.5 * lambda, 0.0});
    const DD r = dd_add({1.0, 0.0}, {-e1.h, -e1.l});
    // power = r^(2 k0 - 1); 0 where it is far below the last bit (r <= exp(-e1))
    DD power{0.0, 0.0};
    if ((2.0 * k0 - 1.0) * e1.h < 45.0) {
        DD base = r;
        power = {1.0, 0.0};
        for (int m = 2 * k0 - 1; m > 0; m >>= 1) {
            if (m & 1) power = dd_mul(power, base);
            base = dd_mul(base, base);
        }
    }
    const DD r2 = dd_mul(r, r);
    // e_k from r^(2k+1)
    auto e_of = [&](DD pw) {
        const DD rp = dd_mul(pw, r);
        const DD den = dd_add({1.0, 0.0}, {-rp.h, -rp.l}), num = dd_add({1.0, 0.0}, pw);
        return e1.h * num.h / den.h;
    };
    // c_k tables: 1 - e less what the entries before it have too much in all.  A segment
    // starts with an amount of its own, spread over the half units, so that what
    // the segments of a line leave at their ends is not shared either.
    const double golden = 0.6180339887498949 * blockIdx.y;
    double carry = 0x1p-53 * (golden - floor(golden) - 0.5);
    auto entry = [&](double e) {
        if (table_of_e(d, n)) return e;
        const double w = e + carry, ck = 1.0 - w;
        carry = (ck - 1.0) + w;  // exact (|w| < 1)
        return ck;
    };
    if (power.h == 0.0) {
        for (int k = k0; k < k1; ++k) c[(int64_t)k * lines + l] = entry(e1.h);
    } else {
        for (int k = k0; k < k1; ++k) {
            power = dd_mul(power, r2);  // r^(2k+1)
            c[(int64_t)k * lines + l] = entry(e_of(power));
        }
    }
    // the middle: 2 + lambda - 2 c = lambda + 2 e, k = n/2 - 1
    if (k1 == n / 2) c[(int64_t)k1 * lines + l] = 1.0 / (lambda + 2.0 * e_of(power));
}

// c v and c v + d from the table's entry x: c = x, or (E) c = 1 - x
template <bool E>
__device__ inline double times_c(double v, double x) {
    return E ? fma(-x, v, v) : v * x;
}
template <bool E>
__device__ inline double times_c_plus(double v, double x, double d) {
    return E ? v + fma(-x, v, d) : fma(x, v, d);
}

// `count` steps v[k dv] -> f(v[k dv], c[k dc]), k = 0.. ; the operands of kB
// steps are loaded together.  STORE: f's value replaces v[k dv].
constexpr int kB = 8;
template <bool STORE, class F>
__device__ inline void chain(double* __restrict__ v, int64_t dv, const double* __restrict__ c,
                             int64_t dc, int count, F&& f) {
    for (int k0 = 0; k0 < count; k0 += kB) {
        double a[kB], b[kB];
#pragma unroll
        for (int t = 0; t < kB; ++t)
            if (k0 + t < count) {
                a[t] = v[(k0 + t) * dv];
                b[t] = c[(k0 + t) * dc];
            }
#pragma unroll
        for (int t = 0; t < kB; ++t)
            if (k0 + t < count) {
                const double w = f(a[t], b[t]);
                if (STORE) v[(k0 + t) * dv] = w;
            }
    }
}

// 3D: one thread per half line; x along the lanes, threadIdx.y the half (0:
// from k = 1 up, 1: from k = n-1 down), threadIdx.z one of the CTA's rows.
// 3 FP64 instructions and (with the coefficients, read twice) 40 bytes per
// node: 125 us at 257^3, 78% of the FP64 pipe.
__global__ void __launch_bounds__(256) k_lines(double* __restrict__ w, const double* __restrict__ c,
                                               int n, int64_t step, double scale) {
    __shared__ double tip[4][2][32];
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.z;
    const int half = threadIdx.y;
    // column 0 and row 0 of the transformed axes hold no coefficient
    const bool in = x > 0 && x < n && y > 0 && y < n;
    const int m = n / 2;
    const int64_t l = (int64_t)y * n + x;
    double* v = w + l + (half ? (int64_t)n * step : 0);
    const int64_t dir = half ? -step : step;
    const double* cl = c + l;
    double prev = 0.0, dm = 0.0;
    if (in) {
        chain<true>(v + dir, dir, cl + step, step, m - 1,
                    [&](double d, double ck) { return prev = fma(scale, d, prev) * ck; });
        tip[threadIdx.z][half][threadIdx.x] = prev;
        dm = v[m * dir];  // the same entry for both halves, read before it is replaced
    }
    __syncthreads();
    if (!in) return;
    prev = (fma(scale, dm, tip[threadIdx.z][0][threadIdx.x]) +
            tip[threadIdx.z][1][threadIdx.x]) *
           cl[m * step];
    if (half == 0) v[m * dir] = prev;
    chain<true>(v + (m - 1) * dir, -dir, cl + (m - 1) * step, -step, m - 1,
                [&](double d, double ck) { return prev = fma(ck, prev, d); });
}

// 2D has only n - 1 lines, too few for their chains (192 cycles of dependent
// FP64 a node) to be hidden: each half line is cut into kC pieces with a
// thread each.  Both recurrences are linear in what flows into a piece, so a
// first pass over the piece with inflow 0 gives its outflow t and the factor
// p = prod c_k of its inflow, the inflows follow from those, and a second
// pass stores the values.  9 instructions per node instead of 4 (c_k: 7 of 3), a
// chain 1/16 as long: 356 us at 4097^2, 12.0 at 257^2 (one piece a line: 578 and
// 33 with a table of c_k, which would take 319 in pieces).
// X columns to a CTA: 16 (128-byte rows) where that makes enough CTAs, else 8.
constexpr int kC = 16;
// E: the table holds e_k (table_of_e)
template <int X, bool E>
__global__ void __launch_bounds__(2 * X * kC) k_lines_2d(double* __restrict__ w,
                                                      const double* __restrict__ c, int n,
                                                      double scale) {
    __shared__ double out[2][kC][X], fac[2][kC][X];
    const int tx = threadIdx.x, half = threadIdx.y & 1, piece = threadIdx.y >> 1;
    const int x = blockIdx.x * X + tx;
    const bool in = x > 0 && x < n;
    const int m = n / 2, len = (m - 1 + kC - 1) / kC;
    const int k0 = 1 + piece * len, count = max(0, min(len, m - k0));  // k = k0 ..
    const int64_t step = n;
    double* v = w + x + (half ? (int64_t)n * step : 0);
    const int64_t dir = half ? -step : step;
    const double* cl = c + x;
    double t = 0.0, p = 1.0, dm = 0.0;
    if (in) {
        chain<false>(v + k0 * dir, dir, cl + k0 * step, step, count, [&](double d, double e) {
            p = times_c<E>(p, e);
            return t = times_c<E>(fma(scale, d, t), e);
        });
        dm = v[m * dir];  // read before it is replaced
    }
    out[half][piece][tx] = t;
    fac[half][piece][tx] = p;
    __syncthreads();
    // flow[h]: what flows into this piece (own half) and into the middle
    double prev = 0.0, tip[2] = {0.0, 0.0};
#pragma unroll
    for (int h = 0; h < 2; ++h)
        for (int i = 0; i < kC; ++i) {
            if (h == half && i == piece) prev = tip[h];
            tip[h] = fma(fac[h][i][tx], tip[h], out[h][i][tx]);
        }
    double mid = 0.0;
    if (in) {
        mid = (fma(scale, dm, tip[0]) + tip[1]) * cl[m * step];
        chain<true>(v + k0 * dir, dir, cl + k0 * step, step, count,
                    [&](double d, double e) { return prev = times_c<E>(fma(scale, d, prev), e); });
        // back substitution from the piece's far end
        t = 0.0;
        chain<false>(v + (k0 + count - 1) * dir, -dir, cl + (k0 + count - 1) * step, -step, count,
                     [&](double d, double e) { return t = times_c_plus<E>(t, e, d); });
    }
    __syncthreads();
    out[half][piece][tx] = t;
    __syncthreads();
    if (!in) return;
    prev = mid;
    for (int i = kC - 1; i > piece; --i) prev = fma(fac[half][i][tx], prev, out[half][i][tx]);
    if (half == 0 && piece == 0) v[m * dir] = mid;
    chain<true>(v + (k0 + count - 1) * dir, -dir, cl + (k0 + count - 1) * step, -step, count,
                [&](double d, double e) { return prev = times_c_plus<E>(prev, e, d); });
}

}  // namespace
}  // namespace fft
}  // namespace gmg

using namespace gmg;
using namespace gmg::fft;

struct gmg_fft_s {
    int d = 3, n = 0, device = 0;
    cudaStream_t user_stream = nullptr, stream = nullptr;
    cudaEvent_t ev = nullptr;
    Plan plan;
    double2* twiddles = nullptr;  // e^{i pi k/n}, k < 2n
    double* coeffs = nullptr;     // the eliminations' coefficients, n/2 + 1 rows
    double* work = nullptr;       // n^d
};

namespace {

// A tile of up to 256 threads holds at most 37 KB (3D n = 128), which needs no opt-in; one
// of 512 threads up to 144 KB (2D n = 8192).  The limit belongs to the kernel,
// not to a plan: it is one value for all of them, so that making one plan does
// not lower it under another's launches.
constexpr size_t kSmem512 = Plan{13, 0, 512}.smem();

cudaError_t allow_smem() {
    cudaError_t e = cudaFuncSetAttribute(k_dst_x<512>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmem512);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_dst_y<512>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmem512);
    return e;
}

void dst_x(gmg_fft h, const double* src, int64_t ssy, int64_t ssz, double* dst, int64_t dsy,
           int64_t dsz, int whole_u) {
    const int64_t m = h->n - 1, lines = h->d == 3 ? m * m : m;
    const unsigned blocks = (unsigned)(((lines + 1) / 2 + h->plan.pairs() - 1) / h->plan.pairs());
    auto kern = h->plan.threads > 256 ? k_dst_x<512> : k_dst_x<256>;
    kern<<<blocks, h->plan.threads, h->plan.smem(), h->stream>>>(src, ssy, ssz, dst, dsy, dsz,
                                                                   lines, h->d, h->plan, whole_u,
                                                                   h->twiddles);
}

void dst_y(gmg_fft h) {
    const int64_t pairs = (int64_t)(h->n - 1) * (h->n / 2);
    const unsigned blocks = (unsigned)((pairs + h->plan.pairs() - 1) / h->plan.pairs());
    auto kern = h->plan.threads > 256 ? k_dst_y<512> : k_dst_y<256>;
    kern<<<blocks, h->plan.threads, h->plan.smem(), h->stream>>>(h->work, pairs, h->plan,
                                                                   h->twiddles);
}

}  // namespace

extern "C" {

gmg_status gmg_fft_destroy(gmg_fft h) {
    if (!h) return GMG_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    cudaFree(h->twiddles);
    cudaFree(h->coeffs);
    cudaFree(h->work);
    if (h->ev) cudaEventDestroy(h->ev);
    if (h->stream) cudaStreamDestroy(h->stream);
    delete h;
    return GMG_OK;
}

gmg_status gmg_fft_create(int d, int n, void* cuda_stream, gmg_fft* out) {
    if (!out) {
        set_error("out is NULL");
        return GMG_ERR_ARG;
    }
    *out = nullptr;
    const int nmax = d == 2 ? 8192 : 1024;
    if ((d != 2 && d != 3) || n < 2 || n > nmax || (n & (n - 1))) {
        set_error("gmg_fft_create: d must be 2 or 3 and n a power of two within limits");
        return GMG_ERR_ARG;
    }
    gmg_fft h = new gmg_fft_s();
    h->d = d;
    h->n = n;
    h->user_stream = (cudaStream_t)cuda_stream;
    h->plan = plan_of(n, d == 3 ? (int64_t)(n - 1) * (n - 1) / 2 : n / 2);
    auto fail = [&](gmg_status s, const std::string& m) {
        set_error("gmg_fft_create: " + m);
        gmg_fft_destroy(h);
        return s;
    };
    if (cudaGetDevice(&h->device) != cudaSuccess) return fail(GMG_ERR_CUDA, "no device");
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev, cudaEventDisableTiming) != cudaSuccess)
        return fail(GMG_ERR_CUDA, "stream/event creation failed");
    const int64_t lines = d == 3 ? (int64_t)n * n : n;
    if (cudaMalloc(&h->twiddles, sizeof(double2) * 2 * n) != cudaSuccess ||
        cudaMalloc(&h->coeffs, sizeof(double) * lines * (n / 2 + 1)) != cudaSuccess ||
        cudaMalloc(&h->work, sizeof(double) * lines * n) != cudaSuccess)
        return fail(GMG_ERR_ALLOC, "cudaMalloc failed");
    if (h->plan.threads > 256 && allow_smem() != cudaSuccess)
        return fail(GMG_ERR_CUDA, "cudaFuncSetAttribute failed");
    // cos and sin of the first octant (long double: every entry correctly rounded up
    // to the rounding of a small argument), the other octants from it
    std::vector<double> t(4 * (size_t)n), oct_c(n / 4 + 1), oct_s(n / 4 + 1);
    for (int r = 0; r <= n / 4; ++r) {
        const long double a = 3.14159265358979323846264338327950288L * r / n;
        oct_c[r] = (double)cosl(a);
        oct_s[r] = (double)sinl(a);
    }
    for (int k = 0; k < 2 * n; ++k) {
        const int oct = (int)((int64_t)4 * k / n), r = k - (int)((int64_t)oct * n / 4);
        double c, s;
        if (n < 4) {  // k multiples of pi/2
            const double cs[4] = {1, 0, -1, 0}, sn[4] = {0, 1, 0, -1};
            c = cs[(k * (2 / n)) & 3];
            s = sn[(k * (2 / n)) & 3];
        } else {
            const bool odd = oct & 1;  // measured back from the octant's end
            const double ca = oct_c[odd ? n / 4 - r : r], sa = oct_s[odd ? n / 4 - r : r];
            const int quad = ((oct + 1) / 2) & 3;  // nearest multiple of pi/2, angle = quad pi/2 +- a
            const double sg = odd ? -1.0 : 1.0;
            const double cc[4] = {ca, -sg * sa, -ca, sg * sa}, ss[4] = {sg * sa, ca, -sg * sa, -ca};
            c = cc[quad];
            s = ss[quad];
        }
        t[2 * k] = c;
        t[2 * k + 1] = s;
    }
    if (cudaMemcpyAsync(h->twiddles, t.data(), sizeof(double) * t.size(), cudaMemcpyHostToDevice,
                        h->stream) != cudaSuccess ||
        cudaMemsetAsync(h->work, 0, sizeof(double) * lines * n, h->stream) != cudaSuccess)
        return fail(GMG_ERR_CUDA, "initialisation failed");
    const unsigned segs = (unsigned)std::max(1, (n / 2 - 1 + kSeg - 1) / kSeg);
    k_coeffs<<<dim3((unsigned)((lines + 127) / 128), segs), 128, 0, h->stream>>>(h->coeffs, d, n);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(h->stream) != cudaSuccess)
        return fail(GMG_ERR_CUDA, "initialisation failed");
    *out = h;
    return GMG_OK;
}

gmg_status gmg_fft_solve(gmg_fft h, const double* f, double* u) {
    if (!h || !f || !u) {
        set_error("gmg_fft_solve: NULL argument");
        return GMG_ERR_ARG;
    }
    const int d = h->d, n = h->n;
    cudaStream_t s = h->stream;
    GMG_CUDA_TRY(cudaEventRecord(h->ev, h->user_stream));
    GMG_CUDA_TRY(cudaStreamWaitEvent(s, h->ev, 0));
    const int64_t m = n + 1, mz = d == 3 ? m * m : 0;
    const int64_t wy = n, wz = d == 3 ? (int64_t)n * n : 0;
    dst_x(h, f, m, mz, h->work, wy, wz, 0);
    if (d == 3) dst_y(h);
    // h^2, the inverse transforms' (2/n)^(d-1) and a half per transform: a power
    // of two, exact
    const double scale = std::pow(0.5 / n, d - 1) / ((double)n * n);
    if (d == 3)
        k_lines<<<dim3((n + 31) / 32, (n + 3) / 4), dim3(32, 2, 4), 0, s>>>(h->work, h->coeffs, n,
                                                                            wz, scale);
    else if (n >= 2048)
        k_lines_2d<16, true><<<n / 16, dim3(16, 2 * kC), 0, s>>>(h->work, h->coeffs, n, scale);
    else if (table_of_e(d, n))
        k_lines_2d<8, true><<<(n + 7) / 8, dim3(8, 2 * kC), 0, s>>>(h->work, h->coeffs, n, scale);
    else
        k_lines_2d<8, false><<<(n + 7) / 8, dim3(8, 2 * kC), 0, s>>>(h->work, h->coeffs, n, scale);
    if (d == 3) dst_y(h);
    dst_x(h, h->work, wy, wz, u, m, mz, 1);
    GMG_CUDA_TRY(cudaGetLastError());
    GMG_CUDA_TRY(cudaStreamSynchronize(s));
    return GMG_OK;
}

}  // extern "C"
