// One level of a 2D FP64 V-cycle in two launches.
//
//   down leg: the pre-smoothing steps, the residual, the restriction;
//   up leg:   the prolongation with correction, the post-smoothing steps.
//
// On the 2D levels up to about 1025^2 a launch per step costs 2.5 to 3 us, of
// which the FP64 work is a fraction (65k nodes x 8 instructions: 1 us of the
// whole chip): 1.25 us of launch, the rest the latency of its L2 loads.  A CTA
// here takes a tile of fine nodes with a halo of one node per smoothing step
// and runs every step in shared memory, each on a region one node smaller,
// so the halo is computed again by its neighbours instead of exchanged.  The
// iterate is read from one array and written to the other (the neighbours
// still read the old one).  Every node value is the level kernels' expression
// of the same operands (level_kernels.cuh), so the results are theirs bit for
// bit.
//
// Tiles: about one per SM (152) as long as the halo allows, since the FP64
// pipe, 1.6 lanes a cycle and SM, is what the steps wait for: 8 x 8 up to 65^2,
// 16 x 8 at 129^2, 32 x 16 at 257^2, 64 x 32 at 513^2.
//
// Measured per leg (a launch per step): weighted Jacobi V(2,2) at 257^2 10 + 6.5
// us (8 + 8.5 with the first sweep done by the restriction), at 129^2 and below
// about 4 + 4 (8 + 8).  Whole solves, launch per step -> legs and a tail from
// 17^2 instead of 33^2: 257^2 Jacobi 1185 -> 887 us, 1025^2 paper variant V(1,1)
// 2199 -> 1762, 2049^2 FMG 2424 -> 2209.  Above 513^2 the steps are bound by the
// FP64 pipe and the halo's work is more than the launches it saves (1025^2 in
// the paper variant: 1762 -> 1814 us; 2049^2 FMG: 2209 -> 2414).
#include <algorithm>

#include "level_kernels.cuh"

namespace gmg {
namespace legs2d {
namespace {

constexpr int kThreads = 512;  // at most (threads_of)
constexpr double kC = 0.25;  // 1/(2d)

// Smoothing steps of one node per halo layer: a weighted-Jacobi sweep, a
// colour of the red-black sweep, or of the paper's four colours 0, (1 and 2),
// 3 -- 1 and 2 are the black nodes and do not touch one another.
enum { WJ = 0, RB = 1, MC = 2 };
__host__ __device__ inline int steps_of(int sm, int sweeps, bool first_done) {
    return (sm == WJ ? 1 : sm == RB ? 2 : 3) * sweeps - (first_done ? 1 : 0);
}

// A tile with its halo: shared-memory entry of fine node (i, j) is
// (j - j0) * pitch + i - i0.
struct Box {
    int i0, j0, pitch, rows;
    __device__ int at(int i, int j) const { return (j - j0) * pitch + i - i0; }
};

// f(i, j) for the nodes of the rectangle [ia, ib] x [ja, jb]; par >= 0: only
// those with i + j = par (mod 2); odd_i >= 0: of these, only those with i =
// odd_i (mod 2), par even then (the paper's colours 0 and 3).
template <class F>
__device__ inline void nodes(int ia, int ib, int ja, int jb, int par, int odd_i, F&& f) {
    if (odd_i >= 0) {
        ia += (ia ^ odd_i) & 1;
        ja += (ja ^ odd_i) & 1;
    }
    const int sx = par < 0 ? 1 : 2, sy = odd_i >= 0 ? 2 : 1;
    // rows of the red-black colours hold (width + 1) / 2 slots, the last of
    // which may be idle
    const int w = (ib - ia + sx) / sx, h = (jb - ja + sy) / sy;
    if (w <= 0 || h <= 0) return;
    const float inv = 1.0f / (float)w;
    for (int idx = threadIdx.x; idx < w * h; idx += blockDim.x) {
        const int y = (int)(((float)idx + 0.5f) * inv);  // exact: idx < 2^15
        const int j = ja + sy * y;
        int i = ia + sx * (idx - y * w);
        if (par >= 0 && odd_i < 0) i += (ia + j + par) & 1;
        if (i <= ib) f(i, j);
    }
}

// The smoothing steps on the box, step s of S on the tile [ti, ti + TX) x
// [tj, tj + TY) widened by lo + S-1-s nodes below and hi + S-1-s above.
// Returns the buffer that holds the iterate (0: u, 1: u2).
template <int SM>
__device__ int smooth(const Box& B, double* u, double* u2, const double* q, int n, int ti, int tj,
                      int TX, int TY, int lo, int hi, int S, bool first_done, bool backward,
                      double omega) {
    int cur = 0;
    for (int s = 0; s < S; ++s) {
        const int e = S - 1 - s;
        const int ia = max(1, ti - lo - e), ib = min(n - 1, ti + TX - 1 + hi + e);
        const int ja = max(1, tj - lo - e), jb = min(n - 1, tj + TY - 1 + hi + e);
        const double* a = SM == WJ && cur ? u2 : u;
        double* b = SM == WJ ? (cur ? u : u2) : u;
        int par = -1, odd = -1;
        if (SM == RB) par = (s + (first_done ? 1 : 0)) & 1;
        if (SM == MC) {
            const int t = (s + (first_done ? 1 : 0)) % 3;
            par = t == 1 ? 1 : 0;
            if (t != 1) odd = (t == 2) != backward ? 1 : 0;  // colours 3 and 0
        }
        nodes(ia, ib, ja, jb, par, odd, [&](int i, int j) {
            const int p = B.at(i, j);
            const double v =
                lk::gs_value<2, false>(kC, lk::nbr_sum<2>(a, p, B.pitch, 0), q[p]);
            b[p] = SM == WJ ? fma(omega, v - a[p], a[p]) : v;
        });
        if (SM == WJ) cur ^= 1;
        __syncthreads();
    }
    return cur;
}

// Load the box's nodes of arrays a (and b) of a dense level n; zero outside the
// grid.  Four nodes per thread in flight.
__device__ inline void load_box(const Box& B, int n, const double* __restrict__ a, double* sa,
                                const double* __restrict__ b, double* sb) {
    constexpr int U = 4;
    const float inv = 1.0f / (float)B.pitch;
    const int total = B.pitch * B.rows;
    for (int e0 = threadIdx.x; e0 < total; e0 += U * blockDim.x) {
        double va[U], vb[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int e = e0 + t * (int)blockDim.x;
            va[t] = vb[t] = 0.0;
            if (e < total) {
                const int y = (int)(((float)e + 0.5f) * inv);
                const int i = B.i0 + e - y * B.pitch, j = B.j0 + y;
                if (i > 0 && i < n && j > 0 && j < n) {
                    const int64_t g = (int64_t)j * (n + 1) + i;
                    va[t] = a[g];
                    if (b) vb[t] = b[g];
                }
            }
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int e = e0 + t * (int)blockDim.x;
            if (e < total) {
                sa[e] = va[t];
                if (b) sb[e] = vb[t];
            }
        }
    }
}

struct Args {
    int n, TX, TY, S;
    int first_done, paper, red_only, init;  // down
    int black;                              // up: a red half sweep follows
    double omega;
};

// Down leg: u -> uo (smoothed), q_c and u_c of the coarse level.
template <int SM>
__global__ void __launch_bounds__(kThreads) k_down(const double* __restrict__ u,
                                                   double* __restrict__ uo,
                                                   const double* __restrict__ q,
                                                   double* __restrict__ qc,
                                                   double* __restrict__ uc, Args A) {
    extern __shared__ double sm[];
    const int n = A.n, TX = A.TX, TY = A.TY, S = A.S;
    const int ti = blockIdx.x * TX, tj = blockIdx.y * TY;
    // the residual on one node around the tile's coarse nodes needs the
    // smoothed iterate on [-2, TX]
    const Box B{ti - 2 - S, tj - 2 - S, TX + 3 + 2 * S, TY + 3 + 2 * S};
    const int size = B.pitch * B.rows;
    double *su = sm, *sq = sm + size, *sr = sm + 2 * size;
    load_box(B, n, u, su, q, sq);
    if (SM == WJ)  // the other buffer's boundary and halo are read too
        for (int e = threadIdx.x; e < size; e += blockDim.x) sr[e] = 0.0;
    __syncthreads();
    const int cur = smooth<SM>(B, su, sr, sq, n, ti, tj, TX, TY, 2, 1, S, A.first_done, false,
                               A.omega);
    double* v = cur ? sr : su;  // smoothed
    double* r = cur ? su : sr;
    if (SM == WJ || !A.red_only) {
        // the residual's zero boundary (and, red only, its black nodes are not read)
        for (int e = threadIdx.x; e < size; e += blockDim.x) r[e] = 0.0;
        __syncthreads();
    }
    nodes(max(1, ti - 1), min(n - 1, ti + TX - 1), max(1, tj - 1), min(n - 1, tj + TY - 1),
          A.red_only ? 0 : -1, -1, [&](int i, int j) {
              const int p = B.at(i, j);
              r[p] = lk::gs_value<2, false>(kC, lk::nbr_sum<2>(v, p, B.pitch, 0), sq[p]) - v[p];
          });
    nodes(max(1, ti), min(n - 1, ti + TX - 1), max(1, tj), min(n - 1, tj + TY - 1), -1, -1,
          [&](int i, int j) { uo[(int64_t)j * (n + 1) + i] = v[B.at(i, j)]; });
    __syncthreads();
    const int nc = n / 2, sy = B.pitch;
    nodes(max(1, ti / 2), min(nc - 1, ti / 2 + TX / 2 - 1), max(1, tj / 2),
          min(nc - 1, tj / 2 + TY / 2 - 1), -1, -1, [&](int I, int J) {
              const int p = B.at(2 * I, 2 * J);
              auto R = [&](int o) { return r[p + o]; };
              double w;
              if (A.paper) {
                  double s = (R(-1) + R(1)) + (R(-sy) + R(sy));
                  s += R(-1 - sy) + R(1 + sy);
                  w = fma(0.5, s, R(0));
              } else {
                  double co = R(-1 - sy) + R(1 - sy);
                  co += R(-1 + sy);
                  co += R(1 + sy);
                  if (A.red_only) {
                      w = fma(0.25, co, R(0));
                  } else {
                      double fc = R(-1) + R(1);
                      fc += R(-sy);
                      fc += R(sy);
                      w = fma(0.25, co, fma(0.5, fc, R(0)));
                  }
              }
              const int64_t P = (int64_t)J * (nc + 1) + I;
              qc[P] = w;
              uc[P] = lk::coarse_init<2>(A.init, A.omega, I, J, 0, w);
          });
}

// Up leg: u + P u_c, smoothed, into uo.
template <int SM>
__global__ void __launch_bounds__(kThreads) k_up(const double* __restrict__ uc,
                                                 const double* __restrict__ u,
                                                 double* __restrict__ uo,
                                                 const double* __restrict__ q, Args A) {
    extern __shared__ double sm[];
    const int n = A.n, TX = A.TX, TY = A.TY, S = A.S;
    const int ti = blockIdx.x * TX, tj = blockIdx.y * TY;
    const Box B{ti - S, tj - S, TX + 2 * S, TY + 2 * S};
    const int size = B.pitch * B.rows;
    double *su = sm, *sq = sm + size, *s2 = sm + 2 * size;
    load_box(B, n, q, sq, nullptr, nullptr);
    if (SM == WJ)
        for (int e = threadIdx.x; e < size; e += blockDim.x) s2[e] = 0.0;
    // the coarse cells that hold the box's nodes
    const int64_t cy = n / 2 + 1;
    const int Ia = B.i0 >> 1, Ib = (B.i0 + B.pitch - 1) >> 1;
    const int Ja = B.j0 >> 1, Jb = (B.j0 + B.rows - 1) >> 1;
    nodes(Ia, Ib, Ja, Jb, -1, -1, [&](int I, int J) {
        auto on = [&](int v) {  // in the box
            const int i = 2 * I + (v & 1), j = 2 * J + (v >> 1);
            return i >= B.i0 && i < B.i0 + B.pitch && j >= B.j0 && j < B.j0 + B.rows;
        };
        auto inner = [&](int v) {
            const int i = 2 * I + (v & 1), j = 2 * J + (v >> 1);
            return i > 0 && i < n && j > 0 && j < n;
        };
        double f[4];
#pragma unroll
        for (int v = 0; v < 4; ++v)
            f[v] = on(v) && inner(v)
                       ? u[(int64_t)(2 * J + (v >> 1)) * (n + 1) + 2 * I + (v & 1)]
                       : 0.0;
        if (I >= 0 && I < n / 2 && J >= 0 && J < n / 2) {
            const int64_t P = J * cy + I;
            const double c00 = uc[P], c10 = uc[P + 1], c01 = uc[P + cy], c11 = uc[P + 1 + cy];
            const double x0 = c00 + c10, y0 = c00 + c01;
            if (!A.black && inner(0)) f[0] = f[0] + c00;
            if (inner(1)) f[1] = fma(0.5, x0, f[1]);
            if (inner(2)) f[2] = fma(0.5, y0, f[2]);
            if (!A.black && inner(3))
                f[3] = A.paper ? fma(0.5, c00 + c11, f[3]) : fma(0.25, x0 + (c01 + c11), f[3]);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (on(v)) su[B.at(2 * I + (v & 1), 2 * J + (v >> 1))] = f[v];
    });
    __syncthreads();
    const int cur = smooth<SM>(B, su, s2, sq, n, ti, tj, TX, TY, 0, 0, S, false, true, A.omega);
    const double* v = cur ? s2 : su;
    nodes(max(1, ti), min(n - 1, ti + TX - 1), max(1, tj), min(n - 1, tj + TY - 1), -1, -1,
          [&](int i, int j) { uo[(int64_t)j * (n + 1) + i] = v[B.at(i, j)]; });
}

void tile_of(int n, int& tx, int& ty) {
    tx = n <= 64 ? 8 : n <= 128 ? 16 : n <= 256 ? 32 : 64;
    ty = n <= 128 ? 8 : n <= 256 ? 16 : 32;
}
int threads_of(int n) { return n <= 256 ? 256 : 512; }
int kind_of(int smoother) {
    return smoother == GMG_WJACOBI ? WJ : smoother == GMG_RBGS ? RB : smoother == GMG_MCGS ? MC : -1;
}

constexpr int kSteps = 6;  // smoothing steps of a leg at most (applies)
constexpr size_t down_bytes(int tx, int ty, int S) {
    return sizeof(double) * 3 * (tx + 3 + 2 * S) * (ty + 3 + 2 * S);
}
constexpr size_t up_bytes(int arrays, int tx, int ty, int S) {
    return sizeof(double) * arrays * (tx + 2 * S) * (ty + 2 * S);
}
// The limit belongs to the kernel, not to the launch: the largest tile's (64 x
// 32, tile_of) for all, so that no thread lowers it between another's limit and
// launch.
constexpr size_t kSmem = std::max(down_bytes(64, 32, kSteps), up_bytes(3, 64, 32, kSteps));
template <class K>
cudaError_t allow(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

}  // namespace

bool applies(int n, int nmax, int smoother, int nu1, int nu2) {
    const int k = kind_of(smoother);
    if (k < 0 || n < 32 || nu1 < 1 || nu2 < 1) return false;
    // six steps: the halo is still smaller than the small tiles
    return steps_of(k, nu1, false) <= kSteps && steps_of(k, nu2, false) <= kSteps &&
           n <= (nmax > 0 ? nmax : 512);
}

cudaError_t down(int n, int smoother, int nu1, bool first_done, double omega, bool paper,
                 bool red_only, int init, const double* u, double* uo, const double* q, double* qc,
                 double* uc, cudaStream_t s) {
    Args A{};
    A.n = n;
    tile_of(n, A.TX, A.TY);
    const int k = kind_of(smoother);
    A.S = steps_of(k, nu1, first_done);
    A.first_done = k != WJ && first_done;
    A.paper = paper;
    A.red_only = red_only;
    A.init = init;
    A.omega = omega;
    const size_t bytes = down_bytes(A.TX, A.TY, A.S);
    auto kern = k == WJ ? k_down<WJ> : k == RB ? k_down<RB> : k_down<MC>;
    cudaError_t e = allow(kern);
    if (e != cudaSuccess) return e;
    kern<<<dim3((n + A.TX - 1) / A.TX, (n + A.TY - 1) / A.TY), threads_of(n), bytes, s>>>(u, uo, q, qc,
                                                                                    uc, A);
    return cudaGetLastError();
}

cudaError_t up(int n, int smoother, int nu2, double omega, bool paper, const double* uc,
               const double* u, double* uo, const double* q, cudaStream_t s) {
    Args A{};
    A.n = n;
    tile_of(n, A.TX, A.TY);
    const int k = kind_of(smoother);
    A.S = steps_of(k, nu2, false);
    A.paper = paper;
    A.black = k == RB;
    A.omega = omega;
    const size_t bytes = up_bytes(k == WJ ? 3 : 2, A.TX, A.TY, A.S);
    auto kern = k == WJ ? k_up<WJ> : k == RB ? k_up<RB> : k_up<MC>;
    cudaError_t e = allow(kern);
    if (e != cudaSuccess) return e;
    kern<<<dim3((n + A.TX - 1) / A.TX, (n + A.TY - 1) / A.TY), threads_of(n), bytes, s>>>(uc, u, uo, q,
                                                                                    A);
    return cudaGetLastError();
}

}  // namespace legs2d
}  // namespace gmg
