// Learned smoother: a per-level convolutional smoother u <- u + N(sigma),
// sigma = (b - A'u)/(2d), N = conv2(ReLU(conv1(sigma))) with conv1: 1 -> 8
// channels and conv2: 8 -> 1 channel, 3^d taps, zero padding at the
// Dirichlet boundary, no biases, BF16 weights with FP32 accumulation.
//
// Training minimises the measured two-grid error contraction
//     L = ||S(CG(S(e0)))||^2 / ||e0||^2,  S e = e - N(A'e/(2d)),
//     CG e = e - P A_c'^{-1} 4 FW(A'e),
// over error samples e0 drawn from plain red-black V(1,1) cycles applied to
// seeded white noise, with this file's forward and backward kernels and an
// Adam step, all on the GPU.  The coarse system inside the loss is solved by
// red-black V(2,2) cycles run to round-off.
//
// Weight layout (host and device): 2 x 8 x T floats, W1[c][t] then W2[c][t],
// tap t = (c3+1)*9 + (b+1)*3 + (a+1) for the offset (a, b, c3) (x fastest);
// T = 27 in 3D, 9 in 2D.
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "gmg_internal.cuh"
#include "level_kernels.cuh"

namespace gmg {
namespace learned {
namespace {

constexpr int H = 8;  // hidden channels

using lk::sy_of;
using lk::sz_of;

template <int DIM>
constexpr int taps() {
    return DIM == 3 ? 27 : 9;
}

template <int DIM>
__device__ inline int64_t tap_offset(int t, int64_t sy, int64_t sz) {
    const int a = t % 3 - 1, b = (t / 3) % 3 - 1, c = DIM == 3 ? t / 9 - 1 : 0;
    return a + b * sy + c * sz;
}

template <int DIM>
__device__ inline void load_weights(const float* W, float* ws) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nt = blockDim.x * blockDim.y;
    for (int i = tid; i < 2 * H * taps<DIM>(); i += nt) ws[i] = W[i];
    __syncthreads();
}

// z_c(p) = sum_t W1[c][t] x(p + o_t) on interior nodes (x is zero on the
// boundary; z's boundary entries are never written and stay zero)
template <int DIM, typename TI>
__global__ void __launch_bounds__(256) k_conv1(const TI* __restrict__ x, float* __restrict__ z,
                                               int n, int64_t zs, const float* __restrict__ W) {
    constexpr int T = taps<DIM>();
    __shared__ float ws[2 * H * T];
    load_weights<DIM>(W, ws);
    const int j = blockIdx.x * blockDim.y + threadIdx.y + 1;
    const int k = DIM == 3 ? blockIdx.y + 1 : 0;
    if (j >= n) return;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t row = k * sz + j * sy;
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const int64_t p = row + i;
        float xv[T];
#pragma unroll
        for (int t = 0; t < T; ++t) xv[t] = (float)x[p + tap_offset<DIM>(t, sy, sz)];
#pragma unroll
        for (int c = 0; c < H; ++c) {
            float acc = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t) acc = fmaf(ws[c * T + t], xv[t], acc);
            z[c * zs + p] = acc;
        }
    }
}

// y(p) = sum_c sum_t W2[c][t] relu(z_c(p + o_t)); mode 0: out = y,
// 1: out += y, 2: out -= y (out in FP64)
template <int DIM, int MODE>
__global__ void __launch_bounds__(256) k_conv2(const float* __restrict__ z, double* __restrict__ out,
                                               int n, int64_t zs, const float* __restrict__ W) {
    constexpr int T = taps<DIM>();
    __shared__ float ws[2 * H * T];
    load_weights<DIM>(W, ws);
    const int j = blockIdx.x * blockDim.y + threadIdx.y + 1;
    const int k = DIM == 3 ? blockIdx.y + 1 : 0;
    if (j >= n) return;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t row = k * sz + j * sy;
    const float* w2 = ws + H * T;
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const int64_t p = row + i;
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < H; ++c)
#pragma unroll
            for (int t = 0; t < T; ++t)
                acc = fmaf(w2[c * T + t], fmaxf(z[c * zs + p + tap_offset<DIM>(t, sy, sz)], 0.f), acc);
        if (MODE == 0)
            out[p] = (double)acc;
        else if (MODE == 1)
            out[p] += (double)acc;
        else
            out[p] -= (double)acc;
    }
}

// gz_c(p) = [z_c(p) > 0] * sum_t W2[c][t] gy(p - o_t)
template <int DIM>
__global__ void __launch_bounds__(256) k_conv2_bwd(const double* __restrict__ gy,
                                                   const float* __restrict__ z,
                                                   float* __restrict__ gz, int n, int64_t zs,
                                                   const float* __restrict__ W) {
    constexpr int T = taps<DIM>();
    __shared__ float ws[2 * H * T];
    load_weights<DIM>(W, ws);
    const int j = blockIdx.x * blockDim.y + threadIdx.y + 1;
    const int k = DIM == 3 ? blockIdx.y + 1 : 0;
    if (j >= n) return;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t row = k * sz + j * sy;
    const float* w2 = ws + H * T;
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const int64_t p = row + i;
        float gv[T];
#pragma unroll
        for (int t = 0; t < T; ++t) gv[t] = (float)gy[p - tap_offset<DIM>(t, sy, sz)];
#pragma unroll
        for (int c = 0; c < H; ++c) {
            float acc = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t) acc = fmaf(w2[c * T + t], gv[t], acc);
            gz[c * zs + p] = z[c * zs + p] > 0.f ? acc : 0.f;
        }
    }
}

// gx(p) = sum_c sum_t W1[c][t] gz_c(p - o_t)
template <int DIM>
__global__ void __launch_bounds__(256) k_conv1_bwd(const float* __restrict__ gz,
                                                   double* __restrict__ gx, int n, int64_t zs,
                                                   const float* __restrict__ W) {
    constexpr int T = taps<DIM>();
    __shared__ float ws[2 * H * T];
    load_weights<DIM>(W, ws);
    const int j = blockIdx.x * blockDim.y + threadIdx.y + 1;
    const int k = DIM == 3 ? blockIdx.y + 1 : 0;
    if (j >= n) return;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t row = k * sz + j * sy;
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const int64_t p = row + i;
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < H; ++c)
#pragma unroll
            for (int t = 0; t < T; ++t)
                acc = fmaf(ws[c * T + t], gz[c * zs + p - tap_offset<DIM>(t, sy, sz)], acc);
        gx[p] = (double)acc;
    }
}

__device__ inline int64_t interior_node(int d, int n, int64_t idx) {
    const int m = n - 1;
    const int i = (int)(idx % m) + 1;
    const int64_t t = idx / m;
    const int j = (int)(t % m) + 1;
    const int k = d == 3 ? (int)(t / m) + 1 : 0;
    return ((int64_t)k * (n + 1) + j) * (n + 1) + i;
}

// Weight-gradient partials over `rpb` consecutive interior rows, one thread
// per (channel, tap):  KIND 1: sum_p gz_c(p) x(p + o_t);  KIND 2: sum_p gy(p)
// relu(z_c(p + o_t)).  FP32 within the block, one double per (block, c, t),
// the nodes in row order.
// Each thread's sum is one chain of dependent FMAs, and a CTA of 216 of them
// per SM is all there is at 65^3, so what matters is how fast a step's two
// operands arrive: rows of up to kSeg nodes are staged in shared memory as
// floats, converted (and ReLU'd) once instead of once per tap and channel --
// the conversions from double run on the FP64 pipe (65^3: 235 -> 83 and 211
// -> 148 us).
constexpr int kSegW = 94;  // + 2 halo nodes: three 32-lane loads a row
template <int DIM, int KIND>
constexpr int wgrad_rows() {  // staged rows: the dense array's, then the channels'
    return KIND == 1 ? (DIM == 3 ? 9 : 3) + H : 1 + H * (DIM == 3 ? 9 : 3);
}
template <int DIM, int KIND>
__global__ void __launch_bounds__(256) k_wgrad(const double* __restrict__ dense,
                                               const float* __restrict__ chan, int n, int64_t zs,
                                               int rpb, double* __restrict__ partial) {
    constexpr int T = taps<DIM>();
    constexpr int NB = DIM == 3 ? 9 : 3;          // neighbour rows (dy, dz)
    constexpr int ND = KIND == 1 ? NB : 1;        // staged rows of the dense array
    constexpr int NC = KIND == 1 ? 1 : NB;        // of each channel
    // nodes i0 - 1 .. i0 + kSegW, rows 3 banks apart (W = 3 mod 32): a warp's 27
    // taps of a channel, and the next channel's, lie in different banks
    constexpr int W = kSegW + 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ float rows_s[wgrad_rows<DIM, KIND>() * W];
    const int ct = threadIdx.x;
    const bool on = ct < H * T;
    const int c = on ? ct / T : 0, t = on ? ct % T : 0;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t rows = DIM == 3 ? (int64_t)(n - 1) * (n - 1) : (n - 1);
    const int64_t r0 = (int64_t)blockIdx.x * rpb;
    const int64_t r1 = r0 + rpb < rows ? r0 + rpb : rows;
    // this thread's two operand rows; the tapped one starts at dx = t % 3
    const float* plain = rows_s + (KIND == 1 ? ND + c : 0) * W + 1;
    const float* tapped = rows_s + (KIND == 1 ? t / 3 : ND + c * NC + t / 3) * W + t % 3;
    float acc = 0.f;
    for (int64_t r = r0; r < r1; ++r) {
        const int j = (int)(r % (n - 1)) + 1;
        const int k = DIM == 3 ? (int)(r / (n - 1)) + 1 : 0;
        for (int i0 = 1; i0 < n; i0 += kSegW) {
            const int cnt = n - i0 < kSegW ? n - i0 : kSegW;
            __syncthreads();
            // element x of staged row g holds node i0 - 1 + x: a warp takes rows
            // g = warp, warp + 8, .., four at a time
            constexpr int R = wgrad_rows<DIM, KIND>();
            for (int g0 = warp; g0 < R; g0 += 32) {
                float v[4][3];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int g = g0 + 8 * q;
                    if (g >= R) break;
                    const bool is_dense = g < ND;
                    const int h = is_dense ? g : g - ND;
                    // neighbour row of the row's (j, k); the centre one if it is alone
                    const int nb = is_dense == (KIND == 1) ? h % NB : NB / 2;
                    const int dy = nb % 3 - 1, dz = DIM == 2 ? 0 : nb / 3 - 1;
                    const int64_t p = (k + dz) * sz + (j + dy) * sy + i0 - 1;
                    const float* cp = chan + (KIND == 1 ? h : h / NB) * zs;
#pragma unroll
                    for (int x3 = 0; x3 < 3; ++x3) {
                        const int x = lane + 32 * x3;
                        v[q][x3] = 0.f;
                        if (x < cnt + 2)
                            v[q][x3] = is_dense    ? (float)dense[p + x]
                                       : KIND == 1 ? cp[p + x]
                                                   : fmaxf(cp[p + x], 0.f);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int x3 = 0; x3 < 3; ++x3)
                        if (g0 + 8 * q < R) rows_s[(g0 + 8 * q) * W + lane + 32 * x3] = v[q][x3];
            }
            __syncthreads();
            if (!on) continue;
#pragma unroll 8
            for (int i = 0; i < cnt; ++i) acc = fmaf(plain[i], tapped[i], acc);
        }
    }
    if (on)
        partial[(int64_t)blockIdx.x * (2 * H * T) + (KIND == 1 ? 0 : H * T) + ct] = (double)acc;
}

// grad[i] += scale * sum_b partial[b][i] (fixed order) for the KIND's half:
// four strided sums per entry, added in order (one thread per entry and part).
__global__ void __launch_bounds__(1024) k_wgrad_reduce(const double* __restrict__ partial,
                                                       int blocks, int half, int base,
                                                       const double* __restrict__ scale_dev,
                                                       double sign, double* __restrict__ grad) {
    __shared__ double part_sum[4][256];
    const int i = threadIdx.x & 255, part = threadIdx.x >> 8;
    double s = 0.0;
    if (i < half) {
#pragma unroll 8
        for (int b = part; b < blocks; b += 4) s += partial[(int64_t)b * 2 * half + base + i];
    }
    part_sum[part][i] = s;
    __syncthreads();
    if (part != 0 || i >= half) return;
    s = ((part_sum[0][i] + part_sum[1][i]) + part_sum[2][i]) + part_sum[3][i];
    grad[base + i] += sign * scale_dev[0] * s;
}

// s = A'e/(2d) = e - c * (sum of neighbours) on interior nodes
template <int DIM>
__global__ void __launch_bounds__(256) k_scaled_apply(const double* __restrict__ e,
                                                      double* __restrict__ s, int n) {
    const double c = DIM == 3 ? 1.0 / 6.0 : 0.25;
    const int j = blockIdx.x * blockDim.y + threadIdx.y + 1;
    const int k = DIM == 3 ? blockIdx.y + 1 : 0;
    if (j >= n) return;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    const int64_t row = k * sz + j * sy;
    for (int i = 1 + threadIdx.x; i < n; i += blockDim.x) {
        const int64_t p = row + i;
        s[p] = e[p] - c * lk::nbr_sum<DIM>(e, p, sy, sz);
    }
}

// y = a * x + y over all nodes (a from a device scalar times a constant)
__global__ void k_axpy(double* __restrict__ y, const double* __restrict__ x, int64_t nodes,
                       double a, const double* __restrict__ a_dev) {
    const double f = a_dev ? a * a_dev[0] : a;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nodes;
         p += (int64_t)gridDim.x * blockDim.x)
        y[p] = fma(f, x[p], y[p]);
}

// out[0] = sum x^2 (deterministic: fixed grid, fixed trees)
__global__ void __launch_bounds__(256) k_sumsq_partial(const double* __restrict__ x, int64_t nodes,
                                                       double* __restrict__ partial) {
    __shared__ double ws[8];
    double acc = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nodes;
         p += (int64_t)gridDim.x * blockDim.x)
        acc = fma(x[p], x[p], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += ws[w];
        partial[blockIdx.x] = s;
    }
}

// scalars: out[0] = op(partials) ; op 0: sum ; 1: 2 / sum (gradient scale) ;
// 2: acc[0] += sum * inv_den[0] / batch (loss)
__global__ void __launch_bounds__(1024) k_scalar(const double* __restrict__ partial, int count,
                                                 int op, double batch,
                                                 const double* __restrict__ inv_den,
                                                 double* __restrict__ out) {
    const double s = fp64::block_sum(partial, count);
    if (threadIdx.x != 0) return;
    if (op == 0) out[0] = s;
    if (op == 1) out[0] = 2.0 / s;
    if (op == 2) out[0] += s * inv_den[0] * 0.5 / batch;
}

// seeded white noise U[-1,1) on interior nodes (splitmix64 of seed and index)
__global__ void k_white_noise(double* __restrict__ e, int d, int n, uint64_t seed) {
    const int64_t m = n - 1;
    const int64_t total = d == 3 ? m * m * m : m * m;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(idx + 1);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z = z ^ (z >> 31);
        e[interior_node(d, n, idx)] = (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
    }
}

// Adam on the master weights; the working copy is their BF16 rounding.
__global__ void k_adam(float* __restrict__ master, float* __restrict__ work,
                       const double* __restrict__ grad, double* __restrict__ m1,
                       double* __restrict__ m2, int count, int step, double lr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double b1 = 0.9, b2 = 0.999, eps = 1e-12;
    const double g = grad[i];
    m1[i] = b1 * m1[i] + (1 - b1) * g;
    m2[i] = b2 * m2[i] + (1 - b2) * g * g;
    const double mh = m1[i] / (1 - pow(b1, step));
    const double vh = m2[i] / (1 - pow(b2, step));
    master[i] = (float)((double)master[i] - lr * mh / (sqrt(vh) + eps));
    work[i] = __bfloat162float(__float2bfloat16_rn(master[i]));
}

__global__ void k_round_bf16(const float* __restrict__ in, float* __restrict__ out, int count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = __bfloat162float(__float2bfloat16_rn(in[i]));
}

lk::RowLaunch rows(int d, int n) { return lk::row_launch(d, n, n); }

int64_t nodes_of(int d, int n) {
    const int64_t m = n + 1;
    return d == 3 ? m * m * m : m * m;
}
int64_t interior_of(int d, int n) {
    const int64_t m = n - 1;
    return d == 3 ? m * m * m : m * m;
}
int flat_blocks(int64_t nodes) { return (int)std::min<int64_t>((nodes + 255) / 256, 152 * 8); }

}  // namespace

// --------------------------------------------------------------- launchers

void conv1(int d, int n, const double* x, float* z, const float* W, cudaStream_t s) {
    auto L = rows(d, n);
    const int64_t zs = nodes_of(d, n);
    if (d == 3)
        k_conv1<3, double><<<L.grid, L.block, 0, s>>>(x, z, n, zs, W);
    else
        k_conv1<2, double><<<L.grid, L.block, 0, s>>>(x, z, n, zs, W);
}

void conv2(int d, int n, const float* z, double* out, int mode, const float* W, cudaStream_t s) {
    auto L = rows(d, n);
    const int64_t zs = nodes_of(d, n);
    if (d == 3) {
        if (mode == 0) k_conv2<3, 0><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
        if (mode == 1) k_conv2<3, 1><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
        if (mode == 2) k_conv2<3, 2><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
    } else {
        if (mode == 0) k_conv2<2, 0><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
        if (mode == 1) k_conv2<2, 1><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
        if (mode == 2) k_conv2<2, 2><<<L.grid, L.block, 0, s>>>(z, out, n, zs, W);
    }
}

void upload_weights(int d, const float* host, float* dev, float* scratch, cudaStream_t s) {
    const int W = 2 * H * (d == 3 ? 27 : 9);
    cudaMemcpyAsync(scratch, host, sizeof(float) * W, cudaMemcpyHostToDevice, s);
    k_round_bf16<<<(W + 255) / 256, 256, 0, s>>>(scratch, dev, W);
}

namespace {

void conv2_bwd(int d, int n, const double* gy, const float* z, float* gz, const float* W,
               cudaStream_t s) {
    auto L = rows(d, n);
    const int64_t zs = nodes_of(d, n);
    if (d == 3)
        k_conv2_bwd<3><<<L.grid, L.block, 0, s>>>(gy, z, gz, n, zs, W);
    else
        k_conv2_bwd<2><<<L.grid, L.block, 0, s>>>(gy, z, gz, n, zs, W);
}

void conv1_bwd(int d, int n, const float* gz, double* gx, const float* W, cudaStream_t s) {
    auto L = rows(d, n);
    const int64_t zs = nodes_of(d, n);
    if (d == 3)
        k_conv1_bwd<3><<<L.grid, L.block, 0, s>>>(gz, gx, n, zs, W);
    else
        k_conv1_bwd<2><<<L.grid, L.block, 0, s>>>(gz, gx, n, zs, W);
}

int wgrad_rpb(int n) { return std::max(1, 2048 / (n - 1)); }
int wgrad_blocks(int d, int n) {
    const int64_t rows = d == 3 ? (int64_t)(n - 1) * (n - 1) : (n - 1);
    return (int)((rows + wgrad_rpb(n) - 1) / wgrad_rpb(n));
}

// grad += sign * scale * (dW1 from (x, gz), dW2 from (gy, z))
void wgrad(int d, int n, const double* x, const float* gz, const double* gy, const float* z,
           double* partial, const double* scale_dev, double sign, double* grad, cudaStream_t s) {
    const int T = d == 3 ? 27 : 9;
    const int blocks = wgrad_blocks(d, n), rpb = wgrad_rpb(n);
    const int64_t zs = nodes_of(d, n);
    if (d == 3) {
        k_wgrad<3, 1><<<blocks, 256, 0, s>>>(x, gz, n, zs, rpb, partial);
        k_wgrad<3, 2><<<blocks, 256, 0, s>>>(gy, z, n, zs, rpb, partial);
    } else {
        k_wgrad<2, 1><<<blocks, 256, 0, s>>>(x, gz, n, zs, rpb, partial);
        k_wgrad<2, 2><<<blocks, 256, 0, s>>>(gy, z, n, zs, rpb, partial);
    }
    const int half = H * T;
    k_wgrad_reduce<<<1, 1024, 0, s>>>(partial, blocks, half, 0, scale_dev, sign, grad);
    k_wgrad_reduce<<<1, 1024, 0, s>>>(partial, blocks, half, half, scale_dev, sign, grad);
}

void scaled_apply(int d, int n, const double* e, double* out, cudaStream_t s) {
    auto L = rows(d, n);
    if (d == 3)
        k_scaled_apply<3><<<L.grid, L.block, 0, s>>>(e, out, n);
    else
        k_scaled_apply<2><<<L.grid, L.block, 0, s>>>(e, out, n);
}

// Work buffers of a training / loss evaluation on one grid.
struct Trainer {
    int d = 3, n = 0, T = 27, coarse_cycles = 30, pair_cycles = 1;
    cudaStream_t s = nullptr;
    int64_t nodes = 0;
    double *e0 = nullptr, *e1 = nullptr, *e2 = nullptr, *e3 = nullptr;  // error states
    double *s1 = nullptr, *s2 = nullptr, *s3 = nullptr;                 // A'e/(2d)
    double *g = nullptr, *gx = nullptr, *w = nullptr;
    float *z1 = nullptr, *z3 = nullptr, *gz = nullptr;
    double *partial = nullptr, *wpart = nullptr, *scal = nullptr;  // scal: [0] 1/||e0||^2*2, [1] loss
    double* grad = nullptr;
    char* extra_mem = nullptr;
    std::vector<Level<double>> coarse;  // hierarchy of the n/2 grid (coarse solve)
    std::vector<Level<double>> pair;    // hierarchy of the n grid (sample generation)
    // one device allocation, dealt out in 256-byte steps: measured first (base
    // NULL), then made
    char* base = nullptr;
    size_t used = 0;
    bool slab16 = false;  // the device places the cluster tail from n = 16 down
    // first error of a launch: the legs and tails opt in to shared memory and
    // clusters, and report (and clear) their own errors
    cudaError_t err = cudaSuccess;

    void note(cudaError_t e) {
        if (err == cudaSuccess) err = e;
    }
    // that error, or the one a plain launch left
    cudaError_t status() {
        note(cudaGetLastError());
        return err;
    }

    cudaError_t alloc(void** p, size_t bytes) {
        *p = base ? base + used : nullptr;
        used += (bytes + 255) / 256 * 256;
        return cudaSuccess;
    }
    void release() {
        cudaFree(base);
        base = nullptr;
    }
    void hierarchy(std::vector<Level<double>>& lv, int nn) {
        int L = 0;
        while ((2 << L) <= nn) ++L;
        lv.resize(L);
        for (int l = 0; l < L; ++l) {
            lv[l].n = nn >> l;
            lv[l].nodes = nodes_of(d, lv[l].n);
            const size_t b = sizeof(double) * lv[l].nodes;
            alloc((void**)&lv[l].u[0], b);
            if (leg_level(lv, l)) alloc((void**)&lv[l].u[1], b);
            alloc((void**)&lv[l].q, b);
            if (l + 1 < L) alloc((void**)&lv[l].r, b);
        }
    }
    void deal(size_t extra) {
        used = 0;
        const size_t b = sizeof(double) * nodes, bz = sizeof(float) * nodes * H;
        for (double** p : {&e0, &e1, &e2, &e3, &s1, &s2, &s3, &g, &gx, &w}) alloc((void**)p, b);
        for (float** p : {&z1, &z3, &gz}) alloc((void**)p, bz);
        alloc((void**)&partial, sizeof(double) * 152 * 8);
        alloc((void**)&wpart, sizeof(double) * wgrad_blocks(d, n) * 2 * H * T);
        alloc((void**)&scal, sizeof(double) * 4);
        alloc((void**)&grad, sizeof(double) * 2 * H * T);
        hierarchy(coarse, n / 2);
        if (pair_cycles >= 0) hierarchy(pair, n);
        alloc((void**)&extra_mem, extra);
    }
    // pc < 0: no samples are drawn.  extra: bytes at extra_mem.  Everything zeroed.
    cudaError_t init(int d_, int n_, int cc, int pc, size_t extra, cudaStream_t st) {
        d = d_;
        n = n_;
        T = d == 3 ? 27 : 9;
        coarse_cycles = cc;
        pair_cycles = pc;
        s = st;
        nodes = nodes_of(d, n);
        cudaGetLastError();  // an error that some other call left is not this one's
        slab16 = d == 3 && n >= 16 && tail::slab_fits<double>(16);
        deal(extra);
        const size_t total = used;
        cudaError_t e = cudaMalloc((void**)&base, total);
        if (e != cudaSuccess) {
            base = nullptr;
            return e;
        }
        deal(extra);
        return cudaMemsetAsync(base, 0, total, s);
    }

    bool leg_level(const std::vector<Level<double>>& lv, int l) const {
        return d == 2 && l + 1 < (int)lv.size() &&
               legs2d::applies(lv[l].n, 0, GMG_RBGS, 1, 1);
    }
    // the cluster tail takes level l of a hierarchy of L
    bool slab_level(const std::vector<Level<double>>& lv, int l) const {
        return slab16 && tail::slab_applies(d, lv[l].n, (int)lv.size() - l, GMG_RBGS, false, true);
    }
    // RB-GS V(nu,nu) cycle on hierarchy lv (level-0 iterate lv[0].u[0], rhs
    // lv[0].q) with the solver's kernels: grid kernels (2D: legs) and the
    // cluster or single-CTA tail.  first_done: the first red half sweep ran.
    void vcycle(std::vector<Level<double>>& lv, int nu, bool first_done = false) {
        const int L = (int)lv.size();
        int lt = L;
        for (int l = 0; l < L && lt == L; ++l)
            if (nu > 0 && (slab_level(lv, l) ||
                           (lv[l].n <= (d == 3 ? 8 : 16) && L - l >= 2)))
                lt = l;
        std::vector<char> done(L + 1, 0);
        done[0] = first_done;
        int down = 0;  // levels run by grid kernels or legs
        for (int l = 0; l < lt && l + 1 < L; ++l, ++down) {
            Level<double>&F = lv[l], &C = lv[l + 1];
            const int init = C.n == 2 ? INIT_EXACT : nu > 0 ? INIT_RED : INIT_ZERO;
            done[l + 1] = init == INIT_RED;
            if (leg_level(lv, l) && F.u[1]) {
                note(legs2d::down(F.n, GMG_RBGS, nu, done[l], 0.0, false, true, init, F.u[0], F.u[1],
                                  F.q, C.q, C.u[0], s));
                continue;
            }
            half_sweeps(F, nu, done[l]);
            lk::residual<double>(d, F.n, F.u[0], F.q, F.r, nu > 0, s);
            lk::restrict_fw<double>(d, F.n, F.r, C.q, C.u[0], nu > 0, init, s);
        }
        if (lt < L) {
            Level<double>& t = lv[lt];
            const Lay lay = dense_lay(d, t.n);
            if (slab_level(lv, lt))
                note(tail::launch_slab<double>(lay, L - lt, t.u[0], t.q, GMG_RBGS, nu, nu, 0, s, false,
                                               done[lt]));
            else
                note(tail::launch<double>(d, lay, L - lt, t.u[0], t.q, GMG_RBGS, 0.8, nu, nu, 0, s,
                                          false, false, done[lt]));
        } else if (L == 1) {
            half_sweeps(lv[0], nu, first_done);
        }
        for (int l = down - 1; l >= 0; --l) {
            Level<double>&F = lv[l], &C = lv[l + 1];
            if (leg_level(lv, l) && F.u[1]) {
                note(legs2d::up(F.n, GMG_RBGS, nu, 0.0, false, C.u[0], F.u[1], F.u[0], F.q, s));
                continue;
            }
            lk::prolong_add<double>(d, C.n, C.u[0], F.u[0], s, nu > 0);
            half_sweeps(F, nu, false);
        }
    }
    void half_sweeps(Level<double>& F, int nu, bool first_done) {
        for (int k = first_done ? 1 : 0; k < 2 * nu; ++k)
            lk::rb_half<double>(d, F.n, F.u[0], F.q, k & 1, s);
    }

    // u_c = (2d) A_c'^{-1} q_c with q_c = 4 FW(src) restricted from src (fine)
    void coarse_solve_of(double* src) {
        Level<double>& C = coarse[0];
        // q_c, and u_c after the first red half sweep from zero (or u_c = q_c on a
        // one-unknown grid)
        lk::restrict_fw<double>(d, n, src, C.q, C.u[0], false, C.n == 2 ? INIT_EXACT : INIT_RED, s);
        if (C.n > 2)
            for (int k = 0; k < coarse_cycles; ++k) vcycle(coarse, 2, k == 0);
    }

    // e_out = e_in - P u_c (error-form coarse-grid correction), s2 = A'e_in/(2d)
    void cgc(const double* e_in, double* e_out) {
        scaled_apply(d, n, e_in, s2, s);
        coarse_solve_of(s2);
        cudaMemcpyAsync(e_out, e_in, sizeof(double) * nodes, cudaMemcpyDeviceToDevice, s);
        cudaMemsetAsync(w, 0, sizeof(double) * nodes, s);
        lk::prolong_add<double>(d, coarse[0].n, coarse[0].u[0], w, s);
        k_axpy<<<flat_blocks(nodes), 256, 0, s>>>(e_out, w, nodes, -1.0, nullptr);
    }

    // g <- g - (A'/(2d)) P u_c' with u_c' = (2d) A_c'^{-1} 4FW(g)
    void cgc_adjoint(double* gg) {
        coarse_solve_of(gg);
        cudaMemsetAsync(w, 0, sizeof(double) * nodes, s);
        lk::prolong_add<double>(d, coarse[0].n, coarse[0].u[0], w, s);
        scaled_apply(d, n, w, gx, s);
        k_axpy<<<flat_blocks(nodes), 256, 0, s>>>(gg, gx, nodes, -1.0, nullptr);
    }

    // e_out = e_in - N(s_in), s_in = A'e_in/(2d), keeping z
    void smooth(const double* e_in, double* s_in, float* z, double* e_out, const float* W) {
        scaled_apply(d, n, e_in, s_in, s);
        conv1(d, n, s_in, z, W, s);
        cudaMemcpyAsync(e_out, e_in, sizeof(double) * nodes, cudaMemcpyDeviceToDevice, s);
        conv2(d, n, z, e_out, 2, W, s);
    }

    void sumsq(const double* x, int op, double batch) {
        const int blocks = flat_blocks(nodes);
        k_sumsq_partial<<<blocks, 256, 0, s>>>(x, nodes, partial);
        k_scalar<<<1, 1024, 0, s>>>(partial, blocks, op, batch, scal, op == 2 ? scal + 1 : scal);
    }

    // loss (accumulated into scal[1] / batch) and, if want_grad, its
    // gradient (accumulated into grad / batch) for the sample in e0
    void loss_grad(const float* W, double batch, bool want_grad) {
        smooth(e0, s1, z1, e1, W);
        cgc(e1, e2);
        smooth(e2, s3, z3, e3, W);
        sumsq(e0, 1, batch);         // scal[0] = 2 / ||e0||^2
        sumsq(e3, 2, batch);         // scal[1] += ||e3||^2 / ||e0||^2 / batch
        if (!want_grad) return;
        // g3 = 2 e3 / ||e0||^2 (scaled by 1/batch in the weight reduction)
        cudaMemsetAsync(g, 0, sizeof(double) * nodes, s);
        k_axpy<<<flat_blocks(nodes), 256, 0, s>>>(g, e3, nodes, 1.0, scal);
        // post-smoother: dtheta -= J^T g ; g2 = g - (A'/(2d)) J_x^T g
        conv2_bwd(d, n, g, z3, gz, W, s);
        wgrad(d, n, s3, gz, g, z3, wpart, scal + 2, -1.0, grad, s);
        conv1_bwd(d, n, gz, gx, W, s);
        scaled_apply(d, n, gx, w, s);
        k_axpy<<<flat_blocks(nodes), 256, 0, s>>>(g, w, nodes, -1.0, nullptr);
        // coarse-grid correction adjoint
        cgc_adjoint(g);
        // pre-smoother weight gradient
        conv2_bwd(d, n, g, z1, gz, W, s);
        wgrad(d, n, s1, gz, g, z1, wpart, scal + 2, -1.0, grad, s);
    }

    // e0 = error after pair_cycles plain RB-GS V(1,1) cycles from white noise
    void sample(uint64_t seed) {
        Level<double>& F = pair[0];
        k_white_noise<<<flat_blocks(interior_of(d, n)), 256, 0, s>>>(F.u[0], d, n, seed);
        for (int k = 0; k < pair_cycles; ++k) vcycle(pair, 1);
        cudaMemcpyAsync(e0, F.u[0], sizeof(double) * nodes, cudaMemcpyDeviceToDevice, s);
    }
};

gmg_status check_dn(int d, int n) {
    if (d != 2 && d != 3) {
        set_error("d must be 2 or 3");
        return GMG_ERR_ARG;
    }
    const int nmax = d == 3 ? 512 : 4096;
    if (n < 4 || n > nmax || (n & (n - 1))) {
        set_error("n must be a power of two in [4, " + std::to_string(nmax) + "]");
        return GMG_ERR_ARG;
    }
    return GMG_OK;
}

}  // namespace
}  // namespace learned
}  // namespace gmg

using namespace gmg;
using namespace gmg::learned;

#define GMG_TRY_CUDA_RELEASE(expr, tr)                                             \
    do {                                                                           \
        cudaError_t e_ = (expr);                                                   \
        if (e_ != cudaSuccess) {                                                   \
            set_error(std::string(#expr) + ": " + cudaGetErrorString(e_));        \
            (tr).release();                                                        \
            return e_ == cudaErrorMemoryAllocation ? GMG_ERR_ALLOC : GMG_ERR_CUDA; \
        }                                                                          \
    } while (0)

extern "C" {

gmg_status gmg_learned_conv(int d, int n, const float* weights, const double* x, double* y,
                            int tensor_cores, void* cuda_stream) {
    gmg_status st = check_dn(d, n);
    if (st != GMG_OK) return st;
    if (!weights || !x || !y) {
        set_error("weights, x, y must be non-NULL");
        return GMG_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int T = d == 3 ? 27 : 9;
    float *wd = nullptr, *wr = nullptr, *z = nullptr;
    const int64_t nodes = nodes_of(d, n);
    GMG_CUDA_TRY(cudaMalloc(&wd, sizeof(float) * 2 * H * T * 2));
    wr = wd + 2 * H * T;
    cudaError_t e = cudaMalloc(&z, sizeof(float) * H * nodes);
    if (e == cudaSuccess) e = cudaMemsetAsync(z, 0, sizeof(float) * H * nodes, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(wd, weights, sizeof(float) * 2 * H * T, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        k_round_bf16<<<(2 * H * T + 255) / 256, 256, 0, s>>>(wd, wr, 2 * H * T);
        if (tensor_cores) {
            conv_tc(d, n, x, y, 0, wr, s);
        } else {
            conv1(d, n, x, z, wr, s);
            conv2(d, n, z, y, 0, wr, s);
        }
        e = cudaStreamSynchronize(s);
    }
    cudaFree(wd);
    cudaFree(z);
    if (e != cudaSuccess) {
        set_error(std::string("gmg_learned_conv: ") + cudaGetErrorString(e));
        return GMG_ERR_CUDA;
    }
    return GMG_OK;
}

gmg_status gmg_learned_loss_grad(int d, int n, const float* weights, const double* e0,
                                 int coarse_cycles, double* loss_out, double* grad_out,
                                 void* cuda_stream) {
    gmg_status st = check_dn(d, n);
    if (st != GMG_OK) return st;
    if (!weights || !e0 || !loss_out || coarse_cycles < 1) {
        set_error("weights, e0, loss_out must be non-NULL and coarse_cycles >= 1");
        return GMG_ERR_ARG;
    }
    Trainer tr;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int W = 2 * H * (d == 3 ? 27 : 9);
    GMG_TRY_CUDA_RELEASE(tr.init(d, n, coarse_cycles, -1, sizeof(float) * 2 * W, s), tr);
    float* wd = reinterpret_cast<float*>(tr.extra_mem);
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(wd, weights, sizeof(float) * W, cudaMemcpyHostToDevice, s),
                         tr);
    k_round_bf16<<<(W + 255) / 256, 256, 0, s>>>(wd, wd + W, W);
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(tr.e0, e0, sizeof(double) * tr.nodes,
                                         cudaMemcpyDeviceToDevice, s),
                         tr);
    // scal[2] = 1 (the batch scale of the weight-gradient reduction)
    const double one = 1.0;
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(tr.scal + 2, &one, sizeof(double), cudaMemcpyHostToDevice, s),
                         tr);
    tr.loss_grad(wd + W, 1.0, grad_out != nullptr);
    GMG_TRY_CUDA_RELEASE(tr.status(), tr);
    double sc[2];
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(sc, tr.scal, sizeof(double) * 2, cudaMemcpyDeviceToHost, s),
                         tr);
    if (grad_out)
        GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(grad_out, tr.grad, sizeof(double) * W,
                                             cudaMemcpyDeviceToHost, s),
                             tr);
    GMG_TRY_CUDA_RELEASE(cudaStreamSynchronize(s), tr);
    *loss_out = sc[1];
    tr.release();
    return GMG_OK;
}

gmg_status gmg_learned_train(int d, int n, int steps, int batch, int pair_cycles, int coarse_cycles,
                             double lr, uint64_t seed, const float* w_init, float* w_out,
                             double* loss_history, void* cuda_stream) {
    gmg_status st = check_dn(d, n);
    if (st != GMG_OK) return st;
    if (steps < 1 || steps > 1000000 || batch < 1 || batch > 4096 || pair_cycles < 0 ||
        pair_cycles > 16 || coarse_cycles < 1 || coarse_cycles > 200 || !(lr > 0.0) || !w_init ||
        !w_out) {
        set_error("gmg_learned_train: bad arguments");
        return GMG_ERR_ARG;
    }
    Trainer tr;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int W = 2 * H * (d == 3 ? 27 : 9);
    GMG_TRY_CUDA_RELEASE(tr.init(d, n, coarse_cycles, pair_cycles,
                                 (sizeof(float) + sizeof(double)) * 2 * W, s), tr);
    double* m1 = reinterpret_cast<double*>(tr.extra_mem);
    double* m2 = m1 + W;
    float* master = reinterpret_cast<float*>(m2 + W);
    float* work = master + W;
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(master, w_init, sizeof(float) * W, cudaMemcpyHostToDevice, s),
                         tr);
    k_round_bf16<<<(W + 255) / 256, 256, 0, s>>>(master, work, W);
    const double inv_batch = 1.0 / batch;
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(tr.scal + 2, &inv_batch, sizeof(double),
                                         cudaMemcpyHostToDevice, s),
                         tr);
    std::vector<double> hloss(1);
    for (int it = 0; it < steps; ++it) {
        cudaMemsetAsync(tr.grad, 0, sizeof(double) * W, s);
        cudaMemsetAsync(tr.scal + 1, 0, sizeof(double), s);
        for (int b = 0; b < batch; ++b) {
            tr.sample(seed * 1000003ull + (uint64_t)it * 4096ull + (uint64_t)b);
            tr.loss_grad(work, (double)batch, true);
        }
        k_adam<<<(W + 255) / 256, 256, 0, s>>>(master, work, tr.grad, m1, m2, W, it + 1, lr);
        GMG_TRY_CUDA_RELEASE(tr.status(), tr);
        if (loss_history) {
            GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(&loss_history[it], tr.scal + 1, sizeof(double),
                                                 cudaMemcpyDeviceToHost, s),
                                 tr);
        }
    }
    GMG_TRY_CUDA_RELEASE(cudaMemcpyAsync(w_out, master, sizeof(float) * W, cudaMemcpyDeviceToHost, s),
                         tr);
    GMG_TRY_CUDA_RELEASE(cudaStreamSynchronize(s), tr);
    tr.release();
    return GMG_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Fused tensor-core network for the V-cycle: u += N(sigma) in one kernel.
//
// One CTA (8 warps) owns a TX x TY x TZ tile of output nodes.  sigma is
// staged in shared memory as BF16 on the tile plus a 2-node halo; conv1 runs
// on the tile plus a 1-node halo as a [16 nodes x 32 taps] x [32 taps x 8
// channels] product per 16 nodes (two mma.sync m16n8k16 BF16, FP32
// accumulate, taps 27..31 zero), its ReLU'd result stored channel-last in
// BF16 (16 bytes per node, zero outside the interior); conv2 runs per 16
// consecutive output nodes as sum over tap pairs of [16 nodes x (2 taps x 8
// channels)] x [16 x 8] with ldmatrix gathering each node's 8 channels at
// the tapped position and only column 0 of the B operand non-zero.  Hidden
// activations and sigma therefore enter the tensor cores in BF16; weights
// are BF16; every sum accumulates in FP32.
namespace gmg {
namespace learned {
namespace {

template <int DIM>
struct TcTile {
    // TX = 14: a halo-1 x-row is exactly 16 nodes, one conv1 mma group
    static constexpr int TX = 14, TY = DIM == 3 ? 8 : 16, TZ = DIM == 3 ? 8 : 1;
    static constexpr int HZ = DIM == 3 ? 1 : 0;                   // halo in z
    static constexpr int X1 = TX + 2, Y1 = TY + 2, Z1 = TZ + 2 * HZ;  // halo-1 region
    static constexpr int X2 = TX + 4, Y2 = TY + 4, Z2 = TZ + 4 * HZ;  // halo-2 region
    static constexpr int N1 = X1 * Y1 * Z1;
    static constexpr int N2 = X2 * Y2 * Z2;
    static constexpr int T = DIM == 3 ? 27 : 9;
    static constexpr int K1 = (T + 15) / 16;  // conv1 k-steps of 16 taps
    static constexpr int P2 = (T + 1) / 2;    // conv2 tap pairs
};

__device__ inline uint32_t pack_bf16(float lo, float hi) {
    const uint32_t l = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
    const uint32_t h = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
    return l | (h << 16);
}

__device__ inline void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ inline void ldmatrix_x4(uint32_t* r, const void* smem_row) {
    const uint32_t addr = (uint32_t)__cvta_generic_to_shared(smem_row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

template <int DIM>
__device__ inline int tap_dx(int t) { return t % 3 - 1; }
template <int DIM>
__device__ inline int tap_dy(int t) { return (t / 3) % 3 - 1; }
template <int DIM>
__device__ inline int tap_dz(int t) { return DIM == 3 ? t / 9 - 1 : 0; }

// MODE 1: u += N(sigma);  MODE 0: u = N(sigma) (interior nodes)
template <int DIM, int MODE>
__global__ void __launch_bounds__(256) k_conv_tc(const double* __restrict__ sigma,
                                                 double* __restrict__ u, int n,
                                                 const float* __restrict__ W) {
    using G = TcTile<DIM>;
    __shared__ __nv_bfloat16 xs[G::N2];
    __shared__ __align__(16) uint4 zs[G::N1];  // 8 BF16 channels per node
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gid = lane >> 2, tig = lane & 3;
    const int i0 = 1 + G::TX * blockIdx.x, j0 = 1 + G::TY * blockIdx.y,
              k0 = DIM == 3 ? 1 + G::TZ * blockIdx.z : 0;
    const int64_t sy = sy_of(n), sz = sz_of<DIM>(n);
    auto inside = [&](int i, int j, int k) {
        return i >= 1 && i < n && j >= 1 && j < n && (DIM == 2 || (k >= 1 && k < n));
    };
    // 1. sigma on the halo-2 region, BF16, zero outside the interior
    for (int m = threadIdx.x; m < G::N2; m += blockDim.x) {
        const int hx = m % G::X2, hy = (m / G::X2) % G::Y2, hz = m / (G::X2 * G::Y2);
        const int i = i0 - 2 + hx, j = j0 - 2 + hy, k = DIM == 3 ? k0 - 2 + hz : 0;
        const float v = inside(i, j, k) ? (float)sigma[k * sz + j * sy + i] : 0.f;
        xs[m] = __float2bfloat16_rn(v);
    }
    // B operands (weights) in registers
    uint32_t b1w[G::K1][2];
#pragma unroll
    for (int kh = 0; kh < G::K1; ++kh) {
        const int t0 = 16 * kh + 2 * tig;
        auto w1 = [&](int t) { return t < G::T ? W[gid * G::T + t] : 0.f; };
        b1w[kh][0] = pack_bf16(w1(t0), w1(t0 + 1));
        b1w[kh][1] = pack_bf16(w1(t0 + 8), w1(t0 + 9));
    }
    uint32_t b2w[G::P2][2];
#pragma unroll
    for (int pp = 0; pp < G::P2; ++pp) {
        const float* W2 = W + 8 * G::T;
        const int ta = 2 * pp, tb = 2 * pp + 1;
        auto w2 = [&](int c, int t) { return (gid == 0 && t < G::T) ? W2[c * G::T + t] : 0.f; };
        b2w[pp][0] = pack_bf16(w2(2 * tig, ta), w2(2 * tig + 1, ta));
        b2w[pp][1] = pack_bf16(w2(2 * tig, tb), w2(2 * tig + 1, tb));
    }
    __syncthreads();
    // 2. conv1 on the halo-1 region: groups of 16 nodes, one group per warp
    // turn.  This lane's taps (fixed per lane) as offsets in the halo-2 tile.
    constexpr int NT1 = 4 * G::K1;
    int toff[NT1];
    bool tok[NT1];
#pragma unroll
    for (int q = 0; q < NT1; ++q) {
        const int kh = q / 4, sub = q % 4;
        const int t = 16 * kh + 2 * tig + (sub & 1) + (sub >> 1) * 8;
        tok[q] = t < G::T;
        const int tt = tok[q] ? t : 0;
        toff[q] = (tap_dz<DIM>(tt) * G::Y2 + tap_dy<DIM>(tt)) * G::X2 + tap_dx<DIM>(tt);
    }
    static_assert(G::X1 == 16, "a halo-1 row must be one 16-node mma group");
    // this lane's two nodes of a row: x = gid and gid + 8 of the halo-1 row
    const bool xin0 = i0 - 1 + gid >= 1 && i0 - 1 + gid < n;
    const bool xin1 = i0 - 1 + gid + 8 >= 1 && i0 - 1 + gid + 8 < n;
    const unsigned short* xr = reinterpret_cast<const unsigned short*>(xs);
    const int rows1 = G::Y1 * G::Z1;
    for (int g = warp; g < rows1; g += 8) {
        const int hy = g % G::Y1, hz = g / G::Y1;
        const int j = j0 - 1 + hy, k = DIM == 3 ? k0 - 1 + hz : 0;
        const bool yzin = j >= 1 && j < n && (DIM == 2 || (k >= 1 && k < n));
        // centre of node (gid, hy, hz) in the halo-2 tile
        const int m0 = ((hz + G::HZ) * G::Y2 + (hy + 1)) * G::X2 + (gid + 1);
        const int m1 = m0 + 8;
        auto xb = [&](int m, int q) -> uint32_t {
            return tok[q] ? (uint32_t)xr[m + toff[q]] : 0u;
        };
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kh = 0; kh < G::K1; ++kh) {
            const int q = 4 * kh;
            uint32_t a[4];
            a[0] = xb(m0, q) | (xb(m0, q + 1) << 16);
            a[1] = xb(m1, q) | (xb(m1, q + 1) << 16);
            a[2] = xb(m0, q + 2) | (xb(m0, q + 3) << 16);
            a[3] = xb(m1, q + 2) | (xb(m1, q + 3) << 16);
            mma_bf16(c, a, b1w[kh][0], b1w[kh][1]);
        }
        // relu, BF16, channel-last; zero outside the interior
        uint32_t* z0 = reinterpret_cast<uint32_t*>(&zs[16 * g + gid]);
        uint32_t* z1 = reinterpret_cast<uint32_t*>(&zs[16 * g + gid + 8]);
        z0[tig] = (yzin && xin0) ? pack_bf16(fmaxf(c[0], 0.f), fmaxf(c[1], 0.f)) : 0u;
        z1[tig] = (yzin && xin1) ? pack_bf16(fmaxf(c[2], 0.f), fmaxf(c[3], 0.f)) : 0u;
    }
    __syncthreads();
    // 3. conv2 on 16-node x-rows of the output tile
    const int rows2 = G::TY * G::TZ;
    for (int row = warp; row < rows2; row += 8) {
        const int oy = row % G::TY, oz = row / G::TY;
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        const int mtx = lane >> 3, rr = lane & 7;  // ldmatrix: this lane's matrix and row
        // rows past the tile's last x (TX..15) are computed but discarded: read
        // the last column's neighbourhood there so every address stays in its row
        const int ox = min((mtx & 1) * 8 + rr, G::TX - 1);
        const int mc = ((oz + G::HZ) * G::Y1 + (oy + 1)) * G::X1 + (ox + 1);
        const int hi = mtx >> 1;
#pragma unroll
        for (int pp = 0; pp < G::P2; ++pp) {
            // tap 2pp (matrices 0, 1) or 2pp + 1 (matrices 2, 3); a padding tap
            // reads the centre row (its weight is zero)
            const int ta = 2 * pp, tb = 2 * pp + 1 < G::T ? 2 * pp + 1 : G::T / 2;
            const int oa = (tap_dz<DIM>(ta) * G::Y1 + tap_dy<DIM>(ta)) * G::X1 + tap_dx<DIM>(ta);
            const int ob = (tap_dz<DIM>(tb) * G::Y1 + tap_dy<DIM>(tb)) * G::X1 + tap_dx<DIM>(tb);
            uint32_t a[4];
            ldmatrix_x4(a, &zs[mc + (hi ? ob : oa)]);
            mma_bf16(c, a, b2w[pp][0], b2w[pp][1]);
        }
        if (tig == 0) {
            const int j = j0 + oy, k = DIM == 3 ? k0 + oz : 0;
            for (int h = 0; h < 2; ++h) {
                const int ox_ = gid + 8 * h;
                const int i = i0 + ox_;
                if (ox_ >= G::TX || !inside(i, j, k)) continue;
                const int64_t p = k * sz + j * sy + i;
                const double y = (double)c[2 * h];
                if (MODE == 1)
                    u[p] += y;
                else
                    u[p] = y;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// z-streaming 3D network: u += N(sigma), the hidden layer in registers.
//
// A warp owns 14 x kR output columns and walks the planes of its CTA's chunk (one
// halo plane on either side).  Per plane kk and per hidden row y of 16 halo-1
// nodes (mma.sync m16n8k16 / m16n8k8, BF16 operands, FP32 sums):
//  1. conv1 is a [16 nodes x 48] x [48 x 8 channels] product, K = 3 dy x 4 groups
//     (three planes, one zero-weight group) x 4 dx slots (dx = -1, 0, +1, one
//     zero-weight slot).  One sigma row is one A operand of four registers, used
//     with the three dy's weights by the three hidden rows it belongs to: a
//     lane loads 4 words a row instead of 12.  sigma sits in a ring of four BF16
//     planes stored twice (element e, and shifted by one), so each pair is one
//     aligned word.
//  2. The ReLU'd accumulators, rounded to BF16, are the A operand of conv2 as
//     they are: two rows' make K = 16.  Output row y takes rows y-1 .. y+1 as a
//     pair in one m16n8k16 and one in m16n8k8; the columns are the three dx of the
//     three open output planes (4 columns each: two n-tiles), and the FP32
//     accumulators stay in the tensor core's registers from plane to plane.
//     The output plane's number modulo 3 is its column group, so the B operands
//     rotate (the plane loop is unrolled by 3) instead of the sums.
//  3. The plane that is complete adds its three dx columns, shifted by one
//     node against each other (4 shuffles a row), and u += y runs over full
//     warps (an FP64 instruction costs the same with 8 lanes on).  The
//     conversions from and to double run on the integer pipe, with the casts'
//     results (df.cuh): as casts they took 30% of the FP64 pipe.
// Nothing of the hidden layer goes through shared memory; the kernel this
// replaces kept the 27 contributions of a node there and was bound by that: 501
// us per application at 257^3 and 315 M warp instructions, 291 us and 139 M now.
// What bounds it now is latency at two CTAs per SM (128 registers: 24 of them
// weights, 32 accumulators): 47% of the issue slots, 31% of the tensor pipe.
// The hidden activations and sigma enter the tensor cores in BF16, weights
// are BF16, every sum is FP32 -- the numerics of k_conv_tc, with the taps
// summed in a different order.
constexpr int kR = 4;                      // output rows per warp
constexpr int kWX = 2, kWY = 4;            // warps of a CTA along x, y
constexpr int kTX = 14 * kWX, kTY = kR * kWY;  // output tile
constexpr int kSX = kTX + 4, kSY = kTY + 4;    // sigma tile (halo 2): kSX = 32
constexpr int kSRow = kSX + 2;             // elements per row (the last pair's pad)
// words per plane and to the shifted copy: 11 and 5 banks apart, so that a
// warp's four runs of 5 words (two copies, two planes) rarely meet in a bank
constexpr int kPlaneW = 363, kCopyW = 4 * kPlaneW + 25;
constexpr int kSmemW = kCopyW + 4 * kPlaneW;
static_assert(kSX == 32 && kSY * kSRow / 2 <= kPlaneW && kPlaneW % 32 == 11 && kCopyW % 32 == 5,
              "sigma ring layout");
constexpr int kPF = (kSX * kSY + 255) / 256;  // sigma elements fetched per thread

// d = A B, from zero accumulators
__device__ inline void mma_bf16_first(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ inline void mma_bf16_k8(float* c, uint32_t a0, uint32_t a1, uint32_t b0) {
    asm(
        "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(b0));
}

// BF16 of max(lo, 0) and max(hi, 0) (rounding and the maximum commute; NaN -> 0)
__device__ inline uint32_t relu_pack(float lo, float hi) {
    const __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(lo, hi), __float2bfloat162_rn(0.f));
    return *reinterpret_cast<const uint32_t*>(&v);
}

// MODE 1: u += N(sigma);  MODE 0: u = N(sigma) (interior nodes)
template <int MODE>
__global__ void __launch_bounds__(256, 2) k_conv_zs(const double* __restrict__ sigma,
                                                    double* __restrict__ u, int n,
                                                    const float* __restrict__ W, int planes) {
    __shared__ __align__(16) uint32_t ring[kSmemW];
    __shared__ float ybuf[8][kR][16];
    __nv_bfloat16* sa = reinterpret_cast<__nv_bfloat16*>(ring);
    __nv_bfloat16* sb = reinterpret_cast<__nv_bfloat16*>(ring + kCopyW);  // shifted copy
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gid = lane >> 2, tig = lane & 3, hf = tig >> 1;
    const int wx = warp % kWX, wy = warp / kWX;
    const int i0 = 1 + kTX * blockIdx.x, j0 = 1 + kTY * blockIdx.y;
    const int k0 = 1 + planes * blockIdx.z;
    const int kend = min(k0 + planes, n);  // output planes k0 .. kend-1
    const int64_t sy = (int64_t)n + 1, sz = sy * sy;

    for (int e = threadIdx.x; e < kSmemW; e += 256) ring[e] = 0u;

    // conv1 B operands, one per dy: k = 0..7 are the lane halves' first planes (half
    // 0 dz = -1, half 1 dz = +1), k = 8..15 their second (half 0 dz = 0, half 1 none)
    uint32_t b1w[3][2];
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) {
        const int sl = 2 * (tig & 1);
        auto w1 = [&](int dz, int slot) {
            return slot < 3 ? W[gid * 27 + dz * 9 + dy * 3 + slot] : 0.f;
        };
        const int dz0 = hf ? 2 : 0;
        b1w[dy][0] = pack_bf16(w1(dz0, sl), w1(dz0, sl + 1));
        b1w[dy][1] = hf ? 0u : pack_bf16(w1(1, sl), w1(1, sl + 1));
    }
    // conv2 B operands [phase][n-tile][dy] of this lane's column
    uint32_t b2w[3][2][3];
    {
        const float* W2 = W + 8 * 27;
#pragma unroll
        for (int ph = 0; ph < 3; ++ph)  // t % 3, t = plane - (k0 - 1)
#pragma unroll
            for (int tile = 0; tile < 2; ++tile) {
                const int s = 2 * tile + (gid >> 2), dx = gid & 3;
                // group s holds the output plane k0 + p with p % 3 = s, p = t, t - 1, t - 2
                const int back = (ph - s + 3) % 3;  // 0: dz = -1, 1: dz = 0, 2: dz = +1
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    auto w2 = [&](int c) {
                        return (s < 3 && dx < 3) ? W2[c * 27 + back * 9 + dy * 3 + dx] : 0.f;
                    };
                    b2w[ph][tile][dy] = pack_bf16(w2(2 * tig), w2(2 * tig + 1));
                }
            }
    }

    // sigma tile elements of this thread (row m >> 5, column m & 31): offset in a
    // plane of sigma (-1 outside the interior) and in a ring slot.  They stay
    // doubles until they are stored, a plane later, so that nothing waits for
    // the loads.
    double pf[kPF];
    int goff[kPF];
    const int soff = (threadIdx.x >> 5) * kSRow + lane;  // element r: 8 r rows on
#pragma unroll
    for (int r = 0; r < kPF; ++r) {
        const int m = threadIdx.x + 256 * r;
        const int i = i0 - 2 + (m & 31), j = j0 - 2 + (m >> 5);
        const bool in = m < kSX * kSY && i >= 1 && i < n && j >= 1 && j < n;
        goff[r] = in ? j * (n + 1) + i : -1;
    }
    auto fetch = [&](int k) {
        const double* plane = sigma + (int64_t)k * sz;
        const bool kin = k >= 1 && k < n;
#pragma unroll
        for (int r = 0; r < kPF; ++r) pf[r] = kin && goff[r] >= 0 ? plane[goff[r]] : 0.0;
    };
    auto store = [&](int k) {  // the fetched plane k -> ring slot k & 3, both copies
        __nv_bfloat16* a = sa + (k & 3) * 2 * kPlaneW;
        __nv_bfloat16* b = sb + (k & 3) * 2 * kPlaneW;
#pragma unroll
        for (int r = 0; r < kPF; ++r) {
            const int m = threadIdx.x + 256 * r;
            if (m < kSX * kSY) {
                const __nv_bfloat16 v = __float2bfloat16_rn(cvt::narrow(pf[r]));
                a[soff + 8 * r * kSRow] = v;
                if (lane) b[soff + 8 * r * kSRow - 1] = v;
            }
        }
    };
    __syncthreads();
    for (int k = k0 - 2; k <= k0; ++k) {
        fetch(k);
        store(k);
    }
    fetch(k0 + 1);

    // the word of this lane's first node (x = gid) in row 0 of the warp's sigma rows:
    // columns x + (0, 1) for tig even, x + (2, 3) for tig odd
    const uint32_t* src = ring + ((gid & 1) ? kCopyW : 0) +
                          (kR * wy * kSRow + 14 * wx + gid - (gid & 1) + 2 * (tig & 1)) / 2;
    // hidden nodes outside the interior are zero: masks of the warp's two node
    // sets and its first and last row, for the warps that have any outside
    const int ia = i0 - 1 + 14 * wx + gid;
    const uint32_t xm0 = ia >= 1 && ia < n ? ~0u : 0u, xm1 = ia + 8 >= 1 && ia + 8 < n ? ~0u : 0u;
    const int jw = j0 - 1 + kR * wy;  // global row of hidden row 0
    const bool edge_warp = i0 - 1 + 14 * wx < 1 || i0 - 1 + 14 * wx + 15 >= n || jw < 1 ||
                           jw + kR + 1 >= n;

    // the two outputs of this lane: rows o / 14, columns o % 14 of the warp's tile
    int ooff[2];
    const float* yout[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int o = lane + 32 * h;
        const int i = i0 + 14 * wx + o % 14, j = j0 + kR * wy + o / 14;
        ooff[h] = o < 14 * kR && i < n && j < n ? j * (n + 1) + i : -1;
        yout[h] = &ybuf[warp][o / 14 % kR][1 + o % 14];
    }

    float acc[kR][2][4];
#pragma unroll
    for (int y = 0; y < kR; ++y)
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[y][t][e] = 0.f;

    // plane kk, the PH-th modulo 3 from k0 - 1 on
    auto plane_step = [&](auto phase, int kk) {
        constexpr int PH = decltype(phase)::value;
        constexpr int FIN = (PH + 1) % 3;       // the column group complete after this plane
        constexpr int FT = FIN == 2 ? 1 : 0;    // its n-tile
        constexpr int FL = FIN == 1 ? 2 : 0;    // its lanes: tig = FL (dx = -1, 0), FL + 1 (+1)
        // u of the outputs finished this plane, read early
        double* uo = u + (int64_t)(kk - 1) * sz;
        const bool out = kk - 1 >= k0;
        double u_old[2] = {0.0, 0.0};
        if (MODE == 1 && out) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (ooff[h] >= 0) u_old[h] = uo[ooff[h]];
        }
        __syncthreads();  // sigma planes kk-1 .. kk+1 stored
        const bool kin = kk >= 1 && kk < n, masked = edge_warp || !kin;
        // this lane's planes: half 0 kk-1 and kk, half 1 kk+1 (twice)
        const uint32_t* p0 = src + ((kk + (hf ? 1 : -1)) & 3) * kPlaneW;
        const uint32_t* p1 = src + ((kk + hf) & 3) * kPlaneW;
        // sigma row r of the warp as conv1's A operand: nodes gid, gid + 8 of the two
        // planes (the same registers serve the three hidden rows it belongs to)
        uint32_t sg[3][4];
        auto load_row = [&](int r) {
            sg[r % 3][0] = p0[r * (kSRow / 2)];
            sg[r % 3][1] = p0[r * (kSRow / 2) + 4];
            sg[r % 3][2] = p1[r * (kSRow / 2)];
            sg[r % 3][3] = p1[r * (kSRow / 2) + 4];
        };
        load_row(0);
        load_row(1);
        // hidden rows of the nodes gid, gid + 8, two rows to an A operand; two rows at
        // a time, so that two to four independent products are in flight
        uint32_t h[(kR + 2) / 2][4];
#pragma unroll
        for (int hp = 0; hp < (kR + 2) / 2; ++hp) {
            const int ra = 2 * hp;  // rows ra, ra + 1
            load_row(ra + 2);
            uint32_t last[4] = {p0[(ra + 3) * (kSRow / 2)], p0[(ra + 3) * (kSRow / 2) + 4],
                                p1[(ra + 3) * (kSRow / 2)], p1[(ra + 3) * (kSRow / 2) + 4]};
            float ca[4], cb[4];
            mma_bf16_first(ca, sg[ra % 3], b1w[0][0], b1w[0][1]);
            mma_bf16_first(cb, sg[(ra + 1) % 3], b1w[0][0], b1w[0][1]);
            mma_bf16(ca, sg[(ra + 1) % 3], b1w[1][0], b1w[1][1]);
            mma_bf16(cb, sg[(ra + 2) % 3], b1w[1][0], b1w[1][1]);
            mma_bf16(ca, sg[(ra + 2) % 3], b1w[2][0], b1w[2][1]);
            mma_bf16(cb, last, b1w[2][0], b1w[2][1]);
#pragma unroll
            for (int e = 0; e < 4; ++e) sg[ra % 3][e] = last[e];  // row ra + 3
            h[hp][0] = relu_pack(ca[0], ca[1]);
            h[hp][1] = relu_pack(ca[2], ca[3]);
            h[hp][2] = relu_pack(cb[0], cb[1]);
            h[hp][3] = relu_pack(cb[2], cb[3]);
            if (masked) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int j = jw + ra + r;
                    const uint32_t ym = kin && j >= 1 && j < n ? ~0u : 0u;
                    h[hp][2 * r] &= xm0 & ym;
                    h[hp][2 * r + 1] &= xm1 & ym;
                }
            }
            if (hp == 0) continue;
            // output rows ya = ra - 2 (hidden rows ra - 2, ra - 1 | ra) and yb = ra - 1
            // (ra - 1 | ra, ra + 1): a pair of rows that shares an operand in one
            // m16n8k16, the third in one m16n8k8
            const int ya = ra - 2, yb = ra - 1;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                mma_bf16(acc[ya][t], h[hp - 1], b2w[PH][t][0], b2w[PH][t][1]);
                mma_bf16(acc[yb][t], h[hp], b2w[PH][t][1], b2w[PH][t][2]);
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                mma_bf16_k8(acc[ya][t], h[hp][0], h[hp][1], b2w[PH][t][2]);
                mma_bf16_k8(acc[yb][t], h[hp - 1][2], h[hp - 1][3], b2w[PH][t][0]);
            }
        }
        // out(x) = [x-1][dx = -1] + [x][0] + [x+1][+1] of group FIN, nodes x = gid, gid + 8
#pragma unroll
        for (int y = 0; y < kR; ++y) {
            float* d = acc[y][FT];
            const float m0 = __shfl_sync(0xffffffffu, d[0], (lane - 4) & 31);
            const float m1 = __shfl_sync(0xffffffffu, d[2], (lane - 4) & 31);
            const float q0 = __shfl_sync(0xffffffffu, d[0], (lane + 5) & 31);
            const float q1 = __shfl_sync(0xffffffffu, d[2], (lane + 5) & 31);
            if (tig == FL) {
                ybuf[warp][y][gid] = (m0 + d[1]) + (gid == 7 ? q1 : q0);
                ybuf[warp][y][gid + 8] = ((gid == 0 ? m0 : m1) + d[3]) + q1;
            }
            // the group starts its next plane from zero
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] = FIN == 2 || hf == FIN ? 0.f : d[e];
        }
        store(kk + 2);  // slot (kk + 2) & 3 is not read by this plane's conv1
        fetch(kk + 3);
        __syncwarp();
        if (out) {
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (ooff[e] >= 0) uo[ooff[e]] = u_old[e] + cvt::widen(*yout[e]);
        }
        __syncwarp();
    };
    for (int kk = k0 - 1; kk <= kend; kk += 3) {
        plane_step(std::integral_constant<int, 0>{}, kk);
        if (kk + 1 <= kend) plane_step(std::integral_constant<int, 1>{}, kk + 1);
        if (kk + 2 <= kend) plane_step(std::integral_constant<int, 2>{}, kk + 2);
    }
}

}  // namespace

// 3D uses the z-streaming kernel unless GMG_CONV_ZS=0 (then the tile kernel;
// the two agree to FP32 rounding of the conv2 sums).
bool conv_zs_enabled() {
    static const bool on = [] {
        const char* v = std::getenv("GMG_CONV_ZS");
        return !(v && v[0] == '0');
    }();
    return on;
}

void conv_tc(int d, int n, const double* sigma, double* u, int mode, const float* W,
             cudaStream_t s) {
    if (d == 3 && conv_zs_enabled()) {
        // planes per CTA: the number with the fewest plane steps in all waves of two
        // CTAs per SM, where a CTA also computes two halo planes and spends
        // about four steps' time on its operands
        const int tx = (n - 1 + kTX - 1) / kTX, ty = (n - 1 + kTY - 1) / kTY;
        int planes = 2;
        int64_t best = INT64_MAX;
        for (int p = 2; p <= 64; ++p) {
            const int64_t ctas = (int64_t)tx * ty * ((n - 1 + p - 1) / p);
            const int64_t steps = (ctas + 2 * 152 - 1) / (2 * 152) * (p + 6);
            if (steps < best) {
                best = steps;
                planes = p;
            }
        }
        const dim3 grid(tx, ty, (n - 1 + planes - 1) / planes);
        if (mode == 1)
            k_conv_zs<1><<<grid, 256, 0, s>>>(sigma, u, n, W, planes);
        else
            k_conv_zs<0><<<grid, 256, 0, s>>>(sigma, u, n, W, planes);
        return;
    }
    if (d == 3) {
        using G = TcTile<3>;
        dim3 grid((n - 1 + G::TX - 1) / G::TX, (n - 1 + G::TY - 1) / G::TY,
                  (n - 1 + G::TZ - 1) / G::TZ);
        if (mode == 1)
            k_conv_tc<3, 1><<<grid, 256, 0, s>>>(sigma, u, n, W);
        else
            k_conv_tc<3, 0><<<grid, 256, 0, s>>>(sigma, u, n, W);
    } else {
        using G = TcTile<2>;
        dim3 grid((n - 1 + G::TX - 1) / G::TX, (n - 1 + G::TY - 1) / G::TY, 1);
        if (mode == 1)
            k_conv_tc<2, 1><<<grid, 256, 0, s>>>(sigma, u, n, W);
        else
            k_conv_tc<2, 0><<<grid, 256, 0, s>>>(sigma, u, n, W);
    }
}

}  // namespace learned
}  // namespace gmg
