#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

// ---------------------------------------------------------------------------
// the price-space time loop (Sec. 3.3 on the paper's grid), FP64
// ---------------------------------------------------------------------------
namespace pide {

namespace {
constexpr int kBX = 32, kBY = 8;
__device__ __forceinline__ int clampi(int v, int hi) { return v < 0 ? 0 : (v > hi ? hi : v); }
}  // namespace

// D v (Sec. 3.2.1) at node (m1, m2): per-axis three-point coefficients a1 (first
// difference) and b2 (second difference), boundary rows encoded in the tables
__device__ __forceinline__ double ps_dv(const PsDiff& d, const double* v, int m1, int m2) {
    const int n = d.n1, N = n - 1;
    double d2x = 0.0, d2y = 0.0, mix = 0.0;
#pragma unroll
    for (int i = -1; i <= 1; ++i) {
        const int q1 = clampi(m1 + i, N), q2 = clampi(m2 + i, N);
        d2x += d.b2[m1 * 3 + i + 1] * v[(size_t)m2 * n + q1];
        d2y += d.b2[m2 * 3 + i + 1] * v[(size_t)q2 * n + m1];
        const double a2 = d.a1[m2 * 3 + i + 1];
        if (a2 != 0.0) {
#pragma unroll
            for (int j = -1; j <= 1; ++j) mix += a2 * d.a1[m1 * 3 + j + 1] * v[(size_t)q2 * n + clampi(m1 + j, N)];
        }
    }
    const double x1 = d.x[m1], x2 = d.x[m2];
    return 0.5 * d.A11 * x1 * x1 * d2x + d.A12 * x1 * x2 * mix + 0.5 * d.A22 * x2 * x2 * d2y;
}

// out = alpha v + beta D v + gamma w (w may be NULL)
__global__ void k_ps_diff(PsDiff d, const double* __restrict__ v, double alpha, double beta,
                          const double* __restrict__ w, double gamma, double* __restrict__ out) {
    const int m1 = blockIdx.x * blockDim.x + threadIdx.x, m2 = blockIdx.y * blockDim.y + threadIdx.y;
    if (m1 >= d.n1 || m2 >= d.n1) return;
    const size_t i = (size_t)m2 * d.n1 + m1;
    double r = alpha * v[i] + beta * ps_dv(d, v, m1, m2);
    if (w) r += gamma * w[i];
    out[i] = r;
}

// inverse of the diagonal of c0 I - c1 D (Jacobi preconditioner)
__global__ void k_ps_diag_inv(PsDiff d, double c0, double c1, double* __restrict__ dinv) {
    const int m1 = blockIdx.x * blockDim.x + threadIdx.x, m2 = blockIdx.y * blockDim.y + threadIdx.y;
    if (m1 >= d.n1 || m2 >= d.n1) return;
    const double x1 = d.x[m1], x2 = d.x[m2];
    const double dd = 0.5 * d.A11 * x1 * x1 * d.b2[m1 * 3 + 1] + d.A12 * x1 * x2 * d.a1[m2 * 3 + 1] * d.a1[m1 * 3 + 1] +
                      0.5 * d.A22 * x2 * x2 * d.b2[m2 * 3 + 1];
    dinv[(size_t)m2 * d.n1 + m1] = 1.0 / (c0 - c1 * dd);
}

// Y^{n,0} = sum_i c_i V^{n-i} (eq. 3.26), and, BV given, its B_w Y by the same sum of B_w V^{n-i}
__global__ void k_ps_start(size_t n, PsHistory h, double* __restrict__ Y, double* __restrict__ BY) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double y = h.c[0] * h.V[0][i];
    for (int k = 1; k < h.count; ++k) y += h.c[k] * h.V[k][i];
    Y[i] = y;
    if (!BY) return;
    double b = h.c[0] * h.BV[0][i];
    for (int k = 1; k < h.count; ++k) b += h.c[k] * h.BV[k][i];
    BY[i] = b;
}

// before an implicit solve: B_w Y += ZZ (the jump of the last increment, or NULL), its right-hand
// side B = h_t theta B_w Y + W, and its start X = Y
__global__ void k_ps_rhs(size_t n, double htt, const double* __restrict__ W, const double* __restrict__ ZZ,
                         const double* __restrict__ Y, double* __restrict__ BY, double* __restrict__ B,
                         double* __restrict__ X) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double by = BY[i];
    if (ZZ) BY[i] = by += ZZ[i];
    B[i] = htt * by + W[i];
    X[i] = Y[i];
}

// after it: the increment T = X - Y, Y = X, and eq. 3.25's maximum per block
__global__ void k_ps_update(size_t n, const double* __restrict__ X, double* __restrict__ Y, double* __restrict__ T,
                            double* __restrict__ part) {
    __shared__ double red[256];
    double m = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double x = X[i], t = x - Y[i];
        m = fmax(m, fabs(t) / fmax(1.0, fabs(x)));
        T[i] = t;
        Y[i] = x;
    }
    red[threadIdx.x] = m;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// the maximum of per-block partials into res[0]
__global__ void k_ps_finish(const double* __restrict__ part, int nblocks, double* __restrict__ res) {
    __shared__ double red[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) s = fmax(s, part[b]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) res[0] = red[0];
}

constexpr int kPsRedBlocks = 304;      // 2 x 152 SMs

cudaError_t launch_ps_diff(const PsDiff& d, const double* v, double alpha, double beta, const double* w, double gamma,
                           double* out, cudaStream_t s) {
    const dim3 blk(kBX, kBY), grd((d.n1 + kBX - 1) / kBX, (d.n1 + kBY - 1) / kBY);
    k_ps_diff<<<grd, blk, 0, s>>>(d, v, alpha, beta, w, gamma, out);
    return cudaGetLastError();
}
cudaError_t launch_ps_diag_inv(const PsDiff& d, double c0, double c1, double* dinv, cudaStream_t s) {
    const dim3 blk(kBX, kBY), grd((d.n1 + kBX - 1) / kBX, (d.n1 + kBY - 1) / kBY);
    k_ps_diag_inv<<<grd, blk, 0, s>>>(d, c0, c1, dinv);
    return cudaGetLastError();
}
cudaError_t launch_ps_start(size_t n, const PsHistory& h, double* Y, double* BY, cudaStream_t s) {
    k_ps_start<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, h, Y, BY);
    return cudaGetLastError();
}
cudaError_t launch_ps_rhs(size_t n, double htt, const double* W, const double* ZZ, const double* Y, double* BY, double* B,
                          double* X, cudaStream_t s) {
    k_ps_rhs<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, htt, W, ZZ, Y, BY, B, X);
    return cudaGetLastError();
}
int ps_reduction_blocks() { return kPsRedBlocks; }
// ---------------------------------------------------------------------------
// Jacobi-preconditioned BiCGSTAB for (c0 I - c1 D) X = B as one cooperative kernel.
// A block owns tiles of 32 x 8 nodes; a product with the matrix takes its vector
// from shared memory, where the tile and its ring of neighbours are formed from the
// recurrences (p = r + beta p - beta omega v, y = p/diag; s = r - alpha v, z = s/diag), so
// an iteration is three passes with one grid barrier and one reduction each.  Every
// block sums the blocks' partial dot products in the same order and so takes the same
// scalars and the same decision to stop.  Bound by the latency of the three barriers;
// NIG1, N_x = 150, 75 steps: 103 us a system, 535 -> 506 ms for the whole solve against
// sixteen kernels an iteration.
// ---------------------------------------------------------------------------
namespace {
constexpr int kTX = 32, kTY = 8, kPsThreads = kTX * kTY;
constexpr unsigned kSpinLimit = 1u << 22;            // a barrier gives up after a few seconds
}  // namespace

// all blocks of the (cooperative) grid; false once any block gave up waiting
__device__ __forceinline__ bool ps_barrier(PsBicg* st, unsigned& gen) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        gen += gridDim.x;
        __threadfence();
        atomicAdd(&st->arrived, 1u);
        unsigned spins = 0;
        while (*(volatile unsigned*)&st->arrived < gen && ++spins < kSpinLimit) {}
        __threadfence();
        ok = spins < kSpinLimit;
        if (!ok) st->stalled = 1;
    }
    __syncthreads();
    return ok != 0;
}

// sums over the grid of NV values per thread, in a fixed order; part: NV doubles per block
template <int NV>
__device__ __forceinline__ bool ps_grid_sum(double* v, double* part, PsBicg* st, unsigned& gen) {
    __shared__ double red[NV][kPsThreads / 32];
    __shared__ double tot[NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto warp_sum = [](double x) {
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    };
    __syncthreads();                                  // red and tot of the previous call are read
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const double x = warp_sum(v[k]);
        if (lane == 0) red[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double x = 0.0;
        for (int u = 0; u < kPsThreads / 32; ++u) x += red[threadIdx.x][u];
        part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = x;
    }
    if (!ps_barrier(st, gen)) return false;
    if (w < NV) {
        double x = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) x += __ldcg(part + (size_t)w * gridDim.x + b);
        x = warp_sum(x);
        if (lane == 0) tot[w] = x;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = tot[k];
    return true;
}

__global__ void __launch_bounds__(kPsThreads) k_ps_bicg(PsBicgArgs a) {
    __shared__ double sv[kTY + 2][kTX + 2];
    const int n1 = a.d.n1, N = n1 - 1;
    const int ntx = (n1 + kTX - 1) / kTX, nty = (n1 + kTY - 1) / kTY, ntiles = ntx * nty;
    const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX;
    unsigned gen = 0;
    // vec(i) at the nodes of a tile and their ring into sv, then f(i, A vec at node i, vec) at
    // the tile's nodes, A = c0 I - c1 D
    auto product = [&](auto vec, auto f) {
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int x0 = (tile % ntx) * kTX, y0 = (tile / ntx) * kTY;
            __syncthreads();
            for (int q = threadIdx.x; q < (kTX + 2) * (kTY + 2); q += kPsThreads) {
                const int cy = q / (kTX + 2), cx = q - cy * (kTX + 2);
                const int q1 = x0 - 1 + cx, q2 = y0 - 1 + cy;
                if (q1 < 0 || q2 < 0 || q1 > N || q2 > N) continue;
                const bool own = cx >= 1 && cx <= kTX && cy >= 1 && cy <= kTY;
                sv[cy][cx] = vec((size_t)q2 * n1 + q1, own);
            }
            __syncthreads();
            const int m1 = x0 + tx, m2 = y0 + ty;
            if (m1 > N || m2 > N) continue;
            double d2x = 0.0, d2y = 0.0, mix = 0.0;
#pragma unroll
            for (int i = -1; i <= 1; ++i) {
                const int c1 = clampi(m1 + i, N) - m1 + tx + 1, c2 = clampi(m2 + i, N) - m2 + ty + 1;
                d2x += a.d.b2[m1 * 3 + i + 1] * sv[ty + 1][c1];
                d2y += a.d.b2[m2 * 3 + i + 1] * sv[c2][tx + 1];
                const double a2 = a.d.a1[m2 * 3 + i + 1];
                if (a2 != 0.0) {
#pragma unroll
                    for (int j = -1; j <= 1; ++j)
                        mix += a2 * a.d.a1[m1 * 3 + j + 1] * sv[c2][clampi(m1 + j, N) - m1 + tx + 1];
                }
            }
            const double x1 = a.d.x[m1], x2 = a.d.x[m2];
            const double dv = 0.5 * a.d.A11 * x1 * x1 * d2x + a.d.A12 * x1 * x2 * mix + 0.5 * a.d.A22 * x2 * x2 * d2y;
            const double c = sv[ty + 1][tx + 1];
            f((size_t)m2 * n1 + m1, a.c0 * c - a.c1 * dv, c);
        }
    };
    // the block's own nodes
    auto own_nodes = [&](auto f) {
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int m1 = (tile % ntx) * kTX + tx, m2 = (tile / ntx) * kTY + ty;
            if (m1 <= N && m2 <= N) f((size_t)m2 * n1 + m1);
        }
    };
    PsBicg q{};
    q.rho = q.alpha = q.omega = 1.0;
    double acc[3] = {0.0, 0.0, 0.0};
    product([&](size_t i, bool) { return a.X[i]; },
            [&](size_t i, double av, double) {
                const double b = a.B[i], r = b - av;
                a.r[i] = r;
                a.rh[i] = r;
                acc[0] += b * b;
                acc[1] += r * r;
            });
    if (!ps_grid_sum<2>(acc, a.part + 6 * (size_t)gridDim.x, a.st, gen)) return;
    const double bn = sqrt(acc[0]);
    q.lim = 1e-13 * (bn > 0.0 ? bn : 1.0);
    q.rn = sqrt(acc[1]);
    q.rho_new = acc[1];
    while (q.rn > q.lim && q.it < a.maxit) {
        // the old p and v are read at neighbours while the new ones are written: two of each
        double* const pn = q.it & 1 ? a.p1 : a.p0;
        double* const vn = q.it & 1 ? a.v1 : a.v0;
        const double* const po = q.it & 1 ? a.p0 : a.p1;
        const double* const vo = q.it & 1 ? a.v0 : a.v1;
        const double beta = (q.rho_new / q.rho) * (q.alpha / q.omega), bo = -beta * q.omega;
        const bool first = q.it == 0;
        acc[0] = 0.0;
        product([&](size_t i, bool own) {
                    double p = __ldcg(a.r + i);
                    if (!first) p = p + beta * __ldcg(po + i) + bo * __ldcg(vo + i);
                    if (own) pn[i] = p;
                    return p * a.dinv[i];
                },
                [&](size_t i, double av, double) {
                    vn[i] = av;
                    acc[0] += a.rh[i] * av;
                });
        if (!ps_grid_sum<1>(acc, a.part, a.st, gen)) return;
        q.alpha = q.rho_new / acc[0];
        acc[0] = acc[1] = acc[2] = 0.0;
        product([&](size_t i, bool own) {
                    const double sn = __ldcg(a.r + i) - q.alpha * __ldcg(vn + i);
                    if (own) a.s[i] = sn;
                    return sn * a.dinv[i];
                },
                [&](size_t i, double av, double) {
                    const double sn = a.s[i];         // written by this block, before the tile's barrier
                    a.t[i] = av;
                    acc[0] += av * sn;
                    acc[1] += av * av;
                    acc[2] += sn * sn;
                });
        // (three regions of partial sums in turn: a block may still be reading the previous ones)
        if (!ps_grid_sum<3>(acc, a.part + 3 * (size_t)gridDim.x, a.st, gen)) return;
        q.it += 1;
        const double sn = sqrt(acc[2]);
        if (sn <= q.lim) {
            q.rn = sn;
            q.done = 1;
            own_nodes([&](size_t i) { a.X[i] = a.X[i] + q.alpha * (pn[i] * a.dinv[i]); });
            break;
        }
        q.omega = acc[0] / acc[1];
        acc[0] = acc[1] = 0.0;
        own_nodes([&](size_t i) {
            const double di = a.dinv[i], s = a.s[i];
            a.X[i] = a.X[i] + q.alpha * (pn[i] * di) + q.omega * (s * di);
            const double r = s - q.omega * a.t[i];
            a.r[i] = r;
            acc[0] += r * r;
            acc[1] += a.rh[i] * r;
        });
        if (!ps_grid_sum<2>(acc, a.part + 6 * (size_t)gridDim.x, a.st, gen)) return;
        q.rho = q.rho_new;
        q.rn = sqrt(acc[0]);
        q.rho_new = acc[1];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.st->rn = q.rn;
        a.st->lim = q.lim;
        a.st->it = q.it;
        a.st->done = q.done;
    }
}

// blocks of the solve: one per tile, as many as are resident together (0 on error)
int ps_bicg_blocks(int n1) {
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_ps_bicg, kPsThreads, 0) != cudaSuccess)
        return 0;
    const int tiles = ((n1 + kTX - 1) / kTX) * ((n1 + kTY - 1) / kTY);
    return std::min(std::min(tiles, per * sms), kPsRedBlocks);
}

cudaError_t launch_ps_bicg(const PsBicgArgs& a, int blocks, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(a.st, 0, sizeof(PsBicg), s);
    if (e != cudaSuccess) return e;
    PsBicgArgs b = a;
    void* args[] = {&b};
    return cudaLaunchCooperativeKernel((const void*)k_ps_bicg, dim3(blocks), dim3(kPsThreads), args, 0, s);
}

cudaError_t launch_ps_update(size_t n, const double* X, double* Y, double* T, double* part, double* res, cudaStream_t s) {
    k_ps_update<<<kPsRedBlocks, 256, 0, s>>>(n, X, Y, T, part);
    k_ps_finish<<<1, 256, 0, s>>>(part, kPsRedBlocks, res);
    return cudaGetLastError();
}

}  // namespace pide

namespace pide {

// W[m2][m1] = sum_{b,c} w2[m2][b] w1[m1][c] Z[s2[m2]+b][s1[m1]+c]: the departure interpolation T_SL
__global__ void k_ps_sl(int n1, const int* __restrict__ s1, const double* __restrict__ w1, const int* __restrict__ s2,
                        const double* __restrict__ w2, const double* __restrict__ Z, double* __restrict__ W) {
    const int m1 = blockIdx.x * blockDim.x + threadIdx.x, m2 = blockIdx.y * blockDim.y + threadIdx.y;
    if (m1 >= n1 || m2 >= n1) return;
    const int a1 = s1[m1], a2 = s2[m2];
    double acc = 0.0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const double* row = Z + (size_t)(a2 + b) * n1 + a1;
        double r = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) r += w1[m1 * 4 + c] * row[c];
        acc += w2[m2 * 4 + b] * r;
    }
    W[(size_t)m2 * n1 + m1] = acc;
}

cudaError_t launch_ps_sl(int n1, const int* s1, const double* w1, const int* s2, const double* w2, const double* Z,
                         double* W, cudaStream_t s) {
    const dim3 blk(kBX, kBY), grd((n1 + kBX - 1) / kBX, (n1 + kBY - 1) / kBY);
    k_ps_sl<<<grd, blk, 0, s>>>(n1, s1, w1, s2, w2, Z, W);
    return cudaGetLastError();
}

}  // namespace pide
