// FP64 CUDA kernels of the hot path: Kronecker-structured transport and
// mass applies (eq. AR, bMebMo with eq. tpmv), the scattering and eigenbasis
// contractions (eq. bKebKo, Lemma apply_high_order_pre), the coarse-matrix
// apply, per-RHS reductions, and the setup-time quadrature of S^+ / S^-.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>

#include "device.h"
#include "rte_internal.h"

namespace rte {

namespace {

constexpr int kThreads = 256;

inline unsigned grid_for(size_t n, int threads = kThreads) {
    size_t b = (n + threads - 1) / threads;
    const size_t cap = 65535ull * 32ull;
    return (unsigned)std::max<size_t>(1, std::min(b, cap));
}

// ------------------------------------------------------------------ GEMM
// Row-major C = alpha * (A B) .* F + beta * C: TM x TN tiles, 16-deep K steps,
// 256 threads with a TM / 16 x TN / 16 register tile each, the next step's
// operands loaded into registers under the current one's products.
//
// What bounds it: the FP64 units (about two fused multiply-adds per clock and
// SM), so what counts is that every SM has the same share of them: 64 x 64
// tiles leave 152 SMs two thirds idle on a 32 x 32 mesh (96 tiles) and nine
// tenths on the smallest calls (18).  gemm_f64 takes the tile with the least
// products on the busiest SM.  Every output sums over k in the same order
// whatever the tile.  Measured: one E - K^+ on 9 x 9 cells, 64
// directions, two right-hand sides (324 x 192 x 128) 450 -> 80 us; a 32 x 32
// solve in FP64 (2048 x 192 x 128) 22.4 -> 17.8 ms.
template <int EPI, int TM, int TN>
__global__ void __launch_bounds__(256)
k_gemm_f64(int M, int N, int K, const double* __restrict__ A, int lda,
           const double* __restrict__ B, int ldb, double* C, int ldc,
           double alpha, double beta, const double* __restrict__ at,
           const double* __restrict__ as, const double* __restrict__ lam,
           int rows) {
    constexpr int RM = TM / 16, RN = TN / 16;   // outputs, and operands to load, per thread
    __shared__ double As[16][TM + 1];
    __shared__ double Bs[16][TN + 2];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    // one-dimensional grid, column tiles fastest: the row tiles of a tall call
    // (one per 16 rows of nrhs n_R^-) exceed the 65535 of the grid's y
    const int ntn = (N + TN - 1) / TN;
    const int m0 = (int)(blockIdx.x / ntn) * TM, n0 = (int)(blockIdx.x % ntn) * TN;
    double acc[RM][RN], a[RM], b[RN];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = 0.0;
    auto load = [&](int k0) {
#pragma unroll
        for (int t = 0; t < RM; ++t) {
            const int gr = m0 + ty + 16 * t, gc = k0 + tx;
            a[t] = (gr < M && gc < K) ? A[(size_t)gr * lda + gc] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < RN; ++t) {
            const int e = threadIdx.x + t * 256, br = e / TN, bc = e % TN;
            b[t] = (k0 + br < K && n0 + bc < N) ? B[(size_t)(k0 + br) * ldb + n0 + bc] : 0.0;
        }
    };
    load(0);
    for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
        for (int t = 0; t < RM; ++t) As[tx][ty + 16 * t] = a[t];
#pragma unroll
        for (int t = 0; t < RN; ++t) {
            const int e = threadIdx.x + t * 256;
            Bs[e / TN][e % TN] = b[t];
        }
        __syncthreads();
        if (k0 + 16 < K) load(k0 + 16);
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            double x[RM], y[RN];
#pragma unroll
            for (int i = 0; i < RM; ++i) x[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < RN; ++j) y[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < RN; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int r = m0 + ty + 16 * i;
        if (r >= M) continue;
        double fat = 0.0, fas = 0.0;
        if (EPI != 0) {
            const int rr = r % rows;
            fat = at[rr];
            fas = as[rr];
        }
#pragma unroll
        for (int j = 0; j < RN; ++j) {
            const int c = n0 + tx + 16 * j;
            if (c >= N) continue;
            double v = acc[i][j];
            if (EPI == 1) v = v / (fat - lam[c] * fas);
            if (EPI == 2) v = v * (1.0 / (fat - lam[c] * fas) - 1.0 / fat);
            v *= alpha;
            double* dst = C + (size_t)r * ldc + c;
            if (beta != 0.0) v += beta * *dst;
            *dst = v;
        }
    }
}

// (M^- - K^-) z = at_j (z_j M_S^-) - as_j (z_j S^-),  G = Z S^- precomputed
__global__ void k_mk_combine(int nRm, int nSp, int nrhs,
                             const double* __restrict__ at,
                             const double* __restrict__ as,
                             const double* __restrict__ MSm,
                             const double* __restrict__ Z,
                             const double* __restrict__ G, double* __restrict__ Y) {
    const unsigned total = (unsigned)nrhs * nRm * nSp;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += gridDim.x * blockDim.x) {
        const int k = (int)(e % (unsigned)nSp);
        const unsigned rj = e / (unsigned)nSp;
        const int j = (int)(rj % (unsigned)nRm);
        const size_t base = rj * 3 * nSp + 3 * k;
        const double z[3] = {Z[base], Z[base + 1], Z[base + 2]};
        const double* M = MSm + 9 * k;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double mz = M[3 * c] * z[0] + M[3 * c + 1] * z[1] + M[3 * c + 2] * z[2];
            Y[base + c] = at[j] * mz - as[j] * G[base + c];
        }
    }
}

// Y = (B M_S^{-1}) / at   (the high-order part of eq. MmKprecond)
__global__ void k_mk_minv_scale(int nRm, int nSp, int nrhs,
                                const double* __restrict__ at,
                                const double* __restrict__ MSm_inv,
                                const double* __restrict__ B, double* __restrict__ Y) {
    const unsigned total = (unsigned)nrhs * nRm * nSp;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += gridDim.x * blockDim.x) {
        const int k = (int)(e % (unsigned)nSp);
        const unsigned rj = e / (unsigned)nSp;
        const int j = (int)(rj % (unsigned)nRm);
        const size_t base = rj * 3 * nSp + 3 * k;
        const double b[3] = {B[base], B[base + 1], B[base + 2]};
        const double* M = MSm_inv + 9 * k;
        const double inv = 1.0 / at[j];
#pragma unroll
        for (int c = 0; c < 3; ++c)
            Y[base + c] = (M[3 * c] * b[0] + M[3 * c + 1] * b[1] + M[3 * c + 2] * b[2]) * inv;
    }
}

__global__ void k_rhs_source(int nRp, int nSp, int nrhs, int nnz,
                             const int* __restrict__ st_ptr,
                             const int* __restrict__ st_col,
                             const double* __restrict__ sval,
                             const double* __restrict__ m,
                             const double* __restrict__ qn, double* __restrict__ q) {
    const size_t total = (size_t)nrhs * nRp * nSp;
    const double* Mu = sval + (size_t)kMu * nnz;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e % nSp);
        const size_t ri = e / nSp;
        const int i = (int)(ri % nRp);
        const int r = (int)(ri / nRp);
        double s = 0.0;
        for (int p = st_ptr[i]; p < st_ptr[i + 1]; ++p)
            s += Mu[p] * qn[(size_t)r * nRp + st_col[p]];
        q[e] = s * m[k];
    }
}

// Inflow part of l^+ (Section 2.4): 2 (|s.n| g, phi_i mu_k) over the
// incoming half of the boundary.  On face f with outward normal n, exactly
// one triangle of pair k has s.n < 0 (the octahedral sphere mesh has no
// triangle across a coordinate plane): half[f][k] says which.  Its integral
// of |s.n| is half of omega_k (omega^x on the faces x = 0, 1, omega^y on
// y = 0, 1), and the data is P1 along the face, so
//   q[i(f, j)][k] += omega_k sum_j' B1[j][j'] g[f][j'][2k + half[f][k]]
// with B1 the face's 1-D P1 mass (h/3 at the ends, 2h/3 inside, h/6 off the
// diagonal, h = 1/m).  One launch takes the two opposite faces f0, f0 + 1,
// whose nodes are disjoint, so no two threads add to one entry.
__global__ void k_inflow(int m, int nSp, int nrhs, int f0, const int* __restrict__ half,
                         const double* __restrict__ omx, const double* __restrict__ omy,
                         const double* __restrict__ g, double* __restrict__ q) {
    const int nf = m + 1, nRp = nf * nf;
    const size_t total = (size_t)nrhs * 2 * nf * nSp;
    const double h = 1.0 / m;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e % nSp);
        size_t rest = e / nSp;
        const int j = (int)(rest % nf);
        rest /= nf;
        const int f = f0 + (int)(rest % 2);
        const int r = (int)(rest / 2);
        const int hk = half[f * nSp + k];
        const double* gf = g + ((size_t)r * 4 + f) * nf * 2 * nSp + 2 * k + hk;
        const double gj = gf[(size_t)j * 2 * nSp];
        double acc = (j == 0 || j == m ? h / 3.0 : 2.0 * h / 3.0) * gj;
        if (j > 0) acc += h / 6.0 * gf[(size_t)(j - 1) * 2 * nSp];
        if (j < m) acc += h / 6.0 * gf[(size_t)(j + 1) * 2 * nSp];
        const double om = f < 2 ? omx[k] : omy[k];
        // node of face f's j-th point: x = 0 / x = 1 run along y, y = 0 / y = 1 along x
        const int i = f == 0 ? j * nf : f == 1 ? j * nf + m : f == 2 ? j : m * nf + j;
        q[((size_t)r * nRp + i) * nSp + k] += om * acc;
    }
}

// ------------------------------------------------------------ reductions
template <int BS>
__device__ double block_sum(double v) {
    __shared__ double sh[BS / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < BS / 32 ? sh[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;  // valid in thread 0
}

// x[e] uniform in [-1, 1) from the SplitMix64 mix of (seed, e) (Steele,
// Lea and Flood, "Fast splittable pseudorandom number generators", 2014).
__global__ void k_fill_uniform(double* __restrict__ x, size_t n, unsigned long long seed) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
         e += (size_t)gridDim.x * blockDim.x) {
        unsigned long long z = seed + (e + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        x[e] = (double)(z >> 11) * 0x1.0p-52 - 1.0;
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_dot_partial(const T* __restrict__ x, const T* __restrict__ y,
              size_t len, double* __restrict__ partial) {
    const int r = blockIdx.y;
    const T* xr = x + (size_t)r * len;
    const T* yr = y + (size_t)r * len;
    double s = 0.0;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < len;
         e += (size_t)gridDim.x * blockDim.x)
        s = fma((double)xr[e], (double)yr[e], s);
    s = block_sum<256>(s);
    if (threadIdx.x == 0) partial[(size_t)r * 1024 + blockIdx.x] = s;
}

__global__ void __launch_bounds__(256)
k_dot_final(const double* __restrict__ partial, int nb, double* __restrict__ out) {
    const int r = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += partial[(size_t)r * 1024 + b];
    s = block_sum<256>(s);
    if (threadIdx.x == 0) out[r] = s;
}

template <typename T>
__global__ void k_axpby(const T* __restrict__ x, T* __restrict__ y,
                        size_t len, int nrhs, const double* __restrict__ a,
                        double ca, const double* __restrict__ b, double cb) {
    const unsigned total = (unsigned)(len * nrhs);
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += gridDim.x * blockDim.x) {
        const int r = nrhs == 1 ? 0 : (int)(e / (unsigned)len);
        const T av = static_cast<T>(a ? a[r] : ca);
        const T bv = static_cast<T>(b ? b[r] : cb);
        const T yv = bv == T(0) ? T(0) : bv * y[e];
        y[e] = (x ? av * x[e] : T(0)) + yv;
    }
}

// W consecutive values a thread: 4 where the pointers and n allow it (2048 x
// 16384 FP64 to BF16: 107 -> 62 us, bound by memory), else 1
template <typename TI, typename TO, int W>
__global__ void k_convert(const TI* __restrict__ x, TO* __restrict__ y, size_t n) {
    struct alignas(sizeof(TI) * W) In { TI v[W]; };
    struct alignas(sizeof(TO) * W) Out { TO v[W]; };
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n / W;
         e += (size_t)gridDim.x * blockDim.x) {
        const In a = reinterpret_cast<const In*>(x)[e];
        Out b;
#pragma unroll
        for (int w = 0; w < W; ++w) b.v[w] = static_cast<TO>(a.v[w]);
        reinterpret_cast<Out*>(y)[e] = b;
    }
}

// --------------------------------------------------------- coarse apply
// Y[r, i, a] = sum_p sum_b Ec[p, a, b] X[r, col(p), b]
__global__ void k_coarse_apply(int nRp, int d, int nrhs, const int* __restrict__ st_ptr,
                               const int* __restrict__ st_col,
                               const double* __restrict__ ec,
                               const double* __restrict__ X, double* __restrict__ Y) {
    const size_t total = (size_t)nrhs * nRp * d;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int a = (int)(e % d);
        const size_t ri = e / d;
        const int i = (int)(ri % nRp);
        const int r = (int)(ri / nRp);
        const double* Xr = X + (size_t)r * nRp * d;
        double s = 0.0;
        for (int p = st_ptr[i]; p < st_ptr[i + 1]; ++p) {
            const double* blk = ec + ((size_t)p * d + a) * d;
            const double* xv = Xr + (size_t)st_col[p] * d;
            for (int b = 0; b < d; ++b) s = fma(blk[b], xv[b], s);
        }
        Y[e] = s;
    }
}

// ------------------------------------------------ quadrature of S^+, S^-
__device__ __forceinline__ double hg_eval(double mu, double g, double c0) {
    const double t = 1.0 + g * g - 2.0 * g * mu;
    return c0 / (t * sqrt(t));
}

// Far rule for every pair: one thread per (k, k').
__global__ void k_scatter_far(int n, double g, const double* __restrict__ pts,
                              const double* __restrict__ w,
                              const double* __restrict__ psi, int qf,
                              double* __restrict__ Sp, double* __restrict__ Sm) {
    const size_t pair = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (pair >= (size_t)n * n) return;
    const int k = (int)(pair / n), kk = (int)(pair % n);
    const double c0 = (1.0 - g * g) / (4.0 * 3.14159265358979323846);
    double sp = 0.0, sm[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int p = 0; p < qf; ++p) {
        const double* s = pts + ((size_t)k * qf + p) * 3;
        const double wp = w[(size_t)k * qf + p];
        const double* ps = psi + ((size_t)k * qf + p) * 3;
        double rowp = 0.0, rowm[3] = {0, 0, 0};
        for (int q = 0; q < qf; ++q) {
            const double* t = pts + ((size_t)kk * qf + q) * 3;
            const double mu = s[0] * t[0] + s[1] * t[1] + s[2] * t[2];
            const double kp = hg_eval(mu, g, c0), km = hg_eval(-mu, g, c0);
            const double wq = w[(size_t)kk * qf + q];
            const double* pq = psi + ((size_t)kk * qf + q) * 3;
            rowp += wq * (kp + km);
            const double dk = wq * (kp - km);
            rowm[0] += dk * pq[0];
            rowm[1] += dk * pq[1];
            rowm[2] += dk * pq[2];
        }
        sp += wp * rowp;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) sm[3 * i + j] += wp * ps[i] * rowm[j];
    }
    Sp[(size_t)k * n + kk] = 2.0 * sp;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            Sm[(size_t)(3 * k + i) * 3 * n + 3 * kk + j] = 2.0 * sm[3 * i + j];
}

// Near rule for vertex-sharing pairs: one block per (k, k'), one thread per
// node of K_k.
__global__ void __launch_bounds__(256)
k_scatter_near(int n, double g, const double* __restrict__ pts,
               const double* __restrict__ w, const double* __restrict__ psi, int qn,
               const int* __restrict__ near_ptr, const int* __restrict__ near_idx,
               const int* __restrict__ pair_row, double* __restrict__ Sp,
               double* __restrict__ Sm) {
    const int pidx = blockIdx.x;
    const int k = pair_row[pidx];
    const int kk = near_idx[pidx];
    const double c0 = (1.0 - g * g) / (4.0 * 3.14159265358979323846);
    double sp = 0.0, sm[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int p = threadIdx.x; p < qn; p += blockDim.x) {
        const double* s = pts + ((size_t)k * qn + p) * 3;
        const double wp = w[(size_t)k * qn + p];
        const double* ps = psi + ((size_t)k * qn + p) * 3;
        double rowp = 0.0, rowm[3] = {0, 0, 0};
        for (int q = 0; q < qn; ++q) {
            const double* t = pts + ((size_t)kk * qn + q) * 3;
            const double mu = s[0] * t[0] + s[1] * t[1] + s[2] * t[2];
            const double kp = hg_eval(mu, g, c0), km = hg_eval(-mu, g, c0);
            const double wq = w[(size_t)kk * qn + q];
            const double* pq = psi + ((size_t)kk * qn + q) * 3;
            rowp += wq * (kp + km);
            const double dk = wq * (kp - km);
            rowm[0] += dk * pq[0];
            rowm[1] += dk * pq[1];
            rowm[2] += dk * pq[2];
        }
        sp += wp * rowp;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) sm[3 * i + j] += wp * ps[i] * rowm[j];
    }
    sp = block_sum<256>(sp);
    if (threadIdx.x == 0) Sp[(size_t)k * n + kk] = 2.0 * sp;
    for (int c = 0; c < 9; ++c) {
        const double v = block_sum<256>(sm[c]);
        if (threadIdx.x == 0)
            Sm[(size_t)(3 * k + c / 3) * 3 * n + 3 * kk + c % 3] = 2.0 * v;
    }
}

__global__ void k_symmetrise(int n, double* __restrict__ S) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e >= (size_t)n * n) return;
    const int i = (int)(e / n), j = (int)(e % n);
    if (j <= i) return;
    const double v = 0.5 * (S[(size_t)i * n + j] + S[(size_t)j * n + i]);
    S[(size_t)i * n + j] = v;
    S[(size_t)j * n + i] = v;
}

__global__ void k_e0_coef(int nRp, int nSp, const double* __restrict__ ell6,
                          const double* __restrict__ e0s, double* __restrict__ coef,
                          float* __restrict__ coef_f) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const size_t per = (size_t)7 * nRp;
    if (e >= per * nSp) return;
    const size_t di = e / nSp;          // dir * nRp + i
    const int k = (int)(e % nSp);
    double c = 0.0;
    for (int q = 0; q < 6; ++q) c += e0s[6 * k + q] * ell6[(size_t)q * per + di];
    coef[e] = c;
    if (coef_f) coef_f[e] = (float)c;
}

__global__ void k_near_rows(int n, const int* __restrict__ near_ptr, int* __restrict__ row) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    for (int p = near_ptr[k]; p < near_ptr[k + 1]; ++p) row[p] = k;
}

// ------------------------------------------- structured-mesh versions
// The m x m "/"-mesh: node (x, y) = y (m+1) + x; square (I, J) holds cells
// 2 (J m + I) (lower: (I,J),(I+1,J),(I+1,J+1)) and 2 (J m + I) + 1 (upper:
// (I,J),(I+1,J+1),(I,J+1)).  Adjacency is computed, not looked up.
template <typename TIn, typename TOut, typename TC>
__global__ void k_apply_A_s(int m, int nSp, int nrhs, const TC* __restrict__ cell_D,
                            const TC* __restrict__ A1, const TC* __restrict__ A2,
                            const TIn* __restrict__ U, TOut* __restrict__ Z) {
    const int nRm = 2 * m * m, nRp = (m + 1) * (m + 1);
    const unsigned total = (unsigned)nrhs * nRm * nSp;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += gridDim.x * blockDim.x) {
        const int k = (int)(e % (unsigned)nSp);
        const unsigned rj = e / (unsigned)nSp;
        const int j = (int)(rj % (unsigned)nRm);
        const int r = (int)(rj / (unsigned)nRm);
        const int q = j >> 1, I = q % m, J = q / m;
        const int n00 = J * (m + 1) + I;
        const int nd[3] = {n00, (j & 1) ? n00 + m + 2 : n00 + 1,
                           (j & 1) ? n00 + m + 1 : n00 + m + 2};
        const TIn* Ur = U + (size_t)r * nRp * nSp + k;
        TC g1 = 0, g2 = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const TC u = static_cast<TC>(Ur[(size_t)nd[a] * nSp]);
            g1 = fma(cell_D[6 * j + a], u, g1);
            g2 = fma(cell_D[6 * j + 3 + a], u, g2);
        }
        TOut* z = Z + (size_t)rj * (3 * (size_t)nSp) + 3 * k;
#pragma unroll
        for (int c = 0; c < 3; ++c)
            z[c] = static_cast<TOut>(A1[3 * k + c] * g1 + A2[3 * k + c] * g2);
    }
}

// Y = [A^T Zp] + [M^+ X + R X] - [M_s^+ V] on the structured mesh; ell4 holds
// M_t^+, M_s^+, B_x, B_y in ELL form [4][7][nRp].
template <typename T>
__global__ void k_apply_even_s(int m, int nSp, int nrhs, int flags,
                               const T* __restrict__ cell_D, const T* __restrict__ A1,
                               const T* __restrict__ A2, const T* __restrict__ ell4,
                               const T* __restrict__ mk, const T* __restrict__ omx,
                               const T* __restrict__ omy, const T* __restrict__ Zp,
                               const T* __restrict__ X, const T* __restrict__ V,
                               T* __restrict__ Y) {
    const int nRp = (m + 1) * (m + 1), nRm = 2 * m * m;
    const unsigned total = (unsigned)nrhs * nRp * nSp;
    const int off[7] = {0, 1, -1, m + 1, -(m + 1), m + 2, -(m + 2)};
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += gridDim.x * blockDim.x) {
        const int k = (int)(e % (unsigned)nSp);
        const unsigned ri = e / (unsigned)nSp;
        const int i = (int)(ri % (unsigned)nRp);
        const int r = (int)(ri / (unsigned)nRp);
        const int x = i % (m + 1), y = i / (m + 1);
        T acc = 0;
        if (flags & 1) {
            const T a1[3] = {A1[3 * k], A1[3 * k + 1], A1[3 * k + 2]};
            const T a2[3] = {A2[3 * k], A2[3 * k + 1], A2[3 * k + 2]};
            const T* Zr = Zp + (size_t)r * nRm * 3 * nSp + 3 * k;
            // the six cells around node (x, y) and the node's local index
            const int cI[6] = {x, x, x - 1, x - 1, x - 1, x};
            const int cJ[6] = {y, y, y, y - 1, y - 1, y - 1};
            const int up[6] = {0, 1, 0, 0, 1, 1};
            const int loc[6] = {0, 0, 1, 2, 1, 2};
#pragma unroll
            for (int t = 0; t < 6; ++t) {
                if (cI[t] < 0 || cJ[t] < 0 || cI[t] >= m || cJ[t] >= m) continue;
                const int j = 2 * (cJ[t] * m + cI[t]) + up[t];
                const T* z = Zr + (size_t)j * 3 * nSp;
                const T z0 = z[0], z1 = z[1], z2 = z[2];
                const T t1 = a1[0] * z0 + a1[1] * z1 + a1[2] * z2;
                const T t2 = a2[0] * z0 + a2[1] * z1 + a2[2] * z2;
                acc += cell_D[6 * j + loc[t]] * t1 + cell_D[6 * j + 3 + loc[t]] * t2;
            }
        }
        if (flags & 6) {
            const T mkv = mk[k], ox = omx[k], oy = omy[k];
            const T* Xr = X + (size_t)r * nRp * nSp + k;
            const T* Vr = V ? V + (size_t)r * nRp * nSp + k : nullptr;
            const size_t sl = (size_t)7 * nRp;
#pragma unroll
            for (int dir = 0; dir < 7; ++dir) {
                int jn = i + off[dir];
                jn = jn < 0 ? 0 : (jn >= nRp ? nRp - 1 : jn);
                const size_t pe = (size_t)dir * nRp + i;
                if (flags & 2)
                    acc += (mkv * ell4[pe] + ox * ell4[2 * sl + pe] + oy * ell4[3 * sl + pe]) *
                           Xr[(size_t)jn * nSp];
                if (flags & 4) acc -= ell4[sl + pe] * Vr[(size_t)jn * nSp];
            }
        }
        Y[e] = acc;
    }
}

// ------------------------------------------- the eigenbasis route's E
// (M^- - K^-)^{-1} between A and A^T needs only what A's odd values carry:
// A u = A_1 (x) D_1 u + A_2 (x) D_2 u has two spatial derivatives per cell and
// direction, not three free values, and A^T takes two projections back.  So
// with W = [A_1 A_2]^T V (2 n_S^+ x n_S^-, V the eigenvectors) the
// contractions run from and to the derivatives, 2/3 of their work, and the
// two kernels below need 8 products per square, direction and node where A
// and A^T on three odd values took 12 and 48.
//
// W consecutive directions per thread: 2 where the pointers are aligned for it,
// else 1.
constexpr int kMaxSpmm = 512;   // threads a block, at most (autotuned: 128, 256, 512)
template <typename T, int N>
struct alignas(sizeof(T) * N) Pack {
    T v[N];
};

// G[r, j, 2k + d] = sign (D_d U_r)[j, k] for both cells of every square.  On
// the "/"-mesh each hat function of a cell has a derivative along x or along y
// only, but for one: the terms that are zero are left out.
template <int W>
__global__ void __launch_bounds__(kMaxSpmm)
k_grad(int m, int nSp, int nrhs, double sign, const double* __restrict__ cell_D,
       const double* __restrict__ U, double* __restrict__ G) {
    const unsigned nk = (unsigned)nSp / W, total = (unsigned)nrhs * m * m * nk;
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const int k = (int)(e % nk) * W;
    const unsigned rq = e / nk;
    const int q = (int)(rq % (unsigned)(m * m)), r = (int)(rq / (unsigned)(m * m));
    const int I = q % m, J = q / m;
    const size_t n00 = ((size_t)r * (m + 1) * (m + 1) + (size_t)J * (m + 1) + I) * nSp + k;
    using PI = Pack<double, W>;
    auto node = [&](size_t o) { return *reinterpret_cast<const PI*>(U + o); };
    const PI u00 = node(n00), u10 = node(n00 + nSp), u01 = node(n00 + (size_t)(m + 1) * nSp),
             u11 = node(n00 + (size_t)(m + 2) * nSp);
    const double *lo = cell_D + 12 * (size_t)q, *up = lo + 6;   // D_1 of the three vertices, then D_2
    Pack<double, 2 * W> a, b;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const double x00 = u00.v[i], x10 = u10.v[i], x01 = u01.v[i], x11 = u11.v[i];
        a.v[2 * i] = sign * fma(lo[0], x00, lo[1] * x10);
        a.v[2 * i + 1] = sign * fma(lo[4], x10, lo[5] * x11);
        b.v[2 * i] = sign * fma(up[1], x11, up[2] * x01);
        b.v[2 * i + 1] = sign * fma(up[3], x00, up[5] * x01);
    }
    double* g = G + ((size_t)rq * 2 * nSp + k) * 2;
    *reinterpret_cast<Pack<double, 2 * W>*>(g) = a;
    *reinterpret_cast<Pack<double, 2 * W>*>(g + 2 * (size_t)nSp) = b;
}

// Y = sum_d D_d^T G_d + [M^+ X + R X] - [M_s^+ V] - [Q] (the terms whose
// pointer is set), G as k_grad lays it out.  The stencil sums come before the
// direction's factors, and the boundary terms on boundary nodes alone.
template <int W>
__global__ void __launch_bounds__(kMaxSpmm)
k_even_grad(int m, int nSp, int nrhs, const double* __restrict__ cell_D, const double* __restrict__ ell4,
            const double* __restrict__ mk, const double* __restrict__ omx, const double* __restrict__ omy,
            const double* __restrict__ G, const double* __restrict__ X, const double* __restrict__ V,
            const double* __restrict__ Q, double* __restrict__ Y) {
    const int n1 = m + 1, nRp = n1 * n1;
    const unsigned nk = (unsigned)nSp / W, total = (unsigned)nrhs * nRp * nk;
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const int k = (int)(e % nk) * W;
    const unsigned ri = e / nk;
    const int i = (int)(ri % (unsigned)nRp), r = (int)(ri / (unsigned)nRp);
    const int y = i / n1, x = i - y * n1;
    using P = Pack<double, W>;
    auto at = [&](const double* p, int node) {
        return *reinterpret_cast<const P*>(p + ((size_t)r * nRp + node) * nSp + k);
    };
    double acc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) acc[w] = 0.0;
    // the six cells around the node: square, cell of the square, and which of
    // the two derivatives the node's hat function has there
    const double* Gr = G + (size_t)r * 4 * m * m * nSp + 2 * k;
    auto cell = [&](int I, int J, int up, int loc, bool d1, bool d2) {
        const int j = 2 * (J * m + I) + up;
        const Pack<double, 2 * W> g = *reinterpret_cast<const Pack<double, 2 * W>*>(Gr + (size_t)j * 2 * nSp);
        const double* D = cell_D + 6 * (size_t)j + loc;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            if (d1) acc[w] = fma(D[0], g.v[2 * w], acc[w]);
            if (d2) acc[w] = fma(D[3], g.v[2 * w + 1], acc[w]);
        }
    };
    const bool l = x > 0, rt = x < m, dn = y > 0, tp = y < m;
    if (rt && tp) {
        cell(x, y, 0, 0, true, false);
        cell(x, y, 1, 0, false, true);
    }
    if (l && tp) cell(x - 1, y, 0, 1, true, true);
    if (l && dn) {
        cell(x - 1, y - 1, 0, 2, false, true);
        cell(x - 1, y - 1, 1, 1, true, false);
    }
    if (rt && dn) cell(x, y - 1, 1, 2, true, true);
    // neighbours in the order of the ELL form; one outside takes the node
    // itself (its coefficient is zero)
    const int nb[7] = {i, rt ? i + 1 : i, l ? i - 1 : i, tp ? i + n1 : i, dn ? i - n1 : i,
                       rt && tp ? i + n1 + 1 : i, l && dn ? i - n1 - 1 : i};
    const size_t sl = (size_t)7 * nRp;
    if (X) {
        double mass[W], bx[W], by[W];
#pragma unroll
        for (int w = 0; w < W; ++w) mass[w] = bx[w] = by[w] = 0.0;
        const bool edge = !(l && rt && dn && tp);
#pragma unroll
        for (int dir = 0; dir < 7; ++dir) {
            const size_t pe = (size_t)dir * nRp + i;
            const P u = at(X, nb[dir]);
            const double c = ell4[pe];
#pragma unroll
            for (int w = 0; w < W; ++w) mass[w] = fma(c, u.v[w], mass[w]);
            if (edge) {
                const double cx = ell4[2 * sl + pe], cy = ell4[3 * sl + pe];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    bx[w] = fma(cx, u.v[w], bx[w]);
                    by[w] = fma(cy, u.v[w], by[w]);
                }
            }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            acc[w] = fma(mk[k + w], mass[w], acc[w]);
            if (edge) acc[w] = fma(omx[k + w], bx[w], fma(omy[k + w], by[w], acc[w]));
        }
    }
    if (V) {
#pragma unroll
        for (int dir = 0; dir < 7; ++dir) {
            const P v = at(V, nb[dir]);
            const double c = -ell4[sl + (size_t)dir * nRp + i];
#pragma unroll
            for (int w = 0; w < W; ++w) acc[w] = fma(c, v.v[w], acc[w]);
        }
    }
    const size_t o = (size_t)ri * nSp + k;
    P out;
    if (Q) {
        const P q = *reinterpret_cast<const P*>(Q + o);
#pragma unroll
        for (int w = 0; w < W; ++w) out.v[w] = acc[w] - q.v[w];
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) out.v[w] = acc[w];
    }
    *reinterpret_cast<P*>(Y + o) = out;
}

// ------------------------------------------- the mixed modes' inner E
// A u and A^T z + M^+ x + R x - M_s^+ v on three odd values per direction, in
// FP32: between the derivatives instead (as above) the BF16 or TF32 operands
// of the contractions lose three to four times as much on smooth fields (7.5e-2
// against 1.9e-2 of E u on a 128 x 128 solution in BF16).  Bound by memory
// once a thread takes four directions (16-byte accesses, the cell and stencil
// coefficients loaded once for four) and leaves out the derivatives that are
// zero.  Measured on 128 x 128 / 256 directions: A u 56 us before, 19 now, the gather 94
// before, 50 now.
template <typename TOut>
__global__ void __launch_bounds__(kMaxSpmm)
k_odd_lo(int m, int nSp, int nrhs, const float* __restrict__ cell_D, const float* __restrict__ A1,
         const float* __restrict__ A2, const float* __restrict__ U, TOut* __restrict__ Z) {
    const unsigned nk = (unsigned)nSp / 4, total = (unsigned)nrhs * m * m * nk;
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const int k = (int)(e % nk) * 4;
    const unsigned rq = e / nk;
    const int q = (int)(rq % (unsigned)(m * m)), r = (int)(rq / (unsigned)(m * m));
    const int I = q % m, J = q / m;
    const size_t n00 = ((size_t)r * (m + 1) * (m + 1) + (size_t)J * (m + 1) + I) * nSp + k;
    using P4 = Pack<float, 4>;
    auto node = [&](size_t o) { return *reinterpret_cast<const P4*>(U + o); };
    const P4 u00 = node(n00), u10 = node(n00 + nSp), u01 = node(n00 + (size_t)(m + 1) * nSp),
             u11 = node(n00 + (size_t)(m + 2) * nSp);
    float a1[12], a2[12];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        *reinterpret_cast<P4*>(a1 + 4 * i) = *reinterpret_cast<const P4*>(A1 + 3 * k + 4 * i);
        *reinterpret_cast<P4*>(a2 + 4 * i) = *reinterpret_cast<const P4*>(A2 + 3 * k + 4 * i);
    }
    const float *lo = cell_D + 12 * (size_t)q, *up = lo + 6;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float z[12];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float g1 = c == 0 ? fmaf(lo[0], u00.v[i], lo[1] * u10.v[i])
                                    : fmaf(up[1], u11.v[i], up[2] * u01.v[i]);
            const float g2 = c == 0 ? fmaf(lo[4], u10.v[i], lo[5] * u11.v[i])
                                    : fmaf(up[3], u00.v[i], up[5] * u01.v[i]);
#pragma unroll
            for (int j = 0; j < 3; ++j) z[3 * i + j] = a1[3 * i + j] * g1 + a2[3 * i + j] * g2;
        }
        TOut* out = Z + ((size_t)rq * 2 + c) * 3 * nSp + 3 * k;
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            Pack<TOut, 4> w;
#pragma unroll
            for (int i = 0; i < 4; ++i) w.v[i] = static_cast<TOut>(z[4 * p + i]);
            *reinterpret_cast<Pack<TOut, 4>*>(out + 4 * p) = w;
        }
    }
}

__global__ void __launch_bounds__(kMaxSpmm)
k_even_lo(int m, int nSp, int nrhs, const float* __restrict__ cell_D, const float* __restrict__ A1,
          const float* __restrict__ A2, const float* __restrict__ ell4,
          const float* __restrict__ mk, const float* __restrict__ omx,
          const float* __restrict__ omy, const float* __restrict__ Z, const float* __restrict__ X,
          const float* __restrict__ V, float* __restrict__ Y) {
    const int n1 = m + 1, nRp = n1 * n1;
    const unsigned nk = (unsigned)nSp / 4, total = (unsigned)nrhs * nRp * nk;
    const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const int k = (int)(e % nk) * 4;
    const unsigned ri = e / nk;
    const int i = (int)(ri % (unsigned)nRp), r = (int)(ri / (unsigned)nRp);
    const int y = i / n1, x = i - y * n1;
    using P4 = Pack<float, 4>;
    auto at = [&](const float* p, int node) {
        return *reinterpret_cast<const P4*>(p + ((size_t)r * nRp + node) * nSp + k);
    };
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, a1[12], a2[12];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        *reinterpret_cast<P4*>(a1 + 4 * p) = *reinterpret_cast<const P4*>(A1 + 3 * k + 4 * p);
        *reinterpret_cast<P4*>(a2 + 4 * p) = *reinterpret_cast<const P4*>(A2 + 3 * k + 4 * p);
    }
    const float* Zr = Z + (size_t)r * 6 * m * m * nSp + 3 * k;
    auto cell = [&](int I, int J, int up, int loc, bool d1, bool d2) {
        const int j = 2 * (J * m + I) + up;
        const float* zp = Zr + (size_t)j * 3 * nSp;
        float z[12];
#pragma unroll
        for (int p = 0; p < 3; ++p)
            *reinterpret_cast<P4*>(z + 4 * p) = *reinterpret_cast<const P4*>(zp + 4 * p);
        const float* D = cell_D + 6 * (size_t)j + loc;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (d1)
                acc[w] = fmaf(D[0], a1[3 * w] * z[3 * w] + a1[3 * w + 1] * z[3 * w + 1] + a1[3 * w + 2] * z[3 * w + 2], acc[w]);
            if (d2)
                acc[w] = fmaf(D[3], a2[3 * w] * z[3 * w] + a2[3 * w + 1] * z[3 * w + 1] + a2[3 * w + 2] * z[3 * w + 2], acc[w]);
        }
    };
    const bool l = x > 0, rt = x < m, dn = y > 0, tp = y < m;
    if (rt && tp) {
        cell(x, y, 0, 0, true, false);
        cell(x, y, 1, 0, false, true);
    }
    if (l && tp) cell(x - 1, y, 0, 1, true, true);
    if (l && dn) {
        cell(x - 1, y - 1, 0, 2, false, true);
        cell(x - 1, y - 1, 1, 1, true, false);
    }
    if (rt && dn) cell(x, y - 1, 1, 2, true, true);
    const int nb[7] = {i, rt ? i + 1 : i, l ? i - 1 : i, tp ? i + n1 : i, dn ? i - n1 : i,
                       rt && tp ? i + n1 + 1 : i, l && dn ? i - n1 - 1 : i};
    const size_t sl = (size_t)7 * nRp;
    const bool edge = !(l && rt && dn && tp);
    float mass[4] = {0.f, 0.f, 0.f, 0.f}, bx[4] = {0.f, 0.f, 0.f, 0.f}, by[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int dir = 0; dir < 7; ++dir) {
        const size_t pe = (size_t)dir * nRp + i;
        const P4 u = at(X, nb[dir]);
        const float c = ell4[pe];
#pragma unroll
        for (int w = 0; w < 4; ++w) mass[w] = fmaf(c, u.v[w], mass[w]);
        if (edge) {
            const float cx = ell4[2 * sl + pe], cy = ell4[3 * sl + pe];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                bx[w] = fmaf(cx, u.v[w], bx[w]);
                by[w] = fmaf(cy, u.v[w], by[w]);
            }
        }
        if (V) {
            const P4 v = at(V, nb[dir]);
            const float cs = -ell4[sl + pe];
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[w] = fmaf(cs, v.v[w], acc[w]);
        }
    }
    P4 out;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        acc[w] = fmaf(mk[k + w], mass[w], acc[w]);
        if (edge) acc[w] = fmaf(omx[k + w], bx[w], fmaf(omy[k + w], by[w], acc[w]));
        out.v[w] = acc[w];
    }
    *reinterpret_cast<P4*>(Y + (size_t)ri * nSp + k) = out;
}

// ------------------------------------ vector passes of the mixed iteration
// The P_1 steps and the update of the outer iteration as few passes over the
// vectors: each kernel below reads what it needs once and writes every form
// (FP64, and the FP32 copy the inner operator takes) of its result, and sums
// what is needed of it; the separate copies, conversions, axpys and dots took
// 45 array passes and 30 launches an iteration more.  Bound by memory, and on
// small meshes by the launches.  Measured, whole solve with the iteration's
// one synchronisation in place of two: 128 x 128 / 512 triangles 76.2 -> 71.2
// ms, 77 x 77 with three right-hand sides 51.5 -> 41.9, 32 x 32 / 128
// triangles 3.5 -> 2.9.  W as above; one right-hand side per blockIdx.y, len
// values each.

// per-block sums of NS products into partial[(q nrhs + r) 1024 + block]
template <int NS>
__device__ void store_partials(double (&s)[NS], double* __restrict__ partial) {
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const double v = block_sum<256>(s[q]);
        if (threadIdx.x == 0)
            partial[((size_t)q * gridDim.y + blockIdx.y) * 1024 + blockIdx.x] = v;
    }
}

// P = Y, F = Y in FP32, partial sums of R.Y
template <int W>
__global__ void __launch_bounds__(256)
k_p1_start(const double* __restrict__ R, const double* __restrict__ Y, double* __restrict__ P,
           float* __restrict__ F, size_t len, double* __restrict__ partial) {
    const size_t o = (size_t)blockIdx.y * len;
    double s[1] = {0.0};
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * W; e < len; e += (size_t)gridDim.x * 256 * W) {
        const Pack<double, W> r = *reinterpret_cast<const Pack<double, W>*>(R + o + e);
        const Pack<double, W> y = *reinterpret_cast<const Pack<double, W>*>(Y + o + e);
        Pack<float, W> f;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            f.v[w] = (float)y.v[w];
            s[0] = fma(r.v[w], y.v[w], s[0]);
        }
        *reinterpret_cast<Pack<double, W>*>(P + o + e) = y;
        *reinterpret_cast<Pack<float, W>*>(F + o + e) = f;
    }
    store_partials<1>(s, partial);
}

// partial sums of P.F2 (F2 the FP32 result of an inner apply)
__global__ void __launch_bounds__(256)
k_p1_dot(const double* __restrict__ P, const float* __restrict__ F2, size_t len,
         double* __restrict__ partial) {
    const size_t o = (size_t)blockIdx.y * len;
    double s[1] = {0.0};
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * 2; e < len; e += (size_t)gridDim.x * 512) {
        const double2 p = *reinterpret_cast<const double2*>(P + o + e);
        const float2 f = *reinterpret_cast<const float2*>(F2 + o + e);
        s[0] = fma(p.x, (double)f.x, s[0]);
        s[0] = fma(p.y, (double)f.y, s[0]);
    }
    store_partials<1>(s, partial);
}

// One P_1 step: Z = alpha P (first) or Z += alpha P; R = B - alpha F2 unless
// it is the last one (B: the right-hand side on the first step, R itself
// after), which leaves F = Z in FP32 instead.
template <int W>
__global__ void __launch_bounds__(256)
k_p1_step(const double* __restrict__ alpha, int first, int last, const double* __restrict__ P,
          const float* __restrict__ F2, const double* B, double* Z, double* R,
          float* __restrict__ F, size_t len) {
    const size_t o = (size_t)blockIdx.y * len;
    const double a = alpha[blockIdx.y];
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * W; e < len; e += (size_t)gridDim.x * 256 * W) {
        const Pack<double, W> p = *reinterpret_cast<const Pack<double, W>*>(P + o + e);
        Pack<double, W> z, b;
        if (!last) b = *reinterpret_cast<const Pack<double, W>*>(B + o + e);   // before Z, which may be B
        if (!first) z = *reinterpret_cast<const Pack<double, W>*>(Z + o + e);
#pragma unroll
        for (int w = 0; w < W; ++w) z.v[w] = first ? a * p.v[w] : a * p.v[w] + z.v[w];
        *reinterpret_cast<Pack<double, W>*>(Z + o + e) = z;
        if (last) {
            Pack<float, W> f;
#pragma unroll
            for (int w = 0; w < W; ++w) f.v[w] = (float)z.v[w];
            *reinterpret_cast<Pack<float, W>*>(F + o + e) = f;
        } else {
            const Pack<float, W> g = *reinterpret_cast<const Pack<float, W>*>(F2 + o + e);
#pragma unroll
            for (int w = 0; w < W; ++w) b.v[w] = -a * (double)g.v[w] + b.v[w];
            *reinterpret_cast<Pack<double, W>*>(R + o + e) = b;
        }
    }
}

// P = Y + beta P, F = P in FP32
__global__ void __launch_bounds__(256)
k_p1_direction(const double* __restrict__ beta, const double* __restrict__ Y, double* __restrict__ P,
               float* __restrict__ F, size_t len) {
    const size_t o = (size_t)blockIdx.y * len;
    const double b = beta[blockIdx.y];
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * 2; e < len; e += (size_t)gridDim.x * 512) {
        const double2 y = *reinterpret_cast<const double2*>(Y + o + e);
        double2 p = *reinterpret_cast<const double2*>(P + o + e);
        p.x = y.x + b * p.x;
        p.y = y.y + b * p.y;
        *reinterpret_cast<double2*>(P + o + e) = p;
        *reinterpret_cast<float2*>(F + o + e) = make_float2((float)p.x, (float)p.y);
    }
}

__device__ void copy_state(const IterStateSrc& src, IterState* state) {
    state->status = *src.status;
    state->e0_flag = *src.e0_flag;
    state->tc_flag = *src.tc_flag;
}

__global__ void k_gather_state(IterStateSrc src, IterState* state) { copy_state(src, state); }

// Sum of a right-hand side's partials, and the scalar it gives: op 0: out =
// sum; 1: out = rho / sum (a step length); 2: out = sum / rho and rho = sum (a
// direction's factor).  blockIdx.x: sum q nrhs + r.  state set: the iteration's
// state beside the sums, so that one copy brings both to the host.
__global__ void __launch_bounds__(256)
k_sum_scalar(const double* __restrict__ partial, int nb, int op, double* rho,
             double* __restrict__ out, IterStateSrc src, IterState* state) {
    const int r = blockIdx.x;
    if (state && r == 0 && threadIdx.x == 32) copy_state(src, state);
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) s += partial[(size_t)r * 1024 + b];
    s = block_sum<256>(s);
    if (threadIdx.x != 0) return;
    if (op == 0) {
        out[r] = s;
    } else if (op == 1) {
        out[r] = s != 0.0 ? rho[r] / s : 0.0;
    } else {
        out[r] = rho[r] != 0.0 ? s / rho[r] : 0.0;
        rho[r] = s;
    }
}

// partial sums of R.R and, with D, D.R and D.Rp
template <bool ALL>
__global__ void __launch_bounds__(256)
k_residual_sums(const double* __restrict__ R, const double* __restrict__ D,
                const double* __restrict__ Rp, size_t len, double* __restrict__ partial) {
    const size_t o = (size_t)blockIdx.y * len;
    double s[ALL ? 3 : 1] = {};
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * 2; e < len; e += (size_t)gridDim.x * 512) {
        const double2 r = *reinterpret_cast<const double2*>(R + o + e);
        s[0] = fma(r.x, r.x, s[0]);
        s[0] = fma(r.y, r.y, s[0]);
        if constexpr (ALL) {
            const double2 d = *reinterpret_cast<const double2*>(D + o + e);
            const double2 p = *reinterpret_cast<const double2*>(Rp + o + e);
            s[1] = fma(d.x, r.x, s[1]);
            s[1] = fma(d.y, r.y, s[1]);
            s[2] = fma(d.x, p.x, s[2]);
            s[2] = fma(d.y, p.y, s[2]);
        }
    }
    store_partials<ALL ? 3 : 1>(s, partial);
}

// U -= S, D = -S
template <int W>
__global__ void __launch_bounds__(256)
k_update(const double* __restrict__ S, double* __restrict__ U, double* __restrict__ D, size_t n) {
    for (size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * W; e < n; e += (size_t)gridDim.x * 256 * W) {
        const Pack<double, W> v = *reinterpret_cast<const Pack<double, W>*>(S + e);
        Pack<double, W> u = *reinterpret_cast<const Pack<double, W>*>(U + e), d;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            u.v[w] -= v.v[w];
            d.v[w] = -v.v[w];
        }
        *reinterpret_cast<Pack<double, W>*>(U + e) = u;
        *reinterpret_cast<Pack<double, W>*>(D + e) = d;
    }
}

// whether pointers allow W = 2 accesses of T (null ones do)
template <typename T, typename... Ps>
bool paired(const Ps*... p) {
    return (((reinterpret_cast<uintptr_t>(p) & (2 * sizeof(T) - 1)) == 0) && ...);
}

}  // namespace

void apply_grad(cudaStream_t s, const DevSystem& d, const double* U, double* G, int nrhs,
                double sign) {
    // G is the library's own work array: aligned for four values
    const bool two = paired<double>(U);
    const size_t total = (size_t)nrhs * d.m * d.m * (d.nSp / (two ? 2 : 1));
    const unsigned blocks = (unsigned)((total + d.tpb_A - 1) / d.tpb_A);
    count_launches(1);
    if (two) k_grad<2><<<blocks, d.tpb_A, 0, s>>>(d.m, d.nSp, nrhs, sign, d.cell_D, U, G);
    else k_grad<1><<<blocks, d.tpb_A, 0, s>>>(d.m, d.nSp, nrhs, sign, d.cell_D, U, G);
}

void apply_even_grad(cudaStream_t s, const DevSystem& d, const double* G, const double* X,
                     const double* V, const double* Q, double* Y, int nrhs) {
    const bool two = paired<double>(X, V, Q, Y);
    const size_t total = (size_t)nrhs * d.nRp * (d.nSp / (two ? 2 : 1));
    const unsigned blocks = (unsigned)((total + d.tpb_even - 1) / d.tpb_even);
    count_launches(1);
    auto run = [&](auto kern) {
        kern<<<blocks, d.tpb_even, 0, s>>>(d.m, d.nSp, nrhs, d.cell_D, d.ell4, d.ang_m, d.ang_omx,
                                           d.ang_omy, G, X, V, Q, Y);
    };
    if (two) run(k_even_grad<2>);
    else run(k_even_grad<1>);
}

void apply_A_lo(cudaStream_t s, const DevSystem& d, const float* U, void* Z, bool bf16, int nrhs) {
    const size_t total = (size_t)nrhs * d.m * d.m * (d.nSp / 4);
    const unsigned blocks = (unsigned)((total + d.tpb_A_lo - 1) / d.tpb_A_lo);
    count_launches(1);
    if (bf16)
        k_odd_lo<__nv_bfloat16><<<blocks, d.tpb_A_lo, 0, s>>>(
            d.m, d.nSp, nrhs, d.lo.cell_D, d.lo.A1, d.lo.A2, U, static_cast<__nv_bfloat16*>(Z));
    else
        k_odd_lo<float><<<blocks, d.tpb_A_lo, 0, s>>>(
            d.m, d.nSp, nrhs, d.lo.cell_D, d.lo.A1, d.lo.A2, U, static_cast<float*>(Z));
}

void apply_even_lo(cudaStream_t s, const DevSystem& d, const float* Zp, const float* X,
                   const float* V, float* Y, int nrhs) {
    const size_t total = (size_t)nrhs * d.nRp * (d.nSp / 4);
    count_launches(1);
    k_even_lo<<<(unsigned)((total + d.tpb_even_lo - 1) / d.tpb_even_lo), d.tpb_even_lo, 0, s>>>(
        d.m, d.nSp, nrhs, d.lo.cell_D, d.lo.A1, d.lo.A2, d.lo.ell4, d.lo.m, d.lo.omx, d.lo.omy, Zp,
        X, V, Y);
}

static std::atomic<long long> g_launches{0};
void count_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches_total() { return g_launches.load(std::memory_order_relaxed); }

int device_sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

template <int EPI, typename... Args>
static int gemm_f64_epi(cudaStream_t s, int M, int N, Args... args) {
    // Products on the busiest SM, per step of K, and 8 % more for the operand
    // traffic of each smaller tile, so that calls with many tiles stay at 64 x
    // 64.  Both sides (us, 64 x 64, 32 x 64, 32 x 32, 16 x 32; taken: *):
    // 324 x 192 x 128 147, 77, 43, 26*; 512 x 192 x 128 147, 77, 43*, 41;
    // 2048 x 192 x 128 148, 145, 111*, 111; 6400 x 192 x 128 284*, 284, 284, 286;
    // 1152 x 512 x 768 789*, 773, 773, 778; 8192 x 768 x 512 5728*, 5462, 5349,
    // 5305 (the 8 % could be less: the operands come from L2 in time).
    const int tiles[4][2] = {{64, 64}, {32, 64}, {32, 32}, {16, 32}};
    const double sms = device_sm_count();
    int best = 0;
    double cost = 1e300;
    for (int t = 0; t < 4; ++t) {
        const double blocks = std::ceil((double)M / tiles[t][0]) * std::ceil((double)N / tiles[t][1]);
        const double c = std::ceil(blocks / sms) * tiles[t][0] * tiles[t][1] * (1.0 + 0.08 * t);
        if (c < cost) {
            cost = c;
            best = t;
        }
    }
    const long long grid = ((N + tiles[best][1] - 1LL) / tiles[best][1]) *
                           ((M + tiles[best][0] - 1LL) / tiles[best][0]);
    if (grid > 0x7fffffffLL) return fail(RTE_ERR_ARG, "FP64 GEMM: too many tiles for one launch");
    const unsigned g = (unsigned)grid;
    switch (best) {
        case 0: k_gemm_f64<EPI, 64, 64><<<g, 256, 0, s>>>(M, N, args...); break;
        case 1: k_gemm_f64<EPI, 32, 64><<<g, 256, 0, s>>>(M, N, args...); break;
        case 2: k_gemm_f64<EPI, 32, 32><<<g, 256, 0, s>>>(M, N, args...); break;
        default: k_gemm_f64<EPI, 16, 32><<<g, 256, 0, s>>>(M, N, args...); break;
    }
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

int gemm_f64(cudaStream_t s, int M, int N, int K, const double* A, int lda,
             const double* B, int ldb, double* C, int ldc, double alpha,
             double beta, int epi, const double* at, const double* as,
             const double* lam, int rows) {
    if (M <= 0 || N <= 0) return RTE_OK;
    count_launches(1);
    if (epi == 1) return gemm_f64_epi<1>(s, M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, at, as, lam, rows);
    if (epi == 2) return gemm_f64_epi<2>(s, M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, at, as, lam, rows);
    return gemm_f64_epi<0>(s, M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, at, as, lam, rows);
}

void apply_A(cudaStream_t s, const DevSystem& d, const double* U, double* Z, int nrhs) {
    const size_t total = (size_t)nrhs * d.nRm * d.nSp;
    count_launches(1);
    k_apply_A_s<double, double, double><<<grid_for(total, d.tpb_A), d.tpb_A, 0, s>>>(
        d.m, d.nSp, nrhs, d.cell_D, d.ang_A1, d.ang_A2, U, Z);
}

void apply_even(cudaStream_t s, const DevSystem& d, const double* Zp, const double* X,
                const double* V, double* Y, int nrhs, int flags) {
    const size_t total = (size_t)nrhs * d.nRp * d.nSp;
    count_launches(1);
    k_apply_even_s<double><<<grid_for(total, d.tpb_even), d.tpb_even, 0, s>>>(
        d.m, d.nSp, nrhs, flags, d.cell_D, d.ang_A1, d.ang_A2, d.ell4, d.ang_m, d.ang_omx,
        d.ang_omy, Zp, X, V, Y);
}

void mk_combine(cudaStream_t s, const DevSystem& d, const double* Z, const double* G,
                double* Y, int nrhs) {
    const size_t total = (size_t)nrhs * d.nRm * d.nSp;
    count_launches(1);
    k_mk_combine<<<grid_for(total), kThreads, 0, s>>>(d.nRm, d.nSp, nrhs, d.cell_at,
                                                      d.cell_as, d.ang_MSm, Z, G, Y);
}

void mk_minv_scale(cudaStream_t s, const DevSystem& d, const double* B, double* Y,
                   int nrhs) {
    const size_t total = (size_t)nrhs * d.nRm * d.nSp;
    count_launches(1);
    k_mk_minv_scale<<<grid_for(total), kThreads, 0, s>>>(d.nRm, d.nSp, nrhs, d.cell_at,
                                                         d.ang_MSm_inv, B, Y);
}

void inflow_source(cudaStream_t s, const DevSystem& d, const double* g, double* q, int nrhs) {
    const size_t total = (size_t)nrhs * 2 * (d.m + 1) * d.nSp;
    for (int f0 = 0; f0 < 4; f0 += 2)
        k_inflow<<<grid_for(total), kThreads, 0, s>>>(d.m, d.nSp, nrhs, f0, d.inflow_half,
                                                     d.ang_omx, d.ang_omy, g, q);
    count_launches(2);
}

void rhs_source(cudaStream_t s, const DevSystem& d, const double* qn, double* q, int nrhs) {
    const size_t total = (size_t)nrhs * d.nRp * d.nSp;
    count_launches(1);
    k_rhs_source<<<grid_for(total), kThreads, 0, s>>>(d.nRp, d.nSp, nrhs, d.nnz, d.st_ptr,
                                                      d.st_col, d.sval, d.ang_m, qn, q);
}

template <typename T>
void dot_impl(cudaStream_t s, const T* x, const T* y, size_t len, int nrhs, double* partial,
              double* out) {
    int nb = (int)std::min<size_t>(1024, std::max<size_t>(1, (len + 2047) / 2048));
    count_launches(2);
    k_dot_partial<T><<<dim3(nb, nrhs), 256, 0, s>>>(x, y, len, partial);
    k_dot_final<<<nrhs, 256, 0, s>>>(partial, nb, out);
}

void dot_per_rhs(cudaStream_t s, const double* x, const double* y, size_t len, int nrhs,
                 double* partial, double* out) {
    dot_impl(s, x, y, len, nrhs, partial, out);
}

void dot_per_rhs(cudaStream_t s, const float* x, const float* y, size_t len, int nrhs,
                 double* partial, double* out) {
    dot_impl(s, x, y, len, nrhs, partial, out);
}

void axpby_per_rhs(cudaStream_t s, const double* x, double* y, size_t len, int nrhs,
                   const double* a, double ca, const double* b, double cb) {
    count_launches(1);
    k_axpby<double><<<grid_for(len * nrhs), kThreads, 0, s>>>(x, y, len, nrhs, a, ca, b, cb);
}

void axpby_per_rhs(cudaStream_t s, const float* x, float* y, size_t len, int nrhs,
                   const double* a, double ca, const double* b, double cb) {
    count_launches(1);
    k_axpby<float><<<grid_for(len * nrhs), kThreads, 0, s>>>(x, y, len, nrhs, a, ca, b, cb);
}

// blocks of a vector pass over len values, and of its partial sums (<= 1024)
static int pass_blocks(size_t len) {
    return (int)std::min<size_t>(1024, std::max<size_t>(1, (len + 2047) / 2048));
}

void p1_start(cudaStream_t s, const double* R, const double* Y, double* P, float* F, size_t len,
              int nrhs, double* partial, double* rho) {
    const int nb = pass_blocks(len);
    count_launches(2);
    if (paired<double>(R))
        k_p1_start<2><<<dim3(nb, nrhs), 256, 0, s>>>(R, Y, P, F, len, partial);
    else
        k_p1_start<1><<<dim3(nb, nrhs), 256, 0, s>>>(R, Y, P, F, len, partial);
    k_sum_scalar<<<nrhs, 256, 0, s>>>(partial, nb, 0, nullptr, rho, {}, nullptr);
}

void p1_length(cudaStream_t s, const double* P, const float* F2, size_t len, int nrhs,
               double* partial, double* rho, double* alpha) {
    const int nb = pass_blocks(len);
    count_launches(2);
    k_p1_dot<<<dim3(nb, nrhs), 256, 0, s>>>(P, F2, len, partial);
    k_sum_scalar<<<nrhs, 256, 0, s>>>(partial, nb, 1, rho, alpha, {}, nullptr);
}

void p1_step(cudaStream_t s, const double* alpha, bool first, bool last, const double* P,
             const float* F2, const double* B, double* Z, double* R, float* F, size_t len, int nrhs) {
    const int nb = pass_blocks(len);
    count_launches(1);
    if (paired<double>(B, Z))
        k_p1_step<2><<<dim3(nb, nrhs), 256, 0, s>>>(alpha, first, last, P, F2, B, Z, R, F, len);
    else
        k_p1_step<1><<<dim3(nb, nrhs), 256, 0, s>>>(alpha, first, last, P, F2, B, Z, R, F, len);
}

void p1_direction(cudaStream_t s, const double* R, const double* Y, double* P, float* F, size_t len,
                  int nrhs, double* partial, double* rho, double* beta) {
    const int nb = pass_blocks(len);
    count_launches(3);
    k_dot_partial<double><<<dim3(nb, nrhs), 256, 0, s>>>(R, Y, len, partial);
    k_sum_scalar<<<nrhs, 256, 0, s>>>(partial, nb, 2, rho, beta, {}, nullptr);
    k_p1_direction<<<dim3(nb, nrhs), 256, 0, s>>>(beta, Y, P, F, len);
}

void residual_sums(cudaStream_t s, const double* R, const double* D, const double* Rp, size_t len,
                   int nrhs, double* partial, double* out, const IterStateSrc& src, IterState* state) {
    const int nb = pass_blocks(len);
    count_launches(2);
    if (D) k_residual_sums<true><<<dim3(nb, nrhs), 256, 0, s>>>(R, D, Rp, len, partial);
    else k_residual_sums<false><<<dim3(nb, nrhs), 256, 0, s>>>(R, D, Rp, len, partial);
    k_sum_scalar<<<(D ? 3 : 1) * nrhs, 256, 0, s>>>(partial, nb, 0, nullptr, out, src, state);
}

void gather_state(cudaStream_t s, const IterStateSrc& src, IterState* state) {
    count_launches(1);
    k_gather_state<<<1, 1, 0, s>>>(src, state);
}

void update_solution(cudaStream_t s, const double* S, double* U, double* D, size_t n) {
    const unsigned blocks = (unsigned)std::min<size_t>((n + 511) / 512, 65535);
    count_launches(1);
    if (paired<double>(U)) k_update<2><<<blocks, 256, 0, s>>>(S, U, D, n);
    else k_update<1><<<blocks, 256, 0, s>>>(S, U, D, n);
}

void fill_uniform(cudaStream_t s, double* x, size_t n, unsigned long long seed) {
    count_launches(1);
    k_fill_uniform<<<grid_for(n), kThreads, 0, s>>>(x, n, seed);
}


// ------------------------------------------ restriction and prolongation
// qc[row][j] = sum_k x[row][k] W[k][j], one warp per row: lanes stride over
// k with 16 partial sums each, reduced across the warp by halving exchanges
// (31 shuffles leave lane j holding the sum of column j mod 16).
// SUB: of x - sub instead.  (The variants of these two kernels are compiled
// apart, and their loops written apart below: with the choice made at run time
// the plain ones ran 1.0 to 1.15 and 1.05 to 1.9 times as long.)
template <typename T, bool SUB>
__global__ void __launch_bounds__(256) k_restrict(int rows, int nSp, int dP, const double* __restrict__ x,
                                                  const float* __restrict__ sub,
                                                  const T* __restrict__ W, double* __restrict__ qc) {
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= rows) return;
    T v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = T(0);
    const double* xr = x + (size_t)row * nSp;
    for (int k = lane; k < nSp; k += 32) {
        const T xv = (T)(SUB ? __ldg(xr + k) - (double)__ldg(sub + (size_t)row * nSp + k) : __ldg(xr + k));
        const T* w = W + (size_t)k * dP;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < dP) v[j] = fma(xv, __ldg(w + j), v[j]);
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], 16);
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const T send = up ? v[i] : v[i + o];
            const T keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    if (lane < dP) qc[(size_t)row * dP + lane] = (double)v[0];
}

// x[row][k] = beta x[row][k] + sum_j uc[row][j] WT[j][k], one warp per row.
// UPDATE (the outer iteration's): x stays, U -= that and D = -that, unless the
// coarse solve's status says that it gave up.
template <typename T, bool UPDATE>
__global__ void __launch_bounds__(256) k_prolong(int rows, int nSp, int dP, const double* __restrict__ uc,
                                                 const T* __restrict__ WT, double* __restrict__ x,
                                                 double beta, double* __restrict__ U,
                                                 double* __restrict__ D,
                                                 const SolveStatus* __restrict__ status) {
    if (UPDATE && status->timed_out) return;
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= rows) return;
    const T mine = lane < dP ? (T)uc[(size_t)row * dP + lane] : T(0);
    T u[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) u[j] = __shfl_sync(0xffffffffu, mine, j);
    double* xr = x + (size_t)row * nSp;
    auto value = [&](int k) {
        T acc = T(0);
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < dP) acc = fma(u[j], __ldg(WT + (size_t)j * nSp + k), acc);
        return (double)acc;
    };
    if constexpr (UPDATE) {
        // four trips' loads at once in FP32 (96 x 96 / 2048 triangles: 92 us,
        // 168 one by one); in FP64 that takes 88 registers and is slower (64 x
        // 64 / 512: 61 us against 47)
        double *Ur = U + (size_t)row * nSp, *Dr = D + (size_t)row * nSp;
#pragma unroll (sizeof(T) == 4 ? 4 : 1)
        for (int k = lane; k < nSp; k += 32) {
            const double x0 = beta == 0.0 ? 0.0 : xr[k], u0 = Ur[k], v = beta * x0 + value(k);
            Ur[k] = u0 - v;
            Dr[k] = -v;
        }
    } else {
        for (int k = lane; k < nSp; k += 32) {
            const double v = value(k);
            xr[k] = beta == 0.0 ? v : beta * xr[k] + v;
        }
    }
}

bool restrict_rows(cudaStream_t s, int rows, int nSp, int dP, const double* x, const double* W,
                   const float* W32, double* qc, const float* sub) {
    if (dP < 1 || dP > 16 || rows <= 0) return false;
    const unsigned blocks = (unsigned)(((size_t)rows * 32 + 255) / 256);
    count_launches(1);
    auto run = [&](auto kern, auto w) { kern<<<blocks, 256, 0, s>>>(rows, nSp, dP, x, sub, w, qc); };
    if (W32) sub ? run(k_restrict<float, true>, W32) : run(k_restrict<float, false>, W32);
    else sub ? run(k_restrict<double, true>, W) : run(k_restrict<double, false>, W);
    return true;
}

bool prolong_rows(cudaStream_t s, int rows, int nSp, int dP, const double* uc, const double* WT,
                  const float* WT32, double* x, double beta, double* U, double* D,
                  const SolveStatus* status) {
    if (dP < 1 || dP > 16 || rows <= 0) return false;
    const unsigned blocks = (unsigned)(((size_t)rows * 32 + 255) / 256);
    count_launches(1);
    auto run = [&](auto kern, auto w) {
        kern<<<blocks, 256, 0, s>>>(rows, nSp, dP, uc, w, x, beta, U, D, status);
    };
    if (WT32) U ? run(k_prolong<float, true>, WT32) : run(k_prolong<float, false>, WT32);
    else U ? run(k_prolong<double, true>, WT) : run(k_prolong<double, false>, WT);
    return true;
}

template <typename TI, typename TO>
static void convert_launch(cudaStream_t s, const TI* x, TO* y, size_t n) {
    count_launches(1);
    const bool four = n % 4 == 0 && reinterpret_cast<uintptr_t>(x) % (4 * sizeof(TI)) == 0 &&
                      reinterpret_cast<uintptr_t>(y) % (4 * sizeof(TO)) == 0;
    if (four) k_convert<TI, TO, 4><<<grid_for(n / 4), kThreads, 0, s>>>(x, y, n);
    else k_convert<TI, TO, 1><<<grid_for(n), kThreads, 0, s>>>(x, y, n);
}

void convert(cudaStream_t s, const double* x, float* y, size_t n) {
    convert_launch(s, x, y, n);
}

void convert(cudaStream_t s, const float* x, double* y, size_t n) {
    convert_launch(s, x, y, n);
}

void convert(cudaStream_t s, const float* x, __nv_bfloat16* y, size_t n) {
    convert_launch(s, x, y, n);
}

void convert(cudaStream_t s, const double* x, __nv_bfloat16* y, size_t n) {
    convert_launch(s, x, y, n);
}

void coarse_apply(cudaStream_t s, const DevSystem& d, const double* X, double* Y, int nrhs) {
    const size_t total = (size_t)nrhs * d.nRp * d.dP;
    count_launches(1);
    k_coarse_apply<<<grid_for(total), kThreads, 0, s>>>(d.nRp, d.dP, nrhs, d.st_ptr,
                                                        d.st_col, d.ec_val, X, Y);
}

void e0_coefficients(cudaStream_t s, int nRp, int nSp, const double* ell6, const double* e0s,
                     double* coef, float* coef_f) {
    const size_t n = (size_t)7 * nRp * nSp;
    k_e0_coef<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(nRp, nSp, ell6, e0s, coef, coef_f);
}

void assemble_scattering(cudaStream_t s, int n, double g, const QuadDev& q, double* Sp,
                         double* Sm) {
    const size_t pairs = (size_t)n * n;
    k_scatter_far<<<(unsigned)((pairs + 127) / 128), 128, 0, s>>>(
        n, g, q.far_pts, q.far_w, q.far_psi, q.qf, Sp, Sm);
    // near pairs: row index of every entry of the near list
    int npairs = 0;
    cudaMemcpyAsync(&npairs, q.near_ptr + n, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    int* rows = nullptr;
    if (npairs > 0 && cudaMallocAsync(&rows, sizeof(int) * npairs, s) == cudaSuccess) {
        k_near_rows<<<(n + 127) / 128, 128, 0, s>>>(n, q.near_ptr, rows);
        k_scatter_near<<<npairs, 256, 0, s>>>(n, g, q.near_pts, q.near_w, q.near_psi, q.qn,
                                              q.near_ptr, q.near_idx, rows, Sp, Sm);
        cudaFreeAsync(rows, s);
    }
    k_symmetrise<<<grid_for(pairs), kThreads, 0, s>>>(n, Sp);
    const size_t pm = (size_t)9 * n * n;
    k_symmetrise<<<grid_for(pm), kThreads, 0, s>>>(3 * n, Sm);
}

}  // namespace rte
