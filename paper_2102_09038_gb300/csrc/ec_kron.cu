// E_c^{-1} by one persistent multigrid-preconditioned CG on the Kronecker
// form of the levels, E_c = sum_q S_q (x) G_q (the default coarse route).
//
// What bounds it: latency.  A level holds at most a few megabytes (the CG's
// 250,000 unknowns at 128 x 128 take 1 MB in FP32, its stencils 6 MB, the
// inverse diagonal blocks 15 MB), all of it in L2, so a phase costs one round
// of L2 loads, a chain of small products and a grid-wide barrier, whatever
// its level; the coarsest level's dense inverse (75 MB for 289 nodes of 15)
// is the one phase bound by bandwidth.  Hence:
//  * few phases: a level's first smoothing step x = w D^{-1} b runs where its
//    b is made (the restriction, or the CG update on level 0), prolongation
//    runs inside the smoothing step after it, the direction update inside the
//    product E_c p, the r.z sum inside the last smoothing step: with two
//    sweeps 3 + 5 (L - 1) phases per CG iteration on L levels, against 26
//    for L = 4 before (now 18), and none for the V-cycle that no further
//    iteration would use;
//  * short phases: the loads of a phase are independent and issued first; the
//    d x d products take their operands as 16-byte broadcasts from shared
//    memory, four accumulators each, unrolled for d = 15, 6, 1, and a warp
//    skips the terms none of its nodes has (most nodes see one sigma class
//    and no boundary: 4 products of the 12); a lane group
//    (16 lanes, or 8 for d <= 8; lane a owns component a) takes two nodes at
//    a time where there are more nodes than groups, sharing the G_q it loads;
//  * a cheap barrier: one block of 512 threads per SM, at most.
// Vectors of the CG stay FP64, the V-cycle FP32.
//
// Measured, ms per solve (CG iterations): 128 x 128 / 512 triangles to 0.3
// (6): 2.65 -> 0.88; 32 x 32 / 128 triangles (3): 0.53 -> 0.16; 77 x 77, three right-hand
// sides (5): 4.85 -> 0.68; 32 x 32 in FP64 to 1e-12 (33): 4.92 -> 2.03.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "device.h"
#include "mg.h"
#include "mg_device.cuh"
#include "persist.cuh"
#include "rte_internal.h"

namespace rte {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kDenseRhs = 4;    // right-hand sides per pass over the dense inverse
constexpr int kPartRhs = 16;    // right-hand sides summed in shared memory first

struct KronArgs {
    int nRp, m, nrhs, maxit, nu, L, Q;
    int N, cld, rb;           // dense coarsest system, its row stride, rhs per pass
    double tol2;
    const double* ec;         // FP64 blocks [7][nRp][b][a] of the CG's products, or
                              // null: FP32 products on level 0
    const double* B;
    double *X, *R, *P0, *P1, *AP;   // P1: FP64 products only
    double* acc;              // rr, rz, pap: [3][3 slots][nrhs]
    double* bb;               // ||b||^2 [nrhs]
    GridBar* bar;
    SolveStatus* status;
    const float* cinv;
    const float* Gq;
    const MGDeviceLevel* lev;
};

// Per right-hand-side sums of a phase.  A lane adds its values; a lane group
// reduces them when its right-hand side changes and at the end, into its own
// row of shared memory (no atomics), and the block adds each sum once.
template <int GS>
struct PhaseSum {
    double v = 0.0;
    int r = -1;
    double* part;     // this group's row [nrhs], or null: straight to dst
    double* dst;
    int gl;
    unsigned mask;
    __device__ void flush() {
        if (r < 0) return;
#pragma unroll
        for (int o = GS / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
        if (gl == 0) {
            if (part) part[r] += v;
            else if (v != 0.0) atomicAdd(dst + r, v);
        }
        v = 0.0;
    }
    // every lane of the group calls this for the same rr
    __device__ void add(double x, int rr) {
        if (rr != r) {
            flush();
            r = rr;
        }
        v += x;
    }
};

// Shared memory of a block, in floats: the dense angular blocks (Ox, Oy and
// four per class) with a row pitch free of bank conflicts, then the lane
// groups' scratch (two nodes, four terms or seven FP64 directions), which the
// dense phase uses for b.
__host__ __device__ constexpr int group_lanes(int D) { return D <= 8 ? 8 : 16; }
__host__ __device__ constexpr int row_pitch(int D) { return group_lanes(D) == 16 ? 20 : 12; }
__host__ __device__ constexpr int dense_floats(int D, int NC) { return (2 + 4 * NC) * group_lanes(D) * row_pitch(D); }
__host__ __device__ constexpr int scratch_floats(int D) { return 16 * group_lanes(D); }

// All blocks of the (co-resident) grid meet here for the target / gridDim.x-th
// time.  One counter that only grows: an arrival is a fire-and-forget
// reduction and the wait one poll after the last of them, where a barrier
// with a generation word and a reset takes four dependent round trips to L2.
// Bounded like grid_sync (persist.cuh).
__device__ __forceinline__ bool meet(GridBar* gb, unsigned& target) {
    target += gridDim.x;
    __syncthreads();
    int bad = 0;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->count) : "memory");
        unsigned long long t0 = 0, lim = 0;
        unsigned spins = 0, now;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(&gb->count) : "memory");
            if ((int)(now - target) >= 0) break;
            if ((++spins & 255u) != 0) continue;
            if (*(volatile int*)&gb->err) {
                bad = 1;
                break;
            }
            if (t0 == 0) {
                t0 = global_ns();
                lim = gb->limit_ns ? gb->limit_ns : kWaitLimitNs;
            } else if (global_ns() - t0 > lim) {
                atomicExch(&gb->err, 1);
                bad = 1;
                break;
            }
        }
        if (blockIdx.x == 0 && gb->trace && gb->n < gb->cap) gb->trace[gb->n++] = global_ns();
    }
    return !__syncthreads_or(bad);
}

// D = d^+, NC = sigma classes.  The terms are q = 0: M_t (x) I, 1: M_s (x)
// -Lambda, 2 and 3: B_x (x) Ox, B_y (x) Oy, then four per class, and a level
// stores them node-major, four to a 16-byte word: word 0 of a direction the
// first four, word 1 + c class c.
template <int D, int NC>
__global__ void __launch_bounds__(kThreads, 1) k_ec_kron(KronArgs a) {
    constexpr int GS = group_lanes(D);       // lanes per item
    constexpr int PITCH = row_pitch(D);
    constexpr int QS = 1 + NC;               // 16-byte words per node and direction
    constexpr int GPB = kThreads / GS;       // groups per block
    extern __shared__ __align__(16) float sm[];
    float* sG = sm;                          // [2 + 4 NC][GS][PITCH]
    float* sU = sG + dense_floats(D, NC);    // group scratch, or the dense phase's b
    __shared__ MGDeviceLevel slev[kMaxMGLevels];
    // scalars of a phase per right-hand side (up to kPartRhs of them): step
    // length or direction factor, and whether it still iterates
    __shared__ double s_fac[kPartRhs];
    __shared__ int s_act[kPartRhs];
    unsigned target = 0;
    __shared__ double s_part[GPB * kPartRhs];
    const int lane = threadIdx.x & 31, gib = threadIdx.x / GS, gl = threadIdx.x % GS;
    // items go to the warps of all blocks in turn: few items then use every
    // SM (its FP64 units and load paths) instead of filling the first blocks
    const unsigned ng = gridDim.x * GPB,
                   gid = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * (32 / GS) + lane / GS;
    const unsigned gmask = (GS == 16 ? 0xffffu : 0xffu) << (lane / GS * GS);
    float* st = sU + gib * scratch_floats(D);   // this group's scratch
    const int nrhs = a.nrhs;
    const bool mine = gl < D;

    for (int t = threadIdx.x; t < dense_floats(D, NC); t += kThreads) {
        const int q = t / (GS * PITCH) + 2, row = t / PITCH % GS, c = t % PITCH;
        sG[t] = row < D && c < D ? __ldg(a.Gq + ((size_t)q * D + row) * D + c) : 0.f;
    }
    const float neglam = mine ? __ldg(a.Gq + ((size_t)D + gl) * D + gl) : 0.f;
    for (int t = threadIdx.x; t < a.L; t += kThreads) slev[t] = a.lev[t];
    for (int t = threadIdx.x; t < GPB * kPartRhs; t += kThreads) s_part[t] = 0.0;
    __syncthreads();

    PhaseSum<GS> sum;
    sum.part = nrhs <= kPartRhs ? s_part + gib * kPartRhs : nullptr;
    sum.gl = gl;
    sum.mask = gmask;
    auto sum_to = [&](double* dst) { sum.dst = dst; };
    auto sum_end = [&]() {
        sum.flush();
        sum.r = -1;
        if (!sum.part) return;
        __syncthreads();
        for (int r = threadIdx.x; r < nrhs; r += kThreads) {
            double v = 0.0;
            for (int g = 0; g < GPB; ++g) {
                v += s_part[g * kPartRhs + r];
                s_part[g * kPartRhs + r] = 0.0;
            }
            if (v != 0.0) atomicAdd(sum.dst + r, v);
        }
    };
    // f(N, first) for every N items first, first + ng, ... of `total`; all
    // lanes of a warp make the same trips (items past the end have e >= total)
    auto items = [&](unsigned total, auto&& f) {
        if (total > ng) {
            for (unsigned t = 0; t < total; t += 2 * ng) f(std::integral_constant<int, 2>{}, t + gid);
        } else {
            f(std::integral_constant<int, 1>{}, gid);
        }
    };
    auto split_item = [&](unsigned e, int nn, int& r, int& i) {
        r = nrhs == 1 ? 0 : (int)(e / (unsigned)nn);
        i = nrhs == 1 ? (int)e : (int)(e % (unsigned)nn);
    };
    // Neighbours of node i of an m-mesh; one outside takes the node itself
    // (its coefficient is zero).
    auto neighbours = [&](int i, int m, int (&j)[7]) {
        const int w = m + 1, y = i / w, x = i - y * w;
        const bool l = x > 0, r = x < m, d = y > 0, u = y < m;
        j[0] = i;
        j[1] = r ? i + 1 : i;
        j[2] = l ? i - 1 : i;
        j[3] = u ? i + w : i;
        j[4] = d ? i - w : i;
        j[5] = r && u ? i + w + 1 : i;
        j[6] = l && d ? i - w - 1 : i;
        return (y << 16) | x;
    };
    // y[n] += row gl of sum_k G_k t_k[n] over K dense blocks from `first` on
    auto blocks = [&](auto nc, auto kc, int first,
                      const float (&t)[decltype(nc)::value][decltype(kc)::value],
                      float (&y)[decltype(nc)::value]) {
        constexpr int N = decltype(nc)::value, K = decltype(kc)::value;
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
            for (int k = 0; k < K; ++k) st[(n * K + k) * GS + gl] = t[n][k];
        __syncwarp();
        float c[N][4];
#pragma unroll
        for (int n = 0; n < N; ++n) c[n][0] = c[n][1] = c[n][2] = c[n][3] = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int b = 0; b < (D + 3) / 4; ++b) {
                const float4 g =
                    *reinterpret_cast<const float4*>(sG + ((first + k) * GS + gl) * PITCH + 4 * b);
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const float4 v = *reinterpret_cast<const float4*>(st + (n * K + k) * GS + 4 * b);
                    c[n][0] = fmaf(g.x, v.x, c[n][0]);
                    c[n][1] = fmaf(g.y, v.y, c[n][1]);
                    c[n][2] = fmaf(g.z, v.z, c[n][2]);
                    c[n][3] = fmaf(g.w, v.w, c[n][3]);
                }
            }
        __syncwarp();
#pragma unroll
        for (int n = 0; n < N; ++n) y[n] += (c[n][0] + c[n][1]) + (c[n][2] + c[n][3]);
    };
    // y[n] = row gl of (sum_q S_q (x) G_q) x for N nodes, from component gl
    // of x at the seven neighbours: t_q = sum_dir S_q x, then y = sum_q G_q t_q.
    // The first two terms are diagonal in the components; the boundary terms
    // and a class's terms are skipped where no node of the warp has them
    // (mask: bit c for class c, bit 7 for the boundary).
    auto kron = [&](auto nc, const float (&xv)[decltype(nc)::value][7],
                    const float4* const (&sk)[decltype(nc)::value],
                    const unsigned (&mask)[decltype(nc)::value],
                    float (&y)[decltype(nc)::value]) {
        constexpr int N = decltype(nc)::value;
        unsigned any = mask[0];
        if constexpr (N == 2) any |= mask[1];
        any = __reduce_or_sync(0xffffffffu, any);
        float tb[N][2];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            float t0 = 0.f, t1 = 0.f;
            tb[n][0] = tb[n][1] = 0.f;
#pragma unroll
            for (int dir = 0; dir < 7; ++dir) {
                const float4 s4 = __ldg(sk[n] + dir * QS);
                t0 = fmaf(s4.x, xv[n][dir], t0);
                t1 = fmaf(s4.y, xv[n][dir], t1);
                tb[n][0] = fmaf(s4.z, xv[n][dir], tb[n][0]);
                tb[n][1] = fmaf(s4.w, xv[n][dir], tb[n][1]);
            }
            y[n] = fmaf(neglam, t1, t0);
        }
        if (any & 0x80u) blocks(nc, std::integral_constant<int, 2>{}, 0, tb, y);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (!(any >> c & 1u)) continue;
            float t[N][4];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                t[n][0] = t[n][1] = t[n][2] = t[n][3] = 0.f;
#pragma unroll
                for (int dir = 0; dir < 7; ++dir) {
                    const float4 s4 = __ldg(sk[n] + dir * QS + 1 + c);
                    t[n][0] = fmaf(s4.x, xv[n][dir], t[n][0]);
                    t[n][1] = fmaf(s4.y, xv[n][dir], t[n][1]);
                    t[n][2] = fmaf(s4.z, xv[n][dir], t[n][2]);
                    t[n][3] = fmaf(s4.w, xv[n][dir], t[n][3]);
                }
            }
            blocks(nc, std::integral_constant<int, 4>{}, 2 + 4 * c, t, y);
        }
    };
    // row gl of the inverse diagonal block of a node (0 for idle lanes)
    auto load_dinv = [&](const float* dinv, int i, bool act, float (&dr)[D]) {
#pragma unroll
        for (int b = 0; b < D; ++b)
            dr[b] = act ? __ldg(dinv + (unsigned)i * (D * D) + b * D + gl) : 0.f;
    };
    // dx[n] = row gl of D^{-1} v, v[n] held by component
    auto dmul = [&](auto nc, const float (&dr)[decltype(nc)::value][D],
                    const float (&v)[decltype(nc)::value], float (&dx)[decltype(nc)::value]) {
        constexpr int N = decltype(nc)::value;
#pragma unroll
        for (int n = 0; n < N; ++n) st[n * GS + gl] = v[n];
        __syncwarp();
#pragma unroll
        for (int n = 0; n < N; ++n) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int b = 0; b < D; b += 4) {
                const float4 u = *reinterpret_cast<const float4*>(st + n * GS + b);
                c[0] = fmaf(dr[n][b], u.x, c[0]);
                if (b + 1 < D) c[1] = fmaf(dr[n][b + 1 < D ? b + 1 : 0], u.y, c[1]);
                if (b + 2 < D) c[2] = fmaf(dr[n][b + 2 < D ? b + 2 : 0], u.z, c[2]);
                if (b + 3 < D) c[3] = fmaf(dr[n][b + 3 < D ? b + 3 : 0], u.w, c[3]);
            }
            dx[n] = (c[0] + c[1]) + (c[2] + c[3]);
        }
        __syncwarp();
    };
    // xo = x + w D^{-1} (b - A x) on level l, where x has the prolongation of
    // xc (level l + 1) added first when xc is set; res: xo = b - A x instead;
    // rz: add r.xo to the phase sum (level 0)
    auto smooth = [&](int l, const float* x, float* xo, const float* xc, bool res, bool rz) {
        const MGDeviceLevel& Lv = slev[l];
        const int nn = Lv.n, mm = Lv.m, ncn = xc ? slev[l + 1].n : 0;
        const unsigned total = (unsigned)nrhs * nn;
        items(total, [&](auto nc, unsigned first) {
            constexpr int N = decltype(nc)::value;
            float xv[N][7], bv[N], y[N], dr[N][D];
            const float4* sk[N];
            bool act[N];
            int r[N], i[N];
            unsigned e[N], mask[N];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const bool ok = first + n * ng < total;
                e[n] = ok ? first + n * ng : 0u;
                act[n] = ok && mine;
                split_item(e[n], nn, r[n], i[n]);
                const float* xr = x + (unsigned)r[n] * nn * D + gl;
                int j[7];
                const int yx = neighbours(i[n], mm, j);
                mask[n] = act[n] ? __ldg(Lv.kmask + i[n]) : 0u;
#pragma unroll
                for (int dir = 0; dir < 7; ++dir) xv[n][dir] = act[n] ? ldg2(xr + j[dir] * D) : 0.f;
                if (xc) {
                    // the coarse mesh is the floor(m / 2)-mesh; for odd m the
                    // last column and row repeat the ones before them
                    const int mc = mm / 2, top = 2 * mc, cw = mc + 1;
                    const float* cr = xc + (unsigned)r[n] * ncn * D + gl;
                    constexpr int dx[7] = {0, 1, -1, 0, 0, 1, -1}, dy[7] = {0, 0, 0, 1, -1, 1, -1};
#pragma unroll
                    for (int dir = 0; dir < 7; ++dir) {
                        const bool in = dir == 0 || j[dir] != i[n];
                        const int X = min((yx & 0xffff) + (in ? dx[dir] : 0), top);
                        const int Y = min((yx >> 16) + (in ? dy[dir] : 0), top);
                        const int c0 = (Y >> 1) * cw + (X >> 1);
                        const int c1 = c0 + (X & 1) + (Y & 1) * cw;
                        const float w1 = c1 == c0 ? 0.f : 0.5f, w0 = 1.f - w1;
                        if (act[n]) xv[n][dir] += w0 * ldg2(cr + c0 * D) + w1 * ldg2(cr + c1 * D);
                    }
                }
                bv[n] = act[n] ? ldg2(Lv.B + e[n] * D + gl) : 0.f;
                sk[n] = reinterpret_cast<const float4*>(Lv.sv) + (unsigned)i[n] * 7 * QS;
                if (N == 1 && !res) load_dinv(Lv.dinv, i[n], act[n], dr[n]);
            }
            kron(nc, xv, sk, mask, y);
            if (res) {
#pragma unroll
                for (int n = 0; n < N; ++n)
                    if (act[n]) xo[e[n] * D + gl] = bv[n] - y[n];
                return;
            }
            float v[N], dx[N];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                // (two nodes' blocks do not fit the registers any earlier)
                if (N > 1) load_dinv(Lv.dinv, i[n], act[n], dr[n]);
                v[n] = act[n] ? bv[n] - y[n] : 0.f;
            }
            dmul(nc, dr, v, dx);
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const float xn = xv[n][0] + kOmega * dx[n];
                if (act[n]) xo[e[n] * D + gl] = xn;
                if (rz && first + n * ng < total)
                    sum.add(act[n] ? ldg2(a.R + e[n] * D + gl) * (double)xn : 0.0, r[n]);
            }
        });
    };
    // b of level l + 1 from the residual t of level l, and the first
    // smoothing step there (unless that level is solved densely)
    auto restrict_to = [&](int l, const float* t) {
        const MGDeviceLevel& Cv = slev[l + 1];
        const int nn = Cv.n, nf = slev[l].n, wid = Cv.rwid;
        const bool first_step = l + 2 < a.L;
        const unsigned total = (unsigned)nrhs * nn;
        items(total, [&](auto nc, unsigned first) {
            constexpr int N = decltype(nc)::value;
            float v[N], dx[N], dr[N][D];
            unsigned e[N];
            bool act[N];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const bool ok = first + n * ng < total;
                e[n] = ok ? first + n * ng : 0u;
                act[n] = ok && mine;
                int r, i;
                split_item(e[n], nn, r, i);
                v[n] = 0.f;
                const float* tr = t + (unsigned)r * nf * D + gl;
                if (act[n]) {
#pragma unroll 8
                    for (int q = 0; q < wid; ++q) {
                        float w;
                        const int f = restrict_src(Cv, i, q, w);
                        v[n] += w * ldg2(tr + f * D);
                    }
                    Cv.B[e[n] * D + gl] = v[n];
                }
                if (first_step) load_dinv(Cv.dinv, i, act[n], dr[n]);
            }
            if (!first_step) return;
            dmul(nc, dr, v, dx);
#pragma unroll
            for (int n = 0; n < N; ++n)
                if (act[n]) Cv.X[e[n] * D + gl] = kOmega * dx[n];
        });
    };
    // x = A^{-1} b on the coarsest level: two rows of the inverse per warp at
    // a time, b of up to rb right-hand sides in shared memory
    auto dense = [&](bool rz) {
        const MGDeviceLevel& Lv = slev[a.L - 1];
        const int N = a.N, ld4 = a.cld / 4;
        const int nw = gridDim.x * kWarps, gw = blockIdx.x * kWarps + (threadIdx.x >> 5);
        auto rows = [&](auto rc, int r0, int nr) {
            constexpr int RB = decltype(rc)::value;
            const float4* sb = reinterpret_cast<const float4*>(sU);
            for (int q = gw; q < N; q += 2 * nw) {
                const int q2 = q + nw < N ? q + nw : q;
                const float4* m0 = reinterpret_cast<const float4*>(a.cinv) + (size_t)q * ld4;
                const float4* m1 = reinterpret_cast<const float4*>(a.cinv) + (size_t)q2 * ld4;
                float c0[RB], c1[RB];
#pragma unroll
                for (int r = 0; r < RB; ++r) c0[r] = c1[r] = 0.f;
#pragma unroll (RB == 1 ? 8 : 4)
                for (int j = lane; j < ld4; j += 32) {
                    const float4 u = __ldcg(m0 + j), w = __ldcg(m1 + j);
#pragma unroll
                    for (int r = 0; r < RB; ++r)
                        if (r < nr) {
                            const float4 v = sb[r * ld4 + j];
                            c0[r] = fmaf(u.x, v.x, fmaf(u.y, v.y, fmaf(u.z, v.z, fmaf(u.w, v.w, c0[r]))));
                            c1[r] = fmaf(w.x, v.x, fmaf(w.y, v.y, fmaf(w.z, v.z, fmaf(w.w, v.w, c1[r]))));
                        }
                }
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    if (r >= nr) break;
                    for (int o = 16; o > 0; o >>= 1) {
                        c0[r] += __shfl_xor_sync(0xffffffffu, c0[r], o);
                        c1[r] += __shfl_xor_sync(0xffffffffu, c1[r], o);
                    }
                    const size_t o0 = (size_t)(r0 + r) * N + q, o1 = (size_t)(r0 + r) * N + q2;
                    if (lane == 0) {
                        Lv.X[o0] = c0[r];
                        if (q2 != q) Lv.X[o1] = c1[r];
                    }
                    if (rz) {   // a single level: this is z on level 0
                        double v = 0.0;
                        if (lane == 0) {
                            v = ldg2(a.R + o0) * (double)c0[r];
                            if (q2 != q) v += ldg2(a.R + o1) * (double)c1[r];
                        }
                        sum.add(v, r0 + r);
                    }
                }
            }
        };
        for (int r0 = 0; r0 < nrhs; r0 += a.rb) {
            const int nr = min(a.rb, nrhs - r0);
            __syncthreads();
            for (int t = threadIdx.x; t < nr * a.cld; t += kThreads) {
                const int r = t / a.cld, c = t % a.cld;
                sU[t] = c < N ? ldg2(Lv.B + (size_t)(r0 + r) * N + c) : 0.f;
            }
            __syncthreads();
            // one right-hand side (the usual solve) keeps twice as many
            // loads of the matrix in flight
            if (nr == 1) rows(std::integral_constant<int, 1>{}, r0, nr);
            else rows(std::integral_constant<int, kDenseRhs>{}, r0, nr);
        }
    };
    auto buf = [&](int l, unsigned cur) { return (cur >> l & 1u) ? slev[l].Xt : slev[l].X; };
    // z = one V-cycle for b = B0 (level 0's first step done), rz_slot += r.z
    auto vcycle = [&](float*& z, double* rz_slot) -> bool {
        unsigned cur = 0;   // bit l: level l's iterate is in Xt
        sum_to(rz_slot);
        for (int l = 0; l + 1 < a.L; ++l) {
            // nu - 1 more smoothing steps, then the residual
            for (int k = 1; k <= a.nu; ++k) {
                smooth(l, buf(l, cur), buf(l, cur ^ 1u << l), nullptr, k == a.nu, false);
                if (k < a.nu) cur ^= 1u << l;
                if (!meet(a.bar, target)) return false;
            }
            restrict_to(l, buf(l, cur ^ 1u << l));
            if (!meet(a.bar, target)) return false;
        }
        dense(a.L == 1);
        if (a.L == 1) sum_end();
        if (!meet(a.bar, target)) return false;
        for (int l = a.L - 2; l >= 0; --l)
            for (int k = 0; k < a.nu; ++k) {
                const bool rz = l == 0 && k == a.nu - 1;
                smooth(l, buf(l, cur), buf(l, cur ^ 1u << l), k == 0 ? buf(l + 1, cur) : nullptr,
                       false, rz);
                cur ^= 1u << l;
                if (rz) sum_end();
                if (!meet(a.bar, target)) return false;
            }
        z = buf(0, cur);
        return true;
    };
    const unsigned total0 = (unsigned)nrhs * a.nRp;
    auto rr = [&](int k) { return k == 0 ? a.bb : a.acc + (size_t)(k % 3) * nrhs; };
    auto rz = [&](int k) { return a.acc + (size_t)(3 + k % 3) * nrhs; };
    auto pap = [&](int k) { return a.acc + (size_t)(6 + k % 3) * nrhs; };
    // level 0's first smoothing step from b (one value per lane and item)
    auto start0 = [&](auto nc, const unsigned (&e)[decltype(nc)::value],
                      const bool (&act)[decltype(nc)::value],
                      const int (&i)[decltype(nc)::value],
                      const float (&b)[decltype(nc)::value]) {
        constexpr int N = decltype(nc)::value;
        const MGDeviceLevel& Lv = slev[0];
        float dr[N][D], dx[N];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            if (act[n]) Lv.B[e[n] * D + gl] = b[n];
            if (a.L > 1) load_dinv(Lv.dinv, i[n], act[n], dr[n]);
        }
        if (a.L == 1) return;
        dmul(nc, dr, b, dx);
#pragma unroll
        for (int n = 0; n < N; ++n)
            if (act[n]) Lv.X[e[n] * D + gl] = kOmega * dx[n];
    };
    sum_to(a.bb);
    items(total0, [&](auto nc, unsigned first) {
        constexpr int N = decltype(nc)::value;
        unsigned e[N];
        bool act[N];
        int i[N];
        float b[N];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const bool ok = first + n * ng < total0;
            e[n] = ok ? first + n * ng : 0u;
            act[n] = ok && mine;
            int r;
            split_item(e[n], a.nRp, r, i[n]);
            const unsigned o = e[n] * D + gl;
            const double bd = act[n] ? a.B[o] : 0.0;
            if (act[n]) {
                a.X[o] = 0.0;
                a.R[o] = bd;
            }
            if (ok) sum.add(bd * bd, r);
            b[n] = (float)bd;
        }
        start0(nc, e, act, i, b);
    });
    sum_end();
    if (!meet(a.bar, target)) return;
    float* z = nullptr;
    int it = 0;
    // The phase's scalars: one division per right-hand side and block, not
    // one per lane (an FP64 division costs a lane group hundreds of cycles).
    // More right-hand sides than the table holds compute their own.
    auto live = [&](int r) { return ldg2(rr(it) + r) > a.tol2 * ldg2(a.bb + r); };
    auto scalars = [&](auto&& f) {
        if (nrhs > kPartRhs) return;
        if (threadIdx.x < nrhs) {
            s_fac[threadIdx.x] = f(threadIdx.x);
            s_act[threadIdx.x] = live(threadIdx.x);
        }
        __syncthreads();
    };
    auto active = [&](int r) { return nrhs > kPartRhs ? live(r) : s_act[r] != 0; };
    auto factor = [&](int r, auto&& f) { return nrhs > kPartRhs ? f(r) : s_fac[r]; };
    bool stop = false;
    double *P = a.P0, *Pn = a.P1;
    for (;;) {
        if (!vcycle(z, rz(it))) return;
        // p = z + beta p and AP = E_c p, pap += p.AP; right-hand sides that
        // are done stay as they are
        if (blockIdx.x == 0)
            for (int c = threadIdx.x; c < nrhs; c += kThreads) rr(it + 1)[c] = rz(it + 1)[c] = 0.0;
        sum_to(pap(it));
        auto beta_of = [&](int r) {
            const double o = it > 0 ? ldg2(rz(it - 1) + r) : 0.0;
            return o != 0.0 ? ldg2(rz(it) + r) / o : 0.0;
        };
        scalars(beta_of);
        if (!a.ec) {
            // FP32 products: E_c z from the exact FP32 z, and E_c p by the
            // recurrence of p itself
            items(total0, [&](auto nc, unsigned first) {
                constexpr int N = decltype(nc)::value;
                float xv[N][7], y[N];
                const float4* sk[N];
                int r[N], i[N];
                bool act[N];
                unsigned e[N], mask[N];
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const bool ok = first + n * ng < total0;
                    e[n] = ok ? first + n * ng : 0u;
                    split_item(e[n], a.nRp, r[n], i[n]);
                    act[n] = ok && mine && active(r[n]);
                    const float* zr = z + (unsigned)r[n] * a.nRp * D + gl;
                    int j[7];
                    neighbours(i[n], a.m, j);
                    mask[n] = act[n] ? __ldg(slev[0].kmask + i[n]) : 0u;
#pragma unroll
                    for (int dir = 0; dir < 7; ++dir) xv[n][dir] = act[n] ? ldg2(zr + j[dir] * D) : 0.f;
                    sk[n] = reinterpret_cast<const float4*>(slev[0].sv) + (unsigned)i[n] * 7 * QS;
                }
                kron(nc, xv, sk, mask, y);
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    double s = 0.0;
                    if (act[n]) {
                        const unsigned o = e[n] * D + gl;
                        double p = (double)xv[n][0], ap = (double)y[n];
                        if (it > 0) {
                            const double beta = factor(r[n], beta_of);
                            p = fma(beta, P[o], p);
                            ap = fma(beta, a.AP[o], ap);
                        }
                        P[o] = p;
                        a.AP[o] = ap;
                        s = p * ap;
                    }
                    if (first + n * ng < total0) sum.add(s, r[n]);
                }
            });
        } else {
            // FP64 products of p itself, formed at the node and its
            // neighbours, stored at the node
            double* sd = reinterpret_cast<double*>(st);   // [7][GS]
            for (unsigned t = 0; t < total0; t += ng) {
                const bool ok = t + gid < total0;
                const unsigned e = ok ? t + gid : 0u;
                double pv[7], y[7];
                int r, i, j[7];
                split_item(e, a.nRp, r, i);
                const bool act = ok && mine && active(r);
                const double beta = act ? factor(r, beta_of) : 0.0;
                const float* zr = z + (unsigned)r * a.nRp * D + gl;
                const double* pr = P + (unsigned)r * a.nRp * D + gl;
                neighbours(i, a.m, j);
#pragma unroll
                for (int dir = 0; dir < 7; ++dir) {
                    pv[dir] = 0.0;
                    if (act) {
                        pv[dir] = (double)ldg2(zr + j[dir] * D);
                        if (it > 0) pv[dir] = fma(beta, ldg2(pr + j[dir] * D), pv[dir]);
                    }
                    sd[dir * GS + gl] = pv[dir];
                    y[dir] = 0.0;
                }
                if (act) Pn[e * D + gl] = pv[0];
                __syncwarp();
                if (act) {
#pragma unroll
                    for (int dir = 0; dir < 7; ++dir) {
                        const double* blk = a.ec + ((size_t)dir * a.nRp + i) * D * D + gl;
#pragma unroll
                        for (int b = 0; b < D; ++b)
                            y[dir] = fma(__ldg(blk + b * D), sd[dir * GS + b], y[dir]);
                    }
                }
                __syncwarp();
                const double s = ((y[0] + y[1]) + (y[2] + y[3])) + ((y[4] + y[5]) + y[6]);
                if (act) a.AP[e * D + gl] = s;
                if (ok) sum.add(act ? s * pv[0] : 0.0, r);
            }
            double* t = P;   // P: the direction of this iteration
            P = Pn;
            Pn = t;
        }
        sum_end();
        if (!meet(a.bar, target)) return;
        // x += alpha p, r -= alpha AP, and level 0's b and first step
        if (blockIdx.x == 0)
            for (int c = threadIdx.x; c < nrhs; c += kThreads) pap(it + 1)[c] = 0.0;
        sum_to(rr(it + 1));
        auto alpha_of = [&](int r) {
            const double q = ldg2(pap(it) + r);
            return q != 0.0 ? ldg2(rz(it) + r) / q : 0.0;
        };
        scalars(alpha_of);
        items(total0, [&](auto nc, unsigned first) {
            constexpr int N = decltype(nc)::value;
            unsigned e[N];
            bool act[N];
            int i[N];
            float b[N];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const bool ok = first + n * ng < total0;
                e[n] = ok ? first + n * ng : 0u;
                act[n] = ok && mine;
                int r;
                split_item(e[n], a.nRp, r, i[n]);
                const unsigned o = e[n] * D + gl;
                b[n] = 0.f;
                double s = 0.0;
                if (active(r)) {
                    if (act[n]) {
                        const double alpha = factor(r, alpha_of);
                        a.X[o] += alpha * P[o];
                        const double rv = a.R[o] - alpha * a.AP[o];
                        a.R[o] = rv;
                        b[n] = (float)rv;
                        s = rv * rv;
                    }
                } else if (i[n] == 0 && gl == 0) {
                    s = ldg2(rr(it) + r);   // done: its residual is carried along
                }
                if (ok) sum.add(s, r);
            }
            start0(nc, e, act, i, b);
        });
        sum_end();
        if (!meet(a.bar, target)) return;
        ++it;
        int more = 0;
        for (int c = threadIdx.x; c < nrhs; c += kThreads)
            if (ldg2(rr(it) + c) > a.tol2 * ldg2(a.bb + c)) more = 1;
        stop = !__syncthreads_or(more);
        if (stop || it >= a.maxit) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.status->iterations = it;
        a.status->converged = stop;
        a.status->timed_out = 0;
    }
}

template <int D, int NC>
int launch(cudaStream_t s, const KronArgs& a) {
    constexpr int GS = group_lanes(D), kScratch = kThreads / GS * scratch_floats(D);
    const size_t sm = (dense_floats(D, NC) + std::max((size_t)kScratch, (size_t)a.rb * a.cld)) * sizeof(float);
    const void* fn = (const void*)k_ec_kron<D, NC>;
    // the most any mesh needs, whatever the call: a call never shrinks the
    // attribute under another's launch
    constexpr int kMaxSm =
        (dense_floats(D, NC) + std::max(kScratch, kDenseRhs * (kDenseCoarseNodes * D + 4))) * 4;
    static_assert(kMaxSm <= 200 * 1024, "shared memory of the coarse solve");
    RTE_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSm));
    // a block per SM at most (the barrier needs them resident); fewer when
    // neither the nodes nor the dense rows (two per warp) fill them
    const size_t groups = (size_t)a.nrhs * a.nRp, per = kThreads / GS;
    const size_t want = std::max((groups + per - 1) / per, ((size_t)a.N + 2 * kWarps - 1) / (2 * kWarps));
    const int grid = (int)std::min<size_t>(std::max<size_t>(want, 1), device_sm_count());
    KronArgs args = a;
    void* p[] = {&args};
    RTE_CUDA_TRY(cudaLaunchCooperativeKernel(fn, grid, kThreads, p, sm, s));
    count_launches(1);
    return RTE_OK;
}

template <int D>
int launch_classes(cudaStream_t s, const KronArgs& a) {
    switch (a.Q) {
        case 8: return launch<D, 1>(s, a);
        case 12: return launch<D, 2>(s, a);
        default: return launch<D, 3>(s, a);
    }
}

}  // namespace

bool ec_kron_takes(const DevSystem& d, int nrhs) {
    const MGDevice& g = d.ecmg;
    const bool direct = d.eclu32 != nullptr || d.eclu64 != nullptr;
    return !direct && (g.Q == 8 || g.Q == 12 || g.Q == 16) && g.dense && g.L >= 1 && g.lev[0].n == d.nRp &&
           (d.dP == 1 || d.dP == 6 || d.dP == 15) &&
           // 32-bit offsets into the vectors, the blocks and the stencils
           (double)nrhs * d.nRp * d.dP < 1e9 && 225.0 * d.nRp < 2e9;
}

int ec_kron_cg(cudaStream_t s, const DevSystem& d, const double* B, double* X, int nrhs,
               double tol, int maxit, void* work, SolveStatus* status_dev, bool f32_products,
               unsigned long long limit_ns, unsigned long long* trace, int cap) {
    const MGDevice& g = d.ecmg;
    const size_t n = (size_t)nrhs * d.nRp * d.dP;
    char* p = static_cast<char*>(work);
    KronArgs a{};
    a.R = carve<double>(p, n);
    a.P0 = carve<double>(p, n);
    a.P1 = carve<double>(p, n);
    a.AP = carve<double>(p, n);
    char* zero = p;
    a.acc = carve<double>(p, 9 * (size_t)nrhs);
    a.bb = carve<double>(p, nrhs);
    a.bar = carve<GridBar>(p, 1);
    RTE_CUDA_TRY(cudaMemsetAsync(zero, 0, (size_t)(p - zero), s));
    if (limit_ns || trace) {   // otherwise the zeroed barrier has its defaults
        GridBar h{};
        h.trace = trace;
        h.cap = cap;
        h.limit_ns = limit_ns;
        RTE_CUDA_TRY(cudaMemcpyAsync(a.bar, &h, sizeof(GridBar), cudaMemcpyHostToDevice, s));
    }
    // a launch that gives up leaves timed_out set; one that ends clears it
    RTE_CUDA_TRY(cudaMemsetAsync(status_dev, 0xff, sizeof(SolveStatus), s));
    const MGDeviceLevel& c = g.lev[g.L - 1];
    a.nRp = d.nRp;
    a.m = g.lev[0].m;
    a.nrhs = nrhs;
    a.maxit = maxit;
    a.nu = g.nu;
    a.L = g.L;
    a.Q = g.Q;
    a.N = c.n * d.dP;
    a.cld = g.cld;
    a.rb = std::min(nrhs, kDenseRhs);
    a.tol2 = tol * tol;
    a.ec = f32_products ? nullptr : d.ec_ell;
    a.B = B;
    a.X = X;
    a.status = status_dev;
    a.cinv = g.cinv;
    a.Gq = g.G;
    a.lev = g.dev_lev;
    switch (d.dP) {
        case 1: return launch_classes<1>(s, a);
        case 6: return launch_classes<6>(s, a);
        default: return launch_classes<15>(s, a);
    }
}

}  // namespace rte
