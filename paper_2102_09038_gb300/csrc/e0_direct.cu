// E_0^{-1} by a direct factorisation of its direction blocks, the route of
// the paper's experiments (Section 6: E_0's blocks solved by a sparse direct
// factorisation), laid out for the GPU.
//
// Block k of E_0 (eq. equivalence_bE_bE0) is the 7-point stencil of the
// "/"-mesh with the direction's weights.  With the nodes in lexicographic
// order (x fastest) it is block tridiagonal over the mesh rows y = 0..m, each
// block of size b = m + 1:
//   A_yy      tridiagonal (self, +x, -x),
//   A_y,y-1   two diagonals (-y: node (x, y-1), -x-y: node (x-1, y-1)),
//   A_y,y+1 = A_y+1,y^T   (+y: node (x, y+1), +x+y: node (x+1, y+1)).
// The rows are eliminated from both ends towards the middle row h = b / 2:
// S_0 = A_00, S_y = A_yy - A_y,y-1 S_y-1^{-1} A_y-1,y for y < h, the same from
// the last row upwards for y > h, and S_h with both corrections.  Kept are
// the explicit inverses S_y^{-1} (dense, symmetric, b x b).  The solve runs
// both chains at once, each by one block of a two-block cluster:
//   towards h   w_y = S_y^{-1} (b_y - A_y,y' w_y')       y' the row before
//   at h        x_h = S_h^{-1} (b_h - A_h,h-1 w_h-1 - A_h,h+1 w_h+1)
//               (each block, after exchanging the two w)
//   back        x_y = w_y - S_y^{-1} (A_y,y' x_y')       y' the row after
// so a direction takes b dependent steps of two blocks instead of 2 b - 1 of
// one.
//
// What bounds it: reading the factor, twice, from HBM on large meshes; on
// small ones the chain of steps, each a wait for its record, a few products
// and three block barriers.  Hence each S_y^{-1} is kept by the tiles of its
// upper triangle (8 x 8, the diagonal ones full: 0.59 of the dense rows at
// b = 129), in one record with its row's coupling coefficients, so a step is
// one bulk copy into a ring of shared-memory slots; as many blocks share an
// SM as the slots allow, and where a chain's right-hand side fits in shared
// memory (small meshes) the steps touch no global memory but the copies and
// the stores of x.  Measured, us per solve (one right-hand side): 128 x 128 /
// 256 directions FP32 1075 -> 640, FP64 10580 -> 5000;
// 32 x 32 / 64 directions FP32 137 -> 37, FP64 325 -> 66; 96 x 96 / 1024
// directions FP32 2480 -> 1230.
//
// Setup factorises in FP64 (two blocks per direction, S_y in shared memory,
// Gauss-Jordan inversion); the factor is kept in FP64 (FP64 mode) or FP32
// (mixed modes, where E_0^{-1} is a preconditioner under the FP64 outer
// residual).
#include <cuda_runtime.h>

#include <algorithm>

#include "device.h"
#include "rte_internal.h"

namespace rte {

namespace {

constexpr int kThreads = 256;        // of the factorisation
constexpr int kRB = 4;               // right-hand sides per sweep of the factor
constexpr int kMaxParts = 6;         // groups that share a tile row, at most
// largest mesh of the route: the set-up holds one b x b FP64 matrix in
// shared memory
constexpr int kMaxM = 156;
constexpr int kSmemPerSm = 226 * 1024;

// Limit of one wait for a factor record (SM clock cycles; ~2 s at 2 GHz),
// and the flag a wait that ran out sets.
__device__ long long g_e0_wait_cycles = 4000000000ll;
__device__ int g_e0_error = 0;

__device__ __forceinline__ double cf(const double* coef, int nRp, int nSp, int dir, int node,
                                     int k) {
    return coef[((size_t)dir * nRp + node) * nSp + k];
}

// Threads of the solve's products for one and for up to kRB right-hand sides,
// at most (one more warp copies): with four blocks on an SM 48 and 64
// registers each.
__host__ __device__ constexpr int e0_threads(int NR) { return NR == 1 ? 288 : 224; }

// A row's record, in elements: [A pair | tiles | B pair] with nt = ceil(b / 8)
// tile rows and bp = 8 nt; the A pair holds the coefficients towards row y - 1
// (-y at x, then bp later -x-y at x), the B pair those towards y + 1 (+y, then
// +x+y); pairs are padded to whole tiles.
__host__ __device__ __forceinline__ int e0_nt(int m) { return (m + 8) / 8; }
__host__ __device__ __forceinline__ int e0_tiles(int nt) { return nt * (nt + 1) / 2; }
__host__ __device__ __forceinline__ int e0_pair(int nt) { return (16 * nt + 63) / 64 * 64; }
__host__ __device__ __forceinline__ int e0_record(int nt) { return 64 * e0_tiles(nt) + 2 * e0_pair(nt); }
// tile (I, J), I <= J, and element (r, c) of tile t: rows permuted by the
// tile and 16-byte pieces by the row, so that eight lanes reading one row
// each (16 bytes) and four times eight lanes reading one row of neighbouring
// tiles (one element each) both meet distinct banks
__host__ __device__ __forceinline__ int e0_tile(int nt, int I, int J) {
    return I * nt - I * (I - 1) / 2 + J - I;
}
template <typename T>
__host__ __device__ __forceinline__ int e0_elem(int t, int r, int c) {
    constexpr int CH = 16 / sizeof(T), NCH = 8 / CH;   // elements per piece, pieces per row
    return 64 * t + ((r ^ (t & 3)) * 8) + (((c / CH) ^ (r / (8 / NCH))) * CH) + c % CH;
}

// One chain (or the middle row) of direction block k = blockIdx.x: part 0 the
// rows 0 .. h-1 downwards, 1 the rows b-1 .. h+1 upwards, 2 the row h.  G:
// FP64 scratch of two b x b per direction (the last inverse of either chain);
// out32 / out64: the records [k][y].
__global__ void __launch_bounds__(kThreads) k_e0_factor(int m, int nSp, int middle,
                                                        const double* __restrict__ coef,
                                                        double* __restrict__ G,
                                                        float* __restrict__ out32,
                                                        double* __restrict__ out64) {
    extern __shared__ double sm[];
    const int b = m + 1, nRp = b * b, k = blockIdx.x, h = b / 2;
    const int part = middle ? 2 : (int)blockIdx.y;
    const int nt = e0_nt(m), bp = 8 * nt, rec = e0_record(nt);
    double* S = sm;                 // b x b, row-major, leading dimension b
    double* colp = S + b * b;       // column p before elimination
    double* rowp = colp + b;        // row p after scaling
    const int bb = b * b;
    double* Gk = G + (size_t)k * 2 * bb;
    const int rows = part == 0 ? h : part == 1 ? b - 1 - h : 1;
    for (int n = 0; n < rows; ++n) {
        const int y = part == 0 ? n : part == 1 ? b - 1 - n : h;
        // S_y = A_yy - sum over the rows y' eliminated before it (y - 1 and /
        // or y + 1) of A_y,y' S_y'^{-1} A_y',y
        for (int e = threadIdx.x; e < bb; e += blockDim.x) {
            const int r = e / b, c = e - r * b;
            const int nr = y * b + r, nc = y * b + c;
            double v = 0.0;
            if (r == c) v = cf(coef, nRp, nSp, 0, nr, k);
            else if (c == r + 1) v = cf(coef, nRp, nSp, 1, nr, k);
            else if (c == r - 1) v = cf(coef, nRp, nSp, 2, nr, k);
            for (int side = 0; side < 2; ++side) {
                const bool from = side == 0 ? (part != 1 && y > 0)
                                            : (part != 0 && y < b - 1);
                if (!from) continue;
                const double* Gs = Gk + (size_t)side * bb;
                const int d0 = side == 0 ? 4 : 3, d1 = side == 0 ? 6 : 5, s = side == 0 ? -1 : 1;
                const bool hr = r + s >= 0 && r + s < b, hc = c + s >= 0 && c + s < b;
                const double lr0 = cf(coef, nRp, nSp, d0, nr, k);
                const double lr1 = hr ? cf(coef, nRp, nSp, d1, nr, k) : 0.0;
                const double lc0 = cf(coef, nRp, nSp, d0, nc, k);
                const double lc1 = hc ? cf(coef, nRp, nSp, d1, nc, k) : 0.0;
                double a = lr0 * lc0 * Gs[r * b + c];
                if (hc) a += lr0 * lc1 * Gs[r * b + c + s];
                if (hr) a += lr1 * lc0 * Gs[(r + s) * b + c];
                if (hr && hc) a += lr1 * lc1 * Gs[(r + s) * b + c + s];
                v -= a;
            }
            S[e] = v;
        }
        __syncthreads();
        // in-place Gauss-Jordan inversion (S is SPD: no pivoting)
        for (int p = 0; p < b; ++p) {
            const double d = 1.0 / S[p * b + p];
            for (int r = threadIdx.x; r < b; r += blockDim.x) {
                colp[r] = S[r * b + p];
                rowp[r] = r == p ? d : S[p * b + r] * d;
            }
            __syncthreads();
            // (r, c) of entry e advance by the block's stride without a division
            const int sr = blockDim.x / b, sc = blockDim.x - sr * b;
            int r = threadIdx.x / b, c = threadIdx.x - r * b;
            for (int e = threadIdx.x; e < bb; e += blockDim.x) {
                if (r == p) S[e] = rowp[c];
                else if (c == p) S[e] = -colp[r] * d;
                else S[e] = fma(-colp[r], rowp[c], S[e]);
                r += sr;
                c += sc;
                if (c >= b) {
                    c -= b;
                    ++r;
                }
            }
            __syncthreads();
        }
        // symmetrised inverse and couplings to the record, and the inverse
        // to the scratch of the next row
        const size_t o = ((size_t)k * b + y) * rec;
        auto put = [&](int at, double v) {
            if (out32) out32[o + at] = (float)v;
            if (out64) out64[o + at] = v;
        };
        for (int e = threadIdx.x; e < bp * bp; e += blockDim.x) {
            const int r = e / bp, c = e - r * bp, I = r >> 3, J = c >> 3;
            const bool in = r < b && c < b;
            const double v = in ? 0.5 * (S[r * b + c] + S[c * b + r]) : 0.0;
            if (in && part < 2) Gk[(size_t)part * bb + r * b + c] = v;
            if (I > J) continue;
            const int t = e0_tile(nt, I, J);
            put(e0_pair(nt) + (out32 ? e0_elem<float>(t, r & 7, c & 7) : e0_elem<double>(t, r & 7, c & 7)), v);
        }
        const int pw = e0_pair(nt);
        for (int e = threadIdx.x; e < 2 * pw; e += blockDim.x) {
            const int up = e / pw, f = e - up * pw, q = f / bp, x = f - q * bp;
            const int dir = up ? (q ? 5 : 3) : (q ? 6 : 4);
            put(up ? rec - pw + f : f, q < 2 && x < b ? cf(coef, nRp, nSp, dir, y * b + x, k) : 0.0);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ uint32_t sh_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t par) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(par)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of parity `par` of the mbarrier at `bar`.  The
// limit (in global memory) is read only by a wait that has gone on for a
// while: its latency would otherwise be part of every wait that does not
// succeed at once.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t par) {
    if (mbar_try(bar, par)) return true;
    const long long t0 = clock64();
    while (true) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try(bar, par)) return true;
        if (clock64() - t0 > g_e0_wait_cycles) {
            atomicExch(&g_e0_error, 1);
            return false;
        }
    }
}

// One thread: one bulk copy of `bytes` (a multiple of 16, both addresses
// 16-byte aligned) from global src into shared dst, completing on bar.
__device__ __forceinline__ void tma_block(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// all threads of both blocks of the cluster; earlier writes to the peer's
// shared memory are visible after it
__device__ __forceinline__ void cluster_meet() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// loads by shared-memory address: one element, or a 16-byte piece
__device__ __forceinline__ void lds(uint32_t p, float& v) {
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(p));
}
__device__ __forceinline__ void lds(uint32_t p, double& v) {
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(p));
}
__device__ __forceinline__ void lds16(uint32_t p, float* v) {
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(p));
}
__device__ __forceinline__ void lds16(uint32_t p, double* v) {
    asm volatile("ld.shared.v2.f64 {%0,%1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(p));
}

__device__ __forceinline__ void sts(uint32_t p, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void sts(uint32_t p, double v) {
    asm volatile("st.shared.f64 [%0], %1;" ::"r"(p), "d"(v) : "memory");
}
template <typename T>
__device__ __forceinline__ T ldv(uint32_t p) {
    T v;
    lds(p, v);
    return v;
}

// acc[r] += s . v[r] over the eight values at shared address p + r stride, in
// two short chains (they round less than one over the whole row)
template <typename T, int NR>
__device__ __forceinline__ void e0_dot(const T (&s)[8], uint32_t p, uint32_t stride, T (&acc)[NR]) {
    constexpr int CH = 16 / sizeof(T);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        T u[8];
#pragma unroll
        for (int i = 0; i < 8 / CH; ++i) lds16(p + r * stride + 16 * i, u + CH * i);
        T a = s[0] * u[0], c4 = s[4] * u[4];
#pragma unroll
        for (int c = 1; c < 4; ++c) {
            a = fma(s[c], u[c], a);
            c4 = fma(s[4 + c], u[4 + c], c4);
        }
        acc[r] += a + c4;
    }
}

// X = E_0^{-1} B for direction k = blockIdx.x / 2, every right-hand side, in
// sweeps of up to kRB; block side 0 of the cluster takes the rows from 0, side
// 1 those from b - 1, both the middle row.  Eight lanes own eight consecutive
// rows of the product (one each) and read their tiles by rows right of the
// diagonal, by columns left of it; P groups of eight share a tile row and meet
// in `part`.  HIST: the chain's right-hand side, and then its w, stay in
// shared memory; else they are read one step ahead and w waits in X.
template <typename T, bool HIST, int NR>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(e0_threads(NR) + 32, sizeof(T) == 4 ? 4 : 2)
k_e0_solve(int m, int nSp, int nrhs, int P, int slots, const T* __restrict__ fac,
           const double* __restrict__ B, double* __restrict__ X) {
    extern __shared__ __align__(128) unsigned char smraw[];
    constexpr int SZ = sizeof(T), CH = 16 / SZ, NCH = 8 / CH, RB = 8 * SZ, kE = NR;
    const int b = m + 1, nRp = b * b, h = b / 2, nt = e0_nt(m), bp = 8 * nt, rec = e0_record(nt);
    const int k = blockIdx.x >> 1, side = blockIdx.x & 1, tid = threadIdx.x;
    const int n = side == 0 ? h : b - 1 - h;   // rows of the chain
    const int passes = (nrhs + NR - 1) / NR;
    const int nthr = (int)blockDim.x - 32;     // of the products; the last warp copies
    __shared__ __align__(8) unsigned long long bars[16];   // full and empty, per slot
    const uint32_t full0 = sh_addr(bars), empty0 = full0 + 64;
    // Byte addresses in shared memory: the ring (tiles on their own size:
    // their elements' addresses are formed by XOR), the product's right-hand
    // side, the row before, the other chain's last w (twice), the partial
    // products, and with HIST the chain's rows.
    const uint32_t recb = rec * SZ, pairb = e0_pair(nt) * SZ, rowb = (uint32_t)bp * SZ, vecb = NR * rowb;
    const uint32_t ring = (sh_addr(smraw) + 511) & ~511u, aV = ring + slots * recb, aPrev = aV + vecb,
                   aMid = aPrev + vecb, aPart = aMid + 2 * vecb, aHist = aPart + P * vecb;
    const T* fk = fac + (size_t)k * b * rec;
    if (tid == 0) {
        for (int s = 0; s < slots; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8 * s) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty0 + 8 * s), "r"(nthr / 32)
                         : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_meet();   // the peer runs: its shared memory may be written
    if (tid >= nthr) {
        // The last warp keeps the ring full, one record per step and without
        // the pair of coefficients the step does not use.  It has nothing to
        // exchange at the middle row: it arrives there ahead (its copies must
        // go on while the products wait for each other) and waits when the
        // sweep's copies are issued.
        int slot = 0, done = 0;
        uint32_t ph = 1;   // a fresh barrier passes a wait for the phase before
        bool ok = true;
        for (int pass = 0; pass < passes; ++pass) {
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            if (tid == nthr)
                for (int t = 0; t <= 2 * n && ok; ++t) {
                    if (!mbar_wait(empty0 + 8 * slot, ph)) { ok = false; break; }
                    // every read of the slot came before its arrivals: order
                    // them before the copy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    const int j = t < n ? t : 2 * n - t;   // chain row, n: the middle
                    const int y = j == n ? h : side == 0 ? j : b - 1 - j;
                    const bool needA = t == n || (t < n) == (side == 0), needB = t == n || !needA;
                    const uint32_t o0 = needA ? 0 : pairb, o1 = needB ? recb : recb - pairb;
                    tma_block(ring + slot * recb + o0,
                              reinterpret_cast<const char*>(fk + (size_t)y * rec) + o0, o1 - o0,
                              full0 + 8 * slot);
                    ++done;
                    if (++slot == slots) { slot = 0; ph ^= 1; }
                }
            __syncwarp();
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
        // after a timeout: the copies still in flight land before the block
        // leaves
        if (tid == nthr && !ok)
            for (int q = max(0, done - slots); q < done; ++q)
                mbar_wait(full0 + 8 * (q % slots), (uint32_t)(q / slots) & 1u);
        return;
    }
    // barrier of the products' threads alone
    auto block_sync = [&]() { asm volatile("barrier.sync 1, %0;" ::"r"(nthr) : "memory"); };
    const int g = tid >> 3, lane = tid & 7, I = g % nt, p = g / nt;
    const bool work = p < P;
    const int J0 = p * nt / P, J1 = (p + 1) * nt / P;
    // this group's tiles: columns of (J0 .. Jc - 1, I), rows of (I, Jr .. J1 - 1)
    const int Jc = min(J1, I), Jr = max(J0, I), colt = e0_tile(nt, J0, I), rowt = e0_tile(nt, I, Jr);
    const uint32_t aOut = aPart + p * vecb + (8 * I + lane) * SZ;
    // the coefficient pairs towards the row before (forward) and after, and
    // the neighbour in x they reach besides the node itself
    const uint32_t pairA = 0, pairB = recb - pairb;
    const uint32_t fpair = side == 0 ? pairA : pairB, bpair = side == 0 ? pairB : pairA;
    const int fs = side == 0 ? -1 : 1;
    bool ok = true;   // this thread's waits; after one that ran out the steps
                      // go on without stores, so that the cluster meets
    int slot = 0;
    uint32_t ph = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const int r0 = pass * NR, nr = min(NR, nrhs - r0);
        // this thread's elements of a row: one x, and the right-hand sides
        // rfirst, rfirst + rstep, ...; byte offsets of x and of the neighbours
        // in x the two pairs reach (the node itself where there is none: the
        // coefficient is zero there)
        const int rfirst = NR == 1 ? 0 : tid / bp, x = tid - rfirst * bp;
        const int rstep = NR == 1 ? 1 : nthr / bp;
        const bool mine_x = NR == 1 ? tid < bp : rfirst < rstep;
        const uint32_t xb = x * SZ;
        const int nbf = (x + fs >= 0 && x + fs < b) ? fs * SZ : 0;
        const int nbb = (x - fs >= 0 && x - fs < b) ? -fs * SZ : 0;
        bool own[kE], in[kE];
        uint32_t eb[kE];
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            const int r = rfirst + j * rstep;
            // (a last sweep of fewer carries zeros for the others)
            own[j] = mine_x && r < NR;
            in[j] = own[j] && x < b && r < nr;
            eb[j] = r * rowb + xb;
        }
        const size_t at0 = ((size_t)(r0 + rfirst) * nRp + x) * nSp + k,
                     atr = (size_t)rstep * nRp * nSp;
        auto at = [&](int j) { return at0 + j * atr; };   // place in B and X, without the row
        const size_t ystep = (size_t)b * nSp;
        auto chain_at = [&](int j) { return (size_t)(side == 0 ? j : b - 1 - j) * ystep; };
        // read ahead: the next step's b towards the middle, w on the way back
        T nxt[kE];
        auto ahead = [&](const double* src, size_t row) {
#pragma unroll
            for (int j = 0; j < kE; ++j) nxt[j] = in[j] ? (T)src[at(j) + row] : T(0);
        };
        ahead(B, HIST || n == 0 ? h * ystep : chain_at(0));
        if constexpr (HIST) {
            for (int c = 0; c < n; ++c)
#pragma unroll
                for (int j = 0; j < kE; ++j)
                    if (own[j])
                        sts(aHist + c * vecb + eb[j], in[j] ? (T)B[at(j) + chain_at(c)] : T(0));
        }
        // the record of the next step
        auto record = [&]() -> uint32_t {
            if (ok && !mbar_wait(full0 + 8 * slot, ph)) ok = false;
            return ring + slot * recb;
        };
        auto pair = [&](uint32_t c, uint32_t u, int j, int nb) {
            T a = ldv<T>(c + xb) * ldv<T>(u + eb[j]);
            return a + ldv<T>(c + rowb + xb) * ldv<T>(u + eb[j] + nb);
        };
        // sum[j] = element j of S^{-1} v for the record at R, whose slot is
        // then given back
        auto product = [&](uint32_t R, T (&sum)[kE]) {
            block_sync();   // v is complete
            if (work) {
                T acc[NR], s[8];
#pragma unroll
                for (int r = 0; r < NR; ++r) acc[r] = T(0);
                const uint32_t tiles = R + pairb;
                int tl = colt;
#pragma unroll 2
                for (int J = J0; J < Jc; ++J) {
                    const uint32_t q = tiles + tl * 8 * RB + ((tl & 3) * RB) + lane * SZ;
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        lds(q ^ (uint32_t)(c * RB | (c / (8 / NCH)) << 4), s[c]);
                    e0_dot<T, NR>(s, aV + J * RB, rowb, acc);
                    tl += nt - J - 1;
                }
                tl = rowt;
#pragma unroll 2
                for (int J = Jr; J < J1; ++J, ++tl) {
                    const uint32_t q = tiles + tl * 8 * RB + ((lane ^ (tl & 3)) * RB) + ((lane / (8 / NCH)) << 4);
#pragma unroll
                    for (int i = 0; i < NCH; ++i) lds16(q ^ (uint32_t)(i << 4), s + CH * i);
                    e0_dot<T, NR>(s, aV + J * RB, rowb, acc);
                }
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    sts(aOut + r * rowb, acc[r]);
            }
            // the slot is free once every warp has read it
            __syncwarp();
            if ((tid & 31) == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty0 + 8 * slot) : "memory");
            if (++slot == slots) { slot = 0; ph ^= 1; }
            block_sync();   // the partial products are complete
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                T q[kMaxParts];
#pragma unroll
                for (int u = 0; u < kMaxParts; ++u)
                    q[u] = u < P ? ldv<T>(aPart + u * vecb + eb[j]) : T(0);
                sum[j] = ((q[0] + q[1]) + (q[2] + q[3])) + (q[4] + q[5]);
            }
        };
        // towards the middle: w_y
        T sum[kE];
        for (int t = 0; t < n; ++t) {
            const uint32_t R = record();
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                T v = T(0);
                if (in[j]) {
                    v = HIST ? ldv<T>(aHist + t * vecb + eb[j]) : nxt[j];
                    if (t > 0) v -= pair(R + fpair, aPrev, j, nbf);
                }
                sts(aV + eb[j], v);
            }
            if constexpr (!HIST) ahead(B, t + 1 < n ? chain_at(t + 1) : h * ystep);
            product(R, sum);
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                sts(aPrev + eb[j], sum[j]);
                if constexpr (HIST) sts(aHist + t * vecb + eb[j], sum[j]);
                else if (ok && in[j]) X[at(j) + chain_at(t)] = (double)sum[j];
            }
            block_sync();
        }
        // the chains' last rows change hands, and the middle row
        const uint32_t mine = aMid + (pass & 1) * vecb;
        uint32_t peer;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(mine), "r"(side ^ 1));
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            if (!own[j]) continue;
            const T w = n > 0 ? ldv<T>(aPrev + eb[j]) : T(0);
            if constexpr (SZ == 4)
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer + eb[j]), "f"((float)w) : "memory");
            else
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(peer + eb[j]), "d"((double)w) : "memory");
        }
        __syncwarp();
        cluster_meet();
        {
            const uint32_t R = record();
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                T v = T(0);
                if (in[j]) {
                    v = nxt[j];
                    if (n > 0) v -= pair(R + fpair, aPrev, j, nbf);
                    v -= pair(R + bpair, mine, j, nbb);
                }
                sts(aV + eb[j], v);
            }
            product(R, sum);
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                sts(aPrev + eb[j], sum[j]);
                if (ok && in[j] && side == 0) X[at(j) + h * ystep] = (double)sum[j];
            }
            if (!HIST && n > 0) ahead(X, chain_at(n - 1));
            block_sync();
        }
        // and back: x_y = w_y - S^{-1} (the coupling to the row after)
        for (int t = n - 1; t >= 0; --t) {
            const uint32_t R = record();
#pragma unroll
            for (int j = 0; j < kE; ++j)
                if (own[j]) sts(aV + eb[j], in[j] ? pair(R + bpair, aPrev, j, nbb) : T(0));
            product(R, sum);
#pragma unroll
            for (int j = 0; j < kE; ++j) {
                if (!own[j]) continue;
                const T x = (HIST ? ldv<T>(aHist + t * vecb + eb[j]) : nxt[j]) - sum[j];
                sts(aPrev + eb[j], x);
                if (ok && in[j]) X[at(j) + chain_at(t)] = (double)x;
            }
            if (!HIST && t > 0) ahead(X, chain_at(t - 1));
            block_sync();
        }
    }
}

// How the solve is launched: threads and groups per tile row, slots and
// shared memory, and whether the chains' right-hand sides are kept there.
struct SolvePlan {
    int threads, P, slots;
    size_t smem;
    bool hist;
};

template <typename T>
SolvePlan solve_plan(int m, int nSp, int nrhs) {
    SolvePlan pl{};
    const int nt = e0_nt(m), bp = 8 * nt, nr = std::min(nrhs, kRB), b = m + 1;
    pl.P = std::max(1, std::min({nt, e0_threads(nrhs) / (8 * nt), kMaxParts}));
    pl.threads = (8 * nt * pl.P + 31) / 32 * 32;
    const size_t rec = e0_record(nt) * sizeof(T);
    const size_t vec = (size_t)(4 + pl.P) * nr * bp * sizeof(T);
    const size_t hist = (size_t)(b - 1 - b / 2 > b / 2 ? b - 1 - b / 2 : b / 2) * nr * bp * sizeof(T);
    // As many blocks per SM as it takes to have every chain resident, at
    // most 4 (2 in FP64): chains that wait for each other's copies keep HBM
    // busy, while a second wave would leave half the SMs idle at its end.
    const int most = sizeof(T) == 4 ? 4 : 2;
    int per = std::min(most, std::max(1, (2 * nSp + device_sm_count() - 1) / device_sm_count()));
    for (;; --per) {
        const size_t room = kSmemPerSm / per - 2048;   // driver's share, alignment, barriers
        if (vec + rec > room && per > 1) continue;
        pl.hist = vec + hist + 2 * rec <= room;
        const size_t left = room - vec - (pl.hist ? hist : 0);
        pl.slots = (int)std::max<size_t>(1, std::min<size_t>(8, left / rec));
        pl.smem = pl.slots * rec + vec + (pl.hist ? hist : 0) + 512;   // 512: alignment
        return pl;
    }
}

template <typename T, bool HIST, int NR>
int solve_launch(cudaStream_t s, const DevSystem& d, const SolvePlan& pl, const T* fac,
                 const double* B, double* X, int nrhs) {
    auto kern = k_e0_solve<T, HIST, NR>;
    // the attribute is per device and per kernel: every call sets the same
    // value, so none can shrink it under another's launch
    RTE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm));
    kern<<<2 * d.nSp, pl.threads + 32, pl.smem, s>>>(d.m, d.nSp, nrhs, pl.P, pl.slots, fac, B, X);
    count_launches(1);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

template <typename T, int NR>
int solve_nr(cudaStream_t s, const DevSystem& d, const SolvePlan& pl, const T* fac, const double* B,
             double* X, int nrhs) {
    return pl.hist ? solve_launch<T, true, NR>(s, d, pl, fac, B, X, nrhs)
                   : solve_launch<T, false, NR>(s, d, pl, fac, B, X, nrhs);
}

template <typename T>
int solve(cudaStream_t s, const DevSystem& d, const T* fac, const double* B, double* X, int nrhs) {
    const SolvePlan pl = solve_plan<T>(d.m, d.nSp, nrhs);
    switch (std::min(nrhs, kRB)) {
        case 1: return solve_nr<T, 1>(s, d, pl, fac, B, X, nrhs);
        case 2: return solve_nr<T, 2>(s, d, pl, fac, B, X, nrhs);
        case 3: return solve_nr<T, 3>(s, d, pl, fac, B, X, nrhs);
        default: return solve_nr<T, kRB>(s, d, pl, fac, B, X, nrhs);
    }
}

size_t factor_smem(int m) { return (size_t)((m + 1) * (m + 1) + 2 * (m + 1)) * sizeof(double); }

}  // namespace

// m <= 156: the set-up's FP64 Schur complement fits in 200 KB of shared
// memory (and the solve's record, 113 KB in FP64, beside its vectors).
bool e0_direct_fits(int m) { return m >= 1 && m <= kMaxM; }

size_t e0_direct_bytes(int m, int nSp, bool fp64) {
    return (size_t)nSp * (m + 1) * e0_record(e0_nt(m)) * (fp64 ? 8 : 4);
}

size_t e0_direct_scratch_bytes(int m, int nSp) {
    return (size_t)nSp * 2 * (m + 1) * (m + 1) * sizeof(double);
}

int e0_direct_factor(cudaStream_t s, const DevSystem& d, double* scratch, float* out32,
                     double* out64) {
    const int m = d.m;
    if (!e0_direct_fits(m)) return fail(RTE_ERR_ARG, "mesh too large for the direct E_0 route");
    const size_t sm = factor_smem(m);
    RTE_CUDA_TRY(cudaFuncSetAttribute(k_e0_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)factor_smem(kMaxM)));
    count_launches(2);
    k_e0_factor<<<dim3(d.nSp, 2), kThreads, sm, s>>>(m, d.nSp, 0, d.e0coef, scratch, out32, out64);
    k_e0_factor<<<d.nSp, kThreads, sm, s>>>(m, d.nSp, 1, d.e0coef, scratch, out32, out64);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

int e0_direct_solve(cudaStream_t s, const DevSystem& d, const double* B, double* X, int nrhs,
                    bool fp64) {
    if (fp64) {
        if (!d.e0lu64) return fail(RTE_ERR_ARG, "no FP64 direct E_0 factor");
        return solve<double>(s, d, d.e0lu64, B, X, nrhs);
    }
    if (!d.e0lu32) return fail(RTE_ERR_ARG, "no FP32 direct E_0 factor");
    return solve<float>(s, d, d.e0lu32, B, X, nrhs);
}

int e0_direct_flag(const int** flag) {
    RTE_CUDA_TRY(cudaGetSymbolAddress((void**)flag, g_e0_error));
    return RTE_OK;
}

int e0_direct_error_check(cudaStream_t s, int flag) {
    if (!flag) return RTE_OK;
    const int zero = 0;
    cudaMemcpyToSymbolAsync(g_e0_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
    return fail(RTE_ERR_TIMEOUT, "a wait for a staged E_0 factor record timed out");
}

int e0_direct_error(cudaStream_t s) {
    int e = 0;
    RTE_CUDA_TRY(cudaMemcpyFromSymbolAsync(&e, g_e0_error, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
    RTE_CUDA_TRY(cudaStreamSynchronize(s));
    return e0_direct_error_check(s, e);
}

int e0_set_wait_cycles(long long cycles) {
    RTE_CUDA_TRY(cudaMemcpyToSymbol(g_e0_wait_cycles, &cycles, sizeof(cycles)));
    return RTE_OK;
}

}  // namespace rte
