// cluster_chol.cuh -- Cholesky factor and both triangular solves of one
// symmetric positive definite FP64 system per thread-block cluster.
//
// Used for the Gram of the dynamic block: every row of I of a dense A, the
// n x n form, and the coupled rows of a sparse A whose connected component is
// too large for one warp.
//
// What bounds it.  GB300's FP64 unit takes one warp instruction per 64 cycles
// from one warp and one per 17 to 19 cycles from a whole SM (measured: a
// dependent fused multiply-add 64 cycles, CUDA's sqrt 611, division 581), so a
// factor of order 256 is a chain of 256 pivots, each a square root, a quotient
// and one update, with 2.8 million multiply-adds around it.  The design keeps
// the chain short and everything else off it:
//   - panels of 32 columns; the rows below the panel's 32 x 32 diagonal block are
//     dealt over the cluster, every block factors the diagonal block itself
//     (identical operations), so a panel needs no communication;
//   - inside a column two warps form the pivot and divide, with 1 / sqrt(d) taken
//     first and root and quotients from it by fused remainders (pivot.cuh; no call
//     to sqrt or to a division), while six warps apply
//     the previous column to the columns after the next, from registers;
//   - the trailing update of a panel runs over all warps of the cluster (a lane
//     per column, a few rows per warp) from a copy of the panel in shared memory;
//     only its part in the next panel's columns is awaited, the rest runs beside
//     those columns in the block's second half;
//   - the right-hand side is carried as one more row of the matrix, so the
//     forward solve costs nothing extra; the backward solve runs in the
//     cluster's first block, one warp on the 32-row diagonal chain while the
//     others apply the finished rows of the solution further up.
// Two cluster barriers per panel order the traffic through L2.
//
// Measured (16 blocks, one launch; 8 at order 100, 4 at 40): order 256 313 us (mixed
// form's factor 237 us), order 100 116 us, order 40 47 us, order 500 837 us; with the
// whole trailing update awaited 348, 128, 54 and 995 us.  At order 256 about 356 kcycles of
// 622 are the 256 columns and 100 the backward solve.  Before: 15 grid-wide launches
// and a one-block backward solve, 1,003 us at order 256 (dense A); the sparse
// dynamic block, factored by one block of threads, 2,230 us at about 230 coupled
// rows.
//
// Order of operations.  Every entry receives g = fma(-L_aj, L_bj, g) over
// ascending j, then the correctly rounded quotient by
// L_jj, exactly as the one-block right-looking factor and column-oriented
// solves, so the result is the same bit for bit.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "pivot.cuh"

namespace rorbk {

constexpr int kCw = 32;                 // panel width
constexpr int kCwp = kCw + 1;           // row stride of panels in shared memory
constexpr int kCcThreads = 512;          // one system at a time (256 for a block of columns)
constexpr int kCcMaxCluster = 16;       // blocks per cluster
constexpr int kCcMaxRows = 32;          // rows below the diagonal block per block: one per lane

// (.aligned: a warp's lanes arrive together, also where the code before left them
// apart)
__device__ __forceinline__ void cluster_sync_all() {
    __threadfence();
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_blocks() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Rows below the first diagonal block per block of a cluster of C (with the
// right-hand side's row), and the largest order such a cluster takes.
__host__ __device__ constexpr int cc_rows(int K, int C) { return K + 1 <= kCw ? 1 : (K + 1 - kCw + C - 1) / C; }
__host__ __device__ constexpr int cc_max_order(int C) {
    return C * kCcMaxRows + kCw - 1;
}
template <int N>
struct IntC { static constexpr int value = N; };
constexpr int kCcStage = 2 * kCw * kCwp;          // backward solve: one stage (two 32 x 32 tiles)
// Dynamic shared memory for orders up to K: diagonal block, own rows, the
// panel (or the three stages of the backward solve), z, reciprocals.
__host__ __device__ constexpr size_t cc_smem_bytes(int K, int C) {
    const size_t panel = (size_t)(K + 1) * kCwp > 3u * kCcStage ? (size_t)(K + 1) * kCwp : 3u * kCcStage;
    return ((size_t)kCw * kCwp + (size_t)cc_rows(K, C) * kCwp + panel + 2u * (size_t)(K + kCw)) * sizeof(double);
}

// Factor of the w x w diagonal block Ld in step with nr rows R below it (one
// block of threads; see the file comment).  On return Ld and R hold L; the
// diagonal holds L_jj (RC: 1 / L_jj) and rlp[j] its reciprocal (rlp: 2 kCw values).  RC is the
// mixed form's factor: rsqrt on the diagonal, products instead of quotients.
//
// Column j: warp 0 has the diagonal block's column, warp 1 the rows' column.
// Each applies column j - 1, forms the pivot for itself (handing it over
// through shared memory costs more than the repeated operations) and divides.
// Warps 2..7 keep the entries of the columns after j in registers, apply column
// j - 1 to them and put column j + 1 back into shared memory for the next step,
// so one barrier per column is enough.  Their entries are listed by descending
// column: those still to be updated are always the first ones, and a step issues
// as few FP64 instructions as the entries fill.
constexpr int kCcBulk = 256 - 64;
constexpr int kCcTri = kCw * (kCw - 1) / 2;          // entries of columns 1 .. kCw - 1 of the diagonal block
constexpr int kCcGd = (kCcTri + kCcBulk - 1) / kCcBulk;
constexpr int kCcGr = ((kCw - 1) * kCcMaxRows + kCcBulk - 1) / kCcBulk;

// (The panel's 256 threads meet at named barrier 1: in a block of 512 the other
// half works on the previous panel's trailing update meanwhile.)
__device__ __forceinline__ void panel_sync() {
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
}

template <bool RC>
__device__ __forceinline__ void cc_panel(double *Ld, double *R, int w, int nr, double *rlp, int *bad) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, bt = (int)threadIdx.x - 64;
    double gd[kCcGd], gr[kCcGr];
    int pd[kCcGd], pr[kCcGr];                    // row << 8 | column (0: no entry)
    if (warp >= 2) {
#pragma unroll
        for (int k = 0; k < kCcGd; ++k) {        // column w - 1 - t holds t + 1 entries
            const int e = bt + kCcBulk * k;
            int t = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
            while (t * (t + 1) / 2 > e) --t;
            while ((t + 1) * (t + 2) / 2 <= e) ++t;
            const int c = w - 1 - t, i = c + e - t * (t + 1) / 2;
            pd[k] = c > 0 ? i << 8 | c : 0;
            gd[k] = c > 0 ? Ld[i * kCwp + c] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kCcGr; ++k) {
            const int e = bt + kCcBulk * k;
            const int t = nr > 0 ? e / nr : kCw, c = w - 1 - t, u = e - t * nr;
            pr[k] = c > 0 ? u << 8 | c : 0;
            gr[k] = c > 0 ? R[u * kCwp + c] : 0.0;
        }
    }
    for (int j = 0; j < w; ++j) {
        const int p = j - 1;                     // the column to apply (columns before it are applied)
        if (warp < 2) {
            double *row = (warp == 0 ? Ld : R) + lane * kCwp;
            const bool in = warp == 0 ? lane > j && lane < w : lane < nr;
            double d = Ld[j * kCwp + j], v = 0.0;
            if (in) v = row[j];
            if (p >= 0) {
                const double lb = Ld[j * kCwp + p];
                d = sub_prod(d, lb, lb);
                if (in) v = sub_prod(v, row[p], lb);
            }
            if (!positive(d)) {
                d = 1.0;
                if (lane == 0) *bad = 1;
            }
            double q, dg, rl;
            if constexpr (RC) {
                dg = rl = rsqrt(d);
                q = v * rl;
            } else {
                const Pivot pv = pivot(d);
                q = pivot_div(v, pv);
                rl = pv.rl;
                dg = pv.l;
            }
            // Ld's column p and pivot are read by the other warp too: only column j is written
            if (in) row[j] = q;
            if (warp == 0 && lane == j) rlp[j] = rl;
            if (warp == 0 && lane == j) rlp[kCw + j] = dg;
        } else if (p >= 0) {                     // columns j + 1 .. w - 1
            const int left = w - 1 - j, nd = left * (left + 1) / 2, nn = left * nr;
#pragma unroll
            for (int k = 0; k < kCcGd; ++k) {
                if (kCcBulk * k + (bt & ~31) >= nd) break;
                const int i = pd[k] >> 8, c = pd[k] & 255;
                gd[k] = sub_prod(gd[k], Ld[i * kCwp + p], Ld[c * kCwp + p]);
                if (c == j + 1) Ld[i * kCwp + c] = gd[k];
            }
#pragma unroll
            for (int k = 0; k < kCcGr; ++k) {
                if (kCcBulk * k + (bt & ~31) >= nn) break;
                const int u = pr[k] >> 8, c = pr[k] & 255;
                gr[k] = sub_prod(gr[k], R[u * kCwp + p], Ld[c * kCwp + p]);
                if (c == j + 1) R[u * kCwp + c] = gr[k];
            }
        }
        panel_sync();
    }
    if (threadIdx.x < w) Ld[threadIdx.x * kCwp + threadIdx.x] = rlp[kCw + threadIdx.x];
    panel_sync();
}

// The matrix, packed lower row-major in g (order K), and its right-hand side:
// entry c of it is first(c) while the first panel runs, then zbuf[c].  On
// return out(i, x_i) has been called for every i of the solution (by the
// cluster's first block), and *bad is set there if a pivot was not positive.
// Every thread of the cluster calls it with the same K.
//
// OV (blocks of 512 threads): of a panel's trailing update only the next panel's
// 32 columns are awaited; the rest is left to the second half of the block, beside
// the next panel's columns, whose chain leaves half of the FP64 unit free.
// A block of columns keeps blocks of 256, two per SM: its clusters fill the
// device, and two chains on an SM overlap each other.
template <bool RC, bool OV, typename First, typename Out>
__device__ __forceinline__ void cluster_chol_solve(double *g, double *zbuf, int K, double *sm, int *bad,
                                                   First first, Out out) {
    constexpr int NT = OV ? 512 : 256, NW = NT / 32;
    __shared__ double rlp[2 * kCw];               // the panel's 1 / L_jj, and its diagonal
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank(), C = (int)cluster_blocks();
    const int NR = cc_rows(K, C);
    double *Ld = sm, *R = Ld + kCw * kCwp, *P = R + (size_t)NR * kCwp;
    const size_t panel = (size_t)(K + 1) * kCwp > 3u * kCcStage ? (size_t)(K + 1) * kCwp : 3u * kCcStage;
    double *z = P + panel, *rlv = z + K + kCw;    // first block: solution, reciprocals of the pivots
    auto at = [](int i, int j) { return (long long)i * (i + 1) / 2 + j; };
    // The trailing update by the panel before column j1 (P: its rows j1 .. K, row K
    // the right-hand side) of the columns from j1 + bfrom up to j1 + bto, in units of
    // RU rows x 32 columns dealt over the warps of the cluster.
    auto trail = [&](auto ru, int j1, int bfrom, int bto, int wid, int nw) {
        constexpr int RU = decltype(ru)::value;
        const int nb = K + 1 - j1;
        int unit = wid * C + rank;
        for (int b0 = bfrom; b0 < min(bto, K - j1); b0 += kCw) {
            const int groups = (nb - b0 + RU - 1) / RU;
            for (; unit < groups; unit += C * nw) {
                const int a0 = b0 + RU * unit, b = b0 + lane;     // rows and column, from j1
                const bool bin = b < K - j1;
                double acc[RU];
#pragma unroll
                for (int q = 0; q < RU; ++q) {
                    const int a = a0 + q;
                    acc[q] = 0.0;
                    if (bin && a < nb - 1 && b <= a) acc[q] = __ldcg(&g[at(j1 + a, j1 + b)]);
                    if (bin && a == nb - 1) acc[q] = j1 == kCw ? first(j1 + b) : __ldcg(&zbuf[j1 + b]);
                }
                const double *pb = P + (size_t)min(b, nb - 1) * kCwp;
                const double *pa[RU];
#pragma unroll
                for (int q = 0; q < RU; ++q) pa[q] = P + (size_t)min(a0 + q, nb - 1) * kCwp;
#pragma unroll 8
                for (int j = 0; j < kCw; ++j) {
                    const double lb = pb[j];
#pragma unroll
                    for (int q = 0; q < RU; ++q) acc[q] = sub_prod(acc[q], pa[q][j], lb);
                }
#pragma unroll
                for (int q = 0; q < RU; ++q) {
                    const int a = a0 + q;
                    if (bin && a < nb - 1 && b <= a) g[at(j1 + a, j1 + b)] = acc[q];
                    if (bin && a == nb - 1) zbuf[j1 + b] = acc[q];
                }
            }
            unit -= groups;
        }
    };
    for (int j0 = 0; j0 < K; j0 += kCw) {
        const int w = min(kCw, K - j0), j1 = j0 + w;
        const int nr = max(0, (K + 1 - j1 - rank + C - 1) / C);     // rows j1 + rank + C u
        for (int e = tid; e < w * kCw; e += NT) {
            const int i = e >> 5, j = e & 31;
            if (j <= i) Ld[i * kCwp + j] = __ldcg(&g[at(j0 + i, j0 + j)]);
        }
        for (int e = tid; e < nr * kCw; e += NT) {
            const int u = e >> 5, j = e & 31, i = j1 + rank + C * u;
            if (j < w)
                R[u * kCwp + j] = i < K ? __ldcg(&g[at(i, j0 + j)]) : j0 == 0 ? first(j) : __ldcg(&zbuf[j0 + j]);
        }
        __syncthreads();
        if (tid < 256) cc_panel<RC>(Ld, R, w, nr, rlp, bad);
        else if (OV && j0 > 0) trail(IntC<4>(), j0, kCw, K, warp - 8, 8);
        if constexpr (OV) __syncthreads();
        for (int e = tid; e < nr * kCw; e += NT) {
            const int u = e >> 5, j = e & 31, i = j1 + rank + C * u;
            if (j < w) {
                if (i < K) g[at(i, j0 + j)] = R[u * kCwp + j];
                else zbuf[j0 + j] = R[u * kCwp + j];
            }
        }
        if (rank == 0 && tid < w) rlv[j0 + tid] = rlp[tid];
        cluster_sync_all();
        // every block has its copy of the diagonal block: it can be replaced
        if (rank == 0)
            for (int e = tid; e < w * kCw; e += NT) {
                const int i = e >> 5, j = e & 31;
                if (j <= i) g[at(j0 + i, j0 + j)] = Ld[i * kCwp + j];
            }
        if (j1 >= K) break;
        const int nb = K + 1 - j1;
        for (int u0 = warp; u0 < nb; u0 += 8 * NW) {      // a warp per row, eight rows in flight
            double t[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = j1 + u0 + NW * q;
                t[q] = i < K ? __ldcg(&g[at(i, j0 + lane)]) : i == K ? __ldcg(&zbuf[j0 + lane]) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (u0 + NW * q < nb) P[(u0 + NW * q) * kCwp + lane] = t[q];
        }
        __syncthreads();
        if constexpr (OV) trail(IntC<2>(), j1, 0, kCw, warp, NW);
        else trail(IntC<4>(), j1, 0, K, warp, NW);
        cluster_sync_all();
    }
    if (rank != 0) return;
    // ---- backward solve, 32 rows at a time from the last ------------------
    // Stage of block q (buffer q % 3): tile D[j][i] = L[j0 + j][j0 + i] of its
    // diagonal block and tile U[j][i] = L[j0 + j][j0 - 32 + i] above it.
    __threadfence();
    __syncthreads();
    const int nblk = (K + kCw - 1) / kCw;
    auto stage = [&](int q, int t0, int tn) {
        if (q < 0) return;
        double *D = P + (size_t)(q % 3) * kCcStage, *U = D + kCw * kCwp;
        const int j0 = q * kCw, w = min(kCw, K - j0);
        for (int e = t0; e < w * kCw; e += tn) {
            const int j = e >> 5, i = e & 31;
            if (i <= j) D[j * kCwp + i] = __ldcg(&g[at(j0 + j, j0 + i)]);
            if (q > 0) U[j * kCwp + i] = __ldcg(&g[at(j0 + j, j0 - kCw + i)]);
        }
    };
    for (int i = tid; i < K; i += NT) z[i] = __ldcg(&zbuf[i]);
    stage(nblk - 1, tid, NT);
    stage(nblk - 2, tid, NT);
    __syncthreads();
    for (int q = nblk - 1; q >= 0; --q) {
        const int j0 = q * kCw, w = min(kCw, K - j0);
        const double *D = P + (size_t)(q % 3) * kCcStage, *U = D + kCw * kCwp;
        if (warp == 0) {
            double zi = lane < w ? z[j0 + lane] : 0.0;
            const double li = lane < w ? D[lane * kCwp + lane] : 1.0;
            const unsigned okm = __ballot_sync(0xffffffffu, divisor_ok(li));
#pragma unroll 4
            for (int j = w - 1; j >= 0; --j) {
                double zj = __shfl_sync(0xffffffffu, zi, j);
                const double l = D[j * kCwp + j], rl = rlv[j0 + j];
                if constexpr (RC) zj = zj * rl;
                else zj = quotient_rn(zj, __dmul_rn(zj, rl), l, rl, okm >> j & 1u);
                if (lane == j) zi = zj;
                if (lane < j) {
                    const double lji = D[j * kCwp + lane];
                    zi = sub_prod(zi, lji, zj);
                }
            }
            if (lane < w) z[j0 + lane] = zi;
        }
        __syncthreads();                          // this block's part of the solution; the rows above
        if (q == 0) break;                        // have received every later block
        if (warp == 0) {
            double zi = z[j0 - kCw + lane];
#pragma unroll 4
            for (int j = w - 1; j >= 0; --j) {
                const double lji = U[j * kCwp + lane];
                zi = sub_prod(zi, lji, z[j0 + j]);
            }
            z[j0 - kCw + lane] = zi;
            __syncwarp();
        } else {
            stage(q - 2, tid - 32, NT - 32);
            for (int i = tid - 32; i < j0 - kCw; i += NT - 32) {
                double zi = z[i];
#pragma unroll 8
                for (int j = w - 1; j >= 0; --j) {
                    const double lji = __ldcg(&g[at(j0 + j, i)]);
                    zi = sub_prod(zi, lji, z[j0 + j]);
                }
                z[i] = zi;
            }
        }
    }
    for (int i = tid; i < K; i += NT) out(i, z[i]);
}

}  // namespace rorbk
