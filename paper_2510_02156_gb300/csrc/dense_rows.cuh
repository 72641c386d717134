// dense_rows.cuh -- row and column chains over a dense row-major A.
//
// A row's dot product with x is one fused multiply-add chain over its columns,
// so the parallelism of a dense pass is its rows: one lane per row, 32 rows per
// warp.  What bounds such a warp is either the chain itself (GB300: 4.7 cycles
// per FP32 link, 64 per FP64 link) or the bytes it keeps in flight.  Registers
// hold too few of the latter, so the rows go through a ring of stages in shared
// memory, RB bytes of each row and the matching part of x per stage, filled by
// asynchronous 16-byte copies.  A second warp issues the copies: the chain's warp
// is left with the reads of its stage, one pack of values ahead of the chain
// (with the copies in its own instruction stream an FP32 link took 14 cycles and
// an FP64 link 88).  A row of a stage starts RB + 16 bytes after the previous
// one: the lanes' 16-byte reads of their own rows meet no bank conflict.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace rorbk {

template <typename T, typename V, int RB>
struct DenseStage {
    static constexpr int cols = RB / sizeof(V);                  // columns per stage
    static constexpr int pitch = RB + 16;                        // bytes between rows
    static constexpr int bytes = 32 * pitch + cols * (int)sizeof(T);
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, int bytes) {   // the rest of 16 is zeroed
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_elem(unsigned dst, const void *src) {
    static_assert(N == 4 || N == 8, "element copies");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(N) : "memory");
}
// The same with an L2 eviction policy: lines that are the first to be evicted.
__device__ __forceinline__ unsigned long long l2_stream_policy() {
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, int bytes, unsigned long long pol) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(dst), "l"(src), "r"(bytes),
                 "l"(pol)
                 : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_elem(unsigned dst, const void *src, unsigned long long pol) {
    static_assert(N == 4 || N == 8, "element copies");
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(N), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T> struct Pack16;
template <> struct Pack16<float> { using type = float4; };
template <> struct Pack16<double> { using type = double2; };

// A pair of warps: acc_l = sum over j ascending of A0[l * n + j] x[j] (one fused
// chain from 0) for the lanes l < rows, in the warp that calls dense_sum; the
// other warp calls dense_copy for the same rows.  ring: ST stages of
// DenseStage<T, V, RB>::bytes.  vec: every row starts on a 16-byte boundary
// (n * sizeof(V) % 16 == 0); else the rows are copied value by value.  STREAM: A's
// lines are the first that L2 evicts.  The pair meets at named barrier `bar` once
// per stage: behind it stage k has landed and stage k - 1 is free.
__device__ __forceinline__ void pair_sync(int bar) {
    __syncwarp();
    switch (bar) {                                    // an immediate barrier number
        case 1: asm volatile("bar.sync 1, 64;" ::: "memory"); break;
        case 2: asm volatile("bar.sync 2, 64;" ::: "memory"); break;
        case 3: asm volatile("bar.sync 3, 64;" ::: "memory"); break;
        case 4: asm volatile("bar.sync 4, 64;" ::: "memory"); break;
        case 5: asm volatile("bar.sync 5, 64;" ::: "memory"); break;
        case 6: asm volatile("bar.sync 6, 64;" ::: "memory"); break;
        case 7: asm volatile("bar.sync 7, 64;" ::: "memory"); break;
        default: asm volatile("bar.sync 8, 64;" ::: "memory"); break;
    }
}

template <typename T, typename V, int RB, int ST, bool STREAM = false>
__device__ __forceinline__ void dense_copy(const V *__restrict__ A0, int rows, int n, const T *__restrict__ x,
                                           unsigned char *ring, bool vec, int bar) {
    using S = DenseStage<T, V, RB>;
    constexpr int EP = 16 / sizeof(V);                            // values per 16 bytes
    constexpr int RP = 32 / (RB / 16);                            // rows per copy instruction (1 or 2)
    const int lane = threadIdx.x & 31;
    const int nst = (n + S::cols - 1) / S::cols;
    {
        const unsigned rb = smem_u32(ring);
        unsigned long long pol = 0;
        if constexpr (STREAM) pol = l2_stream_policy();
        const int ch = lane % (RB / 16), u0 = lane / (RB / 16);
        auto issue = [&](int k) {
            if (k < nst) {
                const unsigned sb = rb + (unsigned)(k % ST) * S::bytes;
                const int c0 = k * S::cols;
                if (vec) {
                    const int c = c0 + ch * EP, bytes = min(16, (n - c) * (int)sizeof(V));
                    const V *src = A0 + (long long)u0 * n + c;
                    unsigned dst = sb + u0 * S::pitch + ch * 16;
#pragma unroll
                    for (int u = 0; u < 32; u += RP) {
                        if (u + u0 < rows && bytes > 0) {
                            if constexpr (STREAM) cp_async16(dst, src, bytes, pol);
                            else cp_async16(dst, src, bytes);
                        }
                        src += (long long)RP * n;
                        dst += RP * S::pitch;
                    }
                } else {
                    for (int u = 0; u < rows; ++u)
#pragma unroll
                        for (int q = 0; q < S::cols / 32; ++q) {
                            const int c = c0 + 32 * q + lane;
                            const unsigned d = sb + u * S::pitch + (32 * q + lane) * (int)sizeof(V);
                            if (c < n) {
                                if constexpr (STREAM) cp_async_elem<sizeof(V)>(d, A0 + (long long)u * n + c, pol);
                                else cp_async_elem<sizeof(V)>(d, A0 + (long long)u * n + c);
                            }
                        }
                }
#pragma unroll
                for (int q = 0; q < S::cols / 32; ++q) {
                    const int c = c0 + 32 * q + lane;
                    if (c < n) cp_async_elem<sizeof(T)>(sb + 32 * S::pitch + (32 * q + lane) * (int)sizeof(T), x + c);
                }
            }
            cp_async_commit();
        };
#pragma unroll 1
        for (int k = 0; k < ST - 1; ++k) issue(k);
#pragma unroll 1
        for (int k = 0; k < nst; ++k) {
            cp_async_wait<ST - 2>();
            pair_sync(bar);
            issue(k + ST - 1);
        }
        cp_async_wait<0>();
    }
    pair_sync(bar);                                   // the ring is free for the next rows
}

template <typename T, typename V, int RB, int ST>
__device__ __forceinline__ T dense_sum(int n, const unsigned char *ring, int bar) {
    using S = DenseStage<T, V, RB>;
    constexpr int EP = 16 / sizeof(V);
    const int lane = threadIdx.x & 31;
    const int nst = (n + S::cols - 1) / S::cols;
    T acc = T(0);
    {
        constexpr int GP = 4;                                     // packs per group
        constexpr int NG = RB / 16 / GP;
#pragma unroll 1
        for (int k = 0; k < nst; ++k) {
            pair_sync(bar);
            const unsigned char *st = ring + (size_t)(k % ST) * S::bytes;
            const V *row = (const V *)(st + lane * S::pitch);
            const T *xs = (const T *)(st + 32 * S::pitch);
            if (k * S::cols + S::cols <= n) {
                V v[2][GP * EP];
                T xv[2][GP * EP];
                auto fetch = [&](int g, V *vd, T *xd) {
#pragma unroll
                    for (int q = 0; q < GP; ++q) {
                        const typename Pack16<V>::type t = *(const typename Pack16<V>::type *)(row + (g * GP + q) * EP);
                        vd[q * EP] = t.x;
                        vd[q * EP + 1] = t.y;
                        if constexpr (EP == 4) { vd[q * EP + 2] = t.z; vd[q * EP + 3] = t.w; }
                    }
#pragma unroll
                    for (int q = 0; q < GP * EP; q += 16 / (int)sizeof(T)) {
                        const typename Pack16<T>::type t = *(const typename Pack16<T>::type *)(xs + g * GP * EP + q);
                        xd[q] = t.x;
                        xd[q + 1] = t.y;
                        if constexpr (sizeof(T) == 4) { xd[q + 2] = t.z; xd[q + 3] = t.w; }
                    }
                };
                fetch(0, v[0], xv[0]);
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    if (g + 1 < NG) fetch(g + 1, v[(g + 1) & 1], xv[(g + 1) & 1]);
#pragma unroll
                    for (int q = 0; q < GP * EP; ++q) acc = Ar<T>::fma(wide<T>(v[g & 1][q]), xv[g & 1][q], acc);
                }
            } else {
                for (int j = 0; j < n - k * S::cols; ++j) acc = Ar<T>::fma(wide<T>(row[j]), xs[j], acc);
            }
        }
    }
    pair_sync(bar);
    return acc;
}

// One thread: sum over a = 0 .. s-1 ascending of at(a) * y[a] (one fused chain
// from 0), the values read kAhead at a time while the chain runs over the
// previous ones: 24 FP64 links last 1,536 cycles, 64 FP32 links about 300.
template <typename T, typename At>
__device__ __forceinline__ T column_chain(int s, const T *y, At at) {
    constexpr int kAhead = sizeof(T) == 8 ? 24 : 64;
    T acc = T(0), nx[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) nx[u] = u < s ? at(u) : T(0);
#pragma unroll 1
    for (int a = 0; a < s; a += kAhead) {
        T v[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            v[u] = nx[u];
            nx[u] = a + kAhead + u < s ? at(a + kAhead + u) : T(0);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (a + u < s) acc = Ar<T>::fma(v[u], y[a + u], acc);
    }
    return acc;
}

}  // namespace rorbk
