// dense_rows.cuh -- row and column chains over a dense row-major A.
//
// A row's dot product with x is one fused multiply-add chain over its columns,
// so the parallelism of a dense pass is its rows: one lane per row, 32 rows per
// warp.  What bounds such a warp is either the chain itself (GB300: 4.7 cycles
// per FP32 link, 64 per FP64 link) or the bytes it keeps in flight; registers
// hold too few of the latter, so each warp runs a ring of stages in shared
// memory that it fills for itself by asynchronous 16-byte copies (cp.async),
// 256 bytes of each of its rows and the matching part of x per stage.  A row of
// a stage starts 272 bytes after the previous one: the lanes' 16-byte reads of
// their own rows meet no bank conflict.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace rorbk {

template <typename T, typename V>
struct DenseStage {
    static constexpr int cols = 256 / sizeof(V);                 // columns per stage
    static constexpr int pitch = 272;                            // bytes between rows
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
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T> struct Pack16;
template <> struct Pack16<float> { using type = float4; };
template <> struct Pack16<double> { using type = double2; };

// One warp: acc_l = sum over j ascending of A0[l * n + j] x[j] (one fused chain
// from 0) for the lanes l < rows.  ring: ST stages of DenseStage<T, V>::bytes.
// vec: every row starts on a 16-byte boundary (n * sizeof(V) % 16 == 0); else
// the rows are copied value by value.
template <typename T, typename V, int ST>
__device__ __forceinline__ T dense_chain(const V *__restrict__ A0, int rows, int n, const T *__restrict__ x,
                                         unsigned char *ring, bool vec) {
    using S = DenseStage<T, V>;
    constexpr int EP = 16 / sizeof(V);                            // values per 16 bytes
    const int lane = threadIdx.x & 31;
    const int nst = (n + S::cols - 1) / S::cols;
    const unsigned rb = smem_u32(ring);
    auto issue = [&](int k) {
        if (k < nst) {
            const unsigned sb = rb + (unsigned)(k % ST) * S::bytes;
            const int c0 = k * S::cols;
            if (vec) {
                const int ch = lane & 15, c = c0 + ch * EP;
                const int bytes = min(16, (n - c) * (int)sizeof(V));
                const V *src = A0 + (long long)(lane >> 4) * n + c;
                unsigned dst = sb + (lane >> 4) * S::pitch + ch * 16;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    if (2 * u + (lane >> 4) < rows && bytes > 0) cp_async16(dst, src, bytes);
                    src += 2LL * n;
                    dst += 2 * S::pitch;
                }
            } else {
                for (int u = 0; u < rows; ++u)
#pragma unroll
                    for (int q = 0; q < S::cols / 32; ++q) {
                        const int c = c0 + 32 * q + lane;
                        if (c < n)
                            cp_async_elem<sizeof(V)>(sb + u * S::pitch + (32 * q + lane) * (int)sizeof(V),
                                                     A0 + (long long)u * n + c);
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
    __syncwarp();                                     // the ring's earlier readers are done
#pragma unroll 1
    for (int k = 0; k < ST - 1; ++k) issue(k);
    T acc = T(0);
#pragma unroll 1
    for (int k = 0; k < nst; ++k) {
        cp_async_wait<ST - 2>();
        __syncwarp();                                 // stage k is there; stage k - 1 is free
        issue(k + ST - 1);
        const unsigned char *st = ring + (size_t)(k % ST) * S::bytes;
        const V *row = (const V *)(st + lane * S::pitch);
        const T *xs = (const T *)(st + 32 * S::pitch);
        if (k * S::cols + S::cols <= n) {
#pragma unroll 4
            for (int q = 0; q < S::cols / EP; ++q) {
                const typename Pack16<V>::type v = *(const typename Pack16<V>::type *)(row + q * EP);
                T xv[EP];
#pragma unroll
                for (int u = 0; u < EP; u += 16 / (int)sizeof(T)) {
                    const typename Pack16<T>::type t = *(const typename Pack16<T>::type *)(xs + q * EP + u);
                    xv[u] = t.x;
                    xv[u + 1] = t.y;
                    if constexpr (sizeof(T) == 4) { xv[u + 2] = t.z; xv[u + 3] = t.w; }
                }
                acc = Ar<T>::fma(wide<T>(v.x), xv[0], acc);
                acc = Ar<T>::fma(wide<T>(v.y), xv[1], acc);
                if constexpr (EP == 4) {
                    acc = Ar<T>::fma(wide<T>(v.z), xv[2], acc);
                    acc = Ar<T>::fma(wide<T>(v.w), xv[3], acc);
                }
            }
        } else {
            for (int j = 0; j < n - k * S::cols; ++j) acc = Ar<T>::fma(wide<T>(row[j]), xs[j], acc);
        }
    }
    cp_async_wait<0>();
    return acc;
}

// One thread: sum over a = 0 .. s-1 ascending of at(a) * y[a] (one fused chain
// from 0), the values read kAhead at a time while the chain runs over the
// previous ones.
template <typename T, typename At>
__device__ __forceinline__ T column_chain(int s, const T *y, At at) {
    constexpr int kAhead = 16;
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
