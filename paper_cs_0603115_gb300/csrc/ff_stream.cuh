// ff_stream.cuh -- one streaming kernel for every elementwise op.
//
// Each op reads NIN arrays and writes NOUT arrays of the same element type T
// (float2 for float-float values and packed operand pairs, double or float
// for the native baselines).  The body moves 16-byte vectors (two float2,
// two double, four float) with evict-first streaming loads and stores: every
// byte is touched once, so nothing is worth keeping in L1/L2.
//
// Bound by HBM.  A block takes one run of kBlock x U consecutive vectors of each
// array, loads them together and ends; the next block follows on the SM.  So the
// SM always holds blocks that load beside blocks that compute and store, and the
// blocks in flight cover a compact stretch of each array.  Against a grid of 2 to
// 4 resident blocks of 256 per SM that strode through the arrays with a software
// pipeline: mul of 2^28 values 943 -> 887 us (7.26 TB/s), div 944 -> 883, sqrt
// 640 -> 592, dot_backward 1285 -> 1201; div of 2^20 3.5 -> 3.2, dot_backward of
// 2^26 331 -> 303, add of 4096 1.61 -> 1.12.  Strided instead of consecutive
// vectors in such blocks: mul at 2^28 914.
//
// U by size: 1 while the vectors are no more than the resident threads, where a
// second vector only lengthens a thread's chain (div of 2^18 values 1.93 us, 2.15
// with 2); else 2 (sqrt at 2^22 7.1 us, 9.4 with 1; 3 and 4 within 2% of it from
// 2^24 on, slower on the operators with two inputs below).
//
// Alignment: device arrays are only required to be aligned to sizeof(T).
// If all arrays share the same offset modulo 16 bytes, a scalar head of
// `head` elements brings them to a 16-byte boundary and the remainder that
// does not fill a vector is a scalar tail; otherwise the whole range runs on
// scalar accesses (still coalesced).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "ff_core.cuh"
#include "ff_host.cuh"

namespace ffst {

constexpr int kBlock = 128;

template <typename T> struct Vec;
template <> struct Vec<float2> { using V = float4; static constexpr int E = 2; };
template <> struct Vec<double> { using V = double2; static constexpr int E = 2; };
template <> struct Vec<float>  { using V = float4; static constexpr int E = 4; };

template <typename T, int NIN, int NOUT>
struct Args {
    const T* in[NIN];
    T* out[NOUT];
    size_t n;      // elements
    int head;      // scalar elements before the first 16-byte boundary
};

// Split a 16-byte vector into its E values and join them back.  Explicit
// component moves, not a union: with a union the compiler scheduled the
// Add22 kernel measurably worse (about 6.2 instead of 7.1 TB/s on 2^28
// values at the same launch shape), the other operators were unaffected.
__device__ __forceinline__ void unpack(const float4& v, float2 (&e)[2])
{
    e[0] = make_float2(v.x, v.y);
    e[1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ float4 pack(const float2 (&e)[2]) { return make_float4(e[0].x, e[0].y, e[1].x, e[1].y); }
__device__ __forceinline__ void unpack(const double2& v, double (&e)[2])
{
    e[0] = v.x;
    e[1] = v.y;
}
__device__ __forceinline__ double2 pack(const double (&e)[2]) { return make_double2(e[0], e[1]); }
__device__ __forceinline__ void unpack(const float4& v, float (&e)[4])
{
    e[0] = v.x;
    e[1] = v.y;
    e[2] = v.z;
    e[3] = v.w;
}
__device__ __forceinline__ float4 pack(const float (&e)[4]) { return make_float4(e[0], e[1], e[2], e[3]); }

// An operator that reads memory itself takes the wait's zero into its address
// (see ffk::prior_kernel_done).
template <class Op>
__device__ __forceinline__ auto after_wait(Op& op, unsigned zero, int) -> decltype(op.after_wait(zero))
{
    op.after_wait(zero);
}
template <class Op>
__device__ __forceinline__ void after_wait(Op&, unsigned, long)
{
}

template <typename T, int NIN, int NOUT, class Op>
__device__ __forceinline__ void scalar_at(const Args<T, NIN, NOUT>& a, const Op& op, size_t i)
{
    T x[NIN];
    T y[NOUT];
#pragma unroll
    for (int k = 0; k < NIN; ++k) x[k] = a.in[k][i];
    op(x, y);
#pragma unroll
    for (int k = 0; k < NOUT; ++k) a.out[k][i] = y[k];
}

// Apply the op to the E values of one vector per input and store one vector
// per output at vector index j.
template <typename T, int NIN, int NOUT, class Op>
__device__ __forceinline__ void apply_vec(const Op& op, const typename Vec<T>::V (&x)[NIN],
                                          typename Vec<T>::V* const (&out)[NOUT], size_t j)
{
    constexpr int E = Vec<T>::E;
    T xe[NIN][E];
#pragma unroll
    for (int k = 0; k < NIN; ++k) unpack(x[k], xe[k]);
    T ye[NOUT][E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        T xs[NIN];
        T ys[NOUT];
#pragma unroll
        for (int k = 0; k < NIN; ++k) xs[k] = xe[k][e];
        op(xs, ys);
#pragma unroll
        for (int k = 0; k < NOUT; ++k) ye[k][e] = ys[k];
    }
#pragma unroll
    for (int k = 0; k < NOUT; ++k) __stcs(out[k] + j, pack(ye[k]));
}

// Vector path: elements [0, head) and the tail are scalar; the body is
// processed as 16-byte vectors, U consecutive runs of kBlock per block.
template <typename T, int NIN, int NOUT, class Op, int U>
__global__ void __launch_bounds__(kBlock) stream_vec(Args<T, NIN, NOUT> a, Op op)
{
    using V = typename Vec<T>::V;
    constexpr int E = Vec<T>::E;
    const unsigned zero = ffk::prior_kernel_done();
    after_wait(op, zero, 0);
    const size_t block = blockIdx.x + zero;
    const size_t head = static_cast<size_t>(a.head);
    const size_t nv = (a.n - head) / E;            // full vectors
    const size_t tail0 = head + nv * E;            // first tail element

    const V* in[NIN];
    V* out[NOUT];
#pragma unroll
    for (int k = 0; k < NIN; ++k) in[k] = reinterpret_cast<const V*>(a.in[k] + head);
#pragma unroll
    for (int k = 0; k < NOUT; ++k) out[k] = reinterpret_cast<V*>(a.out[k] + head);

    const size_t i = block * (kBlock * U) + threadIdx.x;
    if (i + (U - 1) * kBlock < nv) {
        V x[U][NIN];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < NIN; ++k) x[u][k] = __ldcs(in[k] + i + u * kBlock);
#pragma unroll
        for (int u = 0; u < U; ++u) apply_vec<T, NIN, NOUT>(op, x[u], out, i + u * kBlock);
    } else {
        for (size_t j = i; j < nv; j += kBlock) {
            V x[NIN];
#pragma unroll
            for (int k = 0; k < NIN; ++k) x[k] = __ldcs(in[k] + j);
            apply_vec<T, NIN, NOUT>(op, x, out, j);
        }
    }
    if (block == 0) {
        if (threadIdx.x < head) scalar_at(a, op, threadIdx.x);
        if (threadIdx.x < a.n - tail0) scalar_at(a, op, tail0 + threadIdx.x);
    }
}

// Scalar path for arrays whose offsets modulo 16 bytes differ.
template <typename T, int NIN, int NOUT, class Op, int U>
__global__ void __launch_bounds__(kBlock) stream_scalar(Args<T, NIN, NOUT> a, Op op)
{
    const unsigned zero = ffk::prior_kernel_done();
    after_wait(op, zero, 0);
    const size_t i = static_cast<size_t>(blockIdx.x + zero) * (kBlock * U) + threadIdx.x;
    if (i + (U - 1) * kBlock < a.n) {
        T x[U][NIN];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < NIN; ++k) x[u][k] = __ldcs(a.in[k] + i + u * kBlock);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            T y[NOUT];
            op(x[u], y);
#pragma unroll
            for (int k = 0; k < NOUT; ++k) __stcs(a.out[k] + i + u * kBlock, y[k]);
        }
    } else {
        for (size_t j = i; j < a.n; j += kBlock) scalar_at(a, op, j);
    }
}

template <typename T, int NIN, int NOUT, class Op, int U>
ff_status launch_vec(const Args<T, NIN, NOUT>& a, const Op& op, size_t nv, cudaStream_t s)
{
    const size_t blocks = (nv + kBlock * U - 1) / (kBlock * U);
    return ffh::launch_kernel(&stream_vec<T, NIN, NOUT, Op, U>, static_cast<unsigned>(blocks > 0 ? blocks : 1), kBlock, s,
                              a, op);
}

template <typename T, int NIN, int NOUT, class Op, int U>
ff_status launch_scalar(const Args<T, NIN, NOUT>& a, const Op& op, cudaStream_t s)
{
    const size_t blocks = (a.n + kBlock * U - 1) / (kBlock * U);
    return ffh::launch_kernel(&stream_scalar<T, NIN, NOUT, Op, U>, static_cast<unsigned>(blocks), kBlock, s, a, op);
}

// Host launcher: validates nothing (the caller did), picks the path and the
// vectors per thread, launches on `s`.
template <typename T, int NIN, int NOUT, class Op>
ff_status launch(Args<T, NIN, NOUT> a, Op op, cudaStream_t s)
{
    if (a.n == 0) return FF_OK;
    ffh::DeviceInfo di;
    ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    const size_t resident = static_cast<size_t>(di.sm_count) * static_cast<size_t>(di.max_threads_per_sm);
    constexpr int E = Vec<T>::E;
    // offset of each array modulo 16 bytes, in elements
    uintptr_t phase = reinterpret_cast<uintptr_t>(a.in[0]) & 15u;
    bool same = true;
    for (int k = 1; k < NIN; ++k) same &= ((reinterpret_cast<uintptr_t>(a.in[k]) & 15u) == phase);
    for (int k = 0; k < NOUT; ++k) same &= ((reinterpret_cast<uintptr_t>(a.out[k]) & 15u) == phase);
    if (same && (phase % sizeof(T)) == 0) {
        size_t head = phase ? (16u - phase) / sizeof(T) : 0;
        if (head > a.n) head = a.n;
        a.head = static_cast<int>(head);
        const size_t nv = (a.n - head) / E;
        return nv <= resident ? launch_vec<T, NIN, NOUT, Op, 1>(a, op, nv, s) : launch_vec<T, NIN, NOUT, Op, 2>(a, op, nv, s);
    }
    a.head = 0;   // half the bytes per access: twice as many in flight (sqrt of 2^27 values 409 -> 329 us)
    return a.n <= resident ? launch_scalar<T, NIN, NOUT, Op, 1>(a, op, s) : launch_scalar<T, NIN, NOUT, Op, 4>(a, op, s);
}

}  // namespace ffst
