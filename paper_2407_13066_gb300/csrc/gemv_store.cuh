// Decoding of the stored Fhat formats, shared by the per-frequency product
// kernels (gemv_kernels.cu, gemv_multi.cu).
#pragma once

#include "fftq.cuh"
#include "kernels.h"

namespace btt {

// ------------------------------------------------------ storage decoding
// Store<PREC>: one 16-byte unit of a Fhat row (VPL complex values).
// load_raw fetches the unit (evict-first; the split pair also its lo-plane
// twin at p + lo), decode turns it into FP32 complex values, and load does
// both.  Kernels that keep many units in flight hold raw units and decode
// late.
template <int PREC> struct Store;

template <> struct Store<P_F32> {
    using elem = float2;
    using acc = float;
    using raw = float4;
    static constexpr int VPL = 2;  // complex values per 16-byte load
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t)
    {
        return __ldcs(reinterpret_cast<const float4*>(p));
    }
    static __device__ __forceinline__ void decode(const raw& q, float2 (&f)[VPL])
    {
        f[0] = make_float2(q.x, q.y);
        f[1] = make_float2(q.z, q.w);
    }
    static __device__ __forceinline__ void load(const elem* p, float2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

template <> struct Store<P_F64> {
    using elem = double2;
    using acc = double;
    using raw = double2;
    static constexpr int VPL = 1;
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t) { return __ldcs(p); }
    static __device__ __forceinline__ void decode(const raw& q, double2 (&f)[VPL]) { f[0] = q; }
    static __device__ __forceinline__ void load(const elem* p, double2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

template <> struct Store<P_F16S> {
    using elem = __half2;
    using acc = float;
    using raw = uint4;
    static constexpr int VPL = 4;
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t)
    {
        return __ldcs(reinterpret_cast<const uint4*>(p));
    }
    static __device__ __forceinline__ void decode(const raw& q, float2 (&f)[VPL])
    {
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) f[i] = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
    }
    static __device__ __forceinline__ void load(const elem* p, float2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

template <> struct Store<P_BF16> {
    using elem = __nv_bfloat162;
    using acc = float;
    using raw = uint4;
    static constexpr int VPL = 4;
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t)
    {
        return __ldcs(reinterpret_cast<const uint4*>(p));
    }
    static __device__ __forceinline__ void decode(const raw& q, float2 (&f)[VPL])
    {
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) f[i] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
    }
    static __device__ __forceinline__ void load(const elem* p, float2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

// BF16 hi+lo split pair, stored as two planes of BF16 Fhat: hi at p, lo at
// p + lo (the same [w][s][ldm] layout each, so either plane is also a BF16
// operand of the tensor-core products).
struct SplitRaw {
    uint4 h, l;
};
template <> struct Store<P_BF16X2> {
    using elem = __nv_bfloat162;
    using acc = float;
    using raw = SplitRaw;
    static constexpr int VPL = 4;
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t lo)
    {
        return SplitRaw{__ldcs(reinterpret_cast<const uint4*>(p)), __ldcs(reinterpret_cast<const uint4*>(p + lo))};
    }
    static __device__ __forceinline__ void decode(const raw& q, float2 (&f)[VPL])
    {
        const unsigned h[4] = {q.h.x, q.h.y, q.h.z, q.h.w};
        const unsigned l[4] = {q.l.x, q.l.y, q.l.z, q.l.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h[i]));
            const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&l[i]));
            f[i] = make_float2(a.x + b.x, a.y + b.y);
        }
    }
    static __device__ __forceinline__ void load(const elem* p, float2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

template <> struct Store<P_FP8S> {
    using elem = __nv_fp8x2_storage_t;   // (Re, Im) E4M3 codes of Fhat / s_w
    using acc = float;
    using raw = uint4;
    static constexpr int VPL = 8;
    static __device__ __forceinline__ raw load_raw(const elem* p, int64_t)
    {
        return __ldcs(reinterpret_cast<const uint4*>(p));
    }
    static __device__ __forceinline__ void decode(const raw& q, float2 (&f)[VPL])
    {
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __half2 lo = __half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w[i] & 0xFFFFu), __NV_E4M3));
            const __half2 hi = __half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w[i] >> 16), __NV_E4M3));
            f[2 * i] = __half22float2(lo);
            f[2 * i + 1] = __half22float2(hi);
        }
    }
    static __device__ __forceinline__ void load(const elem* p, float2 (&f)[VPL], int64_t lo) { decode(load_raw(p, lo), f); }
};

// acc += a * b
template <typename V> __device__ __forceinline__ void cfma(V& acc, V a, V b)
{
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}
// acc += conj(a) * b
template <typename V> __device__ __forceinline__ void cfma_conj(V& acc, V a, V b)
{
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(-a.y, b.x, acc.y);
}

// Sums v[0..CNT) over the 32 lanes.  While the count is even a lane sends
// half of its values to its partner and keeps the sums of the other half;
// `base` is the index of the first value it ends with.  Adds the same pairs
// in the same tree as a butterfly over all values, with a fifth of the
// shuffles at CNT = 64.  Returns the number of values a lane ends with;
// lanes that differ only in `dup` bits hold the same ones.
template <int CNT, int O> struct LaneSum {
    static constexpr bool kHalve = CNT % 2 == 0;
    static constexpr int kNext = kHalve ? CNT / 2 : CNT;
    static constexpr int kLeft = LaneSum<kNext, O / 2>::kLeft;
    static constexpr int kDup = (kHalve ? 0 : O) | LaneSum<kNext, O / 2>::kDup;
    template <typename T> static __device__ __forceinline__ void run(T* v, int lane, int& base)
    {
        if constexpr (kHalve) {
            const bool up = lane & O;
#pragma unroll
            for (int i = 0; i < kNext; ++i) {
                const T send = up ? v[i] : v[i + kNext], keep = up ? v[i + kNext] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
            }
            base += up ? kNext : 0;
        } else {
#pragma unroll
            for (int i = 0; i < CNT; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], O);
        }
        LaneSum<kNext, O / 2>::run(v, lane, base);
    }
};
template <int CNT> struct LaneSum<CNT, 0> {
    static constexpr int kLeft = CNT;
    static constexpr int kDup = 0;
    template <typename T> static __device__ __forceinline__ void run(T*, int, int&) {}
};

// Element offset of the lo plane of a split-pair Fhat (0 for other formats).
inline int64_t lo_plane(int prec, int n_freq, int N_d, int ldm)
{
    return prec == P_BF16X2 ? (int64_t)n_freq * N_d * ldm : 0;
}

}  // namespace btt
