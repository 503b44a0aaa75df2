// Setup transform (Alg. 1) in FP64: every first-column series padded to
// 2 N_t, transformed and stored frequency-major in the storage format.
//
// Bound by the FP64 units (GB300: two FP64 lanes per SM and clock, a hundredth
// of what the memory could feed), so the transform is arranged to spend the
// fewest FP64 instructions:
//  * the padding half is never computed: even frequencies are the N_t-point
//    transform of the samples, odd ones that of the samples times w_L^n;
//  * N_t is split into its prime powers, whose transforms combine without
//    twiddles (prime-factor map: n = sum n_i N / N_i, frequency k at digits
//    k mod N_i); twiddles remain only inside a prime power of several passes;
//  * odd radices share their cosine sums between outputs q and R - q, and
//    the unpack's 1/2 rides in the inputs (an exact scaling).
// Two real columns form one complex sequence, as everywhere.  360 x 100 x 4000
// in FP32: 14.6 -> 8.6 ms against the mixed-radix kernel of fft_kernels.cu
// (FP64 pipe 78% -> 83% busy); btt_create, FP32 / FP16 / split pair: 15.6 / 34.5 /
// 17.2 -> 9.7 / 22.9 / 11.3 ms there, 14.7 / 30.3 / 15.8 -> 10.1 / 21.3 / 11.3 ms at
// 1000 x 100 x 1000, 12.6 -> 11.6 ms (FP32) at 2048 x 50 x 1000, where one prime
// power takes four passes with twiddles.
#include "fft.cuh"
#include "kernels.h"

namespace btt {
namespace setup {

constexpr int NT = 256;

__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 mul(double2 a, double2 w)
{
    return make_double2(fma(-a.y, w.y, a.x * w.x), fma(a.y, w.x, a.x * w.y));
}
// tile element i of n
__device__ __forceinline__ double2 get(const double2* buf, int i, int n)
{
    return BTT_IN(i, n, CK_FFT_SMEM) ? buf[i] : make_double2(0., 0.);
}
__device__ __forceinline__ void put(double2* buf, int i, int n, double2 v)
{
    if (BTT_IN(i, n, CK_FFT_SMEM)) buf[i] = v;
}
// a - i b and a + i b
__device__ __forceinline__ double2 sub_i(double2 a, double2 b) { return make_double2(a.x + b.y, a.y - b.x); }
__device__ __forceinline__ double2 add_i(double2 a, double2 b) { return make_double2(a.x - b.y, a.y + b.x); }

template <int R> __device__ __forceinline__ void dft_fwd(double2* v);

template <int R> __device__ __forceinline__ void dft_odd_fwd(double2* v)
{
    constexpr int H = (R - 1) / 2;
    double2 a[H], b[H];
    const double2 v0 = v[0];
    double2 y0 = v0;
#pragma unroll
    for (int p = 1; p <= H; ++p) {
        a[p - 1] = add(v[p], v[R - p]);
        b[p - 1] = sub(v[p], v[R - p]);
        y0 = add(y0, a[p - 1]);
    }
    v[0] = y0;
#pragma unroll
    for (int q = 1; q <= H; ++q) {
        double2 t = v0, u = make_double2(0., 0.);
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            const double c = RootTable<R>::c((p * q) % R), s = RootTable<R>::s((p * q) % R);
            t.x = fma(a[p - 1].x, c, t.x);
            t.y = fma(a[p - 1].y, c, t.y);
            u.x = p == 1 ? b[0].x * s : fma(b[p - 1].x, s, u.x);
            u.y = p == 1 ? b[0].y * s : fma(b[p - 1].y, s, u.y);
        }
        v[q] = sub_i(t, u);
        v[R - q] = add_i(t, u);
    }
}

template <int R> __device__ __forceinline__ void dft_fwd(double2* v)
{
    if constexpr (R == 2) {
        const double2 a = v[0];
        v[0] = add(a, v[1]);
        v[1] = sub(a, v[1]);
    } else if constexpr (R == 4) {
        const double2 s = add(v[0], v[2]), d = sub(v[0], v[2]), e = add(v[1], v[3]), f = sub(v[1], v[3]);
        v[0] = add(s, e);
        v[2] = sub(s, e);
        v[1] = sub_i(d, f);
        v[3] = add_i(d, f);
    } else if constexpr (R == 8) {
        const double h = 0.70710678118654752440084436210485;
        double2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft_fwd<4>(e);
        dft_fwd<4>(o);
        const double2 o1 = make_double2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
        const double2 o3 = make_double2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
        v[0] = add(e[0], o[0]);
        v[4] = sub(e[0], o[0]);
        v[1] = add(e[1], o1);
        v[5] = sub(e[1], o1);
        v[2] = sub_i(e[2], o[2]);
        v[6] = add_i(e[2], o[2]);
        v[3] = add(e[3], o3);
        v[7] = sub(e[3], o3);
    } else if constexpr (R == 9) {   // 3 x 3, twiddles w_9^1, w_9^2, w_9^4
        const double2 w1 = make_double2(0.76604444311897803520239265055542, -0.64278760968653932632264340990726);
        const double2 w2 = make_double2(0.17364817766693034885171662676931, -0.98480775301220805936674302458952);
        const double2 w4 = make_double2(-0.93969262078590838405410927732473, -0.34202014332566873304409961468226);
        double2 t[3][3];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            double2 u[3] = {v[n2], v[3 + n2], v[6 + n2]};
            dft_odd_fwd<3>(u);
            t[0][n2] = u[0];
            t[1][n2] = n2 == 0 ? u[1] : mul(u[1], n2 == 1 ? w1 : w2);
            t[2][n2] = n2 == 0 ? u[2] : mul(u[2], n2 == 1 ? w2 : w4);
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            dft_odd_fwd<3>(t[k1]);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[k1][k2];
        }
    } else {
        dft_odd_fwd<R>(v);
    }
}

// One in-place pass of radix R over both halves: elements `step` apart,
// S sub-positions of I points each (S > 1: twiddles w_{S R}^{n1 k}).
template <int R>
__device__ __forceinline__ void pass(double2* buf, int total, int S, int I, int wcl, int tstep,
                                     const double2* __restrict__ tw)
{
    const int SI = S * I, nb = (total / R) << wcl, step = SI << wcl;
    for (int b = threadIdx.x; b < nb; b += NT) {
        const int c = b & ((1 << wcl) - 1), j = b >> wcl;
        const int hi = j / SI, lo = j - hi * SI;
        const int at = ((hi * R * SI + lo) << wcl) + c;
        double2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = get(buf, at + i * step, total << wcl);
        dft_fwd<R>(v);
        if (S > 1) {
            const int n1 = lo / I;
            if (n1)
#pragma unroll
                for (int k = 1; k < R; ++k)
                    if (BTT_IN(n1 * k * tstep, S * R * tstep, CK_FFT_TABLE)) v[k] = mul(v[k], __ldg(tw + n1 * k * tstep));
        }
#pragma unroll
        for (int i = 0; i < R; ++i) put(buf, at + i * step, total << wcl, v[i]);
    }
    __syncthreads();
}

__device__ __forceinline__ void passes(double2* buf, int total, const SetupPlan& plan, int wcl,
                                       const double2* __restrict__ tw)
{
    for (int p = 0; p < plan.np; ++p) {
        const int S = plan.S[p], I = plan.I[p], ts = plan.tstep[p];
        switch (plan.radix[p]) {
            case 2: pass<2>(buf, total, S, I, wcl, ts, tw); break;
            case 3: pass<3>(buf, total, S, I, wcl, ts, tw); break;
            case 4: pass<4>(buf, total, S, I, wcl, ts, tw); break;
            case 5: pass<5>(buf, total, S, I, wcl, ts, tw); break;
            case 7: pass<7>(buf, total, S, I, wcl, ts, tw); break;
            case 8: pass<8>(buf, total, S, I, wcl, ts, tw); break;
            default: pass<9>(buf, total, S, I, wcl, ts, tw); break;
        }
    }
}

template <int PREC>
__global__ void __launch_bounds__(NT, 2)
k_create_pf(const double* __restrict__ blk, int64_t ldb, int ncols, int64_t col_base, int N_d, int N_m, int ldm,
            SetupPlan plan, int wcl, const double2* __restrict__ tw, const int* __restrict__ tab,
            void* __restrict__ fhat, const float* __restrict__ scales, unsigned long long* __restrict__ maxbits,
            int find_max)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = plan.N, Wc = 1 << wcl, L = 2 * N;
    double2* buf = reinterpret_cast<double2*>(smem_raw);   // [2][N][Wc]: even, odd frequencies
    unsigned long long* smax = reinterpret_cast<unsigned long long*>(buf + ((size_t)L << wcl));
    unsigned short* in = reinterpret_cast<unsigned short*>(smax + (find_max ? N + 1 : 0));
    unsigned short* out = in + N;
    for (int i = threadIdx.x; i < N; i += NT) {
        in[i] = (unsigned short)__ldg(tab + i);
        out[i] = (unsigned short)__ldg(tab + N + i);
    }
    if (find_max)
        for (int i = threadIdx.x; i <= N; i += NT) smax[i] = 0ull;
    const int c = threadIdx.x & (Wc - 1);
    const int ntiles = (ncols + 2 * Wc - 1) / (2 * Wc);
    const bool vec = (ldb & 1) == 0 && (reinterpret_cast<uintptr_t>(blk) & 15) == 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        __syncthreads();   // tables ready; the tile before is stored
        const int col = tile * 2 * Wc + 2 * c;
        const bool both = col + 1 < ncols, one = col < ncols;
        constexpr int U = 4;   // rows requested together
        for (int n0 = threadIdx.x >> wcl; n0 < N; n0 += U * (NT >> wcl)) {
            double2 z[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int n = n0 + u * (NT >> wcl);
                z[u] = make_double2(0., 0.);
                if (n >= N) continue;
                const double* p = blk + (int64_t)n * ldb + col;
                if (vec && both) z[u] = __ldcs(reinterpret_cast<const double2*>(p));
                else if (one) z[u] = make_double2(__ldcs(p), both ? __ldcs(p + 1) : 0.);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int n = n0 + u * (NT >> wcl);
                if (n >= N) break;
                const double2 w = __ldg(tw + n), h = make_double2(0.5 * z[u].x, 0.5 * z[u].y);
                const int at = ((int)in[n] << wcl) + c;
                put(buf, at, N << wcl, h);
                put(buf + (N << wcl), at, N << wcl, mul(h, w));
            }
        }
        __syncthreads();
        passes(buf, L, plan, wcl, tw);
        // where this thread's two columns go
        const unsigned g0 = (unsigned)(col_base + col);
        const unsigned s0 = one ? g0 / (unsigned)N_m : 0u, l0 = g0 - s0 * (unsigned)N_m;
        const bool wrap = l0 + 1 == (unsigned)N_m;   // the second column starts the next row of Fhat
        const int64_t o0 = (int64_t)s0 * ldm + l0, o1 = wrap ? (int64_t)(s0 + 1) * ldm : o0 + 1;
        const bool pairs = both && !wrap && (l0 & 1) == 0;
        for (int i0 = threadIdx.x >> wcl; i0 - (int)(threadIdx.x >> wcl) <= N; i0 += NT >> wcl) {
            const int w = i0, j = w >> 1;
            double2 a = make_double2(0., 0.), d = a;
            if (w <= N) {
                // Z[w] and Z[L - w] (halved): even w = 2 j, partner N - j; odd
                // w = 2 j + 1, partner N - 1 - j
                const double2* half = buf + ((w & 1) ? (N << wcl) : 0);
                const int jj = w & 1 ? N - 1 - j : (j ? N - j : 0);
                const double2 z = get(half, ((int)out[j] << wcl) + c, N << wcl);
                const double2 zc = get(half, ((int)out[jj] << wcl) + c, N << wcl);
                a = make_double2(z.x + zc.x, z.y - zc.y);
                d = make_double2(z.y + zc.y, zc.x - z.x);
            }
            if ((PREC == P_F16S || PREC == P_FP8S) && find_max) {
                // the lanes of a row first, then one shared maximum per row;
                // as bits, in the order of the magnitudes with NaN on top: an
                // entry without a finite part leaves the slice at scale 1
                auto bits = [](double2 z) { return (unsigned long long)__double_as_longlong(fmax(fabs(z.x), fabs(z.y))); };
                unsigned long long m = one && w <= N ? bits(a) : 0ull;
                if (both && w <= N) m = max(m, bits(d));
                for (int o = Wc / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (c == 0 && w <= N) atomicMax(&smax[w], m);
                continue;
            }
            if (w > N || !one) continue;
            if (!BTT_IN(o0, (int64_t)N_d * ldm, CK_FFT_STORE) || (both && !BTT_IN(o1, (int64_t)N_d * ldm, CK_FFT_STORE)))
                continue;
            const int64_t row = (int64_t)w * N_d * ldm;
            if constexpr (PREC == P_F64) {
                double2* f = reinterpret_cast<double2*>(fhat) + row;
                f[o0] = a;
                if (both) f[o1] = d;
            } else if constexpr (PREC == P_F32) {
                float2* f = reinterpret_cast<float2*>(fhat) + row;
                const float2 x = make_float2((float)a.x, (float)a.y), y = make_float2((float)d.x, (float)d.y);
                if (pairs) {
                    *reinterpret_cast<float4*>(f + o0) = make_float4(x.x, x.y, y.x, y.y);
                } else {
                    f[o0] = x;
                    if (both) f[o1] = y;
                }
            } else if constexpr (PREC == P_BF16 || PREC == P_BF16X2) {
                // hi = bf16(fp32(z)); split pairs: lo = bf16(fp32(z - hi)) on a second plane
                __nv_bfloat162* f = reinterpret_cast<__nv_bfloat162*>(fhat) + row;
                const __nv_bfloat162 x = __floats2bfloat162_rn((float)a.x, (float)a.y);
                const __nv_bfloat162 y = __floats2bfloat162_rn((float)d.x, (float)d.y);
                f[o0] = x;
                if (both) f[o1] = y;
                if constexpr (PREC == P_BF16X2) {
                    f += (int64_t)(N + 1) * N_d * ldm;
                    const float2 xf = __bfloat1622float2(x), yf = __bfloat1622float2(y);
                    f[o0] = __floats2bfloat162_rn((float)(a.x - (double)xf.x), (float)(a.y - (double)xf.y));
                    if (both) f[o1] = __floats2bfloat162_rn((float)(d.x - (double)yf.x), (float)(d.y - (double)yf.y));
                }
            } else if constexpr (PREC == P_F16S) {
                __half2* f = reinterpret_cast<__half2*>(fhat) + row;
                const double s_w = (double)scales[w];
                f[o0] = __floats2half2_rn((float)(a.x / s_w), (float)(a.y / s_w));
                if (both) f[o1] = __floats2half2_rn((float)(d.x / s_w), (float)(d.y / s_w));
            } else {   // P_FP8S: E4M3, round to nearest even, saturating
                __nv_fp8x2_storage_t* f = reinterpret_cast<__nv_fp8x2_storage_t*>(fhat) + row;
                const double s_w = (double)scales[w];
                f[o0] = __nv_cvt_float2_to_fp8x2(make_float2((float)(a.x / s_w), (float)(a.y / s_w)), __NV_SATFINITE,
                                                 __NV_E4M3);
                if (both)
                    f[o1] = __nv_cvt_float2_to_fp8x2(make_float2((float)(d.x / s_w), (float)(d.y / s_w)),
                                                     __NV_SATFINITE, __NV_E4M3);
            }
        }
    }
    if (find_max) {
        __syncthreads();
        for (int i = threadIdx.x; i <= N; i += NT)
            if (smax[i]) atomicMax(&maxbits[i], smax[i]);
    }
}

// ------------------------------------------------ FP64 vector transforms
// The transforms of BTT_F64 operators on the same passes.  The inverse runs
// them on conjugates (IDFT(X) = conj DFT(conj X)) of both halves.  Against the
// mixed-radix kernels of fft_kernels.cu (us, one vector; input / inverse of
// N_m columns, averaged with N_d, and middle step of N_d columns):
//   1000 x 100 x 1000  131 / 125 / 88 -> 82 / 86 / 62
//   420 x 37 x 3001    131 / 124 / 44 -> 75 / 73 / 29
//   5000 x 10 x 200    230 / 219 / 441 -> 140 / 160 / 307
// At 64 x 8 x 32 they are latency (a warp's FP64 instruction occupies the
// pipe for 16 clocks): 14.4 / 14.5 / 24 -> 12.3 / 12.3 / 18.6 with event timers.

struct Tables {   // positions of sample n and of frequency k, in shared memory
    unsigned short *in, *out;
    __device__ __forceinline__ Tables(unsigned char* at, int N, const int* __restrict__ tab)
    {
        in = reinterpret_cast<unsigned short*>(at);
        out = in + N;
        for (int i = threadIdx.x; i < N; i += NT) {
            in[i] = (unsigned short)__ldg(tab + i);
            out[i] = (unsigned short)__ldg(tab + N + i);
        }
    }
};

// Rows w = 2 j + odd <= N of one half (values halved) to X.
__device__ __forceinline__ void store_half(const double2* half, int odd, int N, int wcl, const unsigned short* out,
                                           double2* X, int64_t ldx, int col, int ncols)
{
    const int c = threadIdx.x & ((1 << wcl) - 1);
    if (col >= ncols) return;
    for (int j = threadIdx.x >> wcl; 2 * j + odd <= N; j += NT >> wcl) {
        const double2 z = get(half, ((int)out[j] << wcl) + c, N << wcl);
        const double2 zc = get(half, ((int)out[odd ? N - 1 - j : (j ? N - j : 0)] << wcl) + c, N << wcl);
        double2* o = X + (int64_t)(2 * j + odd) * ldx + col;
        o[0] = make_double2(z.x + zc.x, z.y - zc.y);
        if (col + 1 < ncols) o[1] = make_double2(z.y + zc.y, zc.x - z.x);
    }
}

// Conjugates of Z[w] = A + i B and Z[L - w] of every row to their halves.
__device__ __forceinline__ void load_conj(double2* buf, int N, int wcl, const unsigned short* in,
                                          const double2* __restrict__ X, int64_t ldx, int col, int ncols)
{
    const int c = threadIdx.x & ((1 << wcl) - 1);
    for (int w = threadIdx.x >> wcl; w <= N; w += NT >> wcl) {
        double2 a = make_double2(0., 0.), b = a;
        if (col < ncols) a = X[(int64_t)w * ldx + col];
        if (col + 1 < ncols) b = X[(int64_t)w * ldx + col + 1];
        if (w == 0 || w == N) a.y = b.y = 0.;   // real bins
        const int j = w >> 1, jj = w & 1 ? N - 1 - j : (j ? N - j : 0);
        double2* half = buf + (w & 1 ? (N << wcl) : 0);
        put(half, ((int)in[j] << wcl) + c, N << wcl, make_double2(a.x - b.y, -(a.y + b.x)));
        if (jj != j) put(half, ((int)in[jj] << wcl) + c, N << wcl, make_double2(a.x + b.y, a.y - b.x));
    }
}

// blockIdx.z: the half (even or odd frequencies) of this CTA, so that a few
// columns' FP64 work spreads over twice the SMs; the samples are read twice.
__global__ void __launch_bounds__(NT, 2)
k_rfft_pf(const double* __restrict__ x, int64_t ldx, int64_t bsx, int ncols, double2* __restrict__ X, int64_t ldo,
          int64_t bso, SetupPlan plan, int wcl, const double2* __restrict__ tw, const int* __restrict__ tab,
          const double* const* __restrict__ xptr)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = plan.N, odd = blockIdx.z, c = threadIdx.x & ((1 << wcl) - 1);
    const int col = (int)(blockIdx.x << (wcl + 1)) + 2 * c;
    const int64_t b = blockIdx.y;
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const Tables t(smem_raw + ((size_t)N << wcl) * sizeof(double2), N, tab);
    const double* xb = (xptr ? xptr[b] : x + b * bsx) + col;
    __syncthreads();
    for (int n = threadIdx.x >> wcl; n < N; n += NT >> wcl) {
        double2 z = make_double2(0., 0.);
        if (col < ncols) z.x = 0.5 * xb[(int64_t)n * ldx];
        if (col + 1 < ncols) z.y = 0.5 * xb[(int64_t)n * ldx + 1];
        put(buf, ((int)t.in[n] << wcl) + c, N << wcl, odd ? mul(z, __ldg(tw + n)) : z);
    }
    __syncthreads();
    passes(buf, N, plan, wcl, tw);
    store_half(buf, odd, N, wcl, t.out, X + b * bso, ldo, col, ncols);
}

__global__ void __launch_bounds__(NT, 2)
k_irfft_pf(const double2* __restrict__ X, int64_t ldx, int64_t bsx, int ncols, double* __restrict__ y, int64_t ldy,
           int64_t bsy, const double* __restrict__ g, SetupPlan plan, int wcl, const double2* __restrict__ tw,
           const int* __restrict__ tab, double* const* __restrict__ yptr)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = plan.N, c = threadIdx.x & ((1 << wcl) - 1);
    const int col = (int)(blockIdx.x << (wcl + 1)) + 2 * c;
    const int64_t b = blockIdx.y;
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const Tables t(smem_raw + ((size_t)2 * N << wcl) * sizeof(double2), N, tab);
    __syncthreads();
    load_conj(buf, N, wcl, t.in, X + b * bsx, ldx, col, ncols);
    __syncthreads();
    passes(buf, 2 * N, plan, wcl, tw);
    const double inv = 1. / (2. * N);
    double* yb = (yptr ? yptr[b] : y + b * bsy) + col;
    if (col >= ncols) return;
    for (int n = threadIdx.x >> wcl; n < N; n += NT >> wcl) {
        // conj(y) = (E + w_L^n O) / L
        const int at = ((int)t.out[n] << wcl) + c;
        const double2 v = add(get(buf, at, N << wcl), mul(get(buf + (N << wcl), at, N << wcl), __ldg(tw + n)));
        double p = v.x * inv, q = -v.y * inv;
        if (g) {
            p *= g[(int64_t)n * ncols + col];
            if (col + 1 < ncols) q *= g[(int64_t)n * ncols + col + 1];
        }
        yb[(int64_t)n * ldy] = p;
        if (col + 1 < ncols) yb[(int64_t)n * ldy + 1] = q;
    }
}

// In place: X <- rfft(pad(irfft(X)[:N] g)).
__global__ void __launch_bounds__(NT, 2)
k_mid_pf(double2* X, int64_t ldx, int64_t bsx, int ncols, const double* __restrict__ g, SetupPlan plan, int wcl,
         const double2* __restrict__ tw, const int* __restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = plan.N, c = threadIdx.x & ((1 << wcl) - 1);
    const int col = (int)(blockIdx.x << (wcl + 1)) + 2 * c;
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    double2* odd = buf + (N << wcl);
    const Tables t(smem_raw + ((size_t)2 * N << wcl) * sizeof(double2), N, tab);
    double2* Xb = X + blockIdx.y * bsx;
    __syncthreads();
    load_conj(buf, N, wcl, t.in, Xb, ldx, col, ncols);
    __syncthreads();
    passes(buf, 2 * N, plan, wcl, tw);
    const double inv = 0.5 / (2. * N);   // the unpack's 1/2 with it
    for (int n = threadIdx.x >> wcl; n < N; n += NT >> wcl) {
        const int at = ((int)t.out[n] << wcl) + c;
        const double2 v = add(get(buf, at, N << wcl), mul(get(odd, at, N << wcl), __ldg(tw + n)));
        double2 z = make_double2(v.x * inv, -v.y * inv);
        if (g) {
            if (col < ncols) z.x *= g[(int64_t)n * ncols + col];
            if (col + 1 < ncols) z.y *= g[(int64_t)n * ncols + col + 1];
        }
        put(buf, at, N << wcl, z);
    }
    __syncthreads();
    // back to the input positions through the odd half
    for (int n = threadIdx.x >> wcl; n < N; n += NT >> wcl)
        put(odd, ((int)t.in[n] << wcl) + c, N << wcl, get(buf, ((int)t.out[n] << wcl) + c, N << wcl));
    __syncthreads();
    for (int n = threadIdx.x >> wcl; n < N; n += NT >> wcl) {
        const int at = ((int)t.in[n] << wcl) + c;
        const double2 z = get(odd, at, N << wcl);
        put(buf, at, N << wcl, z);
        put(odd, at, N << wcl, mul(z, __ldg(tw + n)));
    }
    __syncthreads();
    passes(buf, 2 * N, plan, wcl, tw);
    store_half(buf, 0, N, wcl, t.out, Xb, ldx, col, ncols);
    store_half(odd, 1, N, wcl, t.out, Xb, ldx, col, ncols);
}

static size_t vec_smem(int N, int halves, int wcl) { return ((size_t)halves * N << wcl) * sizeof(double2) + (size_t)N * 4; }

// Column pairs per CTA: up to 8, two CTAs per SM by shared memory, and as few
// as give two CTAs per SM work (an SM has two FP64 lanes).  Where a tile is
// small, its latency and not the FP64 rate, no more than the 304 CTAs that are
// resident: a second wave took as long again (us, input / inverse / middle step
// with it -> without: 9 steps, 468 columns x 2 12.3 / 14.4 / 23.6 -> 8.2 / 8.3 / 14.4; 64 steps
// 16.4 / 18.5 / 31.1 -> 10.3 / 11.3 / 18.5).  Above 512 points a tile the second wave is the
// better balance (360 steps, 700 columns x 2 47 / 47 / 86 with it, 62 / 59 / 108 without).
static int vec_tile(int N, int halves, int ncols, int nb)
{
    int w = 0;
    while (w < 3 && vec_smem(N, halves, w + 1) <= 113 * 1024) ++w;
    auto ctas = [&](int v) { return (int64_t)(halves == 1 ? 2 : 1) * nb * ((ncols + (2 << v) - 1) / (2 << v)); };
    while (w > 0 && ctas(w) < 2 * 152 && (ctas(w - 1) <= 2 * 152 || (N * halves << w) > 1024)) --w;
    return w;
}

// Shared memory at Wc = 2^wcl column pairs per tile.
static size_t smem_of(int N, int wcl, bool find_max)
{
    return ((size_t)2 * N << wcl) * sizeof(double2) + (size_t)N * 4 + (find_max ? (size_t)(N + 1) * 8 : 0);
}

}  // namespace setup

// Prime powers of N_t, each as passes of the largest radices (8 9 5 7, the
// rest of the power last); np = 0 entries when N_t = 1.
bool make_setup_plan(int N_t, SetupPlan* p)
{
    *p = SetupPlan{};
    p->N = N_t;
    int rest = N_t, inner = N_t;
    for (int prime : {2, 3, 5, 7}) {
        int q = 1;
        while (rest % prime == 0) rest /= prime, q *= prime;
        if (q == 1) continue;
        inner /= q;   // points of the dimensions behind this one
        const int d = p->ndim++;
        p->dim[d] = q;
        int M = q;
        while (M > 1) {
            int R = prime;
            if (prime == 2) R = M % 8 == 0 ? 8 : (M % 4 == 0 ? 4 : 2);
            if (prime == 3) R = M % 9 == 0 ? 9 : 3;
            if (p->np == kSetupPasses) return false;
            p->radix[p->np] = R;
            p->pdim[p->np] = d;
            p->S[p->np] = M / R;
            p->I[p->np] = inner;
            p->tstep[p->np] = 2 * N_t / M;
            ++p->np;
            M /= R;
        }
    }
    return rest == 1;
}

// Host tables: position of sample n (N entries), position of frequency k.
void setup_tables(const SetupPlan& p, int* t)
{
    const int N = p.N;
    int* in = t;
    int* out = t + N;
    // every digit combination (n_1 .. n_d) sits at its mixed-radix index and
    // holds sample sum n_i N / N_i mod N
    for (int at = 0; at < N; ++at) {
        int64_t n = 0;
        int inner = N;
        for (int d = 0; d < p.ndim; ++d) {
            inner /= p.dim[d];
            n += (int64_t)(at / inner % p.dim[d]) * (N / p.dim[d]);
        }
        in[n % N] = at;
    }
    for (int k = 0; k < N; ++k) {
        int at = 0, inner = N;
        for (int d = 0; d < p.ndim; ++d) {
            inner /= p.dim[d];
            int rem = k % p.dim[d], span = p.dim[d], pos = 0;
            for (int s = 0; s < p.np; ++s)
                if (p.pdim[s] == d) {
                    span /= p.radix[s];
                    pos += rem % p.radix[s] * span;
                    rem /= p.radix[s];
                }
            at += pos * inner;
        }
        out[k] = at;
    }
}

bool setup_fits(const SetupPlan& p, bool find_max)
{
    return p.N > 0 && setup::smem_of(p.N, 0, find_max) <= (size_t)kFftSmemMax;
}

cudaError_t prepare_setup_fft()
{
    cudaError_t e = cudaSuccess;
    for (auto k : {setup::k_create_pf<P_F32>, setup::k_create_pf<P_F16S>, setup::k_create_pf<P_BF16>,
                   setup::k_create_pf<P_BF16X2>, setup::k_create_pf<P_F64>, setup::k_create_pf<P_FP8S>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(setup::k_rfft_pf, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(setup::k_irfft_pf, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(setup::k_mid_pf, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax);
    return e;
}

bool pf_rfft(const double* x, int64_t ldx, int64_t bsx, int ncols, double2* X, int64_t ldo, int64_t bso, int nb,
             const FftGeom& g, const double2* tw, cudaStream_t st, const double* const* xptr, cudaError_t* err)
{
    const int N = g.N_t;
    if (!g.setup_tab || setup::vec_smem(N, 1, 0) > (size_t)kFftSmemMax) return false;
    const int w = setup::vec_tile(N, 1, ncols, nb);
    setup::k_rfft_pf<<<dim3((ncols + (2 << w) - 1) / (2 << w), nb, 2), setup::NT, setup::vec_smem(N, 1, w), st>>>(
        x, ldx, bsx, ncols, X, ldo, bso, g.splan, w, tw, g.setup_tab, xptr);
    count_launch();
    *err = cudaGetLastError();
    return true;
}

bool pf_irfft(const double2* X, int64_t ldx, int64_t bsx, int ncols, double* y, int64_t ldy, int64_t bsy,
              const double* gam, int nb, const FftGeom& g, const double2* tw, cudaStream_t st, double* const* yptr,
              cudaError_t* err)
{
    const int N = g.N_t;
    if (!g.setup_tab || setup::vec_smem(N, 2, 0) > (size_t)kFftSmemMax) return false;
    const int w = setup::vec_tile(N, 2, ncols, nb);
    setup::k_irfft_pf<<<dim3((ncols + (2 << w) - 1) / (2 << w), nb), setup::NT, setup::vec_smem(N, 2, w), st>>>(
        X, ldx, bsx, ncols, y, ldy, bsy, gam, g.splan, w, tw, g.setup_tab, yptr);
    count_launch();
    *err = cudaGetLastError();
    return true;
}

bool pf_hess_mid(double2* X, int64_t ldx, int64_t bsx, int ncols, const double* gam, int nb, const FftGeom& g,
                 const double2* tw, cudaStream_t st, cudaError_t* err)
{
    const int N = g.N_t;
    if (!g.setup_tab || setup::vec_smem(N, 2, 0) > (size_t)kFftSmemMax) return false;
    const int w = setup::vec_tile(N, 2, ncols, nb);
    setup::k_mid_pf<<<dim3((ncols + (2 << w) - 1) / (2 << w), nb), setup::NT, setup::vec_smem(N, 2, w), st>>>(
        X, ldx, bsx, ncols, gam, g.splan, w, tw, g.setup_tab);
    count_launch();
    *err = cudaGetLastError();
    return true;
}

bool setup_create(const double* blk, int64_t ldb, int ncols, int64_t col_base, int N_d, int N_m, int ldm, int prec,
                  void* fhat, const float* scales, unsigned long long* maxbits, int pass, const SetupPlan& p,
                  const double2* tw, const int* tab, cudaStream_t st, cudaError_t* err)
{
    const bool find_max = (prec == P_F16S || prec == P_FP8S) && pass == 0;
    if (!tab || !setup_fits(p, find_max)) return false;
    // up to 8 column pairs (128-byte rows), two CTAs per SM where that fits
    int wcl = 0;
    while (wcl < 3 && setup::smem_of(p.N, wcl + 1, find_max) <= 113 * 1024) ++wcl;
    const int ntiles = (ncols + (2 << wcl) - 1) / (2 << wcl);
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int grid = ntiles < 2 * nsm ? ntiles : 2 * nsm;
    const size_t sm = setup::smem_of(p.N, wcl, find_max);
#define BTT_SETUP(P)                                                                                            \
    setup::k_create_pf<P><<<grid, setup::NT, sm, st>>>(blk, ldb, ncols, col_base, N_d, N_m, ldm, p, wcl, tw, tab, \
                                                       fhat, scales, maxbits, find_max ? 1 : 0)
    switch (prec) {
        case P_F32: BTT_SETUP(P_F32); break;
        case P_F64: BTT_SETUP(P_F64); break;
        case P_F16S: BTT_SETUP(P_F16S); break;
        case P_BF16: BTT_SETUP(P_BF16); break;
        case P_BF16X2: BTT_SETUP(P_BF16X2); break;
        case P_FP8S: BTT_SETUP(P_FP8S); break;
        default: *err = cudaErrorInvalidValue; return true;
    }
#undef BTT_SETUP
    count_launch();
    *err = cudaGetLastError();
    return true;
}

}  // namespace btt

#ifdef BTT_CHECK
namespace btt {
BTT_CHECK_TU(check_record_fft_setup)
}  // namespace btt
#endif
