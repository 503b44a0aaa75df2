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
        for (int i = 0; i < R; ++i) v[i] = buf[at + i * step];
        dft_fwd<R>(v);
        if (S > 1) {
            const int n1 = lo / I;
            if (n1)
#pragma unroll
                for (int k = 1; k < R; ++k) v[k] = mul(v[k], __ldg(tw + n1 * k * tstep));
        }
#pragma unroll
        for (int i = 0; i < R; ++i) buf[at + i * step] = v[i];
    }
    __syncthreads();
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
                buf[at] = h;
                buf[(N << wcl) + at] = mul(h, w);
            }
        }
        __syncthreads();
        for (int p = 0; p < plan.np; ++p) {
            const int S = plan.S[p], I = plan.I[p], ts = plan.tstep[p];
            switch (plan.radix[p]) {
                case 2: pass<2>(buf, L, S, I, wcl, ts, tw); break;
                case 3: pass<3>(buf, L, S, I, wcl, ts, tw); break;
                case 4: pass<4>(buf, L, S, I, wcl, ts, tw); break;
                case 5: pass<5>(buf, L, S, I, wcl, ts, tw); break;
                case 7: pass<7>(buf, L, S, I, wcl, ts, tw); break;
                case 8: pass<8>(buf, L, S, I, wcl, ts, tw); break;
                default: pass<9>(buf, L, S, I, wcl, ts, tw); break;
            }
        }
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
                const double2 z = half[((int)out[j] << wcl) + c], zc = half[((int)out[jj] << wcl) + c];
                a = make_double2(z.x + zc.x, z.y - zc.y);
                d = make_double2(z.y + zc.y, zc.x - z.x);
            }
            if ((PREC == P_F16S || PREC == P_FP8S) && find_max) {
                // the lanes of a row first, then one shared maximum per row
                double m = one && w <= N ? fmax(fabs(a.x), fabs(a.y)) : 0.;
                if (both && w <= N) m = fmax(m, fmax(fabs(d.x), fabs(d.y)));
                for (int o = Wc / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (c == 0 && w <= N) atomicMax(&smax[w], (unsigned long long)__double_as_longlong(m));
                continue;
            }
            if (w > N || !one) continue;
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
    return e;
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
