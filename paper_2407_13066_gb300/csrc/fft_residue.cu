// FP32 time transforms of any length N_t, one tile of columns spread over a
// cluster of C thread blocks by frequency residue.
//
// The frequencies w of the length-L transform (L = 2 N_t, S = 2 C divides L)
// fall into S residues w = S j + r, and residue r is an M-point transform,
// M = N_t / C, of folded samples:
//     Z[S j + r] = sum_{n < M} u_r[n] w_M^{n j},
//     u_r[n] = w_L^{r n} sum_{q < C} z[n + q M] w_S^{r q}
// (the padding half of z is zero, so only C of S inputs appear; they give
// the even residues as one C-point DFT and the odd ones as a C-point DFT of
// z w_S^q).  The Hermitian partner L - w of residue r lies in residue S - r, at
// M - 1 - j: CTA r of the cluster owns residues r and S - r (CTA 0: 0 and C),
// so it unpacks and stores its own frequency rows.  Only the folded samples
// cross CTAs: forward, each CTA folds 1/C of the n and writes every u_r to its
// owner (distributed shared memory); inverse, each reads the S values of its
// n's back.  A CTA holds 2 M complex values per column pair instead of 2 N_t, so
// the rows of a tile are C times wider for the same shared memory; the width
// is what bounds these transforms (about 50 G L2 requests/s however narrow).
//
// Columns are handled as quads (fftq.cuh): four real columns, two complex
// sequences per thread, paired FP32.  The M-point transforms run in place with
// run-time radices up to 10 (6 and 10 by the prime-factor map, which needs no
// twiddles between their factors); twiddles and positions sit in shared
// memory (from global memory they missed L1, 736 against 646 us forward at
// 1500 steps).  Output digit order is reversed; complementing every digit of a
// frequency complements its position, so the partner of the value at position
// p is read at M - 1 - p.
//
// Against the one-CTA kernels of fft_kernels.cu, which this replaces wherever
// a plan exists but for few columns of long odd lengths (res_irfft, res_mid;
// us; 8 FP32 vectors, N_t N_m = 6.4 M, rows off 16-byte boundaries; 614 MB, 91 us
// at the measured copy rate):
//   N_t               60    100    250    420   1125   1500   3000   9000
//   input, before    616    530    449    486    692    669    954   1382
//   input, here      189    203    236    246    338    336    373    494
//   inverse, before  490    404    348    369    584    529    869   1108
//   inverse, here    275    296    313    330    461    455    577    722
// Bound by issue and latency (57% / 45% issue active at 24 resident warps,
// 1500 steps), no longer by the L2 requests of narrow rows.
#include <cooperative_groups.h>

#include "fftq.cuh"
#include "kernels.h"

namespace btt {
namespace res {

using fq::cq;
using fq::f2;
using fq::fma;
using fq::mul;

// Threads per CTA (threads_of); 24 warps per SM with 3, 2 or 1 CTAs.
constexpr int kNT = 256, kNTLong = 384, kNTLongest = 768;
constexpr int ctas_per_sm(int nt) { return nt == kNT ? 3 : nt == kNTLong ? 2 : 1; }
// Radices up to 10 run in 80 registers, three CTAs per SM (the inverse on
// clusters of 8 spills 80-88 bytes); up to 16 they take
// 128 (two CTAs), and the passes saved do not make up for the latency left
// uncovered (N_t = 1500, 8 columns on 2 CTAs: 866 / 1147 us against 646 / 911).
constexpr int kMaxRadix = 10;


// cos / sin of 2 pi e / n for the constant twiddles below
template <int N> struct Unit;
template <> struct Unit<9> {
    static __device__ __forceinline__ float c(int e)
    {
        return e == 1 ? 0.76604444311897803520f : e == 2 ? 0.17364817766693034885f : -0.93969262078590838405f;   // e = 4
    }
    static __device__ __forceinline__ float s(int e)
    {
        return e == 1 ? 0.64278760968653932632f : e == 2 ? 0.98480775301220805937f : 0.34202014332566873304f;
    }
};
template <> struct Unit<16> {   // e < 16
    static __device__ __forceinline__ float q(int e)   // cos over a quarter turn
    {
        return e == 0 ? 1.f : e == 1 ? 0.92387953251128675613f : e == 2 ? 0.70710678118654752440f
             : e == 3 ? 0.38268343236508977173f : 0.f;
    }
    static __device__ __forceinline__ float c(int e)
    {
        e &= 15;
        return e <= 4 ? q(e) : e <= 8 ? -q(8 - e) : e <= 12 ? -q(e - 8) : q(16 - e);
    }
    static __device__ __forceinline__ float s(int e) { return c(e + 12); }
};

// v * exp(-SG i theta), c = cos theta, s = sin theta
template <int SG> __device__ __forceinline__ cq rot(cq v, float c, float s)
{
    const f2 cc = fq::dup(c), d = fq::dup(SG > 0 ? s : -s), nd = fq::dup(SG > 0 ? -s : s);
    return {fma(v.im, d, mul(v.re, cc)), fma(v.re, nd, mul(v.im, cc))};
}

// Odd R, inputs p and R - p paired; outputs q and R - q share their cosine sum.
template <int R, int SG> __device__ __forceinline__ void rdft_odd(cq* v)
{
    constexpr int H = (R - 1) / 2;
    cq a[H], b[H];
    const cq v0 = v[0];
    cq y0 = v0;
#pragma unroll
    for (int p = 1; p <= H; ++p) {
        a[p - 1] = fq::cadd(v[p], v[R - p]);
        b[p - 1] = fq::csub(v[p], v[R - p]);
        y0 = fq::cadd(y0, a[p - 1]);
    }
    v[0] = y0;
#pragma unroll
    for (int q = 1; q <= H; ++q) {
        cq t = v0;
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            const f2 c = fq::dup((float)RootTable<R>::c((p * q) % R));
            t.re = fma(a[p - 1].re, c, t.re);
            t.im = fma(a[p - 1].im, c, t.im);
        }
        cq x = t, y = t;
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            const float s = (float)RootTable<R>::s((p * q) % R) * (float)SG;
            const f2 d = fq::dup(s), nd = fq::dup(-s);
            x.re = fma(b[p - 1].im, d, x.re);
            x.im = fma(b[p - 1].re, nd, x.im);
            y.re = fma(b[p - 1].im, nd, y.re);
            y.im = fma(b[p - 1].re, d, y.im);
        }
        v[q] = x;
        v[R - q] = y;
    }
}

template <int R, int SG> __device__ __forceinline__ void rdft(cq* v);

// R = A B, coprime: n = B n1 + A n2 (mod R), k = the residue class of (k1, k2)
template <int A, int B, int SG> __device__ __forceinline__ void dft_pfa(cq* v)
{
    constexpr int R = A * B;
    cq t[A][B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
        cq u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = v[(B * n1 + A * n2) % R];
        rdft<A, SG>(u);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) t[k1][n2] = u[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) rdft<B, SG>(t[k1]);
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = t[k % A][k % B];
}

// R = A A: n = A n1 + n2, k = k1 + A k2, constant twiddles w_R^{n2 k1} between
template <int A, int SG> __device__ __forceinline__ void dft_square(cq* v)
{
    constexpr int R = A * A;
    cq t[A][A];
#pragma unroll
    for (int n2 = 0; n2 < A; ++n2) {
        cq u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = v[A * n1 + n2];
        rdft<A, SG>(u);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1)
            t[k1][n2] = n2 * k1 == 0 ? u[k1] : rot<SG>(u[k1], Unit<R>::c(n2 * k1), Unit<R>::s(n2 * k1));
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        rdft<A, SG>(t[k1]);
#pragma unroll
        for (int k2 = 0; k2 < A; ++k2) v[k1 + A * k2] = t[k1][k2];
    }
}

template <int R, int SG> __device__ __forceinline__ void rdft(cq* v)
{
    if constexpr (R == 1) return;
    else if constexpr (R == 2 || R == 4 || R == 8) fq::dft<R, SG>(v);
    else if constexpr (R % 2 == 1 && R <= 7) rdft_odd<R, SG>(v);
    else if constexpr (R == 9) dft_square<3, SG>(v);
    else dft_pfa<2, R / 2, SG>(v);   // 6, 10
}

// a twiddle for both lanes
__device__ __forceinline__ ulonglong2 quad(float2 w) { return make_ulonglong2(fq::dup(w.x).u, fq::dup(w.y).u); }

// One in-place pass over the CTA's 2 M positions: radix R on sub-blocks of Mp
// (forward: DFT, then twiddles; inverse: conjugate twiddles, then DFT).
template <int NT, int R, bool INV>
__device__ __forceinline__ void pass(ulonglong2* buf, int total, int Mp, unsigned magic, int wql, int tstep,
                                     const float2* tws)
{
    const int S = Mp / R, nb = (total / R) << wql, step = S << wql, wm = (1 << wql) - 1;
    for (int b = threadIdx.x; b < nb; b += NT) {
        const int c = b & wm, j = b >> wql;
        const int blk = S == 1 ? j : (int)__umulhi((unsigned)j, magic), n1 = j - blk * S;
        const int at = ((blk * Mp + n1) << wql) + c;
        cq v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = fq::from_u2(buf[at + i * step]);
        const int e = n1 * tstep;
        if (INV && n1 != 0) {
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = fq::twiddle_conj(v[k], quad(tws[k * e]));
        }
        rdft<R, INV ? -1 : 1>(v);
        if (!INV && n1 != 0) {
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = fq::twiddle(v[k], quad(tws[k * e]));
        }
#pragma unroll
        for (int i = 0; i < R; ++i) buf[at + i * step] = fq::to_u2(v[i]);
    }
    __syncthreads();
}

template <int NT, bool INV>
__device__ __forceinline__ void radix_pass(int R, ulonglong2* buf, int total, int Mp, unsigned magic, int wql,
                                           int tstep, const float2* tws)
{
    switch (R) {
        case 2: pass<NT, 2, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 3: pass<NT, 3, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 4: pass<NT, 4, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 5: pass<NT, 5, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 6: pass<NT, 6, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 7: pass<NT, 7, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 8: pass<NT, 8, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        case 9: pass<NT, 9, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
        default: pass<NT, 10, INV>(buf, total, Mp, magic, wql, tstep, tws); break;
    }
}

// Shared memory of a CTA: the tile [2 M][Wq] quads, the M-point twiddles and
// the position table (position of a frequency).
template <int NT> struct Smem {
    ulonglong2* buf;
    float2* tws;
    unsigned short* pos;
    float* row;   // this warp's 128 values for rows off 16-byte boundaries
    __device__ __forceinline__ Smem(unsigned char* raw, int M, int wql)
    {
        buf = reinterpret_cast<ulonglong2*>(raw);
        float* rows = reinterpret_cast<float*>(buf + ((2 * M) << wql));
        row = rows + (threadIdx.x >> 5) * 128;
        tws = reinterpret_cast<float2*>(rows + NT * 4);
        pos = reinterpret_cast<unsigned short*>(tws + M);
    }
    // step: L / M
    __device__ __forceinline__ void fill(int M, int step, const float2* __restrict__ tw, const int* __restrict__ tab)
    {
        for (int i = threadIdx.x; i < M; i += NT) {
            tws[i] = __ldg(tw + i * step);
            pos[i] = (unsigned short)__ldg(tab + i);
        }
    }
};

// 32-bit shared::cluster address of this CTA's shared byte address a in CTA q
__device__ __forceinline__ uint32_t map(uint32_t a, int q)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(q));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, cq v)
{
    asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(v.re.u), "l"(v.im.u) : "memory");
}
__device__ __forceinline__ cq ld_remote(uint32_t a)
{
    cq v;
    asm volatile("ld.shared::cluster.v2.u64 {%0, %1}, [%2];" : "=l"(v.re.u), "=l"(v.im.u) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int cta_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}

// owner CTA and slot of residue rr (S = 2 C)
template <int C> __device__ __forceinline__ constexpr int owner(int rr) { return rr == 0 || rr == C ? 0 : (rr < C ? rr : 2 * C - rr); }
template <int C> __device__ __forceinline__ constexpr int slot(int rr) { return rr < C ? 0 : 1; }

// z_q w_S^{SG q}, S = 2 C: the inputs (forward) or outputs (inverse) of the odd residues
template <int C, int SG> __device__ __forceinline__ cq odd_root(cq v, int q)
{
    return q == 0 ? v : rot<SG>(v, Unit<16>::c(q * (8 / C)), Unit<16>::s(q * (8 / C)));
}

__device__ __forceinline__ cq load_quad(const float* __restrict__ row, int col, int ncols, bool vec)
{
    float4 x;
    if (vec && col + 3 < ncols) {
        x = __ldcs(reinterpret_cast<const float4*>(row + col));
    } else {
        x.x = col < ncols ? __ldg(row + col) : 0.f;
        x.y = col + 1 < ncols ? __ldg(row + col + 1) : 0.f;
        x.z = col + 2 < ncols ? __ldg(row + col + 2) : 0.f;
        x.w = col + 3 < ncols ? __ldg(row + col + 3) : 0.f;
    }
    return {fq::pack(x.x, x.y), fq::pack(x.z, x.w)};
}

// ------------------------------------------------------------ forward
// Output of one frequency row: columns col .. col+3, spectra a (columns col,
// col+1) and b (col+2, col+3).
struct OutC64 {
    float2* X;
    int64_t ldo, bso;
    // columns col, col + 1 of frequency row w
    __device__ __forceinline__ void row(int64_t b, int w, int col, int ncols, cq a, bool vec) const
    {
        float2* o = X + b * bso + (int64_t)w * ldo + col;
        const float2 v0 = make_float2(fq::lo(a.re), fq::lo(a.im)), v1 = make_float2(fq::hi(a.re), fq::hi(a.im));
        if (vec && col + 1 < ncols) {
            *reinterpret_cast<float4*>(o) = make_float4(v0.x, v0.y, v1.x, v1.y);
        } else {
            if (col < ncols) o[0] = v0;
            if (col + 1 < ncols) o[1] = v1;
        }
    }
    __device__ __forceinline__ bool vec() const { return ((ldo | bso) & 1) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0; }
};

// The BF16 operand of the tensor-core products: conj(X) as BF16 pairs, and
// with lo_off the BF16 remainders (launch_rfft_stack).
struct OutStack {
    __nv_bfloat162* XA;
    int64_t ldm, mt_stride, lo_off;
    static __device__ __forceinline__ void put(__nv_bfloat162* o, int col, int ncols, bool vec, __nv_bfloat162 v0,
                                               __nv_bfloat162 v1)
    {
        if (vec && col + 1 < ncols) {
            *reinterpret_cast<uint2*>(o) = make_uint2(*reinterpret_cast<unsigned*>(&v0), *reinterpret_cast<unsigned*>(&v1));
        } else {
            if (col < ncols) o[0] = v0;
            if (col + 1 < ncols) o[1] = v1;
        }
    }
    __device__ __forceinline__ void row(int64_t b, int w, int col, int ncols, cq a, bool vec) const
    {
        __nv_bfloat162* o = XA + (((int64_t)w * mt_stride + (b >> 6)) * 64 + (b & 63)) * ldm + col;
        const float2 x0 = make_float2(fq::lo(a.re), -fq::lo(a.im)), x1 = make_float2(fq::hi(a.re), -fq::hi(a.im));
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(x0.x, x0.y), h1 = __floats2bfloat162_rn(x1.x, x1.y);
        put(o, col, ncols, vec, h0, h1);
        if (!lo_off) return;
        const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
        put(o + lo_off, col, ncols, vec, __floats2bfloat162_rn(x0.x - f0.x, x0.y - f0.y),
            __floats2bfloat162_rn(x1.x - f1.x, x1.y - f1.y));
    }
    __device__ __forceinline__ bool vec() const
    {
        return ((ldm | lo_off) & 1) == 0 && (reinterpret_cast<uintptr_t>(XA) & 7) == 0;
    }
};

// Row pairs of CTA r: task t is a frequency row w <= N_t; at() gives the
// positions of Z[w] and Z[L - w] in the tile.  CTA r > 0: every frequency j of
// its first residue, partner mirrored in the second (the row is w or L - w).
// CTA 0: half of each residue.
template <int C> struct Rows {
    static constexpr int S = 2 * C;
    int M, r, n0;
    __device__ __forceinline__ Rows(int M_, int r_) : M(M_), r(r_), n0(r_ ? M_ : M_ / 2 + 1) {}
    __device__ __forceinline__ int count() const { return r ? M : n0 + (M + 1) / 2; }
    __device__ __forceinline__ int w(int t) const
    {
        if (r) {
            const int w = S * t + r;
            return w > C * M ? S * M - w : w;
        }
        return t < n0 ? S * t : S * (t - n0) + C;
    }
    // h = 0: position of Z[w], h = 1: of Z[L - w]
    __device__ __forceinline__ int at(int t, int h, const unsigned short* pos) const
    {
        if (r == 0 && t < n0) return pos[h ? (t ? M - t : 0) : t];   // residue 0: partner M - j
        const int p = pos[r ? t : t - n0];
        const int first = r ? p : M + p;             // residue C: partner M - 1 - j, mirrored
        const bool flip = r && S * t + r > C * M;
        return (h != 0) != flip ? 2 * M - 1 - p : first;
    }
};
// exchange with the other half of the quad
__device__ __forceinline__ cq swap_half(cq v)
{
    return {{__shfl_xor_sync(0xffffffffu, v.re.u, 1)}, {__shfl_xor_sync(0xffffffffu, v.im.u, 1)}};
}

template <int C, class Out, int NT>
__global__ void __launch_bounds__(NT, ctas_per_sm(NT))
k_rfft_res(const float* __restrict__ x, int64_t ldx, int64_t bsx, int ncols, Out out, ResPlan plan, int wql,
           const float2* __restrict__ tw, const int* __restrict__ tab, const float* const* __restrict__ xptr)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int S = 2 * C;
    Smem<NT> sm_(smem_raw, plan.M, wql);
    ulonglong2* buf = sm_.buf;
    const int M = plan.M, L = S * M, N = C * M, wm = (1 << wql) - 1;
    const int r = C == 1 ? 0 : cta_rank();
    const int col0 = (blockIdx.x / C) << (wql + 2);
    const int64_t b = blockIdx.y;
    const float* xb = xptr ? xptr[b] : x + b * bsx;
    const bool vin = (ldx & 3) == 0 && (reinterpret_cast<uintptr_t>(xb) & 15) == 0;

    uint32_t dst[C];
    if constexpr (C > 1) {
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(buf);
#pragma unroll
        for (int q = 0; q < C; ++q) dst[q] = map(mine, q);
        // every CTA of the cluster has started: its shared memory may be written
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    }
    sm_.fill(M, S, tw, tab);
    // fold: C rows in, S residues out, U of them per thread so that 8 row
    // loads are in flight
    constexpr int U = 8 / C;
    const int nfold = M << wql, lane = threadIdx.x & 31;
    for (int g0 = r * NT + threadIdx.x; g0 - lane < nfold; g0 += U * C * NT) {
        cq z[U][C];
        if (vin) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int g = g0 + u * C * NT, n = g >> wql, col = col0 + ((g & wm) << 2);
#pragma unroll
                for (int q = 0; q < C; ++q)
                    z[u][q] = g < nfold && BTT_IN(n + q * M, N, CK_FFT_LOAD)
                                  ? load_quad(xb + (int64_t)(n + q * M) * ldx, col, ncols, true)
                                  : cq{fq::dup(0.f), fq::dup(0.f)};
            }
        } else {
            // rows off 16-byte boundaries: the warp's 32 quads are 128
            // consecutive tile elements, loaded 32 at a time and regrouped
            float f[U * C][4];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < C; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = ((g0 - lane + u * C * NT) << 2) + 32 * k + lane;   // tile element
                        const int n = e >> (wql + 2), col = col0 + (e & (4 * wm + 3));
                        f[u * C + q][k] = n < M && col < ncols && BTT_IN(n + q * M, N, CK_FFT_LOAD)
                                              ? __ldcs(xb + (int64_t)(n + q * M) * ldx + col)
                                              : 0.f;
                    }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k) sm_.row[32 * k + lane] = f[u * C + q][k];
                    __syncwarp();
                    z[u][q] = fq::from_u2(reinterpret_cast<const ulonglong2*>(sm_.row)[lane]);
                }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int g = g0 + u * C * NT, n = g >> wql;
            if (g >= nfold) break;
            cq e[C], o[C];
#pragma unroll
            for (int q = 0; q < C; ++q) {
                e[q] = z[u][q];
                o[q] = odd_root<C, 1>(z[u][q], q);
            }
            rdft<C, 1>(e);
            rdft<C, 1>(o);
#pragma unroll
            for (int rr = 0; rr < S; ++rr) {
                cq v = (rr & 1) ? o[rr / 2] : e[rr / 2];
                if (rr) v = fq::twiddle(v, quad(__ldg(tw + rr * n)));
                const int at = slot<C>(rr) * nfold + g;
                if (!BTT_IN(at, 2 * nfold, CK_FFT_REMOTE)) continue;
                if constexpr (C == 1) buf[at] = fq::to_u2(v);
                else st_remote(dst[owner<C>(rr)] + (uint32_t)at * 16u, v);
            }
        }
    }
    if constexpr (C > 1) cooperative_groups::this_cluster().sync();
    else __syncthreads();

    int Mp = M, tstep = 1;
    for (int p = 0; p < plan.np; ++p) {
        radix_pass<NT, false>(plan.radix[p], buf, 2 * M, Mp, plan.magic[p], wql, tstep, sm_.tws);
        Mp /= plan.radix[p];
        tstep *= plan.radix[p];
    }

    // Unpack this CTA's rows, two threads per quad (so that a warp's stores
    // are contiguous): one reads Z[w], the other Z[L - w], they exchange them,
    // and each forms two of the four spectra.
    const bool vout = out.vec();
    const f2 half = fq::dup(0.5f);
    const Rows<C> rows(M, r);
    const int nrow = rows.count(), ntask = nrow << (wql + 1);
    for (int i0 = 0; i0 < ntask; i0 += NT) {
        const int i = i0 + threadIdx.x, h = i & 1, c = (i >> 1) & wm, t = min(i >> (wql + 1), nrow - 1);
        const int w = rows.w(t), col = col0 + (c << 2) + 2 * h;
        const cq mine = fq::from_u2(buf[(rows.at(t, h, sm_.pos) << wql) + c]), other = swap_half(mine);
        cq v;   // h = 0: (Z + conj Z') / 2; h = 1: (Z - conj Z') / (2 i)
        if (h == 0) v = {fq::add(mine.re, other.re), fq::sub(mine.im, other.im)};
        else v = {fq::add(other.im, mine.im), fq::sub(mine.re, other.re)};
        v = {mul(half, v.re), mul(half, v.im)};
        if (i < ntask && BTT_IN(w, N + 1, CK_FFT_STORE)) out.row(b, w, col, ncols, v, vout);
    }
}

// ------------------------------------------------------------ inverse
// columns col, col + 1 of a half spectra row
__device__ __forceinline__ cq load_spectra(const float2* __restrict__ row, int col, int ncols, bool vec)
{
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec && col + 1 < ncols) {
        p = __ldcs(reinterpret_cast<const float4*>(row + col));
    } else {
        if (col < ncols) p.x = row[col].x, p.y = row[col].y;
        if (col + 1 < ncols) p.z = row[col + 1].x, p.w = row[col + 1].y;
    }
    return {fq::pack(p.x, p.z), fq::pack(p.y, p.w)};
}
__device__ __forceinline__ cq load_spectra(const __nv_bfloat162* __restrict__ row, int col, int ncols, bool vec)
{
    uint2 q = make_uint2(0u, 0u);
    if (vec && col + 1 < ncols) {
        q = __ldcs(reinterpret_cast<const uint2*>(row + col));
    } else {
        if (col < ncols) q.x = *reinterpret_cast<const unsigned*>(row + col);
        if (col + 1 < ncols) q.y = *reinterpret_cast<const unsigned*>(row + col + 1);
    }
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
    const float2 d = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
    return {fq::pack(a.x, d.x), fq::pack(a.y, d.y)};
}

template <int C, class TX, int NT>
__global__ void __launch_bounds__(NT, ctas_per_sm(NT))
k_irfft_res(const TX* __restrict__ X, int64_t ldx, int64_t bsx, int ncols, float* __restrict__ y, int64_t ldy,
            int64_t bsy, const float* __restrict__ gam, ResPlan plan, int wql, const float2* __restrict__ tw,
            const int* __restrict__ tab, float* const* __restrict__ yptr)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int S = 2 * C;
    Smem<NT> sm_(smem_raw, plan.M, wql);
    ulonglong2* buf = sm_.buf;
    const int M = plan.M, L = S * M, N = C * M, wm = (1 << wql) - 1;
    const int r = C == 1 ? 0 : cta_rank();
    const int col0 = (blockIdx.x / C) << (wql + 2);
    const int64_t b = blockIdx.y;
    const TX* Xb = X + b * bsx;
    const bool vin = (ldx & 1) == 0 && (reinterpret_cast<uintptr_t>(Xb) & (2 * sizeof(TX) - 1)) == 0;
    const int nfold = M << wql;

    // This CTA's half spectra rows, two threads per quad: one loads the
    // spectra A of columns 0, 1, the other B of columns 2, 3 (contiguous
    // across a warp); they exchange, and one forms Z[w] = A + i B, the other
    // Z[L - w] = conj A + i conj B.  Bins 0 and N_t of a real series are real.
    constexpr int U = 8;
    const Rows<C> rows(M, r);
    const int nrow = rows.count(), ntask = nrow << (wql + 1);
    for (int i0 = 0; i0 < ntask; i0 += U * NT) {
        cq v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * NT + threadIdx.x, h = i & 1, c = (i >> 1) & wm, t = min(i >> (wql + 1), nrow - 1);
            const int w = rows.w(t), col = col0 + (c << 2) + 2 * h;
            v[u] = {fq::dup(0.f), fq::dup(0.f)};
            if (BTT_IN(w, N + 1, CK_FFT_LOAD)) v[u] = load_spectra(Xb + (int64_t)w * ldx, col, ncols, vin);
            if (w == 0 || w == N) v[u].im = fq::dup(0.f);
        }
        if (i0 == 0) {   // the tables arrive behind the first rows
            sm_.fill(M, S, tw, tab);
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * NT >= ntask) break;
            const int i = i0 + u * NT + threadIdx.x, t = min(i >> (wql + 1), nrow - 1);
            const int at = (rows.at(t, i & 1, sm_.pos) << wql) + ((i >> 1) & wm);
            const cq o = swap_half(v[u]);
            cq q;   // Z = A + i B; Z' = conj A + i conj B (h = 1: v = B, o = A)
            if ((i & 1) == 0) q = {fq::sub(v[u].re, o.im), fq::add(v[u].im, o.re)};
            else q = {fq::add(o.re, v[u].im), fq::sub(v[u].re, o.im)};
            if (i < ntask && BTT_IN(at, 2 * nfold, CK_FFT_SMEM)) buf[at] = fq::to_u2(q);
        }
    }
    __syncthreads();

    int Mp = 1, tstep = M;
    for (int p = plan.np - 1; p >= 0; --p) {
        Mp *= plan.radix[p];
        tstep /= plan.radix[p];
        radix_pass<NT, true>(plan.radix[p], buf, 2 * M, Mp, plan.magic[p], wql, tstep, sm_.tws);
    }

    uint32_t src[C];
    if constexpr (C > 1) {
        cooperative_groups::this_cluster().sync();   // every CTA's residues are final
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(buf);
#pragma unroll
        for (int q = 0; q < C; ++q) src[q] = map(mine, q);
    }
    const float inv = 1.f / (float)L;
    float* yb = yptr ? yptr[b] : y + b * bsy;
    const bool vout = (ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(yb) & 15) == 0;
    const bool vgam = (ncols & 3) == 0 && (reinterpret_cast<uintptr_t>(gam) & 15) == 0;
    constexpr int V = C >= 4 ? 1 : 4 / C;   // butterflies whose values are requested together
    const int lane = threadIdx.x & 31;
    for (int g0 = r * NT + threadIdx.x; g0 - lane < nfold; g0 += V * C * NT) {
        cq e[V][C], o[V][C];
        float2 t[V][S];
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const int g = min(g0 + u * C * NT, nfold - 1);
#pragma unroll
            for (int rr = 0; rr < S; ++rr) {
                cq v = {fq::dup(0.f), fq::dup(0.f)};
                const int at = slot<C>(rr) * nfold + g;
                if (BTT_IN(at, 2 * nfold, CK_FFT_REMOTE)) {
                    if constexpr (C == 1) v = fq::from_u2(buf[at]);
                    else v = ld_remote(src[owner<C>(rr)] + (uint32_t)at * 16u);
                }
                ((rr & 1) ? o[u][rr / 2] : e[u][rr / 2]) = v;
                t[u][rr] = rr ? __ldg(tw + rr * (g >> wql)) : make_float2(1.f, 0.f);
            }
        }
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const int g = g0 + u * C * NT, n = g >> wql, col = col0 + ((g & wm) << 2);
            if (g - lane >= nfold) break;
#pragma unroll
            for (int rr = 1; rr < S; ++rr) {
                cq& v = (rr & 1) ? o[u][rr / 2] : e[u][rr / 2];
                v = fq::twiddle_conj(v, quad(t[u][rr]));
            }
            rdft<C, -1>(e[u]);
            rdft<C, -1>(o[u]);
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const cq x = fq::cadd(e[u][q], odd_root<C, -1>(o[u][q], q));
                const f2 k = fq::dup(inv);
                const f2 re = mul(x.re, k), im = mul(x.im, k);
                float4 v = make_float4(fq::lo(re), fq::hi(re), fq::lo(im), fq::hi(im));
                const int64_t row = n + q * M;
                const bool in = g < nfold && BTT_IN(row, N, CK_FFT_STORE);
                if (gam && in) {
                    const cq gv = load_quad(gam + row * ncols, col, ncols, vgam);
                    v.x *= fq::lo(gv.re);
                    v.y *= fq::hi(gv.re);
                    v.z *= fq::lo(gv.im);
                    v.w *= fq::hi(gv.im);
                }
                if (vout) {
                    float* out = yb + row * ldy + col;
                    if (in && col + 3 < ncols) {
                        *reinterpret_cast<float4*>(out) = v;
                    } else if (in) {
                        if (col < ncols) out[0] = v.x;
                        if (col + 1 < ncols) out[1] = v.y;
                        if (col + 2 < ncols) out[2] = v.z;
                    }
                } else {
                    // rows off 16-byte boundaries: the warp's 128 values,
                    // stored 32 consecutive tile elements at a time
                    __syncwarp();
                    reinterpret_cast<float4*>(sm_.row)[lane] = v;
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int el = ((g - lane) << 2) + 32 * k + lane;
                        const int en = el >> (wql + 2), ec = col0 + (el & (4 * wm + 3));
                        if (en < M && ec < ncols && BTT_IN(en + q * M, N, CK_FFT_STORE))
                            yb[(int64_t)(en + q * M) * ldy + ec] = sm_.row[32 * k + lane];
                    }
                }
            }
        }
    }
    if constexpr (C > 1) cooperative_groups::this_cluster().sync();   // the others have read this CTA's memory
}

// ------------------------------------------------------------ host side
template <typename K> static cudaError_t set_smem(K k)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax);
}

template <typename K, typename... A>
static cudaError_t launch(K kern, int C, int threads, int tiles, int nb, size_t sm, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(tiles * C), (unsigned)nb, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

struct Shape {
    int C, wql;
};

// Odd lengths above 2048 have no cluster to spread over, and their CTA leaves
// room for one other on its SM or for none: with 8 warps each the latency of
// a pass was left uncovered.  Inverse, us, the kernels of fft_kernels.cu / 8 warps
// / now: 3125 steps, 8 x 1200 columns 450 / 497 / 365, 30 columns 18 / 25 / 23; 2187 steps
// (two CTAs), 8 x 800 columns 263 / 147 / 135.
static int threads_of(const FftGeom& g, int C)
{
    if (C > 1 || g.N_t <= 2048) return kNT;
    return (size_t)g.N_t * 42 + kNTLong * 16 <= 113 * 1024 ? kNTLong : kNTLongest;
}

static size_t smem_of(const FftGeom& g, int C, int wql)
{
    const size_t M = g.N_t / C;
    return ((2 * M) << wql) * 16 + threads_of(g, C) * 16 + M * 10;
}

// Cluster size and tile width.  Wide rows want few CTAs' worth of shared
// memory per column, latency wants three CTAs per SM (76 KB): the widest
// tile up to 16 columns that leaves three, on the smallest cluster that
// holds it; where only 4 columns would, 8 columns at two per SM.  Measured
// (us, 8 FP32 vectors, N_t N_m = 12.8 M, input transform / inverse):
//   420:  1 CTA  16 columns 468 / 615, 32 845 / 1296, 8 625 / 703
//   1500: 4 CTAs 16 columns 620 / 835; 2 CTAs 8 644 / 785, 16 664 / 864
//   9000: 8 CTAs 8 columns (87 KB) 932 / 1356, 4 (52 KB) 1129 / 1458,
//         16 (157 KB, one CTA per SM) 1190 / 2237; 4 CTAs 4 (100 KB) 1446 / 1306
// Few columns take narrower tiles, so that two CTAs per SM have work, but no
// more CTAs than are resident at once: a second wave of small ones cost more
// than the idle SMs (us, input / inverse, unbounded -> so: 12 steps, 2000
// columns 8.2 / 8.7 -> 6.2 / 6.2; 420 steps 13.0 / 14.4 -> 10.3 / 10.3; 1500 steps, 16
// x 30 columns 19.1 / 21.5 -> 12.4 / 14.4).
static bool pick(const FftGeom& g, int ncols, int nb, Shape* s)
{
    if (!g.res_tab) return false;
    int best = -1;
    for (int i = 0; i < 4; ++i) {
        if (!g.res[i].M) continue;
        int wmax = 2;   // one CTA and few points: up to 128 columns, so that its threads have work
        if (i == 0)
            while (wmax < 5 && (g.res[0].M << wmax) < 2048) ++wmax;
        for (int w = wmax; w >= 0; --w) {
            const size_t sm = smem_of(g, 1 << i, w);
            if (sm > (size_t)kFftSmemMax) continue;
            // 3 per SM: 30 + width; 2 per SM: 8 columns and more beat 4 at 3
            const int per = sm <= 76 * 1024 ? 2 : (sm <= 113 * 1024 ? 1 : 0);
            const int score = per == 2 ? (w ? 30 + w : 10) : per == 1 ? (w ? 20 + w : 5) : 0;
            if (score > best) best = score, s->C = 1 << i, s->wql = w;
        }
    }
    if (best < 0) return false;
    auto ctas = [&](int w) { return (int64_t)s->C * nb * ((ncols + (4 << w) - 1) / (4 << w)); };
    auto resident = [&](int w) {
        const size_t sm = smem_of(g, s->C, w);
        return 152 * (sm <= 76 * 1024 ? 3 : sm <= 113 * 1024 ? 2 : 1);
    };
    while (s->wql > 0 && ctas(s->wql) < 2 * 152 && ctas(s->wql - 1) <= resident(s->wql - 1)) --s->wql;
    return true;
}

static int lg(int C) { return C == 1 ? 0 : C == 2 ? 1 : C == 4 ? 2 : 3; }
static int tiles_of(int ncols, const Shape& s) { return (ncols + (4 << s.wql) - 1) / (4 << s.wql); }

}  // namespace res

// Radices of an M-point transform: the fewest passes, then the smallest
// largest radix; even ones first, so that the last pass (neighbouring
// positions) has an odd stride in shared memory where there is one.
static void res_radices(int m, int last, int* cur, int n, int* best, int* nbest)
{
    static const int kR[] = {10, 9, 8, 7, 6, 5, 4, 3, 2};
    if (m == 1) {
        int sum = 0, bsum = 0;
        for (int i = 0; i < n; ++i) sum += cur[i];
        for (int i = 0; i < *nbest; ++i) bsum += best[i];
        if (*nbest < 0 || n < *nbest || (n == *nbest && n && (cur[0] < best[0] || (cur[0] == best[0] && sum < bsum)))) {
            for (int i = 0; i < n; ++i) best[i] = cur[i];
            *nbest = n;
        }
        return;
    }
    if (n == kResPasses || (*nbest >= 0 && n >= *nbest)) return;
    for (int r : kR)
        if (r <= last && m % r == 0) {
            cur[n] = r;
            res_radices(m / r, r, cur, n + 1, best, nbest);
        }
}

void make_res_plans(FftGeom* g)
{
    int off = 0;
    for (int i = 0; i < 4; ++i) {
        ResPlan& p = g->res[i];
        const int C = 1 << i;
        p = ResPlan{};
        if (g->N_t % C) continue;
        p.M = g->N_t / C;
        int cur[kResPasses], best[kResPasses], nbest = -1;
        res_radices(p.M, res::kMaxRadix, cur, 0, best, &nbest);
        if (nbest < 0) {
            p.M = 0;
            continue;
        }
        p.np = nbest;
        int n = 0;
        for (int odd = 0; odd < 2; ++odd)
            for (int k = 0; k < nbest; ++k)
                if (best[k] % 2 == odd) p.radix[n++] = best[k];
        int Mp = p.M;
        for (int k = 0; k < p.np; ++k) {
            const int S = Mp / p.radix[k];
            p.magic[k] = S > 1 ? (unsigned)((1ull << 32) / S + 1) : 0u;
            Mp = S;
        }
        p.tab = off;
        off += p.M;
    }
    g->res_ints = off;
}

void res_tables(const FftGeom& g, int* t)
{
    for (const ResPlan& p : g.res) {
        if (!p.M) continue;
        int* pos = t + p.tab;
        for (int k = 0; k < p.M; ++k) {
            int rem = k, at = 0, span = p.M;
            for (int s = 0; s < p.np; ++s) {
                span /= p.radix[s];
                at += rem % p.radix[s] * span;
                rem /= p.radix[s];
            }
            pos[k] = at;
        }
    }
}

cudaError_t prepare_res_fft()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](auto k) {
        if (e == cudaSuccess) e = res::set_smem(k);
    };
    auto all = [&](auto c) {
        constexpr int C = decltype(c)::value;
        set(res::k_rfft_res<C, res::OutC64, res::kNT>);
        set(res::k_rfft_res<C, res::OutStack, res::kNT>);
        set(res::k_irfft_res<C, float2, res::kNT>);
        set(res::k_irfft_res<C, __nv_bfloat162, res::kNT>);
    };
    all(std::integral_constant<int, 1>{});
    all(std::integral_constant<int, 2>{});
    all(std::integral_constant<int, 4>{});
    all(std::integral_constant<int, 8>{});
    auto wide = [&](auto nt) {
        constexpr int NT = decltype(nt)::value;
        set(res::k_rfft_res<1, res::OutC64, NT>);
        set(res::k_rfft_res<1, res::OutStack, NT>);
        set(res::k_irfft_res<1, float2, NT>);
        set(res::k_irfft_res<1, __nv_bfloat162, NT>);
    };
    wide(std::integral_constant<int, res::kNTLong>{});
    wide(std::integral_constant<int, res::kNTLongest>{});
    return e;
}

// Dispatch on the cluster size and the threads per CTA.
#define BTT_RES(K, T, ...)                                                                                      \
    (nt == res::kNTLongest ? res::launch(res::K<1, T, res::kNTLongest>, 1, nt, tiles, nb, sm, st, __VA_ARGS__)  \
     : nt == res::kNTLong  ? res::launch(res::K<1, T, res::kNTLong>, 1, nt, tiles, nb, sm, st, __VA_ARGS__)     \
     : s.C == 1            ? res::launch(res::K<1, T, res::kNT>, 1, nt, tiles, nb, sm, st, __VA_ARGS__)         \
     : s.C == 2            ? res::launch(res::K<2, T, res::kNT>, 2, nt, tiles, nb, sm, st, __VA_ARGS__)         \
     : s.C == 4            ? res::launch(res::K<4, T, res::kNT>, 4, nt, tiles, nb, sm, st, __VA_ARGS__)         \
                           : res::launch(res::K<8, T, res::kNT>, 8, nt, tiles, nb, sm, st, __VA_ARGS__))
#define BTT_RES_SETUP                                                       \
    res::Shape s;                                                           \
    if (!res::pick(g, ncols, nb, &s)) return false;                         \
    const ResPlan& plan = g.res[res::lg(s.C)];                              \
    const int tiles = res::tiles_of(ncols, s), nt = res::threads_of(g, s.C); \
    const size_t sm = res::smem_of(g, s.C, s.wql);                          \
    const int* tab = g.res_tab + plan.tab

bool res_rfft(const float* x, int64_t ldx, int64_t bsx, int ncols, float2* X, int64_t ldo, int64_t bso, int nb,
              const FftGeom& g, const float2* tw, cudaStream_t st, const float* const* xptr, cudaError_t* err)
{
    BTT_RES_SETUP;
    const res::OutC64 out{X, ldo, bso};
    *err = BTT_RES(k_rfft_res, res::OutC64, x, ldx, bsx, ncols, out, plan, s.wql, tw, tab, xptr);
    return true;
}

bool res_rfft_stack(const float* x, int64_t ldx, int64_t bsx, int ncols, void* xstack, int ldm, int mt_stride, int nb,
                    const FftGeom& g, const float2* tw, cudaStream_t st, int64_t lo_off, const float* const* xptr,
                    cudaError_t* err)
{
    BTT_RES_SETUP;
    const res::OutStack out{static_cast<__nv_bfloat162*>(xstack), ldm, mt_stride, lo_off};
    *err = BTT_RES(k_rfft_res, res::OutStack, x, ldx, bsx, ncols, out, plan, s.wql, tw, tab, xptr);
    return true;
}

bool res_irfft(const float2* X, int64_t ldx, int64_t bsx, int ncols, float* y, int64_t ldy, int64_t bsy,
               const float* gam, int nb, const FftGeom& g, const float2* tw, cudaStream_t st, float* const* yptr,
               cudaError_t* err)
{
    // Few columns of a long odd length, one CTA's latency: the mixed-radix
    // kernel's is shorter (30 columns, this one / that: 3125 23 / 19 us, 4375
    // 27 / 23, 5145 32 / 25; below 3000 steps they are level).  The number of
    // vectors has no part in it: a vector's result stays the same.
    if (g.N_t % 2 && g.N_t > 3000 && ncols <= 32) return false;
    BTT_RES_SETUP;
    *err = BTT_RES(k_irfft_res, float2, X, ldx, bsx, ncols, y, ldy, bsy, gam, plan, s.wql, tw, tab, yptr);
    return true;
}

// Odd lengths above 2048 (no cluster) take two launches of 20-30 us where the
// columns are few; one launch of the mixed-radix kernel is shorter (us, two
// launches / one; 30 columns, 1 and 8 vectors, then 100 columns and 8):
//   2401  33 / 29  35 / 29  57 / 62     3125  43 / 35  43 / 35  80 / 80
//   4375  55 / 43  55 / 43  102 / 103   5145  68 / 47  68 / 48  131 / 115
bool res_mid(const FftGeom& g, int ncols)
{
    return g.N_t >= 100 && !(g.N_t % 2 && g.N_t > 2048 && ncols <= (g.N_t > 4200 ? 100 : 32));
}

bool res_irfft_bf16(const __nv_bfloat162* X, int64_t ldx, int64_t bsx, int ncols, float* y, int64_t ldy, int64_t bsy,
                    int nb, const FftGeom& g, const float2* tw, cudaStream_t st, float* const* yptr, cudaError_t* err)
{
    BTT_RES_SETUP;
    const float* none = nullptr;
    *err = BTT_RES(k_irfft_res, __nv_bfloat162, X, ldx, bsx, ncols, y, ldy, bsy, none, plan, s.wql, tw, tab, yptr);
    return true;
}

}  // namespace btt

#ifdef BTT_CHECK
namespace btt {
BTT_CHECK_TU(check_record_fft_residue)
}  // namespace btt
#endif
