// Per-frequency products for several right-hand sides on the FP32 units:
//     F :  dhat_n[w][s] = sum_l Fhat[w][s][l] xhat_n[w][l]
//     F*:  mhat_n[w][l] = sum_s conj(Fhat[w][s][l]) dhat_n[w][s]
// for groups of up to 8 vectors n that share one pass over Fhat.  An entry
// feeds 8 flops per vector: at 256 x 200 x 10000 and 8 vectors 0.44 ms of FP32
// time (128 lanes per SM and clock) against 0.61 ms of HBM time for complex64,
// 0.30 for the 4-byte formats and 0.15 for FP8, so the floor is HBM's in FP32
// (up to 11 vectors) and the FP32 units' in the others (from 6 and 3 vectors
// on).  What the kernels are bound by there is issue and latency (issue active
// 63-68%, FMA pipe 47-51%).
// Both kernels spare what stands beside the multiply-adds: a value read from
// shared memory serves four rows (F) or a 16-byte unit of columns (F*).  The
// arithmetic is scalar: paired f32x2 instructions need each Fhat value
// duplicated and each vector value swapped, and those register moves take
// the FMA pipe too (F at 8 vectors 1.44 ms against 1.21 at the same tiling).
//
// Rows on their way are first brought to L2 (cp.async.bulk.prefetch), so the
// 16-20 warps an SM holds at 96-128 registers cover the latency of an L2
// hit and not of HBM (F* at 4 vectors 686 -> 600 us).
//
// 256 x 200 x 10000 (Fhat 4.1 GB in FP32: 0.61 ms of HBM time; 8 vectors:
// 0.44 ms of FP32 time), kernels of gemv_kernels.cu -> these, us per launch:
//   FP32  F  3 vectors 779 -> 661, 8 1513 -> 1004, 32 5890 -> 3807
//         F* 3 vectors 686 -> 595, 8 1062 -> 828, 32 3653 -> 3143
//         F 5 vectors 1493 -> 738, 7 1513 -> 902 (a group's kernel has its own count)
//   BF16  F  8 vectors 1456 -> 983;   F* 8 vectors 860 -> 773
//   FP8   F  8 vectors 1997 -> 905;   F* 8 vectors 800 -> 726
//
// F* sums along s, F per lane along l and then over the lanes in the tree of
// the single-vector kernels; where warps share a row (fwd_slices) every F of the
// operator does.  A vector's result does not depend on the batch it is in.
#include <utility>

#include "gemv_store.cuh"

namespace btt {

// Two neighbouring complex values (16-byte piece h of VPL/2) of a raw unit.
template <int PREC> __device__ __forceinline__ void decode2(const typename Store<PREC>::raw& q, int h, float2 (&f)[2])
{
    if constexpr (PREC == P_F32) {
        f[0] = make_float2(q.x, q.y);
        f[1] = make_float2(q.z, q.w);
    } else if constexpr (PREC == P_BF16X2) {
        const unsigned hw[2] = {h ? q.h.z : q.h.x, h ? q.h.w : q.h.y};
        const unsigned lw[2] = {h ? q.l.z : q.l.x, h ? q.l.w : q.l.y};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw[i]));
            const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&lw[i]));
            f[i] = make_float2(a.x + b.x, a.y + b.y);
        }
    } else if constexpr (PREC == P_FP8S) {
        const unsigned w = h == 0 ? q.x : h == 1 ? q.y : h == 2 ? q.z : q.w;
        f[0] = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w & 0xFFFFu), __NV_E4M3)));
        f[1] = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w >> 16), __NV_E4M3)));
    } else {
        const unsigned w[2] = {h ? q.z : q.x, h ? q.w : q.y};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if constexpr (PREC == P_F16S) f[i] = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
            else f[i] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
        }
    }
}

// Asks for `bytes` (a multiple of 16) from p on to be brought into L2.
__device__ __forceinline__ void l2_prefetch(const void* p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ------------------------------------------------------------ F (Alg. 2)
// CTA = rg warps x 4 rows of one frequency (or 8 warps that share the blocks
// of 4 rows, wk = 8, where rows and frequencies are few) for a group of NB
// vectors; the
// group is the fastest grid dimension, so CTAs sharing a Fhat tile run
// together and repeats hit L2 (the kernel it replaces read Fhat twice from
// HBM at 8 vectors).  A warp streams its rows with 16-byte loads, the next
// block's requested before the current one is used; the group's mhat(w) goes
// through shared memory in chunks of `ch` values per vector (cp.async,
// double buffered), its 16-byte pieces permuted so that the lanes of a warp
// read consecutive ones whatever the unit's width.  Four rows per value
// read: two would need 128 bytes per clock at the full FP32 rate, all the
// shared pipe has.
constexpr int kFwdRows = 4, kFwdWarps = 8;
constexpr int kFwdSmemMax = 128 * 1024;   // set by prepare_gemv_multi

// Whether two blocks' raw units fit beside the accumulators in 128 registers,
// and whether 80 registers (three CTAs of 8 warps per SM) hold the kernel.
// (Most spill up to 36 bytes; FP16 with 8 vectors 156.)
template <int PREC, int NB> constexpr bool fwd_pipelined()
{
    return PREC == P_BF16X2 ? NB <= 3 : (NB <= 6 || PREC == P_F32);
}
template <int PREC, int NB> constexpr int fwd_min_blocks()
{
    return NB <= 2 && PREC != P_BF16X2 ? 3 : (NB == 3 && PREC == P_F32 ? 3 : 2);
}

template <int PREC, int NB>
__global__ void __launch_bounds__(kFwdWarps * 32, (fwd_min_blocks<PREC, NB>()))
k_gemv_fwd_multi(const typename Store<PREC>::elem* __restrict__ fhat, const float* __restrict__ scales, int N_d,
                 int ldm, const float2* __restrict__ xh, int64_t xbs, float2* __restrict__ dh, int64_t dbs, int nrhs,
                 int per, int rg, int wk, int ch, int its_log2, int64_t lo_off)
{
    using S = Store<PREC>;
    using Raw = typename S::raw;
    constexpr int VPL = S::VPL, BLK = 32 * VPL, R = kFwdRows;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* sx = reinterpret_cast<float4*>(smem_raw);   // [2][NB][ch / 2] 16-byte pieces
    const int w = blockIdx.z, b0 = blockIdx.x * per;
    const int nv = min(per, nrhs - b0);                 // vectors of this group (<= NB)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int row_warp = wid % rg, slice = wid / rg;    // this warp's rows and its share of the blocks
    const int r0 = (blockIdx.y * rg + row_warp) * R;
    const bool live = r0 < N_d;
    const int last = N_d - 1 - r0;   // rows past the last one repeat it (their sums are not stored)
    const typename S::elem* row0 = fhat + ((int64_t)w * N_d + min(r0, N_d - 1)) * ldm + lane * VPL;
    int off[R];
#pragma unroll
    for (int r = 0; r < R; ++r) off[r] = max(0, min(r, last)) * ldm;
    const int hp = ch / 2;
    const int nch = (ldm + ch - 1) / ch, nblk = (ldm + BLK - 1) / BLK, nfull = ldm / BLK;

    const float2* x0 = xh + (int64_t)b0 * xbs + (int64_t)w * ldm;
    auto stage = [&](int c) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(sx + (c & 1) * NB * hp);
        for (int i = threadIdx.x; i < hp; i += blockDim.x) {
            const int k = c * ch + 2 * i;
            const int in = i % (BLK / 2);   // piece h of lane `in / (VPL/2)`
            const int at = i - in + (in % (VPL / 2)) * 32 + in / (VPL / 2);
            const float2* src = x0 + (k < ldm ? k : 0);
#pragma unroll
            for (int n = 0; n < NB; ++n) {
                const bool ok = n < nv && k < ldm;   // else zeros
                if (!BTT_IN(at, hp, CK_GEMV_SMEM)) continue;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (n * hp + at) * 16),
                             "l"(ok ? src + (int64_t)n * xbs : x0), "r"(ok ? 16 : 0)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the pieces of the warp's rows kAhead blocks on, on their way to L2
    constexpr int kAhead = 8;
    const bool asks = lane < R && lane <= last;
    const typename S::elem* prow = fhat + ((int64_t)w * N_d + min(r0 + (asks ? lane : 0), N_d - 1)) * ldm;
    auto prefetch = [&](int g) {
        const int n = min(BLK, ldm - g * BLK);
        if (!asks || n <= 0) return;
        l2_prefetch(prow + g * BLK, n * (unsigned)sizeof(typename S::elem));
        if (PREC == P_BF16X2) l2_prefetch(prow + g * BLK + lo_off, n * (unsigned)sizeof(typename S::elem));
    };

    float2 acc[R][NB];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NB; ++n) acc[r][n] = make_float2(0.f, 0.f);

    auto block = [&](const Raw (&q)[R], const float4* sb) {
#pragma unroll
        for (int h = 0; h < VPL / 2; ++h) {
            float2 f[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r) decode2<PREC>(q[r], h, f[r]);
#pragma unroll
            for (int n = 0; n < NB; ++n) {
                const float4 x = sb[n * hp + h * 32];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    cfma(acc[r][n], f[r][0], make_float2(x.x, x.y));
                    cfma(acc[r][n], f[r][1], make_float2(x.z, x.w));
                }
            }
        }
    };

    int c = -1;   // chunk in use
    auto advance = [&]() {
        // the next chunk has arrived; everyone is done with the one before
        ++c;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (c + 1 < nch) stage(c + 1);
    };
    auto load = [&](Raw (&q)[R], int g) {
#pragma unroll
        for (int r = 0; r < R; ++r) q[r] = S::load_raw(row0 + ((unsigned)off[r] + (unsigned)(g * BLK)), lo_off);
    };
    auto use = [&](const Raw (&q)[R], int g) {
        while (c < g >> its_log2) advance();
        prefetch(g + kAhead);
        block(q, sx + (c & 1) * NB * hp + lane + (g - (c << its_log2)) * (BLK / 2));
    };

    stage(0);
    if (live) {
        for (int g = slice; g < kAhead; g += wk) prefetch(g);
        int g = slice;
        Raw qa[R];
        if constexpr (fwd_pipelined<PREC, NB>()) {
            // one block's units are requested before the block ahead of it is used
            Raw qb[R];
            if (g < nfull) load(qa, g);
            while (g < nfull) {
                if (g + wk < nfull) load(qb, g + wk);
                use(qa, g);
                g += wk;
                if (g >= nfull) break;
                if (g + wk < nfull) load(qa, g + wk);
                use(qb, g);
                g += wk;
            }
        } else {
            for (; g < nfull; g += wk) {
                load(qa, g);
                use(qa, g);
            }
        }
        if (g == nfull && nfull < nblk) {   // the last, partial block (ldm is a multiple of VPL)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                qa[r] = Raw{};
                if ((g * 32 + lane) * VPL < ldm && BTT_IN((g * 32 + lane) * VPL + VPL - 1, ldm, CK_GEMV_FHAT))
                    qa[r] = S::load_raw(row0 + ((unsigned)off[r] + (unsigned)(g * BLK)), lo_off);
            }
            use(qa, g);
        }
    }
    while (c < nch - 1) advance();
    constexpr int CNT = R * NB * 2;
    float v[CNT];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            v[(r * NB + n) * 2] = acc[r][n].x;
            v[(r * NB + n) * 2 + 1] = acc[r][n].y;
        }
    using LS = LaneSum<CNT, 16>;
    int base = 0;
    LS::run(v, lane, base);
    const float sc = (PREC == P_F16S || PREC == P_FP8S) ? scales[w] : 1.f;
    auto put = [&](int j, float a) {
        const int c = j & 1, n = (j >> 1) % NB, r = (j >> 1) / NB;
        if (n < nv && r0 + r < N_d && BTT_IN((int64_t)w * N_d + r0 + r, dbs, CK_GEMV_VEC))
            reinterpret_cast<float*>(dh + (int64_t)(b0 + n) * dbs + (int64_t)w * N_d + r0 + r)[c] = a * sc;
    };
    if (wk == 1) {
        if (live && !(lane & LS::kDup))
#pragma unroll
            for (int i = 0; i < LS::kLeft; ++i) put(base + i, v[i]);
        return;
    }
    // the slices' sums, added in their order
    float* red = reinterpret_cast<float*>(smem_raw);   // [warp][CNT]
    __syncthreads();
    if (!(lane & LS::kDup))
#pragma unroll
        for (int i = 0; i < LS::kLeft; ++i) red[wid * CNT + base + i] = v[i];
    __syncthreads();
    if (live && slice == 0)
        for (int j = lane; j < CNT; j += 32) {
            float a = red[row_warp * CNT + j];
            for (int k = 1; k < wk; ++k) a += red[(k * rg + row_warp) * CNT + j];
            put(j, a);
        }
}

// ----------------------------------------------------------- F* (Alg. 3)
// CTA = 128 threads, each the VPL columns of one 16-byte unit, for one
// frequency and a group of NB vectors; a thread walks the N_d rows with UNR
// units requested together (a rolling request per used unit was half as
// fast: the loads in flight then share scoreboards with newer ones) and
// dhat(w) broadcast from shared memory.
constexpr int kAdjThreads = 128;
constexpr int kAdjSmem = 16 * 1024;

template <int PREC, int NB> constexpr int adj_unroll()
{
    return PREC == P_BF16X2 ? 4 : (Store<PREC>::VPL * NB >= 32 ? 6 : 8);
}
template <int PREC, int NB> constexpr int adj_min_blocks()
{
    // 128 registers for 16 or more complex accumulators, 96 below
    return Store<PREC>::VPL * NB >= 16 ? 4 : 5;
}

template <int PREC, int NB>
__global__ void __launch_bounds__(kAdjThreads, adj_min_blocks<PREC, NB>())
k_gemv_adj_multi(const typename Store<PREC>::elem* __restrict__ fhat, const float* __restrict__ scales, int N_d,
                 int N_m, int ldm, const float2* __restrict__ dh, int64_t dbs, float2* __restrict__ mh, int64_t mbs,
                 int nrhs, int per, int sc_rows, int64_t lo_off)
{
    using S = Store<PREC>;
    using Raw = typename S::raw;
    constexpr int VPL = S::VPL, UNR = adj_unroll<PREC, NB>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sd = reinterpret_cast<float2*>(smem_raw);   // [sc_rows][NB]
    const int w = blockIdx.z, b0 = blockIdx.x * per;
    const int nv = min(per, nrhs - b0);
    const int k = (blockIdx.y * kAdjThreads + threadIdx.x) * VPL;
    const bool live = k < ldm && BTT_IN(k + VPL - 1, ldm, CK_GEMV_FHAT);
    const float sc = (PREC == P_F16S || PREC == P_FP8S) ? scales[w] : 1.f;
    const typename S::elem* p = fhat + (int64_t)w * N_d * ldm + (live ? k : 0);

    float2 acc[VPL][NB];
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
        for (int n = 0; n < NB; ++n) acc[v][n] = make_float2(0.f, 0.f);
    // rows to come on their way to L2: one request per row of this CTA's columns
    constexpr int kAhead = 24;
    const int k0 = blockIdx.y * kAdjThreads * VPL;
    const unsigned seg = (unsigned)(min(kAdjThreads * VPL, ldm - k0) * (int)sizeof(typename S::elem));
    auto prefetch = [&](int s) {
        if (s >= N_d) return;
        const typename S::elem* at = fhat + ((int64_t)w * N_d + s) * ldm + k0;
        l2_prefetch(at, seg);
        if (PREC == P_BF16X2) l2_prefetch(at + lo_off, seg);
    };
    if (threadIdx.x >= UNR && threadIdx.x < kAhead) prefetch(threadIdx.x);
    for (int c0 = 0; c0 < N_d; c0 += sc_rows) {   // sc_rows: N_d, or a multiple of UNR
        const int end = min(c0 + sc_rows, N_d);
        if (c0) __syncthreads();
        for (int i = threadIdx.x; i < NB * (end - c0); i += kAdjThreads) {
            const int n = i / (end - c0), s = i - n * (end - c0);
            float2 v = make_float2(0.f, 0.f);
            if (n < nv && BTT_IN((int64_t)w * N_d + c0 + s, dbs, CK_GEMV_VEC))
                v = dh[(int64_t)(b0 + n) * dbs + (int64_t)w * N_d + c0 + s];
            v = cscale(v, sc);
            if (BTT_IN(s * NB + n, sc_rows * NB, CK_GEMV_SMEM)) sd[s * NB + n] = v;
        }
        __syncthreads();
        if (!live) continue;
        auto row = [&](const Raw& cur, int s) {
            const float2* sr = sd + (s - c0) * NB;
#pragma unroll
            for (int h = 0; h < VPL / 2; ++h) {
                float2 f[2];
                decode2<PREC>(cur, h, f);
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    const float2 d = sr[n];
                    cfma_conj(acc[2 * h][n], f[0], d);
                    cfma_conj(acc[2 * h + 1][n], f[1], d);
                }
            }
        };
        int s = c0;
        for (; s + UNR <= end; s += UNR) {
            Raw q[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) q[u] = S::load_raw(p + (int64_t)u * ldm, lo_off);
            p += (int64_t)UNR * ldm;
            if (threadIdx.x < UNR) prefetch(s + kAhead + threadIdx.x);
#pragma unroll
            for (int u = 0; u < UNR; ++u) row(q[u], s + u);
        }
        if (s < end) {   // the last rows, requested together as well
            Raw q[UNR - 1];
#pragma unroll
            for (int u = 0; u < UNR - 1; ++u)
                if (s + u < end) q[u] = S::load_raw(p + (int64_t)u * ldm, lo_off);
#pragma unroll
            for (int u = 0; u < UNR - 1; ++u)
                if (s + u < end) row(q[u], s + u);
            p += (int64_t)(end - s) * ldm;
        }
    }
    if (!live) return;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        if (n >= nv) break;
        float2* out = mh + (int64_t)(b0 + n) * mbs + (int64_t)w * ldm + k;
        // columns past N_m keep the workspace's zeros
        if (k + VPL <= N_m && BTT_IN((int64_t)w * ldm + k + VPL - 1, mbs, CK_GEMV_VEC)) {
#pragma unroll
            for (int v = 0; v < VPL; v += 2)
                *reinterpret_cast<float4*>(out + v) = make_float4(acc[v][n].x, acc[v][n].y, acc[v + 1][n].x, acc[v + 1][n].y);
        } else {
#pragma unroll
            for (int v = 0; v < VPL; ++v)
                if (k + v < N_m) out[v] = acc[v][n];
        }
    }
}

// ---------------------------------------------------------------- launchers
// Warps that share a row of F along l (blocks g, g + 8, ... each): 1, or 8 where
// rows and frequencies are few and the rows long, so that a warp's walk along
// its row is what the launch waits for.  A function of the operator alone: the
// order in which a row is summed must not depend on the batch a vector is in,
// so in those shapes a single vector comes here as well.  Measured (us, one
// warp per row in gemv_kernels.cu -> 8 here, 1 / 2 / 8 / 32 vectors):
//   65 x 7 x 20000    FP32 35 / 61 / 113 / 150 -> 21 / 25 / 43 / 119, BF16 41 / 72 / 131 / 163 ->
//                     17 / 28 / 60 / 197, split pairs 68 / 121 / 141 / 175 -> 21 / 29 / 81 / 265,
//                     FP8 49 / 90 / 103 / 204 -> 15 / 23 / 62 / 196
//   17 x 7 x 2500     FP32 6.3 / 8.3 / 10.5 / 10.5 -> 6.4 / 6.4 / 6.3 / 8.5, BF16 7.7 / 8.4 / 12.4 /
//                     12.5 -> 6.3 / 8.2 / 8.2 / 12.5
// Beyond these lines it loses (mean over 1 .. 32 vectors, time on 8 over the
// better kernel of one warp): FP32 at 457-608 row groups up to 1.15, up to 12
// blocks 1.0-1.15; 16-bit formats and pairs at 153-304 groups 1.06-1.2 up to 40
// blocks, at 305-456 1.1-1.4; FP8 at 153-304 1.03-1.24.
int fwd_slices(int prec, int n_freq, int N_d, int ldm)
{
    const int64_t groups = (int64_t)n_freq * ((N_d + kFwdRows - 1) / kFwdRows);
    const int blk = prec == P_F32 ? 64 : (prec == P_FP8S ? 256 : 128), nblk = (ldm + blk - 1) / blk;
    const bool yes = prec == P_F32    ? groups <= 456 && nblk > 12
                     : prec == P_FP8S ? groups <= 152 && nblk > 12
                                      : (groups <= 152 && nblk > 12) || (groups <= 304 && nblk > 40);
    return yes ? kFwdWarps : 1;
}

template <int PREC, int NB>
static cudaError_t fwd_multi(const void* fhat, const float* scales, int n_freq, int N_d, int ldm, const void* xh,
                             int64_t xbs, void* dh, int64_t dbs, int nrhs, int per, int wk, cudaStream_t st)
{
    using S = Store<PREC>;
    constexpr int BLK = 32 * S::VPL;
    const int nblk = (ldm + BLK - 1) / BLK;
    // Row groups of 4 spread evenly over tiles of at most 8 warps.
    const int groups = (N_d + kFwdRows - 1) / kFwdRows;
    const int64_t vg = (nrhs + per - 1) / per;
    int tiles = (groups + kFwdWarps - 1) / kFwdWarps;
    const int rg = wk > 1 ? 1 : (groups + tiles - 1) / tiles;
    tiles = (groups + rg - 1) / rg;
    // Values per chunk: 512, less for CTAs of up to 4 warps, so that 16 warps of
    // them fit (FP32) or one block (the formats that decode: few values arrive
    // sooner than many; us at 512 / 256 / 128 values): 257 x 10 x 7648, BF16, 3
    // vectors 50 / 48 / 45, 631 x 4 x 2923 25 / 25 / 23; FP32, 8 vectors, 2001 x 2 x
    // 390 25 / 18 / 15.  A block for every warp that shares a row.
    int ch = wk > 1 ? wk * BLK : rg > 4 || PREC == P_F32 ? 512 : BLK;
    while (wk == 1 && ch > BLK && (size_t)2 * NB * ch * sizeof(float2) * (16 / rg) > 220 * 1024) ch /= 2;
    int its_log2 = 0;   // blocks per chunk
    while ((BLK << its_log2) < ch) ++its_log2;
    if (nblk * BLK < ch) ch = nblk * BLK;   // a single chunk
    const size_t need = wk > 1 ? (size_t)wk * kFwdRows * NB * 2 * sizeof(float) : 0;
    size_t sm = (size_t)2 * NB * ch * sizeof(float2);
    if (sm < need) sm = need;
    dim3 grid((unsigned)vg, tiles, n_freq);
    k_gemv_fwd_multi<PREC, NB><<<grid, rg * wk * 32, sm, st>>>(
        static_cast<const typename S::elem*>(fhat), scales, N_d, ldm, static_cast<const float2*>(xh), xbs,
        static_cast<float2*>(dh), dbs, nrhs, per, rg, wk, ch, its_log2, lo_plane(PREC, n_freq, N_d, ldm));
    count_launch();
    return cudaGetLastError();
}

template <int PREC, int NB>
static cudaError_t adj_multi(const void* fhat, const float* scales, int n_freq, int N_d, int N_m, int ldm,
                             const void* dh, int64_t dbs, void* mh, int64_t mbs, int nrhs, int per, cudaStream_t st)
{
    using S = Store<PREC>;
    constexpr int UNR = adj_unroll<PREC, NB>();
    const int cols = kAdjThreads * S::VPL, cap = kAdjSmem / (8 * NB) / UNR * UNR;
    const int rows = N_d < cap ? N_d : cap;
    dim3 grid((nrhs + per - 1) / per, (ldm + cols - 1) / cols, n_freq);
    k_gemv_adj_multi<PREC, NB><<<grid, kAdjThreads, (size_t)rows * NB * sizeof(float2), st>>>(
        static_cast<const typename S::elem*>(fhat), scales, N_d, N_m, ldm, static_cast<const float2*>(dh), dbs,
        static_cast<float2*>(mh), mbs, nrhs, per, rows, lo_plane(PREC, n_freq, N_d, ldm));
    count_launch();
    return cudaGetLastError();
}

// Vectors per group (at most `cap`): the split whose waves of CTAs cost
// least, a CTA's time taken as proportional to its vectors plus one (the
// pass over Fhat).  Large grids take the fewest groups; a grid below one
// wave is widened by smaller groups, and a nearly empty last wave avoided.
static int group_size(int nrhs, int cap, int64_t ctas, int resident)
{
    int best = 0;
    int64_t cost = 0;
    for (int most = cap; most >= 2; --most) {   // (a batch may hold thousands of vectors)
        const int g = (nrhs + most - 1) / most, per = (nrhs + g - 1) / g;
        const int64_t c = (g * ctas + 152 * resident - 1) / (152 * resident) * (per + 1);
        if (!best || c < cost) best = per, cost = c;
    }
    return best;
}

template <int PREC>
static cudaError_t fwd_groups(const void* fhat, const float* scales, int n_freq, int N_d, int ldm, const void* xh,
                              int64_t xbs, void* dh, int64_t dbs, int nrhs, cudaStream_t st)
{
    const int wk = fwd_slices(PREC, n_freq, N_d, ldm), groups = (N_d + kFwdRows - 1) / kFwdRows;
    // (split pairs: a raw unit takes 8 registers, three vectors fill the rest;
    // 8 warps along a row: their chunk in 128 KB, one CTA per SM counted)
    const int cap = PREC == P_BF16X2 ? 3 : wk == 1 || PREC == P_F32 ? 8 : PREC == P_FP8S ? 4 : 5;
    const int per = nrhs == 1 ? 1
                    : wk > 1  ? group_size(nrhs, cap, (int64_t)n_freq * groups, 1)
                              : group_size(nrhs, cap, (int64_t)n_freq * ((groups + kFwdWarps - 1) / kFwdWarps), 2);
#define BTT_FWD(NB) \
    if (per <= NB) return fwd_multi<PREC, NB>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, per, wk, st)
    BTT_FWD(1);
    BTT_FWD(2);
    BTT_FWD(3);
    if constexpr (PREC != P_BF16X2) {
        BTT_FWD(4);
        BTT_FWD(5);
        BTT_FWD(6);
        BTT_FWD(7);
        BTT_FWD(8);
    }
#undef BTT_FWD
    return cudaErrorInvalidValue;
}

template <int PREC>
static cudaError_t adj_groups(const void* fhat, const float* scales, int n_freq, int N_d, int N_m, int ldm,
                              const void* dh, int64_t dbs, void* mh, int64_t mbs, int nrhs, cudaStream_t st)
{
    // FP8 units hold 8 columns: 4 vectors fill the accumulators
    const int cols = kAdjThreads * Store<PREC>::VPL;
    const int per = group_size(nrhs, PREC == P_FP8S ? 4 : 8, (int64_t)n_freq * ((ldm + cols - 1) / cols), 4);
#define BTT_ADJ(NB) \
    if (per <= NB) return adj_multi<PREC, NB>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, per, st)
    BTT_ADJ(2);
    BTT_ADJ(3);
    BTT_ADJ(4);
    if constexpr (PREC != P_FP8S) {
        BTT_ADJ(5);
        BTT_ADJ(6);
        // (16-bit formats: 7 spills 64 bytes, which few rows do not make up for:
        // one shape, 2000 x 7 x 3000 FP16, 128 on 8 against 137 us)
        if (PREC == P_F32 || PREC == P_BF16X2 || N_d > 16) BTT_ADJ(7);
        BTT_ADJ(8);
    }
#undef BTT_ADJ
    return cudaErrorInvalidValue;
}

template <int PREC, int... NB> static cudaError_t fwd_limits(std::integer_sequence<int, NB...>)
{
    cudaError_t e = cudaSuccess;
    ((e = e != cudaSuccess ? e
                           : cudaFuncSetAttribute(k_gemv_fwd_multi<PREC, NB>,
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmemMax)),
     ...);
    return e;
}

// The largest a launch may ask for, once per context: the limit belongs to
// the kernel, so one set per launch to that launch's size may be lowered by
// another thread's launch before the first has been made.
cudaError_t prepare_gemv_multi()
{
    using Groups = std::integer_sequence<int, 1, 2, 3, 4, 5, 6, 7, 8>;
    cudaError_t e = fwd_limits<P_F32>(Groups{});
    if (e == cudaSuccess) e = fwd_limits<P_F16S>(Groups{});
    if (e == cudaSuccess) e = fwd_limits<P_BF16>(Groups{});
    if (e == cudaSuccess) e = fwd_limits<P_BF16X2>(std::integer_sequence<int, 1, 2, 3>{});
    if (e == cudaSuccess) e = fwd_limits<P_FP8S>(Groups{});
    return e;
}

cudaError_t launch_gemv_fwd_multi(int prec, const void* fhat, const float* scales, int n_freq, int N_d, int ldm,
                                  const void* xh, int64_t xbs, void* dh, int64_t dbs, int nrhs, cudaStream_t st)
{
    switch (prec) {
        case P_F32: return fwd_groups<P_F32>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, st);
        case P_F16S: return fwd_groups<P_F16S>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, st);
        case P_BF16: return fwd_groups<P_BF16>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, st);
        case P_BF16X2: return fwd_groups<P_BF16X2>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, st);
        case P_FP8S: return fwd_groups<P_FP8S>(fhat, scales, n_freq, N_d, ldm, xh, xbs, dh, dbs, nrhs, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_gemv_adj_multi(int prec, const void* fhat, const float* scales, int n_freq, int N_d, int N_m,
                                  int ldm, const void* dh, int64_t dbs, void* mh, int64_t mbs, int nrhs,
                                  cudaStream_t st)
{
    switch (prec) {
        case P_F32: return adj_groups<P_F32>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, st);
        case P_F16S: return adj_groups<P_F16S>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, st);
        case P_BF16: return adj_groups<P_BF16>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, st);
        case P_BF16X2: return adj_groups<P_BF16X2>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, st);
        case P_FP8S: return adj_groups<P_FP8S>(fhat, scales, n_freq, N_d, N_m, ldm, dh, dbs, mh, mbs, nrhs, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace btt

#ifdef BTT_CHECK
namespace btt {
BTT_CHECK_TU(check_record_gemv_multi)
}  // namespace btt
#endif
