// Visibility simulator (Sec. 3): the flat-sky map times the primary beam
// (Eq. beam, the MWA tile's sinc^2 pattern, or Eq. A_G, its Gaussian
// approximation), then the direct DFT of Eq. vis at every baseline, with
// Q = 1 (visibilities in map units):
//
//   V(U) = sum over pixels of dtheta^2 A(theta) T(theta) exp(+i 2 pi U.theta),
//   pixel (row b, column a) at theta = ((a - m/2) dtheta, (b - m/2) dtheta).
//
// The phase separates, exp(i 2 pi U.theta) = exp(i 2 pi u theta_x) exp(i 2 pi v theta_y), so
// every visibility's sum is a product of matrices: per row b of the map the real-by-complex
// product R[b] = sum_a W[b][a] exp(i 2 pi u theta_a), two multiply-adds a term, then
// V = sum_b exp(i 2 pi v theta_b) R[b].  A thread owns two visibilities and SIM_A columns whose
// column phases it keeps in registers while it walks the rows (k_dft); the column blocks and
// the row ranges are spread over CTAs and their partial sums added in a fixed order
// (k_dft_reduce).  The phases (hundreds of cycles for baselines of hundreds of wavelengths
// over a radian) are carried as double-float pairs and reduced to their fractional cycle
// before the FP32 sine and cosine.
#include <algorithm>

#include "abs_internal.cuh"

namespace absk {
namespace {

constexpr int SIM_T = 128;       // threads per CTA
constexpr int SIM_V = 2;         // visibilities of a thread
constexpr int SIM_A = 32;        // map columns of a thread (their phases: 2 x SIM_A x SIM_V registers)
constexpr int SIM_R = 4;         // map rows walked together
constexpr int SIM_ROWS = 32;     // map rows staged in shared memory per pass

__global__ void k_sky_weights(int m, double dth, const float *__restrict__ sky, int beam, double bp,
                              float *__restrict__ W) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)m * m) return;
    const int b = (int)(p / m), a = (int)(p - (int64_t)b * m);
    const double tx = (a - m / 2) * dth, ty = (b - m / 2) * dth;
    double A = 1.0;
    if (beam == ABS_BEAM_MWA_TILE) {
        const double x = bp * tx, y = bp * ty;   // sinc(x) = sin(pi x) / (pi x)
        const double sx = x == 0.0 ? 1.0 : sinpi(x) / (M_PI * x);
        const double sy = y == 0.0 ? 1.0 : sinpi(y) / (M_PI * y);
        A = sx * sx * sy * sy;
    } else if (beam == ABS_BEAM_GAUSS) {
        A = exp(-(tx * tx + ty * ty) / (bp * bp));
    }
    W[p] = (float)(dth * dth * A * (double)sky[p]);
}

// x + y for double-float pairs (hi, lo): TwoSum of the high parts, low parts added.
__device__ __forceinline__ void df_add(float xh, float xl, float yh, float yl, float &zh, float &zl) {
    const float s = __fadd_rn(xh, yh);
    const float bp = __fsub_rn(s, xh);
    const float e = __fadd_rn(__fsub_rn(xh, __fsub_rn(s, bp)), __fsub_rn(yh, bp));
    const float t = __fadd_rn(e, __fadd_rn(xl, yl));
    zh = __fadd_rn(s, t);
    zl = __fsub_rn(t, __fsub_rn(zh, s));
}

// k x (hi, lo) for a small integer k, as a double-float pair.
__device__ __forceinline__ void df_scale(float h, float l, float k, float &zh, float &zl) {
    const float p = __fmul_rn(h, k);
    const float e = fmaf(h, k, -p);
    const float t = fmaf(l, k, e);
    zh = __fadd_rn(p, t);
    zl = __fsub_rn(t, __fsub_rn(zh, p));
}

// exp(i 2 pi phi) for a double-float phase phi in cycles: the fractional cycle f, |f| <= 1/2,
// to the nearest quarter turn q and the rest r, |r| <= 1/8, then the Taylor series of sine and
// cosine on |2 pi r| <= pi / 4 (truncation below 2e-9) turned by q quarters.  About 1e-7 at
// most, without the FP64 pipe sincospif keeps busy here or the 4e-7 of the SFU's __sincosf.
__device__ __forceinline__ float2 cis_cycles(float h, float l) {
    const float f = __fadd_rn(__fsub_rn(h, rintf(h)), l);
    const float qf = rintf(4.0f * f);
    const float t = 6.28318531f * fmaf(-0.25f, qf, f), t2 = t * t;
    float s = fmaf(t2, 2.75573192e-6f, -1.98412698e-4f);
    s = fmaf(t2, s, 8.33333333e-3f);
    s = fmaf(t2, s, -1.66666667e-1f);
    s = fmaf(t * t2, s, t);
    float c = fmaf(t2, -2.75573192e-7f, 2.48015873e-5f);
    c = fmaf(t2, c, -1.38888889e-3f);
    c = fmaf(t2, c, 4.16666667e-2f);
    c = fmaf(t2, c, -0.5f);
    c = fmaf(t2, c, 1.0f);
    const int q = (int)qf;
    const float a = (q & 1) ? s : c, b = (q & 1) ? c : s;   // |cos|, |sin| after the quarter turns
    return make_float2(((q + 1) & 2) ? -a : a, (q & 2) ? -b : b);
}

// k (h, l) cycles for an integer k, |k| <= 8192.
__device__ __forceinline__ float2 cis_multiple(float h, float l, int k) {
    float zh, zl;
    df_scale(h, l, (float)k, zh, zl);
    return cis_cycles(zh, zl);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// SIM_V visibilities a thread, SIM_A columns from blockIdx.y SIM_A, rows [blockIdx.z rows_per, + rows_per):
// their sums over them as double-float pairs (re.hi, re.lo, im.hi, im.lo) in part[z gridDim.y + y][vis].
// Per term one half of a packed FFMA2 (two columns) for each of re and im; one map load (LDS.128, a
// broadcast) serves four FFMA2 of each visibility.  The columns' phases take 243 registers a thread, so two
// CTAs an SM: issue 53 %, the FMA pipe 43 %, what is between is the chains' latency (100,000 visibilities of
// 256^2: 0.60 ms against 0.33 of multiply-adds).  The columns' FP32 sums run in chains of
// SIM_A / 2 terms, eight rows' terms are added in FP32 and everything beyond in double-float; a row
// phase is rotated from the one SIM_R rows before, at most SIM_ROWS / SIM_R times from an exact one.
__global__ void __launch_bounds__(SIM_T) k_dft(int m, double dth, const float *__restrict__ W, int64_t n_vis,
                                               const float2 *__restrict__ uv, int rows_per,
                                               float4 *__restrict__ part) {
    __shared__ __align__(16) float ws[SIM_ROWS][SIM_A];
    const int64_t e = (int64_t)blockIdx.x * (SIM_T * SIM_V) + threadIdx.x;
    const int a0 = blockIdx.y * SIM_A, b0 = blockIdx.z * rows_per, b1 = min(m, b0 + rows_per);
    float cvh[SIM_V], cvl[SIM_V];                    // v dtheta in cycles as a double-float pair (from the FP64 product)
    float2 xr[SIM_V][SIM_A / 2], xi[SIM_V][SIM_A / 2];   // the columns' phases, two neighbours to a pair
    float2 turn[SIM_V][SIM_R];                       // one to SIM_R rows further
#pragma unroll
    for (int n = 0; n < SIM_V; ++n) {
        const int64_t en = e + n * SIM_T;
        const float2 U = en < n_vis ? uv[en] : make_float2(0.f, 0.f);
        const double cu = (double)U.x * dth, cv = (double)U.y * dth;
        const float cuh = (float)cu, cul = (float)(cu - (double)cuh);
        cvh[n] = (float)cv;
        cvl[n] = (float)(cv - (double)cvh[n]);
#pragma unroll
        for (int k = 0; k < SIM_A / 2; ++k) {
            const float2 p = cis_multiple(cuh, cul, a0 + 2 * k - m / 2), q = cis_multiple(cuh, cul, a0 + 2 * k + 1 - m / 2);
            xr[n][k] = make_float2(p.x, q.x);
            xi[n][k] = make_float2(p.y, q.y);
        }
#pragma unroll
        for (int r = 0; r < SIM_R; ++r) turn[n][r] = cis_multiple(cvh[n], cvl[n], r + 1);
    }
    float reh[SIM_V] = {}, rel[SIM_V] = {}, imh[SIM_V] = {}, iml[SIM_V] = {};
    for (int r0 = b0; r0 < b1; r0 += SIM_ROWS) {
        const int nr = min(SIM_ROWS, b1 - r0);
        __syncthreads();
        for (int i = threadIdx.x; i < SIM_ROWS * SIM_A; i += SIM_T) {   // zeros past the map and the range
            const int r = i / SIM_A, a = i % SIM_A;
            ws[r][a] = r < nr && a0 + a < m ? W[(int64_t)(r0 + r) * m + a0 + a] : 0.f;
        }
        __syncthreads();
        float2 y[SIM_V], v[SIM_V];   // the phase of the first of SIM_R rows; the FP32 sum of up to 2 SIM_R rows
#pragma unroll
        for (int n = 0; n < SIM_V; ++n) {
            y[n] = cis_multiple(cvh[n], cvl[n], r0 - m / 2);
            v[n] = make_float2(0.f, 0.f);
        }
        for (int r = 0; r < nr; r += SIM_R) {
            float2 sr[SIM_V][SIM_R], si[SIM_V][SIM_R];
#pragma unroll
            for (int n = 0; n < SIM_V; ++n)
#pragma unroll
                for (int q = 0; q < SIM_R; ++q) sr[n][q] = si[n][q] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < SIM_A / 4; ++k) {
#pragma unroll
                for (int q = 0; q < SIM_R; ++q) {
                    const float4 w = ((const float4 *)ws[r + q])[k];
#pragma unroll
                    for (int n = 0; n < SIM_V; ++n) {
                        sr[n][q] = __ffma2_rn(make_float2(w.x, w.y), xr[n][2 * k], sr[n][q]);
                        si[n][q] = __ffma2_rn(make_float2(w.x, w.y), xi[n][2 * k], si[n][q]);
                        sr[n][q] = __ffma2_rn(make_float2(w.z, w.w), xr[n][2 * k + 1], sr[n][q]);
                        si[n][q] = __ffma2_rn(make_float2(w.z, w.w), xi[n][2 * k + 1], si[n][q]);
                    }
                }
            }
#pragma unroll
            for (int n = 0; n < SIM_V; ++n) {
                float2 z = make_float2(sr[n][0].x + sr[n][0].y, si[n][0].x + si[n][0].y);
#pragma unroll
                for (int q = 1; q < SIM_R; ++q) {
                    const float2 t = cmul(turn[n][q - 1], make_float2(sr[n][q].x + sr[n][q].y, si[n][q].x + si[n][q].y));
                    z = make_float2(z.x + t.x, z.y + t.y);
                }
                z = cmul(y[n], z);
                y[n] = cmul(y[n], turn[n][SIM_R - 1]);
                v[n] = make_float2(v[n].x + z.x, v[n].y + z.y);
                if ((r & SIM_R) || r + SIM_R >= nr) {
                    df_add(reh[n], rel[n], v[n].x, 0.f, reh[n], rel[n]);
                    df_add(imh[n], iml[n], v[n].y, 0.f, imh[n], iml[n]);
                    v[n] = make_float2(0.f, 0.f);
                }
            }
        }
    }
#pragma unroll
    for (int n = 0; n < SIM_V; ++n)
        if (e + n * SIM_T < n_vis)
            part[((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * n_vis + e + n * SIM_T] =
                make_float4(reh[n], rel[n], imh[n], iml[n]);
}

// The parts of a visibility added in order.
__global__ void __launch_bounds__(256) k_dft_reduce(int64_t n_vis, int parts, const float4 *__restrict__ part,
                                                    float2 *__restrict__ vis) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_vis) return;
    float reh = 0.f, rel = 0.f, imh = 0.f, iml = 0.f;
    for (int k = 0; k < parts; ++k) {
        const float4 p = part[k * n_vis + e];
        df_add(reh, rel, p.x, p.y, reh, rel);
        df_add(imh, iml, p.z, p.w, imh, iml);
    }
    vis[e] = make_float2(__fadd_rn(reh, rel), __fadd_rn(imh, iml));
}

}  // namespace

abs_status launch_simulate_vis(abs_ctx *ctx, int32_t m, double dtheta, const float *d_sky, int32_t beam,
                               double beam_param, int64_t n_vis, const float *d_uv, float *d_vis) {
    const int64_t npix = (int64_t)m * m;
    float *W = (float *)workspace(ctx, "sim.weights", sizeof(float) * (size_t)npix);
    if (!W) return fail(ctx, ABS_ERR_OOM, "simulator workspace");
    // column blocks and row ranges (whole staged passes) so that the launch holds about eight waves
    // of CTAs, two to an SM by their registers; the visibilities in slabs whose parts take `room` bytes at most
    const int ny = (int)cdiv(m, SIM_A);
    int64_t slab = 0;
    int rows_per = 0, nz = 0;
    auto shape = [&](int64_t room) {
        const int64_t fit = room / (int64_t)sizeof(float4) / ny, unit = SIM_T * SIM_V;
        slab = std::min<int64_t>(n_vis, std::max<int64_t>(fit < unit ? fit : fit / unit * unit, 1));
        const int64_t ctas = std::max<int64_t>(cdiv(slab, unit) * ny, 1), most = slab > 0 ? std::max<int64_t>(fit / slab, 1) : 1;
        const int want = (int)std::min(std::min<int64_t>(cdiv(m, SIM_ROWS), cdiv((int64_t)16 * ctx->sm_count, ctas)), most);
        rows_per = (int)cdiv(cdiv(m, want), SIM_ROWS) * SIM_ROWS;
        nz = (int)cdiv(m, rows_per);
        return sizeof(float4) * (size_t)(ny * nz) * (size_t)slab;
    };
    // 256 MB, or as much as there is: less if the device has not the room, and what an earlier call left in a
    // stream that is being captured, where nothing can be allocated
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &capturing) != cudaSuccess) cudaGetLastError();
    const bool fixed = capturing != cudaStreamCaptureStatusNone;
    const size_t have = ctx->ws["sim.parts"].bytes, least = sizeof(float4) * (size_t)ny;   // one visibility
    size_t bytes = shape((int64_t)256 << 20);
    if (fixed && bytes > have && have >= least) bytes = shape((int64_t)have);
    float4 *part = (float4 *)workspace(ctx, "sim.parts", bytes);
    for (size_t room = bytes / 2; !part && !fixed && room >= least; room /= 2)
        part = (float4 *)workspace(ctx, "sim.parts", shape((int64_t)room));
    if (!part) return fail(ctx, ABS_ERR_OOM, "simulator workspace");
    StageTimer timer(ctx, "simulate_vis");
    k_sky_weights<<<(unsigned)cdiv(npix, 256), 256, 0, ctx->stream>>>(m, dtheta, d_sky, beam, beam_param, W);
    for (int64_t v0 = 0; v0 < n_vis; v0 += slab) {
        const int64_t nv = std::min(slab, n_vis - v0);
        k_dft<<<dim3((unsigned)cdiv(nv, SIM_T * SIM_V), ny, nz), SIM_T, 0, ctx->stream>>>(m, dtheta, W, nv, (const float2 *)d_uv + v0,
                                                                                rows_per, part);
        k_dft_reduce<<<(unsigned)cdiv(nv, 256), 256, 0, ctx->stream>>>(nv, ny * nz, part, (float2 *)d_vis + v0);
    }
    return check_launch(ctx, "visibility simulator");
}

}  // namespace absk
