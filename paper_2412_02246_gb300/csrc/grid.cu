// Stage 1: gridding of visibilities, Eq. vg (Sec. 2).
//
// V_g = sum_i w(U_g - U_i) V(U_i) over the (2r+1)^2 cells around each
// visibility's nearest grid point, every visibility also entered at -U_i with
// V*.  The mirror is applied after accumulation (G(g) + conj G(-g)), which is
// the same sum.
//
// Plan (per baseline set): key every visibility by its 16x16-cell uv tile and
// its cell in the tile and stable-sort positions and original indices by that
// key (LSD radix, two passes up to about 500^2 cells, three beyond); the
// sorted order is cut into work units of UMAX records (fewer for small sets, see grid_unit).
//
// Accumulation (per realisation): one CTA per unit stages the unit in shared
// memory, forms the 1-D Gaussian weights and cuts it into runs of
// visibilities that share a cell (and at every CHUNK-th record); a warp sums
// the (2r+1)^2 footprint cells of a run (lane per pair of footprint cells,
// compensated FP32, input order) and adds them to an FP64 grid.  A final pass
// applies the Hermitian mirror and writes the FP32 outputs.
//
// Weights: w = exp(-(dx - fx)^2 s) exp(-(dy - fy)^2 s), s = 1/(2 sigma^2),
// with the fractional offset f = u/dU - c carried as a float pair (the exact
// division residual) and the exponent argument formed in double-float, so
// that the only sizeable error is that of expf itself.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "abs_internal.cuh"

namespace absk {
namespace {

constexpr int TS = 16;                       // tile side in cells
constexpr int UMAX = 512;                    // visibilities per work unit
constexpr unsigned FULL = 0xffffffffu;

struct GridGeom {
    int n, half, r, ks, tt, off, kernel;
    float du, inv_du, s_hi, s_lo;
    bool by_inv;   // quotients by the correctly rounded reciprocal inv_du (see quotient)
};

// The key space of the plan: every nearest cell whose footprint can reach the grid
// (|c| <= half + r), or, with rings_only (the estimate), only those whose footprint can
// reach a ring cell (|c| <= R + r, R the largest |g_x| of a ring cell): a visibility
// outside adds to no cell the estimate reads, and the smaller key space sorts in fewer
// or narrower passes.  Cells keep their place in the full n x n accumulators either way.
GridGeom geom(const Setup &s, bool rings_only = false) {
    GridGeom g;
    g.n = s.n;
    g.half = s.half;
    g.r = s.kernel == ABS_KERNEL_NGP ? 0 : s.r;
    const int reach = rings_only ? std::min(s.half, std::max(s.R, 0)) : s.half;
    g.ks = 2 * (reach + g.r) + 1;
    g.tt = (int)cdiv(g.ks, TS);
    g.off = reach + g.r;
    g.kernel = s.kernel;
    g.du = s.du;
    // 1 / dU correctly rounded: of the FP32 neighbours of the rounded quotient the one with the smallest
    // |1 - y dU| (exact in FP64)
    g.inv_du = (float)(1.0 / (double)s.du);
    for (float y : {std::nextafter(g.inv_du, 0.f), std::nextafter(g.inv_du, INFINITY)})
        if (std::fabs(1.0 - (double)y * s.du) < std::fabs(1.0 - (double)g.inv_du * s.du)) g.inv_du = y;
    uint32_t bits;
    std::memcpy(&bits, &s.du, sizeof bits);
    g.by_inv = (bits & 0x7fffffu) != 0x7fffffu && s.du > 1e-30f && s.du < 1e30f;
    g.s_hi = s.s_hi;
    g.s_lo = s.s_lo;
    return g;
}

// exp(-(s_hi + s_lo) (d - f_hi - f_lo)^2) for the x and the y offset of a visibility at once, the
// argument in double-float (packed FP32x2).  nf = -f_hi, nfl = -f_lo.  The difference t = d - f_hi and
// its error e are exact: d is an integer and |f_hi| <= |d| unless d = 0 (Fast2Sum).
__device__ __forceinline__ float2 wexp2(float d, float2 nf, float2 nfl, float s_hi, float s_lo) {
    const float2 dd = make_float2(d, d), nd = make_float2(-d, -d), f = make_float2(-nf.x, -nf.y);
    const float2 ns = make_float2(-s_hi, -s_hi), sl = make_float2(s_lo, s_lo);
    const float2 t = __fadd2_rn(dd, nf), nt = __fadd2_rn(nd, f);   // +-(d - f_hi)
    const float2 a_lo = __fadd2_rn(__fadd2_rn(__fadd2_rn(dd, nt), nf), nfl);
    const float2 np = __fmul2_rn(t, nt);                           // -t^2
    const float2 pe = __ffma2_rn(t, t, np);                        // its error
    const float2 qq = __ffma2_rn(__fadd2_rn(t, t), a_lo, pe);
    const float2 narg = __fmul2_rn(ns, np);                        // s_hi t^2 = -arg_hi
    const float2 arg_e = __ffma2_rn(make_float2(s_hi, s_hi), np, narg);   // error of the product
    const float2 arg_lo = __ffma2_rn(sl, np, __ffma2_rn(ns, qq, arg_e));
    const float2 c = __fadd2_rn(make_float2(1.f, 1.f), arg_lo);
    return __fmul2_rn(make_float2(expf(-narg.x), expf(-narg.y)), c);
}

// ------------------------------------------------------------------ plan kernels
// The plan is a stable counting sort of the visibilities by (uv tile, cell in
// the tile): LSD radix with digits of up to DMAX bits (two passes up to about
// 500^2 cells, three beyond), so a tile's visibilities are grouped by cell
// whatever the input order (baseline-major tracks or time-major snapshots)
// and keep their input order inside a cell: the gridded sums are reproducible
// run to run.  The input of a pass is cut into two slices an SM; a pass counts
// the digits of every slice (k_plan_hist), turns the counts into the slices'
// places in every digit's run (k_plan_offsets) and then moves positions, indices
// and keys together (k_plan_scatter).
constexpr int ST_T = 512;              // threads per CTA
constexpr int ST_W = ST_T / 32;
constexpr int ST_R = 8;                // visibilities of a thread at a time
constexpr int RT = ST_T * ST_R;        // a chunk: what a CTA sorts in shared memory at a time
constexpr int DMAX = 9;                // widest digit: 512 bins
constexpr int CB = 8;                  // key bits of the cell inside its tile (TS x TS = 2^CB)
static_assert(TS * TS == 1 << CB, "tile cells must fill CB bits");
static_assert(1 << DMAX <= ST_T, "one digit a thread");

// u / dU rounded to nearest: q0 = u y with y = RN(1 / dU), its exact remainder and one correction,
// q = RN(q0 + RN(u - q0 dU) y), which Markstein's theorem (IBM J. Res. Dev. 34, 1990) makes the
// correctly rounded quotient unless dU's significand is all ones (by_inv is false then).  Three
// instructions; where q0 overflows the result is NaN, and no cell either way.
__device__ __forceinline__ float quotient(const GridGeom &G, float u) {
    if (!G.by_inv) return __fdiv_rn(u, G.du);
    const float q0 = __fmul_rn(u, G.inv_du);
    return __fmaf_rn(__fmaf_rn(-q0, G.du, u), G.inv_du, q0);
}

__device__ __forceinline__ float2 quotients(const GridGeom &G, float2 p) {
    return make_float2(quotient(G, p.x), quotient(G, p.y));
}

// Key of the position with quotients q = (u / dU, v / dU); key_none for non-finite and far ones.
__device__ __forceinline__ uint32_t key_from_q(const GridGeom &G, float2 q, uint32_t key_none) {
    if (!(fabsf(q.x) < 1.0e7f && fabsf(q.y) < 1.0e7f)) return key_none;
    const uint32_t kx = (uint32_t)((int)floorf(__fadd_rn(q.x, 0.5f)) + G.off);
    const uint32_t ky = (uint32_t)((int)floorf(__fadd_rn(q.y, 0.5f)) + G.off);
    if (kx >= (uint32_t)G.ks || ky >= (uint32_t)G.ks) return key_none;
    const uint32_t tile = (ky / TS) * (uint32_t)G.tt + kx / TS;
    return tile << CB | (ky % TS) * TS + kx % TS;
}

__device__ __forceinline__ uint32_t cell_key(const GridGeom &G, float2 p, uint32_t key_none) {
    return key_from_q(G, quotients(G, p), key_none);
}

// Block-wide exclusive scan of one value per thread (blockDim.x a multiple of 32, at most 1024).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *sh, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    const uint32_t warp_base = warp ? sh[warp - 1] : 0u;
    total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return warp_base + x - v;
}

// hist[digit][slice]: the digit counts of one slice (shared-memory counters, whose hardware adds
// merge equal digits of a warp), from the positions (first pass) or the keys.
template <bool FIRST>
__global__ void __launch_bounds__(ST_T) k_plan_hist(GridGeom G, int64_t n, int64_t per_slice,
                                                    const float2 *__restrict__ uv, const uint32_t *__restrict__ keys,
                                                    uint32_t key_none, int shift, int dw, uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[1 << DMAX];
    const int nb = 1 << dw;
    if ((int)threadIdx.x < nb) h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t b0 = blockIdx.x * per_slice;
    const int cnt = (int)(min(n, b0 + per_slice) - b0);   // a slice is far below 2^31
    constexpr int K = 4;                 // visibilities of a thread in flight
    for (int b = threadIdx.x; b < cnt; b += ST_T * K) {
        uint32_t key[K];
        if (FIRST) {
            float2 p[K];
#pragma unroll
            for (int k = 0; k < K; ++k) p[k] = b + k * ST_T < cnt ? uv[b0 + b + k * ST_T] : make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k) key[k] = cell_key(G, p[k], key_none);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) key[k] = b + k * ST_T < cnt ? keys[b0 + b + k * ST_T] : 0u;
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (b + k * ST_T < cnt) atomicAdd(&h[(key[k] >> shift) & (uint32_t)(nb - 1)], 1u);
    }
    __syncthreads();
    if ((int)threadIdx.x < nb) hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// One warp per digit: the counts of its slices become their exclusive sums, in place, and total[digit].
__global__ void __launch_bounds__(256) k_plan_offsets(int nb, int slices, uint32_t *__restrict__ hist,
                                                      uint32_t *__restrict__ total) {
    const int d = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (d >= nb) return;
    uint32_t *h = hist + (size_t)d * slices;
    uint32_t carry = 0;
    for (int c0 = 0; c0 < slices; c0 += 32 * 4) {
        uint32_t v[4], s = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + 4 * lane + k;
            v[k] = c < slices ? h[c] : 0u;
            s += v[k];
        }
        uint32_t x = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        uint32_t run = carry + x - s;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + 4 * lane + k;
            if (c < slices) h[c] = run;
            run += v[k];
        }
        carry += __shfl_sync(FULL, x, 31);
    }
    if (lane == 0) total[d] = carry;
}

// One slice of a pass, stably by its digit, a chunk of up to RT visibilities at a time (warp w
// owns a contiguous part of the chunk):
//  - every item's rank among its warp's earlier items of its digit, on top of the warp's running
//    count of the digit: the lanes of one digit by __match_any_sync for every other row and by a
//    ballot per digit bit for the rest, which spreads the work over the two units that do them (all
//    matches: 77 cycles a row and SM, all ballots: 1 % slower overall than half and half).  DW is a
//    template parameter: with a runtime width the tests between the ballots doubled the kernel's
//    instructions;
//  - the chunk staged in shared memory in digit order and written out in that order: consecutive
//    threads, consecutive addresses within a run.
// FIRST: keys are computed from the positions and the indices are the identity; LAST: no keys are
// written.  Positions travel with the indices, so no pass gathers, and no CTA waits for another (a
// single sweep with look-back spent 8 of 20 us a pass waiting at 1e6 visibilities).  Bound by
// instruction issue and the latency of a chunk's phases.
__host__ __device__ constexpr size_t sort_smem(int nb) {
    return (sizeof(float2) + 2 * sizeof(uint32_t)) * RT + 2 * sizeof(uint32_t) * nb + sizeof(uint16_t) * ST_W * nb;
}
template <int DW, bool FIRST, bool LAST>
__global__ void __launch_bounds__(ST_T, 2) k_plan_scatter(GridGeom G, int64_t n, int64_t per_slice,
                                                          const float2 *__restrict__ uv_in,
                                                          const uint32_t *__restrict__ idx_in,
                                                          const uint32_t *__restrict__ key_in, uint32_t key_none, int shift,
                                                          const uint32_t *__restrict__ offs,
                                                          const uint32_t *__restrict__ total, float2 *__restrict__ uv_out,
                                                          uint32_t *__restrict__ idx_out, uint32_t *__restrict__ key_out) {
    extern __shared__ __align__(16) uint8_t ssm[];
    constexpr int nb = 1 << DW;
    float2 *suv = (float2 *)ssm;                         // [RT] the chunk ordered by digit
    uint32_t *sidx = (uint32_t *)(suv + RT);             // [RT]
    uint32_t *skey = sidx + RT;                          // [RT]
    uint32_t *gbase = skey + RT;                         // [nb] global position of local 0 for the digit
    uint32_t *lstart = gbase + nb;                       // [nb] the digit's first local position
    uint16_t *wcnt = (uint16_t *)(lstart + nb);          // [ST_W][nb] per-warp counts, then offsets
    __shared__ uint32_t sh[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t b0 = blockIdx.x * per_slice;
    const int size = (int)(min(n, b0 + per_slice) - b0);
    uv_in += b0;
    if (!FIRST) {
        idx_in += b0;
        key_in += b0;
    }
    // thread d < nb: global position of the digit's next item
    uint32_t tot, next = block_exclusive_scan(tid < nb ? total[tid] : 0u, sh, tot);
    if (tid < nb) next += offs[(size_t)tid * gridDim.x + blockIdx.x];
    uint16_t *mycnt = wcnt + warp * nb;
    for (int c0 = 0; c0 < size; c0 += RT) {
        const int nloc = min(RT, size - c0);
        const int rows = (nloc + ST_T - 1) / ST_T;       // 32-item rows of a warp
        const int w0 = warp * rows * 32;
        float2 p[ST_R];
        uint32_t ix[ST_R], key[ST_R], rk[ST_R / 2];      // rk: two ranks
#pragma unroll
        for (int k = 0; k < ST_R; ++k) {
            const int e = w0 + k * 32 + lane;
            const bool on = k < rows && e < nloc;
            p[k] = on ? uv_in[c0 + e] : make_float2(0.f, 0.f);
            ix[k] = FIRST ? (uint32_t)b0 + (uint32_t)(c0 + e) : on ? idx_in[c0 + e] : 0u;
            if (!FIRST) key[k] = on ? key_in[c0 + e] : 0u;
        }
        __syncthreads();   // the chunk before has been written out
        for (int i = tid; i < ST_W * nb / 8; i += ST_T) ((uint4 *)wcnt)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ST_R; ++k)
            if (k < rows) {
                const bool on = w0 + k * 32 + lane < nloc;
                if (FIRST) key[k] = cell_key(G, p[k], key_none);
                const uint32_t d = (key[k] >> shift) & (uint32_t)(nb - 1);
                unsigned peers;
                if (k % 2) {
                    peers = __match_any_sync(FULL, on ? d : 1u << DW);
                } else {
                    peers = __ballot_sync(FULL, on);
#pragma unroll
                    for (int b = 0; b < DW; ++b) {
                        const bool bit = (d >> b) & 1u;
                        const unsigned v = __ballot_sync(FULL, bit);
                        peers &= bit ? v : ~v;
                    }
                }
                const uint32_t before = mycnt[d], rank = before + (uint32_t)__popc(peers & lt);
                if (k % 2 == 0) rk[k / 2] = rank;
                else rk[k / 2] |= rank << 16;
                __syncwarp();
                if (on && lane == __ffs(peers) - 1) mycnt[d] = (uint16_t)(before + __popc(peers));
                __syncwarp();
            }
        __syncthreads();
        // per digit: offsets of the warps inside its run; the run's local start and global place
        uint32_t cnt = 0;
        if (tid < nb) {
            uint32_t c[ST_W];
#pragma unroll
            for (int w = 0; w < ST_W; ++w) c[w] = wcnt[w * nb + tid];
#pragma unroll
            for (int w = 0; w < ST_W; ++w) {
                wcnt[w * nb + tid] = (uint16_t)cnt;
                cnt += c[w];
            }
        }
        const uint32_t ls = block_exclusive_scan(cnt, sh, tot);
        if (tid < nb) {
            lstart[tid] = ls;
            gbase[tid] = next - ls;
            next += cnt;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ST_R; ++k)
            if (k < rows && w0 + k * 32 + lane < nloc) {
                const uint32_t d = (key[k] >> shift) & (uint32_t)(nb - 1);
                const uint32_t L = lstart[d] + mycnt[d] + ((rk[k / 2] >> (16 * (k % 2))) & 0xffffu);
                suv[L] = p[k];
                sidx[L] = ix[k];
                skey[L] = key[k];
            }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ST_R; ++k) {
            const int L = k * ST_T + tid;
            if (L < nloc) {
                const uint32_t kk = skey[L], pos = gbase[(kk >> shift) & (uint32_t)(nb - 1)] + (uint32_t)L;
                uv_out[pos] = suv[L];
                idx_out[pos] = sidx[L];
                if (!LAST) key_out[pos] = kk;
            }
        }
    }
}

using ScatterFn = void (*)(GridGeom, int64_t, int64_t, const float2 *, const uint32_t *, const uint32_t *, uint32_t, int,
                           const uint32_t *, const uint32_t *, float2 *, uint32_t *, uint32_t *);
template <int DW>
ScatterFn scatter_of(bool first, bool last) {
    if constexpr (DW == DMAX) {   // a single pass: 9 key bits
        if (first && last) return k_plan_scatter<DW, true, true>;
    }
    return first ? k_plan_scatter<DW, true, false> : last ? k_plan_scatter<DW, false, true> : k_plan_scatter<DW, false, false>;
}
ScatterFn scatter_of(int dw, bool first, bool last) {
    switch (dw) {   // at least 9 key bits, so at least 5 of a digit
        case 5: return scatter_of<5>(first, last);
        case 6: return scatter_of<6>(first, last);
        case 7: return scatter_of<7>(first, last);
        case 8: return scatter_of<8>(first, last);
        default: return scatter_of<9>(first, last);
    }
}

// The whole plan of at most PS_MAX visibilities in one CTA: the passes above with the keys and indices in
// registers and shared memory, the positions gathered at the end.  Latency and launches are all of such a
// plan.  Gridding 1,000 / 5,000 visibilities on 64^2, a call: 53 / 47 us with six dependent kernels, 31 / 33
// with this one; an estimate of 8 rings 54 / 53.5 and 47.5 / 51.5.  At 8,192 on 128^2 the one CTA is the
// longer chain (estimate 63.7 and 67.2 us), so the line lies between.
constexpr int PS_T = 1024, PS_W = PS_T / 32, PS_R = 5, PS_MAX = PS_T * PS_R;
__host__ __device__ constexpr size_t small_smem(int nb) {
    return 2 * sizeof(uint32_t) * PS_MAX + sizeof(uint32_t) * nb + sizeof(uint16_t) * PS_W * nb;
}
__global__ void __launch_bounds__(PS_T) k_plan_small(GridGeom G, int n, const float2 *__restrict__ uv, uint32_t key_none,
                                                     int passes, int dw, float2 *__restrict__ s_uv,
                                                     uint32_t *__restrict__ s_idx) {
    extern __shared__ __align__(16) uint8_t ssm[];
    const int nb = 1 << dw;
    uint16_t *wcnt = (uint16_t *)ssm;                    // [PS_W][nb] per-warp counts, then offsets
    uint32_t *lstart = (uint32_t *)(wcnt + PS_W * nb);   // [nb] the digit's first position
    uint32_t *skey = lstart + nb, *sidx = skey + PS_MAX; // [n] the records ordered by digit
    __shared__ uint32_t sh[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    const int rows = (n + PS_T - 1) / PS_T;              // 32-item rows of a warp
    const int e0 = warp * rows * 32 + lane;
    uint32_t key[PS_R], ix[PS_R], rk[PS_R];
#pragma unroll
    for (int k = 0; k < PS_R; ++k) {
        const int e = e0 + k * 32;
        ix[k] = (uint32_t)e;
        key[k] = k < rows && e < n ? cell_key(G, uv[e], key_none) : 0u;
    }
    uint16_t *mycnt = wcnt + warp * nb;
    for (int ps = 0; ps < passes; ++ps) {
        const int shift = dw * ps;
        for (int i = tid; i < PS_W * nb / 8; i += PS_T) ((uint4 *)wcnt)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PS_R; ++k)
            if (k < rows) {
                const bool on = e0 + k * 32 < n;
                const uint32_t d = (key[k] >> shift) & (uint32_t)(nb - 1);
                unsigned peers = __ballot_sync(FULL, on);
                for (int b = 0; b < dw; ++b) {
                    const bool bit = (d >> b) & 1u;
                    const unsigned v = __ballot_sync(FULL, bit);
                    peers &= bit ? v : ~v;
                }
                const uint32_t before = mycnt[d];
                rk[k] = before + (uint32_t)__popc(peers & lt);
                __syncwarp();
                if (on && lane == __ffs(peers) - 1) mycnt[d] = (uint16_t)(before + __popc(peers));
                __syncwarp();
            }
        __syncthreads();
        uint32_t cnt = 0, tot;
        if (tid < nb)
            for (int w = 0; w < PS_W; ++w) {
                const uint32_t c = wcnt[w * nb + tid];
                wcnt[w * nb + tid] = (uint16_t)cnt;
                cnt += c;
            }
        const uint32_t ls = block_exclusive_scan(cnt, sh, tot);
        if (tid < nb) lstart[tid] = ls;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PS_R; ++k)
            if (k < rows && e0 + k * 32 < n) {
                const uint32_t d = (key[k] >> shift) & (uint32_t)(nb - 1), L = lstart[d] + mycnt[d] + rk[k];
                skey[L] = key[k];
                sidx[L] = ix[k];
            }
        __syncthreads();
        if (ps + 1 < passes)
#pragma unroll
            for (int k = 0; k < PS_R; ++k)
                if (k < rows && e0 + k * 32 < n) {
                    key[k] = skey[e0 + k * 32];
                    ix[k] = sidx[e0 + k * 32];
                }
    }
    for (int L = tid; L < n; L += PS_T) {
        const uint32_t i = sidx[L];
        s_idx[L] = i;
        s_uv[L] = uv[i];
    }
}

// ------------------------------------------------------------------ accumulation
// One CTA per work unit: um consecutive visibilities (at most UMAX) of the sorted order,
// so a unit's visibilities come grouped by cell (any number of cells and
// tiles).  Each visibility's 2 (2r+1) one-dimensional weights are formed
// once and staged in shared memory, and the unit is cut into tasks: runs of
// one cell, also cut at every CHUNK-th item of the unit, so a task holds at
// most CHUNK visibilities.  A warp takes a task; lane (dy, q) owns the
// footprint cells (q, dy) and (q + 4, dy) of the (2r+1)^2 around the run's
// cell (its lanes' FP64 adds cover whole sectors of a grid row) and sums w = wx wy, w Re V, w Im V over the run with packed FP32x2
// arithmetic (plain blocks of GFOLD, as two interleaved chains, folded into
// Kahan sums; a fixed order), then adds its cells to the FP64 grid.  No
// shared accumulators: runs never wait on one another, whether the cell is
// dense (long runs) or sparse.
//
// Staged record of a visibility (RS floats): wx of columns 0, 4, 1, 5, 2, 6, 3
// (a lane's two columns are adjacent; zero beyond 2r), a zero, (wy[d], wy[d])
// for d = 0..6, two pad floats, (Re V, Re V, Im V, Im V).
constexpr int GT = 256;          // threads per gridding CTA (8 warps x UMAX/8 items)
// What the third (and fourth) accumulator plane of a cell holds: the weight sum
// (GW_SUM), the number N_g of visibilities entered (GW_COUNT, Eq. vg), or the
// weight sum and the sum of squared weights (GW_SUM_SQ).
enum { GW_SUM = 0, GW_COUNT = 1, GW_SUM_SQ = 2 };
constexpr int RS = 28;           // floats per staged record
constexpr int R_WY = 8, R_V = 24;
constexpr int GFOLD = 16;
constexpr int CHUNK = 128;       // visibilities per task at most
static_assert(UMAX == 8 * 64, "each of 8 warps holds two rounds of 32 items of a unit");
static_assert(UMAX % CHUNK == 0 && UMAX <= 65535, "task starts are 16-bit unit offsets");
constexpr size_t GRID_SMEM = UMAX * sizeof(float) * RS + sizeof(uint32_t) * UMAX + sizeof(uint16_t) * (UMAX + 8);

// The double with the value of x, built with integer operations only (GB300's
// FP64 pipe is narrow: one hardware conversion per flushed value is what kept
// it busy).  widen: normal x.  is_special: x is zero, subnormal, infinite or NaN, which widen_any
// takes too (subnormal x, |x| < 2^-126, become a zero of the same sign).
__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x);
    return __hiloint2double((int)((((int)b >> 3) & 0x8fffffff) + 0x38000000), (int)(b << 29));
}
__device__ __forceinline__ bool is_special(float x) { return ((__float_as_uint(x) + 0x00800000u) & 0x7f000000u) == 0u; }
__device__ __noinline__ double widen_any(float x) {
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 255u, sign = b & 0x80000000u;
    const uint32_t eh = e == 255u ? 2047u : e + (1023u - 127u);
    const uint32_t hi = e == 0u ? sign : sign | (eh << 20) | ((b >> 3) & 0xFFFFFu);
    return __hiloint2double((int)hi, (int)(e == 0u ? 0u : b << 29));
}

__device__ __forceinline__ void kahan_add2(float2 &s, float2 &c, float2 x) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 y = __ffma2_rn(c, m1, x);                   // x - c
    const float2 t = __fadd2_rn(s, y);
    c = __ffma2_rn(y, m1, __ffma2_rn(s, m1, t));             // (t - s) - y
    s = t;
}

// One staged visibility (record at offset o) into this lane's two footprint
// cells: w = (wx[2q], wx[2q+1]) * wy[dy], re += w Re V, im += w Im V, sum w.
template <int WM>
__device__ __forceinline__ void grid_acc(const float *lw, const float *lwy, const float *lv, int o, float2 &re,
                                         float2 &im, float2 &ws, float2 &ws2) {
    const float2 wxp = *(const float2 *)(lw + o);
    const float2 wyy = *(const float2 *)(lwy + o);
    const float4 vv = *(const float4 *)(lv + o);
    const float2 w = __fmul2_rn(wxp, wyy);
    re = __ffma2_rn(w, make_float2(vv.x, vv.y), re);
    im = __ffma2_rn(w, make_float2(vv.z, vv.w), im);
    if (WM != GW_COUNT) ws = __fadd2_rn(w, ws);
    if (WM == GW_SUM_SQ) ws2 = __ffma2_rn(w, w, ws2);
}

// Inputs of one unit as thread (warp, lane) sees them: items t = ipw warp +
// 32 h + lane, h = 0, 1 (h = 0 only when ipw is 32), in sorted order.
struct UnitIn {
    int cnt;
    float2 p[2];
    uint32_t idx[2];
};

__device__ __forceinline__ void load_unit(UnitIn &in, int64_t u, int64_t nu, int64_t n_vis, int um, int ipw,
                                          const float2 *__restrict__ s_uv, const uint32_t *__restrict__ s_idx,
                                          int warp, int lane) {
    if (u >= nu) return;
    const int64_t b = u * um;
    in.cnt = n_vis - b < um ? (int)(n_vis - b) : um;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int t = warp * ipw + h * 32 + lane;
        if (h * 32 < ipw && t < in.cnt) {
            in.p[h] = s_uv[b + t];
            in.idx[h] = s_idx[b + t];
        }
    }
}

// A run's sums of one footprint cell into the FP64 grid.
template <int WM>
__device__ __forceinline__ void grid_add(double *__restrict__ re, double *__restrict__ im, double *__restrict__ w,
                                         double *__restrict__ w2, float vre, float vim, float vw, float vw2, double run) {
    const bool odd = is_special(vre) || is_special(vim) || (WM != GW_COUNT && is_special(vw)) ||
                     (WM == GW_SUM_SQ && is_special(vw2));
    if (!odd) {
        atomicAdd(re, widen(vre));
        atomicAdd(im, widen(vim));
        atomicAdd(w, WM == GW_COUNT ? run : widen(vw));
        if (WM == GW_SUM_SQ) atomicAdd(w2, widen(vw2));
    } else {
        atomicAdd(re, widen_any(vre));
        atomicAdd(im, widen_any(vim));
        atomicAdd(w, WM == GW_COUNT ? run : widen_any(vw));
        if (WM == GW_SUM_SQ) atomicAdd(w2, widen_any(vw2));
    }
}

template <int WM>
__global__ void __launch_bounds__(GT, 3) k_grid(GridGeom G, int64_t n_vis, int um, uint32_t key_none,
                                             const float2 *__restrict__ s_uv,
                                             const uint32_t *__restrict__ s_idx,
                                             const float2 *__restrict__ vis,
                                             double *__restrict__ acc_re,
                                             double *__restrict__ acc_im,
                                             double *__restrict__ acc_w,
                                             double *__restrict__ acc_w2) {
    extern __shared__ __align__(16) uint8_t dsm[];
    float *st = (float *)dsm;                                          // [UMAX][RS] staged records
    uint32_t *skey = (uint32_t *)(st + UMAX * RS);                     // [UMAX] key of every item
    uint16_t *tstart = (uint16_t *)(skey + UMAX);                      // [UMAX + 1] first item of each task
    __shared__ uint32_t wsum_s[8], wvalid_s[8];
    __shared__ int next_s;   // next task of the unit
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = G.r, fw = 2 * r + 1;
    const bool gauss = G.kernel == ABS_KERNEL_GAUSS;
    // this lane's footprint cells: (qx, dy) and (qx + 4, dy)
    const int dy = lane >> 2, qx = lane & 3;
    const bool on_a = dy < fw && qx < fw, on_b = on_a && qx + 4 < fw;
    const int ipw = um > GT ? 64 : 32;   // items a warp
    const int64_t nu = cdiv(n_vis, um);
    UnitIn nxt;
    load_unit(nxt, blockIdx.x, nu, n_vis, um, ipw, s_uv, s_idx, warp, lane);
    float2 vn[2];   // the next unit's visibilities, gathered one unit ahead
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (blockIdx.x < nu && h * 32 < ipw && warp * ipw + h * 32 + lane < nxt.cnt) vn[h] = vis[nxt.idx[h]];
    for (int64_t u = blockIdx.x; u < nu; u += gridDim.x) {
        const UnitIn cur = nxt;
        const int total = cur.cnt;
        const float2 v[2] = {vn[0], vn[1]};   // this unit's visibilities
        load_unit(nxt, u + gridDim.x, nu, n_vis, um, ipw, s_uv, s_idx, warp, lane);   // in flight during this unit
        __syncthreads();   // previous unit done with the staging buffers
        // keys (the plan's, recomputed from the same positions); invalid items sort last
        float2 q[2];   // u/dU, v/dU of this thread's items
        bool valid[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = warp * ipw + h * 32 + lane;
            valid[h] = false;
            if (h * 32 < ipw && t < total) {
                q[h] = quotients(G, cur.p[h]);
                const uint32_t key = key_from_q(G, q[h], key_none);
                skey[t] = key;
                valid[h] = key != key_none;
            }
        }
        __syncthreads();
        // task starts: a valid item that begins a cell run or sits at a multiple of CHUNK
        bool ts[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = warp * ipw + h * 32 + lane;
            ts[h] = valid[h] && (t % CHUNK == 0 || skey[t] != skey[t - 1]);
        }
        const unsigned b0 = __ballot_sync(FULL, ts[0]), b1 = __ballot_sync(FULL, ts[1]);
        const unsigned nv0 = __ballot_sync(FULL, valid[0]), nv1 = __ballot_sync(FULL, valid[1]);
        if (lane == 0) {
            wsum_s[warp] = (uint32_t)(__popc(b0) + __popc(b1));
            wvalid_s[warp] = (uint32_t)(__popc(nv0) + __popc(nv1));
        }
        __syncthreads();
        uint32_t wbase = 0, ntask = 0, nvalid = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            wbase += w < warp ? wsum_s[w] : 0u;
            ntask += wsum_s[w];
            nvalid += wvalid_s[w];
        }
        const unsigned lt = (1u << lane) - 1u;
        if (ts[0]) tstart[wbase + __popc(b0 & lt)] = (uint16_t)(warp * ipw + lane);
        if (ts[1]) tstart[wbase + __popc(b0) + __popc(b1 & lt)] = (uint16_t)(warp * ipw + 32 + lane);
        if (threadIdx.x == 0) {
            tstart[ntask] = (uint16_t)nvalid;
            next_s = GT / 32;   // the warps' first tasks are their own numbers
        }
        // staging: weights and visibility of every valid item, in place
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = warp * ipw + h * 32 + lane;
            if (valid[h]) {
                const float2 p = cur.p[h], qq = q[h];
                const float cxf = floorf(__fadd_rn(qq.x, 0.5f)), cyf = floorf(__fadd_rn(qq.y, 0.5f));
                const float fxh = __fsub_rn(qq.x, cxf), fyh = __fsub_rn(qq.y, cyf);
                // the division residual (exact by FMA) over dU: a correction of
                // relative size 2^-24, so one rounding of its own does not matter
                const float fxl = __fmul_rn(fmaf(-qq.x, G.du, p.x), G.inv_du);
                const float fyl = __fmul_rn(fmaf(-qq.y, G.du, p.y), G.inv_du);
                const float2 nf = make_float2(-fxh, -fyh), nfl = make_float2(-fxl, -fyl);
                float2 w[7];
#pragma unroll
                for (int k = 0; k < 7; ++k) {
                    w[k] = make_float2(0.f, 0.f);
                    if (k < fw) w[k] = gauss ? wexp2((float)(k - r), nf, nfl, G.s_hi, G.s_lo) : make_float2(1.f, 1.f);
                }
                float4 *rec = (float4 *)(st + t * RS);
                rec[0] = make_float4(w[0].x, w[4].x, w[1].x, w[5].x);
                rec[1] = make_float4(w[2].x, w[6].x, w[3].x, 0.f);
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    rec[R_WY / 4 + k] = make_float4(w[2 * k].y, w[2 * k].y, w[2 * k + 1].y, w[2 * k + 1].y);
                ((float2 *)(rec + R_WY / 4 + 3))[0] = make_float2(w[6].y, w[6].y);
                rec[R_V / 4] = make_float4(v[h].x, v[h].x, v[h].y, v[h].y);
            }
        }
        // the next unit's visibilities: its indices have arrived by now
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (u + gridDim.x < nu && h * 32 < ipw && warp * ipw + h * 32 + lane < nxt.cnt) vn[h] = vis[nxt.idx[h]];
        __syncthreads();
        for (int tk = warp, nx = 0; tk < (int)ntask; tk = nx) {
            if (lane == 0) nx = atomicAdd(&next_s, 1);   // tasks differ in length: the next free one
            nx = __shfl_sync(FULL, nx, 0);
            if (on_a) {   // lanes without a footprint cell take no part in the sums
                const int j_begin = tstart[tk], j_end = tstart[tk + 1];
                const float2 z = make_float2(0.f, 0.f);
                float2 sre = z, cre = z, sim = z, cim = z, sw = z, cw = z, sw2 = z, cw2 = z;
                const float *lw = st + 2 * qx, *lwy = st + R_WY + 2 * dy, *lv = st + R_V;
                for (int j0 = j_begin; j0 < j_end; j0 += GFOLD) {   // plain blocks of GFOLD, folded into Kahan sums
                    float2 bre = z, bim = z, bw = z, bw2 = z;
                    if (j0 + GFOLD <= j_end) {
                        // a full block: unrolled, two independent chains (even, odd visibilities)
                        float2 bre1 = z, bim1 = z, bw1 = z, bw21 = z;
#pragma unroll
                        for (int k = 0; k < GFOLD; k += 2) {
                            grid_acc<WM>(lw, lwy, lv, (j0 + k) * RS, bre, bim, bw, bw2);
                            grid_acc<WM>(lw, lwy, lv, (j0 + k + 1) * RS, bre1, bim1, bw1, bw21);
                        }
                        bre = __fadd2_rn(bre, bre1);
                        bim = __fadd2_rn(bim, bim1);
                        if (WM != GW_COUNT) bw = __fadd2_rn(bw, bw1);
                        if (WM == GW_SUM_SQ) bw2 = __fadd2_rn(bw2, bw21);
                    } else {
                        for (int j = j0; j < j_end; ++j) grid_acc<WM>(lw, lwy, lv, j * RS, bre, bim, bw, bw2);
                    }
                    kahan_add2(sre, cre, bre);
                    kahan_add2(sim, cim, bim);
                    if (WM != GW_COUNT) kahan_add2(sw, cw, bw);
                    if (WM == GW_SUM_SQ) kahan_add2(sw2, cw2, bw2);
                }
                // the run's cell from its key: tile (kx / TS, ky / TS), cell in the tile
                const uint32_t key = skey[j_begin];
                const int tile = (int)(key >> CB), loc = (int)(key & (uint32_t)(TS * TS - 1));
                const int kx = (tile % G.tt) * TS + (loc & (TS - 1)), ky = (tile / G.tt) * TS + (loc >> 4);
                const int gy = ky - G.off + dy - r, gx = kx - G.off + qx - r;
                if (abs(gy) > G.half) continue;
                // the run's sums s - c, rounded once to FP32 (relative 2^-24 of the run)
                const float2 m1 = make_float2(-1.f, -1.f);
                const float2 vre = __ffma2_rn(cre, m1, sre), vim = __ffma2_rn(cim, m1, sim);
                const float2 vw = __ffma2_rn(cw, m1, sw), vw2 = __ffma2_rn(cw2, m1, sw2);
                const double run = WM == GW_COUNT ? (double)(j_end - j_begin) : 0.0;   // visibilities entered at the cell
                const int row = (gy < 0 ? gy + G.n : gy) * G.n;   // n <= 8192: cells fit 32 bits
                if (abs(gx) <= G.half) {
                    const int o = row + (gx < 0 ? gx + G.n : gx);
                    grid_add<WM>(acc_re + o, acc_im + o, acc_w + o, acc_w2 + o, vre.x, vim.x, vw.x, vw2.x, run);
                }
                if (on_b && abs(gx + 4) <= G.half) {
                    const int o = row + (gx + 4 < 0 ? gx + 4 + G.n : gx + 4);
                    grid_add<WM>(acc_re + o, acc_im + o, acc_w + o, acc_w2 + o, vre.y, vim.y, vw.y, vw2.y, run);
                }
            }
        }
    }
}

// Hermitian mirror and FP32 outputs: G(g) + conj G(-g), W(g) + W(-g).  One thread per cell of the
// rows 0 .. n/2 (blockIdx.y), which also writes the mirrored cell, so the accumulators are read once.
// Bound by memory: 24 bytes read and 13 written a cell.
__global__ void __launch_bounds__(256) k_grid_finalize(int n, const double *__restrict__ acc_re,
                                                       const double *__restrict__ acc_im,
                                                       const double *__restrict__ acc_w, float2 *__restrict__ grid,
                                                       float *__restrict__ wsum, uint8_t *__restrict__ mask) {
    const int ix = blockIdx.x * 256 + threadIdx.x, iy = blockIdx.y;
    if (ix >= n) return;
    const int mx = ix == 0 ? 0 : n - ix, my = iy == 0 ? 0 : n - iy;
    const int64_t p = (int64_t)iy * n + ix, pm = (int64_t)my * n + mx;
    float2 g = make_float2(0.f, 0.f);
    float w = 0.f;
    uint8_t on = 0;
    if (ix != n / 2 && iy != n / 2) {
        const double wa = acc_w[p], wb = acc_w[pm];
        g = make_float2((float)(acc_re[p] + acc_re[pm]), (float)(acc_im[p] - acc_im[pm]));
        w = (float)(wa + wb);
        on = wa > 0.0 || wb > 0.0;   // a filled cell has weight > 0
    }
    grid[p] = g;
    wsum[p] = w;
    mask[p] = on;
    if (iy != 0 && iy != n / 2) {
        grid[pm] = make_float2(g.x, -g.y);
        wsum[pm] = w;
        mask[pm] = on;
    }
}

struct PlanBufs {
    uint32_t *s_idx;      // sorted original indices
    float2 *s_uv;         // sorted positions
    int ntiles;
};

bool plan_bufs(abs_ctx *ctx, const GridGeom &G, int64_t n_vis, PlanBufs &b) {
    b.ntiles = G.tt * G.tt;
    const int64_t nv = n_vis > 0 ? n_vis : 1;
    b.s_idx = (uint32_t *)workspace(ctx, "plan.s_idx", sizeof(uint32_t) * nv);
    b.s_uv = (float2 *)workspace(ctx, "plan.s_uv", sizeof(float2) * nv);
    return b.s_idx && b.s_uv;
}

}  // namespace

// The key of an invalid visibility: above every (tile, cell) key.
static uint32_t plan_key_none(const PlanBufs &b) { return (uint32_t)b.ntiles << CB; }

abs_status launch_grid_plan(abs_ctx *ctx, const Setup &s, int64_t n_vis, const float *d_uv, bool rings_only) {
    const GridGeom G = geom(s, rings_only);
    PlanBufs b;
    if (!plan_bufs(ctx, G, n_vis, b)) return fail(ctx, ABS_ERR_OOM, "grid plan workspace");
    if ((uint64_t)b.ntiles << CB >= 0x7fffffffull) return fail(ctx, ABS_ERR_UNSUPPORTED, "uv grid too large");
    if (n_vis == 0) return ABS_OK;   // no visibilities: no units
    const uint32_t key_none = plan_key_none(b);     // invalid visibilities sort last
    int bits = 1;
    while (((uint64_t)1 << bits) <= (uint64_t)key_none) ++bits;
    const int passes = (bits + DMAX - 1) / DMAX;
    const int dw = (bits + passes - 1) / passes, nb = 1 << dw;
    if (n_vis <= PS_MAX) {
        StageTimer timer(ctx, "grid_plan");
        allow_smem(k_plan_small, small_smem(nb));
        k_plan_small<<<1, PS_T, small_smem(nb), ctx->stream>>>(G, (int)n_vis, (const float2 *)d_uv, key_none, passes, dw,
                                                               b.s_uv, b.s_idx);
        return check_launch(ctx, "grid plan");
    }
    // two slices an SM, of whole rows of a CTA
    const int64_t per_slice = cdiv(cdiv(n_vis, 2 * ctx->sm_count), ST_T) * ST_T;
    const int slices = (int)cdiv(n_vis, per_slice);
    uint32_t *hist = (uint32_t *)workspace(ctx, "plan.hist", sizeof(uint32_t) * ((size_t)slices * nb + nb));
    // the passes alternate between the scratch and the sorted arrays, ending in the latter; the keys
    // between two arrays of their own
    const bool two = passes > 1, three = passes > 2;
    float2 *t_uv = two ? (float2 *)workspace(ctx, "plan.t_uv", sizeof(float2) * n_vis) : nullptr;
    uint32_t *t_idx = two ? (uint32_t *)workspace(ctx, "plan.t_idx", sizeof(uint32_t) * n_vis) : nullptr;
    uint32_t *k1 = two ? (uint32_t *)workspace(ctx, "plan.k1", sizeof(uint32_t) * n_vis) : nullptr;
    uint32_t *k2 = three ? (uint32_t *)workspace(ctx, "plan.k2", sizeof(uint32_t) * n_vis) : nullptr;
    if (!hist || (two && (!t_uv || !t_idx || !k1)) || (three && !k2)) return fail(ctx, ABS_ERR_OOM, "grid plan workspace");
    uint32_t *total = hist + (size_t)slices * nb;
    cudaStream_t st = ctx->stream;
    StageTimer timer(ctx, "grid_plan");
    const size_t smem = sort_smem(nb);
    const float2 *uin = (const float2 *)d_uv;
    const uint32_t *iin = nullptr, *kin = nullptr;
    for (int ps = 0; ps < passes; ++ps) {
        const bool first = ps == 0, last = ps == passes - 1, to_out = (passes - 1 - ps) % 2 == 0;
        float2 *uo = to_out ? b.s_uv : t_uv;
        uint32_t *io = to_out ? b.s_idx : t_idx, *ko = last ? nullptr : first ? k1 : k2;
        if (first) k_plan_hist<true><<<slices, ST_T, 0, st>>>(G, n_vis, per_slice, uin, nullptr, key_none, dw * ps, dw, hist);
        else k_plan_hist<false><<<slices, ST_T, 0, st>>>(G, n_vis, per_slice, nullptr, kin, key_none, dw * ps, dw, hist);
        k_plan_offsets<<<(int)cdiv(nb, 8), 256, 0, st>>>(nb, slices, hist, total);
        const ScatterFn scatter = scatter_of(dw, first, last);
        allow_smem(scatter, smem);
        scatter<<<slices, ST_T, smem, st>>>(G, n_vis, per_slice, uin, iin, kin, key_none, dw * ps, hist, total, uo, io, ko);
        uin = uo;
        iin = io;
        kin = ko;
    }
    return check_launch(ctx, "grid plan");
}

int grid_acc_planes(const Setup &s) { return s.weight_mode == ABS_W_NOISE ? 4 : 3; }

void grid_acc_buffers(abs_ctx *ctx, const Setup &s, double **acc) {
    const int64_t cells = (int64_t)s.n * s.n;
    *acc = (double *)workspace(ctx, "grid.acc", sizeof(double) * grid_acc_planes(s) * cells);
}

// Visibilities of a gridding unit: UMAX where that gives every resident CTA a unit, else half or a quarter
// of it (a unit is a chain of staging and sums, and on a small set the longest one is the kernel).  All are
// multiples of CHUNK, so the runs, and with them the results, are the same.
// 5,000 visibilities on 64^2: 27 us with 512 a unit, 12 with 128; 50,000 on 256^2: 35 / 20; 80,000 on 512^2:
// 55 / 36; 160,000 (256 a unit): 59 / 52; equal from 230,000 on.
static int grid_unit(int64_t n_vis, int ctas) {
    int um = UMAX;
    while (um > CHUNK && cdiv(n_vis, um) < ctas) um /= 2;
    return um;
}

abs_status launch_grid_accumulate(abs_ctx *ctx, const Setup &s, int64_t n_vis, const float *d_vis,
                                  float *d_grid, float *d_wsum, uint8_t *d_mask, bool acc_zeroed, abs_ctx *plan) {
    // the estimate path (no FP32 outputs; its plan was made with rings_only) accumulates what
    // its weighting needs
    const bool estimate = !d_grid && !d_wsum;
    const GridGeom G = geom(s, estimate);
    PlanBufs b;
    if (!plan_bufs(plan ? plan : ctx, G, n_vis, b)) return fail(ctx, ABS_ERR_OOM, "grid plan workspace");
    const int64_t cells = (int64_t)s.n * s.n;
    const int wm = !estimate ? GW_SUM
                   : s.weight_mode == ABS_W_PAPER_LITERAL ? GW_COUNT
                   : s.weight_mode == ABS_W_NOISE ? GW_SUM_SQ : GW_SUM;
    const int planes = wm == GW_SUM_SQ ? 4 : 3;
    double *acc = (double *)workspace(ctx, "grid.acc", sizeof(double) * planes * cells);
    if (!acc) return fail(ctx, ABS_ERR_OOM, "grid accumulation workspace");
    cudaStream_t st = ctx->stream;
    if (!acc_zeroed) {
        StageTimer timer(ctx, "grid_zero");
        cudaMemsetAsync(acc, 0, sizeof(double) * planes * cells, st);
    }
    if (n_vis > 0) {
        StageTimer timer(ctx, "grid");
        const int um = grid_unit(n_vis, ctx->sm_count * 3);
        const int blocks = (int)std::min<int64_t>(cdiv(n_vis, um), ctx->sm_count * 3);
        auto run = [&](auto kern) {
            allow_smem(kern, GRID_SMEM);
            kern<<<blocks, GT, GRID_SMEM, st>>>(G, n_vis, um, plan_key_none(b), b.s_uv, b.s_idx, (const float2 *)d_vis,
                                                acc, acc + cells, acc + 2 * cells, acc + 3 * cells);
        };
        if (wm == GW_COUNT)
            run(k_grid<GW_COUNT>);
        else if (wm == GW_SUM_SQ)
            run(k_grid<GW_SUM_SQ>);
        else
            run(k_grid<GW_SUM>);
    }
    if (estimate) return check_launch(ctx, "grid accumulate");   // read from the accumulators
    {
        StageTimer timer(ctx, "grid_finalize");
        k_grid_finalize<<<dim3((unsigned)cdiv(s.n, 256), s.n / 2 + 1), 256, 0, st>>>(s.n, acc, acc + cells, acc + 2 * cells,
                                                                                     (float2 *)d_grid, d_wsum, d_mask);
    }
    return check_launch(ctx, "grid accumulate");
}

}  // namespace absk
