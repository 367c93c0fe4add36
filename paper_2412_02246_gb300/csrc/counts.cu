// Stage 4: exact triangle counts, the denominator of Eq. estimator_t.
//
// With unit-mask fields I_m (X = 1 on the filled cells of a_m) the sum
// N^-2 sum_p I_i I_j I_k is the number T_ijk of ordered closed triangles
// (g1 in a_i, g2 in a_j, g3 in a_k, all filled, g1 + g2 + g3 = 0).  FP32 or
// even FP64 pixel sums cannot return that integer exactly at these sizes, so
// it is counted in integers.  For symmetric cell sets X, Y, Z (closed under
// g -> -g; the origin is in no ring)
//
//   T(X_i, Y_j, Z_k) = 2 #{ (g1, g2) : g1 in X_i upper half plane, g2 in Y_j, g1 + g2 in Z_k }
//
// (the third vertex -(g1+g2) is in Z_k iff g1 + g2 is; negating a triangle
// moves g1 to the other half plane, hence the factor 2).
//
// With A = every cell of the annuli on the grid, F = the filled ones and
// H = A \ F the holes, expanding every F as A - H gives
//
//   T(F,F,F) = T(A,A,A) - [T(H,A,A) + T(A,H,A) + T(A,A,H)]
//              + T(H,A,H) + T(A,H,H) + T(H,H,F),
//
// where T(A,A,A) depends only on the ring geometry (computed once per
// configuration and kept by the context).  The one-hole terms are sums over the
// holes h of n_bc(h), the number of pairs g2 in A_b, -(h + g2) in A_c, which is
// geometry too: it is the same for the (up to eight) images of h under the
// reflections of the square, so it is enumerated once per image class
// ("orbit", represented by 0 <= x <= y) that holds any hole, with the number of
// its holes as weight.  And g2 -> -h - g2 exchanges b and c, so only one of the
// two halves it maps on one another is enumerated: g2 = -u with u in the upper
// half plane and u above h/2 (row-major), the self-mapped g2 = -h/2 apart; above
// h/2, because h + g2 = h - u is then the shorter of the two third vertices'
// candidates and mostly inside the annuli.  T(A,A,A) is enumerated per orbit as well (every orbit,
// weighted by its size).  The two-hole terms are enumerated directly, sum over
// a <= b of |H_a| |H_b| / 2 pairs each.  A channel of the wide-band workload
// (R = 350, 385,000 cells, 33,000 holes in the two outer rings) has 4.6e8 visits
// of the one-hole terms this way and 8.4e8 of the others, against 1.2e10 for the
// form T(A,A,A) - T(H,A,A) - T(F,H,A) - T(F,F,H) without the symmetries.  A
// device-side estimate picks this route or the direct enumeration of T(F,F,F),
// whichever visits fewer pairs; both are exact.
//
// Cell lists are row-major per ring and hold the upper half plane only (the
// lower half is the negation).  The lists of A and of the orbits and the byte
// map of A are geometry, made once per configuration at its first count.  A byte map holds 1 + ring id of
// every cell of a family (0 elsewhere), indexed by |lin(h)| with lin(g) = g_y W +
// g_x, W = 2R + 1: lin is linear and odd, so lin(g1 + g2) = lin(g1) + lin(g2) and
// |lin(h)| = lin(+-h) picks the upper-half-plane representative of h, whose
// ring and membership are those of h.  A pair sum with |h_x| > R is in no ring;
// for |h_x| <= R and |h_y| <= 2R, lin is one-to-one, so a pair is classified
// by one add and compare on x, one add, one abs and one byte load (a map of
// about 4R^2 bytes, in shared memory up to R of about 230).  One CTA per work item
// (pair of rings, chunk of the larger set spread over the threads, chunk of
// the smaller set streamed through shared memory); each thread keeps
// run-length state (consecutive cells in row order usually land in the same
// ring) and adds finished runs into a lane-private shared-memory histogram
// of 16-bit counters (an item adds at most INNER x G1 x 4 to one counter)
// over the third ring, reduced into an int64 table at the end.
#include <algorithm>
#include <cstring>
#include <vector>

#include "abs_internal.cuh"

namespace absk {
namespace {

#ifndef ABS_COUNT_G1
#define ABS_COUNT_G1 4
#endif
#ifndef ABS_COUNT_KU
#define ABS_COUNT_KU 4
#endif
constexpr int G1 = ABS_COUNT_G1;   // g1 cells per thread
constexpr int KU = ABS_COUNT_KU;   // inner cells whose map loads are issued together
constexpr int CT = 256;          // threads per counting CTA (max)
// inner cells per work item: INNER where that gives every CTA a few items, INNER_S where it would not
// (an item of 1,024 x 512 visits takes 25 us, as long as a whole small grid should)
constexpr int INNER = 512, INNER_S = 128;
constexpr int GATHER_FUSED = CT;     // longest triplet list gathered by the pair kernel's last CTA
constexpr unsigned FULL = 0xffffffffu;

struct CountGeom {
    int n, nb, R, W;             // W = 2R + 1
    int K;                       // row pitch of the half-plane key g_y K + g_x (above 3R, so that
                                 // 2 key(u) - key(h) has the sign of (2u - h)_y, then (2u - h)_x)
    int nU, nO;                  // upper-half cells, orbits
    int64_t base;                // 2R W + R: the largest |lin| of a pair sum with |h_x| <= R
    // ring geometry (owned by the setup)
    const short2 *up;            // [nU] cells of A, upper half plane, by ring, then row-major
    const uint8_t *up_ring;      // [nU]
    const int32_t *up_off;       // [nb + 1]
    const uint32_t *orb;         // [nO] orbits by ring, then row-major: x | y << 12 | size / 2 << 24
    const uint8_t *orb_ring;     // [nO]
    const int32_t *orb_off;      // [nb + 1]
    const uint8_t *mapA;
};

// Cells and counters of the filled set, per call.
struct RingTables {
    short2 *F, *H;               // upper-half lists at up_off
    uint32_t *HO;                // orbits with holes at orb_off, packed as orb with the holes' number / 2
    uint8_t *mapF;
    uint8_t *nf;                 // [nO] filled upper-half cells of every orbit
    int32_t *cnt;                // [3][nb]: F, H (upper half), HO
    unsigned long long *fix;     // [nb][nb]: holes (upper half) of ring a with h / 2 in ring b
    int *ctl;                    // [0], [1] items of list 0, 1; [2], [3] next item; [4] the route;
                                 // [5] inner cells of an item
};

__device__ __forceinline__ int64_t cell_index(int n, int gx, int gy) {
    return (int64_t)(gy < 0 ? gy + n : gy) * n + (gx < 0 ? gx + n : gx);
}

// sqrt(v) of a non-negative integer v < 2^31 as a double-float pair h + l
// (relative error about 2^-46), with 32-bit arithmetic only: GB300's FP64 pipe
// (which also converts 64-bit integers) is too narrow for a square root per
// cell.  v = vf + vr exactly; h is the correctly rounded sqrtf(vf), whose
// residual vf - h^2 one FMA gives exactly; l = (v - h^2) / (2h) is the
// first-order (Newton) correction.
__device__ __forceinline__ void df_sqrt_int(int32_t v, float &h, float &l) {
    const float vf = (float)v;
    const float vr = (float)(v - (int32_t)vf);     // exact: |v - vf| <= ulp(vf) / 2 <= 64
    h = sqrtf(vf);
    if (h == 0.f) {
        l = 0.f;
        return;
    }
    const float r = __fadd_rn(fmaf(-h, h, vf), vr);
    l = __fdiv_rn(r, __fmul_rn(2.f, h));
}

// (sh, sl) += (h, l) in double-float (TwoSum of the high parts, then the low parts).
__device__ __forceinline__ void df_add(float &sh, float &sl, float h, float l) {
    const float t = __fadd_rn(sh, h);
    const float bp = __fsub_rn(t, sh);
    const float e = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(h, bp));
    const float lo = __fadd_rn(e, __fadd_rn(sl, l));
    sh = __fadd_rn(t, lo);                          // Fast2Sum renormalisation (|t| >= |lo|)
    sl = __fsub_rn(lo, __fsub_rn(sh, t));
}

// Packed orbit: representative (x, y), 0 <= x <= y, and a weight of at most 4.
__host__ __device__ __forceinline__ uint32_t orb_pack(int x, int y, int w) {
    return (uint32_t)x | (uint32_t)y << 12 | (uint32_t)w << 24;
}
__device__ __forceinline__ int orb_x(uint32_t o) { return (int)(o & 4095u); }
__device__ __forceinline__ int orb_y(uint32_t o) { return (int)((o >> 12) & 4095u); }
__device__ __forceinline__ int orb_w(uint32_t o) { return (int)(o >> 24); }

// Place of this lane's entry (on) in its ring's list: the warp's lanes of one ring are adjacent (the
// cells come by ring), one counter atomic per ring and warp.
__device__ __forceinline__ int ring_slot(bool on, unsigned peers, int lane, int32_t *counter) {
    const unsigned b = __ballot_sync(FULL, on) & peers;
    const int lead = __ffs(peers) - 1;
    int base = 0;
    if (lane == lead && b) base = atomicAdd(counter, __popc(b));
    base = __shfl_sync(FULL, base, lead);
    return base + __popc(b & ((1u << lane) - 1u));
}

// A cell is filled when the mask says so or (accw given) when it or its mirror has a nonzero weight sum.
__device__ __forceinline__ bool cell_filled(int n, const uint8_t *__restrict__ mask,
                                            const unsigned long long *__restrict__ accw, int x, int y) {
    if (accw) return accw[cell_index(n, x, y)] != 0ull || accw[cell_index(n, -x, -y)] != 0ull;
    return mask[cell_index(n, x, y)] != 0;
}

// The first ub blocks: one thread per upper-half cell, which goes to the list of filled cells or of
// holes and into the filled byte map.  The others: one thread per orbit, its filled cells counted
// (for the mean l) and, if it holds a hole, listed with their number.  Bound by latency (two
// dependent loads and an atomic a warp); the transposed images are single sectors each.
__global__ void __launch_bounds__(256) k_ring_cells(CountGeom G, int ub, const uint8_t *__restrict__ mask,
                                                    const unsigned long long *__restrict__ accw, RingTables T) {
    const int lane = threadIdx.x & 31;
    if ((int)blockIdx.x < ub) {
        const int t = blockIdx.x * 256 + threadIdx.x;
        const bool in = t < G.nU;
        const short2 g = in ? G.up[t] : make_short2(0, 0);
        const int m = in ? G.up_ring[t] : 255;
        const bool on = in && cell_filled(G.n, mask, accw, g.x, g.y);
        if (in) T.mapF[g.y * G.W + g.x] = on ? (uint8_t)(m + 1) : (uint8_t)0;
        const unsigned peers = __match_any_sync(FULL, m);
        const int pf = ring_slot(on, peers, lane, T.cnt + m), ph = ring_slot(in && !on, peers, lane, T.cnt + G.nb + m);
        if (on) T.F[G.up_off[m] + pf] = g;
        else if (in) T.H[G.up_off[m] + ph] = g;
        return;
    }
    const int t = (blockIdx.x - ub) * 256 + threadIdx.x;
    const bool in = t < G.nO;
    const uint32_t o = in ? G.orb[t] : 0u;
    const int m = in ? G.orb_ring[t] : 255;
    const int x = orb_x(o), y = orb_y(o);
    int nf = 0;
    if (in) {   // the upper-half images: (x, y), (y, x) if x < y, and their mirrors in x if x > 0
        nf = cell_filled(G.n, mask, accw, x, y);
        if (x > 0) nf += cell_filled(G.n, mask, accw, -x, y);
        if (x < y) {
            nf += cell_filled(G.n, mask, accw, y, x);
            if (x > 0) nf += cell_filled(G.n, mask, accw, -y, x);
        }
        T.nf[t] = (uint8_t)nf;
    }
    const int nh = in ? orb_w(o) - nf : 0;
    const unsigned peers = __match_any_sync(FULL, m);
    const int p = ring_slot(nh > 0, peers, lane, T.cnt + 2 * G.nb + m);
    if (nh > 0) {
        T.HO[G.orb_off[m] + p] = orb_pack(x, y, nh);
        if (!(x & 1) && !(y & 1)) {
            const int b = G.mapA[(y / 2) * G.W + x / 2];
            if (b) atomicAdd(&T.fix[(size_t)m * G.nb + b - 1], (unsigned long long)nh);
        }
    }
}

// Pair-count jobs: (set of g1, set of g2, map looked up).
//   DIRECT  F upper half x F, filled map      Q  H upper half x H, filled map
//   P       H upper half x H, annulus map     M  orbits with holes x A above h / 2, annulus map
//   FULL    orbits x A, annulus map
// DIRECT and Q share a table (one route or the other); FULL is the setup's.
enum { JOB_DIRECT = 0, JOB_Q = 1, JOB_P = 2, JOB_M = 3, JOB_FULL = 4 };

// Ring pair (a <= b) of pair index pr = a nb - a (a - 1) / 2 + (b - a): a from the
// quadratic's root in FP32, corrected by whole steps.
__device__ __forceinline__ void pair_of(int pr, int nb, int &a, int &b) {
    const float B = 2.f * (float)nb + 1.f;
    a = (int)((B - sqrtf(fmaxf(B * B - 8.f * (float)pr, 0.f))) * 0.5f);
    a = max(0, min(a, nb - 1));
    while (a > 0 && a * nb - a * (a - 1) / 2 > pr) --a;
    while (a + 1 < nb && (a + 1) * nb - (a + 1) * a / 2 <= pr) ++a;
    b = a + (pr - (a * nb - a * (a - 1) / 2));
}

// First upper-half cell of ring b above half the lowest orbit of ring a (index in ring b's list).
__device__ __forceinline__ int suffix_start(const CountGeom &G, int a, int b) {
    const uint32_t o = G.orb[G.orb_off[a]];
    const int kh = orb_y(o) * G.K + orb_x(o);
    int lo = 0, hi = G.up_off[b + 1] - G.up_off[b];
    const short2 *U = G.up + G.up_off[b];
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (2 * (U[mid].y * G.K + U[mid].x) > kh) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

struct ItemArgs {
    int chunk, need_full, cap0, cap1;
    int ctas;                                        // of the pair kernel
    int small_ok;                                    // the lists hold items of INNER_S
    int4 *items0, *items1;
    int32_t *err;
    unsigned long long *tab0, *tabP, *tabM, *full;   // [nb^3]; full cleared when need_full
};

// Mean l (block b < nb: ring b), the pair-count tables cleared and the work items written.  Every block
// finds the route by itself from the ring counts; the pairs of every job are dealt to the warps, which
// reserve their items' places in the job's list with one atomic (the items' order does not matter).
// item = (a | b << 8 | job << 16 | outer-is-x << 24, outer start, inner start, suffix start)
__global__ void __launch_bounds__(256) k_ring_finish(CountGeom G, float du, RingTables T, double *__restrict__ ellbar,
                                                     ItemArgs ia) {
    const int nb = G.nb, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (ellbar && (int)blockIdx.x < nb) {   // the sum of |g| over the filled cells, in a fixed order
        __shared__ double part[8];
        const int m = blockIdx.x;
        float sh = 0.f, sl = 0.f;
        for (int t = G.orb_off[m] + threadIdx.x; t < G.orb_off[m + 1]; t += 256) {
            const uint32_t o = G.orb[t];
            const float k = (float)T.nf[t];
            float h, l;
            df_sqrt_int(orb_x(o) * orb_x(o) + orb_y(o) * orb_y(o), h, l);
            const float p = __fmul_rn(h, k);
            df_add(sh, sl, p, fmaf(l, k, fmaf(h, k, -p)));
        }
        // a thread's few terms in double-float, everything beyond in FP64: the partial sums of a whole ring in
        // double-float cost 1.7e-15 rms (R = 350, 128 rings; 4e-16 so)
        double s = (double)sh + (double)sl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == 0) part[warp] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) s += part[w];
            const int32_t c = T.cnt[m];
            ellbar[m] = c > 0 ? 2.0 * 3.14159265358979323846 * (double)du * s / (double)c : nan("");
        }
    }
    if (!ia.items0) return;
    // the route: pairs visited by either (suffix sums over the rings b >= a)
    __shared__ int cF[ABS_MAX_BINS], cH[ABS_MAX_BINS];
    __shared__ int use_holes_s, inner_s;
    for (int i = threadIdx.x; i < nb; i += 256) {
        cF[i] = T.cnt[i];
        cH[i] = T.cnt[nb + i];
    }
    __syncthreads();
    if (warp == 0) {
        unsigned long long dir = 0, hol = 0;
        unsigned long long tf = 0, th = 0;     // filled cells and holes of the rings above this lane's block
        const int per = (nb + 31) / 32, lo = min(nb, lane * per), hi = min(nb, lo + per);
        for (int i = lo; i < hi; ++i) {
            tf += 2 * cF[i];
            th += 2 * cH[i];
        }
        const unsigned long long of = tf, oh = th;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {     // inclusive suffix sums over the lanes
            const unsigned long long yf = __shfl_down_sync(FULL, tf, o), yh = __shfl_down_sync(FULL, th, o);
            if (lane + o < 32) {
                tf += yf;
                th += yh;
            }
        }
        tf -= of;
        th -= oh;
        for (int i = hi - 1; i >= lo; --i) {
            tf += 2 * cF[i];
            th += 2 * cH[i];
            dir += (unsigned long long)cF[i] * tf;
            hol += 2 * (unsigned long long)cH[i] * th + (unsigned long long)T.cnt[2 * nb + i] * G.nU;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dir += __shfl_xor_sync(FULL, dir, o);
            hol += __shfl_xor_sync(FULL, hol, o);
        }
        if (lane == 0) {
            use_holes_s = hol < dir ? 1 : 0;
            const unsigned long long visits = ia.need_full ? ~0ull : hol < dir ? hol : dir;
            inner_s = ia.small_ok && visits / ((unsigned long long)ia.chunk * INNER) < 4ull * ia.ctas ? INNER_S : INNER;
        }
    }
    __syncthreads();
    const int holes = use_holes_s, inner = inner_s;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        T.ctl[4] = holes;
        T.ctl[5] = inner;
    }
    // the tables' rows that will be added to (the holes' route: rings a with holes only)
    const int64_t row = (int64_t)nb * nb;
    for (int a = blockIdx.x; a < nb; a += gridDim.x) {
        if (ia.need_full)
            for (int64_t i = threadIdx.x; i < row; i += 256) ia.full[a * row + i] = 0ull;
        if (holes && cH[a] == 0) continue;
        for (int64_t i = threadIdx.x; i < row; i += 256) {
            ia.tab0[a * row + i] = 0ull;
            if (holes) ia.tabP[a * row + i] = ia.tabM[a * row + i] = 0ull;
        }
    }
    // pairs: [DIRECT or Q][P][M][FULL]
    const int np = nb * (nb + 1) / 2;
    const int n1 = np, n2 = n1 + (holes ? np : 0), n3 = n2 + (holes ? nb * nb : 0), n4 = n3 + (ia.need_full ? np : 0);
    __shared__ int w_pos[8][32];
    __shared__ int4 w_pair[8][32];   // (a | b << 8 | job << 16 | outer-is-x << 24, inner chunks, suffix start, -)
    for (int p0 = (blockIdx.x * 8 + warp) * 32; p0 < n4; p0 += gridDim.x * 256) {
        const int pr = p0 + lane;
        int job = pr < n1 ? (holes ? JOB_Q : JOB_DIRECT) : pr < n2 ? JOB_P : pr < n3 ? JOB_M : JOB_FULL;
        int a = 0, b = 0, start = 0, nx = 0, ny = 0;
        if (pr < n4) {
            if (job == JOB_M) {
                a = (pr - n2) / nb;
                b = (pr - n2) - a * nb;
                nx = T.cnt[2 * nb + a];
                if (nx) {
                    start = suffix_start(G, a, b);
                    ny = G.up_off[b + 1] - G.up_off[b] - start;
                }
            } else {
                pair_of(job == JOB_FULL ? pr - n3 : job == JOB_P ? pr - n1 : pr, nb, a, b);
                nx = job == JOB_FULL ? G.orb_off[a + 1] - G.orb_off[a] : job == JOB_DIRECT ? cF[a] : cH[a];
                ny = 2 * (job == JOB_FULL ? G.up_off[b + 1] - G.up_off[b] : job == JOB_DIRECT ? cF[b] : cH[b]);
            }
        }
        const bool outer_x = nx >= ny;
        const int no = outer_x ? nx : ny, ni = outer_x ? ny : nx;
        const int n_ic = (ni + inner - 1) / inner;
        const int cnt = ni > 0 ? (no + ia.chunk - 1) / ia.chunk * n_ic : 0;
        const int lst = job >= JOB_P ? 1 : 0;
        // places: an inclusive scan over the warp, one reservation a list
        int s0 = lst ? 0 : cnt, s1 = lst ? cnt : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y0 = __shfl_up_sync(FULL, s0, o), y1 = __shfl_up_sync(FULL, s1, o);
            if (lane >= o) {
                s0 += y0;
                s1 += y1;
            }
        }
        const int t0 = __shfl_sync(FULL, s0, 31), t1 = __shfl_sync(FULL, s1, 31), tot = t0 + t1;
        if (tot == 0) continue;
        int base0 = 0, base1 = 0;
        if (lane == 0) {
            if (t0) base0 = atomicAdd(T.ctl, t0);
            if (t1) base1 = atomicAdd(T.ctl + 1, t1);
        }
        base0 = __shfl_sync(FULL, base0, 0);
        base1 = __shfl_sync(FULL, base1, 0);
        if (lane == 0 && (base0 + t0 > ia.cap0 || base1 + t1 > ia.cap1)) atomicCAS(ia.err, 0, DERR_CAPACITY);
        w_pos[warp][lane] = s0 + s1 - cnt;   // lists are adjacent in pair order, so one running position serves both
        w_pair[warp][lane] = make_int4(a | b << 8 | job << 16 | (outer_x ? 1 << 24 : 0), n_ic, start, 0);
        __syncwarp();
        for (int t = lane; t < tot; t += 32) {
            int lo = 0, hi = 31;   // last pair with w_pos <= t
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (w_pos[warp][mid] <= t) lo = mid;
                else hi = mid - 1;
            }
            const int4 P = w_pair[warp][lo];
            const int c = t - w_pos[warp][lo], oc = c / P.y, ic = c - oc * P.y;
            const int4 item = make_int4(P.x, oc * ia.chunk, ic * inner, P.z);
            if (((P.x >> 16) & 7) >= JOB_P) {
                if (base1 + t - t0 < ia.cap1) ia.items1[base1 + t - t0] = item;
            } else if (base0 + t < ia.cap0) {
                ia.items0[base0 + t] = item;
            }
        }
        __syncwarp();
    }
}

struct GatherArgs {   // T_ijk for the listed triplets
    int32_t n_trip;
    const int32_t *ijk;
    int64_t *T;
    const unsigned long long *tab0, *tabP, *tabM, *full;
    unsigned *ticket;    // by the last CTA of k_count_pairs to finish; nullptr: by k_count_gather
};

// Reads the tables' rows of rings with holes only (the others hold nothing).
__device__ __forceinline__ int64_t gather_one(int nb, const RingTables &R, const GatherArgs &ga, bool holes, int t) {
    const int i = ga.ijk[3 * t], j = ga.ijk[3 * t + 1], k = ga.ijk[3 * t + 2];
    if (i < 0 || j < i || k < j || k >= nb) return 0;
    auto at = [nb](int a, int b, int c) { return ((size_t)a * nb + b) * nb + c; };
    if (!holes) return 2 * (int64_t)__ldcg(ga.tab0 + at(i, j, k));
    const bool hi = R.cnt[nb + i] != 0, hj = R.cnt[nb + j] != 0, hk = R.cnt[nb + k] != 0;
    auto one = [&](int a, int b, int c) {
        int64_t v = (int64_t)__ldcg(ga.tabM + at(a, b, c)) + (int64_t)__ldcg(ga.tabM + at(a, c, b));
        if (b == c) v += (int64_t)R.fix[(size_t)a * nb + b];
        return v;
    };
    int64_t s = (int64_t)__ldcg(ga.full + at(i, j, k));
    if (hi) s -= one(i, j, k);
    if (hj) s -= one(j, i, k);
    if (hk) s -= one(k, i, j);
    if (hi && hk) s += (int64_t)__ldcg(ga.tabP + at(i, k, j));
    if (hj && hk) s += (int64_t)__ldcg(ga.tabP + at(j, k, i));
    if (hi && hj) s += (int64_t)__ldcg(ga.tab0 + at(i, j, k));
    return 2 * s;
}

// The lookups of one item's inner cells (staged as lin, x, half-plane key, weight) against this thread's
// G1 outer cells.  WT: weighted cells and the half-plane test (jobs M and FULL).  The map loads of KU
// inner cells are issued before their run-length updates, which never feed a load: KU x G1 lookups in
// flight per thread.
template <bool WT>
__device__ __forceinline__ void count_inner(const int4 *stage, int nin, const uint8_t *__restrict__ map,
                                            const int (&lin1)[G1], const int (&xr1)[G1], const int (&k1)[G1],
                                            const uint32_t (&w1)[G1], uint32_t span, uint16_t *myhist) {
    int cur[G1];
    uint32_t cnt[G1];
#pragma unroll
    for (int q = 0; q < G1; ++q) {
        cur[q] = 0;
        cnt[q] = 0;
    }
    auto flush = [&](int q) { myhist[(size_t)cur[q] * 32] += (uint16_t)(WT ? cnt[q] * w1[q] : cnt[q]); };
    auto look = [&](const int4 &c, int q) {
        const bool in = (uint32_t)(xr1[q] + c.y) <= span && (!WT || k1[q] + c.z > 0);
        return in ? (int)map[abs(lin1[q] + c.x)] : 0;
    };
    auto step = [&](int r, int w, int q) {
        if (r != cur[q]) {
            flush(q);
            cur[q] = r;
            cnt[q] = 0;
        }
        cnt[q] += WT ? (uint32_t)w : 1u;
    };
    int k = 0;
    for (; k + KU <= nin; k += KU) {
        int rr[KU][G1], w2[KU];
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            const int4 c = stage[k + u];
            w2[u] = c.w;
#pragma unroll
            for (int q = 0; q < G1; ++q) rr[u][q] = look(c, q);
        }
#pragma unroll
        for (int u = 0; u < KU; ++u)
#pragma unroll
            for (int q = 0; q < G1; ++q) step(rr[u][q], w2[u], q);
    }
    for (; k < nin; ++k) {
        const int4 c = stage[k];
#pragma unroll
        for (int q = 0; q < G1; ++q) step(look(c, q), c.w, q);
    }
#pragma unroll
    for (int q = 0; q < G1; ++q) flush(q);
}

// Persistent CTAs take the items of list 0 (filled map), then of list 1 (annulus map).
template <bool MAP_IN_SMEM>
__global__ void __launch_bounds__(CT) k_count_pairs(CountGeom G, RingTables T, const int4 *__restrict__ items0,
                                                    const int4 *__restrict__ items1, int cap0, int cap1,
                                                    unsigned long long *__restrict__ tab0,
                                                    unsigned long long *__restrict__ tabP,
                                                    unsigned long long *__restrict__ tabM,
                                                    unsigned long long *__restrict__ full, GatherArgs ga) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int nwarps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hs = G.nb + 1;                       // histogram slots (0 = none)
    uint16_t *hist = (uint16_t *)smem;             // [nwarps][hs][32]
    uint32_t *hist32 = (uint32_t *)smem;           // the same, as pairs of counters (clearing)
    const int hwords = nwarps * hs * 16;
    int4 *stage = (int4 *)(hist + (size_t)nwarps * hs * 32);   // [INNER] inner cells: lin, x, half-plane key, weight
    uint8_t *map_s = (uint8_t *)(stage + INNER);
    uint16_t *myhist = hist + (size_t)warp * hs * 32 + lane;
    const uint32_t span = 2u * (uint32_t)G.R;   // |x1 + x2| <= R  <=>  x1 + R + x2 in [0, 2R]
    __shared__ int it_s;
    __shared__ int4 item_s;
    const int inner = T.ctl[5];
    bool clean = false;
    for (int lst = 0; lst < 2; ++lst) {
        const int ni = min(T.ctl[lst], lst ? cap1 : cap0);
        if (ni <= 0) continue;
        const uint8_t *map_g = lst ? G.mapA : T.mapF, *map = MAP_IN_SMEM ? map_s : map_g;
        const int4 *items = lst ? items1 : items0;
        bool loaded = !MAP_IN_SMEM;
        // thread 0 fetches the next item while the CTA counts this one (dynamic: items differ in size)
        int next = 0;
        int4 nitem = make_int4(0, 0, 0, 0);
        if (threadIdx.x == 0) {
            next = atomicAdd(T.ctl + 2 + lst, 1);
            if (next < ni) nitem = items[next];
        }
        for (;;) {
            if (threadIdx.x == 0) {
                it_s = next;
                item_s = nitem;
            }
            __syncthreads();
            if (it_s >= ni) break;
            const int4 I = item_s;
            if (!loaded) {   // a CTA that takes no item loads no map and clears nothing
                const int64_t mb = G.base + 1, nv = mb / 16;
                for (int64_t i = threadIdx.x; i < nv; i += blockDim.x) ((uint4 *)map_s)[i] = ((const uint4 *)map_g)[i];
                for (int64_t i = nv * 16 + threadIdx.x; i < mb; i += blockDim.x) map_s[i] = map_g[i];
                loaded = true;
            }
            if (!clean) {
                for (int i = threadIdx.x; i < hwords; i += blockDim.x) hist32[i] = 0u;
                clean = true;
            }
            const int a = I.x & 255, b = (I.x >> 8) & 255, job = (I.x >> 16) & 7;
            const bool outer_x = (I.x & (1 << 24)) != 0;
            const bool orbit = job >= JOB_M;       // X holds packed orbits
            // set X: an upper-half list or orbits; set Y: whole (the upper half, then its negation),
            // or (M) the negated upper half from the suffix start on
            const short2 *X = (job == JOB_DIRECT ? T.F : T.H) + G.up_off[a];
            const uint32_t *XO = job == JOB_FULL ? G.orb + G.orb_off[a] : T.HO + G.orb_off[a];
            const short2 *Yu = (job == JOB_DIRECT ? T.F : orbit ? G.up : T.H) + G.up_off[b];
            const int cU = G.up_off[b + 1] - G.up_off[b];
            const int nx = job == JOB_FULL ? G.orb_off[a + 1] - G.orb_off[a]
                                           : T.cnt[(job == JOB_DIRECT ? 0 : orbit ? 2 : 1) * G.nb + a];
            const int hy = orbit ? cU : T.cnt[(job == JOB_DIRECT ? 0 : 1) * G.nb + b];
            const int ny = job == JOB_M ? cU - I.w : 2 * hy;
            auto load_x = [&](int k) {
                if (!orbit) return make_int4(X[k].y * G.W + X[k].x, X[k].x, 0, 1);
                const uint32_t o = XO[k];
                const int x = orb_x(o), y = orb_y(o);
                return make_int4(y * G.W + x, x, job == JOB_M ? -(y * G.K + x) : 0, orb_w(o));
            };
            auto load_y = [&](int k) {   // key 1: the test always holds
                const bool neg = job == JOB_M || k >= hy;
                const short2 g = Yu[job == JOB_M ? k + I.w : neg ? k - hy : k];
                const int l = g.y * G.W + g.x;
                return make_int4(neg ? -l : l, neg ? -g.x : g.x, job == JOB_M ? 2 * (g.y * G.K + g.x) : 1, 1);
            };
            const int no = outer_x ? nx : ny;
            const int nin = min(inner, (outer_x ? ny : nx) - I.z);
            int lin1[G1], xr1[G1], k1[G1];   // lin, x + R and half-plane key of this thread's outer cells
            uint32_t w1[G1];
#pragma unroll
            for (int q = 0; q < G1; ++q) {
                const int k = I.y + q * blockDim.x + threadIdx.x;
                int4 c = make_int4(0, 0, 0, 0);
                if (k < no) c = outer_x ? load_x(k) : load_y(k);
                lin1[q] = c.x;
                // an empty slot fails the x-range test of every lookup (|x2| <= R), so the lookups
                // need no separate validity test
                xr1[q] = k < no ? c.y + G.R : 0x40000000;
                k1[q] = c.z;
                w1[q] = (uint32_t)c.w;
            }
            for (int k = threadIdx.x; k < nin; k += blockDim.x) stage[k] = outer_x ? load_y(I.z + k) : load_x(I.z + k);
            __syncthreads();
            if (threadIdx.x == 0) next = atomicAdd(T.ctl + 2 + lst, 1);
            if (orbit) count_inner<true>(stage, nin, map, lin1, xr1, k1, w1, span, myhist);
            else count_inner<false>(stage, nin, map, lin1, xr1, k1, w1, span, myhist);
            if (threadIdx.x == 0 && next < ni) nitem = items[next];
            __syncthreads();
            unsigned long long *tab = job == JOB_P ? tabP : job == JOB_M ? tabM : job == JOB_FULL ? full : tab0;
            for (int k = 1 + warp; k < hs; k += nwarps) {
                uint64_t sacc = 0;
                for (int w = 0; w < nwarps; ++w) sacc += hist[((size_t)w * hs + k) * 32 + lane];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sacc += __shfl_xor_sync(FULL, sacc, o);
                if (lane == 0 && sacc)
                    atomicAdd(&tab[((size_t)a * G.nb + b) * G.nb + (k - 1)], (unsigned long long)sacc);
            }
            __syncthreads();
            for (int k = threadIdx.x; k < hwords; k += blockDim.x) hist32[k] = 0u;
        }
        __syncthreads();   // everyone has seen the end of the list
    }
    if (!ga.ticket) return;
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ga.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const bool holes = T.ctl[4] != 0;
    for (int t = threadIdx.x; t < ga.n_trip; t += blockDim.x) ga.T[t] = gather_one(G.nb, T, ga, holes, t);
    if (threadIdx.x == 0) *ga.ticket = 0u;
}

__global__ void __launch_bounds__(256) k_count_gather(int nb, RingTables T, GatherArgs ga) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t < ga.n_trip) ga.T[t] = gather_one(nb, T, ga, T.ctl[4] != 0, t);
}

CountGeom cgeom(const Setup &s) {
    CountGeom G;
    G.n = s.n;
    G.nb = s.nb;
    G.R = s.R;
    G.W = 2 * s.R + 1;
    G.K = 2 * (3 * s.R + 1);
    G.nU = (int)s.up_off.back();
    G.nO = s.n_orb;
    G.base = (int64_t)2 * s.R * G.W + s.R;   // largest |lin| of a pair sum with |h_x| <= R
    const uint8_t *p = (const uint8_t *)s.d_ring_geom;
    G.up = (const short2 *)(p + s.rg_at[0]);
    G.up_ring = p + s.rg_at[1];
    G.up_off = (const int32_t *)(p + s.rg_at[2]);
    G.orb = (const uint32_t *)(p + s.rg_at[3]);
    G.orb_ring = p + s.rg_at[4];
    G.orb_off = (const int32_t *)(p + s.rg_at[5]);
    G.mapA = p + s.rg_at[6];
    return G;
}

int64_t map_bytes_of(const CountGeom &G) { return cdiv(G.base + 1, 16) * 16; }

// Threads of a counting CTA: lane-private histograms of 2 (nb + 1) bytes a thread within 96 KB.
int count_warps(int nb) {
    return (int)std::min<size_t>(CT / 32, (96 * 1024) / ((size_t)(nb + 1) * 32 * 2));
}

// The ring geometry's device tables (one allocation) and the counts' item capacities, made on the first
// call that counts or averages over a ring.
bool make_ring_geometry(Setup &s) {
    const int nb = s.nb, R = s.R, W = 2 * R + 1;
    const int64_t nU = s.up_off.back();
    std::vector<short2> up((size_t)nU);
    std::vector<uint8_t> up_ring((size_t)nU), orb_ring, map((size_t)map_bytes_of([&] {
        CountGeom g{};
        g.base = (int64_t)2 * R * W + R;
        return g;
    }()), 0);
    std::vector<uint32_t> orb;
    std::vector<int32_t> up_off(nb + 1), orb_off(nb + 1, 0);
    for (int m = 0; m <= nb; ++m) up_off[m] = (int32_t)s.up_off[m];
    std::vector<std::vector<uint32_t>> by(nb);
    std::vector<int32_t> at(up_off.begin(), up_off.end());
    for (int y = 0; y <= R; ++y)
        for (int x = y == 0 ? 1 : -R; x <= R; ++x) {
            const int64_t r2 = (int64_t)x * x + (int64_t)y * y;
            if (r2 < s.q[0] || r2 >= s.q[nb]) continue;
            const int m = (int)(std::upper_bound(s.q.begin(), s.q.end(), r2) - s.q.begin()) - 1;
            up[at[m]] = make_short2((short)x, (short)y);
            up_ring[at[m]++] = (uint8_t)m;
            map[(size_t)y * W + x] = (uint8_t)(m + 1);
            if (x >= 0 && x <= y) by[m].push_back(orb_pack(x, y, x == 0 || x == y ? 2 : 4));
        }
    for (int m = 0; m < nb; ++m) {
        orb_off[m + 1] = orb_off[m] + (int32_t)by[m].size();
        orb.insert(orb.end(), by[m].begin(), by[m].end());
        orb_ring.insert(orb_ring.end(), by[m].size(), (uint8_t)m);
    }
    s.n_orb = (int)orb.size();
    // work items at most: DIRECT or Q in list 0; P, M and FULL in list 1 (every list at its longest)
    const int64_t chunk = (int64_t)std::max(count_warps(nb), 1) * 32 * G1;
    int64_t c0 = 0, c1 = 0;
    for (int inner : {INNER, INNER_S}) {
        auto items = [&](int64_t x, int64_t y) { return cdiv(std::max(x, y), chunk) * cdiv(std::min(x, y), inner); };
        int64_t n0 = 0, n1 = 0;
        for (int a = 0; a < nb; ++a)
            for (int b = 0; b < nb; ++b) {
                const int64_t ua = up_off[a + 1] - up_off[a], ub = up_off[b + 1] - up_off[b], oa = orb_off[a + 1] - orb_off[a];
                if (a <= b) {
                    n0 += items(ua, 2 * ub);
                    n1 += items(ua, 2 * ub) + items(oa, 2 * ub);
                }
                n1 += items(oa, ub);
            }
        s.small_items = inner == INNER_S && std::max(n0, n1) <= 1 << 21;   // 32 MB a list at most
        if (inner == INNER || s.small_items) {
            c0 = n0;
            c1 = n1;
        }
    }
    s.item_cap[0] = (int)std::min<int64_t>(std::max<int64_t>(c0, 1), 1 << 26);
    s.item_cap[1] = (int)std::min<int64_t>(std::max<int64_t>(c1, 1), 1 << 26);
    const void *src[7] = {up.data(), up_ring.data(), up_off.data(), orb.data(), orb_ring.data(), orb_off.data(), map.data()};
    const size_t bytes[7] = {up.size() * sizeof(short2), up_ring.size(), up_off.size() * sizeof(int32_t),
                             orb.size() * sizeof(uint32_t), orb_ring.size(), orb_off.size() * sizeof(int32_t), map.size()};
    size_t total = 0;
    for (int k = 0; k < 7; ++k) {
        s.rg_at[k] = total;
        total += (bytes[k] + 255) / 256 * 256;
    }
    std::vector<uint8_t> host(total, 0);
    for (int k = 0; k < 7; ++k)
        if (bytes[k]) std::memcpy(host.data() + s.rg_at[k], src[k], bytes[k]);
    if (cudaMalloc(&s.d_ring_geom, total) != cudaSuccess) {
        cudaGetLastError();
        s.d_ring_geom = nullptr;
        return false;
    }
    if (cudaMemcpy(s.d_ring_geom, host.data(), total, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(s.d_ring_geom);
        s.d_ring_geom = nullptr;
        return false;
    }
    return true;
}

// Ring tables of the filled set; with ia the tables and work items of the counts too.
abs_status ring_tables(abs_ctx *ctx, const Setup &s, const uint8_t *d_mask, const double *d_accw, RingTables &T,
                       double *d_ellbar, ItemArgs *ia) {
    if (!s.d_ring_geom && !make_ring_geometry(const_cast<Setup &>(s))) return fail(ctx, ABS_ERR_OOM, "ring geometry");
    const CountGeom G = cgeom(s);
    const int64_t U = std::max(G.nU, 1), O = std::max(G.nO, 1), mb = map_bytes_of(G);
    short2 *lists = (short2 *)workspace(ctx, "ring.lists", sizeof(short2) * 2 * U + sizeof(uint32_t) * O + O);
    // the filled map, the hole table, the counters: cleared together
    const int64_t cb = mb + sizeof(unsigned long long) * s.nb * s.nb + sizeof(int32_t) * 3 * s.nb + sizeof(int) * 8;
    uint8_t *clr = (uint8_t *)workspace(ctx, "ring.maps", cb);
    if (!lists || !clr) return fail(ctx, ABS_ERR_OOM, "ring table workspace");
    T.F = lists;
    T.H = lists + U;
    T.HO = (uint32_t *)(lists + 2 * U);
    T.nf = (uint8_t *)(T.HO + O);
    T.mapF = clr;
    T.fix = (unsigned long long *)(clr + mb);
    T.cnt = (int32_t *)(T.fix + (size_t)s.nb * s.nb);
    T.ctl = (int *)(T.cnt + 3 * s.nb);
    StageTimer timer(ctx, "ring_lists");
    cudaStream_t st = ctx->stream;
    cudaMemsetAsync(clr, 0, cb, st);
    const int ub = (int)cdiv(U, 256), ob = (int)cdiv(O, 256);
    k_ring_cells<<<ub + ob, 256, 0, st>>>(G, ub, d_mask, (const unsigned long long *)d_accw, T);
    const ItemArgs none{};
    // blocks: a ring each for the mean l and the tables, and enough warps for the pairs (32 each)
    const int np = s.nb * s.nb;
    const int blocks = ia ? std::max<int>(s.nb, std::min<int>((int)cdiv(3 * np, 256), 2 * ctx->sm_count)) : s.nb;
    k_ring_finish<<<blocks, 256, 0, st>>>(G, s.du, T, d_ellbar, ia ? *ia : none);
    return check_launch(ctx, "ring lists");
}

}  // namespace

abs_status launch_counts(abs_ctx *ctx, const Setup &s, const uint8_t *d_mask, int32_t n_trip,
                         const int32_t *d_ijk, int64_t *d_count, double *d_ellbar, const double *d_accw) {
    RingTables T;
    if (n_trip == 0 || !d_count) return ring_tables(ctx, s, d_mask, d_accw, T, d_ellbar, nullptr);
    if (!s.d_ring_geom && !make_ring_geometry(const_cast<Setup &>(s))) return fail(ctx, ABS_ERR_OOM, "ring geometry");
    const CountGeom G = cgeom(s);
    const int hs = s.nb + 1;
    const int64_t map_bytes = map_bytes_of(G);
    const int nwarps = count_warps(s.nb);
    if (nwarps < 1) return fail(ctx, ABS_ERR_UNSUPPORTED, "too many rings for the count kernel");
    const int threads = nwarps * 32;
    const int64_t fixed_bytes = (int64_t)nwarps * hs * 32 * 2 + INNER * sizeof(int4);
    const bool map_smem = map_bytes + fixed_bytes <= 220 * 1024;
    const size_t smem = (size_t)fixed_bytes + (map_smem ? map_bytes : 0);
    // resident CTAs an SM (shared memory, threads and registers), for the persistent grid
    const auto kern = map_smem ? k_count_pairs<true> : k_count_pairs<false>;
    int per_sm = 1;
    allow_smem(kern, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    per_sm = std::max(per_sm, 1);
    const int cap0 = s.item_cap[0], cap1 = s.item_cap[1];
    int4 *items0 = (int4 *)workspace(ctx, "count.items0", sizeof(int4) * cap0);
    int4 *items1 = (int4 *)workspace(ctx, "count.items1", sizeof(int4) * cap1);
    unsigned *ticket = (unsigned *)workspace_zeroed(ctx, "count.tickets", sizeof(unsigned));
    const size_t tn = (size_t)s.nb * s.nb * s.nb;
    unsigned long long *tabs = (unsigned long long *)workspace(ctx, "count.tables", 3 * tn * sizeof(unsigned long long));
    // full-annulus counts: a property of the ring geometry, kept per configuration
    Setup &ms = const_cast<Setup &>(s);
    if (!ms.d_full_counts) {
        if (cudaMalloc(&ms.d_full_counts, tn * sizeof(unsigned long long)) != cudaSuccess) {
            cudaGetLastError();
            ms.d_full_counts = nullptr;
        }
    }
    if (!items0 || !items1 || !ticket || !tabs || !ms.d_full_counts) return fail(ctx, ABS_ERR_OOM, "count workspace");
    unsigned long long *tab0 = tabs, *tabP = tabs + tn, *tabM = tabs + 2 * tn, *full = ms.d_full_counts;
    ItemArgs ia{threads * G1, ms.full_counts_ready ? 0 : 1, cap0, cap1, ctx->sm_count * per_sm, s.small_items ? 1 : 0,
                items0, items1, ctx->d_err, tab0, tabP, tabM, full};
    ABS_CHECK(ring_tables(ctx, s, d_mask, d_accw, T, d_ellbar, &ia));
    {
        // long lists are gathered by a launch of their own (one CTA takes 0.3 ms for 1e5 triplets), short
        // ones by the last CTA of the pair kernel
        StageTimer timer(ctx, "count_pairs");
        const bool fused = n_trip <= GATHER_FUSED;
        const GatherArgs ga{n_trip, d_ijk, d_count, tab0, tabP, tabM, full, fused ? ticket : nullptr};
        kern<<<ctx->sm_count * per_sm, threads, smem, ctx->stream>>>(G, T, items0, items1, cap0, cap1, tab0, tabP, tabM,
                                                                     full, ga);
        if (!fused) k_count_gather<<<(int)cdiv(n_trip, 256), 256, 0, ctx->stream>>>(s.nb, T, ga);
    }
    ms.full_counts_ready = true;
    return check_launch(ctx, "counts");
}

abs_status launch_ellbar(abs_ctx *ctx, const Setup &s, const uint8_t *d_mask, double *d_ellbar) {
    RingTables T;
    return ring_tables(ctx, s, d_mask, nullptr, T, d_ellbar, nullptr);
}

}  // namespace absk
