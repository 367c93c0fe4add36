// Stage 3, precision form: the numerator of Eq. estimator_t as a split-BF16
// contraction on the 5th-generation tensor cores (tcgen05), middle-ring major.
//
// Rows r = (j, k), a pair of rings j <= k that closes a triangle with some
// ring i <= j, and columns i:
//   C[r][i] = sum_p A[r][p] B[i][p],  A[r][p] = D_j(p) D_k(p),  B[i][p] = D_i(p),
// so that S_ijk = N^-2 C[(j, k)][i].  B is the plain fields, the same for every
// row, and A the only operand that has to be formed.  Each FP32 operand x is
// split into x_hi = bf16(x) and x_lo = bf16(x - x_hi) (x - x_hi is exact in
// FP32, so the pair carries 16 significant bits) and the three products
// Ah Bh + Ah Bl + Al Bh accumulate into one FP32 accumulator in tensor memory
// (Al Bl is below the FP32 resolution of the sum).
//
// Layout.  The fields are split once per estimate (k_split_fields) into three
// chunk-blocked planes [P_pad / 64][nbp][64] (P_pad = P rounded up to 64
// pixels, zeros past P and past the last ring): BF16 hi, BF16 lo and an FP32
// copy, each row already in the 128-byte swizzle the kernel reads it in, so
// that a window of consecutive rings of one chunk is one contiguous bulk copy
// (cp.async.bulk) that lands in shared memory ready for use.
//
// Rows (j, k) are taken in (j, k) order and cut into blocks of 128 rows; inside
// a block the rows are ordered by (k, j), so that a warp's 32 rows read few
// distinct rings when forming A.  A block's ring columns i (from its lowest i
// rounded down to 8, rounded up to 16) are cut into column tiles of at most
// 128 (the MMA N).  Consecutive tiles form a set of at most two whose
// accumulator columns stay within a budget (autotuned, at most 128); a work item
// is one set over one range of pixels, and a persistent grid of one CTA per SM
// takes items from a queue (one atomic counter), ranges outermost, so that the
// sets that read the same pixels run at about the same time and share them in L2.
//
// Per 64-pixel chunk c of an item, four roles and their mbarriers:
//   loader (warp 0)    bulk copies of chunk c into stage s = c mod n_stages:
//                      the set's window of rings of the hi and lo planes (the
//                      MMA operand B, K-major, 128-byte swizzle) and the window
//                      of rings its rows form A from (FP32), counted on full[s];
//                      it reuses stage s once done[s] says chunk c - n_stages has
//                      finished with it;
//   formers (FW0 ..)   thread = one row (its tensor-memory lane) and 64 / FQ
//                      of the 64 pixels (32 with eight forming warps), for every tile
//                      of the set: A = D_j D_k in FP32, split, packed in BF16
//                      pairs and stored to A buffer (c & 1) of the tile in
//                      tensor memory (tcgen05.st); one arrival on a_full[c & 1]
//                      a warp per chunk.  Buffer (c & 1) is free again once
//                      done[] of chunk c - 2 has completed;
//   MMA issuers (1 ..) per tile, 4 K-steps x 3 MMAs (A from tensor memory, B
//                      from the stage), M = 128, N = the tile's ring columns,
//                      into accumulation region (g & 1) of group g = c / DRAIN;
//                      one tcgen05.commit per chunk to done[s] (the stage and
//                      the A buffers of chunk c are free), and at the end of
//                      a group one to d_full[g & 1];
//   drainers (DW0 ..)  add a complete group's region to long accumulators.
// Tensor-core accumulation in FP32 over long pixel ranges loses accuracy (the
// error grows with the number of chunks summed into one accumulator), so every
// DRAIN chunks the drainers read the group's region back (tcgen05.ld) into FP32
// registers, one long accumulator per (row, column) a thread owns, and release
// it (d_empty); the issuer meanwhile fills the other region.  After the item's
// last chunk the drainers write the long accumulators, column-major by tile
// (lanes contiguous), to the item's pixel range of the partial-sum array.  A
// second kernel adds the pixel ranges in double-float in a fixed order and gathers each
// triplet's entry.
//
// What bounds it: the formers, eight warps each with a serial chain of loads, products,
// splits and stores a tile (1.82 ms on 128 rings of 1,080^2, of which the MMAs alone take
// 0.9; half of the issue slots, ALU 43 %, two thirds of the shared-memory data path).  Draining in warps of
// their own took 0.1 ms off: the long accumulators, 64 registers a thread, had left the
// formers spilling.
//
// Rates that shaped this design, measured on GB300 with microbenchmarks: an MMA
// of M = 128, K = 16 costs max(45.5, N / 2) cycles of the tensor pipe, with A in
// tensor or shared memory alike; a tcgen05.commit between short MMAs costs about
// 270 cycles of issue, hence one per chunk for the whole set; tiled TMA loads
// of 128-byte rows reached about 26 bytes per clock per SM, contiguous bulk
// copies of the pre-swizzled blocks about 2.5 times that.
//
// Every mbarrier wait is bounded: on timeout the role sets a shared abort flag
// and leaves; the CTA then waits (bounded) for its copies and MMAs in flight,
// latches DERR_TIMEOUT, frees its tensor memory and returns.


#include <cuda_bf16.h>

#include <algorithm>
#include <map>

#include "abs_internal.cuh"

namespace absk {
namespace {

constexpr int TM = 128;              // rows per tile (MMA M)
constexpr int KC = 64;               // pixels per chunk (4 MMA K-steps of 16)
#ifndef ABS_TC_FORMERS
#define ABS_TC_FORMERS 8
#endif
constexpr int NFORM = ABS_TC_FORMERS;   // forming warps
constexpr int FQ = NFORM / 4;           // forming warps per tensor-memory lane quadrant
constexpr int FPX = KC / FQ;            // pixels of a chunk per forming thread
#ifndef ABS_TC_MAX_TILES
#define ABS_TC_MAX_TILES 2
#endif
#ifndef ABS_TC_ISSUERS
#define ABS_TC_ISSUERS ABS_TC_MAX_TILES
#endif
// MMA-issuing warps (one thread each): issuer e takes the tiles t with t % NISS == e.  A single
// thread issues at most one tcgen05.mma every ~45 cycles, so the tiles of a set issue in parallel.
constexpr int NISS = ABS_TC_ISSUERS;
constexpr int FW0 = 1 + NISS;           // first forming warp (warp 0 loads, warps 1 .. NISS issue)
constexpr int DW0 = FW0 + NFORM;        // first draining warp
constexpr int NDRAIN = 8;               // draining warps, two a tensor-memory lane quadrant
constexpr int NT = (DW0 + NDRAIN) * 32; // threads per CTA
// registers per thread: the register file is split over the SM's four schedulers (16,384
// each) and warps are dealt to them in turn, so the scheduler with the most warps
// (5 of 19) bounds it, in steps of 8
#define TC_MAXREG 96
#ifndef ABS_TC_ASLOTS
#define ABS_TC_ASLOTS 2
#endif
constexpr int MAX_TILES = ABS_TC_MAX_TILES;   // tiles per set
constexpr int ASLOTS = ABS_TC_ASLOTS;         // chunks whose A buffers are in tensor memory at once (2 or 4)
static_assert(ASLOTS == 2 || ASLOTS == 4, "A slots: a power of two");
constexpr int MAX_STAGES = 8;
constexpr int TMEM_COLS = 512;
constexpr int A_COLS = 64;           // one A buffer: 32 columns of hi pairs, 32 of lo pairs
constexpr int NABUF = ASLOTS * MAX_TILES;   // A buffers: every tile of ASLOTS chunks (formers ahead of the MMAs)
constexpr int B_ROWS = 8;            // B windows start and end on 8-ring boundaries (the swizzle atom)
#ifndef ABS_TC_DRAIN
#define ABS_TC_DRAIN 8
#endif
constexpr int DRAIN = ABS_TC_DRAIN;  // chunks accumulated in tensor memory before the drainers take them
#ifndef ABS_TC_SET_COLS
#define ABS_TC_SET_COLS 128
#endif
// accumulator columns of a set: two accumulation regions beside the A buffers fit tensor
// memory up to 192; the draining threads' long accumulators (set columns / DQ each)
// bound it by registers
constexpr int MAX_SET_COLS = ABS_TC_SET_COLS;
static_assert(NABUF * A_COLS + 2 * MAX_SET_COLS <= TMEM_COLS, "A buffers and two regions fit tensor memory");
constexpr int MAX_TILE_N = 128;      // MMA N of a tile (wider column ranges are cut into several tiles)
constexpr int DQ = NDRAIN / 4;       // draining warps per quadrant
constexpr int MAXBLK = (MAX_SET_COLS / 8 + DQ - 1) / DQ;     // drain blocks of 8 columns per draining thread
constexpr int MAXSLOT = 8 * MAXBLK;  // long accumulators per draining thread
// A wait suspends the warp for up to WAIT_HINT_NS per try (it resumes as soon as the
// phase completes, so waiting warps take no issue slots), at most WAIT_LIMIT tries.
constexpr uint32_t WAIT_HINT_NS = 100000;
constexpr uint32_t WAIT_LIMIT = 1u << 15;

struct TcParams {
    int n_items;                 // sets x pixel ranges
    int n_sets;
    int64_t per_item;            // pixels of a range (a multiple of KC)
    int64_t P_pad;               // pixels per plane row
    int64_t dense;               // accumulator entries of one range (sum over tiles of 128 x N)
    int stage_bytes;             // one shared-memory stage (the largest set's)
    int n_stages;
};

// The split fields, chunk-blocked: [P_pad / 64][nbp][64] (nbp >= n_bins rings a block, zeros past
// n_bins and past P).  BF16 rows are 128 bytes in the 128-byte swizzle of the MMA operand (16-byte
// units XOR-permuted by ring & 7), FP32 rows 256 bytes permuted the same way, so that a set's window
// of rings of one chunk is one contiguous bulk copy and lands in shared memory ready for use.
struct TcPlanes {
    const __nv_bfloat16 *hi, *lo;
    const float *f32;
    int nbp;
};

// Set descriptor: first tile, tiles, B window (first ring, rows), F window (first ring, rows).
struct TcSet {
    int tile0, ntiles;
    int b_lo, b_n;
    int f_lo, f_n;
    int pad0, pad1;
};

// Tile descriptor: first column ring (multiple of 8), MMA N, offset in the dense accumulator.
struct TcTile {
    int i_lo, n;
    int64_t acc_off;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor of a K-major operand in the 128-byte swizzle:
// start address, leading byte offset 16 (unused by this layout), 8-row groups
// 1024 bytes apart, descriptor version 1, layout SWIZZLE_128B.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(16 >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, M x N.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The issuing warps run converged, every value the same in all lanes (uni), and only the issue itself is
// one lane's (elect.sync, always the same lane): so the compiler keeps the MMA's operands in uniform
// registers, where the instruction takes them.  Issued from inside an `if (lane == 0)`, each MMA
// waited for its operands to be moved there: 83 cycles apart instead of the tensor pipe's rate.
constexpr unsigned FULL = 0xffffffffu;
template <class T>
__device__ __forceinline__ T uni(T x) {
    return __shfl_sync(FULL, x, 0);
}

// D (tensor memory) += A (tensor memory) x B (shared-memory descriptor)^T, issued by one lane of the warp.
__device__ __forceinline__ void mma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
        ::"r"(tmem_d), "r"(tmem_a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n"
        ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

// An arrival of the lanes that are `on`, without a branch: the warp stays together.
__device__ __forceinline__ void mbar_arrive_if(uint32_t mbar, bool on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n\t}\n"
        ::"r"(mbar), "r"((int)on) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;\n"
                 ::"r"(mbar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok) : "r"(mbar), "r"(parity), "r"(WAIT_HINT_NS) : "memory");
    return ok != 0;
}

// Non-blocking test of the phase of the given parity.
__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity; false on timeout or once
// another role has given up (abort set).  A phase that has already completed
// is seen by one non-blocking test (cheaper than a suspending try).
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, const volatile int *abort_flag) {
    if (mbar_test(mbar, parity)) return true;
    for (uint32_t it = 0; it < WAIT_LIMIT; ++it) {
        if (mbar_try(mbar, parity)) return true;
        if (*abort_flag) return false;
    }
    return false;
}

// Bounded wait for work already in flight, whatever the abort flag says.
__device__ __forceinline__ bool mbar_drain(uint32_t mbar, uint32_t parity) {
    for (uint32_t it = 0; it < WAIT_LIMIT; ++it)
        if (mbar_try(mbar, parity)) return true;
    return false;
}

// Bulk copy of `bytes` contiguous bytes from global into shared memory, counted on mbar.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}

// Sixteen bytes of shared memory at a 32-bit shared address.  Not volatile, so the compiler may
// schedule it freely: callers derive the address from after_wait(), which keeps it below the
// mbarrier wait that makes the data visible.
__device__ __forceinline__ float4 lds128(uint32_t a) {
    float4 v;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}

// x, passed through an opaque volatile instruction: values computed from it cannot be moved above
// the volatile instructions (mbarrier waits) that precede this one.
__device__ __forceinline__ uint32_t after_wait(uint32_t x) {
    uint32_t y;
    asm volatile("mov.b32 %0, %1;\n" : "=r"(y) : "r"(x) : "memory");
    return y;
}

// Where a forming thread's FP32 values of ring m sit in an F window (rings from f_lo, rows of
// 256 bytes, 16-byte units XOR-permuted by m & 7): unit u = u0 ^ w of the thread's pixels (u0
// its first unit, w < 16 / (u0's step)) is at window + (rel ^ (w << 4)), rel = (m - f_lo) 256
// + ((u0 ^ (m & 7)) << 4), since the window starts on a 256-byte boundary and u0 and w have no
// bit in common.
__device__ __forceinline__ uint32_t frow_rel(int m, int f_lo, int u0) {
    return (uint32_t)((m - f_lo) * 256 + ((u0 ^ (m & 7)) << 4));
}

// Eight consecutive tensor-memory columns of one lane (completion awaited separately).
__device__ __forceinline__ void tmem_ld8(uint32_t ta, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(ta));
}

// Eight packed BF16 pairs of one lane to consecutive tensor-memory columns.
__device__ __forceinline__ void tmem_st(uint32_t ta, const uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n"
        ::"r"(ta), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
        : "memory");
}

// A pair of FP32 values as BF16 hi parts and BF16 residuals, each packed (first value low).
__device__ __forceinline__ void split2(float2 v, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __float22bfloat162_rn(v);
    hi = *(const uint32_t *)&h;
    // the two hi parts as FP32: a shift and a mask (two byte permutes, which the library's conversion
    // takes, both go to the pipe that already does the packing)
    const float2 hf = make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
    const float2 r = __ffma2_rn(hf, make_float2(-1.f, -1.f), v);   // v - hi, exact in FP32
    const __nv_bfloat162 l = __float22bfloat162_rn(r);
    lo = *(const uint32_t *)&l;
}

__global__ void __maxnreg__(TC_MAXREG) k_triple_tc(TcParams G, TcPlanes PL,
                                                     const TcSet *__restrict__ sets,
                                                     const TcTile *__restrict__ tiles,
                                                     const short2 *__restrict__ rowjk,
                                                     float *__restrict__ partial, int *__restrict__ next_item,
                                                     int32_t *__restrict__ err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[MAX_STAGES], done[MAX_STAGES], a_full[ASLOTS * MAX_TILES], d_full[2], d_empty[2], fin;
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_s;
    __shared__ int item_s;
    __shared__ TcSet set_s;
    __shared__ int t_ilo[MAX_TILES], t_n[MAX_TILES], t_col[MAX_TILES], sum_n;
    __shared__ int64_t t_off[MAX_TILES];
    __shared__ short2 rows_s[MAX_TILES][TM];
    __shared__ int blk_col[DQ][MAXBLK], n_blk[DQ];   // drain blocks of 8 columns per draining warp of a quadrant
    __shared__ int64_t blk_out[DQ][MAXBLK];
    // stages on a 1024-byte boundary (the 128-byte swizzle's atom); the launch adds 1 KB of slack
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int warp = uni((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < G.n_stages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&done[s]), NISS);
        }
        for (int b = 0; b < ASLOTS * MAX_TILES; ++b) mbar_init(smem_u32(&a_full[b]), NFORM);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&d_full[b]), NISS);
            mbar_init(smem_u32(&d_empty[b]), NDRAIN);
        }
        mbar_init(smem_u32(&fin), NISS);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(smem_u32(&tmem_holder)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = uni(tmem_holder);

    // role state that lives across items
    int st = 0, su = 0;      // stage and its use (loader, formers and issuer walk the same sequence)
    int cg = 0;              // chunks so far (A slot cg % ASLOTS, its use cg / ASLOTS)
    int hst[ASLOTS], hsu[ASLOTS];   // formers: stage and use of chunks cg - ASLOTS .. cg - 1, oldest first
#pragma unroll
    for (int x = 0; x < ASLOTS; ++x) hst[x] = hsu[x] = 0;
    int grp = 0;             // accumulation groups so far (region grp & 1, its use grp >> 1)
    int issued = 0;          // stages the loader filled (for the drain)
    for (;;) {
        // every thread is between items here, and no role writes the abort flag; the next
        // item comes from the launch's work counter (items in pixel-range order, so the
        // CTAs work on neighbouring ranges at any time and share them in L2)
        __syncthreads();
        if (__any_sync(FULL, abort_s)) break;
        if (threadIdx.x == 0) item_s = atomicAdd(next_item, 1);
        __syncthreads();
        const int e = uni(item_s);
        if (e >= G.n_items) break;
        const int set_id = e % G.n_sets;
        const int64_t p0 = (int64_t)(e / G.n_sets) * G.per_item;
        const int nchunks = (int)(min(G.per_item, G.P_pad - p0) / KC);
        // the set's tiles and rows
        if (threadIdx.x == 0) set_s = sets[set_id];
        __syncthreads();
        const TcSet S = set_s;
        if (threadIdx.x < S.ntiles) {
            const TcTile T = tiles[S.tile0 + threadIdx.x];
            t_ilo[threadIdx.x] = T.i_lo;
            t_n[threadIdx.x] = T.n;
            t_off[threadIdx.x] = T.acc_off;
        }
        for (int x = threadIdx.x; x < S.ntiles * TM; x += NT)
            rows_s[x / TM][x % TM] = rowjk[(size_t)S.tile0 * TM + x];
        __syncthreads();
        if (threadIdx.x == 0) {
            // tile columns inside an accumulation region; drain blocks dealt round robin
            int col = 0, b = 0;
            for (int h = 0; h < DQ; ++h) n_blk[h] = 0;
            for (int t = 0; t < S.ntiles; ++t) {
                t_col[t] = col;
                for (int c0 = 0; c0 < t_n[t]; c0 += 8, ++b) {
                    const int h = b % DQ, k = n_blk[h]++;
                    blk_col[h][k] = col + c0;
                    blk_out[h][k] = t_off[t] + (int64_t)c0 * TM;
                }
                col += t_n[t];
            }
            sum_n = col;
        }
        __syncthreads();
        const int b_bytes = S.b_n * 128;              // one plane of the B window
        const int f_bytes = S.f_n * 256;              // the F window (FP32 rows)
        const uint32_t tx_bytes = (uint32_t)(2 * b_bytes + f_bytes);
        const int region_cols = sum_n;
        // a whole warp's wait: one answer for all its lanes, which stay together for the collective
        // (.sync.aligned) instructions that follow
        auto wait = [&](const uint64_t *bar, int parity) {
            return __all_sync(FULL, mbar_wait(smem_u32(bar), (uint32_t)parity, &abort_s)) != 0;
        };

        if (warp == 0) {
            // ---------------- loader
            if (lane == 0) {
                for (int c = 0; c < nchunks; ++c) {
                    if (su > 0 && !mbar_wait(smem_u32(&done[st]), (uint32_t)((su - 1) & 1), &abort_s)) {
                        abort_s = 1;
                        break;
                    }
                    uint8_t *stage = smem + (size_t)st * G.stage_bytes;
                    const size_t blk = ((size_t)(p0 / KC) + c) * PL.nbp;   // the chunk's block of rings
                    const uint32_t fb = smem_u32(&full[st]);
                    mbar_arrive_tx(fb, tx_bytes);
                    bulk_g2s(smem_u32(stage), PL.hi + (blk + S.b_lo) * KC, (uint32_t)b_bytes, fb);
                    bulk_g2s(smem_u32(stage + b_bytes), PL.lo + (blk + S.b_lo) * KC, (uint32_t)b_bytes, fb);
                    bulk_g2s(smem_u32(stage + 2 * b_bytes), PL.f32 + (blk + S.f_lo) * KC, (uint32_t)f_bytes, fb);
                    ++issued;
                    if (++st == G.n_stages) {
                        st = 0;
                        ++su;
                    }
                }
            }
        } else if (warp <= NISS) {
            // ---------------- MMA issue (the whole warp, one lane's instruction): groups of DRAIN chunks into alternating
            // regions.  Every issuer walks every chunk (waits and commits alike, so that the
            // barriers count NISS arrivals a phase) and issues the MMAs of its own tiles.  The
            // per-chunk path is kept short (tile constants in registers, the stage's descriptor
            // advanced by addition): the tensor pipe idles while an issuer is between chunks.
            const int iss = warp - 1;
            const int ntiles = uni(S.ntiles);
            uint32_t idesc_t[MAX_TILES], col_t[MAX_TILES], rows_t[MAX_TILES];
#pragma unroll
            for (int t = 0; t < MAX_TILES; ++t) {
                idesc_t[t] = uni(t < ntiles ? make_idesc(TM, t_n[t]) : 0u);
                col_t[t] = uni(t < ntiles ? (uint32_t)t_col[t] : 0u);
                rows_t[t] = uni(t < ntiles ? (uint32_t)(t_ilo[t] - S.b_lo) * 8u : 0u);
            }
            const uint32_t cols = uni((uint32_t)region_cols);
            const uint64_t d_stage = (uint64_t)(G.stage_bytes >> 4), d_lo = (uint64_t)uni((uint32_t)b_bytes >> 4);
            const uint64_t d_base = desc_sw128(uni(smem_u32(smem)));
            uint64_t d_cur = d_base + (uint64_t)st * d_stage;   // this chunk's stage, B hi plane
            int gc = 0;                                          // chunk in the group
            for (int c = 0; c < nchunks; ++c) {
                const uint32_t region = (uint32_t)(NABUF * A_COLS) + (grp & 1) * cols;
                bool ok = true;
                if (gc == 0 && grp >= 2) {   // the group before last in this region has been drained
                    ok = wait(&d_empty[grp & 1], ((grp >> 1) - 1) & 1);
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                }
                ok = ok && wait(&full[st], su & 1);
                const uint32_t a_slot = tmem + (uint32_t)((cg & (ASLOTS - 1)) * MAX_TILES * A_COLS);
                const uint32_t first = gc > 0 ? 1u : 0u;
#pragma unroll
                for (int t = 0; t < MAX_TILES; ++t) {
                    if (t >= ntiles || !ok) break;
                    if (t % NISS != iss) continue;
                    // this tile's A buffers, formed ahead
                    ok = wait(&a_full[(cg & (ASLOTS - 1)) * MAX_TILES + t], (cg / ASLOTS) & 1);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    // a tile's rows and a K-step move only the descriptors' start-address field
                    // (16-byte units: 8 per ring row, 2 per 16 pixels)
                    const uint32_t acc = tmem + region + col_t[t];
                    const uint32_t a_hi = a_slot + (uint32_t)(t * A_COLS), a_lo = a_hi + 32;
                    const uint64_t dh0 = d_cur + rows_t[t], dl0 = dh0 + d_lo;
#pragma unroll
                    for (int ks = 0; ks < KC / 16; ++ks) {
                        mma_ts(acc, a_hi + 8u * ks, dh0 + 2u * ks, idesc_t[t], ks > 0 ? 1u : first);
                        mma_ts(acc, a_hi + 8u * ks, dl0 + 2u * ks, idesc_t[t], 1u);
                        mma_ts(acc, a_lo + 8u * ks, dh0 + 2u * ks, idesc_t[t], 1u);
                    }
                }
                if (!ok) {
                    abort_s = 1;
                    break;
                }
                // one commit a chunk: its MMAs done frees the stage and the chunk's A buffers
                mma_commit(smem_u32(&done[st]));
                ++cg;
                if (++st == G.n_stages) {
                    st = 0;
                    ++su;
                    d_cur = d_base;
                } else {
                    d_cur += d_stage;
                }
                if (gc == DRAIN - 1 || c == nchunks - 1) {   // the group is complete: the drainers take it
                    mma_commit(smem_u32(&d_full[grp & 1]));
                    ++grp;
                }
                if (++gc == DRAIN) gc = 0;
            }
        } else if (warp < DW0) {
            // ---------------- formers
            const int q = warp & 3;                   // tensor-memory lanes 32 q .. 32 q + 31
            const int h = (warp - FW0) >> 2;          // pixel part of the chunk (FPX pixels)
            const int row = 32 * q + lane;
            const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
            // this thread's rows of the set's tiles: offsets of D_j and D_k in an F window (a row the tile
            // does not have forms the window's first ring; its sums are never read)
            uint32_t rel_j[MAX_TILES], rel_k[MAX_TILES];
#pragma unroll
            for (int t = 0; t < MAX_TILES; ++t) {
                const short2 jk = t < S.ntiles ? rows_s[t][row] : make_short2(-1, -1);
                rel_j[t] = jk.x >= 0 ? frow_rel(jk.x, S.f_lo, (h * FPX) / 4) : 0u;
                rel_k[t] = jk.x >= 0 ? frow_rel(jk.y, S.f_lo, (h * FPX) / 4) : 0u;
            }
            bool fail_f = false;
            // a barrier test takes over 100 cycles to answer, so the next chunk's two are asked for before the
            // end of this one: the copies have landed; the MMAs that read the next chunk's A slot are done.  A
            // phase may complete between two lanes' tests: the warp goes on where all of them have seen it
            bool full_ok = false, done_ok = false;
            for (int c = 0; c < nchunks; ++c) {
                if (!__all_sync(FULL, full_ok) && !wait(&full[st], su & 1)) {
                    fail_f = true;
                    break;
                }
                // the F window
                const uint8_t *F = smem + (size_t)st * G.stage_bytes + 2 * b_bytes;
                // the A buffers of this chunk's pair were read by the MMAs of chunk cg - 2
                if (!__all_sync(FULL, done_ok) && cg >= ASLOTS && !wait(&done[hst[0]], hsu[0] & 1)) {
                    fail_f = true;
                    break;
                }
#pragma unroll
                for (int x = 0; x + 1 < ASLOTS; ++x) {
                    hst[x] = hst[x + 1];
                    hsu[x] = hsu[x + 1];
                }
                hst[ASLOTS - 1] = st;
                hsu[ASLOTS - 1] = su;
                const int nst = st + 1 == G.n_stages ? 0 : st + 1, nsu = st + 1 == G.n_stages ? su + 1 : su;
                const uint32_t Fs = after_wait(smem_u32(F));
#pragma unroll
                for (int t = 0; t < MAX_TILES; ++t) {
                    if (t >= S.ntiles) break;
                    const uint32_t ta =
                        lane_base + (uint32_t)(((cg & (ASLOTS - 1)) * MAX_TILES + t) * A_COLS + (FPX / 2) * h);
                    const uint32_t pj = Fs + rel_j[t], pk = Fs + rel_k[t];
                    // 16 pixels at a time: products, hi / lo split, 8 packed pairs of each to tensor memory
#pragma unroll
                    for (int part = 0; part < FPX / 16; ++part) {
                        uint32_t hi[8], lo[8];
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            const uint32_t w = (uint32_t)(4 * part + cc) << 4;
                            const float4 x = lds128(pj ^ w), y = lds128(pk ^ w);
                            split2(__fmul2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y)), hi[2 * cc],
                                   lo[2 * cc]);
                            split2(__fmul2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w)), hi[2 * cc + 1],
                                   lo[2 * cc + 1]);
                        }
                        tmem_st(ta + 8u * part, hi);
                        tmem_st(ta + 32u + 8u * part, lo);
                    }
                    if (t == S.ntiles - 1 && c + 1 < nchunks) {
                        full_ok = mbar_test(smem_u32(&full[nst]), (uint32_t)(nsu & 1));
                        done_ok = cg + 1 >= ASLOTS && mbar_test(smem_u32(&done[hst[0]]), (uint32_t)(hsu[0] & 1));
                    }
                    // tile t's A buffers are complete: its issuer may start while the next is formed
                    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    mbar_arrive_if(smem_u32(&a_full[(cg & (ASLOTS - 1)) * MAX_TILES + t]), lane == 0);
                }
                // tiles the set does not have: their barriers keep step with the chunks
                if (lane == 0)
                    for (int t = S.ntiles; t < MAX_TILES; ++t)
                        mbar_arrive(smem_u32(&a_full[(cg & (ASLOTS - 1)) * MAX_TILES + t]));
                ++cg;
                st = nst;
                su = nsu;
            }
            if (fail_f) abort_s = 1;
        } else {
            // ---------------- drainers: every group's accumulation region is added into accl and released
            const int q = warp & 3;
            const int h = (warp - DW0) >> 2;          // drain blocks
            const int row = 32 * q + lane;
            const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
            const int nb_h = n_blk[h];
            bool fail_f = false;
            float accl[MAXSLOT];                      // this thread's long accumulators (FP32, rounded to nearest)
#pragma unroll
            for (int x = 0; x < MAXSLOT; ++x) accl[x] = 0.f;
            for (int c = 0; c < nchunks; c += DRAIN) {
                if (!wait(&d_full[grp & 1], (grp >> 1) & 1)) {
                    fail_f = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t base = lane_base + (uint32_t)(NABUF * A_COLS + (grp & 1) * region_cols);
#pragma unroll
                for (int b = 0; b < MAXBLK; ++b) {   // one block at a time: the accumulators fill the registers
                    if (b >= nb_h) break;
                    uint32_t v[8];
                    tmem_ld8(base + (uint32_t)blk_col[h][b], v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                    for (int x = 0; x < 8; ++x) accl[8 * b + x] += __uint_as_float(v[x]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&d_empty[grp & 1]));
                ++grp;
            }
            if (fail_f) {
                abort_s = 1;
            } else {
                // the long accumulators into the item's range of partials
                float *out = partial + (size_t)(e / G.n_sets) * G.dense + row;
#pragma unroll
                for (int b = 0; b < MAXBLK; ++b)
                    if (b < nb_h) {
                        float *o = out + blk_out[h][b];
#pragma unroll
                        for (int x = 0; x < 8; ++x) o[x * TM] = accl[8 * b + x];
                    }
            }
        }
    }
    // every role is done (or gave up): copies and MMAs in flight land before the memory goes
    __syncthreads();
    if (abort_s) {
        if (warp == 0 && lane == 0) {
            // the loader's last fills of each stage
            for (int s = 0; s < G.n_stages && s < issued; ++s) {
                const int uses = (issued - s + G.n_stages - 1) / G.n_stages;
                if (!mbar_drain(smem_u32(&full[s]), (uint32_t)((uses - 1) & 1))) break;
            }
        }
        if (warp >= 1 && warp <= NISS) {
            // every MMA the issuers issued is done once a fresh commit of each arrives
            mma_commit(smem_u32(&fin));
            mbar_drain(smem_u32(&fin), 0u);
        }
        if (threadIdx.x == 0) atomicCAS(err, 0, DERR_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
}

// The fields [nb][P] FP32 as the three chunk-blocked planes of TcPlanes: BF16 hi, BF16 lo
// and FP32, nbp rings a block (zeros past nb and past P).  One thread per 4 pixels of a ring.
__global__ void __launch_bounds__(256) k_split_fields(int nb, int nbp, int64_t P, int64_t P_pad,
                                                      const float *__restrict__ f, __nv_bfloat16 *__restrict__ hi,
                                                      __nv_bfloat16 *__restrict__ lo, float *__restrict__ f32) {
    const int64_t per = P_pad / 4;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= per * nbp) return;
    const int m = (int)(g / per);
    const int64_t p = (g - (int64_t)m * per) * 4;
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = (m < nb && p + e < P) ? f[(size_t)m * P + p + e] : 0.f;
    uint32_t h[2], l[2];
    split2(make_float2(v[0], v[1]), h[0], l[0]);
    split2(make_float2(v[2], v[3]), h[1], l[1]);
    const int x = (int)(p % KC), key = m & 7;
    const size_t row = ((size_t)(p / KC) * nbp + m) * KC;
    const size_t ob = row + (size_t)((((x >> 3) ^ key) << 3) | (x & 7));   // 8 BF16 per 16-byte unit
    const size_t of = row + (size_t)(((x >> 2) ^ key) << 2);                // 4 FP32 per 16-byte unit
    *(uint2 *)(hi + ob) = make_uint2(h[0], h[1]);
    *(uint2 *)(lo + ob) = make_uint2(l[0], l[1]);
    *(float4 *)(f32 + of) = make_float4(v[0], v[1], v[2], v[3]);
}

// The padding of planes the transform wrote directly: rings nb .. nbp-1 of every
// chunk block, and the pixels past P of the last block's rings (zeros).
__global__ void __launch_bounds__(256) k_split_pad(int nb, int nbp, int64_t P, int64_t P_pad,
                                                   __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo,
                                                   float *__restrict__ f32) {
    const int64_t nblk = P_pad / KC;
    const int64_t rows_pad = nblk * (nbp - nb) * KC;   // whole padding rings
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < rows_pad) {
        const int64_t blk = g / ((int64_t)(nbp - nb) * KC), rem = g - blk * (nbp - nb) * KC;
        const size_t o = (size_t)(blk * nbp + nb) * KC + rem;
        hi[o] = __float2bfloat16_rn(0.f);
        lo[o] = __float2bfloat16_rn(0.f);
        f32[o] = 0.f;
        return;
    }
    const int64_t t = g - rows_pad;
    if (t >= (int64_t)nb * KC) return;
    const int m = (int)(t / KC), u = (int)(t - (int64_t)m * KC), key = m & 7;
    if ((nblk - 1) * KC + u < P) return;
    const size_t row = ((size_t)(nblk - 1) * nbp + m) * KC;
    hi[row + ((((u >> 3) ^ key) << 3) | (u & 7))] = __float2bfloat16_rn(0.f);
    lo[row + ((((u >> 3) ^ key) << 3) | (u & 7))] = __float2bfloat16_rn(0.f);
    f32[row + ((((u >> 2) ^ key) << 2) | (u & 3))] = 0.f;
}

// dense[x] = sum over pixel ranges of partial[r][x] in double-float (TwoSum, then Fast2Sum; about
// 2^-44 relative, in FP32 arithmetic: GB300's FP64 pipe, which also converts, is narrow), widened to
// FP64 once: blockDim.y threads an entry take every blockDim.y-th range, eight loads in flight each,
// and their sums are added in a fixed order.  Bound by memory with many entries, by the latency of a
// thread's loads with few (a small grid's list has some 1e4 entries and 300 ranges: 29 us with one
// thread an entry), hence the threads an entry gets (see tc_run).
constexpr int RED_X = 64;
struct DfSum {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float v, float vl = 0.f) {
        const float t = __fadd_rn(h, v);
        const float bp = __fsub_rn(t, h);
        const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(v, bp));
        const float lo = __fadd_rn(__fadd_rn(l, vl), e);
        h = __fadd_rn(t, lo);
        l = __fsub_rn(lo, __fsub_rn(h, t));
    }
};
__global__ void __launch_bounds__(1024) k_tc_reduce(int64_t dense, int n_ranges, const float *__restrict__ partial,
                                                    double *__restrict__ out) {
    __shared__ float2 part[1024];
    const int64_t x = (int64_t)blockIdx.x * RED_X + threadIdx.x;
    const int step = blockDim.y;
    DfSum s;
    if (x < dense) {
        int r = threadIdx.y;
        for (; r + 7 * step < n_ranges; r += 8 * step) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldcs(&partial[(size_t)(r + u * step) * dense + x]);
#pragma unroll
            for (int u = 0; u < 8; ++u) s.add(v[u]);
        }
        for (; r < n_ranges; r += step) s.add(__ldcs(&partial[(size_t)r * dense + x]));
    }
    part[threadIdx.y * RED_X + threadIdx.x] = make_float2(s.h, s.l);
    __syncthreads();
    if (threadIdx.y || x >= dense) return;
    for (int y = 1; y < step; ++y) {
        const float2 p = part[y * RED_X + threadIdx.x];
        s.add(p.x, p.y);
    }
    out[x] = (double)s.h + (double)s.l;
}

// S[t] = inv_p dense[pos[t]].
__global__ void __launch_bounds__(256) k_tc_gather(int n_trip, double inv_p, const int64_t *__restrict__ pos,
                                                   const double *__restrict__ dense, double *__restrict__ S) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_trip) S[t] = dense[pos[t]] * inv_p;
}

}  // namespace

// The tiling of a triplet list (see the file comment): rows (j, k) in (j, k)
// order, tiles of 128 rows ordered inside by (k, j), sets of consecutive tiles
// whose accumulator columns fit col_budget, each triplet's place in the dense
// accumulator.  A block of 128 rows whose rings i span more than MAX_TILE_N
// columns becomes several tiles with the same rows.  False for a list the
// kernel cannot take (ring out of range, i > j or j > k).
struct TcPlanHost {
    std::vector<TcSet> sets;
    std::vector<TcTile> tiles;
    std::vector<short2> rowjk;
    std::vector<int64_t> pos;
    int64_t dense = 0;
    int max_stage = 0;       // bytes of the largest set's stage
    int plane_rows = 0;      // rings a block of the planes must hold (every set's windows inside it)
    double work = 0;         // sum over tiles of 128 x N (executed MMA columns x rows per pixel)
};

static bool tc_plan(const int32_t *ijk, int n_trip, int nb, int col_budget, int stage_cap, TcPlanHost &pl) {
    std::map<std::pair<int, int>, std::pair<int, int>> rows;   // (j, k) -> (lowest i, highest i)
    for (int t = 0; t < n_trip; ++t) {
        const int i = ijk[3 * t], j = ijk[3 * t + 1], k = ijk[3 * t + 2];
        if (i < 0 || i > j || j > k || k >= nb) return false;
        auto it = rows.find({j, k});
        if (it == rows.end()) rows[{j, k}] = {i, i};
        else {
            it->second.first = std::min(it->second.first, i);
            it->second.second = std::max(it->second.second, i);
        }
    }
    std::vector<std::pair<std::pair<int, int>, std::pair<int, int>>> R(rows.begin(), rows.end());
    const int nblocks = (int)cdiv((int64_t)R.size(), TM);      // blocks of 128 rows
    pl.tiles.clear();
    pl.rowjk.clear();
    std::vector<int> first_tile(nblocks);
    std::map<std::pair<int, int>, int> lane_of;   // (j, k) -> row block * TM + lane
    pl.dense = 0;
    pl.work = 0;
    for (int rb = 0; rb < nblocks; ++rb) {
        const int r0 = rb * TM, r1 = std::min<int>((int)R.size(), r0 + TM);
        int lo = 1 << 30, hi = -1;
        std::vector<std::pair<int, int>> kj;
        for (int r = r0; r < r1; ++r) {
            lo = std::min(lo, R[r].second.first);
            hi = std::max(hi, R[r].second.second);
            kj.push_back({R[r].first.second, R[r].first.first});
        }
        std::sort(kj.begin(), kj.end());
        std::vector<short2> lanes(TM, make_short2(-1, -1));
        for (int x = 0; x < (int)kj.size(); ++x) {
            lanes[x] = make_short2((short)kj[x].second, (short)kj[x].first);
            lane_of[{kj[x].second, kj[x].first}] = rb * TM + x;
        }
        // the block's ring columns, cut into tiles of at most MAX_TILE_N (same rows); a tile that
        // would reach past the last ring (rounded up to 8) moves down to end there, so that no
        // plane needs rings past it (a few columns more at its low end instead)
        const int ilo = lo & ~7;
        const int n_all = (int)cdiv(hi - ilo + 1, 16) * 16;
        const int ring_cap = (int)cdiv(nb, B_ROWS) * B_ROWS;
        first_tile[rb] = (int)pl.tiles.size();
        for (int c0 = 0; c0 < n_all; c0 += MAX_TILE_N) {
            TcTile T;
            T.i_lo = ilo + c0;
            T.n = std::min(MAX_TILE_N, n_all - c0);
            if (T.i_lo + T.n > ring_cap) T.i_lo = std::max(0, (ring_cap - T.n) & ~(B_ROWS - 1));
            if (T.n > col_budget) return false;
            T.acc_off = pl.dense;
            pl.dense += (int64_t)TM * T.n;
            pl.work += (double)TM * T.n;
            pl.tiles.push_back(T);
            pl.rowjk.insert(pl.rowjk.end(), lanes.begin(), lanes.end());
        }
    }
    const int ntiles = (int)pl.tiles.size();
    // sets: greedy runs of tiles within the column budget, the stage cap and MAX_TILES
    pl.sets.clear();
    pl.max_stage = 0;
    pl.plane_rows = nb;
    for (int t = 0; t < ntiles;) {
        TcSet S{};
        S.tile0 = t;
        int cols = 0, blo = 1 << 30, bhi = -1, flo = 1 << 30, fhi = -1;
        while (t < ntiles && S.ntiles < MAX_TILES) {
            const TcTile &T = pl.tiles[t];
            int jmin = 1 << 30, kmax = -1;
            for (int x = 0; x < TM; ++x) {
                const short2 v = pl.rowjk[(size_t)t * TM + x];
                if (v.x < 0) continue;
                jmin = std::min(jmin, (int)v.x);
                kmax = std::max(kmax, (int)v.y);
            }
            const int nblo = std::min(blo, T.i_lo), nbhi = std::max(bhi, T.i_lo + T.n);
            const int nflo = std::min(flo, jmin), nfhi = std::max(fhi, kmax + 1);
            const int bn = (int)cdiv(nbhi - nblo, B_ROWS) * B_ROWS, fn = nfhi - nflo;
            const int stage = (int)cdiv(2 * bn * 128 + fn * 256, 1024) * 1024;   // stages stay 1024-aligned
            if (S.ntiles > 0 && (cols + T.n > col_budget || stage > stage_cap)) break;
            cols += T.n;
            blo = nblo, bhi = nbhi, flo = nflo, fhi = nfhi;
            S.b_lo = blo, S.b_n = bn, S.f_lo = flo, S.f_n = fn;
            ++S.ntiles;
            ++t;
        }
        pl.max_stage = std::max(pl.max_stage, (int)cdiv(2 * S.b_n * 128 + S.f_n * 256, 1024) * 1024);
        pl.plane_rows = std::max(pl.plane_rows, std::max(S.b_lo + S.b_n, S.f_lo + S.f_n));
        pl.sets.push_back(S);
    }
    pl.pos.resize(n_trip);
    for (int t = 0; t < n_trip; ++t) {
        const int i = ijk[3 * t], j = ijk[3 * t + 1], k = ijk[3 * t + 2];
        const int l = lane_of[{j, k}];
        const int tl = first_tile[l / TM] + (i - pl.tiles[first_tile[l / TM]].i_lo) / MAX_TILE_N;
        const TcTile &T = pl.tiles[tl];
        pl.pos[t] = T.acc_off + (int64_t)(i - T.i_lo) * TM + (l % TM);
    }
    return true;
}

// A plan on the device: the host plan and device copies of its tables.  The
// canonical list's plans (one per column budget) are kept in the setup; a
// caller's list is read back and planned into context workspaces on each call.
struct TcPlanDev {
    TcPlanHost h;
    TcSet *d_sets = nullptr;
    TcTile *d_tiles = nullptr;
    short2 *d_rowjk = nullptr;
    int64_t *d_pos = nullptr;
    bool owned = false;
    ~TcPlanDev() {
        if (owned) {
            cudaFree(d_sets);
            cudaFree(d_tiles);
            cudaFree(d_rowjk);
            cudaFree(d_pos);
        }
    }
};
struct TcPlans {
    std::map<int, std::unique_ptr<TcPlanDev>> by_budget;
};

template <class T>
static bool upload_to(T *&dst, const std::vector<T> &v) {
    if (cudaMalloc((void **)&dst, sizeof(T) * std::max<size_t>(v.size(), 1)) != cudaSuccess) {
        cudaGetLastError();
        dst = nullptr;
        return false;
    }
    if (!v.empty() && cudaMemcpy(dst, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

// The split-BF16 launch shape: the accumulator-column budget of a set (how many
// tiles share each chunk) and the work items per CTA (which sets the pixel
// range of an item, at most MAX_RANGE_PIXELS so that one FP32 tensor-memory
// accumulation covers a bounded number of terms).
#ifndef ABS_TC_MAX_RANGE
#define ABS_TC_MAX_RANGE 16384
#endif
constexpr int64_t MAX_RANGE_PIXELS = ABS_TC_MAX_RANGE;
constexpr int BUDGETS[] = {MAX_SET_COLS, MAX_SET_COLS * 3 / 4 / 16 * 16};

struct TcShapeSel {
    int budget = MAX_SET_COLS;
    int waves = 2;
};

// Pixel range per work item for a plan, SM count and waves: items = sets x ranges
// close to waves x SMs, each range a multiple of the chunk and at most MAX_RANGE_PIXELS.
static int64_t tc_range(const TcPlanHost &pl, int64_t P_pad, int sms, int waves) {
    const int64_t nsets = (int64_t)pl.sets.size();
    int64_t ranges = std::max<int64_t>(1, cdiv((int64_t)sms * 4 * waves, nsets));
    int64_t per = cdiv(cdiv(P_pad, ranges), KC) * KC;
    const int64_t cap = std::min<int64_t>(MAX_RANGE_PIXELS, (int64_t)4096 << (waves - 1));
    if (per > cap) per = cap;
    return std::max<int64_t>(per, KC);
}

}  // namespace absk

namespace absk {

// dynamic shared memory for the stages (with 1 KB of alignment slack and the kernel's
// 9 KB of static shared memory, below the 227 KB a CTA may have)
static const int SMEM_BUDGET = 200 * 1024;

// Plan of cfg's canonical list for a column budget (made and uploaded on first use).
static const TcPlanDev *canonical_plan(const Setup &s, int budget) {
    Setup &ms = const_cast<Setup &>(s);
    if (!ms.tc_plan) ms.tc_plan = std::make_shared<TcPlans>();
    TcPlans &pls = *static_cast<TcPlans *>(ms.tc_plan.get());
    auto it = pls.by_budget.find(budget);
    if (it != pls.by_budget.end()) return it->second.get();
    auto pd = std::make_unique<TcPlanDev>();
    if (!tc_plan(s.ijk.data(), (int)(s.ijk.size() / 3), s.nb, budget, SMEM_BUDGET / std::max(2, ASLOTS), pd->h))
        return nullptr;
    pd->owned = true;
    if (!upload_to(pd->d_sets, pd->h.sets) || !upload_to(pd->d_tiles, pd->h.tiles) ||
        !upload_to(pd->d_rowjk, pd->h.rowjk) || !upload_to(pd->d_pos, pd->h.pos))
        return nullptr;
    const TcPlanDev *r = pd.get();
    pls.by_budget[budget] = std::move(pd);
    return r;
}

// One launch of the kernel and its reduction for a plan and shape; events around the kernel when given.
static abs_status tc_run(abs_ctx *ctx, const Setup &s, const TcPlanDev &pd, const TcShapeSel &sh,
                         const TcPlanes &planes, int64_t P_pad, int32_t n_trip, double *d_sum, cudaEvent_t e0,
                         cudaEvent_t e1) {
    const TcPlanHost &pl = pd.h;
    TcParams G;
    G.n_sets = (int)pl.sets.size();
    G.P_pad = P_pad;
    G.per_item = tc_range(pl, P_pad, ctx->sm_count, sh.waves);
    const int64_t ranges = cdiv(P_pad, G.per_item);
    G.n_items = (int)(ranges * G.n_sets);
    G.dense = pl.dense;
    G.stage_bytes = pl.max_stage;
    G.n_stages = std::min(MAX_STAGES, SMEM_BUDGET / std::max(G.stage_bytes, 1));
    // the formers' wait on the MMAs of chunk c - ASLOTS is unambiguous only while a stage serves
    // at most one chunk in that span: at least ASLOTS stages
    if (G.n_stages < std::max(2, ASLOTS))
        return fail(ctx, ABS_ERR_UNSUPPORTED, "split-BF16 stages do not fit shared memory");
    float *partial = (float *)workspace(ctx, "tc.partial", sizeof(float) * (size_t)(ranges * G.dense));
    double *dsum = (double *)workspace(ctx, "tc.dense", sizeof(double) * (size_t)G.dense);
    int *next = (int *)workspace(ctx, "tc.next", sizeof(int));
    if (!partial || !dsum || !next) return fail(ctx, ABS_ERR_OOM, "split-BF16 workspace");
    const size_t smem = 1024 + (size_t)G.n_stages * G.stage_bytes;
    if (!allow_smem(k_triple_tc, smem)) return fail(ctx, ABS_ERR_UNSUPPORTED, "split-BF16: shared memory attribute refused");
    {
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, k_triple_tc) == cudaSuccess && fa.maxThreadsPerBlock < NT)
            return fail(ctx, ABS_ERR_UNSUPPORTED,
                        "split-BF16: kernel needs " + std::to_string(fa.numRegs) + " registers a thread, " +
                            std::to_string(fa.maxThreadsPerBlock) + " threads fit a CTA");
        cudaGetLastError();
    }
    cudaStream_t st = ctx->stream;
    const int grid = std::min(G.n_items, ctx->sm_count);
    {
        StageTimer timer(ctx, e0 ? nullptr : "triple_tc");
        if (e0) cudaEventRecord(e0, st);
        cudaMemsetAsync(next, 0, sizeof(int), st);
        k_triple_tc<<<grid, NT, smem, st>>>(G, planes, pd.d_sets, pd.d_tiles, pd.d_rowjk, partial, next,
                                             ctx->d_err);
    }
    {
        StageTimer timer(ctx, e0 ? nullptr : "tc_reduce");
        // threads an entry: one while the entries alone fill the GPU, up to 16 below
        int per = 1;
        while (per < 16 && G.dense * per < (int64_t)ctx->sm_count * 2048 && per * 8 < ranges) per *= 2;
        k_tc_reduce<<<(int)cdiv(G.dense, RED_X), dim3(RED_X, per), 0, st>>>(G.dense, (int)ranges, partial, dsum);
        k_tc_gather<<<(int)cdiv(n_trip, 256), 256, 0, st>>>(n_trip, 1.0 / (double)s.P, pd.d_pos,
                                                             dsum, d_sum);
    }
    if (e1) cudaEventRecord(e1, st);   // the autotuner times the kernel with its reduction
    return check_launch(ctx, "split-BF16 triple sums");
}

// Planes of nbp rings, in the context's workspace.
struct PlaneBufs {
    __nv_bfloat16 *hi, *lo;
    float *f32;
};
static bool tc_plane_buffers(abs_ctx *ctx, int nbp, int64_t P_pad, PlaneBufs &pl) {
    const size_t plane = (size_t)nbp * P_pad;
    pl.hi = (__nv_bfloat16 *)workspace(ctx, "tc.hi", sizeof(__nv_bfloat16) * plane);
    pl.lo = (__nv_bfloat16 *)workspace(ctx, "tc.lo", sizeof(__nv_bfloat16) * plane);
    pl.f32 = (float *)workspace(ctx, "tc.f32", sizeof(float) * plane);
    return pl.hi && pl.lo && pl.f32;
}

// Rings a plane block must hold for the canonical plans: every window of every budget's tiling.
static int canonical_nbp(const Setup &s) {
    int nbp = 0;
    for (int b : BUDGETS)
        if (const TcPlanDev *pd = canonical_plan(s, b)) nbp = std::max({nbp, s.nb, pd->h.plane_rows});
    return nbp > 0 ? (int)cdiv(nbp, 8) * 8 : 0;
}

abs_status tc_split_target(abs_ctx *ctx, const Setup &s, SplitOut &out) {
    const int nbp = canonical_nbp(s);
    if (nbp == 0) return fail(ctx, ABS_ERR_UNSUPPORTED, "split-BF16: no tiling fits the tensor memory");
    const int64_t P_pad = cdiv(s.P, KC) * KC;
    PlaneBufs pl;
    if (!tc_plane_buffers(ctx, nbp, P_pad, pl)) return fail(ctx, ABS_ERR_OOM, "split-BF16 planes");
    out = SplitOut{pl.hi, pl.lo, pl.f32, nbp, P_pad};
    return ABS_OK;
}

abs_status launch_triple_tc(abs_ctx *ctx, const Setup &s, const float *d_fields, int32_t n_trip,
                            const int32_t *d_ijk, double *d_sum) {
    if (n_trip == 0) return ABS_OK;
    const int64_t P = s.P;
    const int64_t P_pad = cdiv(P, KC) * KC;
    const bool canonical = d_ijk == s.d_ijk;
    if (!d_fields && !canonical) return fail(ctx, ABS_ERR_INVALID_ARG, "split-BF16: planes without fields need the canonical list");
    abs_ctx *root = ctx->parent ? ctx->parent : ctx;
    // the plans: the canonical list's, one per column budget (kept by the setup), or the caller's
    // list read back and planned (one synchronisation)
    TcPlanDev caller;
    std::vector<std::pair<int, const TcPlanDev *>> plans;
    if (canonical) {
        for (int b : BUDGETS)
            if (const TcPlanDev *pd = canonical_plan(s, b)) plans.push_back({b, pd});
        if (plans.empty()) return fail(ctx, ABS_ERR_UNSUPPORTED, "split-BF16: no tiling fits the tensor memory");
    } else {
        std::vector<int32_t> h((size_t)3 * n_trip);
        if (cudaMemcpyAsync(h.data(), d_ijk, sizeof(int32_t) * h.size(), cudaMemcpyDeviceToHost, ctx->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
            cudaGetLastError();
            return fail(ctx, ABS_ERR_CUDA, "split-BF16: reading the triplet list back");
        }
        if (!tc_plan(h.data(), n_trip, s.nb, BUDGETS[0], SMEM_BUDGET / std::max(2, ASLOTS), caller.h))
            return fail(ctx, ABS_ERR_INVALID_ARG, "split-BF16: triplet list outside i <= j <= k < n_bins");
        caller.d_sets = (TcSet *)workspace(ctx, "tc.sets", sizeof(TcSet) * caller.h.sets.size());
        caller.d_tiles = (TcTile *)workspace(ctx, "tc.tiles", sizeof(TcTile) * caller.h.tiles.size());
        caller.d_rowjk = (short2 *)workspace(ctx, "tc.rowjk", sizeof(short2) * caller.h.rowjk.size());
        caller.d_pos = (int64_t *)workspace(ctx, "tc.pos", sizeof(int64_t) * caller.h.pos.size());
        if (!caller.d_sets || !caller.d_tiles || !caller.d_rowjk || !caller.d_pos)
            return fail(ctx, ABS_ERR_OOM, "split-BF16 plan");
        cudaMemcpy(caller.d_sets, caller.h.sets.data(), sizeof(TcSet) * caller.h.sets.size(), cudaMemcpyHostToDevice);
        cudaMemcpy(caller.d_tiles, caller.h.tiles.data(), sizeof(TcTile) * caller.h.tiles.size(),
                   cudaMemcpyHostToDevice);
        cudaMemcpy(caller.d_rowjk, caller.h.rowjk.data(), sizeof(short2) * caller.h.rowjk.size(),
                   cudaMemcpyHostToDevice);
        cudaMemcpy(caller.d_pos, caller.h.pos.data(), sizeof(int64_t) * caller.h.pos.size(), cudaMemcpyHostToDevice);
        plans.push_back({BUDGETS[0], &caller});
    }
    // the three planes, with room for every plan's windows (the canonical ones: as
    // tc_split_target sized them)
    int nbp = canonical ? canonical_nbp(s) : (int)cdiv(std::max(s.nb, caller.h.plane_rows), 8) * 8;
    PlaneBufs pb;
    if (!tc_plane_buffers(ctx, nbp, P_pad, pb)) return fail(ctx, ABS_ERR_OOM, "split-BF16 planes");
    const size_t plane = (size_t)nbp * P_pad;
    if (d_fields) {
        StageTimer timer(ctx, "tc_split");
        k_split_fields<<<(int)cdiv((int64_t)plane / 4, 256), 256, 0, ctx->stream>>>(
            s.nb, nbp, P, P_pad, d_fields, pb.hi, pb.lo, pb.f32);
    } else if (nbp > s.nb || P < P_pad) {
        StageTimer timer(ctx, "tc_pad");
        const int64_t n = (P_pad / KC) * (nbp - s.nb) * KC + (int64_t)s.nb * KC;
        k_split_pad<<<(int)cdiv(n, 256), 256, 0, ctx->stream>>>(s.nb, nbp, P, P_pad, pb.hi, pb.lo, pb.f32);
    }
    {
        const abs_status sl = check_launch(ctx, "split-BF16 planes");
        if (sl != ABS_OK) return sl;
    }
    const TcPlanes planes{pb.hi, pb.lo, pb.f32, nbp};
    if (!canonical) return tc_run(ctx, s, caller, TcShapeSel{}, planes, P_pad, n_trip, d_sum, nullptr, nullptr);
    // the canonical list: the shape measured on this configuration's first eager call
    // (every budget x item length timed twice, kernel and reduction, the faster kept),
    // else the first budget that plans with the middle item length
    auto it = root->tc_shapes.find(s.key);
    TcShapeSel pick;
    pick.budget = plans[0].first;
    if (it != root->tc_shapes.end() && it->second.budget > 0) {
        pick.budget = it->second.budget;
        pick.waves = it->second.waves;
    } else {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(ctx->stream, &cs);
        const bool tune = root->autotune && !ctx->profiling && cs == cudaStreamCaptureStatusNone &&
                          ctx->stream != nullptr;
        if (tune) {
            cudaEvent_t e0 = nullptr, e1 = nullptr;
            if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
                cudaGetLastError();
                if (e0) cudaEventDestroy(e0);
                return fail(ctx, ABS_ERR_CUDA, "autotuner events");
            }
            float best = 1e30f;
            for (const auto &pp : plans)
                for (int w = 1; w <= 3; ++w) {
                    const TcShapeSel c{pp.first, w};
                    float ms_min = 1e30f;
                    for (int rep = 0; rep < 2; ++rep) {
                        const abs_status rs = tc_run(ctx, s, *pp.second, c, planes, P_pad, n_trip, d_sum, e0, e1);
                        if (rs != ABS_OK) {
                            cudaEventDestroy(e0);
                            cudaEventDestroy(e1);
                            return rs;
                        }
                        float t = 0.f;
                        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
                            cudaGetLastError();
                            t = 1e30f;
                        }
                        ms_min = std::min(ms_min, t);
                    }
                    if (ms_min < best) {
                        best = ms_min;
                        pick = c;
                    }
                }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
        }
        if (tune || !root->autotune) {
            abs_ctx::TcShape &c = root->tc_shapes[s.key];
            c.budget = pick.budget;
            c.waves = pick.waves;
            c.measured = tune;
        }
    }
    const TcPlanDev *pd = canonical_plan(s, pick.budget);
    if (!pd) return fail(ctx, ABS_ERR_OOM, "split-BF16 plan");
    return tc_run(ctx, s, *pd, pick, planes, P_pad, n_trip, d_sum, nullptr, nullptr);
}

}  // namespace absk
