// Split-precision exchange on the 5th-generation tensor cores (tcgen05 + TMEM + TMA).
//
// Same arithmetic as split_k.cu (Ozaki slices, exact FP32 chunks, float-float drains), with the products issued
// as tcgen05.mma kind::f16 (BF16 x BF16 -> FP32 in tensor memory):
//   * a CTA works on output tiles of 128 rows x N columns; every Ozaki level L = s + t (0-based) has its own FP32
//     accumulator of N columns in TMEM (S levels, S * N <= 512 columns);
//   * a producer warp streams K-steps of 64 elements with TMA (3-D tensor maps, 128-byte swizzle): the S B slices
//     of a K-step (N x 64 each) once into one of two resident buffers, and the S A slices (128 x 64) through a
//     ring of slots; every buffer is guarded by mbarriers;
//   * an issuing warp: for A slice s, the B slices t < S - s in wide MMAs (4 k16 steps each), then the A slot
//     goes back to the producer, and the B buffer after the K-step's last A slice; a chunk begins once the
//     epilogue has taken the sums of the one before;
//   * four epilogue warps (one per 32 TMEM lanes) read the level sums with tcgen05.ld, scale them by the
//     exact power of two 2^{e_row + e_col - 7 (L + 2)} and add them into per-thread float-float rows, two
//     elements per instruction (f32x2).
// Every mbarrier wait is bounded by a clock budget; on expiry the kernel records DF_E_TIMEOUT in a flag,
// waits (with the full budget) for the copies and MMAs it has already issued, releases its tensor memory and
// returns.
//
// A third mode runs the metric whitening B = L^-1 A (paper eq. 1, third form) the same way with 7 slices:
// A operand = slices of L^-1 rows (one exponent per auxiliary row), B operand = slices of the
// transposed three-index columns (one exponent per pair column), K over the auxiliary index up to the
// end of the lower triangle, exact 448-element chunks (7 slices: a level sum is below 9 * 2^12 per
// term, 448 terms stay below 2^24), output in FP64.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "ozaki.cuh"

namespace dfhf {

namespace {

typedef __nv_bfloat16 bf16;

constexpr int TM = 128;            // output rows per CTA (TMEM lanes)
constexpr int KS = 64;             // K elements per pipeline step (one 128-byte swizzle row)
// pipeline steps per exact chunk: 12 (S = 3), 9 (S = 5), 7 (whitening, S = 7)
template <int S>
constexpr int chunk_steps() {
    return exact_chunk<S>() / KS;
}
// A-slice ring slots (one 128 x 64 slice each): 4, or 3 where that lets two CTAs share an SM
template <int S, int N>
constexpr int ring_slots() {
    return (S >= 7 && N <= 32) || (S == 5 && N == 48) || (S == 3 && N == 64) ? 3 : 4;
}
template <int S, int N>
constexpr int tc_smem_bytes() {
    return ring_slots<S, N>() * TM * KS * 2 + 2 * S * N * KS * 2 + 1024 + 256;
}
// two CTAs share an SM where the accumulators take at most half of its tensor memory and the rings fit twice into
// 228 KB; the kernel's registers are bounded for two there, and only there (3 slices, 80 wide: 372 bytes of spills
// for a second CTA that has no room; Y at n = 800, naux = 2192, 80 occupied 1.86 -> 1.81 ms without)
template <int S, int N>
constexpr int ctas_per_sm() {
    return S * N <= 256 && 2 * (tc_smem_bytes<S, N>() + 1024) <= 228 * 1024 ? 2 : 1;
}
constexpr long long WAIT_CYCLES = 4000000000LL;   // ~2 s at 2 GHz

// ------------------------------------------------------------------------------------------------
// PTX helpers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded pipeline wait: false (and the error flag set) if the barrier did not complete within `budget`
// cycles (WAIT_CYCLES unless the host shortened it). The waits that drain copies and MMAs already issued,
// before the CTA leaves, always keep the full WAIT_CYCLES.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int* err, long long budget) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > budget || *(volatile int*)err) {
            atomicExch(err, DF_E_TIMEOUT);
            return false;
        }
    }
    return true;
}

// the same by a whole warp, with one result for all of its lanes (the code after it stays uniform, so that the
// MMA's operands live in uniform registers)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, unsigned parity, int* err, long long budget) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, err, budget));
}
__device__ __forceinline__ bool elect_one() {
    unsigned p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
        ::"r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// MN-major operand (the M index contiguous in shared memory, 128-byte swizzle): the tile is two 8 KB halves
// of 64 M-values each (one per TMA box), each half 8 K-rows of 128 bytes per 1024-byte atom. One stride
// field steps between the halves (along M), the other between 8-row atoms (along K).
constexpr unsigned MN_LBO = 8192;   // bytes between the two 64-wide M halves
constexpr unsigned MN_SBO = 1024;   // bytes between 8-row atoms along K
__device__ __forceinline__ uint64_t smem_desc_mn(const void* tile) {
    const unsigned a = smem_u32(tile);
    uint64_t d = (uint64_t)((a & 0x3FFFF) >> 4);
    d |= (uint64_t)(MN_LBO >> 4) << 16;
    d |= (uint64_t)(MN_SBO >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row atoms 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc(const void* tile) {
    const unsigned a = smem_u32(tile);
    uint64_t d = (uint64_t)((a & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;                  // leading byte offset (unused with 128-byte swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset: next 8-row atom
    d |= (uint64_t)1 << 46;                  // descriptor version for tcgen05
    d |= (uint64_t)2 << 61;                  // swizzle: 128 bytes
    return d;
}

// instruction descriptor: kind::f16, A and B BF16 (K-major), D FP32, M x N
__host__ __device__ constexpr unsigned instr_desc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(unsigned tmem_d, uint64_t a, uint64_t b, unsigned idesc, unsigned accum) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// 16 accumulator columns of this warp's 32 lanes: the load is issued here, the registers hold it after tmem_wait
__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// waits for the loads issued so far; the registers pass through so that no use moves above the wait
__device__ __forceinline__ void tmem_wait(unsigned (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// pairs of floats (two per 64-bit register): every operation rounds each half as the scalar one does
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(unsigned a, unsigned b) { return (f2)a | ((f2)b << 32); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float lo_of(f2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float hi_of(f2 a) { return __uint_as_float((unsigned)(a >> 32)); }

__device__ __forceinline__ float pow2f(int e) { return e < -126 ? 0.f : __int_as_float((127 + min(e, 127)) << 23); }


// (hi, lo) += v sc by Knuth's TwoSum, sc a power of two (the product v sc is exact, so it folds into the
// multiply-adds): s = hi + v sc, b = s - hi, lo += (hi - (s - b)) + (v sc - b), hi = s
__device__ __forceinline__ void two_sum_acc(f2& hi, f2& lo, f2 v, f2 sc) {
    const f2 m1 = 0xBF800000BF800000ull;   // (-1, -1)
    const f2 s = fma2(v, sc, hi);
    const f2 nb = fma2(s, m1, hi);         // hi - s = -b
    const f2 u = fma2(add2(s, nb), m1, hi);
    lo = add2(lo, add2(u, fma2(v, sc, nb)));
    hi = s;
}

// ------------------------------------------------------------------------------------------------
// Work description. The kernel is persistent: a CTA takes the tiles blockIdx.x, blockIdx.x + gridDim.x, ... and
// its rings run on across them, so that the next tile's loads and products overlap the last drain and the
// output of the one before (a CTA per tile spent the time of about 8 K-steps on its start and end: at n = 832,
// 13 K-steps a tile, two fifths of the kernel).
// MODE 0 (Y = B C): tile = (128 of the rows P np + mu, column tile), column tile fastest; K runs over nu (np),
// exponents constant (row: Be[P np + mu], column: Ce[i]). MODE 3 (Y = B C from the packed slices): tile = (P,
// mu-tile, column tile); B_P is stored as its lower 128 x 128 tiles only, Bs[s][P][t][128][128] with
// t = I (I + 1) / 2 + J for I >= J (diagonal tiles whole), one exponent per P (Be[P]); K-step blocks nu of J > I
// come from the stored tile (J, I) read as an MN-major (transposed) operand. In both only the columns below
// `cols` (the occupied orbitals rounded up to 16) are computed: full tiles of N and a narrower last one.
// MODE 1 (K = sum Y Y^T): tile = (split, 128-row tile, column tile up to the row tile's end), the split slowest so that the CTAs
// resident together stream the same range of the contraction through L2; K runs over the contiguous index
// k = P ldy + i of the Y slices, stored tile-major as Ys[s][k / 64][mu][k % 64] (one TMA box is 16 KB of
// contiguous memory; no padding between auxiliary rows), one exact chunk per block of consecutive k with its own
// exponents Ye[block][mu], Ye[block][nu]; the 16-wide blocks with i >= cols are zero and take no product.
// MODE 2 (whitening): tile = (row tile, column tile), the last row tiles (the longest sums) first.
// ------------------------------------------------------------------------------------------------
struct TcArgs {
    int naux, np, ldy, nsplit;
    int rows;                // MODE 0: naux np
    int cols;                // MODE 0, 1, 3: columns of Y that are not identically zero (a multiple of 16)
    long long KL;            // MODE 1: naux * ldy, the length of the contraction
    int nkb;                 // MODE 1: 64-wide blocks of the contraction, ceil(KL / 64)
    int ntiles;              // MODE 1: tiles of one split
    const int* row_e;        // MODE 0: Be [naux][np]; MODE 1: Ye [nchunk][np]
    const int* col_e;        // MODE 0: Ce [ldy]
    float2* out;             // MODE 0: Y [naux][np][ldy]; MODE 1: Kpart [nsplit][npt][npt]
    int npt;                 // MODE 1: padded dimension of Kpart (multiple of 128)
    int* err;
    // MODE 2 (whitening): rows = naux (np is set to naux), ncols pair columns of this chunk, row_e = L^-1 row
    // exponents, col_e = column exponents, output FP64 rows of stride ldo: a column's elements go to its
    // positions pos (its own, its mirror's; negative: none) of the row
    int ncols;
    const int2* pos;
    double* outd;
    long long ldo;
    long long wait_cycles;   // budget of the pipeline waits (WAIT_CYCLES by default)
    int nB;                  // MODE 3: 128-row blocks of the packed tiles (np padded to 128 nB)
    int total;               // tiles of the launch
};

// one tile: first row and column, its width, K-steps; MODE 0 and 3: auxiliary row; MODE 1: split, its first
// chunk and K-step
struct Tile {
    int m0, n0, nw, ksteps, P, split, chunk0, kb0;
};

// MODE 1: column tiles of width N that row tile I takes (the lower triangle of 128-blocks)
__host__ __device__ __forceinline__ int k_col_tiles(int I, int N) { return ((I + 1) * TM + N - 1) / N; }

template <int S, int N, int MODE>
__device__ __forceinline__ Tile decode_tile(const TcArgs& args, int b) {
    Tile t{0, 0, N, 0, 0, 0, 0, 0};
    if (MODE == 0 || MODE == 3) {
        const int nt = (args.cols + N - 1) / N;
        t.n0 = (b % nt) * N;
        t.nw = min(N, args.cols - t.n0);
        b /= nt;
        if (MODE == 0) {
            t.m0 = b * TM;
            t.ksteps = args.np / KS;
        } else {
            t.m0 = (b % args.nB) * TM;
            t.P = b / args.nB;
            t.ksteps = 2 * args.nB;
        }
    } else if (MODE == 2) {
        const int ntn = args.ncols / N, mt = (args.naux + TM - 1) / TM;
        t.m0 = (mt - 1 - b / ntn) * TM;               // row-tile major: the L^-1 tile is shared in L2
        t.n0 = (b % ntn) * N;
        t.ksteps = (min(args.naux, t.m0 + TM) + KS - 1) / KS;   // L^-1 is lower triangular
    } else {
        constexpr int CH = exact_chunk<S>();
        t.split = b / args.ntiles;
        b -= t.split * args.ntiles;
        int I = 0;
        for (int c; b >= (c = k_col_tiles(I, N)); ++I) b -= c;
        t.m0 = I * TM;
        t.n0 = b * N;
        const long long nchk = (args.KL + CH - 1) / CH;
        const long long c0 = nchk * t.split / args.nsplit, c1 = nchk * (t.split + 1) / args.nsplit;
        t.chunk0 = (int)c0;
        const long long k0 = c0 * CH, k1 = min(args.KL, c1 * CH);
        t.kb0 = (int)(k0 / KS);                                  // chunks are K-step aligned
        t.ksteps = (int)((k1 - k0 + KS - 1) / KS);
    }
    return t;
}

// Where two CTAs share an SM, one drains while the other's products run. What bounds it (measured on a stream of MMAs alone): an MMA of width W
// takes max(W / 2, (4096 + 32 W) / 128) clocks, arithmetic or the read of its shared-memory operands at 128 bytes
// a clock, and the TMA writes of the streamed slices (16 KB of A and 128 N bytes of B per slice and K-step) share
// that memory; so wider tiles do better, up to the 48 columns at which two CTAs still fit (5 slices: 94 % of the
// pipe without the writes, against 84 % at 32). The issuing and the loading warp run their loops as whole warps
// with one elected lane per instruction: the operands (descriptors, addresses, coordinates) then sit in uniform
// registers. As one-lane branches each MMA cost about 100 clocks of register moves.
// Measured, 5 slices at n = 1200, naux = 3288, 120 occupied: Y 18.8 -> 12.7 ms (1.47 PFLOP/s), K 10.6 -> 7.6 ms;
// whitening at naux = 1644, 225280 columns: 23.8 -> 12.8 ms. Of that, at np = 1216: uniform issue 919 -> 1077
// TFLOP/s (K 1035 -> 1250), uniform loads 1172 -> 1233, packed drains + 4 %, persistent tiles over flattened rows
// 1233 -> 1346, 48-wide tiles 1442.
template <int S, int N, int MODE>
__global__ void __launch_bounds__(192, ctas_per_sm<S, N>())
    ozaki_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                    const __grid_constant__ CUtensorMap mapB2, const TcArgs args) {
    constexpr int A_BYTES = TM * KS * 2;          // 16 KB
    constexpr int BSET = S * N * KS * 2;          // every B slice of one K-step (a slice: a multiple of 1024 bytes)
    constexpr int NA = ring_slots<S, N>();
    constexpr int CSTEPS = chunk_steps<S>();
    constexpr int NCOLS = S * N <= 32 ? 32 : (S * N <= 64 ? 64 : (S * N <= 128 ? 128 : (S * N <= 256 ? 256 : 512)));
    static_assert(S * N <= 512, "TMEM holds at most 512 accumulator columns");
    constexpr int MMA_SLICES = 256 / N;            // B slices per MMA (M = 128 allows N <= 256)
    static_assert(N % 16 == 0 && N <= 256, "MMA width");

    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* bbuf = smem + NA * A_BYTES;    // two B sets
    uint64_t* a_full = (uint64_t*)(bbuf + 2 * BSET);
    uint64_t* a_empty = a_full + NA;
    uint64_t* b_full = a_empty + NA;
    uint64_t* b_empty = b_full + 2;
    uint64_t* acc_full = b_empty + 2;
    uint64_t* acc_empty = acc_full + 1;
    uint64_t* mma_done = acc_empty + 1;
    unsigned* tmem_slot = (unsigned*)(mma_done + 1);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    int* err = args.err;
    const long long wait = args.wait_cycles;
    const int total = args.total;

    // ---- set-up: barriers (thread 0), tensor memory (warp 0) ------------------------------------
    if (threadIdx.x == 0) {
        for (int i = 0; i < NA; ++i) {
            mbar_init(&a_full[i], 1);
            mbar_init(&a_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, 128);
        mbar_init(mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(NCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = *tmem_slot;

    if (warp == 4) {
        // ---------------------------------- producer ------------------------------------------
        const bool leader = elect_one();
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((unsigned long long)&mapA) : "memory");
        asm volatile("prefetch.tensormap [%0];\n" ::"l"((unsigned long long)&mapB) : "memory");
        int slot = 0, bs = 0;
        unsigned aph = 0, bph = 0;                // ring phases
        int a_issued = 0, b_issued = 0;           // capped counts: which buffers have copies to wait for
        bool ok = true;
        for (int b = blockIdx.x; b < total && ok; b += gridDim.x) {
            const Tile t = decode_tile<S, N, MODE>(args, b);
            const CUtensorMap* mb = t.nw == N ? &mapB : &mapB2;
            const int bslice = t.nw * KS * 2;
            for (int ks = 0; ks < t.ksteps && ok; ++ks) {
                // x: the contraction coordinate of this K-step; MODE 1 reads the tile-major slices
                // [s][k block][row][64] at x = 0 and z = s nkb + the split's K-step
                const int kx = MODE == 1 ? 0 : ks * KS;
                const int kb = t.kb0 + ks;
                if (!(ok = mbar_wait_warp(&b_empty[bs], bph ^ 1, err, wait))) break;
                if (leader) {
                    mbar_expect_tx(&b_full[bs], S * bslice);
#pragma unroll
                    for (int q = 0; q < S; ++q)
                        tma_load_3d(bbuf + bs * BSET + q * bslice, mb, kx, t.n0, MODE == 1 ? q * args.nkb + kb : q,
                                    &b_full[bs]);
                }
                b_issued = min(b_issued + 1, 2);
                bs ^= 1;
                if (bs == 0) bph ^= 1;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    if (!(ok = mbar_wait_warp(&a_empty[slot], aph ^ 1, err, wait))) break;
                    if (leader) {
                        mbar_expect_tx(&a_full[slot], A_BYTES);
                        unsigned char* dst = smem + slot * A_BYTES;
                        if (MODE == 3) {
                            // two 64-row boxes of one stored tile: rows mu of tile (I, J) at columns nu of this
                            // K-step (K-major), or, above the diagonal, rows nu of tile (J, I) (MN-major halves)
                            const int I = t.m0 / TM, J = ks >> 1, half = ks & 1, za = s * args.naux + t.P;
                            const bool low = I >= J;
                            const int y0 = low ? (I * (I + 1) / 2 + J) * TM : (J * (J + 1) / 2 + I) * TM + half * KS;
                            tma_load_3d(dst, &mapA, low ? half * KS : 0, y0, za, &a_full[slot]);
                            tma_load_3d(dst + A_BYTES / 2, &mapA, low ? half * KS : KS, low ? y0 + KS : y0, za, &a_full[slot]);
                        } else {
                            tma_load_3d(dst, &mapA, kx, t.m0, MODE == 1 ? s * args.nkb + kb : s, &a_full[slot]);
                        }
                    }
                    a_issued = min(a_issued + 1, NA);
                    if (++slot == NA) {
                        slot = 0;
                        aph ^= 1;
                    }
                }
            }
        }
        // copies in flight complete before the kernel may leave: wait (bounded) for the last ones of every
        // slot. After a normal run the MMA issuer has consumed them all and these waits return at once;
        // after a timeout (here or in the issuer, which may give up while this warp has finished its
        // loop) they keep the CTA until its copies have landed. The phase of a slot's last copy: aph for the
        // slots filled since the ring last wrapped, the one before for the others.
        for (int i = 0; i < a_issued; ++i) {
            const int q = (slot + NA - 1 - i) % NA;
            const unsigned ph = q < slot ? aph : aph ^ 1;
            const long long t0 = clock64();
            while (!mbar_try_wait(&a_full[q], ph) && clock64() - t0 < WAIT_CYCLES) {
            }
        }
        for (int i = 0; i < b_issued; ++i) {
            const int q = (bs + 1 - i) & 1;
            const unsigned ph = q < bs ? bph : bph ^ 1;
            const long long t0 = clock64();
            while (!mbar_try_wait(&b_full[q], ph) && clock64() - t0 < WAIT_CYCLES) {
            }
        }
    } else if (warp == 5) {
        // ---------------------------------- MMA issuer ----------------------------------------
        const bool leader = elect_one();
        const uint64_t ad0 = smem_desc(smem), bd0 = smem_desc(bbuf), adm0 = smem_desc_mn(smem);
        int slot = 0, bs = 0;
        unsigned aph = 0, bph = 0, cph = 1;       // cph: phase of the accumulators' release (none awaited at first)
        bool ok = true;
        for (int b = blockIdx.x; b < total && ok; b += gridDim.x) {
            const Tile t = decode_tile<S, N, MODE>(args, b);
            const unsigned nw8 = (unsigned)(MODE == 1 || MODE == 2 ? N : t.nw) >> 3;   // tile width / 8
            const unsigned bslice = nw8 * 64;                              // bytes of a B slice / 16
            // MODE 1: position of the K-step's first 16-block in the period of ldy / 16, of which the first
            // cols / 16 hold orbitals (at most one in the period does not)
            const int kper = MODE == 1 ? args.ldy / 16 : 0, klive = MODE == 1 ? args.cols / 16 : 0;
            int kpos = MODE == 1 ? (int)((long long)t.kb0 * (KS / 16) % kper) : 0;
            int left = 0;                                                  // K-steps left in the chunk
            for (int ks = 0; ks < t.ksteps && ok; ++ks) {
                bool fresh = false;
                if (left == 0) {                  // a new chunk: the epilogue has taken the last one's sums
                    if (!(ok = mbar_wait_warp(acc_empty, cph, err, wait))) break;
                    fence_after();
                    cph ^= 1;
                    left = CSTEPS;
                    fresh = true;
                }
                unsigned live = 0xf;              // 16-blocks of this K-step that take products
                if (MODE == 1 && klive != kper) {
                    live = 0;
#pragma unroll
                    for (int k = 0; k < KS / 16; ++k) {
                        live |= (kpos < klive ? 1u : 0u) << k;
                        kpos = kpos + 1 == kper ? 0 : kpos + 1;
                    }
                }
                if (!(ok = mbar_wait_warp(&b_full[bs], bph, err, wait))) break;
                fence_after();
                const uint64_t bdk = bd0 + (uint64_t)(bs * (BSET >> 4));
                const bool mn = MODE == 3 && t.m0 / TM < (ks >> 1);   // A read transposed from the stored tile
                const unsigned amaj = mn ? (1u << 15) : 0u;
                // the products of one K-step: for A slice s the B slices q < S - s are consecutive tiles of nw rows
                // in shared memory and their levels s + q consecutive accumulators of nw columns in TMEM, so up to
                // 256 / N of them form one MMA (one read of the A tile per MMA instead of one per slice). The first
                // products of a chunk (slice 0 meets every level) overwrite.
                auto products = [&](auto all_live) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        if (!(ok = mbar_wait_warp(&a_full[slot], aph, err, wait))) break;
                        fence_after();
                        const uint64_t adk = (mn ? adm0 : ad0) + (uint64_t)(slot * (A_BYTES >> 4));
                        bool over = fresh && s == 0;
#pragma unroll
                        for (int k = 0; k < KS / 16; ++k) {
                            if (!decltype(all_live)::value && !(live >> k & 1)) continue;
                            // K-major: +32 B per k16; MN-major: +2 atoms of 8 K-rows (2048 B) per k16
                            const uint64_t ad = adk + (mn ? (uint64_t)(k * 128) : (uint64_t)(k * 2));
#pragma unroll
                            for (int q = 0; q < S - s; q += MMA_SLICES) {
                                const int cnt = MMA_SLICES < S - s - q ? MMA_SLICES : S - s - q;
                                if (leader)
                                    mma_bf16(tmem + (unsigned)(s + q) * nw8 * 8, ad, bdk + (uint64_t)(q * bslice + k * 2),
                                             instr_desc(TM, 0) | (cnt * nw8) << 17 | amaj, over ? 0u : 1u);
                            }
                            over = false;
                        }
                        if (leader) mma_commit(&a_empty[slot]);
                        if (++slot == NA) {
                            slot = 0;
                            aph ^= 1;
                        }
                    }
                };
                if (MODE != 1 || live == 0xf) products(std::true_type());
                else products(std::false_type());
                if (!ok) break;
                if (leader) mma_commit(&b_empty[bs]);
                bs ^= 1;
                if (bs == 0) bph ^= 1;
                --left;
                if (left == 0 || ks + 1 == t.ksteps) {   // the chunk's sums are complete
                    if (leader) mma_commit(acc_full);
                    left = 0;
                }
            }
        }
        // every MMA this warp issued has completed before tensor memory is released
        if (leader) mma_commit(mma_done);
        const long long t0 = clock64();
        while (!mbar_try_wait(mma_done, 0) && clock64() - t0 < WAIT_CYCLES) {
        }
    } else {
        // ---------------------------------- epilogue (warps 0-3) ------------------------------
        // MODE 0, 2 and 3: exponents are the same for every chunk, so chunk sums are accumulated with the
        // level factor 2^{-7(L+2)} only and the row/column powers of two are applied once at the end.
        const int row = warp * 32 + lane;               // TMEM lane = tile row
        const unsigned lane_base = tmem + ((unsigned)(warp * 32) << 16);
        constexpr int NG = N / 16;                       // 16-column groups
        unsigned cph = 0;
        bool ok = true;
        for (int b = blockIdx.x; b < total && ok; b += gridDim.x) {
            const Tile t = decode_tile<S, N, MODE>(args, b);
            const int grow = t.m0 + row;
            const int nw = MODE == 1 || MODE == 2 ? N : t.nw;
            const int nchunks = (t.ksteps + CSTEPS - 1) / CSTEPS;
            f2 hi[N / 2], lo[N / 2];
#pragma unroll
            for (int c = 0; c < N / 2; ++c) hi[c] = lo[c] = 0;
            for (int ch = 0; ch < nchunks; ++ch) {
                int erow = 0;
                int ec[(N + 31) / 32];                   // MODE 1: column exponents, one per lane
                if (MODE == 1) {
                    const int* e = args.row_e + (long long)(t.chunk0 + ch) * args.np;
                    erow = grow < args.np ? __ldg(e + grow) : 0;
#pragma unroll
                    for (int g = 0; g < (N + 31) / 32; ++g)
                        ec[g] = t.n0 + g * 32 + lane < args.np ? __ldg(e + t.n0 + g * 32 + lane) : 0;
                }
                if (!(ok = mbar_wait_warp(acc_full, cph, err, wait))) break;
                cph ^= 1;
                fence_after();
                // per element the levels are added in descending order; the next level's load is in flight while
                // this one's sums are added
                unsigned r[2][16];
                tmem_ld16(lane_base + (unsigned)((S - 1) * nw), r[0]);
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    if (g * 16 < nw) {   // (a break here would keep the loop from being unrolled)
                    // MODE 1: the factors 2^{e_row + e_col} of the group's columns; where the lowest level's
                    // factor leaves the normal range (pow2f gives zero there) each is formed by itself
                    f2 cf[8];
                    int ee[16];
                    bool plain = true;
                    if (MODE == 1) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            ee[j] = erow + __shfl_sync(0xffffffffu, ec[g / 2], (g & 1) * 16 + j);
                            plain = plain && ee[j] >= 7 * (S + 1) - 126 && ee[j] <= 127;
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            cf[j] = pack2((unsigned)(127 + ee[2 * j]) << 23, (unsigned)(127 + ee[2 * j + 1]) << 23);
                        plain = __all_sync(0xffffffffu, plain);
                    }
#pragma unroll
                    for (int q = 0; q < S; ++q) {
                        const int L = S - 1 - q, cur = (g * S + q) & 1;
                        tmem_wait(r[cur]);
                        if (q + 1 < S) tmem_ld16(lane_base + (unsigned)((L - 1) * nw + g * 16), r[cur ^ 1]);
                        else if (g + 1 < NG && (g + 1) * 16 < nw)
                            tmem_ld16(lane_base + (unsigned)((S - 1) * nw + (g + 1) * 16), r[cur ^ 1]);
                        const unsigned lv = (unsigned)(127 - 7 * (L + 2)) << 23;
                        const f2 lev = pack2(lv, lv);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            f2 sc = lev;
                            if (MODE == 1) {
                                if (plain) sc = mul2(cf[j], lev);
                                else sc = pack2(__float_as_uint(pow2f(ee[2 * j] - 7 * (L + 2))),
                                                __float_as_uint(pow2f(ee[2 * j + 1] - 7 * (L + 2))));
                            }
                            two_sum_acc(hi[g * 8 + j], lo[g * 8 + j], pack2(r[cur][2 * j], r[cur][2 * j + 1]), sc);
                        }
                    }
                    }
                }
                fence_before();
                mbar_arrive(acc_empty);
            }
            if (!ok) break;
            // output
            if (*(volatile int*)err || grow >= (MODE == 0 ? args.rows : args.np)) continue;
            if (MODE == 2) {
                const int er = args.row_e[grow];
                double* o = args.outd + (long long)grow * args.ldo;
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const f2 h = hi[c / 2], l = lo[c / 2];
                    const double v = scale_pow2(c & 1 ? (double)hi_of(h) + (double)hi_of(l) : (double)lo_of(h) + (double)lo_of(l),
                                                er + __ldg(args.col_e + t.n0 + c));
                    const int2 p = __ldg(args.pos + t.n0 + c);
                    if (p.x >= 0) o[p.x] = v;
                    if (p.y >= 0) o[p.y] = v;
                }
            } else if (MODE == 0 || MODE == 3) {
                const int er = args.row_e[MODE == 3 ? t.P : grow];
                float2* o = args.out + ((MODE == 3 ? (long long)t.P * args.np : 0LL) + grow) * args.ldy + t.n0;
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    if (c < nw) {
                        const float f = pow2f(er + __ldg(args.col_e + t.n0 + c));
                        const f2 h = hi[c / 2], l = lo[c / 2];
                        o[c] = c & 1 ? make_float2(hi_of(h) * f, hi_of(l) * f) : make_float2(lo_of(h) * f, lo_of(l) * f);
                    }
                }
            } else {
                float2* o = args.out + ((long long)t.split * args.npt + grow) * args.npt + t.n0;
#pragma unroll
                for (int c = 0; c < N; c += 2)
                    if (TM % N == 0 || t.n0 + c < args.npt) {   // a width that does not divide 128 may run over
                        o[c] = make_float2(lo_of(hi[c / 2]), lo_of(lo[c / 2]));
                        o[c + 1] = make_float2(hi_of(hi[c / 2]), hi_of(lo[c / 2]));
                    }
            }
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOLS));
}


// ------------------------------------------------------------------------------------------------
// tensor maps through the driver entry point (no link-time dependence on libcuda)
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static std::mutex mu;
    static EncodeTiledFn fn = nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        DF_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
        if (q != cudaDriverEntryPointSuccess || !p) throw Error{DF_E_CUDA, "cuTensorMapEncodeTiled unavailable"};
        fn = (EncodeTiledFn)p;
    }
    return fn;
}

// 3-D BF16 tensor [d2][d1][d0] (d0 contiguous) with box {64, rows, 1}, 128-byte swizzle, zero fill
CUtensorMap make_map(const bf16* base, unsigned long long d0, unsigned long long d1, unsigned long long d2,
                     unsigned rows) {
    CUtensorMap m;
    const cuuint64_t dims[3] = {d0, d1, d2};
    const cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
    const cuuint32_t box[3] = {(cuuint32_t)KS, rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)base, dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) throw Error{DF_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r)};
    return m;
}

// Budget of the kernels' pipeline waits: WAIT_CYCLES, or DFHF_TC_WAIT_CYCLES (a test knob that makes the
// waits run out, to exercise the DF_E_TIMEOUT path; the drains of work already issued keep WAIT_CYCLES)
long long pipeline_wait_cycles() {
    const char* v = std::getenv("DFHF_TC_WAIT_CYCLES");
    const long long c = v ? std::atoll(v) : 0;
    return (c > 0 && c < WAIT_CYCLES) ? c : WAIT_CYCLES;
}

// CTAs that the current device holds at once
template <int S, int N>
int resident_ctas() {
    int dev = 0, sms = 0;
    DF_CUDA(cudaGetDevice(&dev));
    DF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return sms * ctas_per_sm<S, N>();
}

template <int S, int N, int MODE>
void launch_tc(cudaStream_t s, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& b2, const TcArgs& args_in,
               long long total) {
    if (total > INT_MAX - (1 << 20)) throw Error{DF_E_ARG, "tensor-core kernel: too many tiles"};
    constexpr int smem = tc_smem_bytes<S, N>();
    TcArgs args = args_in;
    args.wait_cycles = pipeline_wait_cycles();
    args.total = (int)total;
    DF_CUDA(cudaFuncSetAttribute(ozaki_tc_kernel<S, N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const int grid = MODE == 1 ? (int)total : (int)std::min<long long>(total, resident_ctas<S, N>());
    ozaki_tc_kernel<S, N, MODE><<<grid, 192, smem, s>>>(a, b, b2, args);
    DF_CHECK_LAUNCH();
}

// K[mu][nu] (n x n, FP64) = sum over splits of the float pairs, both triangles: a CTA per 8 rows of a lower
// 32 x 32 tile, the mirrored part through shared memory (reading it transposed instead took 67 us at n = 1200)
__global__ void __launch_bounds__(256) k_tc_reduce_kernel(const float2* __restrict__ Kpart, int nsplit, int npt, int n,
                                                          double* __restrict__ K) {
    __shared__ double t[8][33];
    const int tile = blockIdx.x >> 2, r8 = (blockIdx.x & 3) * 8;
    int I = (int)((sqrt(8.0 * tile + 1.0) - 1.0) * 0.5);
    while ((I + 1) * (I + 2) / 2 <= tile) ++I;
    while (I * (I + 1) / 2 > tile) --I;
    const int J = tile - I * (I + 1) / 2;
    {
        const int c = threadIdx.x & 31, r = threadIdx.x >> 5;
        const int mu = I * 32 + r8 + r, nu = J * 32 + c;
        double s = 0.0;
        if (mu < n && nu <= mu) {
#pragma unroll 4
            for (int q = 0; q < nsplit; ++q) {
                const float2 v = __ldcs(Kpart + ((long long)q * npt + mu) * npt + nu);
                s += (double)v.x + (double)v.y;
            }
            K[(long long)mu * n + nu] = s;
        }
        t[r][c] = s;
    }
    __syncthreads();
    const int c = threadIdx.x & 7, r = threadIdx.x >> 3;
    const int mu = I * 32 + r8 + c, nu = J * 32 + r;   // element (mu, nu) mirrored to row nu
    if (mu < n && nu < mu) K[(long long)nu * n + mu] = t[c][r];
}

}  // namespace

void k_tc_reduce(cudaStream_t s, const float2* Kpart, int nsplit, int npt, int n, double* K) {
    const int nt = (n + 31) / 32;
    k_tc_reduce_kernel<<<2 * nt * (nt + 1), 256, 0, s>>>(Kpart, nsplit, npt, n, K);
    DF_CHECK_LAUNCH();
}

// Y[P][mu][i] (float pairs, i < cols) = B_P C from the slices of B and Cs [S][ldy][np] by tiles of 128 rows x N
// columns (chosen by the autotuner), the last one narrower: MODE 0 from full rows, MODE 3 from packed tiles
template <int S, int N, int MODE>
void y_tc_launch(cudaStream_t s, const CUtensorMap& ma, const bf16* Cs, const TcArgs& a, long long row_tiles) {
    const CUtensorMap mb = make_map(Cs, a.np, a.ldy, S, N);
    const int last = a.cols % N;
    const CUtensorMap mb2 = last ? make_map(Cs, a.np, a.ldy, S, (unsigned)last) : mb;
    launch_tc<S, N, MODE>(s, ma, mb, mb2, a, row_tiles * ((a.cols + N - 1) / N));
}

// N: tile width
template <int MODE>
void y_tc_dispatch(cudaStream_t s, int S, int N, const CUtensorMap& ma, const bf16* Cs, const TcArgs& a, long long row_tiles) {
    if (S == 3 && N == 80) y_tc_launch<3, 80, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 5 && N == 80) y_tc_launch<5, 80, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 3 && N == 64) y_tc_launch<3, 64, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 5 && N == 64) y_tc_launch<5, 64, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 3 && N == 48) y_tc_launch<3, 48, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 5 && N == 48) y_tc_launch<5, 48, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 3 && N == 32) y_tc_launch<3, 32, MODE>(s, ma, Cs, a, row_tiles);
    else if (S == 5 && N == 32) y_tc_launch<5, 32, MODE>(s, ma, Cs, a, row_tiles);
    else throw Error{DF_E_ARG, "tensor-core split Y supports 3 or 5 slices and tile widths 32, 48, 64, 80"};
}

// from full rows Bs [S][naux][np][np], exponents Be [naux][np]
void y_split_tc(cudaStream_t s, int S, int N, const bf16* Bs, const int* Be, const bf16* Cs, const int* Ce, int naux,
                int np, int ldy, int cols, float2* Y, int* err) {
    if ((long long)naux * np > INT_MAX - TM) throw Error{DF_E_ARG, "tensor-core split Y: too many rows"};
    TcArgs a{};
    a.naux = naux;
    a.np = np;
    a.rows = naux * np;
    a.ldy = ldy;
    a.cols = cols;
    a.row_e = Be;
    a.col_e = Ce;
    a.out = Y;
    a.err = err;
    // the rows P np + mu as one dimension: tiles do not stop at an auxiliary row's end
    const CUtensorMap ma = make_map(Bs, np, (unsigned long long)naux * np, S, TM);
    y_tc_dispatch<0>(s, S, N, ma, Cs, a, ((long long)a.rows + TM - 1) / TM);
}

// from the packed slices Bs [S][zrows][nB (nB + 1) / 2][128][128] (lower 128-tiles, one exponent Be[P] per
// auxiliary row): naux rows are computed; the slices of row P sit at z = s * zrows + P (zrows >= naux: the
// buffer's rows)
void y_split_tc_packed(cudaStream_t s, int S, int N, const bf16* Bs, const int* Be, const bf16* Cs, const int* Ce,
                       int naux, int zrows, int np, int nB, int ldy, int cols, float2* Y, int* err) {
    if (np > nB * TM || np % KS) throw Error{DF_E_ARG, "internal: packed tiles do not cover the padded size"};
    if (zrows < naux) throw Error{DF_E_ARG, "internal: slice buffer smaller than the rows computed"};
    TcArgs a{};
    a.naux = zrows;
    a.np = np;
    a.ldy = ldy;
    a.cols = cols;
    a.nB = nB;
    a.row_e = Be;
    a.col_e = Ce;
    a.out = Y;
    a.err = err;
    const unsigned long long ntile = (unsigned long long)nB * (nB + 1) / 2;
    const CUtensorMap ma = make_map(Bs, TM, ntile * TM, (unsigned long long)S * zrows, KS);
    y_tc_dispatch<3>(s, S, N, ma, Cs, a, (long long)naux * nB);
}

// B[P][pos[c]] = sum_Q L^-1[P][Q] A[Q][c] for the ncols columns of one chunk, from the 7 slices
// Ls [7][naux][kp] (row exponents eL) and At [7][ncols][kp] (column exponents eA); rows of `out` have
// stride ldo. kp is naux padded to a multiple of 64 (zero slices beyond naux), ncols a multiple of 64.
template <int N>
void whiten_tc_n(cudaStream_t s, const bf16* Ls, const int* eL, const bf16* At, const int* eA, int naux, int kp,
                 int ncols, const int2* pos, double* out, long long ldo, int* err) {
    constexpr int S = 7;
    if (kp % KS || ncols % N) throw Error{DF_E_ARG, "internal: whitening operands not padded to 64"};
    TcArgs a{};
    a.naux = naux;
    a.np = naux;
    a.row_e = eL;
    a.col_e = eA;
    a.err = err;
    a.ncols = ncols;
    a.pos = pos;
    a.outd = out;
    a.ldo = ldo;
    const CUtensorMap ma = make_map(Ls, kp, naux, S, TM);
    const CUtensorMap mb = make_map(At, kp, ncols, S, N);
    launch_tc<S, N, 2>(s, ma, mb, mb, a, (long long)((naux + TM - 1) / TM) * (ncols / N));
}

// N: output tile width, 64 or 32 (32: two CTAs per SM)
void whiten_tc(cudaStream_t s, int N, const bf16* Ls, const int* eL, const bf16* At, const int* eA, int naux, int kp,
               int ncols, const int2* pos, double* out, long long ldo, int* err) {
    if (N == 64) whiten_tc_n<64>(s, Ls, eL, At, eA, naux, kp, ncols, pos, out, ldo, err);
    else if (N == 32) whiten_tc_n<32>(s, Ls, eL, At, eA, naux, kp, ncols, pos, out, ldo, err);
    else throw Error{DF_E_ARG, "tensor-core whitening supports tile widths 32 and 64"};
}

// K partial sums over the lower triangle of 128-blocks: Kpart [nsplit][npt][npt] (float pairs), from the Y slices
// Ys [S][KL / 64][np][64] (KL = naux ldy over the contraction index k = P ldy + i, tile-major) with exponents
// Ye [chunk][np]. One CTA per tile: the tiles are long (hundreds of K-steps), so the block scheduler's balance is
// worth more than a persistent CTA's overlap of their ends (measured 1341 against 1242 TFLOP/s at n = 1216).
template <int S, int N>
void k_tc_launch(cudaStream_t s, const bf16* Ys, TcArgs a) {
    a.ntiles = 0;
    for (int I = 0; I < a.npt / TM; ++I) a.ntiles += k_col_tiles(I, N);
    const CUtensorMap ma = make_map(Ys, KS, a.np, (unsigned long long)S * a.nkb, TM);
    const CUtensorMap mb = make_map(Ys, KS, a.np, (unsigned long long)S * a.nkb, N);
    launch_tc<S, N, 1>(s, ma, mb, mb, a, (long long)a.ntiles * a.nsplit);
}

// N: column tile width, 32, 48 or 64
void k_split_tc(cudaStream_t s, int S, int N, const bf16* Ys, const int* Ye, int naux, int np, int ldy, int cols, int nsplit,
                float2* Kpart, int npt, int* err) {
    TcArgs a{};
    a.naux = naux;
    a.np = np;
    a.ldy = ldy;
    a.cols = cols;
    a.KL = (long long)naux * ldy;
    a.nkb = (int)((a.KL + KS - 1) / KS);
    a.nsplit = nsplit;
    a.row_e = Ye;
    a.out = Kpart;
    a.npt = npt;
    a.err = err;
    if (S == 3 && N == 64) k_tc_launch<3, 64>(s, Ys, a);
    else if (S == 5 && N == 64) k_tc_launch<5, 64>(s, Ys, a);
    else if (S == 3 && N == 48) k_tc_launch<3, 48>(s, Ys, a);
    else if (S == 5 && N == 48) k_tc_launch<5, 48>(s, Ys, a);
    else if (S == 3 && N == 32) k_tc_launch<3, 32>(s, Ys, a);
    else if (S == 5 && N == 32) k_tc_launch<5, 32>(s, Ys, a);
    else throw Error{DF_E_ARG, "tensor-core split K supports 3 or 5 slices and tile widths 32, 48, 64"};
}

}  // namespace dfhf
