// FP64 dense contractions on the CUDA cores (DFMA).
//
// GB300 does 2 FP64 multiply-adds per clock and SM: one 64 x 64 x 16 tile step alone keeps an SM busy for
// 16 us, and a warp's DFMA occupies its sub-core for 64 clocks. Neither operand staging nor instruction issue
// is near a limit; what costs time is arithmetic on padding and SMs without a tile. So the tiles here are
// small (16 x 8 to 128 x 5 outputs per CTA), their shape is chosen per product by a model of just that
// (pick_and_launch: padding, waves over the SMs, step latency), and batched rows are flattened so that no batch
// entry pads its own last tile. Where the outputs alone do not fill the GPU, dgemm_rows lets the CTAs of a
// thread-block cluster split the contraction and add their partial tiles through distributed shared memory in a
// fixed order (deterministic, no workspace); everything that feeds an SCF keeps each element one chain of
// multiply-adds in ascending order of the contraction, whatever the tile.
//   - dgemm: general row-major C = alpha op(A) op(B) + beta C, never a split contraction (SCF algebra);
//     dgemm_lower: the same for a lower-triangular B (metric inverse).
//   - dgemm_rows: C[b][m][n] = sum_k A[b][m][k] B[k][n] for every batch b at once, any strides (object operations,
//     MP2); its contraction may be split.
//   - dgemv_rows, dgemv_cols: products with one column or one row (the objects' density contractions), bound by HBM.
//   - whiten_fp64_inplace: A <- L A for lower-triangular L, in place (the FP64 whitening, paper eq. 1, third
//     form): one launch, each CTA owning its columns, over the distinct elements mu >= nu only.
//   - y_transform: Y[mu][P nocc + i] = sum_nu B_{P,mu nu} C_{nu i} reading the packed symmetric B (paper eq. 1,
//     first form); each stored off-diagonal tile serves both (I,J) and (J,I).
//   - k_syrk: K = Y Y^T over lower tiles with split partial sums (paper eq. 2, first form), reduced in order.
// The 64 x 64 register tiles that these kernels replace ran the FP64 pipe at its rate too, but half of it on
// padding (8 waters: Y 22.7 ms, now 11.4; K 11.9 ms, now 6.0) or on one SM in three (400 x 400 products).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace dfhf {

namespace {

constexpr int GT = 128;   // threads of every tile kernel
constexpr int GK = 16;    // contraction elements per step

// where the row operand comes from: k contiguous in memory, row index contiguous, or the packed symmetric B
enum { A_KFAST = 0, A_MFAST = 1, A_PACKED = 2 };

struct GemmArgs {
    // row r = (batch b = r / M, m = r % M): A[b aB + m aM + k aK], C[b cB + m cM + n cN]; B[k bK + n bN]
    const double* A;
    long long aB, aM, aK;
    const double* B;
    long long bK, bN;
    double* C;
    long long cB, cM, cN;
    unsigned rows;     // batches x M, below 2^31
    int M, N, K;
    double alpha, beta;
    int split;         // CTAs of a cluster that share one tile's contraction (1, 2, 4 or 8); SYRK: partial sums
    int ntn;           // column tiles
    int b_lower;       // B[k][n] = 0 for k < n: the contraction starts at the tile's first column
    int naux;          // SYRK: partial sum s covers the auxiliary rows [naux s / split, naux (s + 1) / split)
};

// ------------------------------------------------------------------------------------------------
// C tile of BM = (128 / TX) TM rows by BN = TX TN columns: thread (tx, ty) owns rows ty + TY i and columns
// tx + TX j; operand steps of 16 k pass through registers into two shared buffers. SYRK: rows = columns = N,
// B = A, lower tiles only, partial sum `rank` of the contraction into C + rank N N (elements below the diagonal).
// Bound by the FP64 pipe: at 8 waters (n = 400, naux = 1096, 40 occupied) Y runs at 98 % and K at 94 % of the
// unit count's 1.256 TFLOP/s on useful work.
// ------------------------------------------------------------------------------------------------
template <int TX, int TM, int TN, int AMODE, bool SYRK>
__global__ void __launch_bounds__(GT) fgemm_kernel(const GemmArgs g) {
    constexpr int TY = GT / TX, BM = TY * TM, BN = TX * TN;
    constexpr int LDA = BM + 1, LDB = BN + 1;
    constexpr int NA = BM * GK / GT;                 // A elements per thread and step
    constexpr int NB = (BN * GK + GT - 1) / GT;      // B elements per thread and step
    static_assert(2 * GK * (LDA + LDB) >= BM * BN, "the partial tile reuses the operand buffers");
    __shared__ double sm[2 * GK * (LDA + LDB)];
    double* As = sm;                                 // [2][GK][LDA]
    double* Bs = sm + 2 * GK * LDA;                  // [2][GK][LDB]
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int split = g.split;
    const int rank = (int)(blockIdx.x % split);
    const unsigned tile = blockIdx.x / split;
    unsigned r0;
    int n0;
    if (SYRK) {
        // lower tiles column by column: column bj holds the row tiles from the one its first row falls in
        const int nrt = (g.N + BM - 1) / BM;
        int t = (int)tile, bj = 0, first = 0;
        for (;; ++bj) {
            first = bj * BN / BM;
            if (t < nrt - first) break;
            t -= nrt - first;
        }
        r0 = (unsigned)(first + t) * BM;
        n0 = bj * BN;
    } else {
        r0 = (tile / g.ntn) * BM;
        n0 = (int)(tile % g.ntn) * BN;
    }
    // this CTA's part [kbeg, kend) of the contraction
    int kbeg, kend;
    if (SYRK) {
        const int per = g.K / g.naux;   // occupied orbitals
        kbeg = (int)((long long)g.naux * rank / split) * per;
        kend = (int)((long long)g.naux * (rank + 1) / split) * per;
    } else {
        const int step0 = g.b_lower ? n0 / GK : 0, nsteps = (g.K + GK - 1) / GK - step0;
        kbeg = (step0 + (int)((long long)nsteps * rank / split)) * GK;
        kend = min(g.K, (step0 + (int)((long long)nsteps * (rank + 1) / split)) * GK);
    }
    const int steps = kend > kbeg ? (kend - kbeg + GK - 1) / GK : 0;

    // ---- this thread's operand rows --------------------------------------------------------------
    const int ka = AMODE == A_MFAST ? tid / BM : tid & 15;   // first k of this thread's A elements
    constexpr int NP = AMODE == A_MFAST ? 1 : NA;            // distinct rows
    long long aoff[NP];                                      // -1: beyond the last row
    int amu[AMODE == A_PACKED ? NP : 1];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const unsigned r = r0 + (AMODE == A_MFAST ? tid % BM : (tid >> 4) + 8 * q);
        aoff[q] = -1;
        if (r < g.rows) {
            const unsigned b = r / (unsigned)g.M, m = r - b * (unsigned)g.M;
            if (AMODE == A_PACKED) {
                aoff[q] = b * g.aB;
                amu[q] = (int)m;
            } else {
                aoff[q] = b * g.aB + m * g.aM;
            }
        }
    }
    const bool bkfast = SYRK || g.bK == 1;

    double va[NA], vb[NB];
    auto load = [&](int s) {
        const int k0 = kbeg + s * GK;
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            const int k = k0 + (AMODE == A_MFAST ? ka + (GT / BM > 0 ? GT / BM : 1) * q : ka);
            const int p = AMODE == A_MFAST ? 0 : q;
            double v = 0.0;
            if (aoff[p] >= 0 && k < kend) {
                if (AMODE == A_PACKED) {
                    const int I = amu[p] >> 6, J = k >> 6;
                    const long long at = I >= J ? tile_pair(I, J) * (TS * TS) + (amu[p] & 63) * TS + (k & 63)
                                                : tile_pair(J, I) * (TS * TS) + (k & 63) * TS + (amu[p] & 63);
                    v = __ldg(g.A + aoff[p] + at);
                } else {
                    v = __ldg(g.A + aoff[p] + (AMODE == A_KFAST ? (long long)k : k * g.aK));
                }
            }
            va[q] = v;
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int idx = tid + GT * q;
            const int k = bkfast ? idx & 15 : idx / BN, n = bkfast ? idx >> 4 : idx % BN;
            double v = 0.0;
            if (idx < BN * GK && k0 + k < kend && n0 + n < g.N)
                v = __ldg(SYRK ? g.A + (long long)(n0 + n) * g.aM + k0 + k
                               : g.B + (long long)(k0 + k) * g.bK + (long long)(n0 + n) * g.bN);
            vb[q] = v;
        }
    };
    auto store = [&](int buf) {
        double* a = As + buf * GK * LDA;
        double* b = Bs + buf * GK * LDB;
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            if (AMODE == A_MFAST) a[(ka + (GT / BM > 0 ? GT / BM : 1) * q) * LDA + tid % BM] = va[q];
            else a[ka * LDA + (tid >> 4) + 8 * q] = va[q];
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int idx = tid + GT * q;
            const int k = bkfast ? idx & 15 : idx / BN, n = bkfast ? idx >> 4 : idx % BN;
            if (idx < BN * GK) b[k * LDB + n] = vb[q];
        }
    };

    double acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
    if (steps > 0) {
        load(0);
        store(0);
    }
    __syncthreads();
    for (int s = 0; s < steps; ++s) {
        const int cur = s & 1;
        if (s + 1 < steps) load(s + 1);
        const double* a = As + cur * GK * LDA + ty;
        const double* b = Bs + cur * GK * LDB + tx;
#pragma unroll
        for (int k = 0; k < GK; ++k) {
            double x[TM], y[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) x[i] = a[k * LDA + TY * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) y[j] = b[k * LDB + TX * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
        }
        if (s + 1 < steps) store(cur ^ 1);
        __syncthreads();
    }

    auto write = [&](unsigned r, int n, double v) {
        if (SYRK) {
            if ((int)r >= g.N || n > (int)r) return;
            g.C[((long long)rank * g.N + r) * g.N + n] = v;
        } else {
            if (r >= g.rows || n >= g.N) return;
            const unsigned b = r / (unsigned)g.M, m = r - b * (unsigned)g.M;
            double* c = g.C + b * g.cB + m * g.cM + n * g.cN;
            *c = g.alpha * v + (g.beta == 0.0 ? 0.0 : g.beta * *c);
        }
    };
    if (SYRK || split == 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) write(r0 + ty + TY * i, n0 + tx + TX * j, acc[i][j]);
        return;
    }
    // partial tiles of the cluster's CTAs, added in rank order through distributed shared memory
    cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) sm[(ty + TY * i) * BN + tx + TX * j] = acc[i][j];
    cluster.sync();
    for (int e = rank * GT + tid; e < BM * BN; e += split * GT) {
        double v = 0.0;
        for (int q = 0; q < split; ++q) v += cluster.map_shared_rank(sm, q)[e];
        write(r0 + e / BN, n0 + e % BN, v);
    }
    cluster.sync();   // no CTA leaves while its partial tile may still be read
}

// ------------------------------------------------------------------------------------------------
// choice of the tile: the model counts, in SM clocks, the waves of CTAs over the 152 SMs times the tile's
// multiply-adds at 2 per clock (padding included), a floor of STEP_CLOCKS per 16-element step (load latency
// that the one step of prefetch does not hide when a tile is small and alone on its SM), and the operands' L2
// traffic. Measured on 400 x 400 x 400: 0.41 ms with the 64 x 64 tiles before (49 CTAs), 0.11 ms with the
// model's choice (the FP64 pipe's floor is 0.10 ms).
// ------------------------------------------------------------------------------------------------
constexpr int NSM = 152;
constexpr double STEP_CLOCKS = 1000.0;     // one step of a lone small tile, measured order
constexpr double L2_BYTES_PER_CLOCK = 1500.0;

struct TileShape {
    int tx, tm, tn;
    int bm() const { return GT / tx * tm; }
    int bn() const { return tx * tn; }
};

// clocks for `tiles` tiles with a contraction of K split over S CTAs
double tile_cost(const TileShape& t, double tiles, int K, int S) {
    const int steps = ((K + GK - 1) / GK + S - 1) / S;
    const double ctas = tiles * S, waves = std::ceil(ctas / NSM);
    const double together = std::min(waves, 6.0);      // CTAs resident on an SM
    const double step = std::max(together * t.bm() * t.bn() * (GK / 2.0), STEP_CLOCKS);
    const double pipe = waves / together * steps * step + (S > 1 ? 2500.0 : 0.0);
    const double l2 = ctas * steps * GK * 8.0 * (t.bm() + t.bn()) / L2_BYTES_PER_CLOCK;
    // a slight preference for larger tiles among equals (fewer operand reads and addresses per multiply-add)
    return std::max(pipe, l2) * (1.0 + 0.3 / t.bm() + 0.3 / t.bn());
}

template <int TX, int TM, int TN, int AMODE, bool SYRK>
void launch_tile(cudaStream_t s, GemmArgs g, unsigned tiles) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles * g.split);
    cfg.blockDim = dim3(GT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    if (!SYRK && g.split > 1) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = g.split;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
    DF_CUDA(cudaLaunchKernelEx(&cfg, fgemm_kernel<TX, TM, TN, AMODE, SYRK>, g));
}

typedef void (*TileLaunch)(cudaStream_t, GemmArgs, unsigned);
struct TileKernel {
    TileShape shape;
    TileLaunch launch;
};
#define TILE(TX, TM, TN, MODE, SYRK) {{TX, TM, TN}, launch_tile<TX, TM, TN, MODE, SYRK>}
// column widths of 8 to 40, and of 5, 10 and 20 for the few occupied orbitals of small molecules
#define TILES_GENERAL(MODE)                                                                                       \
    TILE(8, 1, 1, MODE, false), TILE(8, 1, 2, MODE, false), TILE(8, 1, 3, MODE, false), TILE(8, 1, 5, MODE, false), \
        TILE(8, 2, 2, MODE, false), TILE(8, 2, 4, MODE, false), TILE(8, 4, 4, MODE, false),                        \
        TILE(8, 4, 5, MODE, false), TILE(4, 1, 5, MODE, false), TILE(2, 1, 5, MODE, false), TILE(1, 1, 5, MODE, false)
const TileKernel KFAST_TILES[] = {TILES_GENERAL(A_KFAST)};
const TileKernel MFAST_TILES[] = {TILES_GENERAL(A_MFAST)};
const TileKernel PACKED_TILES[] = {TILE(8, 1, 1, A_PACKED, false), TILE(8, 4, 2, A_PACKED, false), TILE(8, 4, 3, A_PACKED, false),
                                   TILE(8, 4, 4, A_PACKED, false), TILE(8, 4, 5, A_PACKED, false), TILE(4, 2, 5, A_PACKED, false),
                                   TILE(2, 1, 5, A_PACKED, false), TILE(1, 1, 5, A_PACKED, false)};
const TileKernel SYRK_TILES[] = {TILE(8, 1, 1, A_KFAST, true), TILE(8, 1, 2, A_KFAST, true), TILE(8, 1, 5, A_KFAST, true),
                                 TILE(8, 2, 4, A_KFAST, true), TILE(8, 4, 4, A_KFAST, true), TILE(8, 4, 5, A_KFAST, true)};
#undef TILES_GENERAL
#undef TILE

double count_tiles(const TileShape& t, const GemmArgs& g, bool syrk) {
    const int bm = t.bm(), bn = t.bn();
    if (!syrk) return std::ceil((double)g.rows / bm) * ((g.N + bn - 1) / bn);
    const int nrt = (g.N + bm - 1) / bm;
    double c = 0;
    for (int bj = 0; bj * bn < g.N; ++bj) c += nrt - bj * bn / bm;
    return c;
}

// most_split: the largest cluster that may share a tile's contraction; fixed_split (SYRK): the partial sums
template <size_t NT>
void pick_and_launch(cudaStream_t s, GemmArgs g, const TileKernel (&kernels)[NT], bool syrk, int most_split, int fixed_split) {
    double best = 1e300;
    const TileKernel* pick = &kernels[0];
    int bs = 1;
    for (const TileKernel& k : kernels) {
        const double tiles = count_tiles(k.shape, g, syrk);
        if (tiles * std::max(most_split, fixed_split) > 2.0e9) continue;
        for (int S = fixed_split ? fixed_split : 1; S <= std::max(most_split, fixed_split); S *= 2) {
            if (!fixed_split && S > 1 && S * GK > g.K) break;
            const double c = tile_cost(k.shape, tiles, g.K, S);
            if (c < best) {
                best = c;
                pick = &k;
                bs = S;
            }
        }
    }
    g.split = bs;
    g.ntn = (g.N + pick->shape.bn() - 1) / pick->shape.bn();
    pick->launch(s, g, (unsigned)count_tiles(pick->shape, g, syrk));
}

// K[mu][nu] = sum over the partial sums in order, both triangles: a CTA per 8 rows of a lower 32 x 32 tile, a
// thread per element (the transposed part through shared memory). Bound by the latency of the partial sums'
// reads, eight in flight (n = 100, 68 sums: 26 us on the ten CTAs of whole tiles).
__global__ void __launch_bounds__(256) syrk_reduce_kernel(const double* __restrict__ part, int nsplit, int n,
                                                          double* __restrict__ K) {
    __shared__ double t[8][33];
    const int tile = blockIdx.x >> 2, r8 = (blockIdx.x & 3) * 8;
    int I = (int)((sqrt(8.0 * tile + 1.0) - 1.0) * 0.5);
    while ((I + 1) * (I + 2) / 2 <= tile) ++I;
    while (I * (I + 1) / 2 > tile) --I;
    const int J = tile - I * (I + 1) / 2;
    const long long nn = (long long)n * n;
    {
        const int c = threadIdx.x & 31, r = threadIdx.x >> 5;
        const int mu = I * 32 + r8 + r, nu = J * 32 + c;
        double s = 0.0;
        if (mu < n && nu <= mu) {
            const double* p = part + (long long)mu * n + nu;
            int q = 0;
            for (; q + 8 <= nsplit; q += 8) {
                double v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = p[(q + u) * nn];
#pragma unroll
                for (int u = 0; u < 8; ++u) s += v[u];
            }
            for (; q < nsplit; ++q) s += p[q * nn];
            K[(long long)mu * n + nu] = s;
        }
        t[r][c] = s;
    }
    __syncthreads();
    const int c = threadIdx.x & 7, r = threadIdx.x >> 3;
    const int mu = I * 32 + r8 + c, nu = J * 32 + r;   // element (mu, nu) mirrored to row nu
    if (mu < n && nu < mu) K[(long long)nu * n + mu] = t[c][r];
}

// ------------------------------------------------------------------------------------------------
// matrix-vector products
// ------------------------------------------------------------------------------------------------
// y[r] = sum_k A[r lda + k] x[k]: one cluster of `split` CTAs per row, each a part of the row. Bound by the read
// of A (548 rows of 40000: 50 us for 175 MB; as a column of 64-wide tiles it took 62 ms).
__global__ void __launch_bounds__(256) gemv_dot_kernel(const double* __restrict__ A, long long lda, long long K,
                                                       const double* __restrict__ x, double* __restrict__ y, int split) {
    const long long r = blockIdx.x / split;
    const int rank = (int)(blockIdx.x % split);
    const long long k0 = K * rank / split, k1 = K * (rank + 1) / split;
    const double* a = A + r * lda;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    long long k = k0 + threadIdx.x;
    for (; k + 768 < k1; k += 1024) {
        const double a0 = __ldcs(a + k), a1 = __ldcs(a + k + 256), a2 = __ldcs(a + k + 512), a3 = __ldcs(a + k + 768);
        s0 = fma(a0, __ldg(x + k), s0);
        s1 = fma(a1, __ldg(x + k + 256), s1);
        s2 = fma(a2, __ldg(x + k + 512), s2);
        s3 = fma(a3, __ldg(x + k + 768), s3);
    }
    for (; k < k1; k += 256) s0 = fma(__ldcs(a + k), __ldg(x + k), s0);
    double s = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double part[8];
    __shared__ double total;
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += part[w];
        total = v;
    }
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
        double v = 0.0;
        for (int q = 0; q < split; ++q) v += *cluster.map_shared_rank(&total, q);
        y[r] = v;
    }
    cluster.sync();   // no CTA leaves while its part may still be read
}

// y[c] = sum_k x[k] A[k lda + c]: 32 columns x 8 row groups per CTA, the rows of A split over a cluster of
// `split` CTAs; partial sums added in a fixed order. Bound by the read of A (as above: 52 us, before 50 ms).
__global__ void __launch_bounds__(256) gemv_sweep_kernel(const double* __restrict__ A, long long lda, int K,
                                                         const double* __restrict__ x, long long N,
                                                         double* __restrict__ y, int split) {
    const long long c = (long long)(blockIdx.x / split) * 32 + (threadIdx.x & 31);
    const int rank = (int)(blockIdx.x % split), grp = threadIdx.x >> 5;
    const int parts = 8 * split, p = rank * 8 + grp;
    const int k0 = (int)((long long)K * p / parts), k1 = (int)((long long)K * (p + 1) / parts);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    if (c < N) {
        const double* a = A + c;
        int k = k0;
        for (; k + 4 <= k1; k += 4) {
            const double a0 = __ldcs(a + k * lda), a1 = __ldcs(a + (k + 1) * lda), a2 = __ldcs(a + (k + 2) * lda),
                         a3 = __ldcs(a + (k + 3) * lda);
            s0 = fma(__ldg(x + k), a0, s0);
            s1 = fma(__ldg(x + k + 1), a1, s1);
            s2 = fma(__ldg(x + k + 2), a2, s2);
            s3 = fma(__ldg(x + k + 3), a3, s3);
        }
        for (; k < k1; ++k) s0 = fma(__ldg(x + k), __ldcs(a + k * lda), s0);
    }
    __shared__ double part[8][32];
    __shared__ double total[32];
    part[grp][threadIdx.x & 31] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += part[w][threadIdx.x];
        total[threadIdx.x] = v;
    }
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0 && threadIdx.x < 32 && c < N) {
        double v = total[threadIdx.x];
        for (int q = 1; q < split; ++q) v += cluster.map_shared_rank(total, q)[threadIdx.x];
        y[c] = v;
    }
    cluster.sync();   // no CTA leaves while its part may still be read
}

template <typename... KArgs, typename... Args>
void launch_cluster(cudaStream_t s, void (*kernel)(KArgs...), unsigned grid, unsigned threads, int split, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    DF_CUDA(cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...));
}

// CTAs of a cluster per output block: enough to put about four CTAs on every SM
int vector_split(long long blocks, long long K, long long per) {
    int S = 1;
    while (S < 8 && blocks * S < 4 * NSM && K >= per * S * 2) S *= 2;
    return S;
}

// ------------------------------------------------------------------------------------------------
// A <- L A in place over the packed columns (mu, nu), mu >= nu: a CTA owns BN columns and walks the 32-row
// blocks of L from the last one up; row block I needs rows 0 .. end of block I of its own columns, which later
// (higher) blocks do not change. The packed tiles' padding (zero) and the mirror halves of the diagonal tiles
// (copied) are not computed: at n = 200 that is half of the 64-tiles' elements. Bound by the FP64 pipe.
// ------------------------------------------------------------------------------------------------
template <int TN>
__global__ void __launch_bounds__(GT) whiten_fp64_kernel(const double* __restrict__ L, int m, double* __restrict__ A,
                                                         long long ld, long long npair) {
    constexpr int TX = 8, TY = GT / TX, TM = 2, BM = TY * TM, BN = TX * TN;
    constexpr int LDA = BM + 1, LDB = BN + 1;
    constexpr int NA = BM * GK / GT, NB = BN * GK / GT;
    __shared__ double As[2][GK * LDA], Bs[2][GK * LDB];
    __shared__ long long pos[BN], mir[BN];           // packed position of each column, and of its mirror (-1: none)
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    for (int j = tid; j < BN; j += GT) {
        const long long c = (long long)blockIdx.x * BN + j;
        pos[j] = mir[j] = -1;
        if (c < npair) {
            int mu = (int)((sqrt(8.0 * (double)c + 1.0) - 1.0) * 0.5);
            while ((long long)(mu + 1) * (mu + 2) / 2 <= c) ++mu;
            while ((long long)mu * (mu + 1) / 2 > c) --mu;
            const int nu = (int)(c - (long long)mu * (mu + 1) / 2);
            pos[j] = packed_index(mu, nu);
            if (mu / TS == nu / TS && mu != nu) mir[j] = packed_index(nu, mu);
        }
    }
    __syncthreads();
    long long bpos[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) bpos[q] = pos[(tid + GT * q) % BN];
    for (int r0 = (m - 1) / BM * BM; r0 >= 0; r0 -= BM) {
        const int K = min(m, r0 + BM);               // L is zero beyond the diagonal block
        const int steps = (K + GK - 1) / GK;
        double va[NA], vb[NB];
        auto load = [&](int s) {
            const int k0 = s * GK;
#pragma unroll
            for (int q = 0; q < NA; ++q) {
                const int r = r0 + (tid >> 4) + 8 * q, k = k0 + (tid & 15);
                va[q] = (r < m && k < K) ? __ldg(L + (long long)r * m + k) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                const int k = k0 + (tid + GT * q) / BN;
                vb[q] = (bpos[q] >= 0 && k < K) ? A[(long long)k * ld + bpos[q]] : 0.0;
            }
        };
        auto store = [&](int buf) {
#pragma unroll
            for (int q = 0; q < NA; ++q) As[buf][(tid & 15) * LDA + (tid >> 4) + 8 * q] = va[q];
#pragma unroll
            for (int q = 0; q < NB; ++q) Bs[buf][(tid + GT * q) / BN * LDB + (tid + GT * q) % BN] = vb[q];
        };
        double acc[TM][TN] = {};
        load(0);
        store(0);
        __syncthreads();
        for (int s = 0; s < steps; ++s) {
            const int cur = s & 1;
            if (s + 1 < steps) load(s + 1);
#pragma unroll
            for (int k = 0; k < GK; ++k) {
                double x[TM], y[TN];
#pragma unroll
                for (int i = 0; i < TM; ++i) x[i] = As[cur][k * LDA + ty + TY * i];
#pragma unroll
                for (int j = 0; j < TN; ++j) y[j] = Bs[cur][k * LDB + tx + TX * j];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
            }
            if (s + 1 < steps) store(cur ^ 1);
            __syncthreads();
        }
        // every read of rows r0 .. r0 + BM - 1 (this block's and the earlier, lower ones') is done
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int r = r0 + ty + TY * i;
            if (r >= m) continue;
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const long long p = pos[tx + TX * j], q = mir[tx + TX * j];
                if (p >= 0) A[(long long)r * ld + p] = acc[i][j];
                if (q >= 0) A[(long long)r * ld + q] = acc[i][j];
            }
        }
    }
}

}  // namespace

// C[b][m][n] = alpha sum_k A[b][m][k] B[k][n] + beta C[b][m][n] for b < batches, m < M, n < N (general strides)
void dgemm_rows(cudaStream_t s, long long batches, int M, int N, int K, double alpha, const double* A, long long aB,
                long long aM, long long aK, const double* B, long long bK, long long bN, double beta, double* C,
                long long cB, long long cM, long long cN) {
    if (batches < 1 || M < 1 || N < 1) return;
    const long long most = ((1LL << 31) - 256) / M;   // batches per launch: rows stay below 2^31
    for (long long b0 = 0; b0 < batches; b0 += most) {
        const long long nb = std::min(most, batches - b0);
        GemmArgs g{A + b0 * aB, aB, aM, aK, B, bK, bN, C + b0 * cB, cB, cM, cN, (unsigned)(nb * M), M, N, K, alpha, beta,
                   1, 1, 0, 1};
        if (aM == 1 && aK != 1) pick_and_launch(s, g, MFAST_TILES, false, 8, 0);
        else if (aK == 1) pick_and_launch(s, g, KFAST_TILES, false, 8, 0);
        else throw Error{DF_E_ARG, "internal: dgemm_rows needs a unit stride in A"};
    }
}

void dgemv_rows(cudaStream_t s, int m, long long k, const double* A, long long lda, const double* x, double* y) {
    const int S = vector_split(m, k, 1024);
    launch_cluster(s, gemv_dot_kernel, (unsigned)m * S, 256, S, A, lda, k, x, y, S);
}

void dgemv_cols(cudaStream_t s, int k, long long n, const double* A, long long lda, const double* x, double* y) {
    const long long blocks = (n + 31) / 32;
    const int S = vector_split(blocks, k, 32);
    if (blocks * S >= (1LL << 31)) throw Error{DF_E_ARG, "vector-matrix product: too many columns"};
    launch_cluster(s, gemv_sweep_kernel, (unsigned)(blocks * S), 256, S, A, lda, k, x, n, y, S);
}

// Every element is one chain of multiply-adds in ascending k, whatever tile is picked: the metric's inverse
// factor, whose roundings its conditioning carries into J and K, and the SCF's matrices, whose roundings its
// early 3-slice exchange builds amplify, keep their bits.
void dgemm(cudaStream_t s, bool ta, bool tb, int m, int n, int k, double alpha, const double* A, int lda,
           const double* B, int ldb, double beta, double* C, int ldc) {
    if (m < 1 || n < 1) return;
    GemmArgs g{A, 0, ta ? 1 : lda, ta ? lda : 1, B, tb ? 1 : ldb, tb ? ldb : 1, C, 0, ldc, 1, (unsigned)m, m, n, k,
               alpha, beta, 1, 1, 0, 1};
    if (ta && lda != 1) pick_and_launch(s, g, MFAST_TILES, false, 1, 0);
    else pick_and_launch(s, g, KFAST_TILES, false, 1, 0);
}

// dgemm for B[i][j] = 0 where i < j: the contraction of each column tile starts at its first column
void dgemm_lower(cudaStream_t s, int m, int n, int k, double alpha, const double* A, int lda, const double* B, int ldb,
                 double beta, double* C, int ldc) {
    if (m < 1 || n < 1) return;
    GemmArgs g{A, 0, lda, 1, B, ldb, 1, C, 0, ldc, 1, (unsigned)m, m, n, k, alpha, beta, 1, 1, 1, 1};
    pick_and_launch(s, g, KFAST_TILES, false, 1, 0);
}

// A <- L A in place for lower-triangular L (m x m, row-major) over the packed rows of A (m rows of stride ld
// for n orbital functions)
void whiten_fp64_inplace(cudaStream_t s, int m, int n, const double* L, double* A, long long ld) {
    const long long npair = (long long)n * (n + 1) / 2;
    // column width by the waves it leaves: the CTAs are equal, so the SMs with one more set the time
    int best = 5;
    double cost = 1e300;
    for (int tn = 5; tn >= 2; --tn) {
        const double ctas = std::ceil(npair / (8.0 * tn));
        const double c = std::ceil(ctas / NSM) * tn * (1.0 + 0.1 / tn);
        if (c < cost) {
            cost = c;
            best = tn;
        }
    }
    const unsigned grid = (unsigned)((npair + 8 * best - 1) / (8 * best));
    switch (best) {
        case 2: whiten_fp64_kernel<2><<<grid, GT, 0, s>>>(L, m, A, ld, npair); break;
        case 3: whiten_fp64_kernel<3><<<grid, GT, 0, s>>>(L, m, A, ld, npair); break;
        case 4: whiten_fp64_kernel<4><<<grid, GT, 0, s>>>(L, m, A, ld, npair); break;
        default: whiten_fp64_kernel<5><<<grid, GT, 0, s>>>(L, m, A, ld, npair); break;
    }
    DF_CHECK_LAUNCH();
}

// Y[mu][P nocc + i] (n rows of naux nocc) = sum_nu B_P[mu][nu] C[nu][i] from the packed rows of B (naux rows of
// stride `row`) and C (n x nocc, row-major)
void y_transform_fp64(cudaStream_t s, const double* B, long long row, int n, int naux, const double* C, int nocc,
                      double* Y) {
    const long long most = ((1LL << 31) - 256) / n;
    const long long KL = (long long)naux * nocc;
    for (long long p0 = 0; p0 < naux; p0 += most) {
        const long long np = std::min<long long>(most, naux - p0);
        GemmArgs g{B + p0 * row, row, 0, 0, C, nocc, 1, Y + p0 * nocc, nocc, KL, 1, (unsigned)(np * n), n, nocc, n, 1.0, 0.0,
                   1, 1, 0, 1};
        pick_and_launch(s, g, PACKED_TILES, false, 1, 0);
    }
}

// K = Y Y^T (n x n, both triangles) from the n rows of Y of length naux nocc: nsplit partial sums over ranges of
// the auxiliary index (part: nsplit n n doubles), added in order
void k_syrk_fp64(cudaStream_t s, const double* Y, int n, int naux, int nocc, int nsplit, double* part, double* K) {
    const long long KL = (long long)naux * nocc;
    if (KL >= (1LL << 31) - 64) throw Error{DF_E_ARG, "FP64 exchange: naux x nocc exceeds 2^31"};
    GemmArgs g{Y, 0, KL, 1, nullptr, 1, 0, part, 0, n, 1, (unsigned)n, n, n, (int)KL, 1.0, 0.0, 1, 1, 0, naux};
    pick_and_launch(s, g, SYRK_TILES, true, 1, nsplit);
    const int nt = (n + 31) / 32;
    syrk_reduce_kernel<<<2 * nt * (nt + 1), 256, 0, s>>>(part, nsplit, n, K);
    DF_CHECK_LAUNCH();
}

}  // namespace dfhf
