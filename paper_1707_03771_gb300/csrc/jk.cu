// Per-iteration Coulomb and exchange builds from the packed, whitened B (paper eqs. 1-3).
//
// J (eq. 3): gamma_P = sum_{mu nu} B_{P,mu nu} D_{mu nu} is a dot product of each packed row of B
// with the packed, weighted density Dw (off-diagonal tiles carry weight 2, diagonal tiles are stored
// in full with weight 1), reduced with warp shuffles; J_{mu nu} = sum_P gamma_P B_{P,mu nu} is a
// column sweep over B with coalesced 16-byte loads. Both read B once; on GB300 both are bounded by
// the FP64 pipe (one FMA per 8 bytes needs 0.85 TFMA/s at 6.8 TB/s, above the ~0.5 TFMA/s DFMA rate).
// K (eqs. 1-2, first forms): Y = B C_occ per auxiliary row (dense.cu), then K = sum_P Y_P Y_P^T.
#include <algorithm>

#include "common.cuh"

namespace dfhf {

void k_syrk_fp64(cudaStream_t s, const double* Y, int n, int naux, int nocc, int nsplit, double* part, double* K);

namespace {

// Dw[packed(mu, nu)] = w D[mu][nu]; one block per tile pair (blockIdx.x = I, blockIdx.y = J)
__global__ void pack_density_kernel(const double* __restrict__ D, int n, double* __restrict__ Dw) {
    const int I = blockIdx.x, J = blockIdx.y;
    if (J > I) return;
    const double wgt = (I == J) ? 1.0 : 2.0;
    double* t = Dw + tile_pair(I, J) * TS * TS;
    for (int e = threadIdx.x; e < TS * TS; e += blockDim.x) {
        const int mu = I * TS + e / TS, nu = J * TS + e % TS;
        t[e] = (mu < n && nu < n) ? wgt * D[(long long)mu * n + nu] : 0.0;
    }
}

// M[r][mu][nu] (n x n) from the packed rows r = blockIdx.y
__global__ void unpack_kernel(const double* __restrict__ packed, long long row, int n, double* __restrict__ M) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x, nn = (long long)n * n;
    if (idx >= nn) return;
    M[blockIdx.y * nn + idx] = packed[blockIdx.y * row + packed_index((int)(idx / n), (int)(idx % n))];
}

// The last row of tiles holds n - 64 (nt - 1) rows of the matrix, the rest is zero padding, which the two
// Coulomb kernels leave out: they are bound by the FP64 pipe (one multiply-add per 8 bytes), and at 8 waters
// (n = 400) the padding is a fifth of the packed elements.

// gamma_P = <B_P, Dw>: one block per row, 16-byte loads, shuffle + shared reduction.
// 12 waters (n = 590): 642 -> 571 us, the column sweep below 620 -> 522 us.
__global__ void __launch_bounds__(256) gamma_kernel(const double* __restrict__ B, long long row, int nt, int n,
                                                    const double* __restrict__ Dw, double* __restrict__ gamma) {
    const long long P = blockIdx.x;
    const double2* b = reinterpret_cast<const double2*>(B + P * row);
    const double2* d = reinterpret_cast<const double2*>(Dw);
    constexpr int T2 = TS * TS / 2;                      // double2 per tile, a multiple of the block
    const long long full = (long long)nt * (nt - 1) / 2 * T2;
    double s0 = 0.0, s1 = 0.0;
    auto add = [&](long long i) {
        const double2 x = __ldcs(b + i);
        const double2 y = __ldg(d + i);
        s0 = fma(x.x, y.x, s0);
        s1 = fma(x.y, y.y, s1);
    };
#pragma unroll 4
    for (long long i = threadIdx.x; i < full; i += 256) add(i);
    const int last = (n - TS * (nt - 1)) * (TS / 2);     // double2 of a last-row tile's rows below n
    for (int J = 0; J < nt; ++J)
#pragma unroll 4
        for (int i = threadIdx.x; i < last; i += 256) add(full + (long long)J * T2 + i);
    double s = s0 + s1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = (threadIdx.x < (blockDim.x >> 5)) ? part[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) gamma[P] = s;
    }
}

// Jp[x] = sum_P gamma_P B[P][x]; each thread owns two adjacent columns, blockIdx.y splits P (padding is not
// written)
__global__ void __launch_bounds__(256) coulomb_kernel(const double* __restrict__ B, long long row, int naux, int nt,
                                                      int n, const double* __restrict__ gamma, int nsplit,
                                                      double* __restrict__ Jpart) {
    const long long c2 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c2 * 2 >= row) return;
    if (c2 >= (long long)nt * (nt - 1) / 2 * (TS * TS / 2) &&
        (int)(c2 % (TS * TS / 2)) >= (n - TS * (nt - 1)) * (TS / 2))
        return;
    const int s = blockIdx.y;
    const int p0 = (int)((long long)naux * s / nsplit), p1 = (int)((long long)naux * (s + 1) / nsplit);
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
    for (int P = p0; P < p1; ++P) {
        const double2 x = __ldcs(reinterpret_cast<const double2*>(B + (long long)P * row) + c2);
        const double g = gamma[P];
        a0 = fma(g, x.x, a0);
        a1 = fma(g, x.y, a1);
    }
    reinterpret_cast<double2*>(Jpart + (long long)s * row)[c2] = make_double2(a0, a1);
}

// J[mu][nu] = the partial sums' total, both triangles: a CTA per 8 rows of a tile pair, the mirrored part through
// shared memory
__global__ void __launch_bounds__(256) coulomb_sum_kernel(const double* __restrict__ part, int nsplit, long long row,
                                                          int n, double* __restrict__ J) {
    __shared__ double t[8][TS + 1];
    const int tp = blockIdx.x >> 3, r0 = (blockIdx.x & 7) * 8;
    int I = (int)((sqrt(8.0 * tp + 1.0) - 1.0) * 0.5);
    while ((I + 1) * (I + 2) / 2 <= tp) ++I;
    while (I * (I + 1) / 2 > tp) --I;
    const int Jt = tp - I * (I + 1) / 2;
    if (I * TS + r0 >= n) return;
    for (int e = threadIdx.x; e < 8 * TS; e += 256) {
        const int r = e / TS, c = e % TS, mu = I * TS + r0 + r, nu = Jt * TS + c;
        double s = 0.0;
        if (mu < n && nu < n) {
            const double* p = part + (long long)tp * TS * TS + (r0 + r) * TS + c;
            for (int q = 0; q < nsplit; ++q) s += p[q * row];
            J[(long long)mu * n + nu] = s;
        }
        t[r][c] = s;
    }
    if (I == Jt) return;                                 // a diagonal tile is stored whole
    __syncthreads();
    for (int e = threadIdx.x; e < 8 * TS; e += 256) {
        const int r = e & 7, c = e >> 3, mu = I * TS + r0 + r, nu = Jt * TS + c;
        if (mu < n && nu < n) J[(long long)nu * n + mu] = t[r][c];
    }
}

constexpr int J_SPLIT = 8;

}  // namespace

// partial sums of the FP64 exchange over ranges of the auxiliary index
int k_splits(const df_handle* h) {
    const int tiles = h->pk.nt * (h->pk.nt + 1) / 2;
    int s = (4 * 152 + tiles - 1) / tiles;
    return std::max(1, std::min(s, std::max(1, h->naux / 4)));
}

void ensure_jk_buffers(df_handle* h, int nocc) {
    const Packing& pk = h->pk;
    if (!h->Dw.p) {
        h->Dw.alloc(pk.row);
        h->gamma.alloc(h->naux);
        h->Jp.alloc(pk.row * J_SPLIT);
        h->dD.alloc((size_t)h->n * h->n);
        h->dJ.alloc((size_t)h->n * h->n);
        h->dK.alloc((size_t)h->n * h->n);
        h->Kpart.alloc((size_t)k_splits(h) * h->n * h->n);
        // tile list for the exchange contraction: lower tile pairs
        std::vector<int2> tiles;
        for (int I = 0; I < pk.nt; ++I)
            for (int J = 0; J <= I; ++J) tiles.push_back(make_int2(I, J));
        h->ktiles.alloc(tiles.size());
        DF_CUDA(cudaMemcpyAsync(h->ktiles.p, tiles.data(), tiles.size() * sizeof(int2), cudaMemcpyHostToDevice, h->stream));
    }
    if (nocc > h->nocc_alloc) {
        h->dC.alloc((size_t)h->n * nocc);
        h->nocc_alloc = nocc;
    }
}

void coulomb_fp64(df_handle* h, const double* dD, double* dJ) {
    const Packing& pk = h->pk;
    cudaStream_t s = h->stream;
    PhaseTimer& t = h->timer;
    t.on = h->sync_timing;
    pack_density_kernel<<<dim3(pk.nt, pk.nt), 256, 0, s>>>(dD, h->n, h->Dw.p);
    DF_CHECK_LAUNCH();
    t.mark(PhaseTimer::COULOMB, s);
    gamma_kernel<<<h->naux, 256, 0, s>>>(h->B.p, pk.row, pk.nt, h->n, h->Dw.p, h->gamma.p);
    DF_CHECK_LAUNCH();
    t.mark(PhaseTimer::COULOMB + 1, s);
    const long long c2 = pk.row / 2;
    coulomb_kernel<<<dim3((unsigned)((c2 + 255) / 256), J_SPLIT), 256, 0, s>>>(h->B.p, pk.row, h->naux, pk.nt, h->n,
                                                                             h->gamma.p, J_SPLIT, h->Jp.p);
    DF_CHECK_LAUNCH();
    t.mark(PhaseTimer::COULOMB + 2, s);
    coulomb_sum_kernel<<<(unsigned)(8 * pk.ntp), 256, 0, s>>>(h->Jp.p, J_SPLIT, pk.row, h->n, dJ);
    DF_CHECK_LAUNCH();
}

void exchange_fp64(df_handle* h, const double* dC, int nocc, double* dK) {
    const Packing& pk = h->pk;
    cudaStream_t s = h->stream;
    PhaseTimer& t = h->timer;
    t.on = h->sync_timing;
    t.mark(PhaseTimer::EXCHANGE, s);
    h->exchange_launches = 3;   // Y transform, K contraction, K reduction
    // Y (n rows of naux nocc doubles): the split exchange's Y buffer when the handle has one large enough (8
    // bytes per element as well; both run in order on the handle's stream), else its own, allocated on first use
    const long long KL = (long long)h->naux * nocc;
    const size_t ny = (size_t)KL * h->n;
    double* Y = split_y_buffer(h, (long long)ny);
    if (!Y) {
        if (h->Y.n < ny) h->Y.alloc(ny);
        Y = h->Y.p;
    }
    y_transform_fp64(s, h->B.p, pk.row, h->n, h->naux, dC, nocc, Y);
    t.mark(PhaseTimer::EXCHANGE + 1, s);
    k_syrk_fp64(s, Y, h->n, h->naux, nocc, k_splits(h), h->Kpart.p, dK);
    t.mark(PhaseTimer::EXCHANGE + 2, s);
}

// the phase times of the build whose work is complete on the device (its marks are cleared)
void collect_timings(df_handle* h) {
    PhaseTimer& t = h->timer;
    constexpr int C = PhaseTimer::COULOMB, E = PhaseTimer::EXCHANGE, S = PhaseTimer::SPLIT;
    auto take = [&](int slot, int a, int b) {
        if (t.has(a) && t.has(b)) h->timings_ms[slot] = t.ms(a, b);
    };
    take(4, C, C + 1);
    take(5, C + 1, C + 2);
    take(6, E, E + 1);
    take(7, E + 1, E + 2);
    if (t.has(S + 5)) {
        take(8, S, S + 5);
        take(9, S + 1, S + 2);      // Y = B C (split)
        take(10, S + 3, S + 4);     // K contraction (split)
        h->timings_ms[11] = h->timings_ms[8] - h->timings_ms[9] - h->timings_ms[10];   // slicing, reduce
    }
    t.marked = 0;
}

void jk_fp64(df_handle* h, const double* dD, const double* dC, int nocc, double* dJ, double* dK) {
    ensure_jk_buffers(h, nocc);
    coulomb_fp64(h, dD, dJ);
    exchange_fp64(h, dC, nocc, dK);
}

void unpack_rows(df_handle* h, const double* packed, int p0, int count, double* dout) {
    const long long nn = (long long)h->n * h->n;
    for (int r = 0; r < count; r += 65535) {
        const int c = std::min(65535, count - r);
        unpack_kernel<<<dim3((unsigned)((nn + 255) / 256), c), 256, 0, h->stream>>>(packed + (long long)(p0 + r) * h->pk.row,
                                                                                   h->pk.row, h->n, dout + r * nn);
        DF_CHECK_LAUNCH();
    }
}

double elapsed_ms(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    DF_CUDA(cudaEventElapsedTime(&ms, a, b));
    return ms;
}

}  // namespace dfhf

namespace dfhf {

// The Coulomb build with every scratch buffer supplied by the caller and no split of the auxiliary
// sum: Dw and Jp hold `row` doubles each, gamma `naux`. Each scratch element is written before it
// is read within the call, so nothing has to start at zero. No allocation, no synchronisation.
// Loads the Coulomb kernels on the current device now (under lazy module loading they would otherwise be
// loaded, and their code placed in device memory, at their first launch)
void coulomb_kernels_load() {
    cudaFuncAttributes a;
    DF_CUDA(cudaFuncGetAttributes(&a, pack_density_kernel));
    DF_CUDA(cudaFuncGetAttributes(&a, gamma_kernel));
    DF_CUDA(cudaFuncGetAttributes(&a, coulomb_kernel));
    DF_CUDA(cudaFuncGetAttributes(&a, unpack_kernel));
}

void coulomb_with_scratch(cudaStream_t s, const double* B, const Packing& pk, int naux, int n, const double* dD,
                          double* dJ, double* Dw, double* gamma, double* Jp) {
    pack_density_kernel<<<dim3(pk.nt, pk.nt), 256, 0, s>>>(dD, n, Dw);
    DF_CHECK_LAUNCH();
    gamma_kernel<<<naux, 256, 0, s>>>(B, pk.row, pk.nt, n, Dw, gamma);
    DF_CHECK_LAUNCH();
    const long long c2 = pk.row / 2;
    coulomb_kernel<<<dim3((unsigned)((c2 + 255) / 256), 1), 256, 0, s>>>(B, pk.row, naux, pk.nt, n, gamma, 1, Jp);
    DF_CHECK_LAUNCH();
    const long long nn = (long long)n * n;
    unpack_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(Jp, pk.row, n, dJ);
    DF_CHECK_LAUNCH();
}

}  // namespace dfhf
