// Metric whitening B = L^-1 (Q|mu nu) (paper eq. 1, third form, with M' = L^-1) on the tcgen05 tensor
// cores by Ozaki splitting.
//
// GB300's FP64 rate is ~1 TFLOP/s; the whitening is naux^2 npair / 2 multiply-adds (24.6 TFLOP at 32
// waters). Each row of L^-1 is scaled by its power of two and written as 7 BF16 digit slices, each pair
// column of the three-index tensor likewise (with its own power of two, transposed so the auxiliary
// index is contiguous); the 28 slice pairs with s + t <= 8 are multiplied on the tensor cores in exact
// FP32 chunks and summed in float-float (ozaki_tc_kernel, whitening mode). With 7 slices the result
// differs from an FP64 product L^-1 A by ~3e-10 of max|B| on the 8-water cluster, well inside the
// ~kappa(L) eps |B| by which two correct FP64 whitenings differ (8e-9 there).
//
// The columns are the distinct pairs mu >= nu of the packed rows: the padding of the last tiles (zero) and the
// mirror halves of the diagonal tiles (written beside their originals) are not whitened; at n = 590 they are a
// quarter of the packed elements. The columns are processed in chunks whose transposed slices fit a bounded
// buffer; when the unwhitened tensor is not kept, each chunk's result overwrites the chunk's own columns in place.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <map>
#include <mutex>

#include "common.cuh"
#include "ozaki.cuh"

namespace dfhf {

void whiten_tc(cudaStream_t s, int N, const __nv_bfloat16* Ls, const int* eL, const __nv_bfloat16* At, const int* eA,
               int naux, int kp, int ncols, const int2* pos, double* out, long long ldo, int* err);

namespace {

typedef __nv_bfloat16 bf16;
constexpr int WS = 7;   // slices

// Output tile width of the whitening kernel (64, or 32 with two CTAs per SM), chosen per size bucket
// (naux / 512) by timing the first two column chunks of the first whitening in that bucket with one
// width each: the candidates run on real work, so the choice costs nothing extra.
std::mutex g_wmu;
std::map<int, int> g_wtile;

// L^-1 (naux x naux, row-major, lower) -> Ls[s][P][Q] (kp columns, zero beyond naux), eL[P]
__global__ void __launch_bounds__(256) slice_rows_kernel(const double* __restrict__ L, int naux, int kp,
                                                         bf16* __restrict__ Ls, long long sstr, int* __restrict__ eL) {
    const int P = blockIdx.x;
    const double* row = L + (long long)P * naux;
    double mx = 0.0;
    for (int q = threadIdx.x; q < naux; q += blockDim.x) mx = fmax(mx, fabs(row[q]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ double red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = fmax(mx, red[w]);
    int e = 0;
    if (mx > 0.0) frexp(mx, &e);   // |row| * 2^-e < 1
    if (threadIdx.x == 0) eL[P] = e;
    bf16* o = Ls + (long long)P * kp;
    for (int q = threadIdx.x; q < kp; q += blockDim.x) split_pow2<WS>(q < naux ? row[q] : 0.0, e, o + q, sstr);
}

// positions of column c (the pair mu >= nu) in a packed row: its own and its mirror's in a diagonal tile (-1: none);
// columns beyond the last pair have none
__global__ void __launch_bounds__(256) column_positions_kernel(long long npair, long long count, int2* __restrict__ pos) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= count) return;
    int2 p = make_int2(-1, -1);
    if (c < npair) {
        int mu = (int)((sqrt(8.0 * (double)c + 1.0) - 1.0) * 0.5);
        while ((long long)(mu + 1) * (mu + 2) / 2 <= c) ++mu;
        while ((long long)mu * (mu + 1) / 2 > c) --mu;
        const int nu = (int)(c - (long long)mu * (mu + 1) / 2);
        p.x = (int)packed_index(mu, nu);
        if (mu / TS == nu / TS && mu != nu) p.y = (int)packed_index(nu, mu);
    }
    pos[c] = p;
}

// cmax[c] = max_Q |A[Q][column c]| as the bits of a non-negative double, over the rows of blockIdx.y; pos at the
// chunk's first column
__global__ void __launch_bounds__(256) col_max_kernel(const double* __restrict__ A, long long ld, int naux,
                                                      const int2* __restrict__ pos, int nc,
                                                      unsigned long long* __restrict__ cmax) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const int p = pos[c].x;
    if (p < 0) return;
    const int q0 = (int)((long long)naux * blockIdx.y / gridDim.y), q1 = (int)((long long)naux * (blockIdx.y + 1) / gridDim.y);
    unsigned long long m = 0;
#pragma unroll 8
    for (int q = q0; q < q1; ++q) m = max(m, abs_bits(A[(long long)q * ld + p]));
    atomicMax(cmax + c, m);
}

// eA[c] = e with max 2^-e < 1 (0 for a zero column)
__global__ void col_exponent_kernel(const unsigned long long* __restrict__ cmax, int nc, int* __restrict__ eA) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const double mx = __longlong_as_double((long long)cmax[c]);
    int e = 0;
    if (mx > 0.0) frexp(mx, &e);
    eA[c] = e;
}

// At[s][c][Q] (kp per column, zero beyond naux) = slices of column c 2^-eA[c]; 64 x 64 tiles transposed through
// shared memory (reads run along the packed row, a warp writes 64 neighbours along Q). n = 590, naux = 1619:
// 2.10 -> 1.39 ms
__global__ void __launch_bounds__(256) slice_cols_kernel(const double* __restrict__ A, long long ld, int naux, int kp,
                                                         const int2* __restrict__ pos, const int* __restrict__ eA,
                                                         bf16* __restrict__ At, long long sstr) {
    __shared__ double tile[64][65];
    const int cb = blockIdx.x * 64, q0 = blockIdx.y * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;   // 64 x 4
    const int p = pos[cb + tx].x;
#pragma unroll 4
    for (int r = ty; r < 64; r += 4) {
        const int q = q0 + r;
        tile[r][tx] = (q < naux && p >= 0) ? A[(long long)q * ld + p] : 0.0;
    }
    __syncthreads();
    const int k = (threadIdx.x & 31) * 2;
    for (int r = threadIdx.x >> 5; r < 64; r += 8) {          // r: column within the tile, k: Q within the tile
        const int c = cb + r, e = __ldg(eA + c);
        split_pow2_pair<WS>(tile[k][r], e, tile[k + 1][r], e, At + (long long)c * kp + q0 + k, sstr);
    }
}

}  // namespace

// B = L^-1 A for the packed tensor A of n orbital functions (naux rows of stride ld). `B` may equal `A` (in place,
// chunk by chunk); else its padding is A's. Scratch: the slices of L^-1 and one chunk of transposed slices.
void whiten_ozaki(cudaStream_t s, int naux, int n, long long ld, const double* Linv, const double* A, double* B) {
    if (ld > 0x7fffffff) throw Error{DF_E_ARG, "whitening supports packed rows of at most 2^31 elements"};
    const long long npair = (long long)n * (n + 1) / 2;
    const long long ncol = (npair + 63) / 64 * 64;
    if (B != A) DF_CUDA(cudaMemsetAsync(B, 0, sizeof(double) * (size_t)naux * ld, s));
    const int kp = (naux + 63) / 64 * 64;
    size_t free_b = 0, total_b = 0;
    DF_CUDA(cudaMemGetInfo(&free_b, &total_b));
    const double col_bytes = (double)WS * kp * 2 + 4;
    // the chunk's transposed slices: at most 8 GB (several molecules may whiten at once)
    const double chunk_bytes = std::min(0.4 * (double)free_b, 8.0e9);
    // columns per chunk: at most 2^19 and what the buffer holds, in chunks of nearly equal size
    const long long most = std::max<long long>(64, (long long)std::min<double>(1LL << 19, chunk_bytes / col_bytes) / 64 * 64);
    const long long chunks = (ncol + most - 1) / most;
    const long long nc = ((ncol + chunks - 1) / chunks + 63) / 64 * 64;
    DevBuf<bf16> Ls, At;
    DevBuf<int> eL, eA, err;
    DevBuf<int2> pos;
    DevBuf<unsigned long long> cmax;
    Ls.alloc((size_t)WS * naux * kp);
    eL.alloc(naux);
    At.alloc((size_t)WS * nc * kp);
    eA.alloc(nc);
    pos.alloc(ncol);
    cmax.alloc(nc);
    err.alloc(1);
    err.zero(s);
    try {
    slice_rows_kernel<<<naux, 256, 0, s>>>(Linv, naux, kp, Ls.p, (long long)naux * kp, eL.p);
    DF_CHECK_LAUNCH();
    column_positions_kernel<<<(unsigned)((ncol + 255) / 256), 256, 0, s>>>(npair, ncol, pos.p);
    DF_CHECK_LAUNCH();
    const int bucket = (naux + 511) / 512;
    int tile = 0;
    {
        std::lock_guard<std::mutex> lock(g_wmu);
        auto it = g_wtile.find(bucket);
        if (it != g_wtile.end()) tile = it->second;
    }
    if (const char* f = std::getenv("DFHF_WHITEN_TILE")) {   // fixes the width (tests compare the two)
        const int t = std::atoi(f);
        if (t == 32 || t == 64) tile = t;
    }
    const bool tune = tile == 0 && chunks >= 3;      // two chunks of the same size to compare
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    if (tune)
        for (auto& e : ev) DF_CUDA(cudaEventCreate(&e));
    int k = 0;
    for (long long c0 = 0; c0 < ncol; c0 += nc, ++k) {
        const int w = (int)std::min<long long>(nc, ncol - c0);
        cmax.zero(s);
        // enough row ranges to fill the GPU
        const int ranges = std::max(1, std::min(naux / 16, (16 * 152 * 256 + w - 1) / w));
        col_max_kernel<<<dim3((w + 255) / 256, ranges), 256, 0, s>>>(A, ld, naux, pos.p + c0, w, cmax.p);
        DF_CHECK_LAUNCH();
        col_exponent_kernel<<<(w + 255) / 256, 256, 0, s>>>(cmax.p, w, eA.p);
        DF_CHECK_LAUNCH();
        slice_cols_kernel<<<dim3(w / 64, kp / 64), 256, 0, s>>>(A, ld, naux, kp, pos.p + c0, eA.p, At.p, (long long)w * kp);
        DF_CHECK_LAUNCH();
        int use = tile ? tile : 64;
        if (tune && k < 2) {
            use = k == 0 ? 64 : 32;
            DF_CUDA(cudaEventRecord(ev[2 * k], s));
        }
        whiten_tc(s, use, Ls.p, eL.p, At.p, eA.p, naux, kp, w, pos.p + c0, B, ld, err.p);
        if (tune && k < 2) DF_CUDA(cudaEventRecord(ev[2 * k + 1], s));
        if (tune && k == 1) {
            DF_CUDA(cudaEventSynchronize(ev[3]));
            tile = elapsed_ms(ev[2], ev[3]) < elapsed_ms(ev[0], ev[1]) ? 32 : 64;
            std::lock_guard<std::mutex> lock(g_wmu);
            g_wtile[bucket] = tile;
        }
    }
    if (tune)
        for (auto& e : ev) cudaEventDestroy(e);
    int herr = 0;
    DF_CUDA(cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    DF_CUDA(cudaStreamSynchronize(s));
    if (herr) throw Error{DF_E_TIMEOUT, "tensor-core whitening kernel timed out waiting on a barrier"};
    } catch (...) {
        cudaStreamSynchronize(s);   // queued kernels finish before the scratch buffers are released
        throw;
    }
}

}  // namespace dfhf
