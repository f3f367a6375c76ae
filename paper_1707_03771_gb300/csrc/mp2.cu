// Density-fitted closed-shell MP2 correlation energy (the paper lists MP2 among the programs on the
// density-fitting utilities, section "Program features"), FP64 on the GPU from the handle's B:
//   * Y_{P,mu i} = sum_nu B_{P,mu nu} C_{nu i} (eq. 1, first form; the FP64 half-transform of the exchange);
//   * B^P_{ia} = sum_mu C_{mu a} Y_{P,mu i} (eq. 1 again, on the second index), one product over all P, stored
//     as T[i][a][P];
//   * for each occupied i, V_{ia,jb} = sum_P B^P_{ia} B^P_{jb} for every j <= i in one product
//     (eq. 2, second form);
//   * E2 = sum_{ij ab} (ia|jb) [2 (ia|jb) - (ib|ja)] / (e_i + e_j - e_a - e_b), every orbital correlated,
//     summed per pair and 32 x 32 tile of (a, b) in one block (fixed order), these added on the host in a
//     fixed order.
#include <cmath>
#include <new>
#include <utility>
#include <vector>

#include "common.cuh"

namespace dfhf {

namespace {

constexpr int MT = 32;   // tile of virtual orbitals in the pair energies

// pair energies of occupied i with every j <= i: V holds (ia|jb) at V[a][j nvir + b] (row stride ld). Block
// (t, j) takes the tile pair t = (ta >= tb): with N_ab = 1 / (e_i + e_j - e_a - e_b) the elements ab and ba
// together give N_ab 2 (V_ab^2 + V_ba^2 - V_ab V_ba), so each quotient is taken once; both tiles pass through
// shared memory so that V_ba is read along its rows. pe[j ntp + t] = f x sum, f = 2 for j < i (the pair (j, i)
// too). Bound by the quotients' FP64 work; a block per pair left most SMs idle (0.13 ms a launch at 4 waters).
__global__ void __launch_bounds__(256) pair_energy_kernel(const double* __restrict__ V, long long ld, int i, int nocc,
                                                          int nvir, const double* __restrict__ eps,
                                                          double* __restrict__ pe) {
    __shared__ double P[MT][MT + 1], Q[MT][MT + 1];
    __shared__ double part[8];
    const int t = blockIdx.x, j = blockIdx.y;
    int ta = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
    while ((ta + 1) * (ta + 2) / 2 <= t) ++ta;
    while (ta * (ta + 1) / 2 > t) --ta;
    const int tb = t - ta * (ta + 1) / 2;
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
    const double* v = V + (long long)j * nvir;
    for (int r = r0; r < MT; r += 8) {
        const int a = ta * MT + r, b = tb * MT + c;
        P[r][c] = (a < nvir && b < nvir) ? v[(long long)a * ld + b] : 0.0;          // (ia|jb)
        const int a2 = tb * MT + r, b2 = ta * MT + c;
        Q[r][c] = (a2 < nvir && b2 < nvir) ? v[(long long)a2 * ld + b2] : 0.0;
    }
    __syncthreads();
    const double eij = eps[i] + eps[j];
    const double* ev = eps + nocc;
    double s = 0.0;
    for (int r = r0; r < MT; r += 8) {
        const int a = ta * MT + r, b = tb * MT + c;
        if (a >= nvir || b >= nvir || (ta == tb && b > a)) continue;
        const double x = P[r][c], y = Q[c][r];                                       // V_ab, V_ba
        const double num = (ta == tb && a == b) ? x * x : 2.0 * (x * x + y * y - x * y);
        s += num / (eij - ev[a] - ev[b]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (c == 0) part[r0] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int w = 0; w < 8; ++w) sum += part[w];
        pe[(long long)j * gridDim.x + t] = (j < i ? 2.0 : 1.0) * sum;
    }
}

}  // namespace

double mp2_energy(df_handle* h, const double* C_host, const double* eps_host, int nmo, int nocc) {
    const int n = h->n, naux = h->naux, nvir = nmo - nocc;
    const Packing& pk = h->pk;
    cudaStream_t s = h->stream;
    DevBuf<double> Call, Cocc, Cvir, eps, Y, T, V, pe;
    Call.alloc((size_t)n * nmo);
    Cocc.alloc((size_t)n * nocc);
    Cvir.alloc((size_t)n * nvir);
    eps.alloc(nmo);
    DF_CUDA(cudaMemcpyAsync(Call.p, C_host, sizeof(double) * n * nmo, cudaMemcpyHostToDevice, s));
    DF_CUDA(cudaMemcpyAsync(eps.p, eps_host, sizeof(double) * nmo, cudaMemcpyHostToDevice, s));
    DF_CUDA(cudaMemcpy2DAsync(Cocc.p, sizeof(double) * nocc, Call.p, sizeof(double) * nmo, sizeof(double) * nocc, n,
                              cudaMemcpyDeviceToDevice, s));
    DF_CUDA(cudaMemcpy2DAsync(Cvir.p, sizeof(double) * nvir, Call.p + nocc, sizeof(double) * nmo, sizeof(double) * nvir,
                              n, cudaMemcpyDeviceToDevice, s));
    const long long KL = (long long)naux * nocc;
    Y.alloc((size_t)KL * n);
    y_transform_fp64(s, h->B.p, pk.row, n, naux, Cocc.p, nocc, Y.p);
    // T[i][a][P] = sum_mu Y[mu][P nocc + i] C_vir[mu][a]: rows (P, i), every P in one product
    T.alloc((size_t)KL * nvir);
    dgemm_rows(s, naux, nocc, nvir, n, 1.0, Y.p, nocc, 1, KL, Cvir.p, nvir, 1, 0.0, T.p, 1, (long long)nvir * naux, naux);
    // rows of pair integrals: V = T_i T_{0..i}^T (nvir x (i + 1) nvir) and the pair energies of row i
    const int nt = (nvir + MT - 1) / MT, ntp = nt * (nt + 1) / 2;
    // V in Y's memory, which nothing reads any more (the peak is T and the larger of the two); without a free and an
    // allocation, which cost 0.1 of 9.3 ms at 4 waters
    const size_t nv = (size_t)nvir * nocc * nvir;
    V = std::move(Y);
    if (V.n < nv) V.alloc(nv);
    pe.alloc((size_t)nocc * (nocc + 1) / 2 * ntp);
    for (int i = 0; i < nocc; ++i) {
        const long long ld = (long long)(i + 1) * nvir;
        dgemm_rows(s, 1, nvir, (int)ld, naux, 1.0, T.p + (long long)i * nvir * naux, 0, naux, 1, T.p, 1, naux, 0.0, V.p, 0,
                   ld, 1);
        pair_energy_kernel<<<dim3(ntp, i + 1), 256, 0, s>>>(V.p, ld, i, nocc, nvir, eps.p,
                                                           pe.p + (long long)i * (i + 1) / 2 * ntp);
        DF_CHECK_LAUNCH();
    }
    std::vector<double> host((size_t)nocc * (nocc + 1) / 2 * ntp);
    DF_CUDA(cudaMemcpyAsync(host.data(), pe.p, sizeof(double) * host.size(), cudaMemcpyDeviceToHost, s));
    DF_CUDA(cudaStreamSynchronize(s));
    double e2 = 0.0;
    for (double v : host) e2 += v;
    return e2;
}

}  // namespace dfhf

using namespace dfhf;

extern "C" int df_mp2(df_handle* h, const double* C, const double* eps, int nmo, int nocc, double* e2) {
    if (!h || !C || !eps || !e2 || nocc < 1 || nmo <= nocc || nmo > h->n) return DF_E_ARG;
    if (!h->built || !h->B.p) {
        h->last_error = "df_mp2: B not built";
        return DF_E_STATE;
    }
    try {
        DF_CUDA(cudaSetDevice(h->device));
        *e2 = mp2_energy(h, C, eps, nmo, nocc);
    } catch (const Error& e) {
        h->last_error = e.msg;
        return e.code;
    } catch (const std::bad_alloc&) {
        h->last_error = "df_mp2: host memory exhausted";
        return DF_E_NOMEM;
    }
    return DF_OK;
}
