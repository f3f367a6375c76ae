// Symmetric eigenproblem of small matrices in FP64: cyclic Jacobi (Jacobi 1846; the parallel order of Brent and
// Luk, SIAM J. Sci. Stat. Comput. 6, 69 (1985)) as one cooperative kernel.
//
// cuSOLVER's dsyevd takes 4.0 ms for n = 100 (a hundred-odd dependent launches); an SCF of two waters spent three
// quarters of its time there (93.6 ms, now 33.9; a solve 1.14 ms on average). Here a step of the round-robin order
// rotates n / 2 disjoint pairs at once: every CTA forms all rotations of the step itself from the current matrix,
// the 2 x 2 blocks (pair x pair, half of them by symmetry) and the eigenvectors' elements are dealt to the threads,
// the new matrix goes to a second buffer, and a grid barrier ends the step. A step is a few L2 latencies and the
// barrier, 3.4 us at n = 100; a sweep has n - 1 steps, and a matrix that is nearly diagonal (an SCF's Fock matrix in
// the last iteration's orbitals) needs three or four. The angle is taken in FP32 (it only has to make the element
// small), the rotation is orthogonal to FP64 rounding: c = (1 + t^2)^(-1/2) by one third-order step from the FP32
// value, s = t c.
#include "common.cuh"
#include "grid_barrier.cuh"

namespace dfhf {

namespace {

constexpr int JT = 128;             // threads per CTA
constexpr int MAXP = (JACOBI_MAX + 1) / 2;
static_assert(MAXP <= JT, "a thread per pair");
constexpr int MAX_SWEEPS = 40;
constexpr double OFF_TOL = 4e-15;   // largest off-diagonal element left, relative to the largest diagonal one

struct JacobiArgs {
    int n;
    const double* A;                // row-major, the lower triangle is read
    double *M0, *M1, *V;            // work: n x n each
    double* out;                    // row j: eigenvector of w[j]
    double* w;                      // ascending
    unsigned* count;                // barrier arrivals
    int* top;                       // high word of the largest magnitude in A, zero at the start
    int* err;
    int* info;                      // 0, or 1 if MAX_SWEEPS did not suffice
    long long wait;                 // budget of a barrier's wait
};

__device__ __forceinline__ int high_word(double v) { return __double2hiint(v) & 0x7fffffff; }

__global__ void __launch_bounds__(JT) jacobi_kernel(const JacobiArgs a) {
    __shared__ double sc[MAXP], ss[MAXP];
    __shared__ int red_off[JT / 32], red_max[JT / 32];
    __shared__ int rank[JACOBI_MAX];
    const int n = a.n, N = n + (n & 1), m = N / 2, tid = threadIdx.x;
    const int gt = blockIdx.x * JT + tid, gn = gridDim.x * JT;
    unsigned target = 0;

    int top = 0;
    for (int e = gt; e < n * n; e += gn) {
        const int i = e / n, j = e % n;
        const double v = a.A[i >= j ? e : j * n + i];
        a.M0[e] = v;
        a.V[e] = i == j ? 1.0 : 0.0;
        top = max(top, high_word(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((tid & 31) == 0) atomicMax(a.top, top);
    if (!grid_barrier(a.count, a.err, target, a.wait)) return;
    // a matrix whose magnitude is far from 1 (the change of a density between two iterations may be) has its angles'
    // FP32 operands scaled to the range of floats; others are taken as they are
    top = __ldcg(a.top);
    const bool far = top < 0x7ff00000 && abs((top >> 20) - 1023) > 60;
    const double scale = __hiloint2double(max(1, 2046 - (top >> 20)) << 20, 0);

    // this thread's task in every step: one new row (the pair's first or second) of a block (I, J), I >= J, of
    // pair rows and pair columns (and its mirror image), or element tj of the eigenvectors of pair ti. The launch
    // has a thread for each; a warp's multiply-adds cost 64 clocks each, so the tasks are short.
    const int nb = m * (m + 1), N1 = N - 1;
    int ti = 0, tj = 0;
    const bool block = gt < nb, vector = !block && gt < nb + m * n, second = block && gt >= nb / 2;
    if (block) {
        const int k = second ? gt - nb / 2 : gt;
        ti = (int)((sqrtf(8.f * k + 1.f) - 1.f) * 0.5f);
        while ((ti + 1) * (ti + 2) / 2 <= k) ++ti;
        while (ti * (ti + 1) / 2 > k) --ti;
        tj = k - ti * (ti + 1) / 2;
    } else if (vector) {
        ti = (gt - nb) / n;
        tj = (gt - nb) % n;
    }
    // the round-robin's pair i of step t, p < q; index n, if any, is a dummy
    auto pair_of = [&](int i, int t, int& p, int& q) {
        int x = t + i, y = t - i;
        if (x >= N1) x -= N1;
        if (y < 0) y += N1;
        if (i == 0) x = N1;
        p = min(x, y);
        q = max(x, y);
    };
    double *cur = a.M0, *nxt = a.M1;
    bool done = n == 1 || top == 0;
    for (int sweep = 0; sweep < MAX_SWEEPS && !done; ++sweep) {
        int off = 0, big = 0;                        // largest magnitudes of the sweep, as high words of doubles
        for (int t = 0; t < N1; ++t) {
            // the task's operands, requested before the rotations are formed
            int p1, q1, p2 = 0, q2 = 0;
            double x00 = 0.0, x01 = 0.0, x10 = 0.0, x11 = 0.0;
            pair_of(ti, t, p1, q1);
            if (block) {
                pair_of(tj, t, p2, q2);
                x00 = __ldcg(cur + p1 * n + p2);
                if (q2 < n) x01 = __ldcg(cur + p1 * n + q2);
                if (q1 < n) x10 = __ldcg(cur + q1 * n + p2);
                if (q1 < n && q2 < n) x11 = __ldcg(cur + q1 * n + q2);
            } else if (vector && q1 < n) {
                x00 = __ldcg(a.V + p1 * n + tj);
                x10 = __ldcg(a.V + q1 * n + tj);
            }
            // rotations of the step's pairs (the same in every CTA)
            if (tid < m) {
                int p, q;
                pair_of(tid, t, p, q);
                double c = 1.0, s = 0.0;
                if (q < n) {
                    const double app = __ldcg(cur + p * n + p), aqq = __ldcg(cur + q * n + q), apq = __ldcg(cur + p * n + q);
                    off = max(off, high_word(apq));
                    big = max(big, max(high_word(app), high_word(aqq)));
                    double gap = aqq - app, el = apq;
                    if (far) {
                        gap *= scale;
                        el *= scale;
                    }
                    const float f = (float)el;
                    if (f != 0.f) {
                        const float th = (float)gap / (2.f * f);
                        const double tt = (double)copysignf(1.f / (fabsf(th) + sqrtf(fmaf(th, th, 1.f))), th);
                        const double x = fma(tt, tt, 1.0);
                        const double y = (double)rsqrtf((float)x);
                        const double e = fma(-x * y, y, 1.0);
                        c = fma(y * e, fma(0.375, e, 0.5), y);
                        s = tt * c;
                    }
                }
                sc[tid] = c;
                ss[tid] = s;
            }
            __syncthreads();
            const double c1 = sc[ti], s1 = ss[ti];
            if (block) {
                const double c2 = sc[tj], s2 = ss[tj];
                const bool r2 = q2 < n;
                // the row of the block rotated by pair I, then by pair J
                const double u = second ? s1 : c1, v = second ? c1 : -s1;
                const double y0 = fma(u, x00, v * x10), y1 = fma(u, x01, v * x11);
                const double z0 = fma(c2, y0, -s2 * y1), z1 = fma(s2, y0, c2 * y1);
                const int r = second ? q1 : p1;
                if (r < n) {
                    if (ti == tj) {
                        // a diagonal block's off-diagonal element comes from its second row alone
                        if (!second) {
                            nxt[r * n + p2] = z0;
                        } else {
                            nxt[r * n + p2] = z0;
                            nxt[p2 * n + r] = z0;
                            nxt[r * n + q2] = z1;
                        }
                    } else {
                        nxt[r * n + p2] = z0;
                        nxt[p2 * n + r] = z0;
                        if (r2) {
                            nxt[r * n + q2] = z1;
                            nxt[q2 * n + r] = z1;
                        }
                    }
                }
            } else if (vector && q1 < n && s1 != 0.0) {
                a.V[p1 * n + tj] = fma(c1, x00, -s1 * x10);
                a.V[q1 * n + tj] = fma(s1, x00, c1 * x10);
            }
            if (!grid_barrier(a.count, a.err, target, a.wait)) return;
            double* x = cur;
            cur = nxt;
            nxt = x;
        }
        // largest off-diagonal and diagonal elements met: every CTA saw the same ones
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            off = max(off, __shfl_xor_sync(0xffffffffu, off, o));
            big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
        }
        if ((tid & 31) == 0) {
            red_off[tid >> 5] = off;
            red_max[tid >> 5] = big;
        }
        __syncthreads();
        off = big = 0;
        for (int k = 0; k < JT / 32; ++k) {
            off = max(off, red_off[k]);
            big = max(big, red_max[k]);
        }
        __syncthreads();
        // near the end (the convergence is quadratic) the elements themselves are looked at, which spares the sweep
        // that would only find them small
        const double diag = __hiloint2double(big, 0);
        if (off && __hiloint2double(off, -1) > 1e-4 * diag) continue;
        int left = 0;
        for (int e = tid; e < n * n; e += JT)
            if (e / n != e % n) left = max(left, high_word(__ldcg(cur + e)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) left = max(left, __shfl_xor_sync(0xffffffffu, left, o));
        if ((tid & 31) == 0) red_off[tid >> 5] = left;
        __syncthreads();
        for (int k = 0; k < JT / 32; ++k) left = max(left, red_off[k]);
        __syncthreads();
        done = !left || __hiloint2double(left, -1) <= OFF_TOL * diag;
    }
    // ascending order
    for (int i = tid; i < n; i += JT) {
        const double d = __ldcg(cur + i * n + i);
        int r = 0;
        for (int j = 0; j < n; ++j) {
            const double e = __ldcg(cur + j * n + j);
            r += (e < d || (e == d && j < i)) ? 1 : 0;
        }
        rank[i] = r;
        if (blockIdx.x == 0) a.w[r] = d;
    }
    __syncthreads();
    for (int e = gt; e < n * n; e += gn) a.out[rank[e / n] * n + e % n] = __ldcg(a.V + e);
    if (gt == 0) *a.info = done ? 0 : 1;
}

}  // namespace

size_t jacobi_work_doubles(int n) { return 3 * (size_t)n * n + 1; }

// eigenvalues (ascending, w) and eigenvectors (row j of out) of the symmetric n x n matrix A (row-major, lower
// triangle read), 1 <= n <= JACOBI_MAX; work: jacobi_work_doubles(n). out may be A. info (device) as JacobiArgs; a
// barrier that expires leaves DF_E_TIMEOUT there.
void jacobi_eig(cudaStream_t s, int n, const double* A, double* w, double* out, double* work, int* info) {
    const size_t nn = (size_t)n * n;
    unsigned* sync = reinterpret_cast<unsigned*>(work + 3 * nn);   // arrivals | largest magnitude
    DF_CUDA(cudaMemsetAsync(sync, 0, 2 * sizeof(unsigned), s));
    DF_CUDA(cudaMemsetAsync(info, 0, sizeof(int), s));
    JacobiArgs a{n,    A,    work, work + nn, work + 2 * nn, out, w, sync, reinterpret_cast<int*>(sync + 1),
                 info, info, grid_wait_cycles()};
    const int m = (n + 1) / 2, tasks = m * (m + 1) + m * n;
    const int grid = (tasks + JT - 1) / JT;   // 236 at n = 200: two CTAs per SM
    void* args[] = {&a};
    DF_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(grid), dim3(JT), args, 0, s));
}

}  // namespace dfhf
