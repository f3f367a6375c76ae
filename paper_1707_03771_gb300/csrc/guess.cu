// Learned initial guess: a small MLP maps rotation-invariant features of each water's environment to
// the water's 50 x 50 diagonal density block expressed in the molecule's own frame; the blocks are
// rotated to the laboratory frame with real-solid-harmonic rotation matrices (l <= 2) and assembled
// block-diagonally into D0. A second network maps features of each ordered pair of waters within a cutoff
// (the second water's atoms in the first one's frame, atom-pair distances) to the pair's 50 x 50
// off-diagonal block in the first water's frame. The SCF then starts from the natural orbitals of D0
// (scf_run_guess).
// Training (forward, backward, Adam) and BF16 inference run in this file's CUDA kernels.
// The paper has no learned guess; this is the build's design (its quality is a measured outcome).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <random>
#include <vector>

#include "common.cuh"
#include "grid_barrier.cuh"

struct df_mlp {
    int nin = 0, nh = 0, nlayers = 0, nout = 0;   // nlayers hidden layers of width nh
    std::vector<int> dims;                        // nin, nh, ..., nh, nout
    std::vector<long long> woff, boff;            // offsets of W_l (out x in) and b_l in params
    long long nparams = 0;
    dfhf::DevBuf<float> P, G, Mom, Vel;           // parameters, gradients, Adam moments
    dfhf::DevBuf<__nv_bfloat16> Pbf;              // BF16 copy for inference
    int adam_t = 0;
    cudaStream_t stream = nullptr;
};

namespace dfhf {

namespace {

// ---------------------------------------------------------------------------------------------
// FP32 network: forward, backward and Adam steps as one persistent cooperative kernel
//
// A training step is small (16 to 64 samples, 0.46 M parameters: 45 MFLOP) and its layers depend on one
// another, so its time is the number of dependent phases times their latency: as some 25 launches and two row
// copies a sample, a 16-sample step took 0.53 ms, on 4 to 20 CTAs each. Here one launch runs all steps; a
// phase's tiles are dealt to the CTAs and phases are separated by a grid barrier: per step one phase per layer
// forward, one per layer but the first backward, and one more. Parameter updates (the weight gradient of a
// few outputs, consumed by Adam as it is formed) ride along in the phases after the one that last reads the
// weights. Samples are read through the epoch's permutation. A phase is a few L2 latencies long, so tiles are as
// narrow as the CTAs allow (16 rows x 2 to 16 columns), and a tile's whole operands are requested at once.
// Measured: 4 epochs of 17 steps, 57-256-256-256-1275, 16 samples: 37.7 -> 3.9 ms (of a step, about 50 us,
// the eight barriers take 8 and the weight updates with their quotients and square roots 13). Every number is that
// of the same sums and updates done one by one in ascending order, bit for bit.
// ---------------------------------------------------------------------------------------------
constexpr int NT = 256;             // threads of a CTA
constexpr int STAGE_BYTES = 104 * 1024;   // shared memory of a tile's operands (two CTAs fit an SM)
// contraction elements staged at once for tiles of W columns
template <int W>
constexpr int stage_k() {
    return STAGE_BYTES / 4 / (16 + W) / 256 * 256;
}
constexpr int UO = 4;               // outputs of a weight-update task
constexpr int UR = 64;              // rows of a weight-update task staged at once
constexpr int MAX_SHARED_LAYERS = 32;

struct Layer {
    int ni, no;
    long long w, b;                 // offsets of W (no x ni) and the bias in the parameters
    float *Z, *A, *dZ;              // pre- and post-activations, gradient of the pre-activations (rows x no)
};

struct StepArgs {
    const Layer* layers;
    int L, rows, nsteps;
    float *P, *Mom, *Vel;           // parameters, Adam moments
    float* G;                       // not null: the gradient goes here and nothing is updated
    const float *X, *Y;             // samples; Y null: forward only
    const int* perm;                // sample of row r of step t: perm[t rows + r] (null: r)
    float scale;                    // 1 / (rows nout)
    float* part;                    // loss partials, 256 per step
    const float4* c;                // bias corrections per step (adam_update)
    float lr, b1, b2, eps;
    unsigned* count;                // barrier arrivals
    int* err;
    long long wait;                 // budget of a barrier's wait
};

// kz floats of a row into shared memory (those from kc on, or all of a missing row, as zeros), by one warp: 16
// bytes a lane where source and count allow it, else 4
__device__ __forceinline__ void stage_row(float* dst, const float* src, int kc, int kz, int lane) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (kc % 4 == 0 && ((unsigned long long)src & 15) == 0) {
#pragma unroll 4
        for (int k = lane * 4; k < kz; k += 128)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d + k * 4), "l"(src + (k < kc ? k : 0)),
                         "r"(k < kc ? 16 : 0) : "memory");
    } else {
#pragma unroll 4
        for (int k = lane; k < kz; k += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d + k * 4), "l"(src + (k < kc ? k : 0)),
                         "r"(k < kc ? 4 : 0) : "memory");
    }
}

// one tile of 16 rows x W columns of sum_k A[r][k] B(k, n): all threads stage the operands, thread tid < 16 W sums
// element (tid / W, tid % W), one chain of multiply-adds in ascending k whatever the tile. (Dealt to groups of threads
// the sum is shorter by 0.4 us a phase of 256, but its rounding then depends on the tile; and where a
// pre-activation is within rounding of zero the sign decides a sample's gradient, which Adam's first steps turn
// into changes of the size of the learning rate.) A rows through `row` (offset of row r of the tile, or -1); BT:
// B(k, n) = B[n ldb + k], else B[k ldb + n]. (What other CTAs wrote is visible after the barrier's acquire.)
template <int W, bool BT, typename Row>
__device__ float tile_sum(const float* A, Row row, const float* B, long long ldb, int n0, int nn, int K, float* stage) {
    constexpr int KC = stage_k<W>();
    constexpr int KP = KC + 4;      // padded row: 16-byte reads of eight rows fall on distinct banks
    const int tid = threadIdx.x;
    float* As = stage;              // [16][KP]
    float* Bs = stage + 16 * KP;    // BT: [W][KP], else [KC][W]
    float s = 0.f;
    const int n = tid % W, r = tid / W % 16;
    for (int k0 = 0; k0 < K; k0 += KC) {
        const int kc = min(KC, K - k0);
        const int kz = (kc + 3) / 4 * 4;   // elements up to kz are read
        __syncthreads();
        const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
        for (int q = warp; q < 16; q += NT / 32) {
            const long long ar = row(q);
            stage_row(As + q * KP, A + (ar >= 0 ? ar + k0 : 0), ar >= 0 ? kc : 0, kz, lane);
        }
        if (BT) {
            for (int q = warp; q < W; q += NT / 32) {
                const bool in = n0 + q < nn;
                stage_row(Bs + q * KP, B + (in ? (long long)(n0 + q) * ldb + k0 : 0), in ? kc : 0, kz, lane);
            }
        } else {
            const bool in = n0 + n < nn;
            const float* src = B + (long long)k0 * ldb + (in ? n0 + n : 0);
            const unsigned d = (unsigned)__cvta_generic_to_shared(Bs);
#pragma unroll 4
            for (int k = tid / W; k < kz; k += NT / W) {
                const bool ok = in && k < kc;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d + (k * W + n) * 4),
                             "l"(src + (ok ? (long long)k * ldb : 0)), "r"(ok ? 4 : 0) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        if (tid >= 16 * W) continue;
#pragma unroll 8
        for (int k = 0; k < kz; k += 4) {
            const float4 x = *reinterpret_cast<const float4*>(As + r * KP + k);
            float4 y;
            if (BT) y = *reinterpret_cast<const float4*>(Bs + n * KP + k);
            else y = make_float4(Bs[k * W + n], Bs[(k + 1) * W + n], Bs[(k + 2) * W + n], Bs[(k + 3) * W + n]);
            s = fmaf(x.x, y.x, s);
            s = fmaf(x.y, y.y, s);
            s = fmaf(x.z, y.z, s);
            s = fmaf(x.w, y.w, s);
        }
    }
    return s;
}

template <bool BT, typename Row>
__device__ float tile_sum_w(int W, const float* A, Row row, const float* B, long long ldb, int n0, int nn, int K,
                            float* stage) {
    switch (W) {
        case 16: return tile_sum<16, BT>(A, row, B, ldb, n0, nn, K, stage);
        case 8: return tile_sum<8, BT>(A, row, B, ldb, n0, nn, K, stage);
        case 4: return tile_sum<4, BT>(A, row, B, ldb, n0, nn, K, stage);
        default: return tile_sum<2, BT>(A, row, B, ldb, n0, nn, K, stage);
    }
}

// One layer over many rows: out = in W^T + b (rows x no), with ReLU for a hidden layer; 64 x 64 outputs a CTA, 4 x 4 a
// thread, which needs a quarter of the operand reads per multiply-add of the step kernel's 16 x 16 tiles. Each element
// is the same chain of multiply-adds as tile_sum's, so the outputs are equal bit for bit. A forward pass takes it from
// the row count on at which it is the faster one. Device ms of the step kernel / of these, 57-256-256-256-1275 and
// 26-256-256-256-2500: 512 rows 0.064 / 0.112 and 0.095 / 0.114, 1024 0.116 / 0.117 and 0.178 / 0.135, 4096 0.41 / 0.19
// and 0.65 / 0.28, 65536 6.3 / 2.2 and 10.2 / 3.6.
constexpr int LAYER_TILES_ROWS = 1024;
constexpr int FBM = 64, FBN = 64, FBK = 16;
__global__ void __launch_bounds__(256) layer_tiles_kernel(const float* __restrict__ in, int rows, int ni,
                                                          const float* __restrict__ W, const float* __restrict__ b, int no,
                                                          bool relu, float* __restrict__ out) {
    __shared__ float As[FBK][FBM + 1];
    __shared__ float Bs[FBK][FBN + 1];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16, c = tid % FBK;
    const int nt = (no + FBN - 1) / FBN, n0 = (int)(blockIdx.x % nt) * FBN;
    const long long m0 = (long long)(blockIdx.x / nt) * FBM;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < ni; k0 += FBK) {
        const bool ink = k0 + c < ni;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = tid / FBK + 16 * q;
            As[c][r] = ink && m0 + r < rows ? __ldg(in + (m0 + r) * ni + k0 + c) : 0.f;
            Bs[c][r] = ink && n0 + r < no ? __ldg(W + (long long)(n0 + r) * ni + k0 + c) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < FBK; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(As[k][ty + 16 * i], Bs[k][tx + 16 * j], acc[i][j]);
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int n = n0 + tx + 16 * j;
        if (n >= no) continue;
        const float bias = __ldg(b + n);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const long long m = m0 + ty + 16 * i;
            if (m >= rows) continue;
            const float z = acc[i][j] + bias;
            out[m * no + n] = relu ? fmaxf(z, 0.f) : z;
        }
    }
}

// a / b from y = 1 / b correctly rounded: q = a y is within a unit in the last place, and q + (a - q b) y rounds to the
// quotient (Markstein, IBM J. Res. Dev. 34, 111 (1990)) unless b's mantissa is all ones (y = 0 is passed then) or the
// remainder underflows, where |a| is too small to move a parameter
__device__ __forceinline__ float quotient(float a, float b, float y) {
    if (y == 0.f) return a / b;
    const float q = a * y;
    return fmaf(fmaf(-q, b, a), y, q);
}

// Adam (Kingma & Ba 2015) with bias correction: p -= lr (m / c1) / (sqrt(v / c2) + eps), c = (c1, 1 / c1, c2, 1 / c2)
__device__ __forceinline__ void adam_update(float& p, float g, float& m, float& v, float lr, float b1, float b2, float eps,
                                            float4 c) {
    // the roundings are written out: they do not depend on how this code is compiled into the step kernel
    const float mi = __fmaf_rn(1.f - b1, g, __fmul_rn(b1, m));
    const float vi = __fmaf_rn(__fmul_rn(1.f - b2, g), g, __fmul_rn(b2, v));
    m = mi;
    v = vi;
    p = __fsub_rn(p, __fdiv_rn(__fmul_rn(lr, quotient(mi, c.x, c.y)),
                               __fadd_rn(__fsqrt_rn(quotient(vi, c.z, c.w)), eps)));
}

__global__ void __launch_bounds__(NT, 2) mlp_steps_kernel(const StepArgs s) {
    extern __shared__ __align__(16) float stage[];   // STAGE_BYTES
    __shared__ float red[NT];
    // the layers' table and the step's samples: the barrier drops what the L1 cache holds, so a phase would begin
    // with a chain of L2 reads
    __shared__ Layer slayers[MAX_SHARED_LAYERS];
    __shared__ int sperm[NT];
    const int tid = threadIdx.x;
    const Layer* layers = s.L <= MAX_SHARED_LAYERS ? slayers : s.layers;
    if (s.L <= MAX_SHARED_LAYERS)
        for (int l = tid; l < s.L; l += NT) slayers[l] = s.layers[l];
    const int rt = (s.rows + 15) / 16;
    // tile width of a phase with n columns: the narrowest whose tiles each find a CTA
    auto width = [&](int n) {
        int W = 2;
        while (W < 16 && rt * ((n + W - 1) / W) > (int)gridDim.x) W *= 2;
        return W;
    };
    unsigned target = 0;

    for (int step = 0; step < s.nsteps; ++step) {
        const int* perm = s.perm ? s.perm + (long long)step * s.rows : nullptr;
        const float4 c = s.c ? s.c[step] : make_float4(1.f, 1.f, 1.f, 1.f);
        __syncthreads();   // the last step's samples are no longer read
        if (tid < s.rows) sperm[tid] = perm ? __ldg(perm + tid) : tid;
        __syncthreads();
        auto sample = [&](int r) { return r < NT ? sperm[r] : (perm ? __ldg(perm + r) : r); };

        // forward: Z = in W^T + b, A = relu(Z) but for the last layer, whose tiles also give
        // dY = 2 (Z - Y) / (rows nout)
        for (int l = 0; l < s.L; ++l) {
            const Layer y = layers[l];
            const float* in = l == 0 ? s.X : layers[l - 1].A;
            const int W = width(y.no), nt = (y.no + W - 1) / W;
            for (int t = blockIdx.x; t < rt * nt; t += gridDim.x) {
                const int r0 = t / nt * 16, n0 = t % nt * W;
                auto row = [&](int r) {
                    return r0 + r < s.rows ? (long long)(l == 0 ? sample(r0 + r) : r0 + r) * y.ni : -1LL;
                };
                const int r = r0 + tid / W, n = n0 + tid % W;
                const bool mine = tid < 16 * W && r < s.rows && n < y.no;
                const float bias = mine ? __ldcg(s.P + y.b + n) : 0.f;
                const float goal = mine && l == s.L - 1 && s.Y ? __ldg(s.Y + (long long)sample(r) * y.no + n) : 0.f;
                const float sum = tile_sum_w<true>(W, in, row, s.P + y.w, y.ni, n0, y.no, y.ni, stage);
                if (mine) {
                    const long long at = (long long)r * y.no + n;
                    const float z = sum + bias;
                    y.Z[at] = z;
                    y.A[at] = l < s.L - 1 ? fmaxf(z, 0.f) : z;
                    if (l == s.L - 1 && s.Y) {
                        const float d = z - goal;
                        y.dZ[at] = 2.f * d * s.scale;
                    }
                }
            }
            if (!s.Y && l == s.L - 1) continue;
            if (!grid_barrier(s.count, s.err, target, s.wait)) return;
        }
        if (!s.Y) continue;

        // weight and bias gradients of UO outputs of layer l over 256 inputs at a time (task t), each consumed
        // at once: dW[o][i] = sum_r dZ[r][o] in[r][i], db[o] = sum_r dZ[r][o]; the parameters and moments are
        // requested before the sums
        auto update = [&](int l, int t) {
            const Layer y = layers[l];
            const float* in = l == 0 ? s.X : layers[l - 1].A;
            const int ni = y.ni, no = y.no, it = (ni + NT - 1) / NT;
            const int o0 = t / it * UO, i = t % it * NT + tid;
            const bool bias = t % it == 0 && tid < UO && o0 + tid < no;
            float g[UO], p[UO], m[UO], v[UO], gb = 0.f;
#pragma unroll
            for (int q = 0; q < UO; ++q) {
                g[q] = p[q] = m[q] = v[q] = 0.f;
                if (!s.G && i < ni && o0 + q < no) {
                    const long long at = y.w + (long long)(o0 + q) * ni + i;
                    p[q] = __ldcg(s.P + at);
                    m[q] = __ldcg(s.Mom + at);
                    v[q] = __ldcg(s.Vel + at);
                }
            }
            for (int r0 = 0; r0 < s.rows; r0 += UR) {
                const int nr = min(UR, s.rows - r0);
                __syncthreads();
                {
                    const int r = tid / UO, q = tid % UO;        // UR x UO = 256 elements of dZ
                    red[tid] = (r < nr && o0 + q < no) ? __ldcg(y.dZ + (long long)(r0 + r) * no + o0 + q) : 0.f;
                }
                __syncthreads();
                if (i < ni)
#pragma unroll 16
                    for (int r = 0; r < nr; ++r) {
                        const float x = __ldcg(in + (long long)(l == 0 ? sample(r0 + r) : r0 + r) * ni + i);
#pragma unroll
                        for (int q = 0; q < UO; ++q) g[q] = fmaf(red[r * UO + q], x, g[q]);
                    }
                if (bias)
                    for (int r = 0; r < nr; ++r) gb += red[r * UO + tid];
            }
            if (i < ni)
#pragma unroll
                for (int q = 0; q < UO; ++q)
                    if (o0 + q < no) {
                        const long long at = y.w + (long long)(o0 + q) * ni + i;
                        if (s.G) {
                            s.G[at] = g[q];
                        } else {
                            adam_update(p[q], g[q], m[q], v[q], s.lr, s.b1, s.b2, s.eps, c);
                            s.P[at] = p[q];
                            s.Mom[at] = m[q];
                            s.Vel[at] = v[q];
                        }
                    }
            if (bias) {
                const long long at = y.b + o0 + tid;
                if (s.G) {
                    s.G[at] = gb;
                } else {
                    float pb = __ldcg(s.P + at), mb = __ldcg(s.Mom + at), vb = __ldcg(s.Vel + at);
                    adam_update(pb, gb, mb, vb, s.lr, s.b1, s.b2, s.eps, c);
                    s.P[at] = pb;
                    s.Mom[at] = mb;
                    s.Vel[at] = vb;
                }
            }
        };
        static_assert(UR * UO == NT, "one staged element per thread");
        auto update_tasks = [&](int l) {
            const Layer y = layers[l];
            return (y.no + UO - 1) / UO * ((y.ni + NT - 1) / NT);
        };
        // block q of 256 of the loss: thread partials strided by 65536, then a tree
        auto loss_block = [&](int q) {
            const Layer y = layers[s.L - 1];
            const long long len = (long long)s.rows * y.no;
            float sum = 0.f;
            for (long long i = (long long)q * NT + tid; i < len; i += 256LL * NT) {
                const int r = (int)(i / y.no);
                const float d = __ldcg(y.A + i) - s.Y[(long long)sample(r) * y.no + (i - (long long)r * y.no)];
                sum += d * d;
            }
            __syncthreads();
            red[tid] = sum;
            __syncthreads();
            for (int o = NT / 2; o > 0; o >>= 1) {
                if (tid < o) red[tid] += red[tid + o];
                __syncthreads();
            }
            if (tid == 0) s.part[(long long)step * 256 + q] = red[0] * s.scale;
        };

        // blocks beyond the outputs hold zero from the start
        const int loss_blocks = (int)min(256LL, ((long long)s.rows * layers[s.L - 1].no + NT - 1) / NT);

        // backward phase l: the gradient of the layer below, dZ_{l-1} = (dZ_l W_l) relu'(Z_{l-1}); beside it the
        // updates of layer l + 1 (whose weights the phase before read last), or the loss
        for (int l = s.L - 1; l >= 0; --l) {
            const Layer y = layers[l];
            const int W = width(y.ni), nt = (y.ni + W - 1) / W;
            const int below = l > 0 ? rt * nt : 0;
            const int above = l == s.L - 1 ? loss_blocks : update_tasks(l + 1);
            const int own = l == 0 ? update_tasks(0) : 0;
            for (int t = blockIdx.x; t < below + above + own; t += gridDim.x) {
                if (t < below) {
                    const Layer x = layers[l - 1];
                    const int r0 = t / nt * 16, n0 = t % nt * W;
                    auto row = [&](int r) { return r0 + r < s.rows ? (long long)(r0 + r) * y.no : -1LL; };
                    const int r = r0 + tid / W, n = n0 + tid % W;
                    const bool mine = tid < 16 * W && r < s.rows && n < y.ni;
                    const long long at = (long long)r * y.ni + n;
                    const float z = mine ? __ldcg(x.Z + at) : 0.f;
                    const float sum = tile_sum_w<false>(W, y.dZ, row, s.P + y.w, y.ni, n0, y.ni, y.no, stage);
                    if (mine) x.dZ[at] = z <= 0.f ? 0.f : sum;
                } else if (t < below + above) {
                    if (l == s.L - 1) loss_block(t - below);
                    else update(l + 1, t - below);
                } else {
                    update(0, t - below - above);
                }
            }
            if (!grid_barrier(s.count, s.err, target, s.wait)) return;
        }
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ x, long long n, __nv_bfloat16* __restrict__ y) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = __float2bfloat16_rn(x[i]);
}

// BF16 inference layer: out[r][o] = act(sum_i in[r][i] W[o][i] + b[o]) with BF16 inputs and weights,
// FP32 accumulation; one warp per output element (inputs re-rounded to BF16 between layers)
__global__ void bf16_layer_kernel(const __nv_bfloat16* __restrict__ in, int rows, int nin,
                                  const __nv_bfloat16* __restrict__ W, const __nv_bfloat16* __restrict__ b, int nout,
                                  bool relu, __nv_bfloat16* __restrict__ out_bf, float* __restrict__ out_f) {
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (long long)rows * nout) return;
    const int r = (int)(w / nout), o = (int)(w % nout);
    float s = 0.f;
    for (int i = lane; i < nin; i += 32)
        s = fmaf(__bfloat162float(in[(long long)r * nin + i]), __bfloat162float(W[(long long)o * nin + i]), s);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
        s += __bfloat162float(b[o]);
        if (relu) s = fmaxf(s, 0.f);
        if (out_bf) out_bf[(long long)r * nout + o] = __float2bfloat16_rn(s);
        if (out_f) out_f[(long long)r * nout + o] = s;
    }
}

inline unsigned nb(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

int fail_code(df_handle* h, const Error& e) {
    h->last_error = e.msg;
    return e.code;
}

// buffers of the step kernel for batches of `rows` samples, and its launches
struct Work {
    DevBuf<Layer> layers;
    DevBuf<float> buf, part;
    DevBuf<unsigned> sync;          // barrier arrivals | error word
    float* out = nullptr;           // the last layer's outputs (rows x nout)
    int rows = 0;
    static constexpr int MAX_STEPS = 4096;                 // per launch,
    static constexpr long long MAX_SAMPLES = 1 << 20;      // and rows of all of its steps (4 MB of indices)
    // steps of n rows per launch
    static int launch_steps(long long steps, int n) {
        return (int)std::min(std::min<long long>(steps, MAX_STEPS), std::max(1LL, MAX_SAMPLES / n));
    }
    void alloc(df_mlp* m, int n, int steps) {
        rows = n;
        const int L = (int)m->dims.size() - 1;
        size_t per = 0;
        for (int l = 0; l < L; ++l) per += m->dims[l + 1];
        buf.alloc(3 * per * n);
        part.alloc((size_t)256 * steps);
        part.zero(m->stream);
        sync.alloc(2);
        std::vector<Layer> host(L);
        float* p = buf.p;
        for (int l = 0; l < L; ++l) {
            const size_t c = (size_t)n * m->dims[l + 1];
            host[l] = Layer{m->dims[l], m->dims[l + 1], m->woff[l], m->boff[l], p, p + c, p + 2 * c};
            p += 3 * c;
        }
        out = host[L - 1].A;
        layers.alloc(L);
        DF_CUDA(cudaMemcpyAsync(layers.p, host.data(), sizeof(Layer) * L, cudaMemcpyHostToDevice, m->stream));
        DF_CUDA(cudaStreamSynchronize(m->stream));   // the host array is released on return
    }
};

// 1 / b for quotient()
inline float recip(float b) {
    int e = 0;
    return std::frexp(b, &e) == 1.f - 0x1p-24f ? 0.f : 1.f / b;
}

// runs a.nsteps steps (at most Work::MAX_STEPS) on two CTAs per SM; synchronises
void run_steps(df_mlp* m, Work& w, StepArgs a) {
    a.layers = w.layers.p;
    a.L = (int)m->dims.size() - 1;
    a.rows = w.rows;
    a.scale = 1.f / (float)((long long)w.rows * m->nout);
    a.P = m->P.p;
    a.part = w.part.p;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.count = w.sync.p;
    a.err = reinterpret_cast<int*>(w.sync.p + 1);
    a.wait = grid_wait_cycles();
    DF_CUDA(cudaMemsetAsync(w.sync.p, 0, 2 * sizeof(unsigned), m->stream));
    int dev = 0, sms = 0;
    DF_CUDA(cudaGetDevice(&dev));
    DF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    void* args[] = {&a};
    DF_CUDA(cudaFuncSetAttribute(mlp_steps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_BYTES));
    DF_CUDA(cudaLaunchCooperativeKernel((const void*)mlp_steps_kernel, dim3(2 * sms), dim3(NT), args, STAGE_BYTES, m->stream));
    int herr = 0;
    DF_CUDA(cudaMemcpyAsync(&herr, a.err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
    DF_CUDA(cudaStreamSynchronize(m->stream));
    if (herr) throw Error{DF_E_TIMEOUT, "network kernel timed out waiting on its grid barrier"};
}

// one step's loss from its partials
float step_loss(const float* part) {
    double s = 0;
    for (int q = 0; q < 256; ++q) s += part[q];
    return (float)s;
}

// ---------------------------------------------------------------------------------------------
// geometry: water frames, features and rotation matrices for real solid harmonics (l <= 2)
// ---------------------------------------------------------------------------------------------
struct Frame {
    double O[3];
    double R[3][3];   // columns x, y, z of the molecular frame in laboratory coordinates
};

void normalize(double* v) {
    const double r = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int d = 0; d < 3; ++d) v[d] /= r;
}

// waters as consecutive (O, H, H) atoms; z along the H-O-H bisector, x along H1 - H2
std::vector<Frame> water_frames(const df_atom* atoms, int natom) {
    if (natom % 3) throw Error{DF_E_ARG, "learned guess: atoms must be (O, H, H) triples"};
    std::vector<Frame> fr(natom / 3);
    for (int w = 0; w < natom / 3; ++w) {
        const df_atom &o = atoms[3 * w], &h1 = atoms[3 * w + 1], &h2 = atoms[3 * w + 2];
        if (o.Z != 8 || h1.Z != 1 || h2.Z != 1) throw Error{DF_E_ARG, "learned guess: atoms must be (O, H, H) triples"};
        double z[3], x[3], y[3];
        for (int d = 0; d < 3; ++d) {
            z[d] = (h1.xyz[d] - o.xyz[d]) + (h2.xyz[d] - o.xyz[d]);
            x[d] = h1.xyz[d] - h2.xyz[d];
        }
        normalize(z);
        const double dot = x[0] * z[0] + x[1] * z[1] + x[2] * z[2];
        for (int d = 0; d < 3; ++d) x[d] -= dot * z[d];
        normalize(x);
        y[0] = z[1] * x[2] - z[2] * x[1];
        y[1] = z[2] * x[0] - z[0] * x[2];
        y[2] = z[0] * x[1] - z[1] * x[0];
        for (int d = 0; d < 3; ++d) {
            fr[w].O[d] = o.xyz[d];
            fr[w].R[d][0] = x[d];
            fr[w].R[d][1] = y[d];
            fr[w].R[d][2] = z[d];
        }
    }
    return fr;
}

// D^l(Q) with S_lm(Q u) = sum_m' D_mm' S_lm'(u) for the real solid harmonics of cart_sph.cuh:
// l = 1: S = (y, z, x) = P u, so D = P Q P^T. l = 2: S_m(u) = u^T Q_m u with orthogonal traceless Q_m
// (Frobenius norm^2 = 3/2), so D_mm' = <Q^T Q_m Q, Q_m'> / (3/2).
void rotation_l1(const double Q[3][3], double D[3][3]) {
    const int p[3] = {1, 2, 0};
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) D[a][b] = Q[p[a]][p[b]];
}

void rotation_l2(const double Q[3][3], double D[5][5]) {
    const double s3 = std::sqrt(3.0);
    double Qm[5][3][3] = {};
    Qm[0][0][1] = Qm[0][1][0] = s3 / 2;     // sqrt3 xy
    Qm[1][1][2] = Qm[1][2][1] = s3 / 2;     // sqrt3 yz
    Qm[2][0][0] = Qm[2][1][1] = -0.5;       // z^2 - (x^2 + y^2)/2
    Qm[2][2][2] = 1.0;
    Qm[3][0][2] = Qm[3][2][0] = s3 / 2;     // sqrt3 xz
    Qm[4][0][0] = s3 / 2;                   // sqrt3/2 (x^2 - y^2)
    Qm[4][1][1] = -s3 / 2;
    for (int a = 0; a < 5; ++a) {
        double T[3][3] = {};   // Q^T Qm_a Q
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j)
                for (int k = 0; k < 3; ++k)
                    for (int l = 0; l < 3; ++l) T[i][j] += Q[k][i] * Qm[a][k][l] * Q[l][j];
        for (int b = 0; b < 5; ++b) {
            double s = 0;
            for (int i = 0; i < 3; ++i)
                for (int j = 0; j < 3; ++j) s += T[i][j] * Qm[b][i][j];
            D[a][b] = s / 1.5;
        }
    }
}

// M (nb x nb) for one water's functions: block-diagonal D^l(R^T) per shell; the reference-frame
// function a equals sum_a' M[a][a'] times laboratory function a'
void water_rotation(const df_handle* h, int w, const Frame& f, int nbw, std::vector<double>& M, int& first) {
    double Rt[3][3];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) Rt[i][j] = f.R[j][i];
    double D1[3][3], D2[5][5];
    rotation_l1(Rt, D1);
    rotation_l2(Rt, D2);
    M.assign((size_t)nbw * nbw, 0.0);
    first = -1;
    int off = 0, local = 0;
    for (const df_shell& s : h->basis) {
        const int ns = 2 * s.l + 1;
        if (s.atom >= 3 * w && s.atom < 3 * w + 3) {
            if (first < 0) first = off;
            if (local + ns > nbw) throw Error{DF_E_ARG, "learned guess: unexpected basis layout"};
            for (int a = 0; a < ns; ++a)
                for (int b = 0; b < ns; ++b)
                    M[(size_t)(local + a) * nbw + local + b] = s.l == 0 ? 1.0 : (s.l == 1 ? D1[a][b] : D2[a][b]);
            local += ns;
        }
        off += ns;
    }
    if (local != nbw) throw Error{DF_E_ARG, "learned guess: every water needs the same basis"};
}

int water_nbf(const df_handle* h) {
    int nbw = 0;
    for (const df_shell& s : h->basis)
        if (s.atom < 3) nbw += 2 * s.l + 1;
    return nbw;
}

// features of water w (DF_MLP_NFEAT values): Gaussian radial histograms of O-O, O-H, H1-O, H2-O
// distances (12 centres 3.5 + 0.9 k bohr, width 0.6 bohr, cutoff 15 bohr) and the coordinates of
// the three nearest other O atoms in the molecule's frame (divided by 10 bohr)
constexpr int NRAD = 12;
constexpr int NFEAT = 4 * NRAD + 9;
void water_features(const df_atom* atoms, int natom, const std::vector<Frame>& fr, int w, float* out) {
    for (int i = 0; i < NFEAT; ++i) out[i] = 0.f;
    auto dist = [&](int a, int b) {
        double r2 = 0;
        for (int d = 0; d < 3; ++d) r2 += (atoms[a].xyz[d] - atoms[b].xyz[d]) * (atoms[a].xyz[d] - atoms[b].xyz[d]);
        return std::sqrt(r2);
    };
    auto hist = [&](float* f, double r) {
        if (r > 15.0) return;
        for (int k = 0; k < NRAD; ++k) {
            const double c = 3.5 + 0.9 * k;
            f[k] += (float)std::exp(-(r - c) * (r - c) / (2 * 0.36));
        }
    };
    std::vector<std::pair<double, int>> near;
    for (int a = 0; a < natom; ++a) {
        if (a / 3 == w) continue;
        if (atoms[a].Z == 8) {
            hist(out, dist(3 * w, a));
            hist(out + 2 * NRAD, dist(3 * w + 1, a));
            hist(out + 3 * NRAD, dist(3 * w + 2, a));
            near.push_back({dist(3 * w, a), a});
        } else {
            hist(out + NRAD, dist(3 * w, a));
        }
    }
    std::sort(near.begin(), near.end());
    for (int q = 0; q < 3 && q < (int)near.size(); ++q) {
        const int a = near[q].second;
        for (int c = 0; c < 3; ++c) {
            double v = 0;
            for (int d = 0; d < 3; ++d) v += fr[w].R[d][c] * (atoms[a].xyz[d] - fr[w].O[d]);
            out[4 * NRAD + 3 * q + c] = (float)(v / 10.0);
        }
    }
}

// pair features of the ordered water pair (w1, w2) (DF_MLP_NPFEAT values): the atoms of w2 in w1's frame
// relative to w1's O (divided by 10 bohr), 5 bohr / r for the nine atom pairs between the two waters, and
// a Gaussian expansion of the O-O distance (8 centres 4.5 + 0.5 k bohr, width 0.35 bohr)
constexpr int NPFEAT = 26;
void pair_features(const df_atom* atoms, const std::vector<Frame>& fr, int w1, int w2, float* out) {
    auto dist = [&](int a, int b) {
        double r2 = 0;
        for (int d = 0; d < 3; ++d) r2 += (atoms[a].xyz[d] - atoms[b].xyz[d]) * (atoms[a].xyz[d] - atoms[b].xyz[d]);
        return std::sqrt(r2);
    };
    for (int a = 0; a < 3; ++a)
        for (int c = 0; c < 3; ++c) {
            double v = 0;
            for (int d = 0; d < 3; ++d) v += fr[w1].R[d][c] * (atoms[3 * w2 + a].xyz[d] - fr[w1].O[d]);
            out[3 * a + c] = (float)(v / 10.0);
        }
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) out[9 + 3 * a + b] = (float)(5.0 / dist(3 * w1 + a, 3 * w2 + b));
    const double r = dist(3 * w1, 3 * w2);
    for (int k = 0; k < 8; ++k) {
        const double c = 4.5 + 0.5 * k;
        out[18 + k] = (float)std::exp(-(r - c) * (r - c) / (2 * 0.35 * 0.35));
    }
}

// ordered pairs (w1 != w2) with O-O distance <= cutoff, by w1 then w2
std::vector<std::pair<int, int>> water_pair_list(const df_atom* atoms, int natom, double cutoff) {
    std::vector<std::pair<int, int>> out;
    const int nw = natom / 3;
    for (int w1 = 0; w1 < nw; ++w1)
        for (int w2 = 0; w2 < nw; ++w2) {
            if (w1 == w2) continue;
            double r2 = 0;
            for (int d = 0; d < 3; ++d) {
                const double x = atoms[3 * w1].xyz[d] - atoms[3 * w2].xyz[d];
                r2 += x * x;
            }
            if (r2 <= cutoff * cutoff) out.push_back({w1, w2});
        }
    return out;
}

// C = A B (nb x nb, row-major); tA / tB use the transposes
void small_mm(const std::vector<double>& A, bool tA, const std::vector<double>& B, bool tB, int nb,
              std::vector<double>& C) {
    C.assign((size_t)nb * nb, 0.0);
    for (int i = 0; i < nb; ++i)
        for (int k = 0; k < nb; ++k) {
            const double a = tA ? A[(size_t)k * nb + i] : A[(size_t)i * nb + k];
            if (a == 0.0) continue;
            for (int j = 0; j < nb; ++j) C[(size_t)i * nb + j] += a * (tB ? B[(size_t)j * nb + k] : B[(size_t)k * nb + j]);
        }
}

}  // namespace
}  // namespace dfhf

using namespace dfhf;

extern "C" {

int df_mlp_create(int nin, int nhidden, int nlayers, int nout, unsigned long long seed, df_mlp** out) {
    if (!out || nin < 1 || nhidden < 1 || nlayers < 1 || nout < 1) return DF_E_ARG;
    *out = nullptr;
    df_mlp* m = new df_mlp();
    try {
        m->nin = nin;
        m->nh = nhidden;
        m->nlayers = nlayers;
        m->nout = nout;
        m->dims.push_back(nin);
        for (int l = 0; l < nlayers; ++l) m->dims.push_back(nhidden);
        m->dims.push_back(nout);
        long long off = 0;
        for (size_t l = 0; l + 1 < m->dims.size(); ++l) {
            m->woff.push_back(off);
            off += (long long)m->dims[l] * m->dims[l + 1];
            m->boff.push_back(off);
            off += m->dims[l + 1];
        }
        m->nparams = off;
        // He initialisation from a seeded host generator
        std::vector<float> p(off, 0.f);
        std::mt19937_64 gen(seed);
        for (size_t l = 0; l + 1 < m->dims.size(); ++l) {
            std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / m->dims[l]));
            for (long long i = 0; i < (long long)m->dims[l] * m->dims[l + 1]; ++i) p[m->woff[l] + i] = (float)nd(gen);
        }
        DF_CUDA(cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking));
        m->P.alloc(off);
        m->G.alloc(off);
        m->Mom.alloc(off);
        m->Vel.alloc(off);
        m->Pbf.alloc(off);
        DF_CUDA(cudaMemcpyAsync(m->P.p, p.data(), off * sizeof(float), cudaMemcpyHostToDevice, m->stream));
        m->Mom.zero(m->stream);
        m->Vel.zero(m->stream);
        DF_CUDA(cudaStreamSynchronize(m->stream));
    } catch (const Error& e) {
        df_mlp_free(m);
        return e.code;
    }
    *out = m;
    return DF_OK;
}

void df_mlp_free(df_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    m->P.release();
    m->G.release();
    m->Mom.release();
    m->Vel.release();
    m->Pbf.release();
    if (m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

long long df_mlp_nparams(const df_mlp* m) { return m ? m->nparams : DF_E_ARG; }

int df_mlp_params(df_mlp* m, float* host, int set) {
    if (!m || !host) return DF_E_ARG;
    try {
        if (set) {
            DF_CUDA(cudaMemcpyAsync(m->P.p, host, m->nparams * sizeof(float), cudaMemcpyHostToDevice, m->stream));
            m->adam_t = 0;
            m->Mom.zero(m->stream);
            m->Vel.zero(m->stream);
        } else {
            DF_CUDA(cudaMemcpyAsync(host, m->P.p, m->nparams * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
        }
        DF_CUDA(cudaStreamSynchronize(m->stream));
    } catch (const Error& e) {
        return e.code;
    }
    return DF_OK;
}

int df_mlp_gradients(df_mlp* m, const float* X, const float* Y, int ns, float* grad, float* loss) {
    if (!m || !X || !Y || ns < 1 || !grad) return DF_E_ARG;
    try {
        DevBuf<float> dX, dYt;
        dX.alloc((size_t)ns * m->nin);
        dYt.alloc((size_t)ns * m->nout);
        DF_CUDA(cudaMemcpyAsync(dX.p, X, sizeof(float) * ns * m->nin, cudaMemcpyHostToDevice, m->stream));
        DF_CUDA(cudaMemcpyAsync(dYt.p, Y, sizeof(float) * ns * m->nout, cudaMemcpyHostToDevice, m->stream));
        Work w;
        w.alloc(m, ns, 1);
        StepArgs a{};
        a.nsteps = 1;
        a.G = m->G.p;
        a.X = dX.p;
        a.Y = dYt.p;
        run_steps(m, w, a);
        std::vector<float> part(256);
        DF_CUDA(cudaMemcpyAsync(part.data(), w.part.p, 256 * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
        DF_CUDA(cudaMemcpyAsync(grad, m->G.p, m->nparams * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
        DF_CUDA(cudaStreamSynchronize(m->stream));
        if (loss) *loss = step_loss(part.data());
    } catch (const Error& e) {
        return e.code;
    } catch (const std::bad_alloc&) {
        return DF_E_NOMEM;
    }
    return DF_OK;
}

int df_mlp_train(df_mlp* m, const float* X, const float* Y, int ns, int epochs, int batch, float lr,
                 unsigned long long seed, float* loss_history) {
    if (!m || !X || !Y || ns < 1 || epochs < 1 || batch < 1 || !(lr > 0)) return DF_E_ARG;
    try {
        batch = std::min(batch, ns);
        const int per_epoch = ns / batch;                        // whole batches
        const long long steps = (long long)epochs * per_epoch;
        DevBuf<float> dX, dY;
        dX.alloc((size_t)ns * m->nin);
        dY.alloc((size_t)ns * m->nout);
        DF_CUDA(cudaMemcpyAsync(dX.p, X, sizeof(float) * ns * m->nin, cudaMemcpyHostToDevice, m->stream));
        DF_CUDA(cudaMemcpyAsync(dY.p, Y, sizeof(float) * ns * m->nout, cudaMemcpyHostToDevice, m->stream));
        const int chunk = Work::launch_steps(steps, batch);
        Work w;
        w.alloc(m, batch, chunk);
        DevBuf<int> perm;
        DevBuf<float4> corr;
        perm.alloc((size_t)chunk * batch);
        corr.alloc(chunk);
        std::vector<int> order(ns), hperm((size_t)chunk * batch);
        std::vector<float4> hcorr(chunk);
        std::vector<float> part((size_t)256 * chunk);
        std::vector<double> ep_loss(epochs, 0.0);
        std::mt19937_64 gen(seed);
        for (int i = 0; i < ns; ++i) order[i] = i;
        for (long long t0 = 0; t0 < steps; t0 += chunk) {
            const int nt = (int)std::min<long long>(chunk, steps - t0);
            for (int t = 0; t < nt; ++t) {
                const int b = (int)((t0 + t) % per_epoch);
                if (b == 0) std::shuffle(order.begin(), order.end(), gen);   // a new epoch
                for (int r = 0; r < batch; ++r) hperm[(size_t)t * batch + r] = order[b * batch + r];
                const float b1 = 0.9f, b2 = 0.999f, at = (float)(m->adam_t + t + 1);
                const float c1 = 1.f - std::pow(b1, at), c2 = 1.f - std::pow(b2, at);
                hcorr[t] = make_float4(c1, recip(c1), c2, recip(c2));
            }
            DF_CUDA(cudaMemcpyAsync(perm.p, hperm.data(), sizeof(int) * nt * batch, cudaMemcpyHostToDevice, m->stream));
            DF_CUDA(cudaMemcpyAsync(corr.p, hcorr.data(), sizeof(float4) * nt, cudaMemcpyHostToDevice, m->stream));
            StepArgs a{};
            a.nsteps = nt;
            a.Mom = m->Mom.p;
            a.Vel = m->Vel.p;
            a.X = dX.p;
            a.Y = dY.p;
            a.perm = perm.p;
            a.c = corr.p;
            a.lr = lr;
            run_steps(m, w, a);
            m->adam_t += nt;
            DF_CUDA(cudaMemcpyAsync(part.data(), w.part.p, sizeof(float) * 256 * nt, cudaMemcpyDeviceToHost, m->stream));
            DF_CUDA(cudaStreamSynchronize(m->stream));
            for (int t = 0; t < nt; ++t) ep_loss[(t0 + t) / per_epoch] += step_loss(part.data() + (size_t)256 * t);
        }
        if (loss_history)
            for (int ep = 0; ep < epochs; ++ep) loss_history[ep] = (float)(ep_loss[ep] / per_epoch);
    } catch (const Error& e) {
        return e.code;
    } catch (const std::bad_alloc&) {
        return DF_E_NOMEM;
    }
    return DF_OK;
}

int df_mlp_predict(df_mlp* m, const float* X, int ns, int bf16, float* Y) {
    if (!m || !X || !Y || ns < 1) return DF_E_ARG;
    try {
        const int L = (int)m->dims.size() - 1;
        DevBuf<float> dX, out;
        dX.alloc((size_t)ns * m->nin);
        out.alloc((size_t)ns * m->nout);
        DF_CUDA(cudaMemcpyAsync(dX.p, X, sizeof(float) * ns * m->nin, cudaMemcpyHostToDevice, m->stream));
        if (!bf16 && ns >= LAYER_TILES_ROWS) {
            DevBuf<float> a, b;
            int wide = 1;
            for (int l = 1; l < L; ++l) wide = std::max(wide, m->dims[l]);
            a.alloc((size_t)ns * wide);
            b.alloc((size_t)ns * wide);
            const float* in = dX.p;
            for (int l = 0; l < L; ++l) {
                const int ni = m->dims[l], no = m->dims[l + 1];
                float* to = l == L - 1 ? out.p : (l & 1 ? b.p : a.p);
                const long long tiles = ((long long)ns + FBM - 1) / FBM * ((no + FBN - 1) / FBN);
                layer_tiles_kernel<<<(unsigned)tiles, 256, 0, m->stream>>>(in, ns, ni, m->P.p + m->woff[l], m->P.p + m->boff[l],
                                                                          no, l < L - 1, to);
                DF_CHECK_LAUNCH();
                in = to;
            }
            DF_CUDA(cudaMemcpyAsync(Y, out.p, sizeof(float) * ns * m->nout, cudaMemcpyDeviceToHost, m->stream));
            DF_CUDA(cudaStreamSynchronize(m->stream));
        } else if (!bf16) {
            Work w;
            w.alloc(m, ns, 1);
            StepArgs a{};
            a.nsteps = 1;
            a.X = dX.p;
            run_steps(m, w, a);
            DF_CUDA(cudaMemcpyAsync(Y, w.out, sizeof(float) * ns * m->nout, cudaMemcpyDeviceToHost, m->stream));
            DF_CUDA(cudaStreamSynchronize(m->stream));
        } else {
            to_bf16_kernel<<<nb(m->nparams), 256, 0, m->stream>>>(m->P.p, m->nparams, m->Pbf.p);
            DF_CHECK_LAUNCH();
            int maxw = m->nin;
            for (int d : m->dims) maxw = std::max(maxw, d);
            DevBuf<__nv_bfloat16> a, b;
            a.alloc((size_t)ns * maxw);
            b.alloc((size_t)ns * maxw);
            to_bf16_kernel<<<nb((long long)ns * m->nin), 256, 0, m->stream>>>(dX.p, (long long)ns * m->nin, a.p);
            DF_CHECK_LAUNCH();
            for (int l = 0; l < L; ++l) {
                const int ni = m->dims[l], no = m->dims[l + 1];
                const bool last = l == L - 1;
                bf16_layer_kernel<<<nb((long long)ns * no * 32), 256, 0, m->stream>>>(
                    a.p, ns, ni, m->Pbf.p + m->woff[l], m->Pbf.p + m->boff[l], no, !last, last ? nullptr : b.p,
                    last ? out.p : nullptr);
                DF_CHECK_LAUNCH();
                std::swap(a, b);
            }
            DF_CUDA(cudaMemcpyAsync(Y, out.p, sizeof(float) * ns * m->nout, cudaMemcpyDeviceToHost, m->stream));
            DF_CUDA(cudaStreamSynchronize(m->stream));
            a.release();
            b.release();
        }
        dX.release();
        out.release();
    } catch (const Error& e) {
        return e.code;
    } catch (const std::bad_alloc&) {
        return DF_E_NOMEM;
    }
    return DF_OK;
}

int df_water_features(const df_atom* atoms, int natom, float* out) {
    if (!atoms || natom < 3 || !out) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(atoms, natom);
        for (int w = 0; w < natom / 3; ++w) water_features(atoms, natom, fr, w, out + (size_t)w * NFEAT);
    } catch (const Error& e) {
        return e.code;
    }
    return NFEAT;
}

// reference-frame diagonal blocks of D (host, n x n): out[w] = upper triangle of M D_w M^T
int df_water_blocks(df_handle* h, const double* D, float* out) {
    if (!h || !D || !out) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(h->atoms.data(), (int)h->atoms.size());
        const int nbw = water_nbf(h);
        std::vector<double> M, T((size_t)nbw * nbw);
        const int ntri = nbw * (nbw + 1) / 2;
        for (int w = 0; w < (int)fr.size(); ++w) {
            int first = 0;
            water_rotation(h, w, fr[w], nbw, M, first);
            // T = M Dw M^T
            std::vector<double> MD((size_t)nbw * nbw, 0.0);
            for (int a = 0; a < nbw; ++a)
                for (int c = 0; c < nbw; ++c) {
                    const double mac = M[(size_t)a * nbw + c];
                    if (mac == 0.0) continue;
                    for (int b = 0; b < nbw; ++b) MD[(size_t)a * nbw + b] += mac * D[(size_t)(first + c) * h->n + first + b];
                }
            for (int a = 0; a < nbw; ++a)
                for (int b = 0; b < nbw; ++b) {
                    double s = 0;
                    for (int c = 0; c < nbw; ++c) s += MD[(size_t)a * nbw + c] * M[(size_t)b * nbw + c];
                    T[(size_t)a * nbw + b] = s;
                }
            int k = 0;
            for (int a = 0; a < nbw; ++a)
                for (int b = a; b < nbw; ++b) out[(size_t)w * ntri + k++] = (float)T[(size_t)a * nbw + b];
        }
    } catch (const Error& e) {
        return fail_code(h, e);
    }
    return DF_OK;
}

// learned D0 for a water cluster: features -> MLP (BF16 inference if bf16) -> blocks -> D0 (host)
int df_mlp_guess(df_handle* h, df_mlp* m, int bf16, double* D0) {
    if (!h || !m || !D0) return DF_E_ARG;
    const int natom = (int)h->atoms.size();
    if (natom % 3) return DF_E_ARG;
    const int nw = natom / 3;
    const int nbw = water_nbf(h);
    if (m->nin != NFEAT || m->nout != nbw * (nbw + 1) / 2) {
        h->last_error = "df_mlp_guess: network shape does not match the features / water basis";
        return DF_E_ARG;
    }
    std::vector<float> X((size_t)nw * NFEAT), Y((size_t)nw * m->nout);
    int rc = df_water_features(h->atoms.data(), natom, X.data());
    if (rc < 0) return rc;
    rc = df_mlp_predict(m, X.data(), nw, bf16, Y.data());
    if (rc != DF_OK) return rc;
    return df_water_density(h, Y.data(), D0);
}

int df_water_pairs(const df_atom* atoms, int natom, double cutoff, int* pairs, int max_pairs, float* feats) {
    if (!atoms || natom < 3 || !(cutoff > 0) || max_pairs < 0 || (max_pairs > 0 && !pairs)) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(atoms, natom);
        const auto list = water_pair_list(atoms, natom, cutoff);
        for (int k = 0; k < (int)list.size() && k < max_pairs; ++k) {
            pairs[2 * k] = list[k].first;
            pairs[2 * k + 1] = list[k].second;
            if (feats) pair_features(atoms, fr, list[k].first, list[k].second, feats + (size_t)k * NPFEAT);
        }
        return (int)list.size();
    } catch (const Error& e) {
        return e.code;
    }
}

// out[k] = M_1 D[w1][w2] M_2^T (nb x nb, row-major): the block of the ordered pair in w1's frame (M_2 rotates
// w2's functions by w1's frame)
int df_pair_blocks(df_handle* h, const double* D, const int* pairs, int npairs, float* out) {
    if (!h || !D || npairs < 0 || (npairs > 0 && (!pairs || !out))) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(h->atoms.data(), (int)h->atoms.size());
        const int nbw = water_nbf(h), nw = (int)fr.size();
        std::vector<double> M1, M2, Dl((size_t)nbw * nbw), T1, T;
        for (int k = 0; k < npairs; ++k) {
            const int w1 = pairs[2 * k], w2 = pairs[2 * k + 1];
            if (w1 < 0 || w2 < 0 || w1 >= nw || w2 >= nw || w1 == w2) throw Error{DF_E_ARG, "df_pair_blocks: bad pair"};
            int f1 = 0, f2 = 0;
            water_rotation(h, w1, fr[w1], nbw, M1, f1);
            water_rotation(h, w2, fr[w1], nbw, M2, f2);
            for (int a = 0; a < nbw; ++a)
                for (int b = 0; b < nbw; ++b) Dl[(size_t)a * nbw + b] = D[(size_t)(f1 + a) * h->n + f2 + b];
            small_mm(M1, false, Dl, false, nbw, T1);
            small_mm(T1, false, M2, true, nbw, T);
            for (size_t i = 0; i < T.size(); ++i) out[(size_t)k * nbw * nbw + i] = (float)T[i];
        }
    } catch (const Error& e) {
        return fail_code(h, e);
    }
    return DF_OK;
}

// D0 += the laboratory-frame pair blocks M_1^T T M_2 at [w1][w2] and their transposes at [w2][w1]; a pair
// listed in both orders contributes the mean of its two blocks
int df_pair_density(df_handle* h, const float* blocks, const int* pairs, int npairs, double* D0) {
    if (!h || !D0 || npairs < 0 || (npairs > 0 && (!pairs || !blocks))) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(h->atoms.data(), (int)h->atoms.size());
        const int nbw = water_nbf(h), nw = (int)fr.size();
        std::vector<int> count((size_t)nw * nw, 0);
        for (int k = 0; k < npairs; ++k) {
            const int w1 = pairs[2 * k], w2 = pairs[2 * k + 1];
            if (w1 < 0 || w2 < 0 || w1 >= nw || w2 >= nw || w1 == w2) throw Error{DF_E_ARG, "df_pair_density: bad pair"};
            ++count[(size_t)std::min(w1, w2) * nw + std::max(w1, w2)];
        }
        std::vector<double> M1, M2, T((size_t)nbw * nbw), T1, L;
        for (int k = 0; k < npairs; ++k) {
            const int w1 = pairs[2 * k], w2 = pairs[2 * k + 1];
            const double wgt = 1.0 / count[(size_t)std::min(w1, w2) * nw + std::max(w1, w2)];
            int f1 = 0, f2 = 0;
            water_rotation(h, w1, fr[w1], nbw, M1, f1);
            water_rotation(h, w2, fr[w1], nbw, M2, f2);
            for (size_t i = 0; i < T.size(); ++i) T[i] = blocks[(size_t)k * nbw * nbw + i];
            small_mm(M1, true, T, false, nbw, T1);
            small_mm(T1, false, M2, false, nbw, L);
            for (int a = 0; a < nbw; ++a)
                for (int b = 0; b < nbw; ++b) {
                    const double v = wgt * L[(size_t)a * nbw + b];
                    D0[(size_t)(f1 + a) * h->n + f2 + b] += v;
                    D0[(size_t)(f2 + b) * h->n + f1 + a] += v;
                }
        }
    } catch (const Error& e) {
        return fail_code(h, e);
    }
    return DF_OK;
}

// learned D0 with pair blocks: the diagonal blocks from m (df_mlp_guess) plus the blocks of every water pair
// within `cutoff` bohr (O-O) from mp, in both orders
int df_mlp_guess_pairs(df_handle* h, df_mlp* m, df_mlp* mp, double cutoff, int bf16, double* D0) {
    if (!h || !m || !mp || !D0 || !(cutoff > 0)) return DF_E_ARG;
    const int nbw = water_nbf(h);
    if (mp->nin != NPFEAT || mp->nout != nbw * nbw) {
        h->last_error = "df_mlp_guess_pairs: pair network shape does not match the pair features / water basis";
        return DF_E_ARG;
    }
    int rc = df_mlp_guess(h, m, bf16, D0);
    if (rc != DF_OK) return rc;
    const int natom = (int)h->atoms.size();
    const int np = df_water_pairs(h->atoms.data(), natom, cutoff, nullptr, 0, nullptr);
    if (np < 0) return np;
    if (np == 0) return DF_OK;
    std::vector<int> pairs(2 * (size_t)np);
    std::vector<float> X((size_t)np * NPFEAT), Y((size_t)np * mp->nout);
    rc = df_water_pairs(h->atoms.data(), natom, cutoff, pairs.data(), np, X.data());
    if (rc < 0) return rc;
    rc = df_mlp_predict(mp, X.data(), np, bf16, Y.data());
    if (rc != DF_OK) return rc;
    return df_pair_density(h, Y.data(), pairs.data(), np, D0);
}

// D0 (host n x n) from reference-frame blocks (nwater x ntri): block-diagonal M^T T_w M
int df_water_density(df_handle* h, const float* blocks, double* D0) {
    if (!h || !blocks || !D0) return DF_E_ARG;
    try {
        const std::vector<Frame> fr = water_frames(h->atoms.data(), (int)h->atoms.size());
        const int nbw = water_nbf(h);
        const int ntri = nbw * (nbw + 1) / 2;
        std::fill(D0, D0 + (size_t)h->n * h->n, 0.0);
        std::vector<double> M, T((size_t)nbw * nbw), TM((size_t)nbw * nbw);
        for (int w = 0; w < (int)fr.size(); ++w) {
            int first = 0;
            water_rotation(h, w, fr[w], nbw, M, first);
            int k = 0;
            for (int a = 0; a < nbw; ++a)
                for (int b = a; b < nbw; ++b) T[(size_t)a * nbw + b] = T[(size_t)b * nbw + a] = blocks[(size_t)w * ntri + k++];
            std::fill(TM.begin(), TM.end(), 0.0);
            for (int a = 0; a < nbw; ++a)
                for (int c = 0; c < nbw; ++c) {
                    const double t = T[(size_t)a * nbw + c];
                    for (int b = 0; b < nbw; ++b) TM[(size_t)a * nbw + b] += t * M[(size_t)c * nbw + b];
                }
            for (int a = 0; a < nbw; ++a)
                for (int b = 0; b < nbw; ++b) {
                    double s = 0;
                    for (int c = 0; c < nbw; ++c) s += M[(size_t)c * nbw + a] * TM[(size_t)c * nbw + b];
                    D0[(size_t)(first + a) * h->n + first + b] = s;
                }
        }
    } catch (const Error& e) {
        return fail_code(h, e);
    }
    return DF_OK;
}

}  // extern "C"
