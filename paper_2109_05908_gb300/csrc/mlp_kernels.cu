// The proposal network (an MLP 32 -> 256 -> 256 -> 256, ReLU; outputs read as a
// symmetrised 16 x 16 matrix) in three kernels per training step, FP32 on the
// CUDA cores throughout:
//   1. mlp_rows_kernel: everything that is local to a sample.  A CTA keeps the
//      activations of 16 samples in shared memory through the three layers, the
//      loss and the two backward products, and streams the weights through a
//      double-buffered 32-wide tile (33 tiles, L2-resident), so no activation
//      makes a round trip and no layer boundary is a launch.
//   2. mlp_grad_kernel: the weight gradients H^T dZ, 64 x 64 tiles, the samples
//      split so that the few tiles fill the chip; bias gradients from the same
//      staged tiles.
//   3. mlp_update_kernel: the splits summed in a fixed order, Adam, the bfloat16
//      rounding and the loss.
// Bound by FP32 issue and shared-memory reads in 1 and 2 (1.7 GFLOP at 2000
// samples) and by launch latency below a few hundred samples.  Before: a generic
// GEMM with its own descriptors and allocation per layer, single-thread column
// and loss sums, 24 launches.  2000 samples, call included: 1565 -> 142 us; 700 samples 1120 -> 137 us.
#include "amdd_internal.h"

namespace amdd {
namespace {

constexpr int MR = 16;               // samples per CTA
constexpr int MT = 32;               // k per weight tile
constexpr int MW = 256;              // layer width
constexpr int MLD = MT + 4;          // leading dimension of a backward tile
constexpr int MTILE = MW * MLD;      // floats per tile buffer (forward tiles need MT * MW)
static_assert(PROP_NH == MW && PROP_NO == MW && PROP_NF == MT && PROP_NB * PROP_NB == MW, "network shape");

__device__ __forceinline__ void mlp_cp(float* dst, const float* src, int vec) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (vec)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
#pragma unroll
        for (int u = 0; u < 4; ++u)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * u), "l"(src + u) : "memory");
}
__device__ __forceinline__ void mlp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void mlp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// tile t of the 33: 0 W1; 1..8 W2 forward; 9..16 W3 forward; 17..24 W3 backward; 25..32 W2 backward
__device__ __forceinline__ void mlp_issue(int t, const float* __restrict__ wb, float* buf, int vec) {
    if (t < 17) {  // 32 rows of 256, contiguous
        const float* src = t == 0 ? wb + MLP_OFF_W1 : wb + (t < 9 ? MLP_OFF_W2 : MLP_OFF_W3) + (size_t)((t - 1) & 7) * MT * MW;
        for (int i = threadIdx.x; i < MT * MW / 4; i += 256) mlp_cp(buf + 4 * i, src + 4 * i, vec);
    } else {  // columns [32 q, 32 q + 32) of the 256 rows
        const float* src = wb + (t < 25 ? MLP_OFF_W3 : MLP_OFF_W2) + (size_t)((t - 17) & 7) * MT;
        for (int i = threadIdx.x; i < MT * MW / 4; i += 256)
            mlp_cp(buf + (i >> 3) * MLD + 4 * (i & 7), src + (size_t)(i >> 3) * MW + 4 * (i & 7), vec);
    }
    mlp_commit();
}

// acc[c][r] += w_c a[r] for 8 samples a
__device__ __forceinline__ void mlp_fma(float (&acc)[2][8], float w0, float w1, const float* a) {
    const float4 p = *reinterpret_cast<const float4*>(a), q = *reinterpret_cast<const float4*>(a + 4);
    const float v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        acc[0][r] = fmaf(w0, v[r], acc[0][r]);
        acc[1][r] = fmaf(w1, v[r], acc[1][r]);
    }
}

}  // namespace

// Thread t owns columns t % 128 and t % 128 + 128 for samples 8 (t / 128) .. + 8.
// TRAIN: writes H1, H2, dY, dZ2, dZ1 (n x 256) and each sample's loss; else Q.
template <bool TRAIN>
__global__ void __launch_bounds__(256) mlp_rows_kernel(const float* __restrict__ wb, const float* __restrict__ x,
                                                       const float* __restrict__ qt, int n, float* __restrict__ H1,
                                                       float* __restrict__ H2, float* __restrict__ dY,
                                                       float* __restrict__ dZ2, float* __restrict__ dZ1,
                                                       float* __restrict__ Q, float* __restrict__ part, int vec) {
    extern __shared__ __align__(16) float mlp_smem[];
    float* wt[2] = {mlp_smem, mlp_smem + MTILE};
    float* xs = mlp_smem + 2 * MTILE;  // [k][sample]
    float* h1 = xs + MT * MR;
    float* h2 = h1 + MW * MR;
    float* ys = h2 + MW * MR;
    __shared__ float red[8][8];
    const int tid = threadIdx.x, c0 = tid & 127, rg = (tid >> 7) * 8;
    const int row0 = blockIdx.x * MR;
    mlp_issue(0, wb, wt[0], vec);
    for (int e = tid; e < MT * MR; e += 256) {
        const int r = e / MT, k = e % MT;
        xs[k * MR + r] = row0 + r < n ? x[(size_t)(row0 + r) * MT + k] : 0.0f;
    }
    float acc[2][8];
    auto clear = [&]() {
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[0][r] = acc[1][r] = 0.0f;
    };
    clear();
    constexpr int NT = TRAIN ? 33 : 17;
    for (int t = 0; t < NT; ++t) {
        mlp_wait();
        __syncthreads();  // tile t is there; tile t - 1's buffer and the last layer's inputs are free
        if (t + 1 < NT) mlp_issue(t + 1, wb, wt[(t + 1) & 1], vec);
        const float* w = wt[t & 1];
        if (t < 17) {
            const float* in = (t == 0 ? xs : (t < 9 ? h1 : h2)) + (t == 0 ? 0 : ((t - 1) & 7) * MT * MR) + rg;
#pragma unroll 8
            for (int k = 0; k < MT; ++k) mlp_fma(acc, w[k * MW + c0], w[k * MW + c0 + 128], in + k * MR);
        } else {
            const float* in = (t < 25 ? ys : h2) + ((t - 17) & 7) * MT * MR + rg;
#pragma unroll 2
            for (int k = 0; k < MT; k += 4) {
                const float4 a = *reinterpret_cast<const float4*>(w + c0 * MLD + k);
                const float4 b = *reinterpret_cast<const float4*>(w + (c0 + 128) * MLD + k);
                mlp_fma(acc, a.x, b.x, in + k * MR);
                mlp_fma(acc, a.y, b.y, in + (k + 1) * MR);
                mlp_fma(acc, a.z, b.z, in + (k + 2) * MR);
                mlp_fma(acc, a.w, b.w, in + (k + 3) * MR);
            }
        }
        if (t == 0 || t == 8) {  // a hidden layer is complete
            float* hs = t == 0 ? h1 : h2;
            float* hg = t == 0 ? H1 : H2;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = c0 + 128 * c;
                const float bias = wb[(t == 0 ? MLP_OFF_B1 : MLP_OFF_B2) + j];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float h = fmaxf(acc[c][r] + bias, 0.0f);
                    hs[j * MR + rg + r] = h;
                    if (TRAIN && row0 + rg + r < n) hg[(size_t)(row0 + rg + r) * MW + j] = h;
                }
            }
            clear();
        } else if (t == 16) {  // the outputs are complete: symmetrise, loss and its gradient
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = c0 + 128 * c;
                const float bias = wb[MLP_OFF_B3 + j];
#pragma unroll
                for (int r = 0; r < 8; ++r) ys[j * MR + rg + r] = acc[c][r] + bias;
            }
            clear();
            __syncthreads();
            float d[2][8], loss[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) loss[r] = 0.0f;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = c0 + 128 * c, jt = (j % PROP_NB) * PROP_NB + j / PROP_NB;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int row = row0 + rg + r;
                    const float q = 0.5f * (ys[j * MR + rg + r] + ys[jt * MR + rg + r]);
                    d[c][r] = 0.0f;
                    if (row < n) {
                        if (TRAIN) {
                            const float de = q - qt[(size_t)row * MW + j], dt = q - qt[(size_t)row * MW + jt];
                            loss[r] = fmaf(de, de, loss[r]);
                            d[c][r] = (de + dt) / (float)n;
                            dY[(size_t)row * MW + j] = d[c][r];
                        } else {
                            Q[(size_t)row * MW + j] = q;
                        }
                    }
                }
            }
            if (TRAIN) {
                __syncthreads();  // ys read whole
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int r = 0; r < 8; ++r) ys[(c0 + 128 * c) * MR + rg + r] = d[c][r];
                // each sample's sum over the warp's columns: the lanes first halve the
                // eight samples among them, lane l ends with sample (l >> 2) in bit
                // order 16, 8, 4
                const int lane = tid & 31;
#pragma unroll
                for (int o = 16, h = 4; h > 0; o >>= 1, h >>= 1)
#pragma unroll
                    for (int r = 0; r < h; ++r) {
                        const bool up = (lane & o) != 0;
                        const float give = up ? loss[r] : loss[r + h];
                        loss[r] = (up ? loss[r + h] : loss[r]) + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                loss[0] += __shfl_xor_sync(0xffffffffu, loss[0], 2);
                loss[0] += __shfl_xor_sync(0xffffffffu, loss[0], 1);
                if ((lane & 3) == 0) red[tid >> 5][lane >> 2] = loss[0];
                __syncthreads();
                if (tid < MR && row0 + tid < n) {
                    const float(*w4)[8] = red + 4 * (tid >> 3);  // the four warps of the sample's columns
                    part[row0 + tid] = (w4[0][tid & 7] + w4[1][tid & 7]) + (w4[2][tid & 7] + w4[3][tid & 7]);
                }
            }
        } else if (t == 24 || t == 32) {  // dZ = dH where the unit was on
            float* dg = t == 24 ? dZ2 : dZ1;
            float* hs = t == 24 ? h2 : h1;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = c0 + 128 * c;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float dz = hs[j * MR + rg + r] > 0.0f ? acc[c][r] : 0.0f;
                    hs[j * MR + rg + r] = dz;  // each thread its own entries: the input of the next product
                    if (row0 + rg + r < n) dg[(size_t)(row0 + rg + r) * MW + j] = dz;
                }
            }
            clear();
        }
    }
}

constexpr size_t MLP_ROWS_SMEM = sizeof(float) * (2 * MTILE + MT * MR + 3 * MW * MR);

// G[i][j] = sum over samples of A[s][i] B[s][j], 64 x 64 tile per CTA, 4 x 4 per
// thread; blockIdx.y = split of the samples.  Tiles 0..15 W3 (H2, dY), 16..31 W2
// (H1, dZ2), 32..35 W1 (x, dZ1).  The CTAs of a first tile row also sum B's columns
// (the bias gradient).
__global__ void __launch_bounds__(256) mlp_grad_kernel(const float* __restrict__ x, const float* __restrict__ H1,
                                                       const float* __restrict__ H2, const float* __restrict__ dY,
                                                       const float* __restrict__ dZ2, const float* __restrict__ dZ1,
                                                       int n, int per, float* __restrict__ out, int vec) {
    __shared__ __align__(16) float As[2][MT][64], Bs[2][MT][64];
    const int t = blockIdx.x;
    const int layer = t < 16 ? 3 : (t < 32 ? 2 : 1);
    const int tm = layer == 1 ? 0 : (t & 15) >> 2, tn = t & 3;
    const int M = layer == 1 ? PROP_NF : MW;  // rows of the gradient
    const float* A = layer == 3 ? H2 : (layer == 2 ? H1 : x);
    const float* B = layer == 3 ? dY : (layer == 2 ? dZ2 : dZ1);
    const int s0 = blockIdx.y * per, s1 = min(n, s0 + per);
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int aw = min(64, M - tm * 64);  // 32 for the first layer
    auto issue = [&](int k0, int b) {
        for (int i = tid; i < MT * 16; i += 256) {
            const int k = i >> 4, c = 4 * (i & 15), s = k0 + k;
            if (s < s1) {
                mlp_cp(&Bs[b][k][c], B + (size_t)s * MW + tn * 64 + c, vec);
                if (c < aw) mlp_cp(&As[b][k][c], A + (size_t)s * M + tm * 64 + c, vec);
            } else {
                *reinterpret_cast<float4*>(&Bs[b][k][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(&As[b][k][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (c >= aw) *reinterpret_cast<float4*>(&As[b][k][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        mlp_commit();
    };
    float acc[4][4], bsum = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    if (s0 < s1) issue(s0, 0);
    int b = 0;
    for (int k0 = s0; k0 < s1; k0 += MT, b ^= 1) {
        mlp_wait();
        __syncthreads();
        if (k0 + MT < s1) issue(k0 + MT, b ^ 1);
#pragma unroll 8
        for (int k = 0; k < MT; ++k) {
            const float4 a4 = *reinterpret_cast<const float4*>(&As[b][k][4 * ty]);
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[b][k][4 * tx]);
            const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        if (tm == 0 && tid < 64)
            for (int k = 0; k < MT; ++k) bsum += Bs[b][k][tid];
    }
    float* g = out + (size_t)blockIdx.y * MLP_NPARAM;
    float* gw = g + (layer == 3 ? MLP_OFF_W3 : (layer == 2 ? MLP_OFF_W2 : MLP_OFF_W1));
    float* gb = g + (layer == 3 ? MLP_OFF_B3 : (layer == 2 ? MLP_OFF_B2 : MLP_OFF_B1));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = tm * 64 + 4 * ty + i;
        if (r < M)
#pragma unroll
            for (int j = 0; j < 4; ++j) gw[(size_t)r * MW + tn * 64 + 4 * tx + j] = acc[i][j];
    }
    if (tm == 0 && tid < 64) gb[tn * 64 + tid] = bsum;
}

// grad = sum of the splits (in order), then, with W, one Adam step (Kingma and Ba)
// on the FP32 master weights and their bfloat16-rounded copy; the last CTA sums the
// samples' losses in FP64.
__global__ void __launch_bounds__(256) mlp_update_kernel(const float* __restrict__ parts, int splits,
                                                         float* __restrict__ grad, float* __restrict__ W,
                                                         float* __restrict__ Wb, float* __restrict__ m,
                                                         float* __restrict__ v, float lr, float b1, float b2, float eps,
                                                         float c1, float c2, const float* __restrict__ lpart, int n,
                                                         float* __restrict__ loss) {
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t < (int)MLP_NPARAM) {
        float g = parts[t];
        for (int s = 1; s < splits; ++s) g += parts[(size_t)s * MLP_NPARAM + t];
        if (splits > 1) grad[t] = g;
        if (W) {
            const float mt = b1 * m[t] + (1.0f - b1) * g;
            const float vt = b2 * v[t] + (1.0f - b2) * g * g;
            m[t] = mt;
            v[t] = vt;
            const float w = W[t] - lr * (mt / c1) / (sqrtf(vt / c2) + eps);
            W[t] = w;
            Wb[t] = bf16_round(w);
        }
    }
    if (blockIdx.x + 1 == gridDim.x) {  // a CTA of its own: the loss
        __shared__ double red[8];
        double s = 0.0;
        for (int k = threadIdx.x; k < n; k += 256) s += lpart[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < 8; ++k) s += red[k];
            loss[0] = (float)(s / n);
        }
    }
}

static int mlp_vec(const void* a, const void* b, const void* c) {
    return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}

void launch_mlp_forward(const float* wb, const float* x, int n, float* q, cudaStream_t s) {
    if (n <= 0) return;
    cudaFuncSetAttribute(mlp_rows_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MLP_ROWS_SMEM);
    mlp_rows_kernel<false><<<(n + MR - 1) / MR, 256, MLP_ROWS_SMEM, s>>>(wb, x, nullptr, n, nullptr, nullptr, nullptr,
                                                                         nullptr, nullptr, q, nullptr,
                                                                         mlp_vec(wb, nullptr, nullptr));
}

// work: 9 n 256 + n floats (amdd_mlp_sizes): H1, H2, dY, dZ2, dZ1, the samples' losses,
// then the gradient splits, as many as fit (at most 8, at least 128 samples each)
void launch_mlp_step(float* w, float* wb, float* m, float* v, int t, float lr, const float* x, const float* qt, int n,
                     float* grad, float* work, float* loss, cudaStream_t s) {
    if (n <= 0) return;
    const size_t L = (size_t)n * MW;
    float *H1 = work, *H2 = H1 + L, *dY = H2 + L, *dZ2 = dY + L, *dZ1 = dZ2 + L, *parts = dZ1 + L;
    float* lpart = work + 9 * L;
    const int fit = (int)(4 * L / MLP_NPARAM < 8 ? 4 * L / MLP_NPARAM : 8);
    const int want = fit < n / 128 ? fit : n / 128;
    const int per = want > 1 ? ((n + want - 1) / want + MT - 1) / MT * MT : n;
    const int splits = (n + per - 1) / per;
    const int nl = (n + MR - 1) / MR;
    const int vec = mlp_vec(wb, x, work);
    cudaFuncSetAttribute(mlp_rows_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MLP_ROWS_SMEM);
    mlp_rows_kernel<true><<<nl, 256, MLP_ROWS_SMEM, s>>>(wb, x, qt, n, H1, H2, dY, dZ2, dZ1, nullptr, lpart, vec);
    float* out = splits > 1 ? parts : grad;
    mlp_grad_kernel<<<dim3(36, splits), 256, 0, s>>>(x, H1, H2, dY, dZ2, dZ1, n, per, out, vec);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    mlp_update_kernel<<<((int)MLP_NPARAM + 255) / 256 + 1, 256, 0, s>>>(out, splits, grad, lr > 0.0f ? w : nullptr, wb, m, v,
                                                                    lr, b1, b2, 1e-8f, c1, c2, lpart, n, loss);
}

}  // namespace amdd
