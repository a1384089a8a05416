// Learned radial surrogate: a 1 -> H -> H -> F multilayer perceptron with SiLU activations that maps a pair
// distance to the F = n_max (l_max+1) o-GTO radial integrals I^o_nl(r) (Eq. rad-int-gto-1 after S^-1/2). The paper
// has no such network; its nearest hook is the closing remark of Sec. 'Spline optimization' that the radial basis
// invites numerical optimisation. Conventions (shared with the oracle's mlp.py):
//   t = r / r_cut;  z1 = W1 t + b1;  h1 = silu(z1);  z2 = W2 h1 + b2;  h2 = silu(z2);  y = W3 h2 + b3;
//   I^o_f(r) ~ scale_f y_f, with scale_f = max over r of |I^o_f| so every output is O(1);
//   loss L = mean over batch and outputs of (y - target/scale)^2.
// Parameters are one FP32 vector [W1 (H) | b1 (H) | W2 (H x H, row = output) | b2 (H) | W3 (F x H) | b3 (F)].
//
// Training (FP32, CUDA cores): k_mlp_train takes tiles of samples through forward, backward and their share of the
// weight gradients, k_mlp_reduce sums the shares and applies one bias-corrected Adam step. Targets are the exact FP64
// integrals (rascal_mlp_targets).
//
// Inference (k_mlp_infer): tiles of 128 distances on the tcgen05 tensor cores with BF16 weights and activations and
// FP32 accumulators in TMEM: layer 1 (rank one) on the CUDA cores, layers 2 and 3 as M = 128 MMAs against the
// weights held in shared memory, SiLU epilogues between them, and the input tangent (d/dr) carried as a second
// set of MMAs when derivatives are requested.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "f32x2.cuh"
#include "radial_fp64.cuh"
#include "tcgen05.cuh"

namespace rascal {

__device__ inline float sigmoidf_(float z) { return 1.0f / (1.0f + __expf(-z)); }
__device__ inline float silu_(float z) { return z * sigmoidf_(z); }
__device__ inline float silu_grad_(float z) {
    const float s = sigmoidf_(z);
    return s * (1.0f + z * (1.0f - s));
}

struct MlpLayout {
    int H, F;
    int oW1, ob1, oW2, ob2, oW3, ob3, n;
};

static MlpLayout mlp_layout(int H, int F) {
    MlpLayout L;
    L.H = H;
    L.F = F;
    L.oW1 = 0;
    L.ob1 = H;
    L.oW2 = 2 * H;
    L.ob2 = 2 * H + H * H;
    L.oW3 = 3 * H + H * H;
    L.ob3 = 3 * H + H * H + F * H;
    L.n = 3 * H + H * H + F * H + F;
    return L;
}

// ------------------------------------------------------------------------------------------------ training
// One CTA takes a tile of TS samples through the whole step: forward, the residual, both backward layers and the
// tile's share of every weight gradient, with the weights and all activations in shared memory. A CTA that gets more
// than one tile adds to its own row of `part` [gridDim.x][L.n + 1] (the last word is the loss); k_mlp_reduce sums the
// rows, in order, so the result does not depend on scheduling.
//
// Bound: FP32 FMA issue (6 FMAs per weight and sample, 0.43 GFLOP at 4096 samples and F = 208). Each contraction runs
// as register tiles whose loads are 16-byte rows along the summed index where both operands have it contiguous
// (layers 2 and 3, weight gradients: paired FMAs over even and odd terms, no operand duplication), and as 4 x 4 outer
// products where they do not (the two backward layers, split over the summed index so that all threads work).
// Measured (4096 samples, F = 208, forward to gradient): 958 us as a kernel per layer with one thread per weight
// summing the batch serially (648 us of it) -> 28.7 us.
constexpr int kTrainThreads = 256;
constexpr int kTrainH = 64;       // hidden units: the layouts below are written for it (kMlpH)
constexpr int kTrainP = 68;       // pitch of a 64-wide row in floats: 17 16-byte words, odd, conflict-free

template <int TS>
__host__ __device__ constexpr size_t train_smem_floats(int F) {
    // W3, W2 | H1, H2 by sample | H1, H2, silu'(z2), dz2, dz1 by unit | dY by output | partial sums | t, W1, b1, b2, b3
    return (size_t)F * kTrainP + kTrainH * kTrainP + 2 * TS * kTrainP + 5 * kTrainH * (TS + 4) + (size_t)F * (TS + 4) +
           kTrainThreads * 16 + TS + 3 * kTrainH + F + 8;
}

__device__ inline float f2_sum(uint64_t v) {
    float a, b;
    f2_unpack(v, a, b);
    return a + b;
}

// acc[u][v] += sum over 4 consecutive k of a_u b_v, even and odd terms in the two halves
template <int NU, int NV>
__device__ inline void dot4(uint64_t (&acc)[NU][NV], const float* const (&a)[NU], const float* const (&b)[NV], int k) {
    ulonglong2 av[NU], bv[NV];
#pragma unroll
    for (int u = 0; u < NU; ++u) av[u] = *reinterpret_cast<const ulonglong2*>(a[u] + k);
#pragma unroll
    for (int v = 0; v < NV; ++v) bv[v] = *reinterpret_cast<const ulonglong2*>(b[v] + k);
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            acc[u][v] = f2_fma(av[u].x, bv[v].x, acc[u][v]);
            acc[u][v] = f2_fma(av[u].y, bv[v].y, acc[u][v]);
        }
}

// out[4 x 4 tile (k, s)] of sum_r W[r][k] D[r][s] over r in [r0, r1): W rows at pitch kTrainP, D rows at pitch pd
__device__ inline void outer_sum(float (&acc)[4][4], const float* W, const float* D, int pd, int r0, int r1) {
    uint64_t ap[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u) ap[u][0] = ap[u][1] = 0ull;
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
        const float4 w = *reinterpret_cast<const float4*>(W + r * kTrainP);
        const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(D + r * pd);
        const float ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint64_t wu = f2_pack(ww[u], ww[u]);
            ap[u][0] = f2_fma(wu, d.x, ap[u][0]);
            ap[u][1] = f2_fma(wu, d.y, ap[u][1]);
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        f2_unpack(ap[u][0], acc[u][0], acc[u][1]);
        f2_unpack(ap[u][1], acc[u][2], acc[u][3]);
    }
}

// B samples; `order` (may be NULL) maps sample b of the batch to its row of t_all and y_all
template <int TS>
__global__ void __launch_bounds__(kTrainThreads, 1) k_mlp_train(int B, int F, const float* __restrict__ P, MlpLayout L,
                                                                const int64_t* __restrict__ order,
                                                                const float* __restrict__ t_all,
                                                                const float* __restrict__ y_all, float* __restrict__ part) {
    extern __shared__ __align__(16) float sh[];
    constexpr int H = kTrainH, PT = TS + 4, ST = TS / 4;  // PT / 4 is odd for TS = 8, 16, 32
    float* W3 = sh;                    // [F][kTrainP]
    float* W2 = W3 + F * kTrainP;      // [H][kTrainP]
    float* H1 = W2 + H * kTrainP;      // [TS][kTrainP]
    float* H2 = H1 + TS * kTrainP;     // [TS][kTrainP]
    float* H1T = H2 + TS * kTrainP;    // [H][PT]
    float* H2T = H1T + H * PT;         // [H][PT]
    float* G2T = H2T + H * PT;         // [H][PT] silu'(z2)
    float* D2T = G2T + H * PT;         // [H][PT] dz2
    float* D1T = D2T + H * PT;         // [H][PT] dz1
    float* DYT = D1T + H * PT;         // [F][PT]
    float* red = DYT + F * PT;         // [kTrainThreads][16]
    float* st = red + kTrainThreads * 16;  // [TS] inputs
    float* sW1 = st + TS;
    float* sb1 = sW1 + H;
    float* sb2 = sb1 + H;
    float* sb3 = sb2 + H;              // [F]
    __shared__ float s_loss[kTrainThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < F * 16; e += kTrainThreads)
        *reinterpret_cast<float4*>(W3 + (e >> 4) * kTrainP + 4 * (e & 15)) =
            __ldg(reinterpret_cast<const float4*>(P + L.oW3) + e);
    for (int e = tid; e < H * 16; e += kTrainThreads)
        *reinterpret_cast<float4*>(W2 + (e >> 4) * kTrainP + 4 * (e & 15)) =
            __ldg(reinterpret_cast<const float4*>(P + L.oW2) + e);
    if (tid < H) {
        sW1[tid] = P[L.oW1 + tid];
        sb1[tid] = P[L.ob1 + tid];
        sb2[tid] = P[L.ob2 + tid];
    }
    for (int f = tid; f < F; f += kTrainThreads) sb3[f] = P[L.ob3 + f];
    const float inv = 2.0f / ((float)B * (float)F);
    const int FT = (F + 3) / 4;
    const int tiles = (B + TS - 1) / TS;
    float* G = part + (int64_t)blockIdx.x * (L.n + 1);
    float loss = 0.0f;
    bool first = true;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, first = false) {
        const int b0 = tile * TS, ns = min(TS, B - b0);
        __syncthreads();  // the previous tile's weight gradients are done with the activations
        if (tid < TS) st[tid] = tid < ns ? t_all[order ? order[b0 + tid] : (int64_t)(b0 + tid)] : 0.0f;
        __syncthreads();
        // layer 1; samples past the batch keep zero residuals, so nothing of theirs reaches a sum
        for (int e = tid; e < TS * H; e += kTrainThreads) {
            const int s = e >> 6, k = e & 63;
            const float h = silu_(fmaf(sW1[k], st[s], sb1[k]));
            H1[s * kTrainP + k] = h;
            H1T[k * PT + s] = h;
        }
        __syncthreads();
        // layer 2: tiles of 2 units x 4 samples, rows interleaved so that neighbouring lanes read neighbouring rows
        for (int e = tid; e < 32 * ST; e += kTrainThreads) {
            const int kt = e & 31, s0 = e >> 5;
            const float* a[2] = {W2 + kt * kTrainP, W2 + (kt + 32) * kTrainP};
            const float* b[4];
            uint64_t acc[2][4] = {};
#pragma unroll
            for (int v = 0; v < 4; ++v) b[v] = H1 + (s0 + ST * v) * kTrainP;
#pragma unroll 4
            for (int k = 0; k < H; k += 4) dot4<2, 4>(acc, a, b, k);
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int k = kt + 32 * u, s = s0 + ST * v;
                    const float z = f2_sum(acc[u][v]) + sb2[k], h = silu_(z);
                    H2[s * kTrainP + k] = h;
                    H2T[k * PT + s] = h;
                    G2T[k * PT + s] = silu_grad_(z);
                }
        }
        __syncthreads();
        // layer 3 and the residual: tiles of 4 outputs x 4 samples
        for (int e = tid; e < FT * ST; e += kTrainThreads) {
            const int s0 = e / FT, ft = e - s0 * FT;
            const float *a[4], *b[4], *y[4];
            uint64_t acc[4][4] = {};
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = W3 + min(ft + FT * u, F - 1) * kTrainP;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int s = s0 + ST * v;
                b[v] = H2 + s * kTrainP;
                const int64_t row = s < ns ? (order ? order[b0 + s] : (int64_t)(b0 + s)) : 0;
                y[v] = y_all + row * F;
            }
#pragma unroll 4
            for (int k = 0; k < H; k += 4) dot4<4, 4>(acc, a, b, k);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int f = ft + FT * u;
                if (f >= F) break;
                const float bias = sb3[f];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int s = s0 + ST * v;
                    const float d = s < ns ? f2_sum(acc[u][v]) + bias - __ldg(y[v] + f) : 0.0f;
                    DYT[f * PT + s] = inv * d;
                    loss = fmaf(d, d, loss);
                }
            }
        }
        __syncthreads();
        // backward through layer 3, then layer 2: 16 x ST tiles, the sum split over the thread groups
        constexpr int kTiles = 16 * ST, kSplit = kTrainThreads / kTiles;
        const int tl = tid % kTiles, sp = tid / kTiles;
        const int k0 = 4 * (tl & 15), s0 = 4 * (tl >> 4);
        for (int pass = 0; pass < 2; ++pass) {
            const int n = pass ? H : F, per = (n + kSplit - 1) / kSplit;
            float acc[4][4];
            outer_sum(acc, (pass ? W2 : W3) + k0, (pass ? D2T : DYT) + s0, PT, min(n, sp * per), min(n, (sp + 1) * per));
            if (sp > 0) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) red[((sp - 1) * 16 + 4 * u + v) * kTiles + tl] = acc[u][v];
            }
            __syncthreads();
            if (sp == 0) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
#pragma unroll
                        for (int q = 0; q < kSplit - 1; ++q) acc[u][v] += red[(q * 16 + 4 * u + v) * kTiles + tl];
                        const int k = k0 + u, s = s0 + v;
                        acc[u][v] *= pass ? silu_grad_(fmaf(sW1[k], st[s], sb1[k])) : G2T[k * PT + s];
                    }
                    *reinterpret_cast<float4*>((pass ? D1T : D2T) + (k0 + u) * PT + s0) =
                        make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
                }
            }
            __syncthreads();
        }
        // weight gradients of the tile: 4 x 4 tiles of (output row, hidden unit), summed over the samples; 16
        // neighbouring lanes write 16 neighbouring words
        auto put = [&](int idx, float v) { G[idx] = first ? v : G[idx] + v; };
        for (int e = tid; e < (FT + 16) * 16; e += kTrainThreads) {
            const bool l3 = e < FT * 16;
            const int kt = e & 15, rt = (l3 ? e : e - FT * 16) >> 4, step = l3 ? FT : 16, n = l3 ? F : H;
            const float* D = l3 ? DYT : D2T;
            const float* A = l3 ? H2T : H1T;
            const float *a[4], *b[4];
            uint64_t acc[4][4] = {};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = D + min(rt + step * u, n - 1) * PT;
                b[u] = A + (kt + 16 * u) * PT;
            }
#pragma unroll
            for (int s = 0; s < TS; s += 4) dot4<4, 4>(acc, a, b, s);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = rt + step * u;
                if (r >= n) break;
#pragma unroll
                for (int v = 0; v < 4; ++v) put((l3 ? L.oW3 : L.oW2) + r * H + kt + 16 * v, f2_sum(acc[u][v]));
            }
        }
        for (int e = tid; e < F + 3 * H; e += kTrainThreads) {  // biases and layer 1
            const float* D = e < F ? DYT + e * PT : (e < F + H ? D2T + (e - F) * PT : D1T + ((e - F) & 63) * PT);
            const bool w1 = e >= F + 2 * H;
            float v = 0.0f;
            for (int s = 0; s < TS; ++s) v = w1 ? fmaf(D[s], st[s], v) : v + D[s];
            put(e < F ? L.ob3 + e : (e < F + H ? L.ob2 + e - F : (w1 ? L.oW1 : L.ob1) + ((e - F) & 63)), v);
        }
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) s_loss[warp] = loss;
    __syncthreads();
    if (tid == 0) {
        float v = 0.0f;
        for (int w = 0; w < kTrainThreads / 32; ++w) v += s_loss[w];
        G[L.n] = v / ((float)B * (float)F);
    }
}

// Sums the rows of `part` [rows][n + 1] per parameter (rows in order, in kRedSplit interleaved chains), the loss from
// the last word, and with ADAM applies one bias-corrected Adam step to the parameter. One block covers 32 parameters.
constexpr int kRedSplit = 8;
struct AdamArgs {
    float *P, *m, *v;
    float lr, beta1, beta2, eps, bc1, bc2;
};
template <bool ADAM>
__global__ void __launch_bounds__(32 * kRedSplit) k_mlp_reduce(int n, int rows, const float* __restrict__ part,
                                                               float* __restrict__ G, float* __restrict__ loss, AdamArgs A) {
    __shared__ float sum[kRedSplit][32];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float acc = 0.0f;
    if (i <= n) {
#pragma unroll 8
        for (int r = q; r < rows; r += kRedSplit) acc += part[(int64_t)r * (n + 1) + i];
    }
    sum[q][lane] = acc;
    __syncthreads();
    if (q != 0 || i > n) return;
    for (int k = 1; k < kRedSplit; ++k) acc += sum[k][lane];
    if (i == n) {
        *loss = acc;
        return;
    }
    if (!ADAM) {
        G[i] = acc;
        return;
    }
    const float mi = A.beta1 * A.m[i] + (1.0f - A.beta1) * acc;
    const float vi = A.beta2 * A.v[i] + (1.0f - A.beta2) * acc * acc;
    A.m[i] = mi;
    A.v[i] = vi;
    A.P[i] -= A.lr * (mi / A.bc1) / (sqrtf(vi / A.bc2) + A.eps);
}

// Samples per tile and CTAs of a training step: the smallest tile of 8, 16 or 32 samples that gives every tile an SM of
// its own (whole call at F = 208, one tile per CTA: 23 us with 8 samples, 25 with 16, 29 with 32; a second tile of 32
// adds 25 us, so past 32 samples per SM the largest tile, which reads the weights least often, is taken). A basis so
// wide that 32 samples do not fit beside its weights takes 16, then 8.
struct TrainPlan {
    int ts, grid;
    size_t smem;
};
static TrainPlan train_plan(const rascal_ctx* ctx, int B, int F) {
    auto bytes = [&](int ts) {
        return sizeof(float) * (ts == 32 ? train_smem_floats<32>(F) : (ts == 16 ? train_smem_floats<16>(F) : train_smem_floats<8>(F)));
    };
    int ts = 8;
    while (ts < 32 && (B + ts - 1) / ts > ctx->n_sm && bytes(2 * ts) <= 226 * 1024) ts *= 2;
    const int tiles = (B + ts - 1) / ts;
    return {ts, std::min(tiles, ctx->n_sm), bytes(ts)};
}

// loss and gradient of one batch into G and *loss, or (adam != NULL) the Adam step with them; part holds
// plan.grid (L.n + 1) floats
static int mlp_step(rascal_ctx* ctx, const MlpLayout& L, const TrainPlan& plan, int B, const int64_t* order, const float* t,
                    const float* y, float* part, float* G, float* loss, const AdamArgs* adam) {
    switch (plan.ts) {
        case 32: k_mlp_train<32><<<plan.grid, kTrainThreads, plan.smem, ctx->stream>>>(B, L.F, ctx->mlp_params, L, order, t, y, part); break;
        case 16: k_mlp_train<16><<<plan.grid, kTrainThreads, plan.smem, ctx->stream>>>(B, L.F, ctx->mlp_params, L, order, t, y, part); break;
        default: k_mlp_train<8><<<plan.grid, kTrainThreads, plan.smem, ctx->stream>>>(B, L.F, ctx->mlp_params, L, order, t, y, part); break;
    }
    RASCAL_LAUNCH_CHECK("k_mlp_train");
    const unsigned blocks = (unsigned)div_up(L.n + 1, 32);
    if (adam)
        k_mlp_reduce<true><<<blocks, 32 * kRedSplit, 0, ctx->stream>>>(L.n, plan.grid, part, G, loss, *adam);
    else
        k_mlp_reduce<false><<<blocks, 32 * kRedSplit, 0, ctx->stream>>>(L.n, plan.grid, part, G, loss, AdamArgs{});
    RASCAL_LAUNCH_CHECK("k_mlp_reduce");
    return RASCAL_OK;
}

// ------------------------------------------------------------------------------------------------ targets
// FP64 targets at arbitrary r from a dense FP64 clamped spline of the exact integrals (see rascal_mlp_targets)
__global__ void k_spline64_eval(int64_t n, const double* __restrict__ r, int M, double delta, int F,
                                const double* __restrict__ y, const double* __restrict__ y2, int n_max, int L1,
                                const double* __restrict__ inv_scale, float* __restrict__ out) {
    const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (id >= n * F) return;
    const int64_t p = id / F;
    const int f = (int)(id % F);  // f = l n_max + n
    const int l = f / n_max, nn = f % n_max;
    const double rr = r[p];
    int k = (int)floor(rr / delta);
    k = k < 0 ? 0 : (k > M - 1 ? M - 1 : k);
    const double A = ((k + 1) * delta - rr) / delta, B = 1.0 - A;
    const double yk = y[((int64_t)k * n_max + nn) * L1 + l], yk1 = y[((int64_t)(k + 1) * n_max + nn) * L1 + l];
    const double s0 = y2[(int64_t)f * (M + 1) + k], s1 = y2[(int64_t)f * (M + 1) + k + 1];
    const double v = A * yk + B * yk1 + ((A * A * A - A) * s0 + (B * B * B - B) * s1) * delta * delta / 6.0;
    out[p * F + f] = (float)(v * inv_scale[f]);
}

// ------------------------------------------------------------------------------------------------ inference
struct MlpInferArgs {
    const float4* rij;      // pair vectors (w = r), or NULL when r is given
    const float* r_in;      // distances, or NULL
    int64_t n;
    float* out;             // [n][F] radial values scale_f y_f (f = l n_max + n)
    float* dout;            // [n][F] d/dr, or NULL
    const float* P;         // FP32 parameters (layer 1 and biases are read from here)
    const __nv_bfloat16* W2t;  // W2 as a K-major operand tile (N = H rows, K = H)
    const __nv_bfloat16* W3t;  // W3 as a K-major operand tile (N = F_pad rows, K = H)
    const float* scale;     // [F]
    MlpLayout L;
    int F_pad;              // F rounded up to 16
    float inv_rscale;       // 1 / r_cut
    unsigned* flags;
    uint32_t stall_polls;   // test hook: > 0 makes the first completion wait run out
};

constexpr int kMlpH = 64;
constexpr int kMlpTile = 128;
constexpr int kMlpThreads = 256;
// TMEM: values in columns 0..255, forward tangents (d/dr) in 256..511; without tangents two CTAs share an SM


// offset of element (row, k) in a K-major no-swizzle bf16 tile with K = 64 (8 chunks of 16 bytes per 8-row group)
__device__ __host__ inline int kmajor64_off(int row, int k) {
    return (row >> 3) * 1024 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// Eight bf16 values, one 16-byte chunk of an operand row.
__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
    uint32_t o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const __nv_bfloat162 h = __halves2bfloat162(__float2bfloat16_rn(v[2 * u]), __float2bfloat16_rn(v[2 * u + 1]));
        o[u] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// A tile of 128 distances per step; two threads share a row (its TMEM lane), each with half of the columns of every layer.
// Bound: the chain layer 1, MMA, SiLU, MMA, output of a tile, overlapped only between the two CTAs of an SM (442 000 pairs, 208
// outputs, no derivatives: 0.37 GB written, 55 us). With a thread per row, 2-byte operand stores, 64-byte pieces of output rows
// and sleeping waits the kernel took 341 us there, now 164; outputs bit-identical.
__global__ void __launch_bounds__(kMlpThreads, 2) k_mlp_infer(const MlpInferArgs A) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t s_bar, s_dead;
    __shared__ uint32_t s_tmem;
    const int H = kMlpH, F = A.L.F;
    unsigned char* w2 = smem;                              // 64 x 64 bf16 = 8 KB
    unsigned char* w3 = w2 + 8192;                         // F_pad x 64 bf16
    unsigned char* a1 = w3 + (size_t)A.F_pad * 128;        // 128 x 64 bf16 (h1), 16 KB
    const bool deriv = A.dout != nullptr;
    const uint32_t tm_cols = deriv ? 512u : 256u;
    unsigned char* a1d = a1 + 16384;                       // tangent of h1 (only with derivatives)
    unsigned char* a2 = a1d + (deriv ? 16384 : 0);         // h2
    unsigned char* a2d = a2 + 16384;                       // tangent of h2 (only with derivatives)
    float* s_par = reinterpret_cast<float*>(a2d + (deriv ? 16384 : 0));  // W1, b1, b2 [H each], b3, scale [F each]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, trow = tid & 127, half = tid >> 7;
    // per-warp 32 x 32 output slabs (pitch 36: rows and 16-byte pieces of rows without conflicts)
    float* s_slab = s_par + ((3 * H + 2 * F + 3) & ~3) + warp * 32 * 36;
    // weights into shared memory (already laid out as operand tiles on the host side)
    for (int b = tid; b < 8192 / 16; b += blockDim.x) reinterpret_cast<uint4*>(w2)[b] = reinterpret_cast<const uint4*>(A.W2t)[b];
    for (int b = tid; b < A.F_pad * 128 / 16; b += blockDim.x)
        reinterpret_cast<uint4*>(w3)[b] = reinterpret_cast<const uint4*>(A.W3t)[b];
    for (int k = tid; k < H; k += blockDim.x) {
        s_par[k] = A.P[A.L.oW1 + k];
        s_par[H + k] = A.P[A.L.ob1 + k];
        s_par[2 * H + k] = A.P[A.L.ob2 + k];
    }
    for (int f = tid; f < F; f += blockDim.x) {
        s_par[3 * H + f] = A.P[A.L.ob3 + f];
        s_par[3 * H + F + f] = A.scale[f];
    }
    if (warp == 0) {
        tmem_alloc(&s_tmem, tm_cols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&s_bar, 1);
        mbar_init(&s_dead, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = s_tmem;
    const uint32_t id2 = instr_desc(1u, 128u, (uint32_t)H);
    const uint32_t id3 = instr_desc(1u, 128u, (uint32_t)A.F_pad);
    const uint32_t s_w2 = smem_u32(w2), s_w3 = smem_u32(w3), s_a1 = smem_u32(a1), s_a1d = smem_u32(a1d),
                   s_a2 = smem_u32(a2), s_a2d = smem_u32(a2d);
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const bool vec = F % 4 == 0 && ((reinterpret_cast<uintptr_t>(A.out) | reinterpret_cast<uintptr_t>(A.dout)) & 15) == 0;
    uint32_t phase = 0;
    bool ok = true;
    const int64_t n_tiles = (A.n + kMlpTile - 1) / kMlpTile;
    for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        const int64_t p = tile * kMlpTile + trow;
        const bool valid = p < A.n;
        float r = 0.0f;
        if (valid) r = A.rij ? A.rij[p].w : A.r_in[p];
        const float tt = r * A.inv_rscale;
        // layer 1 on the CUDA cores: row = this thread's distance
#pragma unroll 1
        for (int k0 = H / 2 * half; k0 < H / 2 * (half + 1); k0 += 8) {
            float h[8], d[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float z = fmaf(s_par[k0 + u], tt, s_par[H + k0 + u]);
                h[u] = silu_(z);
                d[u] = deriv ? silu_grad_(z) * s_par[k0 + u] * A.inv_rscale : 0.0f;
            }
            *reinterpret_cast<uint4*>(a1 + kmajor64_off(trow, k0)) = pack8(h);
            if (deriv) *reinterpret_cast<uint4*>(a1d + kmajor64_off(trow, k0)) = pack8(d);
        }
        fence_proxy_async_smem();
        __syncthreads();
        // layer 2: D2 = h1 W2^T (TMEM cols 0..63), tangent in cols 256..319
        if (tid == 0) {
            tc_fence_after();
            for (int kk = 0; kk < H / 16; ++kk) {
                const uint64_t db = smem_desc(s_w2 + kk * 256, 128, 1024);
                mma_bf16_ss(taddr, smem_desc(s_a1 + kk * 256, 128, 1024), db, id2, kk > 0);
                if (deriv) mma_bf16_ss(taddr + 256, smem_desc(s_a1d + kk * 256, 128, 1024), db, id2, kk > 0);
            }
            mma_commit(&s_bar);
        }
        // the test hook makes this wait, a CTA's first, on a barrier that nothing arrives at
        bool done = A.stall_polls ? mbar_wait_bounded(&s_dead, 0u, A.stall_polls) : mbar_wait_spin(&s_bar, phase);
        ok = __syncthreads_and(done) != 0;
        if (!ok) break;
        phase ^= 1u;
        tc_fence_after();
#pragma unroll 1
        for (int c0 = H / 2 * half; c0 < H / 2 * (half + 1); c0 += 16) {
            float z[16], dz[16];
            tmem_ld16(taddr + lane_base + (uint32_t)c0, z);
            if (deriv) tmem_ld16(taddr + lane_base + 256u + (uint32_t)c0, dz);
#pragma unroll
            for (int g = 0; g < 16; g += 8) {
                float h[8], d[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float zz = z[g + u] + s_par[2 * H + c0 + g + u];
                    h[u] = silu_(zz);
                    d[u] = deriv ? silu_grad_(zz) * dz[g + u] : 0.0f;
                }
                *reinterpret_cast<uint4*>(a2 + kmajor64_off(trow, c0 + g)) = pack8(h);
                if (deriv) *reinterpret_cast<uint4*>(a2d + kmajor64_off(trow, c0 + g)) = pack8(d);
            }
        }
        tc_fence_before();
        fence_proxy_async_smem();
        __syncthreads();
        // layer 3: D3 = h2 W3^T (cols 0..F_pad-1), tangent at 256..
        if (tid == 0) {
            tc_fence_after();
            for (int kk = 0; kk < H / 16; ++kk) {
                const uint64_t db = smem_desc(s_w3 + kk * 256, 128, 1024);
                mma_bf16_ss(taddr, smem_desc(s_a2 + kk * 256, 128, 1024), db, id3, kk > 0);
                if (deriv) mma_bf16_ss(taddr + 256, smem_desc(s_a2d + kk * 256, 128, 1024), db, id3, kk > 0);
            }
            mma_commit(&s_bar);
        }
        done = mbar_wait_spin(&s_bar, phase);
        ok = __syncthreads_and(done) != 0;
        if (!ok) break;
        phase ^= 1u;
        tc_fence_after();
        const int64_t row0 = tile * kMlpTile + 32 * (warp & 3);  // this warp's 32 rows (pairs)
        // 32 columns at a time through the slab, values then derivatives: eight lanes store 128 bytes of a row
        auto leave = [&](float* out, uint32_t t0, int c0, bool value) {
            const int n16 = min(32, A.F_pad - c0);
#pragma unroll
            for (int g = 0; g < 32; g += 16) {
                if (g >= n16) break;
                float y[16];
                tmem_ld16(t0 + (uint32_t)(c0 + g), y);
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const int f = min(c0 + g + u, F - 1);
                    const float sc = s_par[3 * H + F + f];
                    y[u] = value ? sc * (y[u] + s_par[3 * H + f]) : sc * y[u];
                }
#pragma unroll
                for (int u = 0; u < 16; u += 4)
                    *reinterpret_cast<float4*>(s_slab + lane * 36 + g + u) = make_float4(y[u], y[u + 1], y[u + 2], y[u + 3]);
            }
            __syncwarp();
            if (vec) {
                const int cl = 4 * (lane & 7), f = c0 + cl;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int rr = 4 * k + (lane >> 3);
                    if (row0 + rr < A.n && cl < n16 && f < F)
                        *reinterpret_cast<float4*>(out + (row0 + rr) * F + f) = *reinterpret_cast<const float4*>(s_slab + rr * 36 + cl);
                }
            } else {
#pragma unroll 4
                for (int rr = 0; rr < 32; ++rr)
                    if (row0 + rr < A.n && lane < n16 && c0 + lane < F) out[(row0 + rr) * F + c0 + lane] = s_slab[rr * 36 + lane];
            }
            __syncwarp();
        };
#pragma unroll 1
        for (int c0 = 32 * half; c0 < A.F_pad; c0 += 64) {
            leave(A.out, taddr + lane_base, c0, true);
            if (deriv) leave(A.dout, taddr + lane_base + 256u, c0, false);
        }
        tc_fence_before();
        __syncthreads();
    }
    if (!ok && tid == 0) atomicOr(A.flags, kFlagTimeout);
    if (!ok) mbar_wait_bounded(&s_bar, phase);  // the MMAs of the wait that ran out, before their TMEM is freed
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(taddr, tm_cols);
    }
}

}  // namespace rascal

using namespace rascal;

// ---------------------------------------------------------------------------------------------------------- API
namespace rascal {

static int mlp_check(rascal_ctx* ctx) {
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (!ctx->mlp_params) return set_error(RASCAL_E_ARG, "no MLP in this context: call rascal_mlp_set_params first");
    return RASCAL_OK;
}

// bf16 operand tiles of W2 (H x H) and W3 (F_pad x H) from the FP32 parameters
__global__ void k_mlp_pack(int H, int F, int F_pad, const float* __restrict__ P, MlpLayout L, __nv_bfloat16* W2t,
                           __nv_bfloat16* W3t) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < H * H) {
        const int row = idx / H, k = idx % H;
        W2t[kmajor64_off(row, k) / 2] = __float2bfloat16_rn(P[L.oW2 + idx]);
    }
    if (idx < F_pad * H) {
        const int row = idx / H, k = idx % H;
        const float v = row < F ? P[L.oW3 + (int64_t)row * H + k] : 0.0f;
        W3t[kmajor64_off(row, k) / 2] = __float2bfloat16_rn(v);
    }
}

int mlp_pack(rascal_ctx* ctx) {
    const MlpLayout L = mlp_layout(ctx->mlp_hidden, ctx->F);
    const int F_pad = (ctx->F + 15) / 16 * 16;
    const int n = std::max(ctx->mlp_hidden * ctx->mlp_hidden, F_pad * ctx->mlp_hidden);
    k_mlp_pack<<<div_up(n, 256), 256, 0, ctx->stream>>>(ctx->mlp_hidden, ctx->F, F_pad, ctx->mlp_params, L,
                                                       reinterpret_cast<__nv_bfloat16*>(ctx->mlp_w2t),
                                                       reinterpret_cast<__nv_bfloat16*>(ctx->mlp_w3t));
    RASCAL_LAUNCH_CHECK("k_mlp_pack");
    return RASCAL_OK;
}

int mlp_infer(rascal_ctx* ctx, int64_t n, const float4* rij, const float* r, float* out, float* dout) {
    if (n == 0) return RASCAL_OK;
    const int F_pad = (ctx->F + 15) / 16 * 16;
    if (F_pad > 256) return set_error(RASCAL_E_UNSUPPORTED, "MLP inference needs n_max*(l_max+1) <= 256");
    MlpInferArgs A;
    A.rij = rij;
    A.r_in = r;
    A.n = n;
    A.out = out;
    A.dout = dout;
    A.P = ctx->mlp_params;
    A.W2t = reinterpret_cast<const __nv_bfloat16*>(ctx->mlp_w2t);
    A.W3t = reinterpret_cast<const __nv_bfloat16*>(ctx->mlp_w3t);
    A.scale = ctx->mlp_scale;
    A.L = mlp_layout(ctx->mlp_hidden, ctx->F);
    A.F_pad = F_pad;
    A.inv_rscale = (float)(1.0 / ctx->r_cut);
    A.flags = ctx->d_flags;
    A.stall_polls = ctx->stall_polls;
    const size_t smem = 8192 + (size_t)F_pad * 128 + (dout ? 4 : 2) * 16384 +
                        sizeof(float) * ((3 * kMlpH + 2 * ctx->F + 3) / 4 * 4 + kMlpThreads / 32 * 32 * 36) + 64;
    const int64_t tiles = (n + kMlpTile - 1) / kMlpTile;
    // one CTA per SM with tangents (all 512 TMEM columns), two without
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, (int64_t)ctx->n_sm * (dout ? 1 : 2));
    k_mlp_infer<<<grid, kMlpThreads, smem, ctx->stream>>>(A);
    RASCAL_LAUNCH_CHECK("k_mlp_infer");
    return RASCAL_OK;
}

int mlp_setup(rascal_ctx* ctx) {
    RASCAL_CUDA(cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    RASCAL_CUDA(cudaFuncSetAttribute(k_mlp_train<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
    RASCAL_CUDA(cudaFuncSetAttribute(k_mlp_train<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
    RASCAL_CUDA(cudaFuncSetAttribute(k_mlp_train<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
    return RASCAL_OK;
}

}  // namespace rascal

extern "C" int rascal_mlp_num_params(const rascal_ctx* ctx, int hidden) {
    if (!ctx || hidden != kMlpH) return -1;
    return mlp_layout(hidden, ctx->F).n;
}

extern "C" int rascal_mlp_set_params(rascal_ctx* ctx, int hidden, const float* h_params, const float* h_scale) {
    clear_error();
    if (!ctx || !h_params || !h_scale) return set_error(RASCAL_E_ARG, "NULL argument");
    if (hidden != kMlpH) return set_error(RASCAL_E_UNSUPPORTED, "the MLP kernels use %d hidden units", kMlpH);
    const MlpLayout L = mlp_layout(hidden, ctx->F);
    const int F_pad = (ctx->F + 15) / 16 * 16;
    if (!ctx->mlp_params) {
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_params, sizeof(float) * L.n));
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_m, sizeof(float) * L.n));
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_v, sizeof(float) * L.n));
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_scale, sizeof(float) * ctx->F));
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_w2t, sizeof(__nv_bfloat16) * hidden * hidden));
        RASCAL_CUDA(cudaMalloc(&ctx->mlp_w3t, sizeof(__nv_bfloat16) * F_pad * hidden));
    }
    ctx->mlp_hidden = hidden;
    ctx->mlp_step = 0;
    RASCAL_CUDA(cudaMemcpyAsync(ctx->mlp_params, h_params, sizeof(float) * L.n, cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(ctx->mlp_scale, h_scale, sizeof(float) * ctx->F, cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaMemsetAsync(ctx->mlp_m, 0, sizeof(float) * L.n, ctx->stream));
    RASCAL_CUDA(cudaMemsetAsync(ctx->mlp_v, 0, sizeof(float) * L.n, ctx->stream));
    int st = mlp_pack(ctx);
    if (st) return st;
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    return RASCAL_OK;
}

extern "C" int rascal_mlp_get_params(rascal_ctx* ctx, float* h_params, float* h_scale) {
    clear_error();
    int st = mlp_check(ctx);
    if (st) return st;
    const MlpLayout L = mlp_layout(ctx->mlp_hidden, ctx->F);
    if (h_params) RASCAL_CUDA(cudaMemcpyAsync(h_params, ctx->mlp_params, sizeof(float) * L.n, cudaMemcpyDeviceToHost, ctx->stream));
    if (h_scale) RASCAL_CUDA(cudaMemcpyAsync(h_scale, ctx->mlp_scale, sizeof(float) * ctx->F, cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    return RASCAL_OK;
}

extern "C" int rascal_mlp_targets(rascal_ctx* ctx, int64_t n, const double* d_r, int dense_intervals, float* d_targets,
                                  float* h_scale_out) {
    clear_error();
    if (!ctx || n < 0 || (n > 0 && (!d_r || !d_targets))) return set_error(RASCAL_E_ARG, "bad argument");
    const int M = dense_intervals > 0 ? dense_intervals : 8192;
    const int n_max = ctx->n_max, L1 = ctx->l_max + 1, F = ctx->F;
    const double delta = ctx->r_cut / M;
    const size_t bytes = carve_bytes((M + 1) * 8, 2 * 8, (size_t)(M + 1) * F * 8, (size_t)2 * F * 8, (size_t)2 * F * 8,
                                     (size_t)F * (M + 1) * 8, (size_t)F * (M + 1) * 8, (size_t)F * 8, (size_t)F * 8);
    void* base;
    int st = arena_get(ctx->scratch, bytes, &base);
    if (st) return st;
    Carver cv(base);
    double* grid = cv.take<double>(M + 1);
    double* ends = cv.take<double>(2);
    double* y = cv.take<double>((size_t)(M + 1) * F);
    double* yend = cv.take<double>((size_t)2 * F);
    double* dyend = cv.take<double>((size_t)2 * F);
    double* cp = cv.take<double>((size_t)F * (M + 1));
    double* y2 = cv.take<double>((size_t)F * (M + 1));
    double* inv_scale = cv.take<double>(F);
    (void)cv.take<double>(F);
    // exact FP64 integrals on the dense grid, clamped spline through them (error ~ 1e-14 at 8192 intervals)
    if ((st = radial_grid_fp64(ctx, M, grid, ends, y, yend, dyend, cp, y2))) return st;
    // per-output scale = max |I| on the grid
    std::vector<double> hy((size_t)(M + 1) * F);
    RASCAL_CUDA(cudaMemcpyAsync(hy.data(), y, sizeof(double) * hy.size(), cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    std::vector<double> inv(F), sc(F);
    for (int f = 0; f < F; ++f) {
        const int l = f / n_max, nn = f % n_max;
        double m = 0.0;
        for (int k = 0; k <= M; ++k) m = std::max(m, std::fabs(hy[((size_t)k * n_max + nn) * L1 + l]));
        sc[f] = m > 0.0 ? m : 1.0;
        inv[f] = 1.0 / sc[f];
        if (h_scale_out) h_scale_out[f] = (float)sc[f];
    }
    RASCAL_CUDA(cudaMemcpyAsync(inv_scale, inv.data(), sizeof(double) * F, cudaMemcpyHostToDevice, ctx->stream));
    if (n > 0) {
        k_spline64_eval<<<(unsigned)div_up(n * F, 256), 256, 0, ctx->stream>>>(n, d_r, M, delta, F, y, y2, n_max, L1,
                                                                             inv_scale, d_targets);
        RASCAL_LAUNCH_CHECK("k_spline64_eval");
    }
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    return RASCAL_OK;
}

extern "C" int rascal_mlp_train(rascal_ctx* ctx, int64_t n_samples, const float* d_t, const float* d_targets,
                                const int64_t* d_order, int batch, int steps, float lr_max, float lr_min, int total_steps,
                                float* d_loss) {
    clear_error();
    int st = mlp_check(ctx);
    if (st) return st;
    if (batch <= 0 || steps < 0 || n_samples < batch || !d_t || !d_targets || !d_order)
        return set_error(RASCAL_E_ARG, "bad training arguments");
    const MlpLayout L = mlp_layout(ctx->mlp_hidden, ctx->F);
    const TrainPlan plan = train_plan(ctx, batch, L.F);
    void* base;
    if ((st = arena_get(ctx->scratch, carve_bytes(sizeof(float) * (size_t)plan.grid * (L.n + 1), sizeof(float) * 4), &base)))
        return st;
    Carver cv(base);
    float* part = cv.take<float>((size_t)plan.grid * (L.n + 1));
    float* loss_sink = cv.take<float>(4);
    const double b1 = 0.9, b2 = 0.999;
    for (int s = 0; s < steps; ++s) {
        const int64_t start = ((int64_t)ctx->mlp_step * batch) % (n_samples - batch + 1);
        ++ctx->mlp_step;
        const int T = total_steps > 0 ? total_steps : steps;
        const double prog = std::min(1.0, (double)(ctx->mlp_step - 1) / std::max(1, T - 1));
        AdamArgs adam;
        adam.P = ctx->mlp_params;
        adam.m = ctx->mlp_m;
        adam.v = ctx->mlp_v;
        adam.lr = (float)(lr_min + 0.5 * (lr_max - lr_min) * (1.0 + std::cos(3.14159265358979 * prog)));
        adam.beta1 = (float)b1;
        adam.beta2 = (float)b2;
        adam.eps = 1e-8f;
        adam.bc1 = (float)(1.0 - std::pow(b1, ctx->mlp_step));
        adam.bc2 = (float)(1.0 - std::pow(b2, ctx->mlp_step));
        if ((st = mlp_step(ctx, L, plan, batch, d_order + start, d_t, d_targets, part, nullptr, d_loss ? d_loss + s : loss_sink, &adam)))
            return st;
    }
    return mlp_pack(ctx);
}

extern "C" int rascal_mlp_gradients(rascal_ctx* ctx, int batch, const float* d_t, const float* d_targets, float* d_grad,
                                    float* d_loss) {
    clear_error();
    int st = mlp_check(ctx);
    if (st) return st;
    if (batch <= 0 || !d_t || !d_targets || !d_grad || !d_loss) return set_error(RASCAL_E_ARG, "bad argument");
    const MlpLayout L = mlp_layout(ctx->mlp_hidden, ctx->F);
    const TrainPlan plan = train_plan(ctx, batch, L.F);
    void* part;
    if ((st = arena_get(ctx->scratch, sizeof(float) * (size_t)plan.grid * (L.n + 1), &part))) return st;
    return mlp_step(ctx, L, plan, batch, nullptr, d_t, d_targets, static_cast<float*>(part), d_grad, d_loss, nullptr);
}

extern "C" int rascal_mlp_eval(rascal_ctx* ctx, int64_t n, const float* d_r, float* d_out, float* d_dout) {
    clear_error();
    int st = mlp_check(ctx);
    if (st) return st;
    if (n < 0 || (n > 0 && (!d_r || !d_out))) return set_error(RASCAL_E_ARG, "bad argument");
    return mlp_infer(ctx, n, nullptr, d_r, d_out, d_dout);
}

extern "C" int rascal_mlp_save(rascal_ctx* ctx, const char* path) {
    clear_error();
    int st = mlp_check(ctx);
    if (st) return st;
    if (!path) return set_error(RASCAL_E_ARG, "NULL path");
    const MlpLayout L = mlp_layout(ctx->mlp_hidden, ctx->F);
    std::vector<float> p(L.n), m(L.n), v(L.n), s(ctx->F);
    RASCAL_CUDA(cudaMemcpyAsync(p.data(), ctx->mlp_params, sizeof(float) * L.n, cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(m.data(), ctx->mlp_m, sizeof(float) * L.n, cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(v.data(), ctx->mlp_v, sizeof(float) * L.n, cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(s.data(), ctx->mlp_scale, sizeof(float) * ctx->F, cudaMemcpyDeviceToHost, ctx->stream));
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    FILE* fh = std::fopen(path, "wb");
    if (!fh) return set_error(RASCAL_E_ARG, "cannot open %s for writing", path);
    const int32_t hdr[8] = {0x52534d4c /* 'RSML' */, 1, ctx->mlp_hidden, ctx->F, ctx->n_max, ctx->l_max, L.n, ctx->mlp_step};
    const double hyp[2] = {ctx->r_cut, ctx->sigma};
    bool okw = std::fwrite(hdr, sizeof(hdr), 1, fh) == 1 && std::fwrite(hyp, sizeof(hyp), 1, fh) == 1 &&
               std::fwrite(p.data(), sizeof(float), L.n, fh) == (size_t)L.n && std::fwrite(m.data(), sizeof(float), L.n, fh) == (size_t)L.n &&
               std::fwrite(v.data(), sizeof(float), L.n, fh) == (size_t)L.n && std::fwrite(s.data(), sizeof(float), ctx->F, fh) == (size_t)ctx->F;
    std::fclose(fh);
    if (!okw) return set_error(RASCAL_E_ARG, "short write to %s", path);
    return RASCAL_OK;
}

extern "C" int rascal_mlp_load(rascal_ctx* ctx, const char* path) {
    clear_error();
    if (!ctx || !path) return set_error(RASCAL_E_ARG, "NULL argument");
    FILE* fh = std::fopen(path, "rb");
    if (!fh) return set_error(RASCAL_E_ARG, "cannot open %s", path);
    int32_t hdr[8];
    double hyp[2];
    bool okr = std::fread(hdr, sizeof(hdr), 1, fh) == 1 && std::fread(hyp, sizeof(hyp), 1, fh) == 1;
    if (!okr || hdr[0] != 0x52534d4c || hdr[1] != 1 || hdr[3] != ctx->F || hdr[4] != ctx->n_max || hdr[5] != ctx->l_max ||
        hyp[0] != ctx->r_cut || hyp[1] != ctx->sigma) {
        std::fclose(fh);
        return set_error(RASCAL_E_ARG, "%s holds an MLP for other hypers or is not an MLP checkpoint", path);
    }
    const MlpLayout L = mlp_layout(hdr[2], ctx->F);
    if (L.n != hdr[6]) {
        std::fclose(fh);
        return set_error(RASCAL_E_ARG, "%s: parameter count mismatch", path);
    }
    std::vector<float> p(L.n), m(L.n), v(L.n), s(ctx->F);
    okr = std::fread(p.data(), sizeof(float), L.n, fh) == (size_t)L.n && std::fread(m.data(), sizeof(float), L.n, fh) == (size_t)L.n &&
          std::fread(v.data(), sizeof(float), L.n, fh) == (size_t)L.n && std::fread(s.data(), sizeof(float), ctx->F, fh) == (size_t)ctx->F;
    std::fclose(fh);
    if (!okr) return set_error(RASCAL_E_ARG, "%s is truncated", path);
    int st = rascal_mlp_set_params(ctx, hdr[2], p.data(), s.data());
    if (st) return st;
    RASCAL_CUDA(cudaMemcpyAsync(ctx->mlp_m, m.data(), sizeof(float) * L.n, cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(ctx->mlp_v, v.data(), sizeof(float) * L.n, cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    ctx->mlp_step = hdr[7];
    return RASCAL_OK;
}
