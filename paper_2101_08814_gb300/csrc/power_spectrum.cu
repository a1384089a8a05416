// Power spectrum (Eq. nu2-basis-coupled) from stored coefficients, p_l = k_l C_l C_l^T per centre and l.
//
// One CTA per centre. The centre's block c[q][lm] comes in as it lies in memory (cp.async, rows at a pitch that keeps the
// loads below off each other's banks); p is staged per group of l over two alternating halves and leaves by bulk copies.
// The Gram itself is too small per centre (48 x 48 x 2l+1 at the batch hypers) for anything but operands in registers:
//   BF16, TF32x3  warp-level tensor-core MMAs (m16n8k16 / m16n8k8). An item is 16 rows x up to four 8-column blocks left
//                 of the diagonal and the two on it, or the six tiles of a 32-row diagonal block; rows serve as A and B
//                 fragments alike, so a block of eight rows is loaded (and rounded or split) once per item. The warps take
//                 a group's items, largest first, as they come free. tcgen05 needs its operands re-tiled in shared memory,
//                 a wait per l and a TMEM read per column block, which at these sizes cost more than the products.
//   FP32          8 x 4 tiles per thread over the rows q1 = t1 + H u and columns q2 = t2 + 2 H w (H = ceil(Q / 8)), paired
//                 FMAs, m in order. A tile is made for every t2 mod H >= t1, which meets every unordered pair once.
//                 Interleaved columns let lanes of neighbouring tiles write neighbouring words.
// Bound: HBM (c in, p out). 20 000 centres, Q = 48, l_max 9, PACKED: BF16 813 -> 283 us (0.70 of HBM), TF32x3 1 454 -> 372 us
// (error against 64 bits 6.4e-7 -> 1.9e-7: the high part of the split is rounded, not cut off), FP32 573 -> 436 us, bit for bit (bound by its
// shared-memory loads, 12 floats for 32 products); FULL: 1 253 -> 465, 2 014 -> 561, 1 391 -> 678 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "f32x2.cuh"
#include "ps_fp32.cuh"
#include "stage.cuh"

namespace rascal {

constexpr int kPsThreads = 256;     // of k_power_spectrum_direct, and of k_power_spectrum at first (ps_plan)
constexpr int kPsMaxThreads = 512;  // of k_power_spectrum (64 registers)
constexpr int kPsStage = 7168;  // floats of the two staging halves (28 KB: four CTAs per SM at the batch hypers)
constexpr int kPsOff = 4;       // 8-column blocks left of the diagonal in one item

struct PsArgs {
    const float* c;
    float* ps;
    int64_t ps_stride;
    const unsigned* items;
    int items_per_l, Q, l_max, pitch, per_l, half, n_half, ps_norm, copy16;
};

// D += A B, the warp-level tensor-core path (FP32 accumulation): A 16 rows, B 8 columns, both as register fragments
__device__ __forceinline__ void mma_bf16_16x8x16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_tf32_16x8x8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// eight rows x K terms of the sum, as A or B fragment (K = 16 BF16, 8 TF32 high and low)
template <int PREC>
struct PsFrag {
    uint32_t h[2], l[PREC == RASCAL_PS_TF32X3 ? 2 : 1];
};

// the lane's row at its first term, `left` terms to the end of the l block (past it: zero)
template <int PREC>
__device__ __forceinline__ PsFrag<PREC> ps_load(const float* p, int t4, int left) {
    PsFrag<PREC> f;
    if (PREC == RASCAL_PS_BF16) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = 2 * t4 + 8 * e;
            const __nv_bfloat162 v = __floats2bfloat162_rn(k < left ? p[k] : 0.0f, k + 1 < left ? p[k + 1] : 0.0f);
            f.h[e] = *reinterpret_cast<const uint32_t*>(&v);
        }
    } else {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = t4 + 4 * e;
            const float x = k < left ? p[k] : 0.0f;
            // high: rounded to the nearest TF32 value; low: what is left, of which the tensor core drops the last bits
            // (below 2^-23 of x, either sign)
            f.h[e] = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
            f.l[PREC == RASCAL_PS_TF32X3 ? e : 0] = __float_as_uint(x - __uint_as_float(f.h[e]));
        }
    }
    return f;
}

template <int PREC>
__device__ __forceinline__ void ps_mma(float (&d)[4], const PsFrag<PREC>& a0, const PsFrag<PREC>& a1, const PsFrag<PREC>& b) {
    if (PREC == RASCAL_PS_BF16) {
        mma_bf16_16x8x16(d, a0.h[0], a1.h[0], a0.h[1], a1.h[1], b.h[0], b.h[1]);
    } else {
        constexpr int k = PREC == RASCAL_PS_TF32X3 ? 1 : 0;
        mma_tf32_16x8x8(d, a0.l[0], a1.l[0], a0.l[k], a1.l[k], b.h[0], b.h[1]);
        mma_tf32_16x8x8(d, a0.h[0], a1.h[0], a0.h[1], a1.h[1], b.l[0], b.l[k]);
        mma_tf32_16x8x8(d, a0.h[0], a1.h[0], a0.h[1], a1.h[1], b.h[0], b.h[1]);
    }
}

// one warp item of l into the staged l block o
template <int PREC, bool FULL>
__device__ __forceinline__ void ps_warp_item(const float* C, int pitch, int Q, int l, unsigned item, float kl, float* o) {
    constexpr int KS = PREC == RASCAL_PS_BF16 ? 16 : 8;
    const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
    const int r0 = (int)(item & 0xff) * 16, j0 = (item >> 8) & 0xff, nj = (item >> 16) & 0xff;
    const bool diag = item >> 24 & 1, pair = item >> 25 & 1;
    const int terms = 2 * l + 1, rows8 = 8 * pitch;
    float acc[6][4];
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.0f;
    const float* a = C + (r0 + g) * pitch + l * l;
    const float* b = C + (8 * j0 + g) * pitch + l * l;
#pragma unroll 1
    for (int k = 0; k < terms; k += KS) {
        const int left = terms - k;
        const PsFrag<PREC> u0 = ps_load<PREC>(a + k, t4, left), u1 = ps_load<PREC>(a + rows8 + k, t4, left);
        if (pair) {  // the lower triangle of a 32-row block
            ps_mma<PREC>(acc[0], u0, u1, u0);
            ps_mma<PREC>(acc[1], u0, u1, u1);
            const PsFrag<PREC> u2 = ps_load<PREC>(a + 2 * rows8 + k, t4, left), u3 = ps_load<PREC>(a + 3 * rows8 + k, t4, left);
            ps_mma<PREC>(acc[2], u2, u3, u0);
            ps_mma<PREC>(acc[3], u2, u3, u1);
            ps_mma<PREC>(acc[4], u2, u3, u2);
            ps_mma<PREC>(acc[5], u2, u3, u3);
        } else {
            if (diag) {
                ps_mma<PREC>(acc[4], u0, u1, u0);
                ps_mma<PREC>(acc[5], u0, u1, u1);
            }
#pragma unroll
            for (int j = 0; j < kPsOff; ++j) {
                if (j >= nj) break;
                ps_mma<PREC>(acc[j], u0, u1, ps_load<PREC>(b + j * rows8 + k, t4, left));
            }
        }
    }
    // Entry (row r, column q), q <= r, of the symmetric block: PACKED at q (2Q - q - 1) / 2 + r, so that lanes of
    // neighbouring rows write neighbouring words; FULL at q Q + r and r Q + q.
    auto put = [&](const float (&d)[4], int r, int q, bool p0, bool p1, bool p2, bool p3) {
        p0 = p0 && r < Q;
        p1 = p1 && r < Q;
        p2 = p2 && r + 8 < Q;
        p3 = p3 && r + 8 < Q;
        float* o0 = o + (FULL ? q * Q : (q * (2 * Q - q - 1)) / 2) + r;
        float* o1 = o0 + (FULL ? Q : Q - 1 - q);  // the next column's
        const float v0 = kl * d[0], v1 = kl * d[1], v2 = kl * d[2], v3 = kl * d[3];
        if (p0) o0[0] = v0;
        if (p1) o1[0] = v1;
        if (p2) o0[8] = v2;
        if (p3) o1[8] = v3;
        if (FULL) {
            float* m = o + r * Q + q;
            if (p0) m[0] = v0;
            if (p1) m[1] = v1;
            if (p2) m[8 * Q] = v2;
            if (p3) m[8 * Q + 1] = v3;
        }
    };
    const int c2 = 2 * t4;
    const bool w0 = c2 <= g, w1 = c2 < g;  // columns c2 and c2 + 1 not right of row g of a diagonal tile
    const int r = r0 + g;
    if (pair) {
        put(acc[0], r, r0 + c2, w0, w1, true, true);
        put(acc[1], r, r0 + 8 + c2, false, false, w0, w1);
        put(acc[2], r + 16, r0 + c2, true, true, true, true);
        put(acc[3], r + 16, r0 + 8 + c2, true, true, true, true);
        put(acc[4], r + 16, r0 + 16 + c2, w0, w1, true, true);
        put(acc[5], r + 16, r0 + 24 + c2, false, false, w0, w1);
        return;
    }
    if (diag) {
        put(acc[4], r, r0 + c2, w0, w1, true, true);
        put(acc[5], r, r0 + 8 + c2, false, false, w0, w1);
    }
#pragma unroll
    for (int j = 0; j < kPsOff; ++j) {
        if (j >= nj) break;
        put(acc[j], r, 8 * (j0 + j) + c2, true, true, true, true);
    }
}

// one thread tile of l (FP32) into the staged l block o; rows and columns past Q are computed and not stored
template <bool FULL>
__device__ __forceinline__ void ps_thread_tile(const float* C, int pitch, int Q, int H, int l, int t1, int t2, float kl, float* o) {
    const float* a = C + t1 * pitch + l * l;
    const float* b = C + t2 * pitch + l * l;
    const int hp = H * pitch;
    uint64_t acc[4][4];  // rows (2 v, 2 v + 1) x column w
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[v][w] = 0ull;
#pragma unroll 1
    for (int m = 2 * l; m >= 0; --m, ++a, ++b) {
        uint64_t x[4], y[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) x[v] = f2_pack(a[2 * v * hp], a[(2 * v + 1) * hp]);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const float z = b[2 * w * hp];
            y[w] = f2_pack(z, z);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[v][w] = f2_fma(x[v], y[w], acc[v][w]);
    }
    // q1 = t1 + H u and q2 = t2 + 2 H w = (t2 mod H) + H e, e = 2 w + (t2 >= H)
    auto value = [&](int u, int w) {
        float x, y;
        f2_unpack(acc[u >> 1][w], x, y);
        return kl * ((u & 1) ? y : x);
    };
    bool in2[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) in2[w] = t2 + 2 * H * w < Q;
    if (FULL) {  // every class pair has its tile: row by row
        float* row = o + t1 * Q + t2;
#pragma unroll
        for (int u = 0; u < 8; ++u, row += H * Q) {
            if (t1 + H * u >= Q) break;
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (in2[w]) row[2 * H * w] = value(u, w);
        }
        return;
    }
    // PACKED entry (q, q'), q <= q', at q (2Q - q - 1) / 2 + q'. The tile has t1 <= t2 mod H, so q1 <= q2 for u <= e and
    // q2 < q1 for u > e, where a tile of equal classes repeats another one's entries.
    const bool odd = t2 >= H, same = t1 == (odd ? t2 - H : t2);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int q1 = t1 + H * u;
        if (q1 >= Q) break;
        float* row = o + (q1 * (2 * Q - q1 - 1)) / 2 + t2;
        if ((u & 1) && odd && in2[u >> 1]) row[2 * H * (u >> 1)] = value(u, u >> 1);  // u = 2 w + 1: here for odd e only
#pragma unroll
        for (int w = (u + 1) >> 1; w < 4; ++w)
            if (in2[w]) row[2 * H * w] = value(u, w);
    }
    if (same) return;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        if (!in2[w]) break;
        const int q2 = t2 + 2 * H * w;
        float* row = o + (q2 * (2 * Q - q2 - 1)) / 2 + t1;
        if (!odd && t1 + H * (2 * w + 1) < Q) row[H * (2 * w + 1)] = value(2 * w + 1, w);
#pragma unroll
        for (int u = 2 * w + 2; u < 8; ++u)
            if (t1 + H * u < Q) row[H * u] = value(u, w);
    }
}

template <int PREC, bool FULL>
__global__ void __launch_bounds__(kPsMaxThreads, 2) k_power_spectrum(const PsArgs A) {
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_next[kMaxLMax + 1];  // next item of each group
    const int Q = A.Q, L1 = A.l_max + 1, n_lm = L1 * L1, pitch = A.pitch, tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
    float* stage = sm;                     // [2][half]
    float* C = sm + 2 * A.half;            // rows past Q are read by edge tiles, whose results are not stored
    const float* c = A.c + (int64_t)blockIdx.x * Q * n_lm;
    if (A.copy16) {  // pitch = n_lm and every centre's block 16-byte aligned
        for (int e = tid; e < Q * n_lm / 4; e += nthr) cp_async16_zfill(C + 4 * e, c + 4 * e, 16u);
    } else {
        for (int q = tid >> 5; q < Q; q += nthr >> 5)
            for (int lm = lane; lm < n_lm; lm += 32) cp_async4(C + q * pitch + lm, c + q * n_lm + lm);
    }
    for (int e = tid; e <= kMaxLMax; e += nthr) s_next[e] = 0;
    cp_async_wait_all();
    __syncthreads();
    float* pout = A.ps + (int64_t)blockIdx.x * A.ps_stride;
    const int H = (Q + 7) >> 3;
    for (int gi = 0, hi = L1; hi > 0; ++gi) {
        const int n = min(A.n_half, hi), lo = hi - n;
        const unsigned* items = A.items + (int64_t)(L1 - hi) * A.items_per_l;
        const int n_items = n * A.items_per_l;
        float* dst = pout + (int64_t)lo * A.per_l;
        float* st = stage + (gi & 1) * A.half + stage_shift(dst);
        if (PREC == RASCAL_PS_FP32) {
            for (int it = tid; it < n_items; it += nthr) {
                const unsigned t = __ldg(items + it);
                const int l = t >> 26;
                ps_thread_tile<FULL>(C, pitch, Q, H, l, t & 0xff, (t >> 8) & 0xff, A.ps_norm ? rsqrtf((float)(2 * l + 1)) : 1.0f,
                                     st + (l - lo) * A.per_l);
            }
        } else {
            for (;;) {  // the warps take the items as they come free
                int it = 0;
                if (lane == 0) it = atomicAdd(&s_next[gi], 1);
                it = __shfl_sync(0xffffffffu, it, 0);
                if (it >= n_items) break;
                const unsigned t = __ldg(items + it);
                const int l = t >> 26;
                ps_warp_item<PREC, FULL>(C, pitch, Q, l, t, A.ps_norm ? rsqrtf((float)(2 * l + 1)) : 1.0f, st + (l - lo) * A.per_l);
            }
        }
        fence_proxy_async_smem();
        if (tid == 0 && gi >= 1) bulk_wait_read<0>();  // the store of gi - 1 is done with the half of gi + 1
        __syncthreads();
        if (tid < 32) store_staged(dst, st, n * A.per_l);
        hi = lo;
    }
    if (tid == 0) bulk_wait_all();
}

// FP32 without staging, for bases whose two staged l blocks do not fit shared memory beside the coefficients: c transposed to
// CT[lm][q], 4 x 4 tiles (ps_fp32.cuh), p stored straight to global memory.
__global__ void __launch_bounds__(kPsThreads) k_power_spectrum_direct(const float* __restrict__ coeffs, int Q, int Qp, int n_lm,
                                                                       int l_max, int ps_norm, const int* __restrict__ tasks,
                                                                       int n_tasks, int layout, int64_t ps_stride,
                                                                       float* __restrict__ ps) {
    extern __shared__ __align__(16) float CT[];  // [n_lm][Qp]
    const int64_t i = blockIdx.x;
    const float* c = coeffs + i * (int64_t)Q * n_lm;
    const int total = Q * n_lm;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int q = e / n_lm, lm = e - q * n_lm;
        CT[lm * Qp + q] = c[e];
    }
    for (int e = threadIdx.x; e < n_lm * (Qp - Q); e += blockDim.x) {
        const int lm = e / (Qp - Q), q = Q + e % (Qp - Q);
        CT[lm * Qp + q] = 0.0f;
    }
    __syncthreads();
    ps_gram_fp32(CT, Qp, Q, l_max, ps_norm, tasks, n_tasks, layout, ps + i * ps_stride);
}

static int power_spectrum_direct(rascal_ctx* ctx, int64_t n_centres, const float* d_coeffs, int layout, float* d_ps) {
    const int Q = ctx->Q, Qp = (Q + 3) / 4 * 4;
    const int64_t stride = (int64_t)(ctx->l_max + 1) * (layout == RASCAL_LAYOUT_PACKED ? (int64_t)Q * (Q + 1) / 2 : (int64_t)Q * Q);
    const size_t smem = sizeof(float) * ctx->n_lm * Qp;
    k_power_spectrum_direct<<<(unsigned)n_centres, kPsThreads, smem, ctx->stream>>>(
        d_coeffs, Q, Qp, ctx->n_lm, ctx->l_max, ctx->ps_norm, ctx->d_pstasks, ctx->n_pstasks, layout, stride, d_ps);
    RASCAL_LAUNCH_CHECK("k_power_spectrum_direct");
    return RASCAL_OK;
}

// Warp items of one l: 32-row diagonal blocks, what lies left of them by 16 rows x kPsOff column blocks, and a last single
// 16-row block with its diagonal. Packed row block (of 16) | first column block (of 8) << 8 | column blocks << 16 |
// diagonal << 24 | 32-row block << 25 | l << 26.
static void ps_warp_items(int Q, int l, std::vector<unsigned>& v) {
    const int mt = (Q + 15) / 16;
    const unsigned hl = (unsigned)l << 26;
    for (int i = 0; i + 1 < mt; i += 2) v.push_back(hl | 1u << 25 | (unsigned)i);
    for (int i = 0; i < mt; ++i) {
        const bool lone = i == mt - 1 && mt % 2 == 1;
        const int n = lone ? 2 * i : 4 * (i / 2);  // column blocks left of the diagonal (block)
        for (int a = 0; a < n || (lone && a == 0); a += kPsOff)
            v.push_back(hl | (unsigned)i | (unsigned)a << 8 | (unsigned)std::min(kPsOff, n - a) << 16 | (lone && a == 0 ? 1u << 24 : 0u));
    }
}
// thread tiles of one l, packed t1 | t2 << 8 | l << 26: PACKED the class pairs with t1 <= t2 mod H, FULL all of them
static void ps_thread_items(int Q, int l, bool full, std::vector<unsigned>& v) {
    const int H = (Q + 7) / 8;
    for (int t1 = 0; t1 < H; ++t1)
        for (int t2 = 0; t2 < 2 * H; ++t2)
            if (full || t1 <= t2 % H) v.push_back((unsigned)l << 26 | (unsigned)t2 << 8 | (unsigned)t1);
}

// Row pitch: the first length from n_lm on at which the loads meet a bank at most twice (the warp items' 8 rows x 4 terms),
// or odd (the thread tiles' neighbouring rows)
static int ps_pitch(int n_lm, int precision) {
    if (precision == RASCAL_PS_FP32) return n_lm | 1;
    for (int p = n_lm;; ++p) {
        int n[32] = {}, worst = 0;
        for (int g = 0; g < 8; ++g)
            for (int t = 0; t < 4; ++t) worst = std::max(worst, ++n[(g * p + (precision == RASCAL_PS_BF16 ? 2 * t : t)) % 32]);
        if (worst <= 2) return p;
    }
}

template <int PREC>
static int ps_set_attr() {
    RASCAL_CUDA(cudaFuncSetAttribute(k_power_spectrum<PREC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    RASCAL_CUDA(cudaFuncSetAttribute(k_power_spectrum<PREC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    return RASCAL_OK;
}

static void ps_plan(const rascal_ctx* ctx, int precision, int layout, int per_sm, PsPlan& P);

int power_spectrum_setup(rascal_ctx* ctx) {
    const int Q4 = (ctx->Q + 3) / 4;
    std::vector<int> tasks;  // of the fused kernel's Gram
    for (int l = ctx->l_max; l >= 0; --l)
        for (int t1 = 0; t1 < Q4; ++t1)
            for (int t2 = t1; t2 < Q4; ++t2) tasks.push_back(l | (t1 << 8) | (t2 << 16));
    ctx->n_pstasks = (int)tasks.size();
    std::vector<unsigned> items;
    for (int kind = 0; kind < 3; ++kind) {
        const size_t before = items.size();
        for (int l = ctx->l_max; l >= 0; --l) kind == 0 ? ps_warp_items(ctx->Q, l, items) : ps_thread_items(ctx->Q, l, kind == 2, items);
        ctx->n_psitems[kind] = (int)((items.size() - before) / (ctx->l_max + 1));
    }
    for (int p = 0; p < 3; ++p)
        for (int layout = 0; layout < 2; ++layout)
            for (int k = 0; k < kPsPlans; ++k) ps_plan(ctx, p, layout, k + 1 < kPsPlans ? k + 1 : 64, ctx->ps_plan[p][layout][k]);
    RASCAL_CUDA(cudaMalloc(&ctx->d_pstasks, sizeof(int) * tasks.size()));
    RASCAL_CUDA(cudaMalloc(&ctx->d_psitems, sizeof(unsigned) * items.size()));
    RASCAL_CUDA(cudaMemcpyAsync(ctx->d_pstasks, tasks.data(), sizeof(int) * tasks.size(), cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaMemcpyAsync(ctx->d_psitems, items.data(), sizeof(unsigned) * items.size(), cudaMemcpyHostToDevice, ctx->stream));
    RASCAL_CUDA(cudaFuncSetAttribute(k_power_spectrum_direct, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    int st;
    if ((st = ps_set_attr<RASCAL_PS_FP32>()) || (st = ps_set_attr<RASCAL_PS_BF16>()) || (st = ps_set_attr<RASCAL_PS_TF32X3>())) return st;
    RASCAL_CUDA(cudaStreamSynchronize(ctx->stream));
    return RASCAL_OK;
}

// How k_power_spectrum is launched for per_sm centres per SM: kPsStage floats of staging and 256 threads at first. Groups of few
// items leave an SM half empty in wide bases (one l of Q = 60, PACKED FP32: 72 threads of a CTA) and in small batches, whose
// single CTA per SM then runs l by l. There the staging grows to the l blocks, and the CTA to the threads, that put most threads
// to work, in larger batches up to half of the l blocks only (what a group stores has to overlap the next one's tiles: whole
// centres at once made 4 000 of Q = 36, l_max 8, FULL 72 -> 93 us), and only where fewer than 480 (tensor cores 448) are at
// work on an SM. Before -> so, 4 000 centres PACKED FP32: (Q 60, l_max 15) 615 -> 342 us, (128, 4) 235 -> 172, (96, 15) 1 212 ->
// 653; one centre: (64, 12) 31 -> 12, TF32x3 FULL (48, 9) 26 -> 13.
static void ps_plan(const rascal_ctx* ctx, int precision, int layout, int per_sm, PsPlan& P) {
    const int Q = ctx->Q, L1 = ctx->l_max + 1;
    const bool full = layout == RASCAL_LAYOUT_FULL, fp32 = precision == RASCAL_PS_FP32;
    const int per_l = full ? Q * Q : Q * (Q + 1) / 2, pitch = ps_pitch(ctx->n_lm, precision);
    const int items = ctx->n_psitems[!fp32 ? 0 : (full ? 2 : 1)] * (fp32 ? 1 : 32);  // threads that an l occupies
    const int rows = fp32 ? (Q + 7) / 8 * 8 : (Q + 15) / 16 * 16;  // of c that edge tiles read
    auto plan = [&](int n, int threads) {
        // a staging half: a block of l each, three floats more for a start that matches its target's alignment
        const int half = (n * per_l + 3 + 3) / 4 * 4;
        return PsPlan{n, threads, half, pitch, sizeof(float) * ((size_t)2 * half + (size_t)rows * pitch + 32)};
    };
    // threads at work: of one CTA, the items of a group over the rounds that they take (FP32: dealt in rounds; else the warps take
    // them as they come free), and of an SM, on average over the waves of its `centres` CTAs
    auto fit = [&](const PsPlan& p) { return std::min({(int)(227 * 1024 / (p.smem + 1024)), 1024 / p.threads, 32}); };
    auto busy = [&](const PsPlan& p, int centres) {
        const int n = p.n_half * items, one = fp32 ? n / ((n + p.threads - 1) / p.threads) : std::min(n, p.threads);
        return centres * one / ((centres + fit(p) - 1) / fit(p));
    };
    const int n0 = std::max(1, std::min(L1, (kPsStage / 2 - 3) / per_l));
    P = plan(n0, std::min(kPsThreads, (int)align_up(n0 * items, 32)));
    if (P.smem > 220 * 1024 || (per_sm > 2 && busy(P, fit(P)) >= (fp32 ? 480 : 448))) return;
    PsPlan best = P;
    for (int n = 1; n <= (per_sm > 4 ? std::max(1, L1 / 2) : L1); ++n) {
        const int rounds = (n * items + kPsMaxThreads - 1) / kPsMaxThreads;
        const PsPlan p = plan(n, (int)align_up((n * items + rounds - 1) / rounds, 32));
        if (p.smem <= 220 * 1024 && busy(p, per_sm) > busy(best, per_sm)) best = p;
    }
    if (busy(best, per_sm) * 10 > busy(P, per_sm) * 13) P = best;
}

bool power_spectrum_fits(const rascal_ctx* ctx, int precision, int layout) {
    return ctx->ps_plan[precision][layout][0].smem <= 220 * 1024;
}

int power_spectrum_warp(rascal_ctx* ctx, int64_t n_centres, const float* d_coeffs, int precision, int layout, float* d_ps) {
    const bool full = layout == RASCAL_LAYOUT_FULL;
    const int Q = ctx->Q, L1 = ctx->l_max + 1;
    int k = 0;
    while (k + 1 < kPsPlans && n_centres > (k + 1LL) * ctx->n_sm) ++k;
    const PsPlan& P = ctx->ps_plan[precision][layout][k];
    if (P.smem > 220 * 1024) return RASCAL_E_UNSUPPORTED;
    PsArgs A;
    A.c = d_coeffs;
    A.ps = d_ps;
    A.Q = Q;
    A.l_max = ctx->l_max;
    A.per_l = full ? Q * Q : Q * (Q + 1) / 2;
    A.ps_stride = (int64_t)L1 * A.per_l;
    A.ps_norm = ctx->ps_norm;
    A.pitch = P.pitch;
    const int kind = precision != RASCAL_PS_FP32 ? 0 : (full ? 2 : 1);
    A.items_per_l = ctx->n_psitems[kind];
    A.items = ctx->d_psitems;
    for (int e = 0; e < kind; ++e) A.items += (int64_t)ctx->n_psitems[e] * L1;
    A.n_half = P.n_half;
    A.half = P.half;
    A.copy16 = A.pitch == ctx->n_lm && Q * ctx->n_lm % 4 == 0 && (reinterpret_cast<uintptr_t>(d_coeffs) & 15) == 0;
    auto kernel = precision == RASCAL_PS_BF16 ? (full ? k_power_spectrum<RASCAL_PS_BF16, true> : k_power_spectrum<RASCAL_PS_BF16, false>)
                  : precision == RASCAL_PS_TF32X3
                      ? (full ? k_power_spectrum<RASCAL_PS_TF32X3, true> : k_power_spectrum<RASCAL_PS_TF32X3, false>)
                      : (full ? k_power_spectrum<RASCAL_PS_FP32, true> : k_power_spectrum<RASCAL_PS_FP32, false>);
    kernel<<<(unsigned)n_centres, P.threads, P.smem, ctx->stream>>>(A);
    RASCAL_LAUNCH_CHECK("k_power_spectrum");
    return RASCAL_OK;
}

}  // namespace rascal

using namespace rascal;

extern "C" int rascal_power_spectrum(rascal_ctx* ctx, int64_t n_centres, const float* d_coeffs, int precision,
                                     int layout, float* d_ps) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (n_centres < 0) return set_error(RASCAL_E_ARG, "negative n_centres");
    if (layout != RASCAL_LAYOUT_PACKED && layout != RASCAL_LAYOUT_FULL) return set_error(RASCAL_E_ARG, "unknown layout");
    if (precision < RASCAL_PS_FP32 || precision > RASCAL_PS_TF32X3) return set_error(RASCAL_E_ARG, "unknown precision");
    if (n_centres == 0) return RASCAL_OK;
    if (!d_coeffs || !d_ps) return set_error(RASCAL_E_ARG, "NULL device pointer");
    if (n_centres > 0x7fffffffLL) return set_error(RASCAL_E_UNSUPPORTED, "more than 2^31-1 centres in one call");
    if (precision != RASCAL_PS_FP32) return power_spectrum_tc(ctx, n_centres, d_coeffs, precision, layout, d_ps);
    const int st = power_spectrum_warp(ctx, n_centres, d_coeffs, precision, layout, d_ps);
    return st != RASCAL_E_UNSUPPORTED ? st : power_spectrum_direct(ctx, n_centres, d_coeffs, layout, d_ps);
}
