// Additive linear energy (Eq. additive-energy-model) and the analytic backward pass (Appendix B).
//
// For E = sum_i G_i . p_i (PACKED p), the pair gradient is
//   dE/dr_ji = sum_{n l m} chat^i_{a_j n l m} grad_r [ f_cut(r) I^o_nl(r) Y_lm(r^) ],
//   chat^i_l = k_l (W_l + W_l^T) C^i_l,   k_l = (2l+1)^-1/2,
// where W_l is G_i's l-block in packed upper-triangular form (zeros below the diagonal). The weights are
// contracted with the coefficients first (the adjoint chat, per centre) and only then with the per-pair feature
// gradients, the order of Eq. gpr-force-order; dc/dr is never stored: each pair's radial values, their
// r-derivatives, Y_lm and its Cartesian gradient are recomputed.
//
// With u = r/|r|, s = sum_lm Y_lm sum_n chat_{n lm} (f I_nl)' and w = sum_lm (sum_n chat_{n lm} f I_nl) dY_lm/du
// (the gradient of the polynomial extension of Y in the unit-vector components),
//   dE/dr_ji = s u + (w - (w.u) u)/|r|.
// Forces: F_j -= dE/dr_ji, F_i += dE/dr_ji (skipped when j is an image of i: the two cancel, Appendix B);
// virial V[a][b] += dE/dr_ji[a] r_ji[b] (images of i included).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "ps_fp32.cuh"
#include "tcgen05.cuh"
#include "ylm_fp32.cuh"

namespace rascal {

// Structure of atom i: the largest s < n_s with offs[s] <= i (offsets non-decreasing, offs[n_s] = the atom count),
// found by one warp in rounds of 32 probes (two rounds for up to 1024 structures); every lane returns it.
__device__ inline int warp_find_structure(const int* __restrict__ offs, int n_s, int i, int lane) {
    int lo = 0, hi = n_s;  // offs[lo] <= i < offs[hi]
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) >> 5;
        const int idx = lo + lane * step;
        const unsigned m = __ballot_sync(0xffffffffu, idx < hi && offs[idx] <= i);  // a prefix of the lanes
        lo += (31 - __clz(m)) * step;
        hi = min(hi, lo + step);
    }
    return lo;
}

// E_s = sum_{i in s} w_{a_i} . p_i, one CTA per centre, FP32 partial sums, FP64 across warps and one atomic per centre.
__global__ void k_linear_energy(int N, int n_s, const int* __restrict__ offs, const int* __restrict__ species,
                                const int* __restrict__ lut, const float* __restrict__ ps, const float* __restrict__ w,
                                int64_t F, double* __restrict__ energy) {
    __shared__ double red[32];
    const int i = blockIdx.x;
    int sid = 0;
    if (threadIdx.x < 32) sid = warp_find_structure(offs, n_s, i, threadIdx.x);  // read by thread 0 at the end
    const int lab = species[i];
    const int a = (lab >= 0 && lab < 256) ? lut[lab] : -1;
    // FP32 partial sums per thread and warp (GB300's FP64 rate is a small fraction of its FP32 rate), FP64 across
    // the warps and the structures
    float acc = 0.0f;
    if (a >= 0) {
        const float* p = ps + (int64_t)i * F;
        const float* wa = w + (int64_t)a * F;
        for (int64_t f = threadIdx.x; f < F; f += blockDim.x) acc = fmaf(p[f], wa[f], acc);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (double)acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += red[k];
        atomicAdd(&energy[sid], v);
    }
}

struct GradArgs {
    const int64_t* offsets;
    const int* nbr_j;
    const float4* rij;
    const int* species;
    const int* lut;
    const int* offs;        // structure offsets
    const float4* table;
    const float* pre_G;  // per-pair radial values and r-derivatives (EXACT / MLP modes) or NULL
    const float* pre_D;
    const int* fmap;
    const float* coeffs;
    const float* grad_ps;   // [N][Fp] or NULL
    const float* weights;   // [S][Fp] or NULL
    const float* wsym;      // weights only: k_l (W_l + W_l^T) per species and l, dense [S][L1][Q][Qw] (Qw = ceil4(Q))
    int Qw, Lp_adj, n_adj_tasks;
    int w_lg, w_rows;       // per-centre dE/dp: packed l blocks staged at once (0: the per-element adjoint), rows of a warp
    int w_off;              // bytes from the pair area (k_gradients: from the start of shared memory) to those blocks
    int aux_off;            // bytes from the pair area to the small tables (past both the pair area and C)
    float* forces;          // FP32 accumulation, converted to the FP64 output afterwards
    double* virial;
    double* energy;         // linear model: per-structure energies, or NULL
    unsigned* flags;
    int N, n_s, n_max, l_max, S, Q, n_lm, F, F_pad, n_pad, Lp, M, chunk, ps_norm;
    int64_t Fp;
    float inv_delta, r_cut, width;
    int lp[kMaxLMax + 2];
};

__device__ inline void cutoff_and_slope(float r, float r_cut, float w, float& f, float& df) {
    if (r <= r_cut - w) {
        f = 1.0f;
        df = 0.0f;
    } else if (r >= r_cut) {
        f = 0.0f;
        df = 0.0f;
    } else {
        const float t = (r - r_cut + w) / w;
        const float ch = cospif(0.5f * t);  // (1 + cos(pi t)) / 2 = cos^2(pi t / 2), no cancellation near r_cut
        f = ch * ch;
        df = -0.5f * 3.14159265358979f / w * sinpif(t);
    }
}

constexpr int kGradThreads = 256;

// Y_lm = q_lm(z) C_m, Y_l-m = q_lm(z) S_m down in m at fixed l, from Legendre's equation differentiated m times:
// q_lm = x z q_{l,m+1} + y (1 - z^2) q_{l,m+2} and dq_lm/dz = w q_{l,m+1} with (x, y, w) = c_ylm_down[l][m], q_ll = c_ylm_K[l].
// In FP32 the errors are 0.6 (l = 8) to 0.5 (l = 12) times those of the recurrence up in l, 0.2 times near the poles.
static __constant__ float4 c_ylm_down[16 * 16];

static cudaError_t upload_ylm_down(cudaStream_t stream) {
    float4 t[256] = {};
    for (int l = 1; l < 16; ++l)
        for (int m = 0; m < l; ++m) {
            const double s = m ? 1.0 : sqrt(0.5), p = (double)(l - m) * (l + m + 1);
            t[l * 16 + m] = make_float4((float)(2.0 * (m + 1) * s / sqrt(p)), (float)(-s * sqrt((l + m + 2.0) * (l - m - 1.0) / p)),
                                        (float)(s * sqrt(p)), 0.0f);
        }
    return cudaMemcpyToSymbolAsync(c_ylm_down, t, sizeof(t), 0, cudaMemcpyHostToDevice, stream);
}

// Floats of a species' H in k_gradients: (l, m >= 0) x n rounded up to even x two signs, an odd number of 16-byte words, so that
// lanes of neighbouring species read different banks; floats of a pair's radial values and slopes: an odd number of 8-byte
// words (F_pad is a multiple of 4).
__host__ __device__ constexpr int grad_h_pitch(int l_max, int n_max) {
    return ((l_max + 1) * (l_max + 2) / 2 * ((n_max + 1) & ~1) * 2 / 4 | 1) * 4;
}
__host__ __device__ constexpr int grad_g_pitch(int F_pad) { return 2 * F_pad + 2; }

// What a call needs before the gradient kernel, in one launch instead of four: dense symmetric adjoint weights (linear model)
// Ws[a][l][k][q] = k_l (W_l + W_l^T)[k][q] from the packed upper-triangular weight rows (entry (q1 <= q2) at
// q1 (2Q - q1 - 1) / 2 + q2), zero in the padding columns q >= Q, and zeros in the sums that the gradient kernel adds to.
__global__ void k_prepare(int S, int L1, int Q, int Qw, int ps_norm, const float* __restrict__ w, int64_t Fp,
                          float* __restrict__ ws, int64_t n3, float* __restrict__ forces, int n_s, double* __restrict__ virial,
                          double* __restrict__ energy) {
    const int64_t total = ws ? (int64_t)S * L1 * Q * Qw : 0;
    const int Qpk = Q * (Q + 1) / 2;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n3; e += (int64_t)gridDim.x * blockDim.x) forces[e] = 0.0f;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 9 * (int64_t)n_s; e += (int64_t)gridDim.x * blockDim.x) {
        virial[e] = 0.0;
        if (energy && e < n_s) energy[e] = 0.0;
    }
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(e % Qw);
        const int64_t r = e / Qw;
        const int k = (int)(r % Q);
        const int al = (int)(r / Q);
        const int l = al % L1, a = al / L1;
        float v = 0.0f;
        if (q < Q) {
            const int lo = min(q, k), hi = max(q, k);
            v = w[(int64_t)a * Fp + (int64_t)l * Qpk + (lo * (2 * Q - lo - 1)) / 2 + hi];
            if (q == k) v *= 2.0f;
            if (ps_norm) v *= rsqrtf((float)(2 * l + 1));
        }
        ws[e] = v;
    }
}

// Hyper shape of a gradient kernel: compile-time constants for the instantiated shapes (kExpShapes), the launch arguments
// otherwise.
template <int SHAPE>
struct GradShape {
    int Nmax, Lmax, Q, Nlm, Npad, Fpad, F, Qw, LpAdj, AdjTasks;
    __device__ __forceinline__ explicit GradShape(const GradArgs& A) {
        constexpr ExpShape C = kExpShapes[SHAPE];
        Nmax = SHAPE ? C.n_max : A.n_max;
        Lmax = SHAPE ? C.l_max : A.l_max;
        Q = SHAPE ? C.n_max * C.S : A.Q;
        Nlm = SHAPE ? (C.l_max + 1) * (C.l_max + 1) : A.n_lm;
        Npad = SHAPE ? exp_npad(C.n_max) : A.n_pad;
        Fpad = SHAPE ? (C.l_max + 1) * exp_npad(C.n_max) : A.F_pad;
        F = SHAPE ? (C.l_max + 1) * C.n_max : A.F;
        Qw = SHAPE ? (C.n_max * C.S + 3) / 4 * 4 : A.Qw;
        LpAdj = SHAPE ? exp_lp(C.l_max + 1) : A.Lp_adj;
        AdjTasks = SHAPE ? (C.n_max * C.S + 3) / 4 * (exp_lp(C.l_max + 1) / 4) : A.n_adj_tasks;
    }
};

// Rows of chat_l for l in [l0, l1) from staged packed symmetric blocks (pitch Wp, odd: lanes of different l read different
// banks): a warp takes R rows q, its lanes the 4-column tiles of the padded rows of C. Whether k lies before, in or past the
// rows, and with it where W[q][k] sits in the packed block, is the same for the whole warp. SPLIT, where the staged l have fewer
// tiles than lanes (small l_max; wide bases, of which few blocks fit at a time) and the rows are more than one round of the
// warps: 2^s sets of rows to a warp, as many as leave every warp some (3 000 centres with 24 pairs: (16, 8, 8) 6 489 -> 1 108 us
// with the larger groups below, (12, 0, 8) 260 -> 78). An instance of its own: beside the plain form it cost that one 2 %.
template <int R, bool SPLIT, class Shape, class Put>
__device__ __forceinline__ void adjoint_rows(const Shape& K, const float* s_C, const float* s_W, int Wp, int l0, int l1, int ps_norm,
                                             Put put) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, Q = K.Q, Lq = K.LpAdj;
    int s = 0;
    while (SPLIT && s < 5 && exp_lp(l1) / 4 - exp_lp(l0) / 4 <= 16 >> s && (R * nwarps << s) < Q) ++s;
    const int across = 32 >> s;
    for (int q0 = R * ((warp << s) + lane / across); q0 < Q; q0 += R * nwarps << s) {
        for (int t = exp_lp(l0) / 4 + lane % across; t < exp_lp(l1) / 4; t += across) {
            int l = l0;
            while (exp_lp(l + 1) <= 4 * t) ++l;
            const float* W = s_W + (l - l0) * Wp;
            const float* C = s_C + 4 * t;
            uint64_t a[R][2];
#pragma unroll
            for (int u = 0; u < R; ++u) a[u][0] = a[u][1] = 0ull;
            auto step = [&](int k, auto&& w) {
                const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(C + k * Lq);
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    const float v = w(u);
                    const uint64_t vv = f2_pack(v, v);
                    a[u][0] = f2_fma(vv, c.x, a[u][0]);
                    a[u][1] = f2_fma(vv, c.y, a[u][1]);
                }
            };
            // the packed entry (lo <= hi) sits at lo (2Q - lo - 1) / 2 + hi
            const float* wr[R];  // rows q0 + u (the last row again for those past it, which are not written)
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int q = min(q0 + u, Q - 1);
                wr[u] = W + (q * (2 * Q - q - 1)) / 2;
            }
            const float* wk = W + q0;
            const int last = Q - 1 - q0;
#pragma unroll 2
            for (int k = 0; k < q0; ++k) {
                step(k, [&](int u) { return wk[min(u, last)]; });
                wk += Q - k - 1;
            }
            for (int k = q0; k < min(q0 + R, Q); ++k)
                step(k, [&](int u) {
                    const int q = min(q0 + u, Q - 1), lo = min(q, k), hi = max(q, k);
                    const float v = W[(lo * (2 * Q - lo - 1)) / 2 + hi];
                    return q == k ? 2.0f * v : v;  // W + W^T
                });
#pragma unroll 2
            for (int k = q0 + R; k < Q; ++k) step(k, [&](int u) { return wr[u][k]; });
            const float kl = ps_norm ? rsqrtf((float)(2 * l + 1)) : 1.0f;
            const int s0 = 4 * t - exp_lp(l);
#pragma unroll
            for (int u = 0; u < R; ++u) {
                if (q0 + u >= Q) break;
                float v[4];
                f2_unpack(a[u][0], v[0], v[1]);
                f2_unpack(a[u][1], v[2], v[3]);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (s0 + e <= 2 * l) put(q0 + u, l, s0 + e, kl * v[e]);
            }
        }
    }
}

// chat = k_l (W + W^T) C of centre i from its coefficients (staged at s_C) and its weights; put(q, l, s, v) takes
// chat[q][l, m = s - l]. W: what the weights may be, kLinear (a species' dense blocks), kPerCentre (dE/dp; s_W: room for
// w_lg packed l blocks, or none) or kPerElement (dE/dp read from global memory). s_C holds nothing else yet; a barrier
// follows before s_C and s_W may be reused. Returns this thread's share of chat . c (linear: twice E_i = w . p_i, which is
// quadratic in c).
// Per-centre dE/dp: with each l block expanded to a dense matrix in turn, two barriers and 12 to 60 tile tasks per l, the
// adjoint was 640 us of the kernel's 818 on 8 960 centres (n_max 12, l_max 9, 4 species); all packed blocks staged at once
// and read as they are, 240 of 557 (0.42 GB of dE/dp: 63 us).
enum { kLinear = 1, kPerCentre = 2, kPerElement = 4, kSplitRows = 8 };
template <int SHAPE, int W, class Put>
__device__ __forceinline__ float adjoint(const GradArgs& A, const GradShape<SHAPE>& K, int i, int a_i, float* s_C, float* s_W, Put put) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int L1 = K.Lmax + 1, Q = K.Q, n_lm = K.Nlm, Qpk = Q * (Q + 1) / 2, QN = Q * n_lm;
    const float* Gp = A.grad_ps ? A.grad_ps + (int64_t)i * A.Fp : (a_i >= 0 ? A.weights + (int64_t)a_i * A.Fp : nullptr);
    const float* c = A.coeffs + (int64_t)i * QN;
    float dot = 0.0f;
    // prefix counts of the adjoint tile tasks per l: ceil(Q / 4) ceil((2l' + 1) / 4) summed over l' < l
    auto adj_pref = [&](int l) { return (Q + 3) / 4 * (exp_lp(l) / 4); };
    // one 4 x 4 register tile of chat_l = Ws_l C_l (rows 4 qt.., columns 4 st.. of the l block), Ws_l dense and
    // symmetric with row pitch Qw in global memory (the linear model)
    auto adjoint_tile = [&](const float* Wl, const float* Cl, int Lq, int l, int qt, int st) {
        // paired FMAs (fma.rn.f32x2): each product rounded exactly as fmaf rounds it
        uint64_t ap[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) ap[u][0] = ap[u][1] = 0ull;
        for (int k = 0; k < Q; ++k) {
            const float4 w4 = __ldg(reinterpret_cast<const float4*>(Wl + k * K.Qw));
            const float4 c4 = *reinterpret_cast<const float4*>(Cl + k * Lq);
            const float ww[4] = {w4.x, w4.y, w4.z, w4.w};
            const uint64_t c01 = f2_pack(c4.x, c4.y), c23 = f2_pack(c4.z, c4.w);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t wu = f2_pack(ww[u], ww[u]);
                ap[u][0] = f2_fma(wu, c01, ap[u][0]);
                ap[u][1] = f2_fma(wu, c23, ap[u][1]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = 4 * qt + u;
            if (q >= Q) break;
            float v[4];
            f2_unpack(ap[u][0], v[0], v[1]);
            f2_unpack(ap[u][1], v[2], v[3]);
            const float4 own = *reinterpret_cast<const float4*>(Cl + q * Lq);  // zero in the padding columns
            dot = fmaf(v[0], own.x, fmaf(v[1], own.y, fmaf(v[2], own.z, fmaf(v[3], own.w, dot))));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int sx = 4 * st + e;
                if (sx <= 2 * l) put(q, l, sx, v[e]);
            }
        }
    };
    const bool linear = (W & kLinear) && A.wsym;
    if (linear || ((W & kPerCentre) && A.w_lg)) {
        // adjoint as 4 x 4 register tiles of chat_l = Ws_l C_l: C staged with every l block padded to a multiple of
        // 4 columns (zeros), so that tiles load float4 rows of C and of the dense symmetric weights
        const int Lq = K.LpAdj;
        // the padding columns of the l blocks (ceil4(2l + 1) - (2l + 1) of them: three for even l, one for odd l)
        // read as zero; they are disjoint from the copied columns, so the barrier after the copies covers both
        const int n_padc = 4 * (L1 >> 1) + 3 * (L1 & 1);
        for (int e = tid; e < Q * n_padc; e += blockDim.x) {
            const int q = e / n_padc, r = e - q * n_padc;
            const bool odd = (r & 3) == 3;
            const int l = 2 * (r >> 2) + (odd ? 1 : 0);
            s_C[q * Lq + exp_lp(l) + 2 * l + 1 + (odd ? 0 : (r & 3))] = 0.0f;
        }
        // lanes over lm, warps over rows
        for (int lm = lane; lm < n_lm; lm += 32) {
            const int l = (int)sqrtf((float)lm);  // l with l^2 <= lm < (l + 1)^2
            const int col = exp_lp(l) + (lm - l * l);
            for (int q = warp; q < Q; q += nwarps) cp_async4(s_C + q * Lq + col, c + q * n_lm + lm);
        }
        cp_async_wait_all();
        __syncthreads();
        const int QT = (Q + 3) >> 2;
        if (linear) {  // linear model: the species' dense blocks, shared by all centres, from global memory (L2)
            const float* Wsa = A.wsym + (int64_t)(a_i < 0 ? 0 : a_i) * L1 * Q * K.Qw;
            for (int t = tid; t < K.AdjTasks && a_i >= 0; t += blockDim.x) {
                int l = 0;
                while (adj_pref(l + 1) <= t) ++l;
                const int r = t - adj_pref(l);
                const int st = r / QT, qt = r - st * QT;
                adjoint_tile(Wsa + (int64_t)l * Q * K.Qw + 4 * qt, s_C + exp_lp(l) + 4 * st, Lq, l, qt, st);
            }
            if (a_i < 0)
                for (int e = tid; e < QN; e += blockDim.x) {
                    const int q = e / n_lm, lm = e - q * n_lm, l = (int)sqrtf((float)lm);
                    put(q, l, lm - l * l, 0.0f);
                }
        } else if constexpr ((W & kPerCentre) != 0) {  // this centre's dE/dp: groups of w_lg packed l blocks staged in shared memory
            const int Wp = Qpk | 1;
            for (int l0 = 0; l0 < L1; l0 += A.w_lg) {
                const int l1 = min(L1, l0 + A.w_lg);
                if (l0) __syncthreads();
                for (int l = l0; l < l1; ++l)
                    for (int e = tid; e < Qpk; e += blockDim.x) cp_async4(s_W + (l - l0) * Wp + e, Gp + (int64_t)l * Qpk + e);
                cp_async_wait_all();
                __syncthreads();
                if (W & kSplitRows)
                    adjoint_rows<4, true>(K, s_C, s_W, Wp, l0, l1, A.ps_norm, put);
                else if (A.w_rows == 6)
                    adjoint_rows<6, false>(K, s_C, s_W, Wp, l0, l1, A.ps_norm, put);
                else
                    adjoint_rows<4, false>(K, s_C, s_W, Wp, l0, l1, A.ps_norm, put);
            }
        }
        return dot;
    }
    if (W == kLinear) return dot;
    for (int e = tid; e < QN; e += blockDim.x) cp_async4(s_C + e, c + e);
    cp_async_wait_all();
    __syncthreads();
    // adjoint chat[q][lm] = k_l sum_k (W + W^T)[q][k] C[k][lm]; the packed entry (q1 <= q2) sits at
    // q1 (2Q - q1 - 1) / 2 + q2, and (W + W^T) doubles the diagonal
    for (int e = tid; e < QN; e += blockDim.x) {
        const int q = e / n_lm, lm = e - q * n_lm;
        const int l = (int)sqrtf((float)lm);
        float acc = 0.0f;
        if (Gp) {
            const float* W = Gp + (int64_t)l * Qpk;
            const float* Cc = s_C + lm;
            int idx = q;  // entry (k, q), k < q
            for (int k = 0; k < q; ++k) {
                acc = fmaf(__ldg(W + idx), Cc[k * n_lm], acc);
                idx += Q - k - 1;
            }
            const int ro = (q * (2 * Q - q - 1)) / 2;  // entries (q, k), k >= q
            acc = fmaf(2.0f * __ldg(W + ro + q), Cc[q * n_lm], acc);
            for (int k = q + 1; k < Q; ++k) acc = fmaf(__ldg(W + ro + k), Cc[k * n_lm], acc);
        }
        put(q, l, lm - l * l, (A.ps_norm ? rsqrtf((float)(2 * l + 1)) : 1.0f) * acc);
    }
    return dot;
}

// E_i = chat . c / 2: FP32 per thread and warp (s_e, a value per warp), FP64 across the warps (read by a warp after a barrier)
// and one atomic per centre.
__device__ __forceinline__ void warp_energy(float dot, float* s_e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if ((threadIdx.x & 31) == 0) s_e[threadIdx.x >> 5] = dot;
}
__device__ __forceinline__ void add_energy(const float* s_e, int nwarps, double* energy) {
    double e = 0.0;
    for (int w = 0; w < nwarps; ++w) e += (double)s_e[w];
    atomicAdd(energy, 0.5 * e);
}

// One CTA per centre i:
//   1. chat = k_l (W + W^T) C (adjoint; with it the linear model's energy), kept as H[a][(l, m >= 0)][n / 2][m, -m][n % 2];
//   2. per chunk of 32 of the centre's pairs (two CTA barriers per chunk):
//      radial values (f I, (f I)') per pair into shared memory (a warp takes two pairs at a time, lanes over (l, n));
//      the contraction: a warp takes an l (and a block of n), its lanes the chunk's pairs. The pair's radial values of that l
//      stay in registers; going down in m it forms u = sum_n chat (f I)' and v = sum_n chat f I for both signs of m from one
//      16-byte load of H per two n and eight products, has q_lm and its slope from a recurrence, and sums over m by Horner's
//      rule in x + iy, so that Y is never stored; it leaves its share of s = sum_lm Y u and w = sum_lm dY/du v per pair;
//      the last warp adds the shares up, one pair per lane: dE/dr_ji, the force scatter, F_i and the virial, and
//      stages the next chunk's records (r_ji, the neighbour's species, j, f_cut, f_cut') beside the others' work.
// Bound: latency at four CTAs of 256 threads per SM between the phases' barriers (issue slots 55 %, shared memory 70 %). Of
// 1 390 us on 32 768 centres with 90 pairs (n_max 10, l_max 8, 3 species), the contraction takes 500, the radial values 420
// (4.2 GB from L2) and the adjoint 180. With a warp per pair, lanes over lm and Y in shared memory (two loads per two
// products) the kernel took 2 328 us; with a warp per m, up in l, radial values loaded for every m, 1 422; with half of n_max
// 10 per task 1 526; with three CTAs per SM 1 510. 4 096 centres with 34 pairs (8, 6, 2): 81 -> 63 us, with CTAs of 128
// threads (below) 45.
template <int SHAPE, int W, int T>
__global__ void __launch_bounds__(T, (W == kLinear ? 4 : 3) * 256 / T) k_gradients(const GradArgs A) {
    const GradShape<SHAPE> K(A);
    constexpr int chunk = 32, nwarps = T / 32;
    const int L1 = K.Lmax + 1, n2 = (K.Nmax + 1) & ~1;             // n in pairs
    const int Hl = 2 * n2, Hs = grad_h_pitch(K.Lmax, K.Nmax);      // floats of an (l, m) and of a species in H
    const int NP = n2 / 2;                                         // pairs of n
    // pairs of n of a task (its radial values stay in registers: all of n_max up to 10, else half), and tasks of an l
    constexpr int kN = kExpShapes[SHAPE].n_max, NB = SHAPE == 0 ? 4 : (kN <= 10 ? (kN + 1) / 2 : (kN + 3) / 4);
    const int NK = (NP + NB - 1) / NB;
    const int Gp = grad_g_pitch(K.Fpad);                           // floats of a pair's radial values
    extern __shared__ __align__(16) float sm[];
    float* s_H = sm;                                               // [S][Hs]
    // per-pair records, two buffers that alternate between chunks
    float4* s_vec = reinterpret_cast<float4*>(s_H + A.S * Hs);     // [2][chunk]
    float4* s_part = s_vec + 2 * chunk;                            // [nwarps][chunk] shares of (s, w)
    float* s_fc = reinterpret_cast<float*>(s_part + nwarps * chunk);  // [2][chunk]
    float* s_dfc = s_fc + 2 * chunk;
    int* s_spc = reinterpret_cast<int*>(s_dfc + 2 * chunk);
    int* s_j = s_spc + 2 * chunk;
    // the coefficients are needed only by the adjoint, before the pair loop: they share the area of the radial values
    float* s_C = reinterpret_cast<float*>(s_j + 2 * chunk);
    float* s_G = s_C;                                              // [chunk][Gp]: f I, then (f I)'
    __shared__ float s_e[nwarps];
    __shared__ float s_acc[12][33];  // per lane of the last warp: sums of F_i and of the virial (odd pitch: read down a lane)
    __shared__ int s_sid;

    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp == nwarps - 1) {  // the centre's structure, for the virial and the energy
        const int sid = warp_find_structure(A.offs, A.n_s, i, lane);
        if (lane == 0) s_sid = sid;
    }
    const int lab_i = A.species[i];
    const int a_i = (lab_i >= 0 && lab_i < 256) ? A.lut[lab_i] : -1;
    // what the adjoint leaves out (m = 0 has no partner, an odd n_max a last n) reads as zero; its first barrier follows
    for (int e = tid; e < A.S * Hs / 4; e += T) reinterpret_cast<float4*>(s_H)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    float* s_W = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(sm) + A.w_off);
    const float dot = adjoint<SHAPE, W>(A, K, i, a_i, s_C, s_W, [&](int q, int l, int s, float v) {
        const int a = q / K.Nmax, n = q - a * K.Nmax, m = s - l;
        s_H[a * Hs + (l * (l + 1) / 2 + abs(m)) * Hl + 4 * (n >> 1) + (n & 1) + (m < 0 ? 2 : 0)] = v;
    });
    if (W == kLinear && A.energy) warp_energy(dot, s_e);
    const int64_t seg_beg = A.offsets[i];
    const int seg_len = (int)(A.offsets[i + 1] - seg_beg);
    const bool last = warp == nwarps - 1;
    auto stage = [&](int pos, int b) {  // last warp: the records of the chunk at pos into buffer b
        if (pos + lane >= seg_len) return;
        const float4 v = __ldg(A.rij + seg_beg + pos + lane);
        const int j = __ldg(A.nbr_j + seg_beg + pos + lane);
        const int lab = A.species[j];
        int a = (lab >= 0 && lab < 256) ? A.lut[lab] : -1;
        if (!(v.w > 1e-6f)) a = -1;
        const int o = b * chunk + lane;
        s_vec[o] = v;
        s_spc[o] = a;
        s_j[o] = j;
        cutoff_and_slope(v.w, A.r_cut, A.width, s_fc[o], s_dfc[o]);
    };
    auto finish = [&](int pos, int b) {  // last warp: dE/dr_ji of the chunk at pos, one pair per lane
        const int o = b * chunk + lane;
        if (pos + lane >= seg_len || s_spc[o] < 0) return;
        float S = 0.0f, Wx = 0.0f, Wy = 0.0f, Wz = 0.0f;
        for (int w = 0; w < nwarps; ++w) {
            const float4 t = s_part[w * chunk + lane];
            S += t.x;
            Wx += t.y;
            Wy += t.z;
            Wz += t.w;
        }
        const float4 v = s_vec[o];
        const float inv_r = 1.0f / v.w;
        const float ux = v.x * inv_r, uy = v.y * inv_r, uz = v.z * inv_r;
        const float wu = Wx * ux + Wy * uy + Wz * uz;
        const float g[3] = {S * ux + (Wx - wu * ux) * inv_r, S * uy + (Wy - wu * uy) * inv_r, S * uz + (Wz - wu * uz) * inv_r};
        const int j = s_j[o];
        const float d[3] = {v.x, v.y, v.z};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            if (j != i) {
                atomicAdd(&A.forces[3 * (int64_t)j + x], -g[x]);
                s_acc[x][lane] += g[x];
            }
#pragma unroll
            for (int y = 0; y < 3; ++y) s_acc[3 + 3 * x + y][lane] = fmaf(g[x], d[y], s_acc[3 + 3 * x + y][lane]);
        }
    };
    if (last) {
#pragma unroll
        for (int k = 0; k < 12; ++k) s_acc[k][lane] = 0.0f;
        stage(0, 0);
    }
    int b = 0;
    for (int pos = 0; pos < seg_len; pos += chunk, b ^= 1) {
        const int nc = min(chunk, seg_len - pos), bo = b * chunk;
        // the chunk's records are staged; the adjoint is done with the coefficients, the chains with the radial values
        __syncthreads();
        auto put = [&](float* gd, int f, float g, float dg) {  // slot f = l n_pad + n of a pair
            gd[f] = g;
            gd[K.Fpad + f] = dg;
        };
        if (pos == 0 && K.Npad != K.Nmax)  // the padding slots are read as zero and written only here
            for (int e = tid; e < chunk * L1 * (K.Npad - K.Nmax); e += T) {
                const int q = K.Npad - K.Nmax, n = e % q, l = e / q % L1;
                put(s_G + e / q / L1 * Gp, l * K.Npad + K.Nmax + n, 0.0f, 0.0f);
            }
        // radial values and slopes: a warp takes two pairs at a time, lanes over (l, n)
        for (int p = 2 * warp; p < nc; p += 2 * nwarps) {
            const bool two = p + 1 < nc;
            const int ob = bo + p, oc = ob + (two ? 1 : 0);
            const float f0 = s_fc[ob], d0 = s_dfc[ob], f1 = s_fc[oc], d1 = s_dfc[oc];
            float* gd = s_G + p * Gp;
            auto slot = [&](int c) { return c + c / K.Nmax * (K.Npad - K.Nmax); };  // column l n_max + n -> l n_pad + n
            if (A.pre_G) {
                const float* pg = A.pre_G + (seg_beg + pos + p) * K.F;
                const float* pd = A.pre_D + (seg_beg + pos + p) * K.F;
                const int64_t o1 = two ? K.F : 0;
#pragma unroll 4
                for (int c = lane; c < K.F; c += 32) {
                    const float g0 = __ldg(pg + c), e0 = __ldg(pd + c), g1 = __ldg(pg + o1 + c), e1 = __ldg(pd + o1 + c);
                    const int f = slot(c);
                    put(gd, f, f0 * g0, d0 * g0 + f0 * e0);
                    if (two) put(gd + Gp, f, f1 * g1, d1 * g1 + f1 * e1);
                }
            } else {
                auto row = [&](int o, float& u) {
                    const float x = s_vec[o].w * A.inv_delta;
                    const int k = min(max((int)x, 0), A.M - 1);
                    u = x - (float)k;
                    return A.table + k * K.F;
                };
                auto value = [&](const float4& cf, float u, float f, float df, float* o, int fp) {
                    // value and slope of the cubic by Horner's scheme twice
                    const float b1 = fmaf(u, cf.w, cf.z), b0 = fmaf(u, b1, cf.y), g = fmaf(u, b0, cf.x);
                    const float dg = fmaf(u, fmaf(u, cf.w, b1), b0);
                    put(o, fp, f * g, fmaf(df, g, f * A.inv_delta * dg));
                };
                float u0, u1;
                const float4 *t0 = row(ob, u0), *t1 = row(oc, u1);
#pragma unroll 4
                for (int c = lane; c < K.F; c += 32) {
                    const float4 c0 = __ldg(t0 + c), c1 = __ldg(t1 + c);
                    const int f = slot(c);
                    value(c0, u0, f0, d0, gd, f);
                    if (two) value(c1, u1, f1, d1, gd + Gp, f);
                }
            }
        }
        if (last && pos > 0) finish(pos - chunk, b ^ 1);  // its shares stand until the barrier below
        __syncthreads();
        // contraction, lanes over the chunk's pairs; a warp's tasks: t = w, 2 nwarps - 1 - w, ...: large l with small ones
        if (lane < nc) {
            float S = 0.0f, Wx = 0.0f, Wy = 0.0f, Wz = 0.0f;
            const float4 v = s_vec[bo + lane];
            const float inv_r = v.w > 1e-6f ? 1.0f / v.w : 0.0f;
            const float x = v.x * inv_r, y = v.y * inv_r, z = v.z * inv_r, xy2 = x * x + y * y;
            const float* Ha = s_H + max(s_spc[bo + lane], 0) * Hs;
            const float* gp = s_G + lane * Gp;
            const int tasks = L1 * NK;
#pragma unroll 1
            for (int k = 0; k * nwarps < tasks; ++k) {
                const int t = k * nwarps + ((k & 1) ? nwarps - 1 - warp : warp);
                if (t >= tasks) continue;
                const int l = K.Lmax - t / NK, n0 = t % NK * NB;  // pairs of n from n0
                uint64_t g[NB], d[NB];
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    if (NP % NB && n0 + n >= NP) break;
                    g[n] = *reinterpret_cast<const uint64_t*>(gp + l * K.Npad + 2 * (n0 + n));
                    d[n] = *reinterpret_cast<const uint64_t*>(gp + K.Fpad + l * K.Npad + 2 * (n0 + n));
                }
                // down in m: q = Y_lm / C_m, dq its z derivative; sums over m of (q u_m - i q u_-m) w^m, the same with v
                // and dq, and of m (q v_m - i q v_-m) w^(m - 1), w = x + iy, by Horner's rule
                float q = c_ylm_K[l], q1 = 0.0f, dq = 0.0f;
                float sr = 0.0f, si = 0.0f, zr = 0.0f, zi = 0.0f, tr = 0.0f, ti = 0.0f;
                auto horner = [&](float& re, float& im, float a, float b) {
                    const float r = fmaf(re, x, fmaf(-im, y, a));
                    im = fmaf(re, y, fmaf(im, x, -b));
                    re = r;
                };
                const ulonglong2* h = reinterpret_cast<const ulonglong2*>(Ha + (l * (l + 1) / 2 + l) * Hl) + n0;
#pragma unroll 1
                for (int m = l;; --m, h -= NP) {
                    uint64_t vp = 0ull, up = 0ull, vn = 0ull, un = 0ull;  // even and odd n
#pragma unroll
                    for (int n = 0; n < NB; ++n) {
                        if (NP % NB && n0 + n >= NP) break;
                        const ulonglong2 c = h[n];  // (chat_m, chat_-m) of two n
                        vp = f2_fma(c.x, g[n], vp);
                        up = f2_fma(c.x, d[n], up);
                        vn = f2_fma(c.y, g[n], vn);
                        un = f2_fma(c.y, d[n], un);
                    }
                    auto sum = [](uint64_t t) {
                        float e, o;
                        f2_unpack(t, e, o);
                        return e + o;
                    };
                    const float v0 = sum(vp), v1 = sum(vn);
                    horner(sr, si, q * sum(up), q * sum(un));
                    horner(zr, zi, dq * v0, dq * v1);
                    if (m == 0) break;
                    const float mq = (float)m * q;
                    horner(tr, ti, mq * v0, mq * v1);
                    const float4 f = c_ylm_down[l * 16 + m - 1];
                    const float qn = fmaf(f.x * z, q, f.y * (xy2 * q1));
                    dq = f.z * q;
                    q1 = q;
                    q = qn;
                }
                S += sr;  // Y_lm = q C_m, Y_l-m = q S_m with w^m = C_m + i S_m
                Wx += tr;
                Wy -= ti;
                Wz += zr;
            }
            s_part[warp * chunk + lane] = make_float4(S, Wx, Wy, Wz);
        }
        if (last && pos + chunk < seg_len) stage(pos + chunk, b ^ 1);  // its last readers finished before the barrier above
    }
    __syncthreads();
    if (last && seg_len > 0) finish((seg_len - 1) / chunk * chunk, b ^ 1);
    // F_i and the virial from the last warp's lanes
    if (!last) return;
    if (W == kLinear && A.energy && lane == 0) add_energy(s_e, nwarps, &A.energy[s_sid]);
    // Across the lanes beyond FP32, as the wide form adds its warps' sums in FP64: lane k + 12 h adds half h of component k's
    // lanes with the roundings' errors kept beside the sum (left out where the sum is not finite). Sixteen FP64 additions instead
    // took 1 to 2 % of the kernel (FP64 issues at a sixty-fourth of the FP32 rate).
    __syncwarp();
    double t = 0.0;
    if (lane < 24) {
        const float* v = s_acc[lane % 12] + lane / 12 * 16;
        float s = v[0], c = 0.0f;
#pragma unroll
        for (int e = 1; e < 16; ++e) {
            const float a = v[e], n = s + a, b = n - s;
            c += (s - (n - b)) + (a - b);
            s = n;
        }
        t = (double)s + (double)(c == c ? c : 0.0f);
    }
    t += __shfl_down_sync(0xffffffffu, t, 12);
    if (lane < 3) {
        if (t != 0.0) atomicAdd(&A.forces[3 * (int64_t)i + lane], (float)t);
    } else if (lane < 12) {
        atomicAdd(&A.virial[9 * (int64_t)s_sid + (lane - 3)], t);
    }
}

// The same for bases whose H and radial values do not fit shared memory beside the coefficients: Y and a few pairs' radial
// values staged per chunk. One CTA per centre i:
//   1. chat = k_l (W + W^T) C from the centre's coefficients (shared memory) and its weight block (global, L1);
//   2. per chunk of the centre's pairs (two CTA barriers per chunk):
//      radial values (f I, (f I)') per pair (one warp per pair, lanes over (l, n));
//      Y and dY/du per pair (warp w runs the m = w chains for all pairs, lanes over pairs);
//      the last warp stages the next chunk's records (r_ji, the neighbour's species, j, f_cut, f_cut') into the
//      other of two buffers;
//      contraction s = sum_lm Y sum_n chat (f I)', w = sum_lm dY/du sum_n chat f I, then dE/dr_ji, the force
//      scatter and the virial (one warp per pair, lanes over lm, warp-shuffle reduction; F_i and the virial summed
//      per lane, FP64 across the warps at the end).
static __global__ void __launch_bounds__(kGradThreads, 5) k_gradients_wide(const GradArgs A) {
    const GradShape<0> K(A);
    const int kNmax = A.n_max, kLmax = A.l_max, kQ = A.Q, kNlm = A.n_lm, kNpad = A.n_pad, kFpad = A.F_pad, kF = A.F;
    constexpr bool kFmapId = false;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int chunk = A.chunk;
    const int QN = kQ * kNlm;
    const int QN4 = (QN + 3) & ~3;                            // keeps the float4 arrays 16-byte aligned
    const int Yp = kNlm | 1;                                // odd pitch: conflict-free float4 rows
    float* s_H = reinterpret_cast<float*>(smem_raw);          // chat [Q][n_lm]
    // per-pair records (r_ji, f_cut, f_cut', species index, j): two buffers that alternate between chunks, so that
    // the next chunk is staged while the current one is processed; they come first in the pair area, so that the
    // first chunk can be staged while the adjoint still reads the coefficients
    float4* s_vec = reinterpret_cast<float4*>(s_H + QN4);     // [2][chunk]
    float* s_fc = reinterpret_cast<float*>(s_vec + 2 * chunk);  // [2][chunk]
    float* s_dfc = s_fc + 2 * chunk;                          // [2][chunk]
    int* s_spc = reinterpret_cast<int*>(s_dfc + 2 * chunk);   // [2][chunk]
    int* s_j = s_spc + 2 * chunk;                             // [2][chunk]
    // the coefficients are needed only by the adjoint, before the pair loop: they share the area of Y and G
    float* s_C = reinterpret_cast<float*>(s_j + 2 * chunk);   // [Q][n_lm], or [Q][Lp_adj] padded per l (tiled adjoint)
    float4* s_Yv = reinterpret_cast<float4*>(s_C);            // [chunk][Yp]  (Y, dY/dux, dY/duy, dY/duz)
    float2* s_GD = reinterpret_cast<float2*>(s_Yv + (size_t)chunk * Yp);  // [chunk][F_pad]  (f I, (f I)')
    int* s_lofm = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(s_vec) + A.aux_off);  // [n_lm] l of lm
    int* s_fmap = s_lofm + kNlm;                            // [F_pad]
    __shared__ double red[kGradThreads / 32][12];
    __shared__ float s_e[kGradThreads / 32];
    __shared__ int s_sid;

    const int i = blockIdx.x;
    if ((threadIdx.x >> 5) == (blockDim.x >> 5) - 1) {  // the last warp: the centre's structure, for the virial
        const int sid = warp_find_structure(A.offs, A.n_s, i, threadIdx.x & 31);
        if ((threadIdx.x & 31) == 0) s_sid = sid;
    }
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int L1 = kLmax + 1;
    for (int lm = tid; lm < kNlm; lm += blockDim.x) s_lofm[lm] = (int)sqrtf((float)lm);  // l with l^2 <= lm
    if (!kFmapId)
        for (int t = tid; t < kFpad; t += blockDim.x) s_fmap[t] = A.fmap[t];
    const int lab_i = A.species[i];
    const int a_i = (lab_i >= 0 && lab_i < 256) ? A.lut[lab_i] : -1;
    const float dot = adjoint<0, kLinear | kPerElement>(
        A, K, i, a_i, s_C, nullptr, [&](int q, int l, int s, float v) { s_H[q * kNlm + l * l + s] = v; });
    if (A.energy) warp_energy(dot, s_e);
    // per-lane sums of F_i (lanes 0..2) and of the virial (lanes 3..11, row-major): FP32 within a warp, FP64 across
    // the warps (GB300's FP64 rate is a small fraction of its FP32 rate)
    float racc = 0.0f;
    const int64_t seg_beg = A.offsets[i], seg_end = A.offsets[i + 1];
    // the last warp stages the pairs (chunk <= 32: one pair per lane), with the next chunk's r_ji and j loaded into
    // registers one chunk ahead
    const bool stager = warp == nwarps - 1;
    float4 nv = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
    int nj = 0;
    if (stager && lane < chunk && seg_beg + lane < seg_end) {
        nv = A.rij[seg_beg + lane];
        nj = A.nbr_j[seg_beg + lane];
    }
    auto stage = [&](int64_t pos, int b) {  // the chunk at pos into record buffer b
        const int t = lane;
        if (t < chunk && pos + t < seg_end) {
            const float4 v = nv;
            const int j = nj;
            if (pos + chunk + t < seg_end) {
                nv = A.rij[pos + chunk + t];
                nj = A.nbr_j[pos + chunk + t];
            }
            const int lab = A.species[j];
            int a = (lab >= 0 && lab < 256) ? A.lut[lab] : -1;
            if (!(v.w > 1e-6f)) a = -1;
            const int o = b * chunk + t;
            s_vec[o] = v;
            s_spc[o] = a;
            s_j[o] = j;
            float f, df;
            cutoff_and_slope(v.w, A.r_cut, A.width, f, df);
            s_fc[o] = f;
            s_dfc[o] = df;
        }
    };
    // the first chunk's records do not overlap the coefficients; the first barrier of the loop also ends the adjoint
    // before Y and G overwrite the coefficients
    if (stager) stage(seg_beg, 0);
    int b = 0;
    for (int64_t pos = seg_beg; pos < seg_end; pos += chunk, b ^= 1) {
        const int nc = (int)((seg_end - pos) < (int64_t)chunk ? (seg_end - pos) : (int64_t)chunk);
        // the chunk's records are staged, and the previous chunk's contraction is done with s_GD and s_Yv
        __syncthreads();
        const int bo = b * chunk;  // this chunk's records: s_vec[bo + p], ...
        // radial values and slopes: one warp per pair, lanes over padded (l, n); the warps without a Y chain first
        for (int p = nwarps - 1 - warp; p < nc; p += nwarps) {
            const float f = s_fc[bo + p], df = s_dfc[bo + p];
            float2* gd = s_GD + p * kFpad;
            if (A.pre_G) {
                const float* pg = A.pre_G + (pos + p) * kF;
                const float* pd = A.pre_D + (pos + p) * kF;
                #pragma unroll
                for (int fp = lane; fp < kFpad; fp += 32) {
                    const int col = kFmapId ? fp : s_fmap[fp];
                    const float g = col >= 0 ? __ldg(pg + col) : 0.0f, dg = col >= 0 ? __ldg(pd + col) : 0.0f;
                    gd[fp] = make_float2(f * g, df * g + f * dg);
                }
            } else {
                const float x = s_vec[bo + p].w * A.inv_delta;
                const int k = min(max((int)x, 0), A.M - 1);
                const float u = x - (float)k;
                const float4* trow = A.table + k * kF;
                #pragma unroll
                for (int fp = lane; fp < kFpad; fp += 32) {
                    const int col = kFmapId ? fp : s_fmap[fp];
                    const float4 cf = col >= 0 ? __ldg(trow + col) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    const float g = fmaf(u, fmaf(u, fmaf(u, cf.w, cf.z), cf.y), cf.x);
                    const float dg = fmaf(u, fmaf(u, 3.0f * cf.w, 2.0f * cf.z), cf.y) * A.inv_delta;
                    gd[fp] = make_float2(f * g, df * g + f * dg);
                }
            }
        }
        // Y and dY/du (gradient of the polynomial extension), forward mode through the recurrence: lanes over the
        // chunk's pairs, one chain of m per lane; a chunk of at most 8 (16) pairs gives each warp four (two) values
        // of m on 8 (16) lanes each, a larger one gives warp w the m = w, w + nwarps, ... chains on all 32 lanes
        const int lpm = nc <= 8 ? 8 : (nc <= 16 ? 16 : 32), mpw = 32 / lpm;
        for (int m = warp * mpw + lane / lpm; m < L1; m += nwarps * mpw) {
            const float km = c_ylm_K[m], fm = (float)m;
#pragma unroll 1
            for (int p = lane % lpm; p < nc; p += lpm) {
                const float4 v = s_vec[bo + p];
                const float inv_r = v.w > 1e-6f ? 1.0f / v.w : 0.0f;
                const float x = v.x * inv_r, y = v.y * inv_r, z = v.z * inv_r;
                float cm = 1.0f, sm = 0.0f, cm1 = 0.0f, sm1 = 0.0f;  // (x+iy)^m and (x+iy)^(m-1)
#pragma unroll 1
                for (int t = 0; t < m; ++t) {
                    cm1 = cm;
                    sm1 = sm;
                    const float nc2 = cm * x - sm * y;
                    sm = cm * y + sm * x;
                    cm = nc2;
                }
                float4* Yrow = s_Yv + p * Yp;
                float q2 = 0.0f, q1 = km, d2 = 0.0f, d1 = 0.0f;
#pragma unroll 1
                for (int l = m; l < L1; ++l) {
                    float q = q1, dq = d1;
                    if (l > m) {
                        const float Al = c_ylm_A[l * 16 + m], Bl = c_ylm_B[l * 16 + m];
                        q = Al * (z * q1 - Bl * q2);
                        dq = Al * (q1 + z * d1 - Bl * d2);
                        q2 = q1;
                        d2 = d1;
                        q1 = q;
                        d1 = dq;
                    }
                    const int l0 = l * l + l;
                    if (m == 0) {
                        Yrow[l0] = make_float4(q, 0.0f, 0.0f, dq);
                    } else {
                        Yrow[l0 + m] = make_float4(q * cm, q * fm * cm1, -q * fm * sm1, dq * cm);
                        Yrow[l0 - m] = make_float4(q * sm, q * fm * sm1, q * fm * cm1, dq * sm);
                    }
                }
            }
        }
        // the next chunk's records go to the other buffer, whose last readers finished before this chunk's barrier
        if (stager && pos + chunk < seg_end) stage(pos + chunk, b ^ 1);
        __syncthreads();
        // contraction with chat, then dE/dr_ji, the force scatter and the virial: one warp per pair, lanes over lm
        for (int p = warp; p < nc; p += nwarps) {
            const int a = s_spc[bo + p];
            if (a < 0) continue;  // warp-uniform
            const float* H = s_H + a * kNmax * kNlm;
            const float2* gd = s_GD + p * kFpad;
            const float4* Yrow = s_Yv + p * Yp;
            float S = 0.0f, Wx = 0.0f, Wy = 0.0f, Wz = 0.0f;
            for (int lm = lane; lm < kNlm; lm += 32) {
                const float2* g = gd + s_lofm[lm] * kNpad;
                const float* h = H + lm;
                float uu = 0.0f, vv = 0.0f;
                for (int n = 0; n < kNmax; ++n) {
                    const float hv = h[n * kNlm];
                    const float2 x = g[n];
                    vv = fmaf(hv, x.x, vv);
                    uu = fmaf(hv, x.y, uu);
                }
                const float4 y = Yrow[lm];
                S = fmaf(uu, y.x, S);
                Wx = fmaf(vv, y.y, Wx);
                Wy = fmaf(vv, y.z, Wy);
                Wz = fmaf(vv, y.w, Wz);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, o);
                Wx += __shfl_xor_sync(0xffffffffu, Wx, o);
                Wy += __shfl_xor_sync(0xffffffffu, Wy, o);
                Wz += __shfl_xor_sync(0xffffffffu, Wz, o);
            }
            const float4 v = s_vec[bo + p];
            const float inv_r = 1.0f / v.w;
            const float ux = v.x * inv_r, uy = v.y * inv_r, uz = v.z * inv_r;
            const float wu = Wx * ux + Wy * uy + Wz * uz;
            const float g0 = S * ux + (Wx - wu * ux) * inv_r, g1 = S * uy + (Wy - wu * uy) * inv_r,
                        g2 = S * uz + (Wz - wu * uz) * inv_r;
            const int ra = lane < 3 ? lane : (lane - 3) / 3;  // lane 3 + 3 ra + rb: virial entry (ra, rb)
            const float ga = ra == 0 ? g0 : (ra == 1 ? g1 : g2);
            if (lane < 3) {
                const int j = s_j[bo + p];
                if (j != i) {
                    atomicAdd(&A.forces[3 * (int64_t)j + lane], -ga);
                    racc += ga;
                }
            } else if (lane < 12) {
                const int rb = (lane - 3) - 3 * ra;
                racc = fmaf(ga, rb == 0 ? v.x : (rb == 1 ? v.y : v.z), racc);
            }
        }
    }
    // block reduction of F_i and the virial
    if (lane < 12) red[warp][lane] = (double)racc;
    __syncthreads();
    if (tid < 12) {
        double s = 0.0;
        for (int w = 0; w < nwarps; ++w) s += red[w][tid];
        if (tid < 3) {
            if (s != 0.0) atomicAdd(&A.forces[3 * (int64_t)i + tid], (float)s);
        } else {
            atomicAdd(&A.virial[9 * (int64_t)s_sid + (tid - 3)], s);
        }
    } else if (tid == 32 && A.energy) {
        add_energy(s_e, nwarps, &A.energy[s_sid]);
    }
}

__global__ void k_forces_f64(int64_t n, const float* __restrict__ f32, double* __restrict__ f64) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        f64[e] = (double)f32[e];
}

// bytes from the pair area to the small tables: the pair records, then the larger of Y and G and the staged
// coefficients
static size_t grad_aux_off(const rascal_ctx* ctx, int chunk, bool tiled) {
    const ExpPlan& P = ctx->plan;
    const size_t QN4 = ((size_t)ctx->Q * ctx->n_lm + 3) / 4 * 4;
    const size_t QL4 = tiled ? ((size_t)ctx->Q * P.Lp + 3) / 4 * 4 : QN4;
    const size_t Yp = (size_t)(ctx->n_lm | 1);
    const size_t records = 2 * (sizeof(float4) + sizeof(float) * 2 + sizeof(int) * 2) * chunk;  // two buffers
    const size_t yg = sizeof(float4) * chunk * Yp + sizeof(float2) * chunk * P.F_pad;  // Y and G, or the coefficients
    return align_up(records + std::max(yg, sizeof(float) * QL4), 16);
}

static size_t grad_smem(const rascal_ctx* ctx, int chunk, bool tiled) {
    const ExpPlan& P = ctx->plan;
    const size_t QN4 = ((size_t)ctx->Q * ctx->n_lm + 3) / 4 * 4;
    return sizeof(float) * QN4 + grad_aux_off(ctx, chunk, tiled) + sizeof(int) * (ctx->n_lm + P.F_pad) + 64;
}

// bytes of k_gradients' shared memory before the area that the coefficients (with the dense weight block of a per-centre
// dE/dp behind them) and then the radial values use, and in all
static size_t grad_c_off(const rascal_ctx* ctx, int threads) {
    return sizeof(float) * ctx->n_species * grad_h_pitch(ctx->l_max, ctx->n_max) + 32 * (2 * 16 + threads / 32 * 16 + 2 * 16);
}
static size_t grad_c_bytes(const rascal_ctx* ctx, bool tiled) {
    return align_up(sizeof(float) * ctx->Q * (tiled ? ctx->plan.Lp : ctx->n_lm), 16);
}
static size_t grad_w_bytes(const rascal_ctx* ctx, int w_lg) { return sizeof(float) * w_lg * ((ctx->Q * (ctx->Q + 1) / 2) | 1); }
static size_t grad_chain_smem(const rascal_ctx* ctx, int threads, bool tiled, int w_lg) {
    const size_t c = grad_c_bytes(ctx, tiled) + grad_w_bytes(ctx, w_lg);
    return grad_c_off(ctx, threads) + std::max(c, sizeof(float) * 32 * grad_g_pitch(ctx->plan.F_pad));
}

using GradKernel = void (*)(GradArgs);
// by threads (256, 128), kind of weights and shape; no shape that is not listed for 128 threads is small enough for them
static const GradKernel kGradKernels[2][2][5] = {
    {{k_gradients<0, kLinear, 256>, k_gradients<1, kLinear, 256>, k_gradients<2, kLinear, 256>, k_gradients<3, kLinear, 256>,
      k_gradients<4, kLinear, 256>},
     {k_gradients<0, kPerCentre, 256>, k_gradients<1, kPerCentre, 256>, k_gradients<2, kPerCentre, 256>,
      k_gradients<3, kPerCentre, 256>, k_gradients<4, kPerCentre, 256>}},
    {{k_gradients<0, kLinear, 128>, nullptr, nullptr, k_gradients<3, kLinear, 128>, nullptr},
     {k_gradients<0, kPerCentre, 128>, nullptr, nullptr, k_gradients<3, kPerCentre, 128>, nullptr}}};
constexpr int kSplitGrad = kPerCentre | kSplitRows;
static const GradKernel kSplitKernels[3] = {k_gradients<0, kSplitGrad, 256>, k_gradients<4, kSplitGrad, 256>, k_gradients<0, kSplitGrad, 128>};
static_assert(kNumExpShapes == 5, "an instance per shape");

int gradients_setup(rascal_ctx* ctx) {
    RASCAL_CUDA(upload_ylm_constants(ctx->stream));
    RASCAL_CUDA(upload_ylm_down(ctx->stream));
    RASCAL_CUDA(cudaFuncSetAttribute(k_gradients_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    for (int t = 0; t < 2; ++t)
        for (int w = 0; w < 2; ++w)
            for (GradKernel k : kGradKernels[t][w])
                if (k) RASCAL_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    for (GradKernel k : kSplitKernels)
        RASCAL_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    return RASCAL_OK;
}

}  // namespace rascal

using namespace rascal;

extern "C" int rascal_linear_energy(rascal_ctx* ctx, const rascal_system* sys, const float* d_ps_packed,
                                    const float* d_weights, double* d_energy) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    int st = validate_system(ctx, sys);
    if (st) return st;
    if (!d_energy) return set_error(RASCAL_E_ARG, "NULL energy");
    RASCAL_CUDA(cudaMemsetAsync(d_energy, 0, sizeof(double) * sys->n_structures, ctx->stream));
    if (sys->n_atoms == 0) return RASCAL_OK;
    if (!d_ps_packed || !d_weights) return set_error(RASCAL_E_ARG, "NULL device pointer");
    const int64_t F = (int64_t)(ctx->l_max + 1) * ctx->Q * (ctx->Q + 1) / 2;
    k_linear_energy<<<sys->n_atoms, 256, 0, ctx->stream>>>(sys->n_atoms, sys->n_structures, sys->d_struct_offsets,
                                                          sys->d_species, ctx->d_lut, d_ps_packed, d_weights, F, d_energy);
    RASCAL_LAUNCH_CHECK("k_linear_energy");
    return RASCAL_OK;
}

static int gradients(rascal_ctx* ctx, const rascal_system* sys, const int64_t* d_offsets, const int* d_nbr_j,
                     const float* d_rij, const float* d_coeffs, const float* d_grad_ps, const float* d_weights,
                     double* d_energy, double* d_forces, double* d_virial) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    int st = validate_system(ctx, sys);
    if (st) return st;
    if (!d_forces || !d_virial) return set_error(RASCAL_E_ARG, "NULL forces or virial");
    if ((d_grad_ps == nullptr) == (d_weights == nullptr))
        return set_error(RASCAL_E_ARG, "exactly one of grad_ps and weights must be given");
    if (sys->n_atoms == 0) {
        RASCAL_CUDA(cudaMemsetAsync(d_virial, 0, sizeof(double) * 9 * sys->n_structures, ctx->stream));
        if (d_energy) RASCAL_CUDA(cudaMemsetAsync(d_energy, 0, sizeof(double) * sys->n_structures, ctx->stream));
        return RASCAL_OK;
    }
    if (!d_offsets || !d_nbr_j || !d_rij || !d_coeffs) return set_error(RASCAL_E_ARG, "NULL device pointer");
    const int L1 = ctx->l_max + 1;
    const int Qw = (ctx->Q + 3) / 4 * 4;
    const size_t n_ws = d_weights ? (size_t)ctx->n_species * L1 * ctx->Q * Qw : 0;
    void* wbase;
    if ((st = arena_get(ctx->scratch_w, carve_bytes(sizeof(float) * 3 * (size_t)sys->n_atoms, sizeof(float) * n_ws),
                        &wbase)))
        return st;
    Carver wcv(wbase);
    float* f32 = wcv.take<float>(3 * (size_t)sys->n_atoms);
    float* ws = wcv.take<float>(n_ws);
    const ExpPlan& P = ctx->plan;
    GradArgs A = {};
    A.offsets = d_offsets;
    A.nbr_j = d_nbr_j;
    A.rij = reinterpret_cast<const float4*>(d_rij);
    A.species = sys->d_species;
    A.lut = ctx->d_lut;
    A.offs = sys->d_struct_offsets;
    A.table = ctx->d_table;
    A.fmap = ctx->d_fmap;
    A.coeffs = d_coeffs;
    A.grad_ps = d_grad_ps;
    A.weights = d_weights;
    A.forces = f32;
    A.virial = d_virial;
    A.energy = d_energy;
    A.flags = ctx->d_flags;
    A.N = sys->n_atoms;
    A.n_s = sys->n_structures;
    A.n_max = ctx->n_max;
    A.l_max = ctx->l_max;
    A.S = ctx->n_species;
    A.Q = ctx->Q;
    A.n_lm = ctx->n_lm;
    A.F = ctx->F;
    A.F_pad = P.F_pad;
    A.n_pad = P.n_pad;
    A.Lp = P.Lp;
    A.M = ctx->M;
    A.ps_norm = ctx->ps_norm;
    A.Fp = (int64_t)(ctx->l_max + 1) * ctx->Q * (ctx->Q + 1) / 2;
    A.inv_delta = ctx->inv_delta;
    A.r_cut = (float)ctx->r_cut;
    A.width = (float)ctx->smooth_width;
    for (int l = 0; l < kMaxLMax + 2; ++l) A.lp[l] = P.lp[l];
    A.wsym = d_weights ? ws : nullptr;
    A.Qw = Qw;
    A.Lp_adj = P.Lp;
    A.n_adj_tasks = (ctx->Q + 3) / 4 * (P.Lp / 4);
    // Small bases take CTAs of 128 threads, of which eight (six with dE/dp) fit an SM: their few l leave half of eight warps
    // without a task, and more CTAs hide each other's barriers: 16 000 centres of 31 pairs (8, 6, 2) 205 -> 155 us, of 25 pairs (7, 5,
    // 2) 293 -> 228, of 29 pairs (5, 3, 1) 227 -> 152; with dE/dp 25 262 centres (5, 4, 2) 519 -> 350.
    const int per_sm = d_weights ? 8 : 6;
    const bool small = grad_chain_smem(ctx, 128, true, d_weights ? 0 : L1) <= 226 * 1024 / per_sm - 2 * 1024;
    const int threads = small ? 128 : 256;
    // a per-centre dE/dp: all its l blocks staged at once where two CTAs per SM still fit, else as many as fit (two CTAs, or one
    // where one block leaves room for no more). Wide bases of a few l read it from global memory (an output per thread): 3 000
    // centres of Q = 128, l_max 0 181 -> 101 us, l_max 2 486 -> 344.
    A.w_lg = d_weights ? 0 : L1;
    const size_t room = (!d_weights && grad_chain_smem(ctx, threads, true, 1) > 112 * 1024 ? 220 : 112) * 1024;
    while (A.w_lg > 1 && grad_chain_smem(ctx, threads, true, A.w_lg) > room) --A.w_lg;
    if (A.w_lg && grad_chain_smem(ctx, threads, true, A.w_lg) > 220 * 1024) A.w_lg = 0;
    if (ctx->Q > 96 && ctx->l_max <= 2) A.w_lg = 0;
    size_t smem = grad_chain_smem(ctx, threads, A.wsym || A.w_lg, A.w_lg);
    const bool chains = smem <= 220 * 1024;  // all but the widest bases (about n_species n_max (l_max + 1)^2 > 24 500)
    {  // rows of a warp: the fewest rounds x (loads of a step)
        const int w = threads / 32;
        auto cost = [&](int r) { return (ctx->Q + r * w - 1) / (r * w) * (r + 4); };
        A.w_rows = cost(6) < cost(4) ? 6 : 4;
    }
    if (chains) {
        A.chunk = 32;
        A.w_off = (int)(grad_c_off(ctx, threads) + grad_c_bytes(ctx, true));
        A.aux_off = 0;
    } else {
        // the largest chunk (<= 32: one warp stages a chunk, a pair per lane) that keeps five CTAs per SM (48 registers)
        const bool tiled = A.wsym != nullptr;
        int chunk = 32;
        while (chunk > 1 && grad_smem(ctx, chunk, tiled) > 44 * 1024) --chunk;
        // the radial and contraction phases deal the chunk's pairs to the 8 warps: a chunk one or two pairs past a
        // multiple of 8 is rounded down, so that no nearly empty last round remains (rounding down only shrinks the
        // shared memory below)
        constexpr int kW = kGradThreads / 32;
        if (chunk > kW && chunk % kW <= 2) chunk -= chunk % kW;
        // every shared-memory offset and the size come from this final chunk
        A.chunk = chunk;
        A.w_lg = 0;
        A.aux_off = (int)grad_aux_off(ctx, chunk, tiled);
        smem = grad_smem(ctx, chunk, tiled);
        if (smem > 220 * 1024) return set_error(RASCAL_E_UNSUPPORTED, "hypers too large for the gradient kernel");
    }
    if ((st = radial_precompute(ctx, sys, d_offsets, d_rij, true, &A.pre_G, &A.pre_D))) return st;
    const int64_t n3 = 3 * (int64_t)sys->n_atoms, n_prep = std::max({n3, (int64_t)n_ws, 9 * (int64_t)sys->n_structures});
    k_prepare<<<(unsigned)std::min<int64_t>((n_prep + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        ctx->n_species, L1, ctx->Q, Qw, ctx->ps_norm, d_weights, A.Fp, d_weights ? ws : nullptr, n3, f32, sys->n_structures,
        d_virial, d_energy);
    RASCAL_LAUNCH_CHECK("k_prepare");
    // a compiled instance for the hyper shape when the plan's sizes match it (kExpShapes), else the generic kernel
    int shape = 0;
    for (int k = 1; k < kNumExpShapes && !shape; ++k) {
        const ExpShape& c = kExpShapes[k];
        if (ctx->n_max == c.n_max && ctx->l_max == c.l_max && ctx->n_species == c.S && P.n_pad == exp_npad(c.n_max) &&
            P.F_pad == (c.l_max + 1) * exp_npad(c.n_max) && P.Lp == exp_lp(c.l_max + 1) && ctx->Q == c.n_max * c.S &&
            ctx->n_lm == (c.l_max + 1) * (c.l_max + 1) && ctx->F == (c.l_max + 1) * c.n_max && (!A.wsym || A.Qw == (ctx->Q + 3) / 4 * 4))
            shape = k;
    }
    if (chains) {
        GradKernel kernel = kGradKernels[small][d_weights ? 0 : 1][shape];
        if (!kernel) kernel = kGradKernels[small][d_weights ? 0 : 1][0];
        bool split = false;  // a group of l with fewer tiles than half a warp's lanes
        for (int l = 0; l < L1 && A.w_lg; l += A.w_lg) split = split || exp_lp(std::min(L1, l + A.w_lg)) - exp_lp(l) <= 4 * 16;
        if (split && ctx->Q > 4 * threads / 32) kernel = kSplitKernels[small ? 2 : (shape == 4 ? 1 : 0)];
        kernel<<<sys->n_atoms, threads, smem, ctx->stream>>>(A);
    } else {
        k_gradients_wide<<<sys->n_atoms, kGradThreads, smem, ctx->stream>>>(A);
    }
    RASCAL_LAUNCH_CHECK("k_gradients");
    k_forces_f64<<<(unsigned)std::min<int64_t>((n3 + 255) / 256, 8192), 256, 0, ctx->stream>>>(n3, f32, d_forces);
    RASCAL_LAUNCH_CHECK("k_forces_f64");
    return RASCAL_OK;
}

extern "C" int rascal_gradients(rascal_ctx* ctx, const rascal_system* sys, const int64_t* d_offsets, const int* d_nbr_j,
                                const float* d_rij, const float* d_coeffs, const float* d_grad_ps, const float* d_weights,
                                double* d_forces, double* d_virial) {
    return gradients(ctx, sys, d_offsets, d_nbr_j, d_rij, d_coeffs, d_grad_ps, d_weights, nullptr, d_forces, d_virial);
}

extern "C" int rascal_linear_gradients(rascal_ctx* ctx, const rascal_system* sys, const int64_t* d_offsets,
                                       const int* d_nbr_j, const float* d_rij, const float* d_coeffs, const float* d_weights,
                                       double* d_energy, double* d_forces, double* d_virial) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (!d_energy) return set_error(RASCAL_E_ARG, "NULL energy");
    if (int st = soap_supported(ctx)) return st;  // the same bases with forces as without (which take a power spectrum)
    return gradients(ctx, sys, d_offsets, d_nbr_j, d_rij, d_coeffs, nullptr, d_weights, d_energy, d_forces, d_virial);
}

namespace rascal {

// Per-pair feature gradient, explicitly (a test hook for small cases): for pair p with vector r = r_ji,
//   d[p][x][n][lm] = d/dr_x [ f_cut(r) I^o_nl(r) Y_lm(r^) ] = (f I)'(r) Y_lm u_x + f I (dY/du - (dY/du . u) u)_x / r,
// the derivative of the pair's term in c^i_{a_j n l m} (Eq. spherical_expansion_coefficients_gaussians, Appendix B).
// One CTA per pair: thread m < l_max + 1 runs the m chain of Y and of its polynomial-extension gradient, then the
// threads cover (n, lm).
__global__ void k_debug_pair_grad(int64_t P, const float4* __restrict__ rij, const float4* __restrict__ table,
                                  const float* __restrict__ pre_G, const float* __restrict__ pre_D, int n_max, int l_max,
                                  int F, int M, float inv_delta, float r_cut, float width, float* __restrict__ out) {
    extern __shared__ float sdbg[];
    const int n_lm = (l_max + 1) * (l_max + 1);
    float4* sY = reinterpret_cast<float4*>(sdbg);  // [n_lm] (Y, dY/dux, dY/duy, dY/duz)
    float2* sR = reinterpret_cast<float2*>(sY + n_lm);  // [F] (f I, (f I)')
    const int64_t p = blockIdx.x;
    const float4 v = rij[p];
    const float inv_r = v.w > 1e-6f ? 1.0f / v.w : 0.0f;
    const float x = v.x * inv_r, y = v.y * inv_r, z = v.z * inv_r;
    const int L1 = l_max + 1;
    for (int m = threadIdx.x; m < L1; m += blockDim.x) {
        float cm = 1.0f, sm = 0.0f, cm1 = 0.0f, sm1 = 0.0f;
        for (int t = 0; t < m; ++t) {
            cm1 = cm;
            sm1 = sm;
            const float nc = cm * x - sm * y;
            sm = cm * y + sm * x;
            cm = nc;
        }
        const float fm = (float)m;
        float q2 = 0.0f, q1 = c_ylm_K[m], d2 = 0.0f, d1 = 0.0f;
        for (int l = m; l < L1; ++l) {
            float q = q1, dq = d1;
            if (l > m) {
                const float Al = c_ylm_A[l * 16 + m], Bl = c_ylm_B[l * 16 + m];
                q = Al * (z * q1 - Bl * q2);
                dq = Al * (q1 + z * d1 - Bl * d2);
                q2 = q1;
                d2 = d1;
                q1 = q;
                d1 = dq;
            }
            const int l0 = l * l + l;
            if (m == 0) {
                sY[l0] = make_float4(q, 0.0f, 0.0f, dq);
            } else {
                sY[l0 + m] = make_float4(q * cm, q * fm * cm1, -q * fm * sm1, dq * cm);
                sY[l0 - m] = make_float4(q * sm, q * fm * sm1, q * fm * cm1, dq * sm);
            }
        }
    }
    float f, df;
    cutoff_and_slope(v.w, r_cut, width, f, df);
    for (int c = threadIdx.x; c < F; c += blockDim.x) {  // column l n_max + n
        float g, dg;
        if (pre_G) {
            g = pre_G[p * F + c];
            dg = pre_D[p * F + c];
        } else {
            const float xk = v.w * inv_delta;
            const int k = min(max((int)xk, 0), M - 1);
            const float u = xk - (float)k;
            const float4 cf = table[(int64_t)k * F + c];
            g = fmaf(u, fmaf(u, fmaf(u, cf.w, cf.z), cf.y), cf.x);
            dg = fmaf(u, fmaf(u, 3.0f * cf.w, 2.0f * cf.z), cf.y) * inv_delta;
        }
        sR[c] = make_float2(f * g, df * g + f * dg);
    }
    __syncthreads();
    const int per = n_max * n_lm;
    float* o = out + p * 3 * per;
    for (int e = threadIdx.x; e < per; e += blockDim.x) {
        const int n = e / n_lm, lm = e - n * n_lm;
        const int l = (int)sqrtf((float)lm);
        const float2 R = sR[l * n_max + n];
        const float4 Yv = sY[lm];
        const float wu = Yv.y * x + Yv.z * y + Yv.w * z;
        o[e] = R.y * Yv.x * x + R.x * (Yv.y - wu * x) * inv_r;
        o[per + e] = R.y * Yv.x * y + R.x * (Yv.z - wu * y) * inv_r;
        o[2 * per + e] = R.y * Yv.x * z + R.x * (Yv.w - wu * z) * inv_r;
    }
}

}  // namespace rascal

extern "C" int rascal_debug_pair_gradients(rascal_ctx* ctx, int64_t n_pairs, const float* d_rij, float* d_dc) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (n_pairs < 0 || n_pairs > (1 << 20)) return set_error(RASCAL_E_ARG, "n_pairs must be in [0, 2^20] (a test hook)");
    if (n_pairs == 0) return RASCAL_OK;
    if (!d_rij || !d_dc) return set_error(RASCAL_E_ARG, "NULL device pointer");
    const float* G = nullptr;
    const float* D = nullptr;
    if (ctx->radial != RASCAL_RADIAL_SPLINE) {
        if (ctx->radial == RASCAL_RADIAL_MLP && !ctx->mlp_params)
            return set_error(RASCAL_E_ARG, "radial mode MLP needs trained parameters");
        const size_t words = (size_t)n_pairs * ctx->F;
        void* base;
        int st = arena_get(ctx->scratch, carve_bytes(words * 4, words * 4), &base);
        if (st) return st;
        Carver cv(base);
        float* g = cv.take<float>(words);
        float* d = cv.take<float>(words);
        const float4* rij = reinterpret_cast<const float4*>(d_rij);
        st = ctx->radial == RASCAL_RADIAL_MLP ? mlp_infer(ctx, n_pairs, rij, nullptr, g, d)
                                              : radial_exact_pairs(ctx, n_pairs, rij, g, d);
        if (st) return st;
        G = g;
        D = d;
    }
    const size_t smem = sizeof(float4) * ctx->n_lm + sizeof(float2) * ctx->F;
    k_debug_pair_grad<<<(unsigned)n_pairs, 128, smem, ctx->stream>>>(
        n_pairs, reinterpret_cast<const float4*>(d_rij), ctx->d_table, G, D, ctx->n_max, ctx->l_max, ctx->F, ctx->M,
        ctx->inv_delta, (float)ctx->r_cut, (float)ctx->smooth_width, d_dc);
    RASCAL_LAUNCH_CHECK("k_debug_pair_grad");
    return RASCAL_OK;
}
