// nu = 2 equivariants (lambda-SOAP, Sec. "Experimental features"): the symmetrised correlation of Eq. body-order-x at
// nu = 2 coupled to rank lambda instead of contracted to an invariant,
//   T^{lambda mu}_{(q1 l1)(q2 l2)} = sum_{m1 m2} R^{l1 l2 lambda}[m1][m2][mu] c_{q1 l1 m1} c_{q2 l2 m2},
// with R the Clebsch-Gordan coefficients <l1 m1; l2 m2 | lambda M> (Condon-Shortley) carried into the basis of the
// real harmonics the coefficients use (no Condon-Shortley phase): R = U_lambda . CG . conj(U_l1) . conj(U_l2), real
// for l1 + l2 + lambda even. Only those proper tensors are formed (the improper-rotation average of Eq. body-order-x
// removes the others), and only l1 <= l2: T(l2, l1) is the transpose of T(l1, l2).
//
// Host: Racah's closed form for the CG coefficients in FP64, the unitary U per l, the real tables per (l1, l2), kept
// as their (at most two) non-zero m1 terms per (mu, m2), cached per lambda in the context. Device: one CTA per centre
// with its coefficients in shared memory; per pair the half-contractions X[q1][m2] = sum_m1 R c_{q1 l1 m1} and the
// output tiles T[q1][q2] = sum_m2 X[q1][m2] c_{q2 l2 m2}. Bound: HBM (the output).
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "f32x2.cuh"

namespace rascal {

struct LsoapTable {
    int lambda = -1;
    int n_pairs = 0;
    int4* d_hdr = nullptr;   // per pair: first slots of l1 and l2 in a padded row, offset of its entries in d_R,
                             // 2 l2 + 1 | ceil(65536 / (2 l2 + 1 rounded up to 4)) << 6
    float4* d_R = nullptr;   // per pair [2 lambda + 1][2 l2 + 1]: the (at most two) non-zero m1 terms of R[mu][.][m2]
                             // as {value0, value1, m1_0, m1_1} (indices as integer bits; value 0 pads)
};

static double fact(int n) {
    double f = 1.0;
    for (int k = 2; k <= n; ++k) f *= k;
    return f;
}

// <l1 m1; l2 m2 | L M>, Racah's closed form
static double cg(int l1, int m1, int l2, int m2, int L, int M) {
    if (m1 + m2 != M || L < std::abs(l1 - l2) || L > l1 + l2 || std::abs(m1) > l1 || std::abs(m2) > l2 || std::abs(M) > L)
        return 0.0;
    const double pref = std::sqrt((2.0 * L + 1.0) * fact(L + l1 - l2) * fact(L - l1 + l2) * fact(l1 + l2 - L) /
                                  fact(l1 + l2 + L + 1) * fact(L + M) * fact(L - M) * fact(l1 - m1) * fact(l1 + m1) *
                                  fact(l2 - m2) * fact(l2 + m2));
    double s = 0.0;
    for (int k = 0; k <= l1 + l2; ++k) {
        const int a[6] = {k, l1 + l2 - L - k, l1 - m1 - k, l2 + m2 - k, L - l2 + m1 + k, L - l1 - m2 + k};
        bool neg = false;
        for (int v : a) neg |= v < 0;
        if (neg) continue;
        double den = 1.0;
        for (int v : a) den *= fact(v);
        s += ((k & 1) ? -1.0 : 1.0) / den;
    }
    return pref * s;
}

// U[(m' + l)(2l+1) + (m + l)]: Y^real_{l m'} = sum_m U Y^CS_{l m}. With Z^m = N P^|m| e^{i m phi}, Y^CS_m = (-1)^m Z^m
// (m > 0) and Z^m (m <= 0); the real harmonics are Z^0, (Z^m + Z^-m)/sqrt 2 and (Z^m - Z^-m)/(i sqrt 2) (index -m).
static std::vector<std::complex<double>> u_matrix(int l) {
    const int d = 2 * l + 1;
    std::vector<std::complex<double>> U((size_t)d * d, 0.0);
    const double r = 1.0 / std::sqrt(2.0);
    const std::complex<double> I(0.0, 1.0);
    U[(size_t)l * d + l] = 1.0;
    for (int m = 1; m <= l; ++m) {
        const double sg = (m & 1) ? -1.0 : 1.0;
        U[(size_t)(l + m) * d + (l + m)] = sg * r;
        U[(size_t)(l + m) * d + (l - m)] = r;
        U[(size_t)(l - m) * d + (l + m)] = sg * r / I;
        U[(size_t)(l - m) * d + (l - m)] = -r / I;
    }
    return U;
}

// real coupling table [mu][m1'][m2'] for (l1, l2) -> L; false if it is not real (never for l1 + l2 + L even)
static bool real_table(int l1, int l2, int L, std::vector<float>& out) {
    const int d1 = 2 * l1 + 1, d2 = 2 * l2 + 1, dL = 2 * L + 1;
    const auto U1 = u_matrix(l1), U2 = u_matrix(l2), UL = u_matrix(L);
    out.assign((size_t)dL * d1 * d2, 0.0f);
    for (int u = 0; u < dL; ++u)
        for (int x = 0; x < d1; ++x)
            for (int y = 0; y < d2; ++y) {
                std::complex<double> acc = 0.0;
                for (int a = 0; a < d1; ++a) {
                    const std::complex<double> ua = std::conj(U1[(size_t)x * d1 + a]);
                    if (ua == 0.0) continue;
                    for (int b = 0; b < d2; ++b) {
                        const int M = (a - l1) + (b - l2);
                        if (std::abs(M) > L) continue;
                        const std::complex<double> ub = std::conj(U2[(size_t)y * d2 + b]);
                        if (ub == 0.0) continue;
                        acc += UL[(size_t)u * dL + (M + L)] * cg(l1, a - l1, l2, b - l2, L, M) * ua * ub;
                    }
                }
                if (std::abs(acc.imag()) > 1e-10) return false;
                out[((size_t)u * d1 + x) * d2 + y] = (float)acc.real();
            }
    return true;
}

static void lsoap_pairs(int l_max, int lam, std::vector<int2>& p) {
    p.clear();
    for (int l1 = 0; l1 <= l_max; ++l1)
        for (int l2 = l1; l2 <= l_max; ++l2)
            if (std::abs(l1 - l2) <= lam && lam <= l1 + l2 && ((l1 + l2 + lam) & 1) == 0) p.push_back(make_int2(l1, l2));
}

// One CTA per centre. Rows and columns of the output go in groups of four: with Q a multiple of 4 (VEC) group g holds
// q = 4 g .. 4 g + 3, so that a thread's four columns are adjacent and leave as one streaming 16-byte store; otherwise it
// holds g, g + QT, g + 2 QT, g + 3 QT (QT = ceil(Q / 4)), so that the scalar stores of neighbouring lanes are adjacent.
// The centre's coefficients are staged once as C[g][v][slot], every l block of a row padded with zeros to a multiple of 4
// slots (exp_lp), so that both contractions read 16-byte pieces along m; a group's 16 bytes of slack make neighbouring
// groups' rows differ by an odd number of 16-byte words (conflict-free).
// Per pair (l1, l2) the row groups of all mu (tau = mu QT + g) are made in chunks: the half-contractions
// X[tau][v][m2] = sum_m1 R c_{q1 l1 m1} of a chunk go to one of two buffers (pads zero; row pitch PX, a compile-time
// constant, so that the loads of a tile's rows need no address arithmetic), one block barrier, then 8 x 4 output tiles
// per thread (two row groups), summed over m2 four at a time: 12 16-byte shared loads and 64 paired FMAs (even and odd m2
// in the two halves of an accumulator, added at the end) for 128 products.
// Bound: HBM (the output). 9 001 centres, Q = 48, l_max 9, lambda 1: 1 017 us with 2 x 4 tiles that loaded one value of X
// per two products (issue-bound, 83 % issue-active); 718 us with 4 x 4 tiles (shared-memory loads 74 % of their rate);
// 637 us = 3.8 TB/s in this form. Four CTAs of 128 threads per SM hide the barriers better than two of 256
// (692 against 844 us with runtime pitches). Where an SM has one or two CTAs at most the pairs follow each other with nothing
// to hide their latency: there a CTA has 256 threads (G = 1) and asks for a thread's first table entry of the next pair before
// it makes this one's tiles (kLsoapPrefetch below).
constexpr int kLsoapThreads = 128, kLsoapCtas = 4;
constexpr int kLsoapGroups = 36;  // row groups per chunk: X takes 11.5 KB (PX = 20) or 20.7 KB (PX = 36) per buffer

template <bool VEC, int PX, int G, int T>
__global__ void __launch_bounds__(T, T > kLsoapThreads ? 2 : (G == 1 ? 6 : kLsoapCtas)) k_lambda_soap(const float* __restrict__ c, int Q, int l_max, int lam,
                                                                           int chunk, unsigned qt_inv, int n_pairs,
                                                                           const int4* __restrict__ hdr,
                                                                           const float4* __restrict__ R,
                                                                           float* __restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    const int64_t i = blockIdx.x;
    const int n_lm = (l_max + 1) * (l_max + 1), pitch = exp_ly(l_max), gs = 4 * pitch + 4, QT = (Q + 3) >> 2;
    const int tid = threadIdx.x, groups = (2 * lam + 1) * QT;
    float* C = sm;                           // [QT][gs]
    float* sX = C + QT * gs;                 // two buffers [chunk][4][PX]
    const float* ci = c + i * Q * n_lm;
    for (int e = tid; e < QT * gs / 4; e += T) reinterpret_cast<float4*>(C)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto div_qt = [&](int x) { return QT == 1 ? x : (int)__umulhi((unsigned)x, qt_inv); };  // x / QT, exact for x < 65536
    __syncthreads();
    {
        const int warp = tid >> 5, lane = tid & 31;
        for (int lm = lane; lm < n_lm; lm += 32) {  // lanes over lm: coalesced, the slot worked out once
            const int l = (int)sqrtf((float)lm);
            float* slot = C + exp_lp(l) + lm - l * l;
#pragma unroll 4
            for (int q = warp; q < Q; q += T / 32) {
                const int v = VEC ? q & 3 : div_qt(q), g = VEC ? q >> 2 : q - v * QT;
                slot[g * gs + v * pitch] = __ldg(ci + q * n_lm + lm);
            }
        }
    }
    // output tiling (fixed for the kernel): each thread owns one column group and a stride of row groups
    const int t_r = div_qt(tid), t_c = tid - t_r * QT, r_step = div_qt(T);
    const bool t_on = t_r < r_step;
    const int64_t pair_floats = (int64_t)(2 * lam + 1) * Q * Q;
    float* op = out + i * n_pairs * pair_floats + (VEC ? 4 * t_c : t_c);
    const int x_floats = chunk * 4 * PX;
    int cur = 0;  // offset of the X buffer in use
    int4 h = __ldg(hdr);
    constexpr bool kLsoapPrefetch = T > 128;
    float4 e0 = make_float4(0.f, 0.f, 0.f, 0.f);  // this thread's first entry of the pair to come
    auto fetch = [&](const int4& n) {
        const int d2 = n.w & 63, dp = (d2 + 3) & ~3, r = (tid * (n.w >> 6)) >> 16, col = tid - r * dp;
        if (col < d2 && r < min(chunk, groups)) e0 = __ldg(R + n.z + col + div_qt(r) * d2);
    };
    if (kLsoapPrefetch) fetch(h);
    __syncthreads();
    for (int p = 0; p < n_pairs; ++p, op += pair_floats) {
        const int d2 = h.w & 63, dp = (d2 + 3) & ~3, inv = h.w >> 6;  // inv = ceil(65536 / dp)
        const int b_r = (tid * inv) >> 16, b_c = tid - b_r * dp, b_s = (T * inv) >> 16;
        const float4* Rp = R + h.z + b_c;
        const float* A = C + h.x;
        const float* Bt = C + h.y + t_c * gs;
        h = __ldg(hdr + min(p + 1, n_pairs - 1));
        for (int g0 = 0; g0 < groups; g0 += chunk, cur = x_floats - cur) {
            const int ng = min(chunk, groups - g0);
            float* X = sX + cur;
            if (b_r < b_s) {
#pragma unroll 2
                for (int r = b_r; r < ng; r += b_s) {
                    const int u = div_qt(g0 + r);
                    float w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    if (b_c < d2) {
                        // the two non-zero m1 of this (mu, m2)
                        const float4 e = kLsoapPrefetch && g0 == 0 && r == b_r ? e0 : __ldg(Rp + u * d2);
                        const float* ag = A + (g0 + r - u * QT) * gs;
                        const float* a0 = ag + __float_as_int(e.z);
                        const float* a1 = ag + __float_as_int(e.w);
#pragma unroll
                        for (int v = 0; v < 4; ++v) w[v] = fmaf(e.x, a0[v * pitch], e.y * a1[v * pitch]);
                    }
                    float* x = X + r * 4 * PX + b_c;
#pragma unroll
                    for (int v = 0; v < 4; ++v) x[v * PX] = w[v];
                }
            }
            if (kLsoapPrefetch && g0 + chunk >= groups) fetch(h);
            __syncthreads();
            if (!t_on) continue;
            const int half = G == 2 ? (ng + 1) >> 1 : ng;  // a thread's row groups: r and, with G = 2, r + half, if there is one
#pragma unroll 1
            for (int r = t_r; r < half; r += r_step) {
                uint64_t acc[4 * G][4];
                const bool two = G == 2 && r + half < ng;
                const float* x0 = X + r * 4 * PX;
                const float* x1 = two ? x0 + half * 4 * PX : x0;
                const float *b0 = Bt, *b1 = Bt + pitch, *b2 = b1 + pitch, *b3 = b2 + pitch;
#pragma unroll
                for (int u = 0; u < 4 * G; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] = 0ull;
#pragma unroll 1
                for (int m = 0; m < dp; m += 4) {
                    ulonglong2 b[4];
                    b[0] = *reinterpret_cast<const ulonglong2*>(b0);
                    b[1] = *reinterpret_cast<const ulonglong2*>(b1);
                    b[2] = *reinterpret_cast<const ulonglong2*>(b2);
                    b[3] = *reinterpret_cast<const ulonglong2*>(b3);
#pragma unroll
                    for (int u = 0; u < 4 * G; ++u) {
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>((u < 4 ? x0 : x1) + (u & 3) * PX);
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            acc[u][v] = f2_fma(x.x, b[v].x, acc[u][v]);
                            acc[u][v] = f2_fma(x.y, b[v].y, acc[u][v]);
                        }
                    }
                    b0 += 4;
                    b1 += 4;
                    b2 += 4;
                    b3 += 4;
                    x0 += 4;
                    x1 += 4;
                }
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    if (k == 1 && !two) break;
                    const int tau = g0 + r + k * half, mu = div_qt(tau), g = tau - mu * QT;
                    float* o = op + (mu * Q + (VEC ? 4 * g : g)) * Q;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!VEC && g + QT * u >= Q) break;
                        float w[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            float lo, hi;
                            f2_unpack(acc[4 * k + u][v], lo, hi);
                            w[v] = lo + hi;
                        }
                        if (VEC) {
                            __stcs(reinterpret_cast<float4*>(o), make_float4(w[0], w[1], w[2], w[3]));
                        } else {
#pragma unroll
                            for (int v = 0; v < 4; ++v)
                                if (t_c + QT * v < Q) __stcs(o + QT * v, w[v]);
                        }
                        o += VEC ? Q : QT * Q;
                    }
                }
            }
        }
    }
}

// row pitch of X: 20 holds the widest pair up to l_max 9 (2 l_max + 1 <= 20), 36 every other; an odd number of 16-byte words
static int lsoap_px(int l_max) { return l_max <= 9 ? 20 : 36; }

// Row groups of a thread's tiles: one where a chunk's 4 x 4 tiles do not exceed the threads (small bases, small ranks), else two;
// with one, six CTAs per SM (78 registers). Two groups (and 2 x 4 tiles) -> one: 4 000 centres, Q = 15, l_max 9, lambda 0 106
// (100) -> 72 us; 9 000 centres, Q = 21, l_max 3, lambda 1 90 (167) -> 72 us; 5 000 centres, Q = 12, l_max 4, lambda 0 53 (45) ->
// 37 us. Past the line two groups win (3 000 centres, Q = 30, l_max 5, lambda 1 62 against 70 us), but for pairs of a few m, which
// are over before two groups pay (5 000 centres, l_max 1: Q = 60, lambda 1 52 -> 47 us, Q = 36, lambda 2 43 -> 37), and, to l_max 4,
// for batches that four CTAs per SM leave a few centres of and six do not (700 centres: Q = 20, l_max 4, lambda 4 41 -> 31 us, Q = 60,
// l_max 2, lambda 2 45 -> 39; l_max 8 loses 7 %).
static bool lsoap_small(int Q, int l_max, int lam) {
    const int QT = (Q + 3) / 4;
    return l_max <= 1 || std::min((2 * lam + 1) * QT, kLsoapGroups) * QT <= kLsoapThreads;
}
enum LsoapForm { kLsoapTwo, kLsoapOne, kLsoapAlone };  // row groups per thread, or the form for one or two CTAs to an SM

template <int G, int T>
static auto lsoap_kernel_of(int Q, int l_max) {
    const bool vec = Q % 4 == 0;
    return lsoap_px(l_max) == 20 ? (vec ? k_lambda_soap<true, 20, G, T> : k_lambda_soap<false, 20, G, T>)
                                 : (vec ? k_lambda_soap<true, 36, G, T> : k_lambda_soap<false, 36, G, T>);
}
static auto lsoap_kernel(int Q, int l_max, LsoapForm form) {
    return form == kLsoapAlone ? lsoap_kernel_of<1, 2 * kLsoapThreads>(Q, l_max)
                               : (form == kLsoapOne ? lsoap_kernel_of<1, kLsoapThreads>(Q, l_max) : lsoap_kernel_of<2, kLsoapThreads>(Q, l_max));
}

int lsoap_table(rascal_ctx* ctx, int lam, int* n_pairs, const int4** hdr, const float4** R) {
    if (lam < 0 || lam > 2 * ctx->l_max) return set_error(RASCAL_E_ARG, "lambda must be in [0, 2 l_max] = [0, %d]", 2 * ctx->l_max);
    LsoapTable*& tab = ctx->lsoap[lam];
    if (!tab) {
        std::vector<int2> P;
        lsoap_pairs(ctx->l_max, lam, P);
        std::vector<int4> h(P.size());
        std::vector<float4> all;
        std::vector<float> one;
        for (size_t k = 0; k < P.size(); ++k) {
            const int l1 = P[k].x, l2 = P[k].y, d1 = 2 * l1 + 1, d2 = 2 * l2 + 1;
            if (!real_table(l1, l2, lam, one))
                return set_error(RASCAL_E_UNSUPPORTED, "coupling (%d, %d) -> %d is not real", l1, l2, lam);
            const int dp = (d2 + 3) / 4 * 4;
            h[k] = make_int4(exp_lp(l1), exp_lp(l2), (int)all.size(), d2 | ((65536 + dp - 1) / dp) << 6);
            for (int u = 0; u < 2 * lam + 1; ++u)
                for (int m2 = 0; m2 < d2; ++m2) {
                    float v[2] = {0.0f, 0.0f};
                    int o[2] = {0, 0}, nz = 0;
                    for (int m1 = 0; m1 < d1; ++m1) {
                        const float r = one[((size_t)u * d1 + m1) * d2 + m2];
                        if (std::fabs(r) < 1e-7f) continue;  // exact zeros up to the rounding of the FP64 sums
                        if (nz == 2)
                            return set_error(RASCAL_E_UNSUPPORTED, "coupling (%d, %d) -> %d has more than two terms",
                                             l1, l2, lam);
                        v[nz] = r;
                        o[nz++] = m1;
                    }
                    float f[2];
                    std::memcpy(f, o, sizeof(f));  // indices travel as integer bits
                    all.push_back(make_float4(v[0], v[1], f[0], f[1]));
                }
        }
        LsoapTable* t = new LsoapTable();
        t->lambda = lam;
        t->n_pairs = (int)P.size();
        cudaError_t e = cudaSuccess;
        for (LsoapForm f : {kLsoapTwo, kLsoapOne, kLsoapAlone})
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(lsoap_kernel(ctx->Q, ctx->l_max, f), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess) e = cudaMalloc(&t->d_hdr, sizeof(int4) * std::max<size_t>(1, h.size()));
        if (e == cudaSuccess) e = cudaMalloc(&t->d_R, sizeof(float4) * std::max<size_t>(1, all.size()));
        if (e == cudaSuccess && !h.empty())
            e = cudaMemcpy(t->d_hdr, h.data(), sizeof(int4) * h.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && !all.empty())
            e = cudaMemcpy(t->d_R, all.data(), sizeof(float4) * all.size(), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            cudaFree(t->d_hdr);
            cudaFree(t->d_R);
            delete t;
            return set_error(RASCAL_E_CUDA, "lambda-SOAP tables: %s", cudaGetErrorString(e));
        }
        tab = t;
    }
    *n_pairs = tab->n_pairs;
    *hdr = tab->d_hdr;
    *R = tab->d_R;
    return RASCAL_OK;
}

void lsoap_free(rascal_ctx* ctx) {
    for (auto& t : ctx->lsoap) {
        if (!t) continue;
        cudaFree(t->d_hdr);
        cudaFree(t->d_R);
        delete t;
        t = nullptr;
    }
}

}  // namespace rascal

using namespace rascal;

extern "C" int rascal_lambda_soap_size(const rascal_ctx* ctx, int lambda, int* n_pairs, int64_t* features_per_centre) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (lambda < 0 || lambda > 2 * ctx->l_max)
        return set_error(RASCAL_E_ARG, "lambda must be in [0, 2 l_max] = [0, %d]", 2 * ctx->l_max);
    std::vector<int2> P;
    lsoap_pairs(ctx->l_max, lambda, P);
    if (n_pairs) *n_pairs = (int)P.size();
    if (features_per_centre) *features_per_centre = (int64_t)P.size() * (2 * lambda + 1) * ctx->Q * ctx->Q;
    return RASCAL_OK;
}

extern "C" int rascal_debug_real_coupling(int l1, int l2, int lambda, float* R) {
    clear_error();
    if (l1 < 0 || l2 < 0 || l1 > kMaxLMax || l2 > kMaxLMax || lambda < std::abs(l1 - l2) || lambda > l1 + l2 ||
        ((l1 + l2 + lambda) & 1) || !R)
        return set_error(RASCAL_E_ARG, "l1, l2 <= %d, |l1 - l2| <= lambda <= l1 + l2, l1 + l2 + lambda even", kMaxLMax);
    std::vector<float> t;
    if (!real_table(l1, l2, lambda, t)) return set_error(RASCAL_E_UNSUPPORTED, "coupling is not real");
    std::memcpy(R, t.data(), t.size() * sizeof(float));
    return RASCAL_OK;
}

extern "C" int rascal_lambda_soap(rascal_ctx* ctx, int64_t n_centres, const float* d_coeffs, int lambda, float* d_out) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    if (n_centres < 0) return set_error(RASCAL_E_ARG, "negative n_centres");
    int np;
    const int4* hdr;
    const float4* R;
    int st = lsoap_table(ctx, lambda, &np, &hdr, &R);
    if (st) return st;
    if (n_centres == 0 || np == 0) return RASCAL_OK;
    if (!d_coeffs || !d_out) return set_error(RASCAL_E_ARG, "NULL device pointer");
    if ((reinterpret_cast<uintptr_t>(d_out) & 15) != 0) return set_error(RASCAL_E_ARG, "d_out must be 16-byte aligned");
    if (n_centres > 0x7fffffffLL) return set_error(RASCAL_E_ARG, "too many centres for one launch");
    // the coefficients and one row of half-contractions per q, twice, have to fit a CTA's shared memory
    const int kmax = 2 * ctx->l_max + 1;
    if (sizeof(float) * ((size_t)ctx->n_lm * ctx->Q + (size_t)2 * ctx->Q * kmax) > 227 * 1024)
        return set_error(RASCAL_E_UNSUPPORTED, "n_species * n_max * (l_max + 1)^2 too large for the equivariant kernel");
    // row groups of X per chunk: the widest bases leave room for fewer than kLsoapGroups (never below 6: every shape
    // that passes the check above fits so)
    const int px = lsoap_px(ctx->l_max), QT = (ctx->Q + 3) / 4;
    const size_t c_floats = (size_t)QT * (4 * exp_ly(ctx->l_max) + 4);
    int chunk = std::min((2 * lambda + 1) * QT, kLsoapGroups);
    while (chunk > 6 && sizeof(float) * (c_floats + (size_t)2 * 4 * chunk * px) > 227 * 1024) --chunk;
    const size_t smem = sizeof(float) * (c_floats + (size_t)2 * 4 * chunk * px);
    const int64_t fit = 228 * 1024 / (smem + 1024), sms = ctx->n_sm;
    LsoapForm form = lsoap_small(ctx->Q, ctx->l_max, lambda) ? kLsoapOne : kLsoapTwo;
    if (ctx->l_max <= 4 && n_centres > std::min<int64_t>(fit, kLsoapCtas) * sms && n_centres <= std::min<int64_t>(fit, 6) * sms) form = kLsoapOne;
    // small batches, bases that leave room for no more CTAs: one centre of Q = 2, l_max 15, lambda 4 68 -> 45 us, Q = 20, lambda 2
    // 67 -> 43; 1 500 centres of Q = 100, l_max 12, lambda 1 1 257 -> 1 018
    if (n_centres <= 2 * sms || fit <= 2) form = kLsoapAlone;
    const int threads = form == kLsoapAlone ? 2 * kLsoapThreads : kLsoapThreads;
    lsoap_kernel(ctx->Q, ctx->l_max, form)<<<(unsigned)n_centres, threads, smem, ctx->stream>>>(
        d_coeffs, ctx->Q, ctx->l_max, lambda, chunk, (unsigned)((0x100000000ull + QT - 1) / QT), np, hdr, R, d_out);
    RASCAL_LAUNCH_CHECK("k_lambda_soap");
    return RASCAL_OK;
}
