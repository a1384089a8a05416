// Sparse GPR energy model with the polynomial kernel on the tcgen05 tensor cores (TF32 operands, FP32 accumulation):
//
//   E_i = sum_{I in M, a_I = a_i} x_I k_I(p_i),   k_I(p_i) = (p^_i . M^_I)^zeta              (Eq. sparse-gp)
//   dE_i/dp_i = (G_i - zeta E_i p^_i) / |p_i|,    G_i = sum_I x_I zeta k_(zeta-1) M^_I   (Eq. gpr-force-order)
//
// with p^ = p/|p| and M^ = M/|M| when the model normalises (else p^ = p, M^ = M and |p| = 1). The active set is
// summed first, as the paper orders the force contraction: G_i is one GEMM over the active set, and G_i . p^_i =
// zeta E_i needs no second pass over the features.
//
// Both contractions are dense GEMMs between the centres of one species and that species' sparse points, so the
// centres are first bucketed by species (k_gpr_count, k_gpr_scatter: a stable counting sort on the device).
//   k_gpr_kernel: D[128 centres][128, 256 or 512 sparse points] = p_rows . M^T over the features, A rows gathered from the
//     feature matrix by cp.async (16-byte copies, zero-filled past the end), B = M^ rows (TF32-rounded at model creation).
//     Epilogue (TMEM -> registers): the row norms (accumulated from the staged A tiles), k^zeta, E partials and the
//     per-(centre, point) factor W = x zeta k^(zeta-1), stored for the gradient GEMM.
//   k_gpr_finish: per structure, E_i summed over the passes, FP64 structure energies, zeta E_i / |p_i|^2 (the
//     normalisation's share of the chain rule; 0 without normalisation).
//   k_gpr_grad: D[128 centres][256 features] = W . M^ over the active set, epilogue dE/dp = D / |p| - zeta E p / |p|^2.
// Operand tiles in shared memory are K-major with 128 bytes of K per row and stage (64 in 512-point tiles), in the 128-byte
// (64-byte) swizzled layout (8-row atoms): TMA writes it for the dense operands (the sparse points, W), the gathered feature
// rows are copied into it by cp.async.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "tcgen05.cuh"

struct rascal_gpr {
    int S;                                  // species of the context the model was built for
    int64_t F, Fk, Fn;                      // features; rounded up to 16 (K of the kernel GEMM, N of the gradient)
    int zeta, normalize;
    int n_sp[rascal::kMaxSpecies];          // sparse points per species
    int n_pad[rascal::kMaxSpecies];         // rounded up to 16
    int64_t row_off[rascal::kMaxSpecies];   // first row of a species in M and x
    int64_t t_off[rascal::kMaxSpecies];     // first element of a species' block [Fn][n_pad] in MT
    int n_pad_max;
    int64_t rows;
    float* d_M;   // [rows][Fk]   M^ rows, TF32-rounded, zero-padded
    float* d_MT;  // per species [Fn][n_pad]: M^ transposed (K-major operand of the gradient GEMM)
    float* d_x;   // [rows] x_I (0 in the padding)
    CUtensorMap tmM, tmM32;                   // TMA maps of d_M (16 and 32 columns a box) and of each species' block of d_MT
    CUtensorMap tmMT[rascal::kMaxSpecies];
};

namespace rascal {

constexpr int kGprThreads = 256;
constexpr int kGprThreads2 = kGprThreads + 64;  // gradient GEMM: eight epilogue warps, the MMAs' and the loads'
// kernel GEMM pipeline depth for tiles of 128 (16 KB per stage), 256 (24 KB) and 512 sparse points (40 KB)
constexpr int gpr_stages(int cols) { return cols == 128 ? 6 : (cols == 256 ? 4 : 5); }
constexpr int gpr_kb(int cols) { return cols == 512 ? 16 : 32; }  // K elements (TF32) per stage
constexpr int kGprStages2 = 2;              // gradient GEMM (48 KB per stage, two CTAs per SM)
constexpr int kGprFT = 256;                  // features of a tile of the gradient GEMM
constexpr int kGprB2 = kGprFT * 128;         // its B stage

struct GprArgs {
    int N, S;
    int64_t F, Fk, Fn;
    int zeta, normalize, vec16;
    const float* p;       // [N][F] features, atom order
    const int* perm;      // [N] atoms sorted by species (stable)
    const int* off;       // [S + 1] species offsets into perm
    const float* M;
    const float* MT;
    const float* x;
    int n_pad[kMaxSpecies];
    int64_t row_off[kMaxSpecies];
    int64_t t_off[kMaxSpecies];
    int n_pad_max, passes_max;
    float* e_part;        // [passes_max][N] energy partials per pass over the sparse points
    float* inv;           // [N] 1/|p_i| (1 without normalisation or for p_i = 0)
    float* W;             // [N sorted][n_pad_max] x zeta k^(zeta-1) (NULL: energies only)
    const float* c2;      // [N] zeta E_i / |p_i|^2
    float* grad;          // [N][F]
    unsigned* flags;
    uint32_t stall_polls; // test hook: > 0 makes the MMAs' first wait run out
    CUtensorMap tmM, tmM32;            // M^ rows [rows][Fk], boxes of 256 rows x 16 or 128 rows x 32 columns
    CUtensorMap tmW;                   // W [N sorted][n_pad_max]
    CUtensorMap tmMT[kMaxSpecies];     // per species M^T [Fn][n_pad]
};


__device__ inline float ipow(float k, int e) {
    float r = 1.0f;
    for (int i = 0; i < e; ++i) r *= k;
    return r;
}

// tile t -> (species, first sorted row, index within the species' tiles); false when t is past the last tile
__device__ inline bool gpr_tile(const int* s_off, int S, const int* per_mtile, int64_t t, int& s, int& row0, int& sub) {
    for (s = 0; s < S; ++s) {
        const int rows = s_off[s + 1] - s_off[s];
        const int64_t n = (int64_t)((rows + 127) / 128) * per_mtile[s];
        if (t < n) {
            row0 = s_off[s] + (int)(t / per_mtile[s]) * 128;
            sub = (int)(t % per_mtile[s]);
            return true;
        }
        t -= n;
    }
    return false;
}

// Bounded-wait failure: flag it, let the tensor core and the copies finish, and stop.
__device__ inline void gpr_fail(const GprArgs& A, uint64_t* done, uint32_t phase) {
    if (threadIdx.x == 0) atomicOr(A.flags, kFlagTimeout);
    mbar_wait_bounded(done, phase);
    cp_async_wait_all();
}

// thread 0: TMA loads still in flight after a failure (k-blocks [from, to) of this CTA) are waited for
__device__ inline void gpr_drain_tma(uint64_t* full, int stages, int64_t from, int64_t to) {
    for (int64_t i = from; i < to; ++i) mbar_wait_bounded(&full[i % stages], (uint32_t)((i / stages) & 1));
}

// stage, phase parity and whether the stage was used before of the k-block number g of a CTA, stepped without divisions
template <int STAGES>
struct GprRing {
    int stage;
    uint32_t phase;
    bool used;
    __device__ __forceinline__ explicit GprRing(int64_t g)
        : stage((int)(g % STAGES)), phase((uint32_t)((g / STAGES) & 1)), used(g >= STAGES) {}
    __device__ __forceinline__ void next() {
        if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
            used = true;
        }
    }
};

// ------------------------------------------------------------------------------------------ kernel GEMM
// Warp-specialised pipeline over the stages (empty -> copies landed -> full -> empty): warps 0-3 gather A (feature rows of the
// tile's centres) by cp.async into the swizzled layout, which arrives on `landed`; warps 4-7 take the row norms from the
// landed tile and, in turns, make it visible to the tensor core and arrive on `full`; one thread of warp 9 loads B (the
// species' sparse points) by TMA onto `full`; one of warp 8 issues the MMAs, which release the stage with the norm warps.
// Bound: the issue of the four MMAs of a k-block and the hand-overs around it (0.49 us per 32 features of a 128 x 128 tile,
// whatever the load on memory). 8 960 centres, 11 760 features, 256 points for each of 4 species: 502 us with 72 tiles of 256
// points, one thread issuing MMAs and loads, 16 features a stage; 376 with 144 tiles of 128 points; 271 with 32 features a
// stage; 181 with the loads and the norms in warps of their own (0.42 GB of features: 63 us).
constexpr int kGprProducers = 128;  // A-copy threads (warps 0-3)
constexpr int kGprThreads1 = 2 * kGprProducers + 64;

template <bool VEC16, int COLS>
__global__ void __launch_bounds__(kGprThreads1, 1) k_gpr_kernel(const __grid_constant__ GprArgs A) {
    constexpr int kKB = gpr_kb(COLS), kRow = 4 * kKB;  // features and bytes of an operand row in a stage
    constexpr int kGprStages = gpr_stages(COLS), kGprB1 = COLS * kRow, kGprATile = 128 * kRow;
    constexpr int kParts = kKB / 16;
    constexpr int kMmaWarp = 2 * kGprProducers / 32;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;                                        // [stages][128 rows of kRow bytes]
    unsigned char* sB = sA + kGprStages * kGprATile;                 // [stages][COLS rows of kRow bytes]
    float* s_x = reinterpret_cast<float*>(sB + kGprStages * kGprB1);  // [COLS]
    float* s_inv = s_x + COLS;                                       // [128]
    float* s_E = s_inv + 128;                                        // [2][128]; [4][128] norm partials before
    int* s_atom = reinterpret_cast<int*>(s_E + 512);                 // [128]
    int* s_off = s_atom + 128;                                       // [S + 1]
    int* s_per = s_off + kMaxSpecies + 1;                            // [S] passes per species
    uint64_t* bars = reinterpret_cast<uint64_t*>(s_per + kMaxSpecies + 1);  // [stages] empty, full, landed; done, dead
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + 3 * kGprStages + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint64_t* empty = bars;
    uint64_t* full = bars + kGprStages;
    uint64_t* landed = bars + 2 * kGprStages;
    uint64_t* done = bars + 3 * kGprStages;
    uint64_t* dead = done + 1;  // nothing arrives at it (test hook)

    for (int s = tid; s <= A.S; s += blockDim.x) s_off[s] = A.off[s];
    for (int s = tid; s < A.S; s += blockDim.x) s_per[s] = (A.n_pad[s] + COLS - 1) / COLS;
    if (warp == 0) {
        tmem_alloc(s_tmem, COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < kGprStages; ++i) {
            mbar_init(&empty[i], 1 + kGprProducers / 32);  // the MMAs and the norm warps
            mbar_init(&full[i], 2);                         // a norm warp and the B load
            mbar_init(&landed[i], kGprProducers);
        }
        mbar_init(done, 1);
        mbar_init(dead, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *s_tmem;
    const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
    int64_t g = 0;          // k-blocks of this CTA so far (stage = g % stages, use = g / stages)
    int64_t g_tma = 0;      // last warp: k-blocks whose B load was issued
    uint32_t done_phase = 0;
    bool ok = true;

    for (int64_t t = blockIdx.x;; t += gridDim.x) {
        int s, row0, pass;
        if (!gpr_tile(s_off, A.S, s_per, t, s, row0, pass)) break;
        const int n_rows = min(128, s_off[s + 1] - row0);
        const int col0 = pass * COLS;
        const int ncols = min(COLS, A.n_pad[s] - col0);
        const int nk = (int)((A.Fk + kKB - 1) / kKB);
        if (tid < 128) s_atom[tid] = tid < n_rows ? A.perm[row0 + tid] : -1;
        for (int c = tid; c < COLS; c += blockDim.x) s_x[c] = c < ncols ? A.x[A.row_off[s] + col0 + c] : 0.0f;
        __syncthreads();

        if (warp < kMmaWarp) {
            // ---- A rows r0 + kStep j (j < kRows), 16-byte chunks c and c + 4, by one producer and one norm thread
            constexpr int kStep = kGprProducers / 4, kRows = 128 / kStep;
            const int r0 = (tid % kGprProducers) >> 2, c = tid & 3;
            // row r0 + kStep j lands kStep kRow j bytes further, its chunk c + 4 64 bytes across
            const uint32_t d0 = kKB == 16 ? sw64_off(r0, c) : sw128_off(r0, c);
            auto at = [&](int t) { return (d0 ^ (uint32_t)(t % kParts * 64)) + kStep * kRow * (t / kParts); };
            GprRing<kGprStages> ring(g);
            if (warp < kGprProducers / 32) {
                const float* pa[kRows];
                int64_t lim[kRows];
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    const int atom = s_atom[r0 + kStep * j];
                    pa[j] = atom >= 0 ? A.p + (int64_t)atom * A.F : A.p;
                    lim[j] = atom >= 0 ? A.F : 0;
                }
                for (int kb = 0; kb < nk; ++kb, ring.next()) {
                    if (!mbar_wait_warp(ring.used, &empty[ring.stage], ring.phase ^ 1u)) {
                        ok = false;
                        break;
                    }
                    const int64_t k0 = (int64_t)kb * kKB + 4 * c;
                    unsigned char* a = sA + ring.stage * kGprATile;
#pragma unroll
                    for (int t = 0; t < kRows * kParts; ++t) {
                        const int j = t / kParts;
                        const int64_t f = k0 + t % kParts * 16;
                        unsigned char* o = a + at(t);
                        if (VEC16) {
                            const bool in = f < lim[j];
                            cp_async16_zfill(o, in ? pa[j] + f : A.p, in ? 16u : 0u);
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const bool in = f + e < lim[j];
                                cp_async4_zfill(o + 4 * e, in ? pa[j] + f + e : A.p, in ? 4u : 0u);
                            }
                        }
                    }
                    cp_async_arrive(&landed[ring.stage]);
                }
                cp_async_wait_all();
            } else {
                float nrm[kRows] = {};
                for (int kb = 0; kb < nk; ++kb, ring.next()) {
                    if (!mbar_wait_warp(true, &landed[ring.stage], ring.phase)) {
                        ok = false;
                        break;
                    }
                    // the norm warps take turns to make the tile visible to the tensor core
                    if (((g + kb) & 3) == (warp & 3)) {
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[ring.stage]);
                    }
                    const unsigned char* a = sA + ring.stage * kGprATile;
#pragma unroll
                    for (int t = 0; t < kRows * kParts; ++t) {
                        const int j = t / kParts;
                        const float4 v = *reinterpret_cast<const float4*>(a + at(t));
                        nrm[j] = fmaf(v.x, v.x, nrm[j]);
                        nrm[j] = fmaf(v.y, v.y, nrm[j]);
                        nrm[j] = fmaf(v.z, v.z, nrm[j]);
                        nrm[j] = fmaf(v.w, v.w, nrm[j]);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[ring.stage]);
                }
#pragma unroll
                for (int j = 0; j < kRows; ++j) s_E[c * 128 + r0 + kStep * j] = nrm[j];  // partials [chunk][row]
            }
        } else if (warp == kMmaWarp) {
            if (lane == 0) {  // ---- MMAs
                const int n0 = min(256, ncols), n1 = ncols - n0;
                const uint32_t id0 = instr_desc(2u, 128u, (uint32_t)n0);
                const uint32_t id1 = instr_desc(2u, 128u, (uint32_t)max(n1, 16));
                auto desc = [&](uint32_t at) { return kKB == 16 ? smem_desc_sw64(at, 512) : smem_desc_sw128(at, 1024); };
                const uint64_t da0 = desc(a_base), db0 = desc(b_base);  // the address is the descriptor's low field, in 16 bytes
                GprRing<kGprStages> use(g);
                if (A.stall_polls) ok = mbar_wait_bounded(dead, 0u, A.stall_polls);
                for (int kb = ok ? 0 : nk; kb < nk; ++kb, use.next()) {
                    if (!mbar_wait_spin(&full[use.stage], use.phase)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t da = da0 + (uint32_t)(use.stage * (kGprATile >> 4)), db = db0 + (uint32_t)(use.stage * (kGprB1 >> 4));
                    const int nkk = (int)min((int64_t)kKB, A.Fk - (int64_t)kb * kKB) / 8;
#pragma unroll
                    for (int kk = 0; kk < kKB / 8; ++kk) {
                        if (kk >= nkk) break;
                        mma_tf32_ss(taddr, da + 2 * kk, db + 2 * kk, id0, (kb | kk) != 0);
                        if (COLS > 256 && n1 > 0)
                            mma_tf32_ss(taddr + 256, da + 2 * kk, db + (256 * kRow >> 4) + 2 * kk, id1, (kb | kk) != 0);
                    }
                    mma_commit(&empty[use.stage]);
                }
                mma_commit(done);
            }
            __syncwarp();  // the other lanes wait here, not in a spin beside lane 0
        } else {
            if (lane == 0) {  // ---- B loads: a TMA issue takes as long as an MMA's, so another warp than the MMAs'
                constexpr int kBoxRows = kKB == 16 ? 256 : 128;
                const int nq = (ncols + kBoxRows - 1) / kBoxRows;
                const int brow = (int)(A.row_off[s] + col0);
                GprRing<kGprStages> ring(g);
                for (int kb = 0; kb < nk; ++kb, ring.next()) {
                    if (ring.used && !mbar_wait_spin(&empty[ring.stage], ring.phase ^ 1u)) {
                        ok = false;
                        break;
                    }
                    unsigned char* b = sB + ring.stage * kGprB1;
                    mbar_expect_tx(&full[ring.stage], (uint32_t)(nq * kBoxRows * kRow));
                    for (int qq = 0; qq < nq; ++qq)
                        tma_load_2d(b + qq * kBoxRows * kRow, kKB == 16 ? &A.tmM : &A.tmM32, kb * kKB, brow + kBoxRows * qq,
                                    &full[ring.stage]);
                    ++g_tma;
                }
            }
            __syncwarp();
        }
        g += nk;
        const bool fin = mbar_wait_bounded(done, done_phase);
        done_phase ^= 1u;
        ok = __syncthreads_and(ok && fin) != 0;
        if (!ok) {
            if (warp == kMmaWarp + 1 && lane == 0)
                gpr_drain_tma(full, kGprStages, g_tma > kGprStages ? g_tma - kGprStages : 0, g_tma);
            gpr_fail(A, done, done_phase ^ 1u);
            break;
        }
        if (tid < 128) {
            const float nn = s_E[tid] + s_E[128 + tid] + s_E[256 + tid] + s_E[384 + tid];
            const float iv = (A.normalize && nn > 0.0f) ? 1.0f / sqrtf(nn) : 1.0f;
            s_inv[tid] = iv;
            if (pass == 0 && s_atom[tid] >= 0) A.inv[s_atom[tid]] = iv;
        }
        __syncthreads();
        tc_fence_after();
        // epilogue: warp -> lane quadrant (rows) and column half
        const int q = warp & 3, h = warp >> 2, row = 32 * q + lane;
        const bool valid = row < n_rows;
        const float iv = s_inv[row];
        float e = 0.0f;
        const int c_end = min(ncols, COLS / 2 * (h + 1));
        float* wrow = A.W ? A.W + (int64_t)(row0 + row) * A.n_pad_max + col0 : nullptr;
        for (int cc = COLS / 2 * h; h < 2 && cc < c_end; cc += 16) {
            float v[16];
            tmem_ld16(taddr + ((uint32_t)(32 * q) << 16) + (uint32_t)cc, v);
            float w[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const float k = v[u] * iv;
                const float kz1 = ipow(k, A.zeta - 1);
                const float xv = s_x[cc + u];
                e = fmaf(xv * kz1, k, e);
                w[u] = xv * (float)A.zeta * kz1;
            }
            if (wrow && valid) {
#pragma unroll
                for (int u = 0; u < 16; u += 4)
                    *reinterpret_cast<float4*>(wrow + cc + u) = make_float4(w[u], w[u + 1], w[u + 2], w[u + 3]);
            }
        }
        __syncthreads();  // the norm partials in s_E are read; the energies may reuse it
        if (h < 2) s_E[h * 128 + row] = e;
        tc_fence_before();
        __syncthreads();
        if (tid < 128 && s_atom[tid] >= 0) A.e_part[(int64_t)pass * A.N + s_atom[tid]] = s_E[tid] + s_E[128 + tid];
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(taddr, COLS);
    }
}

// ---------------------------------------------------------------------------------------- gradient GEMM
// Both operands by TMA: A = W rows, B = the species' M^T rows; one thread of warp 9 loads, one of warp 8 issues the MMAs;
// warps 0-7 share the epilogue and request its first features beside the main loop.
// Bound: reading p and writing dE/dp (0.84 GB, 126 us on the model above) behind a main loop of 8 k-blocks per tile, overlapped
// only between the two CTAs of an SM: 256 us. It took 353 with a lane to a row (16-byte pieces of 32 rows per instruction) and
// six 64-row loads per k-block issued by the MMAs' thread; 333 with eight lanes to a row, 272 with 128-byte rows and the
// features requested early. Rows that are not 16-byte aligned (25 262 centres, 275 features): 189 -> 94 us with 32 lanes to a
// row. Tiles of 128 features, three CTAs per SM: 391 us (the W tile is read twice as often).
__global__ void __launch_bounds__(kGprThreads2, 2) k_gpr_grad(const __grid_constant__ GprArgs A) {
    constexpr int kKB = 32, kGprATile = 128 * 128;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;                                          // [stages][16 KB]
    unsigned char* sB = sA + kGprStages2 * kGprATile;                  // [stages][32 KB]
    int* s_atom = reinterpret_cast<int*>(sB + kGprStages2 * kGprB2);  // [128]
    float* s_inv = reinterpret_cast<float*>(s_atom + 128);             // [128] 1 / |p|
    float* s_c2 = s_inv + 128;                                         // [128] zeta E / |p|^2
    int* s_off = reinterpret_cast<int*>(s_c2 + 128);
    int* s_per = s_off + kMaxSpecies + 1;                              // feature chunks per species
    uint64_t* bars = reinterpret_cast<uint64_t*>(s_per + kMaxSpecies + 1);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + 2 * kGprStages2 + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint64_t* empty = bars;
    uint64_t* full = bars + kGprStages2;
    uint64_t* done = bars + 2 * kGprStages2;
    uint64_t* dead = done + 1;  // nothing arrives at it (test hook)
    const int n_fc = (int)((A.Fn + kGprFT - 1) / kGprFT);

    for (int s = tid; s <= A.S; s += blockDim.x) s_off[s] = A.off[s];
    for (int s = tid; s < A.S; s += blockDim.x) s_per[s] = n_fc;
    if (warp == 0) {
        tmem_alloc(s_tmem, kGprFT);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2 * kGprStages2 + 2; ++i) mbar_init(&bars[i], 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *s_tmem;
    const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
    int64_t g = 0, g_tma = 0;  // k-blocks of this CTA so far; last warp: loads issued
    uint32_t done_phase = 0;
    bool ok = true;

    for (int64_t t = blockIdx.x;; t += gridDim.x) {
        int s, row0, fc;
        if (!gpr_tile(s_off, A.S, s_per, t, s, row0, fc)) break;
        const int n_rows = min(128, s_off[s + 1] - row0);
        const int f0 = fc * kGprFT;
        const int ncols = (int)(A.Fn - f0 < kGprFT ? A.Fn - f0 : kGprFT);
        const int nk = (A.n_pad[s] + kKB - 1) / kKB;
        if (tid < 128) {
            const int atom = tid < n_rows ? A.perm[row0 + tid] : -1;
            s_atom[tid] = atom;
            s_inv[tid] = atom >= 0 && nk > 0 ? A.inv[atom] : 0.0f;
            s_c2[tid] = atom >= 0 && nk > 0 ? A.c2[atom] : 0.0f;
        }
        const int q = warp & 3, h = warp >> 2, rr = lane >> 3, cl = 4 * (lane & 7);
        const int c_end = min(ncols, kGprFT / 2 * (h + 1));
        // the features of 32 columns of this warp's rows, eight lanes to a row
        auto fetch = [&](int c, float4 (&pv)[8]) {
            const int64_t f = f0 + c + cl;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int atom = s_atom[32 * q + 4 * u + rr];
                if (c + cl < c_end && f < A.F && atom >= 0) pv[u] = __ldcs(reinterpret_cast<const float4*>(A.p + (int64_t)atom * A.F + f));
            }
        };
        float4 pn[8];
        if (warp < kGprThreads / 32) {  // requested beside the main loop
            asm volatile("bar.sync 1, %0;" ::"n"(kGprThreads) : "memory");  // s_atom
            if (A.vec16) fetch(kGprFT / 2 * h, pn);
        }
        if (nk > 0) {
            if (warp == kGprThreads / 32) {
                if (lane == 0) {  // ---- MMAs
                    const uint64_t da0 = smem_desc_sw128(a_base, 1024), db0 = smem_desc_sw128(b_base, 1024);
                    const uint32_t id = instr_desc(2u, 128u, (uint32_t)ncols);
                    GprRing<kGprStages2> use(g);
                    if (A.stall_polls) ok = mbar_wait_bounded(dead, 0u, A.stall_polls);
                    for (int kb = ok ? 0 : nk; kb < nk; ++kb, use.next()) {
                        if (!mbar_wait_spin(&full[use.stage], use.phase)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t da = da0 + (uint32_t)(use.stage * (kGprATile >> 4)), db = db0 + (uint32_t)(use.stage * (kGprB2 >> 4));
                        const int nkk = min(kKB, A.n_pad[s] - kb * kKB) / 8;  // columns of W past n_pad are not written
#pragma unroll
                        for (int kk = 0; kk < kKB / 8; ++kk)
                            if (kk < nkk) mma_tf32_ss(taddr, da + 2 * kk, db + 2 * kk, id, (kb | kk) != 0);
                        mma_commit(&empty[use.stage]);
                    }
                    mma_commit(done);
                }
                __syncwarp();
            } else if (warp > kGprThreads / 32) {
                if (lane == 0) {  // ---- loads
                    GprRing<kGprStages2> ring(g);
                    for (int kb = 0; kb < nk; ++kb, ring.next()) {
                        if (ring.used && !mbar_wait_spin(&empty[ring.stage], ring.phase ^ 1u)) {
                            ok = false;
                            break;
                        }
                        mbar_expect_tx(&full[ring.stage], (uint32_t)(kGprATile + kGprB2));
                        tma_load_2d(sA + ring.stage * kGprATile, &A.tmW, kb * kKB, row0, &full[ring.stage]);
                        tma_load_2d(sB + ring.stage * kGprB2, &A.tmMT[s], kb * kKB, f0, &full[ring.stage]);
                        ++g_tma;
                    }
                }
                __syncwarp();
            }
            g += nk;
            const bool fin = mbar_wait_bounded(done, done_phase);
            done_phase ^= 1u;
            ok = __syncthreads_and(ok && fin) != 0;
            if (!ok) {
                if (warp > kGprThreads / 32 && lane == 0)
                    gpr_drain_tma(full, kGprStages2, g_tma > kGprStages2 ? g_tma - kGprStages2 : 0, g_tma);
                gpr_fail(A, done, done_phase ^ 1u);
                break;
            }
            tc_fence_after();
        } else {
            __syncthreads();
        }
        // epilogue: dE/dp = inv * G - c2 * p for this warp's rows and half of the columns
        if (warp < kGprThreads / 32) {
            // 32 columns at a time through shared memory (the stages are free: every load has landed and every MMA is done),
            // so that eight lanes read and write 128 contiguous bytes of a row, or 32 lanes where rows are not 16-byte aligned
            float* buf = reinterpret_cast<float*>(sA) + warp * 32 * 36;  // pitch 36: both directions conflict-free
            for (int c = kGprFT / 2 * h; c < c_end; c += 32) {
                const int64_t f = f0 + c + cl;
                const bool in = c + cl < c_end && f < A.F;
                float4 pv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) pv[u] = pn[u];
                if (A.vec16 && c + 32 < c_end) fetch(c + 32, pn);
#pragma unroll
                for (int w = 0; w < 32; w += 16) {
                    if (c + w >= c_end) break;
                    float v[16];
                    if (nk > 0) {
                        tmem_ld16(taddr + ((uint32_t)(32 * q) << 16) + (uint32_t)(c + w), v);
                    } else {
#pragma unroll
                        for (int u = 0; u < 16; ++u) v[u] = 0.0f;
                    }
#pragma unroll
                    for (int u = 0; u < 16; u += 4)
                        *reinterpret_cast<float4*>(buf + lane * 36 + w + u) = make_float4(v[u], v[u + 1], v[u + 2], v[u + 3]);
                }
                __syncwarp();
                if (A.vec16) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int r = 32 * q + 4 * u + rr, atom = s_atom[r];
                        if (!in || atom < 0) continue;
                        const float iv = s_inv[r], cc = s_c2[r];
                        const float4 v = *reinterpret_cast<const float4*>(buf + (4 * u + rr) * 36 + cl);
                        __stcs(reinterpret_cast<float4*>(A.grad + (int64_t)atom * A.F + f),
                               make_float4(fmaf(iv, v.x, -cc * pv[u].x), fmaf(iv, v.y, -cc * pv[u].y),
                                           fmaf(iv, v.z, -cc * pv[u].z), fmaf(iv, v.w, -cc * pv[u].w)));
                    }
                } else if (c + lane < c_end && f0 + c + lane < A.F) {
#pragma unroll 8
                    for (int u = 0; u < 32; ++u) {
                        const int r = 32 * q + u, atom = s_atom[r];
                        if (atom < 0) continue;
                        const int64_t o = (int64_t)atom * A.F + f0 + c + lane;
                        A.grad[o] = fmaf(s_inv[r], buf[u * 36 + lane], -s_c2[r] * __ldg(A.p + o));
                    }
                }
                __syncwarp();
            }
            fence_proxy_async_smem();  // the next tile's loads come by TMA
        }
        tc_fence_before();
        __syncthreads();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(taddr, kGprFT);
    }
}

// --------------------------------------------------------------------------------------- species buckets
constexpr int kSortBlock = 1024;

__global__ void k_gpr_count(int N, int S, const int* __restrict__ species, const int* __restrict__ lut, int* cnt) {
    __shared__ int c[kMaxSpecies];
    if (threadIdx.x < S) c[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * kSortBlock + threadIdx.x;
    if (i < N) {
        const int lab = species[i];
        const int a = (lab >= 0 && lab < 256) ? lut[lab] : -1;
        if (a >= 0) atomicAdd(&c[a], 1);
    }
    __syncthreads();
    if (threadIdx.x < S) cnt[blockIdx.x * S + threadIdx.x] = c[threadIdx.x];
}

// stable scatter of the atoms into per-species buckets; block 0 also writes the species offsets
__global__ void k_gpr_scatter(int N, int S, const int* __restrict__ species, const int* __restrict__ lut,
                              const int* __restrict__ cnt, int* perm, int* off) {
    __shared__ int base[kMaxSpecies];
    __shared__ int wc[kSortBlock / 32][kMaxSpecies];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nb = gridDim.x;
    if (tid < S) {
        int before = 0, total_lower = 0;
        for (int b = 0; b < nb; ++b) {
            const int* row = cnt + b * S;
            if (b < (int)blockIdx.x) before += row[tid];
            for (int s2 = 0; s2 < tid; ++s2) total_lower += row[s2];
        }
        base[tid] = total_lower + before;
        if (blockIdx.x == 0) {
            off[tid] = total_lower;
            if (tid == S - 1) {
                int tot = 0;
                for (int b = 0; b < nb; ++b)
                    for (int s2 = 0; s2 < S; ++s2) tot += cnt[b * S + s2];
                off[S] = tot;
            }
        }
    }
    for (int s2 = lane; s2 < kMaxSpecies; s2 += 32) wc[warp][s2] = 0;
    __syncthreads();
    const int i = blockIdx.x * kSortBlock + tid;
    int a = -1;
    if (i < N) {
        const int lab = species[i];
        a = (lab >= 0 && lab < 256) ? lut[lab] : -1;
    }
    const unsigned same = __match_any_sync(0xffffffffu, a);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (a >= 0 && rank == 0) wc[warp][a] = __popc(same);
    __syncthreads();
    if (a >= 0) {
        int pos = base[a] + rank;
        for (int w = 0; w < warp; ++w) pos += wc[w][a];
        perm[pos] = i;
    }
}

// per structure: E_i over the passes, zeta E_i / |p_i|^2, and the FP64 structure sum; gridDim.y CTAs share a structure (one CTA
// took 96 us on a single structure of 25 262 atoms), whose sums k_gpr_sum adds in order: the same bits in every run
__global__ void k_gpr_finish(int N, int S, int passes_max, const int* __restrict__ struct_off,
                             const int* __restrict__ species, const int* __restrict__ lut, const int* __restrict__ npass,
                             const float* __restrict__ e_part, const float* __restrict__ inv, int zeta, int normalize,
                             float* atomic, float* c2, double* energy, double* part) {
    __shared__ double red[32];
    const int st = blockIdx.x;
    const int i0 = struct_off[st], i1 = struct_off[st + 1];
    double acc = 0.0;
    for (int i = i0 + (int)(blockIdx.y * blockDim.x + threadIdx.x); i < i1; i += gridDim.y * blockDim.x) {
        const int lab = species[i];
        const int a = (lab >= 0 && lab < 256) ? lut[lab] : -1;
        const int np = a >= 0 ? npass[a] : 0;
        float e = 0.0f;
        for (int k = 0; k < np; ++k) e += e_part[(int64_t)k * N + i];
        if (atomic) atomic[i] = e;
        if (c2) c2[i] = (np > 0 && normalize) ? (float)zeta * e * inv[i] * inv[i] : 0.0f;
        acc += (double)e;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0 && energy) {
            if (gridDim.y == 1)
                energy[st] = v;
            else
                part[(int64_t)st * gridDim.y + blockIdx.y] = v;
        }
    }
    (void)S;
    (void)passes_max;
}

__global__ void k_gpr_sum(int n_s, int n, const double* __restrict__ part, double* __restrict__ energy) {
    const int st = blockIdx.x * blockDim.x + threadIdx.x;
    if (st >= n_s) return;
    double v = 0.0;
    for (int k = 0; k < n; ++k) v += part[(int64_t)st * n + k];
    energy[st] = v;
}

static size_t gpr_smem1(int cols) {
    const int stages = gpr_stages(cols);
    return (size_t)stages * (128 + cols) * 4 * gpr_kb(cols) + sizeof(float) * (cols + 128 + 512) + sizeof(int) * 128 +
           sizeof(int) * 2 * (kMaxSpecies + 1) + sizeof(uint64_t) * (3 * stages + 2) + 16;
}
using GprKernel = void (*)(GprArgs);
static GprKernel gpr_kernel(bool vec16, int cols) {
    if (cols == 128) return vec16 ? k_gpr_kernel<true, 128> : k_gpr_kernel<false, 128>;
    if (cols == 256) return vec16 ? k_gpr_kernel<true, 256> : k_gpr_kernel<false, 256>;
    return vec16 ? k_gpr_kernel<true, 512> : k_gpr_kernel<false, 512>;
}
static size_t gpr_smem2() {
    return (size_t)kGprStages2 * (128 * 128 + kGprB2) + sizeof(int) * 3 * 128 + sizeof(int) * 2 * (kMaxSpecies + 1) +
           sizeof(uint64_t) * (2 * kGprStages2 + 2) + 16;
}

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// TMA map of a row-major FP32 matrix [rows][pitch] (cols used), in boxes of box_cols x box_rows elements:
// 16 columns with 64-byte swizzling (the operand layout of smem_desc_sw64), 32 with 128-byte swizzling (smem_desc_sw128); reads
// past the last row fill zeros
static int tmap_2d(CUtensorMap* m, const float* base, uint64_t cols, uint64_t rows, uint64_t pitch, uint32_t box_cols, uint32_t box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return set_error(RASCAL_E_CUDA, "cuTensorMapEncodeTiled is not available from the CUDA driver library");
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {pitch * sizeof(float)};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t es[2] = {1, 1};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(RASCAL_E_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return RASCAL_OK;
}

// round to the nearest TF32 value (10 explicit mantissa bits), ties to even
static float tf32_round(float v) {
    uint32_t u;
    std::memcpy(&u, &v, 4);
    if ((u & 0x7F800000u) != 0x7F800000u) {
        u += 0xFFFu + ((u >> 13) & 1u);
        u &= ~0x1FFFu;
    }
    std::memcpy(&v, &u, 4);
    return v;
}

}  // namespace rascal

using namespace rascal;

extern "C" int rascal_gpr_create(rascal_ctx* ctx, int64_t n_sparse, int64_t n_features, const double* h_sparse,
                                 const int* h_sparse_species, const double* h_weights, int zeta, int normalize,
                                 rascal_gpr** out) {
    clear_error();
    if (!ctx || !out) return set_error(RASCAL_E_ARG, "NULL context or output pointer");
    *out = nullptr;
    if (n_sparse < 0 || n_features < 1) return set_error(RASCAL_E_ARG, "n_sparse must be >= 0 and n_features >= 1");
    if (n_sparse > 0 && (!h_sparse || !h_sparse_species || !h_weights)) return set_error(RASCAL_E_ARG, "NULL host pointer");
    if (zeta < 1 || zeta > 16) return set_error(RASCAL_E_ARG, "zeta must be in [1, 16]");
    const int S = ctx->n_species;
    std::vector<std::vector<int64_t>> rows(S);
    for (int64_t I = 0; I < n_sparse; ++I) {
        int a = -1;
        for (int s = 0; s < S; ++s)
            if (ctx->species[s] == h_sparse_species[I]) a = s;
        if (a < 0) return set_error(RASCAL_E_ARG, "sparse point %lld has species %d, not one of the context's",
                                    (long long)I, h_sparse_species[I]);
        rows[a].push_back(I);
    }
    rascal_gpr* m = new rascal_gpr();
    std::memset(m, 0, sizeof(*m));
    m->S = S;
    m->F = n_features;
    m->Fk = (n_features + 15) / 16 * 16;
    m->Fn = m->Fk;
    m->zeta = zeta;
    m->normalize = normalize ? 1 : 0;
    int64_t r = 0, t = 0;
    for (int s = 0; s < S; ++s) {
        m->n_sp[s] = (int)rows[s].size();
        m->n_pad[s] = (m->n_sp[s] + 15) / 16 * 16;
        m->row_off[s] = r;
        m->t_off[s] = t;
        r += m->n_pad[s];
        t += m->Fn * m->n_pad[s];
        m->n_pad_max = std::max(m->n_pad_max, m->n_pad[s]);
    }
    m->rows = r;
    std::vector<float> hM((size_t)std::max<int64_t>(r, 1) * m->Fk, 0.0f), hMT((size_t)std::max<int64_t>(t, 1), 0.0f),
        hx((size_t)std::max<int64_t>(r, 1), 0.0f);
    for (int s = 0; s < S; ++s) {
        for (int k = 0; k < m->n_sp[s]; ++k) {
            const int64_t I = rows[s][k];
            const double* src = h_sparse + I * n_features;
            double nn = 0.0;
            for (int64_t f = 0; f < n_features; ++f) nn += src[f] * src[f];
            const double sc = (m->normalize && nn > 0.0) ? 1.0 / std::sqrt(nn) : 1.0;
            const int64_t row = m->row_off[s] + k;
            for (int64_t f = 0; f < n_features; ++f) {
                const float v = tf32_round((float)(src[f] * sc));
                hM[(size_t)(row * m->Fk + f)] = v;
                hMT[(size_t)(m->t_off[s] + f * m->n_pad[s] + k)] = v;
            }
            hx[(size_t)row] = (float)h_weights[I];
        }
    }
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = cudaMalloc(&m->d_M, sizeof(float) * hM.size());
    if (e == cudaSuccess) e = cudaMalloc(&m->d_MT, sizeof(float) * hMT.size());
    if (e == cudaSuccess) e = cudaMalloc(&m->d_x, sizeof(float) * hx.size());
    if (e == cudaSuccess) e = cudaMemcpy(m->d_M, hM.data(), sizeof(float) * hM.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->d_MT, hMT.data(), sizeof(float) * hMT.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->d_x, hx.data(), sizeof(float) * hx.size(), cudaMemcpyHostToDevice);
    for (int cols = 128; cols <= 512; cols *= 2)
        for (int v = 0; v < 2; ++v)
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(gpr_kernel(v, cols), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gpr_smem1(cols));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_gpr_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gpr_smem2());
    if (e != cudaSuccess) {
        cudaFree(m->d_M);
        cudaFree(m->d_MT);
        cudaFree(m->d_x);
        delete m;
        return set_error(RASCAL_E_CUDA, "GPR model upload: %s", cudaGetErrorString(e));
    }
    int st = RASCAL_OK;
    if (m->rows > 0) st = tmap_2d(&m->tmM, m->d_M, (uint64_t)m->Fk, (uint64_t)m->rows, (uint64_t)m->Fk, 16, 256);
    if (m->rows > 0 && !st) st = tmap_2d(&m->tmM32, m->d_M, (uint64_t)m->Fk, (uint64_t)m->rows, (uint64_t)m->Fk, 32, 128);
    for (int s = 0; s < S && !st; ++s)
        if (m->n_pad[s] > 0)
            st = tmap_2d(&m->tmMT[s], m->d_MT + m->t_off[s], (uint64_t)m->n_pad[s], (uint64_t)m->Fn, (uint64_t)m->n_pad[s], 32, kGprFT);
    if (st) {
        rascal_gpr_destroy(m);
        return st;
    }
    *out = m;
    return RASCAL_OK;
}

extern "C" void rascal_gpr_destroy(rascal_gpr* m) {
    if (!m) return;
    cudaFree(m->d_M);
    cudaFree(m->d_MT);
    cudaFree(m->d_x);
    delete m;
}

extern "C" int rascal_gpr_predict(rascal_ctx* ctx, const rascal_gpr* m, const rascal_system* sys, const float* d_features,
                                  float* d_atomic, double* d_energy, float* d_grad) {
    clear_error();
    if (!ctx || !m) return set_error(RASCAL_E_ARG, "NULL context or model");
    if (m->S != ctx->n_species) return set_error(RASCAL_E_ARG, "model built for another species list");
    int st = validate_system(ctx, sys);
    if (st) return st;
    const int N = sys->n_atoms;
    if (d_energy) RASCAL_CUDA(cudaMemsetAsync(d_energy, 0, sizeof(double) * sys->n_structures, ctx->stream));
    if (N == 0) return RASCAL_OK;
    if (!d_features) return set_error(RASCAL_E_ARG, "NULL features");
    const int S = m->S;
    const int nb = (int)div_up(N, kSortBlock);
    const bool grad = d_grad != nullptr;
    // Sparse points of a tile: as many as a species has, but fewer where that leaves SMs without a tile (8 960 centres of 4
    // species are 72 tiles of 256 points or 144 of 128). The features are not split: a product's running sum stays one chain.
    int cols = m->n_pad_max <= 128 ? 128 : (m->n_pad_max <= 256 ? 256 : 512);
    auto tiles = [&](int w) { return ((int64_t)div_up(N, 128) + S - 1) * ((m->n_pad_max + w - 1) / w); };
    while (cols > 128 && tiles(cols / 2) <= ctx->n_sm) cols /= 2;
    const int P = std::max(1, (m->n_pad_max + cols - 1) / cols);  // passes
    const dim3 finish((unsigned)sys->n_structures, (unsigned)std::max(1, std::min(64, N / sys->n_structures / 512)));
    const bool shared = d_energy && finish.y > 1;  // several CTAs to a structure
    void* base;
    st = arena_get(ctx->scratch, carve_bytes(sizeof(int) * N, sizeof(int) * nb * S, sizeof(int) * (S + 1),
                                             sizeof(int) * S, sizeof(float) * N, sizeof(float) * (size_t)P * N,
                                             sizeof(float) * N, sizeof(float) * N,
                                             grad ? sizeof(float) * (size_t)N * std::max(16, m->n_pad_max) : 16,
                                             shared ? sizeof(double) * finish.x * finish.y : 16),
                   &base);
    if (st) return st;
    Carver cv(base);
    int* perm = cv.take<int>(N);
    int* cnt = cv.take<int>((size_t)nb * S);
    int* off = cv.take<int>(S + 1);
    int* npass = cv.take<int>(S);
    float* inv = cv.take<float>(N);
    float* e_part = cv.take<float>((size_t)P * N);
    float* atomic = d_atomic ? d_atomic : cv.take<float>(N);
    if (d_atomic) cv.take<float>(N);
    float* c2 = cv.take<float>(N);
    float* W = grad ? cv.take<float>((size_t)N * std::max(16, m->n_pad_max)) : nullptr;
    double* part = shared ? cv.take<double>((size_t)finish.x * finish.y) : nullptr;

    int hp[kMaxSpecies];
    for (int s = 0; s < S; ++s) hp[s] = (m->n_pad[s] + cols - 1) / cols;
    RASCAL_CUDA(cudaMemcpyAsync(npass, hp, sizeof(int) * S, cudaMemcpyHostToDevice, ctx->stream));
    k_gpr_count<<<nb, kSortBlock, 0, ctx->stream>>>(N, S, sys->d_species, ctx->d_lut, cnt);
    RASCAL_LAUNCH_CHECK("k_gpr_count");
    k_gpr_scatter<<<nb, kSortBlock, 0, ctx->stream>>>(N, S, sys->d_species, ctx->d_lut, cnt, perm, off);
    RASCAL_LAUNCH_CHECK("k_gpr_scatter");

    GprArgs A;
    std::memset(&A, 0, sizeof(A));
    A.N = N;
    A.S = S;
    A.F = m->F;
    A.Fk = m->Fk;
    A.Fn = m->Fn;
    A.zeta = m->zeta;
    A.normalize = m->normalize;
    A.vec16 = (m->F % 4 == 0) && ((reinterpret_cast<uintptr_t>(d_features) & 15) == 0) &&
              (!grad || (reinterpret_cast<uintptr_t>(d_grad) & 15) == 0);
    A.p = d_features;
    A.perm = perm;
    A.off = off;
    A.M = m->d_M;
    A.MT = m->d_MT;
    A.x = m->d_x;
    for (int s = 0; s < S; ++s) {
        A.n_pad[s] = m->n_pad[s];
        A.row_off[s] = m->row_off[s];
        A.t_off[s] = m->t_off[s];
    }
    A.n_pad_max = std::max(16, m->n_pad_max);
    A.passes_max = P;
    A.e_part = e_part;
    A.inv = inv;
    A.W = W;
    A.c2 = c2;
    A.grad = d_grad;
    A.flags = ctx->d_flags;
    A.stall_polls = ctx->stall_polls;
    A.tmM = m->tmM;
    A.tmM32 = m->tmM32;
    for (int s = 0; s < S; ++s) A.tmMT[s] = m->tmMT[s];
    if (grad && (st = tmap_2d(&A.tmW, W, (uint64_t)A.n_pad_max, (uint64_t)N, (uint64_t)A.n_pad_max, 32, 128))) return st;
    if (m->rows > 0) {
        gpr_kernel(A.vec16, cols)<<<ctx->n_sm, kGprThreads1, gpr_smem1(cols), ctx->stream>>>(A);
        RASCAL_LAUNCH_CHECK("k_gpr_kernel");
    }
    k_gpr_finish<<<finish, 256, 0, ctx->stream>>>(N, S, P, sys->d_struct_offsets, sys->d_species, ctx->d_lut, npass, e_part, inv,
                                                  m->zeta, m->normalize, atomic, grad ? c2 : nullptr, d_energy, part);
    RASCAL_LAUNCH_CHECK("k_gpr_finish");
    if (shared) {
        k_gpr_sum<<<(unsigned)div_up(sys->n_structures, 256), 256, 0, ctx->stream>>>(sys->n_structures, (int)finish.y, part, d_energy);
        RASCAL_LAUNCH_CHECK("k_gpr_sum");
    }
    if (grad) {
        k_gpr_grad<<<2 * ctx->n_sm, kGprThreads2, gpr_smem2(), ctx->stream>>>(A);
        RASCAL_LAUNCH_CHECK("k_gpr_grad");
    }
    return RASCAL_OK;
}
