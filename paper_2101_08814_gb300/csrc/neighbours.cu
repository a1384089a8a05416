// Periodic cell-list neighbour search (Appendix B: every j, including periodic replicas, with r_ji < r_cut).
//
// Pipeline (all on the context stream; seven launches, ten from 131 073 atoms on, and one wait of the host, for the pair count):
//   k_struct_setup  a warp or four lanes per structure: inverse cell, perpendicular widths, bins >= r_cut(1+1e-6) wide per axis; the
//                   bin counters and the work list are cleared beside it
//   k_atom_bin      per atom: fractional coordinates, wrap count w, bin, wrapped position p = r - w H split into FP32
//                   hi + lo parts, counting-sort rank within the bin
//   k_bin_scan      one CTA per structure: bin starts (a structure's atoms are contiguous, so its slots start at its first
//                   atom), the list of work items (up to item_cap atoms of a bin or of a run of sparse bins), FP32
//                   classification radii
//   k_atom_scatter  bin-sorted FP32 positions (float4: x, y, z, atom index)
//   k_pairs<count>  one CTA per work item: the candidates of the bin's stencil, shifted to the bin, staged in shared
//                   memory once for all the item's centres; one warp per centre counts the accepted ones
//   k_offsets       CSR offsets, and the counts the host reads written straight to its pinned memory
//   k_pairs<fill>   same walk; accepted (j, n) keys and r_ji vectors sorted by (j, n1, n2, n3) in shared memory and
//                   written to the centre's CSR segment
//
// Bit-exactness with the FP64 definition: a candidate is classified in FP32 from the hi parts. The FP32 error of
// the displacement is bounded by 3.6e-7 (|p_i|_1 + |p_j|_1 + sum_k |t_k| |h_k|_1); with a 5x margin this gives
// delta, and only candidates with |d| within delta of r_cut (a few per million) are re-tested with the FP64
// formula d = (r_j - r_i) + ((n1 h1 + n2 h2) + n3 h3), d.d = (dx dx + dy dy) + dz dz < r_cut r_cut, each
// operation rounded on its own (__dadd_rn / __dmul_rn, no contraction). The output vector r_ji is computed in
// double-single arithmetic (error-free FP32 transforms) and rounded once to FP32.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "common.cuh"

namespace rascal {

struct StructInfo {
    double H[9];     // rows h1, h2, h3
    double Hinv[9];  // s = r Hinv (row vectors)
    float hhi[9], hlo[9];
    int nb[3], reach[3], pbc[3];
    int atom_begin, atom_end;
    float thr_lo2, thr_hi2, thr_tiny2;
    unsigned amax_bits;  // max over atoms of |p_hi|_1, as float bits
    int wmax;            // max over atoms and axes of |w|
    int64_t bin_base;    // first of its bins: 2 bins per atom and 8 more are set aside for every structure
};

constexpr int kPairWarps = 4;      // warps per block in k_pairs
constexpr int kPairCap = 128;      // pairs a warp sorts in shared memory; larger segments use global scratch
constexpr int kNoallocCap = 256;   // lists of up to as many take a second form; rascal_neighbours_noalloc has no other (no scratch)
constexpr int kPairChunk = 768;    // candidates staged at a time
constexpr int kPairEntries = 128;  // stencil bins handled at a time (one per thread)
constexpr int kPairRec = 160;      // accepted candidates a warp collects before it works out their vectors
constexpr int kPackedWrap = 511;   // largest |w| that the packed form beside atom_lo holds

__device__ inline int floordiv(int a, int b) {
    const int q = a / b;
    return (a % b != 0 && ((a < 0) != (b < 0))) ? q - 1 : q;
}
__device__ inline int pack3(int x, int y, int z) { return ((x + 512) << 20) | ((y + 512) << 10) | (z + 512); }
__device__ inline void unpack3(int c, int& x, int& y, int& z) {
    x = ((c >> 20) & 1023) - 512;
    y = ((c >> 10) & 1023) - 512;
    z = (c & 1023) - 512;
}

// `per` lanes per structure (32, or 4 where there are many), an axis (or an element of the matrices) per lane: the FP64 divisions
// and roots of the three axes run side by side (one thread per structure took 18-20 us in its serial FP64 chain; a warp per
// structure 39 us for 5 000 structures, since an FP64 instruction fills its pipe whatever its lanes do: four lanes 13 us). All
// threads clear the bin counters, thread 0 the words that the later kernels count in.
__global__ void k_struct_setup(int n_s, int n_atoms, const int* __restrict__ offs, const double* __restrict__ cells,
                               const int* __restrict__ pbc, double r_cut, StructInfo* info, int* __restrict__ bin_count,
                               int64_t nbins_cap, int* __restrict__ words, unsigned* flags, int per) {
    const int64_t gt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n_gt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = gt; e < nbins_cap; e += n_gt) bin_count[e] = 0;
    if (gt == 0) words[0] = words[1] = 0;
    const int lane = threadIdx.x & 31, sub = lane & (per - 1), k = sub % 3, first = lane - sub, group = 32 / per;
    for (int64_t w0 = (gt >> 5) * group; w0 < n_s; w0 += (n_gt >> 5) * group) {  // this warp's structures
        const int64_t s = min(w0 + lane / per, (int64_t)n_s - 1);
        const bool on = w0 + lane / per < n_s;
        StructInfo& S = info[s];
        const double* H = cells + 9 * s;
        const int a = offs[s], b = offs[s + 1];
        const bool bad_offsets = (a < 0 || b < a || b > n_atoms);
        // lane k: cr_k = h_{k+1} x h_{k+2}, the axis' own vector and lengths
        const double *h = H + 3 * k, *u = H + 3 * ((k + 1) % 3), *v = H + 3 * ((k + 2) % 3);
        const double cr[3] = {u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]};
        const double det = __shfl_sync(0xffffffffu, h[0] * cr[0] + h[1] * cr[1] + h[2] * cr[2], first);
        const double hn = norm3d(h[0], h[1], h[2]), cn = norm3d(cr[0], cr[1], cr[2]);
        const double scale = __shfl_sync(0xffffffffu, hn, first) * __shfl_sync(0xffffffffu, hn, first + 1) *
                             __shfl_sync(0xffffffffu, hn, first + 2);
        const bool bad = !(fabs(det) > 1e-12 * scale);
        const int periodic = pbc ? (pbc[3 * s + k] != 0) : 1;
        const double w = bad ? 0.0 : fabs(det) / cn, rc = r_cut * (1.0 + 1e-6);
        int nb = 1, reach = 1;
        bool thin = false;
        if (!bad && w > 0.0) {
            nb = (int)fmin(floor(w / rc), 1 << 20);
            if (nb < 1) nb = 1;
            if (periodic) {
                thin = w < r_cut / 64.0;
                reach = thin ? 1 : (int)ceil(rc * nb / w);
                if (reach < 1) reach = 1;
            }
        }
        int nbs[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) nbs[q] = __shfl_sync(0xffffffffu, nb, first + q);
        // cap the bin count at 2 N_s + 8 by halving the finest axis (bins only get wider, reach stays valid)
        const long cap = bad_offsets ? 1L : 2L * (b - a) + 8;
        while ((long)nbs[0] * nbs[1] * nbs[2] > cap) {
            int kk = 0;
            if (nbs[1] > nbs[kk]) kk = 1;
            if (nbs[2] > nbs[kk]) kk = 2;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (q == kk) nbs[q] = nbs[q] / 2 > 0 ? nbs[q] / 2 : 1;
        }
        for (int e0 = 0; e0 < 9; e0 += per) {  // Hinv[3 i + k] = cr_k[i] / det
            const int e = e0 + sub;
            const double c0 = __shfl_sync(0xffffffffu, cr[0], first + e % 3), c1 = __shfl_sync(0xffffffffu, cr[1], first + e % 3),
                         c2 = __shfl_sync(0xffffffffu, cr[2], first + e % 3);
            if (on && e < 9) {
                const double g = H[e];
                S.H[e] = g;
                S.hhi[e] = (float)g;
                S.hlo[e] = (float)(g - (double)(float)g);
                S.Hinv[e] = bad ? 0.0 : (e < 3 ? c0 : (e < 6 ? c1 : c2)) / det;
            }
        }
        if (on && sub < 3) {
            S.nb[k] = k == 0 ? nbs[0] : (k == 1 ? nbs[1] : nbs[2]);
            S.reach[k] = reach;
            S.pbc[k] = periodic;
            if (thin) atomicOr(flags, kFlagThinCell);
        }
        if (on && sub == 0) {
            // atoms before the first or past the last offset count as the first or last structure's (find_structure)
            const int begin = s == 0 ? 0 : a, end = s == n_s - 1 ? n_atoms : b;
            S.atom_begin = begin;
            S.atom_end = end;
            S.bin_base = 2 * (int64_t)begin + 8 * s;
            S.amax_bits = 0u;
            S.wmax = 0;
            if (bad_offsets) atomicOr(flags, kFlagBadOffsets);
            if (bad) atomicOr(flags, kFlagGeometry);
        }
    }
}

__device__ inline int find_structure(const int* __restrict__ offs, int n_s, int i) {
    int lo = 0, hi = n_s;  // last s with offs[s] <= i
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (offs[mid] <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Bound: latency (few FP64 operations per atom). A structure's largest |p|_1 and |w| are found per warp first: one
// atomicMax per atom on one address took 27 us for a cell of 32 768 atoms.
__global__ void k_atom_bin(int n_atoms, int n_s, int64_t nbins_cap, const int* __restrict__ offs, const double* __restrict__ pos,
                           const int* __restrict__ species, const int* __restrict__ lut, StructInfo* info,
                           int* __restrict__ bin_count, int* __restrict__ atom_bin, int* __restrict__ atom_rank,
                           int4* __restrict__ atom_wrap, float4* __restrict__ atom_hi, float4* __restrict__ atom_lo,
                           unsigned* flags) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = i < n_atoms;
    const int s = find_structure(offs, n_s, on ? i : n_atoms - 1);
    StructInfo& S = info[s];
    unsigned abits = 0u;
    int wmax = 0;
    if (on) {
        const double r[3] = {pos[3 * (int64_t)i], pos[3 * (int64_t)i + 1], pos[3 * (int64_t)i + 2]};
        // a non-finite position is reported; the clamps below keep its bin and wrap count in range, and its FP32
        // thresholds become NaN, so no pair of its structure is accepted before the call returns the error
        if (!(isfinite(r[0]) && isfinite(r[1]) && isfinite(r[2]))) atomicOr(flags, kFlagNonFinite);
        const int lab = species[i];
        if (!(lab >= 0 && lab < 256) || lut[lab] < 0) atomicOr(flags, kFlagSpecies);
        int w[3], bc[3];
        for (int k = 0; k < 3; ++k) {
            const double sk = r[0] * S.Hinv[k] + r[1] * S.Hinv[3 + k] + r[2] * S.Hinv[6 + k];
            double f = sk;
            w[k] = 0;
            if (S.pbc[k]) {
                const double fl = floor(sk);
                w[k] = (int)fmax(fmin(fl, 1e9), -1e9);
                f = sk - fl;
            }
            double x = floor(f * S.nb[k]);
            x = fmin(fmax(x, 0.0), (double)(S.nb[k] - 1));
            bc[k] = (int)x;
            wmax = max(wmax, abs(w[k]));
        }
        double p[3];
        for (int c = 0; c < 3; ++c)
            p[c] = r[c] - (w[0] * S.H[c] + w[1] * S.H[3 + c] + w[2] * S.H[6 + c]);
        float hi[3], lo[3];
        for (int c = 0; c < 3; ++c) {
            hi[c] = (float)p[c];
            lo[c] = (float)(p[c] - (double)hi[c]);
        }
        const float A = fabsf(hi[0]) + fabsf(hi[1]) + fabsf(hi[2]);
        abits = __float_as_uint(A);
        const int64_t gb64 = S.bin_base + (bc[0] * S.nb[1] + bc[1]) * S.nb[2] + bc[2];
        if (gb64 < 0 || gb64 >= nbins_cap) {  // only reachable with inconsistent structure offsets
            atomicOr(flags, kFlagBadOffsets);
            atom_bin[i] = -1;
            atom_rank[i] = 0;
        } else {
            atom_bin[i] = (int)gb64;
            atom_rank[i] = atomicAdd(&bin_count[gb64], 1);
        }
        const bool packs = max(abs(w[0]), max(abs(w[1]), abs(w[2]))) <= kPackedWrap;
        atom_wrap[i] = make_int4(w[0], w[1], w[2], 0);
        atom_hi[i] = make_float4(hi[0], hi[1], hi[2], A);
        atom_lo[i] = make_float4(lo[0], lo[1], lo[2], __int_as_float(packs ? pack3(w[0], w[1], w[2]) : 0));
    }
    const int s0 = __shfl_sync(0xffffffffu, s, 0);
    if (__all_sync(0xffffffffu, s == s0)) {
        abits = __reduce_max_sync(0xffffffffu, abits);
        wmax = __reduce_max_sync(0xffffffffu, wmax);
        if ((threadIdx.x & 31) != 0) return;
    }
    if (abits) atomicMax(&S.amax_bits, abits);
    if (wmax) atomicMax(&S.wmax, wmax);
}

// One CTA per structure: slots of its bins (atom_begin + exclusive prefix of the bin counts), the classification radii, and the
// work items {structure, first bin, first slot, atoms | bins << 8}. An item is a run of bins along the third axis (whose atoms
// are neighbours in slot order) or, where a run has more than item_cap atoms, an equal part of it. Bins of six atoms and more are
// runs of their own; sparser ones (their occupied bins' mean) are joined to about item_cap atoms, as far as the run's stencil
// fits one table. An item per bin left a CTA to the latencies of an item where bins hold an atom or two (whole search): 150 000
// atoms in bins of 0.8 1 367 -> 458 us, 5 000 structures of 20 atoms in vacuum 459 -> 320; the list made from the finished bin
// starts costs a search of few bins 1 us.
constexpr int kBinsPerThread = 8;
__global__ void __launch_bounds__(1024) k_bin_scan(int n_s, int n_atoms, double r_cut, int item_cap, StructInfo* info,
                                                   const int* __restrict__ bin_count, int* __restrict__ bin_start,
                                                   int4* __restrict__ items, int* __restrict__ words,
                                                   const unsigned* __restrict__ flags) {
    __shared__ int warp_tot[32], s_total, s_occupied;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    if (*flags & kFlagBadOffsets) return;  // the bins may be inconsistent: no item, so no later kernel touches an atom
    for (int s = blockIdx.x; s < n_s; s += gridDim.x) {
        StructInfo& S = info[s];
        if (tid == 0) {
            s_occupied = 0;
            const double amax = (double)__uint_as_float(S.amax_bits);
            double tmax = 0.0;
            for (int k = 0; k < 3; ++k) {
                const double hk = fabs((double)S.hhi[3 * k]) + fabs((double)S.hhi[3 * k + 1]) + fabs((double)S.hhi[3 * k + 2]);
                tmax += (S.reach[k] + 1) * hk;
            }
            const double delta = 2e-6 * (2.0 * amax + tmax) + 1e-6 * r_cut;
            const double lo = fmax(r_cut - delta, 0.0), hi = r_cut + delta;
            S.thr_lo2 = (float)(lo * lo);
            S.thr_hi2 = (float)(hi * hi);
            const double tiny = 1e-3 + delta;
            S.thr_tiny2 = (float)(tiny * tiny);
        }
        const int nb2 = S.nb[2], rows = S.nb[0] * S.nb[1], nbins = rows * nb2;
        const int64_t base = S.bin_base;
        int start = S.atom_begin, occupied = 0;
        for (int b0 = 0; b0 < nbins; b0 += kBinsPerThread * blockDim.x) {
            const int b = b0 + kBinsPerThread * tid;
            int n[kBinsPerThread], own = 0;
#pragma unroll
            for (int q = 0; q < kBinsPerThread; ++q) {
                n[q] = b + q < nbins ? bin_count[base + b + q] : 0;
                own += n[q];
                occupied += n[q] > 0;
            }
            int x = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) warp_tot[warp] = x;
            __syncthreads();
            if (warp == 0) {
                int w = lane < nwarps ? warp_tot[lane] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, w, o);
                    if (lane >= o) w += y;
                }
                warp_tot[lane] = w;
                if (lane == 31) s_total = w;
            }
            __syncthreads();
            int slot = start + (warp ? warp_tot[warp - 1] : 0) + x - own;
#pragma unroll
            for (int q = 0; q < kBinsPerThread; ++q) {
                if (b + q < nbins) bin_start[base + b + q] = slot;
                slot += n[q];
            }
            start += s_total;
            __syncthreads();
        }
        occupied = __reduce_add_sync(0xffffffffu, occupied);
        if (lane == 0 && occupied) atomicAdd(&s_occupied, occupied);
        __syncthreads();  // with it the slots above
        const int n_in = start - S.atom_begin, occ = max(s_occupied, 1);
        const int around = (2 * S.reach[0] + 1) * (2 * S.reach[1] + 1);
        int run = 1;
        if (n_in < 6 * occ) run = (int)min((int64_t)item_cap * occ / max(n_in, 1), (int64_t)min(64, nb2));
        run = max(1, min(run, kPairEntries / around - 2 * S.reach[2]));
        const int per_row = (nb2 + run - 1) / run, n_runs = rows * per_row;
        for (int r0 = 0; r0 < n_runs; r0 += blockDim.x) {
            const int r = r0 + tid, row = r / per_row, z = (r - row * per_row) * run, len = min(run, nb2 - z);
            int first = 0, cnt = 0;
            const int bin = row * nb2 + z;
            if (r < n_runs) {
                first = bin_start[base + bin];
                cnt = bin_start[base + bin + len - 1] + bin_count[base + bin + len - 1] - first;
            }
            const int ni = (cnt + item_cap - 1) / item_cap;
            int x = ni;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            int pos = 0;
            if (lane == 31 && x) pos = atomicAdd(words, x);
            pos = __shfl_sync(0xffffffffu, pos, 31) + x - ni;
            for (int k = 0; k < ni; ++k, ++pos) {
                const int lo = (int)((int64_t)cnt * k / ni), hi = (int)((int64_t)cnt * (k + 1) / ni);
                if (pos < n_atoms) items[pos] = make_int4(s, bin, first + lo, (hi - lo) | len << 8);
            }
        }
        __syncthreads();  // s_occupied
    }
}

__global__ void k_atom_scatter(int n_atoms, const int* __restrict__ atom_bin, const int* __restrict__ atom_rank,
                               const int* __restrict__ bin_start, const float4* __restrict__ atom_hi,
                               float4* __restrict__ sorted_hi, const unsigned* __restrict__ flags) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_atoms || atom_bin[i] < 0 || (*flags & kFlagBadOffsets)) return;
    const int slot = bin_start[atom_bin[i]] + atom_rank[i];
    const float4 h = atom_hi[i];
    sorted_hi[slot] = make_float4(h.x, h.y, h.z, __int_as_float(i));
}

__device__ inline void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ inline void two_prod(float a, float b, float& p, float& e) {
    p = a * b;
    e = fmaf(a, b, -p);
}

// exact FP64 inclusion test and squared distance, same operation order as the definition
__device__ inline double exact_d2(const double* __restrict__ pos, int i, int j, const double* H, const int n[3]) {
    double d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double rel = __dsub_rn(pos[3 * (int64_t)j + c], pos[3 * (int64_t)i + c]);
        const double sv = __dadd_rn(__dadd_rn(__dmul_rn((double)n[0], H[c]), __dmul_rn((double)n[1], H[3 + c])),
                                    __dmul_rn((double)n[2], H[6 + c]));
        d[c] = __dadd_rn(rel, sv);
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

__device__ inline uint64_t pair_key(int j, const int n[3]) {
    return ((uint64_t)(uint32_t)j << 30) | ((uint64_t)(n[0] + 512) << 20) | ((uint64_t)(n[1] + 512) << 10) |
           (uint64_t)(n[2] + 512);
}

struct PairArgs {
    int n_atoms;
    const double* pos;
    const StructInfo* info;
    const int* bin_count;
    const int* bin_start;
    const float4* sorted_hi;
    const int4* atom_wrap;
    const float4* atom_lo;
    const int4* items;
    int* words;              // [0] number of work items, [1] largest count of a centre, [3] the search whose fill may run
    int search;              // fill launched before the host has seen the counts: runs only where words[3] names it; else 0
    double rc2;
    int* counts;             // count: pairs per centre
    const int64_t* offsets;  // fill
    int* out_j;
    int* out_shift;
    float4* out_rij;
    uint64_t* ovf_keys;
    float4* ovf_vec;
    unsigned* flags;
};

// One CTA per work item (persistent: CTAs stride over the list). All centres of an item share their bin's stencil: its
// candidates are staged once, already shifted to the bin's image (x + T), so that a warp's test of 32 candidates for one
// centre is a 16-byte shared load, six FP32 operations and a ballot. (One warp per centre that walked the stencil itself
// spent about 1 400 warp instructions per centre on locating and loading candidates, twice, and waited for them in L2:
// 124 us counting and 206 us filling 1.80 M pairs of 70 820 centres; now 66 and 170 us.) Items of more than
// kPairChunk candidates, or whose stencil has more than kPairEntries bins, restage chunk by chunk for every four centres.
// CAP: pairs a warp sorts in shared memory.
template <bool FILL, int CAP = kPairCap>
__global__ void __launch_bounds__(kPairWarps * 32, CAP <= 128 ? (FILL ? 6 : 8) : 0) k_pairs(const PairArgs A) {
    constexpr int kThreads = kPairWarps * 32;
    __shared__ float4 s_c[kPairChunk];             // x + T, y + T, z + T, j (t = 0) or ~j (another image)
    __shared__ unsigned char s_e[kPairChunk];      // the candidate's stencil entry
    __shared__ int s_pref[kPairEntries], s_beg[kPairEntries], s_t[kPairEntries];
    __shared__ float4 s_T[kPairEntries];
    __shared__ float4 s_Th[FILL ? kPairEntries : 1], s_Tl[FILL ? kPairEntries : 1];
    __shared__ int s_wtot[kPairWarps];
    __shared__ __align__(16) uint64_t s_keys[FILL ? kPairWarps * CAP : 1];
    __shared__ float4 s_vec[FILL ? kPairWarps * CAP : 1];
    __shared__ unsigned short s_rec[FILL ? kPairWarps * kPairRec : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (FILL && A.search && A.words[3] != A.search) return;
    const int n_work = min(A.words[0], A.n_atoms);
    unsigned local_flags = 0;
    int local_max = 0;
    for (int work = blockIdx.x; work < n_work; work += gridDim.x) {
        const int4 item = A.items[work];
        const StructInfo& S = A.info[item.x];
        const int nb0 = S.nb[0], nb1 = S.nb[1], nb2 = S.nb[2], r0 = S.reach[0], r1 = S.reach[1], r2 = S.reach[2];
        const int centres = item.w & 255, w1 = 2 * r1 + 1, w2 = 2 * r2 + (item.w >> 8), n_st = (2 * r0 + 1) * w1 * w2;
        const int bz = item.y % nb2, by = (item.y / nb2) % nb1, bx = item.y / (nb2 * nb1);
        const float thr_lo2 = S.thr_lo2, thr_hi2 = S.thr_hi2, thr_tiny2 = S.thr_tiny2;
        const bool packed = S.wmax <= kPackedWrap;
        // |n| <= 2 wmax + |t|: only where this can pass the key's range is a pair's shift checked
        const int tmax = max((r0 + nb0 - 1) / nb0, max((r1 + nb1 - 1) / nb1, (r2 + nb2 - 1) / nb2)) + 1;
        const bool wide = S.wmax > kMaxShift || 2 * S.wmax + tmax > kMaxShift;
        // keys of 32 bits, 20 of the atom's number in the structure and 4 per shift, where every shift fits them: two
        // instructions per comparison of the rank sort and four keys per load (fill
        // pass 196 -> 170 us for 1.80 M pairs, 188 -> 168 us for the 2.95 M of a dense liquid)
        const bool narrow = S.atom_end - S.atom_begin <= (1 << 20) && S.wmax <= kMaxShift && 2 * S.wmax + tmax <= 7;
        int staged = -1;  // first entry of the batch whose tables are in shared memory, if its candidates fill one chunk
        int n_staged = 0;
        // wrap counts of atom j
        auto wrap_of = [&](int j, int& x, int& y, int& z) {
            const int4 w = A.atom_wrap[j];
            x = w.x;
            y = w.y;
            z = w.z;
        };
        const int rounds = (centres + kPairWarps - 1) / kPairWarps;
        for (int round = 0; round < rounds; ++round) {
            const int cidx = round * kPairWarps + warp;
            const bool mine = cidx < centres;  // warp-uniform
            const float4 phi = A.sorted_hi[item.z + (mine ? cidx : 0)];
            const int i = __float_as_int(phi.w);
            float4 plo = make_float4(0.f, 0.f, 0.f, 0.f);
            int64_t seg_beg = 0, seg_cnt = 0;
            uint64_t* keys = s_keys + (FILL ? warp * CAP : 0);
            uint32_t* keys32 = reinterpret_cast<uint32_t*>(keys);  // narrow, at most CAP pairs
            float4* vecs = s_vec + (FILL ? warp * CAP : 0);
            if (FILL) {
                plo = A.atom_lo[i];
                seg_beg = A.offsets[i];
                seg_cnt = A.offsets[i + 1] - seg_beg;
                if (seg_cnt > CAP) {
                    keys = A.ovf_keys + seg_beg;
                    vecs = A.ovf_vec + seg_beg;
                }
            }
            int wix, wiy, wiz;
            if (packed && FILL) unpack3(__float_as_int(plo.w), wix, wiy, wiz);
            else wrap_of(i, wix, wiy, wiz);
            int count = 0;  // accepted so far
            int done = 0;   // of those, with vectors worked out (fill)
            for (int e0 = 0; e0 < n_st; e0 += kPairEntries) {
                int total = n_staged;
                if (staged != e0) {
                    // tables of up to kPairEntries stencil bins, one per thread: candidates, first slot, image shift
                    __syncthreads();
                    const int e = e0 + tid;
                    int cnt = 0;
                    if (e < n_st) {
                        const int ex = e / (w1 * w2), er = e - ex * w1 * w2, ey = er / w2;
                        const int xs[3] = {bx + ex - r0, by + ey - r1, bz + (er - ey * w2) - r2}, nbs[3] = {nb0, nb1, nb2};
                        int tb[3], t[3];
                        bool valid = true;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            tb[k] = xs[k];
                            t[k] = 0;
                            if (S.pbc[k]) {
                                if (xs[k] < 0 || xs[k] >= nbs[k]) {
                                    t[k] = floordiv(xs[k], nbs[k]);
                                    tb[k] = xs[k] - t[k] * nbs[k];
                                }
                            } else if (xs[k] < 0 || xs[k] >= nbs[k]) {
                                valid = false;
                            }
                        }
                        if (valid) {
                            const int64_t bin = S.bin_base + (tb[0] * nb1 + tb[1]) * nb2 + tb[2];
                            s_beg[tid] = A.bin_start[bin];
                            cnt = A.bin_count[bin];
                            s_t[tid] = pack3(t[0], t[1], t[2]);
                            float Tf[3];
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                // explicit roundings: the count and fill passes must take identical decisions
                                Tf[c] = __fadd_rn(__fadd_rn(__fmul_rn((float)t[0], S.hhi[c]), __fmul_rn((float)t[1], S.hhi[3 + c])),
                                                  __fmul_rn((float)t[2], S.hhi[6 + c]));
                            }
                            s_T[tid] = make_float4(Tf[0], Tf[1], Tf[2], (t[0] | t[1] | t[2]) == 0 ? 1.0f : 0.0f);
                            if (FILL) {
                                float Th[3], Tl[3];
#pragma unroll
                                for (int c = 0; c < 3; ++c) {
                                    float sh = 0.0f, sl = 0.0f;
#pragma unroll
                                    for (int k = 0; k < 3; ++k) {
                                        float pp, pe, s2, e2;
                                        two_prod((float)t[k], S.hhi[3 * k + c], pp, pe);
                                        pe += (float)t[k] * S.hlo[3 * k + c];
                                        two_sum(sh, pp, s2, e2);
                                        sh = s2;
                                        sl += pe + e2;
                                    }
                                    Th[c] = sh;
                                    Tl[c] = sl;
                                }
                                s_Th[FILL ? tid : 0] = make_float4(Th[0], Th[1], Th[2], 0.0f);
                                s_Tl[FILL ? tid : 0] = make_float4(Tl[0], Tl[1], Tl[2], 0.0f);
                            }
                        }
                    }
                    int incl = cnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    if (lane == 31) s_wtot[warp] = incl;
                    __syncthreads();
                    total = 0;
#pragma unroll
                    for (int w = 0; w < kPairWarps; ++w) {
                        if (w < warp) incl += s_wtot[w];
                        total += s_wtot[w];
                    }
                    s_pref[tid] = incl;
                    __syncthreads();
                }
                for (int c0 = 0; c0 < total; c0 += kPairChunk) {
                    const int nc = min(kPairChunk, total - c0);
                    if (staged != e0) {
                        if (c0 > 0) __syncthreads();  // the previous chunk is done with
                        for (int c = tid; c < nc; c += kThreads) {
                            // entry of this candidate: the number of entries whose inclusive prefix is <= its index
                            int k = 0;
#pragma unroll
                            for (int st = kPairEntries / 2; st >= 1; st >>= 1)
                                if (s_pref[k + st - 1] <= c0 + c) k += st;
                            const int first = k ? s_pref[k - 1] : 0;
                            const float4 q = A.sorted_hi[s_beg[k] + (c0 + c - first)];
                            const float4 T = s_T[k];
                            const int j = __float_as_int(q.w);
                            s_c[c] = make_float4(__fadd_rn(q.x, T.x), __fadd_rn(q.y, T.y), __fadd_rn(q.z, T.z),
                                                 __int_as_float(T.w != 0.0f ? j : ~j));
                            s_e[c] = (unsigned char)k;
                        }
                        __syncthreads();
                    }
                    if (mine) {
                        // vectors and keys of the collected candidates [done, count)
                        auto flush = [&]() {
                            __syncwarp();
                            for (int r = done + lane; r < count; r += 32) {
                                const int c = s_rec[FILL ? warp * kPairRec + (r - done) : 0], k = s_e[c];
                                const int w = __float_as_int(s_c[c].w), j = w < 0 ? ~w : w;
                                const float4 q = A.sorted_hi[s_beg[k] + (c0 + c - (k ? s_pref[k - 1] : 0))];
                                const float4 qlo = A.atom_lo[j];
                                int t[3], wj[3];
                                unpack3(s_t[k], t[0], t[1], t[2]);
                                if (packed) unpack3(__float_as_int(qlo.w), wj[0], wj[1], wj[2]);
                                else wrap_of(j, wj[0], wj[1], wj[2]);
                                const int n[3] = {min(max(t[0] - wj[0] + wix, -kMaxShift), kMaxShift),
                                                  min(max(t[1] - wj[1] + wiy, -kMaxShift), kMaxShift),
                                                  min(max(t[2] - wj[2] + wiz, -kMaxShift), kMaxShift)};
                                const float4 Th4 = s_Th[FILL ? k : 0], Tl4 = s_Tl[FILL ? k : 0];
                                const float Th[3] = {Th4.x, Th4.y, Th4.z}, Tl[3] = {Tl4.x, Tl4.y, Tl4.z};
                                const float pj[3] = {q.x, q.y, q.z}, pjl[3] = {qlo.x, qlo.y, qlo.z};
                                const float pi_[3] = {phi.x, phi.y, phi.z}, pil[3] = {plo.x, plo.y, plo.z};
                                float v[3];
#pragma unroll
                                for (int cc = 0; cc < 3; ++cc) {
                                    float s1, e1, s2, e2;
                                    two_sum(pj[cc], Th[cc], s1, e1);
                                    e1 += pjl[cc] + Tl[cc];
                                    two_sum(s1, -pi_[cc], s2, e2);
                                    e2 += e1 - pil[cc];
                                    v[cc] = s2 + e2;
                                }
                                const float rr = sqrtf(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
                                if (r < seg_cnt) {
                                    if (narrow && seg_cnt <= CAP)
                                        keys32[r] = (uint32_t)(j - S.atom_begin) << 12 | (uint32_t)((n[0] + 8) << 8 | (n[1] + 8) << 4 | (n[2] + 8));
                                    else
                                        keys[r] = pair_key(j, n);
                                    vecs[r] = make_float4(v[0], v[1], v[2], rr);
                                }
                            }
                            __syncwarp();
                            done = count;
                        };
#pragma unroll 2
                        for (int base = 0; base < nc; base += 32) {
                            const float4 c = s_c[min(base + lane, kPairChunk - 1)];
                            const float dx = __fsub_rn(c.x, phi.x), dy = __fsub_rn(c.y, phi.y), dz = __fsub_rn(c.z, phi.z);
                            const float dsq = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
                            const int w = __float_as_int(c.w);
                            const bool on = base + lane < nc && w != i;
                            bool accept = on && dsq < thr_lo2;
                            if (__any_sync(0xffffffffu, on && dsq <= thr_hi2 && (!accept || dsq < thr_tiny2 || wide))) {
                                const int j = w < 0 ? ~w : w;
                                if (on && dsq <= thr_hi2) {
                                    int wjx, wjy, wjz, tx, ty, tz;
                                    wrap_of(j, wjx, wjy, wjz);
                                    int vx, vy, vz;
                                    wrap_of(i, vx, vy, vz);
                                    unpack3(s_t[s_e[base + lane]], tx, ty, tz);
                                    const int n[3] = {tx - wjx + vx, ty - wjy + vy, tz - wjz + vz};
                                    if (!accept) accept = exact_d2(A.pos, i, j, S.H, n) < A.rc2;
                                    if (accept && dsq < thr_tiny2 && exact_d2(A.pos, i, j, S.H, n) < 1e-12)
                                        local_flags |= kFlagGeometry;
                                    if (accept && (n[0] < -kMaxShift || n[0] > kMaxShift || n[1] < -kMaxShift ||
                                                   n[1] > kMaxShift || n[2] < -kMaxShift || n[2] > kMaxShift))
                                        local_flags |= kFlagShiftRange;
                                }
                            }
                            const unsigned m = __ballot_sync(0xffffffffu, accept);
                            if (FILL) {
                                if (accept)
                                    s_rec[FILL ? warp * kPairRec + (count - done) + __popc(m & ((1u << lane) - 1u)) : 0] =
                                        (unsigned short)(base + lane);
                                count += __popc(m);
                                if (count - done > kPairRec - 32) flush();
                            } else {
                                count += __popc(m);
                            }
                        }
                        if (FILL) flush();  // the records point into this chunk
                    }
                }
                if (staged != e0) {
                    // the whole stencil fits one batch and one chunk: the item's other centres find it staged
                    const bool keep = n_st <= kPairEntries && total <= kPairChunk;
                    staged = keep ? e0 : -1;
                    n_staged = total;
                }
            }
            if (!mine) continue;
            if (!FILL) {
                if (lane == 0) A.counts[i] = count;
                local_max = max(local_max, count);
                continue;
            }
            // rank sort of the segment by (j, n1, n2, n3) and write-out
            __syncwarp();
            const int k = (int)(seg_cnt < (int64_t)count ? seg_cnt : (int64_t)count);
            auto write = [&](int e, int j, int n0, int n1, int n2, int rank) {
                const int64_t o = seg_beg + rank;
                A.out_j[o] = j;
                A.out_shift[3 * o + 0] = n0;
                A.out_shift[3 * o + 1] = n1;
                A.out_shift[3 * o + 2] = n2;
                A.out_rij[o] = vecs[e];
            };
            auto write64 = [&](int e, uint64_t key, int rank) {
                write(e, (int)(key >> 30), (int)((key >> 20) & 1023) - 512, (int)((key >> 10) & 1023) - 512,
                      (int)(key & 1023) - 512, rank);
            };
            if (narrow && seg_cnt <= CAP) {
                if (lane < ((k + 3) & ~3) - k) keys32[k + lane] = 0xffffffffu;
                __syncwarp();
                for (int e0 = 0; e0 < k; e0 += 64) {  // two keys per lane at a time, every key against them
                    const int ea = e0 + lane, eb = ea + 32;
                    const uint32_t ka = ea < k ? keys32[ea] : 0u, kb = eb < k ? keys32[eb] : 0u;
                    int ra = 0, rb = 0;
#pragma unroll 2
                    for (int f = 0; f < k; f += 4) {
                        const uint4 q = *reinterpret_cast<const uint4*>(keys32 + f);
                        ra += (q.x < ka) + (q.y < ka) + (q.z < ka) + (q.w < ka);
                        rb += (q.x < kb) + (q.y < kb) + (q.z < kb) + (q.w < kb);
                    }
                    auto put = [&](int e, uint32_t key, int rank) {
                        write(e, (int)(key >> 12) + S.atom_begin, (int)((key >> 8) & 15) - 8, (int)((key >> 4) & 15) - 8,
                              (int)(key & 15) - 8, rank);
                    };
                    if (ea < k) put(ea, ka, ra);
                    if (eb < k) put(eb, kb, rb);
                }
            } else if (seg_cnt <= CAP) {
                for (int e = lane; e < k; e += 32) {
                    const uint64_t key = keys[e];
                    int rank = 0;
                    for (int f = 0; f < k; ++f) rank += (keys[f] < key);
                    write64(e, key, rank);
                }
            } else {
                __threadfence_block();
                for (int e = lane; e < k; e += 32) {
                    const uint64_t key = keys[e];
                    int rank = 0;
                    for (int f = 0; f < k; ++f) rank += (keys[f] < key);
                    write64(e, key, rank);
                }
            }
            __syncwarp();
        }
        __syncthreads();  // the next item's tables overwrite this one's
    }
    if (local_flags) atomicOr(A.flags, local_flags);
    if (!FILL && lane == 0 && local_max > 0) atomicMax(A.words + 1, local_max);
}

// CSR offsets of up to kOffsetsMax centres in one launch: every CTA sums the counts before its tile itself (at most
// 512 KB from L2) and scans its tile; the last one, which has seen them all, also reports the total, the largest count
// and the error flags to the host's pinned words. Three launches (scan.cu) and k_report serve larger systems.
constexpr int kOffsetsThreads = 1024;
constexpr int kOffsetsMax = 131072;
// h_words: pairs, largest count of a centre. words[3]: the search's number if a fill pass with these limits fits it.
struct Report {
    int* words;
    const unsigned* flags;
    int64_t* h_words;
    unsigned* h_flags;
    int64_t capacity;
    int largest, search;
    __device__ void operator()(int64_t total) const {
        words[3] = *flags == 0 && total <= capacity && words[1] <= largest ? search : 0;
        h_words[0] = total;
        h_words[1] = words[1];
        *h_flags = *flags;
    }
};
__global__ void __launch_bounds__(kOffsetsThreads) k_offsets(int n, const int* __restrict__ counts, int64_t* __restrict__ offsets,
                                                             const Report report) {
    __shared__ int64_t tot[kOffsetsThreads / 32], pre[kOffsetsThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, base = blockIdx.x * kOffsetsThreads;
    int64_t p = 0;
#pragma unroll 4
    for (int e = tid; e < base; e += kOffsetsThreads) p += counts[e];
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    const int64_t own = base + tid < n ? counts[base + tid] : 0;
    int64_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 0) pre[warp] = p;
    if (lane == 31) tot[warp] = x;
    __syncthreads();
    int64_t before = x - own;
    for (int w = 0; w < kOffsetsThreads / 32; ++w) before += pre[w] + (w < warp ? tot[w] : 0);
    if (base + tid < n) offsets[base + tid] = before;
    if (base + tid == n - 1) {
        offsets[n] = before + own;
        report(before + own);
    }
}
__global__ void k_report(const int64_t* __restrict__ total, const Report report) { report(*total); }

// The scratch of one search: at most 116 bytes per atom and 360 per structure (the no-allocation entry point's array
// holds 32 MiB, and the systems that fit it are part of its contract).
struct NbrScratch {
    StructInfo* info;
    int *bin_count, *bin_start, *atom_bin, *atom_rank, *counts, *words;
    int4 *atom_wrap, *items;
    float4 *atom_hi, *atom_lo, *sorted_hi;
    int64_t* sums;
};
static int64_t nbr_bins(int N, int n_s) { return 2LL * N + 8LL * n_s; }
static int64_t nbr_sums(int N) { return N > kOffsetsMax ? scan_tile_sums_len(N) : 1; }
static size_t nbr_scratch_bytes(int N, int n_s) {
    const size_t nb = (size_t)nbr_bins(N, n_s), n = (size_t)N;
    return carve_bytes(sizeof(StructInfo) * n_s, sizeof(int) * nb, sizeof(int) * nb, sizeof(int) * n, sizeof(int) * n,
                       sizeof(int) * n, sizeof(int) * 4, sizeof(int4) * n, sizeof(int4) * n, sizeof(float4) * n,
                       sizeof(float4) * n, sizeof(float4) * n, sizeof(int64_t) * nbr_sums(N));
}
static NbrScratch nbr_carve(void* base, int N, int n_s) {
    const size_t nb = (size_t)nbr_bins(N, n_s), n = (size_t)N;
    Carver cv(base);
    NbrScratch W;
    W.info = cv.take<StructInfo>(n_s);
    W.bin_count = cv.take<int>(nb);
    W.bin_start = cv.take<int>(nb);
    W.atom_bin = cv.take<int>(n);
    W.atom_rank = cv.take<int>(n);
    W.counts = cv.take<int>(n);
    W.words = cv.take<int>(4);
    W.atom_wrap = cv.take<int4>(n);
    W.items = cv.take<int4>(n);
    W.atom_hi = cv.take<float4>(n);
    W.atom_lo = cv.take<float4>(n);
    W.sorted_hi = cv.take<float4>(n);
    W.sums = cv.take<int64_t>((size_t)nbr_sums(N));
    return W;
}

// The fill pass outlives the call: rascal_set_stream makes another stream wait for it.
static int fill_queued(rascal_ctx* ctx) {
    RASCAL_CUDA(cudaEventRecord(ctx->searched, ctx->stream));
    ctx->fill_queued = true;
    return RASCAL_OK;
}

// Everything up to the pair count: *total pairs and *largest count of a centre, after one synchronisation. With output arrays
// (A.out_j) the fill pass is launched before that synchronisation, which then waits for the counts alone; it writes nothing
// unless the counts fit capacity and CAP and no flag is raised (*filled). Waiting for the counts first left the GPU idle for a
// host round trip: 8 to 10 us of every search.
template <int CAP>
static int nbr_search(rascal_ctx* ctx, const rascal_system* sys, const NbrScratch& W, int64_t capacity, int64_t* d_offsets,
                      int* d_nbr_j, int* d_shift, float* d_rij, PairArgs& A, unsigned* grid, int64_t* total, int* largest,
                      bool* filled) {
    const int N = sys->n_atoms, n_s = sys->n_structures;
    const int64_t nbins_cap = nbr_bins(N, n_s);
    cudaStream_t stream = ctx->stream;
    // lanes for every structure, and threads enough to clear the counters in a few strides
    const int per = n_s > 8 * ctx->n_sm ? 4 : 32;
    const int64_t setup_blocks = std::max<int64_t>(div_up(n_s, 128 / per), std::min<int64_t>(div_up(nbins_cap, 1024), 2LL * ctx->n_sm));
    k_struct_setup<<<(unsigned)setup_blocks, 128, 0, stream>>>(n_s, N, sys->d_struct_offsets, sys->d_cells, sys->d_pbc, ctx->r_cut,
                                                               W.info, W.bin_count, nbins_cap, W.words, ctx->d_flags, per);
    RASCAL_LAUNCH_CHECK("k_struct_setup");
    k_atom_bin<<<(unsigned)div_up(N, 64), 64, 0, stream>>>(N, n_s, nbins_cap, sys->d_struct_offsets, sys->d_positions,
                                                          sys->d_species, ctx->d_lut, W.info, W.bin_count, W.atom_bin,
                                                          W.atom_rank, W.atom_wrap, W.atom_hi, W.atom_lo, ctx->d_flags);
    RASCAL_LAUNCH_CHECK("k_atom_bin");
    // centres per work item: 16 share a staged stencil where there are atoms enough for two items per resident CTA, down
    // to one per warp in small systems, whose few bins would leave most SMs idle
    const int item_cap = (int)std::min<int64_t>(16, std::max<int64_t>(kPairWarps, N / (4LL * ctx->n_sm)));
    // few bins to a structure: small CTAs, more of them
    const int scan_threads = nbins_cap / n_s > 4096 ? 1024 : (nbins_cap / n_s > 512 ? 256 : 64);
    k_bin_scan<<<(unsigned)std::min(n_s, 8 * ctx->n_sm * (scan_threads == 64 ? 4 : 1)), scan_threads, 0, stream>>>(
        n_s, N, ctx->r_cut, item_cap, W.info, W.bin_count, W.bin_start, W.items, W.words, ctx->d_flags);
    RASCAL_LAUNCH_CHECK("k_bin_scan");
    k_atom_scatter<<<(unsigned)div_up(N, 256), 256, 0, stream>>>(N, W.atom_bin, W.atom_rank, W.bin_start, W.atom_hi,
                                                                W.sorted_hi, ctx->d_flags);
    RASCAL_LAUNCH_CHECK("k_atom_scatter");
    std::memset(&A, 0, sizeof(A));
    A.n_atoms = N;
    A.pos = sys->d_positions;
    A.info = W.info;
    A.bin_count = W.bin_count;
    A.bin_start = W.bin_start;
    A.sorted_hi = W.sorted_hi;
    A.atom_wrap = W.atom_wrap;
    A.atom_lo = W.atom_lo;
    A.items = W.items;
    A.words = W.words;
    A.rc2 = ctx->r_cut * ctx->r_cut;
    A.counts = W.counts;
    A.offsets = d_offsets;
    A.flags = ctx->d_flags;
    A.out_j = d_nbr_j;
    A.out_shift = d_shift;
    A.out_rij = reinterpret_cast<float4*>(d_rij);
    ctx->searches = ctx->searches % 0x7fffffff + 1;
    const Report report = {W.words, ctx->d_flags, ctx->h_pinned, ctx->h_flags, capacity, CAP, ctx->searches};
    *grid = (unsigned)std::min<int64_t>(N, 8LL * ctx->n_sm);
    k_pairs<false, CAP><<<*grid, kPairWarps * 32, 0, stream>>>(A);
    RASCAL_LAUNCH_CHECK("k_pairs<count>");
    if (N <= kOffsetsMax) {
        k_offsets<<<(unsigned)div_up(N, kOffsetsThreads), kOffsetsThreads, 0, stream>>>(N, W.counts, d_offsets, report);
        RASCAL_LAUNCH_CHECK("k_offsets");
    } else {
        const int st = scan_exclusive_into(W.counts, d_offsets, N, stream, W.sums);
        if (st) return st;
        k_report<<<1, 1, 0, stream>>>(d_offsets + N, report);
        RASCAL_LAUNCH_CHECK("k_report");
    }
    RASCAL_CUDA(cudaEventRecord(ctx->counted, stream));
    const bool outputs = d_nbr_j && d_shift && d_rij;
    if (outputs) {
        A.search = ctx->searches;
        k_pairs<true, CAP><<<*grid, kPairWarps * 32, 0, stream>>>(A);
        RASCAL_LAUNCH_CHECK("k_pairs<fill>");
        A.search = 0;
        if (const int st = fill_queued(ctx)) return st;
    }
    RASCAL_CUDA(cudaEventSynchronize(ctx->counted));
    const int st = flags_status(ctx, *ctx->h_flags);
    if (st) return st;
    *total = ctx->h_pinned[0];
    *largest = (int)ctx->h_pinned[1];
    *filled = outputs && *total <= capacity && *largest <= CAP;
    return RASCAL_OK;
}

}  // namespace rascal

using namespace rascal;

extern "C" int rascal_neighbours(rascal_ctx* ctx, const rascal_system* sys, int64_t capacity, int64_t* d_offsets,
                                 int* d_nbr_j, int* d_shift, float* d_rij, int64_t* n_pairs) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    int st = validate_system(ctx, sys);
    if (st) return st;
    if (!d_offsets || !n_pairs || capacity < 0) return set_error(RASCAL_E_ARG, "NULL offsets / n_pairs or negative capacity");
    const int N = sys->n_atoms, n_s = sys->n_structures;
    *n_pairs = 0;
    if (N == 0) {
        RASCAL_CUDA(cudaMemsetAsync(d_offsets, 0, sizeof(int64_t), ctx->stream));
        return RASCAL_OK;
    }
    void* base;
    if ((st = arena_get(ctx->scratch, nbr_scratch_bytes(N, n_s), &base))) return st;
    PairArgs A;
    unsigned grid;
    int64_t P;
    int maxc;
    bool filled;
    if ((st = nbr_search<kPairCap>(ctx, sys, nbr_carve(base, N, n_s), capacity, d_offsets, d_nbr_j, d_shift, d_rij, A, &grid,
                                   &P, &maxc, &filled)))
        return st;
    *n_pairs = P;
    if (P > capacity) return set_error(RASCAL_E_CAPACITY, "pair capacity %lld < required %lld", (long long)capacity, (long long)P);
    if (P == 0 || filled) return RASCAL_OK;
    if (!d_nbr_j || !d_shift || !d_rij) return set_error(RASCAL_E_ARG, "NULL pair output arrays");
    if (maxc <= kNoallocCap) {  // 30 000 centres of 137 pairs: 955 us with the sort in scratch, 695 in shared memory
        k_pairs<true, kNoallocCap><<<grid, kPairWarps * 32, 0, ctx->stream>>>(A);
        RASCAL_LAUNCH_CHECK("k_pairs<fill>");
        return fill_queued(ctx);
    }
    {  // a centre has more pairs than a warp sorts in shared memory
        void* ob;
        if ((st = arena_get(ctx->scratch2, carve_bytes(sizeof(uint64_t) * P, sizeof(float4) * P), &ob))) return st;
        Carver oc(ob);
        A.ovf_keys = oc.take<uint64_t>(P);
        A.ovf_vec = oc.take<float4>(P);
    }
    k_pairs<true><<<grid, kPairWarps * 32, 0, ctx->stream>>>(A);
    RASCAL_LAUNCH_CHECK("k_pairs<fill>");
    return fill_queued(ctx);
}

// ---------------------------------------------------------------------------------------------------------
// Neighbour search that allocates nothing: the same kernels as rascal_neighbours, with all scratch carved out of
// one file-scope device array. The array is a module global, so every GPU that loads the library holds it until
// the process exits. Its device address is looked up per device (cudaGetSymbolAddress with that device current)
// when a context is created on it, and cached; all calls on a device share the array.
// ---------------------------------------------------------------------------------------------------------
namespace rascal {

constexpr size_t kStaticNbrScratchBytes = size_t(32) << 20;
static __device__ __align__(256) unsigned char g_nbr_scratch[kStaticNbrScratchBytes];
constexpr int kMaxDevices = 64;
static void* g_nbr_scratch_addr[kMaxDevices];
static std::mutex g_nbr_scratch_mu;

// Caches the device address of the array for ctx->device, which must be the current device. Called by
// rascal_create, so the lookup (which may load the module and reserve the array) happens before any step loop.
int nbr_static_prepare(rascal_ctx* ctx) {
    const int dev = ctx->device;
    if (dev < 0 || dev >= kMaxDevices) return set_error(RASCAL_E_UNSUPPORTED, "device ordinal %d above %d", dev, kMaxDevices - 1);
    std::lock_guard<std::mutex> lock(g_nbr_scratch_mu);
    if (!g_nbr_scratch_addr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_nbr_scratch);
        if (e != cudaSuccess || !p)
            return set_error(RASCAL_E_CUDA, "cudaGetSymbolAddress of the static neighbour scratch: %s", cudaGetErrorString(e));
        g_nbr_scratch_addr[dev] = p;
    }
    return RASCAL_OK;
}

// The cached address for the context's device. The kernels run on ctx->stream, which belongs to ctx->device, so a
// call made while another device is current is refused rather than handed another GPU's copy of the array.
static int static_nbr_scratch(const rascal_ctx* ctx, void** out) {
    int cur = -1;
    const cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return set_error(RASCAL_E_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (cur != ctx->device)
        return set_error(RASCAL_E_ARG, "the current device (%d) is not the context's device (%d)", cur, ctx->device);
    std::lock_guard<std::mutex> lock(g_nbr_scratch_mu);
    *out = g_nbr_scratch_addr[ctx->device];
    if (!*out) return set_error(RASCAL_E_CUDA, "the static neighbour scratch of device %d was not prepared", ctx->device);
    return RASCAL_OK;
}

}  // namespace rascal

extern "C" size_t rascal_neighbours_static_limit(void) { return rascal::kStaticNbrScratchBytes; }

extern "C" int rascal_neighbours_noalloc(rascal_ctx* ctx, const rascal_system* sys, int64_t capacity, int64_t* d_offsets,
                                         int* d_nbr_j, int* d_shift, float* d_rij, int64_t* n_pairs) {
    clear_error();
    if (!ctx) return set_error(RASCAL_E_ARG, "NULL context");
    int st = validate_system(ctx, sys);
    if (st) return st;
    if (!d_offsets || !n_pairs || capacity < 0) return set_error(RASCAL_E_ARG, "NULL offsets / n_pairs or negative capacity");
    const int N = sys->n_atoms, n_s = sys->n_structures;
    *n_pairs = 0;
    if (N == 0) {
        RASCAL_CUDA(cudaMemsetAsync(d_offsets, 0, sizeof(int64_t), ctx->stream));
        return RASCAL_OK;
    }
    // what the entry point's limit counts: 116 bytes per atom, 360 per structure (nbr_scratch_bytes is never more)
    const int64_t nbins_cap = nbr_bins(N, n_s);
    const int64_t sums_len = std::max(scan_tile_sums_len(n_s), std::max(scan_tile_sums_len(nbins_cap), scan_tile_sums_len(N)));
    const size_t bytes = carve_bytes((size_t)280 * n_s, sizeof(int) * (n_s + 1), sizeof(int64_t) * (n_s + 1), sizeof(int) * nbins_cap,
                                     sizeof(int64_t) * (nbins_cap + 1), sizeof(int) * N, sizeof(int) * N, sizeof(int) * N,
                                     sizeof(int4) * N, sizeof(int4) * N, sizeof(float4) * N, sizeof(float4) * N,
                                     sizeof(float4) * N, sizeof(int) * 4, sizeof(int64_t) * sums_len);
    if (bytes > kStaticNbrScratchBytes)
        return set_error(RASCAL_E_UNSUPPORTED,
                         "this system needs %zu bytes of neighbour scratch; the no-allocation entry point holds %zu "
                         "(about 116 bytes per atom and 360 per structure): use rascal_neighbours",
                         bytes, kStaticNbrScratchBytes);
    void* base = nullptr;
    if ((st = static_nbr_scratch(ctx, &base))) return st;
    PairArgs A;
    unsigned grid;
    int64_t P;
    int maxc;
    bool filled;
    // the fill is launched only once the call is known to succeed: its scratch is shared by all contexts of the device, and a
    // refused call leaves nothing queued that reads it
    if ((st = nbr_search<kNoallocCap>(ctx, sys, nbr_carve(base, N, n_s), capacity, d_offsets, nullptr, nullptr, nullptr, A, &grid,
                                      &P, &maxc, &filled)))
        return st;
    *n_pairs = P;
    // checked before the capacity, so that a caller who resizes after RASCAL_E_CAPACITY is not refused afterwards
    if (maxc > kNoallocCap)
        return set_error(RASCAL_E_UNSUPPORTED, "a centre has %d neighbours; the no-allocation entry point sorts at most %d "
                         "per centre (rascal_neighbours has no such limit)", maxc, kNoallocCap);
    if (P > capacity) return set_error(RASCAL_E_CAPACITY, "pair capacity %lld < required %lld", (long long)capacity, (long long)P);
    if (P == 0) return RASCAL_OK;
    if (!d_nbr_j || !d_shift || !d_rij) return set_error(RASCAL_E_ARG, "NULL pair output arrays");
    A.out_j = d_nbr_j;
    A.out_shift = d_shift;
    A.out_rij = reinterpret_cast<float4*>(d_rij);
    k_pairs<true, kNoallocCap><<<grid, kPairWarps * 32, 0, ctx->stream>>>(A);
    RASCAL_LAUNCH_CHECK("k_pairs<fill>");
    return fill_queued(ctx);
}
