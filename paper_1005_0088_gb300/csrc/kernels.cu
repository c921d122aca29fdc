// FP64 kernels of the per-pole factor / selected-inversion path.
//
// Front layout: every supernode J owns a dense f x f complex front (f = |J| + |struct(J)|),
// column-major, J's columns first; only the lower triangle is kept valid.  All poles of a chunk
// are batched in one launch (grid.y = pole), each pole owning one slab of fronts and one slab
// of scratch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "fixed_point.cuh"
#include "kernels.cuh"
#include "pivot.cuh"

namespace ndsi {

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// x 2^e (e = 0 for every entry of a normalised basis).
__device__ __forceinline__ double scale2(double x, int e) {
    if (e == 0) return x;
    return e >= -1022 && e <= 1023 ? x * __hiloint2double((1023 + e) << 20, 0) : ldexp(x, e);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// ---------------------------------------------------------------------------------------------
// Front assembly: F_J = sum over children c of U_c (extend-add through the inverse relative
// index maps), written for the lower triangle of every front of a level.  Zero where no child
// contributes; the original entries are added afterwards by k_scatter.  One CTA per 32 x 32 tile
// (lanes = rows, 8 warps x 4 columns) and several poles, which share the tile's indices: the chain
// tile -> node -> children -> index maps takes as long as the loads themselves.  A thread's eight loads
// are in flight together, and FP64 additions (16 clocks of an SM per warp) are left out where one
// child contributes.  80 poles of a cubic lattice of 16^3 atoms x 4 orbitals: 15.8 -> 10.8 ms, 5.8 TB/s.
__global__ void __launch_bounds__(256) k_assemble(const NodeDev* __restrict__ nodes,
                                                  const NodeTile* __restrict__ tiles, int64_t first,
                                                  const int32_t* __restrict__ inv_map,
                                                  double2* __restrict__ F, int64_t stride, int np) {
    static_assert(kNodeTile == 32, "one lane per tile row, 8 warps x 4 columns");
    constexpr int kCols = kNodeTile / 8;
    const NodeTile t = tiles[first + blockIdx.x];
    const NodeDev& nd = nodes[t.node];
    __shared__ NodeDev ch[2];
    __shared__ int ibs[2][kNodeTile];
    const int tx = threadIdx.x, ty = threadIdx.y, f = nd.f, nchild = nd.nchild;
    if (tx < nchild && ty == 0) ch[tx] = nodes[nd.child[tx]];
    if (ty < nchild) ibs[ty][tx] = t.j0 + tx < f ? inv_map[nd.inv_off[ty] + t.j0 + tx] : -1;
    const int a = t.i0 + tx;
    int ia[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) ia[c] = c < nchild && a < f ? inv_map[nd.inv_off[c] + a] : -1;
    __syncthreads();
    int64_t src[2][kCols];  // element of each child and column, -1: none
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < kCols; ++u) {
            const int q = ty + 8 * u;
            const bool has = ia[c] >= 0 && ibs[c][q] >= 0 && t.j0 + q <= a;
            src[c][u] = has ? ch[c].front_off + ch[c].s + ia[c] + (static_cast<int64_t>(ch[c].s) + ibs[c][q]) * ch[c].f : -1;
        }
    const int64_t dst = nd.front_off + a + static_cast<int64_t>(t.j0 + ty) * f;
    auto run = [&](auto adds) {
        for (int pole = blockIdx.y; pole < np; pole += gridDim.y) {
            double2* Fp = F + pole * stride;
            double2 v[2][kCols];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int u = 0; u < kCols; ++u) {
                    v[c][u] = make_double2(0.0, 0.0);
                    if (src[c][u] >= 0) v[c][u] = Fp[src[c][u]];
                }
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
                const bool one = src[0][u] >= 0, both = one && src[1][u] >= 0;
                double2 o = make_double2(one ? v[0][u].x : v[1][u].x, one ? v[0][u].y : v[1][u].y);
                if (decltype(adds)::value && both) o = cadd(v[0][u], v[1][u]);
                const int b = t.j0 + ty + 8 * u;
                if (b <= a && a < f) Fp[dst + static_cast<int64_t>(8 * u) * f] = o;
            }
        }
    };
    // two loops: an addition that no lane of a warp needs would still take its 64 clocks
    bool both = false;
#pragma unroll
    for (int u = 0; u < kCols; ++u) both |= src[0][u] >= 0 && src[1][u] >= 0;
    if (__any_sync(0xffffffffu, both)) run(std::true_type{});
    else run(std::false_type{});
}

// ---------------------------------------------------------------------------------------------
// Basis scaling (launch_basis_scale): four passes over the pattern, one warp per row, bound by the
// latency of a row's dependent loads (its columns, then their diagonals or scales), so four entries of a lane
// are in flight together (12 us a sweep for 320,000 entries instead of 25 one at a time).  Against scales from S_ii
// alone a sweep takes 6 us longer for 12,000 entries (0.96 -> 0.97 ms) and 16 us for 260,000 (7.84 -> 7.85 ms).
// Exponent of |x| (|x| < 2^e); zero, subnormal and non-finite
// values do not take part.
constexpr int kNoExpo = -4000;
__device__ __forceinline__ int expo_of(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7FF;
    return e == 0 || e == 0x7FF ? kNoExpo : e - 1022;
}
// Exponent that brings S_ii into [1/2, 2); 0 unless S_ii is positive and normal.
__device__ __forceinline__ int norm_expo(double sii) {
    const int b = __double2hiint(sii) >> 20;
    return b > 0 && b < 0x7FF ? -((b - 1022) >> 1) : 0;
}
// Exponent of |z S_ij| + |H_ij| without its cancellation (the size at which the entry is rounded).
__device__ __forceinline__ int entry_expo(double h, double s, int ez) { return max(expo_of(h), expo_of(s) + ez); }

constexpr int kScaleRows = 8;     // rows (warps) per block of the scaling kernels
constexpr int kScaleUnit = 8;     // the row scales g count eighths of a binary place
constexpr int kScaleBias = 1 << 20;
constexpr int kScaleGuard = 12;   // places a diagonal may lie below its row's maximum
// Row scales further than these from their mean (in eighths) bring the scaling about.
constexpr int kScaleBelow = 12, kScaleAbove = 20;

// Mean row scale of a system; `wide`: its rows differ enough to be scaled beyond S_ii.
__device__ __forceinline__ int scale_mean(const ScaleStat& t, bool& wide) {
    const int mean = static_cast<int>(t.sum / max(t.count, 1u)) - kScaleBias;
    wide = mean - (kScaleBias - t.lo) > kScaleBelow || (t.hi - kScaleBias) - mean > kScaleAbove;
    return mean;
}

// Start: exponent of the smallest point of the row's system, S_ii's exponent, and the row scale
// 2^(-D / 2) of its diagonal, D = exponent of |H_ii| + |z S_ii|, at least that of its largest entry
// less kScaleGuard places.  Clears the statistics.
__global__ void __launch_bounds__(32 * kScaleRows) k_scale_start(
    const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, const int64_t* __restrict__ diag,
    const int32_t* __restrict__ entry_sys, int64_t n, const double* __restrict__ H, const double* __restrict__ S,
    const double2* __restrict__ z, int64_t zstride, int nz, int n_sys, ScaleTables t) {
    if (blockIdx.x == 0) {
        for (int s = threadIdx.x; s < n_sys; s += blockDim.x) {
            t.stat[s].sum = 0;
            t.stat[s].lo = t.stat[s].hi = 0;
            t.stat[s].count = 0;
        }
        if (threadIdx.x == 0) *t.any = 0;
    }
    const int lane = threadIdx.x & 31;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kScaleRows + (threadIdx.x >> 5);
    if (i >= n) return;
    const int sys = entry_sys[diag[i]];
    int ez = -kNoExpo;
    for (int q = lane; q < nz; q += 32) {
        const double2 zq = z[sys * zstride + q];
        const int e = max(expo_of(zq.x), expo_of(zq.y));
        if (e > kNoExpo) ez = min(ez, e);
    }
    ez = __reduce_min_sync(0xffffffffu, ez);
    if (ez == -kNoExpo) ez = kNoExpo;  // every point is zero
    const double sii = S[diag[i]];
    const int fi = norm_expo(sii);
    int r = 2 * kNoExpo;
#pragma unroll 4
    for (int64_t k = rowptr[i] + lane; k < rowptr[i + 1]; k += 32)
        r = max(r, entry_expo(H[k], S[k], ez) + fi + norm_expo(S[diag[col[k]]]));
    r = __reduce_max_sync(0xffffffffu, r);
    if (lane == 0) {
        const int d = max(entry_expo(H[diag[i]], sii, ez) + 2 * fi, r - kScaleGuard);
        t.norm[i] = static_cast<int16_t>(fi);
        t.ez[i] = static_cast<int16_t>(ez);
        t.g[0][i] = d < kNoExpo / 2 ? 0 : -(kScaleUnit / 2) * d;
    }
}

// One step of symmetric equilibration in the maximum norm (Ruiz 2001): every row scale moves by half of what
// its largest scaled entry is off.  The first step also gathers the statistics the second one and the
// tables are decided by.
template <bool FIRST>
__global__ void __launch_bounds__(32 * kScaleRows) k_scale_step(
    const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, const int64_t* __restrict__ diag,
    const int32_t* __restrict__ entry_sys, int64_t n, const double* __restrict__ H, const double* __restrict__ S,
    ScaleTables t) {
    __shared__ int gs[kScaleRows], ss[kScaleRows];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kScaleRows + w;
    const int sys = i < n ? entry_sys[diag[i]] : -1;
    bool wide = true;
    if (!FIRST && sys >= 0) scale_mean(t.stat[sys], wide);
    const int* gin = t.g[FIRST ? 0 : 1];
    int g = 0;
    if (sys >= 0 && wide) {
        const int ez = t.ez[i], fi = t.norm[i], gi = gin[i];
        int m = 4 * kScaleUnit * kNoExpo;
#pragma unroll 4
        for (int64_t k = rowptr[i] + lane; k < rowptr[i + 1]; k += 32) {
            const int e = entry_expo(H[k], S[k], ez);
            if (e > kNoExpo / 2) m = max(m, kScaleUnit * (e + fi + t.norm[col[k]]) + gin[col[k]]);
        }
        m = __reduce_max_sync(0xffffffffu, m);
        g = m == 4 * kScaleUnit * kNoExpo ? gi : gi - ((m + gi) >> 1);
        if (lane == 0) t.g[FIRST ? 1 : 0][i] = g;
    }
    if (FIRST) {
        if (lane == 0) {
            gs[w] = g;
            ss[w] = sys;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int a = 0; a < kScaleRows && ss[a] >= 0;) {  // runs of rows of one system
                unsigned long long sum = 0;
                int lo = 0, hi = 0, b = a;
                for (; b < kScaleRows && ss[b] == ss[a]; ++b) {
                    sum += static_cast<unsigned long long>(kScaleBias + gs[b]);
                    lo = max(lo, kScaleBias - gs[b]);
                    hi = max(hi, kScaleBias + gs[b]);
                }
                ScaleStat* st = t.stat + ss[a];
                atomicAdd(&st->sum, sum);
                atomicMax(&st->lo, lo);
                atomicMax(&st->hi, hi);
                atomicAdd(&st->count, static_cast<unsigned>(b - a));
                a = b;
            }
        }
    }
}

__global__ void __launch_bounds__(32 * kScaleRows) k_pair_scale(const int64_t* __restrict__ rowptr,
                                                                const int32_t* __restrict__ col,
                                                                const int64_t* __restrict__ diag,
                                                                const int32_t* __restrict__ entry_sys, int64_t n,
                                                                ScaleTables t) {
    const int lane = threadIdx.x & 31;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kScaleRows + (threadIdx.x >> 5);
    if (i >= n) return;
    bool wide;
    const int mean = scale_mean(t.stat[entry_sys[diag[i]]], wide);
    auto expo = [&](int64_t j) { return t.norm[j] + (wide ? (t.g[0][j] - mean + kScaleUnit / 2) >> 3 : 0); };
    static_assert(kScaleUnit == 8, "the shift by three");
    const int fi = expo(i);
    if (lane == 0) {
        t.f[i] = static_cast<int16_t>(fi);
        if (fi != 0) *t.any = 1;
    }
#pragma unroll 4
    for (int64_t k = rowptr[i] + lane; k < rowptr[i + 1]; k += 32) t.pair[k] = static_cast<int16_t>(fi + expo(col[k]));
}

// X = z S - H on the level's entries (each front element receives at most one entry), scaled by the
// entry's pair exponent.
// z[sys * zstride + pole] is the point of the entry's system (systems of a batch have their own
// mu and kT).
__global__ void __launch_bounds__(256) k_scatter(const int64_t* __restrict__ idx, int64_t first,
                                                 int64_t count, const int64_t* __restrict__ asm_map,
                                                 const int32_t* __restrict__ entry_sys,
                                                 const double* __restrict__ H,
                                                 const double* __restrict__ S,
                                                 const int16_t* __restrict__ pair,
                                                 const double2* __restrict__ z, int64_t zstride,
                                                 double2* __restrict__ F, int64_t stride) {
    double2* Fp = F + static_cast<int64_t>(blockIdx.y) * stride;
    for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < count;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t k = idx[first + e];
        const int64_t off = asm_map[k];
        const double2 zq = z[entry_sys[k] * zstride + blockIdx.y];
        const double h = H[k], s = S[k];
        double2 v = Fp[off];
        const int pe = pair[k];
        v.x += scale2(zq.x * s - h, pe);
        v.y += scale2(zq.y * s, pe);
        Fp[off] = v;
    }
}

// FP64 inverse of a complex-symmetric pivot block (Gauss-Jordan sweeps without pivoting).
// No pivoting is needed: for Im z != 0 and S SPD, Im(X) = Im(z) S is definite, so every leading
// block and every Schur complement of X is nonsingular.  A zero or non-finite pivot sets the
// singular bit of the status word.
template <int NB>
__global__ void __launch_bounds__(256) k_diaginv(const DiagItem* __restrict__ items, int64_t first,
                                                 double2* __restrict__ F, int64_t stride,
                                                 int* __restrict__ status) {
    extern __shared__ double2 smem_dinv[];
    double2 (*a)[NB + 1] = reinterpret_cast<double2 (*)[NB + 1]>(smem_dinv);
    const DiagItem d = items[first + blockIdx.x];
    double2* A = F + static_cast<int64_t>(blockIdx.y) * stride + d.off;
    const int nb = d.nb, ld = d.ld;
    const int tid = threadIdx.x;
    if (nb > NB) {
        if (tid == 0) atomicOr(status, kStatusBadItem);
        return;
    }
    for (int e = tid; e < nb * nb; e += blockDim.x) {
        const int i = e % nb, j = e / nb;
        a[i][j] = i >= j ? A[i + static_cast<int64_t>(j) * ld] : A[j + static_cast<int64_t>(i) * ld];
    }
    __syncthreads();
    constexpr int kPer = (NB * NB + 255) / 256;
    for (int t = 0; t < nb; ++t) {
        const double2 p = a[t][t];
        const double den = p.x * p.x + p.y * p.y;
        if (tid == 0 && !(den > 0.0 && isfinite(den))) atomicOr(status, kStatusSingular);
        const double2 ip = make_double2(p.x / den, -p.y / den);
        double2 nv[kPer];
        #pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int e = tid + u * 256;
            if (e < nb * nb) {
                const int i = e % nb, j = e / nb;
                if (i == t && j == t) {
                    nv[u] = ip;
                } else if (i == t) {
                    nv[u] = cmul(a[t][j], ip);
                } else if (j == t) {
                    const double2 v = cmul(a[i][t], ip);
                    nv[u] = make_double2(-v.x, -v.y);
                } else {
                    const double2 v = cmul(cmul(a[i][t], ip), a[t][j]);
                    nv[u] = make_double2(a[i][j].x - v.x, a[i][j].y - v.y);
                }
            }
        }
        __syncthreads();
        #pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int e = tid + u * 256;
            if (e < nb * nb) a[e % nb][e / nb] = nv[u];
        }
        __syncthreads();
    }
    for (int e = tid; e < nb * nb; e += blockDim.x) {
        const int i = e % nb, j = e / nb;
        if (i >= j) A[i + static_cast<int64_t>(j) * ld] = a[i][j];
    }
}

// Register-resident variant for blocks of up to N = 16 or 32: one warp per (block, pole) running
// the symmetric sweep, the sign convention of Gauss-Jordan elimination that keeps a symmetric
// matrix symmetric.  Pivoting on t with p = a_tt maps a_tt -> -1/p, a_it and a_ti -> a_it/p and
// a_ik -> a_ik - a_it a_tk / p; after all pivots the block holds -A^{-1}.  Because every
// intermediate matrix is symmetric only the N(N+1)/2 lower-triangle elements are updated, half
// the FP64 work of the full elimination.  They are packed onto the lanes: virtual column c
// (c < N/2) is rows c..N-1 of column c followed by rows N-1-c..N-1 of column N-1-c (N+1
// elements), split evenly over 64/N lanes.  Every lane runs the same instruction stream (no
// divergent pivot lane); column t of the current matrix and its scaled copy pass through shared
// memory.  N = 16 serves launches whose pivot blocks are all at most 16 wide (small separators
// and the ragged last block of a front) at about a third of the N = 32 cost.
template <int N>
__global__ void __launch_bounds__(32) k_diaginv_sweep(const DiagItem* __restrict__ items, int64_t first,
                                                      double2* __restrict__ F, int64_t stride,
                                                      int* __restrict__ status) {
    constexpr int VC = N / 2;                  // virtual columns
    constexpr int LPC = 32 / VC;               // lanes per virtual column
    constexpr int SLOTS = (N + 1 + LPC - 1) / LPC;
    __shared__ double2 cs[33], ds[33];
    const int lane = threadIdx.x;
    const DiagItem d = items[first + blockIdx.x];
    double2* A = F + static_cast<int64_t>(blockIdx.y) * stride + d.off;
    const int nb = d.nb, ld = d.ld;
    if (nb > N) {
        if (lane == 0) atomicOr(status, kStatusBadItem);
        return;
    }
    const int c = lane % VC, vbase = (lane / VC) * SLOTS;
    int rc[SLOTS];  // row | column << 8 of each slot (32 = unused slot)
    double2 a[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int v = vbase + s;
        int i = 32, k = 32;
        if (v < N - c) {
            i = c + v;
            k = c;
        } else if (v <= N) {
            i = v - 1;
            k = N - 1 - c;
        }
        rc[s] = i | (k << 8);
        a[s] = make_double2(0.0, 0.0);
        if (i < nb && k < nb) a[s] = A[i + static_cast<int64_t>(k) * ld];
    }
    if (lane == 0) {
        cs[32] = make_double2(0.0, 0.0);
        ds[32] = make_double2(0.0, 0.0);
    }
    bool bad = false;
    for (int t = 0; t < nb; ++t) {
        // column t (= row t) of the current matrix
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            const int i = rc[s] & 255, k = rc[s] >> 8;
            if (k == t) cs[i] = a[s];
            if (i == t) cs[k] = a[s];
        }
        __syncwarp();
        const double2 p = cs[t];
        const double den = p.x * p.x + p.y * p.y;
        bad |= bad_pivot(den);
        const double rden = 1.0 / den;
        const double2 ip = make_double2(p.x * rden, -p.y * rden), nip = make_double2(-ip.x, -ip.y);
        if (lane < N) ds[lane] = cmul(cs[lane], ip);
        __syncwarp();
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            const int i = rc[s] & 255, k = rc[s] >> 8;
            const double2 cv = cs[i], dk = ds[k], di = ds[i];
            const double2 g = make_double2(fma(-cv.x, dk.x, fma(cv.y, dk.y, a[s].x)), fma(-cv.x, dk.y, fma(-cv.y, dk.x, a[s].y)));
            // the pivot row and column take d (the pivot itself -1/p), by selects: a branch here diverges
            const bool kq = k == t, iq = i == t;
            const double2 o = kq ? (iq ? nip : di) : dk;
            a[s] = make_double2(kq | iq ? o.x : g.x, kq | iq ? o.y : g.y);
        }
        __syncwarp();
    }
    if (bad && lane == 0) atomicOr(status, kStatusSingular);
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int i = rc[s] & 255, k = rc[s] >> 8;
        if (i < nb && k < nb) A[i + static_cast<int64_t>(k) * ld] = make_double2(-a[s].x, -a[s].y);
    }
}

// ---------------------------------------------------------------------------------------------
// Whole diagonal block in one launch: the inverse of a complex-symmetric block of up to 128 columns
// by the symmetric block sweep.  With pivot block t (16 wide), P = A_tt^{-1}, C_i = A_it and
// W_i = C_i P the sweep maps
//     A_ij <- A_ij - W_i C_j^T (i, j outside the pivot),   A_it <- W_i,   A_tt <- -P,
// and after every pivot block A holds -A^{-1}; every intermediate matrix is symmetric, so only 8 x 8
// blocks of the lower triangle are kept (in shared memory, FP64) and updated (n^3 / 2 complex
// multiply-adds).  The pivot blocks are inverted in FP64; the panel and update products run in
// fixed point (fixed_point.cuh, three real products), with the panels' digits formed once per pivot step.
// Bound: for 128 columns the updates (16 x 8 units handed out dynamically, 45k of 71k clocks per pivot
// block), for narrow blocks, of which two or three share an SM, the FP64 instructions of the pivot
// block: a sub-partition takes 64 clocks for each and an SM 16, so four warps, one per
// sub-partition, invert the next pivot block, updated first, while the others still update.  40
// poles of a chain of 64 atoms x 8 orbitals (128-column blocks) 1.13 -> 0.96 ms against one pivot warp with
// divisions and twelve multiply-adds per product, twelve uneven systems (batched, 80 columns and fewer)
// 63.0 -> 59.1 ms, density of states of a 30 x 26 x 5 sheet 14.4 -> 13.3 ms.
// Replaces, per 16 columns, a pivot-inverse, panel, update and copy launch each and the backward
// assembly (53 launches for 128 columns).
constexpr int kBlkP = 16;   // pivot width
constexpr int kBlkLd = 17;  // row stride of pivot blocks in shared memory

__host__ __device__ constexpr size_t diag_block_smem(int tile) {
    const int nb8 = tile / 8, rows = tile - kBlkP;
    return static_cast<size_t>(nb8 * (nb8 + 1) / 2) * 64 * sizeof(double2) +        // lower 8 x 8 blocks
           sizeof(int4) * (2 * kBlkP * rows + kBlkP * kBlkLd) +                     // digits of W, C and P
           sizeof(double2) * kBlkP * (kBlkLd + 1) +                                 // pivot block, scaled column
           sizeof(int) * (2 * rows + kBlkP) +                                       // exponents
           sizeof(int) * 4 + sizeof(uint16_t) * nb8 * (nb8 + 1) / 2;                // counters, unit list
}

// Threads per block of up to `tile` columns: narrow blocks leave room for three CTAs (64 columns, 71 KB
// each) or two (80 columns) on an SM, whose pivot inversions then overlap; a 128-column block fills
// one SM's shared memory and uses 16 warps for its updates.
constexpr int diag_block_threads(int tile) { return tile <= 64 ? 128 : tile <= 80 ? 256 : 512; }

__global__ void __launch_bounds__(512) k_diaginv_block(const DiagItem* __restrict__ items, int64_t first,
                                                       double2* __restrict__ F, int64_t stride,
                                                       int* __restrict__ status, int tile) {
    extern __shared__ double2 smem_blk[];
    const int T8 = tile / 8, R = tile - kBlkP;
    double2* M = smem_blk;                                    // block (I, J) at I (I + 1) / 2 + J, column-major
    int4* Wd = reinterpret_cast<int4*>(M + (T8 * (T8 + 1) / 2) * 64);  // [16][R], k-major
    int4 *Cd = Wd + kBlkP * R, *Pd = Cd + kBlkP * R;          // [16][R]; [16][17] symmetric
    double2* XB = reinterpret_cast<double2*>(Pd + kBlkP * kBlkLd);     // [16][17] second copy of the pivot block
    double2* ds = XB + kBlkP * kBlkLd;                        // [16] scaled pivot column
    int* We = reinterpret_cast<int*>(ds + kBlkP);            // row exponents of W, C; column exponents of P
    int *Ce = We + R, *Pe = Ce + R;
    int* ctr = Pe + kBlkP;                                    // [0] next unit, [1] list length
    uint16_t* list = reinterpret_cast<uint16_t*>(ctr + 4);    // update units: row pair I16 << 8 | column block J
    const DiagItem d = items[first + blockIdx.x];
    double2* A = F + static_cast<int64_t>(blockIdx.y) * stride + d.off;
    const int n = d.nb, ld = d.ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (n > tile) {
        if (tid == 0) atomicOr(status, kStatusBadItem);
        return;
    }
    const int nb8 = (n + 7) / 8, nt = (n + kBlkP - 1) / kBlkP;
    auto blk = [&](int I, int J) { return M + (I * (I + 1) / 2 + J) * 64; };
    // load the lower triangle (rows and columns past n are zero)
    for (int b = warp; b < nb8 * (nb8 + 1) / 2; b += nw) {
        int I = 0;
        while ((I + 1) * (I + 2) / 2 <= b) ++I;
        const int J = b - I * (I + 1) / 2;
        for (int e = lane; e < 64; e += 32) {
            const int i = I * 8 + (e & 7), j = J * 8 + (e >> 3);
            M[b * 64 + e] = (i < n && j <= i) ? A[i + static_cast<int64_t>(j) * ld] : make_double2(0.0, 0.0);
        }
    }
    if (tid == 0) {
        int cnt = 0;
        for (int I = 0; I < nt; ++I)
            for (int J = 0; J <= min(2 * I + 1, nb8 - 1); ++J) list[cnt++] = static_cast<uint16_t>(I << 8 | J);
        ctr[1] = cnt;
    }
    const int r8 = lane & 7, cq = lane >> 3;  // a unit's row and first column of this lane
    // inverse of pivot block t by warps 0..3 (rank-1 symmetric sweeps on the lower triangle), written
    // to the block itself (-P) and, as digits, to P.  A step reads one of two copies and writes the
    // other; the warps take turns at the scaled column, which costs twice the FP64 instructions of a
    // warp's share of the update.
    auto pivot = [&](int t) {
        const int nb = min(kBlkP, n - t * kBlkP);
        auto at = [&](int i, int k) { return blk(2 * t + (i >> 3), 2 * t + (k >> 3)) + (k & 7) * 8 + (i & 7); };
        auto barrier = [] { asm volatile("bar.sync 1, 128;" ::: "memory"); };
        double2* XA = reinterpret_cast<double2*>(Pd);
        for (int e = tid; e < kBlkP * kBlkP; e += 128) {
            const int i = e / kBlkP, k = e % kBlkP;
            if (k <= i) XA[i * kBlkLd + k] = i < nb ? *at(i, k) : make_double2(0.0, 0.0);
        }
        // this thread's element among the 120 outside the pivot row and column, counted without them
        const bool own = tid < kBlkP * (kBlkP - 1) / 2;
        int i0 = 0;
        while (own && (i0 + 1) * (i0 + 2) / 2 <= tid) ++i0;
        const int j0 = own ? tid - i0 * (i0 + 1) / 2 : 0;
        const int idx = lane & 15;  // column element of this lane: real part, or imaginary part in lanes 16..31
        const bool im = lane >= 16;
        bool bad = false;
        barrier();
        for (int q = 0; q < nb; ++q) {
            const double2* X = q & 1 ? XB : XA;
            double2* Y = q & 1 ? XA : XB;
            auto tri = [](int r, int c) { return r > c ? r * kBlkLd + c : c * kBlkLd + r; };
            if (warp == (q & 3)) {  // d = c / p, 1 / p in the pivot's place
                const double2 p = X[tri(q, q)];
                const double2 c = idx == q ? make_double2(1.0, 0.0) : X[tri(idx, q)];
                const double den = p.x * p.x + p.y * p.y;
                bad |= bad_pivot(den);
                const double u = im ? c.y : c.x, v = im ? -c.x : c.y;
                const double d = fma(u, p.x, v * p.y) * pivot_rcp(den);
                reinterpret_cast<double*>(ds + idx)[im] = d;
                reinterpret_cast<double*>(Y + tri(idx, q))[im] = idx == q ? -d : d;
            }
            const int i = i0 + (i0 >= q), j = j0 + (j0 >= q);
            const double2 ci = X[tri(i, q)], a = X[tri(i, j)];
            barrier();
            const double2 dj = ds[j];
            if (own)
                Y[tri(i, j)] = make_double2(fma(-ci.x, dj.x, fma(ci.y, dj.y, a.x)), fma(-ci.x, dj.y, fma(-ci.y, dj.x, a.y)));
            barrier();
        }
        if (bad && lane == 0) atomicOr(status, kStatusSingular);
        const double2* X = nb & 1 ? XB : XA;
        for (int e = tid; e < kBlkP * kBlkP; e += 128) {
            const int i = e / kBlkP, k = e % kBlkP;
            if (k <= i && i < nb) *at(i, k) = X[i * kBlkLd + k];
        }
        // digits of P = -X, eight lanes per column, two rows each
        const int col = tid >> 3;
        double2 x[2];
        int emax = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = (tid & 7) + 8 * h;
            const double2 y = X[k > col ? k * kBlkLd + col : col * kBlkLd + k];
            x[h] = k < nb && col < nb ? make_double2(-y.x, -y.y) : make_double2(0.0, 0.0);
            emax = max(emax, expo_bits(x[h]));
        }
#pragma unroll
        for (int o = 1; o < 8; o *= 2) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
        barrier();  // X may be P's own storage
#pragma unroll
        for (int h = 0; h < 2; ++h) Pd[((tid & 7) + 8 * h) * kBlkLd + col] = fix_digits2<kFix3>(x[h], emax >> 20);
        if ((tid & 7) == 0) Pe[col] = fix_expo<kFix3>(emax >> 20);
    };
    __syncthreads();
    if (warp < 4) pivot(0);
    __syncthreads();
    for (int t = 0; t < nt; ++t) {
        const int w8 = min(2, nb8 - 2 * t), kw = 8 * w8, m8 = nb8 - w8, m = 8 * m8;
        // digits of the pivot column: panel row `row` is matrix row row (above the pivot) or
        // row + kw; two threads per row
        if (tid == 0) ctr[0] = 0;
        for (int r0 = warp * 16; r0 < m; r0 += nw * 16) {
            const int row = r0 + (lane & 15), kh = lane >> 4;
            const int I = row >> 3, Ig = I < 2 * t ? I : I + w8, r = row & 7;
            double2 v[kBlkP / 2];
            int emax = 0;
#pragma unroll
            for (int k = 0; k < kBlkP / 2; ++k) {
                v[k] = make_double2(0.0, 0.0);
                if (row < m && 2 * k < kw) {
                    const int kk = 2 * k + kh, K = 2 * t + (kk >> 3);
                    v[k] = Ig < K ? blk(K, Ig)[r * 8 + (kk & 7)] : blk(Ig, K)[(kk & 7) * 8 + r];
                }
                emax = max(emax, expo_bits(v[k]));
            }
            emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16)) >> 20;
            if (row < m) {
#pragma unroll
                for (int k = 0; k < kBlkP / 2; ++k)
                    if (2 * k < kw) Cd[(2 * k + kh) * R + row] = fix_digits2<kFix3>(v[k], emax);
                if (kh == 0) Ce[row] = fix_expo<kFix3>(emax);
            }
        }
        __syncthreads();
        // W = C P, eight rows of W per warp; the pivot column becomes W (its old values stay in C)
        for (int u = warp; u < m8; u += nw) {
            const int row = u * 8 + r8, Ig = u < 2 * t ? u : u + w8;
            Fix3Sum c[4] = {};
#pragma unroll 2
            for (int k = 0; k < kw; ++k) {
                const int4 a = Cd[k * R + row];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (4 * q < kw) fix3_mac(c[q], a, Pd[k * kBlkLd + cq + 4 * q]);
            }
            double2 w[4];
            int emax = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                w[q] = make_double2(0.0, 0.0);
                if (4 * q < kw) w[q] = fix3_value(c[q], Ce[row] + Pe[cq + 4 * q]);
                emax = max(emax, expo_bits(w[q]));
            }
            emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 8));
            emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16)) >> 20;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (4 * q >= kw) continue;
                const int k = cq + 4 * q, K = 2 * t + (k >> 3);
                Wd[k * R + row] = fix_digits2<kFix3>(w[q], emax);
                (Ig < K ? blk(K, Ig)[r8 * 8 + (k & 7)] : blk(Ig, K)[(k & 7) * 8 + r8]) = w[q];
            }
            if (cq == 0) We[row] = fix_expo<kFix3>(emax);
        }
        __syncthreads();
        // A_IJ -= W_I C_J^T for the row blocks 2 I16, 2 I16 + 1 and column block J, one unit per warp
        auto update = [&](int I16, int J) {
            const int I0 = 2 * I16, shift = I0 < 2 * t ? 0 : w8;
            const bool lo = J <= I0, hi = I0 + 1 < nb8;
            const int row = (I0 - shift) * 8 + r8, col = (J < 2 * t ? J : J - w8) * 8 + cq;
            Fix3Sum c[2][2] = {};
            if (lo && hi) {
#pragma unroll 2
                for (int k = 0; k < kw; ++k) {
                    const int4 a0 = Wd[k * R + row], a1 = Wd[k * R + row + 8];
                    const int4 b0 = Cd[k * R + col], b1 = Cd[k * R + col + 4];
                    fix3_mac(c[0][0], a0, b0);
                    fix3_mac(c[0][1], a0, b1);
                    fix3_mac(c[1][0], a1, b0);
                    fix3_mac(c[1][1], a1, b1);
                }
            } else {
                const int r = lo ? row : row + 8, g = lo ? 0 : 1;
                Fix3Sum c0{}, c1{};
#pragma unroll 2
                for (int k = 0; k < kw; ++k) {
                    const int4 a = Wd[k * R + r];
                    fix3_mac(c0, a, Cd[k * R + col]);
                    fix3_mac(c1, a, Cd[k * R + col + 4]);
                }
                if (g == 0) c[0][0] = c0, c[0][1] = c1;
                else c[1][0] = c0, c[1][1] = c1;
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                if (g == 0 ? !lo : !hi) continue;
                double2* dst = blk(I0 + g, J);
                const int ea = We[row + 8 * g];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const double2 p = fix3_value(c[g][q], ea + Ce[col + 4 * q]);
                    double2& v = dst[(cq + 4 * q) * 8 + r8];
                    v = make_double2(v.x - p.x, v.y - p.y);
                }
            }
        };
        // the next pivot block is updated first, in six 8 x 4 pieces over the warps, and the first four
        // warps invert it while the others update the rest
        const bool ahead = t + 1 < nt;
        if (ahead) {
            const int N0 = 2 * t + 2;
            for (int u = warp; u < 6; u += nw) {
                const int I = N0 + (u >= 2), J = N0 + (u >= 4);  // (0,0) (1,0) (1,1) of the pivot block
                if (I >= nb8) continue;
                const int row = (I - w8) * 8 + r8, c4 = cq + 4 * (u & 1), col = (J - w8) * 8 + c4;
                Fix3Sum c{};
#pragma unroll 2
                for (int k = 0; k < kw; ++k) fix3_mac(c, Wd[k * R + row], Cd[k * R + col]);
                const double2 p = fix3_value(c, We[row] + Ce[col]);
                double2& v = blk(I, J)[c4 * 8 + r8];
                v = make_double2(v.x - p.x, v.y - p.y);
            }
            __syncthreads();
            if (warp < 4) pivot(t + 1);
        }
        const int cnt = ctr[1];
        while (true) {
            int u = lane == 0 ? atomicAdd(&ctr[0], 1) : 0;
            u = __shfl_sync(0xffffffffu, u, 0);
            if (u >= cnt) break;
            const int I = list[u] >> 8, J = list[u] & 255;
            if (I == t || (J >> 1) == t || (ahead && I == t + 1 && (J >> 1) == t + 1)) continue;
            update(I, J);
        }
        __syncthreads();
    }
    for (int b = warp; b < nb8 * (nb8 + 1) / 2; b += nw) {
        int I = 0;
        while ((I + 1) * (I + 2) / 2 <= b) ++I;
        const int J = b - I * (I + 1) / 2;
        for (int e = lane; e < 64; e += 32) {
            const int i = I * 8 + (e & 7), j = J * 8 + (e >> 3);
            if (i < n && j <= i) A[i + static_cast<int64_t>(j) * ld] = make_double2(-M[b * 64 + e].x, -M[b * 64 + e].y);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Batched complex FP64 GEMM on the CUDA cores: C = alpha op(A) op(B) + beta C for every tile of
// a schedule step, products in fixed point (fixed_point.cuh, three real products per complex one)
// over chunks of 64 inner indices, every chunk added to C in FP64 as soon as it is complete.  One
// CTA of 256 threads per 32 x 32 output tile; a warp has the groups of 8 rows and 4 columns that
// lie 16 apart, 2 x 2 outputs per thread, so that a ragged tile skips its empty groups in all warps
// alike and a tile on the diagonal of a lower-triangle result those above it; operands are staged
// by cp.async and turned into digits in place, four threads per operand row.
//
// Full tiles are bound by the multiply-adds (heavy FMA pipe 74% busy at 64-wide pivots, 5.1 TF
// counting 8 operations per complex product); fronts of 36-44 columns, whose second tile is nearly empty,
// by latency (49%), which is why sums are added to memory and not kept in registers: 80 registers
// and three CTAs per SM instead of 124 and two, 15.5 -> 14.8 ms for 80 poles of a 2D sheet of 32 x 32
// atoms x 4 orbitals, at 8.0 -> 8.3 ms for 8 points of a 9 x 8 x 7 box x 5.  Four products per complex one
// in chunks of 32 took 16.7 and 9.9 ms, DFMA loops 44.2 and 23.5 ms.
template <int OP>
__device__ __forceinline__ int64_t op_offset(int ld, int r, int c) {
    if (OP == OP_N) return r + static_cast<int64_t>(c) * ld;
    if (OP == OP_T) return c + static_cast<int64_t>(r) * ld;
    const int hi = r > c ? r : c, lo = r > c ? c : r;
    return hi + static_cast<int64_t>(lo) * ld;
}

constexpr int kFixThreads = 256;
using FixTile = int4[kFix3K][kGemmTile + 1];  // op(A) rows or op(B) columns: raw FP64, then digits
constexpr int kFixSmem = 2 * static_cast<int>(sizeof(FixTile));

// kc inner products of a thread's outputs (row + 16 i, col + 16 j); bit 2 i + j of `live`: the group has a
// wanted output (FULL: all have).
template <bool FULL>
__device__ __forceinline__ void fix_products(const int4 (*As)[kGemmTile + 1], const int4 (*Bs)[kGemmTile + 1], int kc,
                                             int row, int col, uint32_t live, Fix3Sum (&c)[2][2]) {
#pragma unroll 1
    for (int k = 0; k < kc; ++k) {
        const int4 b[2] = {Bs[k][col], Bs[k][col + 16]};
        const int2 bs[2] = {fix3_sum(b[0]), fix3_sum(b[1])};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int4 a = As[k][row + 16 * i];  // re h, re l, im h, im l
            const int2 as = fix3_sum(a);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (FULL || (live >> (2 * i + j) & 1)) fix3_mac(c[i][j], a, as, b[j], bs[j]);
        }
    }
}

template <int OPA, int OPB>
__global__ void __launch_bounds__(kFixThreads, 3)
    k_gemm_f64(const GemmItem* __restrict__ items, const GemmTile* __restrict__ tiles, int64_t tfirst, int64_t ifirst,
               const double2* __restrict__ Abuf, int64_t sA, const double2* __restrict__ Bbuf, int64_t sB,
               double2* __restrict__ Cbuf, int64_t sC, double alpha, double beta, int lower) {
    extern __shared__ __align__(16) unsigned char fix_smem[];
    FixTile* sh = reinterpret_cast<FixTile*>(fix_smem);
    __shared__ int ex[2][kGemmTile];
    const GemmTile t = tiles[tfirst + blockIdx.x];
    const GemmItem it = items[ifirst + t.item];
    const int64_t pole = blockIdx.y;
    const double2* A = Abuf + pole * sA + it.a_off;
    const double2* B = Bbuf + pole * sB + it.b_off;
    double2* C = Cbuf + pole * sC + it.c_off;
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int mrem = min(kGemmTile, it.M - t.m0), nrem = min(kGemmTile, it.N - t.n0);
    const int r0 = (warp / 4) * 8, c0 = (warp % 4) * 4;  // the warp's first row and column
    const int row = r0 + lane % 8, col = c0 + lane / 8;
    uint32_t live = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (r0 + 16 * i < mrem && c0 + 16 * j < nrem && !(lower && t.m0 + r0 + 16 * i + 7 < t.n0 + c0 + 16 * j))
                live |= 1u << (2 * i + j);
    for (int k0 = 0; k0 < it.K; k0 += kFix3K) {
        const int kc = min(kFix3K, it.K - k0);
        auto stage = [&](int4* dst, const double2* src, bool ok) {
            const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
        };
#pragma unroll
        for (int u = 0; u < kGemmTile * kFix3K / kFixThreads; ++u) {
            const int g = warp + u % 4 * 8, f = lane + u / 4 * 32;  // for the operand that is contiguous in k
            const int w = warp + u * 8;
            const int m = OPA == OP_T ? g : lane, ka = OPA == OP_T ? f : w;
            if (ka < kc) stage(&sh[0][ka][m], A + (m < mrem ? op_offset<OPA>(it.lda, t.m0 + m, k0 + ka) : 0), m < mrem);
            const int n = OPB == OP_T ? lane : g, kb = OPB == OP_T ? w : f;
            if (kb < kc) stage(&sh[1][kb][n], B + (n < nrem ? op_offset<OPB>(it.ldb, k0 + kb, t.n0 + n) : 0), n < nrem);
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        {
            // four threads per operand row: the largest exponent field of the chunk, then the
            // digits in place
            int4 (*x)[kGemmTile + 1] = sh[warp / 4];
            const int rr = (warp % 4) * 8 + lane % 8, kh = lane / 8;
            int emax = 0;
#pragma unroll 4
            for (int u = 0; u < kFix3K / 4; ++u) {
                const int k = kh + 4 * u;
                if (k < kc) emax = max(emax, max(x[k][rr].y & 0x7FF00000, x[k][rr].w & 0x7FF00000));
            }
            emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 8));
            emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16)) >> 20;
#pragma unroll 4
            for (int u = 0; u < kFix3K / 4; ++u) {
                const int k = kh + 4 * u;
                if (k < kc) x[k][rr] = fix_digits2<kFix3>(*reinterpret_cast<const double2*>(&x[k][rr]), emax);
            }
            if (kh == 0) ex[warp / 4][rr] = fix_expo<kFix3>(emax);
        }
        __syncthreads();
        if (live) {
            Fix3Sum c[2][2] = {};
            if (live == 15u) fix_products<true>(sh[0], sh[1], kc, row, col, live, c);
            else fix_products<false>(sh[0], sh[1], kc, row, col, live, c);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int m = t.m0 + row + 16 * i, n = t.n0 + col + 16 * j;
                    if (m >= it.M || n >= it.N || (lower && m < n)) continue;
                    double2 v = fix3_value(c[i][j], ex[0][row + 16 * i] + ex[1][col + 16 * j]);
                    if (alpha == -1.0) v = make_double2(-v.x, -v.y);
                    else if (alpha != 1.0) v = make_double2(alpha * v.x, alpha * v.y);
                    const double b = k0 == 0 ? beta : 1.0;
                    double2* out = C + m + static_cast<int64_t>(n) * it.ldc;
                    if (b != 0.0) {
                        const double2 old = *out;
                        if (b == 1.0) v = cadd(v, old);
                        else v = make_double2(fma(b, old.x, v.x), fma(b, old.y, v.y));
                    }
                    *out = v;
                }
        }
        __syncthreads();
    }
}

// dst = scale * src for the blocks of a step (SCR -> FRONT).
__global__ void __launch_bounds__(256) k_copy(const CopyItem* __restrict__ items, int64_t first,
                                              const double2* __restrict__ src, int64_t s_src,
                                              double2* __restrict__ dst, int64_t s_dst, double scale) {
    const CopyItem c = items[first + blockIdx.x];
    const double2* S = src + static_cast<int64_t>(blockIdx.y) * s_src + c.src_off;
    double2* D = dst + static_cast<int64_t>(blockIdx.y) * s_dst + c.dst_off;
    // the block's rows x cols elements (column-major, < 2^31) in gridDim.z contiguous ranges, so
    // that short columns still occupy every thread
    const uint32_t rows = static_cast<uint32_t>(c.rows);
    const uint32_t total = rows * static_cast<uint32_t>(c.cols);
    const uint32_t per = (total + gridDim.z - 1) / gridDim.z;
    const uint32_t e0 = blockIdx.z * per, e1 = min(total, e0 + per);
#pragma unroll 4
    for (uint32_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        const uint32_t j = e / rows, i = e - j * rows;
        const double2 v = S[i + static_cast<int64_t>(j) * c.lds];
        D[i + static_cast<int64_t>(j) * c.ldd] = make_double2(scale * v.x, scale * v.y);
    }
}

// G_RR of a node from the full (lower-valid) G front of its parent (Eq. 38's reuse of
// ancestor blocks), through the node's relative index map.
__global__ void __launch_bounds__(256) k_gather(const NodeDev* __restrict__ nodes,
                                                const NodeTile* __restrict__ tiles, int64_t first,
                                                const int32_t* __restrict__ rel_map,
                                                double2* __restrict__ F, int64_t stride) {
    constexpr int kCols = kNodeTile / 8;  // a thread's four loads are in flight together
    const NodeTile t = tiles[first + blockIdx.x];
    const NodeDev& nd = nodes[t.node];
    const NodeDev& pd = nodes[nd.parent];
    const int i = t.i0 + threadIdx.x;
    if (i >= nd.r) return;
    const int64_t row = pd.front_off + rel_map[nd.rel_off + i], dst = nd.front_off + nd.s + i;
    const int j0 = t.j0 + threadIdx.y;
    double2* Fp = F + static_cast<int64_t>(blockIdx.y) * stride;
    double2 v[kCols];
#pragma unroll
    for (int u = 0; u < kCols; ++u)
        if (j0 + 8 * u <= i) v[u] = Fp[row + static_cast<int64_t>(rel_map[nd.rel_off + j0 + 8 * u]) * pd.f];
#pragma unroll
    for (int u = 0; u < kCols; ++u)
        if (j0 + 8 * u <= i) Fp[dst + static_cast<int64_t>(nd.s + j0 + 8 * u) * nd.f] = v[u];
}

// Residue sum of Eq. 8 on the pattern: rho_k (+)= sum_q Re(c_q G_q(k)); per-block partial sums
// of rho_k S_k for Tr(rho S) (Eq. 40), reduced in a fixed order by k_reduce.
constexpr int kAccThreads = 256;

__global__ void __launch_bounds__(kAccThreads) k_accumulate(const int64_t* __restrict__ out_map,
                                                            const int16_t* __restrict__ pair,
                                                            int64_t k0, int64_t nnz,
                                                            const double2* __restrict__ F,
                                                            int64_t stride, int np,
                                                            const double2* __restrict__ c,
                                                            const double* __restrict__ S,
                                                            double* __restrict__ rho, int accumulate,
                                                            int want_trace,
                                                            double* __restrict__ partials) {
    __shared__ double red[kAccThreads / 32];
    const int64_t k = k0 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    double tr = 0.0;
    if (k < k0 + nnz) {
        const int64_t off = out_map[k];
        const int pe = pair[k];
        double sum = accumulate ? scale2(rho[k], -pe) : 0.0;
        for (int q = 0; q < np; ++q) {
            const double2 g = F[static_cast<int64_t>(q) * stride + off];
            const double2 w = c[q];
            sum = fma(w.x, g.x, fma(-w.y, g.y, sum));
        }
        sum = scale2(sum, pe);
        rho[k] = sum;
        tr = sum * S[k];
    }
    if (!want_trace) return;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_down_sync(0xffffffffu, tr, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = tr;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < kAccThreads / 32 ? red[threadIdx.x] : 0.0;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) partials[blockIdx.x] = v;
    }
}

__global__ void __launch_bounds__(1024) k_reduce(const double* __restrict__ partials, int n,
                                                 double* __restrict__ out) {
    __shared__ double red[32];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v += partials[i];
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double w = threadIdx.x < (blockDim.x + 31) / 32 ? red[threadIdx.x] : 0.0;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
        if (threadIdx.x == 0) *out = w;
    }
}

__global__ void __launch_bounds__(256) k_gather_pattern(const int64_t* __restrict__ out_map,
                                                        const int16_t* __restrict__ pair,
                                                        int64_t nnz,
                                                        const double2* __restrict__ F,
                                                        int64_t stride, double2* __restrict__ G,
                                                        int64_t q0) {
    const int64_t q = blockIdx.y;
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const double2 g = F[q * stride + out_map[k]];
        const int pe = pair[k];
        G[(q0 + q) * nnz + k] = make_double2(scale2(g.x, pe), scale2(g.y, pe));
    }
}

// Tiles x poles of the assembly: a block keeps its tile's indices for several poles when there are enough
// blocks all the same (eight rounds of five per SM).
dim3 node_grid(int64_t tiles, int np) {
    const int64_t want = (8 * 5 * 152 + tiles - 1) / tiles;
    return dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(std::min<int64_t>(np, std::max<int64_t>(want, 1))));
}

template <int OPA, int OPB>
cudaError_t gemm_launch(const Plan& P, const DevTables& T, const Launch& l, const Workspace& W,
                        int np, cudaStream_t st) {
    const double2* bufs[2] = {W.fronts, W.scr};
    const int64_t strides[2] = {W.front_stride, W.scr_stride};
    dim3 grid(static_cast<unsigned>(l.tcount), static_cast<unsigned>(np));
    k_gemm_f64<OPA, OPB><<<grid, kFixThreads, kFixSmem, st>>>(
        T.gemm_items, T.gemm_tiles, l.tfirst, l.first, bufs[l.bufA], strides[l.bufA], bufs[l.bufB],
        strides[l.bufB], const_cast<double2*>(bufs[l.bufC]), strides[l.bufC], l.alpha, l.beta, l.lower);
    (void)P;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_step(const Plan& P, const DevTables& T, const Launch& l, const Workspace& W,
                        const double* H, const double* S, const double2* z, int64_t zstride, int np,
                        cudaStream_t st) {
    switch (l.kind) {
        case L_ASSEMBLE: {
            k_assemble<<<node_grid(l.count, np), dim3(32, 8), 0, st>>>(T.nodes, T.node_tiles, l.first, T.inv_map, W.fronts,
                                                                      W.front_stride, np);
            return cudaGetLastError();
        }
        case L_SCATTER: {
            const int64_t blocks = (l.count + 255) / 256;
            dim3 grid(static_cast<unsigned>(blocks < 4096 ? blocks : 4096), static_cast<unsigned>(np));
            k_scatter<<<grid, 256, 0, st>>>(T.scatter_idx, l.first, l.count, T.asm_map, T.entry_sys, H, S,
                                            W.scale.pair, z, zstride, W.fronts, W.front_stride);
            return cudaGetLastError();
        }
        case L_DIAGINV: {
            if (l.fused) {
                k_diaginv_block<<<dim3(static_cast<unsigned>(l.count), static_cast<unsigned>(np)), diag_block_threads(l.tile),
                                  diag_block_smem(l.tile), st>>>(T.diag_items, l.first, W.fronts, W.front_stride, T.status,
                                                                 l.tile);
                return cudaGetLastError();
            }
            dim3 grid(static_cast<unsigned>(l.count), static_cast<unsigned>(np));
            const int b = P.block;
            const size_t sm = static_cast<size_t>(b) * (b + 1) * sizeof(double2);
            if (b <= 32) {
                if (l.tile == 16)
                    k_diaginv_sweep<16><<<grid, 32, 0, st>>>(T.diag_items, l.first, W.fronts, W.front_stride, T.status);
                else
                    k_diaginv_sweep<32><<<grid, 32, 0, st>>>(T.diag_items, l.first, W.fronts, W.front_stride, T.status);
            } else {
                k_diaginv<64><<<grid, 256, sm, st>>>(T.diag_items, l.first, W.fronts, W.front_stride, T.status);
            }
            return cudaGetLastError();
        }
        case L_GEMM: {
            if (l.opA == OP_N && l.opB == OP_S) return gemm_launch<OP_N, OP_S>(P, T, l, W, np, st);
            if (l.opA == OP_N && l.opB == OP_T) return gemm_launch<OP_N, OP_T>(P, T, l, W, np, st);
            if (l.opA == OP_S && l.opB == OP_N) return gemm_launch<OP_S, OP_N>(P, T, l, W, np, st);
            if (l.opA == OP_T && l.opB == OP_N) return gemm_launch<OP_T, OP_N>(P, T, l, W, np, st);
            return cudaErrorInvalidValue;
        }
        case L_COPY: {
            // column slices per item: launches of few items (the upper tree levels) would
            // otherwise leave most SMs idle
            const unsigned zc = l.count * np < 4 * 152 ? 32u : 8u;
            dim3 grid(static_cast<unsigned>(l.count), static_cast<unsigned>(np), zc);
            k_copy<<<grid, 256, 0, st>>>(T.copy_items, l.first, W.scr, W.scr_stride, W.fronts, W.front_stride,
                                         l.alpha);
            return cudaGetLastError();
        }
        case L_GATHER: {
            dim3 grid(static_cast<unsigned>(l.count), static_cast<unsigned>(np));
            k_gather<<<grid, dim3(32, 8), 0, st>>>(T.nodes, T.node_tiles, l.first, T.rel_map, W.fronts,
                                                  W.front_stride);
            return cudaGetLastError();
        }
        default:
            return cudaErrorInvalidValue;
    }
}

cudaError_t launch_basis_scale(const Plan& P, const DevTables& T, const double* H, const double* S, const double2* z,
                               int64_t zstride, int nz, const Workspace& W, cudaStream_t st) {
    const unsigned grid = static_cast<unsigned>((P.n + kScaleRows - 1) / kScaleRows);
    constexpr int threads = 32 * kScaleRows;
    k_scale_start<<<grid, threads, 0, st>>>(T.rowptr, T.col, T.diag, T.entry_sys, P.n, H, S, z, zstride, nz, P.n_systems,
                                            W.scale);
    k_scale_step<true><<<grid, threads, 0, st>>>(T.rowptr, T.col, T.diag, T.entry_sys, P.n, H, S, W.scale);
    k_scale_step<false><<<grid, threads, 0, st>>>(T.rowptr, T.col, T.diag, T.entry_sys, P.n, H, S, W.scale);
    k_pair_scale<<<grid, threads, 0, st>>>(T.rowptr, T.col, T.diag, T.entry_sys, P.n, W.scale);
    return cudaGetLastError();
}

cudaError_t kernels_init() {
    using Gemm = decltype(&k_gemm_f64<OP_N, OP_S>);
    for (Gemm f : {&k_gemm_f64<OP_N, OP_S>, &k_gemm_f64<OP_N, OP_T>, &k_gemm_f64<OP_S, OP_N>, &k_gemm_f64<OP_T, OP_N>}) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kFixSmem);
        if (e != cudaSuccess) return e;
    }
    const int smb = static_cast<int>(diag_block_smem(kDiagBlockMax));
    const cudaError_t e = cudaFuncSetAttribute(k_diaginv_block, cudaFuncAttributeMaxDynamicSharedMemorySize, smb);
    if (e != cudaSuccess) return e;
    const int sm64 = 64 * 65 * static_cast<int>(sizeof(double2));
    return cudaFuncSetAttribute(k_diaginv<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm64);
}

int accumulate_blocks(int64_t nnz) { return static_cast<int>((nnz + kAccThreads - 1) / kAccThreads); }

cudaError_t launch_accumulate(const Plan& P, const DevTables& T, const Workspace& W, int np,
                              const double2* c, const double* S, double* rho, int accumulate,
                              int want_trace, double* partials, cudaStream_t st, int64_t k0, int64_t count) {
    if (count < 0) {
        k0 = 0;
        count = P.nnz;
    }
    const int blocks = accumulate_blocks(count);
    k_accumulate<<<blocks, kAccThreads, 0, st>>>(T.out_map, W.scale.pair, k0, count, W.fronts, W.front_stride, np, c, S, rho,
                                                 accumulate, want_trace, partials);
    return cudaGetLastError();
}

// Order-preserving map of doubles to unsigned keys (larger double -> larger key).
__host__ __device__ inline unsigned long long order_key(double x) {
    unsigned long long u;
    memcpy(&u, &x, sizeof(u));
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__global__ void __launch_bounds__(256) k_gershgorin(const int64_t* __restrict__ rowptr,
                                                    const int32_t* __restrict__ col, int64_t n,
                                                    const double* __restrict__ H,
                                                    const double* __restrict__ S,
                                                    unsigned long long* __restrict__ out) {
    const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    double h = 0.0, soff = 0.0, sdiag = 0.0;
    for (int64_t k = rowptr[i]; k < rowptr[i + 1]; ++k) {
        h += fabs(H[k]);
        if (col[k] == i) sdiag = S[k];
        else soff += fabs(S[k]);
    }
    atomicMax(&out[0], order_key(h));
    atomicMax(&out[1], order_key(soff - sdiag));
}

cudaError_t launch_gershgorin(const DevTables& T, int64_t n, const double* H, const double* S,
                              unsigned long long* out, cudaStream_t st) {
    const unsigned blocks = static_cast<unsigned>((n + 255) / 256);
    k_gershgorin<<<blocks, 256, 0, st>>>(T.rowptr, T.col, n, H, S, out);
    return cudaGetLastError();
}

double gershgorin_value(unsigned long long key) {
    const unsigned long long u = (key >> 63) ? (key & 0x7FFFFFFFFFFFFFFFull) : ~key;
    double x;
    memcpy(&x, &u, sizeof(x));
    return x;
}

__global__ void __launch_bounds__(kAccThreads) k_point_traces(const int64_t* __restrict__ out_map,
                                                              const int16_t* __restrict__ pair, int64_t nnz,
                                                              const double2* __restrict__ F, int64_t stride,
                                                              const double* __restrict__ S,
                                                              double* __restrict__ partials) {
    __shared__ double red[kAccThreads / 32];
    const int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    double v = 0.0;
    if (k < nnz) v = scale2(F[static_cast<int64_t>(blockIdx.y) * stride + out_map[k]].y, pair[k]) * S[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double w = threadIdx.x < kAccThreads / 32 ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
        if (threadIdx.x == 0) partials[static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x] = w;
    }
}

cudaError_t launch_point_traces_range(const int64_t* out_map, const int16_t* pair, int64_t nnz, const double2* F,
                                      int64_t stride, int np, const double* S, double* partials, double* out,
                                      cudaStream_t st) {
    if (nnz <= 0 || np <= 0) return cudaSuccess;
    const int nb = accumulate_blocks(nnz);
    k_point_traces<<<dim3(static_cast<unsigned>(nb), static_cast<unsigned>(np)), kAccThreads, 0, st>>>(
        out_map, pair, nnz, F, stride, S, partials);
    cudaError_t e = cudaGetLastError();
    for (int q = 0; q < np && e == cudaSuccess; ++q) {
        k_reduce<<<1, 1024, 0, st>>>(partials + static_cast<int64_t>(q) * nb, nb, out + q);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_reduce(const double* partials, int nblocks, double* out, cudaStream_t st) {
    k_reduce<<<1, 1024, 0, st>>>(partials, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_gather_pattern(const Plan& P, const DevTables& T, const Workspace& W, int np,
                                  double2* G_out, int64_t q0, cudaStream_t st) {
    const int64_t blocks = (P.nnz + 255) / 256;
    dim3 grid(static_cast<unsigned>(blocks < 2048 ? blocks : 2048), static_cast<unsigned>(np));
    k_gather_pattern<<<grid, 256, 0, st>>>(T.out_map, W.scale.pair, P.nnz, W.fronts, W.front_stride, G_out, q0);
    return cudaGetLastError();
}

}  // namespace ndsi
