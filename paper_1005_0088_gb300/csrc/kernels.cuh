// Device kernels of the FP64 numeric phase (shared declarations).
#pragma once

#include <cuda_runtime.h>

#include "plan.hpp"

namespace ndsi {

// Error bits latched in the device status word.
constexpr int kStatusSingular = 1;
constexpr int kStatusTimeout = 2;
constexpr int kStatusBadItem = 4;  // a schedule item outside what its kernel handles (skipped)

struct DevTables {
    NodeDev* nodes = nullptr;
    int64_t* asm_map = nullptr;
    int64_t* out_map = nullptr;
    int32_t* inv_map = nullptr;
    int32_t* rel_map = nullptr;
    int64_t* scatter_idx = nullptr;
    GemmItem* gemm_items = nullptr;
    GemmTile* gemm_tiles = nullptr;
    CopyItem* copy_items = nullptr;
    DiagItem* diag_items = nullptr;
    NodeTile* node_tiles = nullptr;
    int32_t* entry_sys = nullptr;  // system of each pattern entry
    int64_t* diag = nullptr;       // pattern entry of each row's diagonal
    int64_t* rowptr = nullptr;   // CSR pattern (original order), for the moment features
    int32_t* col = nullptr;
    int* status = nullptr;
    void* blob = nullptr;  // single allocation holding all of the above
};

// Statistics of a system's row scales (biased, so that zero is the empty state).
struct ScaleStat {
    unsigned long long sum;
    int lo, hi;
    unsigned count, pad;
};
// Power-of-two scaling of the basis functions the fronts were assembled with (part of the fronts'
// allocation): exponent f_i per basis function, f_i + f_j per pattern entry, any f_i != 0; the others are
// what they are made from.
struct ScaleTables {
    int* any = nullptr;
    ScaleStat* stat = nullptr;  // per system
    int* g[2] = {};             // row scales
    int16_t* norm = nullptr;    // exponent of S_ii
    int16_t* ez = nullptr;      // exponent of the system's smallest point, per basis function
    int16_t* f = nullptr;
    int16_t* pair = nullptr;
};

// Pole-batched workspace: `np` slabs of fronts and of scratch.
struct Workspace {
    double2* fronts = nullptr;
    double2* scr = nullptr;
    int64_t front_stride = 0;   // complex elements per pole slab
    int64_t scr_stride = 0;
    int32_t np_cap = 0;         // poles the buffers hold
    ScaleTables scale;
};

// Bytes of the scaling tables behind the fronts.
inline size_t scale_bytes(const Plan& P) {
    return 256 + sizeof(ScaleStat) * static_cast<size_t>(P.n_systems) +
           (2 * sizeof(int) + 3 * sizeof(int16_t)) * static_cast<size_t>(P.n) + sizeof(int16_t) * static_cast<size_t>(P.nnz);
}

// Fill the scaling tables of W for H and S (values on the pattern) at nz points per system (z[sys *
// zstride + q]).  The fronts hold D (z S - H) D with D = diag(2^f_i), exactly, and so D^{-1} G D^{-1};
// outputs take the pair exponents (solves the row exponents) again.  The fixed-point and split products
// are exact relative to a row's maximum, so rows of mixed scale would lose what FP64 products keep:
//  * 2^f_i brings S_ii into [1/2, 2), so that basis functions normalised very differently do not matter;
//  * orbitals whose on-site energies or couplings are of another size than the rest (core levels, penalty
//    terms) are brought to the common scale by symmetric equilibration of the normalised |H_ij| + |z S_ij|, z
//    the system's smallest point: the diagonal to 1, then two steps of the maximum norm.  In a model of the
//    elimination (190 orbitals, every 16th one at 10^2 / 10^4 / 10^10 times the others with couplings of its
//    0.4th power) the largest error of G is 4e-14 .. 5e-14 with that, 4e-14 .. 7e-14 with FP64 products and 8e-13 /
//    6e-12 / 1e-9 with S_ii alone.  One table serves all points: far from the spectrum the error is small.
// Systems whose rows lie within 1.5 places below and 2.5 above their mean scale (on-site energies within a
// factor of about eight from the typical one) keep S_ii's exponents: equilibrating them changes the error by no more
// than its spread between inputs (2.2e-14 without, 2.9e-14 with, 4.8e-14 FP64 products, eight inputs).
cudaError_t launch_basis_scale(const Plan& P, const DevTables& T, const double* H, const double* S, const double2* z,
                               int64_t zstride, int nz, const Workspace& W, cudaStream_t st);

// Spectral-moment features of (H, S) for the learned mu seed (mlp.cu).
int mlp_features(const Plan& P, const double* Hd, const double* Sd, const int64_t* rowptr_d,
                 const int32_t* col_d, double n_electrons, double kT, int R, uint64_t seed, float* feat_d,
                 cudaStream_t st);

// One-time kernel attributes (large dynamic shared memory).
cudaError_t kernels_init();

// Launch one schedule step over `np` poles whose slabs start at the workspace base.
// z holds the points of every system: z[sys * zstride + pole].
cudaError_t launch_step(const Plan& P, const DevTables& T, const Launch& l, const Workspace& W,
                        const double* H, const double* S, const double2* z, int64_t zstride, int np,
                        cudaStream_t st);

// rho(k) (+)= sum_q Re(c_q G_q(k)) over the pattern; `partials` receives per-block sums of
// rho(k) S(k) when `want_trace` is set (nblocks = accumulate_blocks(nnz)).
// (entries [k0, k0+count); count < 0 = the whole pattern)
cudaError_t launch_accumulate(const Plan& P, const DevTables& T, const Workspace& W, int np,
                              const double2* c, const double* S, double* rho, int accumulate,
                              int want_trace, double* partials, cudaStream_t st, int64_t k0 = 0,
                              int64_t count = -1);
int accumulate_blocks(int64_t nnz);
cudaError_t launch_reduce(const double* partials, int nblocks, double* out, cudaStream_t st);

// Gershgorin data of (H, S): out[0] = order key of max_i sum_j |H_ij|, out[1] = order key of
// max_i (sum_{j != i} |S_ij| - S_ii); keys decode with gershgorin_value.  out must be zeroed.
cudaError_t launch_gershgorin(const DevTables& T, int64_t n, const double* H, const double* S,
                              unsigned long long* out, cudaStream_t st);
double gershgorin_value(unsigned long long key);

// Per point q of a chunk, over a range of pattern entries (out_map, pair and S offset to its first entry; F holds
// np point slabs of `stride` complex elements): out[q] = sum_k Im F_q[out_map[k]] 2^pair[k] S[k], over a whole
// system Im Tr(G(z_q) S) (the density of states of Eq. 42 up to -2/pi).  partials: np x accumulate_blocks(nnz) doubles.
cudaError_t launch_point_traces_range(const int64_t* out_map, const int16_t* pair, int64_t nnz, const double2* F,
                                      int64_t stride, int np, const double* S, double* partials, double* out,
                                      cudaStream_t st);

// G_out[q*nnz + k] = G_q(k) for the np poles of the workspace.
cudaError_t launch_gather_pattern(const Plan& P, const DevTables& T, const Workspace& W, int np,
                                  double2* G_out, int64_t q0, cudaStream_t st);

}  // namespace ndsi
