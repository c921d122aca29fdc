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
    int64_t* rowptr = nullptr;   // CSR pattern (original order), for the moment features
    int32_t* col = nullptr;
    int* status = nullptr;
    void* blob = nullptr;  // single allocation holding all of the above
};

// Pole-batched workspace: `np` slabs of fronts and of scratch.
struct Workspace {
    double2* fronts = nullptr;
    double2* scr = nullptr;
    int64_t front_stride = 0;   // complex elements per pole slab
    int64_t scr_stride = 0;
    int32_t np_cap = 0;         // poles the buffers hold
    // Power-of-two scaling of the basis functions the fronts were assembled with (part of the fronts'
    // allocation): exponent f_i per basis function, f_i + f_j per pattern entry, any f_i != 0.
    int16_t* scale_f = nullptr;
    int16_t* scale_pair = nullptr;
    int* scale_any = nullptr;
};

// Bytes of the scaling tables behind the fronts.
inline size_t scale_bytes(const Plan& P) { return 256 + sizeof(int16_t) * static_cast<size_t>(P.n + P.nnz); }

// Fill the scaling tables of W from the diagonal of S (values on the pattern): 2^f_i brings S_ii into
// [1/2, 2).  The fronts hold D (z S - H) D with D = diag(2^f_i), exactly, and so D^{-1} G D^{-1}: a
// basis whose functions are normalised very differently does not leave rows of mixed scale for the
// fixed-point and split products.  Outputs take the pair exponents (solves the row exponents) again.
cudaError_t launch_basis_scale(const Plan& P, const DevTables& T, const double* S, const Workspace& W, cudaStream_t st);

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

// Per point q of a chunk: out[q] = sum over the pattern of Im G_q(k) S_k = Im Tr(G(z_q) S) (the
// density of states of Eq. 42 up to -2/pi).  partials: np x accumulate_blocks(nnz) doubles.
// The same over one range of pattern entries (out_map and S offset to its first entry; F holds np
// point slabs of `stride` complex elements): out[q] = sum_k Im F_q[out_map[k]] 2^pair[k] S[k].
cudaError_t launch_point_traces_range(const int64_t* out_map, const int16_t* pair, int64_t nnz, const double2* F,
                                      int64_t stride, int np, const double* S, double* partials, double* out,
                                      cudaStream_t st);
cudaError_t launch_point_traces(const Plan& P, const DevTables& T, const Workspace& W, int np,
                                const double* S, double* partials, double* out, cudaStream_t st);

// G_out[q*nnz + k] = G_q(k) for the np poles of the workspace.
cudaError_t launch_gather_pattern(const Plan& P, const DevTables& T, const Workspace& W, int np,
                                  double2* G_out, int64_t q0, cudaStream_t st);

}  // namespace ndsi
