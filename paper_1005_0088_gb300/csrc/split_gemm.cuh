// Split-precision (emulated FP64) complex GEMM on the tcgen05 tensor cores.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <vector>

#include "plan.hpp"

namespace ndsi {

// Tile of the split GEMM: 128 output rows x NC complex output columns.  Default: one TMEM
// accumulator per slice-product scale t+u (S of them, S x 2NC <= 512 columns: NC = 40 for up to
// six slices, 32 for seven), filled by one wide MMA per A digit.  Optional: NC = 64 with four
// accumulators (t+u = 2, 3, 4 exact, the rest in a tail) or NC = 48 with five (t+u = 2..5 exact).
constexpr int kSplitBM = 128;
constexpr int kSplitBNc = 64;      // complex columns per tile, four-band variant
constexpr int kSplitBNc5 = 48;     // complex columns per tile, five-band variant
constexpr int kSplitBNcX = 40;     // complex columns per tile, one accumulator per scale (S <= 6)
constexpr int kSplitBNcX7 = 32;    // the same for seven slices
// Complex columns per tile of a plan: bands 4 or 5 select the tail variants, 0 one accumulator
// per scale.
constexpr int split_nc(int slices, int bands) {
    return bands == 4 ? kSplitBNc : bands == 5 ? kSplitBNc5 : (slices >= 7 ? kSplitBNcX7 : kSplitBNcX);
}
constexpr int kSplitSliceRows = 32;  // operand rows per slicing block (two-pass slicer)
constexpr int kSplitSlice1Smem = 72 * 1024;       // one-pass slicer budget, 4..32 rows per block
constexpr int kSplitSlice1SmemWide = 200 * 1024;  // budget for very long rows, 1 or 2 rows per block
constexpr int kSplitKB = 32;       // complex K padding: the stacked K (2 Kpad) is a multiple of kSplitStageK
constexpr int kSplitStageK = 64;   // stacked K per pipeline block: 64 BF16 (128-byte rows, 128-byte swizzle)
constexpr int kSplitChunkKB = 256 / kSplitStageK;  // blocks per exact chunk (256 stacked-K elements)
constexpr int kSplitMaxSlices = 7;
// Bytes of one operand's slices a tile group may keep in L2 while the other operand streams
// (a third of GB300's 126 MB L2), and the tiles the persistent GEMM runs at one time (one CTA on
// each of GB300's 152 SMs).
constexpr double kSplitL2Share = 40.0 * 1024 * 1024;
constexpr int kSplitConcurrentTiles = 152;
// Default of ndsi_options.split_far_ratio: density-sweep poles with z_p >= 32 z_1 use one slice
// fewer (32^2 ~ 2^10 covers the 2^8 larger product error of the shorter expansion).
constexpr double kSplitFarRatio = 32.0;

// Where an item's slices and exponents live inside one pole's block of the step buffers.
struct SplitItem {
    int64_t rowA, rowB;     // first slice row of the item's operand (digit t at row + t Mpad, + t Npad)
    int64_t erowA, erowB;   // first exponent of the item
    int32_t Mpad, Npad;     // slice rows per digit: at least the tiles' 128 rows, nc complex columns
    int32_t Kpad, pad;      // multiple of kSplitKB (complex K); stacked K is 2*Kpad
};

// Slices of one operand of a step.  A slice row holds the digits of one row of op(A) or column of op(B):
// parts [Re | Im] of Kpad elements each, and [Re | Im | -Im] for a B operand, whose real and imaginary
// output columns take (Re, -Im) and (Im, Re) of the same rows against A's (Re, Im).
struct SplitOperand {
    int64_t rows, erows;                   // per pole
    int32_t Kcols;                         // row length of the slice buffer
    int32_t parts;                         // 2 or 3
    int32_t buf;                           // slice buffer 0 or 1
    int32_t shared;                        // rows are those of the previous launch's other operand
    int64_t first, count;                  // slicing blocks in the block list
};

// Per GEMM launch: sizes of one pole's block in the step buffers, and the split tile range.
struct SplitStep {
    SplitOperand A, B;
    int32_t nc;                            // complex columns per output tile (64, 48, 40 or 32)
    int32_t slice_rows;                    // operand rows per slicing block
    int32_t slice_ldt;                     // one-pass slicing: shared-memory row stride (0: two passes)
    int32_t fuse_copy;                     // the next launch copies this step's own sliced operand
    int64_t tfirst, tcount;                // tiles in the split tile list
};

// A slicing block: item (relative to the launch) and its first row (A) or complex column (B).
struct SliceBlock {
    int32_t item, r0;
};

// Build the split metadata of every GEMM launch (called by the analysis in split mode).
// bands[li]: accumulator layout of launch li (0 one per scale, 4 or 5 with a tail).
void build_split_schedule(const Plan& P, int slices, const std::vector<int8_t>& bands,
                          std::vector<SplitItem>& items, std::vector<SplitStep>& steps,
                          std::vector<GemmTile>& tiles, std::vector<SliceBlock>& blocks);

struct SplitBuffers {
    uint16_t* slices[2] = {};     // bf16 bit patterns
    int32_t* expo[2] = {};
    size_t cap[2] = {};           // slice elements
    std::vector<CUtensorMap> tmA, tmB;                // one per split step (for np_cap poles)
    int32_t np = 0;
};

// Slice elements (out[0], out[1]) and exponents (out[2], out[3]) of the two buffers for one pole.
void split_buffer_elements(const std::vector<SplitStep>& steps, int64_t out[4]);
cudaError_t split_init();
// Allocate the slice buffers for np poles and encode the tensor maps of every step.
cudaError_t split_alloc(SplitBuffers& B, const std::vector<SplitStep>& steps, int slices, int np);
void split_free(SplitBuffers& B);

// One GEMM launch of the schedule in split precision: slice A and B (split_slice_step; a shared operand
// only when its slices are not `ready` from the previous launch), then the tensor-core product and
// FP64 epilogue (split_mma_step).  With `copy` the slicer of the operand that is not
// shared also writes it to its place in the fronts (the schedule's next launch, SplitStep::fuse_copy).
struct SplitCopy {
    const CopyItem* items = nullptr;
    double2* dst = nullptr;
    int64_t stride = 0;
    double scale = 1.0;
};
cudaError_t split_slice_step(const Launch& l, const GemmItem* items_dev, const SplitItem* sitems_dev,
                             const SliceBlock* blocks_dev, const SplitStep& step, const SplitBuffers& B,
                             int slices, const double2* Abuf, int64_t sA, const double2* Bbuf, int64_t sB,
                             bool ready, const SplitCopy& copy, int np, cudaStream_t st);
cudaError_t split_mma_step(const Launch& l, int step_index, const GemmItem* items_dev,
                           const SplitItem* sitems_dev, const GemmTile* stiles_dev, const SplitStep& step,
                           const SplitBuffers& B, int slices, double2* Cbuf, int64_t sC, int np, int* status,
                           cudaStream_t st);
// Tensor-core flops one pole of the step issues (tiles x 128 x 128 x 2Kpad x pairs x 2).
double split_executed_flops(const Plan& P, const SplitStep& step, const std::vector<SplitItem>& items,
                            const std::vector<GemmTile>& tiles, const Launch& l, int slices);

}  // namespace ndsi
