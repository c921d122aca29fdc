// Choice between the tensor-core and CUDA-core paths of a split plan's GEMM steps.
#pragma once

#include <cstdint>
#include <vector>

namespace ndsi {

// A GEMM step that may run on either path.  A step that `receives` takes the slices of an operand from
// the step before it in the list, and may write its own operand back in place of the copy launch `copy` (-1:
// none): its time on the tensor cores depends on the path of the step before.
struct TuneStep {
    size_t launch;
    bool receives;
    int64_t copy;
    bool decided;  // the tensor cores are faster than the CUDA cores could be: not timed there
};

// Per launch milliseconds of three sweeps: `split` with every step on the tensor cores, `cuda` with every step but
// the decided ones on the CUDA cores and, when given, `mixed` with the paths in `mixed_use`.  Sets use[launch] of
// every step, pairs that share slices together.  Returns whether a choice rests on a pair (CUDA cores, then tensor
// cores) that was not timed as such: with the paths in `use` as `mixed_use` its sweep settles it.
bool choose_paths(const std::vector<TuneStep>& steps, const std::vector<double>& split, const std::vector<double>& cuda,
                  const std::vector<double>* mixed, const std::vector<char>* mixed_use, std::vector<char>& use,
                  std::vector<double>& tensor_ms);

}  // namespace ndsi
