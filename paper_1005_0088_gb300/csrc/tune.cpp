// Choice between the tensor-core and CUDA-core paths of a split plan's GEMM steps from measured times.
#include "tune.hpp"

namespace ndsi {

bool choose_paths(const std::vector<TuneStep>& steps, const std::vector<double>& split, const std::vector<double>& cuda,
                  const std::vector<double>* mixed, const std::vector<char>* mixed_use, std::vector<char>& use,
                  std::vector<double>& tensor_ms) {
    bool open = false;
    tensor_ms = split;
    for (size_t k = 0; k < steps.size(); ++k) {
        const TuneStep& s = steps[k];
        const size_t b = s.launch;
        if (!s.receives) {
            if (k + 1 < steps.size() && steps[k + 1].receives) continue;  // decided with the step it gives slices to
            use[b] = s.decided || split[b] <= cuda[b] ? 1 : 0;
            continue;
        }
        const TuneStep& giver = steps[k - 1];
        const size_t a = giver.launch;
        auto copy = [&](const std::vector<double>& t) { return s.copy >= 0 ? t[s.copy] : 0.0; };
        // giver and receiver on the tensor cores; the cheapest of the configurations that were timed wins
        double best = split[a] + split[b] + copy(split);
        use[a] = use[b] = 1;
        auto offer = [&](double t, int ua, int ub) {
            if (t >= best) return false;
            best = t;
            use[a] = static_cast<char>(ua);
            use[b] = static_cast<char>(ub);
            return true;
        };
        if (!s.decided) offer(split[a] + cuda[b] + copy(cuda), 1, 0);
        if (!s.decided && !giver.decided) offer(cuda[a] + cuda[b] + copy(cuda), 0, 0);
        if (!giver.decided) {
            if (s.decided) {
                // the CUDA-core sweep ran the receiver on the tensor cores
                if (offer(cuda[a] + cuda[b] + copy(cuda), 0, 1)) tensor_ms[b] = cuda[b];
            } else if (!mixed) {
                if (offer(cuda[a] + split[b] + copy(cuda), 0, 1)) open = true;  // without the shared operand's slicing
            } else if (!(*mixed_use)[a] && (*mixed_use)[b]) {
                if (offer(cuda[a] + (*mixed)[b] + copy(*mixed), 0, 1)) tensor_ms[b] = (*mixed)[b];
            }
        }
    }
    return open;
}

}  // namespace ndsi
