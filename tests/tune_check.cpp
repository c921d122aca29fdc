// Path choice of the autotuner from given times: single steps, pairs that share slices in all four
// configurations, the cost of slicing a shared operand again, and the copy a slicer takes over.
// Prints one line per case; exits non-zero on a wrong choice.
#include <cstdio>

#include "tune.hpp"

using namespace ndsi;
using V = std::vector<double>;

int bad = 0;
// launches: 0 giver, 1 receiver, 2 its copy
void pair(const char* what, const V& split, const V& cuda, const V* mixed, bool da, bool db, int ua, int ub, bool open,
          double receiver_ms = 0) {
    const std::vector<TuneStep> steps = {{0, false, -1, da}, {1, true, 2, db}};
    std::vector<char> use(3, 1), mixed_use = {0, 1, 1};
    V ms;
    const bool o = choose_paths(steps, split, cuda, mixed, mixed ? &mixed_use : nullptr, use, ms);
    const bool ok = use[0] == ua && use[1] == ub && o == open && (receiver_ms == 0 || ms[1] == receiver_ms);
    std::printf("%-55s %d %d%s %s\n", what, use[0], use[1], o ? " open" : "", ok ? "ok" : "WRONG");
    if (!ok) ++bad;
}

int main() {
    // the copy costs 2 when no slicer makes it; the receiver's own slicing of the shared operand 3
    pair("both faster on the tensor cores", V{5, 5, 0}, V{9, 9, 2}, nullptr, false, false, 1, 1, false);
    pair("both faster on the CUDA cores", V{5, 9, 0}, V{3, 3, 2}, nullptr, false, false, 0, 0, false);
    // one by one the receiver would leave the tensor cores for 1 and pay 2 for the copy
    pair("receiver kept for the copy it makes", V{5, 5, 0}, V{9, 4, 2}, nullptr, false, false, 1, 1, false);
    // one by one the giver would leave for 1 and the receiver then pay 3 + 2
    pair("giver leaves: not timed yet", V{9, 5, 0}, V{5, 9, 2}, nullptr, false, false, 0, 1, true);
    const V same = {5, 8, 2};
    pair("giver stays: slicing again costs more", V{9, 5, 0}, V{5, 9, 2}, &same, false, false, 1, 1, false, 5);
    const V cheap = {5, 6, 2};
    pair("giver leaves: slicing again is cheap", V{9, 5, 0}, V{5, 9, 2}, &cheap, false, false, 0, 1, false, 6);
    pair("receiver decided, timed with its own slicing", V{9, 5, 0}, V{5, 8, 2}, nullptr, false, true, 1, 1, false);
    pair("receiver decided, giver much faster", V{9, 5, 0}, V{1, 8, 2}, nullptr, false, true, 0, 1, false, 8);
    pair("giver decided", V{5, 9, 0}, V{0, 3, 2}, nullptr, true, false, 1, 0, false);
    pair("both decided", V{5, 5, 0}, V{0, 0, 0}, nullptr, true, true, 1, 1, false);
    {
        const std::vector<TuneStep> steps = {{0, false, -1, false}, {3, false, -1, false}, {4, false, 5, true}};
        std::vector<char> use(6, 1);
        V ms;
        choose_paths(steps, V{5, 0, 0, 4, 3, 0}, V{4, 0, 0, 5, 1, 2}, nullptr, nullptr, use, ms);
        const bool ok = use[0] == 0 && use[3] == 1 && use[4] == 1;
        std::printf("%-55s %s\n", "single steps", ok ? "ok" : "WRONG");
        if (!ok) ++bad;
    }
    return bad ? 1 : 0;
}
