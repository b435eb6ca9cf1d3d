// Host count of a batch's grouped launches: no GPU needed.
// Usage: batch_programs n_outer n_cg form..., a form being two digits: the slice
// has orbits, it has the tensor-core filter.  Prints the launches of the phase
// lists (one for each operator present in a phase; the tensor-core filter is
// launched slice by slice and is left out).
#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>

#include "host_common.h"

using namespace air;

int main(int argc, char **argv) {
    std::vector<SolveForm> forms;
    for (int i = 3; i < argc; ++i) forms.push_back({std::atoi(argv[1]), std::atoi(argv[2]), argv[i][1] == '1', argv[i][0] == '1'});
    const auto progs = batch_programs(forms);
    size_t n = 0;
    for (size_t ph = 0;; ++ph) {
        std::set<int> ops;
        bool any = false;
        for (const auto &p : progs) {
            any |= ph < p.size();
            if (ph < p.size() && p[ph].op != OP_NOP && p[ph].op != OP_RAMP_TC) ops.insert(p[ph].op);
        }
        if (!any) break;
        n += ops.size();
    }
    std::printf("%zu\n", n);
    return 0;
}
