// Prints, for p = 1..4, the weak reference matrices (build_ref_elem: M1, N) and the nodal
// ones (build_nodal_ref: Dx, Dy, lift, ML1, ML2, Wx, Wy) as hexadecimal floats, one line per
// degree.
#include "../paper_2004_09389_gb300/csrc/common.h"

#include <cstdio>

using namespace hdg;

int main() {
    for (int p = 1; p <= 4; ++p) {
        const RefElem r = build_ref_elem(p);
        for (double v : r.M1) std::printf("%a ", v);
        for (double v : r.N) std::printf("%a ", v);
        for (double v : build_nodal_ref(p).packed()) std::printf("%a ", v);
        std::printf("\n");
    }
    return 0;
}
