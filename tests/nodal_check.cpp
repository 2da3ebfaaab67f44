// Checks the nodal reference matrices (build_nodal_ref) against the weak ones
// (build_ref_elem) they replace, p = 1..4: M Dx = Dxi, M Dy = Deta, M lift_i = N_i,
// M ML_l = ML_l (weak), M W = -D^T, the edge node maps, and that every entry the kernels leave out vanishes.
#include "../paper_2004_09389_gb300/csrc/common.h"

#include <algorithm>
#include <cmath>
#include <cstdio>

using namespace hdg;

int main() {
    double worst = 0.0, left_out = 0.0;
    for (int p = 1; p <= 4; ++p) {
        const RefElem r = build_ref_elem(p);
        const NodalRef q = build_nodal_ref(p);
        const int n = r.n, pp = r.pp;
        // max |M A - B| for A [n][w], B [n][w]
        auto diff = [&](const double *A, const double *B, int w) {
            for (int i = 0; i < n; ++i)
                for (int j = 0; j < w; ++j) {
                    double s = -B[i * w + j];
                    for (int k = 0; k < n; ++k) s += r.M[i * n + k] * A[k * w + j];
                    worst = std::max(worst, std::fabs(s));
                }
        };
        diff(q.Dx.data(), r.Dxi.data(), n);
        diff(q.Dy.data(), r.Deta.data(), n);
        diff(q.ML1.data(), r.ML.data() + n * n, n);
        diff(q.ML2.data(), r.ML.data() + 2 * n * n, n);
        std::vector<double> t(size_t(2) * n * n);
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) {
                t[i * n + j] = -r.Dxi[j * n + i];
                t[(n + i) * n + j] = -r.Deta[j * n + i];
            }
        diff(q.Wx.data(), t.data(), n);
        diff(q.Wy.data(), t.data() + n * n, n);
        for (int e = 0; e < 3; ++e)
            for (int j = 0; j < pp; ++j) {
                const int b = edge_cell_node(p, e, j);
                if (node_edge_pos(p, e, b) != j) return 3;
            }
        for (int e = 0; e < 3; ++e) diff(q.lift.data() + e * n * pp, r.N.data() + e * n * pp, pp);
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) {
                if (!nodal_dx_nonzero(p, i, j)) left_out = std::max(left_out, std::fabs(q.Dx[i * n + j]));
                if (!nodal_dy_nonzero(p, i, j)) left_out = std::max(left_out, std::fabs(q.Dy[i * n + j]));
            }
        const NodalOffsets o = nodal_offsets(p);
        if (int(q.packed().size()) != o.total) return 2;
    }
    std::printf("%.3e %.3e\n", worst, left_out);
    return 0;
}
