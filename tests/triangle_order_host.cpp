// Storage order of the triangles: neighbours along the curve on every scale of the mesh.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "fetdpic_internal.h"

using namespace fetdpic;

int main()
{
    // an n x n square of triangles in no order, of side `size` in a domain of size 1, and two triangles at its far end
    for (double size : {1.0, 1e-3, 1e-5, 1e-7}) {
        const int n = 60;
        std::mt19937 g(5);
        std::vector<double> xy;
        std::vector<int> cells(n * n), tri;
        const double h = size / n;
        for (int j = 0; j <= n; ++j)
            for (int i = 0; i <= n; ++i) { xy.push_back(i * h); xy.push_back(j * h); }
        for (int k = 0; k < n * n; ++k) cells[k] = k;
        std::shuffle(cells.begin(), cells.end(), g);
        for (int k : cells) {
            const int a = k / n * (n + 1) + k % n, c = a + n + 1;
            for (int v : {a, a + 1, c + 1, a, c + 1, c}) tri.push_back(v);
        }
        const int m = (int)xy.size() / 2;
        for (double v : {2.0, 2.0, 2.1, 2.0, 2.1, 2.1, 2.0, 2.1}) xy.push_back(v);
        for (int v : {0, 1, 2, 0, 2, 3}) tri.push_back(m + v);
        const int nf = (int)tri.size() / 3;
        std::vector<int> perm = hilbert_order(m + 4, xy.data(), nf, tri.data()), seen = perm;
        std::sort(seen.begin(), seen.end());
        for (int k = 0; k < nf; ++k) if (seen[k] != k) { printf("no permutation\n"); return 1; }
        double sum = 0.0;
        int pairs = 0;
        for (int k = 0; k + 1 < nf; ++k) {
            double d[2] = {0.0, 0.0};
            if (perm[k] >= nf - 2 || perm[k + 1] >= nf - 2) continue;
            for (int v = 0; v < 3; ++v)
                for (int a = 0; a < 2; ++a) d[a] += (xy[2 * tri[3 * perm[k] + v] + a] - xy[2 * tri[3 * perm[k + 1] + v] + a]) / 3.0;
            sum += std::hypot(d[0], d[1]);
            ++pairs;
        }
        if (sum / pairs > 2.0 * h) { printf("size %g: consecutive triangles %.1f edges apart\n", size, sum / pairs / h); return 1; }
    }
    return 0;
}
