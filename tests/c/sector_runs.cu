// Host check of sector.cuh: for random groups of centres, every galaxy within the annulus of a
// centre is listed exactly once over the sectors, inside the catalog, and its direction from the
// centre lies within half a sector plus the angle of the cell's and the group's extents.
// usage: sector_runs seed n side ncx ncy S rows cols Ri Ro holes; prints the number of checked pairs.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <random>
#include <vector>

#include "../../paper_2309_08601_gb300/csrc/sector.cuh"

using namespace mp3;

int main(int argc, char** argv)
{
    if (argc < 12) return 2;
    std::mt19937 rng(atoi(argv[1]));
    const int n = atoi(argv[2]), side = atoi(argv[3]), ncx = atoi(argv[4]), ncy = atoi(argv[5]), S = atoi(argv[6]);
    const int rows = atoi(argv[7]), cols = atoi(argv[8]);
    const double Ri = atof(argv[9]), Ro = atof(argv[10]);
    const bool holes = atoi(argv[11]) != 0;
    const int ex = side * ncx, ey = side * ncy;
    std::vector<int> x(n), y(n), key(n), ord(n), start((size_t)ncx * ncy + 1, 0);
    for (int i = 0; i < n; ++i) {
        do {
            x[i] = rng() % ex;
            y[i] = rng() % ey;
        } while (holes && ((x[i] / (8 * side) + y[i] / (8 * side)) & 1));
        if (i % 50 == 0) x[i] = x[i] / side * side, y[i] = y[i] / side * side;  // on the cells' corners
        key[i] = y[i] / side * ncx + x[i] / side;
        ord[i] = i;
        ++start[key[i] + 1];
    }
    for (size_t k = 1; k < start.size(); ++k) start[k] += start[k - 1];
    std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return key[a] < key[b]; });
    long long checked = 0;
    for (int trial = 0; trial < 40; ++trial) {
        // a group: galaxies of a window of rows x cols cells around a galaxy
        const int f = rng() % n, r0 = y[f] / side / rows * rows, q0 = x[f] / side;
        std::vector<int> grp;
        for (int i = 0; i < n && grp.size() < 8; ++i)
            if (y[i] / side >= r0 && y[i] / side < r0 + rows && x[i] / side >= q0 && x[i] / side < q0 + cols) grp.push_back(i);
        float x0 = 3e38f, x1 = -3e38f, y0 = 3e38f, y1 = -3e38f;
        for (int i : grp) {
            x0 = std::min(x0, (float)x[i]), x1 = std::max(x1, (float)x[i]);
            y0 = std::min(y0, (float)y[i]), y1 = std::max(y1, (float)y[i]);
        }
        SectorGeom g;
        g.gx = 0.5f * (x0 + x1), g.gy = 0.5f * (y0 + y1);
        g.hx = 0.5f * (x1 - x0) + 1.0f, g.hy = 0.5f * (y1 - y0) + 1.0f;
        g.Ro = (float)Ro, g.Ri = (float)Ri, g.S = (float)side, g.iS = 1.0f / g.S, g.ncx = ncx, g.ncy = ncy;
        const double reach = side * (0.7072 + 0.5 * sqrt((double)rows * rows + (double)cols * cols)) + 8.0;
        const double slack = asin(std::min(1.0, reach / Ri));
        std::vector<int> seen(n, 0);
        for (int s = 0; s < S; ++s) {
            const bool upper = s < S / 2;
            const int sp = upper ? s : s - S / 2;
            auto ray = [&](int j) { return j > 0 && j < S / 2 ? (float)(cos(2 * M_PI * j / S) / sin(2 * M_PI * j / S)) : 0.f; };
            const double sa = sin(2 * M_PI * sp / S), sb = sin(2 * M_PI * (sp + 1) / S);
            float iy0, iy1;
            sector_rows(g, upper, (float)std::min(sa, sb), (float)std::max(sa, sb), iy0, iy1);
            for (float iy = iy0; iy <= iy1; iy += 1.0f) {
                int st[2], len[2];
                sector_runs(g, upper, sp == 0, sp == S / 2 - 1, ray(sp), ray(sp + 1), iy, start.data(), st[0], len[0], st[1], len[1]);
                for (int h = 0; h < 2; ++h)
                    for (int j = 0; j < len[h]; ++j) {
                        const int at = st[h] + j;
                        if (at < 0 || at >= n) return printf("run outside the catalog\n"), 1;
                        if (++seen[at] > 1) return printf("galaxy listed twice\n"), 1;
                        for (int i : grp) {
                            const double dx = x[ord[at]] - x[i], dy = y[ord[at]] - y[i], r = hypot(dx, dy);
                            if (r < Ri || r >= Ro) continue;
                            double d = atan2(dy, dx) - 2 * M_PI * (s + 0.5) / S;
                            d -= 2 * M_PI * floor(d / (2 * M_PI) + 0.5);
                            if (fabs(d) > M_PI / S + slack) return printf("direction outside the sector\n"), 1;
                        }
                    }
                if (len[0] < 0 || len[1] < 0) return printf("negative run\n"), 1;
            }
        }
        for (int at = 0; at < n; ++at)
            for (int i : grp) {
                const double r = hypot((double)x[ord[at]] - x[i], (double)y[ord[at]] - y[i]);
                if (r >= Ri && r < Ro) {
                    if (!seen[at]) return printf("galaxy of the annulus not listed\n"), 1;
                    ++checked;
                }
            }
    }
    printf("%lld\n", checked);
    return 0;
}
