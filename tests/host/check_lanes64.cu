// Host check of the compiled FP64 kernel's launch (test program): every cell of a grid is some thread's exactly
// once, and how many warps have a cell at all (an FP64 warp costs the same with one lane as with 32).
// usage: check_lanes64; prints the worst ratio of 32 * busy warps to cells over grids of at least 64 cells
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "window64.cu"

using namespace rtpn;

int main() {
    double worst = 0;
    for (int nx = 1; nx <= 140; ++nx)
        for (int k = 0; k < 6; ++k) {
            const int ny = (const int[]){1, 3, 8, 17, 5, 64}[k], nz = (const int[]){1, 2, 5, 9, 70, 40}[k];
            Geom g{nx, ny, nz, (long long)nx * ny * nz, 0, 1.0, 1.0, 1.0};
            win::Args a;
            a.nx = nx;
            a.ny = ny;
            a.nz = nz;
            a.V = g.V;
            unsigned blocks, threads;
            shape64(g, &a, &blocks, &threads);
            if (threads % 32 || threads > 128) return 3;
            std::vector<int> seen(g.V, 0);
            long long busy = 0;
            for (unsigned b = 0; b < blocks; ++b)
                for (unsigned w = 0; w < threads; w += 32) {
                    bool any = false;
                    for (unsigned t = w; t < w + 32; ++t) {
                        int x, y, z;
                        if (!cell64(a, b, t, threads, &x, &y, &z)) continue;
                        if (x < 0 || x >= nx || y < 0 || y >= ny || z < 0 || z >= nz) return 4;
                        ++seen[((long long)z * ny + y) * nx + x];
                        any = true;
                    }
                    busy += any;
                }
            for (int s : seen)
                if (s != 1) return 5;
            const double r = 32.0 * busy / g.V;
            if (g.V >= 64 && r > worst) worst = r;
        }
    printf("%.4f\n", worst);
    return 0;
}
