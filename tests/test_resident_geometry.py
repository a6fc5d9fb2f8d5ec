"""The brick decomposition of the resident Bi-CG kernels, checked on the CPU:
the same header the kernel uses (resident_geom.h), compiled with the host
compiler.  For every grid size the kernel takes, the bricks cover the interior
once, every tap of every node is a tile entry that its CTA writes (or a node
outside the interior), and all tile entries lie inside the tile."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_05118_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "resident_geom.h"
using namespace excmg;
static void fail(const char* what, int n) { std::printf("%s at n = %d\n", what, n); std::exit(1); }
int main() {
    for (int limit : {152, 132, 72, 16, 1})
    for (int n = 4; n <= 84; ++n) {
        const ResidentGeom g = resident_geometry(n, limit);
        if (g.ctas == 0) {
            if (limit == 152 && n <= 81) fail("no cut", n);
            continue;
        }
        if (g.ctas != g.cx * g.cy * g.cz || g.ctas > limit || g.ctas > kResMaxCtas) fail("CTAs", n);
        const int m = n - 1, tx = g.tx, tp = tx * (g.by + 4), cols = g.bx * g.by;
        if (cols * ((g.bz + g.np - 1) / g.np) > kResThreads) fail("threads", n);
        if (g.halo > resident_nh(g.np) * kResHaloThreads) fail("halo", n);
        std::vector<int> seen((size_t)m * m * m, 0);
        for (int cta = 0; cta < g.ctas; ++cta) {
            const int ox = 1 + cta % g.cx * g.bx, oy = 1 + cta / g.cx % g.cy * g.by, oz = 1 + cta / (g.cx * g.cy) * g.bz;
            std::vector<char> wr(g.tile, 0);
            for (int h = 0; h < g.halo; ++h) {
                int x, y, z;
                res_halo(h, g.bx, g.by, g.bz, &x, &y, &z);
                const int t = (z + 2) * tp + (y + 2) * tx + x + 2;
                if (t < 0 || t >= g.tile) fail("halo entry", n);
                if (wr[t]++) fail("halo entry twice", n);
            }
            const int nz = g.bz < n - oz ? g.bz : n - oz;
            for (int pass = 0; pass < 2; ++pass)
            for (int tid = 0; tid < kResThreads; ++tid) {
                const int grp = tid / cols, col = tid - grp * cols, ly = col / g.bx, lx = col - ly * g.bx, lz = grp * g.np;
                const int t0 = (lz + 2) * tp + (ly + 2) * tx + lx + 2;
                if (!(lz < nz && ox + lx < n && oy + ly < n)) continue;
                // (every plane of the thread's run is read, also beyond its last node)
                if (t0 - 2 * tp < 0 || t0 + (g.np + 1) * tp >= g.tile || t0 + g.np * tp + tx >= g.tile ||
                    t0 + (g.np - 1) * tp + 2 * tx >= g.tile) fail("read outside the tile", n);
                for (int k = 0; k < g.np && lz + k < nz; ++k) {
                    const int t = t0 + k * tp, X = ox + lx, Y = oy + ly, Z = oz + lz + k;
                    if (pass == 0) {
                        if (t >= g.tile || wr[t]++) fail("own entry", n);
                        ++seen[((size_t)(Z - 1) * m + Y - 1) * m + X - 1];
                        continue;
                    }
                    const int d[][3] = {{1,0,0},{2,0,0},{0,1,0},{0,2,0},{0,0,1},{0,0,2},{1,1,0},{1,-1,0},{1,0,1},
                                        {1,0,-1},{0,1,1},{0,1,-1}};
                    for (auto& v : d)
                        for (int s = -1; s <= 1; s += 2) {
                            const int a = X + s * v[0], b = Y + s * v[1], c = Z + s * v[2];
                            if (a < 1 || a > m || b < 1 || b > m || c < 1 || c > m) continue;
                            if (!wr[t + s * (v[2] * tp + v[1] * tx + v[0])]) fail("tap not in the tile", n);
                        }
                }
            }
        }
        for (int s : seen)
            if (s != 1) fail("cover", n);
    }
    // 2D: the same with the second axis as z
    for (int n = 4; n <= 520; n += n < 70 ? 1 : 25) {
        const ResidentGeom g = resident_geometry2d(n, 152);
        if (g.ctas == 0) {
            if (n <= 512) fail("no 2D cut", n);
            continue;
        }
        if (g.ctas != g.cx * g.cz || g.ctas > 152 || g.bx * ((g.bz + g.np - 1) / g.np) > kResThreads ||
            g.halo > g.nh * kResHaloThreads) fail("2D threads", n);
        const int m = n - 1, tx = g.tx;
        std::vector<int> seen((size_t)m * m, 0);
        for (int cta = 0; cta < g.ctas; ++cta) {
            const int ox = 1 + cta % g.cx * g.bx, oz = 1 + cta / g.cx * g.bz, nz = g.bz < n - oz ? g.bz : n - oz;
            std::vector<char> wr(g.tile, 0);
            for (int h = 0; h < g.halo; ++h) {
                int x, z;
                res_halo2(h, g.bx, g.bz, &x, &z);
                const int t = (z + 2) * tx + x + 2;
                if (t < 0 || t >= g.tile || wr[t]++) fail("2D halo entry", n);
            }
            for (int pass = 0; pass < 2; ++pass)
            for (int tid = 0; tid < kResThreads; ++tid) {
                const int lz = tid / g.bx * g.np, lx = tid % g.bx, t0 = (lz + 2) * tx + lx + 2;
                if (!(lz < nz && ox + lx < n)) continue;
                if (t0 - 2 * tx - 2 < 0 || t0 + (g.np + 1) * tx >= g.tile || t0 + g.np * tx + 1 >= g.tile)
                    fail("2D read outside the tile", n);
                for (int k = 0; k < g.np && lz + k < nz; ++k) {
                    const int t = t0 + k * tx, X = ox + lx, Z = oz + lz + k;
                    if (pass == 0) {
                        if (t >= g.tile || wr[t]++) fail("2D own entry", n);
                        ++seen[(size_t)(Z - 1) * m + X - 1];
                        continue;
                    }
                    const int d[][2] = {{1,0},{2,0},{0,1},{0,2},{1,1},{1,-1}};
                    for (auto& v : d)
                        for (int s = -1; s <= 1; s += 2) {
                            const int a = X + s * v[0], c = Z + s * v[1];
                            if (a < 1 || a > m || c < 1 || c > m) continue;
                            if (!wr[t + s * (v[1] * tx + v[0])]) fail("2D tap not in the tile", n);
                        }
                }
            }
        }
        for (int s : seen)
            if (s != 1) fail("2D cover", n);
    }
    return 0;
}
"""


def test_bricks_cover_the_grid_and_their_taps(tmp_path):
    src = tmp_path / "geom.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "geom"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
