// How a small grid is cut into bricks for the resident Bi-CG kernels: plain
// arithmetic, used by the launches and the kernel and checked on the CPU.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define EXCMG_HD __host__ __device__ __forceinline__
#else
#define EXCMG_HD inline
#endif

namespace excmg {

constexpr int kResThreads = 512;
constexpr int kResHaloThreads = kResThreads - 32;   // warp 0 has the exchanges
constexpr int kResMaxCtas = 160;    // slot words per copy (five per lane)
constexpr int kResCopies = 32;      // copies of every slot word
// two sets of slot words and the error word
constexpr size_t kResWords = (size_t)2 * kResCopies * kResMaxCtas + 1;

struct ResidentGeom {
    int cx, cy, cz;     // bricks per axis
    int bx, by, bz;     // nodes per brick and axis (the last one may hold fewer)
    int np, nh;         // nodes per thread along z, nodes around the brick per thread
    int halo;           // nodes around a brick that the taps reach
    int tx;             // row pitch of the shared tile
    int tile;           // entries of the shared tile
    int ctas;
};

// Row pitch of the tile beyond the brick's width: the bx nodes of a row and
// the rows after it then lie on consecutive banks (8-byte entries: 16 of them;
// the 4-byte entries of the FP32 kernel share the layout).
constexpr int kResPad = 16;

// Shared memory of a CTA at most; the kernels are opted in to this much once,
// as the launches of different grids share them.
constexpr size_t kResSmemBytes = 212 * 1024;

// Nodes around the brick per thread of the variant with np nodes per thread.
inline int resident_nh(int np) { return np == 1 ? 2 : np == 2 ? 3 : np == 4 ? 5 : np == 6 ? 6 : 7; }

// Variants with more nodes per thread keep x, r*, p* in shared memory.
constexpr int kResRegNodes = 4;
inline size_t resident_own_bytes(int np) { return np > kResRegNodes ? (size_t)3 * np * kResThreads * 8 : 0; }

// Node h of the nodes around a brick that the taps of its nodes reach: two
// layers on each face and one row along each edge.  Local coordinates
// (0 .. b - 1 inside the brick).
EXCMG_HD void res_halo(int h, int bx, int by, int bz, int* lx, int* ly, int* lz) {
    const int fx = 4 * by * bz, fy = 4 * bx * bz, fz = 4 * bx * by;
    if (h < fz) {
        const int l = h / (bx * by), e = h - l * bx * by;
        *lz = l < 2 ? l - 2 : bz + l - 2;
        *ly = e / bx;
        *lx = e - *ly * bx;
        return;
    }
    h -= fz;
    if (h < fy) {
        const int l = h / (bx * bz), e = h - l * bx * bz;
        *ly = l < 2 ? l - 2 : by + l - 2;
        *lz = e / bx;
        *lx = e - *lz * bx;
        return;
    }
    h -= fy;
    if (h < fx) {
        const int l = h & 3, e = h >> 2;
        *lx = l < 2 ? l - 2 : bx + l - 2;
        *lz = e / by;
        *ly = e - *lz * by;
        return;
    }
    h -= fx;
    if (h < 4 * bx) {
        const int l = h / bx;
        *lx = h - l * bx;
        *ly = (l & 1) ? by : -1;
        *lz = (l & 2) ? bz : -1;
        return;
    }
    h -= 4 * bx;
    if (h < 4 * by) {
        const int l = h / by;
        *ly = h - l * by;
        *lx = (l & 1) ? bx : -1;
        *lz = (l & 2) ? bz : -1;
        return;
    }
    h -= 4 * by;
    const int l = h / bz;
    *lz = h - l * bz;
    *lx = (l & 1) ? bx : -1;
    *ly = (l & 2) ? by : -1;
}

// The same in two dimensions (DIM = 2: x and z), corners at (+-1, +-1).
EXCMG_HD void res_halo2(int h, int bx, int bz, int* lx, int* lz) {
    if (h < 4 * bx) {
        const int l = h / bx;
        *lx = h - l * bx;
        *lz = l < 2 ? l - 2 : bz + l - 2;
        return;
    }
    h -= 4 * bx;
    if (h < 4 * bz) {
        const int l = h & 3;
        *lz = h >> 2;
        *lx = l < 2 ? l - 2 : bx + l - 2;
        return;
    }
    h -= 4 * bz;
    *lx = (h & 1) ? bx : -1;
    *lz = (h & 2) ? bz : -1;
}

// The cut of a grid with n intervals into at most max_ctas bricks that fits
// the kernel's variants, and of those the cheapest iteration.  Cost in
// half cycles: five FP64 instructions for each of a thread's own nodes (p,
// sigma, r, rho; x under way counts as part) and one for each node around, two
// lanes per cycle and SM, plus what two exchanges take longer per CTA (about
// 10 cycles each, 1.62 us at 32 CTAs against 2.21 us at 152).  ctas = 0: none
// fits.
inline ResidentGeom resident_geometry(int n, int max_ctas) {
    ResidentGeom best{};
    long long best_cost = -1;
    const int m = n - 1;
    if (max_ctas > kResMaxCtas) max_ctas = kResMaxCtas;
    for (int bx = 1; bx <= m; ++bx) {
        const int cx = (m + bx - 1) / bx;
        if (cx > max_ctas || (m + cx - 1) / cx != bx) continue;
        for (int by = 1; by <= m; ++by) {
            const int cy = (m + by - 1) / by;
            if (cx * cy > max_ctas || (m + cy - 1) / cy != by) continue;
            for (int bz = 1; bz <= m; ++bz) {
                const int cz = (m + bz - 1) / bz;
                if (cx * cy * cz > max_ctas || (m + cz - 1) / cz != bz) continue;
                const int halo = 4 * (bx * by + bx * bz + by * bz) + 4 * (bx + by + bz);
                for (int np = 1; np <= 8; np += np < 2 ? 1 : 2) {
                    const int threads = bx * by * ((bz + np - 1) / np);
                    const int nh = resident_nh(np);
                    const int runs = (bz + np - 1) / np * np;
                    const int tile = (bx + kResPad) * (by + 4) * (runs + 4);
                    if (threads > kResThreads || halo > nh * kResHaloThreads ||
                        (size_t)tile * 8 + resident_own_bytes(np) > kResSmemBytes)
                        continue;
                    const long long cost = 5LL * np * ((threads + 127) / 128) * 128 + halo + 40LL * cx * cy * cz;
                    if (best_cost < 0 || cost < best_cost) {
                        best_cost = cost;
                        best = ResidentGeom{cx, cy, cz, bx, by, bz, np, nh, halo, bx + kResPad, tile, cx * cy * cz};
                    }
                }
            }
        }
    }
    return best;
}

// The same for a 2D grid (y empty; at most one node around the brick per thread).
inline ResidentGeom resident_geometry2d(int n, int max_ctas) {
    ResidentGeom best{};
    long long best_cost = -1;
    const int m = n - 1;
    if (max_ctas > kResMaxCtas) max_ctas = kResMaxCtas;
    for (int cx = 1; cx <= m && cx <= max_ctas; ++cx) {
        const int bx = (m + cx - 1) / cx;
        if ((m + bx - 1) / bx != cx) continue;
        for (int cz = 1; cz <= m && cx * cz <= max_ctas; ++cz) {
            const int bz = (m + cz - 1) / cz;
            if ((m + bz - 1) / bz != cz) continue;
            const int halo = 4 * (bx + bz) + 4, nh = 1;
            for (int np = 1; np <= 4; np *= 2) {
                const int threads = bx * ((bz + np - 1) / np), runs = (bz + np - 1) / np * np;
                const int tile = (bx + kResPad) * (runs + 4);
                if (threads > kResThreads || halo > nh * kResHaloThreads || (size_t)tile * 8 > kResSmemBytes) continue;
                const long long cost = 5LL * np * ((threads + 127) / 128) * 128 + halo + 40LL * cx * cz;
                if (best_cost < 0 || cost < best_cost) {
                    best_cost = cost;
                    best = ResidentGeom{cx, 1, cz, bx, 1, bz, np, nh, halo, bx + kResPad, tile, cx * cz};
                }
            }
        }
    }
    return best;
}

}  // namespace excmg
