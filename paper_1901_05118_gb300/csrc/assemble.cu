// Right-hand side f_h of eq. (sec) and the boundary values of a level.
//
// Every interior node's row of eq. (method1) is h^4 f; the taps that land on
// boundary nodes carry known values g1 and move to the right-hand side, and
// the +-2 axis taps of nodes one step from a face reach a fictitious node
// whose value eq. (reflection2) / (reflection4) splits into a mirror unknown
// (folded into the operator's diagonal) and known data:
//   first kind:   u_ghost = u_mirror + 2h g2          (g2 = outward du/dn)
//   second kind:  u_ghost = -u_mirror + 2 g1 + h^2 g2  (g2 = d2u/dn2)
// The level's arrays are taken at every stride-th node of the given (finer)
// arrays, as the grids of Alg. 1 are nested.
#include "excmg_internal.cuh"

namespace excmg {
namespace {

struct Src {
    const double* g1;
    const double* g2;
    int np_src;   // n_src + 1
    int stride;
    __device__ __forceinline__ double node(int i, int j, int k) const {
        return g1[((size_t)(k * stride) * np_src + (size_t)(j * stride)) * np_src + (size_t)(i * stride)];
    }
    // face value at the boundary node (i,j,k) of face `face`
    __device__ __forceinline__ double face(int face, int i, int j, int k) const {
        const int axis = face >> 1;
        int a, b;
        if (axis == 0) { a = j; b = k; }
        else if (axis == 1) { a = i; b = k; }
        else { a = i; b = j; }
        return g2[(size_t)face * np_src * np_src + (size_t)(b * stride) * np_src + (size_t)(a * stride)];
    }
};

__device__ __forceinline__ bool on_boundary(int v, int n) { return v == 0 || v == n; }

// f_h at the interior node (i, j, k): h^4 f minus what the 25 taps move over.
__device__ __forceinline__ double rhs_near_boundary(int i, int j, int k, int n, int bc_kind, double h, double rhs,
                                                    const Src& src) {
    const int p[3] = {i, j, k};
    double moved = 0.0;
    // axis taps: +-1 (weight -12) and +-2 (weight +1)
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
        for (int s = -1; s <= 1; s += 2) {
            int q[3] = {p[0], p[1], p[2]};
            q[ax] = p[ax] + s;
            if (on_boundary(q[ax], n)) moved += -12.0 * src.node(q[0], q[1], q[2]);
            q[ax] = p[ax] + 2 * s;
            if (on_boundary(q[ax], n)) {
                moved += src.node(q[0], q[1], q[2]);
            } else if (q[ax] < 0 || q[ax] > n) {
                int bnode[3] = {p[0], p[1], p[2]};
                bnode[ax] = s < 0 ? 0 : n;
                const int face = 2 * ax + (s < 0 ? 0 : 1);
                const double g2v = src.face(face, bnode[0], bnode[1], bnode[2]);
                if (bc_kind == 1)
                    moved += 2.0 * h * g2v;
                else
                    moved += 2.0 * src.node(bnode[0], bnode[1], bnode[2]) + h * h * g2v;
            }
        }
    }
    // in-plane diagonal taps (weight +2)
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a + 1; b < 3; ++b)
#pragma unroll
            for (int sa = -1; sa <= 1; sa += 2)
#pragma unroll
                for (int sb = -1; sb <= 1; sb += 2) {
                    int q[3] = {p[0], p[1], p[2]};
                    q[a] += sa;
                    q[b] += sb;
                    if (on_boundary(q[0], n) || on_boundary(q[1], n) || on_boundary(q[2], n))
                        moved += 2.0 * src.node(q[0], q[1], q[2]);
                }
    return rhs - moved;
}

// The same at a node d = 1 or 2 steps from one face and at least three from
// the others, the terms in the same order: the taps on boundary nodes are the
// face's own node and, for d = 1, its four neighbours on the face.  (The
// general form costs 32 FP64 instructions per node, most of them predicated
// off for such a node: the whole right-hand side at 512^3 555 us with it
// alone, 465 with this form; floor 317.)
__device__ __forceinline__ double rhs_near_face(int ax, bool low, int d, const int (&p)[3], int n, int bc_kind,
                                                double h, double rhs, const Src& src) {
    int q[3] = {p[0], p[1], p[2]};
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (a == ax) q[a] = low ? 0 : n;
    const size_t sx = (size_t)src.stride, sy = sx * src.np_src, sz = sy * src.np_src;
    const double* const g = src.g1 + (size_t)q[2] * sz + (size_t)q[1] * sy + (size_t)q[0] * sx;
    if (d == 2) return rhs - *g;
    const size_t s1 = ax == 0 ? sy : sx, s2 = ax == 2 ? sy : sz;
    const double b = *g, g2v = src.face(2 * ax + (low ? 0 : 1), q[0], q[1], q[2]);
    const double m1 = *(g - s1), p1 = g[s1], m2 = *(g - s2), p2 = g[s2];
    double moved = -12.0 * b;
    if (bc_kind == 1)
        moved += 2.0 * h * g2v;
    else
        moved += 2.0 * b + h * h * g2v;
    moved += 2.0 * m1;
    moved += 2.0 * p1;
    moved += 2.0 * m2;
    moved += 2.0 * p2;
    return rhs - moved;
}

// h^4 f at the nodes that no boundary value reaches, zero on the boundary.  A
// warp takes a row at a time.  One index per node with 64-bit divisions, and
// the boundary rows in the same launch, took 1.14 ms at 512^3: the first and
// the last warp of every row waited for the taps of four nodes.
__global__ void __launch_bounds__(256)
assemble_rhs_kernel(double* __restrict__ fh, int n, const double* __restrict__ f, Src src) {
    const int np = n + 1, lane = threadIdx.x & 31;
    const double h = 1.0 / (double)n;
    const double h4 = h * h * h * h;
    const int warps = gridDim.x * 8, rows = np * np;
    for (int row = blockIdx.x * 8 + (threadIdx.x >> 5); row < rows; row += warps) {
        const int k = row / np, j = row - k * np;
        double* const out = fh + (size_t)row * np;
        const bool in_yz = j >= 1 && j <= n - 1 && k >= 1 && k <= n - 1;
        const bool deep_yz = j >= 3 && j <= n - 3 && k >= 3 && k <= n - 3;
        const double* const fr = f + ((size_t)(k * src.stride) * src.np_src + (size_t)(j * src.stride)) * src.np_src;
        constexpr int U = 4;   // loads of a lane in flight
        for (int i0 = lane; i0 <= n; i0 += 32 * U) {
            double v[U];
#pragma unroll
            for (int c = 0; c < U; ++c) {
                const int i = i0 + 32 * c;
                v[c] = in_yz && i >= 1 && i <= n - 1 ? fr[(size_t)i * src.stride] : 0.0;
            }
#pragma unroll
            for (int c = 0; c < U; ++c) {
                const int i = i0 + 32 * c;
                if (i > n) break;
                const bool inside = in_yz && i >= 1 && i <= n - 1;
                if (!inside || (deep_yz && i >= 3 && i <= n - 3)) out[i] = h4 * v[c];
            }
        }
    }
}

// All of it on small grids, a node per thread: rows by warp left a warp two rounds of
// near nodes one after the other (the whole call on 50^3 from 100^3 data 37.4 us, 34.9 so).
__global__ void __launch_bounds__(256)
assemble_nodes_kernel(double* __restrict__ fh, int n, int bc_kind, const double* __restrict__ f, Src src) {
    const int np = n + 1, t = blockIdx.x * 256 + threadIdx.x;
    if (t >= np * np * np) return;
    const double h = 1.0 / (double)n;
    const double h4 = h * h * h * h;
    const int k = t / (np * np), e = t - k * np * np, j = e / np, i = e - j * np;
    if (i < 1 || i > n - 1 || j < 1 || j > n - 1 || k < 1 || k > n - 1) {
        fh[t] = 0.0;
        return;
    }
    const double rhs = h4 * f[((size_t)(k * src.stride) * src.np_src + (size_t)(j * src.stride)) * src.np_src +
                              (size_t)(i * src.stride)];
    const bool deep = i >= 3 && i <= n - 3 && j >= 3 && j <= n - 3 && k >= 3 && k <= n - 3;
    fh[t] = deep ? rhs : rhs_near_boundary(i, j, k, n, bc_kind, h, rhs, src);
}

// The nodes within two of a face, n >= 9: the layers 1, 2, n - 2, n - 1 along z,
// then those along y of the planes between, then those along x of what is left.
__global__ void __launch_bounds__(256)
assemble_near_kernel(double* __restrict__ fh, int n, int bc_kind, const double* __restrict__ f, Src src) {
    const int np = n + 1, m = n - 1, q = m - 4;
    const int nz = 4 * m * m, ny = q * 4 * m, total = nz + ny + q * q * 4;
    const double h = 1.0 / (double)n;
    const double h4 = h * h * h * h;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        int i, j, k;
        auto layer = [&](int l) { return l < 2 ? 1 + l : n - 4 + l; };
        if (t < nz) {
            const int l = t / (m * m), e = t - l * m * m;
            k = layer(l);
            j = 1 + e / m;
            i = e - (j - 1) * m + 1;
        } else if (t < nz + ny) {
            const int e = t - nz, z = e / (4 * m), r = e - z * 4 * m, l = r / m;
            k = 3 + z;
            j = layer(l);
            i = r - l * m + 1;
        } else {
            const int e = t - nz - ny, z = e / (4 * q), r = e - z * 4 * q;
            k = 3 + z;
            j = 3 + (r >> 2);
            i = layer(r & 3);
        }
        const double rhs = h4 * f[((size_t)(k * src.stride) * src.np_src + (size_t)(j * src.stride)) * src.np_src +
                                  (size_t)(i * src.stride)];
        // the one axis with a face within two steps, if there is just one
        const int p[3] = {i, j, k};
        int ax = -1, near = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (p[a] < 3 || p[a] > n - 3) {
                ax = a;
                ++near;
            }
        const int pa = ax == 0 ? i : ax == 1 ? j : k;
        double v;
        if (near == 1) v = rhs_near_face(ax, pa < 3, pa < 3 ? pa : n - pa, p, n, bc_kind, h, rhs, src);
        else v = rhs_near_boundary(i, j, k, n, bc_kind, h, rhs, src);
        fh[((size_t)k * np + j) * np + i] = v;
    }
}

__global__ void set_boundary_kernel(double* __restrict__ u, int n, Src src) {
    const int np = n + 1;
    const size_t per_face = (size_t)np * np;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < 6 * per_face;
         t += (size_t)gridDim.x * blockDim.x) {
        const int face = (int)(t / per_face);
        const size_t r = t - face * per_face;
        const int a = (int)(r % np), b = (int)(r / np);
        const int fixed = (face & 1) ? n : 0;
        int i, j, k;
        if (face < 2) { i = fixed; j = a; k = b; }
        else if (face < 4) { i = a; j = fixed; k = b; }
        else { i = a; j = b; k = fixed; }
        u[((size_t)k * np + j) * np + i] = src.node(i, j, k);
    }
}

// One launch up to here: a second one costs more than the warps that wait in the first.
constexpr int kOneLaunchMaxN = 64;

int grid_for(size_t work) {
    size_t b = (work + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

cudaError_t launch_assemble_rhs(double* fh, int n, int bc_kind, const double* f, const double* g1,
                                const double* g2, int stride, cudaStream_t s) {
    Src src{g1, g2, n * stride + 1, stride};
    if (n <= kOneLaunchMaxN) {
        assemble_nodes_kernel<<<(unsigned)((node_count(n) + 255) / 256), 256, 0, s>>>(fh, n, bc_kind, f, src);
        return cudaGetLastError();
    }
    const int rows = (n + 1) * (n + 1), want = (rows + 7) / 8;
    const int grid = want < 152 * 8 ? want : 152 * 8, block = 256;
    assemble_rhs_kernel<<<grid, block, 0, s>>>(fh, n, f, src);
    const size_t near = 4 * ((size_t)(n - 1) * (n - 1) + (size_t)(n - 5) * (n - 1) + (size_t)(n - 5) * (n - 5));
    assemble_near_kernel<<<grid_for(near), 256, 0, s>>>(fh, n, bc_kind, f, src);
    return cudaGetLastError();
}

cudaError_t launch_set_boundary(double* u, int n, const double* g1, int stride, cudaStream_t s) {
    Src src{g1, nullptr, n * stride + 1, stride};
    set_boundary_kernel<<<grid_for(face_count(n)), 256, 0, s>>>(u, n, src);
    return cudaGetLastError();
}

}  // namespace excmg
