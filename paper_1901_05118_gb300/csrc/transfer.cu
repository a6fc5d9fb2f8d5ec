// Level-transfer steps of Alg. 1.
//
// EXP_finite (Sec. 4.2.2-4.2.3).  On one cell of the coarsest of three
// nested grids, Steps 1-4 give the 27 nodes shared with the middle grid:
// the corner rule (secfff) is u1 + (u1 - u0)/4, the edge rule (bfsec) adds
// (1/8) of the two end differences, and Steps 3-4 average (bfsec) over the
// 2 face diagonals / 4 space diagonals.  All four are one formula,
//     W = u1 + (1/4) * (mean of d = u1 - u0 over the 2^m coarse nodes
//                       around the node, m = number of odd coordinates),
// which is EXP_true's formula with 1/4 in the place of 1/3 (one kernel serves
// both; shared cells agree by construction).  Step 5 is tri-quadratic Lagrange interpolation
// (eqs. (inter)-(iinter)) of W at the fine nodes: per axis the natural
// coordinate 0, 1/4, 1/2, 3/4, 1 has weights (1,0,0), (3/8,3/4,-1/8),
// (0,1,0), (-1/8,3/4,3/8), (0,0,1) on the cell's three middle-grid nodes.
//
// EXP_true (Sec. 4.2.1, eqs. (t1), (chenlin); Alg. 1's final extrapolation):
//     u~ = u_h + (1/3) * (mean of u_h - u_2h over the 2^m coarse nodes
//                         around the node),
// which is (4 u_h - u_2h)/3 at coarse nodes and (chenlin) at 1D midpoints.

#include "excmg_internal.cuh"
#include "reduce.cuh"

namespace excmg {
namespace {

__device__ __forceinline__ size_t nidx(int np, int i, int j, int k) {
    return ((size_t)k * np + j) * np + i;
}

// Both passes work on tiles of 32 x 8 x 8 fine nodes, one CTA of 32 x 8
// threads each.  The coarser values that a tile needs (17 x 5 x 5) go through
// shared memory, are interpolated along x there, and along y and z in the
// registers of the thread that owns a fine (x, y) column of the tile, so that
// every intermediate value is formed once per tile.  What bounds them: FP64
// issue (a warp instruction takes 64 cycles of an SM sub-partition whatever
// its active lanes), then the stores; the integer index arithmetic is kept to
// constant divisors.
constexpr int TT_X = 32, TT_Y = 8, TT_Z = 8;
constexpr int TT_THREADS = 256;
constexpr int TM_X = TT_X / 2 + 1, TM_Y = TT_Y / 2 + 1, TM_Z = TT_Z / 2 + 1;   // coarse extents (17, 5, 5)

// Row of the tile of a warp: the even rows on warps 0 .. 3, the odd ones, which
// have FP64 work along y, on warps 4 .. 7, one on each sub-partition (on
// every second warp they kept two of the four FP64 pipes idle: 1.08 instead
// of 0.8 ms for Step 5 at 512^3).  The kernels skip that work on the even rows by a
// loop of 0 or 1 trips (opaque in reduce.cuh): as a branch it became
// predicated FP64 instructions, which hold the pipe on every row.
__device__ __forceinline__ int tile_row(int warp) { return 2 * (warp & 3) + (warp >> 2); }

// out = u + kWeight * (mean of d = u - uc over the 1, 2, 4 or 8 coarse nodes
// around each node), u on the grid with nf intervals, uc on the one with nf / 2:
// EXP_true with weight 1/3, Steps 1-4 of EXP_finite with weight 1/4
// (kQuarter), where every scaling is a power of two.
// Measured, EXP_true on 256^3 / 512^3 (42 / 320 us of HBM traffic, about 60 / 480 of
// FP64 issue): 107 / 614 us (124 / 747 with predicated sums along y and one row per warp
// along x; 135 / - with every intermediate value through shared memory).
template <bool kQuarter>
__global__ void __launch_bounds__(TT_THREADS)
extrapolate_tiled_kernel(double* __restrict__ out, const double* __restrict__ u, const double* __restrict__ uc,
                         int nf) {
    __shared__ double Ds[TM_Z * TM_Y][TM_X];
    __shared__ double Sx[TM_Z * TM_Y + 1][TT_X];
    const int tid = threadIdx.x, fx = tid & 31, warp = tid >> 5, fy = tile_row(warp);
    const int np = nf + 1, npc = nf / 2 + 1;
    const int xa = blockIdx.x * TT_X, ya = blockIdx.y * TT_Y, za = blockIdx.z * TT_Z;
    const int cx0 = xa >> 1, cy0 = ya >> 1, cz0 = za >> 1;
    for (int e = tid; e < TM_Z * TM_Y * TM_X; e += TT_THREADS) {
        const int row = e / TM_X, ex = e - row * TM_X, ez = row / TM_Y, ey = row - ez * TM_Y;
        const int ci = cx0 + ex, cj = cy0 + ey, ck = cz0 + ez;
        double d = 0.0;
        if (ci < npc && cj < npc && ck < npc) d = u[nidx(np, 2 * ci, 2 * cj, 2 * ck)] - uc[nidx(npc, ci, cj, ck)];
        Ds[row][ex] = d;
        if (ex < TT_X / 2) Sx[row][2 * ex] = d;
    }
    const int i = xa + fx, j = ya + fy;
    const bool mine = i < np && j < np;
    const int kz = min(TT_Z, np - za);   // planes of the tile
    const size_t o = nidx(np, mine ? i : 0, mine ? j : 0, za);
    const size_t plane = (size_t)np * np;
    double uv[TT_Z];
#pragma unroll
    for (int k = 0; k < TT_Z; ++k) uv[k] = mine && k < kz ? u[o + k * plane] : 0.0;
    __syncthreads();
    // along x: a warp forms the odd nodes of two rows at a time
    for (int pair = warp; 2 * pair < TM_Z * TM_Y; pair += TT_Y) {
        const int row = 2 * pair + (fx >> 4), c = fx & 15;
        if (row < TM_Z * TM_Y) Sx[row][2 * c + 1] = Ds[row][c] + Ds[row][c + 1];
    }
    __syncthreads();
    if (!mine) return;
    double s[TM_Z];
#pragma unroll
    for (int c = 0; c < TM_Z; ++c) s[c] = Sx[c * TM_Y + (fy >> 1)][fx];
    // (a loop in place of a branch: opaque in reduce.cuh)
    const int odd = opaque(fy & 1);
#pragma unroll 1
    for (int once = 0; once < odd; ++once) {
#pragma unroll
        for (int c = 0; c < TM_Z; ++c) s[c] += Sx[c * TM_Y + (fy >> 1) + 1][fx];
    }
    // 1 / (3 2^m) or 1 / (4 2^m), m = number of odd coordinates (tiles start on even ones)
    const int m = (fx & 1) + (fy & 1);
    const double w0 = kQuarter ? (m == 0 ? 0.25 : m == 1 ? 0.125 : 0.0625)
                               : (m == 0 ? 1.0 / 3.0 : m == 1 ? 1.0 / 6.0 : 1.0 / 12.0);
    const double w1 = kQuarter ? (m == 0 ? 0.125 : m == 1 ? 0.0625 : 0.03125)
                               : (m == 0 ? 1.0 / 6.0 : m == 1 ? 1.0 / 12.0 : 1.0 / 24.0);
#pragma unroll
    for (int k = 0; k < TT_Z; ++k)
        if (k < kz) {
            const int c = k >> 1;
            out[o + k * plane] = (k & 1) ? __fma_rn(s[c] + s[c + 1], w1, uv[k]) : __fma_rn(s[c], w0, uv[k]);
        }
}

// the Lagrange value at local offset 1 (first) or 3 of a cell of four fine
// intervals with middle-grid values a, b, c
__device__ __forceinline__ double quad_odd(bool first, double a, double b, double c) {
    const double wa = first ? 0.375 : -0.125, wc = first ? -0.125 : 0.375;
    return __fma_rn(wc, c, __fma_rn(0.75, b, wa * a));
}

// Step 5 at every fine node of the tile: even coordinates are middle-grid
// nodes, odd ones take three products per axis.  EXP_finite at 512^3: 0.87 ms
// (1.14 with predicated products along y).  Along x a warp forms the
// odd nodes of two rows at a time.
__global__ void __launch_bounds__(TT_THREADS)
exp_finite_interp_tiled_kernel(double* __restrict__ w, const double* __restrict__ W, int nf) {
    __shared__ double Ws[TM_Z * TM_Y][TM_X];
    __shared__ double Tx[TM_Z * TM_Y + 1][TT_X];
    const int tid = threadIdx.x, fx = tid & 31, warp = tid >> 5, fy = tile_row(warp);
    const int np = nf + 1, np1 = nf / 2 + 1;
    const int xa = blockIdx.x * TT_X, ya = blockIdx.y * TT_Y, za = blockIdx.z * TT_Z;
    const int mx0 = xa >> 1, my0 = ya >> 1, mz0 = za >> 1;
    for (int e = tid; e < TM_Z * TM_Y * TM_X; e += TT_THREADS) {
        const int row = e / TM_X, ex = e - row * TM_X, ez = row / TM_Y, ey = row - ez * TM_Y;
        const int ci = mx0 + ex, cj = my0 + ey, ck = mz0 + ez;
        const double v = ci < np1 && cj < np1 && ck < np1 ? W[nidx(np1, ci, cj, ck)] : 0.0;
        Ws[row][ex] = v;
        if (ex < TT_X / 2) Tx[row][2 * ex] = v;
    }
    __syncthreads();
    for (int pair = warp; 2 * pair < TM_Z * TM_Y; pair += TT_Y) {
        const int row = 2 * pair + (fx >> 4), c = fx & 15, cell = c >> 1;
        if (row < TM_Z * TM_Y) {
            const double* const v = &Ws[row][2 * cell];
            Tx[row][2 * c + 1] = quad_odd((c & 1) == 0, v[0], v[1], v[2]);
        }
    }
    __syncthreads();
    const int i = xa + fx, j = ya + fy;
    if (i >= np || j >= np) return;
    double t[TM_Z];
#pragma unroll
    for (int c = 0; c < TM_Z; ++c) t[c] = Tx[c * TM_Y + (fy >> 1)][fx];
    const int odd = opaque(fy & 1);   // (a loop in place of a branch)
#pragma unroll 1
    for (int once = 0; once < odd; ++once) {
#pragma unroll
        for (int c = 0; c < TM_Z; ++c) {
            const int r0 = c * TM_Y + 2 * (fy >> 2);
            t[c] = quad_odd((fy & 2) == 0, Tx[r0][fx], Tx[r0 + 1][fx], Tx[r0 + 2][fx]);
        }
    }
    const int kz = min(TT_Z, np - za);
    const size_t o = nidx(np, i, j, za);
    const size_t plane = (size_t)np * np;
    const double h[2] = {0.75 * t[1], 0.75 * t[3]};
#pragma unroll
    for (int k = 0; k < TT_Z; ++k)
        if (k < kz) {
            // the two odd nodes of a cell share the middle product
            const int c = 2 * (k >> 2);
            w[o + k * plane] = (k & 1) == 0 ? t[k >> 1]
                               : (k & 2) == 0 ? __fma_rn(-0.125, t[c + 2], __fma_rn(0.375, t[c], h[k >> 2]))
                                              : __fma_rn(0.375, t[c + 2], __fma_rn(-0.125, t[c], h[k >> 2]));
        }
}

dim3 tiled_grid(int nf) {
    const int np = nf + 1;
    return dim3((np + TT_X - 1) / TT_X, (np + TT_Y - 1) / TT_Y, (np + TT_Z - 1) / TT_Z);
}

}  // namespace

cudaError_t launch_exp_finite(double* w, const double* u1, const double* u0, double* W_scratch,
                              int n_fine, cudaStream_t s) {
    const int n1 = n_fine / 2;
    extrapolate_tiled_kernel<true><<<tiled_grid(n1), TT_THREADS, 0, s>>>(W_scratch, u1, u0, n1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    exp_finite_interp_tiled_kernel<<<tiled_grid(n_fine), TT_THREADS, 0, s>>>(w, W_scratch, n_fine);
    return cudaGetLastError();
}

cudaError_t launch_exp_true(double* ut, const double* uh, const double* u2h, int n_fine,
                            cudaStream_t s) {
    extrapolate_tiled_kernel<false><<<tiled_grid(n_fine), TT_THREADS, 0, s>>>(ut, uh, u2h, n_fine);
    return cudaGetLastError();
}

}  // namespace excmg

// ---------------------------------------------------------------------------
// EXP_finite without allocation.
//
// Some callers cannot allocate device memory when they need this step: code
// whose device memory is all owned by an arena or planner that hands out no
// further blocks (a serving process that sized its pools up front, a job
// held to a hard device-memory budget), or code running where entering the
// CUDA allocator is not allowed (cudaMalloc and cudaFree may synchronise the
// device, which a callback or a latency-critical path must not do).  This
// variant keeps its only scratch -- the middle-grid values W -- in a fixed
// array compiled into the library.  Every GPU that loads the library holds
// that array (2.2 MB) until the process exits.
namespace {

constexpr int kNoAllocMaxFine = 128;
constexpr size_t kNoAllocW =
    (size_t)(kNoAllocMaxFine / 2 + 1) * (kNoAllocMaxFine / 2 + 1) * (kNoAllocMaxFine / 2 + 1);

static __device__ __align__(256) double g_noalloc_W[kNoAllocW];

// The array's device address on the current device.  In host code the name
// g_noalloc_W is only a host-side stand-in, so the address is looked up on
// every call: a cached address would go stale if the device's context were
// reset and the library's device code loaded again elsewhere.  The lookup
// allocates nothing; on a device's first call it also loads the library's
// device code there.
int noalloc_scratch(double** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_W);
    if (e != cudaSuccess || !p) {
        cudaGetLastError();
        return EXCMG_ERR_CUDA;
    }
    *out = (double*)p;
    return EXCMG_OK;
}

}  // namespace

extern "C" int extrapolate_interpolate_noalloc(int n_fine, const double* u_2h, const double* u_4h,
                                               double* w_h) {
    if (n_fine < 8 || n_fine % 4 || !u_2h || !u_4h || !w_h) return EXCMG_ERR_ARG;
    if (n_fine > kNoAllocMaxFine) return EXCMG_ERR_SIZE;
    double* W = nullptr;
    const int st = noalloc_scratch(&W);
    if (st != EXCMG_OK) return st;
    // every entry of W is written before it is read: nothing to clear
    cudaError_t e = excmg::launch_exp_finite(w_h, u_2h, u_4h, W, n_fine, nullptr);
    excmg::note_launches(2);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return EXCMG_ERR_CUDA;
    }
    return EXCMG_OK;
}
