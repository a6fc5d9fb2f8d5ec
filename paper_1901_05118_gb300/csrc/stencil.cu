// Matrix-free 25-point operator A_h of eq. (sec): the interior scheme of
// eq. (method1) with the fictitious nodes folded onto their mirrors by
// eq. (reflection2) (first kind) or eq. (reflection4) (second kind).
//
// Structure: each CTA owns a TX x TY block of (x, y) columns and marches
// along z.  One z-plane of the input (with a 2-node halo in x and y) sits in
// shared memory at a time; every thread turns it into its plane-local
// partial sums and adds them to five register accumulators, one per output
// plane z-2 .. z+2.  The 25 taps split by plane offset:
//   same plane:  (42 + sigma*c) u  - 12 (4 axis nbrs) + (4 nbrs at 2) + 2 (4 diagonals)
//   planes +-1:  -12 u + 2 (4 axis nbrs)
//   planes +-2:  u
// Values outside the interior (boundary nodes and beyond) read as zero: the
// known boundary values belong to the right-hand side.  A ghost folds onto
// its mirror node, which for every ghost of eq. (method1) is the row's own
// node (the +-2 tap of a node one step from a face), so the folding only
// changes the centre weight by sigma = +1 (first kind) or -1 (second kind)
// per axis on which the node is one step from a face.
//
// The transposed operator gathers over the mirrored tap set (p - d instead
// of p + d).  Each tap d has a partner -d of equal weight and the folding is
// diagonal, so this is the same arithmetic; the flag is kept so that A^T is
// applied as Alg. 2 asks (its shadow recurrence multiplies by A^T).
#include <initializer_list>
#include <utility>

#include "excmg_internal.cuh"
#include "grid_sync.cuh"
#include "march_fx.cuh"
#include "march_lap.cuh"
#include "reduce.cuh"

namespace excmg {
namespace {

constexpr int TX = 32;
constexpr int TY = 8;
constexpr int HX = TX + 4;
constexpr int HY = TY + 4;

template <bool kTranspose>
__global__ void __launch_bounds__(TX * TY)
stencil_f64_kernel(const double* __restrict__ u, double* __restrict__ y, const double* __restrict__ b,
                   int n, double sigma, int kz_per_cta, const int* __restrict__ skip) {
    if (skip != nullptr && *skip) return;
    __shared__ double tile[2][HY][HX];
    const int np = n + 1;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int i0 = 1 + blockIdx.x * TX, j0 = 1 + blockIdx.y * TY;
    const int kz0 = 1 + blockIdx.z * kz_per_cta;
    const int kz1 = min(kz0 + kz_per_cta, n);   // output planes [kz0, kz1)
    const int i = i0 + tx, j = j0 + ty;
    const bool active = (i <= n - 1) && (j <= n - 1);
    const int cxy = (i == 1) + (i == n - 1) + (j == 1) + (j == n - 1);
    // mirrored gather for the transpose: offset -d instead of +d
    const int sgn = kTranspose ? -1 : 1;

    double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0, acc4 = 0.0;
    int buf = 0;
    for (int zin = kz0 - 2; zin <= kz1 + 1; ++zin, buf ^= 1) {
        const bool zok = (zin >= 1) && (zin <= n - 1);
        for (int e = tid; e < HX * HY; e += TX * TY) {
            const int ly = e / HX, lx = e - ly * HX;
            const int gi = i0 - 2 + lx, gj = j0 - 2 + ly;
            double v = 0.0;
            if (zok && gi >= 1 && gi <= n - 1 && gj >= 1 && gj <= n - 1)
                v = u[((size_t)zin * np + gj) * np + gi];
            tile[buf][ly][lx] = v;
        }
        __syncthreads();
        const int cy = ty + 2, cx = tx + 2;
        const double a = tile[buf][cy][cx];
        const double n4 = tile[buf][cy][cx - sgn] + tile[buf][cy][cx + sgn] +
                          tile[buf][cy - sgn][cx] + tile[buf][cy + sgn][cx];
        const double f4 = tile[buf][cy][cx - 2 * sgn] + tile[buf][cy][cx + 2 * sgn] +
                          tile[buf][cy - 2 * sgn][cx] + tile[buf][cy + 2 * sgn][cx];
        const double d4 = tile[buf][cy - sgn][cx - sgn] + tile[buf][cy - sgn][cx + sgn] +
                          tile[buf][cy + sgn][cx - sgn] + tile[buf][cy + sgn][cx + sgn];
        const int cz = (zin == 1) + (zin == n - 1);
        const double centre = 42.0 + sigma * (double)(cxy + cz);
        const double p0 = centre * a - 12.0 * n4 + f4 + 2.0 * d4;
        const double p1 = -12.0 * a + 2.0 * n4;
        acc0 += a;
        acc1 += p1;
        acc2 += p0;
        acc3 += p1;
        acc4 += a;
        const int zo = zin - 2;   // this output plane has all five contributions now
        if (active && zo >= kz0 && zo < kz1) {
            const size_t o = ((size_t)zo * np + j) * np + i;
            y[o] = b ? (b[o] - acc0) : acc0;
        }
        acc0 = acc1;
        acc1 = acc2;
        acc2 = acc3;
        acc3 = acc4;
        acc4 = 0.0;
    }
}

// y = A u (K = kMarchApply), or y = b - A u (kMarchSub; as a run-time choice the
// subtraction went through the FP64 pipe in either case).  Two CTAs per SM, as
// with three the register limit costs a fifth more instructions: A u on 100^3 / 133^3
// / 512^3 37 / 50 / 969 us with two, 43 / 53 / 980 with three, 42 / 56 / 1006 with
// four (three, with b at run time: 45 / 57 / 1082).
template <MarchKind K>
__global__ void __launch_bounds__(PP_NT, 2)
stencil_apply_kernel(const double* __restrict__ u, double* __restrict__ y, const double* __restrict__ b, int n,
                     int sigma, int kz_per_cta, const int* __restrict__ skip) {
    extern __shared__ __align__(128) unsigned char march_smem[];
    if (skip != nullptr && *skip) return;
    const int kz0 = 1 + blockIdx.z * kz_per_cta;
    const MarchArrays a{u, nullptr, nullptr, nullptr, b, y, nullptr, nullptr, 0.0, nullptr};
    (void)lap_march<K, true>(a, n, sigma, blockIdx.x, blockIdx.y, kz0, min(kz0 + kz_per_cta, n), march_smem);
}

// Every CTA's share of rr = (r, r): the last one writes the sum to *out, and
// the start of a Bi-CG call (rho_0 = (r*_0, r_0) = rr, r*_0 = r_0) to st.
__device__ __forceinline__ void finish_norm(double v, double* partials, unsigned int* ticket, double* out,
                                            BicgState* st) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    const double s = block_sum(v, sh);
    if (publish_partials(&s, 1, partials, ticket, &am_last)) {
        const double rr = gather_partials(partials, 0, sh);
        if (thread0()) {
            *ticket = 0;
            if (out) *out = rr;
            if (st) {
                st->rho = st->rr = rr;
                st->iter = 0;
                st->alpha = st->beta = st->sigma = 0.0;
                const bool conv = sqrt(rr) <= st->tol * st->bnorm;
                st->done = (conv || st->max_iter <= 0) ? 1 : 0;
                st->status = conv ? kConverged : (st->max_iter <= 0 ? kCapped : kRunning);
            }
        }
    }
}

// r = b - A u: the start of a Bi-CG call, or (r, r) alone, which then writes
// nothing else.  Forming r, the copies p_0, r*_0, p*_0 and the norm in one pass
// took the start of a 512^3 call from 2.4 to 1.5 ms, the norm alone from 1.6 to
// 1.1 ms (residual kernel, cleared buffer, inner product).
template <MarchKind K>
__global__ void __launch_bounds__(PP_NT, 2)
stencil_residual_kernel(MarchArrays a, int n, int sigma, int kz_per_cta, double* partials, unsigned int* ticket,
                        double* out, BicgState* st) {
    extern __shared__ __align__(128) unsigned char march_smem[];
    const int kz0 = 1 + blockIdx.z * kz_per_cta;
    finish_norm(lap_march<K, true>(a, n, sigma, blockIdx.x, blockIdx.y, kz0, min(kz0 + kz_per_cta, n), march_smem),
                partials, ticket, out, st);
}

// Every CTA's share of sigma = (p*, A p); the last one forms alpha = rho / sigma (Alg. 2).
__device__ __forceinline__ void finish_sigma(double dot, double* partials, BicgState* st) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    const double sdot = block_sum(dot, sh);
    if (publish_partials(&sdot, 1, partials, &st->ticket, &am_last)) {
        const double sg = gather_partials(partials, 0, sh);
        if (thread0()) {
            const double rho = st->rho;
            st->sigma = sg;
            if (!(rho != 0.0 && isfinite(rho)) || !(sg != 0.0 && isfinite(sg))) {
                st->status = kBreakdown;
                st->done = 1;
            } else {
                st->alpha = rho / sg;
            }
            st->ticket = 0;
        }
    }
}

// The operator launch of Bi-CG on grids above 64^3, for calls that start from
// r*_0 = p*_0 = r_0 = p_0: q = A p (A^T p* is the same bits, as p* = p),
// sigma and alpha; K = kMarchDir: p = r + beta p_{k-1} and p* formed first
// (the fused schedule).  kElide: the shadow-elided mode (p, q only; the same
// sums).
template <MarchKind K, bool kElide>
__global__ void __launch_bounds__(PP_NT, 2)
stencil_step_kernel(MarchArrays a, int n, int sigma, int kz_per_cta, double* partials, BicgState* st) {
    extern __shared__ __align__(128) unsigned char march_smem[];
    if (st->done) return;
    const int kz0 = 1 + blockIdx.z * kz_per_cta;
    a.beta = st->beta;
    finish_sigma(lap_march<K, kElide>(a, n, sigma, blockIdx.x, blockIdx.y, kz0, min(kz0 + kz_per_cta, n), march_smem),
                 partials, st);
}

// The same for a caller-chosen r*_0: two fields, marched side by side
// (march_fx.cuh).
template <bool kDir>
__global__ void __launch_bounds__(FX_NT, 2)
stencil_two_field_kernel(MarchArrays a, double* qs, int n, int sigma, int kz_per_cta, double* partials, BicgState* st) {
    if (st->done) return;
    const int kz0 = 1 + blockIdx.z * kz_per_cta;
    const FxFields fl{{a.in, a.ins}, {a.out, qs}, {a.r, a.rs}, {a.pn, a.psn}, st->beta};
    finish_sigma(fx_march<2, true, kDir>(fl, nullptr, n, sigma, blockIdx.x, blockIdx.y, kz0,
                                         min(kz0 + kz_per_cta, n)),
                 partials, st);
}

// A u at one interior node (i, j, k) with the integer arithmetic, without
// shared memory: the node's own 25 taps are put on the scale of their
// largest exponent and summed exactly.  Used where grids are so small that
// a z-march would be all latency.  Every tap has its bounds check: a way round
// them for nodes away from the faces costs more than it saves (A u on 64^3 32.3
// against 28.9 us, on 17^3 21.3 against 20.3 us; 32 iterations of the general
// cooperative kernel on 16^3 940 against 650 us).
__device__ __forceinline__ double fx_point(const double* __restrict__ u, int n, int sigma, int i, int j, int k) {
    const int np = n + 1;
    auto val = [&](int a, int b, int c) -> double {
        if (a < 1 || a > n - 1 || b < 1 || b > n - 1 || c < 1 || c > n - 1) return 0.0;
        return u[((size_t)c * np + b) * np + a];
    };
    const double ctr = val(i, j, k);
    double ax[6], far[6], dg[12];
    ax[0] = val(i - 1, j, k); ax[1] = val(i + 1, j, k); ax[2] = val(i, j - 1, k);
    ax[3] = val(i, j + 1, k); ax[4] = val(i, j, k - 1); ax[5] = val(i, j, k + 1);
    far[0] = val(i - 2, j, k); far[1] = val(i + 2, j, k); far[2] = val(i, j - 2, k);
    far[3] = val(i, j + 2, k); far[4] = val(i, j, k - 2); far[5] = val(i, j, k + 2);
    dg[0] = val(i - 1, j - 1, k); dg[1] = val(i - 1, j + 1, k); dg[2] = val(i + 1, j - 1, k); dg[3] = val(i + 1, j + 1, k);
    dg[4] = val(i - 1, j, k - 1); dg[5] = val(i + 1, j, k - 1); dg[6] = val(i, j - 1, k - 1); dg[7] = val(i, j + 1, k - 1);
    dg[8] = val(i - 1, j, k + 1); dg[9] = val(i + 1, j, k + 1); dg[10] = val(i, j - 1, k + 1); dg[11] = val(i, j + 1, k + 1);
    int E = max(1, exponent_of(ctr));
#pragma unroll
    for (int t = 0; t < 6; ++t) E = max(E, max(exponent_of(ax[t]), exponent_of(far[t])));
#pragma unroll
    for (int t = 0; t < 12; ++t) E = max(E, exponent_of(dg[t]));
    long long s_ax = 0, s_far = 0, s_dg = 0;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        s_ax += to_fixed(ax[t], E);
        s_far += to_fixed(far[t], E);
    }
#pragma unroll
    for (int t = 0; t < 12; ++t) s_dg += to_fixed(dg[t], E);
    const int c = (i == 1) + (i == n - 1) + (j == 1) + (j == n - 1) + (k == 1) + (k == n - 1);
    const long long acc = (long long)(42 + sigma * c) * to_fixed(ctr, E) - 12 * s_ax + s_far + 2 * s_dg;
    return fx_result(acc, E, E == 0x7FF);
}

// The single-field forms (A u, b - A u, the start of a Bi-CG call, the norm)
// on small grids, node by node: one round of loads instead of a march of a
// dozen planes that wait for each other (17^3: 14 us).  Boundary nodes of the outputs are set
// to zero.
template <MarchKind K>
__global__ void __launch_bounds__(256)
stencil_point_kernel(MarchArrays a, int n, int sigma, const int* __restrict__ skip, double* partials,
                     unsigned int* ticket, double* out, BicgState* st) {
    if (skip != nullptr && *skip) return;
    const int np = n + 1, total = np * np * np;
    const int t = blockIdx.x * 256 + threadIdx.x;
    double v = 0.0;
    if (t < total) {
        const int k = t / (np * np), e = t - k * np * np, j = e / np, i = e - j * np;
        if (i > 0 && i < n && j > 0 && j < n && k > 0 && k < n) {
            v = fx_point(a.in, n, sigma, i, j, k);
            if (a.b) v = a.b[t] - v;
        }
        if (K == kMarchApply || K == kMarchSub) a.out[t] = v;
        if (K == kMarchStart) {
            if (a.words) a.words[t] = make_ulonglong2((unsigned long long)__double_as_longlong(v), 0ull);
            else a.out[t] = v;
            if (a.pn) a.pn[t] = v;
            if (a.rsn) a.rsn[t] = v;
            if (a.psn) a.psn[t] = v;
        }
    }
    if constexpr (K != kMarchApply && K != kMarchSub) finish_norm(v * v, partials, ticket, out, st);
}

// ---------------------------------------------------------------------------
// Bi-CG iterations of a small grid in one cooperative launch.  On grids of a
// few tens of thousands of unknowns every kernel of an iteration lasts a few
// microseconds and launch gaps dominate; here all CTAs stay resident and run
// the three phases of an iteration (operator pair + sigma, x/r/r* update +
// (r*, r), (r, r), direction update) separated by grid barriers.  Every CTA
// adds the per-CTA partial sums itself, in CTA order, so all CTAs derive the
// same alpha, beta and stopping decision.  The barrier spins a bounded
// number of times; if it gives up, every CTA leaves and the state reports a
// timeout.
struct BicgVectors {
    double* x;
    double* r;
    double* rs;
    double* p;
    double* ps;
    double* q;
    double* qs;
};

// Sum of component c of the per-CTA partials, in CTA order (every CTA).
__device__ __forceinline__ double all_partials(const double* partials, int c, double* sh) {
    const int G = flat_grid();
    const int nthreads = blockDim.x * blockDim.y * blockDim.z;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    double v = 0.0;
    for (int b = tid; b < G; b += nthreads) v += __ldcg(&partials[c * G + b]);
    v = block_sum(v, sh);
    __shared__ double bc;
    if (thread0()) bc = v;
    __syncthreads();
    v = bc;
    __syncthreads();
    return v;
}

// Three phases per iteration: operator pair with sigma; x, r, r* update
// with (r*, r) and (r, r); direction update.
template <bool kPointwise>
__global__ void __launch_bounds__(FX_NT, 2)
bicg_persistent_kernel(BicgVectors v, size_t len, int n, int sigma, int gx, int gy, int slabs, int kz_per,
                       int iters, double* partials, BicgState* st, GridBarrier gb) {
    __shared__ double sh[32];
    const unsigned int G = gridDim.x;
    const int units = gx * gy * slabs;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int nthreads = blockDim.x * blockDim.y;
    double rho = st->rho, rr = st->rr, alpha = st->alpha, beta = st->beta, sigma_s = st->sigma;
    int iter = st->iter, status = st->status, done = st->done;
    const int max_iter = st->max_iter;
    const double stop = st->tol * st->bnorm;
    bool ok = true;
    for (int it = 0; it < iters && !done && ok; ++it) {
        // phase A: q = A p, qs = A^T ps, sigma = (ps, q); per node on the
        // smallest grids, by z-marching tiles otherwise
        double dot = 0.0;
        if (kPointwise) {
            const int m = n - 1, np = n + 1;
            const long long pts = (long long)m * m * m;
            for (long long t = (long long)blockIdx.x * nthreads + tid; t < pts; t += (long long)G * nthreads) {
                const int i = (int)(t % m) + 1, j = (int)((t / m) % m) + 1, k = (int)(t / ((long long)m * m)) + 1;
                const size_t o = ((size_t)k * np + j) * np + i;
                const double qv = fx_point(v.p, n, sigma, i, j, k);
                v.q[o] = qv;
                v.qs[o] = fx_point(v.ps, n, sigma, i, j, k);
                dot += v.ps[o] * qv;
            }
        } else {
            for (int u = blockIdx.x; u < units; u += G) {
                const int bx = u % gx, by = (u / gx) % gy, bz = u / (gx * gy);
                const int kz0 = 1 + bz * kz_per;
                const int kz1 = min(kz0 + kz_per, n);
                __syncthreads();   // the CTA's previous unit is done with the shared buffers
                const FxFields fl{{v.p, v.ps}, {v.q, v.qs}, {nullptr, nullptr}, {nullptr, nullptr}, 0.0};
                dot += fx_march<2, true>(fl, nullptr, n, sigma, bx, by, kz0, kz1);
            }
        }
        dot = block_sum(dot, sh);
        if (thread0()) partials[blockIdx.x] = dot;
        if (!(ok = grid_sync(gb, G))) break;
        sigma_s = all_partials(partials, 0, sh);
        if (!(rho != 0.0 && isfinite(rho)) || !(sigma_s != 0.0 && isfinite(sigma_s))) {
            status = kBreakdown;
            done = 1;
            break;
        }
        alpha = rho / sigma_s;
        // phase B: x += alpha p; r -= alpha q; r* -= alpha q*; (r*, r), (r, r)
        // (entries t, t + S of this thread loaded together,
        // then updated and summed in index order)
        double vr = 0.0, vrr = 0.0;
        const double* const pcur = v.p;
        bool twin = true;   // as in bicg_update_kernel: vr == vrr so far
        const size_t S = (size_t)G * nthreads;
        constexpr int kB = kPointwise ? 1 : 2;   // entries per thread loaded together
        for (size_t t0 = (size_t)blockIdx.x * nthreads + tid; t0 < len; t0 += kB * S) {
            double xv[kB], pv[kB], rv[kB], qv[kB], rsv[kB], qsv[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                const size_t t = t0 + k * S;
                if (t < len) {
                    xv[k] = v.x[t];
                    pv[k] = pcur[t];
                    rv[k] = v.r[t];
                    qv[k] = v.q[t];
                    rsv[k] = v.rs[t];
                    qsv[k] = v.qs[t];
                }
            }
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                const size_t t = t0 + k * S;
                if (t >= len) break;
                v.x[t] = xv[k] + alpha * pv[k];
                const double rn = rv[k] - alpha * qv[k];
                v.r[t] = rn;
                if (__double_as_longlong(rsv[k]) == __double_as_longlong(rv[k]) &&
                    __double_as_longlong(qsv[k]) == __double_as_longlong(qv[k])) {
                    v.rs[t] = rn;
                    if (twin) {
                        vrr += rn * rn;
                    } else {
                        vr += rn * rn;
                        vrr += rn * rn;
                    }
                } else {
                    if (twin) {
                        vr = vrr;
                        twin = false;
                    }
                    const double rsn = rsv[k] - alpha * qsv[k];
                    v.rs[t] = rsn;
                    vr += rsn * rn;
                    vrr += rn * rn;
                }
            }
        }
        if (twin) vr = vrr;
        vr = block_sum(vr, sh);
        vrr = block_sum(vrr, sh);
        if (thread0()) {
            partials[G + blockIdx.x] = vr;
            partials[2 * G + blockIdx.x] = vrr;
        }
        if (!(ok = grid_sync(gb, G))) break;
        const double rho_new = all_partials(partials, 1, sh);
        rr = all_partials(partials, 2, sh);
        beta = rho_new / rho;
        rho = rho_new;
        ++iter;
        if (sqrt(rr) <= stop) {
            status = kConverged;
            done = 1;
            break;
        }
        if (iter >= max_iter) {
            status = kCapped;
            done = 1;
            break;
        }
        {
            // phase C: p = r + beta p; p* = r* + beta p*
            for (size_t t0 = (size_t)blockIdx.x * nthreads + tid; t0 < len; t0 += kB * S) {
                double rv[kB], pv[kB], rsv[kB], psv[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const size_t t = t0 + k * S;
                    if (t < len) {
                        rv[k] = v.r[t];
                        pv[k] = v.p[t];
                        rsv[k] = v.rs[t];
                        psv[k] = v.ps[t];
                    }
                }
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const size_t t = t0 + k * S;
                    if (t >= len) break;
                    v.p[t] = rv[k] + beta * pv[k];
                    v.ps[t] = rsv[k] + beta * psv[k];
                }
            }
            if (!(ok = grid_sync(gb, G))) break;
        }
    }
    if (blockIdx.x == 0 && thread0()) {
        if (!ok) {
            status = kTimeout;
            done = 1;
        }
        st->rho = rho;
        st->rr = rr;
        st->alpha = alpha;
        st->beta = beta;
        st->sigma = sigma_s;
        st->iter = iter;
        st->status = status;
        st->done = done;
    }
}

__global__ void zero_boundary_kernel(BoundaryArrays arrays, int n) {
    // one thread per node of the six faces (faces overlap at edges: harmless)
    const int np = n + 1;
    const size_t per_face = (size_t)np * np;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < 6 * per_face;
         t += (size_t)gridDim.x * blockDim.x) {
        const int face = (int)(t / per_face);
        const size_t r = t - face * per_face;
        const int a = (int)(r % np), bb = (int)(r / np);
        const int fixed = (face & 1) ? n : 0;
        int i, j, k;
        if (face < 2) { i = fixed; j = a; k = bb; }
        else if (face < 4) { i = a; j = fixed; k = bb; }
        else { i = a; j = bb; k = fixed; }
        const size_t o = ((size_t)k * np + j) * np + i;
        for (double* y : arrays.a)
            if (y) y[o] = 0.0;
    }
}

}  // namespace

namespace {

struct StencilGrid {
    dim3 grid, block;
    int kz_per_cta;
    size_t smem = 0;   // dynamic shared memory per CTA
};

// Column tiles x z-slabs.  The slab count is chosen so that the CTAs fill
// whole waves of the GPU's resident slots (SMs x CTAs per SM) while each
// slab stays long enough that its 4 extra halo planes cost little.
StencilGrid stencil_grid(int n, int tx, int rows, int per_sm) {
    const int m = n - 1;  // interior extent
    StencilGrid g;
    const int gx = (m + tx - 1) / tx, gy = (m + rows - 1) / rows;
    const int tiles = gx * gy;
    const int slots = device_sms() * (per_sm > 0 ? per_sm : 1);
    int best = 1;
    double best_eff = -1.0;
    for (int slabs = 1; slabs <= 64; ++slabs) {
        const int planes = (m + slabs - 1) / slabs;
        if (slabs > 1 && planes < 8) break;
        const long long ctas = (long long)tiles * slabs;
        if (slabs > 1 && ctas > 4096) break;   // keeps the fused reductions' partials small
        const long long waves = (ctas + slots - 1) / slots;
        const double eff = (double)ctas / (double)(waves * slots) * planes / (planes + 4.0);
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = slabs;
        }
    }
    g.kz_per_cta = (m + best - 1) / best;
    const int slabs = (m + g.kz_per_cta - 1) / g.kz_per_cta;
    g.grid = dim3(gx, gy, slabs);
    return g;
}

// Resident CTAs per SM of a kernel on the current device (cached per
// kernel and device; opts the kernel in to `smem` bytes of dynamic shared
// memory there first).  Function attributes belong to each device's
// context, so the staged launches call this before every launch.
template <typename K>
int resident_per_sm(K kernel, int threads, size_t smem = 0) {
    return kernel_occupancy((const void*)kernel, threads, smem);
}

StencilGrid march_grid(int n, int per_sm, size_t smem) {
    StencilGrid g = stencil_grid(n, PP_TX, PP_OY, per_sm);
    g.block = dim3(PP_TX, PP_TY, 1);
    g.smem = smem;
    return g;
}

// The single-field operator launch (A u, b - A u).
template <MarchKind K>
StencilGrid apply_grid(int n) {
    constexpr size_t smem = MarchStage<K, true>::kSmem;
    return march_grid(n, resident_per_sm(stencil_apply_kernel<K>, PP_NT, smem), smem);
}

// Node-by-node form of the single-field launches: as long as all nodes are
// in flight at once it takes one memory latency, the march a dozen.
constexpr int kPointFormMaxN = 64;
bool point_form(int n) { return n <= kPointFormMaxN; }
int point_blocks(int n) { return (int)((node_count(n) + 255) / 256); }

// The operator step of Bi-CG: every form of it runs on the grid of the
// two-field one with directions, so that sigma adds the same per-CTA
// partial sums in the shadow-elided mode.
template <MarchKind K, bool kElide>
StencilGrid step_grid(int n) {
    constexpr size_t full = MarchStage<kMarchDir, false>::kSmem;
    const int occ = resident_per_sm(stencil_step_kernel<kMarchDir, false>, PP_NT, full);
    constexpr size_t smem = MarchStage<K, kElide>::kSmem;
    (void)resident_per_sm(stencil_step_kernel<K, kElide>, PP_NT, smem);
    return march_grid(n, occ, smem);
}

StencilGrid f64_grid(int n) {
    const int occ = resident_per_sm(stencil_f64_kernel<false>, TX * TY);
    StencilGrid g = stencil_grid(n, TX, TY, occ);
    g.block = dim3(TX, TY, 1);
    return g;
}

}  // namespace

int stencil_cta_count(int n) {
    const StencilGrid g1 = apply_grid<kMarchApply>(n), g2 = step_grid<kMarchDir, false>(n);
    unsigned most = max(g1.grid.x * g1.grid.y * g1.grid.z, g2.grid.x * g2.grid.y * g2.grid.z);
    const StencilGrid g3 = march_grid(n, 2, 0);   // the residual launches: two CTAs per SM
    most = max(most, g3.grid.x * g3.grid.y * g3.grid.z);
    return (int)most;
}

cudaError_t launch_stencil(const double* u, double* y, const double* b, int n, int bc_kind,
                           bool transpose, const int* skip, cudaStream_t s, int variant) {
    if (variant == kStencilFp64) {
        const StencilGrid g = f64_grid(n);
        const double sigma = bc_kind == 1 ? 1.0 : -1.0;
        if (transpose)
            stencil_f64_kernel<true><<<g.grid, g.block, 0, s>>>(u, y, b, n, sigma, g.kz_per_cta, skip);
        else
            stencil_f64_kernel<false><<<g.grid, g.block, 0, s>>>(u, y, b, n, sigma, g.kz_per_cta, skip);
    } else {
        // A^T u == A u bit for bit in integer arithmetic (see above)
        (void)transpose;
        const int sg = bc_kind == 1 ? 1 : -1;
        if (point_form(n)) {
            const MarchArrays a{u, nullptr, nullptr, nullptr, b, y, nullptr, nullptr, 0.0, nullptr};
            stencil_point_kernel<kMarchApply><<<point_blocks(n), 256, 0, s>>>(a, n, sg, skip, nullptr, nullptr,
                                                                              nullptr, nullptr);
        } else {
            const StencilGrid g = b ? apply_grid<kMarchSub>(n) : apply_grid<kMarchApply>(n);
            (b ? stencil_apply_kernel<kMarchSub> : stencil_apply_kernel<kMarchApply>)<<<g.grid, g.block, g.smem, s>>>(
                u, y, b, n, sg, g.kz_per_cta, skip);
        }
    }
    return cudaGetLastError();
}

namespace {
template <MarchKind K>
cudaError_t launch_residual(const MarchArrays& a, int n, int bc_kind, double* partials, unsigned int* ticket,
                            double* out, BicgState* st, cudaStream_t s) {
    const int sg = bc_kind == 1 ? 1 : -1;
    if (point_form(n)) {
        stencil_point_kernel<K><<<point_blocks(n), 256, 0, s>>>(a, n, sg, nullptr, partials, ticket, out, st);
    } else {
        constexpr size_t smem = MarchStage<K, true>::kSmem;
        const StencilGrid g = march_grid(n, resident_per_sm(stencil_residual_kernel<K>, PP_NT, smem), smem);
        stencil_residual_kernel<K><<<g.grid, g.block, g.smem, s>>>(a, n, sg, g.kz_per_cta, partials, ticket, out, st);
    }
    return cudaGetLastError();
}
}  // namespace

bool stencil_writes_boundary(int n, int variant) { return variant == kStencilExact && point_form(n); }

cudaError_t launch_residual_norm(const double* x, const double* b, int n, int bc_kind, double* partials,
                                 unsigned int* ticket, double* out, cudaStream_t s) {
    const MarchArrays a{x, nullptr, nullptr, nullptr, b, nullptr, nullptr, nullptr, 0.0, nullptr};
    return launch_residual<kMarchNorm>(a, n, bc_kind, partials, ticket, out, nullptr, s);
}

cudaError_t launch_bicg_start(const double* x, const double* b, int n, int bc_kind, double* r, double* rs, double* p,
                              double* ps, void* words, double* partials, unsigned int* ticket, double* out,
                              BicgState* st, cudaStream_t s) {
    const MarchArrays a{x, nullptr, nullptr, nullptr, b, r, p, ps, 0.0, rs, (ulonglong2*)words};
    return launch_residual<kMarchStart>(a, n, bc_kind, partials, ticket, out, st, s);
}

constexpr int kPointwiseMaxN = 32;   // per-node operator on grids up to 32^3

int persistent_grid(int n, int* gx, int* gy, int* slabs, int* kz_per) {
    const int occ_pt = min(2, resident_per_sm(bicg_persistent_kernel<true>, FX_NT));
    const int sms = device_sms();
    const int m = n - 1;
    *gx = (m + FX_TX - 1) / FX_TX;
    *gy = (m + FX_OY - 1) / FX_OY;
    *kz_per = m < 8 ? m : (n <= 64 ? 4 : 8);
    *slabs = (m + *kz_per - 1) / *kz_per;
    if (n > kPointwiseMaxN) {
        // z-march: one CTA per SM, and the shortest slabs (at least two
        // planes) that still give every CTA at most one unit per phase.
        // Measured on 48^3 / 64^3: 22.2 / 27.9 us per iteration, against
        // 31.5 / 34.4 with two CTAs per SM and 4-plane slabs (longer waits
        // at the grid barriers, units the CTAs take in two rounds).
        const int G = sms;
        for (int k = 2; k <= 8; ++k) {
            *kz_per = k;
            *slabs = (m + k - 1) / k;
            if ((*gx) * (*gy) * (*slabs) <= G) break;
        }
        return G;
    }
    // one CTA per ~256 interior nodes, at most every resident slot: fewer
    // CTAs keep the grid barriers short on small grids
    const long long pts = (long long)m * m * m;
    long long want = (pts + 255) / 256;
    if (want < 8) want = 8;
    if (want > (long long)sms * occ_pt) want = (long long)sms * occ_pt;
    return (int)want;
}

cudaError_t launch_bicg_persistent(double* x, double* r, double* rs, double* p, double* ps, double* q, double* qs,
                                   int n, int bc_kind, int iters, double* partials, BicgState* st,
                                   unsigned int* barrier_words, cudaStream_t s) {
    int gx, gy, slabs, kz_per;
    const int G = persistent_grid(n, &gx, &gy, &slabs, &kz_per);
    cudaError_t e = cudaMemsetAsync(barrier_words, 0, 3 * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    BicgVectors v{x, r, rs, p, ps, q, qs};
    size_t len = node_count(n);
    int sigma = bc_kind == 1 ? 1 : -1;
    GridBarrier gb{barrier_words, barrier_words + 1, (int*)(barrier_words + 2), kBarrierSpinLimit};
    void* args[] = {&v, &len, &n, &sigma, &gx, &gy, &slabs, &kz_per, &iters, &partials, &st, &gb};
    const void* fn = n <= kPointwiseMaxN ? (const void*)bicg_persistent_kernel<true>
                                         : (const void*)bicg_persistent_kernel<false>;
    return cudaLaunchCooperativeKernel(fn, dim3(G), dim3(FX_TX, FX_TY, 1), args, 0, s);
}

cudaError_t launch_bicg_stencil_pair_dir(const double* r, const double* rs, const double* p_prev,
                                         const double* ps_prev, double* p, double* ps, double* q, double* qs, int n,
                                         int bc_kind, double* partials, BicgState* st, cudaStream_t s) {
    const MarchArrays a{p_prev, r, ps_prev, rs, nullptr, q, p, ps, 0.0, nullptr};
    const int sg = bc_kind == 1 ? 1 : -1;
    const StencilGrid g = step_grid<kMarchDir, false>(n);
    if (qs == nullptr)
        stencil_step_kernel<kMarchDir, false><<<g.grid, g.block, g.smem, s>>>(a, n, sg, g.kz_per_cta, partials, st);
    else
        stencil_two_field_kernel<true><<<g.grid, g.block, 0, s>>>(a, qs, n, sg, g.kz_per_cta, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_bicg_stencil_pair(const double* p, double* q, const double* ps, double* qs, int n,
                                     int bc_kind, double* partials, BicgState* st, cudaStream_t s) {
    const MarchArrays a{p, nullptr, ps, nullptr, nullptr, q, nullptr, nullptr, 0.0, nullptr};
    const int sg = bc_kind == 1 ? 1 : -1;
    const StencilGrid g = step_grid<kMarchPair, false>(n);
    if (qs == nullptr)
        stencil_step_kernel<kMarchPair, false><<<g.grid, g.block, g.smem, s>>>(a, n, sg, g.kz_per_cta, partials, st);
    else
        stencil_two_field_kernel<false><<<g.grid, g.block, 0, s>>>(a, qs, n, sg, g.kz_per_cta, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_cg_stencil(const double* p, double* q, int n, int bc_kind, double* partials, BicgState* st,
                              cudaStream_t s) {
    const MarchArrays a{p, nullptr, nullptr, nullptr, nullptr, q, nullptr, nullptr, 0.0, nullptr};
    const StencilGrid g = step_grid<kMarchPair, true>(n);
    stencil_step_kernel<kMarchPair, true><<<g.grid, g.block, g.smem, s>>>(a, n, bc_kind == 1 ? 1 : -1, g.kz_per_cta,
                                                                         partials, st);
    return cudaGetLastError();
}

cudaError_t launch_cg_stencil_dir(const double* r, const double* p_prev, double* p, double* q, int n, int bc_kind,
                                  double* partials, BicgState* st, cudaStream_t s) {
    const MarchArrays a{p_prev, r, nullptr, nullptr, nullptr, q, p, nullptr, 0.0, nullptr};
    const StencilGrid g = step_grid<kMarchDir, true>(n);
    stencil_step_kernel<kMarchDir, true><<<g.grid, g.block, g.smem, s>>>(a, n, bc_kind == 1 ? 1 : -1, g.kz_per_cta,
                                                                        partials, st);
    return cudaGetLastError();
}

cudaError_t launch_zero_boundary(const BoundaryArrays& arrays, int n, cudaStream_t s) {
    const size_t total = 6 * (size_t)(n + 1) * (n + 1);
    int blocks = (int)((total + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    zero_boundary_kernel<<<blocks, 256, 0, s>>>(arrays, n);
    return cudaGetLastError();
}

}  // namespace excmg
