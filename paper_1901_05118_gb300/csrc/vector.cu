// Vector kernels of Bi-CG (Alg. 2, M = I): the inner products, the iterate
// and residual updates and the direction updates, with the scalars alpha and
// beta formed on the device.
//
// Reductions are deterministic: a fixed grid (kVecBlocks x kVecThreads)
// walks the vectors with a grid stride, each CTA reduces its values by a
// fixed shuffle tree, and the last CTA to finish (atomic ticket) adds the
// per-CTA partials in CTA order.  The same inputs therefore always give the
// same bits, independent of scheduling.  Multiply-adds are written out, so
// that every variant of a kernel rounds alike.
#include "excmg_internal.cuh"
#include "reduce.cuh"

namespace excmg {
namespace {

// Each thread loads kLd entries, one grid stride apart, before it works on
// them in index order: the sums are those of one entry at a time, but with two
// entries twice as many bytes are in flight.  At 512^3 the update moves 64 B per entry
// at 0.95 of the measured copy bandwidth or more with two entries (1.3 ms; one
// entry: 1.6 ms, three 0.1 ms slower, four at four CTAs per SM: 1.61 ms), and more CTAs
// per SM do not help (1.34-1.5 ms).
//
// Vectors of fewer than kPairStrides grid strides (1.87 million entries) go one
// entry at a time: they lie in L2, and a last group of two that is half empty costs a
// whole one, as its predicated FP64 instructions hold the pipe.  One against two entries:
// 60 2D iterations on 580^2 1.95 / 2.18 ms, on 900^2 2.64 / 2.77, on 1400^2 4.47 / 4.37;
// 40 elided ones on 100^3 1.76 / 1.83, on 120^3 2.17 / 2.25, 40 of the separate schedule on
// 130^3 3.50 / 3.40, on 160^3 5.38 / 5.13.  (A loop of its own for the entries that do
// not fill a group: as fast as one below the line, 2 to 4 % slower than two above it.)
constexpr size_t kPairStrides = 12;
inline bool load_pairs(size_t len) { return len >= kPairStrides * kVecBlocks * kVecThreads; }
#define EXCMG_STRIDED(t0, S) \
    const size_t S = (size_t)gridDim.x * blockDim.x; \
    for (size_t t0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t0 < len; t0 += kLd * S)

template <int kLd>
__global__ void __launch_bounds__(kVecThreads)
dot_kernel(const double* __restrict__ a, const double* __restrict__ b, size_t len,
           double* partials, unsigned int* ticket, double* out) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    double v = 0.0;
    EXCMG_STRIDED(t0, S) {
        double av[kLd], bv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            av[k] = t < len ? a[t] : 0.0;
            bv[k] = t < len ? b[t] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) v = __fma_rn(av[k], bv[k], v);
    }
    double s = block_sum(v, sh);
    if (publish_partials(&s, 1, partials, ticket, &am_last)) {
        const double tot = gather_partials(partials, 0, sh);
        if (thread0()) {
            *out = tot;
            *ticket = 0;
        }
    }
}

// (a, a) over the unknowns (interior nodes) of a grid with n intervals:
// for caller-supplied vectors whose boundary entries need not be zero.
__global__ void __launch_bounds__(kVecThreads)
interior_dot_kernel(const double* __restrict__ a, int n, double* partials, unsigned int* ticket, double* out) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    // one warp per row of m nodes: an index split into three by 64-bit
    // divisions per node took 0.71 ms at 512^3
    const int m = n - 1, np = n + 1, lane = threadIdx.x & 31;
    const int rows = m * m, warps = gridDim.x * (kVecThreads / 32);
    double v = 0.0;
    for (int row = blockIdx.x * (kVecThreads / 32) + (threadIdx.x >> 5); row < rows; row += warps) {
        const int k = row / m, j = row - k * m;
        const double* const ar = a + ((size_t)(k + 1) * np + j + 1) * np + 1;
        for (int i = lane; i < m; i += 32) {
            const double x = ar[i];
            v = __fma_rn(x, x, v);
        }
    }
    double s = block_sum(v, sh);
    if (publish_partials(&s, 1, partials, ticket, &am_last)) {
        const double tot = gather_partials(partials, 0, sh);
        if (thread0()) {
            *out = tot;
            *ticket = 0;
        }
    }
}

// r*_0 = shadow (or r_0), p_0 = r_0, p*_0 = r*_0; rho_0 = (r*_0, r_0),
// rr = (r_0, r_0); st->twin: the shadow is r_0 bit for bit at every unknown of a
// grid with n intervals (the boundary entries may hold anything; the index of an entry is
// split only where the bits differ, and once per thread where that is inside).
template <int kLd>
__global__ void __launch_bounds__(kVecThreads)
bicg_init_kernel(const double* __restrict__ r, const double* __restrict__ shadow, double* __restrict__ rs,
                 double* __restrict__ p, double* __restrict__ ps, size_t len, int n, double* partials, BicgState* st) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    double vr = 0.0, vrr = 0.0;
    const size_t np = (size_t)n + 1;
    auto inner = [&](size_t v) { return v >= 1 && v < (size_t)n; };
    bool differs = false;
    EXCMG_STRIDED(t0, S) {
        double rv[kLd], sv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) {
                rv[k] = r[t];
                sv[k] = shadow ? shadow[t] : rv[k];
            }
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t >= len) break;
            if (!differs && __double_as_longlong(sv[k]) != __double_as_longlong(rv[k]))
                differs = inner(t % np) && inner(t / np % np) && inner(t / (np * np));
            rs[t] = sv[k];
            p[t] = rv[k];
            ps[t] = sv[k];
            vr = __fma_rn(sv[k], rv[k], vr);
            vrr = __fma_rn(rv[k], rv[k], vrr);
        }
    }
    double s2[3];
    s2[0] = block_sum(vr, sh);
    s2[1] = block_sum(vrr, sh);
    s2[2] = __syncthreads_or(differs) ? 1.0 : 0.0;
    if (publish_partials(s2, 3, partials, &st->ticket, &am_last)) {
        const double rho = gather_partials(partials, 0, sh);
        const double rr = gather_partials(partials, 1, sh);
        const double off = gather_partials(partials, 2, sh);
        if (thread0()) {
            st->twin = off == 0.0;
            st->rho = rho;
            st->rr = rr;
            st->iter = 0;
            st->alpha = st->beta = st->sigma = 0.0;
            const bool conv = sqrt(rr) <= st->tol * st->bnorm;
            st->done = (conv || st->max_iter <= 0) ? 1 : 0;
            st->status = conv ? kConverged : (st->max_iter <= 0 ? kCapped : kRunning);
            st->ticket = 0;
        }
    }
}

// sigma_k = (p*_k, A p_k); alpha_k = rho_k / sigma_k.
__global__ void __launch_bounds__(kVecThreads)
bicg_sigma_kernel(const double* __restrict__ ps, const double* __restrict__ q, size_t len,
                  double* partials, BicgState* st) {
    if (st->done) return;
    __shared__ double sh[32];
    __shared__ bool am_last;
    double v = 0.0;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < len;
         t += (size_t)gridDim.x * blockDim.x)
        v += ps[t] * q[t];
    double s = block_sum(v, sh);
    if (publish_partials(&s, 1, partials, &st->ticket, &am_last)) {
        const double sigma = gather_partials(partials, 0, sh);
        if (thread0()) {
            const double rho = st->rho;
            st->sigma = sigma;
            if (!(rho != 0.0 && isfinite(rho)) || !(sigma != 0.0 && isfinite(sigma))) {
                st->status = kBreakdown;
                st->done = 1;
            } else {
                st->alpha = rho / sigma;
            }
            st->ticket = 0;
        }
    }
}

// x += alpha p; r -= alpha A p; r* -= alpha A^T p*;
// rho_{k+1} = (r*, r), beta = rho_{k+1} / rho_k; stopping test on ||r||.
// Where r* and A^T p* equal r and A p bit for bit (always so with
// r*_0 = r_0 and the integer operator) the shadow update gives the same
// bits as the primal one and the product r* r equals r r, so it is formed
// once; a thread that meets a differing entry continues with separate sums
// from the identical partial sums it has so far.  FP64 issue is scarce on
// GB300: this saves two of the five FMAs per entry.
// kOneQ: A^T p* is A p bit for bit and read once, from q (r* is r then, too;
// compared on principle, as in resident.cuh).
template <int kLd, bool kOneQ>
__global__ void __launch_bounds__(kVecThreads)
bicg_update_kernel(double* __restrict__ x, const double* __restrict__ p, double* __restrict__ r,
                   const double* __restrict__ q, double* __restrict__ rs,
                   const double* __restrict__ qs, size_t len, double* partials, BicgState* st) {
    if (st->done) return;
    __shared__ double sh[32];
    __shared__ bool am_last;
    const double alpha = st->alpha;
    double vr = 0.0, vrr = 0.0;
    bool twin = true;   // so far every entry of this thread was a twin: vr == vrr
    EXCMG_STRIDED(t0, S) {
        double xv[kLd], pv[kLd], rv[kLd], qv[kLd], rsv[kLd], qsv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) {
                rv[k] = r[t];
                qv[k] = q[t];
                rsv[k] = rs[t];
                qsv[k] = kOneQ ? qv[k] : qs[t];
                xv[k] = x[t];
                pv[k] = p[t];
            }
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t >= len) break;
            const double rn = __fma_rn(-alpha, qv[k], rv[k]);
            r[t] = rn;
            double rsn = rn;
            if (!twin || __double_as_longlong(rsv[k]) != __double_as_longlong(rv[k]) ||
                __double_as_longlong(qsv[k]) != __double_as_longlong(qv[k])) {
                if (twin) {
                    vr = vrr;
                    twin = false;
                }
                rsn = fma_here(-alpha, qsv[k], rsv[k]);
                vr = fma_here(rsn, rn, vr);
            }
            rs[t] = rsn;
            vrr = __fma_rn(rn, rn, vrr);
            x[t] = __fma_rn(alpha, pv[k], xv[k]);
        }
    }
    if (twin) vr = vrr;
    double s[2];
    s[0] = block_sum(vr, sh);
    s[1] = block_sum(vrr, sh);
    if (publish_partials(s, 2, partials, &st->ticket, &am_last)) {
        const double rho_new = gather_partials(partials, 0, sh);
        const double rr = gather_partials(partials, 1, sh);
        if (thread0()) {
            st->beta = rho_new / st->rho;
            st->rho = rho_new;
            st->rr = rr;
            st->iter += 1;
            if (sqrt(rr) <= st->tol * st->bnorm) {
                st->status = kConverged;
                st->done = 1;
            } else if (st->iter >= st->max_iter) {
                st->status = kCapped;
                st->done = 1;
            }
            st->ticket = 0;
        }
    }
}

// p_{k+1} = r_{k+1} + beta p_k; p*_{k+1} = r*_{k+1} + beta p*_k (one FMA
// where the shadow entries equal the primal ones bit for bit).
template <int kLd>
__global__ void __launch_bounds__(kVecThreads)
bicg_pupdate_kernel(double* __restrict__ p, const double* __restrict__ r, double* __restrict__ ps,
                    const double* __restrict__ rs, size_t len, const BicgState* st) {
    if (st->done) return;
    const double beta = st->beta;
    EXCMG_STRIDED(t0, S) {
        double rv[kLd], pv[kLd], rsv[kLd], psv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) {
                rv[k] = r[t];
                pv[k] = p[t];
                rsv[k] = rs[t];
                psv[k] = ps[t];
            }
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t >= len) break;
            const double pn = __fma_rn(beta, pv[k], rv[k]);
            p[t] = pn;
            double psn = pn;
            if (__double_as_longlong(rsv[k]) != __double_as_longlong(rv[k]) ||
                __double_as_longlong(psv[k]) != __double_as_longlong(pv[k]))
                psn = fma_here(beta, psv[k], rsv[k]);
            ps[t] = psn;
        }
    }
}

// Shadow-elided mode (not Alg. 2 as printed; r* = r and p* = p are not
// stored).  p_0 = r_0, rho_0 = rr = (r_0, r_0): the sums of
// bicg_init_kernel with r*_0 = r_0, in the same order.
__global__ void __launch_bounds__(kVecThreads)
cg_init_kernel(const double* __restrict__ r, double* __restrict__ p, size_t len, double* partials, BicgState* st) {
    __shared__ double sh[32];
    __shared__ bool am_last;
    double vrr = 0.0;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < len;
         t += (size_t)gridDim.x * blockDim.x) {
        const double rv = r[t];
        p[t] = rv;
        vrr = __fma_rn(rv, rv, vrr);
    }
    double s2[2];
    s2[0] = block_sum(vrr, sh);
    s2[1] = s2[0];
    if (publish_partials(s2, 2, partials, &st->ticket, &am_last)) {
        const double rr = gather_partials(partials, 1, sh);
        if (thread0()) {
            st->rho = rr;
            st->rr = rr;
            st->iter = 0;
            st->alpha = st->beta = st->sigma = 0.0;
            const bool conv = sqrt(rr) <= st->tol * st->bnorm;
            st->done = (conv || st->max_iter <= 0) ? 1 : 0;
            st->status = conv ? kConverged : (st->max_iter <= 0 ? kCapped : kRunning);
            st->ticket = 0;
        }
    }
}

// Shadow-elided update: x += alpha p; r -= alpha A p; rho_{k+1} = rr =
// (r, r); beta; stopping test.  Same arithmetic and summation order as
// bicg_update_kernel on twin entries.
template <int kLd>
__global__ void __launch_bounds__(kVecThreads)
cg_update_kernel(double* __restrict__ x, const double* __restrict__ p, double* __restrict__ r,
                 const double* __restrict__ q, size_t len, double* partials, BicgState* st) {
    if (st->done) return;
    __shared__ double sh[32];
    __shared__ bool am_last;
    const double alpha = st->alpha;
    double vrr = 0.0;
    EXCMG_STRIDED(t0, S) {
        double xv[kLd], pv[kLd], rv[kLd], qv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) {
                rv[k] = r[t];
                qv[k] = q[t];
                xv[k] = x[t];
                pv[k] = p[t];
            }
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t >= len) break;
            const double rn = __fma_rn(-alpha, qv[k], rv[k]);
            r[t] = rn;
            vrr = __fma_rn(rn, rn, vrr);
            x[t] = __fma_rn(alpha, pv[k], xv[k]);
        }
    }
    double s[2];
    s[0] = block_sum(vrr, sh);
    s[1] = s[0];
    if (publish_partials(s, 2, partials, &st->ticket, &am_last)) {
        const double rr = gather_partials(partials, 1, sh);
        if (thread0()) {
            st->beta = rr / st->rho;
            st->rho = rr;
            st->rr = rr;
            st->iter += 1;
            if (sqrt(rr) <= st->tol * st->bnorm) {
                st->status = kConverged;
                st->done = 1;
            } else if (st->iter >= st->max_iter) {
                st->status = kCapped;
                st->done = 1;
            }
            st->ticket = 0;
        }
    }
}

// Shadow-elided direction update: p = r + beta p.
template <int kLd>
__global__ void __launch_bounds__(kVecThreads)
cg_pupdate_kernel(double* __restrict__ p, const double* __restrict__ r, size_t len, const BicgState* st) {
    if (st->done) return;
    const double beta = st->beta;
    EXCMG_STRIDED(t0, S) {
        double rv[kLd], pv[kLd];
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) {
                rv[k] = r[t];
                pv[k] = p[t];
            }
        }
#pragma unroll
        for (int k = 0; k < kLd; ++k) {
            const size_t t = t0 + k * S;
            if (t < len) p[t] = __fma_rn(beta, pv[k], rv[k]);
        }
    }
}

}  // namespace

cudaError_t launch_cg_pupdate(double* p, const double* r, size_t len, const BicgState* st, cudaStream_t s) {
    (load_pairs(len) ? cg_pupdate_kernel<2> : cg_pupdate_kernel<1>)<<<kVecBlocks, kVecThreads, 0, s>>>(p, r, len, st);
    return cudaGetLastError();
}

cudaError_t launch_cg_init(const double* r, double* p, size_t len, double* partials, BicgState* st, cudaStream_t s) {
    cg_init_kernel<<<kVecBlocks, kVecThreads, 0, s>>>(r, p, len, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_cg_update(double* x, const double* p, double* r, const double* q, size_t len, double* partials,
                             BicgState* st, cudaStream_t s) {
    (load_pairs(len) ? cg_update_kernel<2> : cg_update_kernel<1>)<<<kVecBlocks, kVecThreads, 0, s>>>(x, p, r, q, len, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_dot(const double* a, const double* b, size_t len, double* partials,
                       unsigned int* ticket, double* out, cudaStream_t s) {
    (load_pairs(len) ? dot_kernel<2> : dot_kernel<1>)<<<kVecBlocks, kVecThreads, 0, s>>>(a, b, len, partials, ticket, out);
    return cudaGetLastError();
}

cudaError_t launch_interior_dot(const double* a, int n, double* partials, unsigned int* ticket, double* out,
                                cudaStream_t s) {
    interior_dot_kernel<<<kVecBlocks, kVecThreads, 0, s>>>(a, n, partials, ticket, out);
    return cudaGetLastError();
}

cudaError_t launch_bicg_init(const double* r, const double* shadow, double* rs, double* p, double* ps, size_t len,
                             int n, double* partials, BicgState* st, cudaStream_t s) {
    (load_pairs(len) ? bicg_init_kernel<2> : bicg_init_kernel<1>)<<<kVecBlocks, kVecThreads, 0, s>>>(r, shadow, rs, p, ps, len, n, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_bicg_sigma(const double* ps, const double* q, size_t len, double* partials,
                              BicgState* st, cudaStream_t s) {
    bicg_sigma_kernel<<<kVecBlocks, kVecThreads, 0, s>>>(ps, q, len, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_bicg_update(double* x, const double* p, double* r, const double* q, double* rs,
                               const double* qs, size_t len, double* partials, BicgState* st,
                               cudaStream_t s) {
    const bool two = load_pairs(len);
    (qs ? (two ? bicg_update_kernel<2, false> : bicg_update_kernel<1, false>)
        : (two ? bicg_update_kernel<2, true> : bicg_update_kernel<1, true>))<<<kVecBlocks, kVecThreads, 0, s>>>(
        x, p, r, q, rs, qs, len, partials, st);
    return cudaGetLastError();
}

cudaError_t launch_bicg_pupdate(double* p, const double* r, double* ps, const double* rs, size_t len,
                                const BicgState* st, cudaStream_t s) {
    (load_pairs(len) ? bicg_pupdate_kernel<2> : bicg_pupdate_kernel<1>)<<<kVecBlocks, kVecThreads, 0, s>>>(p, r, ps, rs, len, st);
    return cudaGetLastError();
}

}  // namespace excmg
