// Bi-CG iterations (Alg. 2, M = I, r*_0 = r_0) of a small grid with every
// vector on chip for the whole launch.
//
// The interior of the grid is cut into bricks, one per CTA (one CTA per SM).
// A CTA keeps x, r, r*, p, p* and q of its own nodes in registers, and p of
// the nodes around the brick that the 25 taps reach.  An iteration crosses
// the GPU twice, both times for an inner product that every CTA needs:
//
//   p = r + beta p on the brick and on the nodes around it (their r from L2,
//   their p kept from the last iteration: the owner forms the same bits);
//   q = A p from a shared tile of p;  sigma = (p*, q)          -- exchange 1
//   r -= alpha q, written to L2;  rho = (r*, r)                -- exchange 2
//   x += alpha p while exchange 2 is under way.
//
// What bounds it: the latency of the exchanges and the FP64 pipe (one warp
// instruction per 64 cycles and SM sub-partition, whatever its active
// lanes), not memory.  Hence
//  * two grid-wide waits per iteration instead of three, and no separate
//    gather of partial sums: a CTA publishes its partial sum beside the
//    exchange's tag in one 16-byte word, and every CTA polls the words of all
//    CTAs (an arrival counter and a gather: 2.0 + 0.5 us; the words: about
//    1 us).  A CTA writes 32 copies and reads the copy picked by its index,
//    as 152 CTAs polling one copy take 5.4 us;
//  * r travels the same way, value and tag in one word, so it needs no
//    fence (0.5 us on either side) and arrives while exchange 2 is under way;
//  * sums across lanes in integers (sum_fx): a 5-step FP64 shuffle tree costs
//    about 510 cycles, the integer form about a third;
//  * scalars formed by one warp and broadcast (a division takes 650 cycles),
//    and no FP64 comparisons: they go through the same pipe;
//  * outputs rounded with integer instructions (brick_result; the hardware
//    conversion goes through the FP64 pipe: the same time here).
// Measured: 200 iterations on 64^3 2.13 ms (the general cooperative kernel:
// 5.63 ms), a whole 32^3 first-kind solve to 1e-10 4.9 ms (14.8 ms); 100
// iterations of the 512^2 problem 1.00 ms (three launches each: 3.08 ms); per
// iteration 72^3 13.8 us, 80^3 18.0 (launched kernels: 36.1, 37.7).
//
// Shadow sequence: the launches start from r*_0 = p*_0 = r_0 = p_0 (a
// caller-chosen r*_0 takes the general kernel in stencil.cu).  A^T p* is A p
// bit for bit where p* = p (march_fx.cuh), so q serves both; r* and p* are
// updated entry by entry, with the primal result reused where the operands
// of a thread agree bit for bit; the other case is kept out of the FP64 pipe's
// way (opaque in reduce.cuh).  From such a start they always agree: the
// comparison is there on principle, so that the full mode's r*, p* are what Alg. 2 makes of
// their own values.  kElide: r*, p* are not kept (the same bits).
//
// DIM = 2: the 2D problem's 13-point rows (excmg2d.cu), with the second axis in
// the place of z and no third one.
//
// T = float: the FP32 correction solves of the mixed-precision mode.  The
// operator sums in FP32, inner products are FP32 inside a CTA and combined in
// FP64 between CTAs, as in the launched FP32 kernels.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "grid_sync.cuh"
#include "march_lap.cuh"
#include "resident_geom.h"

namespace excmg {

// One Bi-CG call on one grid.  Vectors are node arrays, of which the interior
// entries are used.  words: kResWords slot words, none with a tag of this launch
// when it starts; rx: one word per node (the r of the brick surfaces), without a
// tag when a call starts.  r null: r is in the value halves of rx between
// launches, the surfaces' as the exchanges left it (FP64).
template <typename T>
struct ResidentInst {
    T* x;
    T* r;
    T* rs;
    T* p;
    T* ps;
    BicgState* st;
    ulonglong2* words;
    ulonglong2* rx;
    int n, sigma;
};

namespace {

// One 16-byte word, read and written as a whole.
__device__ __forceinline__ ulonglong2 ld_word(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=l"(v.x), "=l"(v.y)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_word(ulonglong2* p, unsigned long long x, unsigned long long y) {
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "l"(x), "l"(y)
                 : "memory");
}

// a node's word: its value, and its tag as the result
__device__ __forceinline__ unsigned long long ld_node(const ulonglong2* w, double* v) {
    const ulonglong2 t = ld_word(w);
    *v = __longlong_as_double((long long)t.x);
    return t.y;
}
__device__ __forceinline__ void st_node(ulonglong2* w, double v, unsigned long long tag) {
    st_word(w, (unsigned long long)__double_as_longlong(v), tag);
}
__device__ __forceinline__ unsigned long long ld_node(const ulonglong2* w, float* v) {
    const ulonglong2 t = ld_word(w);
    *v = __uint_as_float((unsigned)t.x);
    return t.y;
}
__device__ __forceinline__ void st_node(ulonglong2* w, float v, unsigned long long tag) {
    st_word(w, (unsigned long long)__float_as_uint(v), tag);
}

__device__ __forceinline__ unsigned long long bits_of(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ bool same_bits(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_int(a) == __float_as_int(b); }
// finite and not zero
__device__ __forceinline__ bool usable(double v) {
    return (bits_of(v) << 1) != 0ull && exponent_of(v) != 0x7FF;
}

// Sum of C values per lane over the warp (every lane gets it): each value as
// an integer of 2^(E - 1079), E the largest biased exponent, rounded to
// nearest, summed exactly and rounded once.  Error below 32 C / 2 units of
// 2^-57 of the largest value, the order of an FP64 tree's.  C <= 5.
template <int C>
__device__ __forceinline__ double sum_fx(const double (&v)[C]) {
    unsigned e[C], em = 1u;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        e[c] = ((unsigned)__double2hiint(v[c]) >> 20) & 0x7FFu;
        em = max(em, e[c]);
    }
    const int E = (int)__reduce_max_sync(0xffffffffu, em);
    long long s = 0;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[c]);
        const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (e[c] ? 1ull << 52 : 0ull);
        const int d = E - (int)max(e[c], 1u);
        const unsigned long long h = d < 63 ? (m << 5) >> d : 0ull;   // twice the unit
        const long long k = (long long)((h + 1ull) >> 1);
        s += (long long)b < 0 ? -k : k;
    }
    // |s| < 5 * 2^57: three pieces whose 32-lane sums fit in 32 bits
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)s & 0x3FFFFFu);
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)((unsigned long long)s >> 22) & 0x3FFFFFu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(s >> 44));
    // the total of up to 160 values in units of 2^(E - 1076), |Y| < 2^62
    const long long Y = ((long long)hi << 41) + ((((long long)mid << 22) + (long long)lo + 4) >> 3);
    return fx_result(Y, E - 1, E == 0x7FF);
}

// Rare, and out of line so that the compiler does not evaluate them -- 650
// cycles each -- on the way of every iteration.
__device__ __noinline__ double divide_slow(double a, double b) { return a / b; }
__device__ __noinline__ bool root_at_most(double a, double b) { return sqrt(a) <= b; }

// v as an integer of 2^(E - 1077), E the largest biased exponent of the tile,
// rounded to nearest: two bits below the last place of the tile's largest
// values (144 * 2^55 < 2^63, the weights' sum times the largest integer); the
// marches truncate at that place.  The per-node form of the general kernel has a
// scale for the 25 taps of each node, a brick one for all of its nodes: truncated to
// it, A p kept fewer bits.  The error of the iterates against 64 bits after 48
// to 96 iterations on 16^3 .. 32^3 (geometric means of 16 right-hand sides) was then 1.57 times the
// per-node form's (0.75 to 2.5 by grid and kind), it is 0.73 times now (0.43 to 0.99), for
// 0.1 of 10.7 us per iteration on 64^3 and 0.7 % of a 32^3 solve.
__device__ __forceinline__ long long to_brick(double v, int E) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7FFu;
    const unsigned mh = ((hi & 0xFFFFFu) | (e != 0u ? 0x100000u : 0u)) << 3 | lo >> 29, ml = lo << 3;
    const unsigned d = (unsigned)(E - (int)max(e, 1u));
    const unsigned rlo = shr_clamp(__funnelshift_rc(ml, mh, d), (unsigned)max((int)d - 32, 0));
    const unsigned rhi = shr_clamp(mh, d);
    const unsigned long long m = ((((unsigned long long)rhi << 32) | rlo) + 1ull) >> 1;   // from half units
    return (int)hi < 0 ? -(long long)m : (long long)m;
}

// Y * 2^(E - 1077) rounded to nearest even, |Y| < 2^63 (from_fixed's exponent
// field holds for one less than with its |Y| < 2^62).
__device__ __forceinline__ double brick_result(long long acc, int E) {
    if (E >= 55 && E <= 2038) return from_fixed(acc, E - 2);
    return fx_result_slow(acc, E - 2, E == 0x7FF);
}

// a b + c, fused: written out so that every variant of the kernel rounds alike
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// The same where it is rarely reached: not evaluated ahead of its branch.
__device__ __forceinline__ double mad_here(double a, double b, double c) { return fma_here(a, b, c); }
__device__ __forceinline__ float mad_here(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// a sum over the warp in FP32 (every lane gets it)
__device__ __forceinline__ float sum_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// A thread's NP values of one vector: in registers, or (kShared) in shared
// memory at v[k * kResThreads].
template <typename T, int NP, bool kShared>
struct OwnValues {
    T reg[kShared ? 1 : NP];
    T* v;
    __device__ __forceinline__ T& operator[](int k) {
        if constexpr (kShared) return v[k * kResThreads];
        else return reg[k];
    }
};

// NP: nodes of a thread's run along z; NH: nodes around the brick per thread.
template <typename T, int DIM, int NP, int NH, bool kElide>
__global__ void __launch_bounds__(kResThreads, 1)
resident_bicg_kernel(const ResidentInst<T> in, const ResidentGeom g, int iters,
                     unsigned serial, long long spin_limit) {
    constexpr bool kExact = std::is_same<T, double>::value;
    using Fix = typename std::conditional<kExact, long long, float>::type;
    extern __shared__ __align__(16) unsigned char res_smem[];
    Fix* const tile = reinterpret_cast<Fix*>(res_smem);
    __shared__ unsigned wmax[kResThreads / 32];
    __shared__ T red[kResThreads / 32];
    __shared__ double bcast[2];   // alpha or beta, rho
    __shared__ int flags[2];      // stop code of the last exchange, gave up
    __shared__ int lost;          // a thread gave up waiting for r
    BicgState* const st = in.st;
    if (st->done) return;
    const int cta = (int)blockIdx.x, G = g.ctas, n = in.n, np = n + 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int plane = DIM == 3 ? np * np : np;

    // this thread's nodes: NP along z at one (x, y) of the brick
    const int kx = cta % g.cx, ky = (cta / g.cx) % g.cy, kz = cta / (g.cx * g.cy);
    const int ox = 1 + kx * g.bx, oy = 1 + ky * g.by, oz = 1 + kz * g.bz;
    const int cols = g.bx * g.by;
    const int grp = tid / cols, col = tid - grp * cols;
    const int ly = col / g.bx, lx = col - ly * g.bx, lz = grp * NP;
    const int nz = min(g.bz, n - oz);            // planes of the brick
    const bool mine = lz < nz && ox + lx < n && oy + ly < n;
    const int cnt = mine ? min(NP, nz - lz) : 0;   // this thread's nodes
    const int idx0 = !mine ? 0 : DIM == 3 ? ((oz + lz) * np + oy + ly) * np + ox + lx : (oz + lz) * np + ox + lx;
    const int tx = g.tx, tp = DIM == 3 ? tx * (g.by + 4) : tx;
    const int t0 = (lz + 2) * tp + (DIM == 3 ? (ly + 2) * tx : 0) + lx + 2;   // tile entry of the first one
    int cc[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int i = ox + lx, j = oy + ly, z = oz + lz + k;
        const int cy = DIM == 3 ? (j == 1) + (j == n - 1) : 0;
        cc[k] = in.sigma * ((i == 1) + (i == n - 1) + cy + (z == 1) + (z == n - 1));
    }
    // nodes of this thread that other bricks' taps reach
    unsigned surf = 0u;
#pragma unroll
    for (int k = 0; k < NP; ++k)
        if (k < cnt && (lx < 2 || lx >= g.bx - 2 || (DIM == 3 && (ly < 2 || ly >= g.by - 2)) || lz + k < 2 ||
                        lz + k >= g.bz - 2))
            surf |= 1u << k;
    // nodes around the brick, on the warps from 1 up (warp 0 has the
    // exchanges): node index (-1: none, or outside the interior), tile entry
    int hidx[NH], htile[NH];
#pragma unroll
    for (int k = 0; k < NH; ++k) {
        const int h = tid - 32 + k * kResHaloThreads;
        hidx[k] = -1;
        htile[k] = 0;
        if (tid >= 32 && h < g.halo) {
            int hx, hy = 0, hz;
            if (DIM == 3) res_halo(h, g.bx, g.by, g.bz, &hx, &hy, &hz);
            else res_halo2(h, g.bx, g.bz, &hx, &hz);
            const int i = ox + hx, j = oy + hy, z = oz + hz;
            if (i >= 1 && i < n && j >= 1 && j < n && z >= 1 && z < n)
                hidx[k] = DIM == 3 ? (z * np + j) * np + i : z * np + i;
            htile[k] = (hz + 2) * tp + (DIM == 3 ? (hy + 2) * tx : 0) + hx + 2;
        }
    }
    for (int t = tid; t < g.tile; t += kResThreads) tile[t] = Fix(0);
    if (tid == 0) lost = 0;
    __syncthreads();   // (FP32: the first tile is written without another barrier before it)

    T r[NP], p[NP], q[NP], hp[NH], hr[NH];
    OwnValues<T, NP, (NP > kResRegNodes)> x, rs, ps;
    if constexpr (NP > kResRegNodes) {
        T* const own = reinterpret_cast<T*>(res_smem + (size_t)((g.tile + 1) & ~1) * sizeof(Fix)) + tid;
        x.v = own;
        rs.v = own + NP * kResThreads;
        ps.v = own + 2 * NP * kResThreads;
    }
    // (the owner of a word writes it first after exchange 1, which every CTA
    // enters with these values in use)
    auto first_r = [&](int o) -> T {
        if (!kExact || in.r) return in.r[o];
        T v;
        (void)ld_node(in.rx + o, &v);
        return v;
    };
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        x[k] = r[k] = p[k] = q[k] = rs[k] = ps[k] = T(0);
        if (k < cnt) {
            const int o = idx0 + k * plane;
            x[k] = in.x[o];
            r[k] = first_r(o);
            p[k] = in.p[o];
            if (!kElide) {
                rs[k] = in.rs[o];
                ps[k] = in.ps[o];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NH; ++k) {
        hp[k] = hidx[k] >= 0 ? in.p[hidx[k]] : T(0);
        hr[k] = hidx[k] >= 0 ? first_r(hidx[k]) : T(0);
    }

    double rho = st->rho, beta = st->beta;                      // every thread
    double alpha = st->alpha, sigma = st->sigma, rr = st->rr;   // warp 0
    int iter = st->iter;
    const int max_iter = st->max_iter;
    const double stop = st->tol * st->bnorm;
    const double far = stop * stop * (1.0 + 1e-12);   // rr above this: sqrt(rr) > stop
    double inv = 0.0;                                 // warp 0: 1 / rho
    int code = kRunning;
    bool gave_up = false;
    // Tags: the launch's serial number above the number of the exchange or
    // iteration (64 bits; a 32-bit one of the iteration in its call was up to 2 % slower).  Slot
    // words come in two sets: a CTA that publishes exchange e + 2 has read
    // exchange e + 1 from every CTA, which each published after it had read
    // exchange e.  The word of a node needs no second one: its owner writes
    // the next r after exchange 1, which every CTA enters with its r read.
    const unsigned long long tag0 = (unsigned long long)serial << 32;
    unsigned ep = 0;   // exchanges so far
    volatile unsigned* const err = reinterpret_cast<volatile unsigned*>(in.words + kResWords - 1);

    // warp 0: publish this CTA's partial sum, wait for those of all CTAs, add them
    auto publish = [&](double v) {
        st_word(in.words + ((size_t)(ep & 1) * kResCopies + lane) * kResMaxCtas + cta, bits_of(v), tag0 | ep);
    };
    auto collect = [&]() -> double {
        const ulonglong2* const s =
            in.words + ((size_t)(ep & 1) * kResCopies + (cta & (kResCopies - 1))) * kResMaxCtas;
        ulonglong2 b[5];
        long long spins = 0;
        for (;;) {
            bool ok = true;
#pragma unroll
            for (int k = 0; k < 5; ++k) b[k] = lane + 32 * k < G ? ld_word(s + lane + 32 * k) : make_ulonglong2(0ull, tag0 | ep);
#pragma unroll
            for (int k = 0; k < 5; ++k) ok = ok && b[k].y == (tag0 | ep);
            if (__all_sync(0xffffffffu, ok)) break;
            if ((++spins & 255) == 0 && (*err == serial || spins > spin_limit)) {
                *err = serial;
                gave_up = true;
                break;
            }
        }
        ++ep;
        double v[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = __longlong_as_double((long long)b[k].x);
        return sum_fx<5>(v);
    };
    // this CTA's sum of v (valid in warp 0, after the CTA barrier inside)
    auto cta_sum = [&](T v) -> double {
        if constexpr (kExact) {
            const double a[1] = {v};
            const double w = sum_fx<1>(a);
            if (lane == 0) red[warp] = w;
        } else {
            const float w = sum_f32(v);
            if (lane == 0) red[warp] = w;
        }
        __syncthreads();
        if (warp != 0) return 0.0;
        if constexpr (kExact) {
            const double b[1] = {lane < kResThreads / 32 ? red[lane] : 0.0};
            return sum_fx<1>(b);
        } else {
            return (double)sum_f32(lane < kResThreads / 32 ? red[lane] : 0.f);
        }
    };

    for (int it = 0; it < iters; ++it) {
        // p = r + beta p
        if (iter > 0) {
            const T b = (T)beta;
            bool twin = kExact;
            if (kExact && !kElide) {
#pragma unroll
                for (int k = 0; k < NP; ++k) twin = twin && same_bits(rs[k], r[k]) && same_bits(ps[k], p[k]);
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) p[k] = mad(b, p[k], r[k]);
            if (!kElide) {
                T pn[NP];
#pragma unroll
                for (int k = 0; k < NP; ++k) pn[k] = p[k];
                const int general = kExact ? opaque(!twin) : 1;
#pragma unroll 1
                for (int once = 0; once < general; ++once) {
#pragma unroll
                    for (int k = 0; k < NP; ++k) pn[k] = mad_here(b, ps[k], rs[k]);
                }
#pragma unroll
                for (int k = 0; k < NP; ++k) ps[k] = pn[k];
            }
#pragma unroll
            for (int k = 0; k < NH; ++k) hp[k] = mad(b, hp[k], hr[k]);
        }
        // the tile of p: on one power-of-two scale as integers (to_brick), or FP32
        int E = 1;
        if constexpr (kExact) {
            unsigned em = 1u;
#pragma unroll
            for (int k = 0; k < NP; ++k) em = max(em, ((unsigned)__double2hiint(p[k]) >> 20) & 0x7FFu);
#pragma unroll
            for (int k = 0; k < NH; ++k) em = max(em, ((unsigned)__double2hiint(hp[k]) >> 20) & 0x7FFu);
            em = __reduce_max_sync(0xffffffffu, em);
            if (lane == 0) wmax[warp] = em;
            __syncthreads();
            E = (int)__reduce_max_sync(0xffffffffu, wmax[lane & (kResThreads / 32 - 1)]);
        }
        // (every read of the last tile was before the last exchanges' barriers)
#pragma unroll
        for (int k = 0; k < NP; ++k)
            if (k < cnt) {
                if constexpr (kExact)
                    tile[t0 + k * tp] = to_brick(p[k], E);
                else
                    tile[t0 + k * tp] = p[k];
            }
#pragma unroll
        for (int k = 0; k < NH; ++k)
            if (hidx[k] >= 0) {
                if constexpr (kExact)
                    tile[htile[k]] = to_brick(hp[k], E);
                else
                    tile[htile[k]] = hp[k];
            }
        __syncthreads();
        // q = A p: the sum of the axis neighbours inside a plane (DIM = 2: row)
        // serves its own row (-12, -8) and the rows above and below (+2)
        constexpr int kCentre = DIM == 3 ? 42 : 20, kNear = DIM == 3 ? 12 : 8;
        T dot = T(0);
        if (cnt > 0) {
            Fix u[NP + 4], s4[NP + 2];
#pragma unroll
            for (int k = 0; k < NP + 4; ++k) u[k] = tile[t0 + (k - 2) * tp];
#pragma unroll
            for (int k = 0; k < NP + 2; ++k) {
                const int o = t0 + (k - 1) * tp;
                s4[k] = tile[o - 1] + tile[o + 1];
                if (DIM == 3) s4[k] += tile[o - tx] + tile[o + tx];
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int o = t0 + k * tp;
                const Fix n6 = s4[k + 1] + (u[k + 1] + u[k + 3]);
                Fix f6 = (tile[o - 2] + tile[o + 2]) + (u[k] + u[k + 4]);
                Fix d12 = s4[k] + s4[k + 2];
                if (DIM == 3) {
                    f6 += tile[o - 2 * tx] + tile[o + 2 * tx];
                    d12 += (tile[o - tx - 1] + tile[o - tx + 1]) + (tile[o + tx - 1] + tile[o + tx + 1]);
                }
                if (k < cnt) {
                    if constexpr (kExact) {
                        const long long acc =
                            mul_w(u[k + 2], (unsigned)(kCentre + cc[k])) - mul_w(n6, (unsigned)kNear) + f6 + (d12 + d12);
                        q[k] = brick_result(acc, E);
                    } else {
                        q[k] = mad((float)(kCentre + cc[k]), u[k + 2], mad(-(float)kNear, n6, mad(2.f, d12, f6)));
                    }
                    dot = mad(kElide ? p[k] : ps[k], q[k], dot);
                }
            }
        }
        // exchange 1: sigma, alpha (1 / rho, for beta, under way)
        const double ds = cta_sum(dot);
        if (warp == 0) {
            publish(ds);
            inv = 1.0 / rho;
            asm volatile("" : "+d"(inv));   // here, not where it is used
            sigma = collect();
            const bool bad = !usable(rho) || !usable(sigma);
            if (!bad) alpha = rho / sigma;
            if (lane == 0) {
                bcast[0] = alpha;
                flags[0] = bad ? kBreakdown : kRunning;
                flags[1] = gave_up || lost;
            }
        }
        __syncthreads();
        code = flags[0];
        gave_up = flags[1] != 0;
        if (gave_up || code != kRunning) break;
        // r -= alpha q, r* -= alpha q*
        const T a = (T)bcast[0];
        const unsigned long long rtag = tag0 | (unsigned)(it + 1);
        T vr = T(0), rn[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) rn[k] = mad(-a, q[k], r[k]);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            if (surf >> k & 1u) st_node(in.rx + idx0 + k * plane, rn[k], rtag);
        }
        if (!kElide) {
            bool twin = kExact;
            if (kExact) {
#pragma unroll
                for (int k = 0; k < NP; ++k) twin = twin && same_bits(rs[k], r[k]);
            }
            T rsn[NP];
#pragma unroll
            for (int k = 0; k < NP; ++k) rsn[k] = rn[k];
            const int general = kExact ? opaque(!twin) : 1;
#pragma unroll 1
            for (int once = 0; once < general; ++once) {
#pragma unroll
                for (int k = 0; k < NP; ++k) rsn[k] = mad_here(-a, q[k], rs[k]);
            }
#pragma unroll
            for (int k = 0; k < NP; ++k) rs[k] = rsn[k];
        }
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            r[k] = rn[k];
            vr = mad(kElide ? rn[k] : rs[k], rn[k], vr);
        }
        // exchange 2: rho (r* = r bit for bit, so (r, r) is the same sum),
        // beta, the stopping test; x += alpha p and the r of the nodes
        // around the brick under way
        const double dr = cta_sum(vr);
        if (warp == 0) publish(dr);
#pragma unroll
        for (int k = 0; k < NP; ++k) x[k] = mad(a, p[k], x[k]);
        if (warp == 0) {
            rr = collect();
            // rr / rho: the product with 1 / rho and one correction step
            // (Markstein, IBM J. Res. Dev. 34, 1990) where no step leaves the
            // normal range
            double bt = rr * inv;
            bt = __fma_rn(__fma_rn(-bt, rho, rr), inv, bt);
            const int er = exponent_of(rr), ei = exponent_of(inv);
            if (er < 256 || er > 1791 || ei < 256 || ei > 1791) bt = divide_slow(rr, rho);
            int c = kRunning;
            // (rr >= 0: its bits order as integers; NaN is above all)
            if (bits_of(rr) <= bits_of(far) && root_at_most(rr, stop)) c = kConverged;
            else if (iter + 1 >= max_iter) c = kCapped;
            if (lane == 0) {
                bcast[0] = bt;
                bcast[1] = rr;
                flags[0] = c;
                flags[1] = gave_up;
            }
        } else {
            long long spins = 0;
            bool ok;
            do {
                ok = true;
#pragma unroll
                for (int k = 0; k < NH; ++k)
                    if (hidx[k] >= 0) ok = (ld_node(in.rx + hidx[k], &hr[k]) == rtag) && ok;
                if (!ok && (++spins & 255) == 0 && (*err == serial || spins > spin_limit)) {
                    *err = serial;
                    lost = 1;
                    break;
                }
            } while (!ok);
        }
        __syncthreads();
        code = flags[0];
        gave_up = flags[1] != 0;
        if (gave_up) break;
        beta = bcast[0];
        rho = bcast[1];
        ++iter;
        if (code != kRunning) break;
    }
#pragma unroll
    for (int k = 0; k < NP; ++k)
        if (k < cnt) {
            const int o = idx0 + k * plane;
            in.x[o] = x[k];
            if (!kExact || in.r) in.r[o] = r[k];
            else if (!(surf >> k & 1u)) st_node(in.rx + o, r[k], 0u);
            in.p[o] = p[k];
            if (!kElide) {
                in.rs[o] = rs[k];
                in.ps[o] = ps[k];
            }
        }
    if (cta == 0 && tid == 0) {
        if (gave_up || *err == serial) code = kTimeout;
        st->rho = rho;
        // (the sum of an exchange that gave up has words of other exchanges in it)
        if (iter > 0 && code != kTimeout) st->rr = rr;
        st->alpha = alpha;
        st->beta = beta;
        st->sigma = sigma;
        st->iter = iter;
        st->status = code;
        st->done = code != kRunning;
    }
}

}  // namespace
}  // namespace excmg
