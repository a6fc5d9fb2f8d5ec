// The z-march of the operator on one 32 x 16 column tile: A u, b - A u, or
// the operator step of Bi-CG (Alg. 2), in the integer arithmetic of
// march_fx.cuh (each input plane of a CTA on one power-of-two scale, taps
// summed exactly, one rounding per output).
//
// The sum is formed as the square of the seven-point Laplacian.  With
// L u = 6 u - (6 axis neighbours), zero outside the interior, and w = L u kept
// on interior nodes only, the 25-point rows of eq. (method1) with the folded
// reflections are
//     A u = L w + (1 + sigma) c u,
// c the number of faces the node is one step from (for an end node of an axis
// L w misses the tap through the boundary node: 42 - c on the diagonal).
// The integers are the ones of the direct sum, so the results are its bits
// while a CTA's scale does not change.  Why: the direct form
// reads 11 tile entries and takes about 45 integer instructions per output,
// this one 7 (ring nodes included) and about 25, and keeps fewer
// accumulators.
//
// What bounds it: latency and instruction issue of two CTAs per SM (at 512^3
// the step with directions moves 56 B per unknown in 1.4 times the time that HBM
// takes for them, 1.54 ms; A u, 0.97 ms, is far from HBM).  Hence
//  * copies run one plane ahead of their use by 8-byte cp.async (rows of N + 1
//    doubles have no 16-byte alignment) into one stage, which a thread refills
//    as soon as it has read its own slots back, so completing the copies needs
//    no CTA barrier.  More stages were slower (step with directions 1.69 ms
//    with one stage then, 1.75 with two, 2.69 with three and no L1 left), the
//    256-byte L2 prefetch hint is worth 4-6 %;
//  * one CTA barrier per plane publishes the tile of u at plane t, the tile of
//    w at plane t - 1 and the exponent maximum of plane t + 1, and between two
//    barriers a thread has three independent pieces of work: plane t + 2 read
//    back and its directions formed, the sums from the tiles, plane t + 1
//    converted;
//  * p* of the planes on their way to sigma waits in shared memory, not in
//    registers (1.75 against 1.79 ms).
//
// Slots of a thread: its two output columns (0, 1) and at most one node of
// the two-node ring around the tile (2), those next to the tile, where w is
// needed, on the first 96 threads.
//
// The direct form (two rows per thread, 25 taps from one tile, three stages)
// took, at 512^3 and with q* stored: step with directions 1.88 ms, without 1.27,
// A u 1.18.
#pragma once

#include <cuda_runtime.h>

#include "march_fx.cuh"
#include "reduce.cuh"

namespace excmg {
namespace {

constexpr int PP_TX = 32;                       // threads along x
constexpr int PP_TY = 8;                        // threads along y
constexpr int PP_OY = 2 * PP_TY;                // output rows per CTA (2 per thread)
constexpr int PP_HX = PP_TX + 4;                // halo width (36)
constexpr int PP_HY = PP_OY + 4;                // halo height (20)
constexpr int PP_HALO = PP_HX * PP_HY;          // 720 nodes per plane
constexpr int PP_NT = PP_TX * PP_TY;            // 256 threads
constexpr int PP_RING = PP_HALO - PP_TX * PP_OY;   // 208 ring nodes

// 32-bit shared-memory address of a generic pointer into shared memory
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ double lds_f64(unsigned a) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ long long lds_s64(unsigned a) {
    long long v;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts_s64(unsigned a, long long v) {
    asm volatile("st.shared.s64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void cp_async8_u32(unsigned dst, const void* src, unsigned src_bytes) {
    asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// x >> k for 0 <= k, 0 once k >= 32 (PTX clamps the shift amount)
__device__ __forceinline__ unsigned shr_clamp(unsigned x, unsigned k) {
    unsigned r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(k));
    return r;
}

// to_fixed (march_fx.cuh) with the biased exponent e of v already at hand
// and the 64-bit shift written as clamped 32-bit shifts: the same value,
// m >> (E - max(e, 1)) with the sign of v, 0 once the shift reaches 64.
__device__ __forceinline__ long long to_fixed_e(double v, unsigned e, int E) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned mh = (hi & 0xFFFFFu) | (e != 0u ? 0x100000u : 0u);
    const unsigned d = (unsigned)(E - (int)max(e, 1u));
    const unsigned rlo = shr_clamp(__funnelshift_rc(lo, mh, d), (unsigned)max((int)d - 32, 0));
    const unsigned rhi = shr_clamp(mh, d);
    const unsigned sg = (unsigned)((int)hi >> 31);   // 0 or all ones
    const unsigned long long m = ((unsigned long long)(rhi ^ sg) << 32) | (rlo ^ sg);
    return (long long)(m - (unsigned long long)(long long)(int)sg);
}

// a * w for a 64-bit integer a and a small positive weight w (|a w| < 2^63):
// one 32 x 32 -> 64 product of the low word and one multiply-add of the high
// word, instead of a general 64-bit multiplication
__device__ __forceinline__ long long mul_w(long long a, unsigned w) {
    const unsigned long long lo = (unsigned long long)(unsigned)a * w;
    const unsigned hi = (unsigned)((unsigned long long)a >> 32) * w + (unsigned)(lo >> 32);
    return (long long)(((unsigned long long)hi << 32) | (unsigned)lo);
}

// Y * 2^(E - 1075) rounded to nearest even, by the hardware conversion of Y
// to double (the same rounding of Y to 53 bits as from_fixed) and an exact
// power-of-two scaling of the exponent field; valid for 53 <= E <= 2036.
__device__ __forceinline__ double fx_result_cvt(long long acc, int E, bool poisoned) {
    if (!poisoned && E >= 53 && E <= 2036) {
        const double d = (double)acc;
        const long long bits = __double_as_longlong(d) + ((long long)(E - 1075) << 52);
        return acc == 0 ? 0.0 : __longlong_as_double(bits);
    }
    return fx_result_slow(acc, E, poisoned);
}

constexpr int ML_INNER = 96;   // ring nodes next to the tile (its corners are not)

// Halo coordinates (own columns start at 2, 2) of ring node e < PP_RING: the
// nodes next to the tile, then the corners between them, then the outer frame.
__host__ __device__ __forceinline__ void ml_ring(int e, int* lx, int* ly) {
    if (e < 64) {                 // rows below and above the tile
        *ly = e < 32 ? 1 : PP_HY - 2;
        *lx = 2 + (e & 31);
    } else if (e < 96) {          // columns left and right of it
        *lx = (e & 1) ? PP_HX - 2 : 1;
        *ly = 2 + ((e - 64) >> 1);
    } else if (e < 100) {         // corners
        *lx = (e & 1) ? PP_HX - 2 : 1;
        *ly = (e & 2) ? PP_HY - 2 : 1;
    } else if (e < 172) {         // the outer frame: its rows ...
        *ly = e < 136 ? 0 : PP_HY - 1;
        *lx = e - (e < 136 ? 100 : 136);
    } else {                      // ... and columns
        *lx = (e & 1) ? PP_HX - 1 : 0;
        *ly = 1 + ((e - 172) >> 1);
    }
}

// What a march does: A u; b - A u; with r = b - A u the start of a Bi-CG
// call (r, p, and r*, p* where given, and (r, r)) or (r, r) alone; (p, p*) ->
// q with sigma; the same with p = r + beta p, p* = r* + beta p* formed first.
enum MarchKind { kMarchApply, kMarchSub, kMarchStart, kMarchNorm, kMarchPair, kMarchDir };
constexpr bool march_is_step(MarchKind k) { return k == kMarchPair || k == kMarchDir; }

struct MarchArrays {
    const double* in;     // u, p or p_{k-1}
    const double* r;      // kMarchDir
    const double* ins;    // p* or p*_{k-1}
    const double* rs;     // kMarchDir
    const double* b;      // right-hand side (kMarchSub, kMarchStart, kMarchNorm)
    double* out;          // y or q (q* = q: the same bits, not stored again)
    double* pn;           // kMarchDir: p_k (not in: neighbours still read it); kMarchStart: p, may be null
    double* psn;          // the same for p*
    double beta;
    double* rsn;          // kMarchStart: r*, may be null
    ulonglong2* words;    // kMarchStart: the on-chip kernel's words, r in their values, no tag (out is
                          // not written then); may be null
};

// Shared memory: one stage, `in` (and r) on all three slots, p* (and r*), or
// b, on the two own ones; p* of four planes of the own slots; the tiles.
template <MarchKind K, bool kElide>
struct MarchStage {
    static constexpr int kAll = K == kMarchDir ? 2 : 1;
    static constexpr int kOwn = K == kMarchApply ? 0 : !march_is_step(K) ? 1 : kElide ? 0 : kAll;
    static constexpr unsigned kBytes = (kAll * 3 + kOwn * 2) * PP_NT * 8u;
    static constexpr unsigned kHist = !march_is_step(K) ? 0 : 4 * 2 * PP_NT * 8u;
    static constexpr size_t kSmem = kBytes + kHist + 4 * PP_HALO * sizeof(long long);
};

// One CTA's march over the output planes [kz0, kz1) of column tile (bx, by).
// Returns this thread's share of sigma = (p*, q), or of (r, r).  Called by all threads.
template <MarchKind K, bool kElide>
__device__ __forceinline__ double lap_march(const MarchArrays& a, int n, int sigma, int bx, int by, int kz0, int kz1,
                                            unsigned char* smem) {
    using St = MarchStage<K, kElide>;
    constexpr unsigned kCol = PP_NT * 8u;              // one slot of one array
    constexpr unsigned kOwn0 = St::kAll * 3 * kCol;    // first own-only array of a stage
    constexpr unsigned kTile = PP_HALO * 8u;
    __shared__ int wmax[2][PP_NT / 32];
    const unsigned raw = smem_u32(smem);
    const unsigned tiles = raw + St::kBytes + St::kHist;   // u twice, then w twice
    const int np = n + 1;
    const size_t plane8 = (size_t)np * np * 8;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * PP_TX + tx;
    const int lane = tid & 31, warp = tid >> 5;
    const int i0 = 1 + bx * PP_TX, j0 = 1 + by * PP_OY;
    const bool ring = tid < PP_RING, inner = tid < ML_INNER;
    constexpr bool kStep = march_is_step(K);
    constexpr bool has_b = !kStep && K != kMarchApply;

    // in-plane byte offset of each slot, copy size (0: reads as zero), tile entry
    unsigned so[3], sz[3], te[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        int lx = tx + 2, ly = 2 * ty + 2 + s;
        if (s == 2) ml_ring(ring ? tid : 0, &lx, &ly);
        const int gi = i0 - 2 + lx, gj = j0 - 2 + ly;
        const bool in = (s < 2 || ring) && gi >= 1 && gi <= n - 1 && gj >= 1 && gj <= n - 1;
        so[s] = in ? 8u * (unsigned)(gj * np + gi) : 0u;
        sz[s] = in ? 8u : 0u;
        te[s] = 8u * (unsigned)(ly * PP_HX + lx);
    }
    const bool act[2] = {sz[0] != 0u, sz[1] != 0u};
    const int i = i0 + tx, j = j0 + 2 * ty;
    // (1 + sigma) c without the z faces
    const int f = 1 + sigma;
    const int cx = (i == 1) + (i == n - 1);
    const int c0 = f * (cx + (j == 1) + (j == n - 1)), c1 = f * (cx + (j + 1 == 1) + (j + 1 == n - 1));
    const int T = kz1 - kz0 + 4;   // input planes kz0 - 2 .. kz1 + 1
    const unsigned st = raw + 8u * (unsigned)tid;                  // this thread's slots of the stage
    const unsigned hist = raw + St::kBytes + 8u * (unsigned)tid;   // its p* of the last planes

    // start the copies of plane t, with b of the plane that step t - 2 writes
    auto issue = [&](int t) {
        const int z = kz0 - 2 + t;
        if (t < T) {
            const bool zok = z >= 1 && z <= n - 1;
            const size_t zo = (size_t)(zok ? z : 1) * plane8;
            const char* const in = (const char*)a.in + zo;
            const char* const r = K == kMarchDir ? (const char*)a.r + zo : nullptr;
            const char* const ps = St::kOwn && kStep ? (const char*)a.ins + zo : nullptr;
            const char* const rs = St::kOwn == 2 ? (const char*)a.rs + zo : nullptr;
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                if (s < 2 || ring) {
                    const unsigned nb = zok ? sz[s] : 0u;
                    cp_async8_u32(st + s * kCol, in + so[s], nb);
                    if (K == kMarchDir) cp_async8_u32(st + (3 + s) * kCol, r + so[s], nb);
                    if (s < 2 && kStep && !kElide) {
                        cp_async8_u32(st + kOwn0 + s * kCol, ps + so[s], nb);
                        if (K == kMarchDir) cp_async8_u32(st + kOwn0 + (2 + s) * kCol, rs + so[s], nb);
                    }
                }
            }
        }
        if (has_b && z - 4 >= kz0 && z - 4 < kz1) {
            const char* const b = (const char*)a.b + (size_t)(z - 4) * plane8;
#pragma unroll
            for (int s = 0; s < 2; ++s) cp_async8_u32(st + kOwn0 + s * kCol, b + so[s], sz[s]);
        }
    };
    // this thread's slots of one plane as p (directions formed), with the
    // shadow of the own ones
    auto fetch = [&](double (&v)[3], double (&vs)[2]) {
        double po[3], rv[3], ps[2], rsv[2];
#pragma unroll
        for (int s = 0; s < 3; ++s)
            if (s < 2 || ring) {
                po[s] = lds_f64(st + s * kCol);
                if (K == kMarchDir) rv[s] = lds_f64(st + (3 + s) * kCol);
                if (s < 2 && kStep && !kElide) {
                    ps[s] = lds_f64(st + kOwn0 + s * kCol);
                    if (K == kMarchDir) rsv[s] = lds_f64(st + kOwn0 + (2 + s) * kCol);
                }
            }
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            v[s] = 0.0;
            if (s < 2 || ring) v[s] = K == kMarchDir ? __fma_rn(a.beta, po[s], rv[s]) : po[s];
        }
        if (kStep && !kElide) {
            // the same bits in: the same bits out, without another FP64 instruction
            // (always so in the calls that come here; compared on principle, as in resident.cuh)
            long long diff = 0;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                vs[s] = K == kMarchDir ? v[s] : ps[s];
                if (K == kMarchDir)
                    diff |= (__double_as_longlong(ps[s]) ^ __double_as_longlong(po[s])) |
                            (__double_as_longlong(rsv[s]) ^ __double_as_longlong(rv[s]));
            }
            if (K == kMarchDir) {
                const int rare = opaque(diff != 0);
#pragma unroll 1
                for (int once = 0; once < rare; ++once) {
#pragma unroll
                    for (int s = 0; s < 2; ++s) vs[s] = fma_here(a.beta, ps[s], rsv[s]);
                }
            }
        }
    };
    // the warp's largest exponent of a plane's slots, for all warps
    auto publish_max = [&](const double (&v)[3], int w) {
        unsigned em = 0u;
#pragma unroll
        for (int s = 0; s < 3; ++s) em = max(em, ((unsigned)__double2hiint(v[s]) >> 20) & 0x7FFu);
        em = __reduce_max_sync(0xffffffffu, em);
        if (lane == 0) wmax[w][warp] = (int)em;
    };
    auto plane_max = [&](int w) { return (int)__reduce_max_sync(0xffffffffu, (unsigned)wmax[w][lane & 7]); };

    // Own rows: u of planes t, t - 1; w of t - 1, t - 2; g = 6 u - (its
    // neighbours in the plane and in the plane before) of plane t, gq the same
    // of w at plane t - 1, with the faces' share.  Ring node next to the tile: u of t, t - 1, g.
    long long u0[2] = {0, 0}, um1[2] = {0, 0}, wm1[2] = {0, 0}, wm2[2] = {0, 0}, g[2] = {0, 0}, gq[2] = {0, 0};
    long long r0 = 0, rm1 = 0, gr = 0;
    double d = 0.0;

    // Plane t on scale E into the tiles of parity par: u(t), and w(t - 1) =
    // g - u(t) where node and plane are interior; new directions out.
    auto convert = [&](int t, int par, int E, const double (&v)[3], const double (&vs)[2]) {
        const int z = kz0 - 2 + t;
        const unsigned tu = tiles + (unsigned)par * kTile, tw = tu + 2 * kTile;
        const bool zw = z >= 2 && z <= n;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const long long u = to_fixed_e(v[s], ((unsigned)__double2hiint(v[s]) >> 20) & 0x7FFu, E);
            const long long w = zw && act[s] ? g[s] - u : 0;
            sts_s64(tu + te[s], u);
            sts_s64(tw + te[s], w);
            wm2[s] = wm1[s];
            wm1[s] = w;
            um1[s] = u0[s];
            u0[s] = u;
            if (kStep)   // p* for sigma, two steps on
                sts_s64(hist + (unsigned)(t & 3) * (2 * kCol) + s * kCol, __double_as_longlong(kElide ? v[s] : vs[s]));
        }
        if (ring) {
            const long long u = to_fixed_e(v[2], ((unsigned)__double2hiint(v[2]) >> 20) & 0x7FFu, E);
            sts_s64(tu + te[2], u);
            if (inner) {
                sts_s64(tw + te[2], zw && sz[2] != 0u ? gr - u : 0);
                rm1 = r0;
                r0 = u;
            }
        }
        if (K == kMarchDir && z >= kz0 && z < kz1) {
            char* const pz = (char*)a.pn + (size_t)z * plane8;
            char* const psz = (char*)a.psn + (size_t)z * plane8;
#pragma unroll
            for (int s = 0; s < 2; ++s)
                if (act[s]) {
                    *(double*)(pz + so[s]) = v[s];
                    if (!kElide) *(double*)(psz + so[s]) = vs[s];
                }
        }
    };

    double va[3] = {0.0, 0.0, 0.0}, vb[3] = {0.0, 0.0, 0.0}, sa[2] = {0.0, 0.0}, sb[2] = {0.0, 0.0};
    issue(0);
    cp_async_wait_all();
    fetch(va, sa);
    issue(1);
    cp_async_wait_all();
    fetch(vb, sb);
    issue(2);
    publish_max(va, 0);
    publish_max(vb, 1);
    __syncthreads();
    int E = max(1, plane_max(0));
    bool poisoned = E == 0x7FF;
    convert(0, 0, E, va, sa);

    // Step t (par its parity): plane t + 2 fetched into v2 -- first, so that
    // its FP64 instructions run under the integer work --, the outputs of plane
    // t - 2, the in-plane sums of u(t) and w(t - 1), plane t + 1 (v1) converted.
    auto step = [&](int t, int par, double (&v2)[3], double (&s2)[2], const double (&v1)[3], const double (&s1)[2]) {
        __syncthreads();   // u(t), w(t - 1) and the exponent maximum of plane t + 1 published
        const int ep = t + 1 < T ? plane_max(par ^ 1) : 0;
        cp_async_wait_all();
        double bv[2] = {0.0, 0.0};
        if (has_b) {
#pragma unroll
            for (int s = 0; s < 2; ++s) bv[s] = lds_f64(st + kOwn0 + s * kCol);
        }
        if (t + 2 < T) fetch(v2, s2);
        issue(t + 3);
        const unsigned b0 = tiles + (unsigned)par * kTile + te[0], b1 = b0 + 2 * kTile;
#define ML_AT(b, dy, dx) lds_s64((b) + (unsigned)(8 * ((dy) * PP_HX + (dx))))
        const long long su0 = (ML_AT(b0, 0, -1) + ML_AT(b0, 0, 1)) + (ML_AT(b0, -1, 0) + u0[1]);
        const long long su1 = (ML_AT(b0, 1, -1) + ML_AT(b0, 1, 1)) + (ML_AT(b0, 2, 0) + u0[0]);
        const long long sw0 = (ML_AT(b1, 0, -1) + ML_AT(b1, 0, 1)) + (ML_AT(b1, -1, 0) + wm1[1]);
        const long long sw1 = (ML_AT(b1, 1, -1) + ML_AT(b1, 1, 1)) + (ML_AT(b1, 2, 0) + wm1[0]);
        if (inner) {
            const unsigned br = tiles + (unsigned)par * kTile + te[2];
            gr = mul_w(r0, 6u) - ((ML_AT(br, 0, -1) + ML_AT(br, 0, 1)) + (ML_AT(br, -1, 0) + ML_AT(br, 1, 0))) - rm1;
        }
#undef ML_AT
        const int z = kz0 - 2 + t, zo = z - 2;
        if (zo >= kz0) {
            char* const oz = (char*)a.out + (size_t)zo * plane8;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const long long acc = gq[s] - wm1[s];   // L w of plane zo, complete with w(t - 1)
                if (act[s]) {
                    const double val = fx_result_cvt(acc, E, poisoned);
                    if (kStep) {
                        *(double*)(oz + so[s]) = val;
                        d = __fma_rn(lds_f64(hist + (unsigned)((t + 2) & 3) * (2 * kCol) + s * kCol), val, d);
                    } else {
                        const double rv = has_b ? bv[s] - val : val;
                        if (K == kMarchApply || K == kMarchSub) *(double*)(oz + so[s]) = rv;
                        if (K == kMarchStart) {
                            const size_t o = (size_t)zo * plane8 + so[s];
                            if (a.words)
                                a.words[o / 8] = make_ulonglong2((unsigned long long)__double_as_longlong(rv), 0ull);
                            else
                                *(double*)(oz + so[s]) = rv;
                            if (a.pn) *(double*)((char*)a.pn + o) = rv;
                            if (a.rsn) *(double*)((char*)a.rsn + o) = rv;
                            if (a.psn) *(double*)((char*)a.psn + o) = rv;
                        }
                        if (K != kMarchApply && K != kMarchSub) d = __fma_rn(rv, rv, d);
                    }
                }
            }
        }
        const int cz = f * ((z - 1 == 1) + (z - 1 == n - 1));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            g[s] = mul_w(u0[s], 6u) - (s == 0 ? su0 : su1) - um1[s];
            gq[s] = mul_w(wm1[s], 6u) - (s == 0 ? sw0 : sw1) - wm2[s];
            const int c = (s == 0 ? c0 : c1) + cz;
            if (c) gq[s] += mul_w(um1[s], (unsigned)c);
        }
        if (t + 1 < T) {
            // scale of plane t + 1: a larger exponent shifts what is carried on
            if (ep == 0x7FF) poisoned = true;
            if (ep > E) {
                const int dd = min(ep - E, 63);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    u0[s] >>= dd;
                    wm1[s] >>= dd;
                    g[s] >>= dd;
                    gq[s] >>= dd;
                }
                r0 >>= dd;
                gr >>= dd;
                E = ep;
            }
            if (t + 2 < T) publish_max(v2, par);
            convert(t + 1, par ^ 1, E, v1, s1);
        }
    };
    for (int t = 0; t < T; t += 2) {
        step(t, 0, va, sa, vb, sb);
        if (t + 1 < T) step(t + 1, 1, vb, sb, va, sa);
    }
    cp_async_wait_all();
    return d;
}

}  // namespace
}  // namespace excmg
