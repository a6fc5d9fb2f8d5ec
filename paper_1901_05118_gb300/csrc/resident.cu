// Host side of the resident Bi-CG kernels (resident.cuh).
#include "excmg_internal.cuh"
#include "resident.cuh"

#include <atomic>
#include <map>
#include <mutex>

namespace excmg {
namespace {

template <typename T, int DIM, bool kElide>
const void* resident_fn(int np) {
    switch (np) {
        case 1: return (const void*)resident_bicg_kernel<T, DIM, 1, DIM == 3 ? 2 : 1, kElide>;
        case 2: return (const void*)resident_bicg_kernel<T, DIM, 2, DIM == 3 ? 3 : 1, kElide>;
        case 4: return (const void*)resident_bicg_kernel<T, DIM, 4, DIM == 3 ? 5 : 1, kElide>;
        default: break;
    }
    if constexpr (DIM == 3)
        return np == 6 ? (const void*)resident_bicg_kernel<T, 3, 6, 6, kElide>
                       : (const void*)resident_bicg_kernel<T, 3, 8, 7, kElide>;
    return nullptr;
}

std::mutex g_geom_mu;
std::map<std::pair<int, int>, ResidentGeom> g_geom;   // one entry per size (2D: negative) and CTA limit

}  // namespace

ResidentGeom resident_geometry_cached(int dim, int n, int max_ctas) {
    std::lock_guard<std::mutex> lock(g_geom_mu);
    const auto key = std::make_pair(dim == 3 ? n : -n, max_ctas);
    auto it = g_geom.find(key);
    if (it == g_geom.end())
        it = g_geom.emplace(key, dim == 3 ? resident_geometry(n, max_ctas) : resident_geometry2d(n, max_ctas)).first;
    return it->second;
}

int resident_ctas(int n, int max_ctas) {
    if (n > kResidentMaxN) return 0;
    return resident_geometry_cached(3, n, max_ctas > 0 ? max_ctas : device_sms()).ctas;
}

int resident2d_ctas(int n) { return n > kPersistentMaxN2d ? 0 : resident_geometry_cached(2, n, device_sms()).ctas; }

// CTAs of a grid in the batch engine: fewer than a single solve takes, so that several instances run side by
// side, and a number that depends on the grid alone (the sums do, too).  32^3 on 16 CTAs takes about 1.5
// times as long per iteration as on its own 64, and nine fit beside each other.  (64^3 on 72 CTAs: 18 against
// 11 us per iteration; eight mixed requests then take 74 instead of 50 ms, as the last one waits for itself.)
int resident_batch_limit(int n) { return n <= 32 ? 16 : n <= 52 ? 72 : 0; }

namespace {
// The launch's tag: unique in the process, so no word left by another launch matches.
unsigned next_serial() {
    static std::atomic<unsigned> serial{0};
    unsigned v = ++serial;
    while (v == 0) v = ++serial;
    return v;
}
}  // namespace

size_t resident_slot_bytes() { return (kResWords * sizeof(ulonglong2) + 255) / 256 * 256; }

namespace {
template <typename T>
cudaError_t launch(const void* fn, ResidentGeom g, T* x, T* r, T* rs, T* p, T* ps, int n, int bc_kind, int iters,
                   BicgState* st, void* slots, void* node_words, cudaStream_t s) {
    ResidentInst<T> in{x, r, rs, p, ps, st, (ulonglong2*)slots, (ulonglong2*)node_words, n, bc_kind == 1 ? 1 : -1};
    const size_t smem = (size_t)((g.tile + 1) & ~1) * sizeof(T) + resident_own_bytes(g.np) / 8 * sizeof(T);
    (void)kernel_occupancy(fn, kResThreads, kResSmemBytes);   // opts in to the shared memory
    unsigned serial = next_serial();
    long long limit = kBarrierSpinLimit;
    void* args[] = {&in, &g, &iters, &serial, &limit};
    return cudaLaunchCooperativeKernel(fn, dim3(g.ctas), dim3(kResThreads), args, smem, s);
}
}  // namespace

template <typename T>
cudaError_t launch_bicg_resident(T* x, T* r, T* rs, T* p, T* ps, int n, int bc_kind, int iters, BicgState* st,
                                 void* slots, void* node_words, cudaStream_t s, bool elide, int max_ctas) {
    const ResidentGeom g = resident_geometry_cached(3, n, max_ctas > 0 ? max_ctas : device_sms());
    const void* fn = resident_fn<T, 3, false>(g.np);
    if constexpr (sizeof(T) == 8)
        if (elide) fn = resident_fn<T, 3, true>(g.np);
    return launch<T>(fn, g, x, r, rs, p, ps, n, bc_kind, iters, st, slots, node_words, s);
}

cudaError_t launch_bicg2d_resident(double* x, double* r, double* rs, double* p, double* ps, int n, int bc_kind,
                                   int iters, BicgState* st, void* slots, void* node_words, cudaStream_t s) {
    const ResidentGeom g = resident_geometry_cached(2, n, device_sms());
    return launch<double>(resident_fn<double, 2, false>(g.np), g, x, r, rs, p, ps, n, bc_kind, iters, st, slots,
                          node_words, s);
}

template cudaError_t launch_bicg_resident<double>(double*, double*, double*, double*, double*, int, int, int,
                                                  BicgState*, void*, void*, cudaStream_t, bool, int);
template cudaError_t launch_bicg_resident<float>(float*, float*, float*, float*, float*, int, int, int, BicgState*,
                                                 void*, void*, cudaStream_t, bool, int);

}  // namespace excmg
