// Host side of the resident Bi-CG kernels (resident.cuh).
#include "excmg_internal.cuh"
#include "resident.cuh"

#include <atomic>
#include <map>
#include <mutex>

namespace excmg {
namespace {

template <typename T, bool kElide>
const void* resident_fn(int np) {
    switch (np) {
        case 1: return (const void*)resident_bicg_kernel<T, 1, 2, kElide>;
        case 2: return (const void*)resident_bicg_kernel<T, 2, 3, kElide>;
        default: return (const void*)resident_bicg_kernel<T, 4, 5, kElide>;
    }
}

std::mutex g_geom_mu;
std::map<std::pair<int, int>, ResidentGeom> g_geom;   // at most one entry per size and CTA limit

}  // namespace

ResidentGeom resident_geometry_cached(int n, int max_ctas) {
    std::lock_guard<std::mutex> lock(g_geom_mu);
    auto it = g_geom.find({n, max_ctas});
    if (it == g_geom.end()) it = g_geom.emplace(std::make_pair(n, max_ctas), resident_geometry(n, max_ctas)).first;
    return it->second;
}

int resident_ctas(int n, int max_ctas) {
    if (n > kPersistentMaxN) return 0;
    return resident_geometry_cached(n, max_ctas > 0 ? max_ctas : device_sms()).ctas;
}

// CTAs of a grid in the batch engine: fewer than a single solve takes, so that several instances run side by
// side, and a number that depends on the grid alone (the sums do, too).  32^3 on 16 CTAs takes about 1.5
// times as long per iteration as on its own 64, and nine fit beside each other; 64^3 leaves no choice.
int resident_batch_limit(int n) { return n <= 32 ? 16 : n <= 52 ? 72 : 0; }

namespace {
size_t slot_bytes() { return (kResWords * sizeof(ulonglong2) + 255) / 256 * 256; }

// The launch's tag: unique in the process, so no word left by another launch matches.
unsigned next_serial() {
    static std::atomic<unsigned> serial{0};
    unsigned v = ++serial;
    while (v == 0) v = ++serial;
    return v;
}
}  // namespace

size_t resident_bytes(int n) { return slot_bytes() + node_count(n) * sizeof(ulonglong2); }

template <typename T>
cudaError_t launch_bicg_resident(T* x, T* r, T* rs, T* p, T* ps, int n, int bc_kind, int iters, BicgState* st,
                                 void* words, cudaStream_t s, bool elide, int max_ctas) {
    ResidentGeom g = resident_geometry_cached(n, max_ctas > 0 ? max_ctas : device_sms());
    ResidentInst<T> in{x, r, rs, p, ps, st, (ulonglong2*)words, (ulonglong2*)((char*)words + slot_bytes()), n, bc_kind == 1 ? 1 : -1};
    const size_t smem = (size_t)g.tile * (sizeof(T) == 8 ? sizeof(long long) : sizeof(float));
    const void* fn;
    if constexpr (sizeof(T) == 8)
        fn = elide ? resident_fn<T, true>(g.np) : resident_fn<T, false>(g.np);
    else
        fn = resident_fn<T, false>(g.np);
    (void)kernel_occupancy(fn, kResThreads, kResTileBytes);   // opts in to the shared memory
    unsigned serial = next_serial();
    long long limit = kBarrierSpinLimit;
    void* args[] = {&in, &g, &iters, &serial, &limit};
    return cudaLaunchCooperativeKernel(fn, dim3(g.ctas), dim3(kResThreads), args, smem, s);
}

template cudaError_t launch_bicg_resident<double>(double*, double*, double*, double*, double*, int, int, int,
                                                  BicgState*, void*, cudaStream_t, bool, int);
template cudaError_t launch_bicg_resident<float>(float*, float*, float*, float*, float*, int, int, int, BicgState*,
                                                 void*, cudaStream_t, bool, int);

}  // namespace excmg
