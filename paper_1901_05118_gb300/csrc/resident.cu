// Host side of the resident Bi-CG kernels (resident.cuh).
#include "excmg_internal.cuh"
#include "resident.cuh"

#include <atomic>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

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
// side, and a number that depends on the grid alone (the sums do, too).  The on-chip levels of a cascade are
// 16, 20, 24, 28, 32, 40, 48, 56, 64 and 80 (c 2^k, c = 4 .. 8); only between these does it matter where the lines lie.
// Eight first-kind requests on 32^3: 12.7 ms on 16 CTAs, 17.7 on 72 (two: 6.4, 4.5; nine fit beside each other);
// 40^3 does not fit on 16: 29.6 ms on 72, 48.8 on all SMs; 48^3 54.0 and 76.0 (one alone: 15.0, 12.4); 56^3 116
// on 72 and 125 on all (two: 32.4, 33.2), not taken so far; 64^3 74 ms on 72 against 50 for eight mixed requests,
// as the last one waits for itself; 80^3 needs all.
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

int resident_wait_selftest(int exchange, long long limit) {
    constexpr int n = 9;
    const ResidentGeom g = resident_geometry(n, 8);   // four bricks of 4 x 4 x 8
    if (g.ctas < 2 || g.np != 1) return EXCMG_ERR_CUDA;
    const size_t nodes = node_count(n), slots = resident_slot_bytes();
    // slot words, node words, x, r, r*, p, p*, state
    std::vector<unsigned char> host(slots + nodes * 16 + 5 * nodes * 8 + sizeof(BicgState), 0);
    unsigned char* dev = nullptr;
    if (cudaMalloc(&dev, host.size()) != cudaSuccess) {
        cudaGetLastError();
        return EXCMG_ERR_OOM;
    }
    const unsigned serial = next_serial();
    unsigned long long one;
    const double v = 1.0;
    memcpy(&one, &v, 8);
    unsigned long long* const word = (unsigned long long*)host.data();
    for (int c = 0; exchange == 2 && c < kResCopies; ++c) {
        // the missing CTA's sum of exchange 1, and a NaN where that of exchange 2 would be
        unsigned long long* const w1 = word + 2 * ((size_t)c * kResMaxCtas + g.ctas - 1);
        unsigned long long* const w2 = w1 + 2 * (size_t)kResCopies * kResMaxCtas;
        w1[0] = one;
        w1[1] = (unsigned long long)serial << 32;
        w2[0] = w2[1] = ~0ull;
    }
    double* const vec = (double*)(host.data() + slots + nodes * 16);
    for (size_t t = 0; t < 5 * nodes; ++t) vec[t] = 1.0;
    BicgState st{};
    st.rho = st.rr = st.bnorm = 1.0;
    st.beta = 0.5;
    st.iter = 1;   // under way: rr is the kernel's to write
    st.max_iter = 8;
    memcpy(host.data() + host.size() - sizeof st, &st, sizeof st);
    double* const dv = (double*)(dev + slots + nodes * 16);
    BicgState* const ds = (BicgState*)(dv + 5 * nodes);
    ResidentInst<double> in{dv,      dv + nodes, dv + 2 * nodes, dv + 3 * nodes, dv + 4 * nodes, ds, (ulonglong2*)dev,
                            (ulonglong2*)(dev + slots), n, 1};
    const void* fn = resident_fn<double, 3, false>(g.np);
    (void)kernel_occupancy(fn, kResThreads, kResSmemBytes);
    int iters = 8;
    unsigned tag = serial;
    void* args[] = {&in, (void*)&g, &iters, &tag, &limit};
    cudaError_t e = cudaMemcpy(dev, host.data(), host.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel(fn, dim3(g.ctas - 1), dim3(kResThreads), args, (size_t)((g.tile + 1) & ~1) * 8,
                                        nullptr);
    note_launches(1);
    if (e == cudaSuccess) e = cudaMemcpy(&st, ds, sizeof st, cudaMemcpyDeviceToHost);
    cudaFree(dev);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return EXCMG_ERR_CUDA;
    }
    return bicg_outcome(st);
}

}  // namespace excmg
