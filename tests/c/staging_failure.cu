// One launch of a discharge kernel whose wait for the staging copies reports
// failure (the copies themselves have landed): error 2 must be raised and every
// region must stay as it was, active, with no flag left from the sweep before.
// -DVOLUME: the 3D kernel (32x8x4), otherwise the 2D one (32x32, 4-connected).
// Prints "ok" and exits 0, or the first difference and exits 1.
#include <cstdio>
#include <vector>

#include "mf_internal.cuh"

namespace mf {
__device__ bool late_wait(unsigned long long *bar, unsigned phase) {
    mbar_wait(bar, phase);
    return false;
}
}  // namespace mf
#define mbar_wait late_wait
#ifdef VOLUME
#include "ard_discharge3d.cu"
#else
#include "ard_bits2d.cuh"
#endif
#undef mbar_wait

using namespace mf;

template <typename T>
static T *device_copy(const std::vector<T> &h) {
    T *d = nullptr;
    if (cudaMalloc(&d, h.size() * sizeof(T)) != cudaSuccess) return nullptr;
    cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}
template <typename T>
static std::vector<T> host_copy(const T *d, size_t n) {
    std::vector<T> h(n);
    cudaMemcpy(h.data(), d, n * sizeof(T), cudaMemcpyDeviceToHost);
    return h;
}
static int bad(const char *what) {
    printf("%s\n", what);
    return 1;
}

int main() {
#ifdef VOLUME
    constexpr int N = 6;
    Geom g{64, 8, 4, 64 * 8 * 4, 32, 8, 4, 5, 3, 2, 2, 1, 1, 2, 100};
#else
    constexpr int N = 4;
    Geom g{64, 32, 1, 64 * 32, 32, 32, 1, 5, 5, 0, 2, 1, 1, 2, 100};
#endif
    const size_t n = (size_t)g.n;
    std::vector<int> cap(N * n, 3), tcap(n, 1), exc(n, 2), lab(n, 1), bout(N * n, 5), ctr(kCtrWords, 0), hist(kHistBins + 1, 0);
    DevState st{};
    st.cap = device_copy(cap);
    st.tcap = device_copy(tcap);
    st.exc = device_copy(exc);
    st.lab = device_copy(lab);
    st.lab_next = device_copy(lab);
    st.bout = device_copy(bout);
    // region 0 was discharged in the sweep before and nothing was left active in it, region 1 was not discharged
    st.active = device_copy(std::vector<unsigned char>{1, 1});
    st.disc = device_copy(std::vector<unsigned char>{1, 0});
    st.left_active = device_copy(std::vector<unsigned char>{0, 0});
    st.flow_t = device_copy(std::vector<unsigned long long>(1, 0));
    st.flow0 = device_copy(std::vector<long long>(1, 0));
    st.hist = device_copy(hist);
    st.ctr = device_copy(ctr);
    SweepArgs sa{};
    sa.max_rounds = 64;
    sa.active = 2;
    sa.c64 = device_copy(std::vector<Counters64>(1));
    if (cudaDeviceSynchronize() != cudaSuccess || !sa.c64) return bad("set-up");
#ifdef VOLUME
    using C = Cfg3D<8, 4, 128, 4>;
    auto k = ard_discharge3d_kernel<8, 4, 128, 4>;
    const int threads = 128;
#else
    using C = Cfg2D<4, 32, 32, 256>;
    auto k = ard_discharge2d_kernel<4, 32, 32, 256>;
    const int threads = 256;
#endif
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem) != cudaSuccess) return bad("shared memory");
    k<<<g.nreg, threads, C::smem>>>(g, st, sa);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return bad("launch");

    if (host_copy(st.ctr, kCtrWords)[kError] != 2) return bad("error word");
    if (host_copy(st.disc, 2) != std::vector<unsigned char>{0, 0}) return bad("disc: the outflows of the sweep before would be fused");
    if (host_copy(st.left_active, 2) != std::vector<unsigned char>{1, 1}) return bad("left_active: a region would drop out");
    if (host_copy(st.active, 2) != std::vector<unsigned char>{1, 1}) return bad("active");
    if (host_copy(st.cap, N * n) != cap || host_copy(st.tcap, n) != tcap || host_copy(st.exc, n) != exc ||
        host_copy(st.lab, n) != lab || host_copy(st.lab_next, n) != lab || host_copy(st.bout, N * n) != bout)
        return bad("a plane changed");
    if (host_copy(st.flow_t, 1)[0] != 0) return bad("flow");
    printf("ok\n");
    return 0;
}
