// The bit-parallel 2D discharge (ard_bits2d.cuh) for the 4- and 8-connected
// grids: single grids, batches and the dispatch over tile shapes.
#include "ard_bits2d.cuh"

#ifdef MF_DIAG
extern "C" int mf_diag_read(unsigned long long *out, int reset) {
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    if (cudaMemcpyFromSymbol(out, mf::mf_diag, sizeof(unsigned long long) * 32) != cudaSuccess) return 2;
    if (reset) {
        static const unsigned long long z[32] = {0};
        if (cudaMemcpyToSymbol(mf::mf_diag, z, sizeof(z)) != cudaSuccess) return 3;
    }
    return 0;
}
#endif

namespace mf {

// persistent blocks over a work queue of (instance, region) items of a batch
template <int CONN, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT, (Cfg2D<CONN, TX, TY, NT>::MINB))
ard_discharge2d_batch_kernel(const Inst *__restrict__ insts, const int2 *__restrict__ items, const int *count,
                             int *head, const SweepArgs sa) {
    __shared__ int s_it;
    __shared__ __align__(8) unsigned long long s_mbar;
    if (threadIdx.x == 0) mbar_init(&s_mbar, 1);
    unsigned phase = 0;
    for (;;) {
        __syncthreads();  // the previous item is done with s_it and the shared planes
        if (threadIdx.x == 0) s_it = atomicAdd(head, 1);
        __syncthreads();
        const int it = s_it;
        if (it >= *count) break;
        const int2 w = items[it];
        const Inst &I = insts[w.x];
        SweepArgs a = sa;
        a.c64 = I.c64;
        discharge2d_region<CONN, TX, TY, NT>(I.g, I.st, a, w.y, &s_mbar, phase);
    }
}

template <int CONN, int TX, int TY, int NT>
static cudaError_t launch2d_batch(const Inst *insts, const int2 *items, const int *count, int *head,
                                  const SweepArgs &sa, int blocks, cudaStream_t s) {
    using C = Cfg2D<CONN, TX, TY, NT>;
    auto k = ard_discharge2d_batch_kernel<CONN, TX, TY, NT>;
    {
        const cudaError_t e_at = ensure_smem_attr((const void *)k, (int)C::smem);
        if (e_at != cudaSuccess) return e_at;
    }
    const int resident = device_sms() * C::MINB;  // persistent blocks: at least as many as can be resident
    k<<<blocks > resident ? blocks : resident, NT, C::smem, s>>>(insts, items, count, head, sa);
    return cudaGetLastError();
}

bool discharge2d_supported(int conn, int tx, int ty) {
    return (conn == 4 || conn == 8) &&
           ((tx == 64 && ty == 64) || (tx == 32 && ty == 32) || (tx == 64 && ty == 32) || (tx == 32 && ty == 16));
}

cudaError_t launch_discharge2d_batch(int conn, int tx, int ty, const Inst *insts, const int2 *items,
                                     const int *count, int *head, const SweepArgs &sa, int blocks,
                                     cudaStream_t stream) {
    if (conn == 4 && tx == 64 && ty == 64) return launch2d_batch<4, 64, 64, 512>(insts, items, count, head, sa, blocks, stream);
    if (conn == 8 && tx == 64 && ty == 64) return launch2d_batch<8, 64, 64, 512>(insts, items, count, head, sa, blocks, stream);
    if (conn == 4 && tx == 32 && ty == 32) return launch2d_batch<4, 32, 32, 256>(insts, items, count, head, sa, blocks, stream);
    if (conn == 8 && tx == 32 && ty == 32) return launch2d_batch<8, 32, 32, 256>(insts, items, count, head, sa, blocks, stream);
    if (conn == 4 && tx == 64 && ty == 32) return launch2d_batch<4, 64, 32, 256>(insts, items, count, head, sa, blocks, stream);
    if (conn == 8 && tx == 64 && ty == 32) return launch2d_batch<8, 64, 32, 256>(insts, items, count, head, sa, blocks, stream);
    if (conn == 4 && tx == 32 && ty == 16) return launch2d_batch<4, 32, 16, 128>(insts, items, count, head, sa, blocks, stream);
    if (conn == 8 && tx == 32 && ty == 16) return launch2d_batch<8, 32, 16, 128>(insts, items, count, head, sa, blocks, stream);
    return cudaErrorInvalidValue;
}

cudaError_t launch_discharge2d(int conn, const Geom &g, const DevState &st, const SweepArgs &sa,
                               cudaStream_t stream) {
    if (conn == 4 && g.tx == 64 && g.ty == 64) return launch2d<4, 64, 64, 512>(g, st, sa, stream);
    if (conn == 8 && g.tx == 64 && g.ty == 64) return launch2d<8, 64, 64, 512>(g, st, sa, stream);
    if (conn == 4 && g.tx == 32 && g.ty == 32) return launch2d<4, 32, 32, 256>(g, st, sa, stream);
    if (conn == 8 && g.tx == 32 && g.ty == 32) return launch2d<8, 32, 32, 256>(g, st, sa, stream);
    if (conn == 4 && g.tx == 64 && g.ty == 32) return launch2d<4, 64, 32, 256>(g, st, sa, stream);
    if (conn == 8 && g.tx == 64 && g.ty == 32) return launch2d<8, 64, 32, 256>(g, st, sa, stream);
    if (conn == 4 && g.tx == 32 && g.ty == 16) return launch2d<4, 32, 16, 128>(g, st, sa, stream);
    if (conn == 8 && g.tx == 32 && g.ty == 16) return launch2d<8, 32, 16, 128>(g, st, sa, stream);
    return cudaErrorInvalidValue;
}

}  // namespace mf
