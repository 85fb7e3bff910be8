// The region discharge for the synthetic networks of Sec. 7.1 (connectivity
// codes 100 + c, c = 8 .. 28; displacements up to 4), single solves: the
// bit-parallel kernel (ard_bits2d.cuh) on 32x32 tiles; the generic one
// (ard_generic.cuh) for 64x32 / 64x64 tiles at connectivity 8 (the paper's
// default, for the dependence on the number of regions), whose planes leave no
// room for the masks, for PRD and as kernel_variant 1.  A translation unit of
// its own, since the 28-arc instantiations are the slowest code of the library
// to compile.
#include "ard_bits2d.cuh"
#include "ard_generic.cuh"

#ifdef MF_DIAG  // this unit's copy of the counters (each unit that includes ard_bits2d.cuh has one)
extern "C" int mf_diag_paper_read(unsigned long long *out, int reset) {
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

// the generic kernel's tiles
#define MF_PAPER_TILES(X)           \
    X(108, 32, 32, 1, 256)          \
    X(112, 32, 32, 1, 256)          \
    X(116, 32, 32, 1, 256)          \
    X(120, 32, 32, 1, 256)          \
    X(124, 32, 32, 1, 256)          \
    X(128, 32, 32, 1, 256)          \
    X(108, 64, 32, 1, 256)          \
    X(108, 64, 64, 1, 1024)

bool discharge_paper_supported(int conn, int tx, int ty, int tz) {
#define X(c, a, b, z, t) if (conn == c && tx == a && ty == b && tz == z) return true;
    MF_PAPER_TILES(X)
#undef X
    return false;
}

size_t discharge_paper_smem_bytes(int conn, int tx, int ty, int tz) {
#define X(c, a, b, z, t) if (conn == c && tx == a && ty == b && tz == z) return TileCfg<c, a, b, z, t>::smem;
    MF_PAPER_TILES(X)
#undef X
    return 0;
}

cudaError_t launch_discharge_paper(int conn, const Geom &g, const DevState &st, const SweepArgs &sa,
                                   cudaStream_t stream) {
    // the bit-parallel discharge, except for PRD, kernel_variant 1 and the larger tiles
    if (sa.variant == 0 && g.tx == 32 && g.ty == 32) {
        switch (conn) {
            case 108: return launch2d<108, 32, 32, 256>(g, st, sa, stream);
            case 112: return launch2d<112, 32, 32, 256>(g, st, sa, stream);
            case 116: return launch2d<116, 32, 32, 256>(g, st, sa, stream);
            case 120: return launch2d<120, 32, 32, 256>(g, st, sa, stream);
            case 124: return launch2d<124, 32, 32, 256>(g, st, sa, stream);
            case 128: return launch2d<128, 32, 32, 256>(g, st, sa, stream);
            default: return cudaErrorInvalidValue;
        }
    }
#define X(c, a, b, z, t) \
    if (conn == c && g.tx == a && g.ty == b && g.tz == z) return launch_one<c, a, b, z, t>(g, st, sa, stream);
    MF_PAPER_TILES(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace mf
