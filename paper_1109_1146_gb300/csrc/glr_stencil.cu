// Exact region-distance relabel (the global relabel heuristic) for any 2D
// stencil: the grids with the longer displacements of the Sec. 7.1 synthetic
// networks, where the bit-mask relabel of cut2d.cu (unit shifts) does not apply,
// and the 4- and 8-connected grids on 32x32 tiles.
//
// d*(u) = the least number of inter-region arcs on a residual path from u to
// t (the region distance of Sec. 4.1, eq. 3).  Level sets S_0 ⊆ S_1 ⊆ ...:
// S_0 = vertices that reach t through residual arcs inside their own region;
// S_l adds every vertex with a residual inter-region arc into S_{l-1}, then
// closes each region under its inner residual arcs.  A vertex first reached
// at level l gets d := max(d, l); vertices never reached get d_inf (as the 2D
// and 3D relabels).  All levels run in one cooperative launch with a grid
// barrier per level.
//
// 32x32 tiles: one warp per region on bit masks, a lane per tile row (a word of
// 32 vertices); a step of the closure is a shift and an and per arc.  Larger
// tiles: one thread block per region, one byte per vertex in shared memory.
// Bound by latency (grid barriers, L2 round trips).  500x500, connectivity 8,
// 14 relabels of 26 levels: 54.6 ms as blocks on bytes with the capacities
// read again in every pass, 4.9 ms as warps on masks (3.3 ms
// with the labels of a row raised together).  Against the 64x64 blocks of
// cut2d.cu (64-bit words, two rows per lane, every block at every level) on
// 32x32 tiles: 1.02 -> 0.72 ms for the 7 relabels of the 637x419 8-connected
// grid, 0.30 -> 0.22 ms (3, 1024x1024 4-connected), 0.89 -> 0.75 ms (3,
// 2048x2048 8-connected).
#include <algorithm>
#include <climits>

#include <cooperative_groups.h>

#include "mf_internal.cuh"

namespace mf {

namespace cg = cooperative_groups;

// level `level` of region r: S_l(r) from S_{l-1} (in; unused at level 0) into
// out; raises the labels of the vertices it adds; returns whether it added any
template <int CONN, int TX, int TY>
__device__ bool stencil_region_level(const Geom &g, const DevState &st, int r, const unsigned char *in,
                                     unsigned char *out, int level, unsigned char *m) {
    constexpr int N = arcs_of(CONN), V = TX * TY;
    constexpr int SX = TX == 64 ? 6 : 5;  // log2 TX
    const int rx = r % g.RX, ry = r / g.RX;
    const size_t n = (size_t)g.n;
    for (int i = threadIdx.x; i < V; i += blockDim.x) {
        const int x = rx * TX + (i & (TX - 1)), y = ry * TY + (i >> SX);
        unsigned char s = 0;
        if (x < g.X && y < g.Y) {
            const size_t v = (size_t)y * g.X + x;
            if (level == 0) {
                s = st.tcap[v] > 0;
            } else {
                s = in[v];
#pragma unroll
                for (int d = 0; d < N && !s; ++d) {  // a residual arc into S_{l-1} of another region
                    const int wx = x + arc_dx(CONN, d), wy = y + arc_dy(CONN, d);
                    if (wx < 0 || wx >= g.X || wy < 0 || wy >= g.Y) continue;
                    if (wx / TX == rx && wy / TY == ry) continue;
                    s = in[(size_t)wy * g.X + wx] && st.cap[(size_t)d * n + v] > 0;
                }
            }
        }
        m[i] = s;
    }
    __syncthreads();
    // closure inside the region (monotone: a stale read only delays)
    for (;;) {
        int ch = 0;
        for (int i = threadIdx.x; i < V; i += blockDim.x) {
            if (m[i]) continue;
            const int lx = i & (TX - 1), ly = i >> SX;
            const int x = rx * TX + lx, y = ry * TY + ly;
            if (x >= g.X || y >= g.Y) continue;
            const size_t v = (size_t)y * g.X + x;
#pragma unroll
            for (int d = 0; d < N; ++d) {
                const int nx = lx + arc_dx(CONN, d), ny = ly + arc_dy(CONN, d);
                if (nx < 0 || nx >= TX || ny < 0 || ny >= TY) continue;
                if (x + arc_dx(CONN, d) >= g.X || y + arc_dy(CONN, d) >= g.Y) continue;
                if (m[ny * TX + nx] && st.cap[(size_t)d * n + v] > 0) {
                    m[i] = 1;
                    ch = 1;
                    break;
                }
            }
        }
        if (!__syncthreads_or(ch)) break;
    }
    int grew = 0;
    for (int i = threadIdx.x; i < V; i += blockDim.x) {
        const int x = rx * TX + (i & (TX - 1)), y = ry * TY + (i >> SX);
        if (x >= g.X || y >= g.Y) continue;
        const size_t v = (size_t)y * g.X + x;
        out[v] = m[i];
        if (level > 0 && m[i] && !in[v]) {
            grew = 1;
            if (st.lab[v] < level) st.lab[v] = level;
        }
    }
    return __syncthreads_or(grew) != 0;
}

// all levels in one cooperative launch; flags[3] triple-buffered "grew" words
template <int CONN, int TX, int TY>
__global__ void stencil_glr_levels_kernel(const Geom g, const DevState st, unsigned char *A, unsigned char *B,
                                          int *flags, int *levels_out, int max_levels) {
    cg::grid_group grid = cg::this_grid();
    __shared__ unsigned char m[TX * TY];
    for (int r = blockIdx.x; r < g.nreg; r += gridDim.x) stencil_region_level<CONN, TX, TY>(g, st, r, nullptr, B, 0, m);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        flags[1] = 0;
        flags[2] = 0;
    }
    grid.sync();
    int level = 1;
    for (; level < max_levels; ++level) {
        const unsigned char *in = (level & 1) ? B : A;
        unsigned char *out = (level & 1) ? A : B;
        bool grew = false;
        for (int r = blockIdx.x; r < g.nreg; r += gridDim.x)
            grew |= stencil_region_level<CONN, TX, TY>(g, st, r, in, out, level, m);
        if (grew && threadIdx.x == 0) atomicOr(&flags[level % 3], 1);
        if (blockIdx.x == 0 && threadIdx.x == 0) flags[(level + 1) % 3] = 0;
        grid.sync();
        if (!*(volatile int *)&flags[level % 3]) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *levels_out = level + 1;
}

// ---- 32x32 tiles: bit masks ----------------------------------------------------
// Scratch in words: M[N][Y][RX] residual masks (bit x of a word = vertex
// rx * 32 + x), T[Y][RX] residual sink arcs, S[Y][RX] the set, N0 / N1[Y][RX] what
// joined it at the last even / odd level, then a byte per region and parity:
// did anything join (the words of a region that did not grow are not read).
struct StencilBits {
    unsigned *M, *T, *S, *Nw[2];
    unsigned char *grew[2];
};
static __host__ __device__ size_t stencil_words(const Geom &g) { return (size_t)g.Y * g.RX; }
static StencilBits stencil_bits(int conn, const Geom &g, void *scratch) {
    StencilBits b;
    const size_t w = stencil_words(g);
    b.M = (unsigned *)scratch;
    b.T = b.M + (size_t)arcs_of(conn) * w;
    b.S = b.T + w;
    b.Nw[0] = b.S + w;
    b.Nw[1] = b.Nw[0] + w;
    b.grew[0] = (unsigned char *)(b.Nw[1] + w);
    b.grew[1] = b.grew[0] + g.nreg;
    return b;
}

// one warp per word: coalesced reads of every plane, a ballot per arc
template <int CONN>
__global__ void stencil_masks_kernel(const Geom g, const DevState st, const StencilBits sb) {
    constexpr int N = arcs_of(CONN);
    const int lane = threadIdx.x & 31;
    const size_t n = (size_t)g.n, words = stencil_words(g);
    const size_t nw = (size_t)gridDim.x * (blockDim.x >> 5);
    for (size_t w = blockIdx.x * (size_t)(blockDim.x >> 5) + (threadIdx.x >> 5); w < words; w += nw) {
        const int y = (int)(w / g.RX), x = (int)(w - (size_t)y * g.RX) * 32 + lane;
        const bool in = x < g.X;
        const size_t v = (size_t)y * g.X + x;
        unsigned mine = 0;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const unsigned b = __ballot_sync(0xffffffffu, in && st.cap[(size_t)d * n + v] > 0);
            if (lane == d) mine = b;
        }
        const unsigned t = __ballot_sync(0xffffffffu, in && st.tcap[v] > 0);
        if (lane < N) sb.M[lane * words + w] = mine;
        if (lane == N) sb.T[w] = t;
    }
}

__device__ __forceinline__ unsigned fill_row(unsigned f, unsigned pl, unsigned pr) {  // runs along the +-x arcs
    unsigned a = f, p = pl;
    a |= p & (a >> 1);  p &= p >> 1;
    a |= p & (a >> 2);  p &= p >> 2;
    a |= p & (a >> 4);  p &= p >> 4;
    a |= p & (a >> 8);  p &= p >> 8;
    a |= p & (a >> 16);
    p = pr;
    f |= p & (f << 1);  p &= p << 1;
    f |= p & (f << 2);  p &= p << 2;
    f |= p & (f << 4);  p &= p << 4;
    f |= p & (f << 8);  p &= p << 8;
    f |= p & (f << 16);
    return a | f;
}

template <int CONN>
__global__ void __launch_bounds__(128) stencil_glr_bits_kernel(const Geom g, const DevState st, const StencilBits sb,
                                                               int *flags, int *levels_out, int max_levels) {
    constexpr int N = arcs_of(CONN), R = radius_of(CONN);
    constexpr unsigned FULL = 0xffffffffu;
    cg::grid_group grid = cg::this_grid();
    const int lane = threadIdx.x & 31;
    const size_t words = stencil_words(g);
    const int w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), nw = gridDim.x * (blockDim.x >> 5);
    int level = 0;
    for (; level < max_levels; ++level) {
        bool grew = false;
        const unsigned *in = sb.Nw[(level + 1) & 1];
        unsigned *out = sb.Nw[level & 1];
        for (int r = w0; r < g.nreg; r += nw) {
            const int rx = r % g.RX, ry = r / g.RX, y = ry * 32 + lane;
            const bool row = y < g.Y;
            const size_t w = (size_t)y * g.RX + rx;
            // the neighbour regions (3x3, bit 4 is the region itself) that grew at the last level
            unsigned near = 0;
            if (level > 0) {
                const int qx = rx + lane % 3 - 1, qy = ry + lane / 3 - 1;
                const bool f = lane < 9 && lane != 4 && qx >= 0 && qx < g.RX && qy >= 0 && qy < g.RY &&
                               __ldcg(&sb.grew[(level + 1) & 1][qy * g.RX + qx]) != 0;
                near = __ballot_sync(FULL, f);
                if (!near) {
                    if (lane == 0) sb.grew[level & 1][r] = 0;
                    continue;
                }
            }
            unsigned Rm[N];
#pragma unroll
            for (int d = 0; d < N; ++d) Rm[d] = row ? sb.M[d * words + w] : 0u;
            const unsigned old = row && level > 0 ? sb.S[w] : 0u;
            unsigned f = 0;
            if (level == 0) {
                f = row ? sb.T[w] : 0u;
            } else {
                // residual arcs into what joined another region at the last level
#pragma unroll
                for (int dy = -R; dy <= R; ++dy) {
                    const int gy = y + dy, q = (gy >> 5) - ry;
                    unsigned c = 0, lw = 0, rw = 0;
                    if (row && gy >= 0 && gy < g.Y) {
                        const unsigned fl = near >> (3 * (q + 1));
                        const unsigned *p = in + (size_t)gy * g.RX + rx;
                        if (q != 0 && (fl & 2u)) c = __ldcg(p);
                        if (fl & 1u) lw = __ldcg(p - 1);
                        if (fl & 4u) rw = __ldcg(p + 1);
                    }
#pragma unroll
                    for (int d = 0; d < N; ++d) {
                        if (arc_dy(CONN, d) != dy) continue;
                        constexpr int kW = 32;
                        const int dx = arc_dx(CONN, d);
                        unsigned t = c;  // bit x: the head of the arc from column x
                        if (dx > 0) t = (c >> dx) | (rw << (kW - dx));
                        if (dx < 0) t = (c << -dx) | (lw >> (kW + dx));
                        f |= Rm[d] & t;
                    }
                }
            }
            f &= ~old;
            // closure inside the region
            unsigned S = old, fr = fill_row(f, Rm[0] & ~old, Rm[1] & ~old) & ~old;
            while (__any_sync(FULL, fr != 0u)) {
                S |= fr;
                unsigned rows[2 * R + 1], a = 0;
#pragma unroll
                for (int q = 1; q <= R; ++q) {
                    const unsigned u = __shfl_up_sync(FULL, fr, q), d = __shfl_down_sync(FULL, fr, q);
                    rows[R - q] = lane >= q ? u : 0u;
                    rows[R + q] = lane + q < 32 ? d : 0u;
                }
                rows[R] = fr;
#pragma unroll
                for (int d = 0; d < N; ++d) {
                    const int dx = arc_dx(CONN, d);
                    const unsigned t = rows[arc_dy(CONN, d) + R];
                    a |= Rm[d] & (dx > 0 ? t >> dx : t << -dx);
                }
                fr = fill_row(a & ~S, Rm[0] & ~S, Rm[1] & ~S) & ~S;
            }
            const unsigned joined = S & ~old;
            const unsigned rows = __ballot_sync(FULL, joined != 0u);
            if (lane == 0) sb.grew[level & 1][r] = rows != 0u;
            if (level == 0 && row) sb.S[w] = S;
            if (!rows) continue;
            grew = true;
            if (row) {
                sb.S[w] = S;
                out[w] = joined;
            }
            if (level > 0) raise_labels(st.lab, joined, (size_t)y * g.X + (size_t)rx * 32, level);
        }
        if (grew && lane == 0) atomicOr(&flags[level % 3], 1);
        if (blockIdx.x == 0 && threadIdx.x == 0) flags[(level + 1) % 3] = 0;
        grid.sync();
        // (level 0 always continues: the level count is that of the first level that adds nothing)
        if (level > 0 && !*(volatile int *)&flags[level % 3]) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *levels_out = level + 1;
}

// unreached vertices get d_inf; boundary-label histogram and region activity
// (the set as bits, or as the bytes A / B)
template <int CONN>
__global__ void stencil_glr_finish_kernel(const Geom g, const DevState st, const unsigned *bits,
                                          const unsigned char *A, const unsigned char *B) {
    constexpr int SB = 2048;
    const int last = st.ctr[kGlrLevels] - 1;  // level 0 and the even levels wrote B
    const unsigned char *S = (last % 2 == 1) ? A : B;
    __shared__ int sh[SB];
    for (int b = threadIdx.x; b < SB; b += blockDim.x) sh[b] = 0;
    __syncthreads();
    for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < (size_t)g.n; v += (size_t)gridDim.x * blockDim.x) {
        const int y = (int)(v / g.X), x = (int)(v - (size_t)y * g.X);
        int l = st.lab[v];
        if (!(bits ? (bits[(size_t)y * g.RX + (x >> 5)] >> (x & 31)) & 1u : S[v])) {
            l = g.dinf;
            st.lab[v] = l;
        }
        if (l >= g.dinf) continue;
        const int r = (y >> g.sy) * g.RX + (x >> g.sx);
        if (st.exc[v] > 0) st.active[r] = 1;
        bool inB = false;
#pragma unroll
        for (int d = 0; d < arcs_of(CONN); ++d) {
            const int wx = x + arc_dx(CONN, d), wy = y + arc_dy(CONN, d);
            if (wx < 0 || wx >= g.X || wy < 0 || wy >= g.Y) continue;
            inB |= (wy >> g.sy) * g.RX + (wx >> g.sx) != r;
        }
        if (!inB) continue;
        if (l < SB) atomicAdd(&sh[l], 1);
        else atomicAdd(&st.hist[l < kHistBins ? l : kHistBins], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < SB; b += blockDim.x)
        if (sh[b]) atomicAdd(&st.hist[b], sh[b]);
}

__global__ void stencil_glr_count_kernel(const DevState st, int nreg) {
    int c = 0;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nreg; r += gridDim.x * blockDim.x) c += st.active[r] != 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&st.ctr[kActiveRegions], c);
}

template <int CONN>
static cudaError_t stencil_glr_finish(const Geom &g, const DevState &st, const unsigned *bits, const unsigned char *A,
                                      const unsigned char *B, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(st.hist, 0, (kHistBins + 1) * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(st.active, 0, (size_t)g.nreg, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&st.ctr[kActiveRegions], 0, 4, s);
    if (e != cudaSuccess) return e;
    const int nb = (int)std::min<size_t>(((size_t)g.n + 255) / 256, device_sms() * 32);
    stencil_glr_finish_kernel<CONN><<<nb, 256, 0, s>>>(g, st, bits, A, B);
    stencil_glr_count_kernel<<<(g.nreg + 255) / 256, 256, 0, s>>>(st, g.nreg);
    return cudaGetLastError();
}

// 32x32 tiles: masks, then all levels in one cooperative launch
template <int CONN>
static cudaError_t stencil_glr_bits(const Geom &g, const DevState &st, void *scratch, cudaStream_t s) {
    StencilBits sb = stencil_bits(CONN, g, scratch);
    int max_blocks = 0;
    cudaError_t e = coop_max_blocks((const void *)stencil_glr_bits_kernel<CONN>, 128, 0, &max_blocks);
    if (e != cudaSuccess) return e;
    const int mb = (int)std::min<size_t>((stencil_words(g) + 7) / 8, (size_t)device_sms() * 16);
    stencil_masks_kernel<CONN><<<mb, 256, 0, s>>>(g, st, sb);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int nblocks = std::max(1, std::min((g.nreg + 3) / 4, max_blocks));
    int *flags = &st.ctr[kGlrFlags];
    int *lvl = &st.ctr[kGlrLevels];
    int max_levels = 1 << 20;
    Geom gg = g;
    DevState ss = st;
    void *args[] = {&gg, &ss, &sb, &flags, &lvl, &max_levels};
    e = cudaLaunchCooperativeKernel((const void *)stencil_glr_bits_kernel<CONN>, dim3(nblocks), dim3(128), args, 0, s);
    if (e != cudaSuccess) return e;
    return stencil_glr_finish<CONN>(g, st, sb.S, nullptr, nullptr, s);
}

// larger tiles: bytes, a block per region
template <int CONN, int TX, int TY>
static cudaError_t stencil_glr_impl(const Geom &g, const DevState &st, void *scratch, cudaStream_t s) {
    unsigned char *A = (unsigned char *)scratch, *B = A + g.n;
    int max_blocks = 0;
    {
        const cudaError_t e_mb = coop_max_blocks((const void *)stencil_glr_levels_kernel<CONN, TX, TY>, 256, 0, &max_blocks);
        if (e_mb != cudaSuccess) return e_mb;
    }
    const int nblocks = std::max(1, std::min(g.nreg, max_blocks));
    int *flags = &st.ctr[kGlrFlags];
    int *lvl = &st.ctr[kGlrLevels];
    int max_levels = 1 << 20;
    Geom gg = g;
    DevState ss = st;
    void *args[] = {&gg, &ss, &A, &B, &flags, &lvl, &max_levels};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)stencil_glr_levels_kernel<CONN, TX, TY>, dim3(nblocks),
                                                dim3(256), args, 0, s);
    if (e != cudaSuccess) return e;
    return stencil_glr_finish<CONN>(g, st, nullptr, A, B, s);
}

bool stencil_glr_supported(int conn, const Geom &g) {
    if (conn == 4 || conn == 8) return g.tz == 1 && g.tx == 32 && g.ty == 32;  // called by glr2d for these tiles
    return is_paper(conn) && g.tz == 1 &&
           ((g.tx == 32 && g.ty == 32) || (conn == 108 && g.tx == 64 && (g.ty == 32 || g.ty == 64)));
}

size_t stencil_glr_scratch_bytes(int conn, const Geom &g) {
    if (g.tx == 32) return (size_t)(arcs_of(conn) + 4) * stencil_words(g) * 4 + 2 * (size_t)g.nreg;
    return 2 * (size_t)g.n;
}

cudaError_t stencil_glr(int conn, const Geom &g, const DevState &st, void *scratch, cudaStream_t s) {
    if (g.tx == 64) {  // connectivity 8 only
        if (conn != 108) return cudaErrorInvalidValue;
        return g.ty == 64 ? stencil_glr_impl<108, 64, 64>(g, st, scratch, s) : stencil_glr_impl<108, 64, 32>(g, st, scratch, s);
    }
    switch (conn) {
        case 4: return stencil_glr_bits<4>(g, st, scratch, s);
        case 8: return stencil_glr_bits<8>(g, st, scratch, s);
        case 108: return stencil_glr_bits<108>(g, st, scratch, s);
        case 112: return stencil_glr_bits<112>(g, st, scratch, s);
        case 116: return stencil_glr_bits<116>(g, st, scratch, s);
        case 120: return stencil_glr_bits<120>(g, st, scratch, s);
        case 124: return stencil_glr_bits<124>(g, st, scratch, s);
        case 128: return stencil_glr_bits<128>(g, st, scratch, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mf
