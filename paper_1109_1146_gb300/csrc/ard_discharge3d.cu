// Region discharge of P-ARD for 3D 6-connected tiles with bit-parallel graph
// search.
//
// The same computation as ard_discharge.cu and ard_bits2d.cuh (Procedure
// ARD of Sec. 4.2, Procedure Augment in synchronous rounds of "exact BFS from
// T_k, then a layered push from the highest BFS layer down", the ARD
// region-relabel of Sec. 5.1), for tiles 32 voxels wide in x:
//
//   * a "row" is the run of 32 voxels along x at one (y, z) of the tile, row
//     index rho = z * TY + y; every mask holds one 32-bit word per row:
//     R_d[rho] bit x = [c_f(v -> v + D(d)) > 0] for the six arcs
//     d = +x, -x, +y, -y, +z, -z, T[rho] = [c_f(v,t) > 0], E[rho] = [e_f(v) > 0];
//   * warp 0 (the graph warp) holds these masks in registers, lane l the rows
//     l*RPL .. l*RPL+RPL-1, and runs every BFS and reachability flood on them: a
//     step shifts a word for +-x, takes the neighbouring row for +-y (a shuffle
//     across one lane at the ends of a lane's rows) and the row TY away for +-z
//     (a shuffle across TY/RPL lanes); floods close whole x-runs at once
//     (Kogge-Stone fill);
//   * every arc leaving the tile ends in its own halo cell (six faces), so the
//     boundary of T_k is a table over halo cells: hm[h] = d(h) if the arc
//     into h has residual capacity, else infinity;
//   * the graph warp also runs the layered push, a lane per row, unless a layer
//     has many pushing vertices in one row; those layers are pushed by all warps;
//   * all warps do the staging, the labels and the write-back.
#include <climits>
#include <cstdint>
#include <utility>

#include "mf_internal.cuh"

namespace mf {

typedef unsigned int u32;

#ifdef MF_DIAG
__device__ unsigned long long mf_diag3[32];
}  // namespace mf
extern "C" int mf_diag3_read(unsigned long long *out, int reset) {
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    if (cudaMemcpyFromSymbol(out, mf::mf_diag3, sizeof(unsigned long long) * 32) != cudaSuccess) return 2;
    if (reset) {
        static const unsigned long long z[32] = {0};
        if (cudaMemcpyToSymbol(mf::mf_diag3, z, sizeof(z)) != cudaSuccess) return 3;
    }
    return 0;
}
namespace mf {
#define mf_diag mf_diag3
#endif

// MB: resident blocks per SM the registers must allow
template <int TY, int TZ, int NT, int MB>
struct Cfg3D {
    static constexpr int TX = 32, N = 6;
    static constexpr int NR = TY * TZ;            // rows of the tile
    static constexpr int V = TX * NR;             // voxels
    static constexpr int NW = NT / 32;            // warps
    static constexpr bool PART = NR < 32;         // 16-row tiles: lanes 16..31 of the graph warp hold no row
    static constexpr int RPL = PART ? 1 : NR / 32;  // rows per lane of the graph warp
    static constexpr int LZ = TY / RPL;           // lanes between rows rho and rho + TY
    // halo faces: -x, +x (one cell per row), -y, +y (TX per z), -z, +z (TX per y)
    static constexpr int B_MX = 0, B_PX = NR, B_MY = 2 * NR, B_PY = 2 * NR + TX * TZ;
    static constexpr int B_MZ = 2 * NR + 2 * TX * TZ, B_PZ = B_MZ + TX * TY;
    static constexpr int HL = B_PZ + TX * TY;     // halo cells = arcs leaving the tile
    // BFS layers kept as masks (24 let five 32x8x4 tiles share an SM's memory)
    static constexpr int LCAP = MB == 5 ? 24 : 32;
    static constexpr size_t smem = (size_t)(N + 3) * V * 4           // cap, tcap, exc, lab
                                   + (size_t)(N + 4) * NR * 4        // R[N], T, E, inc, vis
                                   + (size_t)(LCAP + 1) * NR * 4     // BFS layers 1..LCAP
                                   + (size_t)HL * 4 + NR + 16;       // halo labels, dirty rows, padding
    // after this many passes of the graph warp over a push layer the rest of it
    // is handed to all warps
    static constexpr int HEAVY = 8;
    static_assert((NR % 32 == 0 || NR == 16) && TY % RPL == 0 && V % NT == 0 && NT % 32 == 0, "tile/threads mismatch");
};

// Kogge-Stone fill inside one 32-bit row: x joins if x+1 is in g and pl[x]
// (arc x -> x+1), or x-1 is in g and pr[x] (arc x -> x-1), repeatedly.
__device__ __forceinline__ u32 row_fill32(u32 g, u32 pl, u32 pr) {
    u32 a = g, p = pl;
    a |= p & (a >> 1);  p &= p >> 1;
    a |= p & (a >> 2);  p &= p >> 2;
    a |= p & (a >> 4);  p &= p >> 4;
    a |= p & (a >> 8);  p &= p >> 8;
    a |= p & (a >> 16);
    u32 b = g;
    p = pr;
    b |= p & (b << 1);  p &= p << 1;
    b |= p & (b << 2);  p &= p << 2;
    b |= p & (b << 4);  p &= p << 4;
    b |= p & (b << 8);  p &= p << 8;
    b |= p & (b << 16);
    return a | b;
}

__device__ __forceinline__ int deep_tag3(int epoch, int L) { return ~((epoch << 16) | L); }

// halo cell of the arc d leaving the tile at tile voxel (lx, ly, lz)
template <int TY, int TZ>
__device__ __forceinline__ int halo3(int d, int lx, int ly, int lz) {
    constexpr int TX = 32, NR = TY * TZ;
    constexpr int B_MX = 0, B_PX = NR, B_MY = 2 * NR, B_PY = 2 * NR + TX * TZ;
    constexpr int B_MZ = 2 * NR + 2 * TX * TZ, B_PZ = B_MZ + TX * TY;
    switch (d) {
        case 0: return B_PX + lz * TY + ly;
        case 1: return B_MX + lz * TY + ly;
        case 2: return B_PY + lz * TX + lx;
        case 3: return B_MY + lz * TX + lx;
        case 4: return B_PZ + ly * TX + lx;
        default: return B_MZ + ly * TX + lx;
    }
}

// tile voxel and arc of halo cell h (inverse of halo3); the cell itself lies
// one step along the arc
template <int TY, int TZ>
__device__ __forceinline__ void halo3_src(int h, int &lx, int &ly, int &lz, int &d) {
    constexpr int TX = 32, NR = TY * TZ;
    if (h < NR) { lx = 0; ly = h % TY; lz = h / TY; d = 1; return; }
    if (h < 2 * NR) { const int q = h - NR; lx = TX - 1; ly = q % TY; lz = q / TY; d = 0; return; }
    int q = h - 2 * NR;
    if (q < TX * TZ) { lx = q % TX; lz = q / TX; ly = 0; d = 3; return; }
    q -= TX * TZ;
    if (q < TX * TZ) { lx = q % TX; lz = q / TX; ly = TY - 1; d = 2; return; }
    q -= TX * TZ;
    if (q < TX * TY) { lx = q % TX; ly = q / TX; lz = 0; d = 5; return; }
    q -= TX * TY;
    lx = q % TX; ly = q / TX; lz = TZ - 1; d = 4;
}

// highest set bit of a row word; `other` if there is none
__device__ __forceinline__ int top_bit3(u32 m, int other) {
    int x;
    asm("bfind.u32 %0, %1;" : "=r"(x) : "r"(m));
    return m ? x : other;
}
// Predicated shared-memory store at a constant offset (bytes) from an address,
// and the planes after the vertex at `a` (the address of its cap[0]) sent dl
// along arc D; c and rc: the residuals of the arc and of its reverse before.
// An arc has one writer per step, the excess of its head may have several.
// (Predicated stores and an add that is always executed: timings in ard_bits2d.cuh.)
template <int OFF>
__device__ __forceinline__ void st_if3(bool p, unsigned a, int v) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared.u32 [%0+%3], %1;\n}\n" ::"r"(a), "r"(v),
                 "r"((unsigned)p), "n"(OFF)
                 : "memory");
}
template <int TY, int V, int D>
__device__ __forceinline__ void send_arc3(unsigned a, int c, int rc, int dl) {
    constexpr int off = D == 0 ? 1 : D == 1 ? -1 : D == 2 ? 32 : D == 3 ? -32 : D == 4 ? 32 * TY : -32 * TY;
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n @q st.shared.u32 [%0+%4], %1;\n @q st.shared.u32 [%0+%5], %2;\n"
        " red.shared.add.u32 [%0+%6], %3;\n}\n" ::"r"(a),
        "r"(c - dl), "r"(rc + dl), "r"(dl), "n"(4 * D * V), "n"(4 * ((D ^ 1) * V + off)), "n"(4 * (7 * V + off))
        : "memory");
}
template <int TY, int V, int... D>
__device__ __forceinline__ void send_arcs3(unsigned a, const int (&c)[sizeof...(D)], const int (&rc)[sizeof...(D)],
                                           const int (&dl)[sizeof...(D)], std::integer_sequence<int, D...>) {
    (send_arc3<TY, V, D>(a, c[D], rc[D], dl[D]), ...);
}

// One region's discharge, organised as in 2D (ard_bits2d.cuh): the graph
// warp keeps the masks in registers, runs the searches and pushes the layers
// by itself, a lane per row; crowded layers, labels to write and the end of
// the stages are commands to all warps.
// Bound by one region's chain of dependent steps (11-12 rounds of 8 BFS layers
// and 5-6 push layers per discharge).  By all warps, a row per warp with a
// block barrier per layer and the masks rebuilt after a round, a push layer took
// 2100-2400 cycles and a BFS layer 320-350, now 1000 and 95.  Discharge time of a
// solve: 382 -> 178 ms (512x512x384), 12.4 -> 6.5 ms (128^3), 6.1 -> 3.2 ms
// (61x75x53); of that the search of the next stage in a bit set of the halo labels
// instead of a pass per stage 181 -> 178, 6.7 -> 6.5 and 3.4 -> 3.2 ms.  128 threads
// per 32x8x4 region in single solves (the graph warp without register spills:
// 210 -> 203 ms on 512x512x384), 256 in batches (62 against 65 ms for the batch of
// 48 2D and 16 3D grids, with 46 bytes spilled at 64 registers).  32x8x8 does not
// spill either; 32x16x8 spills 202 bytes at its 128 registers, 32x4x4 and 32x8x2 94
// at 64 (eight blocks per SM).
template <int TY, int TZ, int NT, int MB>
__device__ __forceinline__ void discharge3d_region(const Geom &g, const DevState &st, const SweepArgs &sa,
                                                   const int r, unsigned long long *mbar, unsigned &mphase) {
    using C = Cfg3D<TY, TZ, NT, MB>;
    constexpr int TX = 32, N = 6, V = C::V, NR = C::NR, RPL = C::RPL, NW = C::NW, LCAP = C::LCAP, LZ = C::LZ;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smraw[];
    // (16 bytes of padding first: the reverse arc of the first cell's -x arc is read unconditionally)
    int *s_cap = (int *)(smraw + 16);       // [N][V] residual of arc i -> i + D(d)
    int *s_tcap = s_cap + N * V;            // [V]
    int *s_exc = s_tcap + V;                // [V]
    int *s_lab = s_exc + V;                 // [V] region label (deep BFS layers: negative tags)
    u32 *s_R = (u32 *)(s_lab + V);          // [N][NR] residual masks (rows rebuilt from the planes)
    u32 *s_T = s_R + N * NR;                // [NR]
    u32 *s_E = s_T + NR;                    // [NR]
    u32 *s_inc = s_E + NR;                  // [NR] vertices that joined the closure
    u32 *s_vis = s_inc + NR;                // [NR] final closure (during Augment rounds: excess received)
    u32 *s_layer = s_vis + NR;              // [LCAP+1][NR]
    int *s_hl = (int *)(s_layer + (LCAP + 1) * NR);  // [HL] labels of B^R
    // [NR] rows whose planes changed (2: by the current command's pushes)
    unsigned char *s_dirty = (unsigned char *)(s_hl + C::HL);
    __shared__ int s_ctl[5];                // command, its argument, epoch, any augmentation, stage
    __shared__ unsigned long long s_flow;
    enum { kDone = 0, kLabel = 1, kPush = 2 };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // does this lane of the graph warp hold tile rows (all do unless the tile has 16 rows)
    const bool lrow = !C::PART || lane < NR;
    DIAG_DECL
    const long long diag_t0 = clock64();
    (void)diag_t0;
    const int rx = r % g.RX, ry = (r / g.RX) % g.RY, rz = r / (g.RX * g.RY);
    const int ox = rx * TX, oy = ry * TY, oz = rz * TZ;
    const size_t n = (size_t)g.n;
    const int dinf = g.dinf;
    if (tid == 0) s_flow = 0;

    // voxel index i = rho * TX + x, rho = z * TY + y; plane and row offset of each arc
    auto arc_off = [](int d) -> int {
        return d == 0 ? 1 : d == 1 ? -1 : d == 2 ? TX : d == 3 ? -TX : d == 4 ? TX * TY : -TX * TY;
    };
    auto row_off = [](int d) -> int { return d < 2 ? 0 : d == 2 ? 1 : d == 3 ? -1 : d == 4 ? TY : -TY; };
    // does arc d from row rho stay in the tile along y / z (x handled by the word shifts)
    auto row_has = [](int d, int rho) -> bool {
        const int y = rho % TY, z = rho / TY;
        return d == 2 ? y < TY - 1 : d == 3 ? y > 0 : d == 4 ? z < TZ - 1 : d == 5 ? z > 0 : true;
    };
    // masks of tile row rho from the planes (one warp)
    auto rebuild_row = [&](int rho) {
        const int i = rho * TX + lane;
        unsigned b[N];
#pragma unroll
        for (int d = 0; d < N; ++d) b[d] = __ballot_sync(FULL, s_cap[d * V + i] > 0);
        const unsigned bt = __ballot_sync(FULL, s_tcap[i] > 0), be = __ballot_sync(FULL, s_exc[i] > 0);
        if (lane == 0) {
#pragma unroll
            for (int d = 0; d < N; ++d) s_R[d * NR + rho] = b[d];
            s_T[rho] = bt;
            s_E[rho] = be;
        }
    };

    // ---- stage the tile --------------------------------------------------------
    const bool full = ox + TX <= g.X && oy + TY <= g.Y && oz + TZ <= g.Z;
    // bulk copies need every row on a 16-byte boundary; planes in host memory
    // are read with plain loads
    const bool vec = full && (g.X % 4) == 0 && !st.host;
    if (vec) {
        // one bulk copy per row of every plane (cap[N], tcap, exc are adjacent in
        // shared memory) against the block's transaction barrier, spread over
        // all threads; the labels start at 0 and the halo is gathered meanwhile
        fence_proxy_async_smem();
        if (tid == 0) mbar_arrive_expect_tx(mbar, (unsigned)((N + 2) * V * 4));
        __syncthreads();  // earlier accesses of the planes and the byte count precede the copies
        for (int c = tid; c < (N + 2) * NR; c += NT) {
            const int p = c / NR, rho = c % NR;
            const int *plane = p < N ? st.cap + (size_t)p * n : p == N ? st.tcap : st.exc;
            const size_t v0 = ((size_t)(oz + rho / TY) * g.Y + (oy + rho % TY)) * g.X + ox;
            bulk_g2s(s_cap + p * V + rho * TX, plane + v0, TX * 4, mbar);
        }
        for (int i4 = tid; i4 < V / 4; i4 += NT) *(int4 *)&s_lab[i4 * 4] = make_int4(0, 0, 0, 0);
    } else {
        for (int i = tid; i < V; i += NT) {
            const int lx = i % TX, rho = i / TX;
            const int x = ox + lx, y = oy + rho % TY, z = oz + rho / TY;
            const bool in = x < g.X && y < g.Y && z < g.Z;
            const size_t v = ((size_t)z * g.Y + y) * g.X + x;
#pragma unroll
            for (int d = 0; d < N; ++d) s_cap[d * V + i] = in ? st.cap[d * n + v] : 0;
            s_tcap[i] = in ? st.tcap[v] : 0;
            s_exc[i] = in ? st.exc[v] : 0;
            s_lab[i] = 0;
        }
    }
    for (int rho = tid; rho < NR; rho += NT) s_dirty[rho] = 0;
    for (int h = tid; h < C::HL; h += NT) {
        int lx, ly, lz, d;
        halo3_src<TY, TZ>(h, lx, ly, lz, d);
        const int x = ox + lx + arc_dx(6, d), y = oy + ly + arc_dy(6, d), z = oz + lz + arc_dz(6, d);
        const bool ing = x >= 0 && x < g.X && y >= 0 && y < g.Y && z >= 0 && z < g.Z;
        s_hl[h] = ing ? st.lab[((size_t)z * g.Y + y) * g.X + x] : dinf;
    }
    if (vec) {
        bool landed = mbar_wait(mbar, mphase);
        if (!landed) landed = mbar_wait(mbar, mphase);  // once more (bounded) before giving up
        mphase ^= 1u;
        if (__syncthreads_or(!landed)) {  // never expected: report and leave the region untouched
            if (tid == 0) {
                region_not_staged(st, r);
                atomicExch(&st.ctr[kError], 2);
            }
            return;
        }
    }
    __syncthreads();
    for (int rho = warp; rho < NR; rho += NW) rebuild_row(rho);
    __syncthreads();
    DIAG_LAP(0);

    // ---- the graph warp's state and searches -----------------------------------
    // (Rm holds no arcs that leave the tile in y or z; those that leave it in x
    // meet no bit in a shifted word)
    u32 Rm[N][RPL], T[RPL], E[RPL], Cl[RPL], sdB[RPL];
    u32 recv[RPL];  // vertices that received excess in this round's push
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        const int rho = lane * RPL + j;
#pragma unroll
        for (int d = 0; d < N; ++d) Rm[d][j] = warp == 0 && lrow && row_has(d, rho) ? s_R[d * NR + rho] : 0;
        T[j] = warp == 0 && lrow ? s_T[rho] : 0;
        E[j] = warp == 0 && lrow ? s_E[rho] : 0;
        Cl[j] = sdB[j] = recv[j] = 0;
    }
    bool pushed[RPL] = {};  // rows that pushed
    // the halo labels below d_inf as bits above the least of them: the next stage
    // is a bit search, not a pass over 832 cells (12 passes per discharge)
    int hlo = INT_MAX;
    unsigned long long hbits = 0;
    bool hmore = false;  // labels past the 64 bits
    if (warp == 0) {
        for (int h = lane; h < C::HL; h += 32) hlo = min(hlo, s_hl[h] < dinf ? s_hl[h] : INT_MAX);
        hlo = __reduce_min_sync(FULL, hlo);
        for (int h = lane; h < C::HL; h += 32) {
            const int v = s_hl[h], q = v - hlo;
            if (v < dinf) {
                if (q < 64) hbits |= 1ull << q;
                else hmore = true;
            }
        }
        hbits = __reduce_or_sync(FULL, (unsigned)hbits) | (unsigned long long)__reduce_or_sync(FULL, (unsigned)(hbits >> 32)) << 32;
        hmore = __any_sync(FULL, hmore);
    }
    // next stage value above k: min{d(w)+1 > k : w in B^R, d(w) < d_inf}
    auto next_stage = [&](int k) -> int {
        const int q = max(k - hlo, 0);
        if (q < 64 && (hbits >> q)) return hlo + q + __ffsll((long long)(hbits >> q));
        if (!hmore) return INT_MAX;
        int best = INT_MAX;
        for (int h = lane; h < C::HL; h += 32) {
            const int v = s_hl[h];
            if (v < dinf && v + 1 > k && v + 1 < best) best = v + 1;
        }
        return __reduce_min_sync(FULL, best);
    };
    // boundary part of the seed rows of T_k: a residual arc to a halo cell w with
    // d(w) < k.  The masks of arcs that leave the tile stay in s_R (push_out
    // keeps them up to date).
    auto seed_boundary = [&](int k) {
        u32 my[RPL], py[RPL], mz[RPL], pz[RPL];
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const int rho = lane * RPL + j;
            u32 s = 0u;
            my[j] = py[j] = mz[j] = pz[j] = 0u;
            if (lrow) {
                if (s_hl[C::B_MX + rho] < k) s |= s_R[1 * NR + rho] & 1u;
                if (s_hl[C::B_PX + rho] < k) s |= s_R[rho] & (1u << (TX - 1));
                py[j] = row_has(2, rho) ? 0u : s_R[2 * NR + rho];
                my[j] = row_has(3, rho) ? 0u : s_R[3 * NR + rho];
                pz[j] = row_has(4, rho) ? 0u : s_R[4 * NR + rho];
                mz[j] = row_has(5, rho) ? 0u : s_R[5 * NR + rho];
            }
            sdB[j] = s;
        }
#pragma unroll
        for (int z = 0; z < TZ; ++z) {
            const u32 bm = __ballot_sync(FULL, s_hl[C::B_MY + z * TX + lane] < k);
            const u32 bp = __ballot_sync(FULL, s_hl[C::B_PY + z * TX + lane] < k);
#pragma unroll
            for (int j = 0; j < RPL; ++j)
                if ((lane * RPL + j) / TY == z) sdB[j] |= (bm & my[j]) | (bp & py[j]);
        }
#pragma unroll
        for (int y = 0; y < TY; ++y) {
            const u32 bm = __ballot_sync(FULL, s_hl[C::B_MZ + y * TX + lane] < k);
            const u32 bp = __ballot_sync(FULL, s_hl[C::B_PZ + y * TX + lane] < k);
#pragma unroll
            for (int j = 0; j < RPL; ++j)
                if ((lane * RPL + j) % TY == y) sdB[j] |= (bm & mz[j]) | (bp & pz[j]);
        }
    };
    // the words of the rows one step along each arc direction (2..5) from the
    // lane's rows; wrong where the row lies outside the tile (masked by row_has)
    struct Beside { u32 yp[RPL], ym[RPL], zp[RPL], zm[RPL]; };
    auto beside = [&](const u32 (&f)[RPL]) -> Beside {
        Beside o;
        const u32 up = __shfl_up_sync(FULL, f[RPL - 1], 1);
        const u32 dn = __shfl_down_sync(FULL, f[0], 1);
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            o.zm[j] = __shfl_up_sync(FULL, f[j], LZ);
            o.zp[j] = __shfl_down_sync(FULL, f[j], LZ);
            o.ym[j] = j == 0 ? up : f[j > 0 ? j - 1 : 0];
            o.yp[j] = j == RPL - 1 ? dn : f[j + 1 < RPL ? j + 1 : j];
        }
        return o;
    };
    // one backward BFS step: vertices with a residual arc into f
    auto expand = [&](const u32 (&f)[RPL], u32 (&out)[RPL]) {
        const Beside o = beside(f);
#pragma unroll
        for (int j = 0; j < RPL; ++j)
            out[j] = (Rm[0][j] & (f[j] >> 1)) | (Rm[1][j] & (f[j] << 1)) | (Rm[2][j] & o.yp[j]) | (Rm[3][j] & o.ym[j]) |
                     (Rm[4][j] & o.zp[j]) | (Rm[5][j] & o.zm[j]);
    };
    // words sent along the arcs 2..5 by each row, received by the rows they lead
    // to: f(d, j) is what the lane's row j sends along arc d, take(d, j, m) gets
    // what arrives at row j along arc d
    auto along = [&](auto &&f, auto &&take) {
        const u32 yp = __shfl_up_sync(FULL, f(2, RPL - 1), 1);   // row - 1 sends to this lane's first row
        const u32 ym = __shfl_down_sync(FULL, f(3, 0), 1);       // row + 1 sends to its last row
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const int rho = lane * RPL + j;
            const u32 zp = __shfl_up_sync(FULL, f(4, j), LZ), zm = __shfl_down_sync(FULL, f(5, j), LZ);
            take(2, j, row_has(3, rho) ? (j == 0 ? yp : f(2, j > 0 ? j - 1 : 0)) : 0u);
            take(3, j, row_has(2, rho) ? (j == RPL - 1 ? ym : f(3, j + 1 < RPL ? j + 1 : j)) : 0u);
            take(4, j, row_has(5, rho) ? zp : 0u);
            take(5, j, row_has(4, rho) ? zm : 0u);
        }
    };
    auto flood = [&]() {
        u32 fr[RPL], inc[RPL];
        bool any = false;
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const u32 f = row_fill32((T[j] | sdB[j]) & ~Cl[j], Rm[0][j] & ~Cl[j], Rm[1][j] & ~Cl[j]);
            Cl[j] |= f;
            inc[j] = f;
            fr[j] = f;
            any |= f != 0u;
        }
        while (__any_sync(FULL, any)) {
            u32 nf[RPL];
            expand(fr, nf);
            any = false;
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const u32 f = row_fill32(nf[j] & ~Cl[j], Rm[0][j] & ~Cl[j], Rm[1][j] & ~Cl[j]);
                Cl[j] |= f;
                inc[j] |= f;
                fr[j] = f;
                any |= f != 0u;
            }
        }
        if (lrow) {
#pragma unroll
            for (int j = 0; j < RPL; ++j) s_inc[lane * RPL + j] = inc[j];
        }
    };
    auto write_labels = [&](int k) {
        for (int rho = warp; rho < NR; rho += NW)
            if ((s_inc[rho] >> lane) & 1u) s_lab[rho * TX + lane] = k;
    };

    long long flow_acc = 0;
    // what the vertex at column x of row rho with excess e, in layer 1, sends
    // into B^R; returns the rest.  seed: has it still a residual arc into T_k's
    // boundary vertices
    auto push_out = [&](int x, int rho, int e, int k, bool &seed) -> int {
        const int ly = rho % TY, lz = rho / TY, i = rho * TX + x;
        seed = false;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const bool in = d == 0 ? x < TX - 1 : d == 1 ? x > 0 : row_has(d, rho);
            if (in) continue;
            const int c = s_cap[d * V + i], h = halo3<TY, TZ>(d, x, ly, lz);
            if (c > 0 && s_hl[h] < k) {
                const int b = min(e, c);
                s_cap[d * V + i] = c - b;
                e -= b;
                if (b == c) atomicAnd(&s_R[d * NR + rho], ~(1u << x));
                else seed = true;
            }
        }
        return e;
    };
    // The vertices of BFS layer L in row rho that have excess (bit `act` of this
    // lane) push it one layer down, to T_k from layer 1.  Returns the vertices
    // that pushed along each arc; bpush tells of pushes into B^R.
    struct PushOut { u32 to[N]; bool bpush; };
    auto push_row = [&](int rho, bool act, int L, int k, int epoch, u32 sd, PushOut &o) {
        const int x = lane, i = rho * TX + x;
        o.bpush = false;
        if (L == 1) {
            int e = act ? s_exc[i] : 0;
            const int tc = act ? s_tcap[i] : 0;
            const int dl = min(e, tc);
            if (dl > 0) {
                s_tcap[i] = tc - dl;
                e -= dl;
                flow_acc += dl;
            }
            o.bpush = (__ballot_sync(FULL, e > 0) & sd) != 0;
            bool seed;
            if (o.bpush && e > 0) e = push_out(x, rho, e, k, seed);
            if (act) s_exc[i] = e;
#pragma unroll
            for (int d = 0; d < N; ++d) o.to[d] = 0;
            return;
        }
        bool adm[N];
        if (L - 1 <= LCAP) {
            const u32 *lay = s_layer + (L - 1) * NR;
            const u32 bit = 1u << x, l0 = lay[rho];
            adm[0] = (l0 & (bit << 1)) != 0;
            adm[1] = (l0 & (bit >> 1)) != 0;
#pragma unroll
            for (int d = 2; d < N; ++d) adm[d] = row_has(d, rho) && (lay[rho + row_off(d)] & bit);
        } else {
            const int tg = deep_tag3(epoch, L - 1);
#pragma unroll
            for (int d = 0; d < N; ++d) {
                const bool in = d == 0 ? x < TX - 1 : d == 1 ? x > 0 : row_has(d, rho);
                adm[d] = in && s_lab[i + arc_off(d)] == tg;
            }
        }
        int e = act ? s_exc[i] : 0;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const int c = s_cap[d * V + i];
            const int dl = adm[d] ? min(e, c) : 0;
            e -= dl;
            if (dl > 0) {
                s_cap[d * V + i] = c - dl;
                s_cap[(d ^ 1) * V + i + arc_off(d)] += dl;
                atomicAdd(&s_exc[i + arc_off(d)], dl);
            }
            o.to[d] = __ballot_sync(FULL, dl > 0);
        }
        if (act) s_exc[i] = e;
    };

    const int klimit = sa.partial ? (sa.sweep_dev ? *sa.sweep_dev : sa.sweep) : INT_MAX;
    int rounds = 0, stages = 0, epoch = 0;
    bool err = false, any_aug = false;
    bool cl_valid = true;  // Cl is the closure of T_k on the current graph (empty at start)

    // ---- ARD stages: the graph warp decides, all warps execute its commands ------
    enum { kFlood, kRound, kNext };
    int phase = kFlood, k = 0, kn = 0, round = 0, resume = 0;
    for (;;) {
        if (warp == 0) {
            int cmd = kDone, arg = 0;
            for (;;) {
                if (phase == kFlood) {
                    DIAG_MARK();
                    DIAG_ADD(2, 1);
                    if (!cl_valid) {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) Cl[j] = 0;
                        cl_valid = true;
                    }
                    seed_boundary(k);
                    flood();
                    bool m = false;
#pragma unroll
                    for (int j = 0; j < RPL; ++j) m |= (Cl[j] & E[j]) != 0;
                    const bool reach = __any_sync(FULL, m);
                    kn = next_stage(k);
                    const bool aug = k <= klimit && !err;
                    if (aug) ++stages;
                    DIAG_LAP(1);
                    if (aug && reach) {
                        phase = kRound;
                        round = 0;
                        any_aug = true;
                    } else {
                        phase = kNext;
                        if (!any_aug) {  // labels stay exact until the first augmentation
                            cmd = kLabel;
                            arg = k;
                            break;
                        }
                    }
                    continue;
                }
                if (phase == kNext) {
                    // nothing left to learn: labels are recomputed at the end anyway
                    if (kn == INT_MAX || (any_aug && (kn > klimit || err))) break;
                    k = kn;
                    phase = kFlood;
                    continue;
                }
                // a round of Augment(R, T_k): exact BFS + layered push
                if (resume == 0 && round >= sa.max_rounds) {
                    err = true;
                    cl_valid = false;
                    phase = kNext;
                    continue;
                }
                int L = resume;  // > 0: the block has pushed the layers above
                resume = 0;
                if (L == 0) {
                    if (++epoch >= 32767) {  // deep-layer tags wrap: clear them
                        for (int i = lane; i < V; i += 32) s_lab[i] = 0;
                        __syncwarp();
                        epoch = 1;
                    }
                    DIAG_MARK();
                    DIAG_ADD(5, 1);
                    int lmax = 0;
                    u32 vis[RPL], fr[RPL], want[RPL];
                    bool pending = false;
#pragma unroll
                    for (int j = 0; j < RPL; ++j) {
                        const u32 ex = E[j] & Cl[j];  // excess that can reach T_k lies in the closure
                        recv[j] = 0;
                        vis[j] = fr[j] = T[j] | sdB[j];
                        if (lrow) s_layer[1 * NR + lane * RPL + j] = fr[j];
                        if (fr[j] & ex) lmax = 1;
                        want[j] = ex & ~vis[j];
                        pending |= want[j] != 0u;
                    }
                    L = 1;
                    bool go = __any_sync(FULL, pending);
                    // two layers per vote: a layer too many is an empty or unused mask
                    while (go && L + 2 <= LCAP) {
                        bool any = false;
                        pending = false;
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            u32 nf[RPL];
                            expand(fr, nf);
                            ++L;
#pragma unroll
                            for (int j = 0; j < RPL; ++j) {
                                nf[j] &= ~vis[j];
                                vis[j] |= nf[j];
                                fr[j] = nf[j];
                                if (lrow) s_layer[L * NR + lane * RPL + j] = nf[j];
                                if (nf[j] & want[j]) lmax = L;
                                want[j] &= ~nf[j];
                            }
                        }
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            any |= fr[j] != 0u;
                            pending |= want[j] != 0u;
                        }
                        const bool a = __any_sync(FULL, any), b = __any_sync(FULL, pending);
                        go = a && b;
                    }
                    while (go) {  // layers past the masks: label tags
                        u32 nf[RPL];
                        expand(fr, nf);
                        ++L;
                        bool any = false;
                        pending = false;
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            const int rho = lane * RPL + j;
                            nf[j] &= ~vis[j];
                            any |= nf[j] != 0u;
                            vis[j] |= nf[j];
                            fr[j] = nf[j];
                            if (L <= LCAP) {
                                if (lrow) s_layer[L * NR + rho] = nf[j];
                            } else {
                                const int tg = deep_tag3(epoch, L);
                                for (u32 m = nf[j]; m; m &= m - 1) s_lab[rho * TX + __ffs((int)m) - 1] = tg;
                            }
                            if (nf[j] & want[j]) lmax = L;
                            want[j] &= ~nf[j];
                            pending |= want[j] != 0u;
                        }
                        const bool a = __any_sync(FULL, any), b = __any_sync(FULL, pending);
                        go = a && b;
                    }
                    DIAG_ADD(6, L);
                    lmax = __reduce_max_sync(FULL, lmax);
                    __syncwarp();
                    DIAG_LAP(4);
                    if (lmax == 0) {  // no excess vertex reaches T_k: stage done
                        cl_valid = false;
                        phase = kNext;
                        continue;
                    }
                    ++rounds;
                    ++round;
                    DIAG_ADD(8, lmax);
                    L = lmax;
                }
                // layered push, top layer first: layer L pushes only to layer L-1
                // (to T_k from layer 1), so every arc has one writer per step.
                // Only vertices that had excess when the round began or received
                // some in an earlier step of it can push.  A lane takes the
                // vertices of its own rows one after another.
                DIAG_MARK();
                u32 to[N][RPL];  // vertices that pushed along arc d in this round
#pragma unroll
                for (int j = 0; j < RPL; ++j)
#pragma unroll
                    for (int d = 0; d < N; ++d) to[d][j] = 0;
                if (L <= LCAP) {  // (layers without masks are left to the block)
                    // the lane's words of layers L, L - 1 and L - 2 (loaded a step ahead;
                    // layer 0 is unused space), and the rows beside of layer L - 1
                    u32 lw[RPL], lo[RPL], ln[RPL];
                    auto layer_word = [&](int l, int j) -> u32 { return lrow ? s_layer[l * NR + lane * RPL + j] : 0u; };
#pragma unroll
                    for (int j = 0; j < RPL; ++j) {
                        lw[j] = layer_word(L, j);
                        lo[j] = layer_word(L - 1, j);
                    }
                    Beside bo = beside(lo);
                    bool heavy = false;
                    for (; L > 1; --L) {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) ln[j] = layer_word(L - 2, j);
                        const Beside bn = beside(ln);
                        u32 P[RPL];
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            P[j] = lw[j] & (E[j] | recv[j]);
                            pushed[j] |= P[j] != 0u;
                        }
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            const int rho = lane * RPL + j;
                            u32 src[N];  // bit x: the head of arc d from column x lies in layer L - 1
                            src[0] = lo[j] >> 1;
                            src[1] = lo[j] << 1;
                            src[2] = row_has(2, rho) ? bo.yp[j] : 0u;
                            src[3] = row_has(3, rho) ? bo.ym[j] : 0u;
                            src[4] = row_has(4, rho) ? bo.zp[j] : 0u;
                            src[5] = row_has(5, rho) ? bo.zm[j] : 0u;
                            int x = top_bit3(P[j], lane);
                            // no branches inside: lanes without a vertex run along with
                            // amounts of 0, in a column of their own (no bank conflicts)
                            for (int it = 0;; ++it) {
                                const u32 bit = (1u << x) & P[j];
                                const int i = rho * TX + x;
                                int c[N], rc[N], dl[N];
#pragma unroll
                                for (int d = 0; d < N; ++d) {
                                    c[d] = s_cap[d * V + i];
                                    rc[d] = s_cap[(d ^ 1) * V + i + arc_off(d)];
                                }
                                int e = s_exc[i];
                                P[j] ^= bit;
                                x = top_bit3(P[j], lane);
                                const bool again = __any_sync(FULL, P[j] != 0u);
#pragma unroll
                                for (int d = 0; d < N; ++d) {
                                    dl[d] = (src[d] & bit) ? min(e, c[d]) : 0;
                                    e -= dl[d];
                                }
                                send_arcs3<TY, V>(smem_u32(s_cap + i), c, rc, dl, std::make_integer_sequence<int, N>());
#pragma unroll
                                for (int d = 0; d < N; ++d) {  // (an arc with c = 0 has no bit in Rm)
                                    if (dl[d] != 0) to[d][j] |= bit;
                                    if (dl[d] == c[d]) Rm[d][j] &= ~bit;
                                }
                                st_if3<4 * (N + 1) * V>(bit != 0u, smem_u32(s_cap + i), e);
                                E[j] = (E[j] & ~bit) | (e > 0 ? bit : 0u);
                                if (!again) break;
                                if (it == C::HEAVY) {  // the rest of a crowded layer is left to the block
                                    heavy = true;
                                    break;
                                }
                            }
                        }
                        // who received (marks of earlier layers are sent again: harmless)
#pragma unroll
                        for (int j = 0; j < RPL; ++j) recv[j] |= (to[0][j] << 1) | (to[1][j] >> 1);
                        along([&](int d, int j) { return to[d][j]; }, [&](int, int j, u32 m) { recv[j] |= m; });
                        __syncwarp();
                        if (heavy) {  // layer L shrinks to the vertices that have not pushed
#pragma unroll
                            for (int j = 0; j < RPL; ++j)
                                if (lrow) s_layer[L * NR + lane * RPL + j] = P[j];
                            break;
                        }
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            lw[j] = lo[j];
                            lo[j] = ln[j];
                        }
                        bo = bn;
                    }
                    if (!heavy) {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            const int rho = lane * RPL + j;
                            u32 P = lw[j] & (E[j] | recv[j]);
                            pushed[j] |= P != 0u;
                            int x = top_bit3(P, lane);
                            for (bool again = true; again;) {
                                const u32 bit = (1u << x) & P;
                                const int xv = x, i = rho * TX + x;
                                int e = bit ? s_exc[i] : 0;
                                const int tc = s_tcap[i];
                                P ^= bit;
                                x = top_bit3(P, lane);
                                again = __any_sync(FULL, P != 0u);
                                const int dl = min(e, tc);
                                e -= dl;
                                flow_acc += dl;
                                const bool out = e > 0 && (sdB[j] & bit);
                                if (__any_sync(FULL, out)) {
                                    if (out) {
                                        bool seed;
                                        e = push_out(xv, rho, e, k, seed);
                                        if (!seed) sdB[j] &= ~bit;
                                    }
                                }
                                st_if3<4 * N * V>(bit != 0u, smem_u32(s_cap + i), tc - dl);
                                st_if3<4 * (N + 1) * V>(bit != 0u, smem_u32(s_cap + i), e);
                                T[j] &= dl == tc ? ~bit : ~0u;
                                E[j] = (E[j] & ~bit) | (e > 0 ? bit : 0u);
                            }
                        }
                        __syncwarp();
                        L = 0;
                    }
                }
                // the reverse arcs of the pushes are residual now
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    Rm[1][j] |= to[0][j] << 1;
                    Rm[0][j] |= to[1][j] >> 1;
                }
                along([&](int d, int j) { return to[d][j]; }, [&](int d, int j, u32 m) { Rm[d ^ 1][j] |= m; });
                DIAG_LAP(7);
                if (L >= 1) {
                    cmd = kPush;
                    arg = L;
                    break;
                }
            }
            if (cmd == kPush) {
#pragma unroll
                for (int j = 0; j < RPL; ++j)
                    if (lrow) {
                        s_E[lane * RPL + j] = E[j];
                        s_vis[lane * RPL + j] = recv[j];
                        s_inc[lane * RPL + j] = sdB[j];
                    }
            }
            if (lane == 0) {
                s_ctl[0] = cmd;
                s_ctl[1] = arg;
                s_ctl[2] = epoch;
                s_ctl[3] = any_aug;
                s_ctl[4] = k;
            }
        }
        __syncthreads();
        const int cmd = s_ctl[0], arg = s_ctl[1];
        if (cmd == kDone) break;
        if (cmd == kLabel) {
            write_labels(arg);
            __syncthreads();
            continue;
        }
        DIAG_MARK();
        // the push layers from arg down by all warps: warp w takes the busy
        // rows w, w + NW, .. of each layer, while a layer is crowded
        const int ep = s_ctl[2], kk = s_ctl[4];
        u32 *s_recv = s_vis;
        int L = arg;
        for (; L >= 1; --L) {
            u32 mine[RPL];
            bool many = false;
            int rank0 = 0;
#pragma unroll
            for (int q = 0; q < RPL; ++q) {
                const int rho = lane + 32 * q;
                u32 P = 0;
                // (deep layers: every row, as marks of the step itself would show in the word)
                if (rho < NR) P = L <= LCAP ? s_layer[L * NR + rho] & (s_E[rho] | s_recv[rho]) : FULL;
                many |= __popc(P) > C::HEAVY / 2;
                const unsigned busy = __ballot_sync(FULL, P != 0u);
                const int rank = rank0 + __popc(busy & ((1u << lane) - 1u));
                mine[q] = __ballot_sync(FULL, P != 0u && rank % NW == warp);
                rank0 += __popc(busy);
            }
            if (!__any_sync(FULL, many)) break;  // (the same in every warp) back to the graph warp
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                for (u32 mm = mine[q]; mm; mm &= mm - 1) {
                    const int rho = 32 * q + __ffs((int)mm) - 1;
                    const u32 P = (L <= LCAP ? s_layer[L * NR + rho] : FULL) & (s_E[rho] | s_recv[rho]);
                    bool act = (P >> lane) & 1u;
                    if (L > LCAP) act = act && s_lab[rho * TX + lane] == deep_tag3(ep, L);
                    if (!__any_sync(FULL, act)) continue;
                    PushOut o;
                    push_row(rho, act, L, kk, ep, s_inc[rho], o);
                    if (lane < 5) {  // the row itself and the rows beside
                        const int d = lane == 0 ? 0 : lane + 1;
                        const u32 v = lane == 0 ? (o.to[0] << 1) | (o.to[1] >> 1) : lane == 1 ? o.to[2] : lane == 2 ? o.to[3]
                                                                                  : lane == 3 ? o.to[4] : o.to[5];
                        if (v) atomicOr(&s_recv[rho + row_off(d)], v);
                        if (v || lane == 0) s_dirty[rho + row_off(d)] = 2;
                    }
                }
            __syncthreads();
        }
        for (int rho = warp; rho < NR; rho += NW)
            if (s_dirty[rho] == 2) rebuild_row(rho);
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const int rho = lane * RPL + j;
                if (lrow && s_dirty[rho] == 2) {
#pragma unroll
                    for (int d = 0; d < N; ++d) Rm[d][j] = row_has(d, rho) ? s_R[d * NR + rho] : 0u;
                    T[j] = s_T[rho];
                    E[j] = s_E[rho];
                    s_dirty[rho] = 1;
                }
                recv[j] = lrow ? s_recv[rho] : 0u;
            }
            __syncwarp();
            seed_boundary(k);
            resume = L;
        }
        DIAG_LAP(13);
    }

    // ---- region-relabel after augmentation: d(u) = min{k : u -> T_k} -------------
    if (s_ctl[3]) {
        DIAG_MARK();
        __syncthreads();  // the last command has been read
        if (warp == 0) {
#pragma unroll
            for (int j = 0; j < RPL; ++j) Cl[j] = 0;
        }
        for (int k2 = 0;;) {
            if (warp == 0) {
                seed_boundary(k2);
                flood();
                const int n2 = next_stage(k2);
                if (lane == 0) s_ctl[0] = n2;
            }
            __syncthreads();
            write_labels(k2);
            const int n2 = s_ctl[0];
            __syncthreads();
            if (n2 == INT_MAX) break;
            k2 = n2;
        }
        DIAG_LAP(9);
    }
    if (warp == 0 && lrow) {
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const int rho = lane * RPL + j;
            s_vis[rho] = Cl[j];
            if (pushed[j]) {  // rows to write back: those that pushed and the rows beside
                s_dirty[rho] = 1;
#pragma unroll
                for (int d = 2; d < N; ++d)
                    if (row_has(d, rho)) s_dirty[rho + row_off(d)] = 1;
            }
        }
    }
    __syncthreads();
    DIAG_MARK();

    // ---- write back: planes of rows that changed; labels and boundary flows always
    int left = 0;
    for (int i = tid; i < V; i += NT) {
        const int lx = i % TX, rho = i / TX, ly = rho % TY, lz = rho / TY;
        const int x = ox + lx, y = oy + ly, z = oz + lz;
        if (!(x < g.X && y < g.Y && z < g.Z)) continue;
        const size_t v = ((size_t)z * g.Y + y) * g.X + x;
        const bool dirty = s_dirty[rho] != 0;
        bool perim = false;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const int nx = lx + arc_dx(6, d), ny = ly + arc_dy(6, d), nz = lz + arc_dz(6, d);
            const int gx = x + arc_dx(6, d), gy = y + arc_dy(6, d), gz = z + arc_dz(6, d);
            const bool intile = nx >= 0 && nx < TX && ny >= 0 && ny < TY && nz >= 0 && nz < TZ;
            const bool ing = gx >= 0 && gx < g.X && gy >= 0 && gy < g.Y && gz >= 0 && gz < g.Z;
            if (intile) {
                if (dirty) st.cap[d * n + v] = s_cap[d * V + i];
            } else if (ing) {
                perim = true;
                if (dirty) {
                    const int c = s_cap[d * V + i];
                    st.bout[d * n + v] = st.cap[d * n + v] - c;  // flow pushed across the boundary
                    st.cap[d * n + v] = c;
                } else {
                    st.bout[d * n + v] = 0;
                }
            }
        }
        if (dirty) {
            st.tcap[v] = s_tcap[i];
            st.exc[v] = s_exc[i];
        }
        const int lab = ((s_vis[rho] >> lx) & 1u) ? s_lab[i] : dinf;
        if (perim) st.lab_next[v] = lab;
        else st.lab[v] = lab;
        if (s_exc[i] > 0 && lab < dinf) left = 1;
    }
    left = __syncthreads_or(left);
    unsigned long long f = (unsigned long long)flow_acc;
    for (int o = 16; o > 0; o >>= 1) f += __shfl_down_sync(FULL, f, o);
    if (lane == 0 && f) atomicAdd(&s_flow, f);
    __syncthreads();
    if (tid == 0) {
        DIAG_LAP(10);
        DIAG_ADD(11, clock64() - diag_t0);
        DIAG_ADD(12, 1);
        DIAG_ADD(14, rounds);
        DIAG_FLUSH();
        if (s_flow) atomicAdd(st.flow_t, s_flow);
        st.disc[r] = 1;
        st.left_active[r] = (unsigned char)left;
        if (err) atomicExch(&st.ctr[kError], 1);
        atomicAdd(&sa.c64->stages, (unsigned long long)stages);
        atomicAdd(&sa.c64->rounds, (unsigned long long)rounds);
        atomicAdd(&sa.c64->discharges, 1ull);
        const unsigned long long live =
            (unsigned long long)min(TX, g.X - ox) * min(TY, g.Y - oy) * min(TZ, g.Z - oz);
        atomicAdd(&sa.c64->discharged_vertices, live);
    }
}

template <int TY, int TZ, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) ard_discharge3d_kernel(const Geom g, const DevState st, const SweepArgs sa) {
    const int r = blockIdx.x;
    if (!region_to_discharge(st, r)) return;
    __shared__ __align__(8) unsigned long long s_mbar;
    if (threadIdx.x == 0) mbar_init(&s_mbar, 1);
    __syncthreads();
    unsigned phase = 0;
    discharge3d_region<TY, TZ, NT, MB>(g, st, sa, r, &s_mbar, phase);
}

template <int TY, int TZ, int NT, int MB>
__global__ void __launch_bounds__(NT, MB)
ard_discharge3d_batch_kernel(const Inst *__restrict__ insts, const int2 *__restrict__ items, const int *count,
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
        discharge3d_region<TY, TZ, NT, MB>(I.g, I.st, a, w.y, &s_mbar, phase);
    }
}

template <int TY, int TZ, int NT, int MB>
static cudaError_t launch3d(const Geom &g, const DevState &st, const SweepArgs &sa, cudaStream_t s) {
    using C = Cfg3D<TY, TZ, NT, MB>;
    auto k = ard_discharge3d_kernel<TY, TZ, NT, MB>;
    {
        const cudaError_t e_at = ensure_smem_attr((const void *)k, (int)C::smem);
        if (e_at != cudaSuccess) return e_at;
    }
    k<<<g.nreg, NT, C::smem, s>>>(g, st, sa);
    return cudaGetLastError();
}

template <int TY, int TZ, int NT, int MB>
static cudaError_t launch3d_batch(const Inst *insts, const int2 *items, const int *count, int *head,
                                  const SweepArgs &sa, int blocks, cudaStream_t s) {
    using C = Cfg3D<TY, TZ, NT, MB>;
    auto k = ard_discharge3d_batch_kernel<TY, TZ, NT, MB>;
    {
        const cudaError_t e_at = ensure_smem_attr((const void *)k, (int)C::smem);
        if (e_at != cudaSuccess) return e_at;
    }
    // persistent blocks: at least as many as can be resident
    const int resident = device_sms() * MB;
    k<<<blocks > resident ? blocks : resident, NT, C::smem, s>>>(insts, items, count, head, sa);
    return cudaGetLastError();
}

bool discharge3d_supported(int tx, int ty, int tz) {
    return tx == 32 && ((ty == 16 && tz == 8) || (ty == 8 && tz == 8) || (ty == 8 && tz == 4) || (ty == 4 && tz == 4) ||
                        (ty == 8 && tz == 2));
}

constexpr int kMany3d = 48;  // active regions per SM from which five are resident

cudaError_t launch_discharge3d(const Geom &g, const DevState &st, const SweepArgs &sa, cudaStream_t stream) {
    if (g.tx == 32 && g.ty == 16 && g.tz == 8) return launch3d<16, 8, 512, 1>(g, st, sa, stream);
    if (g.tx == 32 && g.ty == 8 && g.tz == 8) return launch3d<8, 8, 256, 2>(g, st, sa, stream);
    if (g.tx == 32 && g.ty == 8 && g.tz == 4) {
        // Five regions per SM only where many wait for a place: each is slower (95
        // registers a thread instead of 109), the SM does more of them.  Discharge
        // time of a solve with four / five: 128^3 (2048 regions) 6.7 / 7.2 ms, 192^3
        // (6912) 16.2 / 16.4, 256x256x128 (8192) 19.1 / 19.3 and 18.95 with five
        // for the sweeps above the bound, 256^3 (16384) 36.2 / 34.2, 512x512x384
        // (98304) 203 / 181.
        if (sa.active > kMany3d * device_sms()) return launch3d<8, 4, 128, 5>(g, st, sa, stream);
        return launch3d<8, 4, 128, 4>(g, st, sa, stream);
    }
    if (g.tx == 32 && g.ty == 4 && g.tz == 4) return launch3d<4, 4, 128, 8>(g, st, sa, stream);
    if (g.tx == 32 && g.ty == 8 && g.tz == 2) return launch3d<8, 2, 128, 8>(g, st, sa, stream);
    return cudaErrorInvalidValue;
}

cudaError_t launch_discharge3d_batch(int tx, int ty, int tz, const Inst *insts, const int2 *items, const int *count,
                                     int *head, const SweepArgs &sa, int blocks, cudaStream_t stream) {
    if (tx == 32 && ty == 16 && tz == 8) return launch3d_batch<16, 8, 512, 1>(insts, items, count, head, sa, blocks, stream);
    if (tx == 32 && ty == 8 && tz == 8) return launch3d_batch<8, 8, 256, 2>(insts, items, count, head, sa, blocks, stream);
    if (tx == 32 && ty == 8 && tz == 4) return launch3d_batch<8, 4, 256, 4>(insts, items, count, head, sa, blocks, stream);
    if (tx == 32 && ty == 4 && tz == 4) return launch3d_batch<4, 4, 128, 8>(insts, items, count, head, sa, blocks, stream);
    if (tx == 32 && ty == 8 && tz == 2) return launch3d_batch<8, 2, 128, 8>(insts, items, count, head, sa, blocks, stream);
    return cudaErrorInvalidValue;
}

}  // namespace mf
