// Region discharge of P-ARD for 2D tiles with bit-parallel graph search: the
// 4- and 8-connected grids (tiles 64 or 32 wide) and, on 32x32 tiles, the
// stencils of Sec. 7.1 with displacements up to 4.
//
// Same computation as ard_discharge.cu (Procedure ARD of Sec. 4.2 with
// Procedure Augment done in synchronous rounds of "BFS from T_k, then a
// layered push from the highest BFS layer down", and the ARD region-relabel
// of Sec. 5.1), organised for a 64- or 32-wide tile:
//
//   * the residual graph of the tile is also kept as bit masks, one word per
//     tile row (32 or 64 bits): R_d[y] bit x = [c_f((x,y) -> (x,y)+D(d)) > 0],
//     T[y] bit x = [c_f(v,t) > 0], E[y] bit x = [e_f(v) > 0];
//   * warp 0 (the "graph warp") holds these masks in registers, lane l the rows
//     l*RPL .. l*RPL+RPL-1, and runs every BFS and reachability flood on them:
//     a BFS step is a few shifts/ands per row plus two shuffles for the rows
//     above and below; floods also close whole row runs at once (Kogge-Stone
//     fill along the row);
//   * it also runs the layered push, a lane per row, unless a layer has many
//     pushing vertices in one row; those layers are pushed by all warps;
//   * all warps do the staging, the labels and the write-back.
//
// Stage checks ("does an excess vertex reach T_k?") use a reachability closure
// C_k extended stage by stage; its increments are the region labels
// d(u) = min{k : u -> T_k}.  Augmentation invalidates the closure; it is then
// rebuilt for the next check, and the labels are recomputed once at the end.
#pragma once

#include <climits>
#include <cstdint>
#include <utility>

#include "mf_internal.cuh"

namespace mf {

typedef unsigned long long u64;

#ifdef MF_DIAG
static __device__ unsigned long long mf_diag[32];
#endif

template <int TX> struct RowWord { typedef u64 type; };
template <> struct RowWord<32> { typedef unsigned type; };

template <int CONN, int TX, int TY, int NT>
struct Cfg2D {
    typedef typename RowWord<TX>::type W;               // one tile row as a bit mask
    static constexpr bool PAPER = is_paper(CONN);       // a stencil of Sec. 7.1
    static constexpr int R = radius_of(CONN);           // its longest displacement
    static constexpr int N = arcs_of(CONN);
    static constexpr int V = TX * TY;
    static constexpr int NW = NT / 32;                  // warps
    static constexpr bool PART = TY < 32;               // 32x16 tiles: lanes 16..31 of the graph warp hold no row
    static constexpr int RPL = PART ? 1 : TY / 32;      // rows per lane of the graph warp
    static constexpr int HW = TX / 32;                  // 32-bit halves per row
    // halo cells (B^R plus unused corners): a ring, or the padded tile
    static constexpr int HL = PAPER ? (TX + 2 * R) * (TY + 2 * R) : 2 * (TX + 2) + 2 * TY;
    // slots of boundary vertices: the perimeter (top, bottom, left, right), or every vertex
    static constexpr int PER = PAPER ? V : 2 * TX + 2 * TY;
    static constexpr int LCAP = PART || PAPER ? 48 : 64;  // BFS layers kept as masks; deeper layers use label tags
    // resident blocks per SM the registers must allow (shared memory allows
    // four 8-connected 32x32 tiles, eight 32x16 tiles, two 64x32 tiles)
    // (the stencils: 62 KB at 8 arcs, 113 KB at 20, 146 KB at 28)
    static constexpr int MINB = PAPER ? (N <= 8 ? 3 : N <= 20 ? 2 : 1) : PART ? 8 : TX == 32 ? 4 : (TX * TY == 2048) ? 2 : 1;
    // after this many passes of the graph warp over a push layer the rest of it
    // is handed to all warps (1: 12% slower on the 1024x1024 4-connected grid;
    // 4, 8 and 16 within 3% of each other everywhere)
    static constexpr int HEAVY = 8;
    static constexpr size_t smem = (size_t)(N + 3) * V * 4                  // cap, tcap, exc, lab
                                   + (size_t)(N + 4) * TY * sizeof(W)       // R[N], T, E, inc, vis
                                   + (size_t)(LCAP + 1) * TY * sizeof(W)    // BFS layers 1..LCAP
                                   + (size_t)(HL + PER) * 4 + 16;           // halo labels, hmin, padding
    static_assert(TX == 32 || TX == 64, "row width must be 32 or 64");
    static_assert((TY % 32 == 0 || (TY == 16 && TX == 32)) && TY <= 64 && V % NT == 0 && NT % 32 == 0,
                  "tile/threads mismatch");
    static_assert(!PAPER || (TX == 32 && TY == 32), "the stencils run on 32x32 tiles");
};

// halo cell index of (hx, hy), a cell just outside the tile
template <int CONN, int TX, int TY>
__device__ __forceinline__ int halo_idx(int hx, int hy) {
    if constexpr (is_paper(CONN)) {
        constexpr int R = radius_of(CONN);
        return (hy + R) * (TX + 2 * R) + hx + R;
    }
    if (hy < 0) return hx + 1;
    if (hy >= TY) return (TX + 2) + hx + 1;
    if (hx < 0) return 2 * (TX + 2) + hy;
    return 2 * (TX + 2) + TY + hy;
}

// Kogge-Stone fill inside one row: x joins if x+1 is in g and pl[x] (arc x -> x+1),
// or x-1 is in g and pr[x] (arc x -> x-1), repeatedly (a whole run at once).
template <typename W>
__device__ __forceinline__ W row_fill(W g, W pl, W pr) {
    W a = g, p = pl;
    a |= p & (a >> 1);  p &= p >> 1;
    a |= p & (a >> 2);  p &= p >> 2;
    a |= p & (a >> 4);  p &= p >> 4;
    a |= p & (a >> 8);  p &= p >> 8;
    a |= p & (a >> 16);
    if (sizeof(W) == 8) { p &= p >> 16;  a |= p & (a >> (sizeof(W) * 4)); }
    W b = g;
    p = pr;
    b |= p & (b << 1);  p &= p << 1;
    b |= p & (b << 2);  p &= p << 2;
    b |= p & (b << 4);  p &= p << 4;
    b |= p & (b << 8);  p &= p << 8;
    b |= p & (b << 16);
    if (sizeof(W) == 8) { p &= p << 16;  b |= p & (b << (sizeof(W) * 4)); }
    return a | b;
}

// distance tag of a deep BFS layer (negative: never equal to a label >= 0)
__device__ __forceinline__ int deep_tag(int epoch, int L) { return ~((epoch << 16) | L); }

__device__ __forceinline__ int first_bit(unsigned m) { return __ffs((int)m) - 1; }
__device__ __forceinline__ int count_bits(unsigned m) { return __popc(m); }
__device__ __forceinline__ int count_bits(u64 m) { return __popcll(m); }
__device__ __forceinline__ int first_bit(u64 m) { return __ffsll((long long)m) - 1; }

// highest set bit of a row word; `other` if there is none
__device__ __forceinline__ int top_bit(unsigned m, int other) {
    int x;
    asm("bfind.u32 %0, %1;" : "=r"(x) : "r"(m));
    return m ? x : other;
}
__device__ __forceinline__ int top_bit(u64 m, int other) {
    int x;
    asm("bfind.u64 %0, %1;" : "=r"(x) : "l"(m));
    return m ? x : other;
}
// Shared-memory accesses of the push at constant offsets (bytes) from an
// address: predicated stores, and an add that is always executed (an amount of
// 0 changes nothing).  Timed in one warp: a predicated store 4.6 cycles, an
// unconditional add 4.3, a predicated add 37, a taken branch 23 and a divergent
// one 45-70.  The lane-per-row push written with C++ conditions ran a solve's
// discharge 1.35 times as fast as the push by all warps, this 1.8 times.
template <int OFF>
__device__ __forceinline__ void st_if(bool p, unsigned a, int v) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared.u32 [%0+%3], %1;\n}\n" ::"r"(a), "r"(v),
                 "r"((unsigned)p), "n"(OFF)
                 : "memory");
}
template <int OFF>
__device__ __forceinline__ void red_add(unsigned a, int v) {
    asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF) : "memory");
}
// arc D of the vertex at `a` (the address of its cap[0]) took dl; c and rc: the
// residuals of the arc and of its reverse before.  An arc has one writer per
// step, the excess of its head may have several.
template <int CONN, int TX, int V, int D>
__device__ __forceinline__ void send_arc(unsigned a, int c, int rc, int dl) {
    constexpr int off = arc_dy(CONN, D) * TX + arc_dx(CONN, D);
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n @q st.shared.u32 [%0+%4], %1;\n @q st.shared.u32 [%0+%5], %2;\n"
        " red.shared.add.u32 [%0+%6], %3;\n}\n" ::"r"(a),
        "r"(c - dl), "r"(rc + dl), "r"(dl), "n"(4 * D * V), "n"(4 * ((D ^ 1) * V + off)),
        "n"(4 * ((arcs_of(CONN) + 1) * V + off))
        : "memory");
}
template <int CONN, int TX, int V, int... D>
__device__ __forceinline__ void send_arcs(unsigned a, const int (&c)[sizeof...(D)], const int (&rc)[sizeof...(D)],
                                          const int (&dl)[sizeof...(D)], std::integer_sequence<int, D...>) {
    (send_arc<CONN, TX, V, D>(a, c[D], rc[D], dl[D]), ...);
}

// One region's discharge.  The graph warp decides what comes next and runs the
// searches and the push layers by itself, with no block barrier between layers
// or rounds; it keeps its masks exact while it pushes.  Crowded push layers,
// labels to write and the end of the stages are commands to all warps.
//
// What bounds it: one region's chain of dependent steps (per discharge about 8
// rounds of 14 BFS layers and 9 push layers), at 4 cycles per dependent
// instruction and 23 per taken branch.  A push layer has 2 to 20 pushing
// vertices in 2 to 11 rows, so a lane per row does it in 2.3 passes on average
// (1024x1024 4-connected grid); by all warps, a row per warp with a block
// barrier per layer and the masks rebuilt from the planes after a round, a
// layer took 2400 cycles, now 900, and a BFS layer 310, now 75.  Discharge time
// of a solve: 2.35 -> 1.29 ms (1024x1024 4-connected, 12 sweeps), 9.5 -> 6.8 ms
// (2048x2048 8-connected, hard seeds), 7.5 -> 4.8 ms (637x419 8-connected).
// 64 or 128 threads per region instead of 256: 5-20% slower (staging,
// write-back and crowded layers), also with five or six regions per SM.
// The masks stay in registers on the 4-connected 32x32 and all 64x32 tiles; the
// register limits of MINB spill 114 bytes on 8-connected 32x32 tiles, 118 (12) on
// 32x16 with 8 (4) arcs, 290 on 8-connected 64x64 and 34 at 20 stencil arcs.
// The stencils of Sec. 7.1 on the same code, against the vertex-by-vertex kernel
// (ard_generic.cuh): 325 -> 17 ms discharge time of a 500x500 solve at
// connectivity 8, 60 sweeps.
template <int CONN, int TX, int TY, int NT>
__device__ __forceinline__ void discharge2d_region(const Geom &g, const DevState &st, const SweepArgs &sa,
                                                   const int r, unsigned long long *mbar, unsigned &mphase) {
    using C = Cfg2D<CONN, TX, TY, NT>;
    typedef typename C::W W;
    constexpr int N = C::N, V = C::V, RPL = C::RPL, NW = C::NW, HW = C::HW, LCAP = C::LCAP, R = C::R;
    constexpr bool PAPER = C::PAPER;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smraw[];
    // (16 bytes of padding first: the reverse arc of the first cell's -x arc is read unconditionally)
    int *s_cap = (int *)(smraw + 16);     // [N][V] residual of arc i -> i + D(d)
    int *s_tcap = s_cap + N * V;          // [V]
    int *s_exc = s_tcap + V;              // [V]
    int *s_lab = s_exc + V;               // [V] region label (deep BFS layers: negative tags)
    W *s_R = (W *)(s_lab + V);            // [N][TY] residual masks (rows rebuilt from the planes)
    W *s_T = s_R + N * TY;                // [TY] residual arc to t
    W *s_E = s_T + TY;                    // [TY] positive excess
    W *s_inc = s_E + TY;                  // [TY] vertices that joined the closure
    W *s_vis = s_inc + TY;                // [TY] final closure (during Augment rounds: excess received)
    W *s_layer = s_vis + TY;              // [LCAP+1][TY] BFS layers
    int *s_hl = (int *)(s_layer + (LCAP + 1) * TY);  // [HL] labels of B^R
    int *s_hmin = s_hl + C::HL;           // [PER] min label over residual boundary arcs of a perimeter vertex
    __shared__ int s_ctl[5];              // command, its argument, epoch, any augmentation, stage
    __shared__ unsigned s_rd[2], s_bd[2];  // rows changed by the block's push / rows with pushes into B^R
    __shared__ unsigned long long s_flow;
    enum { kDone = 0, kLabel = 1, kPush = 2 };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // does this lane of the graph warp hold tile rows (all do unless the tile has 16 rows)
    const bool lrow = !C::PART || lane < TY;
    DIAG_DECL
    const long long diag_t0 = clock64();
    (void)diag_t0;
    const int rx = r % g.RX, ry = r / g.RX;
    const int ox = rx * TX, oy = ry * TY;
    const size_t n = (size_t)g.n;
    const int dinf = g.dinf;
    if (tid == 0) s_flow = 0;

    // masks of tile row y from the planes (one warp; a ballot gives half a row word)
    auto rebuild_row = [&](int y) {
#pragma unroll
        for (int h = 0; h < HW; ++h) {
            const int i = y * TX + lane + 32 * h, hw = y * HW + h;
            unsigned b[N];
#pragma unroll
            for (int d = 0; d < N; ++d) b[d] = __ballot_sync(FULL, s_cap[d * V + i] > 0);
            const unsigned bt = __ballot_sync(FULL, s_tcap[i] > 0), be = __ballot_sync(FULL, s_exc[i] > 0);
            if (lane == 0) {
#pragma unroll
                for (int d = 0; d < N; ++d) ((unsigned *)s_R)[d * TY * HW + hw] = b[d];
                ((unsigned *)s_T)[hw] = bt;
                ((unsigned *)s_E)[hw] = be;
            }
        }
    };
    // slot p -> tile coordinates (perimeter: top row, bottom row, left column, right column)
    auto per_xy = [](int p, int &x, int &y) {
        if (PAPER) { x = p % TX; y = p / TX; }
        else if (p < TX) { x = p; y = 0; }
        else if (p < 2 * TX) { x = p - TX; y = TY - 1; }
        else if (p < 2 * TX + TY) { x = 0; y = p - 2 * TX; }
        else { x = TX - 1; y = p - 2 * TX - TY; }
    };
    // hmin[p] = min{d(w) : residual arc from the perimeter vertex to w in B^R},
    // slots p0, p0 + step, .. whose row is in `rows`
    auto rebuild_hmin = [&](int p0, int step, u64 rows) {
        for (int p = p0; p < C::PER; p += step) {
            int x, y;
            per_xy(p, x, y);
            if (!((rows >> y) & 1ull)) continue;
            int m = INT_MAX;
#pragma unroll
            for (int d = 0; d < N; ++d) {
                const int hx = x + arc_dx(CONN, d), hy = y + arc_dy(CONN, d);
                if (hx >= 0 && hx < TX && hy >= 0 && hy < TY) continue;
                if (s_cap[d * V + y * TX + x] > 0) m = min(m, s_hl[halo_idx<CONN, TX, TY>(hx, hy)]);
            }
            s_hmin[p] = m;
        }
    };

    // ---- stage the tile --------------------------------------------------------
    const bool full = ox + TX <= g.X && oy + TY <= g.Y;
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
        for (int c = tid; c < (N + 2) * TY; c += NT) {
            const int p = c / TY, ly = c % TY;
            const int *plane = p < N ? st.cap + (size_t)p * n : p == N ? st.tcap : st.exc;
            bulk_g2s(s_cap + p * V + ly * TX, plane + (size_t)(oy + ly) * g.X + ox, TX * 4, mbar);
        }
        for (int i4 = tid; i4 < V / 4; i4 += NT) *(int4 *)&s_lab[i4 * 4] = make_int4(0, 0, 0, 0);
    } else {
        for (int i = tid; i < V; i += NT) {
            const int lx = i % TX, ly = i / TX;
            const int x = ox + lx, y = oy + ly;
            const bool in = x < g.X && y < g.Y;
            const size_t v = (size_t)y * g.X + x;
#pragma unroll
            for (int d = 0; d < N; ++d) s_cap[d * V + i] = in ? st.cap[d * n + v] : 0;
            s_tcap[i] = in ? st.tcap[v] : 0;
            s_exc[i] = in ? st.exc[v] : 0;
            s_lab[i] = 0;
        }
    }
    for (int h = tid; h < C::HL; h += NT) {
        int hx, hy;
        if constexpr (PAPER) {
            hx = h % (TX + 2 * R) - R;
            hy = h / (TX + 2 * R) - R;
            bool head = false;  // cells outside the tile that are the head of some stencil arc from it
#pragma unroll
            for (int d = 0; d < N; ++d) {
                const int sx = hx - arc_dx(CONN, d), sy = hy - arc_dy(CONN, d);
                head |= sx >= 0 && sx < TX && sy >= 0 && sy < TY;
            }
            const bool out = hx < 0 || hx >= TX || hy < 0 || hy >= TY;
            const int x = ox + hx, y = oy + hy;
            s_hl[h] = (head && out && x >= 0 && x < g.X && y >= 0 && y < g.Y) ? st.lab[(size_t)y * g.X + x] : dinf;
            continue;
        }
        if (h < TX + 2) { hx = h - 1; hy = -1; }
        else if (h < 2 * (TX + 2)) { hx = h - (TX + 2) - 1; hy = TY; }
        else if (h < 2 * (TX + 2) + TY) { hx = -1; hy = h - 2 * (TX + 2); }
        else { hx = TX; hy = h - 2 * (TX + 2) - TY; }
        const bool corner = (hx < 0 || hx >= TX) && (hy < 0 || hy >= TY);
        const int x = ox + hx, y = oy + hy;
        const bool ing = x >= 0 && x < g.X && y >= 0 && y < g.Y;
        s_hl[h] = (ing && (CONN == 8 || !corner)) ? st.lab[(size_t)y * g.X + x] : dinf;
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
    for (int y = warp; y < TY; y += NW) rebuild_row(y);
    rebuild_hmin(tid, NT, ~0ull);
    __syncthreads();
    DIAG_LAP(0);

    // ---- the graph warp's state and searches -----------------------------------
    // (Rm holds no arcs that leave the tile up or down; those that leave it to
    // the left or right meet no bit in a shifted word)
    auto stays = [](int y, int d) -> bool { return y + arc_dy(CONN, d) >= 0 && y + arc_dy(CONN, d) < TY; };
    W Rm[N][RPL], T[RPL], E[RPL], Cl[RPL], sdB[RPL];
    W recv[RPL];  // vertices that received excess in this round's push
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        const int y = lane * RPL + j;
#pragma unroll
        for (int d = 0; d < N; ++d) Rm[d][j] = warp == 0 && lrow && stays(y, d) ? s_R[d * TY + y] : 0;
        T[j] = warp == 0 && lrow ? s_T[y] : 0;
        E[j] = warp == 0 && lrow ? s_E[y] : 0;
        Cl[j] = sdB[j] = recv[j] = 0;
    }
    bool pushed[RPL] = {};   // rows that pushed
    u64 block_rows = 0;      // rows changed by pushes of the whole block
    auto row_set = [&](const bool (&f)[RPL]) -> u64 {  // bit per row from a flag per row of every lane
        if (RPL == 1) return __ballot_sync(FULL, f[0]);
        u64 m = 0;
#pragma unroll
        for (int j = 0; j < RPL; ++j)
            for (unsigned b = __ballot_sync(FULL, f[j]); b; b &= b - 1) m |= 1ull << ((__ffs((int)b) - 1) * RPL + j);
        return m;
    };
    // next stage value above k: min{d(w)+1 > k : w in B^R, d(w) < d_inf}
    auto next_stage = [&](int k) -> int {
        int best = INT_MAX;
        for (int h = lane; h < C::HL; h += 32) {
            const int v = s_hl[h];
            if (v < dinf && v + 1 > k && v + 1 < best) best = v + 1;
        }
        return __reduce_min_sync(FULL, best);
    };
    // boundary part of the seed rows of T_k: a residual arc to w in B^R with d(w) < k
    auto seed_boundary = [&](int k) {
        if constexpr (PAPER) {
            W s = 0;
#pragma unroll 8
            for (int y = 0; y < TY; ++y) {
                const unsigned b = __ballot_sync(FULL, s_hmin[y * TX + lane] < k);
                if (lane == y) s = b;
            }
            sdB[0] = s;
            return;
        }
        W top = 0, bot = 0;
#pragma unroll
        for (int h = 0; h < HW; ++h) {
            const int x = lane + 32 * h;
            top |= (W)__ballot_sync(FULL, s_hmin[x] < k) << (32 * h);
            bot |= (W)__ballot_sync(FULL, s_hmin[TX + x] < k) << (32 * h);
        }
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const int y = lane * RPL + j;
            W s = 0;
            if (lrow) {
                if (s_hmin[2 * TX + y] < k) s |= (W)1;
                if (s_hmin[2 * TX + TY + y] < k) s |= (W)1 << (TX - 1);
                if (y == 0) s |= top;
                if (y == TY - 1) s |= bot;
            }
            sdB[j] = s;
        }
    };
    // bit x of the result = bit x - dx
    auto shift_x = [](W b, int dx) -> W { return dx > 0 ? (W)(b << dx) : (W)(b >> -dx); };
    // (stencils) the words of the rows y - R .. y + R of the lane's row y; a row
    // outside the tile gives the lane's own word: callers mask it
    auto rows_beside = [&](W f, W (&row)[2 * R + 1]) {
        row[R] = f;
#pragma unroll
        for (int q = 1; q <= R; ++q) {
            row[R - q] = __shfl_up_sync(FULL, f, q);
            row[R + q] = __shfl_down_sync(FULL, f, q);
        }
    };
    // one backward BFS step on the masks: vertices with a residual arc into f
    auto expand = [&](const W (&f)[RPL], W (&out)[RPL]) {
        if constexpr (PAPER) {
            W row[2 * R + 1], a = 0;
            rows_beside(f[0], row);
#pragma unroll
            for (int d = 0; d < N; ++d) a |= Rm[d][0] & shift_x(row[arc_dy(CONN, d) + R], -arc_dx(CONN, d));
            out[0] = a;
            return;
        }
        const W up = __shfl_up_sync(FULL, f[RPL - 1], 1);
        const W dn = __shfl_down_sync(FULL, f[0], 1);
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const W fa = j == 0 ? up : f[j - 1];        // row y-1
            const W fb = j == RPL - 1 ? dn : f[j + 1];  // row y+1
            W a = (Rm[0][j] & (f[j] >> 1)) | (Rm[1][j] & (f[j] << 1)) | (Rm[2][j] & fb) | (Rm[3][j] & fa);
            if (CONN == 8)
                a |= (Rm[4][j] & (fb >> 1)) | (Rm[5][j] & (fa << 1)) | (Rm[6][j] & (fb << 1)) | (Rm[7][j] & (fa >> 1));
            out[j] = a;
        }
    };
    // closure Cl := Cl U {u : u -> T_k} (residual reachability); increments to s_inc
    auto flood = [&]() {
        W fr[RPL], inc[RPL];
        bool any = false;
#pragma unroll
        for (int j = 0; j < RPL; ++j) {
            const W f = row_fill<W>((T[j] | sdB[j]) & ~Cl[j], Rm[0][j] & ~Cl[j], Rm[1][j] & ~Cl[j]);
            Cl[j] |= f;
            inc[j] = f;
            fr[j] = f;
            any |= f != 0;
        }
        while (__any_sync(FULL, any)) {
            W nf[RPL];
            expand(fr, nf);
            any = false;
            DIAG_ADD(3, 1);
#pragma unroll
            for (int j = 0; j < RPL; ++j) {
                const W f = row_fill<W>(nf[j] & ~Cl[j], Rm[0][j] & ~Cl[j], Rm[1][j] & ~Cl[j]);
                Cl[j] |= f;
                inc[j] |= f;
                fr[j] = f;
                any |= f != 0;
            }
        }
        if (lrow) {
#pragma unroll
            for (int j = 0; j < RPL; ++j) s_inc[lane * RPL + j] = inc[j];
        }
    };
    // all threads: label the vertices of s_inc with k
    auto write_labels = [&](int k) {
        for (int y = warp; y < TY; y += NW) {
            const W m = s_inc[y];
            if (!m) continue;
#pragma unroll
            for (int h = 0; h < HW; ++h) {
                const int x = lane + 32 * h;
                if ((m >> x) & 1) s_lab[y * TX + x] = k;
            }
        }
    };

    long long flow_acc = 0;
    auto off = [](int d) -> int { return arc_dy(CONN, d) * TX + arc_dx(CONN, d); };
    auto send = [&](int i, const int (&c)[N], const int (&rc)[N], const int (&dl)[N]) {
        send_arcs<CONN, TX, V>(smem_u32(s_cap + i), c, rc, dl, std::make_integer_sequence<int, N>());
    };
    // what vertex (x, y) with excess e, in layer 1, sends into B^R; returns the rest
    auto push_out = [&](int x, int y, int e, int k) -> int {
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const int hx = x + arc_dx(CONN, d), hy = y + arc_dy(CONN, d);
            if (hx >= 0 && hx < TX && hy >= 0 && hy < TY) continue;
            const int c = s_cap[d * V + y * TX + x];
            if (e > 0 && c > 0 && s_hl[halo_idx<CONN, TX, TY>(hx, hy)] < k) {
                const int b = min(e, c);
                s_cap[d * V + y * TX + x] = c - b;
                e -= b;
            }
        }
        return e;
    };
    // The vertices of BFS layer L in half row h of row y that have excess
    // (bit `act` of this lane) push it one layer down, to T_k from layer 1.
    // Amounts follow the arc order.  Returns the vertices that pushed along each
    // arc (to[d], a bit per column of the half row) and whether any pushed into
    // B^R; sd: the row's boundary seeds.
    struct PushOut { unsigned to[N]; bool bpush; };
    auto push_half = [&](int y, int h, bool act, int L, int k, int epoch, unsigned sd, PushOut &o) {
        const int x = lane + 32 * h, i = y * TX + x;
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
            if (o.bpush && e > 0) e = push_out(x, y, e, k);
            if (act) s_exc[i] = e;
#pragma unroll
            for (int d = 0; d < N; ++d) o.to[d] = 0;
            return;
        }
        int e = act ? s_exc[i] : 0;
        bool adm[N];
        if (L - 1 <= LCAP) {
            const W *lay = s_layer + (L - 1) * TY;
            const W bit = (W)1 << x;
            W row[2 * R + 1];
#pragma unroll
            for (int q = -R; q <= R; ++q) row[q + R] = y + q >= 0 && y + q < TY ? lay[y + q] : 0;
#pragma unroll
            for (int d = 0; d < N; ++d) adm[d] = (row[arc_dy(CONN, d) + R] & shift_x(bit, arc_dx(CONN, d))) != 0;
        } else {
            const int tg = deep_tag(epoch, L - 1);
#pragma unroll
            for (int d = 0; d < N; ++d) {
                const int nx = x + arc_dx(CONN, d), ny = y + arc_dy(CONN, d);
                adm[d] = nx >= 0 && nx < TX && ny >= 0 && ny < TY && s_lab[ny * TX + nx] == tg;
            }
        }
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const int c = s_cap[d * V + i], dl = adm[d] ? min(e, c) : 0;
            e -= dl;
            if (dl > 0) {
                s_cap[d * V + i] = c - dl;
                s_cap[(d ^ 1) * V + i + off(d)] += dl;
                atomicAdd(&s_exc[i + off(d)], dl);
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
                    {
                        W vis[RPL], fr[RPL], want[RPL];
                        bool pending = false;
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            // excess that can reach T_k lies inside the (older) closure
                            const W ex = E[j] & Cl[j];
                            recv[j] = 0;
                            vis[j] = fr[j] = T[j] | sdB[j];
                            if (lrow) s_layer[1 * TY + lane * RPL + j] = fr[j];
                            if (fr[j] & ex) lmax = 1;
                            want[j] = ex & ~vis[j];
                            pending |= want[j] != 0;
                        }
                        L = 1;
                        bool go = __any_sync(FULL, pending);
                        // two layers per vote: a layer too many is an empty or unused mask
                        while (go && L + 2 <= LCAP) {
                            bool any = false;
                            pending = false;
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                W nf[RPL];
                                expand(fr, nf);
                                ++L;
#pragma unroll
                                for (int j = 0; j < RPL; ++j) {
                                    nf[j] &= ~vis[j];
                                    vis[j] |= nf[j];
                                    fr[j] = nf[j];
                                    if (lrow) s_layer[L * TY + lane * RPL + j] = nf[j];
                                    if (nf[j] & want[j]) lmax = L;
                                    want[j] &= ~nf[j];
                                }
                            }
#pragma unroll
                            for (int j = 0; j < RPL; ++j) {
                                any |= fr[j] != 0;
                                pending |= want[j] != 0;
                            }
                            const bool a = __any_sync(FULL, any), b = __any_sync(FULL, pending);
                            go = a && b;
                        }
                        while (go) {  // layers past the masks: label tags
                            W nf[RPL];
                            expand(fr, nf);
                            ++L;
                            bool any = false;
                            pending = false;
#pragma unroll
                            for (int j = 0; j < RPL; ++j) {
                                const int y = lane * RPL + j;
                                nf[j] &= ~vis[j];
                                any |= nf[j] != 0;
                                vis[j] |= nf[j];
                                fr[j] = nf[j];
                                if (L <= LCAP) {
                                    if (lrow) s_layer[L * TY + y] = nf[j];
                                } else {
                                    const int tg = deep_tag(epoch, L);
                                    for (W m = nf[j]; m; m &= m - 1) s_lab[y * TX + first_bit(m)] = tg;
                                }
                                if (nf[j] & want[j]) lmax = L;
                                want[j] &= ~nf[j];
                                pending |= want[j] != 0;
                            }
                            const bool a = __any_sync(FULL, any), b = __any_sync(FULL, pending);
                            go = a && b;
                        }
                        DIAG_ADD(6, L);
                    }
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
                // layered push, top layer first: a vertex of layer L pushes only
                // to layer L-1 (to T_k from layer 1), so every arc has one writer
                // per step.  Only vertices that had excess when the round began
                // or received some in an earlier step of it can push.  A lane
                // takes the vertices of its own rows one after another, all rows
                // side by side.
                DIAG_MARK();
                bool bnd[RPL] = {};  // rows with pushes into B^R
                W to[N][RPL];  // vertices that pushed along arc d in this round
#pragma unroll
                for (int j = 0; j < RPL; ++j)
#pragma unroll
                    for (int d = 0; d < N; ++d) to[d][j] = 0;
                if (L <= LCAP) {  // (layers without masks are left to the block)
                    // the lane's words of layers L, L - 1 and L - 2 (loaded a step ahead;
                    // layer 0 is unused space), and the rows beside of layers L - 1 and L - 2
                    W lw[RPL], lo[RPL], ln[RPL];
                    constexpr int NB = PAPER ? 2 * R + 1 : 2;
                    W nb[NB], nn[NB];
                    auto layer_word = [&](int l, int j) -> W { return lrow ? s_layer[l * TY + lane * RPL + j] : 0; };
                    auto beside = [&](const W (&f)[RPL], W (&o)[NB]) {
                        if constexpr (PAPER) {
                            rows_beside(f[0], o);
#pragma unroll
                            for (int q = -R; q <= R; ++q)
                                if (lane + q < 0 || lane + q >= TY) o[q + R] = 0;
                        } else {
                            const W up = __shfl_up_sync(FULL, f[RPL - 1], 1), dn = __shfl_down_sync(FULL, f[0], 1);
                            o[0] = lane == 0 ? (W)0 : up;
                            o[1] = lane == 31 ? (W)0 : dn;
                        }
                    };
#pragma unroll
                    for (int j = 0; j < RPL; ++j) {
                        lw[j] = layer_word(L, j);
                        lo[j] = layer_word(L - 1, j);
                    }
                    beside(lo, nb);
                    bool heavy = false;
                    for (; L > 1; --L) {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) ln[j] = layer_word(L - 2, j);
                        beside(ln, nn);
                        W ru = 0, rd = 0;  // received by the row above the lane's first / below its last row
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            const int y = lane * RPL + j;
                            // layer L - 1 in the row that lies dy below
                            auto src_row = [&](int dy) -> W {
                                if constexpr (PAPER) return nb[dy + R];
                                else return dy == 0 ? lo[j] : dy < 0 ? (j == 0 ? nb[0] : lo[j > 0 ? j - 1 : 0])
                                                                     : (j == RPL - 1 ? nb[1] : lo[j + 1 < RPL ? j + 1 : j]);
                            };
                            W P = lw[j] & (E[j] | recv[j]);
                            pushed[j] |= P != 0;
                            int x = top_bit(P, lane);
                            // No branches inside: lanes without a vertex run along
                            // with amounts of 0 (a branch costs 23 cycles here, a
                            // divergent one 70, more than the work it would skip), in a
                            // column of their own: no bank conflicts
                            for (int it = 0;; ++it) {
                                const W bit = ((W)1 << x) & P;
                                const int i = y * TX + x;
                                int c[N], rc[N], dl[N];
#pragma unroll
                                for (int d = 0; d < N; ++d) {
                                    c[d] = s_cap[d * V + i];
                                    rc[d] = s_cap[(d ^ 1) * V + i + off(d)];
                                }
                                int e = s_exc[i];
                                P ^= bit;
                                x = top_bit(P, lane);
                                const bool again = __any_sync(FULL, P != 0);
#pragma unroll
                                for (int d = 0; d < N; ++d) {
                                    dl[d] = (src_row(arc_dy(CONN, d)) & shift_x(bit, arc_dx(CONN, d))) ? min(e, c[d]) : 0;
                                    e -= dl[d];
                                }
                                send(i, c, rc, dl);
#pragma unroll
                                for (int d = 0; d < N; ++d) {  // (an arc with c = 0 has no bit in Rm)
                                    if (dl[d] != 0) to[d][j] |= bit;
                                    if (dl[d] == c[d]) Rm[d][j] &= ~bit;
                                }
                                st_if<4 * (N + 1) * V>(bit != 0, smem_u32(s_cap + i), e);
                                E[j] = (E[j] & ~bit) | (e > 0 ? bit : 0);
                                if (!again) break;
                                if (it == C::HEAVY) {  // the rest of a crowded layer is left to the block
                                    heavy = true;
                                    break;
                                }
                            }
                            lw[j] = P;
                            // (marks of earlier layers are sent again: harmless)
                            if constexpr (!PAPER)
#pragma unroll
                            for (int d = 0; d < N; ++d) {
                                const W m = shift_x(to[d][j], arc_dx(CONN, d));
                                if (arc_dy(CONN, d) == 0) recv[j] |= m;
                                else if (arc_dy(CONN, d) < 0) {
                                    if (j == 0) ru |= m;
                                    else recv[j - 1] |= m;
                                } else {
                                    if (j == RPL - 1) rd |= m;
                                    else recv[j + 1] |= m;
                                }
                            }
                        }
                        if constexpr (PAPER) {
#pragma unroll
                            for (int q = -R; q <= R; ++q) {  // what the rows send q rows down
                                W m = 0;
#pragma unroll
                                for (int d = 0; d < N; ++d)
                                    if (arc_dy(CONN, d) == q) m |= shift_x(to[d][0], arc_dx(CONN, d));
                                if (q > 0) m = __shfl_up_sync(FULL, m, q > 0 ? q : 0);
                                if (q < 0) m = __shfl_down_sync(FULL, m, q < 0 ? -q : 0);
                                recv[0] |= lane - q >= 0 && lane - q < TY ? m : (W)0;
                            }
                        } else {
                            const W fu = __shfl_up_sync(FULL, rd, 1), fd = __shfl_down_sync(FULL, ru, 1);
                            recv[0] |= lane > 0 ? fu : (W)0;
                            recv[RPL - 1] |= lane < 31 ? fd : (W)0;
                        }
                        __syncwarp();
                        if (heavy) break;
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            lw[j] = lo[j];
                            lo[j] = ln[j];
                        }
#pragma unroll
                        for (int q = 0; q < NB; ++q) nb[q] = nn[q];
                    }
                    if (heavy) {  // layer L shrinks to the vertices that have not pushed
#pragma unroll
                        for (int j = 0; j < RPL; ++j)
                            if (lrow) s_layer[L * TY + lane * RPL + j] = lw[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) {
                            const int y = lane * RPL + j;
                            W P = lw[j] & (E[j] | recv[j]);
                            pushed[j] |= P != 0;
                            int x = top_bit(P, lane);
                            for (bool again = true; again;) {
                                const W bit = ((W)1 << x) & P;
                                const int i = y * TX + x;
                                int e = bit ? s_exc[i] : 0;
                                const int tc = s_tcap[i];
                                P ^= bit;
                                x = top_bit(P, lane);
                                again = __any_sync(FULL, P != 0);
                                const int dl = min(e, tc);
                                e -= dl;
                                flow_acc += dl;
                                const bool out = e > 0 && (sdB[j] & bit);
                                if (__any_sync(FULL, out)) {
                                    if (out) e = push_out(i % TX, y, e, k);
                                    bnd[j] |= out;
                                }
                                st_if<4 * N * V>(bit != 0, smem_u32(s_cap + i), tc - dl);
                                st_if<4 * (N + 1) * V>(bit != 0, smem_u32(s_cap + i), e);
                                T[j] &= dl == tc ? ~bit : ~(W)0;
                                E[j] = (E[j] & ~bit) | (e > 0 ? bit : 0);
                            }
                        }
                        __syncwarp();
                        L = 0;
                    }
                }
                // the reverse arcs of the pushes are residual now
#pragma unroll
                for (int d = 0; d < N; ++d) {
                    const int dy = arc_dy(CONN, d), dx = arc_dx(CONN, d);
                    if constexpr (PAPER) {
                        W m = shift_x(to[d][0], dx);
                        if (dy > 0) m = __shfl_up_sync(FULL, m, dy > 0 ? dy : 0);
                        if (dy < 0) m = __shfl_down_sync(FULL, m, dy < 0 ? -dy : 0);
                        Rm[d ^ 1][0] |= lane - dy >= 0 && lane - dy < TY ? m : (W)0;
                    } else if (dy == 0) {
#pragma unroll
                        for (int j = 0; j < RPL; ++j) Rm[d ^ 1][j] |= shift_x(to[d][j], dx);
                    } else if (dy > 0) {
                        const W m = __shfl_up_sync(FULL, shift_x(to[d][RPL - 1], dx), 1);
                        if (lane > 0) Rm[d ^ 1][0] |= m;
#pragma unroll
                        for (int j = 1; j < RPL; ++j) Rm[d ^ 1][j] |= shift_x(to[d][j - 1], dx);
                    } else {
                        const W m = __shfl_down_sync(FULL, shift_x(to[d][0], dx), 1);
                        if (lane < 31) Rm[d ^ 1][RPL - 1] |= m;
#pragma unroll
                        for (int j = 0; j + 1 < RPL; ++j) Rm[d ^ 1][j] |= shift_x(to[d][j + 1], dx);
                    }
                }
                DIAG_LAP(7);
                const u64 rows = row_set(bnd);
                if (rows) {
                    rebuild_hmin(lane, 32, rows);
                    __syncwarp();
                    seed_boundary(k);
                }
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
                s_rd[0] = s_rd[1] = s_bd[0] = s_bd[1] = 0;
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
        // rows w, w + NW, .. of each layer
        const int ep = s_ctl[2];
        const int kk = s_ctl[4];
        W *s_recv = s_vis;
        int L = arg;
        for (; L >= 1; --L) {
            // a lane per row: the busy rows; the warp's own are every NW-th of them
            u64 mine = 0;
            bool many = false;
            int rank0 = 0;
#pragma unroll
            for (int q = 0; q < (TY + 31) / 32; ++q) {
                const int y = lane + 32 * q;
                W P = 0;
                // (deep layers: every row, as marks of the step itself would show in the word)
                if (y < TY) P = L <= LCAP ? s_layer[L * TY + y] & (s_E[y] | s_recv[y]) : (W)~(W)0;
                many |= count_bits(P) > C::HEAVY / 2;
                const unsigned busy = __ballot_sync(FULL, P != 0);
                const int rank = rank0 + __popc(busy & ((1u << lane) - 1u));
                mine |= (u64)__ballot_sync(FULL, P != 0 && rank % NW == warp) << (32 * q);
                rank0 += __popc(busy);
            }
            if (!__any_sync(FULL, many)) break;  // (the same in every warp) back to the graph warp
            for (; mine; mine &= mine - 1) {
                const int y = first_bit(mine);
                const W Py = (L <= LCAP ? s_layer[L * TY + y] : (W)~(W)0) & (s_E[y] | s_recv[y]);
                const W sd = s_inc[y];
                W rv[2 * R + 1] = {};
                bool any = false, bp = false;
#pragma unroll
                for (int h = 0; h < HW; ++h) {
                    bool act = (Py >> (lane + 32 * h)) & 1;
                    if (L > LCAP) act = act && s_lab[y * TX + lane + 32 * h] == deep_tag(ep, L);
                    const unsigned ab = __ballot_sync(FULL, act);
                    if (!ab) continue;
                    any = true;
                    PushOut o;
                    push_half(y, h, act, L, kk, ep, (unsigned)(sd >> (32 * h)), o);
                    bp |= o.bpush;
                    if (L > 1) {
#pragma unroll
                        for (int d = 0; d < N; ++d)
                            rv[arc_dy(CONN, d) + R] |= shift_x((W)o.to[d] << (32 * h), arc_dx(CONN, d));
                    }
                }
                if (any) {
                    if (L > 1) {
                        W v = 0;
#pragma unroll
                        for (int q = 0; q <= 2 * R; ++q)
                            if (lane == q) v = rv[q];
                        if (v) atomicOr(&s_recv[y - R + lane], v);
                    }
                    if (lane == 31) {
                        u64 m = 1ull << y;
                        if (L > 1)
#pragma unroll
                            for (int q = 1; q <= R; ++q) m |= (1ull << y) << q | (1ull << y) >> q;
                        atomicOr(&s_rd[0], (unsigned)m);
                        if (TY > 32) atomicOr(&s_rd[1], (unsigned)(m >> 32));
                        if (bp) atomicOr(&s_bd[y >> 5], 1u << (y & 31));
                    }
                }
            }
            __syncthreads();
        }
        {
            u64 rows = s_rd[0] | (u64)s_rd[1] << 32;
            if (TY < 64) rows &= (1ull << (TY & 63)) - 1;
            int idx = 0;
            for (u64 m = rows; m; m &= m - 1, ++idx)
                if (idx % NW == warp) rebuild_row(first_bit(m));
            const u64 bd = s_bd[0] | (u64)s_bd[1] << 32;
            if (bd) rebuild_hmin(tid, NT, bd);
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int j = 0; j < RPL; ++j) {
                    const int y = lane * RPL + j;
                    if (lrow && ((rows >> y) & 1ull)) {
#pragma unroll
                        for (int d = 0; d < N; ++d) Rm[d][j] = stays(y, d) ? s_R[d * TY + y] : 0;
                        T[j] = s_T[y];
                        E[j] = s_E[y];
                    }
                }
#pragma unroll
                for (int j = 0; j < RPL; ++j) recv[j] = lrow ? s_recv[lane * RPL + j] : 0;
                if (bd) seed_boundary(k);
                resume = L;
                block_rows |= rows;
            }
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
                DIAG_ADD(2, 1);
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
        for (int j = 0; j < RPL; ++j) s_vis[lane * RPL + j] = Cl[j];
    }
    if (warp == 0) {  // the rows to write back: those that pushed and their neighbours
        u64 m = row_set(pushed) | block_rows;
        const u64 own = m;
#pragma unroll
        for (int q = 1; q <= R; ++q) m |= own << q | own >> q;
        if (lane == 0) {
            s_rd[0] = (unsigned)m;
            s_rd[1] = (unsigned)(m >> 32);
        }
    }
    __syncthreads();
    DIAG_MARK();

    // ---- write back: planes of rows that changed; labels and boundary flows always
    int left = 0;
    for (int i = tid; i < V; i += NT) {
        const int lx = i % TX, ly = i / TX;
        const int x = ox + lx, y = oy + ly;
        if (!(x < g.X && y < g.Y)) continue;
        const size_t v = (size_t)y * g.X + x;
        const bool dirty = (s_rd[ly >> 5] >> (ly & 31)) & 1u;
        bool perim = false;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const int nx = lx + arc_dx(CONN, d), ny = ly + arc_dy(CONN, d);
            const int gx = x + arc_dx(CONN, d), gy = y + arc_dy(CONN, d);
            const bool intile = nx >= 0 && nx < TX && ny >= 0 && ny < TY;
            const bool ing = gx >= 0 && gx < g.X && gy >= 0 && gy < g.Y;
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
        const int lab = ((s_vis[ly] >> lx) & 1) ? s_lab[i] : dinf;
        if (perim) st.lab_next[v] = lab;
        else st.lab[v] = lab;
        if (s_exc[i] > 0 && lab < dinf) left = 1;
    }
    left = __syncthreads_or(left);
    unsigned long long f = (unsigned long long)flow_acc;
    for (int o = 16; o > 0; o >>= 1) f += __shfl_down_sync(0xffffffffu, f, o);
    if (lane == 0 && f) atomicAdd(&s_flow, f);
    __syncthreads();
    if (tid == 0) {
        DIAG_LAP(10);
        DIAG_ADD(11, clock64() - diag_t0);
        DIAG_ADD(12, 1);
        DIAG_FLUSH();
        if (s_flow) atomicAdd(st.flow_t, s_flow);
        st.disc[r] = 1;
        st.left_active[r] = (unsigned char)left;
        if (err) atomicExch(&st.ctr[kError], 1);
        atomicAdd(&sa.c64->stages, (unsigned long long)stages);
        atomicAdd(&sa.c64->rounds, (unsigned long long)rounds);
        atomicAdd(&sa.c64->discharges, 1ull);
        const unsigned long long live = (unsigned long long)min(TX, g.X - ox) * min(TY, g.Y - oy);
        atomicAdd(&sa.c64->discharged_vertices, live);
    }
}

// one block per region of one grid; regions without active vertices are skipped (Sec. 5.3)
template <int CONN, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT, (Cfg2D<CONN, TX, TY, NT>::MINB)) ard_discharge2d_kernel(const Geom g, const DevState st, const SweepArgs sa) {
    const int r = blockIdx.x;
    if (!region_to_discharge(st, r)) return;
    __shared__ __align__(8) unsigned long long s_mbar;
    if (threadIdx.x == 0) mbar_init(&s_mbar, 1);
    __syncthreads();
    unsigned phase = 0;
    discharge2d_region<CONN, TX, TY, NT>(g, st, sa, r, &s_mbar, phase);
}

template <int CONN, int TX, int TY, int NT>
static cudaError_t launch2d(const Geom &g, const DevState &st, const SweepArgs &sa, cudaStream_t s) {
    using C = Cfg2D<CONN, TX, TY, NT>;
    auto k = ard_discharge2d_kernel<CONN, TX, TY, NT>;
    {
        const cudaError_t e_at = ensure_smem_attr((const void *)k, (int)C::smem);
        if (e_at != cudaSuccess) return e_at;
    }
    k<<<g.nreg, NT, C::smem, s>>>(g, st, sa);
    return cudaGetLastError();
}

}  // namespace mf
