// fr_halo.cu -- local phase over halo-extended tiles for MFD (slope-split)
// forward accumulation and for the adjoints of both routing rules.
//
// Same decomposition as the D8 forward kernel: each CTA solves an inner tile
// plus an H-cell halo exactly in shared memory (a per-subdomain high-to-low solve,
// Sec. 2.4, on overlapping subdomains), and only cells whose dependencies
// reach outside the extended region go to the global phase.  With several
// receivers per cell (App. A) dependency sets spread wider than D8 basins, so
// the halo is deeper: 8 cells leave 0.7 % of the cells of a rough fractal DEM
// global (6 cells 1.3 %, 4 cells 3.3 %, none about 20 %).  A region of 96x80
// cells (80x64 inner, 1.5 region cells per inner cell) fills an SM's shared
// memory with all that its solve reads: values, the fraction of every edge,
// dependency bytes and the cell list, about 29 bytes a cell.
//
// The three modes differ only in the direction of the dependencies:
//   forward MFD   w_c = r_c    + sum over donors j    of f_{j->c} w_j
//   adjoint       g_c = gbar_c + sum over receivers k of f_{c->k} g_k
// (g = A^{-T} gbar, the transposed system of Eq. Aw=f: each cell's adjoint
// is its own gbar plus the fraction-weighted adjoints of its receivers; f = 1
// for D8).  A forward cell waits for its donors and then notifies its
// receivers; an adjoint cell waits for its receivers and notifies its donors.
// Fractions f_{j->k} = u_{j->k} / S_j (u = s^p, S_j the sum of cell j's
// weights) are computed once per cell by a fully parallel pass (mfd_fracs8)
// and read here, so the tile solve evaluates no powers.  The eight direction
// terms of a cell are accumulated in the fixed order of df_dot8, exactly as
// the global phase does, so a cell's value does not depend on which kernel
// computed it.
//
// Cells are finalised level by level, a topological order (Sec. 3.2): level 0
// has no dependency, level l + 1 the cells whose last dependency lies in level
// l.
//  - The levels are found on bits: one thread holds, for 32 cells of a region
//    row, the eight masks "has a dependency in direction k" in registers, and a
//    level is the AND over k of (no dependency, or the neighbour's done bit),
//    the neighbours' bits being funnel shifts of the nine words around.  That
//    takes the place of a counter per cell and an atomic per edge.
//  - Meanwhile the other warps read the fractions, whole rows at a time, into
//    one slot per edge of the region (an edge carries water one way only).
//    Reading them from global memory when a cell is solved costs a cache-line
//    look-up per cell and direction: 3.1 to 4.4 ms of the 8192^2 solve.
//  - The cells of each level go to a list, packed, so that a level is solved
//    with full warps.  One lane finalises one cell: its (up to eight)
//    dependency terms are loaded side by side and summed in the fixed order,
//    so the result does not depend on which lane computed it.
// Cells that never become ready depend on cells outside the region (or lie on
// a cycle of a caller's routing) and are left to the global phase.
//
// What bounds it: about 34 levels per region, 500 cycles each to find (two
// barriers' worth of latency for little work) and 900 to solve (bank conflicts
// of the scattered reads while levels are wide, latency when they are narrow),
// 66 K cycles per region in all.  8192^2: 5.37 ms forward and 5.38 adjoint with
// the queue of ready cells that this replaces (270 K warp instructions per 64x64
// tile at 14 busy lanes), 2.83 and 2.91 ms now.
#include "fr_engine.cuh"

namespace fr {
namespace {

constexpr int kHaloTX = kMfdTileX, kHaloTY = kMfdTileY, kHaloH = 8;
constexpr int kHaloNT = 1024;

struct HaloGeo {
    static constexpr int TX = kHaloTX, TY = kHaloTY, H = kHaloH;
    static constexpr int EX = TX + 2 * H, EY = TY + 2 * H, NE = EX * EY;  // extended region
    static constexpr int RX = EX + 2, RY = EY + 2;                       // plus a one-cell ring
    static constexpr int CP = EX + 8, NR = CP * RY;  // padded rows: ring cell (rx, ry) at byte ry * CP + rx + 3,
                                                     // so region cell (ex, ey) at (ey + 1) * CP + ex + 4
    static constexpr int WR = EX / 32, NWD = WR * EY;        // 32-cell words per row, in all
    static constexpr int FP = WR + 2, NF = FP * (EY + 2);    // done bits with a border of zero words
    static constexpr int OW = (NWD + 31) / 32;               // warps that hold words
    static_assert(EX % 32 == 0 && EX <= 128 && EY <= 128, "rows are whole words; list entries are 7 + 7 bits");
    static_assert(TX % 4 == 0 && H % 4 == 0, "four-cell groups");
    static_assert(NWD <= kHaloNT && 32 * NWD <= NR, "a word per thread; the masks fit the receiver bytes' place");
};

template <Mode M>
struct HaloMode {
    static constexpr bool kAdj = (M == Mode::AdjMfd || M == Mode::AdjD8);
    static constexpr bool kMfd = (M == Mode::FwdMfd || M == Mode::AdjMfd);
};

constexpr int kHaloLevels = 64;  // levels found before they are solved (then the next ones)

template <bool MFD>
struct SmemHalo {
    static constexpr int NE = HaloGeo::NE, NWD = HaloGeo::NWD;
    union {
        float2 v[NE];                       // value (water or adjoint), leading and trailing word
        uint32_t found[kHaloLevels][NWD];   // before the values: the cells of each level
    };
    // fraction of each edge of the region (of its higher cell, towards the
    // lower): E, S, SE and SW of a cell; the other four are its neighbours'
    float edge[MFD ? 4 : 1][MFD ? NE : 1];
    uint16_t list[NE];                  // the cells (ey << 7 | ex), level after level
    uint32_t done[2][HaloGeo::NF];      // done bits by level parity, zero border
    alignas(8) uint8_t rb[HaloGeo::NR]; // receiver masks of region + ring (0 outside the grid); then the
                                        // words' dependency masks, direction k at [k * NWD]
    alignas(4) uint8_t dm[NE];          // dependencies (donors forward, receivers adjoint)
    int lev[kHaloLevels + 1];           // where level l starts in the list
    int nlev, cnt;                      // levels found; cells of one more level
    int wide, narrow;                   // from level `wide` on at most kHaloMid cells each, from `narrow` 32
    unsigned int ndone;
};
constexpr int kHaloMid = 512;

// Plane and offset in `edge` of the edge from a cell in direction k.
__device__ __forceinline__ constexpr int edge_plane(int k) {
    return k == 0 || k == 2 ? 0 : k == 1 || k == 3 ? 1 : k == 5 || k == 7 ? 2 : 3;  // E/W, N/S, NW/SE, NE/SW
}
__device__ __forceinline__ constexpr int edge_off(int k) {
    return k == 0 || k == 3 || k == 6 || k == 7 ? 0 : offy(k) * HaloGeo::EX + offx(k);
}

// The byte vectors (left, centre, right neighbours) of the four cells of word
// w of a padded row.
struct HRow3 {
    uint32_t l, c, r;
};
__device__ __forceinline__ HRow3 hrow3(const uint32_t* w) {
    const uint32_t a = w[-1], b = w[0], d = w[1];
    return {__byte_perm(a, b, 0x6543), b, __byte_perm(b, d, 0x4321)};
}

// Barrier `id` among the first n threads' warps (n a multiple of 32); the
// second form returns whether p holds in any thread.
__device__ __forceinline__ void bar_n(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ bool bar_or(int id, int n, bool p) {
    int r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %3, 0;\n bar.red.or.pred q, %1, %2, p;\n selp.s32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"(id), "r"(n), "r"((int)p)
        : "memory");
    return r != 0;
}

// Marks the global inner cells of a warp (all 32 lanes call; glob: this
// lane's cell gi is global): their bits, list entries reserved with one
// atomic per warp, and their values pending (see k_global_poll).
__device__ __forceinline__ void mark_global_cells(const Prob& P, EngineGlobals* G, int64_t gi,
                                                  int pid, bool glob) {
    const unsigned m = __ballot_sync(0xffffffffu, glob);
    if (!m) return;
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long base = 0;
    if (lane == (unsigned)(__ffs(m) - 1)) base = atomicAdd(&G->glist_count, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
    if (glob) {
        atomicOr(P.gbits + (gi >> 5), 1u << (gi & 31));
        const unsigned long long slot = base + __popc(m & ((1u << lane) - 1u));
        if (FR_OK((int64_t)slot, P.glist_cap, 17))
            P.glist[slot] = ((unsigned long long)pid << 40) | (unsigned long long)gi;
        wr_f(P.out_hi, P, gi, __uint_as_float(kPending), 27);
        wr_f(P.out_lo, P, gi, __uint_as_float(kPending), 28);
    }
}

// Problem and tile of this CTA in a batched launch: the problem whose tiles
// [prefix[p], prefix[p+1]) hold blockIdx.x.
__device__ __forceinline__ int batch_problem_halo(const int64_t* __restrict__ prefix, int nprob,
                                                  int64_t& lt) {
    int lo = 0, hi = nprob - 1;
    const int64_t b = (int64_t)blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    lt = b - prefix[lo];
    return lo;
}

template <Mode M, bool BATCH>
__global__ void __launch_bounds__(kHaloNT, 1) k_local_halo(Prob Pone, EngineGlobals* G,
                                                           const Prob* __restrict__ probs,
                                                           const int64_t* __restrict__ prefix,
                                                           int nprob) {
    using HM = HaloMode<M>;
    constexpr int TX = HaloGeo::TX, TY = HaloGeo::TY, H = HaloGeo::H;
    constexpr int EX = HaloGeo::EX, EY = HaloGeo::EY;
    constexpr int RX = HaloGeo::RX, RY = HaloGeo::RY;
    constexpr int WR = HaloGeo::WR, NWD = HaloGeo::NWD, FP = HaloGeo::FP;
    constexpr int NT = kHaloNT, NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using Sm = SmemHalo<HM::kMfd>;
    Sm& S = *reinterpret_cast<Sm*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int64_t lt = (int64_t)blockIdx.x;
    const int pid = BATCH ? batch_problem_halo(prefix, nprob, lt) : 0;
    const Prob& P = BATCH ? probs[pid] : Pone;
    const int64_t tiles_x = (P.nx + TX - 1) / TX;
    const int64_t ty = lt / tiles_x, tx = lt - ty * tiles_x;
    const int64_t x0 = tx * TX, y0 = ty * TY;
    const int64_t ox = x0 - H - 1, oy = y0 - H - 1;  // ring origin (may be negative)
    // a tile whose ring lies inside the grid skips the bounds checks
    const bool interior = ox >= 0 && oy >= 0 && ox + RX <= P.nx && oy + RY <= P.ny;

    // ---- region + ring: receiver masks
    const bool vec = HM::kMfd && interior && x0 >= H + 4 && x0 + EX - H + 4 <= P.nx && (P.nx & 3) == 0 &&
                     ((uintptr_t)P.rb & 3) == 0;
    if (vec) {
        // whole padded rows (byte b is grid x = x0 - H - 4 + b), a word a lane
        constexpr int U = (RY + NW - 1) / NW, W4 = HaloGeo::CP / 4;
        static_assert(W4 <= 32, "a row of words per warp");
        uint32_t m[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ry = warp + u * NW;
            m[u] = 0;
            if (ry < RY && lane < W4)
                m[u] = __ldg(reinterpret_cast<const uint32_t*>(P.rb + (oy + ry) * P.nx + (x0 - H - 4)) + lane);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ry = warp + u * NW;
            if (ry < RY && lane < W4) reinterpret_cast<uint32_t*>(S.rb)[ry * W4 + lane] = m[u];
        }
    } else {
        constexpr int U = 3, C = (RX + 31) / 32;
        for (int r0 = warp; r0 < RY; r0 += U * NW) {
            uint8_t m[U][C];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int ry = r0 + u * NW;
                const int64_t gy = oy + ry;
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int rx = lane + 32 * q;
                    const int64_t gx = ox + rx;
                    m[u][q] = HM::kMfd ? 0 : kSink;
                    if (ry < RY && rx < RX && (interior || (gx >= 0 && gy >= 0 && gx < P.nx && gy < P.ny)))
                        m[u][q] = rd_rb(P, gy * P.nx + gx);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int ry = r0 + u * NW;
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int rx = lane + 32 * q;
                    if (ry >= RY || rx >= RX) continue;
                    uint32_t b = recv_mask<HM::kMfd>(m[u][q]);
                    if (!interior) b &= grid_mask(ox + rx, oy + ry, P.nx, P.ny);
                    S.rb[ry * HaloGeo::CP + rx + 3] = (uint8_t)b;
                }
            }
        }
    }
    for (int i = tid; i < HaloGeo::NF; i += NT) S.done[0][i] = S.done[1][i] = 0u;
    if (tid == 0) S.ndone = 0;
    __syncthreads();

    // ---- dependency bytes, four cells a step
    for (int g = tid; g < HaloGeo::NE / 4; g += NT) {
        const int ey = g / (EX / 4), ex = (g - ey * (EX / 4)) * 4;
        const uint32_t* row = reinterpret_cast<const uint32_t*>(S.rb + (ey + 1) * HaloGeo::CP + ex + 4);
        uint32_t d;
        if constexpr (HM::kAdj) {
            d = row[0];
        } else {
            // the donor in direction k has receiver bit opp(k) = k ^ 2 set
            const HRow3 up = hrow3(row - HaloGeo::CP / 4), mid = hrow3(row), dn = hrow3(row + HaloGeo::CP / 4);
            d = ((mid.r >> 2) & 0x01010101u) | ((up.c >> 2) & 0x02020202u);
            d |= ((mid.l << 2) & 0x04040404u) | ((dn.c << 2) & 0x08080808u);
            d |= ((up.r >> 2) & 0x10101010u) | ((up.l >> 2) & 0x20202020u);
            d |= ((dn.l << 2) & 0x40404040u) | ((dn.r << 2) & 0x80808080u);
        }
        reinterpret_cast<uint32_t*>(S.dm)[g] = d;
    }
    __syncthreads();

    // ---- this thread's word: dependency masks by direction (a transposition of
    // the 32 bytes), the cells that can become ready, level 0
    uint32_t open = 0, fin = 0, ndep[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const bool owner = tid < NWD;
    int fw = 0, wy = 0, wx = 0;  // index of the word's done bits; its first cell
    uint32_t* const dep_s = reinterpret_cast<uint32_t*>(S.rb) + tid;
    if (owner) {
        wy = tid / WR;
        wx = (tid - wy * WR) * 32;
        fw = (wy + 1) * FP + (tid - wy * WR) + 1;
        uint32_t dep[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t b = reinterpret_cast<const uint32_t*>(S.dm + wy * EX + wx)[q];
#pragma unroll
            for (int k = 0; k < 8; ++k)  // bits k of the four bytes, gathered at bits 28..31
                dep[k] |= ((((b >> k) & 0x01010101u) * 0x10204080u) >> 28) << (4 * q);
        }
        const int64_t gy = oy + wy + 1, gx = ox + wx + 1;
        uint32_t valid = gy >= 0 && gy < P.ny ? ~0u : 0u;
        if (gx < 0) valid = gx > -32 ? valid & (~0u << -gx) : 0u;
        if (gx + 32 > P.nx) valid = gx < P.nx ? valid & (~0u >> (gx + 32 - P.nx)) : 0u;
        uint32_t shut = 0;  // a dependency outside the region
        if (wy == 0) shut |= dep[1] | dep[4] | dep[5];
        if (wy == EY - 1) shut |= dep[3] | dep[6] | dep[7];
        if (wx == 0) shut |= (dep[2] | dep[5] | dep[6]) & 1u;
        if (wx == EX - 32) shut |= (dep[0] | dep[4] | dep[7]) & 0x80000000u;
        open = valid & ~shut;
        fin = open & ~(dep[0] | dep[1] | dep[2] | dep[3] | dep[4] | dep[5] | dep[6] | dep[7]);
        S.done[0][fw] = fin;
#pragma unroll
        for (int k = 0; k < 8; ++k) ndep[k] = ~dep[k];
    }
    // ---- the edges' fractions, by the warps that hold no bits, while the
    // others find the levels: each cell's row of eight goes to the edges it
    // gives to (the float4s of a region row are contiguous)
    if constexpr (HM::kMfd) {
        if (warp >= HaloGeo::OW) {
            constexpr int N4 = 2 * HaloGeo::NE, STEP = NT - HaloGeo::OW * 32, U = 4;
            for (int i0 = tid - HaloGeo::OW * 32; i0 < N4; i0 += U * STEP) {
                float4 f[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * STEP, c = i >> 1, ey = c / EX, ex = c - ey * EX;
                    const int64_t gx = ox + ex + 1, gy = oy + ey + 1;
                    f[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i < N4 && (interior || (gx >= 0 && gy >= 0 && gx < P.nx && gy < P.ny)))
                        f[u] = __ldg(reinterpret_cast<const float4*>(P.frac) + 2 * (gy * P.nx + gx) + (i & 1));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * STEP, c = i >> 1, ey = c / EX, ex = c - ey * EX;
                    if (i >= N4) break;
                    uint32_t m = S.rb[(ey + 1) * HaloGeo::CP + ex + 4];
                    if (ex == 0) m &= ~0x64u;       // edges that leave the region: W NW SW
                    if (ex == EX - 1) m &= ~0x91u;  // E NE SE
                    if (ey == 0) m &= ~0x32u;       // N NE NW
                    if (ey == EY - 1) m &= ~0xC8u;  // S SW SE
                    if (i & 1) {
                        if (m & 0x10u) S.edge[3][c + edge_off(4)] = f[u].x;
                        if (m & 0x20u) S.edge[2][c + edge_off(5)] = f[u].y;
                        if (m & 0x40u) S.edge[3][c] = f[u].z;
                        if (m & 0x80u) S.edge[2][c] = f[u].w;
                    } else {
                        if (m & 0x01u) S.edge[0][c] = f[u].x;
                        if (m & 0x02u) S.edge[1][c + edge_off(1)] = f[u].y;
                        if (m & 0x04u) S.edge[0][c + edge_off(2)] = f[u].z;
                        if (m & 0x08u) S.edge[1][c] = f[u].w;
                    }
                }
            }
        }
    }

    // ---- up to kHaloLevels levels, by the warps that hold bits
    int cur = 0;
    // the cells of this thread's word that level `cur` makes ready
    auto next_ready = [&](const uint32_t (&nd)[8]) -> uint32_t {
        uint32_t ready = open & ~fin;
        if (!ready) return 0u;
        const uint32_t* d = S.done[cur] + fw;
        const uint32_t ul = d[-FP - 1], uc = d[-FP], ur = d[-FP + 1];
        const uint32_t ml = d[-1], mr = d[1];
        const uint32_t dl = d[FP - 1], dc = d[FP], dr = d[FP + 1];
        // bit x of each: the neighbour of cell x in that direction is done
        ready &= (nd[0] | __funnelshift_r(fin, mr, 1)) & (nd[1] | uc);
        ready &= (nd[2] | __funnelshift_l(ml, fin, 1)) & (nd[3] | dc);
        ready &= (nd[4] | __funnelshift_r(uc, ur, 1)) & (nd[5] | __funnelshift_l(ul, uc, 1));
        ready &= (nd[6] | __funnelshift_l(dl, dc, 1)) & (nd[7] | __funnelshift_r(dc, dr, 1));
        return ready;
    };
    if (warp < HaloGeo::OW) {
        constexpr int NO = HaloGeo::OW * 32;
        int l = 0;
        bar_n(1, NO);  // the done bits of level 0
        for (; l < kHaloLevels; ++l) {
            const uint32_t ready = next_ready(ndep);
            fin |= ready;
            cur ^= 1;
            if (owner) {
                S.done[cur][fw] = fin;
                S.found[l][tid] = ready;
            }
            if (!bar_or(1, NO, ready != 0)) break;
        }
        if (tid == 0) {
            S.nlev = l;
            S.cnt = 0;
        }
    }
    __syncthreads();
    const int nlev = S.nlev;
    // the masks move to the receiver bytes' place (needed only if there are
    // more levels)
    if (owner && nlev == kHaloLevels) {
#pragma unroll
        for (int k = 0; k < 8; ++k) dep_s[k * NWD] = ndep[k];
    }
    // ---- initial values (rain forward; gbar adjoint): loads
    constexpr int NV = (HaloGeo::NE + NT - 1) / NT;
    df vi[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        const int c = tid + u * NT, ey = c / EX, ex = c - ey * EX;
        const int64_t gx = ox + ex + 1, gy = oy + ey + 1, gi = gy * P.nx + gx;
        vi[u] = df_make(0.0f);
        if (c >= HaloGeo::NE || !(interior || (gx >= 0 && gy >= 0 && gx < P.nx && gy < P.ny))) continue;
        if constexpr (!HM::kAdj) {
            vi[u].hi = P.init ? rd_in(P.init, P, gi, 8) : 1.0f;
        } else if (P.init) {
            vi[u].hi = rd_in(P.init, P, gi, 8);
        } else if (!S.dm[c]) {
            // L = sum over sinks of w^2: gbar = 2 w at a sink, 0 elsewhere
            // (doubled below, so that no load is waited for here)
            vi[u].hi = rd_in(P.wf, P, gi, 9);
            if (P.wf_lo) vi[u].lo = rd_in(P.wf_lo, P, gi, 10);
        }
    }
    // ---- the levels' cells, packed: a warp per level (two at most) counts,
    // the counts become list positions, the warp writes
    {
        constexpr int LW = kHaloLevels / NW, WPL = (NWD + 31) / 32;
        static_assert(LW * NW == kHaloLevels, "levels per warp");
        int mine[LW];
#pragma unroll
        for (int q = 0; q < LW; ++q) {
            const int l = warp + q * NW;
            int n = 0;
            if (l < nlev) {
#pragma unroll
                for (int j = 0; j < WPL; ++j)
                    if (j * 32 + lane < NWD) n += __popc(S.found[l][j * 32 + lane]);
            }
            mine[q] = n;
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) S.lev[l + 1] = n;
        }
        __syncthreads();
        if (warp == 0) {
            int base = 0, wide = 0, narrow = 0;
#pragma unroll
            for (int q = 0; q < kHaloLevels / 32; ++q) {
                const int n = S.lev[32 * q + lane + 1];
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += u;
                }
                S.lev[32 * q + lane + 1] = base + incl;
                base += __shfl_sync(0xffffffffu, incl, 31);
                const unsigned bw = __ballot_sync(0xffffffffu, n > kHaloMid), bn = __ballot_sync(0xffffffffu, n > 32);
                if (bw) wide = 32 * q + 32 - __clz(bw);
                if (bn) narrow = 32 * q + 32 - __clz(bn);
            }
            if (lane == 0) {
                S.lev[0] = 0;
                S.wide = wide;
                S.narrow = narrow;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < LW; ++q) {
            const int l = warp + q * NW;
            if (l >= nlev) break;
            int incl = mine[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            int pos = S.lev[l] + incl - mine[q];
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                const int w = j * 32 + lane, y = w / WR;
                if (w >= NWD) break;
                const int e = y << 7 | (w - y * WR) * 32;
                for (uint32_t m = S.found[l][w]; m; m &= m - 1) S.list[pos++] = (uint16_t)(e + __ffs(m) - 1);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        const int c = tid + u * NT;
        if (c >= HaloGeo::NE) break;
        // a cell without dependencies is final: as a sum without terms leaves it
        if (HM::kAdj && !S.dm[c]) {
            if (!P.init) vi[u] = {__fmul_rn(2.0f, vi[u].hi), __fmul_rn(2.0f, vi[u].lo)};
            vi[u] = df_norm(vi[u].hi, vi[u].lo);
        }
        S.v[c] = make_float2(vi[u].hi, vi[u].lo);
    }
    __syncthreads();
    // ---- the levels in order: all warps, then half of them, then one as
    // the levels shrink (the barrier among fewer warps is the shorter: halves at 128,
    // 256, 384 and 512 cells 209, 206, 204 and 203 us at 2048^2)
    auto solve = [&](int c, uint32_t m) {
        float f[8];
        df vv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            f[k] = 0.0f;
            vv[k] = df_make(0.0f);
            if (!((m >> k) & 1u)) continue;
            const float2 a = S.v[c + offy(k) * EX + offx(k)];
            vv[k] = {a.x, a.y};
            if constexpr (HM::kMfd) f[k] = S.edge[edge_plane(k)][c + edge_off(k)];
            else f[k] = 1.0f;
        }
        const float2 o = S.v[c];
        const df v = df_dot8(df{o.x, o.y}, f, vv);
        S.v[c] = make_float2(v.hi, v.lo);
    };
    auto cell_of = [&](int i) {
        const int x = S.list[i];
        return (x >> 7) * EX + (x & 127);
    };
    {
        int l = 0;
        for (int stage = 0; stage < 3; ++stage) {
            const int nthr = stage == 0 ? NT : stage == 1 ? kHaloMid : 32;
            const int end = stage == 0 ? S.wide : stage == 1 ? S.narrow : nlev;
            if (tid >= nthr) break;
            int e = -1;
            uint32_t dm = 0;
            auto load = [&](int lv) {  // this thread's cell of level lv
                e = -1;
                if (lv >= end) return;
                const int i = S.lev[lv] + tid;
                if (i >= S.lev[lv + 1]) return;
                e = cell_of(i);
                dm = S.dm[e];
            };
            load(l);
            for (; l < end; ++l) {
                if (e >= 0) {
                    solve(e, dm);
                    for (int i = S.lev[l] + tid + nthr; i < S.lev[l + 1]; i += nthr) {
                        const int c = cell_of(i);
                        solve(c, S.dm[c]);
                    }
                }
                load(l + 1);
                if (nthr == NT) __syncthreads();
                else if (nthr == kHaloMid) bar_n(2, kHaloMid);
                else __syncwarp();
            }
        }
    }
    __syncthreads();
    // ---- chains longer than kHaloLevels (not on rough terrain): level by level
    while (nlev == kHaloLevels) {
        if (warp < HaloGeo::OW) {
            uint32_t nd[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) nd[k] = owner ? dep_s[k * NWD] : 0u;
            const uint32_t ready = next_ready(nd);
            fin |= ready;
            cur ^= 1;
            if (owner) S.done[cur][fw] = fin;
            if (ready) {
                int pos = atomicAdd(&S.cnt, __popc(ready));
                for (uint32_t m = ready; m; m &= m - 1) S.list[pos++] = (uint16_t)(wy << 7 | (wx + __ffs(m) - 1));
            }
        }
        __syncthreads();
        const int n = S.cnt;
        if (n == 0) break;
        for (int i = tid; i < n; i += NT) {
            const int c = cell_of(i);
            solve(c, S.dm[c]);
        }
        __syncthreads();
        if (tid == 0) S.cnt = 0;
        __syncthreads();
    }
    if (owner) S.done[0][fw] = fin;
    __syncthreads();

    // ---- inner tile: publish final cells, list the others as global (every
    // lane of a warp runs the same steps, as mark_global_cells needs).  The
    // trailing word goes out for every cell: 4 bytes more per cell cost less
    // than finding the cells the global phase will pull from.
    const uint32_t* fd = S.done[0];
    unsigned done = 0;
    for (int ly = warp; ly < TY; ly += NW) {
        const int64_t gy = y0 + ly;
        for (int lx0 = 0; lx0 < TX; lx0 += 32) {  // warp-uniform steps
            const int lx = lx0 + lane;
            const int64_t gx = x0 + lx;
            const bool in_grid = lx < TX && gx < P.nx && gy < P.ny;
            const int ex = lx + H, ey = ly + H;
            const int64_t gi = gy * P.nx + gx;
            const bool fin1 = in_grid && ((fd[(ey + 1) * FP + (ex >> 5) + 1] >> (ex & 31)) & 1u);
            mark_global_cells(P, G, gi, pid, in_grid && !fin1);
            if (!fin1) continue;
            ++done;
            const float2 a = S.v[ey * EX + ex];
            wr_f(P.out_hi, P, gi, final_word(a.x), 27);
            wr_f(P.out_lo, P, gi, a.y, 28);
        }
    }
    done = __reduce_add_sync(0xffffffffu, done);
    if (lane == 0 && done) atomicAdd(&S.ndone, done);
    __syncthreads();
    if (tid == 0 && S.ndone) atomicAdd(&G->done_cells, (unsigned long long)S.ndone);
}

template <Mode M, bool BATCH>
cudaError_t launch_local_halo(const Prob& P, EngineGlobals* G, const Prob* probs,
                              const int64_t* prefix, int nprob, int64_t tiles, cudaStream_t s) {
    constexpr size_t sm = sizeof(SmemHalo<HaloMode<M>::kMfd>);
    static std::atomic<unsigned long long> set_on{0};
    cudaError_t e = smem_limit_once(k_local_halo<M, BATCH>, sm, set_on);
    if (e != cudaSuccess) return e;
    if (tiles > 0)
        k_local_halo<M, BATCH><<<(unsigned)tiles, kHaloNT, sm, s>>>(P, G, probs, prefix, nprob);
    return cudaGetLastError();
}

template <Mode M>
cudaError_t launch_halo_single(const Prob& P, EngineGlobals* G, cudaStream_t s) {
    const int64_t tiles = ((P.nx + kHaloTX - 1) / kHaloTX) * ((P.ny + kHaloTY - 1) / kHaloTY);
    cudaError_t e = launch_local_halo<M, false>(P, G, nullptr, nullptr, 1, tiles, s);
    if (e != cudaSuccess) return e;
    return launch_global<M, true, false>(nullptr, P, G, (unsigned long long)(P.nx * P.ny), s);
}

}  // namespace

// MFD forward accumulation: halo-tile local phase + global phase.
cudaError_t launch_mfd_forward(const Prob& P, EngineGlobals* G, cudaStream_t s) {
    return launch_halo_single<Mode::FwdMfd>(P, G, s);
}

// Adjoint (D8 or MFD): halo-tile local phase + global phase.
cudaError_t launch_adjoint(bool mfd, const Prob& P, EngineGlobals* G, cudaStream_t s) {
    return mfd ? launch_halo_single<Mode::AdjMfd>(P, G, s) : launch_halo_single<Mode::AdjD8>(P, G, s);
}

// Batched MFD forward: the CTAs of all problems' tiles in one launch, then one
// global phase.
cudaError_t launch_mfd_forward_batch(const Prob* probs, const int64_t* prefix, int nprob,
                                     int64_t tiles, unsigned long long total_cells,
                                     EngineGlobals* G, cudaStream_t s) {
    Prob none{};
    cudaError_t e = launch_local_halo<Mode::FwdMfd, true>(none, G, probs, prefix, nprob, tiles, s);
    if (e != cudaSuccess) return e;
    return launch_global<Mode::FwdMfd, true, false>(probs, none, G, total_cells, s);
}

}  // namespace fr
