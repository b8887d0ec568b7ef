// fr_fill.cu -- depression filling, the step before the path: the paper routes
// a depression-filled DEM (Sec. 4).  The filled surface F is the least F >= z
// that keeps every edge cell at its own elevation and gives every interior
// cell a neighbour (of 8) lower by at least one fp32 step, i.e. the solution of
//     F_c = z_c                                             (edge cells)
//     F_c = max(z_c, succ(min over neighbours n of F_n))    (elsewhere),
// succ(x) being the next fp32 value above x.  D8 routing on F has sinks only
// on the edge.
//
// GPU form (Planchon-Darboux relaxation): F starts at z on the edge and +inf
// inside; every update lowers a cell to the right-hand side above, which is
// never below the solution, so the updates can run in any order and the
// iteration ends exactly at the solution.  The host repeats sweeps until one
// changes nothing: then every cell meets its equation, and the surface is the
// unique solution, bit for bit.
//
// A sweep here is one launch over 64x64 tiles (up to eight of them are one sweep
// of the caller's).  A tile that has work loads F and z
// with a one-cell ring into shared memory as integers ordered like the floats
// (succ is then +1) and relaxes them in directional passes: warps run down,
// up, right and left at once (two per direction, half the lines each), each
// carrying a row (column) of values in registers from line to line, a cell
// taking the least of the three cells of the previous line.  A pass settles
// every path that is monotone in one of the four directions, where a pass
// that relaxes each cell once moves a path by one cell: that took up to 120
// passes per visit of a 64x32 tile, 22 on average, against about 3 here.  A
// visit stops after `passes` passes (a tile still moving runs again in the
// next sweep): the slowest tile of a sweep holds back all others.  Measured at
// 4096^2: 2 passes 2.42 ms, 3 passes 2.61, 4 passes 2.86; one warp per
// direction 2.44 and four 3.97 ms.
//
// Which tiles run: a tile whose new boundary value lowers a ring cell, by the
// ring's values as it loaded them (never below the current ones), flags that
// cell's tile for the next sweep.  Terrain that stands above its neighbours'
// water flags nobody, so only tiles on the moving front run.  Rings read
// neighbouring tiles that are being rewritten in the same sweep; either value
// is an upper bound.  The first sweep reads no F: it writes the start values.
//
// What bounds it: about 45 000 visits of 4096 tiles in 50 sweeps at 4096^2,
// each some 28 K warp instructions (2.1 per SM and cycle), and in the first and
// last sweeps the latency of one visit (about 20 us).  4096^2 (beta 2, tilt
// 0.01) took 13.3 ms with the cell-by-cell relaxation and takes 2.4 ms; 8192^2
// without tilt 68 ms and 17 ms.
#include "fr_internal.h"

namespace fr {
namespace {

constexpr int kFT = 64;           // tile side
constexpr int kFSeg = 2;          // warps per direction: each takes kFT / kFSeg lines
constexpr int kFNT = 4 * 32 * kFSeg;
constexpr int kFR = kFT + 2;      // with the ring
constexpr int kFP = kFR + 1;      // row pitch: odd, so rows and columns are both free of bank conflicts
constexpr int kInf = 0x7f800000;  // key of +inf, above every key in use

// Order-preserving integer of a float: one more is the next float up; both
// zeros are 0.
__device__ __forceinline__ int fkey(float x) {
    const int b = __float_as_int(x);
    return b >= 0 ? b : -(b & 0x7fffffff);
}
__device__ __forceinline__ float funkey(int k) {
    return __int_as_float(k >= 0 ? k : (int)(0x80000000u | (unsigned)-k));
}

struct FillSmem {
    int f[kFR * kFP], z[kFR * kFP];
    unsigned flags;
};

// One pass of this warp along its direction: lines off + step, off + 2 step,
// ... with cells at lane strides ls; line 0 is the ring's.  Lane l holds cells
// 2 l and 2 l + 1 of a line, the next line's loads run ahead of the chain
// through the shuffles.  Returns whether a cell was lowered.  The stores need
// no atomics: a value that two warps lower at once ends at one of the two, and
// the warp that found the other lowers it again in the next pass.
__device__ __forceinline__ bool fill_pass(FillSmem& S, int off, int step, int ls) {
    const int l = threadIdx.x & 31;
    const int oa = (2 * l + 1) * ls, ob = oa + ls;
    const int oe = l == 31 ? (kFR - 1) * ls : 0;  // the line's ends, for lanes 31 and 0
    volatile int* f = S.f;
    int pa = f[off + oa], pb = f[off + ob], pe = f[off + oe];
    int moved = 0;
    int at = off + step;
    int fa = f[at + oa], fb = f[at + ob], fe = f[at + oe], za = S.z[at + oa], zb = S.z[at + ob];
#pragma unroll 4
    for (int s = 0; s < kFT / kFSeg; ++s) {
        // the line after this one (the last step's read is unused)
        const int nx = at + step;
        const int na = f[nx + oa], nb = f[nx + ob], ne = f[nx + oe];
        const int nza = S.z[nx + oa], nzb = S.z[nx + ob];
        int lf = __shfl_up_sync(0xffffffffu, pb, 1), rt = __shfl_down_sync(0xffffffffu, pa, 1);
        if (l == 0) lf = pe;
        if (l == 31) rt = pe;
        const int pm = min(pa, pb);
        const int va = min(fa, max(za, min(pm, lf) + 1)), vb = min(fb, max(zb, min(pm, rt) + 1));
        if (va < fa) f[at + oa] = va;
        if (vb < fb) f[at + ob] = vb;
        moved |= (va - fa) | (vb - fb);
        pa = va;
        pb = vb;
        pe = fe;
        at = nx;
        fa = na;
        fb = nb;
        fe = ne;
        za = nza;
        zb = nzb;
    }
    return moved != 0;
}

// Boundary cell b of a tile, 0 <= b < 4 kFT - 4, in ring coordinates.
__device__ __forceinline__ void fill_boundary(int b, int& x, int& y) {
    if (b < kFT) {
        x = b + 1;
        y = 1;
    } else if (b < 2 * kFT) {
        x = b - kFT + 1;
        y = kFT;
    } else {
        b -= 2 * kFT;
        y = (b >> 1) + 2;
        x = (b & 1) ? kFT : 1;
    }
}

template <bool FIRST>
__global__ void __launch_bounds__(kFNT) k_fill_sweep(const float* __restrict__ z, int64_t nx,
                                                     int64_t ny, float* F, uint8_t* act,
                                                     uint8_t* act_next, int passes, unsigned long long* changed) {
    __shared__ FillSmem S;
    if (!FIRST && !act[blockIdx.x]) return;
    const int tiles_x = (int)((nx + kFT - 1) / kFT);
    const int tiles_y = (int)((ny + kFT - 1) / kFT);
    const int ty = (int)blockIdx.x / tiles_x, tx = (int)blockIdx.x - ty * tiles_x;
    const int64_t x0 = (int64_t)tx * kFT, y0 = (int64_t)ty * kFT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // extent inside the grid, in ring coordinates: cells [1, ex] x [1, ey]
    const int ex = (int)(nx - x0 < kFT ? nx - x0 : kFT), ey = (int)(ny - y0 < kFT ? ny - y0 : kFT);
    // no cell of the tile or its ring on the grid's edge
    const bool inner = x0 >= 2 && y0 >= 2 && x0 + kFT + 1 < nx && y0 + kFT + 1 < ny;
    if (FIRST && inner) {
        for (int y = warp; y < kFT; y += kFNT / 32) {
            float* row = F + (y0 + y) * nx + x0;
            row[lane] = __int_as_float(kInf);
            row[lane + 32] = __int_as_float(kInf);
        }
        return;
    }
    // ---- load: the 66 ring rows in groups of four cells (and the two ring
    // columns apart), several groups' loads in flight
    const bool vec = inner && (nx & 3) == 0 && (((uintptr_t)F | (uintptr_t)z) & 15) == 0;
    // keys of grid cell (gx, gy) from its values
    auto keys = [&](int64_t gx, int64_t gy, float zz, float ff, int& zk, int& fk) {
        const bool edge = !inner && (gx == 0 || gy == 0 || gx == nx - 1 || gy == ny - 1);
        zk = fkey(zz);
        fk = FIRST ? kInf : fkey(ff);
        if (!(zz == zz)) zk = edge ? kInf : (int)0x80000000;  // a NaN (outside the contract) bounds nothing
        if (edge) fk = zk;                                    // F = z stays
    };
    auto in_grid = [&](int64_t gx, int64_t gy) { return inner || (gx >= 0 && gy >= 0 && gx < nx && gy < ny); };
    auto put = [&](int r, int x, float zz, float ff) {  // ring coordinates
        const int64_t gx = x0 + x - 1, gy = y0 + r - 1;
        int zk = kInf, fk = kInf;  // off the grid: never moves, lowers nobody
        if (in_grid(gx, gy)) keys(gx, gy, zz, ff, zk, fk);
        S.z[r * kFP + x] = zk;
        S.f[r * kFP + x] = fk;
    };
    {
        // ring columns: one cell of each a thread
        const int r = threadIdx.x;
        float cz[2] = {0.f, 0.f}, cf[2] = {0.f, 0.f};
        if (r < kFR) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int64_t gx = s ? x0 + kFT : x0 - 1, gy = y0 + r - 1;
                if (!in_grid(gx, gy)) continue;
                cz[s] = __ldg(z + gy * nx + gx);
                if (!FIRST) cf[s] = __ldcg(F + gy * nx + gx);
            }
        }
        constexpr int U = 3, NQ = kFR * (kFT / 4), NB = (NQ + kFNT - 1) / kFNT;
        for (int b0 = 0; b0 < NB; b0 += U) {
            float4 zv[U], fv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = (b0 + u) * kFNT + threadIdx.x;
                zv[u] = fv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i >= NQ) continue;
                const int64_t gy = y0 + (i >> 4) - 1, gx = x0 + 4 * (i & 15), g = gy * nx + gx;
                if (vec) {
                    zv[u] = __ldg(reinterpret_cast<const float4*>(z + g));
                    if (!FIRST) fv[u] = __ldcg(reinterpret_cast<const float4*>(F + g));
                } else {
                    const bool row = in_grid(x0, gy);
                    const int n = row ? (int)(nx - gx < 4 ? nx - gx : 4) : 0;  // cells of the group in the grid
                    if (n > 0) zv[u].x = __ldg(z + g);
                    if (n > 1) zv[u].y = __ldg(z + g + 1);
                    if (n > 2) zv[u].z = __ldg(z + g + 2);
                    if (n > 3) zv[u].w = __ldg(z + g + 3);
                    if (!FIRST) {
                        if (n > 0) fv[u].x = __ldcg(F + g);
                        if (n > 1) fv[u].y = __ldcg(F + g + 1);
                        if (n > 2) fv[u].z = __ldcg(F + g + 2);
                        if (n > 3) fv[u].w = __ldcg(F + g + 3);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = (b0 + u) * kFNT + threadIdx.x;
                if (i >= NQ) continue;
                const int r = i >> 4, x = 4 * (i & 15) + 1;
                put(r, x, zv[u].x, fv[u].x);
                put(r, x + 1, zv[u].y, fv[u].y);
                put(r, x + 2, zv[u].z, fv[u].z);
                put(r, x + 3, zv[u].w, fv[u].w);
            }
        }
        if (r < kFR) {
            put(r, 0, cz[0], cf[0]);
            put(r, kFR - 1, cz[1], cf[1]);
        }
    }
    if (threadIdx.x == 0) S.flags = 0;
    __syncthreads();
    // this record serves the sweep after next again; cleared behind the barrier,
    // when every thread of the block has read it
    if (!FIRST && threadIdx.x == 0) act[blockIdx.x] = 0;
    // the boundary's values as loaded
    constexpr int NB = 4 * kFT - 4;
    constexpr int NQB = (NB + kFNT - 1) / kFNT;  // boundary cells a thread
    int old[NQB], rb[NQB];
#pragma unroll
    for (int q = 0; q < NQB; ++q) {
        int x = 1, y = 1;
        const int b = threadIdx.x + q * kFNT;
        if (b < NB) fill_boundary(b, x, y);
        rb[q] = y * kFP + x;
        old[q] = S.f[rb[q]];
    }
    __syncthreads();
    // direction (down, up, right, left) and segment of this warp
    const int dir = warp & 3, seg = warp >> 2;
    const int ls = dir < 2 ? 1 : kFP, ds = dir < 2 ? kFP : 1, step = (dir & 1) ? -ds : ds;
    const int off = ((dir & 1) ? (kFR - 1) * ds : 0) + seg * (kFT / kFSeg) * step;
    bool any = false, moving = true;
    for (int pass = 0; pass < passes && moving; ++pass) {
        moving = __syncthreads_or(fill_pass(S, off, step, ls));
        any |= moving;
    }
    if (!FIRST && !any) return;
    // ---- flag the tiles whose ring cells the new boundary lowers (bit 3 dy +
    // dx + 4), and this one if it was still moving
    unsigned fl = moving ? 1u << 4 : 0u;
#pragma unroll
    for (int q = 0; q < NQB; ++q) {
        if (threadIdx.x + q * kFNT >= NB) continue;
        const int v = S.f[rb[q]];
        if (v >= old[q]) continue;
        const int y = rb[q] / kFP, x = rb[q] - y * kFP;
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int xn = x + dx, yn = y + dy;
                const int bx = xn < 1 ? -1 : xn > kFT ? 1 : 0, by = yn < 1 ? -1 : yn > kFT ? 1 : 0;
                if (!(bx | by)) continue;
                const int j = yn * kFP + xn;
                if (max(S.z[j], v + 1) < S.f[j]) fl |= 1u << (3 * by + bx + 4);
            }
    }
    fl = __reduce_or_sync(0xffffffffu, fl);
    if (lane == 0 && fl) atomicOr(&S.flags, fl);
    __syncthreads();
    // ---- write the tile back: edge cells keep z (written by the first sweep),
    // unraised cells their own bits
    for (int y = warp + 1; y <= ey; y += kFNT / 32) {
        const int64_t gy = y0 + y - 1;
        for (int x = lane + 1; x <= ex; x += 32) {
            const int64_t gx = x0 + x - 1, gi = gy * nx + gx;
            const int v = S.f[y * kFP + x];
            if (!inner && (gx == 0 || gy == 0 || gx == nx - 1 || gy == ny - 1)) {
                if (FIRST) F[gi] = z[gi];
            } else {
                F[gi] = v == 0 && S.z[y * kFP + x] == 0 ? z[gi] : funkey(v);
            }
        }
    }
    if (threadIdx.x < 9 && ((S.flags >> threadIdx.x) & 1u)) {
        const int uy = ty + (int)threadIdx.x / 3 - 1, ux = tx + (int)threadIdx.x % 3 - 1;
        if (ux >= 0 && uy >= 0 && ux < tiles_x && uy < tiles_y) act_next[uy * tiles_x + ux] = 1;
    }
    if (threadIdx.x == 0 && any) atomicAdd(changed, 1ull);
}

}  // namespace

int64_t fill_tiles(int64_t nx, int64_t ny) {
    return ((nx + kFT - 1) / kFT) * ((ny + kFT - 1) / kFT);
}

cudaError_t fill_sweep(const float* z, int64_t nx, int64_t ny, float* F, uint8_t* act,
                       uint8_t* act_next, bool first, int passes, unsigned long long* changed,
                       cudaStream_t s) {
    const unsigned grid = (unsigned)fill_tiles(nx, ny);
    if (first)
        k_fill_sweep<true><<<grid, kFNT, 0, s>>>(z, nx, ny, F, act, act_next, passes, changed);
    else
        k_fill_sweep<false><<<grid, kFNT, 0, s>>>(z, nx, ny, F, act, act_next, passes, changed);
    return cudaGetLastError();
}

}  // namespace fr
