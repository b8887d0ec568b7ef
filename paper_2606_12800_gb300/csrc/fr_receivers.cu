// fr_receivers.cu -- local flow routing kernels (paper Sec. 2.1 for D8,
// App. A for the multi-receiver split).
//
// D8 codes come from the TMA-pipelined kernel, or by warps marching down strips
// where TMA cannot address the grid; their donor counts from the codes; donor
// counts of the slope split, D-infinity and batched slope splits from blocks that
// stage a (TY+4) x (TX+4) elevation tile (two-cell halo) in shared memory, which
// outside the grid holds +inf, never strictly lower than anything.
#include <cmath>
#include <type_traits>

#include "fr_internal.h"
#include "fr_tma.cuh"

namespace fr {

namespace {

constexpr int RTX = kRecvTileX;  // receiver tile width (cells)
constexpr int RTY = kRecvTileY;  // receiver tile height
constexpr int RNT = 256;  // threads
constexpr int HX = RTX + 4, HY = RTY + 4;
constexpr int RX = RTX + 2, RY = RTY + 2;

__device__ __forceinline__ void load_z_tile(float* zs, const float* __restrict__ z, int64_t nx,
                                            int64_t ny, int64_t x0, int64_t y0) {
    const float inf = __int_as_float(0x7f800000);
    for (int i = threadIdx.x; i < HX * HY; i += RNT) {
        int ly = i / HX, lx = i - ly * HX;
        int64_t gx = x0 + lx - 2, gy = y0 + ly - 2;
        float v = inf;
        if (gx >= 0 && gy >= 0 && gx < nx && gy < ny && FR_OK(gy * nx + gx, nx * ny, 40))
            v = __ldg(z + gy * nx + gx);
        zs[i] = v;
    }
}

__device__ __forceinline__ void tile_origin(int64_t nx, int64_t& x0, int64_t& y0) {
    const int64_t tiles_x = (nx + RTX - 1) / RTX;
    const int64_t ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
    x0 = tx * RTX;
    y0 = ty * RTY;
}

constexpr int kStrip = 4;  // rows of a strip (a tile is RTY / kStrip strips)

// D8 codes of RTX x kStrip cells by one warp, without shared memory or
// barriers: lane l holds columns l, l + 32, l + 64 and l + 96 and marches down
// the rows with three rows in registers, neighbours along a row coming by
// shuffles.  For grids TMA cannot address and for batches: every load is
// coalesced whatever the rows' alignment.  Bound by instruction issue.  1537x2603
// 23 us by staged tiles, 16 us; batch of 32 tiles, 18 M cells, 160 us by staged
// tiles of a block, 73 us (strips of 16 rows loaded as they go 116 us).
// BITS: the codes also go to `bits` (rows of kBitsPitch bytes), one bit each.
constexpr int kBitsPitch = RTX + 8;
__device__ __forceinline__ uint8_t code_bit(uint32_t code) { return (uint8_t)(code < 8 ? 1u << code : 0u); }

template <bool LOWEST, bool D4, bool INTERIOR, bool BITS>
__device__ __forceinline__ void recv_d8_strip_t(const float* __restrict__ z, int64_t nx, int64_t ny,
                                              float c_orth, float c_diag, bool edge_route,
                                              uint8_t* __restrict__ dir, int64_t x0, int64_t y0, uint8_t* bits) {
    static_assert(RTX == 128, "four columns a lane");
    const float inf = __int_as_float(0x7f800000);
    const int lane = threadIdx.x & 31;
    struct Row {
        float v[4], e;  // the lane's cells; lanes 0 and 31: the cell beside the strip
    };
    auto load = [&](int64_t gy, Row& w) {
        const bool row = INTERIOR || (gy >= 0 && gy < ny);
        const float* p = z + gy * nx + x0 + lane;
#pragma unroll
        for (int g = 0; g < 4; ++g) w.v[g] = INTERIOR || (row && x0 + lane + 32 * g < nx) ? __ldg(p + 32 * g) : inf;
        w.e = inf;
        if ((lane == 0 || lane == 31) && row && (INTERIOR || (lane ? x0 + RTX < nx : x0 > 0)))
            w.e = __ldg(p + (lane ? 97 : -1));
    };
    struct Win {
        float l[4], c[4], r[4];
    };
    auto spread = [&](const Row& w, Win& n) {
        float up[4], dn[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            up[g] = __shfl_sync(0xffffffffu, w.v[g], (lane + 31) & 31);
            dn[g] = __shfl_sync(0xffffffffu, w.v[g], (lane + 1) & 31);
            n.c[g] = w.v[g];
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            n.l[g] = lane ? up[g] : g ? up[g > 0 ? g - 1 : 0] : w.e;
            n.r[g] = lane < 31 ? dn[g] : g < 3 ? dn[g < 3 ? g + 1 : 3] : w.e;
        }
    };
    Row rows[kStrip + 2];  // all loads issued before the first is used
#pragma unroll
    for (int r = 0; r < kStrip + 2; ++r) load(y0 + r - 1, rows[r]);
    Win a, b, c;
    spread(rows[0], a);
    spread(rows[1], b);
#pragma unroll
    for (int r = 0; r < kStrip; ++r) {
        const int64_t gy = y0 + r;
        if (!INTERIOR && gy >= ny) break;
        spread(rows[r + 2], c);
        uint32_t codes[4];
        float m[4];
        struct Around {
            float z[8];
        };
        auto around = [&](int g) -> Around {
            return {{b.r[g], a.c[g], b.l[g], c.c[g], D4 ? inf : a.r[g], D4 ? inf : a.l[g], D4 ? inf : c.l[g],
                     D4 ? inf : c.r[g]}};
        };
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            codes[g] = d8_code_max<LOWEST>(b.c[g], around(g).z, c_orth, c_diag, m[g]);
            if (!INTERIOR && x0 + lane + 32 * g >= nx) m[g] = 1.0f;  // off the grid: no key
        }
        if (d8_unsure<LOWEST>(m, [&](int g) { return d8_any_lower(b.c[g], around(g).z); })) {
#pragma unroll 1
            for (int g = 0; g < 4; ++g) {
                const int64_t gx = x0 + lane + 32 * g;
                if (gx >= nx) break;
                float zn[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int64_t xn = gx + offx(k), yn = gy + offy(k);
                    zn[k] = (k >= 4 && D4) || xn < 0 || yn < 0 || xn >= nx || yn >= ny ? inf : __ldg(z + yn * nx + xn);
                }
                const uint32_t code = d8_code(__ldg(z + gy * nx + gx), zn, c_orth, c_diag, LOWEST);
                codes[0] = g == 0 ? code : codes[0];
                codes[1] = g == 1 ? code : codes[1];
                codes[2] = g == 2 ? code : codes[2];
                codes[3] = g == 3 ? code : codes[3];
            }
        }
        uint8_t* o = dir + gy * nx + x0 + lane;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int64_t gx = x0 + lane + 32 * g;
            if (!INTERIOR) {
                if (gx >= nx) continue;
                if (!edge_route && is_edge(gx, gy, nx, ny)) codes[g] = kSink;
            }
            o[32 * g] = (uint8_t)codes[g];
            if (BITS) bits[r * kBitsPitch + lane + 32 * g] = code_bit(codes[g]);
        }
        a = b;
        b = c;
    }
}

template <bool LOWEST, bool D4, bool BITS = false>
__device__ __forceinline__ void recv_d8_strip(const float* __restrict__ z, int64_t nx, int64_t ny,
                                              float c_orth, float c_diag, bool edge_route,
                                              uint8_t* __restrict__ dir, int64_t x0, int64_t y0,
                                              uint8_t* bits = nullptr) {
    if (x0 >= 1 && y0 >= 1 && x0 + RTX + 1 <= nx && y0 + kStrip + 1 <= ny)
        recv_d8_strip_t<LOWEST, D4, true, BITS>(z, nx, ny, c_orth, c_diag, edge_route, dir, x0, y0, bits);
    else
        recv_d8_strip_t<LOWEST, D4, false, BITS>(z, nx, ny, c_orth, c_diag, edge_route, dir, x0, y0, bits);
}

// Codes and donor counts: a strip per warp, eight strips to a block, the codes
// also as bits in shared memory, with the ring around the block's tile (its codes
// cell by cell); a donor test is then a shift and a mask for four cells.
// Codes and counts of 4096x8192: 320 us by blocks that chose each cell of a staged
// tile and ring in turn, 183 with four-cell windows there, 142 now; 160x192 15, 13
// and 10 us, 1023x1025 21, 17 and 13 (codes first and counts in a second kernel: 143,
// 16 and 18).
constexpr int kCountRows = kStrip * RNT / 32;

template <bool LOWEST, bool D4>
__global__ void __launch_bounds__(RNT) k_receivers_d8_indeg(const float* __restrict__ z, int64_t nx,
                                                            int64_t ny, float c_orth, float c_diag,
                                                            uint32_t flags, uint8_t* __restrict__ dir,
                                                            uint8_t* __restrict__ indeg) {
    // cell (lx, ly) of the tile at (ly + 1) * kBitsPitch + lx + 4
    __shared__ alignas(4) uint8_t bits[(kCountRows + 2) * kBitsPitch];
    const int64_t tiles_x = (nx + RTX - 1) / RTX;
    const int64_t ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
    const int64_t x0 = tx * RTX, y0 = ty * kCountRows;
    const bool edge_route = flags & kEdgeRoute;
    for (int i = threadIdx.x; i < (int)sizeof(bits) / 4; i += RNT) reinterpret_cast<uint32_t*>(bits)[i] = 0u;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (y0 + kStrip * warp < ny)
        recv_d8_strip<LOWEST, D4, true>(z, nx, ny, c_orth, c_diag, edge_route, dir, x0, y0 + kStrip * warp,
                                        bits + (1 + kStrip * warp) * kBitsPitch + 4);
    for (int i = threadIdx.x; i < 2 * RX + 2 * kCountRows; i += RNT) {
        const int j = i - 2 * RX;
        const int rx = i < 2 * RX ? (i < RX ? i : i - RX) : (j & 1) * (RX - 1);
        const int ry = i < 2 * RX ? (i < RX ? 0 : kCountRows + 1) : 1 + (j >> 1);
        const int64_t gx = x0 + rx - 1, gy = y0 + ry - 1;
        if (gx < 0 || gy < 0 || gx >= nx || gy >= ny || (!edge_route && is_edge(gx, gy, nx, ny))) continue;
        float zn[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int64_t xn = gx + offx(k), yn = gy + offy(k);
            zn[k] = (k >= 4 && D4) || xn < 0 || yn < 0 || xn >= nx || yn >= ny ? __int_as_float(0x7f800000)
                                                                              : __ldg(z + yn * nx + xn);
        }
        bits[ry * kBitsPitch + rx + 3] = code_bit(d8_code(__ldg(z + gy * nx + gx), zn, c_orth, c_diag, LOWEST));
    }
    __syncthreads();
    const bool aligned = (nx & 3) == 0 && ((uintptr_t)indeg & 3) == 0;
    const int64_t gx = x0 + 4 * lane;
    if (gx >= nx) return;
    for (int ly = warp; ly < kCountRows; ly += RNT / 32) {
        const int64_t gy = y0 + ly;
        if (gy >= ny) break;
        const Row3 up = row3(bits + ly * kBitsPitch, lane + 1), mid = row3(bits + (ly + 1) * kBitsPitch, lane + 1);
        const Row3 dn = row3(bits + (ly + 2) * kBitsPitch, lane + 1);
        const uint32_t n = popc_bytes(donor_bits(up, mid, dn));
        uint8_t* o = indeg + gy * nx + gx;
        if (aligned) {
            *reinterpret_cast<uint32_t*>(o) = n;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (gx + q < nx) o[q] = (uint8_t)(n >> (8 * q));
        }
    }
}

// A strip per warp.
template <bool LOWEST, bool D4>
__global__ void __launch_bounds__(RNT) k_receivers_d8(const float* __restrict__ z, int64_t nx,
                                                      int64_t ny, float c_orth, float c_diag,
                                                      uint32_t flags, uint8_t* __restrict__ dir,
                                                      int64_t ntiles) {
    const int64_t t = (int64_t)blockIdx.x * (RNT / 32) + (threadIdx.x >> 5);
    if (t >= ntiles) return;
    const int64_t tiles_x = (nx + RTX - 1) / RTX, ty = t / tiles_x, tx = t - ty * tiles_x;
    recv_d8_strip<LOWEST, D4>(z, nx, ny, c_orth, c_diag, flags & kEdgeRoute, dir, tx * RTX, ty * kStrip);
}

// ---------------------------------------------------------------- TMA path
// D8 codes without donor counts, by a persistent kernel: each CTA walks its
// tiles of TTX x TTY cells, the elevations of a tile plus a one-cell halo
// arriving by TMA into one of TNS shared-memory stages while the previous tiles
// are computed.  The box starts 4 cells left of the tile (its x coordinate a
// multiple of 4, as TMA requires), so it is TTX + 8 wide.  The kernel is bound
// by instruction issue and the ALU pipe (the eight directions' keys and their
// selection): 32768^2 2.38 ms with a running best over the directions (66
// instructions per cell), 2.04 ms with d8_code_max (56), 1.92 ms with two rows per
// step and zero keys settled by minima (51).  128x64 tiles in
// two stages (three CTAs per SM) measured 4.7 % faster than 128x32 in three
// (four CTAs per SM) at 32768^2: fewer halo rows and fewer per-tile waits and
// barriers.
constexpr int TTX = 128, TTY = 64, TNS = 2;
constexpr int TBX = TTX + 8, TBY = TTY + 2;
constexpr unsigned kTileBytes = TBX * TBY * 4;
static_assert((TBX * 4) % 16 == 0, "TMA box rows are whole 16-byte units");

// Set when a TMA wait ran out (read and cleared by fr_get_status).
__device__ unsigned g_tma_wait_error;

struct alignas(128) TmaStage {  // TMA writes whole boxes to 128-byte aligned addresses
    float v[TBY * TBX];
};
struct TmaSmem {
    TmaStage buf[TNS];
    alignas(8) uint64_t bar[TNS];
};

template <bool LOWEST, bool D4>
__global__ void __launch_bounds__(256) k_receivers_d8_tma(const __grid_constant__ CUtensorMap zmap,
                                                          int64_t nx, int64_t ny, float c_orth,
                                                          float c_diag, uint32_t flags,
                                                          uint8_t* __restrict__ dir, int64_t ntiles,
                                                          int tiles_x, unsigned long long limit_ns) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    TmaSmem& S = *reinterpret_cast<TmaSmem*>(smem_raw);
    const bool edge_route = flags & kEdgeRoute, aligned = ((uintptr_t)dir & 3) == 0;
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int s = 0; s < TNS; ++s) mbar_init(&S.bar[s], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto issue = [&](int64_t t, int s) {
        const int64_t ty = t / tiles_x, tx = t - ty * tiles_x;
        mbar_expect_tx(&S.bar[s], kTileBytes);
        tma_load_2d(S.buf[s].v, &zmap, (int)(tx * TTX - 4), (int)(ty * TTY - 1), &S.bar[s]);
    };
    if (tid == 0)
        for (int s = 0; s < TNS; ++s) {
            const int64_t t = (int64_t)blockIdx.x + (int64_t)s * gridDim.x;
            if (t < ntiles) issue(t, s);
        }
    const int lane = tid & 31, warp = tid >> 5, qx = 4 * lane;
    int i = 0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
        const int s = i % TNS;
        const bool ok = mbar_wait(&S.bar[s], (unsigned)(i / TNS) & 1u, limit_ns);
        if (__syncthreads_or(!ok)) {
            // the copy did not arrive: report, let the other copies in flight
            // land (bounded), and leave (the whole block takes this branch)
            if (tid == 0) {
                atomicOr(&g_tma_wait_error, 1u);
                for (int k = 1; k < TNS; ++k) {
                    const int64_t tk = t + (int64_t)k * gridDim.x;
                    if (tk < ntiles) mbar_wait(&S.bar[(i + k) % TNS], (unsigned)((i + k) / TNS) & 1u, limit_ns);
                }
            }
            __syncthreads();
            return;
        }
        const int64_t ty = t / tiles_x, tx = t - ty * tiles_x;
        const int64_t x0 = tx * TTX, y0 = ty * TTY;
        const bool interior = x0 >= 1 && y0 >= 1 && x0 + TTX + 1 <= nx && y0 + TTY + 1 <= ny;
        const float* b = S.buf[s].v;
        // two rows per step: they share two of the window's four rows.  Row width
        // and tile origin are multiples of four (the tensor map's condition), so
        // a group of four cells lies in the grid or outside it.
        uint8_t* const out = dir + y0 * nx + x0 + qx;
        const int rows = x0 + qx < nx ? (int)(ny - y0 < TTY ? ny - y0 : TTY) : 0;  // none for a lane off the grid
        for (int r = 2 * warp; r < rows; r += 16) {
            // buffer rows r .. r + 3, columns qx + 3 .. qx + 8 (tile column c
            // sits at buffer column c + 4)
            float w[4][6];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float* row = b + (r + a) * TBX + qx;
                const float4 f = *reinterpret_cast<const float4*>(row + 4);
                w[a][0] = row[3];
                w[a][1] = f.x;
                w[a][2] = f.y;
                w[a][3] = f.z;
                w[a][4] = f.w;
                w[a][5] = row[8];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t codes[4];
                float m[4];
                struct Around {
                    float z[8];
                };
                auto around = [&](int q) -> Around {
                    const int c = q + 1;  // window column of the cell
                    const float inf = __int_as_float(0x7f800000);
                    return {{w[h + 1][c + 1], w[h][c], w[h + 1][c - 1], w[h + 2][c], D4 ? inf : w[h][c + 1],
                             D4 ? inf : w[h][c - 1], D4 ? inf : w[h + 2][c - 1], D4 ? inf : w[h + 2][c + 1]}};
                };
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    codes[q] = d8_code_max<LOWEST>(w[h + 1][q + 1], around(q).z, c_orth, c_diag, m[q]);
                if (d8_unsure<LOWEST>(m, [&](int q) { return d8_any_lower(w[h + 1][q + 1], around(q).z); })) {
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {
                        const float* c = b + (r + h + 1) * TBX + qx + 4 + q;
                        float zn[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            zn[k] = k >= 4 && D4 ? __int_as_float(0x7f800000) : c[offy(k) * TBX + offx(k)];
                        const uint32_t code = d8_code(*c, zn, c_orth, c_diag, LOWEST);
                        codes[0] = q == 0 ? code : codes[0];
                        codes[1] = q == 1 ? code : codes[1];
                        codes[2] = q == 2 ? code : codes[2];
                        codes[3] = q == 3 ? code : codes[3];
                    }
                }
                if (!interior) {
                    if (r + h >= rows) continue;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (!edge_route && is_edge(x0 + qx + q, y0 + r + h, nx, ny)) codes[q] = kSink;
                }
                uint8_t* const o = out + (int64_t)(r + h) * nx;
                if (aligned) {
                    *reinterpret_cast<uint32_t*>(o) =
                        __byte_perm(__byte_perm(codes[0], codes[1], 0x0040), __byte_perm(codes[2], codes[3], 0x0040),
                                    0x5410);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[q] = (uint8_t)codes[q];
                }
            }
        }
        __syncthreads();  // every thread is done with stage s
        if (tid == 0) {
            const int64_t tn = t + (int64_t)TNS * gridDim.x;
            if (tn < ntiles) {
                fence_proxy_async_smem();
                issue(tn, s);
            }
        }
    }
}

template <bool FRAC, bool INDEG>
__device__ __forceinline__ void recv_mfd_tile(const float* __restrict__ z, int64_t nx, int64_t ny,
                                              const MfdConst& mc, uint32_t flags,
                                              uint8_t* __restrict__ mask, float* __restrict__ frac,
                                              uint8_t* __restrict__ indeg, int64_t x0, int64_t y0) {
    __shared__ float zs[HX * HY];
    __shared__ uint8_t ms[RX * RY];
    load_z_tile(zs, z, nx, ny, x0, y0);
    __syncthreads();
    const bool edge_route = flags & kEdgeRoute;
    const int rx0 = INDEG ? 0 : 1, ry0 = INDEG ? 0 : 1;
    const int rw = INDEG ? RX : RTX, rh = INDEG ? RY : RTY;
    for (int i = threadIdx.x; i < rw * rh; i += RNT) {
        int ry = ry0 + i / rw, rx = rx0 + i % rw;
        int64_t gx = x0 + rx - 1, gy = y0 + ry - 1;
        uint8_t m = 0;
        if (gx >= 0 && gy >= 0 && gx < nx && gy < ny &&
            (edge_route || !is_edge(gx, gy, nx, ny))) {
            float zc = zs[(ry + 1) * HX + (rx + 1)];
            if (flags & kDinf) {
                float zn[8], f[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) zn[k] = zs[(ry + 1 + offy(k)) * HX + (rx + 1 + offx(k))];
                m = (uint8_t)dinf_cell(zc, zn, grid_mask8(gx, gy, nx, ny), mc.co_hi, mc.cd_hi, f);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (zs[(ry + 1 + offy(k)) * HX + (rx + 1 + offx(k))] < zc) m |= (uint8_t)(1u << k);
            }
        }
        ms[ry * RX + rx] = m;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < RTX * RTY; i += RNT) {
        int ly = i / RTX, lx = i - ly * RTX;
        int64_t gx = x0 + lx, gy = y0 + ly;
        if (gx >= nx || gy >= ny) continue;
        int64_t gi = gy * nx + gx;
        if (!FR_OK(gi, nx * ny, 42)) continue;
        uint8_t m = ms[(ly + 1) * RX + lx + 1];
        mask[gi] = m;
        if (FRAC) {
            float zn[8], f[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) zn[k] = zs[(ly + 2 + offy(k)) * HX + (lx + 2 + offx(k))];
            if (flags & kDinf) {
                if (m) dinf_cell(zs[(ly + 2) * HX + (lx + 2)], zn, grid_mask8(gx, gy, nx, ny), mc.co_hi,
                                 mc.cd_hi, f);
                else
#pragma unroll
                    for (int k = 0; k < 8; ++k) f[k] = 0.0f;
            } else {
                mfd_fracs8(zs[(ly + 2) * HX + (lx + 2)], zn, m, mc, f);
            }
            float4* fo = reinterpret_cast<float4*>(frac + gi * 8);
            fo[0] = make_float4(f[0], f[1], f[2], f[3]);
            fo[1] = make_float4(f[4], f[5], f[6], f[7]);
        }
        if (INDEG) {
            int n = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                n += (ms[(ly + 1 + offy(k)) * RX + (lx + 1 + offx(k))] >> opp(k)) & 1;
            indeg[gi] = (uint8_t)n;
        }
    }
}

template <bool FRAC, bool INDEG>
__global__ void __launch_bounds__(RNT) k_receivers_mfd(const float* __restrict__ z, int64_t nx,
                                                       int64_t ny, MfdConst mc, uint32_t flags,
                                                       uint8_t* __restrict__ mask,
                                                       float* __restrict__ frac,
                                                       uint8_t* __restrict__ indeg) {
    int64_t x0, y0;
    tile_origin(nx, x0, y0);
    recv_mfd_tile<FRAC, INDEG>(z, nx, ny, mc, flags, mask, frac, indeg, x0, y0);
}

// ------------------------------------------------- slope split by edges
// Masks and fractions of the slope split.  The weight u = s^p of an edge is the
// same number whichever of its two cells is asked, and only the higher one
// gives water along it, so it is computed once per edge: four powers a cell
// (E, S, SE, SW; 4.25 with the tile's rim), each by a lane that needs it, where
// asking each cell for its lower neighbours runs all eight under masks.  Bound
// by instruction issue (the power is about 45 operations).  8192^2: masks and
// fractions 1.61 ms per cell, 1.19 by edges, 1.05 with the shorter power of
// mfd_pow_normal, 1.00 in 64x32 tiles; fractions of given masks 1.49, 1.16, 1.02
// and 0.97 ms.
constexpr int WTX = 64, WTY = 32;                     // tile (64x16 1.05 ms, 64x24 and 128x16 1.01)
constexpr int WZX = WTX + 2, WZY = WTY + 2;           // elevations with a one-cell rim
constexpr int WEN = WZX * (WTY + 1);                  // edges: rows -1 .. WTY - 1, columns -1 .. WTX

// GIVEN: masks come from `given` (bits off the grid are ignored), else from the
// elevations into mask_out.
template <bool GIVEN>
__global__ void __launch_bounds__(RNT) k_mfd_weights(const float* __restrict__ z,
                                                     const uint8_t* __restrict__ given, int64_t nx,
                                                     int64_t ny, MfdConst mc, uint32_t flags,
                                                     uint8_t* __restrict__ mask_out,
                                                     float* __restrict__ frac) {
    __shared__ float zs[WZX * WZY];
    __shared__ float us[4][WEN];  // weights of the edges to E, S, SE, SW
    const int64_t tiles_x = (nx + WTX - 1) / WTX;
    const int64_t ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
    const int64_t x0 = tx * WTX, y0 = ty * WTY;
    const float off = __int_as_float(0x7fffffff);  // off the grid: compares false with everything
    constexpr int NZ = (WZX * WZY + RNT - 1) / RNT;
    float zl[NZ];
#pragma unroll
    for (int q = 0; q < NZ; ++q) {
        const int i = threadIdx.x + q * RNT, ly = i / WZX, lx = i - ly * WZX;
        const int64_t gx = x0 + lx - 1, gy = y0 + ly - 1;
        zl[q] = off;
        if (i < WZX * WZY && gx >= 0 && gy >= 0 && gx < nx && gy < ny && FR_OK(gy * nx + gx, nx * ny, 40))
            zl[q] = __ldg(z + gy * nx + gx);
    }
#pragma unroll
    for (int q = 0; q < NZ; ++q)
        if (threadIdx.x + q * RNT < WZX * WZY) zs[threadIdx.x + q * RNT] = zl[q];
    __syncthreads();
    for (int i = threadIdx.x; i < WEN; i += RNT) {
        const int ly = i / WZX, lx = i - ly * WZX;
        const float zc = zs[i];
        // E, S, SE, SW neighbours (the rim's outermost lack some; their edges
        // are not used)
        const float zn[4] = {lx + 1 < WZX ? zs[i + 1] : off, zs[i + WZX], lx + 1 < WZX ? zs[i + WZX + 1] : off,
                             lx > 0 ? zs[i + WZX - 1] : off};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float hi = fmaxf(zc, zn[e]), lo = fminf(zc, zn[e]);
            us[e][i] = zc > zn[e] || zn[e] > zc ? mfd_u(hi, lo, e < 2 ? 0 : 4, mc) : 0.0f;
        }
    }
    __syncthreads();
    const bool edge_route = flags & kEdgeRoute;
    for (int i = threadIdx.x; i < WTX * WTY; i += RNT) {
        const int ly = i / WTX, lx = i - ly * WTX;
        const int64_t gx = x0 + lx, gy = y0 + ly;
        if (gx >= nx || gy >= ny) continue;
        const int64_t gi = gy * nx + gx;
        if (!FR_OK(gi, nx * ny, 43)) continue;
        const int c = (ly + 1) * WZX + lx + 1;
        const float zc = zs[c];
        float zn[8];
        uint32_t low = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            zn[k] = zs[c + offy(k) * WZX + offx(k)];
            low |= (uint32_t)(zn[k] < zc) << k;
        }
        uint32_t m;
        if constexpr (GIVEN) m = given[gi] & grid_mask8(gx, gy, nx, ny);
        else m = edge_route || !is_edge(gx, gy, nx, ny) ? low : 0u;
        if constexpr (!GIVEN) mask_out[gi] = (uint8_t)m;
        float f[8];
        if (m & ~low) {
            mfd_fracs8(zc, zn, m, mc, f);  // a caller's mask that points uphill: as the rule gives it
        } else {
            float u[8] = {us[0][c], us[1][c - WZX], us[0][c - 1], us[1][c],
                          us[3][c - WZX + 1], us[2][c - WZX - 1], us[3][c], us[2][c]};
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (!((m >> k) & 1u)) u[k] = 0.0f;
            mfd_fracs_of(u, m, f);
        }
        float4* fo = reinterpret_cast<float4*>(frac + gi * 8);
        fo[0] = make_float4(f[0], f[1], f[2], f[3]);
        fo[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
}

// Masks of the slope split alone: four consecutive cells of a row per thread
// from a 3 x 6 window, read through the cache (a cell's elevation is used by
// three rows of threads), no shared memory.  2048^2: 27 us by tiles, 14 now.
__global__ void __launch_bounds__(RNT) k_mfd_masks(const float* __restrict__ z, int64_t nx, int64_t ny,
                                                   uint32_t flags, uint8_t* __restrict__ mask) {
    const int64_t quads = (nx + 3) / 4, q = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
    const int64_t y = (int64_t)blockIdx.y * (RNT / 32) + (threadIdx.x >> 5), x0 = 4 * q;
    if (q >= quads || y >= ny) return;
    const float off = __int_as_float(0x7fffffff);
    float w[3][6];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 6; ++b) {
            const int64_t gx = x0 + b - 1, gy = y + a - 1;
            w[a][b] = gx >= 0 && gy >= 0 && gx < nx && gy < ny ? __ldg(z + gy * nx + gx) : off;
        }
    const bool edge_route = flags & kEdgeRoute;
    uint32_t packed = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float zc = w[1][c + 1];
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) m |= (uint32_t)(w[1 + offy(k)][c + 1 + offx(k)] < zc) << k;
        if (!edge_route && is_edge(x0 + c, y, nx, ny)) m = 0;
        packed |= m << (8 * c);
    }
    uint8_t* out = mask + y * nx + x0;
    if (x0 + 3 < nx && ((uintptr_t)out & 3) == 0) {
        *reinterpret_cast<uint32_t*>(out) = packed;
    } else {
        for (int c = 0; c < 4 && x0 + c < nx; ++c) out[c] = (uint8_t)(packed >> (8 * c));
    }
}

// D-infinity fractions of given receiver masks (a cell with an empty mask gives
// nothing): one cell per thread, elevations staged like the receiver tiles.
__global__ void __launch_bounds__(RNT) k_dinf_fractions(const float* __restrict__ z,
                                                        const uint8_t* __restrict__ mask,
                                                        int64_t nx, int64_t ny, MfdConst mc,
                                                        float* __restrict__ frac) {
    __shared__ float zs[HX * HY];
    int64_t x0, y0;
    tile_origin(nx, x0, y0);
    load_z_tile(zs, z, nx, ny, x0, y0);
    __syncthreads();
    for (int i = threadIdx.x; i < RTX * RTY; i += RNT) {
        const int ly = i / RTX, lx = i - ly * RTX;
        const int64_t gx = x0 + lx, gy = y0 + ly;
        if (gx >= nx || gy >= ny) continue;
        const int64_t gi = gy * nx + gx;
        if (!FR_OK(gi, nx * ny, 43)) continue;
        const uint32_t gm = grid_mask8(gx, gy, nx, ny);
        float zn[8], f[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            zn[k] = zs[(ly + 2 + offy(k)) * HX + (lx + 2 + offx(k))];
            f[k] = 0.0f;
        }
        if (mask[gi] & gm) dinf_cell(zs[(ly + 2) * HX + (lx + 2)], zn, gm, mc.co_hi, mc.cd_hi, f);
        float4* fo = reinterpret_cast<float4*>(frac + gi * 8);
        fo[0] = make_float4(f[0], f[1], f[2], f[3]);
        fo[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
}

// Problem and receiver tile number w of a batch: prefix[p] is the first tile of
// problem p (prefix[nprob] = total).
__device__ __forceinline__ int batch_tile(const int64_t* __restrict__ prefix, int nprob, int64_t w,
                                          const Prob* __restrict__ probs, int64_t& x0, int64_t& y0) {
    int lo = 0, hi = nprob - 1;  // last p with prefix[p] <= w
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= w) lo = mid;
        else hi = mid - 1;
    }
    const int64_t lt = w - prefix[lo], tiles_x = (probs[lo].nx + RTX - 1) / RTX;
    const int64_t ty = lt / tiles_x, tx = lt - ty * tiles_x;
    x0 = tx * RTX;
    y0 = ty * RTY;
    return lo;
}

// Batched D8 receivers: persistent warps take strips of any problem.
template <bool LOWEST, bool D4>
__global__ void __launch_bounds__(RNT) k_receivers_batch_d8(const Prob* __restrict__ probs,
                                                            const int64_t* __restrict__ prefix,
                                                            int nprob, uint32_t flags) {
    constexpr int kSub = RTY / kStrip;
    const int64_t total = prefix[nprob] * kSub;
    for (int64_t w = (int64_t)blockIdx.x * (RNT / 32) + (threadIdx.x >> 5); w < total;
         w += (int64_t)gridDim.x * (RNT / 32)) {
        int64_t x0, y0;
        const Prob& P = probs[batch_tile(prefix, nprob, w / kSub, probs, x0, y0)];
        y0 += w % kSub * kStrip;
        recv_d8_strip<LOWEST, D4>(P.z, P.nx, P.ny, P.mc.co_hi, P.mc.cd_hi, flags & kEdgeRoute,
                                  const_cast<uint8_t*>(P.rb), x0, y0);
    }
}

// Batched MFD receivers with fractions: persistent CTAs.
__global__ void __launch_bounds__(RNT) k_receivers_batch_mfd(const Prob* __restrict__ probs,
                                                             const int64_t* __restrict__ prefix,
                                                             int nprob, uint32_t flags, EngineGlobals* G) {
    __shared__ int64_t s_work;
    const int64_t total = prefix[nprob];
    while (true) {
        if (threadIdx.x == 0) s_work = (int64_t)atomicAdd(&G->recv_next, 1ull);
        __syncthreads();
        const int64_t w = s_work;
        __syncthreads();
        if (w >= total) break;
        int64_t x0, y0;
        const Prob& P = probs[batch_tile(prefix, nprob, w, probs, x0, y0)];
        recv_mfd_tile<true, false>(P.z, P.nx, P.ny, P.mc, flags, const_cast<uint8_t*>(P.rb),
                                   const_cast<float*>(P.frac), nullptr, x0, y0);
        __syncthreads();
    }
}

__global__ void k_count_nonfinite(const float* __restrict__ z, int64_t n,
                                  unsigned long long* count) {
    unsigned long long local = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        local += !isfinite(z[i]);
    for (int o = 16; o; o >>= 1) local += __shfl_down_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(count, local);
}

// Linear index of each cell's receiver (-1 for sinks and for codes that
// point out of the grid), four cells per thread step.
template <class I>
__global__ void __launch_bounds__(256) k_receiver_index(const uint8_t* __restrict__ dir, int64_t nx,
                                                        int64_t n, I* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t k = __ldg(dir + i);
        I r = (I)-1;
        if (k < 8) {
            const int64_t y = i / nx, x = i - y * nx;
            const int64_t xr = x + offx((int)k), yr = y + offy((int)k);
            if (xr >= 0 && yr >= 0 && xr < nx && yr * nx + xr < n) r = (I)(yr * nx + xr);
        }
        out[i] = r;
    }
}

template <bool LOWEST, bool D4>
cudaError_t launch_d8_tma(const CUtensorMap& map, int64_t nx, int64_t ny, float co, float cd,
                          uint32_t flags, uint8_t* dir, cudaStream_t s) {
    constexpr size_t sm = sizeof(TmaSmem);
    static std::atomic<unsigned long long> set_on{0};
    static int grid_per_sm = 0, sms = 0;
    cudaError_t e = smem_limit_once(k_receivers_d8_tma<LOWEST, D4>, sm, set_on);
    if (e != cudaSuccess) return e;
    if (!grid_per_sm) {
        int dev = 0, per = 0, n = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_receivers_d8_tma<LOWEST, D4>, 256, sm)) !=
            cudaSuccess)
            return e;
        sms = n;
        grid_per_sm = per > 0 ? per : 1;
    }
    const int tiles_x = (int)((nx + TTX - 1) / TTX);
    const int64_t ntiles = (int64_t)tiles_x * ((ny + TTY - 1) / TTY);
    int64_t grid = (int64_t)sms * grid_per_sm;
    if (grid > ntiles) grid = ntiles;
    k_receivers_d8_tma<LOWEST, D4><<<(unsigned)grid, 256, sm, s>>>(map, nx, ny, co, cd, flags, dir, ntiles,
                                                                   tiles_x, wait_limit_ns());
    return cudaGetLastError();
}

}  // namespace

bool encode_tile_map_f32(CUtensorMap* map, const float* base, int64_t nx, int64_t ny, int box_x,
                         int box_y) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    // cuTensorMapEncodeTiled from the CUDA driver API, looked up once (thread-safe static
    // initialisation)
    static const Encode fn = []() -> Encode {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<Encode>(p);
        return nullptr;
    }();
    if (!fn || (nx & 3) || ((uintptr_t)base & 15) || nx > (int64_t)1 << 31 || ny > (int64_t)1 << 31) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)ny};
    const cuuint64_t strides[1] = {(cuuint64_t)nx * 4};
    const cuuint32_t box[2] = {(cuuint32_t)box_x, (cuuint32_t)box_y};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NAN_REQUEST_ZERO_FMA) == CUDA_SUCCESS;
}

cudaError_t read_clear_tma_error(unsigned* out, cudaStream_t s) {
    unsigned zero = 0;
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_tma_wait_error);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(out, p, sizeof(unsigned), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    if (*out == 0) return cudaSuccess;
    if ((e = cudaMemcpyAsync(p, &zero, sizeof(unsigned), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

cudaError_t launch_receiver_index(const uint8_t* dir, int64_t nx, int64_t ny, bool wide, void* out,
                                  cudaStream_t s) {
    const int64_t n = nx * ny;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (wide)
        k_receiver_index<int64_t><<<(unsigned)blocks, 256, 0, s>>>(dir, nx, n, (int64_t*)out);
    else
        k_receiver_index<int32_t><<<(unsigned)blocks, 256, 0, s>>>(dir, nx, n, (int32_t*)out);
    return cudaGetLastError();
}

cudaError_t launch_receivers_d8(const float* z, int64_t nx, int64_t ny, double dx,
                                uint32_t flags, uint8_t* dir, uint8_t* indeg, cudaStream_t s) {
    float co = (float)(1.0 / dx);
    float cd = (float)(1.0 / (std::sqrt(2.0) * dx));
    const bool lowest = flags & kD8Lowest;
    // codes alone on a TMA-addressable grid that gives most SMs a tile: the
    // pipelined persistent kernel (below 2^20 cells the strips are the faster:
    // 512^2 5.8 us against 6.8, 768^2 6.5 and 7.0, 1024^2 7.0 and 7.2, 1280^2 11.0 and
    // 9.2, 2048^2 18.9 and 14.4, 4096^2 54 and 37)
    CUtensorMap map;
    if (!indeg && nx * ny >= (int64_t)1 << 20 && encode_tile_map_f32(&map, z, nx, ny, TBX, TBY)) {
        const bool d4 = flags & kD4;
        if (lowest) return d4 ? launch_d8_tma<true, true>(map, nx, ny, co, cd, flags, dir, s)
                              : launch_d8_tma<true, false>(map, nx, ny, co, cd, flags, dir, s);
        return d4 ? launch_d8_tma<false, true>(map, nx, ny, co, cd, flags, dir, s)
                  : launch_d8_tma<false, false>(map, nx, ny, co, cd, flags, dir, s);
    }
    const int64_t tiles = ((nx + RTX - 1) / RTX) * ((ny + kStrip - 1) / kStrip);
    const unsigned wgrid = (unsigned)((tiles + RNT / 32 - 1) / (RNT / 32));
    const unsigned cgrid = (unsigned)(((nx + RTX - 1) / RTX) * ((ny + kCountRows - 1) / kCountRows));
    auto run = [&](auto low, auto d4) {
        constexpr bool L = decltype(low)::value, D = decltype(d4)::value;
        if (indeg) k_receivers_d8_indeg<L, D><<<cgrid, RNT, 0, s>>>(z, nx, ny, co, cd, flags, dir, indeg);
        else k_receivers_d8<L, D><<<wgrid, RNT, 0, s>>>(z, nx, ny, co, cd, flags, dir, tiles);
    };
    if (lowest && (flags & kD4)) run(std::true_type{}, std::true_type{});
    else if (lowest) run(std::true_type{}, std::false_type{});
    else if (flags & kD4) run(std::false_type{}, std::true_type{});
    else run(std::false_type{}, std::false_type{});
    return cudaGetLastError();
}

namespace {
unsigned weight_tiles(int64_t nx, int64_t ny) {
    return (unsigned)(((nx + WTX - 1) / WTX) * ((ny + WTY - 1) / WTY));
}
}  // namespace

cudaError_t launch_receivers_mfd(const float* z, int64_t nx, int64_t ny, double dx, double p,
                                 uint32_t flags, uint8_t* mask, float* frac, uint8_t* indeg,
                                 cudaStream_t s) {
    const unsigned grid = (unsigned)(((nx + RTX - 1) / RTX) * ((ny + RTY - 1) / RTY));
    MfdConst mc = make_mfd_const(dx, p);
    if (!indeg && !(flags & kDinf) && frac) {  // the slope split without donor counts: by edges
        k_mfd_weights<false><<<weight_tiles(nx, ny), RNT, 0, s>>>(z, nullptr, nx, ny, mc, flags, mask, frac);
        return cudaGetLastError();
    }
    if (!indeg && !(flags & kDinf) && ny <= 65535ll * (RNT / 32)) {
        const dim3 g((unsigned)((nx + 127) / 128), (unsigned)((ny + RNT / 32 - 1) / (RNT / 32)));
        k_mfd_masks<<<g, RNT, 0, s>>>(z, nx, ny, flags, mask);
        return cudaGetLastError();
    }
    if (frac && indeg)
        k_receivers_mfd<true, true><<<grid, RNT, 0, s>>>(z, nx, ny, mc, flags, mask, frac, indeg);
    else if (frac)
        k_receivers_mfd<true, false><<<grid, RNT, 0, s>>>(z, nx, ny, mc, flags, mask, frac, nullptr);
    else if (indeg)
        k_receivers_mfd<false, true><<<grid, RNT, 0, s>>>(z, nx, ny, mc, flags, mask, nullptr, indeg);
    else
        k_receivers_mfd<false, false><<<grid, RNT, 0, s>>>(z, nx, ny, mc, flags, mask, nullptr,
                                                           nullptr);
    return cudaGetLastError();
}

cudaError_t launch_mfd_fractions(const float* z, const uint8_t* mask, int64_t nx, int64_t ny,
                                 double dx, double p, uint32_t flags, float* frac, cudaStream_t s) {
    if (!(flags & kDinf)) {
        k_mfd_weights<true><<<weight_tiles(nx, ny), RNT, 0, s>>>(z, mask, nx, ny, make_mfd_const(dx, p), flags,
                                                                 nullptr, frac);
        return cudaGetLastError();
    }
    const unsigned grid = (unsigned)(((nx + RTX - 1) / RTX) * ((ny + RTY - 1) / RTY));
    k_dinf_fractions<<<grid, RNT, 0, s>>>(z, mask, nx, ny, make_mfd_const(dx, p), frac);
    return cudaGetLastError();
}

cudaError_t launch_receivers_batch(int kind, const Prob* probs, const int64_t* prefix, int nprob,
                                   uint32_t flags, EngineGlobals* G, int grid, cudaStream_t s) {
    const bool low = flags & kD8Lowest, d4 = flags & kD4;
    if (kind != 0) k_receivers_batch_mfd<<<grid, RNT, 0, s>>>(probs, prefix, nprob, flags, G);
    else if (low && d4) k_receivers_batch_d8<true, true><<<grid, RNT, 0, s>>>(probs, prefix, nprob, flags);
    else if (low) k_receivers_batch_d8<true, false><<<grid, RNT, 0, s>>>(probs, prefix, nprob, flags);
    else if (d4) k_receivers_batch_d8<false, true><<<grid, RNT, 0, s>>>(probs, prefix, nprob, flags);
    else k_receivers_batch_d8<false, false><<<grid, RNT, 0, s>>>(probs, prefix, nprob, flags);
    return cudaGetLastError();
}

cudaError_t launch_count_nonfinite(const float* z, int64_t n, unsigned long long* count,
                                   cudaStream_t s) {
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_count_nonfinite<<<(unsigned)blocks, 256, 0, s>>>(z, n, count);
    return cudaGetLastError();
}

}  // namespace fr

#ifdef FR_DEBUG_BOUNDS
// Debug builds only: first out-of-range access seen by the receiver kernels.
extern "C" unsigned long long fr_debug_bad_receivers(void) {
    unsigned long long v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, fr::fr_debug_bad, sizeof(v));
    cudaMemcpyToSymbol(fr::fr_debug_bad, &z, sizeof(z));
    return v;
}
#endif
