// Map precompute: exact squared Euclidean distance transform (the EDT lookup
// table of Sec. III-A item 3, used by the likelihood field of Eq. 23 and the
// distance statistics of Eq. 29-30), its clamped padded copy for TAM, and the
// tiled occupancy bitmap for ray casting (Eq. 13) with, per walk frame, the
// empty squares of tiles ahead of every tile.
//
// The clamped field is stored in bands of 8 rows (field_index) with a border
// of P cells holding C on every side, P at least the longest beam in cells, so
// every beam endpoint of TAM falls inside the array and needs no bounds test.
//
// The distance passes themselves are in edt_band.cuh; the tile pass here also
// lays out the walk frames and, where the caller's grid allows it, writes the
// map's own copy of the grid.
#include <cuda_runtime.h>
#include <stdint.h>

#include "edt_band.cuh"
#include "relo_internal.h"

namespace relo {

namespace {

// Occupancy tiles, column summaries and walk frames: the map's word as is, and, with the cells outside the map set, the
// four walk frames: as is, and mirrored in x (x' = 8 TW - 1 - x: tile TW - 1 - tx, bits reversed within each row), in y
// (rows reversed) and in both (all 64 bits reversed), which the ray cast uses so that every ray travels towards +x and
// +y.  A thread reads a tile's 8 rows of 8 bytes with 8 loads in flight (32 bytes a row of the warp are 8 tiles wide); a
// ballot per row of 32 columns with a byte load per cell took 26 us on the 4096 x 4096 warehouse, this takes 9 us
// (with the copy of the grid, which was another 9 us).
__global__ void __launch_bounds__(256) k_edt_tiles(const int8_t *__restrict__ grid, EdtTiles t, bool vec, int8_t *copy,
                                                   uint64_t *wf) {
    edt_tiles(grid, t, vec, copy, [&](uint64_t w, int tx, int ty) {
        const size_t WB = (size_t)t.TW + 1, n = walk_frame_words(t.TW, t.TH);
        const uint64_t rev = __brevll(w);   // both mirrors
        const uint64_t ymir = ((uint64_t)__byte_perm((uint32_t)w, 0u, 0x0123u) << 32) |
                              (uint64_t)__byte_perm((uint32_t)(w >> 32), 0u, 0x0123u);
        const uint64_t xmir = ((uint64_t)__byte_perm((uint32_t)rev, 0u, 0x0123u) << 32) |
                              (uint64_t)__byte_perm((uint32_t)(rev >> 32), 0u, 0x0123u);
        const int mx = t.TW - 1 - tx, my = t.TH - 1 - ty;
        wf[(size_t)ty * WB + tx] = w;
        wf[n + (size_t)ty * WB + mx] = xmir;
        wf[2 * n + (size_t)my * WB + tx] = ymir;
        wf[3 * n + (size_t)my * WB + mx] = rev;
    });
}

EdtTiles tiles_of(const MapDev &m) { return EdtTiles{m.bits, m.summ, edt_span_of(m), m.far, m.W, m.H, m.TW, m.TH}; }

// the border of the padded field: every cell outside the map reads C (d = d_max)
__global__ void k_field_border(uint16_t *__restrict__ fieldp, int W, int H, int P, int Wp, int Hp, int C) {
    const size_t n = (size_t)Hp * Wp;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t c = i >> 3;   // column of a band, then the row inside the band (field_index)
        const int y = (int)(c / Wp) * 8 + (int)(i & 7) - P, x = (int)(c % Wp) - P;
        if (x < 0 || y < 0 || x >= W || y >= H) fieldp[i] = (uint16_t)C;
    }
}

// Which walk-frame tiles are empty, one bit per tile: word [row][k] of a
// frame row holds tiles 32 k .. 32 k + 31 (tiles past the row count as not
// empty, and one more word of zeros ends every row).
__global__ void k_walk_empty(const uint64_t *__restrict__ wf, int TW, uint32_t *__restrict__ emp) {
    const unsigned WB = (unsigned)TW + 1u, SW = walk_empty_row_words(TW);
    const unsigned x = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t row = blockIdx.y;   // frame * (TH + 1) + ty
    const unsigned bal = __ballot_sync(0xffffffffu, x < WB && wf[row * WB + x] == 0ull);
    if ((threadIdx.x & 31) == 0 && (x >> 5) < SW) emp[row * SW + (x >> 5)] = bal;
}

// The empty boxes ahead of every walk-frame tile (MapDev::reach).  A warp
// takes 32 tiles of a row: lanes k < kReachMax load the emptiness word of row
// ty + k covering its tiles and lanes kReachMax + k the next word.  For each
// of the kReachMax rows from theirs, a lane shifts the 64 bits of that pair
// down by its own position, so bit i says whether the tile i to its right is
// empty (i + 31 < 64: a window of kReachMax + 1 bits always fits).  Its row
// run is the block of set bits from bit 0 of the first row, its column run
// the rows that keep bit 0, and its square the largest s whose s rows' AND
// keeps bits 0 .. s - 1.
__global__ void k_walk_reach(const uint32_t *__restrict__ emp, int TW, int TH, uint16_t *__restrict__ reach) {
    static_assert(2 * kReachMax <= 32, "one emptiness word per lane");
    const int lane = threadIdx.x & 31;
    const unsigned WB = (unsigned)TW + 1u, HB = (unsigned)TH + 1u, SW = walk_empty_row_words(TW);
    const unsigned strip = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (strip * 32u >= WB) return;   // the whole warp lies past the row
    const unsigned fy = blockIdx.y, ty = fy % HB;   // frame * HB + ty
    const unsigned k = (unsigned)lane % kReachMax, y = ty + k;
    const uint32_t wv = y < HB ? emp[(size_t)(fy + k) * SW + strip + lane / kReachMax] : 0u;
    uint32_t e0 = 0u, a = ~0u;
    int s = 0, yr = 0;
    bool sq = true, col = true;
#pragma unroll
    for (int r = 0; r < kReachMax; ++r) {
        const uint32_t e = __funnelshift_r(__shfl_sync(0xffffffffu, wv, r),
                                           __shfl_sync(0xffffffffu, wv, r + kReachMax), (unsigned)lane);
        if (r == 0) e0 = e;
        col = col && (e & 1u);
        if (col) yr = r + 1;
        a &= e;
        const uint32_t mr = (2u << r) - 1u;   // bits 0 .. r
        sq = sq && (a & mr) == mr;
        if (sq) s = r + 1;
        if (!__any_sync(0xffffffffu, sq || col)) break;   // no lane's boxes grow further
    }
    // the sentinel bit caps the row run at kReachMax
    const int xr = __ffs((int)(~e0 | (1u << kReachMax))) - 1;
    const unsigned xa = strip * 32u + lane;
    if (xa < WB) reach[(size_t)fy * WB + xa] = (uint16_t)(s | (xr << 5) | (yr << 10));
}

// the last column and row of tiles of each walk frame: every bit set
__global__ void k_walk_border(uint64_t *__restrict__ wf, int TW, int TH) {
    uint64_t *f = wf + (size_t)blockIdx.x * walk_frame_words(TW, TH);
    const int WB = TW + 1;
    for (int i = threadIdx.x; i <= TH; i += blockDim.x) f[(size_t)i * WB + TW] = ~0ull;
    for (int i = threadIdx.x; i < TW; i += blockDim.x) f[(size_t)TH * WB + i] = ~0ull;
}

// The tables row-major: a thread takes kCols columns (4 where rows and buffers are aligned for vector stores, else 1) of
// one field band (8 rows, each column 16 contiguous bytes of the field), so every field load is 16 bytes and the lanes
// of a warp store neighbouring columns; one cell per thread read 2 of every 16 field bytes and divided for its
// coordinates (87 us on 4001 x 3500, now 38).
template <int kCols>
__global__ void __launch_bounds__(128) k_map_tables(const int32_t *__restrict__ d2s, const uint16_t *__restrict__ fs,
                                                    const uint64_t *__restrict__ bs, int W, int H, int TW, int P, int Wp,
                                                    int32_t *__restrict__ d2, uint16_t *__restrict__ field,
                                                    uint8_t *__restrict__ occ) {
    const int B = (P >> 3) + (int)blockIdx.y, y0 = 8 * B - P, x0 = kCols * ((int)blockIdx.x * 128 + (int)threadIdx.x);
    if (x0 >= W) return;   // kCols divides W
    uint4 f[kCols] = {};
    if (field)
#pragma unroll
        for (int i = 0; i < kCols; ++i) f[i] = *reinterpret_cast<const uint4 *>(fs + 8 * ((size_t)B * Wp + (x0 + i + P)));
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int y = y0 + u;
        if (y < 0 || y >= H) continue;
        const size_t at = (size_t)y * W + x0;
        uint32_t h[kCols];
#pragma unroll
        for (int i = 0; i < kCols; ++i) {
            const uint32_t w = u < 2 ? f[i].x : u < 4 ? f[i].y : u < 6 ? f[i].z : f[i].w;
            h[i] = w >> (16 * (u & 1)) & 0xffffu;
        }
        uint32_t o = 0u;   // the cells' occupancy bits (of one tile row)
        if (occ) o = (uint32_t)(bs[(size_t)(y >> 3) * TW + (x0 >> 3)] >> (((y & 7) << 3) | (x0 & 7)));
        if constexpr (kCols == 4) {
            if (d2) *reinterpret_cast<int4 *>(d2 + at) = *reinterpret_cast<const int4 *>(d2s + at);
            if (field) *reinterpret_cast<uint2 *>(field + at) = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
            if (occ)
                *reinterpret_cast<uint32_t *>(occ + at) = (o & 1u) | (o & 2u) << 7 | (o & 4u) << 14 | (o & 8u) << 21;
        } else {
            if (d2) d2[at] = d2s[at];
            if (field) field[at] = (uint16_t)h[0];
            if (occ) occ[at] = (uint8_t)(o & 1u);
        }
    }
}

__global__ void k_check_cells(const int2 *__restrict__ cells, int n, const uint64_t *__restrict__ bits, int W,
                              int H, int TW, int *bad) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int2 c = cells[i];
    bool ok = (unsigned)c.x < (unsigned)W && (unsigned)c.y < (unsigned)H;
    if (ok) ok = !((bits[(size_t)(c.y >> 3) * TW + (c.x >> 3)] >> (((c.y & 7) << 3) | (c.x & 7))) & 1ull);
    if (!ok) atomicAdd(bad, 1);
}

// Hypotheses given in metres (Eq. 6): the containing cell (floor((x - ox) /
// res), floor((y - oy) / res)) in FP64, each operation rounded as IEEE
// prescribes, so the cells equal those of the same expression on the host.
// flags[0] counts points off the map (or not finite), flags[1] points on
// occupied cells; an off-map point's cell is written as (0, 0).
__global__ void k_xy_cells(const double2 *__restrict__ xy, int n, double ox, double oy, double res,
                           const uint64_t *__restrict__ bits, int W, int H, int TW, int2 *__restrict__ cells,
                           int *flags) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 p = xy[i];
    const double fx = floor((p.x - ox) / res), fy = floor((p.y - oy) / res);
    if (!(fx >= 0.0 && fy >= 0.0 && fx < (double)W && fy < (double)H)) {
        cells[i] = make_int2(0, 0);
        atomicAdd(flags, 1);
        return;
    }
    const int cx = (int)fx, cy = (int)fy;
    cells[i] = make_int2(cx, cy);
    if ((bits[(size_t)(cy >> 3) * TW + (cx >> 3)] >> (((cy & 7) << 3) | (cx & 7))) & 1ull) atomicAdd(flags + 1, 1);
}

}  // namespace

cudaError_t launch_xy_cells(const double *xy, int n, double ox, double oy, double res, const MapDev &m, int2 *cells,
                            int *flags, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_xy_cells<<<(n + 255) / 256, 256, 0, s>>>(reinterpret_cast<const double2 *>(xy), n, ox, oy, res, m.bits, m.W,
                                               m.H, m.TW, cells, flags);
    return cudaGetLastError();
}

cudaError_t launch_edt_tiles(const MapDev &m, const int8_t *grid, cudaStream_t s) {
    const EdtTiles t = tiles_of(m);
    const bool vec = (m.W & 7) == 0 && (reinterpret_cast<uintptr_t>(grid) & 7) == 0;
    int8_t *copy = grid != m.grid ? m.grid : nullptr;
    if (copy && !vec) {
        const cudaError_t e = cudaMemcpyAsync(m.grid, grid, (size_t)m.W * m.H, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return e;
        return launch_edt_tiles(m, m.grid, s);
    }
    k_edt_tiles<<<dim3((m.TW + 31) / 32, edt_summary_rows(m.H)), dim3(32, 8), 0, s>>>(grid, t, vec, copy,
                                                                                      m.bits + (size_t)m.TW * m.TH);
    if (m.reach) {
        // the walk frames' empty boxes (their border tiles, full, were written when the map was loaded)
        const unsigned WB = (unsigned)m.TW + 1u, SW = walk_empty_row_words(m.TW), rows = 4u * ((unsigned)m.TH + 1u);
        uint32_t *emp = walk_empty_bits(m.reach, m.TW, m.TH);
        k_walk_empty<<<dim3((32u * SW + 255u) / 256u, rows), 256, 0, s>>>(m.bits + (size_t)m.TW * m.TH, m.TW, emp);
        k_walk_reach<<<dim3((WB + 255u) / 256u, rows), 256, 0, s>>>(emp, m.TW, m.TH, m.reach);
    }
    return cudaGetLastError();
}

cudaError_t launch_edt_field(const MapDev &m, int n_sm, cudaStream_t s) {
    return launch_edt_bands(tiles_of(m), EdtOut{m.d2, m.field, m.C, m.P, m.Wp}, n_sm, s);
}

cudaError_t launch_edt(const MapDev &m, int n_sm, cudaStream_t s) {
    cudaError_t e = launch_edt_tiles(m, m.grid, s);
    return e == cudaSuccess ? launch_edt_field(m, n_sm, s) : e;
}

cudaError_t launch_field_border(const MapDev &m, cudaStream_t s) {
    k_field_border<<<1024, 256, 0, s>>>(m.field, m.W, m.H, m.P, m.Wp, m.Hp, m.C);
    k_walk_border<<<4, 256, 0, s>>>(m.bits + (size_t)m.TW * m.TH, m.TW, m.TH);
    return cudaGetLastError();
}

cudaError_t launch_map_tables(const MapDev &m, int32_t *d2, uint16_t *field, uint8_t *occ, cudaStream_t s) {
    const bool vec = (m.W & 3) == 0 && (reinterpret_cast<uintptr_t>(d2) & 15) == 0 &&
                     (reinterpret_cast<uintptr_t>(field) & 7) == 0 && (reinterpret_cast<uintptr_t>(occ) & 3) == 0;
    const int bands = edt_bands(m.H, m.P);
    if (vec)
        k_map_tables<4><<<dim3((m.W + 511) / 512, bands), 128, 0, s>>>(m.d2, m.field, m.bits, m.W, m.H, m.TW, m.P, m.Wp,
                                                                       d2, field, occ);
    else
        k_map_tables<1><<<dim3((m.W + 127) / 128, bands), 128, 0, s>>>(m.d2, m.field, m.bits, m.W, m.H, m.TW, m.P, m.Wp,
                                                                       d2, field, occ);
    return cudaGetLastError();
}

cudaError_t launch_check_cells(const int2 *cells, int n, const MapDev &m, int *bad, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_check_cells<<<(n + 255) / 256, 256, 0, s>>>(cells, n, m.bits, m.W, m.H, m.TW, bad);
    return cudaGetLastError();
}

}  // namespace relo
