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

EdtTiles tiles_of(const MapDev &m) { return EdtTiles{m.bits, m.summ, edt_span_of(m), m.far,
                                                    m.reach ? walk_empty_bits(m.reach, m.TW, m.TH) : nullptr, m.W, m.H, m.TW, m.TH}; }

// the border of the padded field: every cell outside the map reads the code of C (d = d_max), the last rank
__global__ void k_field_border(uint16_t *__restrict__ fieldp, int W, int H, int P, int Wp, int Hp, uint32_t code) {
    const size_t n = (size_t)Hp * Wp;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t c = i >> 3;   // column of a band, then the row inside the band (field_index)
        const int y = (int)(c / Wp) * 8 + (int)(i & 7) - P, x = (int)(c % Wp) - P;
        if (x < 0 || y < 0 || x >= W || y >= H) fieldp[i] = (uint16_t)code;
    }
}

// The rows of emptiness that a warp's 32 tiles of a frame row see ahead: lanes k < kReachMax hold the emptiness bits of
// row ty + k covering the tiles, lanes kReachMax + k the next 32.  For each of the kReachMax rows from theirs, a lane
// shifts the 64 bits of that pair down by its own position (row_ahead), so bit i says whether the tile i to its right is
// empty (i + 31 < 64: a window of kReachMax + 1 bits always fits).  The map's emptiness is stored once; a frame mirrored
// in x reads the window from the other end, reversed, and tiles outside the map count as not empty.
__device__ __forceinline__ uint32_t rows_ahead(const uint32_t *__restrict__ emp, int TW, int TH, unsigned strip) {
    static_assert(2 * kReachMax <= 32, "one emptiness word per lane");
    const int lane = threadIdx.x & 31, HB = TH + 1, words = walk_empty_row_words(TW);
    const int frame = (int)blockIdx.y / HB, y = (int)blockIdx.y % HB + lane % kReachMax, s = (int)strip + lane / kReachMax;
    if (y >= TH) return 0u;
    const uint32_t *row = emp + (size_t)(frame & 2 ? TH - 1 - y : y) * words;
    if (!(frame & 1)) return s < words ? row[s] : 0u;
    const int p = TW - 32 * (s + 1), q = p >> 5;   // the map's tiles p .. p + 31
    const uint32_t lo = q >= 0 ? row[q] : 0u, hi = q + 1 >= 0 && q + 1 < words ? row[q + 1] : 0u;
    return __brev(__funnelshift_r(lo, hi, (unsigned)(p & 31)));
}
__device__ __forceinline__ uint32_t row_ahead(uint32_t words, int r) {
    return __funnelshift_r(__shfl_sync(0xffffffffu, words, r), __shfl_sync(0xffffffffu, words, r + kReachMax),
                           threadIdx.x & 31);
}

// The empty boxes ahead of every walk-frame tile, per slope class (MapDev::reach).  A warp takes 32 tiles of a row.  With
// h rows' windows ANDed, the run of set bits from bit 0 is the widest box of height h; a class keeps the (w, h) whose far
// edges a ray from the tile's middle at its angle reaches last, min((w - 1/2) / cos, (h - 1/2) / sin).  That value in
// 1/128 tiles above the box's code is one integer, so a candidate is a product, a minimum, an OR and a maximum; a class
// looks no further down than the height that no width up to kReachMax can use (2, 4 and 9 rows for the shallow ones).
// Bound by those; with float values and a box beside each 39 us on the 4096 x 4096 warehouse (1.05 M tiles, 7 classes).
__global__ void __launch_bounds__(256) k_walk_reach(const uint32_t *__restrict__ emp, int TW, int TH,
                                                    uint16_t *__restrict__ reach) {
    // 64 / cos and 64 / sin of the classes' middles: 3, 11, 26, 45, 64, 79 and 87 degrees
    constexpr uint32_t kInvC[kReachClasses] = {64, 65, 71, 91, 146, 335, 1223};
    constexpr uint32_t kInvS[kReachClasses] = {1223, 335, 146, 91, 71, 65, 64};
    const int lane = threadIdx.x & 31;
    const unsigned WB = (unsigned)TW + 1u, HB = (unsigned)TH + 1u;
    const unsigned strip = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (strip * 32u >= WB) return;   // the whole warp lies past the row
    const uint32_t words = rows_ahead(emp, TW, TH, strip);
    uint32_t a = ~0u, best[kReachClasses];
#pragma unroll
    for (int c = 0; c < kReachClasses; ++c) best[c] = 8u | 8u << 8 | 1u;   // not empty: the tile alone
#pragma unroll
    for (int r = 0; r < kReachMax; ++r) {
        a &= row_ahead(words, r);
        const uint32_t w = (uint32_t)__ffs((int)(~a | (1u << kReachMax))) - 1u;   // the sentinel bit caps the run
        if (!__any_sync(0xffffffffu, w > 0u)) break;
        if (w > 0u) {
            const uint32_t w2 = 2u * w - 1u, e = 8u * w | 8u * (uint32_t)(r + 1) << 8;
#pragma unroll
            for (int c = 0; c < kReachClasses; ++c) {
                // rows that r - 1 already offered at any width add nothing
                if (r > 0 && (2u * r - 1u) * kInvS[c] >= (2u * kReachMax - 1u) * kInvC[c]) continue;
                best[c] = max(best[c], min(w2 * (kInvC[c] << 16), ((2u * r + 1u) * kInvS[c]) << 16) | e);
            }
        }
    }
    const unsigned xa = strip * 32u + lane, frame = blockIdx.y / HB, ty = blockIdx.y % HB;
    const size_t n = walk_frame_words(TW, TH);
    if (xa < WB) {
        uint16_t *out = reach + (size_t)frame * kReachClasses * n + (size_t)ty * WB + xa;
#pragma unroll
        for (int c = 0; c < kReachClasses; ++c) out[c * n] = (uint16_t)best[c];
    }
}

// The exported boxes (relo_map_walk_boxes_dev): the row run is the block of set bits from bit 0 of the first row, the
// column run the rows that keep bit 0, the square the largest s whose s rows' AND keeps bits 0 .. s - 1.
__global__ void k_walk_export(const uint32_t *__restrict__ emp, int TW, int TH, uint16_t *__restrict__ boxes) {
    const int lane = threadIdx.x & 31;
    const unsigned WB = (unsigned)TW + 1u;
    const unsigned strip = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (strip * 32u >= WB) return;
    const uint32_t words = rows_ahead(emp, TW, TH, strip);
    uint32_t e0 = 0u, a = ~0u;
    int s = 0, yr = 0;
    bool sq = true, col = true;
#pragma unroll
    for (int r = 0; r < kReachMax; ++r) {
        const uint32_t e = row_ahead(words, r);
        if (r == 0) e0 = e;
        col = col && (e & 1u);
        if (col) yr = r + 1;
        a &= e;
        const uint32_t mr = (2u << r) - 1u;   // bits 0 .. r
        sq = sq && (a & mr) == mr;
        if (sq) s = r + 1;
    }
    const int xr = __ffs((int)(~e0 | (1u << kReachMax))) - 1;
    const unsigned xa = strip * 32u + lane;
    if (xa < WB) boxes[(size_t)blockIdx.y * WB + xa] = (uint16_t)(s | (xr << 5) | (yr << 10));
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
                                                    uint8_t *__restrict__ occ, const uint16_t *__restrict__ value,
                                                    int n_rank) {
    extern __shared__ uint16_t s_value[];   // the value of every rank
    if (field)
        for (int i = threadIdx.x; i < n_rank; i += 128) s_value[i] = __ldg(value + i);
    __syncthreads();
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
            h[i] = field ? s_value[(w >> (16 * (u & 1)) & 0xffffu) - kFieldBias] : 0u;
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
    return cudaGetLastError();
}

cudaError_t launch_walk_reach(const MapDev &m, cudaStream_t s) {
    if (m.reach) {
        // the walk frames' empty boxes (their border tiles, full, were written when the map was loaded)
        const unsigned WB = (unsigned)m.TW + 1u, rows = 4u * ((unsigned)m.TH + 1u);
        k_walk_reach<<<dim3((WB + 255u) / 256u, rows), 256, 0, s>>>(walk_empty_bits(m.reach, m.TW, m.TH), m.TW, m.TH,
                                                                    m.reach);
    }
    return cudaGetLastError();
}

cudaError_t launch_edt_field(const MapDev &m, int n_sm, cudaStream_t s) {
    return launch_edt_bands(tiles_of(m), EdtOut{m.d2, m.field, m.code, m.C, m.P, m.Wp}, n_sm, s);
}

cudaError_t launch_edt(const MapDev &m, int n_sm, cudaStream_t s) {
    cudaError_t e = launch_edt_tiles(m, m.grid, s);
    return e == cudaSuccess ? launch_edt_field(m, n_sm, s) : e;
}

cudaError_t launch_walk_boxes(const MapDev &m, uint16_t *boxes, cudaStream_t s) {
    const unsigned WB = (unsigned)m.TW + 1u, rows = 4u * ((unsigned)m.TH + 1u);
    k_walk_export<<<dim3((WB + 255u) / 256u, rows), 256, 0, s>>>(walk_empty_bits(m.reach, m.TW, m.TH), m.TW, m.TH, boxes);
    return cudaGetLastError();
}

cudaError_t launch_field_border(const MapDev &m, cudaStream_t s) {
    k_field_border<<<1024, 256, 0, s>>>(m.field, m.W, m.H, m.P, m.Wp, m.Hp, kFieldBias + (uint32_t)m.n_rank - 1u);
    k_walk_border<<<4, 256, 0, s>>>(m.bits + (size_t)m.TW * m.TH, m.TW, m.TH);
    return cudaGetLastError();
}

cudaError_t launch_map_tables(const MapDev &m, int32_t *d2, uint16_t *field, uint8_t *occ, cudaStream_t s) {
    const bool vec = (m.W & 3) == 0 && (reinterpret_cast<uintptr_t>(d2) & 15) == 0 &&
                     (reinterpret_cast<uintptr_t>(field) & 7) == 0 && (reinterpret_cast<uintptr_t>(occ) & 3) == 0;
    const int bands = edt_bands(m.H, m.P);
    const size_t smem = field ? (size_t)m.n_rank * sizeof(uint16_t) : 0;
    if (vec)
        k_map_tables<4><<<dim3((m.W + 511) / 512, bands), 128, smem, s>>>(m.d2, m.field, m.bits, m.W, m.H, m.TW, m.P, m.Wp,
                                                                          d2, field, occ, m.value, m.n_rank);
    else
        k_map_tables<1><<<dim3((m.W + 127) / 128, bands), 128, smem, s>>>(m.d2, m.field, m.bits, m.W, m.H, m.TW, m.P, m.Wp,
                                                                          d2, field, occ, m.value, m.n_rank);
    return cudaGetLastError();
}

cudaError_t launch_check_cells(const int2 *cells, int n, const MapDev &m, int *bad, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_check_cells<<<(n + 255) / 256, 256, 0, s>>>(cells, n, m.bits, m.W, m.H, m.TW, bad);
    return cudaGetLastError();
}

}  // namespace relo
