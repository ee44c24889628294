// The exact squared EDT of a grid from its occupancy tiles, shared by the map
// precompute (edt.cu) and the allocation-free entry point (edt_noalloc.cu).
//
// d2(x, y) = min over occupied (x', y') of (x - x')^2 + (y - y')^2 separates
// into g(x', y), the distance to the nearest occupied cell of column x', and
// the row minimum d2(x, y) = min over x' of (x - x')^2 + g(x', y)^2.
//
// k_edt_tiles reads the grid once, a thread per 8x8 tile, and writes the tiles'
// occupancy words and, per segment of kSegTiles tile rows, the first and last
// occupied row of every column.  k_edt_spans gives every column of every tile
// row its nearest occupied rows above and below (4 bytes per 8 cells; searching
// for them in the next kernel cost it more than half its time in dependent
// loads).  k_edt_band takes bands of 8 rows: g of a column from its bits and
// spans, then the minimum over the columns on packed 16-bit squares, two rows
// per instruction.  The column distances never go to memory.
//
// 16 bits hold a squared distance up to 181 cells.  Cells that no column within
// kReach proves to be nearer than that are left to k_edt_far, which does the
// same in 32 bits for the bands that have any (open areas with more than 8.8 m
// of clearance at 5 cm).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "relo_internal.h"

namespace {

constexpr int kSegTiles = 8;          // tile rows per column segment
constexpr uint32_t kCap = 0x7fffu;    // "no occupied cell within 181 rows": kCap + dx^2 fits 16 bits up to dx = 181
constexpr int kReach = 176;           // columns to each side that k_edt_band looks at, for every cell
constexpr int kHalo = kReach + 4;     // and those its blocks of 4 may touch
constexpr int kNear2 = (kReach + 1) * (kReach + 1);   // a result up to this is final
constexpr int kFarMark = -2;          // d2 of a cell left to k_edt_far

// Occupancy words, bit 8 (y & 7) + (x & 7), of tiles [TH][TW]; the segments' first and last occupied rows (-1: none),
// [ceil(TH / kSegTiles)][W]; per tile row and column, the nearest occupied rows above and below the tile row (-1: none),
// [TH][W]; per band, whether k_edt_far has work (TH + 1 bands at most); which tiles have no occupied cell and lie inside
// the map (nullptr: not wanted), a bit per tile, [TH][ceil(TW / 32)].
struct EdtTiles {
    uint64_t *words;
    short2 *summ;
    short2 *span;
    int *far;
    uint32_t *empty;
    int W, H, TW, TH;
};

__host__ __device__ inline int edt_summary_rows(int H) { return ((H + 7) / 8 + kSegTiles - 1) / kSegTiles; }

// 8 cells from byte offset idx of the grid, 4 + 4: cells past the grid's end read 0.  Aligned words, so any width and
// any base address; only the words at the ends of the grid are put together from bytes.
__device__ __forceinline__ uint2 load8(const int8_t *__restrict__ grid, size_t idx, size_t cells, bool vec) {
    if (vec) return __ldg(reinterpret_cast<const uint2 *>(grid + idx));
    const uintptr_t a = reinterpret_cast<uintptr_t>(grid + idx), a0 = a & ~(uintptr_t)3;
    if (a0 >= reinterpret_cast<uintptr_t>(grid) && a0 + 12 <= reinterpret_cast<uintptr_t>(grid + cells)) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(a0);
        const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
        const unsigned sh = 8u * (unsigned)(a & 3);
        return make_uint2(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh));
    }
    uint32_t v[2] = {0u, 0u};
    for (int i = 0; i < 8; ++i)
        if (idx + i < cells) v[i >> 2] |= (uint32_t)(uint8_t)grid[idx + i] << (8 * (i & 3));
    return make_uint2(v[0], v[1]);
}

// bit i set where byte i (signed) is at least 65
__device__ __forceinline__ uint32_t occupied4(uint32_t v) {
    const uint32_t t = ((v & 0x7f7f7f7fu) + 0x3f3f3f3fu) & ~v & 0x80808080u;   // bit 7 of each such byte
    return ((t >> 7) * 0x01020408u >> 24) & 0xfu;
}

// the 8 rows of column c of a tile word, row u at bit u
__device__ __forceinline__ uint32_t column_bits(uint64_t word, int c) {
    return (uint32_t)(((word >> c) & 0x0101010101010101ull) * 0x0102040810204080ull >> 56);
}

// One thread per tile, 32 x 8 tiles per CTA.  FRAMES(word with the cells outside the map set, tx, ty) takes the tile for
// the caller's further layouts; copy (if not null; needs vec) receives the grid.
template <typename F>
__device__ __forceinline__ void edt_tiles(const int8_t *__restrict__ grid, const EdtTiles &t, bool vec, int8_t *copy,
                                          F &&frames) {
    static_assert(kSegTiles == 8, "a CTA's tile rows are one segment");
    __shared__ uint64_t s_word[8][33];
    const int tx = blockIdx.x * 32 + threadIdx.x, ty = blockIdx.y * 8 + threadIdx.y;
    const size_t cells = (size_t)t.W * t.H;
    uint64_t word = 0ull;
    bool free = false;
    if (tx < t.TW && ty < t.TH) {
        uint2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int y = 8 * ty + u;
            v[u] = make_uint2(0u, 0u);
            if (y < t.H) v[u] = load8(grid, (size_t)y * t.W + 8 * tx, cells, vec);
        }
        const int cols = min(8, t.W - 8 * tx), rows = min(8, t.H - 8 * ty);
        const uint64_t inside = (0x0101010101010101ull * ((1u << cols) - 1u)) & (rows < 8 ? (1ull << 8 * rows) - 1ull : ~0ull);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (copy && 8 * ty + u < t.H)
                *reinterpret_cast<uint2 *>(copy + (size_t)(8 * ty + u) * t.W + 8 * tx) = v[u];
            word |= (uint64_t)(occupied4(v[u].x) | occupied4(v[u].y) << 4) << (8 * u);
        }
        word &= inside;
        t.words[(size_t)ty * t.TW + tx] = word;
        frames(word | ~inside, tx, ty);
        free = (word | ~inside) == 0ull;
        if (tx == 0) t.far[ty] = 0;
        if (tx == 0 && ty == 0) t.far[t.TH] = 0;
    }
    if (t.empty) {   // a warp is 32 tiles of a row
        const unsigned bal = __ballot_sync(0xffffffffu, free);
        if (threadIdx.x == 0 && ty < t.TH) t.empty[(size_t)ty * gridDim.x + blockIdx.x] = bal;
    }
    s_word[threadIdx.y][threadIdx.x] = word;
    __syncthreads();
    const int c = threadIdx.y * 32 + threadIdx.x, x = blockIdx.x * 256 + c;   // a column of the CTA's 256
    if (x < t.W) {
        int first = -1, last = -1;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t m = column_bits(s_word[b][c >> 3], c & 7);
            const int y = 8 * ((int)blockIdx.y * 8 + b);
            if (m) {
                if (first < 0) first = y + __ffs((int)m) - 1;
                last = y + 31 - __clz((int)m);
            }
        }
        t.summ[(size_t)blockIdx.y * t.W + x] = make_short2((short)first, (short)last);
    }
}

// A thread per (column, segment): the nearest occupied rows outside the segment from the other segments, then the
// segment's tile rows downwards and upwards.
__global__ void __launch_bounds__(128) k_edt_spans(EdtTiles t) {
    const int x = blockIdx.x * 128 + threadIdx.x, sgm = blockIdx.y, segs = gridDim.y;
    if (x >= t.W) return;
    uint32_t m[kSegTiles];
#pragma unroll
    for (int b = 0; b < kSegTiles; ++b) {
        const int ty = sgm * kSegTiles + b;
        m[b] = ty < t.TH ? column_bits(__ldg(t.words + (size_t)ty * t.TW + (x >> 3)), x & 7) : 0u;
    }
    // the nearest segments first, eight loads at a time (a corridor's columns may cross the whole map)
    int last = -1, next = -1;
    for (int k = 1; k <= sgm && last < 0; k += 8) {
        int v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = sgm - k - i >= 0 ? t.summ[(size_t)(sgm - k - i) * t.W + x].y : -1;
#pragma unroll
        for (int i = 7; i >= 0; --i) last = v[i] >= 0 ? v[i] : last;
    }
    for (int k = 1; sgm + k < segs && next < 0; k += 8) {
        int v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = sgm + k + i < segs ? t.summ[(size_t)(sgm + k + i) * t.W + x].x : -1;
#pragma unroll
        for (int i = 7; i >= 0; --i) next = v[i] >= 0 ? v[i] : next;
    }
    short below[kSegTiles];
#pragma unroll
    for (int b = kSegTiles - 1; b >= 0; --b) {
        below[b] = (short)next;
        if (m[b]) next = 8 * (sgm * kSegTiles + b) + __ffs((int)m[b]) - 1;
    }
#pragma unroll
    for (int b = 0; b < kSegTiles; ++b) {
        const int ty = sgm * kSegTiles + b;
        if (ty < t.TH) t.span[(size_t)ty * t.W + x] = make_short2((short)last, below[b]);
        if (m[b]) last = 8 * ty + 31 - __clz((int)m[b]);
    }
}

// The distances g of column x at the 8 rows y0 .. y0 + 7 (rows off the map included): g[u], far when no cell of the
// column is occupied.
__device__ __forceinline__ void column_distances(const EdtTiles &t, int x, int y0, int far, int (&g)[8]) {
    const int tx = x >> 3, c = x & 7, t0 = y0 >> 3, r0 = y0 & 7;
    // the band lies in tile rows t0 and t0 + 1, of which one may be off the map
    const bool has_a = t0 >= 0, has_b = t0 + 1 < t.TH;
    const uint64_t wa = has_a ? __ldg(t.words + (size_t)t0 * t.TW + tx) : 0ull;
    const uint64_t wb = has_b ? __ldg(t.words + (size_t)(t0 + 1) * t.TW + tx) : 0ull;
    int last = has_a ? t.span[(size_t)t0 * t.W + x].x : -1;             // above tile row t0
    int next = has_b ? t.span[(size_t)(t0 + 1) * t.W + x].y : -1;       // below tile row t0 + 1
    const uint32_t col = column_bits(wa, c) | column_bits(wb, c) << 8;   // rows 8 t0 .. 8 t0 + 15
    const uint32_t m = col >> r0 & 0xffu, above = col & ((1u << r0) - 1u), below = col >> (r0 + 8);
    if (above) last = 8 * t0 + 31 - __clz((int)above);
    if (below) next = y0 + 8 + __ffs((int)below) - 1;
    int d = last >= 0 ? y0 - 1 - last : far;   // at row y0 - 1
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        d = m >> u & 1u ? 0 : d + 1;
        g[u] = d;
    }
    d = next >= 0 ? next - (y0 + 8) : far;   // at row y0 + 8
#pragma unroll
    for (int u = 7; u >= 0; --u) {
        d = m >> u & 1u ? 0 : d + 1;
        g[u] = min(min(g[u], d), far);
    }
}

// Where the results go: d2 row-major [H][W] (-1 when the map has no occupied cell), and, if field is not null, the code
// of min(d2, C), code[0 .. C], in 8-row bands with a border of P cells (relo_internal.h, field_index).
struct EdtOut {
    int32_t *d2;
    uint16_t *field;
    const uint16_t *code;
    int C, P, Wp;
};

// CTA (strip of kCols columns, band).  The band's rows are those of one field band (y + P = 8 B .. 8 B + 7), so a
// column's results are contiguous there.  Shared memory holds the squares of the strip and kHalo columns to each side,
// rows two by two in a word.  A thread takes 4 columns x 8 rows (or, split in two, 4 rows) and goes outward in blocks of
// 4 columns to each side: a 16-byte load gives 4 columns' squares for two rows, and each pair of own and other column is
// one packed add-minimum, so a candidate costs half an instruction per cell and an eighth of a shared-memory word (one
// thread per cell, four columns at a time, took 250 instructions per cell at 45 candidates).  It stops when the next
// block is farther than its worst cell.  Bound by the ALU pipe (packed add-minimum runs at half rate).  With
// k_edt_spans: 65 us on 4001 x 3500, 13 on 1024 x 1024 (column pass and row pass: 129 and 16); strips of 512 columns x
// 4 rows or 2048 x 8 there: 62 and 59 against 56 for the band pass.
template <int kCols, int kSplit>
__global__ void __launch_bounds__(kCols / 4 * kSplit) k_edt_band(EdtTiles t, EdtOut o) {
    constexpr int kRow = kCols + 2 * kHalo, kGroups = kCols / 4, T = kGroups * kSplit, kPairs = 4 / kSplit;
    __shared__ __align__(16) uint32_t sq[4][kRow];
    extern __shared__ uint16_t s_code[];   // [C + 1], with a field
    if (o.field)
        for (int i = threadIdx.x; i <= o.C; i += T) s_code[i] = __ldg(o.code + i);
    const int B = (o.P >> 3) + (int)blockIdx.y, y0 = 8 * B - o.P, X0 = (int)blockIdx.x * kCols;
#pragma unroll 2
    for (int i = threadIdx.x; i < kRow; i += T) {
        const int x = X0 - kHalo + i;
        uint32_t v[4] = {kCap | kCap << 16, kCap | kCap << 16, kCap | kCap << 16, kCap | kCap << 16};
        if (x >= 0 && x < t.W) {
            int g[8];
            column_distances(t, x, y0, 1 << 20, g);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const uint32_t a = g[2 * p] > 181 ? kCap : (uint32_t)(g[2 * p] * g[2 * p]);
                const uint32_t b = g[2 * p + 1] > 181 ? kCap : (uint32_t)(g[2 * p + 1] * g[2 * p + 1]);
                v[p] = a | b << 16;
            }
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) sq[p][i] = v[p];
    }
    __syncthreads();
    const int grp = (int)threadIdx.x % kGroups, p0 = (int)threadIdx.x / kGroups * kPairs;
    const int x0 = X0 + 4 * grp;
    if (x0 >= t.W) return;
    const int c0 = kHalo + 4 * grp;
    uint32_t best[kPairs][4];   // [row pair][column]
#pragma unroll
    for (int p = 0; p < kPairs; ++p) {
        const uint4 w4 = *reinterpret_cast<const uint4 *>(&sq[p0 + p][c0]);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            best[p][i] = w[i];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c != i) best[p][i] = __viaddmin_u16x2(w[c], (uint32_t)((c - i) * (c - i)) * 0x10001u, best[p][i]);
        }
    }
    for (int j = 4; j <= kReach; j += 4) {
        uint32_t worst = 0u;
#pragma unroll
        for (int p = 0; p < kPairs; ++p)
            worst = __vmaxu2(worst, __vmaxu2(__vmaxu2(best[p][0], best[p][1]), __vmaxu2(best[p][2], best[p][3])));
        if ((uint32_t)((j - 3) * (j - 3)) >= max(worst & 0xffffu, worst >> 16)) break;
        uint32_t d[7];   // (j - 3 .. j + 3)^2 for both rows
#pragma unroll
        for (int k = 0; k < 7; ++k) d[k] = (uint32_t)((j + k - 3) * (j + k - 3)) * 0x10001u;
#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
            const uint4 r4 = *reinterpret_cast<const uint4 *>(&sq[p0 + p][c0 + j]);
            const uint4 l4 = *reinterpret_cast<const uint4 *>(&sq[p0 + p][c0 - j]);
            const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w}, l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    best[p][i] = __viaddmin_u16x2(r[c], d[3 + c - i], best[p][i]);
                    best[p][i] = __viaddmin_u16x2(l[c], d[3 + i - c], best[p][i]);
                }
        }
    }
    bool far = false;
    // 16-byte stores where every row of d2 is aligned for them: the allocation-free entry point's output is the caller's
    const bool whole = x0 + 4 <= t.W && (t.W & 3) == 0 && (reinterpret_cast<uintptr_t>(o.d2) & 15) == 0;
#pragma unroll
    for (int u = 0; u < 2 * kPairs; ++u) {
        const int y = y0 + 2 * p0 + u;
        if (y < 0 || y >= t.H) continue;
        int v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = (int)(best[u >> 1][i] >> (16 * (u & 1)) & 0xffffu);
            if (v[i] > kNear2) {
                v[i] = kFarMark;
                far = far || x0 + i < t.W;
            }
        }
        int32_t *out = o.d2 + (size_t)y * t.W + x0;
        if (whole) {
            *reinterpret_cast<int4 *>(out) = make_int4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (x0 + i < t.W) out[i] = v[i];
        }
    }
    if (far) t.far[blockIdx.y] = 1;   // every writer writes 1
    if (!o.field) return;
    // the code of min(d2, C), C's for the rows off the map (the border's value); what is left to k_edt_far is above kNear2
    const uint32_t C = (uint32_t)o.C, C2 = C | C << 16;
    uint32_t off[kPairs];   // halves to replace by C
#pragma unroll
    for (int p = 0; p < kPairs; ++p) {
        const int y = y0 + 2 * (p0 + p);
        off[p] = (y < 0 || y >= t.H ? 0xffffu : 0u) | (y + 1 < 0 || y + 1 >= t.H ? 0xffff0000u : 0u);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (x0 + i >= t.W) continue;
        uint32_t f[kPairs];
#pragma unroll
        for (int p = 0; p < kPairs; ++p) {
            const uint32_t b = (__vminu2(best[p][i], C2) & ~off[p]) | (C2 & off[p]);
            f[p] = (uint32_t)s_code[b & 0xffffu] | (uint32_t)s_code[b >> 16] << 16;
        }
        uint16_t *to = o.field + 8 * ((size_t)B * o.Wp + (x0 + i + o.P)) + 2 * p0;
        if constexpr (kPairs == 4) *reinterpret_cast<uint4 *>(to) = make_uint4(f[0], f[1], f[2], f[3]);
        else *reinterpret_cast<uint2 *>(to) = make_uint2(f[0], f[1]);
    }
}

// The cells that k_edt_band left.  A CTA takes a band that has any, puts its columns' distances into shared memory (16
// bits each; 8 rows, or 4 and 4 on the widest maps) and lists the groups of 4 columns of a row with a cell to do, which
// its threads then share evenly.  A group goes outward in blocks of 4 columns as above, in 32 bits, until the next block
// is farther than its worst cell.  (One thread per cell of a row, 512 at a time over whole rows, spent 615 us on the
// 4096 x 4096 warehouse, whose far cells lie in one strip along its edge; this takes 114 us there by itself,
// most of it beside SMAD and the top-K.)
constexpr int kFarThreads = 256;
constexpr int kFarNone = 30000;               // no occupied cell in the column: its square is above any distance
constexpr int kFarList = 8 * kFarThreads;
constexpr size_t kFarStatic = sizeof(int) * kFarList + 64;   // k_edt_far's static shared memory at most

__host__ __device__ inline int far_rows(int W) { return W <= 8192 ? 8 : 4; }
__host__ __device__ inline int far_width(int W) { return (W + 3) & ~3; }

__global__ void __launch_bounds__(kFarThreads) k_edt_far(EdtTiles t, EdtOut o, int bands) {
    extern __shared__ __align__(16) uint16_t s_g[];   // [far_rows(W)][far_width(W)]
    __shared__ int s_list[kFarList];
    __shared__ int s_n;
    const int W4 = far_width(t.W), R = far_rows(t.W), groups = W4 / 4;
    for (int band = blockIdx.x; band < bands; band += gridDim.x) {
        if (!t.far[band]) continue;
        const int B = (o.P >> 3) + band, y0 = 8 * B - o.P;
        for (int u0 = 0; u0 < 8; u0 += R) {
            __syncthreads();   // the previous rows are done
            for (int x = threadIdx.x; x < W4; x += kFarThreads) {
                int g[8] = {kFarNone, kFarNone, kFarNone, kFarNone, kFarNone, kFarNone, kFarNone, kFarNone};
                if (x < t.W) column_distances(t, x, y0, kFarNone, g);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u >= u0 && u < u0 + R) s_g[(size_t)(u - u0) * W4 + x] = (uint16_t)g[u];
            }
            if (threadIdx.x == 0) s_n = 0;
            __syncthreads();
            const int items = R * groups;
            int n = 0;   // groups on the list: the barrier's own count, since the next round's appends change s_n at once
            for (int i0 = 0; i0 < items; i0 += kFarThreads) {
                const int it = i0 + (int)threadIdx.x, u = it / groups, x0 = 4 * (it - u * groups), y = y0 + u0 + u;
                bool any = false;
                if (it < items && y >= 0 && y < t.H) {
                    for (int i = 0; i < 4; ++i) any = any || (x0 + i < t.W && o.d2[(size_t)y * t.W + x0 + i] == kFarMark);
                    if (any) s_list[atomicAdd(&s_n, 1)] = u << 16 | x0;
                }
                n += __syncthreads_count(any);
                if (n > kFarList - kFarThreads || i0 + kFarThreads >= items) {   // the list is full, or complete
                    for (int k = threadIdx.x; k < n; k += kFarThreads) {
                        const int lu = s_list[k] >> 16, lx = s_list[k] & 0xffff, ly = y0 + u0 + lu;
                        const uint16_t *row = s_g + (size_t)lu * W4;
                        int best[4];
                        auto block = [&](int at, int dx0) {   // columns at .. at + 3, dx0 to the right of the group
                            const uint2 v = *reinterpret_cast<const uint2 *>(row + at);
                            const int g[4] = {(int)(v.x & 0xffffu), (int)(v.x >> 16), (int)(v.y & 0xffffu), (int)(v.y >> 16)};
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int g2 = g[c] * g[c];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const int dx = dx0 + c - i;
                                    best[i] = min(best[i], g2 + dx * dx);
                                }
                            }
                        };
#pragma unroll
                        for (int i = 0; i < 4; ++i) best[i] = kFarNone * kFarNone;
                        block(lx, 0);
                        for (int j = 4; lx - j >= 0 || lx + j < W4; j += 4) {
                            if ((j - 3) * (j - 3) >= max(max(best[0], best[1]), max(best[2], best[3]))) break;
                            if (lx + j < W4) block(lx + j, j);
                            if (lx - j >= 0) block(lx - j, -j);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            int32_t *out = o.d2 + (size_t)ly * t.W + lx + i;
                            if (lx + i >= t.W || *out != kFarMark) continue;
                            *out = best[i] >= kFarNone * kFarNone ? -1 : best[i];
                            if (o.field)
                                o.field[8 * ((size_t)B * o.Wp + (lx + i + o.P)) + u0 + lu] =
                                    __ldg(o.code + (best[i] > o.C ? o.C : best[i]));
                        }
                    }
                    __syncthreads();
                    if (threadIdx.x == 0) s_n = 0;
                    n = 0;
                    __syncthreads();
                }
            }
        }
    }
}

inline int edt_bands(int H, int P) { return ((H - 1 + P) >> 3) - (P >> 3) + 1; }

// The distance passes over tiles that k_edt_tiles wrote.  Strips of 1024 columns on large maps; narrower ones (a
// larger share of halo columns), with the rows of a band split between threads, while the wider leave SMs without work.
inline cudaError_t launch_edt_bands(const EdtTiles &t, const EdtOut &o, int n_sm, cudaStream_t s) {
    const int bands = edt_bands(t.H, o.P);
    k_edt_spans<<<dim3((t.W + 127) / 128, edt_summary_rows(t.H)), 128, 0, s>>>(t);
    auto strips = [&](int cols) { return (t.W + cols - 1) / cols; };
    const size_t code = o.field ? ((size_t)o.C + 1) * sizeof(uint16_t) : 0;   // at most 16 KB
    if ((long long)strips(1024) * bands >= 4ll * n_sm)
        k_edt_band<1024, 1><<<dim3(strips(1024), bands), 256, code, s>>>(t, o);
    else if ((long long)strips(512) * bands >= 2ll * n_sm)
        k_edt_band<512, 2><<<dim3(strips(512), bands), 256, code, s>>>(t, o);
    else
        k_edt_band<256, 2><<<dim3(strips(256), bands), 128, code, s>>>(t, o);
    const size_t smem = (size_t)far_rows(t.W) * far_width(t.W) * sizeof(uint16_t);
    if (smem > 48 * 1024 - kFarStatic) {   // without leave, a kernel has 48 KB for both
        const cudaError_t e = relo::allow_smem((const void *)k_edt_far, smem);
        if (e != cudaSuccess) return e;
    }
    k_edt_far<<<bands < 2 * n_sm ? bands : 2 * n_sm, kFarThreads, smem, s>>>(t, o, bands);
    return cudaGetLastError();
}

}  // namespace
