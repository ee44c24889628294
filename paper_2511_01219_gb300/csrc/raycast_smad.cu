// Ray-cast panoramic synthesized scans (Eq. 13) and SMAD (Eq. 16-20).
//
// Two kernels per batch.  k_cast casts every ray of every hypothesis, 32
// neighbouring directions per warp (lane = ray, so the lanes of a warp trace
// rays of similar length), into a per-request table of Q16 ranges.  Work
// items run over the hypotheses for one 32-direction chunk after another, so
// the warps in flight share a few directions' tables (they stay in L1).  k_smad
// then reads a hypothesis's row, forms chunk prefixes that
// give the cyclic prefix sum S of Eq. 17 at any index, evaluates the window
// sums of Eq. 18 for the orientations m of Eq. 15 with two lookups per FoV
// interval, and minimises the integer SMAD numerator |sum R_real - W_m| of
// Eq. 19 over m (Eq. 20; ties keep the smaller m; the shared denominator of
// the two means cancels from every comparison).
//
// Ray traversal.  From the hypothesis cell centre along the Q30 direction D,
// cells are entered in the order of the ray's grid-line crossings: with k x-
// and l y-crossings so far, x is stepped when (2k+1)|Dy| <= (2l+1)|Dx| (a
// corner tie steps x).  The recurrence tracks the difference e = (2l+1)|Dx| -
// (2k+1)|Dy| incrementally (e -= 2|Dy| after an x step, e += 2|Dx| after a y
// step); it always lies in [-2^31, 2^31), so a 32-bit integer holds it
// exactly.  The ray stops on leaving the map, on entering a cell whose centre
// lies beyond the maximum range, or on entering an occupied cell; the range of
// a hit is floor(sqrt(|d|^2 * 2^32)) (cells, Q16), else 0 (the placeholder of
// the invalid beam).  Occupancy comes from the 8x8-tile bitmap.  The default
// traversal (walk_ray) moves tile by tile with per-direction tables built
// once per (N_s, range limit); cast_ray steps cell by cell with the same
// recurrence.
//
// A panoramic synthesized scan depends only on the map, the hypothesis, the
// beam grid N_s and the range limit, not on the real scan.  The table a
// request casts into is either its scratch (kScanCast) or a resident table
// (kScanStore) that later requests with the same map, hypotheses, N_s and
// limit read without casting (kScanRead).
#include <cuda_runtime.h>

#include <algorithm>
#include <stdint.h>

#include "chain.cuh"
#include "relo_internal.h"
#include "scan_prep.cuh"

namespace relo {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint32_t isqrt_q16(int c2) {
    // floor(sqrt(c2 * 2^32)).  Up to 2^20 (1024 cells: every range limit of 50 m at 5 cm) the float estimate is off
    // by less than 8 (2 roundings of 2^-24 on a root below 2^26), so err = c2 2^32 - r^2 lies within 2 r 8 < 2^30 and
    // 32-bit arithmetic holds it (the low word of c2 2^32 is 0); a few steps then make it exact.
    if ((unsigned)c2 <= (1u << 20)) {
        uint32_t r = (uint32_t)(sqrtf((float)c2) * 65536.0f);
        int err = (int)(0u - r * r);
        while (err < 0) {
            --r;
            err += (int)(2u * r + 1u);
        }
        while (err > (int)(2u * r)) {
            err -= (int)(2u * r + 1u);
            ++r;
        }
        return r;
    }
    // else float estimate, one Newton correction, exact fix-up
    const unsigned long long N = (unsigned long long)(unsigned)c2 << 32;
    unsigned long long r = (unsigned long long)(sqrtf((float)c2) * 65536.0f);
    long long err = (long long)(N - r * r);
    r = (unsigned long long)((long long)r + (long long)__fdividef((float)err, 2.0f * (float)r + 1.0f));
    while (r * r > N) --r;
    while ((r + 1) * (r + 1) <= N) ++r;
    return (uint32_t)r;
}

// State of one ray's traversal.  advance() enters the next cell, or crosses a
// whole empty tile at once, and reports whether the ray has stopped.
//
// Empty tiles are crossed in one move.  Inside a tile whose 64-bit word is 0
// no cell can stop the ray except by leaving the map or the range, and both
// of those only grow along the ray, so jumping straight to the first cell
// past the tile gives the same answer as stepping through it.  With nx
// x-steps and ny y-steps left to the tile's x and y boundaries, the ray
// leaves through the x boundary iff its nx-th x crossing comes no later than
// its ny-th y crossing: e + 2(ny-1)|Dx| - 2(nx-1)|Dy| >= 0.  It then also
// makes the j y-steps whose crossings come strictly earlier, j = the smallest
// integer with 2 j |Dx| >= 2(nx-1)|Dy| - e; leaving through y, it makes the i
// x-steps whose crossings come no later (ties step x first), i = 0 if
// B = e + 2(ny-1)|Dx| < 0, else floor(B / (2|Dy|)) + 1.  Both counts are at
// most 7.
struct Ray {
    int ax, ay, sx, sy, e, cx, cy, adx, ady, c2, n, tile;
    unsigned long long word;

    __device__ __forceinline__ void init(int2 d, int hx, int hy, int tile0, unsigned long long word0) {
        ax = d.x < 0 ? -d.x : d.x;
        ay = d.y < 0 ? -d.y : d.y;
        sx = d.x > 0 ? 1 : -1;
        sy = d.y > 0 ? 1 : -1;
        e = ax - ay;
        cx = hx;
        cy = hy;
        adx = ady = c2 = n = 0;
        tile = tile0;
        word = word0;
    }

    // true once the ray stopped; *range = Q16 range of a hit, else 0
    __device__ __forceinline__ bool advance(const uint64_t *__restrict__ bits, int W, int H, int TW, int lim,
                                            uint32_t *range) {
        if (word == 0ull) {
            const int nx = sx > 0 ? 8 - (cx & 7) : (cx & 7) + 1;
            const int ny = sy > 0 ? 8 - (cy & 7) : (cy & 7) + 1;
            bool xexit;
            if (ay == 0) xexit = true;
            else if (ax == 0) xexit = false;
            else xexit = (long long)e + 2ll * (ny - 1) * ax - 2ll * (nx - 1) * ay >= 0;
            if (xexit) {
                // j = smallest integer with j * 2|Dx| >= A (0 when A <= 0), A = 2(nx-1)|Dy| - e
                const long long A = 2ll * (nx - 1) * ay - e;
                const long long dd = 2ll * ax;
                int j = 0;
                if (A > 0) {
                    j = (int)ceilf((float)A / (float)dd);
                    if ((long long)(j - 1) * dd >= A) --j;
                    if ((long long)j * dd < A) ++j;
                }
                e = (int)((long long)e - 2ll * nx * ay + 2ll * j * ax);
                cx += sx * nx;
                cy += sy * j;
                adx += nx;
                ady += j;
                n += nx + j;
            } else {
                // i = 0 if B < 0, else floor(B / (2|Dy|)) + 1, B = e + 2(ny-1)|Dx|
                const long long B = (long long)e + 2ll * (ny - 1) * ax;
                const long long dd = 2ll * ay;
                int i = 0;
                if (B >= 0) {
                    i = (int)floorf((float)B / (float)dd) + 1;
                    if ((long long)(i - 1) * dd > B) --i;
                    if ((long long)i * dd <= B) ++i;
                }
                e = (int)((long long)e + 2ll * ny * ax - 2ll * i * ay);
                cx += sx * i;
                cy += sy * ny;
                adx += i;
                ady += ny;
                n += ny + i;
            }
            c2 = adx * adx + ady * ady;
        } else if (e >= 0) {
            cx += sx;
            e = (int)((uint32_t)e - 2u * (uint32_t)ay);
            c2 += 2 * adx + 1;
            ++adx;
            ++n;
        } else {
            cy += sy;
            e = (int)((uint32_t)e + 2u * (uint32_t)ax);
            c2 += 2 * ady + 1;
            ++ady;
            ++n;
        }
        if ((unsigned)cx >= (unsigned)W || (unsigned)cy >= (unsigned)H || c2 > lim) {
            *range = 0u;
            return true;
        }
        const int t = (cy >> 3) * TW + (cx >> 3);
        if (t != tile) {
            tile = t;
            word = __ldg(bits + t);
        }
        if ((word >> (((cy & 7) << 3) | (cx & 7))) & 1ull) {
            *range = isqrt_q16(c2);
            return true;
        }
        return false;
    }
};

// whole ray: Q16 range (0 = no hit); *hit receives cy*W+cx or -1, *steps the cells entered
__device__ __forceinline__ uint32_t cast_ray(const uint64_t *__restrict__ bits, int W, int H, int TW, int lim, int hx,
                                             int hy, int2 d, int *hit, int *steps) {
    Ray ray;
    const int tile0 = (hy >> 3) * TW + (hx >> 3);
    ray.init(d, hx, hy, tile0, __ldg(bits + tile0));
    uint32_t r = 0u;
    while (!ray.advance(bits, W, H, TW, lim, &r)) {
    }
    *hit = r ? ray.cy * W + ray.cx : -1;
    *steps = ray.n;
    return r;
}

// Tile walk with the per-direction tables (RayTables).  The ray moves from
// tile to tile in its own frame, the map mirrored in x when D_x <= 0 (x' =
// 8 TW - 1 - x) and in y when D_y <= 0, so that it always travels towards +x
// and +y.  Each of the four frames is stored as a walk frame: cells outside
// the map are set and a last column and row of full tiles follow the map, so
// the first cell outside the map stops the ray like an occupied one and is
// recognised after the loop, which needs no bounds test per tile.
//
// The walk's state is the cell (cx, cy) alone: a cell k steps from the start
// (fx, fy) has cx + cy = fx + fy + k, so a table's step index of a far edge
// gives the other coordinate there with one subtraction, and the rows of the
// tables are linear in cx, cy and cx + cy (the start is folded into the bases).
// A tile is read through its box entry first (MapDev::reach, of the ray's slope class).  A box of empty tiles is left at
// its far edges, at the cell of step min(selx[|dx| at the x edge], sely[|dy| at the y edge]), since no cell inside it can
// stop the ray.  In a tile that is not empty (bit 0 of its entry), the word moved to the current cell is ANDed with the
// table's bit board of the cells still ahead; on a staircase that only moves +x and +y the cell order along the ray is
// the row-major bit order, so the lowest common bit is the hit; without one the ray leaves the tile as a box of one tile.
// Only such tiles load their word and board, together with the exit steps: two memory round trips and at most five loads
// per move.  Same cells, same hit, same range as cast_ray.
//
// Registers bound the kernel's warps: the tables share one allocation, and a
// map's boxes lie behind its words in another, so a direction holds two 64-bit
// bases and 32-bit indexes.
struct RayDir {   // what the walks of one direction share
    const uint64_t *__restrict__ bq;    // the direction's walk frame
    const uint64_t *__restrict__ mk;    // the tables (RayTables)
    unsigned rq;                        // the frame's boxes, 2-byte units from bq
    unsigned selx, sely, jm;            // the direction's column: 2-byte units from mk, 8-byte units from mk
    unsigned WB, ns;
    int mx, my;                         // 8 TW - 1 (mirrored in x) or -1; 8 TH - 1 or -1

    __device__ __forceinline__ void init(const uint64_t *bits, const uint16_t *reach, int TW, int TH,
                                         const RayTables &t, int ns_, int j, int2 d) {
        const bool xneg = d.x <= 0, yneg = d.y <= 0;
        mx = xneg ? 8 * TW - 1 : -1;
        my = yneg ? 8 * TH - 1 : -1;
        WB = (unsigned)TW + 1u;   // walk frame row, with the border column
        ns = (unsigned)ns_;
        const size_t frame = (size_t)((xneg ? 1 : 0) + (yneg ? 2 : 0)) * walk_frame_words(TW, TH);
        bq = bits + (size_t)TW * TH + frame;
        // the class of the slope: any class's boxes are empty, so the split need not be exact
        const float ax = fabsf((float)d.x), ay = fabsf((float)d.y), lo = fminf(ax, ay), hi = fmaxf(ax, ay);
        const int c = lo < 0.1051f * hi ? 0 : lo < 0.3249f * hi ? 1 : lo < 0.7265f * hi ? 2 : 3;
        const size_t box = frame * kReachClasses + (size_t)(ay > ax ? kReachClasses - 1 - c : c) * walk_frame_words(TW, TH);
        rq = (unsigned)(reach + box - reinterpret_cast<const uint16_t *>(bq));
        mk = t.mask;
        selx = t.selx + (unsigned)j;
        sely = t.sely + (unsigned)j;
        jm = (unsigned)j;
    }
    // between the map's x (y) and the frame's: the same involution both ways
    __device__ __forceinline__ int flip_x(int x) const { return mx < 0 ? x : mx - x; }
    __device__ __forceinline__ int flip_y(int y) const { return my < 0 ? y : my - y; }
};

__device__ __forceinline__ uint32_t walk_ray(const RayDir &r, int W, int H, unsigned kmax, int hx, int hy, int *hit,
                                             int *steps) {
    const int fx = r.flip_x(hx), fy = r.flip_y(hy);
    const unsigned S = (unsigned)(fx + fy);
    const uint16_t *__restrict__ sel = reinterpret_cast<const uint16_t *>(r.mk);
    const uint16_t *__restrict__ rch = reinterpret_cast<const uint16_t *>(r.bq);
    // unsigned 32-bit indexes: every table and map index fits, and the bases may wrap below zero before the row
    // term brings the sum back
    const unsigned bx = r.selx - (unsigned)fx * r.ns, by = r.sely - (unsigned)fy * r.ns, bm = r.jm - S * r.ns;
    // The loop only finds where the ray stops; the range is computed after it,
    // once for the whole warp, rather than in a divergent branch per lane.
    unsigned cx = (unsigned)fx, cy = (unsigned)fy;
    int stop;   // 1 hit (or left the map), 2 range limit
    for (;;) {
        const unsigned ti = (cy >> 3) * r.WB + (cx >> 3);
        const unsigned box = __ldg(rch + (r.rq + ti));
        const unsigned ex = (cx & ~7u) + (box & 0xf8u), ey = (cy & ~7u) + (box >> 8);   // the box's far edges
        const unsigned kx = __ldg(sel + (ex * r.ns + bx));
        const unsigned ky = __ldg(sel + (ey * r.ns + by));
        if (box & 1u) {   // not empty
            const uint64_t word = __ldg(r.bq + ti);
            const uint64_t board = __ldg(r.mk + ((cx + cy) * r.ns + bm));
            // move the current cell to bit 0; bits that wrap into the row below
            // sit in columns the board's column mask removes
            const unsigned lx = cx & 7u, ly = cy & 7u;
            const uint32_t cm = 0x01010101u * (0xffu >> lx);   // board columns dx <= 7 - lx, every row
            const uint64_t hm = board & (((uint64_t)cm << 32) | cm) & (word >> (lx + 8u * ly));
            if (hm) {
                const unsigned b = (unsigned)__ffsll((long long)hm) - 1u;
                cx += b & 7u;
                cy += b >> 3;
                stop = 1;
                break;
            }
        }
        const unsigned k = min(kx, ky);
        if (k == kSelNone) {   // the next cell lies beyond the range limit
            stop = 2;
            break;
        }
        const unsigned sk = S + k;   // cx + cy at the exit
        cx = kx < ky ? ex : sk - ey;
        cy = sk - cx;
    }
    const unsigned ax = (unsigned)r.flip_x((int)cx), ay = (unsigned)r.flip_y((int)cy);   // the map's cell
    *steps = stop == 2 ? __ldg(reinterpret_cast<const int32_t *>(r.mk) + kmax) + 1 : (int)(cx + cy - S);
    if (stop == 1 && (ax >= (unsigned)W || ay >= (unsigned)H)) stop = 3;   // the first cell outside the map
    *hit = stop == 1 ? (int)ay * W + (int)ax : -1;
    const int adx = (int)cx - fx, ady = (int)cy - fy;
    const uint32_t q = isqrt_q16(stop == 1 ? adx * adx + ady * ady : 0);   // a hit lies within the range limit
    return stop == 1 ? q : 0u;
}

// One thread per direction: the DDA of cast_ray from (0, 0), recorded.  The
// forward pass writes the step indexes into selx / sely and, as scratch, the
// kind of step k + 1 into mask row k; the backward pass turns those into the
// bit boards, mask(k) = cell k plus mask(k + 1) moved one cell back along
// step k + 1 (cells that fall off the 8x8 board are dropped).  mask rows must
// start at 0 and selx / sely at kSelNone.
__global__ void k_ray_tables(const int2 *__restrict__ D, int ns, int lim, uint64_t *mask, uint16_t *selx,
                             uint16_t *sely, int32_t *kmax) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ns) return;
    const int2 d = D[j];
    const int ax = d.x < 0 ? -d.x : d.x, ay = d.y < 0 ? -d.y : d.y;
    int e = ax - ay, adx = 0, ady = 0, k = 0;
    for (;;) {
        const bool xs = e >= 0;
        const long long nx = adx + (xs ? 1 : 0), ny = ady + (xs ? 0 : 1);
        if (nx * nx + ny * ny > (long long)lim) break;
        mask[(size_t)k * ns + j] = xs ? 1ull : 0ull;
        e = xs ? (int)((uint32_t)e - 2u * (uint32_t)ay) : (int)((uint32_t)e + 2u * (uint32_t)ax);
        adx = (int)nx;
        ady = (int)ny;
        ++k;
        if (xs) selx[(size_t)adx * ns + j] = (uint16_t)k;
        else sely[(size_t)ady * ns + j] = (uint16_t)k;
    }
    kmax[j] = k;
    uint64_t R = 1ull;
    for (int kk = k; kk >= 0; --kk) {
        if (kk < k) {
            const bool xs = mask[(size_t)kk * ns + j] != 0ull;
            R = 1ull | (xs ? ((R & ~0x8080808080808080ull) << 1) : (R << 8));
        }
        mask[(size_t)kk * ns + j] = kk == 0 ? (R & ~1ull) : R;   // the start cell itself is never tested
    }
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long t = __shfl_xor_sync(kFull, v, o);
        v = t < v ? t : v;
    }
    return v;
}

// shared memory of one SMAD warp: in-chunk prefixes [ns_pad + 32] of type P and chunk prefixes [ns_pad / 32 + 1]
template <typename P>
__host__ __device__ __forceinline__ size_t smad_inner_bytes(int ns_pad) {
    return ((size_t)(ns_pad + 32) * sizeof(P) + 7) & ~(size_t)7;
}
template <typename P>
__host__ __device__ __forceinline__ size_t smad_warp_bytes(int ns_pad) {
    return (smad_inner_bytes<P>(ns_pad) + (size_t)(ns_pad / 32 + 1) * 8 + 15) & ~(size_t)15;
}

// Casting.  The batch's rays form one list of work items (request r owns
// items [chunk_base_r, chunk_base_r + ceil(n_hyp_r / G) * N_s_pad / 32), G =
// cast_hyps hypotheses for one chunk of 32 directions each, hypothesis group
// by hypothesis group); every warp takes items from a device counter until
// none is left, casts its 32 neighbouring directions (lane = ray) from each
// of the item's hypotheses in turn (the directions' setup is shared) and
// writes their ranges into the request's scan table, 128 contiguous bytes per
// hypothesis.  No
// warp waits for another, so long and short rays, hypotheses and requests
// mix freely across the GPU.
constexpr int kCastThreads = 256;

template <int G>
__global__ void __launch_bounds__(kCastThreads, 5) k_cast(const ReqDesc *__restrict__ reqs, int R, int total_chunks,
                                                       BatchState *bs) {
    __shared__ int s_base[kMaxBatchRequests + 1];
    chain_wait();
    chain_go();
    const int lane = threadIdx.x & 31;
    // first the scan preparation, which the later stages need and the cast does
    // not: every CTA fills its share of the TAM scores, CTA r prepares request r
    for (int r = 0; r < R; ++r) scan_prep_fill(reqs[r], blockIdx.x, gridDim.x);
    if ((int)blockIdx.x < R) scan_prep_request(reqs[blockIdx.x]);
    for (int r = threadIdx.x; r < R; r += blockDim.x) s_base[r] = reqs[r].chunk_base;
    if (threadIdx.x == 0) s_base[R] = total_chunks;
    __syncthreads();
    unsigned long long my_steps = 0;
    for (;;) {
        int g = 0;
        if (lane == 0) g = (int)atomicAdd(&bs->cast_work, 1u);
        g = __shfl_sync(kFull, g, 0);
        if (g >= total_chunks) break;
        int lo = 0, hi = R - 1;   // last request whose chunk_base <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_base[mid] <= g) lo = mid;
            else hi = mid - 1;
        }
        const ReqDesc &d = reqs[lo];
        const int local = g - s_base[lo];
        const int nhc = (d.n_hyp + G - 1) / G;   // items per direction chunk (G = d.cast_hyps)
        const int jc = local / nhc;   // hypothesis-minor: concurrent warps share 32 directions' tables
        const int h0 = (local - jc * nhc) * G, h1 = min(h0 + G, d.n_hyp);
        const int j = (jc << 5) + lane;
        if (j < d.ns) {
            const int2 dir = d.D[j];
            uint32_t *out = d.scan_table + (size_t)h0 * d.ns + j;
            int hit, steps = 0;
            if (d.rt.mask) {
                RayDir r;
                r.init(d.bits, d.reach, d.TW, d.TH, d.rt, d.ns, j, dir);
                for (int h = h0; h < h1; ++h, out += d.ns) {
                    const int2 hc = d.hyps[h];
                    *out = walk_ray(r, d.W, d.H, d.rt.kmax + (unsigned)j, hc.x, hc.y, &hit, &steps);
                    my_steps += (unsigned)steps;
                }
            } else {
                for (int h = h0; h < h1; ++h, out += d.ns) {
                    const int2 hc = d.hyps[h];
                    *out = cast_ray(d.bits, d.W, d.H, d.TW, d.lim, hc.x, hc.y, dir, &hit, &steps);
                    my_steps += (unsigned)steps;
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_steps += __shfl_xor_sync(kFull, my_steps, o);
    if (lane == 0 && my_steps) atomicAdd(&bs->dda_steps, my_steps);
}

constexpr int kSmadLoads = 16;   // 32-range chunks a SMAD warp has in flight
constexpr int kSmadVecs = 6;      // 128-range blocks it has in flight with 16-byte loads

// The sum of row[x .. x + len) (no wrap) over the lanes' parts: 16 bytes per load between the aligned bounds when rows
// are aligned.
__device__ __forceinline__ long long lane_sum(const uint32_t *__restrict__ row, int x, int len, bool vec) {
    const int lane = threadIdx.x & 31, end = x + len;
    long long w = 0;
    int a = x, b = x;   // the aligned middle [a, b)
    if (vec) {
        a = min((x + 3) & ~3, end);
        b = max(a, end & ~3);
        const uint4 *__restrict__ v = reinterpret_cast<const uint4 *>(row);
#pragma unroll 4
        for (int i = (a >> 2) + lane; i < b >> 2; i += 32) {
            const uint4 q = __ldg(v + i);
            w += (long long)((unsigned long long)q.x + q.y + ((unsigned long long)q.z + q.w));
        }
    }
    for (int t = x + lane; t < a; t += 32) w += __ldg(row + t);
    for (int t = b + lane; t < end; t += 32) w += __ldg(row + t);
    return w;
}

// SMAD.  One warp per hypothesis, taken from a device counter over the
// batch's hypothesis list (request r owns slots [hyp_base_r, hyp_base_r +
// n_hyp_r)).  The warp turns the hypothesis's N_s ranges into exclusive prefixes
// of their 32-range chunk and the 64-bit prefix of the chunks; P(t) = chunkP[t /
// 32] + inner[t] is then the cyclic prefix sum of Eq. 17 for t in [0, N_s].  With
// rows that are 16-byte aligned (N_s a multiple of 4) a lane takes four
// neighbouring ranges of a 128-range block, so a chunk is 8 lanes and a block
// takes 3 shuffles for the scan and 4 for the chunk totals; one range per lane
// takes 6 shuffles for every 32 (the other rows).  The lanes split the
// orientations, evaluate Eq. 18-19 per m and reduce the minimum (Eq. 20).  With a
// single orientation (m = 0) the warp sums the row over the FoV intervals
// directly.  No CTA barrier: each warp owns its slice of shared memory.  Bound
// by issue and the latency of the row's loads.  16 requests of 4000 hypotheses
// on average x 540 to 2880 ranges: 304 us with one range per lane, 189 with
// four (2, 4 or 5 blocks in flight instead of 6: 227, 210, 202); 20000 x 1440
// row sums 62 and 37 us (115 MB: 17 us at the copy rate).
// P: the type of a chunk's prefixes, 32 bits while 32 ranges fit them (kSmadNarrowLim), else 64 (one range per lane): 5000
// hypotheses x 1440 ranges, 360 orientations, 19 us with a limit of 2040 cells, 34.5 with 2060 (973 by direct window sums).
template <typename P>
__global__ void __launch_bounds__(256) k_smad(const ReqDesc *__restrict__ reqs, int R, int total_hyp,
                                              BatchState *bs, int warp_bytes) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_base[kMaxBatchRequests + 1];
    chain_wait();
    chain_go();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = threadIdx.x; r < R; r += blockDim.x) s_base[r] = reqs[r].hyp_base;
    if (threadIdx.x == 0) s_base[R] = total_hyp;
    __syncthreads();
    unsigned char *mine = smem + (size_t)warp * warp_bytes;
    for (;;) {
        int g = 0;
        if (lane == 0) g = (int)atomicAdd(&bs->ray_work, 1u);
        g = __shfl_sync(kFull, g, 0);
        if (g >= total_hyp) break;
        int lo = 0, hi = R - 1;   // last request whose base <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_base[mid] <= g) lo = mid;
            else hi = mid - 1;
        }
        const ReqDesc &d = reqs[lo];
        const int h = g - s_base[lo];
        const int ns = d.ns, ns_pad = d.ns_pad, nch = ns_pad >> 5;
        const uint32_t *__restrict__ row = d.scan_table + (size_t)h * ns;
        if (d.n_m == 1) {
            // a single orientation, m = 0 (Eq. 20 when lambda >= 0.9): W_0 is the row summed over the FoV
            // intervals, read once and coalesced; no prefixes are needed
            long long w = 0;
            for (int k = 0; k < d.n_iv; ++k) {
                const int2 iv = d.iv[k];
                const int n0 = min(iv.y, ns - iv.x);   // up to the row's end, then from its start
                w += lane_sum(row, iv.x, n0, (ns & 3) == 0);
                if (n0 < iv.y) w += lane_sum(row, 0, iv.y - n0, (ns & 3) == 0);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
            if (lane == 0) {
                long long dnum = d.scan->sum_real - w;
                if (dnum < 0) dnum = -dnum;
                d.keys[h] = ((unsigned long long)dnum << kHypBits) | (unsigned long long)h;
                d.smad_num[h] = dnum;
                d.smad_m[h] = 0;
            }
            continue;
        }
        P *inner = reinterpret_cast<P *>(mine);
        long long *chunkP = reinterpret_cast<long long *>(mine + smad_inner_bytes<P>(ns_pad));
        long long carry = 0;
        if (sizeof(P) == 4 && (ns & 3) == 0) {
            const uint4 *__restrict__ row4 = reinterpret_cast<const uint4 *>(row);
            const int n4 = ns >> 2, nblk = (ns_pad + 127) >> 7;
            for (int b0 = 0; b0 < nblk; b0 += kSmadVecs) {
                uint4 r[kSmadVecs];
#pragma unroll
                for (int u = 0; u < kSmadVecs; ++u) {
                    const int i = ((b0 + u) << 5) + lane;
                    r[u] = i < n4 ? __ldg(row4 + i) : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
                for (int u = 0; u < kSmadVecs; ++u) {
                    if (b0 + u >= nblk) break;
                    const uint32_t s1 = r[u].x + r[u].y, s2 = s1 + r[u].z, all = s2 + r[u].w;
                    uint32_t sc = all;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(kFull, sc, o, 8);
                        if ((lane & 7) >= o) sc += t;
                    }
                    const uint32_t ex = sc - all;
                    const int j = ((b0 + u) << 7) + 4 * lane;
                    if (j < ns_pad)   // the last block may reach beyond the padded row
                        *reinterpret_cast<uint4 *>(inner + j) = make_uint4(ex, ex + r[u].x, ex + s1, ex + s2);
                    long long mine = carry;   // lane c < 4: the prefix of the block's chunk c
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t t = __shfl_sync(kFull, sc, 8 * c + 7);
                        if (lane > c) mine += t;
                        carry += t;
                    }
                    const int ch = 4 * (b0 + u) + lane;
                    if (lane < 4 && ch < nch) chunkP[ch] = mine;
                }
            }
        } else
        for (int c0 = 0; c0 < nch; c0 += kSmadLoads) {
            uint32_t r[kSmadLoads];
#pragma unroll
            for (int u = 0; u < kSmadLoads; ++u) {   // kSmadLoads loads in flight
                const int jj = ((c0 + u) << 5) + lane;
                r[u] = (c0 + u < nch && jj < ns) ? __ldg(row + jj) : 0u;
            }
#pragma unroll
            for (int u = 0; u < kSmadLoads; ++u) {
                if (c0 + u >= nch) break;
                P sc = r[u];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const P t = __shfl_up_sync(kFull, sc, o);
                    if (lane >= o) sc += t;
                }
                inner[((c0 + u) << 5) + lane] = sc - r[u];
                if (lane == 0) chunkP[c0 + u] = carry;
                carry += __shfl_sync(kFull, sc, 31);
            }
        }
        inner[ns_pad + lane] = 0;   // P(t) for t in [ns_pad, ns_pad + 32) adds nothing
        if (lane == 0) chunkP[nch] = carry;
        __syncwarp();
        const long long sum_real = d.scan->sum_real;
        unsigned long long best = ~0ull;
        for (int q = lane; q < d.n_m; q += 32) {
            const int m = q * d.n_enum;
            long long Wm = 0;
            for (int k = 0; k < d.n_iv; ++k) {
                const int2 iv = d.iv[k];
                int s0 = iv.x + m;
                if (s0 >= ns) s0 -= ns;
                const int e = s0 + iv.y;
                const long long p0 = chunkP[s0 >> 5] + inner[s0];
                if (e <= ns) {
                    Wm += chunkP[e >> 5] + inner[e] - p0;
                } else {
                    const int e2 = e - ns;
                    Wm += (chunkP[ns >> 5] + inner[ns] - p0) + (chunkP[e2 >> 5] + inner[e2]);
                }
            }
            long long dnum = sum_real - Wm;
            if (dnum < 0) dnum = -dnum;
            const unsigned long long key = ((unsigned long long)dnum << 20) | (unsigned)q;
            best = key < best ? key : best;
        }
        best = warp_min_u64(best);
        if (lane == 0) {
            const unsigned long long num = best >> 20;
            const int q = (int)(best & 0xfffffu);
            d.keys[h] = (num << kHypBits) | (unsigned long long)h;
            d.smad_num[h] = (long long)num;
            d.smad_m[h] = q * d.n_enum;
        }
        __syncwarp();   // the orientation reads are done before the next hypothesis rewrites the prefixes
    }
}

// Window tables.  k_win_build: one CTA per hypothesis of the build list.
// It scans the hypothesis's row into prefixes (as k_smad), evaluates W_m of
// Eq. 18 for every m of Theta, takes the SMAD minimum as k_smad does, and
// sorts the keys W_m << 13 | q ascending (bitonic, in shared memory) into the
// request's window table.
__device__ __forceinline__ int list_request(const int *s_base, int R, int g) {   // last request whose base <= g
    int lo = 0, hi = R - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_base[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename P>   // as in k_smad
__global__ void __launch_bounds__(256) k_win_build(const ReqDesc *__restrict__ reqs, int R, int total, int nm_pad_max) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_base[kMaxBatchRequests + 1];
    __shared__ unsigned long long s_best[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    chain_wait();
    chain_go();
    const int nwarps = blockDim.x >> 5;
    for (int r = threadIdx.x; r < R; r += blockDim.x) s_base[r] = reqs[r].wbuild_base;
    if (threadIdx.x == 0) s_base[R] = total;
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(smem);   // [nm_pad_max]
    unsigned char *rest = smem + (size_t)nm_pad_max * 8;
    for (int g = blockIdx.x; g < total; g += gridDim.x) {
        __syncthreads();   // s_base ready; the previous hypothesis is done with shared memory
        const int r = list_request(s_base, R, g);
        const ReqDesc &d = reqs[r];
        const int h = g - s_base[r];
        const int ns = d.ns, ns_pad = d.ns_pad, nch = ns_pad >> 5, n_m = d.n_m;
        P *inner = reinterpret_cast<P *>(rest);
        long long *chunkP = reinterpret_cast<long long *>(rest + smad_inner_bytes<P>(ns_pad));
        if (threadIdx.x < 32) inner[ns_pad + lane] = 0;
        const uint32_t *__restrict__ row = d.scan_table + (size_t)h * ns;
        for (int c = warp; c < nch; c += nwarps) {
            const int jj = (c << 5) + lane;
            const uint32_t rv = jj < ns ? __ldg(row + jj) : 0u;
            P sc = rv;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const P t = __shfl_up_sync(kFull, sc, o);
                if (lane >= o) sc += t;
            }
            inner[jj] = sc - rv;
            if (lane == 31) chunkP[c + 1] = (long long)sc;
        }
        __syncthreads();
        if (warp == 0) {
            long long carry = 0;
            for (int c0 = 0; c0 < nch; c0 += 32) {
                const int c = c0 + lane;
                long long v = c < nch ? chunkP[c + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const long long t = __shfl_up_sync(kFull, v, o);
                    if (lane >= o) v += t;
                }
                if (c < nch) chunkP[c + 1] = carry + v;
                carry += __shfl_sync(kFull, v, 31);
            }
            if (lane == 0) chunkP[0] = 0;
        }
        __syncthreads();
        int nm_pad = 1;
        while (nm_pad < n_m) nm_pad <<= 1;
        const long long sum_real = d.scan->sum_real;
        unsigned long long best = ~0ull;
        for (int q = threadIdx.x; q < nm_pad; q += blockDim.x) {
            if (q >= n_m) {
                keys[q] = ~0ull;
                continue;
            }
            const int m = q * d.n_enum;
            long long Wm = 0;
            for (int k = 0; k < d.n_iv; ++k) {
                const int2 iv = d.iv[k];
                int s0 = iv.x + m;
                if (s0 >= ns) s0 -= ns;
                const int e = s0 + iv.y;
                const long long p0 = chunkP[s0 >> 5] + inner[s0];
                if (e <= ns) {
                    Wm += chunkP[e >> 5] + inner[e] - p0;
                } else {
                    const int e2 = e - ns;
                    Wm += (chunkP[ns >> 5] + inner[ns] - p0) + (chunkP[e2 >> 5] + inner[e2]);
                }
            }
            keys[q] = ((unsigned long long)Wm << kWinQBits) | (unsigned)q;
            long long dnum = sum_real - Wm;
            if (dnum < 0) dnum = -dnum;
            const unsigned long long key = ((unsigned long long)dnum << 20) | (unsigned)q;
            best = key < best ? key : best;
        }
        best = warp_min_u64(best);
        if (lane == 0) s_best[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long b = s_best[0];
            for (int w = 1; w < nwarps; ++w) b = s_best[w] < b ? s_best[w] : b;
            const unsigned long long num = b >> 20;
            const int q = (int)(b & 0xfffffu);
            d.keys[h] = (num << kHypBits) | (unsigned long long)h;
            d.smad_num[h] = (long long)num;
            d.smad_m[h] = q * d.n_enum;
        }
        // bitonic sort of the keys, ascending
        for (int k = 2; k <= nm_pad; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < nm_pad; i += blockDim.x) {
                    const int p = i ^ j;
                    if (p > i) {
                        const unsigned long long a = keys[i], b = keys[p];
                        if ((a > b) == ((i & k) == 0)) {
                            keys[i] = b;
                            keys[p] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
        unsigned long long *out = d.win + (size_t)h * n_m;
        for (int i = threadIdx.x; i < n_m; i += blockDim.x) out[i] = keys[i];
    }
}

// k_win_read: one thread per hypothesis of the read list.  With S = sum
// R_real, the nearest W_m at or above S is the first key >= S << 13, and the
// nearest below is the key before it; each run of equal W_m starts with its
// smallest q, so the run start found by a second search is the smaller m of
// that value.  The closer of the two wins and a tie goes to the smaller m:
// exactly the minimum k_smad takes (Eq. 20).
__device__ __forceinline__ int lower_bound_u64(const unsigned long long *__restrict__ a, int n, unsigned long long x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(a + mid) < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(256) k_win_read(const ReqDesc *__restrict__ reqs, int R, int total) {
    __shared__ int s_base[kMaxBatchRequests + 1];
    chain_wait();
    chain_go();
    for (int r = threadIdx.x; r < R; r += blockDim.x) s_base[r] = reqs[r].wread_base;
    if (threadIdx.x == 0) s_base[R] = total;
    __syncthreads();
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const int r = list_request(s_base, R, g);
        const ReqDesc &d = reqs[r];
        const int h = g - s_base[r];
        const int n_m = d.n_m;
        const unsigned long long *keys = d.win + (size_t)h * n_m;
        const long long S = d.scan->sum_real;
        const unsigned long long qmask = (1ull << kWinQBits) - 1ull;
        const int pa = lower_bound_u64(keys, n_m, (unsigned long long)S << kWinQBits);
        long long dist = -1;
        unsigned q = 0;
        if (pa < n_m) {
            const unsigned long long ka = __ldg(keys + pa);
            dist = (long long)(ka >> kWinQBits) - S;
            q = (unsigned)(ka & qmask);
        }
        if (pa > 0) {
            const unsigned long long wb = __ldg(keys + pa - 1) >> kWinQBits;
            const long long db = S - (long long)wb;
            if (dist < 0 || db <= dist) {
                const int pb = lower_bound_u64(keys, pa - 1, wb << kWinQBits);   // start of the run of wb
                const unsigned qb = (unsigned)(__ldg(keys + pb) & qmask);
                if (dist < 0 || db < dist || qb < q) q = qb;
                dist = db;
            }
        }
        d.keys[h] = ((unsigned long long)dist << kHypBits) | (unsigned long long)h;
        d.smad_num[h] = dist;
        d.smad_m[h] = (int)q * d.n_enum;
    }
}

// One warp per (chunk of 32 directions, cell), cells fastest, as the ray cast
// orders its work: the warps in flight then share a few directions' tables in
// L1, and each stores whole 128-byte lines.
__global__ void __launch_bounds__(256) k_synth(RayArgs a, uint32_t *__restrict__ ranges, int32_t *__restrict__ hits) {
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int jc = (int)(warp / a.n_hyp), h = (int)(warp - (long long)jc * a.n_hyp), j = (jc << 5) + lane;
    if (j >= a.ns) return;
    const int2 hc = a.hyps[h];
    int hit, steps;
    uint32_t r;
    if (a.tab.mask) {
        RayDir dir;
        dir.init(a.bits, a.reach, a.TW, a.TH, a.tab, a.ns, j, a.D[j]);
        r = walk_ray(dir, a.W, a.H, a.tab.kmax + (unsigned)j, hc.x, hc.y, &hit, &steps);
    } else {
        r = cast_ray(a.bits, a.W, a.H, a.TW, a.lim, hc.x, hc.y, a.D[j], &hit, &steps);
    }
    ranges[(size_t)h * a.ns + j] = r;
    if (hits) hits[(size_t)h * a.ns + j] = hit;
}

}  // namespace

cudaError_t launch_cast(const ReqDesc *reqs, int R, int total_chunks, int cast_hyps, BatchState *bs, int n_sm,
                        int ctas_per_sm, cudaStream_t s) {
    if (R < 1 || R > kMaxBatchRequests) return cudaErrorInvalidValue;
    if (total_chunks <= 0) return cudaSuccess;
    // one instance per group size: a single hypothesis keeps the loop-free body
    void (*kern)(const ReqDesc *, int, int, BatchState *) =
        cast_hyps == 4 ? k_cast<4> : cast_hyps == 2 ? k_cast<2> : cast_hyps == 1 ? k_cast<1> : nullptr;
    if (!kern) return cudaErrorInvalidValue;
    int occ = 0;
    cudaError_t e = resident_ctas((const void *)kern, kCastThreads, 0, &occ);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    if (ctas_per_sm > 0 && ctas_per_sm < occ) occ = ctas_per_sm;   // a tuned launch shape
    const long long warps = (long long)total_chunks;
    long long grid = (long long)n_sm * occ;
    if (grid * (kCastThreads / 32) > warps) grid = (warps + kCastThreads / 32 - 1) / (kCastThreads / 32);
    if (grid < R) grid = R;   // one CTA per request for the scan preparation
    return launch_chained(kern, dim3((unsigned)grid), kCastThreads, 0, s, reqs, R, total_chunks, bs);
}

cudaError_t launch_smad(const ReqDesc *reqs, int R, int total_hyp, int max_ns_pad, bool wide, BatchState *bs, int n_sm,
                        cudaStream_t s) {
    if (R < 1 || R > kMaxBatchRequests) return cudaErrorInvalidValue;
    void (*const kern)(const ReqDesc *, int, int, BatchState *, int) = wide ? k_smad<unsigned long long> : k_smad<uint32_t>;
    // no request takes prefixes: no scratch
    const size_t wb = max_ns_pad <= 0 ? 0
                      : wide          ? smad_warp_bytes<unsigned long long>(max_ns_pad)
                                      : smad_warp_bytes<uint32_t>(max_ns_pad);
    // warps per CTA: the most resident warps per SM that shared memory allows
    // (a long row's scratch fills an SM before its thread limit; smaller CTAs
    // waste less of it), the larger CTA on ties
    int wpc = 0, occ = 0;
    for (int w = 8; w >= 1; --w) {
        if ((size_t)w * wb > (size_t)200 * 1024) continue;
        int o = 0;
        const cudaError_t e = resident_ctas((const void *)kern, w * 32, (size_t)w * wb, &o);
        if (e != cudaSuccess) return e;
        if (o * w > occ * wpc) {
            wpc = w;
            occ = o;
        }
    }
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const size_t smem = (size_t)wpc * wb;
    long long grid = (long long)n_sm * occ;
    const long long need = ((long long)total_hyp + wpc - 1) / wpc;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    return launch_chained(kern, dim3((unsigned)grid), wpc * 32, smem, s, reqs, R, total_hyp, bs, (int)wb);
}

cudaError_t launch_win_build(const ReqDesc *reqs, int R, int total, int max_ns_pad, int max_nm, bool wide,
                             cudaStream_t s) {
    if (R < 1 || R > kMaxBatchRequests) return cudaErrorInvalidValue;
    if (total <= 0) return cudaSuccess;
    void (*const kern)(const ReqDesc *, int, int, int) = wide ? k_win_build<unsigned long long> : k_win_build<uint32_t>;
    int nm_pad = 1;
    while (nm_pad < max_nm) nm_pad <<= 1;
    const size_t smem = (size_t)nm_pad * 8 + (size_t)(max_ns_pad / 32 + 1) * 8 +
                        (wide ? smad_inner_bytes<unsigned long long>(max_ns_pad) : smad_inner_bytes<uint32_t>(max_ns_pad));
    int occ = 0, dev = 0, n_sm = 0;
    cudaError_t e = resident_ctas((const void *)kern, 256, smem, &occ);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const int grid = total < n_sm * occ ? total : n_sm * occ;
    return launch_chained(kern, dim3((unsigned)grid), 256, smem, s, reqs, R, total, nm_pad);
}

cudaError_t launch_win_read(const ReqDesc *reqs, int R, int total, cudaStream_t s) {
    if (R < 1 || R > kMaxBatchRequests) return cudaErrorInvalidValue;
    if (total <= 0) return cudaSuccess;
    return launch_chained(k_win_read, dim3((unsigned)((total + 255) / 256)), 256, 0, s, reqs, R, total);
}

cudaError_t launch_ray_tables(const int2 *D, int ns, int lim, void *tab, cudaStream_t s) {
    const size_t mask_bytes = sizeof(uint64_t) * (size_t)ray_mask_rows(lim) * ns;
    const RayTables t = ray_tables_at(tab, ns, lim);
    uint64_t *mask = static_cast<uint64_t *>(tab);
    uint16_t *sel = static_cast<uint16_t *>(tab);
    cudaError_t e = cudaMemsetAsync(mask, 0, mask_bytes, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(sel + t.selx, 0xff, ray_tables_bytes(ns, lim) - mask_bytes, s);
    if (e != cudaSuccess) return e;
    k_ray_tables<<<(ns + 127) / 128, 128, 0, s>>>(D, ns, lim, mask, sel + t.selx, sel + t.sely,
                                                  static_cast<int32_t *>(tab) + t.kmax);
    return cudaGetLastError();
}

cudaError_t launch_synth(const RayArgs &a, uint32_t *ranges, int32_t *hit, cudaStream_t s) {
    if (a.n_hyp <= 0) return cudaSuccess;
    const long long warps = (long long)a.n_hyp * (a.ns_pad >> 5);
    k_synth<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(a, ranges, hit);
    return cudaGetLastError();
}

}  // namespace relo
