// CAER ranking (Eq. 21, Remark 5): for every hypothesis and orientation m of
// the SMAD set, sum over the beams |R_i - row[(b_i + m) mod N_s]| (invalid beams
// carry R = 0, as in SMAD), minimised over m (ties to the smaller m) and written
// like a SMAD numerator, so the ranking that follows is unchanged.  O(beams) per
// orientation, where SMAD's window sums are O(intervals).
//
// One warp per hypothesis.  A lane keeps kA consecutive orientations.  Along
// the beams of one residue class mod n_enum, the row value that orientation a
// meets at a beam is the one orientation a + 1 met at the beam before, so the
// lane's kA values slide by one: one shared-memory load and one beam's R serve
// kA differences.  The row is stored by residue class, so lanes read at a
// stride of kA words.  When the orientations need fewer than 32 lanes, the
// lanes split the beams as well.  Differences are added in 32 bits for as many
// beams as the range limit allows, then moved to 64.
//
// Bound by integer issue (a difference and its sum per beam and orientation;
// 487 M of them for 2500 hypotheses x 360 orientations x 541 beams: 78 us,
// 393 us with the lanes over the beams of one orientation at a time, which
// loaded the beam's index, its range and the row for every difference).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "relo_internal.h"

namespace relo {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kCaerWarps = 4;
constexpr int kA = 12;   // orientations per lane: 360 in one pass of a warp

// Adds the beams s0 .. s1 - 1 of one residue class: the beam's R is at rbeam + s * n_enum (cyclic in n_beams, rbeam the
// index of the class's first beam), the row value of orientation a at row[(k0 + s + a) mod no].
__device__ __forceinline__ void add_class(const int32_t *__restrict__ Rall, int n_beams, int rbeam, int n_enum,
                                          const uint32_t *row, int no, int k0, int s0, int s1, int room,
                                          unsigned (&acc)[kA], unsigned long long (&sum)[kA], int &held) {
    uint32_t w[kA];
    int kk = k0 + s0;   // < 2 no + beams of the class: reduced to the row value of orientation 0 at beam s0
    while (kk >= no) kk -= no;
#pragma unroll
    for (int a = 0; a < kA - 1; ++a) {
        w[a] = row[kk];
        kk = kk + 1 == no ? 0 : kk + 1;
    }
    int i = rbeam + s0 * n_enum;
    while (i >= n_beams) i -= n_beams;
    for (int s = s0; s < s1; s += kA) {
        if (held + kA > room) {
#pragma unroll
            for (int a = 0; a < kA; ++a) {
                sum[a] += acc[a];
                acc[a] = 0u;
            }
            held = 0;
        }
        held += kA;
#pragma unroll
        for (int j = 0; j < kA; ++j) {
            if (s + j < s1) {
                const unsigned R = (unsigned)__ldg(Rall + i);
                i += n_enum;
                if (i >= n_beams) i -= n_beams;
                w[(j + kA - 1) % kA] = row[kk];
                kk = kk + 1 == no ? 0 : kk + 1;
#pragma unroll
                for (int a = 0; a < kA; ++a) acc[a] = __usad(R, w[(j + a) % kA], acc[a]);
                if (room < kA) {   // ranges beyond 5459 cells: 32 bits hold one difference, not a block's
#pragma unroll
                    for (int a = 0; a < kA; ++a) {
                        sum[a] += acc[a];
                        acc[a] = 0u;
                    }
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kCaerWarps * 32) k_caer(const ReqDesc *__restrict__ reqs, int R, int total_hyp,
                                                          BatchState *bs, int warp_words) {
    extern __shared__ __align__(16) uint32_t s_rows[];
    __shared__ int s_base[kMaxBatchRequests + 1];
    chain_wait();
    chain_go();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = threadIdx.x; r < R; r += blockDim.x) s_base[r] = reqs[r].hyp_base;
    if (threadIdx.x == 0) s_base[R] = total_hyp;
    __syncthreads();
    uint32_t *row = s_rows + (size_t)warp * warp_words;   // [n_enum][no]: the row by residue class mod n_enum
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
        const int h = g - s_base[lo], ns = d.ns, n_enum = d.n_enum, no = d.n_orient, n = d.n_beams, n_m = d.n_m;
        const uint32_t *__restrict__ src = d.scan_table + (size_t)h * ns;
        {
            int c = lane % n_enum, k = lane / n_enum;
            const int dc = 32 % n_enum, dk = 32 / n_enum;
#pragma unroll 4
            for (int j = lane; j < ns; j += 32) {
                row[c * no + k] = __ldg(src + j);
                c += dc;
                k += dk;
                if (c >= n_enum) {
                    c -= n_enum;
                    ++k;
                }
            }
        }
        __syncwarp();
        // a difference is at most the longer of the two ranges, below (sqrt(lim) + 2) cells
        const int room = (int)(65535.0f / (sqrtf((float)d.lim) + 2.0f));
        unsigned long long best = ~0ull;
        for (int q0 = 0; q0 < n_m; q0 += 32 * kA) {
            // lanes over orientation groups (a power of two of them), the rest over the beams
            int lq = 1;
            while (lq < 32 && lq * kA < n_m - q0) lq <<= 1;
            const int parts = 32 / lq, part = lane / lq, qg = q0 + (lane & (lq - 1)) * kA;
            unsigned acc[kA];
            unsigned long long sum[kA];
#pragma unroll
            for (int a = 0; a < kA; ++a) {
                acc[a] = 0u;
                sum[a] = 0ull;
            }
            int held = 0;
            for (int v = 0; v < d.n_iv; ++v) {
                const int2 iv = d.iv[v];
                // the beam on the interval's first direction (b_cyc and Rall are in cyclic order, b_0 anywhere): the beam
                // whose direction lies (iv.x - b_0) mod N_s past the first's, found by bisection
                const int b0 = __ldg(d.b_cyc);
                int want = iv.x - b0;
                if (want < 0) want += ns;
                int bl = 0, bh = n - 1;
                while (bl < bh) {
                    const int mid = (bl + bh) >> 1;
                    int at = __ldg(d.b_cyc + mid) - b0;
                    if (at < 0) at += ns;
                    if (at < want) bl = mid + 1;
                    else bh = mid;
                }
                for (int r = 0; r < n_enum && r < iv.y; ++r) {
                    const int S = (iv.y - r + n_enum - 1) / n_enum;   // beams of this class
                    const int per = (S + parts - 1) / parts, s0 = min(S, part * per), s1 = min(S, s0 + per);
                    const int first = iv.x + r, c = first % n_enum, k0 = first / n_enum + qg;
                    int rb = bl + r;
                    if (rb >= n) rb -= n;
                    add_class(d.Rall, n, rb, n_enum, row + c * no, no, k0, s0, s1, room, acc, sum, held);
                }
            }
#pragma unroll
            for (int a = 0; a < kA; ++a) {
                unsigned long long e = sum[a] + acc[a];
                for (int o = lq; o < 32; o <<= 1) e += __shfl_xor_sync(kFull, e, o);
                const int q = qg + a;
                const unsigned long long key = e << 20 | (unsigned)q;
                if (q < n_m && key < best) best = key;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(kFull, best, o);
            best = t < best ? t : best;
        }
        if (lane == 0) {
            const unsigned long long num = best >> 20;
            d.keys[h] = (num << kHypBits) | (unsigned long long)h;
            d.smad_num[h] = (long long)num;
            d.smad_m[h] = (int)(best & 0xfffffu) * n_enum;
        }
        __syncwarp();   // the row reads are done before the next hypothesis rewrites it
    }
}

}  // namespace

cudaError_t launch_caer(const ReqDesc *reqs, int R, int total_hyp, int max_ns_pad, BatchState *bs, int n_sm,
                        cudaStream_t s) {
    if (R < 1 || R > kMaxBatchRequests || max_ns_pad < 1) return cudaErrorInvalidValue;
    const int warp_words = max_ns_pad;
    const size_t smem = (size_t)kCaerWarps * warp_words * 4;   // at most 128 KB
    int occ = 0;
    const cudaError_t e = resident_ctas((const void *)k_caer, kCaerWarps * 32, smem, &occ);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const long long need = ((long long)total_hyp + kCaerWarps - 1) / kCaerWarps;
    const long long grid = std::max(1ll, std::min((long long)n_sm * occ, need));
    return launch_chained(k_caer, dim3((unsigned)grid), kCaerWarps * 32, smem, s, reqs, R, total_hyp, bs, warp_words);
}

}  // namespace relo
