// TAM scoring (Eq. 22-31), and the stand-alone launch of the scan
// preparation (scan_prep.cuh) for batches that cast no rays.
//
// k_tam: one warp per (survivor, orientation m).  For each valid beam i the
// endpoint cell is hypothesis + round-half-up(R_i * D_{(b_i + m) mod N_s} /
// 2^46); its clamped squared distance b = min(d2, C) is read from the padded
// field, whose border holds C (off-map endpoints take d = d_max), so the read
// needs no bounds test.  The field is stored in bands of 8 rows (field_index):
// a cache line holds an 8 x 8 block of cells, so the endpoints of
// neighbouring beams share lines whichever way the contour runs, and an
// endpoint's offset from its hypothesis depends on the hypothesis only
// through its band phase (y + P) % 8.  The field holds not b but its code
// (field_code): the rank of b among the values that a clamped squared distance
// can take, as a positive fp16 bit pattern.  Ranks order like the values, so the
// likelihood l (Eq. 23), which falls strictly as b grows, falls with the rank:
// the descending sort of Eq. 24 is the ascending order of ranks.  The warp finds
// the k-th smallest rank by bisection with register-resident codes, two beams
// per instruction, and the top-k sum of l is
// sum_{b <= b_k} l(b) - (#{b <= b_k} - k) l(b_k), the count being the one the
// search ends on.  A shared-memory table holds l(b) and sqrt(C) - sqrt(b) by
// rank; the exact integer sum of b comes from the latter (its root is within
// 0.002 of an integer's), and the warp evaluates Eq. 27-30 and, after the block's
// orientations, one lane per orientation takes the exponential and Eq. 31:
//     wp = exp(Lbar),  d_max - dbar = res * sum(sqrt(C) - sqrt(b)) / N,
//     s_d = min(d_max - dbar, d_max - d_min) / (d_max - d_min),
//     var = res^2 * sum(b) / N - dbar^2,  c = exp(-var / 2),
//     T = cbrt(wp * s_d * c).
// Summing sqrt(C) - sqrt(b) (never negative) instead of sqrt(b) keeps s_d
// accurate when dbar is close to d_max.  Each score is written out and folded
// into a per-survivor 64-bit key (the score's order-preserving code, then
// smaller m) with atomicMax: that is the orientation argmax of Eq. 22.
//
// The scoring metric can be switched to those the paper compares TAM with:
// TAM_mean = (wp + s_d + c) / 3 (Eq. 34) from the same components, and the
// likelihood-field sum wp_LF = sum of l over every valid beam (Eq. 32) or its
// normalised form (exp(wp_LF / N) s_d)^(1/2) (Eq. 33), which keep every beam
// (k = N: no retention and no search).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "relo_internal.h"
#include "scan_prep.cuh"

namespace relo {

namespace {

constexpr unsigned kFull = 0xffffffffu;
// The likelihood table in shared memory.  An 8-byte entry's bank pair would be its rank mod 16, and a warp's lookups
// then serialise on the banks that its ranks share (3.0 to 3.2 wavefronts per lookup of 32 where 2 move the bytes,
// counted over both workloads; 2, 4 or 8 copies of the table make it worse, since lanes with the same rank no longer
// share a read).  With kLutCopies copies, entry by entry, each lane of a half-warp reads its own copy, which lies in its
// own bank pair, and no lookup conflicts.  505 ranks and the entry of no beam (C = 1600) take 65 KB that way, one CTA per
// SM; tables whose copies do not fit, maps with different tables in one launch and calls too small to repay the filling
// keep one.  TAM, us, with 16 copies and with one, 1024 survivors x 720 orientations x 1440 beams: C = 100 812 / 797, 400
// 843 / 846, 1600 868 / 876, 2500 878 / 885, 3600 919 / 891, 4096 919 / 894 (their copies leave room for fewer stages),
// 6400 and 8100 (one copy in any case) 901 and 903; 256 x 360 x 1081: C = 400 104 / 105, 1600 109 / 111, 4096 118 / 113.
constexpr int kLutCopies = 16;

// The smallest rank b in [0, C] with count_le(b) >= k, given count_le(C) = n_C >= k
// (C the last rank: every valid beam is <= C); cnt receives count_le(b).  hint < 0: bisection
// over [0, C].  Otherwise the search starts at hint: two counts confirm an
// unchanged answer; else it gallops away from hint in doubling steps to a
// bracket [lo, hi] with count_le(lo - 1) < k <= count_le(hi) and bisects it.
// The count at hi is carried along, so the answer's count costs nothing.
template <typename F>
__device__ __forceinline__ int kth_smallest(F &&count_le, int k, int C, int n_C, int hint, int &cnt) {
    int lo = 0, hi = C, c_hi = n_C;
    if (hint >= 0) {
        const int ch = count_le(hint);
        if (ch >= k) {
            const int cm = hint == 0 ? 0 : count_le(hint - 1);
            if (cm < k) {
                cnt = ch;
                return hint;
            }
            hi = hint - 1;
            c_hi = cm;
            for (int step = 1;; step <<= 1) {
                const int p = hi - step;
                if (p < 0) {
                    lo = 0;
                    break;
                }
                const int cp = count_le(p);
                if (cp < k) {
                    lo = p + 1;
                    break;
                }
                hi = p;
                c_hi = cp;
            }
        } else {
            lo = hint + 1;   // count_le(lo - 1) < k
            for (int step = 1;; step <<= 1) {
                const int p = lo + step - 1;
                if (p >= C) break;   // hi = C
                const int cp = count_le(p);
                if (cp >= k) {
                    hi = p;
                    c_hi = cp;
                    break;
                }
                lo = p + 1;
            }
        }
    }
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const int cm = count_le(mid);
        if (cm >= k) {
            hi = mid;
            c_hi = cm;
        } else {
            lo = mid + 1;
        }
    }
    cnt = c_hi;
    return lo;
}

// Per-lane stride of the endpoint offsets in shared memory: slot s of lane l
// (beam 32 s + l) sits at l * stride + s, so a lane reads four offsets with one
// 16-byte load; stride / 4 odd keeps the eight lanes of each load phase on
// distinct banks.
__host__ __device__ constexpr int tam_offs_stride(int vpl) {
    return ((vpl + 3) & ~3) + ((((vpl + 3) & ~3) / 4) % 2 == 0 ? 4 : 0);
}

// CTA (request, 0) does the scan preparation of scan_prep.cuh and all CTAs
// (request, y) share the fill of its TAM scores with NaN; this launch serves
// batches whose requests all read resident synthesized scans (otherwise the
// ray-cast launch does the same work first).
__global__ void __launch_bounds__(1024) k_scan_prep(const ReqDesc *__restrict__ reqs) {
    chain_wait();
    chain_go();
    const ReqDesc &d = reqs[blockIdx.x];
    scan_prep_fill(d, blockIdx.y, gridDim.y);
    if (blockIdx.y == 0) scan_prep_request(d);
}


// Work is split into tasks (request, chunk of survivors of one band phase,
// block of kTamQ consecutive orientations); the top-K launch builds the chunks
// on the device (tam_offsets.cuh).  A CTA holds a few staged tasks in shared
// memory: the block's endpoint offsets for the chunk's phase (computed from the
// request's table of endpoint cells) and the task's constants, beside the
// likelihood table.  Its warps run through the stages without a CTA barrier:
// each takes survivors of the stage one by one from a shared counter and scores
// them over the block's orientations (every gather one add to the survivor's
// base), and moves on to the next stage when none is left; the last warp to
// leave a stage takes the next task from the launch's counter and stages it
// there while the others work on the next one.  What bounds the kernel is the
// L1 data path (gathers, table lookups, offsets) and, for the shorter scans,
// the latency of the searches; with three CTA barriers per task every warp
// waited for the slowest search of its task, and a table copy and offsets for
// each of 4 to 6 CTAs per SM left the gathers a third of L1.  TAM, us, before
// and with the stages: 256 survivors x 360 orientations x 1081 beams 140 -> 117,
// 1024 x 720 x 1440 1127 -> 1060, 16 mixed requests 2733 -> 2140; with ranks,
// conflict-free lookups and one CTA per SM 112, 975 and 1973 (the L1 data path
// is then 95% busy in the 1024 x 720 launch).
//
// Selection.  The k-th smallest clamped d2 of a survivor rarely changes from
// one orientation to the next (neighbouring orientations see nearly the same
// contour), so each orientation after the block's first starts from the
// previous answer h: two counts confirm it (#{b <= h} >= k and #{b <= h-1} <
// k); otherwise the search gallops away from h in doubling steps and bisects
// the bracket.  Every step is a warp-wide count, and the result is the same
// smallest b with #{b' <= b} >= k as a bisection over [0, C].
constexpr int kTamQ = 4;
constexpr int kTamStages = 8;   // at most

// Warps of the SM's CTA by values-per-lane class: the register budget they leave each other (64 for up to 24 values, then
// 72, 80 and 96; fewer spill) against the warps that hide the gathers.  Measured (TAM, us): 18 values 32 / 30 / 28 warps
// 101 / 102 / 103; 30 values 32 / 28 / 24 177 / 175 / 176; 34 values 32 / 28 / 24 / 20 202 / 198 / 197 / 204; 38 values
// 220 / 213 / 213 / 213; 46 values 32 / 28 / 24 / 22 / 20 / 16 (1024 x 720) 1152 / 1009 / 975 / 989 / 975 / 1070; 64
// values 28 / 24 / 20 / 16 395 / 360 / 327 / 384.  An even share of the four schedulers counts: 24 and 20, not 22.
__host__ __device__ constexpr int tam_warps(int vpl) { return vpl <= 24 ? 32 : vpl <= 30 ? 28 : vpl <= 40 ? 24 : 20; }

// One staged task.
struct TamTask {
    unsigned long long full;   // mbarrier: completes when the stage is filled
    const uint16_t *field;
    const int2 *perm;          // the chunk's survivors: (position, base of the cell's column in its band)
    float *T;
    unsigned long long *best_key;
    const float2 *lut_src;     // the table the stage's copy came from (it stays when the next task shares it)
    int n;                     // survivors, -1 when there are no more tasks
    int q0, nq, n_orient;
    int N, k, top, C, fine;    // top: the last rank, C's
    float root_C;              // sqrt(C), an integer
    float inv_k, res_N, span, inv_span, res2_N, d_max;   // 1 / k, res / N, span of Eq. 29, res^2 / N
    int next, left;            // the next survivor to take; warps that have left the stage
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Waits for phase parity of the barrier.  Gives up after two seconds (a staging takes microseconds), so that a fault
// of this protocol would end the launch with an error instead of hanging it.
__device__ __forceinline__ bool wait_full(unsigned long long *bar, uint32_t parity) {
    const uint32_t addr = smem_u32(bar);
    unsigned long long start = 0;
    for (;;) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(addr), "r"(parity)
                     : "memory");
        if (ok) return true;
        unsigned long long now;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
        if (!start) start = now;
        else if (now - start > 2000000000ull) return false;
    }
}

// Stages task `task` of the launch (or, past the last, its end) by the threads tid, tid + nt, ...: the caller
// synchronises them, records the returned table in lut_src and completes the stage's barrier.
template <int VPL>
__device__ __forceinline__ const float2 *stage_task(const ReqDesc *__restrict__ reqs, int R, const TamSeg *__restrict__ segs,
                                                    const int *s_base, int task, TamTask &t, float2 *lut,
                                                    int lut_tables, int copies, int *offs,
                                                    int tid, int nt) {
    constexpr int kS = tam_offs_stride(VPL);
    if (task >= s_base[R]) {
        if (tid == 0) t.n = -1;
        return t.lut_src;
    }
    int lo = 0, hi = R - 1;   // the request whose tasks hold this one: last r with s_base[r] <= task
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_base[mid] <= task) lo = mid;
        else hi = mid - 1;
    }
    const ReqDesc &d = reqs[lo];
    const int local = task - s_base[lo];
    const int nblk = (d.n_orient + kTamQ - 1) / kTamQ;
    const int4 ck = d.tam_chunks[d.chunk_cnt[segs[lo].batch_lo] + local / nblk];   // (phase, first, end)
    const int q0 = (local % nblk) * kTamQ, nq = min(kTamQ, d.n_orient - q0);
    const float2 *src = lut_tables > 1 || !t.lut_src ? d.lut_rank : t.lut_src;
    if (t.lut_src != src)
        for (int i = tid, sh = copies > 1 ? 4 : 0; i < (d.n_rank + 1) * copies; i += nt) lut[i] = __ldg(src + (i >> sh));
    {
        // the block's endpoint cells (packed x, y offsets), nq x 32 x kS contiguous, to field offsets from a cell of
        // the chunk's band phase (field_index is linear in x, and in y through the bands crossed)
        const int Wp8 = 8 * d.Wp, ph = ck.x;
        const int4 *from = reinterpret_cast<const int4 *>(d.tam_offs + (size_t)q0 * 32 * kS);
        int4 *to = reinterpret_cast<int4 *>(offs);
        const int n4 = nq * 32 * kS / 4;
        auto off = [&](int p) {
            const int v = ph + (p >> 16);
            return 8 * (int)(short)p + Wp8 * (v >> 3) + (v & 7);
        };
#pragma unroll 4
        for (int i = tid; i < n4; i += nt) {
            const int4 p = __ldg(from + i);
            to[i] = make_int4(off(p.x), off(p.y), off(p.z), off(p.w));
        }
    }
    if (tid == 0) {
        const int N = d.scan->n_valid;
        // the likelihood-field metrics (Eq. 32-33) keep every beam: no retention, no k-th value to find
        const int k = d.fine < kFineBaseline ? d.scan->k_ret : N;
        t.field = d.field;
        t.perm = d.surv_perm + ck.y;
        t.T = d.T;
        t.best_key = d.best_key;
        t.n = ck.z - ck.y;
        t.q0 = q0;
        t.nq = nq;
        t.n_orient = d.n_orient;
        t.N = N;
        t.k = k;
        t.top = d.n_rank - 1;
        t.C = d.C;
        t.root_C = sqrtf((float)d.C);
        t.fine = d.fine;
        t.inv_k = 1.0f / (float)k;
        t.res_N = d.res / (float)N;
        t.span = d.d_max - d.d_min;
        t.inv_span = 1.0f / (d.d_max - d.d_min);
        t.res2_N = d.res2 / (float)N;
        t.d_max = d.d_max;
        t.next = 0;
        t.left = 0;
    }
    return src;
}

__device__ __forceinline__ float2 lds_float2(uint32_t addr) {
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// The scores of one survivor (position s, base field pointer fh) over the orientations [ql, qh) of the staged block, by
// one warp.  lut0: the shared address that entry code 0 of this lane's copy of the table would have; stride: bytes
// between its entries.
template <int VPL>
__device__ __forceinline__ void score_survivor(const TamTask &tk, uint32_t lut0, uint32_t stride, const int *offs, int s,
                                               const uint16_t *__restrict__ fh, int ql, int qh) {
    constexpr int kS = tam_offs_stride(VPL);
    const int lane = threadIdx.x & 31;
    const int N = tk.N, k = tk.k, top = tk.top;
    const uint32_t none = kFieldBias + (uint32_t)top + 1u;   // table entry with zero weight
    const float root_C = tk.root_C;
    int hint = -1;   // the previous orientation's k-th smallest rank
    float e_arg = 0.0f, e_sd = 0.0f;   // lane qi: orientation qi's exponent and s_d
    for (int qi = ql; qi < qh; ++qi) {
        const int *ol = offs + (qi * 32 + lane) * kS;   // this lane's offsets, slot s = beam 32 s + lane
        unsigned sumb = 0u;
        float sgs = 0.0f, sl = 0.0f;
        int bk;
        int cle;   // #{b <= bk} over the valid beams
        uint32_t hv[VPL / 2];   // codes of slots 2t (low half) and 2t + 1
#pragma unroll
        for (int u = 0; u < (VPL + 3) / 4; ++u) {
            const int4 o4 = *reinterpret_cast<const int4 *>(ol + 4 * u);
            const int oo[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const int t = 2 * u + e / 2;   // pair of slots 2t, 2t + 1
                if (t < VPL / 2) {
                    const int i0 = (t << 6) + lane, i1 = i0 + 32;
                    uint32_t b0 = none, b1 = none;
                    if (i0 < N) b0 = (uint32_t)__ldg(fh + oo[e]);
                    if (i1 < N) b1 = (uint32_t)__ldg(fh + oo[e + 1]);
                    hv[t] = b0 | (b1 << 16);
                }
            }
        }
        // #{b > x} on a lane: f(b) - f(x) saturated to [0, 1] is 1 exactly when b > x (f maps rank b to the fp16 number
        // of bits kFieldBias + b, numbers >= 1024 at least 1 apart; the exact difference is then >= 1, else <= 0, and
        // rounding keeps both); then #{b <= x} over the warp is the 32 VPL slots less those (no-beam slots are > top)
        auto count_le = [&](int x) -> int {
            const unsigned short fxb = (unsigned short)(kFieldBias + (uint32_t)x);
            const __half2 fx = __halves2half2(__ushort_as_half(fxb), __ushort_as_half(fxb));
            // two chains (half the add latency); the low half starts at 1024, so the
            // total 1024 + c (c <= 64) has the fp16 bits 0x6400 + c
            __half2 acc0 = __halves2half2(__ushort_as_half((unsigned short)0x6400), __float2half(0.0f));
            __half2 acc1 = __float2half2_rn(0.0f);
#pragma unroll
            for (int t = 0; t < VPL / 2; t += 2) {
                acc0 = __hadd2(acc0, __hsub2_sat(*reinterpret_cast<const __half2 *>(&hv[t]), fx));
                if (t + 1 < VPL / 2)
                    acc1 = __hadd2(acc1, __hsub2_sat(*reinterpret_cast<const __half2 *>(&hv[t + 1]), fx));
            }
            const __half2 sum = __hadd2(acc0, acc1);
            const __half2 tot = __hadd2(sum, __lowhigh2highlow(sum));
            const int gt = __reduce_add_sync(kFull, (int)(__half_as_ushort(__low2half(tot)) & 0x3ffu));
            return 32 * VPL - gt;
        };
        if (tk.fine < kFineBaseline) {
            bk = kth_smallest(count_le, k, top, N, hint, cle);
        } else {
            bk = top;   // every valid beam
            cle = N;
        }
        const uint32_t bkb = kFieldBias + (uint32_t)bk;
        // b of an entry: (sqrt(C) - g)^2 is within 0.002 of it (g is rounded to 2^-18 at most, sqrt(C) exact), so adding
        // 1.5 2^23 leaves it as the low bits; the sum of those bit patterns, mod 2^32, is sum b + 32 VPL patterns of 0
        // + C for every slot without a beam (g = 0 there)
#pragma unroll
        for (int t = 0; t < VPL / 2; ++t) {
            const uint32_t p0 = hv[t] & 0xffffu, p1 = hv[t] >> 16;
            const float2 g0 = lds_float2(lut0 + p0 * stride), g1 = lds_float2(lut0 + p1 * stride);
            const float t0 = root_C - g0.y, t1 = root_C - g1.y;
            sgs += g0.y + g1.y;   // the entry of no beam adds zero
            sumb += __float_as_uint(fmaf(t0, t0, 12582912.0f)) + __float_as_uint(fmaf(t1, t1, 12582912.0f));
            if (p0 <= bkb) sl += g0.x;
            if (p1 <= bkb) sl += g1.x;
        }
        hint = bk;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sgs += __shfl_xor_sync(kFull, sgs, o);
            sl += __shfl_xor_sync(kFull, sl, o);
        }
        sumb = __reduce_add_sync(kFull, sumb) - 32u * VPL * 0x4b400000u - (unsigned)(tk.C * (32 * VPL - N));
        {
            // Eq. 27-30 from the warp totals every lane holds; the top-k sum of l is every
            // b <= bk less the cle - k ties at bk beyond the k-th; lane qi keeps what its
            // orientation's score still needs: for TAM the exponent of exp(Lbar) exp(-var / 2)
            // and s_d
            const float topsum = sl - (float)(cle - k) * lds_float2(lut0 + bkb * stride).x;
            const float lbar = topsum * tk.inv_k;
            const float dd = tk.res_N * sgs;   // d_max - dbar
            const float dbar = tk.d_max - dd;
            const float var = fmaxf(tk.res2_N * (float)(int)sumb - dbar * dbar, 0.0f);
            const float sd = fminf(dd, tk.span) * tk.inv_span;
            const int fine = tk.fine;
            float a = lbar - 0.5f * var;
            if (fine == kFineTamMean) a = expf(lbar) + expf(-0.5f * var);   // wp + c (Eq. 34)
            else if (fine == kFineBaseline) a = lbar;                       // wp_LF / N (Eq. 33)
            else if (fine == kFineLF) a = topsum;                           // wp_LF (Eq. 32)
            if (lane == qi) {
                e_arg = a;
                e_sd = sd;
            }
        }
    }
    if (lane >= ql && lane < qh) {   // the score of orientation q0 + lane
        const int q = tk.q0 + lane;
        const int fine = tk.fine;
        float T = cbrtf(expf(e_arg) * e_sd);                                   // TAM, Eq. 31
        if (fine == kFineTamMean) T = (e_arg + e_sd) * (1.0f / 3.0f);         // Eq. 34
        else if (fine == kFineBaseline) T = sqrtf(expf(e_arg) * e_sd);        // Eq. 33
        else if (fine == kFineLF) T = e_arg;                                  // Eq. 32
        tk.T[(size_t)s * tk.n_orient + q] = T;
        const unsigned long long key = ((unsigned long long)score_code(T) << 32) |
                                       (unsigned long long)(0xffffffffu - (unsigned)q);
        atomicMax(tk.best_key + s, key);
    }
}

template <int VPL>
__global__ void __launch_bounds__(tam_warps(VPL) * 32, 1) k_tam(const ReqDesc *__restrict__ reqs, int R,
                                                                TamSeg *__restrict__ segs, int stages, int lut_bytes,
                                                                int lut_tables, int copies, BatchState *bs) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_base[kMaxBatchRequests + 1];
    __shared__ int s_warp[kMaxBatchRequests / 32];
    __shared__ TamTask task[kTamStages];
    constexpr int kWarps = tam_warps(VPL), kThreads = kWarps * 32;
    static_assert(kThreads >= kMaxBatchRequests, "a thread per request");
    constexpr int kOffs = kTamQ * 32 * tam_offs_stride(VPL);
    // one table for all stages when every request of the launch has the same, else one per stage
    auto lut_of = [&](int i) { return reinterpret_cast<float2 *>(smem + (lut_tables > 1 ? i * lut_bytes : 0)); };
    int *const offs0 = reinterpret_cast<int *>(smem + lut_tables * lut_bytes);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    chain_wait();
    chain_go();
    unsigned int *counter = reinterpret_cast<unsigned int *>(&segs[R].batch_lo);   // tasks taken after the first ones
    // each request's tasks: its chunks in the launch's batches x its orientation blocks (counted on the device); none
    // once it has terminated early or when it has no valid beam
    {
        const int r = threadIdx.x;
        int n = 0;
        if (r < R) {
            const TamSeg sg = segs[r];
            const ReqDesc &d = reqs[r];
            if (sg.batch_hi > sg.batch_lo && !d.state->done && d.scan->n_valid > 0)
                n = (d.chunk_cnt[sg.batch_hi] - d.chunk_cnt[sg.batch_lo]) * ((d.n_orient + kTamQ - 1) / kTamQ);
        }
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        if (r < kMaxBatchRequests && lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (r < kMaxBatchRequests) {
            int before = 0;
            for (int w = 0; w < warp; ++w) before += s_warp[w];
            if (r < R) s_base[r] = before + incl - n;
            if (r == R - 1) s_base[R] = before + incl;
        }
        if (threadIdx.x == 0)
            for (int i = 0; i < kTamStages; ++i) {
                task[i].lut_src = nullptr;
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&task[i].full)) : "memory");
            }
        __syncthreads();
    }
    auto arrive = [](TamTask &t) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&t.full)) : "memory");
    };
    for (int i = 0; i < stages; ++i) {   // the first tasks, staged by the whole CTA
        const float2 *src = stage_task<VPL>(reqs, R, segs, s_base, (int)blockIdx.x + i * (int)gridDim.x, task[i],
                                            lut_of(i), lut_tables, copies, offs0 + i * kOffs, threadIdx.x, kThreads);
        __syncthreads();
        if (threadIdx.x == 0) {
            // a table that all stages share is filled by the first task; the others take it as theirs
            for (int j = i; j < (lut_tables > 1 ? i + 1 : stages); ++j) task[j].lut_src = src;
            arrive(task[i]);
        }
        __syncthreads();
    }
    unsigned dead = 0;   // stages that hold no further task
    uint32_t parity = 0;
    for (int i = 0; dead != (1u << stages) - 1u;) {
        if (!(dead >> i & 1u)) {
            TamTask &t = task[i];
            float2 *lut = lut_of(i);
            int *offs = offs0 + i * kOffs;
            const uint32_t stride = 8u * (uint32_t)copies;
            const uint32_t lut0 = smem_u32(lut) + 8u * ((uint32_t)lane & (uint32_t)(copies - 1)) - kFieldBias * stride;
            if (!wait_full(&t.full, parity)) {
                if (lane == 0) atomicExch(&bs->error, 1u);
                return;
            }
            const int n = t.n;
            if (n < 0) {
                dead |= 1u << i;
            } else {
                // with too few survivors for the warps, each takes one orientation of one (its search then starts
                // from no neighbour's answer): the smallest calls wait for one score instead of a block's
                const int part = kTamQ * n <= kWarps ? 1 : t.nq, parts = part == 1 ? t.nq : 1;
                for (;;) {
                    int j = 0;
                    if (lane == 0) j = atomicAdd(&t.next, 1);
                    j = __shfl_sync(kFull, j, 0);
                    if (j >= n * parts) break;
                    const int js = parts == 1 ? j : j / parts, ql = parts == 1 ? 0 : j - js * parts;
                    const int2 sv = __ldg(t.perm + js);
                    score_survivor<VPL>(t, lut0, stride, offs, sv.x, t.field + (unsigned)sv.y, ql, ql + part);
                }
                __syncwarp();   // every lane's reads of the stage come before the warp counts itself out
                int last = 0;
                if (lane == 0) {
                    __threadfence_block();
                    last = atomicAdd(&t.left, 1) == kWarps - 1;
                    __threadfence_block();
                }
                last = __shfl_sync(kFull, last, 0);
                __syncwarp();
                if (last) {   // all warps have left: refill the stage
                    int nt = 0;
                    if (lane == 0) nt = (int)(atomicAdd(counter, 1u) + (unsigned)stages * gridDim.x);
                    nt = __shfl_sync(kFull, nt, 0);
                    const float2 *src = stage_task<VPL>(reqs, R, segs, s_base, nt, t, lut, lut_tables, copies, offs, lane, 32);
                    __syncwarp();
                    if (lane == 0) {
                        t.lut_src = src;
                        arrive(t);
                    }
                }
            }
        }
        if (++i == stages) {
            i = 0;
            parity ^= 1u;
        }
    }
}

template <int VPL>
cudaError_t run_tam(const ReqDesc *reqs, int R, TamSeg *segs, const TamPlan &tp, BatchState *bs, cudaStream_t s) {
    // plan_tam has asked for this shape's residency, which also lets the kernel use its shared memory
    return launch_chained(k_tam<VPL>, dim3((unsigned)tp.grid), tam_warps(VPL) * 32, tp.smem, s, reqs, R, segs,
                          tp.stages, tp.lut_bytes, tp.lut_tables, tp.copies, bs);
}

template <int VPL>
int tam_occupancy(size_t smem) {
    int occ = 0;
    if (resident_ctas((const void *)k_tam<VPL>, tam_warps(VPL) * 32, smem, &occ) != cudaSuccess) {
        cudaGetLastError();   // more than an SM has: no CTA fits
        return 0;
    }
    return occ;
}

#define RELO_TAM_VPLS(X)                                                                                       \
    X(8) X(10) X(12) X(14) X(16) X(18) X(20) X(22) X(24) X(26) X(28) X(30) X(32) X(34) X(36) X(38) X(40) X(42) X(44) \
        X(46) X(48) X(50) X(52) X(54) X(56) X(58) X(60) X(62) X(64)

int vpl_bucket(int max_beams) {
    const int need = (max_beams + 31) / 32;
#define RELO_TAM_PICK(V) \
    if (need <= V) return V;
    RELO_TAM_VPLS(RELO_TAM_PICK)
#undef RELO_TAM_PICK
    return -1;
}

int occupancy_for(int vpl, size_t smem) {
#define RELO_TAM_OCC(V) \
    if (vpl == V) return tam_occupancy<V>(smem);
    RELO_TAM_VPLS(RELO_TAM_OCC)
#undef RELO_TAM_OCC
    return 0;
}

}  // namespace

int tam_vpl_for(int max_beams) { return vpl_bucket(max_beams); }

cudaError_t launch_scan_prep(const ReqDesc *reqs, int R, cudaStream_t s) {
    return launch_chained(k_scan_prep, dim3((unsigned)R, 8), 1024, 0, s, reqs);
}

// The launch for the batches [batch_lo[r], batch_hi[r]) of every request:
// its kernel class (values per lane for the longest scan), its table and
// stages, and a grid of one CTA per SM; the tasks are counted by the kernel
// from the device-built chunk tables.  chunk: survivors of a usual task; luts: 1
// when all requests share one likelihood table (of max_rank ranks at most);
// poses: survivors x orientations of the launch.  segs: R entries and the task
// counter.
//
// A stage is refilled once its slowest survivor is done, so the stages together hold about twice the survivors that
// the warps work on, never fewer than two stages if they fit.  The copied table wants two stages beside it and a
// launch that gives a warp several poses.
TamPlan plan_tam(const int *batch_lo, const int *batch_hi, int R, int max_beams, int max_rank, int n_sm, int chunk,
                 int luts, long long poses, TamSeg *segs) {
    TamPlan tp{0, 0, vpl_bucket(max_beams), 0, 1, 0, 1, 1};
    if (tp.vpl < 0) return tp;
    const size_t table = (size_t)(max_rank + 1) * sizeof(float2);
    const size_t offs = (size_t)kTamQ * 32 * tam_offs_stride(tp.vpl) * sizeof(int);
    const int want = std::min(kTamStages, std::max(3, (9 * tam_warps(tp.vpl) + 4 * chunk - 1) / (4 * chunk)));
    const bool many = luts == 1 && poses >= 4ll * 32 * n_sm;
    for (int copies = many ? kLutCopies : 1; copies >= 1 && !tp.smem; copies /= kLutCopies) {
        const size_t lut = (table * copies + 15) & ~(size_t)15;
        for (int st = want; st >= (copies > 1 ? 2 : 1) && !tp.smem; --st) {
            const size_t bytes = lut * (luts > 1 ? st : 1) + st * offs;
            if (bytes > 220 * 1024 || occupancy_for(tp.vpl, bytes) < 1) continue;
            tp.stages = st;
            tp.smem = bytes;
            tp.copies = copies;
            tp.lut_bytes = (int)lut;
        }
    }
    if (!tp.smem) {
        tp.vpl = -1;
        return tp;
    }
    tp.lut_tables = luts > 1 ? tp.stages : 1;
    bool any = false;
    for (int r = 0; r < R; ++r) {
        segs[r] = TamSeg{batch_lo[r], batch_hi[r]};
        any = any || batch_hi[r] > batch_lo[r];
    }
    segs[R] = TamSeg{0, 0};
    tp.total_tasks = any ? 1 : 0;
    tp.grid = n_sm;
    return tp;
}

int tam_offs_stride_for(int vpl) { return tam_offs_stride(vpl); }

cudaError_t launch_tam(const ReqDesc *reqs, int R, TamSeg *segs, const TamPlan &tp, BatchState *bs, cudaStream_t s) {
    if (tp.total_tasks <= 0) return cudaSuccess;
#define RELO_TAM_RUN(V)                                                                 \
    if (tp.vpl == V)                                                                    \
        return run_tam<V>(reqs, R, segs, tp, bs, s);
    RELO_TAM_VPLS(RELO_TAM_RUN)
#undef RELO_TAM_RUN
    return cudaErrorInvalidValue;
}

}  // namespace relo
