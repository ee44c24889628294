// Coarse ranking and batched selection.
//
// k_topk: the K hypotheses with the smallest SMAD (or CAER; Sec. III intro:
// the coarse metric orders all positions, the ordered set is cut into
// batches).  Keys are numerator << 21 | index, so they are unique and
// ascending key order is (numerator, index) order.  One CTA histograms the keys' digits (octave and the bits below its
// leading one), finds the digit holding the K-th smallest key, moves the keys up to that digit to their digit's range and
// counts each key's rank within it (keys are unique), keeping the first K; when a digit holds many keys it sorts them
// instead, and when too many share the K-th key's digit it falls back to an MSB-first radix select over 8-bit digits.
// The launch is a chain of short phases in one CTA per request, so latency bounds it, not bandwidth (20000 keys are
// 160 KB).  With digits of equal width the best keys shared one (5000 keys, K = 256: the radix select; 20000, K = 1024: a
// sorting network of 66 barriers, half of the launch).  Stage, us, before and now: 20.5 -> 12.2 and 41 -> 22.5; 16
// requests of up to 8000 keys, K = 512, 67 -> 23 (there the endpoint tables of the launch's other CTAs counted most).
//
// k_select_batch: after TAM has scored one batch, the per-hypothesis
// orientation argmax of Eq. 22 (already reduced by TAM into one 64-bit key per
// survivor), the batch's local top-k by TAM (ties to the earlier survivor) by
// rank counting, the running best over batches, and the early-termination
// flag once a batch's best reaches tau (Remark 2).
//
// With ICP refinement on, k_select_batch stops at the local top-k; k_icp
// (icp.cu) refines and re-scores those poses, and k_icp_best takes the
// running best and the early-termination test on the re-evaluated scores (the
// overview of Sec. III).
//
// The last selection launch also writes the selected pose and counters into
// each request's relo_result.
#include <cuda_runtime.h>

#include <algorithm>
#include <math.h>
#include <stdint.h>

#include "../../include/relo.h"
#include "chain.cuh"
#include "icp_points.cuh"
#include "relo_internal.h"
#include "tam_offsets.cuh"

namespace relo {

namespace {

constexpr int kTopkThreads = 1024;
// Keys a thread holds in registers from the one load to the last pass: up to kHold * kTopkThreads keys (20480) cost one
// read, all its loads in flight; more are read from memory in every pass, kLoads in flight.  The two ways are near each
// other: top-K stage, us, K = 256 / 1024: 20000 keys 20.2 / 21.8, 20480 20.7 / 22.1, 20481 22.4 / 23.7, 24000 22.7 / 24.5,
// 40000 30.4 / 31.6 (event times step by 2 us); with 10 keys a thread, so that all of these are read again, 20.2 / 22.5,
// 20.6 / 22.4, 20.6 / 22.6, 21.0 / 23.0 and 28.5 / 30.6.
constexpr int kHold = 20;
constexpr int kLoads = 8;

__device__ void bitonic_sort(unsigned long long *v, int n_pow2) {
    for (int k = 2; k <= n_pow2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n_pow2; i += blockDim.x) {
                int p = i ^ j;
                if (p > i) {
                    unsigned long long a = v[i], b = v[p];
                    bool up = (i & k) == 0;
                    if ((a > b) == up) {
                        v[i] = b;
                        v[p] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
}

constexpr int kRankMax = 512;   // up to this many keys, rank counting (one barrier) beats the sorting network

// The first K of n unique keys v[0 .. n) (v has room for the next power of two)
// in ascending order into the survivor list: by rank counting (each key's
// position is the number of smaller keys) for a few keys, else by sorting.
__device__ void order_out(unsigned long long *v, int n, int K, int32_t *survivors) {
    if (n <= kRankMax) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const unsigned long long me = v[i];
            int rank = 0;
            for (int k = 0; k < n; ++k) rank += v[k] < me ? 1 : 0;   // every thread reads the same v[k]
            if (rank < K) survivors[rank] = (int32_t)(me & ((1ull << kHypBits) - 1));
        }
        return;
    }
    int P = 1;
    while (P < n) P <<= 1;
    for (int i = n + threadIdx.x; i < P; i += blockDim.x) v[i] = ~0ull;
    __syncthreads();
    bitonic_sort(v, P);
    for (int i = threadIdx.x; i < K; i += blockDim.x) survivors[i] = (int32_t)(v[i] & ((1ull << kHypBits) - 1));
}

// First pass: a key's digit is its octave (the position of its highest set bit) and as many bits below that as 2048 digits
// for all octaves present allow.  The best SMADs of thousands of hypotheses lie far below the largest, so digits of equal
// width would put them all in one.
constexpr int kTopkBins = 2048;

struct KeyDigits {
    int lowest, bits;   // the lowest octave present; bits below the highest set bit
    // ascending with the key
    __device__ __forceinline__ int operator()(unsigned long long k) const {
        const int e = 63 - __clzll((long long)(k | 1ull));
        const unsigned long long m = e >= bits ? k >> (e - bits) : k << (bits - e);
        return ((e - lowest) << bits) | (int)((unsigned)m & ((1u << bits) - 1u));
    }
};
// Keys of one digit up to which ranks are counted within the digit: the longest digit is then one short loop per key,
// where the sorting network takes 55 to 66 barriers for 1024 to 2048 keys (42000 cycles
// for the 1024 of 20000).
constexpr int kDigitRankMax = 512;

// The first K keys of request d in ascending order into its survivor list,
// by one CTA (sm: the launch's dynamic shared memory).
__device__ __forceinline__ void topk_request(const ReqDesc &d, unsigned long long *sm, int Kp_cap) {
    const unsigned long long *__restrict__ keys = d.keys;
    const int n = d.n_hyp, K = d.K;
    unsigned long long *sortbuf = sm;                                          // [2 * Kp_cap]
    unsigned int *hist = reinterpret_cast<unsigned int *>(sm + 2 * Kp_cap);    // [kTopkBins]
    __shared__ int s_low, s_high;
    __shared__ int s_digit, s_below, s_cnt, s_sel;
    __shared__ unsigned int s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool held = n <= kHold * kTopkThreads;
    unsigned long long mine[kHold];
    // f(key, in) for the thread's keys; whole warps in every round, in false past the last key
    auto each_key = [&](auto f) {
        if (held) {
#pragma unroll
            for (int u = 0; u < kHold; ++u) {
                if (u * kTopkThreads >= n) break;
                f(mine[u], u * kTopkThreads + (int)threadIdx.x < n);
            }
            return;
        }
        for (int i0 = 0; i0 < n; i0 += kLoads * kTopkThreads) {
            unsigned long long k[kLoads];
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int i = i0 + u * kTopkThreads + (int)threadIdx.x;
                k[u] = i < n ? keys[i] : 0ull;
            }
#pragma unroll
            for (int u = 0; u < kLoads; ++u) f(k[u], i0 + u * kTopkThreads + (int)threadIdx.x < n);
        }
    };

    if (threadIdx.x == 0) { s_low = 63; s_high = 0; s_cnt = 0; }
    if (held) {
#pragma unroll
        for (int u = 0; u < kHold; ++u) {
            const int i = u * kTopkThreads + (int)threadIdx.x;
            mine[u] = i < n ? keys[i] : 0ull;
        }
    }
    for (int i = threadIdx.x; i < kTopkBins; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    int low = 63, top = 0;
    each_key([&](unsigned long long k, bool in) {
        const int e = 63 - __clzll((long long)(k | 1ull));
        if (in) {
            low = min(low, e);
            top = max(top, e);
        }
    });
    low = __reduce_min_sync(0xffffffffu, low);
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) {
        atomicMin(&s_low, low);
        atomicMax(&s_high, top);
    }
    __syncthreads();
    low = s_low;
    top = max(s_high, low);
    const KeyDigits digit{low, 31 - __clz(kTopkBins / (top - low + 1))};

    // One pass over the digits finds the digit b* of the K-th smallest key;
    // the keys with digit < b* are all in, those with digit b* are ordered with
    // them and the first K kept.
    each_key([&](unsigned long long k, bool in) {
        if (in) atomicAdd(&hist[digit(k)], 1u);
    });
    __syncthreads();
    bool long_digit;
    {
        const unsigned a = hist[2 * threadIdx.x], b = hist[2 * threadIdx.x + 1];   // 1024 threads x 2 bins
        unsigned incl = a + b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned v = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            s_warp[lane] = v - s_warp[lane];   // exclusive prefix of the warp totals
        }
        __syncthreads();
        const unsigned excl = s_warp[warp] + incl - (a + b);
        if (excl < (unsigned)K && excl + a + b >= (unsigned)K) {
            if (excl + a >= (unsigned)K) {
                s_digit = 2 * threadIdx.x;
                s_sel = (int)(excl + a);
            } else {
                s_digit = 2 * threadIdx.x + 1;
                s_sel = (int)(excl + a + b);
            }
        }
        hist[2 * threadIdx.x] = excl;   // where each digit's keys begin
        hist[2 * threadIdx.x + 1] = excl + a;
        __syncthreads();
        const int first = 2 * threadIdx.x;
        long_digit = __syncthreads_or((a > kDigitRankMax && first <= s_digit) || (b > kDigitRankMax && first < s_digit));
    }
    const int dstar = s_digit;
    const int n_sel = s_sel;   // keys with digit <= b*
    if (n_sel <= 2 * Kp_cap) {
        each_key([&](unsigned long long k, bool in) {
            const int g = digit(k);
            if (in && g <= dstar) sortbuf[atomicAdd(&hist[g], 1u)] = k;
        });
        __syncthreads();   // hist[g] is now where digit g ends
        if (long_digit) {
            order_out(sortbuf, n_sel, K, d.survivors);
            return;
        }
        for (int i = threadIdx.x; i < n_sel; i += blockDim.x) {
            const unsigned long long me = sortbuf[i];
            const int g = digit(me);
            const int lo = g ? (int)hist[g - 1] : 0, hi = (int)hist[g];
            int rank = lo;
            for (int k = lo; k < hi; ++k) rank += sortbuf[k] < me ? 1 : 0;
            if (rank < K) d.survivors[rank] = (int32_t)(me & ((1ull << kHypBits) - 1));
        }
        return;
    }

    // Many keys share the digit b*: MSB-first radix select over 8-bit digits.
    unsigned long long prefix = 0, mask = 0;
    int remaining = K;
    for (int shift = (top / 8) * 8; shift >= 0; shift -= 8) {
        __syncthreads();
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        each_key([&](unsigned long long k, bool in) {
            if (in && (k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
        });
        __syncthreads();
        if (threadIdx.x < 32) {
            unsigned int local = 0;
            for (int dg = 0; dg < 8; ++dg) local += hist[lane * 8 + dg];
            unsigned int incl = local;
            for (int o = 1; o < 32; o <<= 1) {
                unsigned int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            unsigned int excl = incl - local;
            bool here = excl < (unsigned)remaining && incl >= (unsigned)remaining;
            if (here) {
                unsigned int cum = excl;
                for (int dg = 0; dg < 8; ++dg) {
                    unsigned int c = hist[lane * 8 + dg];
                    if (cum + c >= (unsigned)remaining) {
                        s_digit = lane * 8 + dg;
                        s_below = (int)cum;
                        break;
                    }
                    cum += c;
                }
            }
        }
        __syncthreads();
        prefix |= (unsigned long long)s_digit << shift;
        mask |= 255ull << shift;
        remaining -= s_below;
    }
    // prefix is now the K-th smallest key; one slot reservation per warp
    each_key([&](unsigned long long k, bool in) {
        const bool take = in && k <= prefix;
        const unsigned bal = __ballot_sync(0xffffffffu, take);
        int base = 0;
        if (lane == 0 && bal) base = atomicAdd(&s_cnt, __popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) sortbuf[base + __popc(bal & ((1u << lane) - 1u))] = k;
    });
    __syncthreads();
    order_out(sortbuf, K, K, d.survivors);
}

// One CTA per request ranks it and then builds its TAM work order from the
// survivors; the CTAs after the first R compute the requests' TAM endpoint
// offsets and, for ICP, the beams' sensor-frame points meanwhile (they need the scan preparation, not the ranking).
__global__ void __launch_bounds__(kTopkThreads) k_topk(const ReqDesc *__restrict__ reqs, int Kp_cap, int R,
                                                       int max_n_orient, int off_block, int icp_chunks) {
    extern __shared__ __align__(16) unsigned long long sm[];
    chain_wait();
    chain_go();
    if ((int)blockIdx.x >= R) {
        const int blocks = (max_n_orient + off_block - 1) / off_block;
        for (int t = (int)blockIdx.x - R; t < R * blocks; t += (int)gridDim.x - R) {
            const ReqDesc &o = reqs[t / blocks];
            const int q = t % blocks * off_block;
            if (q < o.n_orient && !o.state->done && o.tam_offs) tam_offsets_block(o, q, min(off_block, o.n_orient - q));
        }
        for (int t = (int)gridDim.x - 1 - (int)blockIdx.x; t < R * icp_chunks; t += (int)gridDim.x - R)
            if (reqs[t / icp_chunks].icp_iters > 0) icp_points_chunk(reqs[t / icp_chunks], t % icp_chunks);
        return;
    }
    const ReqDesc &d = reqs[blockIdx.x];
    topk_request(d, sm, Kp_cap);
    __syncthreads();   // every survivor is written
    tam_chunks_one(d, reinterpret_cast<int2 *>(sm));   // room for 2 Kp_cap >= K cells
}

// The request's pose, score and counters into its relo_result (one thread).
__device__ void finalize_request(const ReqDesc &d) {
    relo_result r;
    const SelectState st = *d.state;
    const unsigned tb = (unsigned)(st.best >> 32);
    const int s = (int)(0xffffffffu - (unsigned)(st.best & 0xffffffffu));
    r.n_batches = st.n_batches;
    r.n_tam_evals = st.n_tam_evals;
    r.n_smad_evals = d.n_smad_evals;
    const bool failed = d.bs->error != 0u;
    if (failed || d.scan->n_valid <= 0 || st.n_batches == 0) {
        r.status = failed ? RELO_E_CUDA : RELO_E_NO_VALID_BEAMS;
        r.x = r.y = r.theta = r.tam = r.smad = 0.0;
        r.smad_num = 0;
        r.hyp = -1;
        r.m = -1;
        r.n_tam_evals = 0;
    } else {
        const int h = d.survivors[s];
        const int m = d.best_m[s];
        const int2 c = d.hyps[h];
        r.status = RELO_OK;
        r.hyp = h;
        r.m = m;
        r.tam = (double)score_of(tb);
        double th;
        if (d.icp_iters > 0) {   // the refined continuous pose
            const double *ps = d.ref_pose + 3 * (size_t)s;
            r.x = d.ox + ps[0];
            r.y = d.oy + ps[1];
            th = remainder(ps[2], 2.0 * M_PI);
        } else {
            r.x = d.ox + ((double)c.x + 0.5) * d.resd;
            r.y = d.oy + ((double)c.y + 0.5) * d.resd;
            th = (double)m * (2.0 * M_PI) / (double)d.ns;
        }
        if (th >= M_PI) th -= 2.0 * M_PI;
        r.theta = th;
        r.smad_num = d.smad_num[h];
        r.smad = (double)r.smad_num / d.fov / 65536.0 * d.resd;
    }
    *reinterpret_cast<relo_result *>(d.result) = r;
}

// one CTA per request: selection of batches batch_lo .. batch_hi - 1 (those the
// request has; with early termination none after it terminated).  Keys (TAM
// descending, then survivor position) are unique, so each survivor's rank is
// the number of smaller keys of its batch; ranks below L fill the local top-k
// directly.  Without early termination as many batches as fit v are ranked
// together: one by one each was another chain of loads and barriers
// (1024 survivors
// in 6 batches 22.5 -> 16.3 us, 16 requests of 512 in 3 batches 18 -> 14).  With last, the launch also writes every request's result.  With
// icp the launch stops at the local top-k and the counters: k_icp refines and
// re-scores them, k_icp_best takes their best.
__global__ void __launch_bounds__(1024) k_select_batch(const ReqDesc *__restrict__ reqs, int batch_lo, int batch_hi,
                                                       int last, int icp) {
    __shared__ unsigned long long v[kMaxBatch];
    __shared__ unsigned long long s_best[kMaxBatches];
    __shared__ int s_skip;
    chain_wait();
    chain_go();
    const ReqDesc &d = reqs[blockIdx.x];
    const bool early = d.early_stop;
    const int B = d.B, K = d.K, L = d.L;
    const int end = d.scan->n_valid > 0 ? min(batch_hi, d.n_batches) : batch_lo;
    const int step = early ? 1 : kMaxBatch / B;
    for (int first = batch_lo; first < end; first += step) {
        __syncthreads();   // the state updates of the batches before are done
        if (early) {
            if (threadIdx.x == 0) s_skip = d.state->done;
            __syncthreads();
            if (s_skip) break;
        }
        const int count = min(step, end - first);   // batches
        const int s_begin = first * B, n = min(K, s_begin + count * B) - s_begin;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int s = s_begin + i;
            const unsigned long long k = d.best_key[s];
            const unsigned tb = (unsigned)(k >> 32);
            const unsigned q = 0xffffffffu - (unsigned)(k & 0xffffffffu);
            d.best_m[s] = (int)q * d.n_enum;
            v[i] = ((unsigned long long)(~tb) << 32) | (unsigned)s;   // ascending = TAM desc, survivor asc
        }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const unsigned long long me = v[i];
            const int b = i / B, hi = min(n, (b + 1) * B);
            int rank = 0;
#pragma unroll 8
            for (int k = b * B; k < hi; ++k) rank += v[k] < me ? 1 : 0;
            if (rank < L) d.local[(size_t)(first + b) * L + rank] = (int)(me & 0xffffffffu);
            if (rank == 0) s_best[b] = ~me;   // (score, 2^32 - 1 - survivor)
        }
        for (int r = threadIdx.x; r < count * L; r += blockDim.x)
            if (r % L >= min(B, n - r / L * B)) d.local[(size_t)first * L + r] = -1;
        __syncthreads();
        if (threadIdx.x == 0) {
            SelectState st = *d.state;
            st.n_batches += count;
            st.n_tam_evals += (long long)n * d.n_orient;
            if (!icp) {
                for (int b = 0; b < count; ++b) {
                    if (s_best[b] > st.best) st.best = s_best[b];
                    if (early && (double)score_of((unsigned)(s_best[b] >> 32)) >= d.tau) st.done = 1;
                }
            }
            *d.state = st;
        }
    }
    if (last) {
        __syncthreads();   // the selection state of this launch is complete
        if (threadIdx.x == 0) finalize_request(d);
    }
}

// One warp per request, after k_icp: for batches batch_lo .. batch_hi - 1
// in order (each skipped when the request has fewer or already terminated),
// the best re-evaluated local top-k pose (ties to the earlier survivor) joins
// the running best, and early termination follows its score (the overview of
// Sec. III: the test is made on the re-evaluated score).  With last, the
// result.
__global__ void __launch_bounds__(32) k_icp_best(const ReqDesc *__restrict__ reqs, int batch_lo, int batch_hi, int last) {
    chain_wait();
    chain_go();
    const ReqDesc &d = reqs[blockIdx.x];
    const int lane = threadIdx.x;
    SelectState *st = d.state;
    if (d.scan->n_valid > 0) {
        bool done = st->done;
        unsigned long long best = st->best;
        for (int b = batch_lo; b < batch_hi && b < d.n_batches && !done; ++b) {
            unsigned long long top = 0ull;
            for (int i = lane; i < d.L; i += 32) {
                const int s = d.local[(size_t)b * d.L + i];
                if (s < 0) continue;
                const unsigned long long key = ((unsigned long long)score_code(d.reev[s]) << 32) |
                                               (0xffffffffu - (unsigned)s);
                top = key > top ? key : top;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long t = __shfl_xor_sync(0xffffffffu, top, o);
                top = t > top ? t : top;
            }
            if (top == 0ull) continue;
            if (top > best) best = top;
            if (d.early_stop && (double)score_of((unsigned)(top >> 32)) >= d.tau) done = true;
        }
        __syncwarp();   // every lane has read the state
        if (lane == 0) {
            st->best = best;
            st->done = done ? 1 : 0;
        }
    }
    if (last && lane == 0) finalize_request(d);
}

}  // namespace

cudaError_t launch_topk(const ReqDesc *reqs, int R, int max_n_hyp, int max_K, int max_n_orient, int icp_beams, int n_sm,
                        cudaStream_t s) {
    int Kp = 1;
    while (Kp < max_K) Kp <<= 1;
    const size_t smem = (size_t)2 * Kp * 8 + (size_t)kTopkBins * 4;
    const cudaError_t e = allow_smem((const void *)k_topk, smem);
    if (e != cudaSuccess) return e;
    // one CTA per SM for the offsets
    const int n_orient = std::max(max_n_orient, 1), n_off = std::max(1, std::min(R * n_orient, n_sm));
    // orientations per task: as many as leave every CTA a task, at most the loads a thread keeps in flight
    const int off_block = std::max(1, std::min(R * n_orient / n_off, kOffBlock));
    return launch_chained(k_topk, dim3((unsigned)(R + n_off)), kTopkThreads, smem, s, reqs, Kp, R, n_orient, off_block,
                          (icp_beams + 31) / 32);
}

cudaError_t launch_select_batch(const ReqDesc *reqs, int R, int batch_lo, int batch_hi, bool last, bool icp,
                                cudaStream_t s) {
    return launch_chained(k_select_batch, dim3((unsigned)R), 1024, 0, s, reqs, batch_lo, batch_hi, last ? 1 : 0,
                          icp ? 1 : 0);
}

cudaError_t launch_icp_best(const ReqDesc *reqs, int R, int batch_lo, int batch_hi, bool last, cudaStream_t s) {
    return launch_chained(k_icp_best, dim3((unsigned)R), 32, 0, s, reqs, batch_lo, batch_hi, last ? 1 : 0);
}

}  // namespace relo
