// TAM's inputs that the top-K launch prepares (select.cu): each request's
// work order (survivors grouped by band phase, in chunks), built by its
// ranking CTA once the survivors are known, and the endpoint offsets of its
// plan (Eq. 13's endpoint cells), computed
// by the other CTAs of the launch beside the ranking ones.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "relo_internal.h"

namespace relo {

// Every request's endpoint cells, once per batch: for orientation q (m = q
// n_enum) and valid beam i, the offsets round-half-up(R_i * D_{(b_i + m) mod
// N_s} / 2^46) per axis (each below 2^15), packed y << 16 | x, laid out
// [q][lane][slot] with the TAM kernel's per-lane stride, so one block of
// orientations is one contiguous span.  TAM turns a block's cells into field
// offsets for its task's band phase as it stages them: a table per phase (8
// times the bytes) cost the batched workload more to write and read back than
// those few operations per task.  One CTA writes the n <= kOffBlock
// orientations from q: a thread reads its beam once and has all their
// directions in flight, where a task per orientation was a chain of dependent
// loads for one store each (16 requests of 360 orientations: the launch 64
// -> 27 us).
constexpr int kOffBlock = 8;
__device__ __forceinline__ void tam_offsets_block(const ReqDesc &d, int q, int n) {
    const int N = d.scan->n_valid;
    const int kS = d.tam_stride, ns = d.ns, n_enum = d.n_enum;
    const int2 *__restrict__ D = d.D;
    int32_t *oq = d.tam_offs + (size_t)q * 32 * kS;
    // k walks an orientation's table in memory order (lane-major), so every store is coalesced
    for (int k = threadIdx.x; k < 32 * kS; k += blockDim.x) {
        const int i = (k % kS) * 32 + k / kS;   // the beam in slot k % kS of lane k / kS
        if (i >= N) continue;
        const int2 bR = d.vbR[i];
        int j = bR.x + q * n_enum;
        if (j >= ns) j -= ns;
        int2 dir[kOffBlock];
#pragma unroll
        for (int u = 0; u < kOffBlock; ++u) {
            if (u < n) dir[u] = D[j];
            j += n_enum;
            if (j >= ns) j -= ns;
        }
#pragma unroll
        for (int u = 0; u < kOffBlock; ++u) {
            if (u >= n) break;
            const int ox = (int)(((long long)bR.y * dir[u].x + (1ll << 45)) >> 46);
            const int oy = (int)(((long long)bR.y * dir[u].y + (1ll << 45)) >> 46);
            // |ox|, |oy| < P keeps every endpoint inside the field's border
            oq[(size_t)u * 32 * kS + k] = (int)((unsigned)oy << 16 | ((unsigned)ox & 0xffffu));
        }
    }
}

// TAM's work order of request d, by one CTA once its survivors are written:
// within each batch (with early termination; without it TAM scores every
// batch in one launch, so all K positions form one group), the survivor
// positions grouped by the band phase (y + P) % 8 of their cell (the order
// inside a group is immaterial: every position's scores are its own), then
// cut into chunks of at most tam_chunk positions of one phase, so that a TAM
// task uses one phase's endpoint offsets for all its survivors.  cells: shared
// memory for the K survivors' cells, read from global memory once.
__device__ __forceinline__ void tam_chunks_one(const ReqDesc &d, int2 *cells) {
    __shared__ int s_cnt[8], s_next[8];
    if (threadIdx.x == 0) d.chunk_cnt[0] = 0;
    int chunks = 0;   // so far (the first warp's)
    const int groups = d.early_stop ? d.n_batches : 1;
    for (int b = 0; b < groups; ++b) {
        const int lo = b * d.B, hi = d.early_stop ? min(d.K, lo + d.B) : d.K;
        if (threadIdx.x < 8) s_cnt[threadIdx.x] = 0;
        __syncthreads();
        for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const int2 c = d.hyps[d.survivors[i]];
            cells[i] = c;
            atomicAdd(&s_cnt[(c.y + d.P) & 7], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {   // lane p: phase p's positions, and its chunks after those of the phases before
            const int p = threadIdx.x, n = p < 8 ? s_cnt[p] : 0;
            const int parts = (n + d.tam_chunk - 1) / d.tam_chunk;   // of equal size, within one
            int run = n, nc = parts;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, run, o), c = __shfl_up_sync(0xffffffffu, nc, o);
                if (p >= o) {
                    run += a;
                    nc += c;
                }
            }
            const int total = __shfl_sync(0xffffffffu, nc, 7);
            run += lo - n;
            nc += chunks - parts;
            if (p < 8) s_next[p] = run;
            for (int c = 0; c < parts; ++c)
                d.tam_chunks[nc + c] = make_int4(p, run + n * c / parts, run + n * (c + 1) / parts, 0);
            chunks += total;
            if (d.early_stop) {
                if (p == 0) d.chunk_cnt[b + 1] = chunks;
            } else {
                for (int j = 1 + p; j <= d.n_batches; j += 32) d.chunk_cnt[j] = chunks;
            }
        }
        __syncthreads();
        for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const int2 c = cells[i];   // this thread's own
            const unsigned base = 8u * ((unsigned)((c.y + d.P) >> 3) * (unsigned)d.Wp + (unsigned)(c.x + d.P));
            d.surv_perm[atomicAdd(&s_next[(c.y + d.P) & 7], 1)] = make_int2(i, (int)base);
        }
        __syncthreads();
    }
}

}  // namespace relo
