// Traversability-constrained hypothesis sampling on the GPU (Algorithm 1,
// Sec. III-A, Remark 4).
//
// Algorithm 1 grows the tree one point at a time: every random point extends
// from its nearest node among all nodes so far.  Here a round's points go in
// sub-batches of kRrtSub, one launch (k_rrt_step) each.  Its first cluster of
// 8 CTAs resolves sub-batch s, a warp per point: the point's nearest tree node
// and the extension from it, then passes over the sub-batch's other points: a
// point whose nearest node is one accepted earlier in the sub-batch (strictly
// nearer than its tree node, so ties keep the lower index as in the serial
// search) is extended again from that one, and the passes repeat until no
// point's result changes.  Point k's result depends on points before k only, so
// the state the passes end in is unique: the serial algorithm's for the same
// random points and the same float32 arithmetic.  The points' results travel
// through distributed shared memory, every CTA holding the whole sub-batch.
// The other CTAs of the launch meanwhile search the tree for sub-batch s + 1 by
// brute force, each a slice of the nodes known before s; the nodes that s adds
// (at most kRrtSub) are searched by the launch of s + 1 itself.
//
// What bounds it: latency, a chain of a launch, a few dependent L2 reads and
// two or more passes of a cluster barrier per sub-batch (late in a run; while
// the tree is small the passes follow its growth): issue slots are 24% busy, the
// warps wait at barriers and for shared memory.  Taking the points one by
// one in a single warp, with three launches per sub-batch, took 72 us per
// sub-batch on the 1024 x 1024 office (161 ms per call).  Whole calls at rho =
// 0.6 m from six seeds, 464 to 2407 sub-batches: 34 to 219 ms then, 6.8 to 43.5
// now (74 to 91 and 14 to 18 us per sub-batch, more as the tree grows).
//
// A voxel of side rho is represented by its lowest-index node; a round's gain
// is the number of voxels it claimed, and sampling stops once a round gains at
// most eps_gain.  The node count lives on the device, so a round waits on the
// host once, for its gain.
//
// Per sample i of round r: p_rand from a counter-based hash (splitmix64 of
// seed ^ (r << 40 | i << 1 | k), k = 0, 1 for x, y), in [0, W res) x [0, H res);
// NearestNode by brute force (squared distance, ties to the lower index);
// AdaptiveExpandDist eta = eta_max when the clearance d at the nearest node is
// >= 2 r_robot, r_robot when d <= r_robot, linear between; ExtendPoint moves
// min(eta, |p_rand - p_nearest|) towards p_rand; the new point must lie in the
// map rectangle, and every point of the segment at spacing res / 2 (both ends
// included) must have clearance >= r_robot (clearance: a per-cell table in
// metres, 0 off the map).  Positions are float32 metres, and every operation
// is an explicitly rounded float32 one (no contraction), so a host program
// with the same steps gets the same tree.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/relo.h"
#include "relo_internal.h"

namespace relo {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRrtSub = 256;            // points per sub-batch: a warp of the resolving cluster each
constexpr int kCluster = 8;             // CTAs per cluster
constexpr int kStepThreads = 1024;
constexpr int kSlots = kRrtSub / 32;    // points of a sub-batch per lane of a warp that looks at all of them
constexpr int kNearTile = 1024;         // nodes staged in shared memory at a time
constexpr int kNearSubs = kStepThreads / (kRrtSub / 2);   // node subsets of a tile: a thread takes two points
constexpr int kMaxNear = 256;           // searching CTAs at most
static_assert(kCluster * kStepThreads / 32 == kRrtSub, "a warp per point");

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {   // Steele, Lea and Flood (2014)
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ float unit_draw(uint64_t seed, int round, int i, int k) {
    const uint64_t c = seed ^ (((uint64_t)round << 40) | ((uint64_t)i << 1) | (uint64_t)k);
    return (float)((double)(splitmix64(c) >> 11) * (1.0 / 9007199254740992.0));
}

struct RrtArgs {
    const float *clr;   // [H*W] clearance, metres
    int W, H;
    float res, rho, eta_max, r_robot;
    float Wm, Hm;       // map extent, metres: float(W) * res, float(H) * res
    uint64_t seed;
};

__device__ __forceinline__ float clearance_at(const RrtArgs &a, float x, float y) {
    const int cx = (int)floorf(__fdiv_rn(x, a.res)), cy = (int)floorf(__fdiv_rn(y, a.res));
    if (cx < 0 || cy < 0 || cx >= a.W || cy >= a.H) return 0.0f;
    return a.clr[(size_t)cy * a.W + cx];
}

__device__ __forceinline__ float dist2(float2 p, float rx, float ry) {
    const float ex = __fsub_rn(p.x, rx), ey = __fsub_rn(p.y, ry);
    return __fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey));
}

// ExtendPoint from node pn (clearance dn) towards (rx, ry), by the whole warp
// (all lanes pass the same arguments; each checks every 32nd segment point).
// *out receives the new point and *c_out the clearance there; returns whether
// the extension is accepted.
__device__ __forceinline__ int warp_extend(const RrtArgs &a, float2 pn, float dn, float rx, float ry, float2 *out,
                                           float *c_out) {
    const int lane = threadIdx.x & 31;
    float eta;
    if (dn >= 2.0f * a.r_robot) eta = a.eta_max;
    else if (dn <= a.r_robot) eta = a.r_robot;
    else eta = __fadd_rn(a.r_robot, __fdiv_rn(__fmul_rn(__fsub_rn(a.eta_max, a.r_robot), __fsub_rn(dn, a.r_robot)),
                                              a.r_robot));
    const float vx = __fsub_rn(rx, pn.x), vy = __fsub_rn(ry, pn.y);
    const float L = __fsqrt_rn(__fadd_rn(__fmul_rn(vx, vx), __fmul_rn(vy, vy)));
    *out = pn;
    *c_out = dn;
    if (!(L > 0.0f)) return 0;
    const float step = fminf(eta, L);
    const float nx = __fadd_rn(pn.x, __fmul_rn(__fdiv_rn(vx, L), step));
    const float ny = __fadd_rn(pn.y, __fmul_rn(__fdiv_rn(vy, L), step));
    *out = make_float2(nx, ny);
    *c_out = 0.0f;
    if (!(nx >= 0.0f && ny >= 0.0f && nx < a.Wm && ny < a.Hm)) return 0;
    const int nseg = (int)ceilf(__fdiv_rn(step, 0.5f * a.res));
    const float sx = __fsub_rn(nx, pn.x), sy = __fsub_rn(ny, pn.y);
    int good = 1;
    for (int t = lane; t <= nseg; t += 32) {
        const float f = nseg ? __fdiv_rn((float)t, (float)nseg) : 0.0f;
        if (clearance_at(a, __fadd_rn(pn.x, __fmul_rn(sx, f)), __fadd_rn(pn.y, __fmul_rn(sy, f))) < a.r_robot)
            good = 0;
    }
    *c_out = clearance_at(a, nx, ny);
    return __all_sync(kFull, good);
}

__device__ __forceinline__ int voxel_of(float2 p, float rho, int vw) {
    return (int)floorf(__fdiv_rn(p.y, rho)) * vw + (int)floorf(__fdiv_rn(p.x, rho));
}

// Running state on the device: tree[s & 3] is the node count before sub-batch s, gain[r & 1] the voxels claimed in
// round r.
struct RrtState {
    int tree[4];
    int gain[2];
    int count;   // representatives written
};

// A sub-batch: its points i0 .. i0 + n - 1 of its round.
struct RrtBatch {
    int i0, n, round;
};

// The nearest of the first n nodes to each point of batch b, slice by slice: CTA c of nc scans nodes [c per, (c + 1)
// per), staged through shared memory; a thread takes two points and one subset of each tile, in groups of four nodes
// whose smallest distance is kept with the group (ascending, so the first smallest wins); its node is found again at
// the end.  part[c][k] receives point k's (squared distance, index), (+inf, INT_MAX) for an empty slice.
__device__ void near_slice(const RrtArgs &a, const float2 *__restrict__ nodes, int n, const RrtBatch &b, int c, int nc,
                           int2 *__restrict__ part) {
    __shared__ __align__(16) float2 tile[kNearTile];
    __shared__ int2 s_best[kNearSubs][kRrtSub];
    constexpr int kPairs = kRrtSub / 2, kSub = kNearTile / kNearSubs;
    const int pair = threadIdx.x % kPairs, sub = threadIdx.x / kPairs;
    const int per = (n + nc - 1) / nc;
    const int lo = min(n, c * per), hi = min(n, lo + per);
    float rx[2], ry[2], best[2] = {INFINITY, INFINITY};
    int group[2] = {-1, -1};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int k = pair + u * kPairs;
        rx[u] = __fmul_rn(unit_draw(a.seed, b.round, b.i0 + k, 0), a.Wm);
        ry[u] = __fmul_rn(unit_draw(a.seed, b.round, b.i0 + k, 1), a.Hm);
    }
    for (int t0 = lo; t0 < hi; t0 += kNearTile) {
        __syncthreads();
        // past the slice: so far away that the squared distance is +inf, which is never smaller
        tile[threadIdx.x] = t0 + (int)threadIdx.x < hi ? nodes[t0 + threadIdx.x] : make_float2(1e30f, 1e30f);
        __syncthreads();
        const int end = min(kSub, hi - t0 - sub * kSub);
        for (int i = 0; i < end; i += 4) {
            const float4 p = *reinterpret_cast<const float4 *>(&tile[sub * kSub + i]);
            const float4 q = *reinterpret_cast<const float4 *>(&tile[sub * kSub + i + 2]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float m = fminf(fminf(dist2(make_float2(p.x, p.y), rx[u], ry[u]),
                                            dist2(make_float2(p.z, p.w), rx[u], ry[u])),
                                      fminf(dist2(make_float2(q.x, q.y), rx[u], ry[u]),
                                            dist2(make_float2(q.z, q.w), rx[u], ry[u])));
                if (m < best[u]) {
                    best[u] = m;
                    group[u] = t0 + sub * kSub + i;
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        int id = 0x7fffffff;
        if (group[u] >= 0)
            for (int i = 3; i >= 0; --i)
                if (group[u] + i < hi && dist2(nodes[group[u] + i], rx[u], ry[u]) == best[u]) id = group[u] + i;
        s_best[sub][pair + u * kPairs] = make_int2(__float_as_int(best[u]), id);
    }
    __syncthreads();
    if (threadIdx.x < kRrtSub) {
        int2 v = s_best[0][threadIdx.x];
        for (int j = 1; j < kNearSubs; ++j) {
            const int2 w = s_best[j][threadIdx.x];
            const float dv = __int_as_float(v.x), dw = __int_as_float(w.x);
            if (dw < dv || (dw == dv && w.y < v.y)) v = w;
        }
        part[(size_t)c * kRrtSub + threadIdx.x] = v;
    }
}

// A point's result as the passes exchange it.
struct __align__(16) RrtPoint {
    float x, y, c;   // the extension's end and the clearance there
    int ok;          // accepted
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The shared-memory address of p in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {
    uint32_t out;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}

// Sub-batch cur (step s), and the nearest-node search of the next one.  part_in: the slices' nearest nodes of cur among
// the tree before step s - 1 (written by the previous launch); part_out: those of next among the tree before step s.
// cur.n == 0: the search alone (the first launch).
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kStepThreads, 1)
    k_rrt_step(RrtArgs a, float2 *nodes, float *nclr, const int2 *__restrict__ part_in, int2 *part_out, int step,
               RrtBatch cur, RrtBatch next, RrtState *st, int node_cap, int vw, int *voxel) {
    const int nc = (int)gridDim.x - kCluster;   // searching CTAs
    const int n0 = st->tree[step & 3];          // nodes before this sub-batch
    if ((int)blockIdx.x >= kCluster) {
        near_slice(a, nodes, n0, next, (int)blockIdx.x - kCluster, nc, part_out);
        return;
    }
    if (cur.n == 0) return;   // the whole cluster
    __shared__ RrtPoint table[2][kRrtSub];
    __shared__ int changed[2];
    const int lane = threadIdx.x & 31, k = (int)blockIdx.x * (kStepThreads / 32) + (int)(threadIdx.x >> 5);
    const int base = st->tree[(step + 3) & 3];   // nodes the slices were searched among
    if (threadIdx.x < 2) changed[threadIdx.x] = -1;
    if (blockIdx.x == 0 && threadIdx.x == 0 && cur.i0 == 0) st->gain[(cur.round + 1) & 1] = 0;   // the next round's
    const bool live = k < cur.n;
    float rx = 0.0f, ry = 0.0f, best2 = INFINITY;
    RrtPoint tree = {0.0f, 0.0f, 0.0f, 0};   // the extension from the nearest tree node
    if (live) {
        rx = __fmul_rn(unit_draw(a.seed, cur.round, cur.i0 + k, 0), a.Wm);
        ry = __fmul_rn(unit_draw(a.seed, cur.round, cur.i0 + k, 1), a.Hm);
        int best = 0x7fffffff;
        auto take = [&](float d2, int id) {
            if (d2 < best2 || (d2 == best2 && id < best)) {
                best2 = d2;
                best = id;
            }
        };
        for (int b = lane; b < nc; b += 32) {
            const int2 v = part_in[(size_t)b * kRrtSub + k];
            take(__int_as_float(v.x), v.y);
        }
        for (int i = base + lane; i < n0; i += 32) take(dist2(nodes[i], rx, ry), i);   // the previous sub-batch's nodes
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {   // the warp's smallest (d2, index); every lane ends with it
            const float od = __shfl_xor_sync(kFull, best2, o);
            const int oj = __shfl_xor_sync(kFull, best, o);
            take(od, oj);
        }
        float2 nw;
        float cw;
        tree.ok = warp_extend(a, nodes[best], nclr[best], rx, ry, &nw, &cw);
        tree.x = nw.x;
        tree.y = nw.y;
        tree.c = cw;
    }
    RrtPoint mine = tree;
    auto publish = [&](int buf) {   // to every CTA of the cluster, one per lane
        if (lane < kCluster)
            asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr(&table[buf][k], lane)),
                         "r"(__float_as_int(mine.x)), "r"(__float_as_int(mine.y)), "r"(__float_as_int(mine.c)),
                         "r"(mine.ok)
                         : "memory");
    };
    cluster_sync();   // every CTA has started (its shared memory may be written) and has set its flags
    publish(0);
    cluster_sync();
    // Pass p reads table[p & 1] and writes table[(p + 1) & 1]; a warp whose result changes says so in changed[p & 1].
    // A CTA can be at most one barrier ahead of another, so neither is overwritten while it is read.  Each pass
    // settles at least one more point, so there are at most cur.n + 1.
    int parent = -1, p = 0;   // -1: the tree node; else the point of the sub-batch it was extended from
    float2 ppos = make_float2(0.0f, 0.0f);
    for (;; ++p) {
        const RrtPoint *now = table[p & 1];
        if (live) {
            float bd = INFINITY;
            int bj = 0x7fffffff;
#pragma unroll
            for (int s = 0; s < kSlots; ++s) {
                const int j = lane + 32 * s;
                if (j < k) {
                    const RrtPoint q = now[j];
                    const float d2 = dist2(make_float2(q.x, q.y), rx, ry);
                    if (q.ok && d2 < bd) {
                        bd = d2;
                        bj = j;
                    }
                }
            }
            // squared distances are >= +0 (or +inf), so their bit patterns order like the values
            const unsigned mn = __reduce_min_sync(kFull, __float_as_uint(bd));
            const RrtPoint was = mine;
            if (__uint_as_float(mn) < best2) {   // a point accepted earlier in this sub-batch is nearer
                const int jj = (int)__reduce_min_sync(kFull, __float_as_uint(bd) == mn ? (unsigned)bj : 0xffffffffu);
                const RrtPoint q = now[jj];
                // the same parent at the same place (its clearance is that place's) gives the same extension
                if (jj != parent || q.x != ppos.x || q.y != ppos.y) {
                    parent = jj;
                    ppos = make_float2(q.x, q.y);
                    float2 nw;
                    float cw;
                    mine.ok = warp_extend(a, ppos, q.c, rx, ry, &nw, &cw);
                    mine.x = nw.x;
                    mine.y = nw.y;
                    mine.c = cw;
                }
            } else {
                parent = -1;
                mine = tree;
            }
            const bool differs = mine.ok != was.ok || mine.x != was.x || mine.y != was.y;
            if (differs && lane < kCluster)
                asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(cluster_addr(&changed[p & 1], lane)), "r"(p)
                             : "memory");
        }
        publish((p + 1) & 1);
        cluster_sync();
        if (*(volatile int *)&changed[p & 1] != p || p > kRrtSub) break;   // the same in every CTA
    }
    // Accepted points in sample order are nodes n0, n0 + 1, ... (at most node_cap in all); each claims its voxel, and
    // the first claim of a voxel counts towards the round's gain.
    const RrtPoint *fin = table[(p + 1) & 1];
    int rank = 0, total = 0;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
        const unsigned bal = __ballot_sync(kFull, fin[lane + 32 * s].ok != 0);
        total += __popc(bal);
        if (32 * s + 32 <= k) rank += __popc(bal);
        else if (32 * s <= k) rank += __popc(bal & ((1u << (k & 31)) - 1u));
    }
    if (lane == 0 && mine.ok && rank < node_cap - n0) {
        const float2 at = make_float2(mine.x, mine.y);
        nodes[n0 + rank] = at;
        nclr[n0 + rank] = mine.c;
        if (atomicMin(voxel + voxel_of(at, a.rho, vw), n0 + rank) == 0x7fffffff) atomicAdd(&st->gain[cur.round & 1], 1);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->tree[(step + 1) & 3] = min(n0 + total, max(n0, node_cap));
}

// The first node: p0, its clearance and its voxel; one node, no gain.
__global__ void k_rrt_init(RrtArgs a, float2 p0, float2 *nodes, float *nclr, int vw, int *voxel, RrtState *st) {
    if (threadIdx.x != 0) return;
    nodes[0] = p0;
    nclr[0] = clearance_at(a, p0.x, p0.y);
    voxel[voxel_of(p0, a.rho, vw)] = 0;
    for (int i = 0; i < 4; ++i) st->tree[i] = 1;
    st->gain[0] = st->gain[1] = 0;
}

// One CTA: the voxel representatives among nodes [0, n), those that hold their voxel, in order to dst[0 ..), at most
// cap of them; *count receives the number written.
__global__ void __launch_bounds__(1024) k_rrt_compact(const float2 *__restrict__ src, const int *__restrict__ voxel,
                                                      float rho, int vw, int n, float2 *__restrict__ dst, int cap,
                                                      int *count) {
    __shared__ int warp_cnt[32];
    __shared__ int s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        const float2 at = i < n ? src[i] : make_float2(0.0f, 0.0f);
        const bool take = i < n && voxel[voxel_of(at, rho, vw)] == i;
        const unsigned bal = __ballot_sync(kFull, take);
        if (lane == 0) warp_cnt[warp] = __popc(bal);
        __syncthreads();
        if (warp == 0) {
            const int v = lane < nwarps ? warp_cnt[lane] : 0;
            int incl = v;
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            warp_cnt[lane] = incl - v;
        }
        __syncthreads();
        if (take) {
            const int pos = s_base + warp_cnt[warp] + __popc(bal & ((1u << lane) - 1u));
            if (pos < cap) dst[pos] = at;
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) s_base += warp_cnt[warp] + __popc(bal);
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = min(cap, s_base);
}

__global__ void k_fill_int(int *p, size_t n, int v) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = v;
}

}  // namespace

int rrt_sample_dev(const float *clr, int W, int H, double res, double p0x, double p0y, double rho, double eta_max,
                   double r_robot, int eps_gain, uint64_t seed, int max_rounds, int node_cap, float *xy_out, int cap,
                   int *n_out, int *rounds_out, int *nodes_out, cudaStream_t s, const char **err) {
    const double Wm = W * res, Hm = H * res;
    if (!(p0x >= 0 && p0y >= 0 && p0x < Wm && p0y < Hm)) {
        *err = "the start point lies off the map";
        return RELO_E_INVALID_ARG;
    }
    const long long n_s_ll = (long long)ceil((double)W * H * res * res / (rho * rho));
    if (n_s_ll < 1 || n_s_ll > (1ll << 26)) {
        *err = "rho gives too many samples per round";
        return RELO_E_INVALID_ARG;
    }
    const int n_s = (int)n_s_ll;
    const int vw = (int)ceil(Wm / rho) + 1, vh = (int)ceil(Hm / rho) + 1;
    const size_t n_vox = (size_t)vw * vh;
    float2 *nodes = nullptr;
    float *nclr = nullptr;
    int2 *part = nullptr;
    int *voxel = nullptr;
    RrtState *st = nullptr;
    cudaError_t e = cudaSuccess;
    // one CTA per SM in clusters of 8: as many as are resident at once, the first resolving, the others searching
    int clusters = 0;
    {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kCluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(kCluster);
        cfg.blockDim = dim3(kStepThreads);
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&clusters, k_rrt_step, &cfg);
        clusters = std::max(2, std::min(clusters, kMaxNear / kCluster + 1));
    }
    const int near = (clusters - 1) * kCluster;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes ? bytes : 1);
    };
    alloc((void **)&nodes, sizeof(float2) * (size_t)node_cap);
    alloc((void **)&nclr, sizeof(float) * (size_t)node_cap);
    alloc((void **)&part, sizeof(int2) * 2 * (size_t)near * kRrtSub);
    alloc((void **)&voxel, sizeof(int) * n_vox);
    alloc((void **)&st, sizeof(RrtState));
    int rc = RELO_OK, n = 1, rounds = 0;
    if (e == cudaSuccess) {
        const float fres = (float)res;
        RrtArgs a{clr, W, H, fres, (float)rho, (float)eta_max, (float)r_robot, (float)W * fres, (float)H * fres, seed};
        k_fill_int<<<256, 256, 0, s>>>(voxel, n_vox, 0x7fffffff);
        k_rrt_init<<<1, 32, 0, s>>>(a, make_float2((float)p0x, (float)p0y), nodes, nclr, vw, voxel, st);
        int step = 0;
        auto batch = [&](int i0, int round) {   // the sub-batch from i0, or the next round's first
            if (i0 >= n_s) return RrtBatch{0, std::min(kRrtSub, n_s), round + 1};
            return RrtBatch{i0, std::min(kRrtSub, n_s - i0), round};
        };
        auto launch = [&](RrtBatch cur, RrtBatch next) {   // searches into the half of part that the next launch reads
            const size_t half = (size_t)near * kRrtSub;
            k_rrt_step<<<clusters * kCluster, kStepThreads, 0, s>>>(a, nodes, nclr, part + (step & 1) * half,
                                                                    part + ((step + 1) & 1) * half, step, cur, next, st,
                                                                    node_cap, vw, voxel);
        };
        step = 3;   // the search for sub-batch 0 alone (every count is 1 so far)
        launch(RrtBatch{0, 0, 0}, batch(0, 0));
        step = 0;
        while ((e = cudaGetLastError()) == cudaSuccess) {
            for (int i0 = 0; i0 < n_s; i0 += kRrtSub, ++step) launch(batch(i0, rounds), batch(i0 + kRrtSub, rounds));
            RrtState host;
            e = cudaMemcpyAsync(&host, st, sizeof host, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) break;
            n = host.tree[step & 3];
            const int gain = host.gain[rounds & 1];
            ++rounds;
            if (gain <= eps_gain || rounds >= max_rounds || n >= node_cap) break;
        }
        // the voxel representatives in order of node index
        if (e == cudaSuccess) {
            k_rrt_compact<<<1, 1024, 0, s>>>(nodes, voxel, a.rho, vw, n, reinterpret_cast<float2 *>(xy_out), cap,
                                             &st->count);
            int reps = 0;
            e = cudaMemcpyAsync(&reps, &st->count, sizeof(int), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            *n_out = reps;
            *rounds_out = rounds;
            *nodes_out = n;
        }
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        *err = cudaGetErrorString(e);
        rc = RELO_E_CUDA;
    }
    cudaFree(nodes);
    cudaFree(nclr);
    cudaFree(part);
    cudaFree(voxel);
    cudaFree(st);
    return rc;
}

namespace {

// The grid the clearance EDT runs on: the map with a ring of one cell around
// it, every cell occupied (100) that the RRT may not stand on (occupied,
// v >= 65, or unknown, v < 0) and every ring cell occupied (the outside of
// the map is blocked); traversable cells 0.
__global__ void k_rrt_blocked(const int8_t *__restrict__ grid, int W, int H, int8_t *__restrict__ out) {
    const int pw = W + 2, ph = H + 2;
    const long long n = (long long)pw * ph;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(i / pw) - 1, x = (int)(i % pw) - 1;
        bool blocked = true;
        if (x >= 0 && y >= 0 && x < W && y < H) {
            const int v = grid[(size_t)y * W + x];
            blocked = v < 0 || v >= 65;
        }
        out[i] = blocked ? (int8_t)100 : (int8_t)0;
    }
}

// MinDistToObstacle as a per-cell table (Sec. III-A item 3): res times the
// distance from the cell centre to the nearest blocked cell centre, from the
// exact squared EDT of the ringed grid (never -1: the ring is blocked); the
// square root and the product in FP64, rounded once to float32.
__global__ void k_rrt_clearance(const int32_t *__restrict__ d2p, int W, int H, double res, float *__restrict__ clr) {
    const long long n = (long long)W * H;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(i / W), x = (int)(i % W);
        const int32_t v = d2p[(size_t)(y + 1) * (W + 2) + (x + 1)];
        clr[i] = (float)(res * sqrt((double)v));
    }
}

}  // namespace

cudaError_t launch_rrt_blocked(const int8_t *grid, int W, int H, int8_t *out, cudaStream_t s) {
    k_rrt_blocked<<<1024, 256, 0, s>>>(grid, W, H, out);
    return cudaGetLastError();
}

cudaError_t launch_rrt_clearance(const int32_t *d2p, int W, int H, double res, float *clr, cudaStream_t s) {
    k_rrt_clearance<<<1024, 256, 0, s>>>(d2p, W, H, res, clr);
    return cudaGetLastError();
}

}  // namespace relo
