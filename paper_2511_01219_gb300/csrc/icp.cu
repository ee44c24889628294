// ICP refinement of the local top-k poses and their re-evaluation (the last
// step of the framework overview, Sec. III: the local top-k poses are aligned
// to the whole map and scored again; Remark 2 names the refinement operator).
//
// k_icp: one cluster of CTAs per local top-k pose.  The pose starts at its hypothesis
// cell centre and orientation theta_m.  Beam i is the sensor-frame point
// (z_i, a_i), z_i = R_i res / 2^16 (its Q16 range) and a_i = 2 pi b_i / N_s (its
// panoramic grid angle); its sensor-frame point s_i = (z_i cos a_i, z_i sin
// a_i) is computed once per request (icp_points.cuh).  An iteration maps every valid beam to its world
// point w = p + R(theta) s (each product and sum rounded on its own, as the
// oracle does; its cell is floor(w * (1 / res))), pairs it with the centre of
// the nearest occupied cell to the cell it
// falls in (the radius is the exact EDT value there; ties go to the smaller
// dy, then the smaller dx; pairs farther than the TAM clamp C = (d_max /
// res)^2 are dropped), and applies the rigid motion that minimises the
// squared pair distances: with the centroids mw, mc and the centred cross and
// dot sums, phi = atan2(cross, dot) (whose cosine and sine are the two sums over
// their length) and t = mc - R(phi) mw.  It stops after
// icp_iters iterations, when fewer than 2 pairs remain, or when the motion is
// below 1e-9 rad and 1e-9 m.  All pose arithmetic is FP64.
//
// What bounds it is the chain of dependent steps, FP64 at two lanes per clock
// and SM and barriers (20 poses over 160 CTAs: issue slots 4% and FP64 pipes 16%
// busy), so a pose is spread over as many SMs as there are to spare:
// the CTAs of a cluster share its beams, their sums meet in the first CTA's
// shared memory, one warp there solves for the motion and writes the pose to
// all.  With one CTA per pose whose every thread solved the motion and made its
// own beams' points, 20 poses of 1027 beams took 420 us for 10 iterations; this
// takes 130 (with the angle evaluated in every iteration 172).
//
// The refined pose is then scored like TAM: each beam ends in the cell of its
// world point, takes min(d2, C) (C off the map), and the k-th smallest
// value, the likelihood table and the epilogue of Eq. 23-31 (or the metric
// fine_metric selects) give the score, in the FP32 arithmetic of k_tam with
// sums in FP64, by one warp.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "chain.cuh"
#include "relo_internal.h"

namespace relo {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kIcpThreads = 128;
constexpr int kIcpWarps = kIcpThreads / 32;
constexpr int kIcpCluster = 8;   // CTAs per pose at most

// The nearest occupied cell to cell (x, y) when its squared distance is at
// most cap (<= C): the cells at exactly the EDT distance, by increasing dy,
// then dx, from the map's table of the offsets at each squared distance, eight
// at a time (most distances have no more; one by one, every candidate waited
// for two loads).
__device__ bool nearest_occupied(const ReqDesc &d, const int32_t *sq_off, const short2 *sq_rep, int x, int y, int cap,
                                 int &ox, int &oy) {
    if (x < 0 || y < 0 || x >= d.W || y >= d.H) return false;
    const int d2 = d.d2map[(size_t)y * d.W + x];
    if (d2 < 0 || d2 > cap) return false;
    if (d2 == 0) {
        ox = x;
        oy = y;
        return true;
    }
    const int e1 = sq_off[d2 + 1];
    for (int e = sq_off[d2]; e < e1; e += 8) {
        short2 o[8];
        int8_t v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = e + i < e1 ? sq_rep[e + i] : make_short2(0, 0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int cx = x + o[i].y, cy = y + o[i].x;
            const bool in = e + i < e1 && cx >= 0 && cy >= 0 && cx < d.W && cy < d.H;
            v[i] = in ? __ldg(d.grid + (size_t)cy * d.W + cx) : (int8_t)0;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (v[i] >= 65) {
                ox = x + o[i].y;
                oy = y + o[i].x;
                return true;
            }
    }
    return false;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Sums of 4 values over the warp with 6 additions instead of 20: each exchange halves the values a lane carries.  The
// lane ends with the total of value sum_index(lane).
__device__ __forceinline__ double warp_sums4(double (&v)[4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 2, o = 16; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < n; ++j) {
            const double send = up ? v[j] : v[j + n], keep = up ? v[j + n] : v[j];
            v[j] = keep + __shfl_xor_sync(kFull, send, o);
        }
    }
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], o);
    return v[0];
}
__device__ __forceinline__ int sum_index(int lane) { return (lane >> 4 & 1) * 2 + (lane >> 3 & 1); }

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {   // p in CTA `rank` of the cluster
    uint32_t out;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}
__device__ __forceinline__ void cluster_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, int v) {
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// world point and cell of a sensor-frame point at pose (x, y) with ct, st = cos, sin of theta
__device__ __forceinline__ void world_point(double x, double y, double ct, double st, double sx, double sy,
                                            double inv_res, double &wx, double &wy, int &cx, int &cy) {
    wx = __dadd_rn(x, __dsub_rn(__dmul_rn(ct, sx), __dmul_rn(st, sy)));
    wy = __dadd_rn(y, __dadd_rn(__dmul_rn(st, sx), __dmul_rn(ct, sy)));
    cx = __double2int_rd(__dmul_rn(wx, inv_res));
    cy = __double2int_rd(__dmul_rn(wy, inv_res));
}

__device__ __forceinline__ int clamped_d2(const ReqDesc &d, int x, int y) {
    if (x < 0 || y < 0 || x >= d.W || y >= d.H) return d.C;
    const int v = d.d2map[(size_t)y * d.W + x];
    return (v < 0 || v > d.C) ? d.C : v;
}

// The pose: position, cos and sin of theta.  The rotation applied so far is carried as its cosine and sine (c, s),
// renormalised after every step, and theta is read off it once at the end: an FP64 atan2, sine and cosine in every
// iteration were half of the iteration's time.
struct IcpPose {
    double x, y, ct, st, c, s;
    int stop;
};

// (c, s) scaled to unit length (its length is 1 within rounding: one Newton step of the reciprocal square root)
__device__ __forceinline__ void unit_rotation(double &c, double &s) {
    const double r = 1.5 - 0.5 * (c * c + s * s);
    c *= r;
    s *= r;
}

constexpr int kIcpTableBytes = 28 * 1024;   // the pairing table is staged up to this size (C = 1600: 26 KB)

// dynamic shared memory: [per] the CTA's sensor-frame points, then in the first CTA [max_beams] the clamped d2 of the
// refined endpoints, then with staged the map's pairing table; per: beams per CTA of the cluster for the longest scan
__global__ void __launch_bounds__(kIcpThreads) k_icp(const ReqDesc *__restrict__ reqs, int batch_lo, int batch_hi,
                                                     int per, int max_beams, bool staged) {
    extern __shared__ __align__(16) unsigned char icp_smem[];
    __shared__ double part[kIcpCluster * kIcpWarps][4];   // the first CTA's: every warp's sums
    __shared__ int parti[kIcpCluster * kIcpWarps][4];
    __shared__ IcpPose pose;
    double2 *pts = reinterpret_cast<double2 *>(icp_smem);
    int *qv = reinterpret_cast<int *>(icp_smem + sizeof(double2) * (size_t)per);
    chain_wait();
    chain_go();
    uint32_t cs, cr;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cs));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(cr));
    const ReqDesc &d = reqs[blockIdx.y];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the conditions below are the same in every CTA of the cluster
    const int slot = (int)(blockIdx.x / cs);
    if (slot >= (batch_hi - batch_lo) * d.L) return;
    const int b = batch_lo + slot / d.L;
    if (b >= d.n_batches) return;
    const int s = d.local[(size_t)b * d.L + slot % d.L];
    const int N = d.scan->n_valid;
    if (s < 0 || N <= 0) return;
    const int i0 = (int)cr * per, n = max(0, min(N - i0, per));   // this CTA's beams
    const double2 *src = reinterpret_cast<const double2 *>(d.icp_pts) + i0;
    for (int i = tid; i < n; i += kIcpThreads) pts[i] = src[i];
    // the pairing table next to the beams: two of the four loads that a pairing waits for in turn
    const int32_t *sq_off = d.sq_off;
    const short2 *sq_rep = d.sq_rep;
    if (staged) {   // 16 bytes at a time: the tables end in padding
        const int reps = __ldg(sq_off + d.C + 1), o4 = (d.C + 2 + 3) / 4, r4 = (reps + 3) / 4;
        int4 *off = reinterpret_cast<int4 *>(qv + ((max_beams + 3) & ~3)), *rep = off + o4;
#pragma unroll 4
        for (int i = tid; i < o4; i += kIcpThreads) off[i] = __ldg(reinterpret_cast<const int4 *>(sq_off) + i);
#pragma unroll 4
        for (int i = tid; i < r4; i += kIcpThreads) rep[i] = __ldg(reinterpret_cast<const int4 *>(sq_rep) + i);
        sq_off = reinterpret_cast<const int32_t *>(off);
        sq_rep = reinterpret_cast<const short2 *>(rep);
    }
    const double res = d.resd, inv_res = 1.0 / res, half = 0.5 * res;
    auto tell = [&](const IcpPose &p) {   // by warp 0 of the first CTA: the pose to every CTA, one per lane
        if (lane < (int)cs) {
            const uint32_t a = cluster_addr(&pose, lane);
            cluster_store(a, p.x);
            cluster_store(a + 8, p.y);
            cluster_store(a + 16, p.ct);
            cluster_store(a + 24, p.st);
            cluster_store(a + 32, p.c);
            cluster_store(a + 40, p.s);
            cluster_store(a + 48, p.stop);
        }
    };
    const double th0 = __ddiv_rn(__dmul_rn((double)d.best_m[s], 2.0 * M_PI), (double)d.ns);
    cluster_sync();   // every CTA has started: its shared memory may be written
    if (cr == 0 && warp == 0) {
        const int2 hc = d.hyps[d.survivors[s]];
        IcpPose p;
        p.x = __dmul_rn((double)hc.x + 0.5, res);
        p.y = __dmul_rn((double)hc.y + 0.5, res);
        p.ct = cos(th0);
        p.st = sin(th0);
        p.c = 1.0;
        p.s = 0.0;
        p.stop = d.icp_iters <= 0;
        tell(p);
    }
    cluster_sync();
    for (int it = 1; !pose.stop; ++it) {
        const IcpPose p = pose;
        double v[4] = {0, 0, 0, 0};   // sums of w, of w.c and of w x c
        int np = 0, sox = 0, soy = 0;   // pairs and sums of their cells, exact
        for (int i = tid; i < n; i += kIcpThreads) {
            double wx, wy;
            int ex, ey, ox, oy;
            world_point(p.x, p.y, p.ct, p.st, pts[i].x, pts[i].y, inv_res, wx, wy, ex, ey);
            if (!nearest_occupied(d, sq_off, sq_rep, ex, ey, d.C, ox, oy)) continue;
            const double cx = fma((double)ox, res, half), cy = fma((double)oy, res, half);
            ++np;
            sox += ox;
            soy += oy;
            v[0] += wx;
            v[1] += wy;
            v[2] = fma(wx, cx, fma(wy, cy, v[2]));
            v[3] = fma(wx, cy, fma(-wy, cx, v[3]));
        }
        __syncwarp();
        const double w = warp_sums4(v);
        const int k0 = cr * kIcpWarps + warp;
        np = __reduce_add_sync(kFull, np);
        sox = __reduce_add_sync(kFull, sox);
        soy = __reduce_add_sync(kFull, soy);
        if ((lane & 7) == 0) cluster_store(cluster_addr(&part[k0][sum_index(lane)], 0), w);
        if (lane < 3) cluster_store(cluster_addr(&parti[k0][lane], 0), lane == 0 ? np : lane == 1 ? sox : soy);
        cluster_sync();   // the sums have arrived, and every thread has read the pose
        if (cr == 0 && warp == 0) {
            const int parts = (int)cs * kIcpWarps;
            double t = 0.0;
            for (int k = lane >> 2; k < parts; k += 8) t += part[k][lane & 3];
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) t += __shfl_xor_sync(kFull, t, o);
            const double swx = __shfl_sync(kFull, t, 0), swy = __shfl_sync(kFull, t, 1), sdot = __shfl_sync(kFull, t, 2),
                         scr = __shfl_sync(kFull, t, 3);
            const int pairs = __reduce_add_sync(kFull, lane < parts ? parti[lane][0] : 0);
            const int nox = __reduce_add_sync(kFull, lane < parts ? parti[lane][1] : 0);
            const int noy = __reduce_add_sync(kFull, lane < parts ? parti[lane][2] : 0);
            const double np = (double)pairs;
            IcpPose q = p;
            if (np < 2.0) {
                q.stop = 1;
            } else {
                // the four means by four lanes, so one division's latency; then the cross sum (even lanes) and the
                // dot sum (odd lanes)
                const int which = lane & 3;
                const double mean = (which == 0 ? swx : which == 1 ? swy : which == 2 ? ((double)nox + 0.5 * np) * res
                                                                                     : ((double)noy + 0.5 * np) * res) / np;
                const double mwx = __shfl_sync(kFull, mean, 0), mwy = __shfl_sync(kFull, mean, 1);
                const double mcx = __shfl_sync(kFull, mean, 2), mcy = __shfl_sync(kFull, mean, 3);
                const bool odd = lane & 1;
                const double a1 = odd ? mcx : mcy, a2 = odd ? mcy : mcx;
                const double cd = (odd ? sdot : scr) - np * (odd ? mwx * a1 + mwy * a2 : mwx * a1 - mwy * a2);
                const double cross = __shfl_sync(kFull, cd, 0), dot = __shfl_sync(kFull, cd, 1);
                // the motion's rotation: cos and sin of atan2(cross, dot) (the identity for two zero sums)
                const double len2 = cross * cross + dot * dot, inv = len2 > 0.0 ? rsqrt(len2) : 0.0;
                double cf = len2 > 0.0 ? dot * inv : 1.0, sf = cross * inv;
                unit_rotation(cf, sf);
                q.ct = p.ct * cf - p.st * sf;
                q.st = p.st * cf + p.ct * sf;
                unit_rotation(q.ct, q.st);
                q.c = p.c * cf - p.s * sf;
                q.s = p.s * cf + p.c * sf;
                unit_rotation(q.c, q.s);
                const double tx = __dsub_rn(mcx, __dsub_rn(__dmul_rn(cf, mwx), __dmul_rn(sf, mwy)));
                const double ty = __dsub_rn(mcy, __dadd_rn(__dmul_rn(sf, mwx), __dmul_rn(cf, mwy)));
                q.x = __dadd_rn(__dsub_rn(__dmul_rn(cf, p.x), __dmul_rn(sf, p.y)), tx);
                q.y = __dadd_rn(__dadd_rn(__dmul_rn(sf, p.x), __dmul_rn(cf, p.y)), ty);
                const double moved = fabs(q.x - p.x) + fabs(q.y - p.y);
                q.stop = (fabs(sf) < 1e-9 && cf > 0.0 && moved < 1e-9) || it >= d.icp_iters;
            }
            tell(q);
        }
        cluster_sync();
    }
    // the refined pose scored again: the clamped d2 of every endpoint to the first CTA
    const IcpPose p = pose;
    for (int i = tid; i < n; i += kIcpThreads) {
        double wx, wy;
        int ex, ey;
        world_point(p.x, p.y, p.ct, p.st, pts[i].x, pts[i].y, inv_res, wx, wy, ex, ey);
        cluster_store(cluster_addr(&qv[i0 + i], 0), clamped_d2(d, ex, ey));
    }
    cluster_sync();
    if (cr != 0 || warp != 0) return;
    int sumb = 0;
    for (int i = lane; i < N; i += 32) sumb += qv[i];
    sumb = __reduce_add_sync(kFull, sumb);
    const int C = d.C;
    const int k = d.fine < kFineBaseline ? d.scan->k_ret : N;
    auto count_le = [&](int x) {
        int c = 0;
        for (int i = lane; i < N; i += 32) c += qv[i] <= x ? 1 : 0;
        return __reduce_add_sync(kFull, c);
    };
    int bk = C, cle = N;
    if (k < N) {   // the smallest b with #{q <= b} >= k, by bisection over [0, C]
        int lo = 0, hi = C, c_hi = N;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const int c = count_le(mid);
            if (c >= k) {
                hi = mid;
                c_hi = c;
            } else {
                lo = mid + 1;
            }
        }
        bk = lo;
        cle = c_hi;
    }
    double dl = 0.0, dg = 0.0;
    for (int i = lane; i < N; i += 32) {
        const float2 g = d.lut[qv[i]];
        dg += (double)g.y;
        if (qv[i] <= bk) dl += (double)g.x;
    }
    const float sl = (float)warp_sum_d(dl), sgs = (float)warp_sum_d(dg);
    if (lane == 0) {
        // Eq. 27-31 as k_tam evaluates them
        const float topsum = sl - (float)(cle - k) * d.lut[bk].x;
        const float lbar = topsum * (1.0f / (float)k);
        const float dd = d.res / (float)N * sgs;   // d_max - dbar
        const float dbar = d.d_max - dd;
        const float var = fmaxf(d.res2 / (float)N * (float)sumb - dbar * dbar, 0.0f);
        const float sd = fminf(dd, d.d_max - d.d_min) * (1.0f / (d.d_max - d.d_min));
        float T = cbrtf(expf(lbar - 0.5f * var) * sd);
        if (d.fine == kFineTamMean) T = (expf(lbar) + sd + expf(-0.5f * var)) * (1.0f / 3.0f);
        else if (d.fine == kFineBaseline) T = sqrtf(expf(lbar) * sd);
        else if (d.fine == kFineLF) T = topsum;
        double *ps = d.ref_pose + 3 * (size_t)s;
        ps[0] = p.x;
        ps[1] = p.y;
        ps[2] = th0 + atan2(p.s, p.c);
        d.reev[s] = T;
    }
}

}  // namespace

cudaError_t launch_icp(const ReqDesc *reqs, int R, int batch_lo, int batch_hi, int max_L, int max_beams, int max_C,
                       int max_reps, int n_sm, cudaStream_t s) {
    const int slots = (batch_hi - batch_lo) * max_L;
    if (R < 1 || slots < 1) return cudaSuccess;
    const int beams = max_beams > 0 ? max_beams : 1;
    // as many CTAs per pose as give every SM about two (each adds its share of the barriers, not of the FP64 work)
    int cs = kIcpCluster;
    while (cs > 1 && (long long)R * slots * cs > 5ll * n_sm / 2) cs >>= 1;
    const int per = (beams + cs - 1) / cs;
    const size_t table = 16 * ((size_t)(max_C + 2 + 3) / 4 + (size_t)(max_reps + 3) / 4);
    const bool staged = table <= (size_t)kIcpTableBytes;
    const size_t smem = sizeof(double2) * (size_t)per + sizeof(int) * (size_t)((beams + 3) & ~3) + (staged ? table : 0);
    if (smem > 46 * 1024) {
        const cudaError_t e = allow_smem((const void *)k_icp, smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_chained
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(cs * slots, R);
    cfg.blockDim = dim3(kIcpThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_icp, reqs, batch_lo, batch_hi, per, beams, staged);
}

}  // namespace relo
