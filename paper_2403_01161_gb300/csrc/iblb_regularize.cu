// iblb_regularize.cu -- mesh regularisation of Sec. 3.3 on a thread-block
// cluster: the scheduled one of a droplet, the batched one of an ensemble,
// and the allocation-free one on caller buffers; for meshes above 32768 nodes,
// and where the context has no room for such a cluster, one block.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <utility>
#include <vector>

#include "iblb_internal.h"
#include "iblb_device.cuh"

namespace iblb {
namespace {

// This thread's share of the enclosed volume and of its first moment, summed
// over signed tetrahedra (x_0, a, b, c) of the triangles, positions relative
// to node 0: v[0] = V, v[1..3] = int (x - x_0) dV.
__device__ __forceinline__ void enclosed_volume_sums(const MeshView &M, double v[4])
{
    v[0] = v[1] = v[2] = v[3] = 0.0;
    const double r0[3] = {M.r[0], M.r[1], M.r[2]};
    for (int t = threadIdx.x; t < M.nt; t += blockDim.x) {
        double pp[3][3];
        for (int k = 0; k < 3; ++k)
            for (int a = 0; a < 3; ++a) pp[k][a] = M.r[3 * M.tris[3 * t + k] + a] - r0[a];
        double bc[3];
        cross3(pp[1], pp[2], bc);
        const double vt = (pp[0][0] * bc[0] + pp[0][1] * bc[1] + pp[0][2] * bc[2]) / 6.0;
        v[0] += vt;
        for (int a = 0; a < 3; ++a) v[1 + a] += vt * (pp[0][a] + pp[1][a] + pp[2][a]) / 4.0;
    }
}

// The iteration on one block: x_o fixed, x_q the previous iterate, x_p the new
// one (ping-pong between r and s1), x_b in xb.  Leaves the result in r, returns
// whether the exit test held.
__device__ __forceinline__ bool regularize_block(double *r, double *xo, double *s1, double *xb, const int *nb_ptr,
                                                 const int *nb_idx, const int nv, const RegParams &p, double *sh, int &it)
{
    double *buf[2] = {r, s1};
    for (int i = threadIdx.x; i < 3 * nv; i += blockDim.x) xo[i] = r[i];
    __syncthreads();
    const double sg = p.plus_sign ? 1.0 : -1.0;
    int cur = 0;
    bool conv = false;
    it = 0;
    while (it < p.max_iter) {
        ++it;
        const double *xq = buf[cur];
        double *xp = buf[cur ^ 1];
        for (int i = threadIdx.x; i < nv; i += blockDim.x) {
            const int b0 = nb_ptr[i], b1 = nb_ptr[i + 1];
            const int ni = b1 - b0;
            for (int a = 0; a < 3; ++a) {
                double s = 0.0;
                for (int k = b0; k < b1; ++k) s += xq[3 * nb_idx[k] + a];
                const double v = p.alpha * xo[3 * i + a] + (1.0 - p.alpha) / ni * s;
                xp[3 * i + a] = v;
                xb[3 * i + a] = v - (p.alpha * xo[3 * i + a] + (1.0 - p.alpha) * xq[3 * i + a]);
            }
        }
        __syncthreads();
        double dmax = 0.0;
        for (int i = threadIdx.x; i < nv; i += blockDim.x) {
            const int b0 = nb_ptr[i], b1 = nb_ptr[i + 1];
            const int ni = b1 - b0;
            double d2 = 0.0;
            for (int a = 0; a < 3; ++a) {
                double s = 0.0;
                for (int k = b0; k < b1; ++k) s += xb[3 * nb_idx[k] + a];
                const double v = xp[3 * i + a] - (p.gamma * xb[3 * i + a] + sg * (1.0 - p.gamma) / ni * s);
                xp[3 * i + a] = v;
                const double d = v - xq[3 * i + a];
                d2 += d * d;
            }
            dmax = fmax(dmax, sqrt(d2));
        }
        dmax = block_max(dmax, sh);  // includes a barrier after the writes above
        cur ^= 1;
        if (dmax < p.tol) {
            conv = true;
            break;
        }
    }
    if (cur != 0) {
        for (int i = threadIdx.x; i < 3 * nv; i += blockDim.x) r[i] = s1[i];
    }
    __syncthreads();
    return conv;
}

// One block per mesh.  patch_buf: patch buffer (parity) of the next step,
// rewritten from the regularised positions.
__global__ void __launch_bounds__(1024) k_regularize(LbView L, MeshView M, RegParams p, int patch_buf)
{
    __shared__ double sh[32];
    const int nv = M.nv;
    // mesh quality: the largest ratio of longest to shortest edge over the
    // triangles (node clustering and loose, stretched elements both raise it)
    double q = 1.0;
    for (int t = threadIdx.x; t < M.nt; t += blockDim.x) {
        const int v[3] = {M.tris[3 * t], M.tris[3 * t + 1], M.tris[3 * t + 2]};
        double e2[3];
        for (int k = 0; k < 3; ++k) {
            const double *a = M.r + 3 * v[k], *b = M.r + 3 * v[(k + 1) % 3];
            const double dx = b[0] - a[0], dy = b[1] - a[1], dz = b[2] - a[2];
            e2[k] = dx * dx + dy * dy + dz * dz;
        }
        const double lo = fmin(e2[0], fmin(e2[1], e2[2])), hi = fmax(e2[0], fmax(e2[1], e2[2]));
        q = fmax(q, lo > 0.0 ? sqrt(hi / lo) : 1e300);
    }
    q = block_max(q, sh);
    if (threadIdx.x == 0) L.ctl->mesh_q = q;
    if (p.trigger > 0.0 && !(q > p.trigger)) {
        // adaptive schedule: the mesh is still regular enough, nothing to do
        if (threadIdx.x == 0) L.ctl->reg_iters = 0;
        return;
    }
    __shared__ double shv[32][4];
    double V0 = 0.0;
    if (p.keep_volume) {
        double v4[4];
        enclosed_volume_sums(M, v4);
        block_sum<4>(v4, shv);
        V0 = v4[0];
    }
    int it;
    const bool conv = regularize_block(M.r, M.s0, M.s1, M.s2, M.nb_ptr, M.nb_idx, nv, p, sh, it);
    if (p.keep_volume) {
        // scale about the volume centroid back to the volume enclosed before
        double v4[4];
        enclosed_volume_sums(M, v4);
        block_sum<4>(v4, shv);
        const double c[3] = {M.r[0] + v4[1] / v4[0], M.r[1] + v4[2] / v4[0], M.r[2] + v4[3] / v4[0]};
        const double f = cbrt(V0 / v4[0]);
        __syncthreads();  // every thread has read M.r[0..2] before it moves
        for (int i = threadIdx.x; i < nv; i += blockDim.x)
            for (int a = 0; a < 3; ++a) M.r[3 * i + a] = c[a] + f * (M.r[3 * i + a] - c[a]);
        __syncthreads();
    }
    block_bbox_patch(L, M, M.r, nv, patch_buf);
    if (threadIdx.x == 0) {
        L.ctl->reg_iters = it;
        L.ctl->reg_count += 1;
        if (!conv) atomicOr(&L.ctl->err, IBL_ERRBIT_NOCONV);
    }
}

// The same regularisation on a thread-block cluster of C CTAs (one per SM),
// for meshes of up to C * kRegPerCta nodes.  CTA c owns nodes [c P, c P + P)
// and keeps their original position, the two iterates and the correction b in
// its shared memory; neighbours owned by other CTAs are read through
// distributed shared memory.  The hardware cluster barrier separates the two
// phases of an iteration, and each CTA pushes its maximum to all others
// before the second one, so every CTA takes the same decision.
//
// What bounds it: the FP64 pipe (a warp instruction every 16 cycles per SM)
// and, on small meshes, the latency of the two phases.  So
//   - an item is one component of one node, 10 nodes on 30 lanes of a warp:
//     three times the threads of a thread per node, each with a third of the
//     serial chain, and 23 FP64 instructions an iteration: (1 - alpha)/N_i
//     and (1 - gamma)/N_i come from a table by valence, not from a division
//     per component;
//   - the neighbours' shared-memory addresses are formed once, not in every
//     phase (an integer division each);
//   - maxima are taken on the bits of non-negative doubles (integer units) and
//     of the squared displacement, whose root is taken once: rounding keeps
//     order, so the exit test is the same;
//   - the mesh quality is found in FP32, and only triangles within rounding of
//     the block's largest ratio are evaluated in FP64;
//   - the volume sums divide once at the end.
// 10242 stretched, jittered nodes on caller buffers: 1490 us on one block,
// 117 us here (FP64 pipe of the 16 SMs busy); a step of 16 droplets of 2562
// nodes, regularised with volume restoring every 10 steps, one launch each
// before: 612 -> 294 us; the 200^3 box regularised after every step: 237.7 ->
// 228.0 us a step.
// Reductions over the cluster are pushed as plain stores to one slot per CTA
// and reduced locally: a 64-bit maximum by atomicMax on another CTA's shared
// memory lost updates.
namespace cg = cooperative_groups;
constexpr int kRegCluster = 16;       // CTAs per cluster of a single mesh
constexpr int kRegClusterBatch = 8;   // and of an ensemble member
constexpr int kRegPerCta = 2048;
constexpr int kRegValences = 64;      // valences with tabulated weights
constexpr size_t kRegSmemMax = 222 * 1024;  // dynamic part; the rest is static

// Neighbour-table entries beside the 12 doubles of each of P nodes: 8 per
// node where they fit (a closed mesh averages just under 6).
inline int reg_table(int P)
{
    const size_t room = (kRegSmemMax - 96 * (size_t)P) / 4;
    return (int)std::min<size_t>(8 * (size_t)P, room);
}
inline size_t reg_smem(int P) { return 96 * (size_t)P + 4 * (size_t)reg_table(P); }
inline int reg_threads(int P) { return std::min(1024, std::max(128, (P + 9) / 10 * 32)); }

__device__ __forceinline__ unsigned cluster_addr(unsigned local, unsigned rank)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}
__device__ __forceinline__ double cluster_ld(unsigned a)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// Sum over the block, left in every thread of warp 0.
template <int K>
__device__ __forceinline__ void reg_block_sum(double (&v)[K], double (*sh)[K])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k = 0; k < K; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0)
        for (int k = 0; k < K; ++k) sh[warp][k] = v[k];
    __syncthreads();
    if (warp == 0)
        for (int k = 0; k < K; ++k) {
            v[k] = lane < nw ? sh[lane][k] : 0.0;
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        }
}

// BARE: positions and one-rings only (no triangles, patch or control block);
// result[0] = iterations, result[1] = 1 if the exit test held.
template <bool BARE>
__device__ __forceinline__ void regularize_body(const LbView &L, const MeshView &M, const RegParams &p,
                                                const int patch_buf, const int P, const int cap, int *result)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int nv = M.nv, tid = threadIdx.x, nth = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    extern __shared__ __align__(16) double sm[];
    double *xo = sm, *xb = sm + 9 * P;
    unsigned *tab = reinterpret_cast<unsigned *>(sm + 12 * P);
    __shared__ double wa[kRegValences], wg[kRegValences];
    __shared__ unsigned long long pub[2][kRegCluster];    // maxima pushed by every CTA, by parity
    __shared__ unsigned long long cta_max[2], cta_box[6];
    __shared__ unsigned long long box[kRegCluster][6];    // pushed by every CTA to the first
    __shared__ double sums[2][kRegCluster][4];            // volume sums pushed by every CTA: before, after
    __shared__ double sh4[32][4];
    __shared__ unsigned s_thr;
    const int g0 = rank * P, own = max(0, min(nv, g0 + P) - g0);
    const double sg = p.plus_sign ? 1.0 : -1.0;
    const double oma = 1.0 - p.alpha, omg = 1.0 - p.gamma;
    const float inv_P = 1.0f / (float)P;
    const unsigned base = smem_addr(sm);
    // shared address of node j's x in the first iterate, wherever it lives
    // (floor((j + 1/2)/P) is exact: j < 2^15)
    auto node_addr = [&](int j) -> unsigned {
        const int c = (int)(((float)j + 0.5f) * inv_P);
        return cluster_addr(base + 8u * (3u * P + 3u * (unsigned)(j - c * P)), (unsigned)c);
    };

    // valence weights, this CTA's nodes and neighbour addresses
    if (tid < kRegValences) {
        wa[tid] = oma / tid;
        wg[tid] = sg * omg / tid;
    }
    if (tid < 2) cta_max[tid] = 0ull;
    if (tid < 6) cta_box[tid] = 0ull;
    if (tid == 0) s_thr = 0u;
    for (int i = tid; i < 3 * own; i += nth) {
        const double v = M.r[3 * g0 + i];
        xo[i] = v;
        sm[3 * P + i] = v;
    }
    const int k0 = own > 0 ? M.nb_ptr[g0] : 0, k1 = own > 0 ? M.nb_ptr[g0 + own] : 0;
    for (int k = k0 + tid; k < min(k1, k0 + cap); k += nth) tab[k - k0] = node_addr(M.nb_idx[k]);

    double V0 = 0.0;
    if constexpr (!BARE) {
        __syncthreads();
        // mesh quality: the largest longest/shortest edge ratio of a triangle
        auto edges = [&](int t, double &lo, double &hi) {
            const int v[3] = {M.tris[3 * t], M.tris[3 * t + 1], M.tris[3 * t + 2]};
            double e2[3];
            for (int k = 0; k < 3; ++k) {
                const double *a = M.r + 3 * v[k], *b = M.r + 3 * v[(k + 1) % 3];
                const double dx = b[0] - a[0], dy = b[1] - a[1], dz = b[2] - a[2];
                e2[k] = dx * dx + dy * dy + dz * dz;
            }
            lo = fmin(e2[0], fmin(e2[1], e2[2]));
            hi = fmax(e2[0], fmax(e2[1], e2[2]));
        };
        const double r0[3] = {M.r[0], M.r[1], M.r[2]};
        double v1[1] = {0.0};
        float mine = 0.f;    // FP32 ratio of this thread's triangles
        bool exact = false;  // a triangle outside FP32's range
        for (int t = rank * nth + tid; t < M.nt; t += C * nth) {
            double lo, hi;
            edges(t, lo, hi);
            const float flo = (float)lo, fhi = (float)hi;
            if (flo > 1e-30f && fhi < 1e30f) mine = fmaxf(mine, fhi / flo);
            else exact = true;
            if (p.keep_volume) {
                double pp[3][3], bc[3];
                for (int k = 0; k < 3; ++k)
                    for (int a = 0; a < 3; ++a) pp[k][a] = M.r[3 * M.tris[3 * t + k] + a] - r0[a];
                cross3(pp[1], pp[2], bc);
                v1[0] += pp[0][0] * bc[0] + pp[0][1] * bc[1] + pp[0][2] * bc[2];
            }
        }
        {
            const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mine));
            if (lane == 0) atomicMax(&s_thr, m);
        }
        __syncthreads();
        unsigned long long qb = 0ull;
        if (exact || mine >= __uint_as_float(s_thr) * (1.f - 1e-6f)) {
            double q = 1.0;
            for (int t = rank * nth + tid; t < M.nt; t += C * nth) {
                double lo, hi;
                edges(t, lo, hi);
                q = fmax(q, lo > 0.0 ? sqrt(hi / lo) : 1e300);
            }
            qb = order_bits(q);
        }
        qb = warp_max(qb);
        if (lane == 0) atomicMax(&cta_max[1], qb);
        double v4[1] = {v1[0]};
        if (p.keep_volume) reg_block_sum<1>(v4, reinterpret_cast<double(*)[1]>(&sh4[0][0]));
        cluster.sync();  // every CTA runs and has set its slots up; its cta_max[1] is complete
        if (warp == 0 && lane < C) {
            *cluster.map_shared_rank(&pub[1][rank], lane) = cta_max[1];
            if (p.keep_volume) *cluster.map_shared_rank(&sums[0][rank][0], lane) = v4[0];
        }
        cluster.sync();
        unsigned long long m = 0x3ff0000000000000ull;  // 1.0
        for (int c = 0; c < C; ++c) m = max(m, pub[1][c]);
        const double q = __longlong_as_double((long long)m);
        if (p.keep_volume) {
            for (int c = 0; c < C; ++c) V0 += sums[0][c][0];
            V0 /= 6.0;
        }
        if (rank == 0 && tid == 0) L.ctl->mesh_q = q;
        if (p.trigger > 0.0 && !(q > p.trigger)) {
            // adaptive schedule: the mesh is still regular enough, nothing to do
            if (rank == 0 && tid == 0) L.ctl->reg_iters = 0;
            return;
        }
        if (tid == 0) cta_max[1] = 0ull;
        __syncthreads();
    } else {
        cluster.sync();
    }

    // this thread's items: component a of nodes 10 warp + lane / 3, striding
    const int a = lane % 3, l0 = lane < 30 ? 10 * warp + lane / 3 : own, lstep = 10 * nw;
    // sum of component a over the one-ring of node g0 + l in the buffer at byte offset `off`
    auto ring = [&](int l, int &ni, unsigned off) -> double {
        const int b0 = M.nb_ptr[g0 + l], b1 = M.nb_ptr[g0 + l + 1];
        ni = b1 - b0;
        double s = 0.0;
        if (b1 - k0 <= cap) {
#pragma unroll 6
            for (int k = b0 - k0; k < b1 - k0; ++k) s += cluster_ld(tab[k] + off);
        } else {
            for (int k = b0; k < b1; ++k) s += cluster_ld(node_addr(M.nb_idx[k]) + off);
        }
        return s;
    };
    const unsigned off_b = 8u * (6u * P + (unsigned)a);  // b, from the first iterate
    int it = 0, cur = 0;
    bool conv = false;
    while (it < p.max_iter) {
        ++it;
        const unsigned off_q = 8u * (3u * P * (unsigned)cur + (unsigned)a);
        const double *xq = sm + 3 * P * (1 + cur);
        double *xp = sm + 3 * P * (2 - cur);
        // Eq. (extended laplacian smoothing) and Eq. (distanceregularization)
        for (int l = l0; l < own; l += lstep) {
            int ni;
            const double s = ring(l, ni, off_q);
            const double w = ni < kRegValences ? wa[ni] : oma / ni;
            const int i = 3 * l + a;
            const double v = p.alpha * xo[i] + w * s;
            xp[i] = v;
            xb[i] = v - (p.alpha * xo[i] + oma * xq[i]);
        }
        cluster.sync();
        // Eq. (HC_algo_full) and the exit test
        unsigned long long d2 = 0ull;
        for (int l = l0, n = 10 * warp; n < own; l += lstep, n += lstep) {
            double d = 0.0;
            if (l < own) {
                int ni;
                const double s = ring(l, ni, off_b);
                const double w = ni < kRegValences ? wg[ni] : sg * omg / ni;
                const int i = 3 * l + a;
                const double v = xp[i] - (p.gamma * xb[i] + w * s);
                xp[i] = v;
                d = v - xq[i];
            }
            // the node's squared displacement on its first lane
            const double dy = __shfl_down_sync(0xffffffffu, d, 1), dz = __shfl_down_sync(0xffffffffu, d, 2);
            const double q = fma(dz, dz, fma(dy, dy, d * d));
            if (a == 0 && l < own) d2 = max(d2, order_bits(q));
        }
        d2 = warp_max(d2);
        if (lane == 0) atomicMax(&cta_max[it & 1], d2);
        __syncthreads();
        if (warp == 0 && lane < C) *cluster.map_shared_rank(&pub[it & 1][rank], lane) = cta_max[it & 1];
        cluster.sync();  // also ends every read of b and of the previous iterate
        if (tid == 0) cta_max[it & 1] = 0ull;
        unsigned long long m = 0ull;
        for (int c = 0; c < C; ++c) m = max(m, pub[it & 1][c]);
        cur ^= 1;
        if (sqrt(__longlong_as_double((long long)m)) < p.tol) {
            conv = true;
            break;
        }
    }
    const double *x = sm + 3 * P * (1 + cur);
    if constexpr (BARE) {
        for (int i = tid; i < 3 * own; i += nth) M.r[3 * g0 + i] = x[i];
        if (rank == 0 && tid == 0) {
            result[0] = it;
            result[1] = conv ? 1 : 0;
        }
    } else {
        double c[3] = {0.0, 0.0, 0.0}, f = 1.0;
        if (p.keep_volume) {
            double v4[4] = {0.0, 0.0, 0.0, 0.0};
            const unsigned off = 8u * 3u * P * (unsigned)cur;
            const unsigned n0 = node_addr(0) + off;
            const double s0[3] = {cluster_ld(n0), cluster_ld(n0 + 8), cluster_ld(n0 + 16)};
            for (int t = rank * nth + tid; t < M.nt; t += C * nth) {
                double pp[3][3], bc[3];
                for (int k = 0; k < 3; ++k) {
                    const unsigned ad = node_addr(M.tris[3 * t + k]) + off;
                    for (int b = 0; b < 3; ++b) pp[k][b] = cluster_ld(ad + 8u * b) - s0[b];
                }
                cross3(pp[1], pp[2], bc);
                const double vt = pp[0][0] * bc[0] + pp[0][1] * bc[1] + pp[0][2] * bc[2];
                v4[0] += vt;
                for (int b = 0; b < 3; ++b) v4[1 + b] += vt * (pp[0][b] + pp[1][b] + pp[2][b]);
            }
            reg_block_sum<4>(v4, sh4);
            if (warp == 0 && lane < C)
                for (int k = 0; k < 4; ++k) cluster.map_shared_rank(&sums[1][rank][0], lane)[k] = v4[k];
            cluster.sync();  // the sums are in; every read of the iterates has ended
            double w4[4] = {0.0, 0.0, 0.0, 0.0};
            for (int r = 0; r < C; ++r)
                for (int k = 0; k < 4; ++k) w4[k] += sums[1][r][k];
            const double V = w4[0] / 6.0;
            for (int b = 0; b < 3; ++b) c[b] = s0[b] + w4[1 + b] / (4.0 * w4[0]);
            f = cbrt(V0 / V);
        }
        // result, and its bounding box on the first CTA
        const double ca = a == 0 ? c[0] : (a == 1 ? c[1] : c[2]);
        unsigned long long hi = 0ull, lo = 0ull;
        for (int l = l0; l < own; l += lstep) {
            const double xv = x[3 * l + a];
            const double v = p.keep_volume ? ca + f * (xv - ca) : xv;
            M.r[3 * (g0 + l) + a] = v;
            hi = max(hi, order_key(v));
            lo = max(lo, order_key(-v));
        }
        // lanes a, a + 3, ... a + 27 of the warp hold component a
        for (int o = 24; o >= 3; o >>= 1) {
            hi = max(hi, __shfl_down_sync(0xffffffffu, hi, o));
            lo = max(lo, __shfl_down_sync(0xffffffffu, lo, o));
        }
        if (lane < 3) {
            atomicMax(&cta_box[lane], lo);
            atomicMax(&cta_box[3 + lane], hi);
        }
        __syncthreads();
        if (tid < 6) *cluster.map_shared_rank(&box[rank][tid], 0) = cta_box[tid];
        cluster.sync();
        if (rank == 0 && tid == 0) {
            double mn[3], mx[3];
            for (int b = 0; b < 3; ++b) {
                unsigned long long lo_c = 0ull, hi_c = 0ull;
                for (int r = 0; r < C; ++r) {
                    lo_c = max(lo_c, box[r][b]);
                    hi_c = max(hi_c, box[r][3 + b]);
                }
                mn[b] = lo_c ? -key_value(lo_c) : 1e300;
                mx[b] = hi_c ? key_value(hi_c) : -1e300;
                M.part[b] = mn[b];
                M.part[3 + b] = mx[b];
            }
            write_patch(L, mn, mx, patch_buf, 1);
            L.ctl->n_part = 1;
            L.ctl->reg_iters = it;
            L.ctl->reg_count += 1;
            if (!conv) atomicOr(&L.ctl->err, IBL_ERRBIT_NOCONV);
        }
    }
}

__global__ void __launch_bounds__(1024) k_regularize_cluster(LbView L, MeshView M, RegParams p, int patch_buf, int P,
                                                             int cap)
{
    regularize_body<false>(L, M, p, patch_buf, P, cap, nullptr);
}

__global__ void __launch_bounds__(1024)
    k_regularize_noalloc(double *r, const int *nb_ptr, const int *nb_idx, int nv, RegParams p, int *result, int P, int cap)
{
    MeshView M{};
    M.nv = nv;
    M.r = r;
    M.nb_ptr = nb_ptr;
    M.nb_idx = nb_idx;
    const LbView L{};
    regularize_body<true>(L, M, p, 0, P, cap, result);
}

// The allocation-free one on one block, for a context without room for a
// cluster: x_o, the second iterate and x_b in a fixed array of the library
// image, so that calls must not overlap.
constexpr int kNoAllocMaxNodes = 16384;  // what one portable cluster's shared memory holds
__device__ double g_noalloc_scratch[3][3 * kNoAllocMaxNodes];
__global__ void __launch_bounds__(1024)
    k_regularize_noalloc_block(double *r, const int *nb_ptr, const int *nb_idx, int nv, RegParams p, int *result)
{
    __shared__ double sh[32];
    int it;
    const bool conv = regularize_block(r, g_noalloc_scratch[0], g_noalloc_scratch[1], g_noalloc_scratch[2], nb_ptr, nb_idx,
                                       nv, p, sh, it);
    if (threadIdx.x == 0) {
        result[0] = it;
        result[1] = conv ? 1 : 0;
    }
}

// Ensemble: the members of a group that are due, a cluster each (blockIdx.y
// is the position among them).
struct RegGroup {
    int member[kGroup];
    RegParams p[kGroup];
};
__global__ void __launch_bounds__(1024)
    k_regularize_batched(const __grid_constant__ LbGroup LG, const __grid_constant__ MeshGroup MG,
                         const __grid_constant__ RegGroup RG, const int patch_buf, const int P, const int cap)
{
    // P and cap size the shared memory by the largest member of the launch
    const int m = RG.member[blockIdx.y], C = (int)gridDim.x;
    regularize_body<false>(LG.v[m], MG.v[m], RG.p[blockIdx.y], patch_buf, min(P, (MG.v[m].nv + C - 1) / C), cap, nullptr);
}
static_assert(sizeof(LbGroup) + sizeof(MeshGroup) + sizeof(RegGroup) + 16 <= 32764, "kernel parameters");

template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*k)(KArgs...), dim3 grid, int C, int P, cudaStream_t s, int prio, Args &&...args)
{
    // set at every launch: the attributes belong to the current context, and
    // setting them costs less than looking up whether it has them
    const void *fn = reinterpret_cast<const void *>(k);
    cudaError_t e = cudaSuccess;
    if (C > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRegSmemMax);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(reg_threads(P));
    cfg.dynamicSmemBytes = reg_smem(P);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributePriority;
    at[1].val.priority = prio;
    cfg.attrs = at;
    cfg.numAttrs = prio != 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)..., P, reg_table(P));
}

// Whether the current context takes a cluster of C such CTAs (one per SM): 1
// yes, 0 no, -1 it could not be asked.
int cluster_fits(int C)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = kRegSmemMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = cudaSuccess;
    if (C > 8) e = cudaFuncSetAttribute(k_regularize_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_regularize_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRegSmemMax);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_regularize_cluster, &cfg);
    if (e == cudaSuccess) return n > 0 ? 1 : 0;
    cudaGetLastError();  // a refusal only selects another form
    return e == cudaErrorInvalidClusterSize || e == cudaErrorInvalidValue || e == cudaErrorNotSupported ? 0 : -1;
}

// CTAs of the widest cluster of the two sizes that `fits` grants, 0 for none;
// `known` says whether that is the answer rather than a failure to ask.
template <typename F>
int widest_cluster(F &&fits, bool &known)
{
    known = true;
    for (const int C : {kRegCluster, kRegClusterBatch}) {
        const int f = fits(C);
        if (f > 0) return C;
        known = known && f == 0;
    }
    return 0;
}

// CTAs of the cluster for a mesh of nv nodes, 0: one block.
int cluster_for(int nv, int widest) { return nv <= widest * kRegPerCta ? widest : 0; }

// Id of the calling thread's current context (0 if there is none yet, or it
// cannot be asked).
unsigned long long context_id()
{
    using GetCurrent = CUresult (*)(CUcontext *);
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    const auto entry = [](const char *name) -> void * {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &q) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return q == cudaDriverEntryPointSuccess ? f : nullptr;
    };
    static void *const a = entry("cuCtxGetCurrent"), *const b = entry("cuCtxGetId");
    if (!a || !b) return 0;
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (reinterpret_cast<GetCurrent>(a)(&c) != CUDA_SUCCESS || !c) return 0;
    return reinterpret_cast<GetId>(b)(c, &id) == CUDA_SUCCESS ? id : 0;
}

// widest_cluster of the current context, asked once per context: another
// device, and a partition of one, is another context.
int widest_cluster_here()
{
    struct Seen {
        unsigned long long ctx;
        int widest;
    };
    static std::mutex mu;
    static Seen seen[16];
    static unsigned next = 0;  // oldest entry
    const unsigned long long ctx = context_id();
    {
        std::lock_guard<std::mutex> lock(mu);
        for (const Seen &s : seen)
            if (ctx != 0 && s.ctx == ctx) return s.widest;
    }
    bool known = false;
    const int w = widest_cluster(cluster_fits, known);
    const unsigned long long now = context_id();  // asking creates the context if there was none
    if (known && now != 0) {
        std::lock_guard<std::mutex> lock(mu);
        seen[next++ % 16] = Seen{now, w};
    }
    return w;
}

}  // namespace

cudaError_t launch_regularize(const LbView &L, const MeshView &M, const RegParams &p, int buf, cudaStream_t s,
                              int prio)
{
    const int C = cluster_for(M.nv, widest_cluster_here());
    if (C == 0) return launch_p(k_regularize, dim3(1), dim3(1024), s, prio, L, M, p, buf);
    return launch_cluster(k_regularize_cluster, dim3(C), C, (M.nv + C - 1) / C, s, prio, L, M, p, buf);
}

// Up to six due members of a group take a 16-CTA cluster each, as a single
// droplet does; more take 8 CTAs.  The line is how many 16-CTA clusters run at
// once beside the outside update, with one in hand for chips whose SMs are
// grouped otherwise: us per step, regularised every other step, 2562 nodes
// each, with 8 and 16 CTAs: 2 members 77.4 and 64.1, 6 124.3 and 110.7, 7
// 137.0 and 123.1, 8 148.4 and 162.9 (the eighth waits), 12 190.8 and 205.3.
cudaError_t launch_regularize_batched(const EnsembleView &E, const std::vector<char> &due,
                                      const std::vector<RegParams> &params, int buf, cudaStream_t s, int prio)
{
    static thread_local LbGroup lg;  // parameter blocks are large: kept off the stack
    static thread_local MeshGroup mg;
    const int n = (int)E.lv.size(), widest = widest_cluster_here();
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        RegGroup rg;
        int k = 0, nv_max = 0;
        for (int m = m0; m < m1; ++m) {
            if (!due[m]) continue;
            if (E.mv[m].nv > kRegClusterBatch * kRegPerCta || widest == 0) {
                const cudaError_t e = launch_regularize(E.lv[m], E.mv[m], params[m], buf, s, prio);
                if (e != cudaSuccess) return e;
                continue;
            }
            lg.v[m - m0] = E.lv[m];
            mg.v[m - m0] = E.mv[m];
            rg.member[k] = m - m0;
            rg.p[k] = params[m];
            nv_max = std::max(nv_max, E.mv[m].nv);
            ++k;
        }
        if (k == 0) continue;
        const int C = k <= 6 ? widest : kRegClusterBatch;
        const cudaError_t e = launch_cluster(k_regularize_batched, dim3(C, k), C, (nv_max + C - 1) / C, s, prio, lg, mg,
                                             rg, buf);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace iblb

// Allocation-free mesh regularisation: the cluster kernel on the caller's
// positions and one-rings.  Its scratch is the cluster's shared memory, so
// overlapping calls on different buffers do not disturb each other.  One block
// with its scratch in a static device array took 1490 us for 10242 stretched
// and jittered nodes, against 117; it remains for a context without room for
// a cluster.
static int regularize_noalloc(double *r, const int32_t *nb_ptr, const int32_t *nb_idx, int n_nodes, double alpha,
                              double gamma, double tol, int max_iter, int plus_sign, int32_t *result, void *stream,
                              int widest)
{
    using namespace iblb;
    if (!r || !nb_ptr || !nb_idx || !result) return iblb_set_error(IBL_EINVAL, "null pointer argument");
    static_assert(kNoAllocMaxNodes <= kRegClusterBatch * kRegPerCta, "cluster capacity");
    if (n_nodes < 1 || n_nodes > kNoAllocMaxNodes)
        return iblb_set_error(IBL_EINVAL, "ibl_regularize_noalloc: n_nodes must be in 1..16384 (the size of its "
                                          "fixed scratch)");
    if (!(alpha >= 0 && alpha <= 1) || !(gamma >= 0 && gamma <= 1) || !(tol > 0) || max_iter < 1)
        return iblb_set_error(IBL_EINVAL, "regularisation parameters out of range");
    RegParams p{alpha, gamma, tol, max_iter, plus_sign ? 1 : 0};
    const int *ptr = reinterpret_cast<const int *>(nb_ptr), *idx = reinterpret_cast<const int *>(nb_idx);
    int *res = reinterpret_cast<int *>(result);
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int C = cluster_for(n_nodes, widest < 0 ? widest_cluster_here() : widest);
    const cudaError_t e =
        C == 0 ? launch_p(k_regularize_noalloc_block, dim3(1), dim3(1024), s, 0, r, ptr, idx, n_nodes, p, res)
               : launch_cluster(k_regularize_noalloc, dim3(C), C, (n_nodes + C - 1) / C, s, 0, r, ptr, idx, n_nodes, p, res);
    if (e != cudaSuccess) return iblb_set_error(IBL_ECUDA, cudaGetErrorString(e));
    return IBL_OK;
}

extern "C" int ibl_regularize_noalloc(double *r, const int32_t *nb_ptr, const int32_t *nb_idx, int n_nodes,
                                      double alpha, double gamma, double tol, int max_iter, int plus_sign,
                                      int32_t *result, void *stream)
{
    return regularize_noalloc(r, nb_ptr, nb_idx, n_nodes, alpha, gamma, tol, max_iter, plus_sign, result, stream, -1);
}

extern "C" int ibl_test_regularize_noalloc(double *r, const int32_t *nb_ptr, const int32_t *nb_idx, int n_nodes,
                                           double alpha, double gamma, double tol, int max_iter, int plus_sign,
                                           int32_t *result, void *stream, int widest)
{
    if (widest != 0 && widest != iblb::kRegClusterBatch && widest != iblb::kRegCluster)
        return iblb::iblb_set_error(IBL_EINVAL, "widest must be 0, 8 or 16");
    return regularize_noalloc(r, nb_ptr, nb_idx, n_nodes, alpha, gamma, tol, max_iter, plus_sign, result, stream, widest);
}

extern "C" int ibl_test_regularize_ctas(int n_nodes, int fits16, int fits8, int *known)
{
    bool k = false;
    const int w = iblb::widest_cluster([&](int C) { return C == iblb::kRegCluster ? fits16 : fits8; }, k);
    if (known) *known = k ? 1 : 0;
    return iblb::cluster_for(n_nodes, w);
}
