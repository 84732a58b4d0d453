// clusters.cuh -- pair traversal of a box by clusters of 32 atoms with bounding boxes.
//
// Atoms are ordered along a Hilbert curve of small cells, so 32 consecutive atoms (a cluster,
// one per lane of a warp) fill a compact region, about 7 A wide in a liquid, and 32 consecutive
// clusters (a super-cluster) one of about 22 A. A work item is one i-cluster (and one of `parts`
// interleaved shares of its partners): the warp tests the boxes of the super-clusters, then of
// the clusters of the near ones, one per lane, then every atom of a near cluster against the
// i-cluster's box, and the atoms left are compacted into a per-warp list which all 32 i-atoms
// scan together. Of the pairs so scanned about a third lie inside the range, against 0.4 % of
// all pairs and 15 % of the pairs of neighbouring range-wide cells.
//
// Fast coordinates: relative to the centre c of the i-cluster's box, j' = wrap(x_j - c) and
// i' = x_i - c as FP32. With h the half width of the box, |i'| <= h <= 2^23 is exact, and an
// atom inside the range R of some i has |j'| <= R + h; where 2 (R + h) < L the difference j' - i'
// is the minimum image of every pair in range, and where R + h <= 2^25 it is off by the rounding of
// j', at most one grid unit and only when |j'| >= 2^24, where the component is longer than 2^24 -
// 2^23 = 2^23 units, and by its own, one more from 2^24 units on: either is at most 2^-23 of the
// component, so the squared distance carries a relative error below 2^-21 + 2^-22 (rounding of the
// squares), its root half of that. Clusters that do not meet the three conditions (boxes less
// than about twice the range wide, sparse boxes, fine grids) keep integer coordinates in the
// list and take the integer minimum image per pair.
#pragma once

#include "epsr_device.cuh"
#include "epsr_internal.h"

namespace epsr {

// ---- two FP32 values per 64-bit register (packed f32x2 instructions of sm_100 and later) ------
__device__ __forceinline__ uint64_t pk2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t r, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// Square root with relative error at most 2^-23 (no denormal inputs here: 0 or at least 1).
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Per-warp list of partner atoms: slots 2q and 2q + 1 share a[q] = {x, x, y, y} and b[q] =
// {z, z, w, w}, so that a broadcast 128-bit load gives packed operands. Fast clusters hold
// FP32 coordinates relative to the i-cluster's centre, the others the grid coordinates (int
// bits); w is the caller's value per partner, idx its position in the cluster order.
constexpr int kListCap = 64;
struct __align__(16) JList {
    float4 a[kListCap / 2];
    float4 b[kListCap / 2];
    int idx[kListCap];

    __device__ __forceinline__ void put(int s, float x, float y, float z, float w, int i)
    {
        float *pa = reinterpret_cast<float *>(&a[s >> 1]) + (s & 1);
        float *pb = reinterpret_cast<float *>(&b[s >> 1]) + (s & 1);
        pa[0] = x; pa[2] = y;
        pb[0] = z; pb[2] = w;
        idx[s] = i;
    }
    // slots [32, n) move to [0, n - 32), n <= 64 (whole warp)
    __device__ __forceinline__ void shift_down(int n, int lane)
    {
        const int s = 32 + lane;
        float x = 0.f, y = 0.f, z = 0.f, w = 0.f;
        int i = 0;
        __syncwarp();
        if (s < n) {
            const float *pa = reinterpret_cast<const float *>(&a[s >> 1]) + (s & 1);
            const float *pb = reinterpret_cast<const float *>(&b[s >> 1]) + (s & 1);
            x = pa[0]; y = pa[2]; z = pb[0]; w = pb[2];
            i = idx[s];
        }
        __syncwarp();
        if (s < n) put(lane, x, y, z, w, i);
        __syncwarp();
    }
};

// Lower bound of the periodic distance between two boxes (centre, half width) against r2.
__device__ __forceinline__ bool boxes_near(int4 c, int4 h, int4 cj, int4 hj, int L, float r2)
{
    const float x = (float)max(0, mi_abs(c.x - cj.x, L) - h.x - hj.x);
    const float y = (float)max(0, mi_abs(c.y - cj.y, L) - h.y - hj.y);
    const float z = (float)max(0, mi_abs(c.z - cj.z, L) - h.z - hj.z);
    return fmaf(x, x, fmaf(y, y, z * z)) < r2;
}

__device__ __forceinline__ int wrap_half(int t, int L)   // t in (-L, L) -> about [-L/2, L/2]
{
    const int hl = L >> 1;
    if (t > hl) t -= L;
    else if (t < -hl) t += L;
    return t;
}

// The i-cluster of a work item.
struct ICluster {
    int4 c, h;         // centre and atom count; half widths and first position in cluster order
    int4 p;            // this lane's atom (grid coordinates, type), or zeros
    int pos;           // its position in cluster order, or -1
    bool fast;
    float fx, fy, fz;  // relative coordinates (fast); 1e9 where the lane has no atom
};

__device__ __forceinline__ ICluster load_icluster(const ClArgs &A, int cl, int L, int r_fx, int lane)
{
    ICluster I;
    I.c = A.cl_c[cl];
    I.h = A.cl_h[cl];
    I.pos = lane < I.c.w ? I.h.w + lane : -1;
    I.p = I.pos >= 0 ? A.coords[I.pos] : make_int4(0, 0, 0, 0);
    const int hm = max(I.h.x, max(I.h.y, I.h.z));
    I.fast = hm <= (1 << 23) && (long long)r_fx + hm <= (1LL << 25) && 2 * ((long long)r_fx + hm) < L;
    I.fx = I.pos >= 0 ? (float)(I.p.x - I.c.x) : 1e9f;
    I.fy = (float)(I.p.y - I.c.y);
    I.fz = (float)(I.p.z - I.c.z);
    return I;
}

// Visits the partners of an i-cluster in later clusters, or (ALL) in every other cluster (share
// `part` of 2^plog): calls
// scan(list, n) for up to 32 listed partners at a time (n <= 32, the tail of an item may be
// shorter), every lane taking its own i-atom against each. value(j) gives the list's w.
template <bool ALL, class Value, class Scan>
__device__ __forceinline__ void visit_partners(const ClArgs &A, const ClBox &cb, const ICluster &I, int ci, int part,
                                               int plog, int L, float r2, JList &list, int lane, Value value, Scan scan)
{
    const unsigned lt = (1u << lane) - 1u;
    int cnt = 0;
    for (int s0 = ALL ? 0 : ci >> 5; s0 < cb.n_su; s0 += 32) {
        const int s = s0 + lane;
        bool near = s < cb.n_su;
        if (near) near = boxes_near(I.c, I.h, A.su_c[cb.su0 + s], A.su_h[cb.su0 + s], L, r2);
        for (unsigned ms = __ballot_sync(0xffffffffu, near); ms; ms &= ms - 1u) {
            const int jc = ((s0 + __ffs(ms) - 1) << 5) + lane;
            bool nj = (ALL ? jc != ci : jc > ci) && jc < cb.n_cl && (jc & ((1 << plog) - 1)) == part;
            int first = 0, num = 0;
            if (nj) {
                const int4 cj = A.cl_c[cb.cl0 + jc], hj = A.cl_h[cb.cl0 + jc];
                nj = boxes_near(I.c, I.h, cj, hj, L, r2);
                first = hj.w;
                num = cj.w;
            }
            unsigned mj = __ballot_sync(0xffffffffu, nj);
            if (!mj) continue;
            // the atoms of the next near cluster are loaded while those of the last are scanned
            int src = __ffs(mj) - 1;
            int jp = __shfl_sync(0xffffffffu, first, src) + lane;
            bool in = lane < __shfl_sync(0xffffffffu, num, src);
            int4 pj = in ? A.coords[jp] : make_int4(0, 0, 0, 0);
            while (mj) {
                mj &= mj - 1u;
                const int4 q = pj;
                const int qp = jp;
                const bool qin = in;
                if (mj) {
                    src = __ffs(mj) - 1;
                    jp = __shfl_sync(0xffffffffu, first, src) + lane;
                    in = lane < __shfl_sync(0xffffffffu, num, src);
                    pj = in ? A.coords[jp] : make_int4(0, 0, 0, 0);
                }
                const int dx = wrap_half(q.x - I.c.x, L), dy = wrap_half(q.y - I.c.y, L), dz = wrap_half(q.z - I.c.z, L);
                const float ax = (float)max(0, abs(dx) - I.h.x), ay = (float)max(0, abs(dy) - I.h.y),
                            az = (float)max(0, abs(dz) - I.h.z);
                const bool keep = qin && fmaf(ax, ax, fmaf(ay, ay, az * az)) < r2;
                const unsigned mk = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int slot = cnt + __popc(mk & lt);
                    const float w = value(q);
                    if (I.fast) list.put(slot, (float)dx, (float)dy, (float)dz, w, qp);
                    else list.put(slot, __int_as_float(q.x), __int_as_float(q.y), __int_as_float(q.z), w, qp);
                }
                cnt += __popc(mk);
                if (cnt >= 32) {
                    __syncwarp();
                    scan(list, 32);
                    list.shift_down(cnt, lane);
                    cnt -= 32;
                }
            }
        }
    }
    if (cnt) {
        __syncwarp();
        scan(list, cnt);
        __syncwarp();
    }
}

// Work of the persistent CTAs: each starts at the box that holds its share of the clusters and
// goes on to any box with items left. Returns the next box with unclaimed items at or after
// `from` (cyclically, `tried` boxes seen), or -1; called by the whole CTA.
__device__ __forceinline__ int next_box(const ClArgs &A, int from, int *s_found)
{
    const int nb = A.n_boxes;
    for (int v0 = 0; v0 < nb; v0 += blockDim.x) {
        __syncthreads();
        if (threadIdx.x == 0) *s_found = 1 << 30;
        __syncthreads();
        const int v = v0 + threadIdx.x;
        if (v < nb) {
            const int b = from + v < nb ? from + v : from + v - nb;
            if (ld_relaxed_gpu(&A.next_item[b]) < (A.box[b].n_cl << A.plog)) atomicMin(s_found, v);
        }
        __syncthreads();
        const int f = *s_found;
        if (f < (1 << 30)) return from + f < nb ? from + f : from + f - nb;
    }
    return -1;
}

// First box of a CTA: the one holding cluster blockIdx / gridDim of all clusters.
__device__ __forceinline__ int start_box(const ClArgs &A)
{
    const long long c = A.box[0].cl0 + (long long)blockIdx.x * A.n_cl_total / gridDim.x;
    int lo = 0, hi = A.n_boxes;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (A.box[mid].cl0 <= c) lo = mid;
        else hi = mid;
    }
    return lo;
}

}  // namespace epsr
