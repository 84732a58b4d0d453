// k_cluster.cu -- Hilbert-ordered clusters of 32 atoms (clusters.cuh) and the pair histograms
// N_ab(r) over them (Sec. 2.3), on sm_103a.
//
// Per call: Hilbert key and rank of every atom (one atomic per atom), exclusive scan of the key
// counts, scatter, then one kernel that gathers the coordinates in order and reduces the boxes
// of clusters and super-clusters.
#include "clusters.cuh"

namespace epsr {

__global__ void cluster_key_kernel(const BoxDev *boxes, const ClBox *cbox, const int *atom_box, const int4 *coords,
                                   int *key, int *rank, int *count, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int b = atom_box[i];
        const int4 c = coords[i];
        const int L = boxes[b].L, bits = cbox[b].bits;
        const uint64_t rcp = boxes[b].sc_rcp;
        const unsigned m = 1u << bits;
        const unsigned h = hilbert3(__umulhi(scale32(c.x, L, rcp), m), __umulhi(scale32(c.y, L, rcp), m),
                                    __umulhi(scale32(c.z, L, rcp), m), bits);
        const int k = cbox[b].key0 + (int)h;
        key[i] = k;
        rank[i] = atomicAdd(&count[k], 1);
    }
}

// Exclusive scan in one launch: every block sums the counts before its own 4096 (from L2; at
// most kScanOneMax of them), then scans its own.
constexpr int kScanThreads = 1024;

__device__ __forceinline__ int block_excl(int v, int *ws, int &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        int t = ws[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    total = ws[31];
    return x - v + (w ? ws[w - 1] : 0);
}

__global__ void __launch_bounds__(kScanThreads) scan_one_kernel(const int *count, int n, int *offset)
{
    __shared__ int ws[32];
    const int begin = blockIdx.x * 4 * kScanThreads;
    int before = 0;
    const int4 *c4 = reinterpret_cast<const int4 *>(count);
    for (int i = threadIdx.x; i < begin / 4; i += kScanThreads) {
        const int4 v = c4[i];
        before += v.x + v.y + v.z + v.w;
    }
    int base;
    block_excl(before, ws, base);
    const int i0 = begin + 4 * threadIdx.x;
    int v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = i0 + u < n ? count[i0 + u] : 0;
    int total;
    int run = base + block_excl(v[0] + v[1] + v[2] + v[3], ws, total);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (i0 + u < n) offset[i0 + u] = run;
        run += v[u];
    }
}

int launch_scan_one(const int *count, int n, int *offset, cudaStream_t stream)
{
    scan_one_kernel<<<(n + 4 * kScanThreads - 1) / (4 * kScanThreads), kScanThreads, 0, stream>>>(count, n, offset);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "scan");
}

// One CTA per super-cluster, one warp per cluster: gathers the coordinates in cluster order and
// reduces the boxes.
__global__ void __launch_bounds__(1024) cluster_boxes_kernel(const BoxDev *boxes, const ClBox *cbox, const int *su_box,
                                                             const int *index, const int4 *coords, int4 *s_coords,
                                                             int4 *cl_c, int4 *cl_h, int4 *su_c, int4 *su_h)
{
    __shared__ int lo[3][32], hi[3][32];
    const int b = su_box[blockIdx.x];
    const ClBox cb = cbox[b];
    const int s = blockIdx.x - cb.su0, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int cl = s * 32 + w;
    const int num = min(32, boxes[b].n_atoms - cl * 32);          // <= 0: no such cluster
    int4 p = make_int4(0, 0, 0, 0);
    const int first = (int)boxes[b].atom0 + cl * 32;
    const bool in = lane < num;
    if (in) {
        p = coords[index[first + lane]];
        s_coords[first + lane] = p;
    }
    const int v[3] = {p.x, p.y, p.z};
    int mn[3], mx[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        mn[a] = __reduce_min_sync(0xffffffffu, in ? v[a] : 0x7fffffff);
        mx[a] = __reduce_max_sync(0xffffffffu, in ? v[a] : -1);
    }
    if (lane < 3) {
        const int l = lane == 0 ? mn[0] : lane == 1 ? mn[1] : mn[2], u = lane == 0 ? mx[0] : lane == 1 ? mx[1] : mx[2];
        lo[lane][w] = l;
        hi[lane][w] = u;
    }
    if (lane == 0 && num > 0) {
        int c[3], h[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            c[a] = mn[a] + ((mx[a] - mn[a]) >> 1);
            h[a] = mx[a] - c[a];
        }
        cl_c[cb.cl0 + cl] = make_int4(c[0], c[1], c[2], num);
        cl_h[cb.cl0 + cl] = make_int4(h[0], h[1], h[2], first);
    }
    __syncthreads();
    if (w == 0) {
        int c[3], h[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int l = __reduce_min_sync(0xffffffffu, lo[a][lane]), u = __reduce_max_sync(0xffffffffu, hi[a][lane]);
            c[a] = l + ((u - l) >> 1);
            h[a] = u - c[a];
        }
        if (lane == 0) {
            su_c[blockIdx.x] = make_int4(c[0], c[1], c[2], 0);
            su_h[blockIdx.x] = make_int4(h[0], h[1], h[2], 0);
        }
    }
}

int launch_clusters(const BoxDev *boxes, const int *atom_box, const int4 *coords, long long n, const ClScratch &sc,
                    bool ordered, const int **order, cudaStream_t stream)
{
    const int grid = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    // the item counters of the traversal lie behind the key counts: one clear for both
    cudaError_t e = cudaMemsetAsync(sc.count, 0, (size_t)(sc.n_keys_pad + sc.n_boxes) * sizeof(int), stream);
    if (e != cudaSuccess) return set_cuda_error(e, "clusters: clear");
    cluster_key_kernel<<<grid, 256, 0, stream>>>(boxes, sc.box, atom_box, coords, sc.key, sc.rank, sc.count, n);
    note_launch();
    int rc = launch_scan(sc.count, sc.n_keys, sc.offset, sc.block, stream);
    if (rc) return rc;
    if ((rc = launch_scatter(sc.key, sc.rank, sc.offset, sc.index, n, stream))) return rc;
    // the ranks came from atomics; in order of the atoms' numbers (into the ranks' buffer) they do not matter
    if (ordered && (rc = launch_cell_order(sc.key, sc.count, sc.offset, sc.index, sc.rank, n, stream))) return rc;
    const int *index = ordered ? sc.rank : sc.index;
    if (order) *order = index;
    cluster_boxes_kernel<<<sc.n_su, 1024, 0, stream>>>(boxes, sc.box, sc.su_box, index, coords, sc.coords, sc.cl_c,
                                                       sc.cl_h, sc.su_c, sc.su_h);
    note_launch();
    e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "clusters");
}

// ---- exact pair histogram -------------------------------------------------------------------------
// A CTA counts in shared memory, one bin row per ordered type pair (so that the row is the sum of
// a value of i and one of j, whatever the number of types), folded into the caller's pairs when it
// leaves a box. The bin comes from the FP32 squared distance; within its error of a bin edge
// (x 2^-20 of the distance x in bins; the errors of clusters.cuh, of sqrt_approx and of the scale
// add up to less than x (2^-22 + 2^-23 + 2 2^-23)) the exact integer distance and the threshold table decide.
constexpr int kClThreads = 256;
constexpr int kClWarps = kClThreads / 32;

// Exact bin of a pair of grid points (off the main path: about one pair in 10^3), counted in
// the row of its ordered types.
__device__ __noinline__ void gr_count_exact(unsigned *row, const long long *T, long long tmax, float inv, int L, int nb,
                                            int4 pi, int4 pj)
{
    const Sep sp = sep(pi, pj, L);
    const long long d2 = d2_of(sp);
    if (d2 < tmax) atomicAdd(&row[bin_of(d2, g2_of(sp), T, nb, inv)], 1u);
}

// Two squared distances at once: the distances in bins less a half (u), rounded to integers in
// the low bits of t; lane q of `sure` is set when the bin of distance q is certain.
struct Bins2 {
    int k0, k1;
    bool sure0, sure1;
};
__device__ __forceinline__ Bins2 bins2(float g0, float g1, uint64_t INV)
{
    const uint64_t M = pk2(12582912.f, 12582912.f), NM = pk2(-12582912.f, -12582912.f);
    const uint64_t U = fma2(pk2(sqrt_approx(g0), sqrt_approx(g1)), INV, pk2(-0.5f, -0.5f));
    const uint64_t T = add2(U, M);
    const uint64_t D = sub2(U, add2(T, NM));
    const uint64_t E = fma2(U, pk2(-0x1p-20f, -0x1p-20f), pk2(0.5f - 0x1p-20f, 0.5f - 0x1p-20f));
    float t0, t1, d0, d1, e0, e1;
    upk2(T, t0, t1);
    upk2(D, d0, d1);
    upk2(E, e0, e1);
    Bins2 b;
    b.k0 = __float_as_int(t0) - 0x4B400000;
    b.k1 = __float_as_int(t1) - 0x4B400000;
    b.sure0 = fabsf(d0) < e0;
    b.sure1 = fabsf(d1) < e1;
    return b;
}

__global__ void __launch_bounds__(kClThreads, 4) gr_clusters_kernel(ClArgs A)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ int s_found;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    JList &list = reinterpret_cast<JList *>(dyn)[warp];
    unsigned *s_hist = reinterpret_cast<unsigned *>(reinterpret_cast<JList *>(dyn) + kClWarps);
    for (int k = tid; k < A.hist_cap; k += kClThreads) s_hist[k] = 0u;

    int b = start_box(A);
    while ((b = next_box(A, b, &s_found)) >= 0) {
        const BoxDev &bx = A.boxes[b];
        const ClBox cb = A.box[b];
        const int L = bx.L, nt = bx.n_types, nb = bx.n_bins;
        const float hi = bx.tmax_hi, r2 = hi * 1.0001f, inv = bx.inv_dr_fx;
        const uint64_t INV = pk2(inv, inv);
        const int n_items = cb.n_cl << A.plog;
        for (;;) {
            int it = 0;
            if (lane == 0) it = atomicAdd(&A.next_item[b], 1);
            it = __shfl_sync(0xffffffffu, it, 0);
            if (it >= n_items) break;
            const int ci = it >> A.plog, part = it & ((1 << A.plog) - 1);
            const ICluster I = load_icluster(A, cb.cl0 + ci, L, cb.r_fx, lane);
            unsigned *rowi = s_hist + I.p.w * nt * nb;
            // one pair by its grid coordinates
            auto count = [&](int4 pj, int row) {
                const float g2 = g2_of(sep(I.p, pj, L));
                if (g2 >= hi) return;
                const Bins2 k = bins2(g2, g2, INV);
                if (k.sure0) atomicAdd(&rowi[row + k.k0], 1u);
                else gr_count_exact(rowi + row, A.thresholds + bx.tbl_off, bx.tmax, inv, L, nb, I.p, pj);
            };
            if (part == 0) {
                // pairs inside the cluster: lane i with lane i + o, o = 1 .. 16
                for (int o = 1; o <= 16; ++o) {
                    const int src = (lane + o) & 31;
                    const int4 pj = make_int4(__shfl_sync(0xffffffffu, I.p.x, src), __shfl_sync(0xffffffffu, I.p.y, src),
                                              __shfl_sync(0xffffffffu, I.p.z, src), __shfl_sync(0xffffffffu, I.p.w, src));
                    if (lane < I.c.w && src < I.c.w && (o < 16 || lane < 16)) count(pj, pj.w * nb);
                }
            }
            auto value = [nb](const int4 &q) { return __int_as_float(q.w * nb); };
            if (I.fast) {
                const uint64_t XI = pk2(I.fx, I.fx), YI = pk2(I.fy, I.fy), ZI = pk2(I.fz, I.fz);
                visit_partners<false>(A, cb, I, ci, part, A.plog, L, r2, list, lane, value, [&](JList &l, int n) {
                    if ((n & 1) && lane == 0) l.put(n, 3e9f, 0.f, 0.f, 0.f, 0);     // pads the last pair: out of every lane's range
                    __syncwarp();
                    const int np = (n + 1) >> 1;
#pragma unroll 2
                    for (int q = 0; q < np; ++q) {
                        const float4 a = l.a[q], c = l.b[q];
                        const uint64_t DX = sub2(pk2(a.x, a.y), XI), DY = sub2(pk2(a.z, a.w), YI), DZ = sub2(pk2(c.x, c.y), ZI);
                        float g0, g1;
                        upk2(fma2(DX, DX, fma2(DY, DY, mul2(DZ, DZ))), g0, g1);
                        const Bins2 k = bins2(g0, g1, INV);
                        const bool in0 = g0 < hi, in1 = g1 < hi;
                        const int r0 = __float_as_int(c.z), r1 = __float_as_int(c.w);
                        if (in0 && k.sure0) atomicAdd(&rowi[r0 + k.k0], 1u);
                        if (in1 && k.sure1) atomicAdd(&rowi[r1 + k.k1], 1u);
                        const bool x0 = in0 && !k.sure0, x1 = in1 && !k.sure1;
                        if (x0 || x1) {
                            const long long *T = A.thresholds + bx.tbl_off;
                            if (x0) gr_count_exact(rowi + r0, T, bx.tmax, inv, L, nb, I.p, A.coords[l.idx[2 * q]]);
                            if (x1) gr_count_exact(rowi + r1, T, bx.tmax, inv, L, nb, I.p, A.coords[l.idx[2 * q + 1]]);
                        }
                    }
                });
            } else {
                visit_partners<false>(A, cb, I, ci, part, A.plog, L, r2, list, lane, value, [&](JList &l, int n) {
                    if (I.pos < 0) return;
                    for (int s = 0; s < n; ++s) {
                        const float *pa = reinterpret_cast<const float *>(&l.a[s >> 1]) + (s & 1);
                        const float *pb = reinterpret_cast<const float *>(&l.b[s >> 1]) + (s & 1);
                        count(make_int4(__float_as_int(pa[0]), __float_as_int(pa[2]), __float_as_int(pb[0]), 0),
                              __float_as_int(pb[2]));
                    }
                });
            }
        }
        __syncthreads();
        // fold the ordered type pairs into the caller's (upper triangle) histogram
        unsigned long long *out = A.hist + bx.hist_off;
        for (int k = tid; k < nt * nt * nb; k += kClThreads) {
            const unsigned v = s_hist[k];
            if (!v) continue;
            const int r = k / nb;
            atomicAdd(out + pair_index(r / nt, r % nt, nt) * nb + k % nb, (unsigned long long)v);
            s_hist[k] = 0u;
        }
    }
}

size_t gr_clusters_smem(int hist_cap) { return kClWarps * sizeof(JList) + (size_t)hist_cap * sizeof(unsigned); }

int launch_gr_clusters(const ClArgs &args, int grid, cudaStream_t stream)
{
    const size_t smem = gr_clusters_smem(args.hist_cap);
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(gr_clusters_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kClMaxSmem);
        if (e != cudaSuccess) return set_cuda_error(e, "cudaFuncSetAttribute(gr clusters)");
        attr_set = true;
    }
    gr_clusters_kernel<<<grid, kClThreads, smem, stream>>>(args);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "gr clusters");
}

}  // namespace epsr
