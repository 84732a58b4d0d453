// k_mc.cu -- Metropolis Monte Carlo sweep (Sec. 2.2 item III) with the per-move energy
// change of the moved molecule against all atoms (Sec. 2.3), on sm_103a.
//
// Two kernels per chunk of moves:
//  1. mc_moves_kernel, one thread per (box, move): everything about a move that does not
//     depend on the configuration -- the Philox words, the molecule, the shift, the
//     rotation matrix (FP64, rounded to 2^-30 fixed point) and the Metropolis threshold
//     -kT ln u (rounded up to FP32, which makes `dU < threshold` in FP32 the same test
//     as in FP64). GB300's FP64 unit is narrow, so this runs once per move on the whole
//     GPU instead of once per move in every CTA.
//  2. mc_sweep_kernel, a cooperative persistent kernel: every box of the handle owns a
//     contiguous group of CTAs; each CTA keeps a slice of its box's atoms (the partners)
//     resident in shared memory for the whole sweep: a contiguous run of every type's Hilbert
//     order, so a compact region, in chunks of 32 slots with bounding boxes.
//
// Batching without changing the chain: moves are taken in batches of up to K
// consecutive moves with distinct molecules (a batch ends before the first molecule that
// repeats; K <= 64). The CTA computes the partial dU of every move against its slice as it
// stood at the start of the batch. One grid barrier per batch gathers the per-CTA partials; every
// CTA sums them in the same fixed order and resolves the batch in order: move k's dU is
// its batch-start value plus, for every earlier accepted move k' of the batch, the exact
// change of the pair energies between the two moved molecules,
// u(new,new') - u(old,new') - u(new,old') + u(old,old'). That is the energy change
// against the state after moves 0..k-1, i.e. the sequential Metropolis chain. Where such a change
// cancels most of the batch-start value (a trial on top of a molecule that an earlier move of the
// batch takes away), the batch is cut before that move, which goes into the next one.
//
// Every device-side wait is bounded by a time limit and an iteration limit; on expiry
// the kernel records a timeout in the status word and all CTAs return.
#include "epsr_device.cuh"
#include "epsr_internal.h"

namespace epsr {

constexpr int kMcThreads = 512;
constexpr int kMcWarps = kMcThreads / 32;
constexpr int kBatchMax = kMcBatchMax;         // moves per batch: warp w takes moves w, w + 16, w + 32, w + 48
constexpr int kPerWarp = kBatchMax / kMcWarps;  // moves per warp and batch
constexpr int kMoveRing = 2 * kBatchMax;        // move records held: a batch and the 64 moves after it
constexpr int kCorrItems = kMcCorrItems;       // >= 496 pairs x 8 atoms (coarse items at G = 1)
constexpr int kQueue = kBatchMax * kBatchMax / 2;   // near items of one round (in the corrections' buffer)
constexpr int kNoAtom = -1;                    // .w of a slot past the end of its type
constexpr int kEscMax = 256;                   // largest escapee_cap that epsr_mc_set_cells accepts
static_assert(kMcCorrPerCta == kBatchMax * (kBatchMax - 1) / 2 && kMcSlotStride == kBatchMax + kMcCorrPerCta,
              "barrier slot layout");
static_assert(kMcThreads == 8 * kBatchMax, "gather: 8 threads per move");
constexpr int kGatherLoads = 5;                 // gather: 16-byte loads per thread in flight (CTA groups up to 160)
static_assert(kPerWarp == 4 && kBatchMax == 64, "phase A / F: two moves per lane of warp 0; phase B: the four moves of a warp in 8-lane groups");
static_assert(kMaxMolAtoms <= 8, "phase B: one lane per atom in 8-lane groups");

// ---- 1. configuration-independent part of each move ----------------------------------------
// A block takes 128 consecutive moves of one box; the molecules of the 192 moves before them are
// drawn again, so that every move knows how long ago its molecule was last moved (the batches of
// the sweep and the coordinates in flight between them follow from that without any search).
constexpr int kMovesThreads = 128;

__global__ void __launch_bounds__(kMovesThreads) mc_moves_kernel(const BoxDev *boxes, const int *mol_start, int n_boxes,
                                                                 long long chunk, long long n, unsigned long long seed,
                                                                 unsigned long long move0, MoveRec *out)
{
    __shared__ int s_mol[kMovePrevWindow + kMovesThreads];
    const long long per_box = (n + kMovesThreads - 1) / kMovesThreads;
    for (long long blk = blockIdx.x; blk < per_box * n_boxes; blk += gridDim.x) {
        const int b = (int)(blk / per_box);
        const long long t = (blk % per_box) * kMovesThreads + threadIdx.x;
        const BoxDev &bx = boxes[b];
        __syncthreads();
        for (int i = threadIdx.x; i < kMovePrevWindow + kMovesThreads; i += kMovesThreads) {
            const long long ti = t - threadIdx.x - kMovePrevWindow + i;
            int mol = -1;
            if (ti >= 0 && ti < n) {
                const unsigned long long mi = move0 + (unsigned long long)ti;
                const U32x4 r = philox4x32_10((uint32_t)mi, (uint32_t)(mi >> 32), (uint32_t)b, 0u, (uint32_t)seed,
                                              (uint32_t)(seed >> 32));
                mol = (int)(((unsigned long long)r.v[0] * (unsigned long long)bx.n_mol) >> 32);
            }
            s_mol[i] = mol;
        }
        __syncthreads();
        if (t >= n) continue;
        const long long e = b * chunk + t;
        const unsigned long long mv = move0 + (unsigned long long)t;
        const bool flex = bx.move_kind == EPSR_MOVE_FLEXIBLE_MOLECULE;
        uint32_t w[16];
#pragma unroll
        for (int lane = 0; lane < 4; ++lane) {
            if (lane == 3 && !flex) break;
            const U32x4 r = philox4x32_10((uint32_t)mv, (uint32_t)(mv >> 32), (uint32_t)b,
                                          (uint32_t)lane, (uint32_t)seed, (uint32_t)(seed >> 32));
#pragma unroll
            for (int i = 0; i < 4; ++i) w[4 * lane + i] = r.v[i];
        }
        MoveRec m;
        m.mol = s_mol[kMovePrevWindow + threadIdx.x];
        m.prev = kMovePrevNone;
        for (int d = kMovePrevWindow; d > 0; --d)
            if (s_mol[kMovePrevWindow + threadIdx.x - d] == m.mol) m.prev = d;
        m.a0 = mol_start[bx.mol0 + m.mol];
        m.m = mol_start[bx.mol0 + m.mol + 1] - m.a0;
        const unsigned span = 2u * (unsigned)bx.max_shift + 1u;
        for (int a = 0; a < 3; ++a) m.shift[a] = (int)(w[1 + a] % span) - bx.max_shift;
        // kind: 0 translate every atom, 1 rotate about the centre (then translate, for rigid
        // molecules), 2 translate one atom; flexible molecules draw the kind from w12 and the
        // atom from w13, and their rotations are not translated
        m.kind = (short)(flex ? (int)(w[12] % 3u) : (bx.move_kind == EPSR_MOVE_RIGID_MOLECULE ? 1 : 0));
        m.atom = (short)(flex ? (int)(w[13] % (uint32_t)m.m) : 0);
        if (flex && m.kind == 1) m.shift[0] = m.shift[1] = m.shift[2] = 0;
        if (m.kind == 1) {
            const double vx = __dmul_rn(bx.h_rot, __dsub_rn(__dmul_rn(2.0, uniform53(w[4], w[5])), 1.0));
            const double vy = __dmul_rn(bx.h_rot, __dsub_rn(__dmul_rn(2.0, uniform53(w[6], w[7])), 1.0));
            const double vz = __dmul_rn(bx.h_rot, __dsub_rn(__dmul_rn(2.0, uniform53(w[8], w[9])), 1.0));
            rotation_fixed(vx, vy, vz, m.R);
        } else {
            for (int i = 0; i < 9; ++i) m.R[i] = 0;
        }
        const double u = uniform53(w[10], w[11]);
        m.u_acc = u;
        // accept iff dU <= 0 or dU < -kT ln u; a float rounded up from the FP64 threshold
        // gives the identical comparison for FP32 dU
        m.thr = __double2float_ru(-bx.kT * log(u));
        out[e] = m;
    }
}

int launch_mc_moves(const BoxDev *boxes, const int *mol_start, int n_boxes, long long chunk,
                    long long n, unsigned long long seed, unsigned long long move0, MoveRec *out,
                    cudaStream_t stream)
{
    const long long blocks = (n + kMovesThreads - 1) / kMovesThreads * n_boxes;
    const int grid = (int)(blocks < 8192 ? blocks : 8192);
    mc_moves_kernel<<<grid, kMovesThreads, 0, stream>>>(boxes, mol_start, n_boxes, chunk, n, seed, move0, out);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EPSR_OK : set_cuda_error(e, "mc_moves");
}

// ---- 2. persistent sweep ----------------------------------------------------------------------
// One batch of moves. Two are held: the next one is prepared while the grid barrier of the
// current one is on its way.
struct McBatch {
    int nb;                                  // moves
    int mm;                                  // largest molecule
    int mol[kBatchMax];
    int acc[kBatchMax];
    int4 newp[kBatchMax][kMaxMolAtoms];
    int4 oldp[kBatchMax][kMaxMolAtoms];
    int natoms[kBatchMax];
    int a0[kBatchMax];
    int spos[kBatchMax][kMaxMolAtoms];   // type-major sorted position of each moved atom
    float hw2[kBatchMax];                // square of the near radius around old atom 0 (2^32-periodic grid)
    // per move and partner type: bit a of the low (high) byte set when moved atom a has a
    // Lennard-Jones (near-only) row with the type
    unsigned short rows[kBatchMax][kMaxTypes];
    int lj_atoms[kBatchMax];                 // moved atoms with a Lennard-Jones row
    // first three atoms of each move on the 2^32-periodic grid, new and old: [move][atom][axis]
    unsigned scn[kBatchMax][3][3];
    unsigned sco[kBatchMax][3][3];
    float thr[kBatchMax];
    double u_acc[kBatchMax];
    float intra[kBatchMax];                 // flexible molecules: change of the springs
};

struct McShared {
    BoxDev bx;
    McBatch b[2];
    MoveRec ring[kMoveRing];                 // move t at t mod kMoveRing, copied in ahead of use
    int nb_min;                              // first move of the next batch that repeats a molecule
    int cut;                                 // first move of the batch whose dU the corrections cancel
    int n_queue;                             // near items of the batch
    // this CTA's partners: per type t, the chunks first[t], first[t] + G, .. of its sorted order, held
    // as its chunks [cbase[t], cbase[t + 1]); chunk c at slice slots [c 2^cs, (c + 1) 2^cs)
    int first[kMaxTypes];
    int cbase[kMaxTypes + 1];
    float part[kBatchMax];
    float base[kBatchMax];
    float dU[kBatchMax];
    float acc_du[2 * kBatchMax];            // rank 0: dU of the decided moves if accepted, else 0
    int abort_flag;
    // leader-only running statistics
    long long st_att, st_acc, st_nonfinite;
    double st_sum;
};
static_assert(sizeof(McShared) + kMcMaxDynSmem <= 227 * 1024, "static plus dynamic shared memory per CTA");


// s += x, the rounding error added to e (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float &s, float &e, float x)
{
    const float t = s + x, b = t - s;
    e += (s - (t - b)) + (x - b);
    s = t;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Warp-wide FP64 sum of v[0..n) (lane-strided, then a fixed shuffle tree), added to acc by lane 0.
__device__ __forceinline__ void block_sum_du(const float *v, int n, int lane, double &acc)
{
    double s = 0.0;
    for (int i = lane; i < n; i += 32) s += (double)v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) acc += s;
}

// Correction of local pair u: the sum over atoms a of move k of the sum over atoms b of move
// k1 of [du(a; b new) - du(a; b old)], in that order. `fine` items hold each du separately;
// otherwise each item already holds the sum over b (same operations, same order).
// Metropolis test of a move with energy change d against its threshold thr = -kT ln u:
// accepted when d <= 0 or d < thr (Sec. 2.2); false for a NaN d.
__device__ __forceinline__ bool metropolis(float d, float thr) { return (d <= 0.f) || (d < thr); }

// True when the corrections of the accepted moves, of magnitude w in all, cancel the batch-start value d
// of a move down to f: what the FP32 sums of d lost below 2^-24 of it would then show in f. The bar is
// a rounding of 6e-5 kJ/mol, and 4e-6 of f: below that f is as good as any FP32 sum. Random boxes with
// steps up to 2 A, worst error against 1e-5 of the condition scale + 1e-4 kJ/mol: 260 times without the cut
// (15 times with batches of 16), 0.2 with it. 99,999-atom water 751 -> 754 us for 3,000 moves.
constexpr float kCancelled = 512.f;
__device__ __forceinline__ bool cancelled(float d, float w, float f)
{
    return !(w <= kCancelled) && !(fabsf(f) >= (fabsf(d) + w) * 0x1p-6f);
}

// Later move k of batch pair pq = k (k - 1) / 2 + k1 (0 <= k1 < k): a float estimate of
// the root of k (k - 1) / 2 = pq, corrected by one step either way.
__device__ __forceinline__ int pair_hi(int pq)
{
    int k = (int)((1.f + sqrtf(8.f * (float)pq + 1.f)) * 0.5f);
    if (k * (k - 1) / 2 > pq) --k;
    if ((k + 1) * k / 2 <= pq) ++k;
    return k;
}

__device__ __forceinline__ float corr_sum(const float *part, int u, int mm, bool fine)
{
    float c = 0.f;
    for (int a = 0; a < mm; ++a) {
        float ca = 0.f;
        if (fine)
            for (int b = 0; b < mm; ++b) {
                const float *v = part + ((u * mm + a) * mm + b) * 2;
                ca += v[0] - v[1];
            }
        else
            ca = part[u * mm + a];
        c += ca;
    }
    return c;
}

__device__ __forceinline__ int floordiv32(int a, int b)   // b > 0
{
    int q = a / b;
    if ((a % b) != 0 && a < 0) --q;
    return q;
}

// Out-of-line copy of pair_du for code that runs once per batch (keeps the kernel small).
template <bool CUT>
__device__ __noinline__ float pair_du_cold(Sep sn, Sep so, const PairRow &pr, const BoxDev &bx,
                                           const long long *T, const float *ep)
{
    return pair_du<CUT>(sn, so, pr, bx, T, ep);
}

// Two FP32 values in one 64-bit register, operated on by the packed f32x2 instructions of
// sm_100 and later: one instruction for the same operation on the two partners of a lane.
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t r, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float rcp_approx(float x)      // 1 ulp
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// floor(x 2^32 / L) or one less, for 0 <= x < L, from rcp = floor((2^64 - 1) / L): the coordinate
// on the 2^32-periodic grid, where a 32-bit difference wraps to the minimum image. The sweep uses
// it for far pairs and for chunk boxes only, so one unit (2^-32 of the box side) does not matter.
__device__ __forceinline__ unsigned scale32_near(int x, uint64_t rcp)
{
    return (unsigned)x * (unsigned)(rcp >> 32) + __umulhi((unsigned)x, (unsigned)rcp);
}

// Lennard-Jones change u(r') - u(r) of two far partners p and q (one f32x2 lane pair) on the
// 2^32-periodic grid, against a moved atom's new and old position there: a 32-bit difference
// wraps to the minimum image, so a separation component costs one subtraction and one
// conversion, and the two partners share every FP32 instruction. r and r' share a reciprocal,
// 1/r'^2 = r^2 / (r^2 r'^2) (neither is 0: such a partner is near): 1.5e6-atom water 602 -> 591 us
// for 400 moves against four root reciprocals. Taken directly: its rounding is a few ulp of |u|,
// which is small beyond the near radius.
struct LjSource {
    unsigned nx, ny, nz, ox, oy, oz;
    float c12, nc6;
    int type;
};
__device__ __forceinline__ uint64_t far_du2(uint4 p, uint4 q, const LjSource &s, uint64_t S2)
{
    const uint64_t XN = f2_pack((float)(int)(p.x - s.nx), (float)(int)(q.x - s.nx));
    const uint64_t YN = f2_pack((float)(int)(p.y - s.ny), (float)(int)(q.y - s.ny));
    const uint64_t ZN = f2_pack((float)(int)(p.z - s.nz), (float)(int)(q.z - s.nz));
    const uint64_t XO = f2_pack((float)(int)(p.x - s.ox), (float)(int)(q.x - s.ox));
    const uint64_t YO = f2_pack((float)(int)(p.y - s.oy), (float)(int)(q.y - s.oy));
    const uint64_t ZO = f2_pack((float)(int)(p.z - s.oz), (float)(int)(q.z - s.oz));
    const uint64_t RN = f2_mul(f2_fma(XN, XN, f2_fma(YN, YN, f2_mul(ZN, ZN))), S2);
    const uint64_t RO = f2_mul(f2_fma(XO, XO, f2_fma(YO, YO, f2_mul(ZO, ZO))), S2);
    float p0, p1;
    f2_unpack(f2_mul(RN, RO), p0, p1);
    const uint64_t I = f2_pack(rcp_approx(p0), rcp_approx(p1));      // 1/r'^2 = r^2 / (r^2 r'^2)
    const uint64_t IN = f2_mul(I, RO), IO = f2_mul(I, RN);
    const uint64_t S6N = f2_mul(f2_mul(IN, IN), IN), S6O = f2_mul(f2_mul(IO, IO), IO);
    const uint64_t C12 = f2_pack(s.c12, s.c12), NC6 = f2_pack(s.nc6, s.nc6), MC12 = f2_pack(-s.c12, -s.c12),
                   C6 = f2_pack(-s.nc6, -s.nc6);
    return f2_fma(f2_fma(C12, S6N, NC6), S6N, f2_mul(f2_fma(MC12, S6O, C6), S6O));
}

// Moved atom a of move k (the coefficients are set per partner type).
__device__ __forceinline__ LjSource lj_source(const McBatch &b, int k, int a, const BoxDev &bx)
{
    LjSource s;
    s.type = b.oldp[k][a].w;
    if (a < 3) {
        s.nx = b.scn[k][a][0]; s.ny = b.scn[k][a][1]; s.nz = b.scn[k][a][2];
        s.ox = b.sco[k][a][0]; s.oy = b.sco[k][a][1]; s.oz = b.sco[k][a][2];
    } else {
        const int4 n = b.newp[k][a], o = b.oldp[k][a];
        s.nx = scale32_near(n.x, bx.sc_rcp); s.ny = scale32_near(n.y, bx.sc_rcp); s.nz = scale32_near(n.z, bx.sc_rcp);
        s.ox = scale32_near(o.x, bx.sc_rcp); s.oy = scale32_near(o.y, bx.sc_rcp); s.oz = scale32_near(o.z, bx.sc_rcp);
    }
    s.c12 = s.nc6 = 0.f;
    return s;
}

// Lennard-Jones terms of one moved atom each of two moves (s0, s1) with the groups of 32 slots
// lo .. up - 1 that are in their masks m0, m1 (sx: the 2^32-periodic copy from group 0 on; a group
// past `up` may be loaded, and is in neither mask). A lane takes one partner each of two groups per step,
// and both moves share their loads: four independent packed chains.
__device__ __forceinline__ void far_groups(float &acc0, float &acc1, const LjSource &s0, const LjSource &s1, unsigned m0,
                                           unsigned m1, int lo, int up, const uint4 *sx, uint64_t S2, int lane)
{
    const uint4 *pp = sx + lo * 32 + lane;
    m0 >>= lo;
    m1 >>= lo;
    for (int n = up - lo; n > 0; n -= 2, pp += 64, m0 >>= 2, m1 >>= 2) {
        if (!((m0 | m1) & 3u)) continue;
        const uint4 p = pp[0], q = pp[32];
        float a0, a1, b0, b1;
        f2_unpack(far_du2(p, q, s0, S2), a0, a1);
        f2_unpack(far_du2(p, q, s1, S2), b0, b1);
        const bool vp = p.w != (unsigned)kNoAtom, vq = q.w != (unsigned)kNoAtom;
        if (vp && (m0 & 1u)) acc0 += a0;
        if (vq && (m0 & 2u)) acc0 += a1;
        if (vp && (m1 & 1u)) acc1 += b0;
        if (vq && (m1 & 2u)) acc1 += b1;
    }
}

// u(r') - u(r) for one partner as pair_du takes it, without branches, so that the atoms of a
// molecule run side by side: every term is formed and selected. Sets `rare` where a squared
// distance lies within its FP32 error of a cutoff, of the table's end or of a bin edge, or the new
// distance is zero; the caller then takes pair_du.
template <bool CUT>
__device__ __forceinline__ float near_pair(Sep sn, Sep so, const PairRow &pr, const BoxDev &bx, const float *ep, bool &rare)
{
    const DuCore c = du_core(sn, so, bx.inv_s2);
    float du = 0.f;
    rare |= c.g2n == 0.f;
    if (pr.c12 != 0.f || pr.c6 != 0.f) {                         // one row for the whole warp
        const float lj = lj_du(c, pr.c12, pr.c6);
        if (!CUT || !bx.lj_cut) {
            du = lj;
        } else {
            const bool ln = c.g2n < bx.lj2_lo, lo = c.g2o < bx.lj2_lo;
            rare |= (!ln && c.g2n <= bx.lj2_hi) || (!lo && c.g2o <= bx.lj2_hi);
            const float a2 = ln ? c.an * c.an : c.ao * c.ao;
            const float s6 = a2 * a2 * a2;
            const float u = fmaf(pr.c12, s6, -pr.c6) * s6;
            du = ln && lo ? lj : ln ? u : lo ? -u : 0.f;
        }
    }
    if (pr.kqq != 0.f) {
        const bool cn = c.g2n < bx.rc2_lo, co = c.g2o < bx.rc2_lo;
        rare |= (!cn && c.g2n <= bx.rc2_hi) || (!co && c.g2o <= bx.rc2_hi);
        const float p = c.an * c.ao;
        const float both = c.dr2 * __fdividef(p * p, c.an + c.ao);       // 2 ulp; an + ao ~ 0.1..10
        du = fmaf(pr.kqq, cn && co ? both : cn ? c.an : co ? -c.ao : 0.f, du);
    }
    if (bx.has_ep) {
        const float *row = ep + pr.pair * bx.n_bins;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float g2 = h ? c.g2o : c.g2n;
            float r;
            asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(g2));
            const float u = fmaf(r, bx.inv_dr_fx, -0.5f);
            const float t = u + 12582912.f;                      // u rounded to an integer in the low bits
            const float d = u - (t - 12582912.f);
            const bool in = g2 < bx.tmax_lo;
            rare |= (!in && g2 <= bx.tmax_hi) || (in && !(fabsf(d) < fmaf(u, -0x1p-20f, 0.5f - 0x1p-20f)));
            const float e = row[in ? min(max(__float_as_int(t) - 0x4B400000, 0), bx.n_bins - 1) : 0];
            du += in ? (h ? -e : e) : 0.f;
        }
    }
    return du;
}

// Near item: the change of one move's energy with one partner of every lane (grid point pj, of a
// type t; valid: a partner, not an atom of the move), over the moved atoms in `todo`.
template <int M, bool CUT>
__device__ __forceinline__ float near_du(const int4 *np, const int4 *op, int m, unsigned todo, int4 pj, int t, bool valid,
                                         const BoxDev &bx, const long long *T, const float *ep)
{
    float acc = 0.f;
    const int L = bx.L;
    bool rare = M == 0;
    if (M > 0) {
#pragma unroll
        for (int a = 0; a < M; ++a) {
            if (!((todo >> a) & 1u)) continue;
            const int4 n = np[a], o = op[a];
            acc += near_pair<CUT>(sep(n, pj, L), sep(o, pj, L), bx.row[n.w * kMaxTypes + t], bx, ep, rare);
        }
    }
    if (rare && valid) {
        acc = 0.f;
        for (int a = 0; a < m; ++a)
            if ((todo >> a) & 1u) {
                const int4 n = np[a], o = op[a];
                acc += pair_du_cold<CUT>(sep(n, pj, L), sep(o, pj, L), bx.row[n.w * kMaxTypes + t], bx, T, ep);
            }
    }
    return valid ? acc : 0.f;
}

// Signed minimum image of a difference of two coordinates, in (-L/2, L/2] (hl = floor(L / 2)).
__device__ __forceinline__ int mi_signed32(int d, int L, int hl)
{
    if (d > hl) return d - L;
    if (d <= hl - L) return d + L;
    return d;
}

// x + e wrapped to [0, L), for x in [0, L).
__device__ __forceinline__ int wrap_near(int x, int e, int L)
{
    if (e >= L || e <= -L) return wrap_coord((long long)x + e, L);
    const int t = (int)((unsigned)x + (unsigned)e);  // negative, or past 2^31 - 1 as unsigned
    if (e < 0) return t < 0 ? t + L : t;
    return (unsigned)t >= (unsigned)L ? (int)((unsigned)t - (unsigned)L) : t;
}

// Trial coordinates and what follows from them alone, for the moves of batch b (from move record
// tn on): thread t takes atom t mod 2^lanes_log of move t >> lanes_log, all three axes; 2^lanes_log
// (4 or 8) holds the box's largest molecule, so that half the warps do this where they can. oldp
// holds the current coordinates.
template <bool CUT>
__device__ __noinline__ void trial_moves(McBatch &b, const MoveRec *ring, long long tn, int nb, const BoxDev &bx)
{
    const int L = bx.L, nt = bx.n_types, lg = bx.lanes_log;
    const int k = threadIdx.x >> lg;
    const int kk = threadIdx.x & ((1 << lg) - 1);
    const bool act = k < nb;
    const MoveRec &mr = ring[(tn + (act ? k : 0)) & (kMoveRing - 1)];
    const int a0 = mr.a0, m = act ? mr.m : 0;
    int4 np4 = make_int4(0, 0, 0, 0), op4 = make_int4(0, 0, 0, 0);
    if (kk < m) {
        const int4 *op = b.oldp[k];
        op4 = op[kk];
        int nx, ny, nz;
        if (mr.kind == 1) {
            // minimum-image offsets from atom 0, summed over the molecule, and this atom's own (sums in 64
            // bits: below 2^25 where a box is made, but atoms without springs may drift apart)
            const int4 b0 = op[0];
            const int hl = L >> 1;
            long long sx = 0, sy = 0, sz = 0;
            int ox = 0, oy = 0, oz = 0;
            for (int i = 0; i < m; ++i) {
                const int4 c = op[i];
                const int dx = mi_signed32(c.x - b0.x, L, hl), dy = mi_signed32(c.y - b0.y, L, hl),
                          dz = mi_signed32(c.z - b0.z, L, hl);
                sx += dx; sy += dy; sz += dz;
                if (i == kk) { ox = dx; oy = dy; oz = dz; }
            }
            const long long ux = (long long)m * ox - sx, uy = (long long)m * oy - sy, uz = (long long)m * oz - sz;
            const int *R = mr.R;
            // per axis: s 2^30 + R (m o - s), then floor((. + m 2^29) / 2^30) (32 bits) and
            // floor division by m
            const long long numx = sx * 1073741824LL + R[0] * ux + R[1] * uy + R[2] * uz;
            const long long numy = sy * 1073741824LL + R[3] * ux + R[4] * uy + R[5] * uz;
            const long long numz = sz * 1073741824LL + R[6] * ux + R[7] * uy + R[8] * uz;
            const long long half = (long long)m * 536870912LL;
            nx = wrap_near(b0.x, floordiv32((int)((numx + half) >> 30), m) + mr.shift[0], L);
            ny = wrap_near(b0.y, floordiv32((int)((numy + half) >> 30), m) + mr.shift[1], L);
            nz = wrap_near(b0.z, floordiv32((int)((numz + half) >> 30), m) + mr.shift[2], L);
        } else {
            const bool moved = mr.kind != 2 || kk == mr.atom;
            nx = wrap_near(op4.x, moved ? mr.shift[0] : 0, L);
            ny = wrap_near(op4.y, moved ? mr.shift[1] : 0, L);
            nz = wrap_near(op4.z, moved ? mr.shift[2] : 0, L);
        }
        np4 = make_int4(nx, ny, nz, op4.w);
        b.newp[k][kk] = np4;
        if (kk < 3) {
            b.scn[k][kk][0] = scale32_near(nx, bx.sc_rcp);
            b.scn[k][kk][1] = scale32_near(ny, bx.sc_rcp);
            b.scn[k][kk][2] = scale32_near(nz, bx.sc_rcp);
            b.sco[k][kk][0] = scale32_near(op4.x, bx.sc_rcp);
            b.sco[k][kk][1] = scale32_near(op4.y, bx.sc_rcp);
            b.sco[k][kk][2] = scale32_near(op4.z, bx.sc_rcp);
        }
    }
    __syncwarp();
    if (act && kk == 0) {
        // flexible molecules: change of the intra-molecular springs, written without
        // cancellation: k[(r' - d)^2 - (r - d)^2] = k (r' - r)(r' + r - 2d), with
        // r' - r = (r'^2 - r^2) / (r' + r) from the exact integer squared distances
        float di = 0.f;
        if (bx.move_kind == EPSR_MOVE_FLEXIBLE_MOLECULE)
            for (int i = 0; i < m; ++i)
                for (int j = i + 1; j < m; ++j) {
                    const int4 ni = b.newp[k][i], nj = b.newp[k][j];
                    const int t = ni.w * kMaxTypes + nj.w;
                    if (bx.bond_k[t] == 0.0) continue;
                    const long long d2n = dist2(ni, nj, L), d2o = dist2(b.oldp[k][i], b.oldp[k][j], L);
                    if (d2n == d2o) continue;
                    const float rn = sqrtf((float)d2n * bx.inv_s2), ro = sqrtf((float)d2o * bx.inv_s2);
                    const float dr = (float)(d2n - d2o) * bx.inv_s2 / (rn + ro);
                    di = fmaf((float)bx.bond_k[t] * dr, rn + ro - 2.f * (float)bx.bond_d[t], di);
                }
        b.intra[k] = di;
        atomicMax(&b.mm, m);
        b.natoms[k] = m;
        b.lj_atoms[k] = 0;
        b.a0[k] = a0;
        b.thr[k] = mr.thr;
        b.u_acc[k] = mr.u_acc;
    }
    // near sphere: every old and new atom position lies within `reach` of old atom 0 (a bound in
    // FP32, rounded up by the margin), so a partner beyond near_fx + reach of it has no near term
    float reach2 = 0.f;
    if (kk < m) {
        const int4 o = b.oldp[k][0];
        reach2 = fmaxf(g2_of(sep(op4, o, L)), g2_of(sep(np4, o, L)));
    }
    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) reach2 = fmaxf(reach2, __shfl_xor_sync(0xffffffffu, reach2, o));
    if (act && kk == 0) {
        const float r = (((float)bx.near_fx + sqrtf(reach2)) * 1.0001f + 2.f) * bx.sc_k + 8.f;
        b.hw2[k] = r * r;
    }
    __syncwarp();                        // lj_atoms is cleared
    // rows of the moved atoms with each partner type (an atom that stays where it is has none)
    for (int t = kk; act && t < nt; t += 1 << lg) {
        unsigned lj = 0u, nr = 0u;
        for (int a = 0; a < m; ++a) {
            const int4 n = b.newp[k][a], o = b.oldp[k][a];
            if (n.x == o.x && n.y == o.y && n.z == o.z) continue;
            const PairRow &pr = bx.row[n.w * kMaxTypes + t];
            if (lj_full_row<CUT>(pr, bx)) lj |= 1u << a;
            else if (near_row<CUT>(pr, bx)) nr |= 1u << a;
        }
        b.rows[k][t] = (unsigned short)(lj | (nr << 8));
        if (lj) atomicOr(&b.lj_atoms[k], (int)lj);
    }
    __syncwarp();
}

// Half width (2^32-periodic grid, rounded up) that reaches a point at wrapped difference d.
__device__ __forceinline__ int grow_half(unsigned d)
{
    return (int)min((unsigned)abs((int)d) + 8u, 0x7fffffffu);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// GSLICE: the partner slices live in global memory ([grid][slice_cap], read through L1/L2)
// because they do not fit in shared memory; the EP table and the chunk boxes stay in shared
// memory either way, and so do the thresholds where there is room (pairs within the FP32 error of a
// bin edge read them, about one in 10^3: from global memory silica with an empirical potential took
// 1480 instead of 1452 us).
template <bool GSLICE, bool CUT>
__global__ void __launch_bounds__(kMcThreads, 1) mc_sweep_kernel(McArgs A)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ McShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x;
    const int box = A.cta_box[cta];

    if (tid == 0) {
        sh.bx = A.boxes[box];
        sh.b[0].nb = sh.b[1].nb = 0;
        sh.b[0].mm = sh.b[1].mm = 0;
        sh.nb_min = 1 << 30;
        sh.cut = 1 << 30;
        sh.n_queue = 0;
        sh.abort_flag = 0;
        sh.st_att = sh.st_acc = sh.st_nonfinite = 0;
        sh.st_sum = 0.0;
    }
    __syncthreads();
    const BoxDev &bx = sh.bx;

    const int G = bx.n_cta;
    const int rank = cta - bx.cta0;
    const int L = bx.L;
    const int nt = bx.n_types;
    // Partners of this CTA: every type's Hilbert order is cut into chunks of 2^cs atoms (compact
    // regions), dealt out in turn: chunk c of a type that follows f chunks of earlier types goes to
    // CTA (f + c) mod G of the group. A move's near chunks so fall on as many CTAs as there are
    // chunks, instead of all on the one that owns the region (the barrier waits for the busiest).
    const int cs = A.chunk_log;
    if (tid == 0) {
        int c = 0;
        long long f = 0;
        for (int t = 0; t < nt; ++t) {
            const int nch = (int)((bx.count[t] + (1 << cs) - 1) >> cs);            // chunks of the type
            const int first = (int)(((long long)rank - f % G + G) % G);           // this CTA's first chunk
            sh.first[t] = first;
            sh.cbase[t] = c;
            c += first < nch ? (nch - first + G - 1) / G : 0;
            f += nch;
        }
        sh.cbase[nt] = c;
    }
    __syncthreads();
    const int n_chunks = sh.cbase[nt], n_words = (n_chunks + 31) >> 5;

    // shared memory: partner slice {x, y, z, type | atom << 3} and its 2^32-periodic copy {X, Y, Z,
    // atom} (or, with the slice in global memory, a staged part of the copy), thresholds, empirical
    // potential, correction tables, chunk boxes (centre and half width per axis, one column per mask
    // bit) and near masks
    int4 *slice = GSLICE ? A.slice_g + (size_t)cta * A.slice_cap : reinterpret_cast<int4 *>(dyn);
    uint4 *sx = GSLICE ? reinterpret_cast<uint4 *>(dyn) : reinterpret_cast<uint4 *>(slice + A.slice_cap);
    long long *s_T = reinterpret_cast<long long *>(sx + (GSLICE ? A.stage : A.slice_cap));
    const long long *T = A.tbl_cap ? s_T : A.thresholds + bx.tbl_off;
    float *ep = reinterpret_cast<float *>(s_T + A.tbl_cap);
    float (*corr)[kBatchMax] = reinterpret_cast<float (*)[kBatchMax]>(ep + A.ep_cap);
    float *corr_part = &corr[kBatchMax][0];                                              // [kCorrItems]
    int *queue = reinterpret_cast<int *>(&corr[0][0]);                                  // [kQueue], during phase C
    float *q_res = reinterpret_cast<float *>(queue + kQueue);                           // [kQueue]
    const int cols = A.words_cap * 32;
    int *cb = reinterpret_cast<int *>(corr_part + kCorrItems);                         // [6][cols]
    unsigned *near = reinterpret_cast<unsigned *>(cb + 6 * cols);                      // [kBatchMax][words_cap]
    unsigned *far = near + kBatchMax * A.words_cap;                                    // [kBatchMax][words_cap]
    unsigned char *ct = reinterpret_cast<unsigned char *>(far + kBatchMax * A.words_cap);   // [cols] type of each chunk
    for (int c = tid; c < cols; c += kMcThreads) {
        int t = 0;
        while (t + 1 < nt && c >= sh.cbase[t + 1]) ++t;
        ct[c] = (unsigned char)t;
    }
    __syncthreads();
    for (int i = tid; i < n_chunks << cs; i += kMcThreads) {
        const int t = ct[i >> cs];
        const long long pos = ((long long)(sh.first[t] + ((i >> cs) - sh.cbase[t]) * G) << cs) + (i & ((1 << cs) - 1));
        if (pos >= bx.count[t]) {                        // the end of a type's last chunk
            slice[i] = make_int4(0, 0, 0, kNoAtom);
            if (!GSLICE) sx[i] = make_uint4(0u, 0u, 0u, (unsigned)kNoAtom);
            continue;
        }
        const int atom = A.sorted_index[bx.atom0 + bx.type_start[t] + pos] - (int)bx.atom0;
        int4 c = A.coords[bx.atom0 + atom];
        c.w = c.w | (atom << 3);
        slice[i] = c;
        if (!GSLICE)
            sx[i] = make_uint4(scale32_near(c.x, bx.sc_rcp), scale32_near(c.y, bx.sc_rcp), scale32_near(c.z, bx.sc_rcp),
                               (unsigned)atom);
    }
    if (A.tbl_cap)
        for (int k = tid; k <= bx.n_bins; k += kMcThreads) s_T[k] = A.thresholds[bx.tbl_off + k];
    if (bx.has_ep)
        for (int k = tid; k < bx.n_pairs * bx.n_bins; k += kMcThreads) ep[k] = A.ep[bx.ep_off + k];
    __syncthreads();
    // boxes of the chunks (coordinates in [0, L); a chunk of Hilbert neighbours seldom meets the
    // seam, and its box is then merely wide)
    for (int c = warp; c < n_chunks; c += kMcWarps) {
        int lo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, hi[3] = {-1, -1, -1};
        for (int i = (c << cs) + lane; i < (c + 1) << cs; i += 32) {
            const int4 p = slice[i];
            if (p.w == kNoAtom) continue;
            lo[0] = min(lo[0], p.x); hi[0] = max(hi[0], p.x);
            lo[1] = min(lo[1], p.y); hi[1] = max(hi[1], p.y);
            lo[2] = min(lo[2], p.z); hi[2] = max(hi[2], p.z);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int l = __reduce_min_sync(0xffffffffu, lo[a]), u = __reduce_max_sync(0xffffffffu, hi[a]);
            if (lane == 0) {
                // centre and half width on the 2^32-periodic grid, rounded up
                const int ce = l + ((u - l) >> 1);
                const unsigned h = scale32_near(u - ce, bx.sc_rcp);
                cb[a * cols + c] = (int)scale32_near(ce, bx.sc_rcp);
                cb[(3 + a) * cols + c] = (int)min(h + 8u, 0x7fffffffu);
            }
        }
    }
    __syncthreads();

    // moves per batch: as set, else the most (the per-batch phases amortise over more moves: 0.27
    // against 0.41 us a move with 32, 99,999-atom water); above 32 only with 8 or more CTAs per box,
    // so that a CTA's share of the batch-pair corrections fits its item buffer
    const int batch_k = min(A.batch_k > 0 ? A.batch_k : kBatchMax, G >= 8 ? kBatchMax : 32);
    const int4 *moves = reinterpret_cast<const int4 *>(A.moves + (size_t)box * A.chunk);
    constexpr int kRecI4 = (int)(sizeof(MoveRec) / sizeof(int4));
    // copies the records of moves [m0, m1) into the ring (asynchronously, 16 bytes a thread)
    auto copy_records = [&](long long m0, long long m1) {
        const unsigned r0 = (unsigned)m0 & (kMoveRing - 1);
        for (unsigned i = tid; i < (unsigned)(m1 - m0) * kRecI4; i += kMcThreads) {
            const unsigned t = i / kRecI4, w = i - t * kRecI4;
            cp_async16(reinterpret_cast<int4 *>(&sh.ring[(r0 + t) & (kMoveRing - 1)]) + w, moves + m0 * kRecI4 + i);
        }
    };
    long long held = min(A.n_moves, (long long)kMoveRing);      // records copied so far
    copy_records(0, held);
    cp_async_wait();
    __syncthreads();

    unsigned seq = 0;
    int par = 0, nb = 0;             // the current batch: b[par], moves [t0, t0 + nb)
    int n_du = 0;                    // entries of acc_du (rank 0)
    const int gk = tid >> 3, gsub = tid & 7;   // gather group: move gk, member gsub
    const bool prep_warp = (warp * 32 >> bx.lanes_log) < kBatchMax;      // has moves in trial_moves
    int n_local = 0, mm = 0;         // this CTA's share of the current batch's corrections
    bool fine = false;
    long long t0 = 0;
    // Looks up the moves from tn on, the current batch being b[par] (nb moves before tn): thread gsub
    // of move gk takes atom gsub. Current coordinates come from the current batch's old ones (as if it
    // were not accepted) or the previous batch's accepted move, b[par ^ 1] (its global update may not be
    // visible yet), else from the global array, which holds every earlier one. The batch ends before
    // its first repeated molecule.
    int4 gc = make_int4(0, 0, 0, 0);
    int gp = 0, mol = -1, last = -1;     // last: index in the current batch of the molecule, or -1
    bool mine = false;
    auto look_up = [&](long long tn) {
        const McBatch &cur = sh.b[par], &nxt = sh.b[par ^ 1];
        mine = gk < (int)min((long long)batch_k, A.n_moves - tn);
        last = -1;
        if (!mine) return;
        const MoveRec &mr = sh.ring[(tn + gk) & (kMoveRing - 1)];
        mol = mr.mol;
        mine = gsub < mr.m;
        if (gsub == 0 && mr.prev <= gk) atomicMin(&sh.nb_min, gk);
        last = nb + gk - mr.prev;
        const int before = last + nxt.nb;                           // index in the previous batch
        if (mine) {
            gp = A.pos_of[bx.atom0 + mr.a0 + gsub];
            if (last >= 0 && last < nb) gc = cur.oldp[last][gsub];
            else if (last < 0 && before >= 0) gc = nxt.acc[before] ? nxt.newp[before][gsub] : nxt.oldp[before][gsub];
            else gc = __ldcg(&A.coords[bx.atom0 + mr.a0 + gsub]);
        }
        if (last >= nb) last = -1;
    };
    look_up(0);
    __syncthreads();
    for (;;) {
        McBatch &cur = sh.b[par], &nxt = sh.b[par ^ 1];
        long long tn = t0 + nb;
        int nb_next = 0;
        bool redo = false;                // the next batch is prepared again
        // ---- A, B. the next batch, while the partials of the current one reach the other CTAs --------
        // Its current and trial coordinates (integer arithmetic). The decisions of the current batch are
        // not known yet: the few molecules that they move are taken up again after them. (A single CTA
        // waits for nobody, and takes them once, after the decisions: 300 moves of 3 atoms 1275 -> 1105 us,
        // of 60 atoms 343 -> 303, of one water molecule 2990 -> 2445.)
        if (tn < A.n_moves) {
            nb_next = min((int)min((long long)batch_k, A.n_moves - tn), sh.nb_min);
            if (tid == 0) nxt.nb = nb_next;
            copy_records(held, min(A.n_moves, tn + kMoveRing));
            held = min(A.n_moves, tn + kMoveRing);
            if (mine && gk < nb_next) {
                nxt.oldp[gk][gsub] = gc;
                nxt.spos[gk][gsub] = gp - (int)bx.atom0;
                if (gsub == 0) nxt.mol[gk] = mol;
            }
            if (G > 1) {
                __syncthreads();
                if (prep_warp) trial_moves<CUT>(nxt, sh.ring, tn, nb_next, bx);
            }
        }
        bool again = false;
        if (nb > 0) {
            // ---- D. gather the partials of the box's CTA group (one bounded grid barrier) -------
            // Lane 0 of warp 0 polls the group's counter with acquire loads; the CTA barrier after it
            // orders every thread's reads after the acquire.
            const bool gin = gk < nb;
            float cv[8];                          // corrections (j, gk), j = gsub + 8 i < gk
            float gv = 0.f, ge = 0.f, gw = 0.f;   // sum of the partials, its rounding error, magnitude of the corrections
#pragma unroll
            for (int i = 0; i < 8; ++i) cv[i] = 0.f;
            if (G > 1) {
                const float *ps = A.slots + (size_t)(seq & 1u) * A.grid * kMcSlotStride;
                const float *pc = ps + (size_t)kBatchMax * A.grid + (size_t)bx.cta0 * kMcCorrPerCta;
                if (tid == 0) {
                    const unsigned target = seq * (unsigned)G;
                    const uint64_t t_start = globaltimer_ns();
                    long long it = 0;
                    bool timed_out = false;
                    while (ld_acquire_gpu(&A.flags[box]) < target) {
                        if ((++it & 255) == 0 &&
                            ((globaltimer_ns() - t_start > A.timeout_ns) || it > A.max_spin ||
                             ld_relaxed_gpu(A.status) != 0)) {
                            timed_out = true;
                            break;
                        }
                    }
                    if (timed_out) {
                        atomicOr(A.status, kStatusTimeout);
                        sh.abort_flag = 1;
                    }
                }
                __syncthreads();
                if (sh.abort_flag) {
                    cp_async_wait();
                    return;
                }
                // 8 threads per move k: every 8th CTA's partial and every 8th correction (j, k),
                // j < k, all loads in flight at once (one L2 round trip)
                if (gin) {
                    const float *pk = ps + (size_t)gk * A.grid + bx.cta0;
                    const float *ck = pc + gk * (gk - 1) / 2;
                    float4 pv[kGatherLoads];             // four CTAs' partials each, where the rows are aligned
                    if (((A.grid | bx.cta0) & 3) == 0) {
#pragma unroll
                        for (int i = 0; i < kGatherLoads; ++i) {
                            const int r = 4 * (gsub + 8 * i);
                            pv[i] = r < G ? __ldcg(reinterpret_cast<const float4 *>(pk + r)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            if (r + 1 >= G) pv[i].y = 0.f;
                            if (r + 2 >= G) pv[i].z = 0.f;
                            if (r + 3 >= G) pv[i].w = 0.f;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < kGatherLoads; ++i) {
                            const int r = gsub + 8 * i;
                            pv[i].x = r < G ? __ldcg(&pk[r]) : 0.f;
                            pv[i].y = r + 8 * kGatherLoads < G ? __ldcg(&pk[r + 8 * kGatherLoads]) : 0.f;
                            pv[i].z = r + 16 * kGatherLoads < G ? __ldcg(&pk[r + 16 * kGatherLoads]) : 0.f;
                            pv[i].w = r + 24 * kGatherLoads < G ? __ldcg(&pk[r + 24 * kGatherLoads]) : 0.f;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int j = gsub + 8 * i;
                        cv[i] = j < gk ? __ldcg(&ck[j]) : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < kGatherLoads; ++i) {
                        two_sum(gv, ge, pv[i].x);
                        two_sum(gv, ge, pv[i].y);
                        two_sum(gv, ge, pv[i].z);
                        two_sum(gv, ge, pv[i].w);
                    }
                    for (int r = gsub + 32 * kGatherLoads; r < G; r += 8) two_sum(gv, ge, __ldcg(&pk[r]));
                }
            } else if (gin) {
                gv = gsub == 0 ? sh.part[gk] : 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int j = gsub + 8 * i;
                    cv[i] = j < gk ? corr_sum(corr_part, gk * (gk - 1) / 2 + j, mm, fine) : 0.f;
                }
            }
            // the group's sums in a fixed shuffle tree (the same order in every run): the move's
            // partial dU and the magnitude sum of its corrections. Plain FP32 sums of 152 partials put the
            // error of dU 7 % above that of sums of 20 (2-norm, 9,999-atom water with an empirical potential:
            // 1.05e-7 of dU; with the rounding errors added up 0.84e-7)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = gsub + 8 * i;
                if (gin && j < gk) corr[j][gk] = cv[i];
                gw += fabsf(cv[i]);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const float v = __shfl_xor_sync(0xffffffffu, gv, o);
                ge += __shfl_xor_sync(0xffffffffu, ge, o);
                two_sum(gv, ge, v);
                gw += __shfl_xor_sync(0xffffffffu, gw, o);
            }
            // (an infinite sum has no error: a pair of coincident atoms)
            if (isfinite(gv)) gv += ge;
            // ---- F. Metropolis decisions of the batch, in order: move k's dU includes the
            // corrections of every earlier accepted move. Fast path: when no move's decision can
            // change with any subset of its earlier corrections (|dU - threshold| beyond the sum of
            // their magnitudes plus the FP32 rounding of that many additions), every group decides
            // its move at once and then adds its accepted corrections (fixed tree order); otherwise
            // warp 0 decides one move after the other (lane l holds moves l and l + 32) and adds
            // the corrections in the chain's order. Both give the same decisions.
            {
                const float d = gin ? gv + cur.intra[gk] : 0.f;
                const float thr = gin ? cur.thr[gk] : 0.f;
                const float wv = gw + (fabsf(d) + gw) * 0x1p-16f;
                const bool sure = !gin || metropolis(d + wv, thr) || !metropolis(d - wv, thr);
                if (gin && gsub == 0) {
                    sh.base[gk] = gv;
                    sh.part[gk] = gw;              // (its partial has been read)
                }
                if (__syncthreads_and(sure)) {
                    const bool acc = gin && metropolis(d, thr);
                    if (gin && gsub == 0) cur.acc[gk] = acc;
                    __syncthreads();
                    float c = 0.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int j = gsub + 8 * i;
                        if (j < gk && cur.acc[j]) c += cv[i];
                    }
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                    if (gin && gsub == 0) sh.dU[gk] = d + c;
                    if (__any_sync(0xffffffffu, !(gw <= kCancelled))) {
                        float w = 0.f;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int j = gsub + 8 * i;
                            if (j < gk && cur.acc[j]) w += fabsf(cv[i]);
                        }
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
                        if (gin && gsub == 0 && cancelled(d, w, d + c)) atomicMin(&sh.cut, gk);
                    }
                } else if (warp == 0) {
                    const bool in0 = lane < nb, in1 = lane + 32 < nb;
                    float d0 = in0 ? sh.base[lane] + cur.intra[lane] : 0.f;
                    float d1 = in1 ? sh.base[lane + 32] + cur.intra[lane + 32] : 0.f;
                    const float thr0 = in0 ? cur.thr[lane] : 0.f, thr1 = in1 ? cur.thr[lane + 32] : 0.f;
                    const float b0 = d0, b1 = d1;
                    int acc0 = 0, acc1 = 0;
#pragma unroll 8
                    for (int j = 0; j < 32; ++j) {
                        if (j < nb) {
                            const float c0 = corr[j][lane], c1 = corr[j][lane + 32];
                            const int aj = __shfl_sync(0xffffffffu, metropolis(d0, thr0), j);
                            if (lane == j) acc0 = aj;
                            if (aj) {
                                if (lane > j) d0 += c0;
                                d1 += c1;
                            }
                        }
                    }
#pragma unroll 8
                    for (int j = 32; j < kBatchMax; ++j) {
                        if (j < nb) {
                            const float c1 = corr[j][lane + 32];
                            const int aj = __shfl_sync(0xffffffffu, metropolis(d1, thr1), j - 32);
                            if (lane == j - 32) acc1 = aj;
                            if (aj && lane + 32 > j) d1 += c1;
                        }
                    }
                    if (in0) {
                        sh.dU[lane] = d0;
                        cur.acc[lane] = acc0;
                    }
                    if (in1) {
                        sh.dU[lane + 32] = d1;
                        cur.acc[lane + 32] = acc1;
                    }
                    if (__any_sync(0xffffffffu, (in0 && !(sh.part[lane] <= kCancelled)) || (in1 && !(sh.part[lane + 32] <= kCancelled)))) {
                        float w0 = 0.f, w1 = 0.f;
                        for (int j = 0; j < nb; ++j) {
                            const int aj = __shfl_sync(0xffffffffu, j < 32 ? acc0 : acc1, j & 31);
                            if (aj && lane > j) w0 += fabsf(corr[j][lane]);
                            if (aj && lane + 32 > j) w1 += fabsf(corr[j][lane + 32]);
                        }
                        if (in0 && cancelled(b0, w0, d0)) atomicMin(&sh.cut, lane);
                        if (in1 && cancelled(b1, w1, d1)) atomicMin(&sh.cut, lane + 32);
                    }
                }
            }
            __syncthreads();
            if (sh.cut < nb) {                   // (the same in every CTA of the group; move 0 has no corrections)
                nb = sh.cut;
                tn = t0 + nb;
                redo = true;
                if (tid == 0) cur.nb = nb;
            }
            if (rank == 0 && warp == 0) {
                // counts now; the FP64 sum of accepted dU over a few batches at once
                const bool in0 = lane < nb, in1 = lane + 32 < nb;
                const bool acc0 = in0 && cur.acc[lane], acc1 = in1 && cur.acc[lane + 32];
                const float d0 = in0 ? sh.dU[lane] : 0.f, d1 = in1 ? sh.dU[lane + 32] : 0.f;
                const unsigned b_acc = __ballot_sync(0xffffffffu, acc0), b_acc1 = __ballot_sync(0xffffffffu, acc1);
                const unsigned b_nf = __ballot_sync(0xffffffffu, in0 && !isfinite(d0)),
                               b_nf1 = __ballot_sync(0xffffffffu, in1 && !isfinite(d1));
                if (in0) sh.acc_du[n_du + lane] = acc0 ? d0 : 0.f;
                if (in1) sh.acc_du[n_du + lane + 32] = acc1 ? d1 : 0.f;
                if (lane == 0) {
                    sh.st_att += nb;
                    sh.st_acc += __popc(b_acc) + __popc(b_acc1);
                    sh.st_nonfinite += __popc(b_nf) + __popc(b_nf1);
                }
                __syncwarp();
                if (n_du + nb > kBatchMax) block_sum_du(sh.acc_du, n_du + nb, lane, sh.st_sum);
            }
            n_du = n_du + nb > kBatchMax ? 0 : n_du + nb;
            // ---- G. apply accepted moves: shared slice, global coordinates, log ------------------
            for (int it = tid; it < nb * kMaxMolAtoms; it += kMcThreads) {
                const int k = it / kMaxMolAtoms, a = it % kMaxMolAtoms;
                if (!cur.acc[k] || a >= cur.natoms[k]) continue;
                const int ja = cur.a0[k] + a;
                const int4 p = cur.newp[k][a];
                const int t = p.w, sp = cur.spos[k][a] - bx.type_start[t], ch = (sp >> cs) - sh.first[t];
                if (ch >= 0 && ch % G == 0) {
                    const int col = sh.cbase[t] + ch / G, slot = (col << cs) + (sp & ((1 << cs) - 1));
                    slice[slot] = make_int4(p.x, p.y, p.z, t | (ja << 3));
                    // the chunk's box grows to hold the new position
                    const unsigned X = scale32_near(p.x, bx.sc_rcp), Y = scale32_near(p.y, bx.sc_rcp),
                                   Z = scale32_near(p.z, bx.sc_rcp);
                    atomicMax(&cb[3 * cols + col], grow_half(X - (unsigned)cb[col]));
                    atomicMax(&cb[4 * cols + col], grow_half(Y - (unsigned)cb[cols + col]));
                    atomicMax(&cb[5 * cols + col], grow_half(Z - (unsigned)cb[2 * cols + col]));
                    if (!GSLICE) sx[slot] = make_uint4(X, Y, Z, (unsigned)ja);
                }
                if (rank == 0) A.coords[bx.atom0 + ja] = p;
            }
            if (rank == 0 && A.log && tid < nb) {
                epsr_move_log *lg = A.log + (size_t)box * A.log_stride + (size_t)(A.log_off + t0 + tid);
                lg->mol = cur.mol[tid];
                lg->accepted = cur.acc[tid];
                lg->dU = sh.dU[tid];
                lg->n_atoms = cur.natoms[tid];
                lg->u_acc = cur.u_acc[tid];
                for (int a = 0; a < kMaxMolAtoms; ++a) {
                    const int4 p = a < cur.natoms[tid] ? cur.newp[tid][a] : make_int4(0, 0, 0, 0);
                    lg->trial[a][0] = p.x; lg->trial[a][1] = p.y; lg->trial[a][2] = p.z;
                }
            }
            // ---- the moves of the next batch whose molecules the current one has moved --------------
            if (redo) {
                // another next batch: its records again, and its molecules looked up again, those of earlier
                // batches in the global array (their updates came before the partials gathered above)
                cp_async_wait();
                __syncthreads();
                held = min(A.n_moves, tn + kMoveRing);
                copy_records(tn, held);
                cp_async_wait();
                if (tid == 0) {
                    sh.nb_min = 1 << 30;
                    nxt.nb = nxt.mm = 0;
                }
                __syncthreads();
                look_up(tn);
                __syncthreads();
                nb_next = min((int)min((long long)batch_k, A.n_moves - tn), sh.nb_min);
                if (tid == 0) nxt.nb = nb_next;
                if (mine && gk < nb_next) {
                    nxt.oldp[gk][gsub] = gc;
                    nxt.spos[gk][gsub] = gp - (int)bx.atom0;
                    if (gsub == 0) nxt.mol[gk] = mol;
                }
            }
            if (nb_next > 0) {
                again = gk < nb_next && last >= 0 && cur.acc[last];
                if (again && gsub < cur.natoms[last]) nxt.oldp[gk][gsub] = cur.newp[last][gsub];
            }
        }
        if (nb_next == 0) break;
        par ^= 1;
        t0 = tn;
        nb = nb_next;
        if (__syncthreads_or(again || redo || G == 1)) {
            if (prep_warp) trial_moves<CUT>(nxt, sh.ring, tn, nb_next, bx);
            __syncthreads();
        }
        McBatch &now = sh.b[par];
        if (tid == 0) {
            sh.nb_min = 1 << 30;
            sh.cut = 1 << 30;
            sh.b[par ^ 1].mm = 0;
        }
        // ---- E. pair-energy corrections between the batch's moved molecules -----------------
        // Pair pq = (k1 < k) is computed by CTA pq mod G of the box's group, as items (pq, atom
        // a of move k) against the whole molecule of move k1, spread one per warp before the
        // partner sums; the per-pair sums travel with the partials through the grid barrier.
        // Items are (pair, a, b, side): atom a of move k (old and new) against atom b of
        // move k1 at its new (side 0) or old (side 1) position, one pair_du each, so a CTA's
        // share (18 items for water with G >= 120) runs as one warp's lanes in parallel.
        const int npq = nb * (nb - 1) / 2;
        mm = now.mm;
        n_local = npq > rank ? (npq - rank + G - 1) / G : 0;
        const int n_items = n_local * mm * mm * 2;
        if (n_items <= kCorrItems) {
            for (int it = tid; it < n_items; it += kMcThreads) {
                const int side = it & 1, b = (it >> 1) % mm, a = ((it >> 1) / mm) % mm;
                const int pq = rank + ((it >> 1) / mm / mm) * G;
                const int k = pair_hi(pq);
                const int k1 = pq - k * (k - 1) / 2;
                float v = 0.f;
                if (a < now.natoms[k] && b < now.natoms[k1]) {
                    const int4 na = now.newp[k][a], oa = now.oldp[k][a];
                    const int4 p1 = side ? now.oldp[k1][b] : now.newp[k1][b];
                    v = pair_du<CUT>(sep(na, p1, L), sep(oa, p1, L), bx.row[na.w * kMaxTypes + p1.w], bx, T, ep);
                }
                corr_part[it] = v;
            }
        } else {                                  // large molecules and few CTAs: items (pair, a)
            for (int it = tid; it < n_local * mm; it += kMcThreads) {
                const int a = it % mm, pq = rank + (it / mm) * G;
                const int k = pair_hi(pq);
                const int k1 = pq - k * (k - 1) / 2;
                float ca = 0.f;
                if (a < now.natoms[k]) {
                    const int4 na = now.newp[k][a], oa = now.oldp[k][a];
                    for (int b = 0; b < now.natoms[k1]; ++b) {
                        const int4 nb1 = now.newp[k1][b], ob1 = now.oldp[k1][b];
                        const PairRow &pr = bx.row[na.w * kMaxTypes + nb1.w];
                        ca += pair_du_cold<CUT>(sep(na, nb1, L), sep(oa, nb1, L), pr, bx, T, ep) -
                              pair_du_cold<CUT>(sep(na, ob1, L), sep(oa, ob1, L), pr, bx, T, ep);
                    }
                }
                corr_part[it] = ca;
            }
        }
        fine = n_items <= kCorrItems;
        // ---- C. partial dU of the batch's moves against this CTA's slice ---------------------
        // Near chunks: those whose box meets the near sphere of the move. A (move, chunk) item
        // takes all pairs of the moved atoms with the chunk's partners in the cancellation-free form,
        // and the items of the CTA are spread over its warps: in a large box the few moves near this
        // CTA's region would otherwise keep single warps busy. The other chunks have at most
        // Lennard-Jones terms, scanned by the move's warp without any test per pair.
        const unsigned ltm = (1u << lane) - 1u;
        int n_near[kPerWarp], base[kPerWarp];          // near chunks of the warp's moves, and their first items
        {
            unsigned ox[kPerWarp], oy[kPerWarp], oz[kPerWarp];
            float hw2[kPerWarp];
            int cnt[kPerWarp];
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) {
                const int k = min(warp + q * kMcWarps, nb - 1);
                ox[q] = now.sco[k][0][0];
                oy[q] = now.sco[k][0][1];
                oz[q] = now.sco[k][0][2];
                hw2[q] = warp + q * kMcWarps >= nb ? -1.f : A.near_all ? 3e38f : now.hw2[k];
                cnt[q] = 0;
            }
            for (int w = 0; w < n_words; ++w) {
                const int c = w * 32 + lane, col = min(c, n_chunks - 1), t = ct[col];
                const int cx = cb[col], cy = cb[cols + col], cz = cb[2 * cols + col];
                const int hx = cb[3 * cols + col], hy = cb[4 * cols + col], hz = cb[5 * cols + col];
#pragma unroll
                for (int q = 0; q < kPerWarp; ++q) {
                    const int k = warp + q * kMcWarps;
                    const float x = (float)max(0, abs((int)(ox[q] - (unsigned)cx)) - hx);
                    const float y = (float)max(0, abs((int)(oy[q] - (unsigned)cy)) - hy);
                    const float z = (float)max(0, abs((int)(oz[q] - (unsigned)cz)) - hz);
                    const unsigned rw = c < n_chunks ? now.rows[min(k, nb - 1)][t] : 0u;
                    const bool in = fmaf(x, x, fmaf(y, y, z * z)) < hw2[q];
                    const unsigned mk = __ballot_sync(0xffffffffu, in && rw != 0u);
                    const unsigned fk = __ballot_sync(0xffffffffu, !in && (rw & 0xFFu));
                    if (lane == 0 && k < nb) {
                        near[k * A.words_cap + w] = mk;
                        far[k * A.words_cap + w] = fk;
                    }
                    cnt[q] += __popc(mk);
                }
            }
            // the warp's moves take consecutive places in the item queue (the order of the warps does not
            // matter: every move sums its own items in their order)
            int all = 0;
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) {
                n_near[q] = cnt[q];
                base[q] = all;
                all += cnt[q];
            }
            int first = 0;
            if (lane == 0 && all) first = atomicAdd(&sh.n_queue, all);
            first = __shfl_sync(0xffffffffu, first, 0);
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) base[q] += first;
        }
        __syncwarp();
        ++seq;
        float *ps = A.slots + (size_t)(seq & 1u) * A.grid * kMcSlotStride;
        const bool arrive = G > 1 && cta != A.skip_arrival_cta;
        float acc[kPerWarp];
#pragma unroll
        for (int q = 0; q < kPerWarp; ++q) acc[q] = 0.f;
        int n_all = 0;
        for (int r0 = 0; r0 == 0 || r0 < n_all; r0 += kQueue) {
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) {
                const int k = warp + q * kMcWarps;
                if (n_near[q] == 0) continue;
                int at = base[q] - r0;
                for (int w = 0; w < n_words; ++w) {
                    const unsigned mk = near[k * A.words_cap + w];
                    const int i = at + __popc(mk & ltm);
                    if (((mk >> lane) & 1u) && i >= 0 && i < kQueue) queue[i] = k | ((w * 32 + lane) << 8);
                    at += __popc(mk);
                }
            }
            if (r0 == 0 && !(CUT && bx.lj_cut)) {
                // Lennard-Jones terms with the far chunks, atom by atom for two moves at a time
                const uint64_t S2 = f2_pack(bx.sc_s2, bx.sc_s2);
                const int all_groups = n_chunks << (cs - 5);              // groups of 32 slots
                for (int g0 = 0; g0 < all_groups; g0 += GSLICE ? A.stage / 32 : all_groups) {
                    if (GSLICE) {
                        // stage the copy of the next partners, read once for the whole batch
                        __syncthreads();
                        for (int i = tid; i < min(A.stage, (all_groups - g0) * 32); i += kMcThreads) {
                            const int4 p = __ldcg(&slice[g0 * 32 + i]);
                            sx[i] = make_uint4(scale32_near(p.x, bx.sc_rcp), scale32_near(p.y, bx.sc_rcp),
                                               scale32_near(p.z, bx.sc_rcp), (unsigned)(p.w == kNoAtom ? kNoAtom : 0));
                        }
                        __syncthreads();
                    }
                    const int g1 = GSLICE ? min(all_groups, g0 + A.stage / 32) : all_groups;
#pragma unroll 1
                    for (int h = 0; h < kPerWarp; h += 2) {               // (one copy of the scan's code)
                        const int k0 = warp + h * kMcWarps;
                        if (k0 >= nb) break;
                        const bool two = k0 + kMcWarps < nb;
                        const int k1 = two ? k0 + kMcWarps : k0;
                        const unsigned atoms0 = (unsigned)now.lj_atoms[k0], atoms1 = two ? (unsigned)now.lj_atoms[k1] : 0u;
                        float f0 = 0.f, f1 = 0.f;
                        for (unsigned todo = atoms0 | atoms1; todo; todo &= todo - 1u) {
                            const int a = __ffs(todo) - 1;
                            LjSource s0 = lj_source(now, (atoms0 >> a) & 1u ? k0 : k1, a, bx);
                            LjSource s1 = lj_source(now, (atoms1 >> a) & 1u ? k1 : k0, a, bx);
                            for (int gw = g0; gw < g1; gw += 32) {
                                // far groups of each move in this word
                                unsigned m0, m1;
                                if (!GSLICE) {
                                    m0 = far[k0 * A.words_cap + (gw >> 5)];
                                    m1 = two ? far[k1 * A.words_cap + (gw >> 5)] : 0u;
                                } else {
                                    const int c = min(gw + lane, g1 - 1) >> (cs - 5);        // chunks of 2^(cs - 5) groups
                                    const bool in = gw + lane < g1;
                                    m0 = __ballot_sync(0xffffffffu, in && ((far[k0 * A.words_cap + (c >> 5)] >> (c & 31)) & 1u));
                                    m1 = __ballot_sync(0xffffffffu, in && two && ((far[k1 * A.words_cap + (c >> 5)] >> (c & 31)) & 1u));
                                }
                                for (int t = 0; t < nt; ++t) {
                                    // groups of type t in this word
                                    const int lo = max(0, (sh.cbase[t] << (cs - 5)) - gw), up = min(32, (sh.cbase[t + 1] << (cs - 5)) - gw);
                                    if (lo >= up) continue;
                                    unsigned tm = (up == 32 ? 0xFFFFFFFFu : (1u << up) - 1u) & ~((1u << lo) - 1u);
                                    const unsigned t0m = (now.rows[k0][t] >> a) & 1u ? m0 & tm : 0u;
                                    const unsigned t1m = (now.rows[k1][t] >> a) & 1u ? m1 & tm : 0u;
                                    if (!(t0m | t1m)) continue;
                                    const PairRow &ra = bx.row[s0.type * kMaxTypes + t], &rb = bx.row[s1.type * kMaxTypes + t];
                                    s0.c12 = ra.c12; s0.nc6 = -ra.c6;
                                    s1.c12 = rb.c12; s1.nc6 = -rb.c6;
                                    far_groups(f0, f1, s0, s1, t0m, t1m, lo, up, sx + (gw - (GSLICE ? g0 : 0)) * 32, S2, lane);
                                }
                            }
                        }
#pragma unroll
                        for (int u = 0; u < kPerWarp; u += 2)
                            if (u == h) {
                                acc[u] += f0;
                                acc[u + 1] += f1;
                            }
                    }
                }
            }
            if (r0 == 0) cp_async_wait();                // records of the next batch
            __syncthreads();
            n_all = sh.n_queue;
            // (its loads run while the items do)
            if (r0 == 0 && t0 + nb < A.n_moves) look_up(t0 + nb);
            if (r0 == 0 && arrive) {
                // the CTA's corrections go out now; the partials of every move from its own warp below
                float *pc = ps + (size_t)kBatchMax * A.grid + (size_t)bx.cta0 * kMcCorrPerCta;
                for (int u = kMcThreads - 1 - tid; u < n_local; u += kMcThreads) pc[rank + u * G] = corr_sum(corr_part, u, mm, fine);
            }
            // near items, one per warp at a time
            for (int i = warp; i < min(kQueue, n_all - r0); i += kMcWarps) {
                const int e = queue[i], k = e & 0xFF, col = e >> 8;
                const int t = ct[col], m = now.natoms[k], a0 = now.a0[k];
                const unsigned rw = now.rows[k][t], todo = (rw | (rw >> 8)) & 0xFFu;
                const int4 *np = now.newp[k], *op = now.oldp[k];
                float v = 0.f;
                for (int o = col << cs; o < ((col + 1) << cs); o += 32) {
                    const int4 pj = slice[o + lane];
                    const int ja = pj.w >> 3;
                    const bool valid = pj.w != kNoAtom && !(ja >= a0 && ja < a0 + m);
                    v += m == 1 ? near_du<1, CUT>(np, op, m, todo, pj, t, valid, bx, T, ep)
                         : m <= 3 ? near_du<3, CUT>(np, op, m, todo, pj, t, valid, bx, T, ep)
                                  : near_du<0, CUT>(np, op, m, todo, pj, t, valid, bx, T, ep);
                }
                v = warp_sum(v);
                if (lane == 0) q_res[i] = v;
            }
            __syncthreads();
            // each move's items of the round, in order (lane-strided, then the warp's sum below)
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) {
                const int k = warp + q * kMcWarps;
                if (k >= nb) continue;
                for (int i = lane; i < n_near[q]; i += 32) {
                    const int at = base[q] + i - r0;
                    if (at >= 0 && at < kQueue) acc[q] += q_res[at];
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < kPerWarp; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
        // lane q writes the sum of the warp's move q
        {
            float v = acc[0];
#pragma unroll
            for (int q = 1; q < kPerWarp; ++q) v = lane == q ? acc[q] : v;
            const int k = warp + lane * kMcWarps;
            if (lane < kPerWarp && k < nb) {
                if (G == 1) sh.part[k] = v;
                else if (arrive) ps[(size_t)k * A.grid + cta] = v;
            }
        }
        // Arrival: the CTA barrier and the release (cumulative) put every thread's writes before the
        // group's counter. Slot buffer, per parity: partials [kBatchMax][grid] (one move's partials of
        // the group are contiguous), then corrections, the box's pair pq at cta0 * kMcCorrPerCta + pq.
        __syncthreads();
        if (tid == 0) {
            sh.n_queue = 0;
            if (arrive) red_add_release_gpu(&A.flags[box], 1u);
        }
    }
    if (rank == 0 && warp == 0) block_sum_du(sh.acc_du, n_du, lane, sh.st_sum);
    if (rank == 0 && tid == 0) {
        epsr_mc_stats *st = A.stats + box;
        st->attempted += sh.st_att;
        st->accepted += sh.st_acc;
        st->nonfinite += sh.st_nonfinite;
        st->sum_dU += sh.st_sum;
    }
}

int launch_mc_sweep(const McArgs &args, int grid, size_t smem, cudaStream_t stream)
{
    // instantiations: partner slices in shared or global memory x Lennard-Jones uncut or cut
    const void *fns[2][2] = {{(const void *)mc_sweep_kernel<false, false>, (const void *)mc_sweep_kernel<false, true>},
                             {(const void *)mc_sweep_kernel<true, false>, (const void *)mc_sweep_kernel<true, true>}};
    static bool attr_set = false;
    if (!attr_set) {
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j) {
                cudaError_t e = cudaFuncSetAttribute(fns[i][j], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)kMcMaxDynSmem);
                if (e != cudaSuccess) return set_cuda_error(e, "cudaFuncSetAttribute(mc)");
            }
        attr_set = true;
    }
    const void *fn = fns[args.slice_g ? 1 : 0][args.lj_cut ? 1 : 0];
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kMcThreads, smem);
    if (e != cudaSuccess) return set_cuda_error(e, "occupancy(mc)");
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (per_sm * sms < grid)
        return set_error(EPSR_ELAUNCH, "mc sweep: %d CTAs cannot be co-resident (%d per SM x %d SMs)",
                         grid, per_sm, sms);
    McArgs a = args;
    void *params[] = {&a};
    e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kMcThreads), params, smem, stream);
    if (e == cudaErrorCooperativeLaunchTooLarge)
        return set_error(EPSR_ELAUNCH, "mc sweep: cooperative launch of %d CTAs refused", grid);
    if (e != cudaSuccess) return set_cuda_error(e, "cudaLaunchCooperativeKernel(mc)");
    note_launch();
    return EPSR_OK;
}

int mc_escapee_max() { return kEscMax; }
int mc_batch_max() { return kBatchMax; }

}  // namespace epsr
