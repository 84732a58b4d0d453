// epsr_internal.h -- host-side declarations shared by libepsr's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <string>

#include "epsr.h"

namespace epsr {

struct BoxDev;
struct MoveRec;

// ---- errors (thread-local last error, see epsr_last_error_detail) -------------------------
int set_error(int status, const char *fmt, ...);
int set_cuda_error(cudaError_t e, const char *what);

// ---- launch accounting (epsr_launch_count): called once after every kernel enqueue ----------
void note_launch();

// ---- autotuner support (epsr_tune.cu): the shape a tuning is cached under --------------------
std::string box_shape_key(const epsr_box *box);
struct BoxSummary {
    int n_boxes, n_pairs, n_bins;
    double rho;             // atoms per A^3
};
int box_summary(const epsr_box *box, int b, BoxSummary *out);
int box_sms(const epsr_box *box);
std::string sq_plan_key(const epsr_sq_plan *p, int n_cols, int cols_per_set, bool totals);
int sq_plan_mode(const epsr_sq_plan *p);
void sq_plan_dims(const epsr_sq_plan *p, int *nQ, int *n_bins, int *max_cols);
int sq_plan_stages(const epsr_sq_plan *p);

// ---- Monte Carlo kernel ----------------------------------------------------------------------
constexpr size_t kMcMaxDynSmem = 161 * 1024;   // with 66 KB of static shared memory, under the 227 KB per CTA
// exchange buffer of the sweep, per parity: the partial dU of every move of a batch from every
// CTA ([kMcBatchMax][grid]), then kMcSlotStride - kMcBatchMax = kMcCorrPerCta floats per CTA of
// which a box group uses its first CTA's share onwards for the batch-pair corrections
constexpr int kMcBatchMax = 64;           // moves per batch of the sweep, at most
constexpr int kMcCorrPerCta = kMcBatchMax * (kMcBatchMax - 1) / 2;   // batch-pair corrections
constexpr int kMcSlotStride = kMcBatchMax + kMcCorrPerCta;
// correction items of one batch in shared memory (>= 496 pairs x 8 atoms: batches above 32 moves
// need 8 or more CTAs per box)
constexpr int kMcCorrItems = 4096;
// partners staged at once in shared memory when the slices live in global memory, and with
// empirical-potential tables that leave no room for as many
constexpr int kMcStageChunk = 2048, kMcStageLeast = 256;
constexpr int kMcMaxWords = 24;           // chunk mask words per CTA of such a slice, at most

struct McArgs {
    const BoxDev *boxes;
    int4 *coords;                 // [n_atoms_total] {x, y, z, type}
    const long long *thresholds;  // concatenated [n_bins + 1] per box
    const float *ep;              // concatenated [n_pairs * n_bins] per box
    const int *cta_box;           // [grid]
    float *slots;                 // [2][grid * kMcSlotStride]: partials [kBatchMax][grid], then corrections
                                  // [grid][kMcCorrPerCta] (a box group uses cta0 * kMcCorrPerCta onwards)
    unsigned *flags;              // [grid] arrival sequence numbers (zeroed per launch)
    epsr_mc_stats *stats;         // [n_boxes] running totals (device)
    epsr_move_log *log;           // nullable [n_boxes][log_stride]
    const MoveRec *moves;         // [n_boxes][chunk] this launch's moves
    const int *sorted_index;      // [n_atoms_total] atom at each type-major sorted position
    const int *pos_of;            // [n_atoms_total] sorted position of each atom
    long long chunk;              // move-table stride per box
    long long log_off;            // log index of this launch's first move
    int *status;                  // device status word
    long long n_moves;
    long long log_stride;
    long long max_spin;           // iteration limit of one barrier wait
    unsigned long long timeout_ns;// time limit of one barrier wait
    int grid;
    int lj_cut;                   // 1: some box truncates Lennard-Jones (the cut instantiation runs)
    int batch_k;
    int slice_cap;                // int4 capacity of the shared partner slice
    int tbl_cap;                  // capacity (entries) of the shared threshold table, 0: read from global memory
    int stage;                    // partners staged at once (slices in global memory)
    int ep_cap;                   // capacity (entries) of the shared empirical-potential table
    int4 *slice_g;                // [grid][slice_cap] partner slices in global memory, or NULL
    int chunk_log;                // log2 of the slots per chunk (5; more for slices in global memory)
    int words_cap;                // chunk mask words per CTA, at most
    int near_all;                 // 1: every chunk is near (no box queries)
    int skip_arrival_cta;         // test hook: this CTA never arrives (-1: none)
};

int launch_mc_sweep(const McArgs &args, int grid, size_t smem, cudaStream_t stream);
int launch_mc_moves(const BoxDev *boxes, const int *mol_start, int n_boxes, long long chunk,
                    long long n, unsigned long long seed, unsigned long long move0, MoveRec *out,
                    cudaStream_t stream);
int launch_intra_energy(const BoxDev *boxes, int n_boxes, const int4 *coords, const int *mol_start, double *U,
                        cudaStream_t stream);
int mc_escapee_max();
int mc_batch_max();

// ---- pair histogram kernels ---------------------------------------------------------------
struct GrTile {           // one (i-tile, j-tile) pair of one box
    int box;
    int ti, tj;
    int pad;
};

struct GrArgs {
    const BoxDev *boxes;
    const int4 *coords;          // [n_atoms_total]
    const uint4 *scaled;         // [n_atoms_total] {x', y', z', type} on the 2^32-periodic grid
    const long long *thresholds;
    const GrTile *tiles;
    long long tile_begin, tile_end;
    unsigned long long *hist;    // accumulated output
    int max_pairs_bins;          // max over boxes of n_pairs * n_bins (shared histogram size)
    int max_bins1;               // max over boxes of n_bins + 1
};

constexpr int kGrTile = 1024;    // atoms per tile (both sides)

// ---- clusters of 32 atoms in Hilbert order (clusters.cuh) ------------------------------------
struct ClBox {            // one box
    int cl0, n_cl;        // first cluster and number of clusters
    int su0, n_su;        // the same of super-clusters (32 clusters)
    int key0, bits;       // first sort key; bits per axis of the Hilbert cells
    int r_fx;             // histogram range in grid units, rounded up (at most 2^30)
    int pad;
};
struct ClScratch {        // device buffers of one handle
    const ClBox *box;
    const int *su_box;    // box of every super-cluster
    int *count;           // [n_keys_pad], then the work counters [n_boxes]
    int *offset, *block;  // [n_keys], [ceil(n_keys / 1024)]
    int *key, *rank, *index;
    int4 *coords;         // coordinates in cluster order
    int4 *cl_c, *cl_h;    // cluster boxes: centre and atom count; half widths and first position
    int4 *su_c, *su_h;    // super-cluster boxes
    int n_keys, n_keys_pad, n_boxes, n_su;
};
struct ClArgs {           // one traversal
    const BoxDev *boxes;
    const ClBox *box;
    const int4 *coords, *cl_c, *cl_h, *su_c, *su_h;
    int *next_item;       // [n_boxes] next unclaimed work item
    const long long *thresholds;
    unsigned long long *hist;
    long long n_cl_total;
    int n_boxes;
    int plog;             // a cluster's partners are split into 2^plog work items
    int hist_cap;         // max over boxes of n_types^2 * n_bins
};
constexpr int kClMaxSmem = 200 * 1024;
size_t gr_clusters_smem(int hist_cap);
// ordered: the order, and so the clusters, depend on the coordinates alone (one launch more); otherwise
// atoms of one Hilbert cell may change places from call to call. *order: the atom at each position.
int launch_clusters(const BoxDev *boxes, const int *atom_box, const int4 *coords, long long n, const ClScratch &sc,
                    bool ordered, const int **order, cudaStream_t stream);
int launch_cell_order(const int *key, const int *count, const int *offset, const int *index, int *out, long long n,
                      cudaStream_t stream);
int launch_gr_clusters(const ClArgs &args, int grid, cudaStream_t stream);
// exclusive scan of n counts (block: scratch [ceil(n / 1024)]), and the scatter of a counting sort
int launch_scan(const int *count, int n, int *offset, int *block, cudaStream_t stream);
int launch_scan_one(const int *count, int n, int *offset, cudaStream_t stream);
int launch_scatter(const int *key, const int *rank, const int *offset, int *index, long long n, cudaStream_t stream);
constexpr int kScanOneMax = 1 << 18;   // counts scanned by the one-launch form at most

int launch_scale_coords(const BoxDev *boxes, const int *atom_box, const int4 *coords,
                        uint4 *scaled, long long n, cudaStream_t stream);
int launch_partial_gr(const GrArgs &args, int grid, cudaStream_t stream);

struct SortScratch {      // device scratch of the spatial sort
    int *count;           // [total_cells]
    int *offset;          // [total_cells]
    int *block;           // [ceil(total_cells / 1024)]
    int *key, *rank;      // [n_atoms_total]
    int *index;           // [n_atoms_total] atom index at each sorted position
};
int launch_spatial_sort(const BoxDev *boxes, const int *atom_box, const uint4 *scaled,
                        const int4 *coords, long long n, int total_cells, int type_major,
                        SortScratch sc, uint4 *s_scaled, int4 *s_coords, int *pos_of,
                        cudaStream_t stream);
int launch_normalize_g(const BoxDev *boxes, int n_boxes, const unsigned long long *hist,
                       float *g, long long n_configs, long long hist_len, const long long *hist_box,
                       cudaStream_t stream);
int launch_total_energy(const BoxDev *boxes, const int4 *coords, const int *atom_mol,
                        const long long *thresholds, const float *ep, const GrTile *tiles,
                        long long n_tiles, double *U, int grid, cudaStream_t stream);

// ---- smeared histogram and adjoint -----------------------------------------------------------
// Node grid of one box (k_smear.cu): h = dr / S, nodes 0 .. nodes - 1 up to r_max + 5 sigma,
// bins in reach of a node within `reach` nodes of the bin, n_off = S + 2 reach + 1 offsets.
struct SmearGrid {
    double h;
    int S, nodes, reach, n_off;
};
constexpr int kSmOffsets = 2048;      // offsets of the weight table, at most
constexpr int kSmMaxS = 16;           // nodes per bin, at most
// Workspace of a handle: per box moments or derivative table (4 x 8 bytes a node and type pair), then
// weights (5 doubles an offset). Handles of many boxes take them in groups of as many as fit.
constexpr size_t kSmWorkspace = 64u << 20;
constexpr int kSmMaxGroup = 32768;    // boxes in grid.y
// h = sigma / 12, or as fine as nodes_cap nodes allow; S = 0 when that leaves it above sigma / 8.
inline
#ifdef __CUDACC__
__host__ __device__
#endif
SmearGrid smear_grid(int n_bins, double dr, double sigma, int nodes_cap)
{
    SmearGrid g;
    const double fine = 12.0 * dr / sigma, least = 8.0 * dr / sigma;
    for (int S = fine < kSmMaxS ? (int)fine + 1 : kSmMaxS;; --S) {
        g.S = S;
        if ((double)S < least || S < 1) { g.S = 0; return g; }
        g.h = dr / (double)S;
        g.reach = (int)(5.0 * sigma / g.h) + 2;
        g.nodes = n_bins * S + g.reach;
        g.n_off = S + 2 * g.reach + 1;
        if (g.nodes <= nodes_cap) break;
    }
    if (g.n_off > kSmOffsets) g.S = 0;
    return g;
}

struct SmearArgs {
    const int *index;          // atom at each position in cluster order
    double sigma;
    int nodes_cap;             // nodes per type pair that fit in shared memory
    long long stride;          // nodes x type pairs per box, at most
    long long *moments;        // forward, nodes: [n_boxes][4 stride], per box [4][n_pairs][nodes], accumulated
    const float4 *table;       // backward, nodes: [n_boxes][stride], per box [n_pairs][nodes]
    unsigned long long *acc;   // forward, direct: weights * 2^20, accumulated
    const float *lambda;       // backward, direct: dL/dHt [hist_len]
    float *grad;               // backward output [n_atoms_total][3] (accumulated)
};
size_t smear_smem(bool table, long long rows);
int smear_warps_per_cta();
int launch_smear(const ClArgs &c, const SmearArgs &a, bool backward, bool table, size_t smem, int grid, cudaStream_t stream);
// weights W [n_boxes][5][offs]; moments and table as in SmearArgs; hist_box the first rows of these boxes,
// of which Ht and gt rows h0 .. h1 - 1 are formed
int launch_smear_weights(const BoxDev *boxes, int n_boxes, double sigma, int nodes_cap, int offs, double *W, cudaStream_t stream);
int launch_smear_bins(const BoxDev *boxes, int n_boxes, double sigma, int nodes_cap, int offs, long long stride,
                      const long long *moments, const double *W, double *Ht, float *gt, long long h0, long long h1,
                      const long long *hist_box, cudaStream_t stream);
int launch_smear_table(const BoxDev *boxes, int n_boxes, double sigma, int nodes_cap, int offs, long long stride,
                       const double *W, const float *lam, float4 *table, cudaStream_t stream);
int launch_smear_norm(const BoxDev *boxes, int n_boxes, const unsigned long long *acc, double *Ht,
                      float *gt, long long hist_len, const long long *hist_box, cudaStream_t stream);
int launch_smear_lambda(const BoxDev *boxes, int n_boxes, const float *dgt, float *lam, long long hist_len,
                        const long long *hist_box, cudaStream_t stream);

// ---- empirical-potential update -------------------------------------------------------------
constexpr int kEpMaxData = 16;     // measured datasets
constexpr int kEpMaxBasis = 40;    // Poisson functions per pair
constexpr int kEpMaxPairs = EPSR_MAX_TYPES * (EPSR_MAX_TYPES + 1) / 2;

struct EpArgs {
    const float *dS;     // [n_data][nQ] device
    const float *Q;      // [nQ] device
    int nQ, n_data, n_pairs, n_basis, n_bins;
    double w[kEpMaxData * kEpMaxPairs];   // [n_data][n_pairs] Eq. (1) weights (barn)
    double s, gamma, alpha, kT, rho, dr;
    double *F;           // [n_basis][nQ] scratch
    double *Y;           // [n_pairs][nQ] scratch
    double *B;           // [n_basis][n_bins] scratch
    double *C_out;       // [n_pairs][n_basis] device
    double *change;      // [1] device: largest change of the table (kJ/mol)
    float *ep;           // [n_pairs][n_bins] the box's table, updated in place
};
int launch_ep_update(const EpArgs &a, cudaStream_t stream);
// epsr_ep_update, also returning the largest change it makes to the table (kJ/mol)
int ep_update_change(epsr_box *box, int32_t b, const float *dS, int32_t n_data, const double *w, const float *Q, int32_t nQ,
                     int32_t n_basis, double s_basis, double gamma, double alpha, double *C_out, double *change,
                     epsr_stream_t stream);

struct ChiParams {
    int P, n_basis;
    double s, rho;
    double W[kEpMaxPairs];     // Eq. (1) weights (2 - delta) c_a c_b b_a b_b, barn
    double *res_scratch;       // [nQ] residuals
    double *F_scratch;         // [n_basis][nQ] basis values F_n(Q)
};
int launch_chi2(const float *S, const float *target, const float *Q, int nQ, const ChiParams &prm,
                const double *C, double *chi2, float *dS, double *dC, cudaStream_t stream);

}  // namespace epsr
