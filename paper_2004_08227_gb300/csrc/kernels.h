// kernels.h -- host-visible launch interfaces of the solver's kernels.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace mplpp {

// Arguments of the Handshake kernels (one struct, passed by value).
struct HsParams {
    const EdgeDesc *edges;
    const float *tab;
    ulonglong2 *agg;         // reparametrized unaries (agg layout, versioned double-float entries)
    ulonglong2 *msg;         // messages (msg layout, versioned double-float entries)
    const int *items;        // looped: edge ids of the phase being launched
    const int *work_off;     // persistent: [clusters + 1] offsets into work
    const WorkItem *work;    // persistent: per-cluster item lists (one iteration)
    int *err;                // device error word (ERR_*)
    long long spin_limit;    // polls before a wait gives up
    int iterations;          // persistent: iterations to run
    int test_wait;           // testing: first item of worker 0 waits for an update that never comes
    int rr;                  // launch the variant with register-resident passes
    int pw;                  // persistent, with rr: the last warp of a CTA polls node u (no rows)
    int C;                   // CTAs per edge (cluster size)
    int tile_floats;         // capacity of one table buffer (floats)
    int workers;             // warp driver: number of warp workers (lists in work_off / work)
    int lw;                  // warp driver: per-warp vector capacity (entries, multiple of 4)
    int cap;                 // warp driver: floats per table buffer (>= 32 rows of any table)
    int rmax;                // capacity of row vectors (floats, multiple of 4)
    int ldmax;               // capacity of column vectors (floats, multiple of 4)
    unsigned long long *queue;  // queue driver: next item index (0 before the launch)
    long long queue_items;      // queue driver: items per iteration (the list in work)
    int queue_entries;          // ... and the mean entries of a table
};

// Update counts an item expects of its inputs (persistent drivers): node u's
// and node v's entries carry u / v (earlier updates of the node in this
// launch), the edge's messages carry e (earlier updates of the edge); the
// item writes u + 1, v + 1, e + 1.  `bump` is added to what the u side waits
// for (testing the bounded wait: an update that never comes).
struct Versions {
    unsigned u, v, e, bump;
};

size_t hs_smem_bytes(int nbuf, int tile_floats, int rmax, int ldmax, int threads, int C);
size_t hs_queue_smem_bytes(int rmax, int ldmax, int threads);
bool hs_queue_batches(int ldmax, int entries);

// warp.cu: one warp per edge (persistent).  Shared memory per warp for vector
// capacity lw and table buffers of cap floats: the work record, two
// mbarriers, two buffers, double-float uh and vh, FP32 w1, alpha, beta.
__host__ __device__ inline size_t hs_warp_bytes_per_warp(int lw, int cap)
{
    return sizeof(WorkItem) + 16 + 8 * static_cast<size_t>(cap) + 28 * static_cast<size_t>(lw);
}
constexpr int kWarpMaxL = 128;  // largest label count (and row stride) the warp driver takes
cudaError_t hs_warp_prepare(size_t smem_bytes);
int hs_warp_max_blocks(int threads, size_t smem_bytes);  // co-resident blocks on the device
cudaError_t hs_launch_warp(const HsParams &p, int blocks, int threads, size_t smem, cudaStream_t st);
cudaError_t hs_prepare(size_t smem_bytes);
cudaError_t hs_launch_looped(const HsParams &p, int n_items, int threads, size_t smem, cudaStream_t st);
cudaError_t hs_launch_persistent(const HsParams &p, int clusters, int threads, size_t smem, cudaStream_t st);
int hs_max_active_clusters(int C, int threads, size_t smem, bool rr);
bool hs_rr_fits(int nr_max, int Q_max, int threads, int tile_floats);
bool hs_pw_fits(int nr_max, int Q_max, int threads, int tile_floats);  // rr_fits with a poller warp
// queue driver (one launch, a global item queue, tables streamed from memory)
cudaError_t hs_launch_queue(const HsParams &p, int blocks, int threads, size_t smem, cudaStream_t st);
int hs_queue_max_blocks(int ldmax, int entries, int threads, size_t smem);  // co-resident blocks on the device

// resident.cu: one CTA per model, the model's state in shared memory for all
// iterations, a block barrier between matchings (label counts <= kResMaxL);
// groups of res_lanes(lmax) lanes update one edge each.
constexpr int kResMaxL = 32;
constexpr int kResWarpBytes = 3 * 32 * 4;  // per-warp vectors (3 words per lane)
__host__ __device__ constexpr int res_lanes(int lmax)
{
    return lmax <= 8 ? 8 : (lmax <= 16 ? 16 : 32);
}
struct ResModel {
    long long agg_base, agg_n;  // the model's entries in agg
    long long msg_base, msg_n;  // ... and in msg
    long long tab_base;         // ... and its first table in tab (floats)
    long long desc;             // its first descriptor in sched_desc
    int steps;                  // steps per iteration (each: one edge per group)
    int full;                   // every label count equals res_lanes
};
// A scheduled edge of the resident driver, relative to its model (16 bytes,
// one load): x = first table entry (floats after the model's first table),
// y = node u's | node v's first agg entry << 16, z = phi_{v->u}'s | phi_{u->v}'s
// first msg entry << 16 (entries after the model's first), w = L_u | L_v << 8 |
// ld << 16 | kResSync in every descriptor of a matching's first step.
constexpr int kResSync = 1 << 24;
constexpr int kResSpare = 2 * 32;  // entries of the spare slot after a model's messages
struct ResParams {
    const float *tab;
    ulonglong2 *agg;
    ulonglong2 *msg;
    const ResModel *models;
    const int4 *sched_desc;   // per model and step: one descriptor per group, as above
    int iterations;
};
cudaError_t res_prepare(size_t smem);
cudaError_t launch_resident(const ResParams &p, int n_models, int threads, size_t smem, int lmax, cudaStream_t st);

// narrow.cu: the persistent driver for label counts <= kResMaxL, a group of
// res_lanes(lmax) lanes per edge, one warp per block.  A warp's steps: up to
// 32 / res_lanes(lmax) edges of one matching each (no edge: Lu = Lv = 0).
struct NarrowRec {
    long long toff;             // table (floats in tab)
    unsigned au, av, mu, mv;    // node vectors in agg, messages in msg (entries)
    int pos_u, pos_v;           // earlier updates of each end within an iteration
    int deg_u, deg_v;           // updates of each end per iteration
    unsigned char Lu, Lv, ld, pad[5];
};
static_assert(sizeof(NarrowRec) == 48, "NarrowRec layout");
struct NarrowParams {
    const float *tab;
    ulonglong2 *agg;
    ulonglong2 *msg;
    const int *step_off;    // [warps + 1] first step of every warp
    const NarrowRec *recs;  // [steps][32 / res_lanes]
    int iterations;
    int test_wait;          // testing: the first step of warp 0 waits for an update that never comes
    int *err;
    long long spin_limit;
};
int narrow_max_warps(int lmax);  // co-resident warps on the device
cudaError_t launch_narrow(const NarrowParams &p, int warps, int lmax, cudaStream_t st);

// rules.cu: the MPLP (eq. (M)) and uniform (eq. (U)) updates of Sec. 4, one
// CTA per edge, one launch per matching.
constexpr int kRuleH = 0, kRuleM = 1, kRuleU = 2;  // the MPLPP_RULE_* values
struct RuleParams {
    const EdgeDesc *edges;
    const int *items;  // edge ids of the matching being launched
    const float *tab;
    ulonglong2 *agg;
    ulonglong2 *msg;
};
size_t rule_smem_bytes(int lumax, int ldmax);  // lumax >= every L_u, ldmax >= every row stride
cudaError_t rule_prepare(size_t smem_bytes);
cudaError_t launch_rule(const RuleParams &p, int rule, int n_items, size_t smem, cudaStream_t st);

// structured.cu: the Handshake update for truncated-linear costs
// w min(|s - t|, tau) in O(L) per minimization and for truncated-quadratic
// costs w min((s - t)^2, tau) over a window, one warp per edge, looped.
constexpr int kStructMaxL = 256;  // largest label count the structured kernel takes
struct StructParams {
    const EdgeDesc *edges;
    const int *items;      // edge ids of the matching being launched
    int n_items;
    int lmax;              // >= every label count of the solver, multiple of 4
    const float2 *param;   // [edges] (w, tau) per edge id
    const int *kind;       // [edges] MPLPP_PAIR_* per edge id
    ulonglong2 *agg;
    ulonglong2 *msg;
    // persistent form (struct_queue_kernel): every warp takes the next item of
    // the queue driver's list (work, queue_items per iteration); versioned waits
    const WorkItem *work;
    unsigned long long *queue;
    long long queue_items;
    int iterations;
    int test_wait;
    int *err;
    long long spin_limit;
};
constexpr int kStructPad = 16;
// uh, vh double-float; h, m FP32; then one of: the scans' indices, the envelope
// (value, index; one entry more than labels), a window's vector with kStructPad
// entries to either side
__host__ __device__ inline size_t struct_bytes_per_warp(int lmax)
{
    const size_t l = static_cast<size_t>(lmax), envelope = 8 * (l + 2), window = 4 * (l + 2 * kStructPad);
    return 24 * l + (envelope > window ? envelope : window);
}
cudaError_t struct_prepare(int lmax);
cudaError_t launch_struct(const StructParams &p, cudaStream_t st);
cudaError_t launch_struct_queue(const StructParams &p, int blocks, cudaStream_t st);
int struct_queue_max_blocks(int lmax);  // co-resident blocks of 8 warps
// tables of n consecutive edges from their (w, tau) and kind: w min(|s - t|,
// tau) or w min((s - t)^2, tau), rows padded with +inf; a negative or
// non-finite parameter sets ERR_NONFINITE
cudaError_t launch_materialize(const EdgeDesc *edges, const float2 *param, const int *kind, int n, float *tab,
                               int *err, cudaStream_t st);
constexpr int kPairLinear = 1, kPairQuad = 2;  // the MPLPP_PAIR_TRUNC_* values

// dual.cu
// Packs the costs of n_models <= kPackModels consecutive models, the first one
// model0, and sets phi = 0: edges, nodes: theirs; msg, n_msg: their messages;
// unary, pair: the caller's arrays per model on the device (pair nullptr: tables
// not packed).  lmax: the largest label count.
constexpr int kPackModels = 128;
cudaError_t launch_pack(int n_models, const float *const *unary, const float *const *pair, int model0,
                        const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes, int lmax, float *tab,
                        float *un0, ulonglong2 *agg, ulonglong2 *msg, long long n_msg, int *err, unsigned *stamp, cudaStream_t st);
// part: [n_models * kSumSlices] FP64 scratch of the sums; max_terms: the
// largest model's edges + nodes; emin: ~0 in every entry, and left so.
constexpr int kSumSlices = 64;
cudaError_t launch_bound(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes,
                         const float *tab, const ulonglong2 *agg, const ulonglong2 *msg, unsigned long long *emin,
                         double *nmin, const int *model_node_off, const int *model_edge_off, int n_models,
                         int max_terms, int exact, int lmax, double *part, double *out,
                         cudaStream_t st);  // lmax >= every label count and row stride
// Primal rounding, then the energies.  order: the nodes by level of the
// rounding order (a node's earlier neighbours lie in lower levels); labels has
// room for one entry more (the queue's counter); max_label: the largest label
// count; spin_limit: polls of a wait for a label; test_wait: testing (the last
// node waits for labels that it never sees).
cudaError_t launch_round(const EdgeDesc *edges, const NodeDesc *nodes, int n_nodes, const int *in_off,
                         const InRec *in_rec, const int *order, const int *model_node_off, const int *model_edge_off,
                         int n_models, const float *tab, const ulonglong2 *agg, const ulonglong2 *msg, const float *un0,
                         int *labels, double *energy, int *err, int max_label, int max_terms, double *part,
                         long long spin_limit, int test_wait, cudaStream_t st);
int sum_slices(int max_terms);  // partial sums per model of a sum over its edges and nodes (> 1: one launch more)
// stamp[0]: nonzero if a state entry may carry a version other than 0.  A full
// pack (stamp given) and a reset clear it; who lets a kernel write versions
// without launch_restamp before it sets it.
cudaError_t launch_init_state(const float *un0, ulonglong2 *agg, long long n_agg, ulonglong2 *msg, long long n_msg,
                              unsigned *stamp, cudaStream_t st);
// Sets the version of every state entry to 0, keeping the values (nothing to do
// if stamp[0] is 0), and stamp[0] for the run that follows.
cudaError_t launch_restamp(ulonglong2 *agg, long long n_agg, ulonglong2 *msg, long long n_msg, unsigned *stamp,
                           cudaStream_t st);

}  // namespace mplpp
