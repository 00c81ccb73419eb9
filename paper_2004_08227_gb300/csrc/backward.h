// backward.h -- FP64 replay of the iterations and the reverse sweep (gradient
// of the dual bound with respect to the original costs).
#pragma once
#include <cstddef>

#include <cuda_runtime.h>

#include "mplpp.h"
#include "common.cuh"

namespace mplpp {

// record.cu
size_t rec64_smem_bytes(int lmax);
cudaError_t launch_rec64_phase(const EdgeDesc *edges, const int *items, int n_items, const float *tab, double *agg,
                               double *msg, unsigned char *rec, const long long *rec_off, int lmax, cudaStream_t st);
cudaError_t launch_widen(const float *src, double *dst, long long n, cudaStream_t st);
// the same update with an FP32 screen and FP64 only for the candidates (bit for
// bit the same minima and argmins); tab_floats >= L_u * (ld | 1) of every edge;
// descs and rec_off: the matching's edges and record offsets in schedule order
size_t rec_screen_smem_bytes(int lmax, long long tab_floats);
cudaError_t launch_rec_screen_phase(const EdgeDesc *descs, int n_items, const float *tab,
                                    double *agg, double *msg, unsigned char *rec, const long long *rec_off, int lmax,
                                    long long tab_floats, cudaStream_t st);

// One update of the backward's queue kernels.
struct BwItem {
    EdgeDesc ed;
    int pos_u, pos_v;   // earlier updates of each end within an iteration, in the queue's order
    int deg_u, deg_v;   // updates of each end per iteration
    long long rec_off;  // byte offset of the edge's argmins within an iteration's records
};
static_assert(sizeof(BwItem) == 96, "BwItem layout");
// A queue kernel: the updates of `iterations` iterations in the order of items
// (repeated), blocks taking the next one; the state in versioned FP64 entries.
struct BwQueue {
    const BwItem *items;
    long long n_items;
    int iterations;
    unsigned done;           // iterations the entries' versions count already
    ulonglong2 *agg, *msg;
    long long rec_stride;    // bytes of an iteration's records
    unsigned long long *queue;
    int *err;
    long long spin_limit;
    int lmax;
    unsigned test_wait;      // testing: 1 if the first update waits for one of node u that never comes
};
#ifdef __CUDACC__
// Place g of the queue: iteration and item (in 32 bits: launches hold fewer than
// 2^32 updates, or are split)
__device__ __forceinline__ uint2 bw_place(const BwQueue &p, long long g)
{
    const unsigned n = static_cast<unsigned>(p.n_items), u = static_cast<unsigned>(g), it = u / n;
    return make_uint2(it, u - it * n);
}

// a - m once they carry versions va and vm (both requested at once; a bounded
// wait, after which the kernel drains without waiting)
__device__ __forceinline__ double bw_poll_diff(const BwQueue &p, const ulonglong2 *a, const ulonglong2 *m, unsigned va,
                                               unsigned vm, bool &drain, double *first = nullptr)
{
    ulonglong2 x = ld_se(a), y = ld_se(m);
    for (long long spins = 1; !drain && !(se_ok(x, va) && se_ok(y, vm)); ++spins) {
        if (spins > p.spin_limit) {
            atomicCAS(p.err, 0, ERR_TIMEOUT);
            drain = true;
        } else if ((spins & 63) == 0 && *reinterpret_cast<volatile int *>(p.err) == ERR_TIMEOUT) {
            drain = true;
        }
        if (spins > 64) __nanosleep(32);
        if (!se_ok(x, va)) x = ld_se(a);
        if (!se_ok(y, vm)) y = ld_se(m);
    }
    if (first) *first = se64_val(x);
    return first ? se64_val(y) : se64_val(x) - se64_val(y);
}
#endif
// the replay for label counts up to 128 in one launch; rec: the records of the
// first of the iterations, or nullptr; max_items: the largest matching
bool rec_group_fits(int lmax);
cudaError_t launch_rec_queue(const BwQueue &p, int max_items, const float *tab, unsigned char *rec, cudaStream_t st);
// FP64 values to entries of version 0, and back
cudaError_t launch_to_entries(const double *src, ulonglong2 *dst, long long n, cudaStream_t st);
cudaError_t launch_from_entries(const ulonglong2 *src, double *dst, long long n, cudaStream_t st);

// backward.cu
cudaError_t launch_bw_init(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes, const float *tab,
                           const double *agg, const double *msg, const float *dD, double *adj_agg, double *adj_msg,
                           double *gtab, int lmax, cudaStream_t st);
size_t bw_sweep_smem_bytes(int lmax);
// the reverse sweep over `iterations` iterations, the last one first: p.items in
// reverse schedule order, p.agg / p.msg the adjoints, rec the first iteration's
// records; gtab: the tables' gradient, added to
cudaError_t launch_bw_sweep(const BwQueue &p, int max_items, const unsigned char *rec, double *gtab, cudaStream_t st);
cudaError_t launch_unpack_grad(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes,
                               const long long *pair_base, const long long *unary_base, const double *gtab,
                               const double *adj_agg, float *grad_pair, float *grad_un, cudaStream_t st);

}  // namespace mplpp
