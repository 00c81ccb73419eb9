// dual.cu -- packing of the inputs, the dual lower bound (Sec. 3, eq.
// LP-lower-bound), sequential primal rounding (Sec. 4, Primal Rounding) and
// the energy (eq. energy-min) on sm_103a.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "bound_scan.cuh"
#include "kernels.h"

namespace mplpp {

namespace {

constexpr int kThreads = 256;

// Packs the costs of up to kPackModels consecutive models: the caller's
// row-major tables into the padded layout (row stride ld, pad +inf), the unaries
// into un0 (FP32) and agg (double-float entries, version 0), pad 0, and sets the
// messages to 0 (version 0): the state phi = 0.  Flags non-finite costs.  Models
// with structured costs (pair == nullptr) get their tables elsewhere.
// A copy, bound by HBM: 16-byte stores everywhere, 16-byte loads where the
// caller's rows allow them (no padding, aligned), and no division per entry --
// a thread steps from chunk to chunk of a row with a carry.  One launch for all
// models, the pointers as launch arguments.  16 x K_50 with 64 labels (643 MB
// moved): 446 us in 32 launches with a 64-bit division per entry, 92 us so (7.0 TB/s).
struct PackPtrs {
    const float *unary[kPackModels];
    const float *pair[kPackModels];
};

__device__ __forceinline__ bool finite4(float4 v)
{
    return isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w);
}

// One table by a team of TEAM threads (ti: the thread's index in it).
template <int TEAM>
__device__ __forceinline__ bool pack_table(const EdgeDesc &ed, const float *src, float *tab, int ti)
{
    constexpr int kB = 4;  // chunks in flight per thread
    bool ok = true;
    const int Lv = ed.Lv, Q = ed.ld >> 2;
    const long long nq = static_cast<long long>(ed.Lu) * Q;
    float4 *dst = reinterpret_cast<float4 *>(tab + ed.toff);
    if (Lv == ed.ld && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const float4 *s4 = reinterpret_cast<const float4 *>(src);
        for (long long n = ti; n < nq; n += kB * TEAM) {
            float4 v[kB];
#pragma unroll
            for (int r = 0; r < kB; ++r)
                if (n + r * TEAM < nq) v[r] = s4[n + r * TEAM];
#pragma unroll
            for (int r = 0; r < kB; ++r)
                if (n + r * TEAM < nq) {
                    ok = ok && finite4(v[r]);
                    dst[n + r * TEAM] = v[r];
                }
        }
        return ok;
    }
    int s = ti / Q, q = ti - s * Q;
    const int ds = TEAM / Q, dq = TEAM - ds * Q;
    for (long long n = ti; n < nq; n += TEAM) {
        const float *p = src + static_cast<long long>(s) * Lv + 4 * q;
        float4 v = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        const int left = Lv - 4 * q;  // >= 1
        v.x = p[0];
        if (left > 1) v.y = p[1];
        if (left > 2) v.z = p[2];
        if (left > 3) v.w = p[3];
        ok = ok && isfinite(v.x) && (left <= 1 || isfinite(v.y)) && (left <= 2 || isfinite(v.z)) &&
             (left <= 3 || isfinite(v.w));
        dst[n] = v;
        q += dq;
        s += ds;
        if (q >= Q) {
            q -= Q;
            ++s;
        }
    }
    return ok;
}

// Blocks [0, edge_blocks): tables (a warp per edge, or a CTA per edge); the next
// node_blocks: unaries, a warp per node; the rest: messages.
template <bool WARP>
__global__ void __launch_bounds__(kThreads) pack_kernel(PackPtrs ptrs, int model0, const EdgeDesc *edges, int n_edges,
                                                        int edge_blocks, const NodeDesc *nodes, int n_nodes,
                                                        int node_blocks, float *tab, float *un0, ulonglong2 *agg,
                                                        ulonglong2 *msg, long long n_msg, int *err, unsigned *stamp)
{
    if (stamp && blockIdx.x == 0 && threadIdx.x == 0) stamp[0] = 0u;  // as init_state_kernel
    constexpr int W = kThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int b = blockIdx.x;
    bool ok = true;
    if (b < edge_blocks) {
        for (int e = WARP ? b * W + warp : b; e < n_edges; e += edge_blocks * (WARP ? W : 1)) {
            const EdgeDesc ed = edges[e];
            const float *src = ptrs.pair[ed.model - model0];
            if (!src) continue;
            ok = pack_table<WARP ? 32 : kThreads>(ed, src + ed.poff, tab, WARP ? lane : static_cast<int>(threadIdx.x)) && ok;
        }
    } else if ((b -= edge_blocks) < node_blocks) {
        for (int u = b * W + warp; u < n_nodes; u += node_blocks * W) {
            const NodeDesc nd = nodes[u];
            const float *src = ptrs.unary[nd.model - model0] + nd.uoff;
            const int Lp = (nd.L + 3) & ~3;
            for (int s = lane; s < Lp; s += 32) {
                const float v = s < nd.L ? src[s] : 0.f;
                ok = ok && isfinite(v);
                un0[nd.aoff + s] = v;
                agg[nd.aoff + s] = se_make(make_float2(v, 0.f), 0u);
            }
        }
    } else {
        b -= node_blocks;
        const long long stride = static_cast<long long>(gridDim.x - edge_blocks - node_blocks) * kThreads;
        for (long long i = static_cast<long long>(b) * kThreads + threadIdx.x; i < n_msg; i += stride)
            msg[i] = se_make(make_float2(0.f, 0.f), 0u);
    }
    if (!ok) atomicCAS(err, 0, ERR_NONFINITE);
}

// emin[e] = min_{s,t} (theta_uv(s,t) - phi_{v->u}(s)) - phi_{u->v}(t) as an
// order-preserving key of its FP64 value (bound_scan.cuh: screened in FP32 and
// double-float, the survivors in FP64), and nmin[u] = min_s theta^phi_u(s).
// Bound by the one read of the tables.  A warp per edge where tables are small
// and many (TEAM = 32), else a CTA per block of rows of an edge (TEAM = 256;
// `parts` blocks per edge, so that wide tables spread over the SMs).  The few
// entries that reach FP64 (a converged 64 x 64 table has near 50 tied ones) are
// collected over a warp's edges and evaluated 32 at a time: an FP64 instruction
// holds the pipe for a whole warp however few lanes are active.  For the same
// reason floats are widened by integer operations: four FP64 instructions per
// 32 entries instead of nine (kNN, 57,000 tables of 64 x 64: 256 -> 231 us).  They
// meet in emin by atomicMin, so emin must hold ~0 before (bound_sum_kernel leaves
// it so).
struct Final {  // an entry to evaluate in FP64
    float th;
    float2 p1, p2;
    int e;
};
constexpr int kFinals = 64;  // per warp

template <int TEAM>
__host__ __device__ constexpr size_t bound_smem_bytes(int lw)
{
    return (kThreads / 32) * (kScanChunks * sizeof(int) + kFinals * sizeof(Final)) +
           8 * static_cast<size_t>(lw) * (TEAM == 32 ? kThreads / 32 : 1);
}

// nmin[u] by the blocks from `first` on, a warp per node
__device__ __forceinline__ void node_minima(const NodeDesc *nodes, int n_nodes, const ulonglong2 *agg, double *nmin,
                                            int first)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int W = kThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (static_cast<int>(gridDim.x) - first) * W;
    for (int u = (static_cast<int>(blockIdx.x) - first) * W + warp; u < n_nodes; u += nw) {
        const NodeDesc nd = nodes[u];
        // double-floats are normalized: ordered by hi, then lo
        float2 m = make_float2(INFINITY, 0.f);
        auto low = [&](float2 v) {
            if (v.x < m.x || (v.x == m.x && v.y < m.y)) m = v;
        };
        for (int s = lane; s < nd.L; s += 32) low(se_df(agg[nd.aoff + s]));
        for (int o = 16; o > 0; o >>= 1) low(make_float2(__shfl_xor_sync(kAll, m.x, o), __shfl_xor_sync(kAll, m.y, o)));
        if (lane == 0) nmin[u] = df_to_d(m);
    }
}

// The same minimum for at most G = 8 or 16 labels: G lanes per edge, lane s with
// row s in registers, so that a warp takes 32 / G edges and the chain of an edge
// (descriptor, messages, screens) is shared by as many.  The screen in double-
// float is that of bound_scan.cuh's lists (its bound B), over every entry; what it
// leaves, a row's tied minimum as a rule, is evaluated in FP64.  Bound by
// instructions.  2,048 K_20 of 8 labels: 295 -> 99 us, K_600 of 13: 198 -> 131 us
// (a warp's list and its passes cost as much for 16 chunks of a table as for 1,024).
template <int G>
__global__ void __launch_bounds__(kThreads) bound_small_kernel(const EdgeDesc *edges, int n_edges, int edge_blocks,
                                                               const float *tab, const ulonglong2 *msg,
                                                               unsigned long long *emin, const NodeDesc *nodes,
                                                               int n_nodes, const ulonglong2 *agg, double *nmin)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int W = kThreads / 32, P = 32 / G;
    if (static_cast<int>(blockIdx.x) >= edge_blocks) {
        node_minima(nodes, n_nodes, agg, nmin, edge_blocks);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = lane & (G - 1), g0 = lane & ~(G - 1);
    for (int base = (static_cast<int>(blockIdx.x) * W + warp) * P; base < n_edges; base += edge_blocks * W * P) {
        const int e = min(base + lane / G, n_edges - 1);  // a group without an edge repeats the last one's
        const EdgeDesc ed = edges[e];
        const float4 *row = reinterpret_cast<const float4 *>(tab + ed.toff) + s * (ed.ld >> 2);
        float th[G];
#pragma unroll
        for (int c = 0; c < G / 4; ++c) {
            const float4 v = s < ed.Lu && 4 * c < ed.Lv ? __ldg(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            th[4 * c] = v.x;
            th[4 * c + 1] = v.y;
            th[4 * c + 2] = v.z;
            th[4 * c + 3] = v.w;
        }
        const float2 zero = make_float2(0.f, 0.f);
        const float2 a = s < ed.Lu ? se_df(msg[ed.mu + s]) : zero, b = s < ed.Lv ? se_df(msg[ed.mv + s]) : zero;
        float lo[G], H = INFINITY;
        const int tmax = __reduce_max_sync(kAll, ed.Lv);
#pragma unroll
        for (int t = 0; t < G; ++t) {
            lo[t] = INFINITY;
            if (t >= tmax) continue;  // the same in every lane
            const float2 c = make_float2(__shfl_sync(kAll, b.x, g0 + t), __shfl_sync(kAll, b.y, g0 + t));
            const float2 o = df_sub(df_sub(make_float2(th[t], 0.f), a), c);
            const float S = __fadd_ru(fabsf(th[t]), __fadd_ru(fabsf(a.x), fabsf(c.x)));
            const float B = __fadd_ru(__fadd_ru(__fmul_ru(0x1p-43f, S), 0x1p-120f), fabsf(o.y));
            lo[t] = __fsub_rd(o.x, B);
            if (s < ed.Lu && t < ed.Lv) H = fminf(H, __fadd_ru(o.x, B));
        }
        for (int q = G >> 1; q > 0; q >>= 1) H = fminf(H, __shfl_xor_sync(kAll, H, q));
        unsigned left = 0u;
#pragma unroll
        for (int t = 0; t < G; ++t)
            if (s < ed.Lu && t < ed.Lv && !(lo[t] > H)) left |= 1u << t;
        const double da = d_of_f(a.x) + d_of_f(a.y), db = d_of_f(b.x) + d_of_f(b.y);
        unsigned long long best = ~0ull;
#pragma unroll 1
        while (__any_sync(kAll, left != 0u)) {
            const int t = left ? __ffs(left) - 1 : 0;
            const double c = __shfl_sync(kAll, db, g0 + t);
            if (left) {
                const double v = (d_of_f(__ldg(reinterpret_cast<const float *>(row) + t)) - da) - c;
                if (!isnan(v)) best = min(best, f64_key(v));
            }
            left &= left - 1u;
        }
        for (int q = G >> 1; q > 0; q >>= 1) best = min(best, __shfl_xor_sync(kAll, best, q));
        if (s == 0 && base + lane / G < n_edges) emin[e] = best;
    }
}

template <int TEAM>
__global__ void __launch_bounds__(kThreads, 4) bound_scan_kernel(const EdgeDesc *edges, int n_edges, int parts,
                                                                 int edge_blocks, const float *tab,
                                                                 const ulonglong2 *msg, int lw,
                                                                 unsigned long long *emin, const NodeDesc *nodes,
                                                                 int n_nodes, const ulonglong2 *agg, double *nmin)
{
    extern __shared__ __align__(16) char smem_raw[];
    __shared__ float red[2][kThreads / 32];
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int W = kThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (static_cast<int>(blockIdx.x) >= edge_blocks) {
        node_minima(nodes, n_nodes, agg, nmin, edge_blocks);
        return;
    }
    // the vectors first (read as float4), then the lists of the warps
    float *vec = reinterpret_cast<float *>(smem_raw);
    Final *fin = reinterpret_cast<Final *>(vec + 2 * lw * (TEAM == 32 ? W : 1)) + warp * kFinals;
    int *list = reinterpret_cast<int *>(reinterpret_cast<Final *>(vec + 2 * lw * (TEAM == 32 ? W : 1)) + W * kFinals) +
                warp * kScanChunks;
    float *d2 = vec + (TEAM == 32 ? 2 * warp * lw : 0), *d1 = d2 + lw;  // lw: a multiple of 4
    const int ti = TEAM == 32 ? lane : static_cast<int>(threadIdx.x);
    int nf = 0;  // entries in fin (the same in every lane)
    auto finish = [&]() {
        __syncwarp();
        for (int i = lane; i < nf; i += 32) {
            const Final f = fin[i];
            const double v = (d_of_f(f.th) - (d_of_f(f.p1.x) + d_of_f(f.p1.y))) - (d_of_f(f.p2.x) + d_of_f(f.p2.y));
            if (!isnan(v)) atomicMin(&emin[f.e], f64_key(v));
        }
        __syncwarp();
        nf = 0;
    };
    const int units = n_edges * parts;
    const int u0 = TEAM == 32 ? static_cast<int>(blockIdx.x) * W + warp : static_cast<int>(blockIdx.x);
    const int ustep = TEAM == 32 ? edge_blocks * W : edge_blocks;
    for (int unit = u0; unit < units; unit += ustep) {
        const int e = TEAM == 32 ? unit : unit / parts;
        const EdgeDesc ed = edges[e];
        int s0 = 0, nr = ed.Lu;
        if (TEAM != 32) {
            const int R = (ed.Lu + parts - 1) / parts;
            s0 = (unit - e * parts) * R;
            nr = min(R, ed.Lu - s0);
            if (nr <= 0) continue;  // the same in every thread
        }
        const int Q = ed.ld >> 2, nq = nr * Q;
        const float4 *th4 = reinterpret_cast<const float4 *>(tab + ed.toff) + static_cast<long long>(s0) * Q;
        float4 first[kScanBatch];
        scan_load<TEAM>(th4, ti, nq, first);
        const ulonglong2 *mu = msg + ed.mu, *mv = msg + ed.mv;
        const float2 r1 = se_df(mu[s0]), r2 = se_df(mv[0]);
        float D1 = 0.f, D2 = 0.f;
        for (int t = ti; t < ed.ld; t += TEAM) {
            const float d = t < ed.Lv ? df_to_f(df_sub(se_df(mv[t]), r2)) : 0.f;
            d2[t] = d;
            D2 = fabsf(d) > D2 || isnan(d) ? fabsf(d) : D2;
        }
        for (int s = s0 + ti; s < s0 + nr; s += TEAM) {
            const float d = df_to_f(df_sub(se_df(mu[s]), r1));
            d1[s] = d;
            D1 = fabsf(d) > D1 || isnan(d) ? fabsf(d) : D1;
        }
        D1 = redux_max_abs(D1);
        D2 = redux_max_abs(D2);
        if (TEAM == 32) {
            __syncwarp();
        } else {
            if (lane == 0) {
                red[0][warp] = D1;
                red[1][warp] = D2;
            }
            __syncthreads();
            D1 = redux_max_abs(red[0][lane & (W - 1)]);
            D2 = redux_max_abs(red[1][lane & (W - 1)]);
        }
        scan_table<TEAM>(
            th4, nq, Q, ed.Lv, s0, first, d1, d2, scan_slack(D1, D2, r1.x, r2.x), list,
            [&](int s) { return se_df(mu[s]); }, [&](int t) { return se_df(mv[t]); },
            [&](bool on, int s, int t, float th) {
                const unsigned mask = __ballot_sync(kAll, on);
                if (nf > kFinals - 32) finish();
                if (on) fin[nf + __popc(mask & ((1u << lane) - 1u))] = Final{th, se_df(mu[s]), se_df(mv[t]), e};
                nf += __popc(mask);
            });
        if (TEAM == 32)
            __syncwarp();  // d1, d2 are rewritten for the next edge
        else
            __syncthreads();
    }
    finish();
}

// Fixed-order FP64 sum (deterministic): thread i adds elements i, i+T, ...,
// then a fixed tree.
template <int T>
__device__ double block_sum_fixed(double v, double *red)
{
    red[threadIdx.x] = v;
    __syncthreads();
    for (int o = T / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

// Block (m, c) adds model m's node and edge minima of slice c (FP64 additions
// run at two lanes per cycle and SM, so a large model is summed by many
// blocks; sum_parts_kernel adds the slices in order).  emin is set back to ~0
// for the next call.
__global__ void __launch_bounds__(kThreads) bound_sum_kernel(const int *model_node_off, const int *model_edge_off,
                                                             const double *nmin, unsigned long long *emin, int exact,
                                                             double *out)
{
    __shared__ double red[kThreads];
    const int m = blockIdx.x, first = blockIdx.y * kThreads + threadIdx.x, step = gridDim.y * kThreads;
    double acc = 0.0;
    for (int u = model_node_off[m] + first; u < model_node_off[m + 1]; u += step) acc += nmin[u];
    if (exact)
        for (int e = model_edge_off[m] + first; e < model_edge_off[m + 1]; e += step) {
            acc += emin[e] == ~0ull ? static_cast<double>(INFINITY) : f64_of_key(emin[e]);
            emin[e] = ~0ull;
        }
    const double D = block_sum_fixed<kThreads>(acc, red);
    if (threadIdx.x == 0) out[static_cast<size_t>(m) * gridDim.y + blockIdx.y] = D;
}

// out[m] = the sum of model m's `slices` partial sums, in order
__global__ void sum_parts_kernel(const double *part, int slices, int n_models, double *out)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n_models) return;
    double acc = 0.0;
    for (int c = 0; c < slices; ++c) acc += part[static_cast<size_t>(m) * slices + c];
    out[m] = acc;
}

// Primal rounding: node u's objective over its labels is its reparametrized
// unary plus, for every earlier neighbour v in increasing order,
// theta^phi_vu(x_v, s) = (theta_vu(x_v,s) - phi_{u->v}(x_v)) - phi_{v->u}(s);
// FP64 sums in that order, argmin with the lowest index.
// GB300's FP64 rate is far below its FP32 rate, so every label's objective
// is first evaluated in double-float (FP32 operations), O(s), with
//   |O(s) - exact| and |FP64 value - exact| <= B(s) = (K + 8) 2^-43 S(s),
// S(s) = |agg_u(s)| + sum_k (|theta| + |phi_{u->v}| + |phi_{v->u}(s)|), K
// earlier neighbours (each double-float addition errs by at most
// 3 * 2^-48 (|a| + |b|), and a label's terms are summed by up to 16 threads
// whose partial sums are then added in a tree: at most K + 4 additions per
// label plus two per term; B carries a factor of more than 10 of margin, so
// the order of the terms does not matter).  With O(s)
// bracketed in FP32 (upward / downward rounding) as [lo(s), hi(s)], a label
// with lo(s) > H = min_s hi(s) can neither attain the FP64 minimum nor tie
// with it.  A single remaining candidate is therefore the FP64 argmin without
// any FP64 work; several (ties, near-ties) are summed in FP64 in neighbour
// order and compared, so the decision always equals the all-FP64 one.

// FP64 objective of node u's label s, summed in neighbour order; the loads of
// kSumBatch neighbours at a time are independent of each other.  A neighbour that
// a team no longer waits for (ERR_TIMEOUT is set) may still be undecided, -1: it
// counts as label 0 here too.
constexpr int kSumBatch = 8;
__device__ double round_sum64(const InRec *rec, int K, const int *labels, const float *tab, const ulonglong2 *msg,
                              double a, int s)
{
    for (int k0 = 0; k0 < K; k0 += kSumBatch) {
        double t[kSumBatch];
#pragma unroll
        for (int j = 0; j < kSumBatch; ++j)
            if (k0 + j < K) {
                const InRec r = rec[k0 + j];
                const int xv = max(*reinterpret_cast<const volatile int *>(labels + r.gu), 0);
                t[j] = (static_cast<double>(tab[r.toff + static_cast<long long>(xv) * r.ld + s]) - se_d(msg[r.mu + xv])) -
                       se_d(msg[r.mv + s]);
            }
#pragma unroll
        for (int j = 0; j < kSumBatch; ++j)
            if (k0 + j < K) a = a + t[j];
    }
    return a;
}

__device__ __forceinline__ void low_label(double &best, int &bi, double v, int i)
{
    if (v < best || (v == best && i < bi)) {
        best = v;
        bi = i;
    }
}

__device__ __forceinline__ void warp_low_label(double &best, int &bi)
{
    for (int o = 16; o > 0; o >>= 1)
        low_label(best, bi, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, bi, o));
}

// Dataflow form, one launch for all models: a team of warps takes the next
// node of one queue (order: nodes by level, level(u) = 1 + the largest level
// of u's earlier neighbours) and adds each earlier neighbour's terms as soon as
// that neighbour's label is there.  labels is -1 until decided, so the label
// itself is the signal: the chain from one decision to the next is one L2 round
// trip for the label, one for its table row and the argmin, instead of a walk
// over all of a node's neighbours or a launch per level.  A team waits only
// for nodes taken earlier by running teams, so the waits end; they are bounded
// all the same (spin_limit polls, then ERR_TIMEOUT and no more waiting).
// A team is one warp for nodes of at most 32 NL labels, else TW warps of 32 NL
// labels each (TW > 1: the whole block).  With at most 16 labels the lanes split
// into 32 / G groups of G, each adding its share of the neighbours.
// Bound by that chain, about 2 us a node or level.  Against one CTA per model
// walking its nodes: K_600 with 13 labels 4.91 -> 1.18 ms, K_60 with 300 labels
// 471 -> 84 us, 2,048 K_20 941 -> 94 us; against a launch per level: a 128 x 128
// grid with 64 labels 1.43 (and 0.7 of gaps) -> 0.63 ms, 2,000-node kNN 625 ->
// 189 us.  A single ready neighbour is added by a loop of its own (K_600: 1.60 ms
// without).  A warp that waits for its last 4 neighbours or fewer requests their
// tables and messages into L2, so that the row the label selects is near: K_600
// 1.15 -> 1.04 ms, the grid 0.63 -> 0.57 ms, kNN 191 -> 170 us, 16 K_50 with 64
// labels 89 -> 82 us (8 or 16 neighbours: K_600 1.06, 1.11 ms; with wider labels,
// a block per node, nothing: 85 us).
constexpr int kRoundFetch = 4;  // the last undecided neighbours, fetched ahead
constexpr int kRoundWarps = 4;  // warps per block of one-warp teams
constexpr int kRoundMaxWarps = 16;

template <int NL, bool TEAM>
__global__ void __launch_bounds__(TEAM ? 32 * kRoundMaxWarps : 32 * kRoundWarps)
    round_flow_kernel(const NodeDesc *nodes, const int *order, int n_nodes, const int *in_off, const InRec *in_rec,
                      const float *tab, const ulonglong2 *agg, const ulonglong2 *msg, int *labels, int *queue, int *err,
                      long long spin_limit, int test_wait)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kRows = NL == 1 ? 8 : (NL == 2 ? 4 : 2);  // neighbours whose loads are in flight together
    __shared__ int s_ticket;
    __shared__ float rh[kRoundMaxWarps];
    __shared__ int rc[kRoundMaxWarps], ri[kRoundMaxWarps];
    __shared__ double rv[kRoundMaxWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, TW = TEAM ? static_cast<int>(blockDim.x >> 5) : 1;
    const int w = TEAM ? warp : 0;
    bool drain = false;
    for (;;) {
        int ticket = 0;
        if (TEAM) {
            __syncthreads();  // the shared results of the previous node have been read
            if (threadIdx.x == 0) s_ticket = atomicAdd(queue, 1) + 1;  // the queue starts at -1
            __syncthreads();
            ticket = s_ticket;
        } else {
            if (lane == 0) ticket = atomicAdd(queue, 1) + 1;
            ticket = __shfl_sync(kAll, ticket, 0);
        }
        if (ticket >= n_nodes) return;
        const int u = order[ticket];
        const NodeDesc nd = nodes[u];
        const int L = nd.L, k0 = in_off[u], K = in_off[u + 1] - k0;
        const InRec *rec = in_rec + k0;
        // lanes per group of neighbours and this lane's labels
        int G = 32;
        if (NL == 1 && !TEAM && L <= 16) G = L <= 4 ? 4 : (L <= 8 ? 8 : 16);
        const int sub = lane / G, P = 32 / G;
        const int s0 = w * 32 * NL + (lane & (G - 1));
        float2 o[NL];
        float sa[NL];
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            o[i] = make_float2(0.f, 0.f);
            sa[i] = 0.f;
            if (s0 + 32 * i < L && sub == 0) {
                o[i] = se_df(agg[nd.aoff + s0 + 32 * i]);
                sa[i] = fabsf(o[i].x);
            }
        }
        for (int b = 0; b < K; b += 32) {
            const bool on = b + lane < K;
            InRec r = {};
            if (on) r = rec[b + lane];
            unsigned pending = __ballot_sync(kAll, on);
            long long spins = 0;
            bool fetched = false;
            while (pending) {
                int x = -1;
                if ((pending >> lane) & 1u) x = *reinterpret_cast<volatile int *>(labels + r.gu);
                if (test_wait && ticket == n_nodes - 1) x = -1;  // testing: the last node sees no label
                if (drain && x < 0) x = 0;
                unsigned ready = __ballot_sync(kAll, x >= 0) & pending;
                if (!ready) {
                    if (!TEAM && !fetched && __popc(pending) <= kRoundFetch) {
                        // their tables (at most 16 KB each) and messages into L2
                        fetched = true;
                        for (unsigned left = pending; left; left &= left - 1u) {
                            const int src = __ffs(left) - 1;
                            const float *t = tab + __shfl_sync(kAll, r.toff, src);
                            const ulonglong2 *pu = msg + __shfl_sync(kAll, r.mu, src), *pv = msg + __shfl_sync(kAll, r.mv, src);
                            const int Lx = nodes[__shfl_sync(kAll, r.gu, src)].L, n = Lx * __shfl_sync(kAll, r.ld, src);
                            for (int i = 32 * lane; i < n; i += 1024) asm volatile("prefetch.global.L2 [%0];" ::"l"(t + i));
                            for (int i = 8 * lane; i < Lx; i += 256) asm volatile("prefetch.global.L2 [%0];" ::"l"(pu + i));
                            for (int i = 8 * lane; i < L; i += 256) asm volatile("prefetch.global.L2 [%0];" ::"l"(pv + i));
                        }
                        continue;
                    }
                    if (++spins > spin_limit || ((spins & 255) == 0 && *reinterpret_cast<volatile int *>(err) == ERR_TIMEOUT)) {
                        if (lane == 0) atomicCAS(err, 0, ERR_TIMEOUT);
                        drain = true;
                    }
                    if (spins > 64) __nanosleep(32);
                    continue;
                }
                pending &= ~ready;
                // the ready neighbours' row and phi_{u->v}(x_v), one neighbour per lane
                long long row = 0;
                float2 ph = make_float2(0.f, 0.f);
                if ((ready >> lane) & 1u) {
                    row = r.toff + static_cast<long long>(x) * r.ld;
                    ph = se_df(msg[r.mu + x]);
                }
                // the terms of R neighbours per group of lanes, their loads in flight together
                auto add_rows = [&](auto rows) {
                    constexpr int R = decltype(rows)::value;
                    float tv[R][NL];
                    ulonglong2 mv[R][NL];
                    float2 f1[R];
                    unsigned has = 0u;
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        // neighbour number sub of the next P ready ones
                        unsigned mine = ready;
                        for (int j = 0; j < sub; ++j) mine &= mine - 1u;
                        for (int j = 0; j < P; ++j) ready &= ready - 1u;
                        const int src = mine ? __ffs(mine) - 1 : 0;
                        const long long rw = __shfl_sync(kAll, row, src);
                        const long long mo = __shfl_sync(kAll, r.mv, src);
                        f1[q] = make_float2(__shfl_sync(kAll, ph.x, src), __shfl_sync(kAll, ph.y, src));
                        if (mine) {
                            has |= 1u << q;
#pragma unroll
                            for (int i = 0; i < NL; ++i)
                                if (s0 + 32 * i < L) {
                                    tv[q][i] = tab[rw + s0 + 32 * i];
                                    mv[q][i] = msg[mo + s0 + 32 * i];
                                }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < R; ++q)
                        if ((has >> q) & 1u) {
#pragma unroll
                            for (int i = 0; i < NL; ++i)
                                if (s0 + 32 * i < L) {
                                    const float2 f2 = se_df(mv[q][i]);
                                    o[i] = df_add(o[i], df_sub(df_sub(make_float2(tv[q][i], 0.f), f1[q]), f2));
                                    sa[i] += fabsf(tv[q][i]) + fabsf(f1[q].x) + fabsf(f2.x);
                                }
                        }
                };
                if (__popc(ready) <= P)  // as a rule on the chain: the last neighbour alone
                    add_rows(std::integral_constant<int, 1>{});
                while (ready) add_rows(std::integral_constant<int, kRows>{});
            }
        }
        if (NL == 1)  // the groups' partial sums of a label, added in a tree
            for (int q = G; q < 32; q <<= 1) {
                o[0] = df_add(o[0], make_float2(__shfl_xor_sync(kAll, o[0].x, q), __shfl_xor_sync(kAll, o[0].y, q)));
                sa[0] += __shfl_xor_sync(kAll, sa[0], q);
            }
        // the screen
        float lo[NL], H = INFINITY;
        const float cK = static_cast<float>(K + 8);
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            lo[i] = INFINITY;
            if (s0 + 32 * i < L && sub == 0) {
                const float bnd = __fadd_ru(__fmul_ru(cK, __fadd_ru(__fmul_ru(0x1.1p-43f, sa[i]), 0x1p-120f)), fabsf(o[i].y));
                lo[i] = __fsub_rd(o[i].x, bnd);
                H = fminf(H, __fadd_ru(o[i].x, bnd));
            }
        }
        H = redux_min_f32(H);
        if (TEAM) {
            if (lane == 0) rh[warp] = H;
            __syncthreads();
            H = redux_min_f32(lane < TW ? rh[lane] : INFINITY);
        }
        int ncand = 0, only = INT_MAX;  // candidates of the team, and one of them
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const bool c = s0 + 32 * i < L && sub == 0 && lo[i] <= H;
            const unsigned m = __ballot_sync(kAll, c);
            ncand += __popc(m);
            if (m) only = w * 32 * NL + 32 * i + __ffs(m) - 1;
        }
        if (TEAM) {
            if (lane == 0) {
                rc[warp] = ncand;
                ri[warp] = only;
            }
            __syncthreads();
            const int c = lane < TW ? rc[lane] : 0;
            ncand = __reduce_add_sync(kAll, c);
            only = __reduce_min_sync(kAll, c ? ri[lane] : INT_MAX);
        }
        if (ncand != 1) {
            // ties or near-ties (or none: every objective NaN): FP64 sums in neighbour order
            double best = INFINITY;
            int bi = INT_MAX;
#pragma unroll
            for (int i = 0; i < NL; ++i)
                if (s0 + 32 * i < L && sub == 0 && lo[i] <= H)
                    low_label(best, bi, round_sum64(rec, K, labels, tab, msg, se_d(agg[nd.aoff + s0 + 32 * i]), s0 + 32 * i),
                              s0 + 32 * i);
            warp_low_label(best, bi);
            if (TEAM) {
                __syncthreads();  // ri has been read
                if (lane == 0) {
                    rv[warp] = best;
                    ri[warp] = bi;
                }
                __syncthreads();
                best = lane < TW ? rv[lane] : static_cast<double>(INFINITY);
                bi = lane < TW ? ri[lane] : INT_MAX;
                warp_low_label(best, bi);
            }
            only = bi;
            if (bi == INT_MAX) {
                only = 0;
                if (threadIdx.x == 0 || !TEAM) atomicCAS(err, 0, ERR_NONFINITE);
            }
        }
        if (lane == 0 && w == 0) *reinterpret_cast<volatile int *>(labels + u) = only;
    }
}

// One CTA per model walking its nodes in order, for label counts beyond the
// dataflow form's.  Latency: the in-edges of node u + 1 whose neighbour is
// already decided are staged (table row offset, messages) and their table rows
// prefetched into L2 by the threads without labels while node u is decided.
constexpr int kRoundThreads = 512;

__global__ void __launch_bounds__(kRoundThreads) round_kernel(const NodeDesc *nodes, const int *in_off,
                                                              const InRec *in_rec, const int *model_node_off,
                                                              const float *tab,
                                                              const ulonglong2 *agg, const ulonglong2 *msg,
                                                              int *labels, int *err)
{
    constexpr int T = kRoundThreads;
    __shared__ double rv[T / 32];
    __shared__ int ri[T / 32];
    __shared__ float rh[T / 32];
    // staged earlier neighbours (up to T per chunk), two sets: node u's and,
    // prepared meanwhile, node u + 1's
    __shared__ long long k_row[2][T], k_mv[2][T];
    __shared__ float2 k_phf[2][T];
    const int m = blockIdx.x;
    const int tid = threadIdx.x;
    const int w = tid >> 5, l = tid & 31;
    constexpr int kBatch = 16;  // rows of different tables miss in L2: loads in flight
    const int u0 = model_node_off[m], u1 = model_node_off[m + 1];
    auto stage_one = [&](int set, int slot, const InRec &r, int xv) {
        k_row[set][slot] = r.toff + static_cast<long long>(xv) * r.ld;
        k_mv[set][slot] = r.mv;
        const double ph = se_d(msg[r.mu + xv]);
        const float hi = static_cast<float>(ph);
        k_phf[set][slot] = make_float2(hi, static_cast<float>(ph - static_cast<double>(hi)));
    };
    bool pre = false;  // node u's set was staged (except a neighbour u - 1) during node u - 1
    for (int u = u0; u < u1; ++u) {
        const int set = (u - u0) & 1;
        const NodeDesc nd = nodes[u];
        const int L = nd.L;
        const int k0 = in_off[u], k1 = in_off[u + 1], K = k1 - k0;
        const bool chunked = K > T;
        // threads per label: the largest power of two (<= 16) leaving half the
        // block free to prepare the next node; labels beyond T / P loop (P = 1)
        int P = 1;
        while (P < 16 && 2 * P * L <= T / 2) P *= 2;
        const int s_of = tid / P, part = tid % P;
        const int nlab = T / P;  // labels per sweep
        // node u's staged neighbours: complete the set (the neighbour u - 1 was
        // still undecided) or stage it now
        if (!chunked) {
            if (pre) {
                if (K > 0 && tid == K - 1) {
                    const InRec r = in_rec[k0 + tid];
                    if (r.gu == u - 1) stage_one(set, tid, r, labels[r.gu]);
                }
            } else if (tid < K) {
                const InRec r = in_rec[k0 + tid];
                stage_one(set, tid, r, labels[r.gu]);
            }
            __syncthreads();
        }
        // the next node's neighbours decided by now, by threads without labels
        const int busy = ((L < nlab ? L : nlab) * P + 31) & ~31;
        const bool prep = u + 1 < u1 && in_off[u + 2] - in_off[u + 1] <= T && T - busy >= 32;
        if (prep && tid >= busy) {
            const int Ln = nodes[u + 1].L;
            for (int k = in_off[u + 1] + tid - busy; k < in_off[u + 2]; k += T - busy) {
                const InRec r = in_rec[k];
                if (r.gu < u) {
                    const int xv = labels[r.gu];
                    stage_one(set ^ 1, k - in_off[u + 1], r, xv);
                    const float *pr = tab + r.toff + static_cast<long long>(xv) * r.ld;
                    for (int q = 0; q < Ln; q += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(pr + q));
                }
            }
        }
        // double-float screen; thread (s, part) sums neighbours k = part, part + P, ...
        float hsel = INFINITY;
        float lo_own = INFINITY;
        float2 o = make_float2(0.f, 0.f);
        float sa = 0.f;
        const int s = s_of;
        const bool mine = s < L && s < nlab;
        if (mine && part == 0) {
            o = se_df(agg[nd.aoff + s]);
            sa = fabsf(o.x);
        }
        for (int c0 = k0; c0 < k1; c0 += T) {
            const int nc = min(T, k1 - c0);
            if (chunked) {  // long neighbour lists: staged chunk by chunk
                __syncthreads();
                if (tid < nc) {
                    const InRec r = in_rec[c0 + tid];
                    stage_one(set, tid, r, labels[r.gu]);
                }
                __syncthreads();
            }
            if (mine)
                for (int kb = part; kb < nc; kb += kBatch * P) {
                    float tv[kBatch];
                    ulonglong2 mv[kBatch];
#pragma unroll
                    for (int q = 0; q < kBatch; ++q) {
                        const int k = kb + q * P;
                        if (k < nc) {
                            tv[q] = tab[k_row[set][k] + s];
                            mv[q] = msg[k_mv[set][k] + s];
                        }
                    }
#pragma unroll
                    for (int q = 0; q < kBatch; ++q) {
                        const int k = kb + q * P;
                        if (k < nc) {
                            const float2 f1 = k_phf[set][k], f2 = se_df(mv[q]);
                            o = df_add(o, df_sub(df_sub(make_float2(tv[q], 0.f), f1), f2));
                            sa += fabsf(tv[q]) + fabsf(f1.x) + fabsf(f2.x);
                        }
                    }
                }
        }
        // the P partial sums of a label (consecutive lanes), added in a tree
        for (int q = 1; q < P; q <<= 1) {
            const float ox = __shfl_xor_sync(0xffffffffu, o.x, q), oy = __shfl_xor_sync(0xffffffffu, o.y, q);
            o = df_add(o, make_float2(ox, oy));
            sa += __shfl_xor_sync(0xffffffffu, sa, q);
        }
        if (mine) {
            const float cK = static_cast<float>(K + 8);
            const float b = __fadd_ru(__fmul_ru(cK, __fadd_ru(__fmul_ru(0x1.1p-43f, sa), 0x1p-120f)), fabsf(o.y));
            lo_own = __fsub_rd(o.x, b);
            hsel = __fadd_ru(o.x, b);
        }
        for (int q = 16; q > 0; q >>= 1) hsel = fminf(hsel, __shfl_xor_sync(0xffffffffu, hsel, q));
        if (l == 0) rh[w] = hsel;
        __syncthreads();
        float H = rh[0];
        for (int q = 1; q < T / 32; ++q) H = fminf(H, rh[q]);
        bool cand = mine && part == 0 && lo_own <= H;
        // labels beyond one sweep (L > T, P = 1) are never screened: decided the
        // exact way below
        const bool extra = L > nlab;
        const int ncand = __syncthreads_count(cand);
        if (ncand == 1 && !extra) {
            // the only label that can attain the FP64 minimum
            if (cand) labels[u] = s;
            __syncthreads();
        } else {
            // several candidates (ties or near-ties), none (NaN objectives), or
            // labels beyond one sweep: FP64 sums in neighbour order
            double best = INFINITY;
            int bi = INT_MAX;
            if (cand) {
                double a = se_d(agg[nd.aoff + s]);
                for (int k = k0; k < k1; ++k) {
                    const InRec r = in_rec[k];
                    const int xv = labels[r.gu];
                    a = a + ((static_cast<double>(tab[r.toff + static_cast<long long>(xv) * r.ld + s]) -
                              se_d(msg[r.mu + xv])) -
                             se_d(msg[r.mv + s]));
                }
                best = a;
                bi = s;
            }
            if (extra && part == 0)
                for (int s2 = nlab + s_of; s2 < L; s2 += nlab) {
                    double a = se_d(agg[nd.aoff + s2]);
                    for (int k = k0; k < k1; ++k) {
                        const InRec r = in_rec[k];
                        const int xv = labels[r.gu];
                        a = a + ((static_cast<double>(tab[r.toff + static_cast<long long>(xv) * r.ld + s2]) -
                                  se_d(msg[r.mu + xv])) -
                                 se_d(msg[r.mv + s2]));
                    }
                    if (a < best || (a == best && s2 < bi)) {
                        best = a;
                        bi = s2;
                    }
                }
            for (int o2 = 16; o2 > 0; o2 >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, best, o2);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o2);
                if (ov < best || (ov == best && oi < bi)) {
                    best = ov;
                    bi = oi;
                }
            }
            if (l == 0) {
                rv[w] = best;
                ri[w] = bi;
            }
            __syncthreads();
            if (tid == 0) {
                double bb = INFINITY;
                int i = INT_MAX;
                for (int q = 0; q < T / 32; ++q)
                    if (ri[q] != INT_MAX && (rv[q] < bb || (rv[q] == bb && ri[q] < i))) {
                        bb = rv[q];
                        i = ri[q];
                    }
                if (i == INT_MAX) {  // no candidate: every objective value was NaN
                    i = 0;
                    atomicCAS(err, 0, ERR_NONFINITE);
                }
                labels[u] = i;
            }
            __syncthreads();
        }
        pre = prep;
    }
}

// E(x | original costs) in FP64 (eq. energy-min), fixed-order sums; block (m, c):
// slice c of model m, as in bound_sum_kernel.
__global__ void __launch_bounds__(kThreads) energy_kernel(const EdgeDesc *edges, const NodeDesc *nodes,
                                                          const int *model_node_off, const int *model_edge_off,
                                                          const float *tab, const float *un0, const int *labels,
                                                          double *energy)
{
    __shared__ double red[kThreads];
    const int m = blockIdx.x, first = blockIdx.y * kThreads + threadIdx.x, step = gridDim.y * kThreads;
    double acc = 0.0;
    for (int u = model_node_off[m] + first; u < model_node_off[m + 1]; u += step)
        acc += static_cast<double>(un0[nodes[u].aoff + labels[u]]);
    for (int e = model_edge_off[m] + first; e < model_edge_off[m + 1]; e += step) {
        const EdgeDesc ed = edges[e];
        acc += static_cast<double>(tab[ed.toff + static_cast<long long>(labels[ed.gu]) * ed.ld + labels[ed.gv]]);
    }
    const double En = block_sum_fixed<kThreads>(acc, red);
    if (threadIdx.x == 0) energy[static_cast<size_t>(m) * gridDim.y + blockIdx.y] = En;
}

// Whether an entry of the state may carry a version other than 0: stamp[0].  A
// word on the device, set and read in stream order, so that it holds for graphs
// and captured streams too; stamp[1] counts restamp_kernel's blocks.
//
// agg := (un0, 0), msg := 0: the state phi = 0 (version 0)
__global__ void __launch_bounds__(kThreads) init_state_kernel(const float *un0, ulonglong2 *agg, long long n_agg,
                                                              ulonglong2 *msg, long long n_msg, unsigned *stamp)
{
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    const long long i0 = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (i0 == 0) stamp[0] = 0u;
#pragma unroll 4
    for (long long i = i0; i < n_agg; i += stride) agg[i] = se_make(make_float2(un0[i], 0.f), 0u);
#pragma unroll 4
    for (long long i = i0; i < n_msg; i += stride) msg[i] = se_make(make_float2(0.f, 0.f), 0u);
}

// version := 0 in both words of every entry, unless every one is 0 (after a reset
// of 256 models, 36 million entries: 220 us of reading and writing, 3 us so); the
// run that follows leaves other versions, so the last block sets stamp[0].
__global__ void __launch_bounds__(kThreads) restamp_kernel(ulonglong2 *agg, long long n_agg, ulonglong2 *msg,
                                                           long long n_msg, unsigned *stamp)
{
    if (__syncthreads_or(threadIdx.x == 0 && *reinterpret_cast<volatile unsigned *>(stamp) != 0u)) {
        const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
        const long long i0 = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
        const unsigned long long keep = 0xffffffffull;
#pragma unroll 4
        for (long long i = i0; i < n_agg; i += stride) {
            const ulonglong2 e = agg[i];
            agg[i] = make_ulonglong2(e.x & keep, e.y & keep);
        }
#pragma unroll 4
        for (long long i = i0; i < n_msg; i += stride) {
            const ulonglong2 e = msg[i];
            msg[i] = make_ulonglong2(e.x & keep, e.y & keep);
        }
    }
    if (threadIdx.x == 0 && atomicAdd(&stamp[1], 1u) == gridDim.x - 1) {  // every block has read the flag
        stamp[1] = 0u;
        stamp[0] = 1u;
    }
}

// a grid of few blocks per SM, for grid-stride loops over n entries
int stride_grid(long long n)
{
    return static_cast<int>(std::max<long long>(1, std::min<long long>((n + kThreads - 1) / kThreads, 152 * 8)));
}

}  // namespace

cudaError_t launch_pack(int n_models, const float *const *unary, const float *const *pair, int model0,
                        const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes, int lmax, float *tab,
                        float *un0, ulonglong2 *agg, ulonglong2 *msg, long long n_msg, int *err, unsigned *stamp, cudaStream_t st)
{
    PackPtrs ptrs = {};
    for (int m = 0; m < n_models; ++m) {
        ptrs.unary[m] = unary[m];
        ptrs.pair[m] = pair[m];
    }
    // tables of at most 32 labels a side are less than a CTA's chunks
    const bool warp = lmax <= 32;
    const int edge_blocks = static_cast<int>(std::min<long long>(warp ? (n_edges + 7) / 8 : n_edges, 1 << 20));
    const int node_blocks = std::min((n_nodes + 7) / 8, 1 << 16);
    const int msg_blocks = static_cast<int>(std::min<long long>((n_msg + 8 * kThreads - 1) / (8 * kThreads), 152 * 8));
    const int blocks = edge_blocks + node_blocks + msg_blocks;
    if (blocks <= 0) return cudaSuccess;
    const auto kernel = warp ? pack_kernel<true> : pack_kernel<false>;
    kernel<<<blocks, kThreads, 0, st>>>(ptrs, model0, edges, n_edges, edge_blocks, nodes, n_nodes, node_blocks, tab, un0,
                                        agg, msg, n_msg, err, stamp);
    return cudaGetLastError();
}

cudaError_t launch_init_state(const float *un0, ulonglong2 *agg, long long n_agg, ulonglong2 *msg, long long n_msg,
                              unsigned *stamp, cudaStream_t st)
{
    init_state_kernel<<<stride_grid(std::max(n_agg, n_msg)), kThreads, 0, st>>>(un0, agg, n_agg, msg, n_msg, stamp);
    return cudaGetLastError();
}

cudaError_t launch_restamp(ulonglong2 *agg, long long n_agg, ulonglong2 *msg, long long n_msg, unsigned *stamp,
                           cudaStream_t st)
{
    restamp_kernel<<<stride_grid(std::max(n_agg, n_msg)), kThreads, 0, st>>>(agg, n_agg, msg, n_msg, stamp);
    return cudaGetLastError();
}

// Slices per model of the sums over its edges: a block per 2,048 terms of the
// largest model, at most kSumSlices.
int sum_slices(int max_terms)
{
    return std::max(1, std::min(kSumSlices, max_terms / 2048));
}

cudaError_t launch_bound(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes, const float *tab,
                         const ulonglong2 *agg, const ulonglong2 *msg, unsigned long long *emin, double *nmin,
                         const int *model_node_off, const int *model_edge_off, int n_models, int max_terms, int exact,
                         int lmax, double *part, double *out, cudaStream_t st)
{
    const int lw = (std::max(lmax, 1) + 3) & ~3;
    const int node_blocks = n_nodes > 0 ? std::min((n_nodes + 7) / 8, 152 * 8) : 0;
    const bool warp = scan_by_warps(lw, n_edges), small = warp && lw <= 16;
    int edge_blocks = 0, parts = 1;
    if (exact && n_edges > 0) {
        if (small) {  // 2 or 4 edges per warp (figures at the kernel)
            edge_blocks = std::min((n_edges + 15) / 16, 152 * 16);
        } else if (warp) {
            edge_blocks = std::min((n_edges + 7) / 8, 152 * 16);
        } else {
            // a table in parts only as far as that gives every SM six blocks: a part costs a
            // block's start, its messages and a list however few rows it has (K_60, 300 labels,
            // parts of 32 KB: 250 us, whole tables: 139 us; 40 to 300 labels: 166 / 62 us)
            parts = static_cast<int>(std::max(1LL, std::min({64LL, 4LL * lw * lw / kPartBytes, (152LL * 6 + n_edges - 1) / n_edges})));
            edge_blocks = static_cast<int>(std::min(1LL * n_edges * parts, 1LL << 20));
        }
    }
    if (edge_blocks && small) {
        const auto kernel = lw <= 8 ? bound_small_kernel<8> : bound_small_kernel<16>;
        kernel<<<edge_blocks + node_blocks, kThreads, 0, st>>>(edges, n_edges, edge_blocks, tab, msg, emin, nodes, n_nodes,
                                                               agg, nmin);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    } else if (edge_blocks + node_blocks > 0) {
        const size_t smem = warp ? bound_smem_bytes<32>(lw) : bound_smem_bytes<kThreads>(lw);
        const auto kernel = warp ? bound_scan_kernel<32> : bound_scan_kernel<kThreads>;
        if (edge_blocks && smem > 48 * 1024) {
            cudaError_t e = raise_smem_limit(kernel, smem);
            if (e != cudaSuccess) return e;
        }
        kernel<<<edge_blocks + node_blocks, kThreads, edge_blocks ? smem : 0, st>>>(
            edges, n_edges, parts, edge_blocks, tab, msg, lw, emin, nodes, n_nodes, agg, nmin);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const int slices = sum_slices(max_terms);
    bound_sum_kernel<<<dim3(n_models, slices), kThreads, 0, st>>>(model_node_off, model_edge_off, nmin, emin, exact,
                                                                  slices > 1 ? part : out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || slices == 1) return e;
    sum_parts_kernel<<<(n_models + kThreads - 1) / kThreads, kThreads, 0, st>>>(part, slices, n_models, out);
    return cudaGetLastError();
}

cudaError_t launch_round(const EdgeDesc *edges, const NodeDesc *nodes, int n_nodes, const int *in_off,
                         const InRec *in_rec, const int *order, const int *model_node_off, const int *model_edge_off,
                         int n_models, const float *tab, const ulonglong2 *agg, const ulonglong2 *msg, const float *un0,
                         int *labels, double *energy, int *err, int max_label, int max_terms, double *part,
                         long long spin_limit, int test_wait, cudaStream_t st)
{
    if (max_label <= 32 * 4 * kRoundMaxWarps) {
        // labels and the queue's counter behind them: -1
        cudaError_t e = cudaMemsetAsync(labels, 0xff, sizeof(int) * (static_cast<size_t>(n_nodes) + 1), st);
        if (e != cudaSuccess) return e;
        // labels per lane: one, two (a warp up to 64 labels, 16 warps up to 1,024), else four
        const int NL = max_label <= 32 ? 1 : (max_label <= 64 * kRoundMaxWarps ? 2 : 4);
        const int tw = (max_label + 32 * NL - 1) / (32 * NL);
        const auto kernel = NL == 1   ? round_flow_kernel<1, false>
                            : tw == 1 ? round_flow_kernel<2, false>
                            : NL == 2 ? round_flow_kernel<2, true>
                                      : round_flow_kernel<4, true>;
        const int threads = 32 * (tw == 1 ? kRoundWarps : tw);
        const int teams = tw == 1 ? kRoundWarps : 1;  // per block
        const int per_sm = 1536 / threads;            // enough to fill an SM; any grid is safe
        const int blocks = static_cast<int>(std::min<long long>((n_nodes + teams - 1) / teams, 152LL * per_sm));
        kernel<<<blocks, threads, 0, st>>>(nodes, order, n_nodes, in_off, in_rec, tab, agg, msg, labels,
                                           labels + n_nodes, err, spin_limit, test_wait);
    } else {
        round_kernel<<<n_models, kRoundThreads, 0, st>>>(nodes, in_off, in_rec, model_node_off, tab, agg, msg, labels,
                                                         err);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int slices = sum_slices(max_terms);
    energy_kernel<<<dim3(n_models, slices), kThreads, 0, st>>>(edges, nodes, model_node_off, model_edge_off, tab, un0,
                                                               labels, slices > 1 ? part : energy);
    e = cudaGetLastError();
    if (e != cudaSuccess || slices == 1) return e;
    sum_parts_kernel<<<(n_models + kThreads - 1) / kThreads, kThreads, 0, st>>>(part, slices, n_models, energy);
    return cudaGetLastError();
}

}  // namespace mplpp
