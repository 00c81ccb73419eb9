// backward.cu -- gradient of the dual bound after T Handshake iterations with
// respect to the original unary and pairwise costs, by reverse-mode
// differentiation of the message-form iteration (handshake.cu).
//
// D is piecewise linear in the costs; inside one linear piece every minimum is
// attained at a fixed argument, so D is a sum of selected entries.  The
// iterations are replayed in FP64 (record.cu) from phi = 0, recording the
// argmins of the three minimizations of every update (all of them where they
// fit, else with a state checkpoint every k iterations and, segment by segment
// from the last, a second replay):
//   t1(s) = argmin_t [theta(s,t) + vh(t)],  s2(t) = argmin_s [theta(s,t) + alpha(s)],
//   t3(s) = argmin_t [theta(s,t) + beta(t)]          (lowest index on ties)
// and the updates are replayed in reverse schedule order.  With the adjoints
// Au, Phu (of agg_u and phi_{v->u} after the update) and Av, Phv:
//   cbar = Au + Phu;  uhbar = Au;  bbar = Av + Phv;  vhbar = -Phv
//   betabar(t) = sum_{s: t3(s)=t} cbar(s);  thetabar(s, t3(s)) += cbar(s)
//   vhbar += betabar;  bbar -= betabar;  vhbar += bbar
//   alphabar(s) = sum_{t: s2(t)=s} bbar(t); thetabar(s2(t), t) += bbar(t)
//   uhbar += alphabar / 2   (alpha = uh - a, a = (m1 + uh) / 2)
//   m1bar = -alphabar / 2;  thetabar(s, t1(s)) += m1bar(s);
//   vhbar(t) += sum_{s: t1(s)=t} m1bar(s)
// and the adjoints before the update are Au = uhbar, Phu = -uhbar,
// Av = vhbar, Phv = -vhbar.  The sums over argmin preimages are taken in a
// fixed order, so the result is deterministic.  Updates wait for those that
// share a node with them, as in the forward.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "backward.h"
#include "bound_scan.cuh"
#include "kernels.h"
#include "solver.h"

namespace mplpp {

namespace {

constexpr int kThreads = 256;
constexpr int kSweepLabels = 3 * kThreads;  // the largest label count of a backward

// Adjoint of D = sum_u min agg_u + sum_e min residual_e at the final state.
__global__ void bw_init_nodes_kernel(const NodeDesc *nodes, int n_nodes, const double *agg, const float *dD,
                                     double *adj_agg)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int u = warp; u < n_nodes; u += nw) {
        const NodeDesc nd = nodes[u];
        double m = INFINITY;
        int mi = INT_MAX;
        for (int s = lane; s < nd.L; s += 32) {
            const double v = agg[nd.aoff + s];
            if (v < m) {
                m = v;
                mi = s;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double om = __shfl_xor_sync(0xffffffffu, m, o);
            const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
            if (om < m || (om == m && oi < mi)) {
                m = om;
                mi = oi;
            }
        }
        if (lane == 0 && mi != INT_MAX) adj_agg[nd.aoff + mi] += static_cast<double>(dD[nd.model]);
    }
}

// The edges' part: the table entry that attains the residual's FP64 minimum
// (lowest index on ties) gets the edge's weight, its two messages minus it.  The
// scan is the exact bound's (bound_scan.cuh, as are the team sizes), on FP64
// messages; what survives its screens is compared in FP64 at once.
__device__ __forceinline__ float2 df_of(double v)
{
    const float hi = static_cast<float>(v);
    return make_float2(hi, static_cast<float>(v - static_cast<double>(hi)));
}

template <int TEAM>
__global__ void __launch_bounds__(kThreads, 4)
    bw_init_edges_kernel(const EdgeDesc *edges, int n_edges, const float *tab, const double *msg, const float *dD, int lw,
                         double *adj_msg, double *gtab)
{
    extern __shared__ __align__(16) float vec[];
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int W = kThreads / 32;
    __shared__ float red[2][W];
    __shared__ unsigned long long rk[W];
    __shared__ long long ri[W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *list = reinterpret_cast<int *>(vec + 2 * lw * (TEAM == 32 ? W : 1)) + warp * kScanChunks;
    float *d2 = vec + (TEAM == 32 ? 2 * warp * lw : 0), *d1 = d2 + lw;  // lw: a multiple of 4
    const int ti = TEAM == 32 ? lane : static_cast<int>(threadIdx.x);
    const int e0 = TEAM == 32 ? static_cast<int>(blockIdx.x) * W + warp : static_cast<int>(blockIdx.x);
    const int step = TEAM == 32 ? static_cast<int>(gridDim.x) * W : static_cast<int>(gridDim.x);
    for (int e = e0; e < n_edges; e += step) {
        const EdgeDesc ed = edges[e];
        const int Q = ed.ld >> 2, nq = ed.Lu * Q;
        const float4 *th4 = reinterpret_cast<const float4 *>(tab + ed.toff);
        float4 first[kScanBatch];
        scan_load<TEAM>(th4, ti, nq, first);
        const double *mu = msg + ed.mu, *mv = msg + ed.mv;
        const float2 r1 = df_of(mu[0]), r2 = df_of(mv[0]);
        float D1 = 0.f, D2 = 0.f;
        for (int t = ti; t < ed.ld; t += TEAM) {
            const float d = t < ed.Lv ? df_to_f(df_sub(df_of(mv[t]), r2)) : 0.f;
            d2[t] = d;
            D2 = fabsf(d) > D2 || isnan(d) ? fabsf(d) : D2;
        }
        for (int s = ti; s < ed.Lu; s += TEAM) {
            const float d = df_to_f(df_sub(df_of(mu[s]), r1));
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
        unsigned long long key = ~0ull;  // this lane's best entry
        long long mi = LLONG_MAX;
        auto low = [&](unsigned long long k, long long i) {
            if (k < key || (k == key && i < mi)) {
                key = k;
                mi = i;
            }
        };
        scan_table<TEAM>(
            th4, nq, Q, ed.Lv, 0, first, d1, d2, scan_slack(D1, D2, r1.x, r2.x), list,
            [&](int s) { return df_of(mu[s]); }, [&](int t) { return df_of(mv[t]); },
            [&](bool on, int s, int t, float th) {
                if (on) {
                    const double r = (static_cast<double>(th) - mu[s]) - mv[t];
                    const unsigned long long z = static_cast<unsigned long long>(__double_as_longlong(r));
                    if (!isnan(r)) low((z << 1) ? f64_key(r) : f64_key(0.0), static_cast<long long>(s) * ed.Lv + t);
                }
            });
        for (int o = 16; o > 0; o >>= 1) low(__shfl_xor_sync(kAll, key, o), __shfl_xor_sync(kAll, mi, o));
        if (TEAM != 32) {
            if (lane == 0) {
                rk[warp] = key;
                ri[warp] = mi;
            }
            __syncthreads();
            for (int j = 0; j < W; ++j) low(rk[j], ri[j]);
        }
        if (ti == 0 && mi != LLONG_MAX) {
            const int s = static_cast<int>(mi / ed.Lv);
            const int t = static_cast<int>(mi - static_cast<long long>(s) * ed.Lv);
            const double d = static_cast<double>(dD[ed.model]);
            gtab[ed.toff + static_cast<long long>(s) * ed.ld + t] += d;
            adj_msg[ed.mu + s] -= d;
            adj_msg[ed.mv + t] -= d;
        }
        if (TEAM == 32)
            __syncwarp();  // d1, d2 are rewritten for the next edge
        else
            __syncthreads();
    }
}

// Sum of val over the lanes of this lane's group (grp: the lanes of the warp
// with an equal key), valid in the group's lowest lane: every step adds to each
// remaining lane the value of the next one above it, and every second lane
// drops out, so a group of m takes ceil(log2 m) additions one after the other.
// The order is fixed by the lanes: the sum is deterministic.
__device__ __forceinline__ double peer_sum(double val, unsigned grp, int lane)
{
    constexpr unsigned kAll = 0xffffffffu;
    unsigned above = grp & ~((2u << lane) - 1u);
    int rank = __popc(grp & ((1u << lane) - 1u));
    while (__any_sync(kAll, above != 0u)) {
        const int next = __ffs(above) - 1;
        const double v = __shfl_sync(kAll, val, next < 0 ? lane : next);
        if (next >= 0) val += v;
        above &= __ballot_sync(kAll, !(rank & 1));
        rank >>= 1;
    }
    return val;
}

// Reverse of one Handshake update per CTA at a time, a thread per label: T
// threads, and for more than T labels (BIG, beyond kThreads) several labels per
// thread.  One launch sweeps all iterations, blocks taking the updates from one
// queue in reverse schedule order, the adjoints in versioned entries (as the
// replay, record.cu).  Sums over argmin preimages: within a warp over the lanes
// of equal argmins (peer_sum), the warps' partial sums through shared memory
// (part[w][key], left zero by the reader), added in warp order.
// Bound by the chain of FP64 additions (70 cycles each) and barriers, so nothing
// else is on it: argmins, their groups, descriptor and the next update are
// prepared while the adjoints are waited for, a thread keeps its label's values
// in registers, the three sums have partials of their own (three barriers an
// update), and the three additions to the table's gradient are left to L2 (the
// barriers between them order those that meet in one entry).
// 16 x K_50 with 64 labels, per matching: 10.5 us with a launch each, 8 warps
// and serial group sums, 4.0 us so; 8 edges of up to 21 labels: 7.7 -> 3.3 us.
template <bool BIG>
__global__ void __launch_bounds__(kThreads) bw_sweep_kernel(BwQueue p, const unsigned char *rec_all, double *gtab)
{
    extern __shared__ __align__(16) double sh[];
    __shared__ __align__(16) BwItem s_it[2];  // the update at work and the next one
    __shared__ long long s_g[2];              // their places in the queue
    constexpr int kQ = static_cast<int>(sizeof(BwItem) / sizeof(int4));
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kPer = BIG ? kSweepLabels / kThreads : 1;  // labels per thread
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = T >> 5;
    const int lm = p.lmax;
    double *part3 = sh, *part2 = part3 + W * lm, *part1 = part2 + W * lm;  // [W][lm] each
    const long long total = p.n_items * p.iterations;
    // the records of the update at place g (the last iteration first)
    auto records = [&](const BwItem &it, long long g) {
        return reinterpret_cast<const unsigned short *>(
            rec_all + (p.iterations - 1 - static_cast<long long>(bw_place(p, g).x)) * p.rec_stride + it.rec_off);
    };
    if (tid == 0) s_g[0] = static_cast<long long>(atomicAdd(p.queue, 1ull));
    for (int i = tid; i < 3 * W * lm; i += T) sh[i] = 0.0;
    __syncthreads();
    long long g = s_g[0];
    if (g >= total) return;
    if (tid < kQ)
        reinterpret_cast<int4 *>(&s_it[0])[tid] = __ldg(reinterpret_cast<const int4 *>(p.items + bw_place(p, g).y) + tid);
    __syncthreads();
    unsigned short r1[kPer], r2[kPer], r3[kPer];  // the argmins, requested ahead
    auto request = [&](const BwItem &it, long long at) {
        const unsigned short *rec = records(it, at);
        const int Lu = it.ed.Lu, Lv = it.ed.Lv;
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int j = tid + c * T;
            r1[c] = r2[c] = r3[c] = 0;
            if (j < Lu) {
                r1[c] = rec[j];
                r3[c] = rec[Lu + Lv + j];
            }
            if (j < Lv) r2[c] = rec[Lu + j];
        }
    };
    request(s_it[0], g);
    bool drain = false;
    for (int turn = 0; g < total; ++turn) {
        const BwItem &it = s_it[turn & 1];
        const EdgeDesc ed = it.ed;
        const int Lu = ed.Lu, Lv = ed.Lv;
        const unsigned ve = p.done + bw_place(p, g).x;
        const unsigned vu = ve * static_cast<unsigned>(it.deg_u) + static_cast<unsigned>(it.pos_u);
        const unsigned vv = ve * static_cast<unsigned>(it.deg_v) + static_cast<unsigned>(it.pos_v);
        if (tid == 0) s_g[(turn + 1) & 1] = static_cast<long long>(atomicAdd(p.queue, 1ull));
        double *gt = gtab + ed.toff;
        // recorded indices are < L for finite values; clamp so that no record
        // can address outside the table
        int t1[kPer], s2[kPer], t3[kPer];
        unsigned g1[kPer], g2s[kPer], g3[kPer];
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int j = tid + c * T;
            t1[c] = min(static_cast<int>(r1[c]), Lv - 1);
            t3[c] = min(static_cast<int>(r3[c]), Lv - 1);
            s2[c] = min(static_cast<int>(r2[c]), Lu - 1);
            // (idle lanes never match an active one)
            g1[c] = __match_any_sync(kAll, j < Lu ? t1[c] : -1 - lane);
            g3[c] = __match_any_sync(kAll, j < Lu ? t3[c] : -1 - lane);
            g2s[c] = __match_any_sync(kAll, j < Lv ? s2[c] : -1 - lane);
        }
        double cb[kPer], uhb[kPer], bb[kPer], vhb[kPer];
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int j = tid + c * T;
            cb[c] = uhb[c] = bb[c] = vhb[c] = 0.0;
            if (j < Lu) {
                const double Pu = bw_poll_diff(p, p.agg + ed.au + j, p.msg + ed.mu + j, g > 0 ? vu : vu + p.test_wait, ve,
                                               drain, &uhb[c]);
                cb[c] = uhb[c] + Pu;
            }
            if (j < Lv) {
                double Av;
                const double Pv = bw_poll_diff(p, p.agg + ed.av + j, p.msg + ed.mv + j, vv, ve, drain, &Av);
                bb[c] = Av + Pv;
                vhb[c] = -Pv;
            }
        }
        // a sum's partials: the lowest lane of every group stores its warp's
        auto scatter = [&](const double (&val)[kPer], const unsigned (&grp)[kPer], const int (&key)[kPer], int n,
                           double *part) {
#pragma unroll
            for (int c = 0; c < kPer; ++c) {
                const double sum = peer_sum(val[c], grp[c], lane);
                if (tid + c * T < n && (grp[c] & ((1u << lane) - 1u)) == 0u) {
                    double *const to = &part[warp * lm + key[c]];
                    *to = c > 0 ? *to + sum : sum;
                }
                if (BIG) __syncwarp();  // another lane may lead the same key's next group
            }
        };
        auto gather = [&](double *part, int j) {  // ... and a key's, in warp order
            double acc = 0.0;
            for (int w = 0; w < W; ++w) {
                acc += part[w * lm + j];
                part[w * lm + j] = 0.0;
            }
            return acc;
        };
        // pass 3 reversed: c(s) = theta(s, t3(s)) + beta(t3(s)) + uh(s)
#pragma unroll
        for (int c = 0; c < kPer; ++c)
            if (tid + c * T < Lu) atomicAdd(&gt[static_cast<long long>(tid + c * T) * ed.ld + t3[c]], cb[c]);
        scatter(cb, g3, t3, Lu, part3);
        __syncthreads();
        const long long g2 = s_g[(turn + 1) & 1];
        int4 nrec = make_int4(0, 0, 0, 0);
        if (g2 < total && tid < kQ) nrec = __ldg(reinterpret_cast<const int4 *>(p.items + bw_place(p, g2).y) + tid);
        // beta = vh - b;  b = m2 + vh
        // pass 2 reversed: m2(t) = theta(s2(t), t) + alpha(s2(t))
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int t = tid + c * T;
            if (t < Lv) {
                const double acc = gather(part3, t);
                bb[c] = bb[c] - acc;
                vhb[c] = (vhb[c] + acc) + bb[c];
                atomicAdd(&gt[static_cast<long long>(s2[c]) * ed.ld + t], bb[c]);
            }
        }
        scatter(bb, g2s, s2, Lv, part2);
        if (tid < kQ) reinterpret_cast<int4 *>(&s_it[(turn + 1) & 1])[tid] = nrec;
        __syncthreads();
        if (g2 < total) request(s_it[(turn + 1) & 1], g2);
        // alpha = uh - a;  a = (m1 + uh) / 2
        // pass 1 reversed: m1(s) = theta(s, t1(s)) + vh(t1(s))
        double m1b[kPer];
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int s = tid + c * T;
            m1b[c] = 0.0;
            if (s < Lu) {
                const double acc = gather(part2, s);
                m1b[c] = -0.5 * acc;
                uhb[c] = (uhb[c] + acc) + m1b[c];
                st_se(p.agg + ed.au + s, se64_make(uhb[c], vu + 1u));
                atomicAdd(&gt[static_cast<long long>(s) * ed.ld + t1[c]], m1b[c]);
            }
        }
        scatter(m1b, g1, t1, Lu, part1);
        __syncthreads();
        // uh = agg_u - phi_{v->u}, vh = agg_v - phi_{u->v} (values before the update)
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int t = tid + c * T;
            if (t < Lv) {
                vhb[c] += gather(part1, t);
                st_se(p.agg + ed.av + t, se64_make(vhb[c], vv + 1u));
            }
        }
        // The messages are read by this edge's next update only, which adds to
        // the same table: the fence orders its additions after these.
        __threadfence();
#pragma unroll
        for (int c = 0; c < kPer; ++c) {
            const int j = tid + c * T;
            if (j < Lv) st_se(p.msg + ed.mv + j, se64_make(-vhb[c], ve + 1u));
            if (j < Lu) st_se(p.msg + ed.mu + j, se64_make(-uhb[c], ve + 1u));
        }
        g = g2;
    }
}

__global__ void unpack_grad_kernel(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes,
                                   const long long *pair_base, const long long *unary_base, const double *gtab,
                                   const double *adj_agg, float *grad_pair, float *grad_un)
{
    // a warp per row; rows without padding are one run (no index per entry)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    for (int e = blockIdx.x; e < n_edges; e += gridDim.x) {
        const EdgeDesc ed = edges[e];
        float *dst = grad_pair + pair_base[ed.model] + ed.poff;
        const double *src = gtab + ed.toff;
        if (ed.Lv == ed.ld) {
            const long long n = static_cast<long long>(ed.Lu) * ed.Lv;
            if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
                for (long long i = 4LL * threadIdx.x; i < n; i += 4LL * blockDim.x) {
                    const double2 a = *reinterpret_cast<const double2 *>(src + i);
                    const double2 b = *reinterpret_cast<const double2 *>(src + i + 2);
                    *reinterpret_cast<float4 *>(dst + i) =
                        make_float4(static_cast<float>(a.x), static_cast<float>(a.y), static_cast<float>(b.x),
                                    static_cast<float>(b.y));
                }
            } else {
                for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = static_cast<float>(src[i]);
            }
        } else {
            for (int s = warp; s < ed.Lu; s += W)
                for (int t = lane; t < ed.Lv; t += 32)
                    dst[static_cast<long long>(s) * ed.Lv + t] =
                        static_cast<float>(src[static_cast<long long>(s) * ed.ld + t]);
        }
    }
    for (int u = blockIdx.x; u < n_nodes; u += gridDim.x) {
        const NodeDesc nd = nodes[u];
        for (int s = threadIdx.x; s < nd.L; s += blockDim.x)
            grad_un[unary_base[nd.model] + nd.uoff + s] = static_cast<float>(adj_agg[nd.aoff + s]);
    }
}

}  // namespace

cudaError_t launch_bw_init(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes, const float *tab,
                           const double *agg, const double *msg, const float *dD, double *adj_agg, double *adj_msg,
                           double *gtab, int lmax, cudaStream_t st)
{
    if (n_nodes > 0) {
        bw_init_nodes_kernel<<<std::max(1, std::min(65535, (n_nodes + 7) / 8)), kThreads, 0, st>>>(nodes, n_nodes, agg,
                                                                                                  dD, adj_agg);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (n_edges > 0) {
        const int lw = (lmax + 3) & ~3;
        const bool warp = scan_by_warps(lw, n_edges);
        const size_t smem = 2 * sizeof(float) * static_cast<size_t>(lw) * (warp ? kThreads / 32 : 1) +
                            (kThreads / 32) * kScanChunks * sizeof(int);
        const auto kernel = warp ? bw_init_edges_kernel<32> : bw_init_edges_kernel<kThreads>;
        if (smem > 48 * 1024) {
            cudaError_t e = raise_smem_limit(kernel, smem);
            if (e != cudaSuccess) return e;
        }
        const int blocks = warp ? std::min((n_edges + 7) / 8, 152 * 16) : std::min(n_edges, 1 << 20);
        kernel<<<blocks, kThreads, smem, st>>>(edges, n_edges, tab, msg, dD, lw, adj_msg, gtab);
        return cudaGetLastError();
    }
    return cudaSuccess;
}

static int bw_threads(int lmax) { return std::min(kThreads, (lmax + 31) & ~31); }

size_t bw_sweep_smem_bytes(int lmax)
{
    return static_cast<size_t>(lmax) * 3 * (bw_threads(lmax) / 32) * sizeof(double);
}

cudaError_t launch_bw_sweep(const BwQueue &p, int max_items, const unsigned char *rec, double *gtab, cudaStream_t st)
{
    if (p.n_items <= 0 || p.iterations <= 0) return cudaSuccess;
    const size_t smem = bw_sweep_smem_bytes(p.lmax);
    const int threads = bw_threads(p.lmax);
    const auto kernel = p.lmax <= kThreads ? bw_sweep_kernel<false> : bw_sweep_kernel<true>;
    int per_sm = 0;
    cudaError_t e = cudaMemsetAsync(p.queue, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = raise_smem_limit(kernel, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    const int blocks = std::max(1, std::min(per_sm * 152, 2 * max_items));
    kernel<<<blocks, threads, smem, st>>>(p, rec, gtab);
    return cudaGetLastError();
}

cudaError_t launch_unpack_grad(const EdgeDesc *edges, int n_edges, const NodeDesc *nodes, int n_nodes,
                               const long long *pair_base, const long long *unary_base, const double *gtab,
                               const double *adj_agg, float *grad_pair, float *grad_un, cudaStream_t st)
{
    const int grid = std::max(1, std::min(std::max(n_edges, n_nodes), 1 << 20));
    unpack_grad_kernel<<<grid, kThreads, 0, st>>>(edges, n_edges, nodes, n_nodes, pair_base, unary_base, gtab, adj_agg,
                                                  grad_pair, grad_un);
    return cudaGetLastError();
}

}  // namespace mplpp

using namespace mplpp;

namespace {

mplpp_status bfail(mplpp_solver *s, mplpp_status st, const std::string &m)
{
    s->err = m;
    return st;
}

#define BCK(call)                                                                                          \
    do {                                                                                                   \
        cudaError_t e_ = (call);                                                                           \
        if (e_ != cudaSuccess) return bfail(s, MPLPP_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

constexpr long long kRecordAllBytes = 1LL << 30;  // argmin records kept for a one-replay backward

template <typename T>
cudaError_t ensure(mplpp_solver *s, T **p, size_t count)
{
    if (*p) return cudaSuccess;
    return s->alloc(p, count);
}

// One FP64 iteration, a launch per matching (screened kernel when the largest
// table fits shared memory, tab_floats > 0; else all-FP64 scans).
cudaError_t rec64_iteration(mplpp_solver *s, unsigned char *rec, int lmax, long long tab_floats, cudaStream_t st)
{
    for (int ph = 0; ph < s->P; ++ph) {
        const int *items = s->d_phase_edges + s->phase_off[ph];
        const int n = s->phase_off[ph + 1] - s->phase_off[ph];
        const int f = s->phase_off[ph];
        cudaError_t e = tab_floats > 0 ? launch_rec_screen_phase(s->d_sched_desc + f, n, s->d_tab, s->d_agg64,
                                                                 s->d_msg64, rec, s->d_sched_rec_off + f, lmax,
                                                                 tab_floats, st)
                                       : launch_rec64_phase(s->d_edges, items, n, s->d_tab, s->d_agg64, s->d_msg64, rec,
                                                            s->d_rec_off, lmax, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

extern "C" mplpp_status mplpp_backward(mplpp_solver *s, const float *dD, float *grad_unary, float *grad_pairwise)
{
    if (!s || !dD || !grad_unary || (s->sum_pair > 0 && !grad_pairwise)) return MPLPP_E_INVALID;
    s->err.clear();
    const int k = s->opt.record_every;
    if (k <= 0) return bfail(s, MPLPP_E_STATE, "backward needs options.record_every > 0");
    if (!s->history_valid)
        return bfail(s, MPLPP_E_STATE, "the state was loaded: the iterations since phi = 0 are unknown");
    const long long Ttot = s->iterations;
    const int nm = static_cast<int>(s->models.size());
    cudaStream_t st = s->stream;
    int lmax = 1;
    for (auto &nd : s->h_nodes) lmax = std::max(lmax, nd.L);
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->device);
    if (lmax > kSweepLabels)
        return bfail(s, MPLPP_E_UNSUPPORTED, "backward supports at most " + std::to_string(kSweepLabels) + " labels per node");
    long long tab_floats = 0;  // the screened replay stages the largest table in shared memory
    for (auto &ed : s->h_edges) tab_floats = std::max(tab_floats, 1LL * ed.Lu * (ed.ld | 1));
    if ((s->opt.test_backward & 1) || rec_screen_smem_bytes(lmax, tab_floats) > static_cast<size_t>(optin))
        tab_floats = 0;

    // buffers
    if (!s->d_rec_off) {
        std::vector<long long> off(s->EE);
        long long acc = 0;
        for (int e = 0; e < s->EE; ++e) {
            off[e] = acc;
            acc += 2LL * (2LL * s->h_edges[e].Lu + s->h_edges[e].Lv);
            acc = (acc + 3) & ~3LL;
        }
        s->rec_stride = std::max(4LL, acc);
        // the same in schedule order, with the edges' descriptors: a block of
        // the replay reads both at once; and the queue kernels' items, for the
        // replay in schedule order, for the reverse sweep from its end
        std::vector<EdgeDesc> sd(s->EE);
        std::vector<long long> so(s->EE);
        std::vector<BwItem> fwd(s->EE), bwd(s->EE);
        std::vector<int> pos(s->N, 0);
        for (int j = 0; j < s->EE; ++j) {
            sd[j] = s->h_edges[s->phase_edges[j]];
            so[j] = off[s->phase_edges[j]];
            fwd[j] = BwItem{sd[j], pos[sd[j].gu]++, pos[sd[j].gv]++, 0, 0, so[j]};
        }
        for (int j = 0; j < s->EE; ++j) {  // pos: every node's updates per iteration by now
            BwItem &f = fwd[j];
            f.deg_u = pos[f.ed.gu];
            f.deg_v = pos[f.ed.gv];
            BwItem &b = bwd[s->EE - 1 - j];
            b = f;
            b.pos_u = f.deg_u - 1 - f.pos_u;
            b.pos_v = f.deg_v - 1 - f.pos_v;
        }
        BCK(s->alloc(&s->d_bw_fwd, std::max(1, s->EE)));
        BCK(s->alloc(&s->d_bw_rev, std::max(1, s->EE)));
        BCK(s->alloc(&s->d_bw_queue, 1));
        BCK(cudaMemcpyAsync(s->d_bw_fwd, fwd.data(), sizeof(BwItem) * s->EE, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(s->d_bw_rev, bwd.data(), sizeof(BwItem) * s->EE, cudaMemcpyHostToDevice, st));
        BCK(s->alloc(&s->d_rec_off, std::max(1, s->EE)));
        BCK(s->alloc(&s->d_sched_desc, std::max(1, s->EE)));
        BCK(s->alloc(&s->d_sched_rec_off, std::max(1, s->EE)));
        BCK(cudaMemcpyAsync(s->d_rec_off, off.data(), sizeof(long long) * s->EE, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(s->d_sched_desc, sd.data(), sizeof(EdgeDesc) * s->EE, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(s->d_sched_rec_off, so.data(), sizeof(long long) * s->EE, cudaMemcpyHostToDevice, st));
        BCK(cudaStreamSynchronize(st));
    }
    if (!s->d_pbase) {
        std::vector<long long> pb(nm), ub(nm);
        long long a = 0, b = 0;
        for (int m = 0; m < nm; ++m) {
            pb[m] = a;
            ub[m] = b;
            a += s->models[m].pair_size;
            b += s->models[m].unary_size;
        }
        BCK(s->alloc(&s->d_pbase, nm));
        BCK(s->alloc(&s->d_ubase, nm));
        BCK(cudaMemcpyAsync(s->d_pbase, pb.data(), sizeof(long long) * nm, cudaMemcpyHostToDevice, st));
        BCK(cudaMemcpyAsync(s->d_ubase, ub.data(), sizeof(long long) * nm, cudaMemcpyHostToDevice, st));
        BCK(cudaStreamSynchronize(st));
    }
    BCK(ensure(s, &s->d_agg64, s->aggN));
    BCK(ensure(s, &s->d_msg64, s->msgN));
    BCK(ensure(s, &s->d_adj_agg, s->aggN));
    BCK(ensure(s, &s->d_adj_msg, s->msgN));
    BCK(ensure(s, &s->d_gtab, s->tabN));
    BCK(ensure(s, &s->d_adj_agg_v, s->aggN));
    BCK(ensure(s, &s->d_adj_msg_v, s->msgN));
    const bool queued = tab_floats > 0 && rec_group_fits(lmax);  // the replay's form
    if (queued) {
        BCK(ensure(s, &s->d_agg64_v, s->aggN));
        BCK(ensure(s, &s->d_msg64_v, s->msgN));
    }
    BwQueue q = {};
    q.n_items = s->EE;
    q.rec_stride = s->rec_stride;
    q.queue = s->d_bw_queue;
    q.err = s->d_err;
    q.spin_limit = s->own_wait_limit();
    q.test_wait = s->opt.test_unreachable_wait ? 1u : 0u;
    q.lmax = lmax;
    // `n` iterations of the FP64 replay, `done` of them already in the state; rec:
    // the records of the first one, or nullptr
    // (a launch takes at most 2^31 updates)
    const long long most = std::max(1LL, (1LL << 31) / std::max(1, s->EE) - 1);
    auto replay = [&](long long n, long long done, unsigned char *rec) -> cudaError_t {
        if (queued) {
            BwQueue r = q;
            r.items = s->d_bw_fwd;
            r.agg = s->d_agg64_v;
            r.msg = s->d_msg64_v;
            for (long long i = 0; i < n; i += most) {
                r.iterations = static_cast<int>(std::min(most, n - i));
                r.done = static_cast<unsigned>(done + i);
                cudaError_t e =
                    launch_rec_queue(r, s->max_phase, s->d_tab, rec ? rec + i * s->rec_stride : nullptr, st);
                if (e != cudaSuccess) return e;
            }
            return cudaSuccess;
        }
        for (long long i = 0; i < n; ++i) {
            cudaError_t e = rec64_iteration(s, rec ? rec + i * s->rec_stride : nullptr, lmax, tab_floats, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    };
    auto to_entries = [&]() -> cudaError_t {  // the plain FP64 state into the replay's form, from update count 0
        if (!queued) return cudaSuccess;
        cudaError_t e = launch_to_entries(s->d_agg64, s->d_agg64_v, s->aggN, st);
        return e != cudaSuccess ? e : launch_to_entries(s->d_msg64, s->d_msg64_v, s->msgN, st);
    };
    auto from_entries = [&](double *agg, double *msg) -> cudaError_t {  // ... and the state out of it
        if (!queued) {
            cudaError_t e = cudaSuccess;
            if (agg != s->d_agg64) {
                e = cudaMemcpyAsync(agg, s->d_agg64, sizeof(double) * s->aggN, cudaMemcpyDeviceToDevice, st);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(msg, s->d_msg64, sizeof(double) * s->msgN, cudaMemcpyDeviceToDevice, st);
            }
            return e;
        }
        cudaError_t e = launch_from_entries(s->d_agg64_v, agg, s->aggN, st);
        return e != cudaSuccess ? e : launch_from_entries(s->d_msg64_v, msg, s->msgN, st);
    };
    // When the argmin records of every iteration fit kRecordAllBytes, the one
    // replay records them all (no checkpoints, no second replay); otherwise a
    // state checkpoint every k iterations and each segment replayed again,
    // recording, before its reverse sweep.
    const bool record_all = Ttot > 0 && s->rec_stride * Ttot <= kRecordAllBytes && !(s->opt.test_backward & 2);
    const long long rec_slots = record_all ? Ttot : k;
    if (s->rec_slots < rec_slots) {
        BCK(s->release(s->d_rec));
        s->d_rec = nullptr;
        BCK(s->alloc(&s->d_rec, static_cast<size_t>(s->rec_stride) * rec_slots));
        s->rec_slots = rec_slots;
    }
    BCK(ensure(s, &s->d_dD, nm));
    const long long nseg = record_all ? 0 : (Ttot + k - 1) / k;
    while (static_cast<long long>(s->ckpt64.size()) < nseg) {
        double *c = nullptr;
        BCK(s->alloc(&c, static_cast<size_t>(s->aggN + s->msgN)));
        s->ckpt64.push_back(c);
    }

    // FP64 replay from phi = 0: recording every iteration, or a checkpoint every k
    BCK(launch_widen(s->d_un0, s->d_agg64, s->aggN, st));
    BCK(cudaMemsetAsync(s->d_msg64, 0, sizeof(double) * s->msgN, st));
    BCK(to_entries());
    if (record_all) {
        BCK(replay(Ttot, 0, s->d_rec));
    } else {
        for (long long it = 0; it < Ttot; it += k) {
            BCK(from_entries(s->ckpt64[it / k], s->ckpt64[it / k] + s->aggN));
            BCK(replay(std::min<long long>(k, Ttot - it), it, nullptr));
        }
    }
    BCK(from_entries(s->d_agg64, s->d_msg64));
    BCK(cudaMemcpyAsync(s->d_dD, dD, sizeof(float) * nm, cudaMemcpyHostToDevice, st));
    BCK(cudaMemsetAsync(s->d_adj_agg, 0, sizeof(double) * s->aggN, st));
    BCK(cudaMemsetAsync(s->d_adj_msg, 0, sizeof(double) * s->msgN, st));
    BCK(cudaMemsetAsync(s->d_gtab, 0, sizeof(double) * s->tabN, st));
    BCK(launch_bw_init(s->d_edges, s->EE, s->d_nodes, s->N, s->d_tab, s->d_agg64, s->d_msg64, s->d_dD, s->d_adj_agg,
                       s->d_adj_msg, s->d_gtab, lmax, st));

    // the reverse sweep, on the adjoints in entries; `swept` iterations are done
    BCK(launch_to_entries(s->d_adj_agg, s->d_adj_agg_v, s->aggN, st));
    BCK(launch_to_entries(s->d_adj_msg, s->d_adj_msg_v, s->msgN, st));
    long long swept = 0;
    auto sweep = [&](long long n) -> cudaError_t {
        BwQueue r = q;
        r.items = s->d_bw_rev;
        r.agg = s->d_adj_agg_v;
        r.msg = s->d_adj_msg_v;
        for (long long left = n; left > 0;) {
            r.iterations = static_cast<int>(std::min(most, left));
            left -= r.iterations;
            r.done = static_cast<unsigned>(swept);
            swept += r.iterations;
            cudaError_t e = launch_bw_sweep(r, s->max_phase, s->d_rec + left * s->rec_stride, s->d_gtab, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    };
    if (record_all) BCK(sweep(Ttot));
    for (long long j = nseg - 1; j >= 0; --j) {
        const long long len = std::min<long long>(k, Ttot - j * k);
        BCK(cudaMemcpyAsync(s->d_agg64, s->ckpt64[j], sizeof(double) * s->aggN, cudaMemcpyDeviceToDevice, st));
        BCK(cudaMemcpyAsync(s->d_msg64, s->ckpt64[j] + s->aggN, sizeof(double) * s->msgN, cudaMemcpyDeviceToDevice,
                            st));
        BCK(to_entries());
        BCK(replay(len, 0, s->d_rec));
        BCK(sweep(len));
    }
    BCK(launch_from_entries(s->d_adj_agg_v, s->d_adj_agg, s->aggN, st));
    float *d_gu = nullptr, *d_gp = nullptr;
    float *gu = grad_unary, *gp = grad_pairwise;
    if (!s->opt.inputs_on_device) {
        BCK(cudaMalloc(&d_gu, sizeof(float) * std::max(1LL, s->sum_unary)));
        cudaError_t e = cudaMalloc(&d_gp, sizeof(float) * std::max(1LL, s->sum_pair));
        if (e != cudaSuccess) {
            cudaFree(d_gu);
            return bfail(s, MPLPP_E_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
        }
        gu = d_gu;
        gp = d_gp;
    }
    cudaError_t e = launch_unpack_grad(s->d_edges, s->EE, s->d_nodes, s->N, s->d_pbase, s->d_ubase, s->d_gtab,
                                       s->d_adj_agg, gp, gu, st);
    if (e == cudaSuccess && !s->opt.inputs_on_device) {
        e = cudaMemcpyAsync(grad_unary, d_gu, sizeof(float) * s->sum_unary, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && s->sum_pair)
            e = cudaMemcpyAsync(grad_pairwise, d_gp, sizeof(float) * s->sum_pair, cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (d_gu) cudaFree(d_gu);
    if (d_gp) cudaFree(d_gp);
    if (e != cudaSuccess) return bfail(s, MPLPP_E_CUDA, std::string("backward: ") + cudaGetErrorString(e));
    return mplpp_sync(s);
}
