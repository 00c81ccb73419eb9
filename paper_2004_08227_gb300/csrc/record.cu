// record.cu -- the Handshake update in FP64, optionally recording argmins, for
// the backward pass.
//
// The gradient of D_T is the gradient of one linear piece of a piecewise
// linear function, selected by the argmins of the forward.  A binary32
// trajectory drifts from the exact one by ~1e-6 relative over many
// iterations, enough to select different pieces at near-ties; the backward
// therefore replays the iterations in binary64 (same message-form arithmetic
// and association as handshake.cu, on a double copy of the state), so that its
// argmins are those of the exact-arithmetic trajectory up to binary64 rounding.
// One CTA per edge of a matching; one launch per matching (label counts up to
// 128: one launch for all iterations, rec_queue_kernel).
#include <algorithm>
#include <climits>

#include "backward.h"
#include "kernels.h"

namespace mplpp {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void amin_d(double &m, int &i, double v, int j)
{
    if (v < m || (v == m && j < i)) {
        m = v;
        i = j;
    }
}

__device__ __forceinline__ void warp_amin_d(double &m, int &i)
{
    for (int o = 16; o > 0; o >>= 1) {
        const double om = __shfl_xor_sync(0xffffffffu, m, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        amin_d(m, i, om, oi);
    }
}

template <bool REC>
__global__ void __launch_bounds__(kThreads) rec64_phase_kernel(const EdgeDesc *edges, const int *items,
                                                               const float *tab, double *agg, double *msg,
                                                               unsigned char *rec, const long long *rec_off, int lmax)
{
    extern __shared__ __align__(16) double shd[];
    double *uh = shd;           // [Lu]
    double *alpha = uh + lmax;  // [Lu]
    double *vh = alpha + lmax;  // [Lv]
    double *bv = vh + lmax;     // [Lv]
    double *beta = bv + lmax;   // [Lv]
    const int e = items[blockIdx.x];
    const EdgeDesc ed = edges[e];
    const int Lu = ed.Lu, Lv = ed.Lv, ld = ed.ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const float *th = tab + ed.toff;
    unsigned short *t1 = nullptr, *s2 = nullptr, *t3 = nullptr;
    if (REC) {
        t1 = reinterpret_cast<unsigned short *>(rec + rec_off[e]);
        s2 = t1 + Lu;
        t3 = s2 + Lv;
    }
    for (int s = tid; s < Lu; s += blockDim.x) uh[s] = agg[ed.au + s] - msg[ed.mu + s];
    for (int t = tid; t < Lv; t += blockDim.x) vh[t] = agg[ed.av + t] - msg[ed.mv + t];
    __syncthreads();
    // pass 1: a(s) = 1/2 (min_t [theta(s,t) + vh(t)] + uh(s)),  alpha = uh - a
    for (int s = warp; s < Lu; s += nw) {
        double m = INFINITY;
        int mi = INT_MAX;
        for (int t = lane; t < Lv; t += 32) {
            const double v = static_cast<double>(th[static_cast<long long>(s) * ld + t]) + vh[t];
            if (v < m) {
                m = v;
                mi = t;
            }
        }
        warp_amin_d(m, mi);
        if (lane == 0) {
            const double a = 0.5 * (m + uh[s]);
            alpha[s] = uh[s] - a;
            if (REC) t1[s] = static_cast<unsigned short>(mi);
        }
    }
    __syncthreads();
    // pass 2: b(t) = min_s [theta(s,t) + alpha(s)] + vh(t),  beta = vh - b
    for (int t = tid; t < Lv; t += blockDim.x) {
        double m = INFINITY;
        int mi = 0;
        for (int s = 0; s < Lu; ++s) {
            const double v = static_cast<double>(th[static_cast<long long>(s) * ld + t]) + alpha[s];
            if (v < m) {
                m = v;
                mi = s;
            }
        }
        const double b = m + vh[t];
        bv[t] = b;
        beta[t] = vh[t] - b;
        if (REC) s2[t] = static_cast<unsigned short>(mi);
    }
    __syncthreads();
    // pass 3: c(s) = min_t [theta(s,t) + beta(t)] + uh(s)
    for (int s = warp; s < Lu; s += nw) {
        double m = INFINITY;
        int mi = INT_MAX;
        for (int t = lane; t < Lv; t += 32) {
            const double v = static_cast<double>(th[static_cast<long long>(s) * ld + t]) + beta[t];
            if (v < m) {
                m = v;
                mi = t;
            }
        }
        warp_amin_d(m, mi);
        if (lane == 0) {
            const double c = m + uh[s];
            agg[ed.au + s] = c;
            msg[ed.mu + s] = c - uh[s];
            if (REC) t3[s] = static_cast<unsigned short>(mi);
        }
    }
    for (int t = tid; t < Lv; t += blockDim.x) {
        agg[ed.av + t] = bv[t];
        msg[ed.mv + t] = bv[t] - vh[t];
    }
}

// ---------------------------------------------------------------------------
// The same update with FP64 work only where it can decide a minimum.  GB300
// runs FP64 at a small fraction of its FP32 rate, so every minimization is
// first screened in FP32 and only its surviving candidates are evaluated in
// FP64, with exactly the FP64 expression of rec64_phase_kernel above; the
// minima and argmins are therefore bit for bit those of the all-FP64 kernel.
//
// Screen of min_j V(j), V(j) = theta(j) + x(j) (x the FP64 vector of the
// minimization, theta the FP32 table entries along a row or a column):
//   w(j) = fl32(x(j) - x(0)) (the difference taken in FP64),
//   c(j) = fl32(theta(j) + w(j)).
// With D = max_j |w(j)| and h = max_j |theta(j)| over the row / column,
//   |c(j) - (theta(j) + w(j))| <= 2^-24 (h + D),
//   |w(j) - (x(j) - x(0))|     <= 2^-24 D (1 + 2^-24) + 2^-53 |x(j) - x(0)|,
// so |c(j) - (V(j) - x(0))| <= 2^-22 (h + D) = e1 (a factor 2 to spare); and
// the FP64 value v(j) = fl64(theta(j) + x(j)) errs from V(j) by at most
// 2^-53 (h + D + |x(0)|)(1 + 2^-22) <= 2^-50 (h + D + |x(0)|) = e2.  If j* is
// the FP64 argmin and c(jc) the FP32 minimum, then
//   c(j*) <= V(j*) - x(0) + e1 <= v(j*) - x(0) + e1 + e2
//         <= v(jc) - x(0) + e1 + e2 <= c(jc) + 2 e1 + 2 e2,
// so every j with c(j) <= c(jc) + 2 e1 + 2 e2 (threshold rounded upwards) is a
// candidate, and the FP64 argmin (the lowest index among equal FP64 minima)
// is among the candidates.  One group of G threads (a power of two, G lines
// per block of threads; the groups of a warp hold consecutive lines) handles
// a line: both FP32 scans and the bound from the line's own h and
// max |w(j)|.  The warp's candidates are appended to a per-warp list and
// evaluated in FP64 32 at a time (one candidate per lane: GB300 issues an FP64
// instruction at the cost of a full warp however few lanes are active), and
// merged into their line's minimum with 64-bit shared-memory atomics on an
// order-preserving key (value first, then the lowest index among equal
// values), so neither the order of the list nor of the lanes matters.  A warp
// whose list overflows scans its lines in FP64 entirely.  One block barrier
// per pass.  The table is staged in shared memory with an odd row stride.
namespace {

constexpr int kScrThreads = 256;
constexpr int kWarpCands = 128;  // candidates per warp and pass
constexpr int kSpanReg = 16;     // a thread's sums of a line kept in registers (up to this many)

__device__ __forceinline__ unsigned long long order_key(double v)
{
    unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
    b = (b << 1) ? b : 0ull;  // -0 -> +0: equal values get equal keys
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__device__ __forceinline__ double key_value(unsigned long long k)
{
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double(static_cast<long long>(b));
}

// m(i) = min_j [theta(i, j) + x(j)], j < len, for every line i < n (rows of the
// staged table when ROWS, else columns), with its lowest argmin; w(j) =
// fl32(x(j) - x(0)).  key / arg: [n] per-line scratch; cand: this warp's list
// [kWarpCands].  emit(i, m, argmin) runs on the line group's first thread.
template <bool ROWS, typename F>
__device__ __forceinline__ void screened_lines(const float *tab, int ldp, int n, int len, const double *xv,
                                               const float *w, unsigned long long *key, int *arg, int2 *cand, F emit)
{
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    int G = 32;
    while (G > 1 && G * n > T) G >>= 1;
    const int k = tid & (G - 1), g0 = tid / G, ng = T / G;
    const float ax0 = __double2float_ru(fabs(xv[0]));
    auto th = [&](int i, int j) { return ROWS ? tab[i * ldp + j] : tab[j * ldp + i]; };
    const int span = (len + G - 1) / G;  // elements of a line per thread
    const bool reg = span <= kSpanReg;
    for (int base = 0; base < n; base += ng) {  // the same trip count in every thread
        const int i = base + g0;
        const bool on = i < n;
        float mn = INFINITY, h = 0.f, d = 0.f;
        float sv[kSpanReg];  // the FP32 sums, for the candidate test
#pragma unroll
        for (int r = 0; r < kSpanReg; ++r) {
            const int j = k + r * G;
            sv[r] = INFINITY;
            if (on && j < len) {
                const float t = th(i, j);
                const float wj = w[j];
                sv[r] = t + wj;
                mn = fminf(mn, sv[r]);
                h = fmaxf(h, fabsf(t));
                d = fmaxf(d, fabsf(wj));
            }
        }
        if (on)
            for (int j = k + kSpanReg * G; j < len; j += G) {
                const float t = th(i, j);
                const float wj = w[j];
                mn = fminf(mn, t + wj);
                h = fmaxf(h, fabsf(t));
                d = fmaxf(d, fabsf(wj));
            }
        for (int o = G >> 1; o > 0; o >>= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            h = fmaxf(h, __shfl_xor_sync(0xffffffffu, h, o));
            d = fmaxf(d, __shfl_xor_sync(0xffffffffu, d, o));
        }
        // c(jc) + 2 e1 + 2 e2, every operation rounded upwards (d bounds |w| on the line)
        const float e1 = __fmul_ru(0x1p-22f, __fadd_ru(h, d));
        const float e2 = __fmul_ru(0x1p-50f, __fadd_ru(__fadd_ru(h, d), ax0));
        const float thr = __fadd_ru(__fadd_ru(mn, __fmul_ru(2.f, e1)), __fadd_ru(__fmul_ru(2.f, e2), 0x1p-126f));
        if (on && k == 0) {
            key[i] = ~0ull;
            arg[i] = INT_MAX;
        }
        // the warp's candidates into its list (warp-uniform trip count; the
        // list's order does not matter)
        int nc = 0;
        bool over = false;
        if (reg) {
            // a mask of the thread's candidates, a prefix sum of the counts over the warp
            unsigned m = 0u;
#pragma unroll
            for (int r = 0; r < kSpanReg; ++r)  // +inf beyond the line; a thread without a line has no finite thr
                if (on && sv[r] <= thr) m |= 1u << r;
            const int cnt = __popc(m);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            nc = __shfl_sync(0xffffffffu, incl, 31);
            for (int slot = incl - cnt; m; m &= m - 1u, ++slot)
                if (slot < kWarpCands) cand[slot] = make_int2(i, k + (__ffs(m) - 1) * G);
        } else {
            for (int r = 0; r < span; ++r) {
                const int j = k + r * G;
                const bool c = on && j < len && th(i, j) + w[j] <= thr;
                const unsigned mask = __ballot_sync(0xffffffffu, c);
                const int slot = nc + __popc(mask & ((1u << lane) - 1u));
                if (c && slot < kWarpCands) cand[slot] = make_int2(i, j);
                nc += __popc(mask);
            }
        }
        if (nc > kWarpCands) {
            over = true;
            nc = 0;
        }
        __syncwarp();
        if (!over) {
            // FP64 values, 32 candidates per instruction, merged per line; the
            // keys stay in registers for the argmin step (FP64 is computed once)
            unsigned long long kv[kWarpCands / 32];
#pragma unroll
            for (int r = 0; r < kWarpCands / 32; ++r) {
                const int c = lane + 32 * r;
                if (c < nc) {
                    const int2 q = cand[c];
                    kv[r] = order_key(static_cast<double>(th(q.x, q.y)) + xv[q.y]);
                    atomicMin(&key[q.x], kv[r]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kWarpCands / 32; ++r) {
                const int c = lane + 32 * r;
                if (c < nc) {
                    const int2 q = cand[c];
                    if (kv[r] == key[q.x]) atomicMin(&arg[q.x], q.y);
                }
            }
            __syncwarp();
        } else if (on && k == 0) {
            // too many near-ties in this warp's lines: every element in FP64
            double m = INFINITY;
            int mi = 0;
            for (int j = 0; j < len; ++j) {
                const double v = static_cast<double>(th(i, j)) + xv[j];
                if (v < m) {
                    m = v;
                    mi = j;
                }
            }
            key[i] = order_key(m);
            arg[i] = mi;
        }
        __syncwarp();
        if (on && k == 0) emit(i, key_value(key[i]), arg[i]);
    }
}

template <bool REC>
// descs, rec_off: the matching's edges and their record offsets, in schedule
// order (one independent load each per block)
__global__ void __launch_bounds__(kScrThreads, 4) rec_screen_kernel(const EdgeDesc *descs, const float *tab,
                                                                 double *agg, double *msg, unsigned char *rec,
                                                                 const long long *rec_off, int lmax)
{
    extern __shared__ __align__(16) double shd[];
    const EdgeDesc ed = descs[blockIdx.x];
    const int Lu = ed.Lu, Lv = ed.Lv, ld = ed.ld, ldp = ld | 1;
    const int T = blockDim.x, tid = threadIdx.x, warp = tid >> 5;
    double *uh = shd, *vh = uh + lmax, *al = vh + lmax, *be = al + lmax, *bv = be + lmax;
    unsigned long long *key = reinterpret_cast<unsigned long long *>(bv + lmax);  // [lmax] per-line minima
    int2 *cand = reinterpret_cast<int2 *>(key + lmax) + warp * kWarpCands;      // this warp's list
    int *arg = reinterpret_cast<int *>(reinterpret_cast<int2 *>(key + lmax) + (kScrThreads / 32) * kWarpCands);
    float *w = reinterpret_cast<float *>(arg + lmax);  // [lmax] the current pass's shifted vector
    float *st = w + lmax;                              // [Lu][ldp] staged table
    unsigned short *t1 = nullptr, *s2 = nullptr, *t3 = nullptr;
    if (REC) {
        t1 = reinterpret_cast<unsigned short *>(rec + rec_off[blockIdx.x]);
        s2 = t1 + Lu;
        t3 = s2 + Lv;
    }
    // the node vectors (requested first), the table (16-byte chunks, a
    // thread's next eight requested before any is stored, so the loads
    // overlap), shifted vh
    const double vh0 = agg[ed.av] - msg[ed.mv];
    for (int s = tid; s < Lu; s += T) uh[s] = agg[ed.au + s] - msg[ed.mu + s];
    for (int t = tid; t < Lv; t += T) vh[t] = agg[ed.av + t] - msg[ed.mv + t];
    const float4 *th4 = reinterpret_cast<const float4 *>(tab + ed.toff);
    const int Q = ld >> 2, nq = Lu * Q;
    for (int base = tid; base < nq; base += 8 * T) {
        float4 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (base + r * T < nq) v[r] = th4[base + r * T];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int c = base + r * T;
            if (c < nq) {
                const int s = c / Q;
                float *d = st + s * ldp + 4 * (c - s * Q);
                d[0] = v[r].x;
                d[1] = v[r].y;
                d[2] = v[r].z;
                d[3] = v[r].w;
            }
        }
    }
    for (int t = tid; t < Lv; t += T) w[t] = static_cast<float>(vh[t] - vh0);
    __syncthreads();
    // pass 1: a(s) = 1/2 (min_t [theta(s,t) + vh(t)] + uh(s)),  alpha = uh - a
    screened_lines<true>(st, ldp, Lu, Lv, vh, w, key, arg, cand, [&](int s, double m, int mi) {
        const double a = 0.5 * (m + uh[s]);
        al[s] = uh[s] - a;
        if (REC) t1[s] = static_cast<unsigned short>(mi);
    });
    __syncthreads();
    for (int s = tid; s < Lu; s += T) w[s] = static_cast<float>(al[s] - al[0]);
    __syncthreads();
    // pass 2: b(t) = min_s [theta(s,t) + alpha(s)] + vh(t),  beta = vh - b
    screened_lines<false>(st, ldp, Lv, Lu, al, w, key, arg, cand, [&](int t, double m, int mi) {
        const double b = m + vh[t];
        bv[t] = b;
        be[t] = vh[t] - b;
        if (REC) s2[t] = static_cast<unsigned short>(mi);
    });
    __syncthreads();
    for (int t = tid; t < Lv; t += T) {
        w[t] = static_cast<float>(be[t] - be[0]);
        agg[ed.av + t] = bv[t];
        msg[ed.mv + t] = bv[t] - vh[t];
    }
    __syncthreads();
    // pass 3: c(s) = min_t [theta(s,t) + beta(t)] + uh(s)
    screened_lines<true>(st, ldp, Lu, Lv, be, w, key, arg, cand, [&](int s, double m, int mi) {
        const double c = m + uh[s];
        agg[ed.au + s] = c;
        msg[ed.mu + s] = c - uh[s];
        if (REC) t3[s] = static_cast<unsigned short>(mi);
    });
}

// ---------------------------------------------------------------------------
// The same screened update for label counts up to 128 (4 lanes per line).
// What bounds it is the chain from one matching to the next, not work: 400
// edges of 64 x 64 labels are 2.6 blocks per SM.  So:
// - one launch runs all iterations: blocks take the updates from one queue in
//   schedule order, and the FP64 state lives in versioned entries (common.cuh)
//   that a thread polls until they carry the update count it expects.  Every
//   wait is on an update taken earlier by a running block (a block holds the one
//   it works on and the next one, whose record and table it requests meanwhile),
//   so the waits end; they are bounded all the same;
// - a block has 4 threads per label and keeps each row in the registers of its
//   4 lanes (NC 16-byte chunks each) for passes 1 and 3; a copy in shared memory
//   serves the columns of pass 2 (row stride = 8 mod 32 words: the 8 columns x 4
//   rows a warp reads fall into 32 banks);
// - the reference of the shifted vector is 0 (w = x rounded towards zero to
//   FP32), and D is the largest |w| of the vector.  |c - V| <= 2^-24 |c| +
//   2^-23 D, so c lies within eps(c) = 2^-22 (|c| + D) of V and of its FP64 value
//   with more than a factor 2 to spare, and the FP64 minimizer's c* <= c + 4
//   eps(c) for any c of its line (as in bound_scan.cuh): no largest |theta|, no
//   reduction per line but the minimum's.  The padding of w keeps entries beyond
//   the labels at +inf;
// - the screen only finds the argmin.  A line with one candidate (nearly all)
//   needs no FP64 comparison; the others compare their candidates' FP64 values.
//   The minimum's value, and all FP64 vector arithmetic, is formed by one thread
//   per label: an FP64 instruction costs the same for one lane as for 32, so
//   full warps of them are the cheapest.
// 16 x K_50 with 64 labels, per matching: 16.2 us in the general kernel, 8 us
// as dependent launches of this update, 5.8 us so (4 blocks an SM at 64 registers
// instead of 3: 5.9); 8 edges of up to 21 labels: 16.3 -> 2.9 us.
constexpr int kGrpLabels = 128;

template <int NC>
__host__ __device__ constexpr int grp_labels()  // the label counts NC covers
{
    return 16 * NC;
}

__host__ __device__ inline int grp_stride(int ld)  // words, = 8 mod 32, >= ld
{
    return ld + ((8 - ld) & 31);
}

// Argmin of one line from its 4 lanes' screen sums: sv[r] <= thr are the
// candidates, index(r) their positions, value(j) the FP64 value at position j.
// Valid in every lane of the line; INT_MAX without a candidate.
template <int N, typename Index, typename Value>
__device__ __forceinline__ int line_argmin(const float (&sv)[N], float thr, Index index, Value value)
{
    constexpr unsigned kAll = 0xffffffffu;
    unsigned m = 0u;
#pragma unroll
    for (int r = 0; r < N; ++r)
        if (sv[r] <= thr) m |= 1u << r;  // +inf beyond the line; thr is finite
    int cnt = __popc(m);
    cnt += __shfl_xor_sync(kAll, cnt, 1);
    cnt += __shfl_xor_sync(kAll, cnt, 2);
    int arg = m ? index(__ffs(m) - 1) : INT_MAX;
    if (__any_sync(kAll, cnt > 1)) {
        unsigned long long key = ~0ull;
        if (cnt > 1) {
            arg = INT_MAX;
            for (; m; m &= m - 1u) {
                const int j = index(__ffs(m) - 1);
                const unsigned long long v = order_key(value(j));
                if (v < key || (v == key && j < arg)) {
                    key = v;
                    arg = j;
                }
            }
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            const unsigned long long ok = __shfl_xor_sync(kAll, key, o);
            const int oa = __shfl_xor_sync(kAll, arg, o);
            if (ok < key || (ok == key && oa < arg)) {
                key = ok;
                arg = oa;
            }
        }
    } else {
        arg = min(arg, __shfl_xor_sync(kAll, arg, 1));
        arg = min(arg, __shfl_xor_sync(kAll, arg, 2));
    }
    return arg;
}

// The screen's threshold from the line's smallest sum, rounded upwards.  From
// 2^125 on a sum may overflow that the FP64 minimum does not exceed (or all of
// them, as in a table of 1.7e38 against a vector of 1.8e38): no candidate then.
__device__ __forceinline__ float line_threshold(float mn, float d)
{
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
    const float e4 = __fadd_ru(__fmul_ru(0x1p-20f, __fadd_ru(fabsf(mn), d)), 0x1p-122f);
    return e4 < 0x1p105f ? __fadd_ru(mn, e4) : -INFINITY;
}

// Argmin of a line without a candidate: all of it in FP64, by one thread.
__device__ __forceinline__ int line_argmin_all(const float *th, int stride, const double *x, int n)
{
    unsigned long long key = ~0ull;
    int arg = 0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const unsigned long long v = order_key(d_of_f(th[j * stride]) + x[j]);
        if (v < key) {
            key = v;
            arg = j;
        }
    }
    return arg;
}

template <int NC>
__host__ __device__ constexpr int grp_blocks()  // per SM at least (a register cap)
{
    return NC == 8 ? 1 : 12 / NC;
}

template <int NC, bool REC>
__global__ void __launch_bounds__(4 * grp_labels<NC>(), grp_blocks<NC>())
    rec_queue_kernel(BwQueue p, const float *tab, unsigned char *rec)
{
    extern __shared__ __align__(16) double shd[];
    __shared__ float dred[3][kGrpLabels / 32];
    __shared__ __align__(16) BwItem s_it[2];  // the update at work and the next one
    __shared__ long long s_g[2];              // their places in the queue
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kQ = static_cast<int>(sizeof(BwItem) / sizeof(int4));
    const int lmax = p.lmax;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    constexpr int V = NC > 2 ? NC / 2 : 1;  // warps with a thread per label
    const int i = tid >> 2, k = tid & 3;  // this thread's line and its lane of the line
    double *uh = shd, *vh = uh + lmax, *al = vh + lmax, *be = al + lmax;
    float *w = reinterpret_cast<float *>(be + lmax);  // [32 V] the current pass's vector in FP32
    int *arg = reinterpret_cast<int *>(w + 32 * V);     // [32 V] argmins of the pass
    float *st = reinterpret_cast<float *>(arg + 32 * V);  // [16 NC][ldp] the table
    const float4 inf4 = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
    const long long total = p.n_items * p.iterations;
    // this thread's chunks k, k + 4, ... of row i
    auto load_rows = [&](const EdgeDesc &ed, float4 (&r)[NC]) {
        const float4 *th4 = reinterpret_cast<const float4 *>(tab + ed.toff);
        const int Q = ed.ld >> 2;
#pragma unroll
        for (int c = 0; c < NC; ++c) r[c] = (i < ed.Lu && k + 4 * c < Q) ? __ldg(th4 + i * Q + k + 4 * c) : inf4;
    };
    if (tid == 0) s_g[0] = static_cast<long long>(atomicAdd(p.queue, 1ull));
    __syncthreads();
    long long g = s_g[0];
    if (g >= total) return;
    if (tid < kQ)
        reinterpret_cast<int4 *>(&s_it[0])[tid] = __ldg(reinterpret_cast<const int4 *>(p.items + bw_place(p, g).y) + tid);
    __syncthreads();
    float4 row[NC], nrow[NC];
    load_rows(s_it[0].ed, row);
    bool drain = false;
    for (int turn = 0; g < total; ++turn) {
        const BwItem &it = s_it[turn & 1];
        const EdgeDesc ed = it.ed;
        const int Lu = ed.Lu, Lv = ed.Lv, Q = ed.ld >> 2, ldp = grp_stride(ed.ld);
        const unsigned n_it = bw_place(p, g).x;  // iterations before this one in this launch
        const unsigned ve = p.done + n_it;       // ... and in all: updates of this edge
        const unsigned vu = ve * static_cast<unsigned>(it.deg_u) + static_cast<unsigned>(it.pos_u);
        const unsigned vv = ve * static_cast<unsigned>(it.deg_v) + static_cast<unsigned>(it.pos_v);
        if (tid == 0) s_g[(turn + 1) & 1] = static_cast<long long>(atomicAdd(p.queue, 1ull));
        unsigned short *t1 = nullptr, *s2 = nullptr, *t3 = nullptr;
        if (REC) {
            t1 = reinterpret_cast<unsigned short *>(rec + n_it * p.rec_stride + it.rec_off);
            s2 = t1 + Lu;
            t3 = s2 + Lv;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (i < Lu && k + 4 * c < Q) *reinterpret_cast<float4 *>(st + i * ldp + 4 * (k + 4 * c)) = row[c];
        // the vectors: the first V warps node v's, the last V warps node u's (the same warps if V = W)
        // w(j) and the vector's largest |w|; pad: w beyond the labels
        auto shifted = [&](int pass, int j, int n, double x, float pad) {
            const float f = j < n ? f_of_d(x) : 0.f;
            w[j] = j < n ? f : pad;
            const float d = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(fabsf(f))));
            if (lane == 0) dred[pass][warp] = d;
        };
        const int vt = tid, ut = tid - (W - V) * 32;  // this thread's label of node v / node u (0 <= . < 32 V)
        if (warp < V) {
            double x = 0.0;
            if (vt < Lv) vh[vt] = x = bw_poll_diff(p, p.agg + ed.av + vt, p.msg + ed.mv + vt, vv, ve, drain);
            shifted(0, vt, Lv, x, 0.f);
        }
        if (warp >= W - V && ut < Lu)
            uh[ut] = bw_poll_diff(p, p.agg + ed.au + ut, p.msg + ed.mu + ut, g > 0 ? vu : vu + p.test_wait, ve, drain);
        __syncthreads();
        const long long g2 = s_g[(turn + 1) & 1];
        int4 nrec = make_int4(0, 0, 0, 0);
        if (g2 < total && tid < kQ) nrec = __ldg(reinterpret_cast<const int4 *>(p.items + bw_place(p, g2).y) + tid);
        auto largest = [&](int pass) {
            float d = dred[pass][0];
            for (int q = 1; q < V; ++q) d = fmaxf(d, dred[pass][q]);
            return d;
        };
        const float4 *w4 = reinterpret_cast<const float4 *>(w);
        // argmin of row i of theta + x (w: x in FP32)
        auto scan_rows = [&](int pass, const double *x, unsigned short *out) {
            float sv[4 * NC], mn = INFINITY;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float4 v = k + 4 * c < Q ? add4(row[c], w4[k + 4 * c]) : inf4;
                sv[4 * c] = v.x;
                sv[4 * c + 1] = v.y;
                sv[4 * c + 2] = v.z;
                sv[4 * c + 3] = v.w;
                mn = min3f(min3f(mn, v.x, v.y), v.z, v.w);
            }
            const float thr = line_threshold(mn, largest(pass));
            const float *st_i = st + i * ldp;
            const int a = line_argmin(
                sv, i < Lu ? thr : -INFINITY, [&](int r) { return 4 * (k + 4 * (r >> 2)) + (r & 3); },
                [&](int j) { return d_of_f(st_i[j]) + x[j]; });
            if (k == 0 && i < Lu) {
                const int j = a == INT_MAX ? line_argmin_all(st_i, 1, x, Lv) : a;
                arg[i] = j;
                if (REC) out[i] = static_cast<unsigned short>(j);
            }
        };
        // pass 1: a(s) = 1/2 (min_t [theta(s,t) + vh(t)] + uh(s)),  alpha = uh - a
        scan_rows(0, vh, t1);
        __syncthreads();
        if (warp < V) {
            double x = 0.0;
            if (tid < Lu) {
                const int j = arg[tid];
                const double u = uh[tid];
                al[tid] = x = fma(-0.5, (d_of_f(st[tid * ldp + j]) + vh[j]) + u, u);  // u - a, 0.5 (...) is exact
            }
            shifted(1, tid, Lu, x, INFINITY);
        }
        if (tid < kQ) reinterpret_cast<int4 *>(&s_it[(turn + 1) & 1])[tid] = nrec;
        __syncthreads();
        if (g2 < total) load_rows(s_it[(turn + 1) & 1].ed, nrow);
        // pass 2: b(t) = min_s [theta(s,t) + alpha(s)] + vh(t),  beta = vh - b
        {
            float sv[4 * NC], mn = INFINITY;
#pragma unroll
            for (int r = 0; r < 4 * NC; ++r) {
                sv[r] = st[(k + 4 * r) * ldp + i] + w[k + 4 * r];  // rows beyond Lu: w is +inf (a NaN is ignored)
                mn = fminf(mn, sv[r]);
            }
            const float thr = line_threshold(mn, largest(1));
            const int a = line_argmin(
                sv, i < Lv ? thr : -INFINITY, [&](int r) { return k + 4 * r; },
                [&](int j) { return d_of_f(st[j * ldp + i]) + al[j]; });
            if (k == 0 && i < Lv) {
                const int j = a == INT_MAX ? line_argmin_all(st + i, ldp, al, Lu) : a;
                arg[i] = j;
                if (REC) s2[i] = static_cast<unsigned short>(j);
            }
        }
        __syncthreads();
        if (warp < V) {
            double x = 0.0;
            if (tid < Lv) {
                const int j = arg[tid];
                const double v = vh[tid], b = (d_of_f(st[j * ldp + tid]) + al[j]) + v;
                st_se(p.agg + ed.av + tid, se64_make(b, vv + 1u));
                be[tid] = x = v - b;
                st_se(p.msg + ed.mv + tid, se64_make(-x, ve + 1u));
            }
            shifted(2, tid, Lv, x, 0.f);
        }
        __syncthreads();
        // pass 3: c(s) = min_t [theta(s,t) + beta(t)] + uh(s)
        scan_rows(2, be, t3);
        __syncthreads();
        if (tid < Lu) {
            const int j = arg[tid];
            const double u = uh[tid], c = (d_of_f(st[tid * ldp + j]) + be[j]) + u;
            st_se(p.agg + ed.au + tid, se64_make(c, vu + 1u));
            st_se(p.msg + ed.mu + tid, se64_make(c - u, ve + 1u));
        }
        __syncthreads();  // vectors and table are rewritten for the next update
        g = g2;
#pragma unroll
        for (int c = 0; c < NC; ++c) row[c] = nrow[c];
    }
}

}  // namespace

// FP64 values to versioned entries (version 0), and back
__global__ void to_entries_kernel(const double *src, ulonglong2 *dst, long long n)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        dst[i] = se64_make(src[i], 0u);
}

__global__ void from_entries_kernel(const ulonglong2 *src, double *dst, long long n)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        dst[i] = se64_val(src[i]);
}

__global__ void widen_kernel(const float *src, double *dst, long long n)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        dst[i] = static_cast<double>(src[i]);
}

}  // namespace

size_t rec64_smem_bytes(int lmax)
{
    return static_cast<size_t>(lmax) * 5 * sizeof(double);
}

size_t rec_screen_smem_bytes(int lmax, long long tab_floats)
{
    // uh, vh, alpha, beta, b (FP64), keys; the warps' candidate lists; args; w (FP32); the staged table
    return static_cast<size_t>(lmax) * (6 * 8 + 4 + 4) + sizeof(int2) * (kScrThreads / 32) * kWarpCands +
           4 * static_cast<size_t>(tab_floats);
}

cudaError_t launch_rec_screen_phase(const EdgeDesc *descs, int n_items, const float *tab,
                                    double *agg, double *msg, unsigned char *rec, const long long *rec_off, int lmax,
                                    long long tab_floats, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    const size_t smem = rec_screen_smem_bytes(lmax, tab_floats);
    if (rec) {
        cudaError_t e = raise_smem_limit(rec_screen_kernel<true>, smem);
        if (e != cudaSuccess) return e;
        rec_screen_kernel<true><<<n_items, kScrThreads, smem, st>>>(descs, tab, agg, msg, rec, rec_off, lmax);
    } else {
        cudaError_t e = raise_smem_limit(rec_screen_kernel<false>, smem);
        if (e != cudaSuccess) return e;
        rec_screen_kernel<false><<<n_items, kScrThreads, smem, st>>>(descs, tab, agg, msg, nullptr, nullptr, lmax);
    }
    return cudaGetLastError();
}

size_t rec_group_smem_bytes(int lmax)
{
    const int l4 = (lmax + 3) & ~3;
    const size_t rows = lmax <= 16 ? 16 : (lmax <= 32 ? 32 : (lmax <= 64 ? 64 : 128));  // 16 NC
    return 4 * sizeof(double) * static_cast<size_t>(lmax) + 8 * std::max<size_t>(32, rows) + 4 * rows * grp_stride(l4);
}

bool rec_group_fits(int lmax)
{
    return lmax <= kGrpLabels;
}

namespace {
template <int NC, bool REC>
cudaError_t launch_queue_nc(const BwQueue &p, int max_items, const float *tab, unsigned char *rec, cudaStream_t st)
{
    const size_t smem = rec_group_smem_bytes(p.lmax);
    const int threads = 4 * ((p.lmax + 7) & ~7);
    int per_sm = 0;
    cudaError_t e = raise_smem_limit(rec_queue_kernel<NC, REC>, smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rec_queue_kernel<NC, REC>, threads, smem);
    if (e != cudaSuccess) return e;
    // (blocks beyond two matchings' updates would only poll)
    const int blocks = std::max(1, std::min(per_sm * 152, 2 * max_items));
    rec_queue_kernel<NC, REC><<<blocks, threads, smem, st>>>(p, tab, rec);
    return cudaGetLastError();
}

template <bool REC>
cudaError_t launch_queue_for(const BwQueue &p, int max_items, const float *tab, unsigned char *rec, cudaStream_t st)
{
    if (p.lmax <= grp_labels<1>()) return launch_queue_nc<1, REC>(p, max_items, tab, rec, st);
    if (p.lmax <= grp_labels<2>()) return launch_queue_nc<2, REC>(p, max_items, tab, rec, st);
    if (p.lmax <= grp_labels<4>()) return launch_queue_nc<4, REC>(p, max_items, tab, rec, st);
    return launch_queue_nc<8, REC>(p, max_items, tab, rec, st);
}
}  // namespace

cudaError_t launch_rec_queue(const BwQueue &p, int max_items, const float *tab, unsigned char *rec, cudaStream_t st)
{
    if (p.n_items <= 0 || p.iterations <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(p.queue, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    return rec ? launch_queue_for<true>(p, max_items, tab, rec, st)
               : launch_queue_for<false>(p, max_items, tab, nullptr, st);
}

cudaError_t launch_rec64_phase(const EdgeDesc *edges, const int *items, int n_items, const float *tab, double *agg,
                               double *msg, unsigned char *rec, const long long *rec_off, int lmax, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    const size_t smem = rec64_smem_bytes(lmax);
    if (rec) {
        if (smem > 48 * 1024) {
            cudaError_t e = raise_smem_limit(rec64_phase_kernel<true>, smem);
            if (e != cudaSuccess) return e;
        }
        rec64_phase_kernel<true><<<n_items, kThreads, smem, st>>>(edges, items, tab, agg, msg, rec, rec_off, lmax);
    } else {
        if (smem > 48 * 1024) {
            cudaError_t e = raise_smem_limit(rec64_phase_kernel<false>, smem);
            if (e != cudaSuccess) return e;
        }
        rec64_phase_kernel<false><<<n_items, kThreads, smem, st>>>(edges, items, tab, agg, msg, nullptr, nullptr, lmax);
    }
    return cudaGetLastError();
}

namespace {
unsigned blocks_for(long long n)
{
    return static_cast<unsigned>(std::min<long long>((n + 255) / 256, 65535LL * 8));
}
}  // namespace

cudaError_t launch_to_entries(const double *src, ulonglong2 *dst, long long n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    to_entries_kernel<<<blocks_for(n), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_from_entries(const ulonglong2 *src, double *dst, long long n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    from_entries_kernel<<<blocks_for(n), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_widen(const float *src, double *dst, long long n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const long long blocks = std::min<long long>((n + 255) / 256, 65535LL * 8);
    widen_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

}  // namespace mplpp
