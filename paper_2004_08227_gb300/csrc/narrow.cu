// narrow.cu -- the persistent driver for small label counts (<= 32): one launch
// for all iterations, a group of LM = 8, 16 or 32 lanes per edge (group.cuh).
// A warp walks a fixed list of steps in schedule order, each up to 32 / LM edges
// of one matching; an edge belongs to the same lanes in every iteration.
//
// One warp per block.  As in the persistent driver of handshake.cu the state
// lives in versioned entries (common.cuh): a lane polls the two node entries of
// its label until they carry the update count it expects, and the new entries
// are the signal to their readers.  Every wait is on an earlier matching, which
// no step waiting in the same warp can hold up, and all warps are co-resident,
// so the waits end; they are bounded (spin_limit; then ERR_TIMEOUT is recorded
// and the kernel drains without waiting).
//
// Bound by the chain from one matching to the next: a store and a polling round
// trip through L2, then the update.  What else a step needs -- its table, the
// edge's messages, which the same lanes wrote an iteration ago, and its record --
// is copied into shared memory two steps ahead by cp.async (the messages only
// where the copy comes a step or more after they were stored, which a warp
// barrier separates: with one or two steps in an iteration they are loaded at
// their turn).  K_600 with 13 labels, per matching: 2.44 us with a CTA of 128
// threads per edge, 1.53 us with these loads prefetched into registers (a warp
// has six load scoreboards: its wait for the node entries took in the prefetches
// behind them), 1.15 us so. Node vectors in the distributed shared memory of a
// cluster of 16 CTAs, with a cluster barrier per matching, took 1.86 us: 16 SMs
// issue too slowly for 300 edges.
#include <cfloat>
#include <cstdint>

#include "group.cuh"
#include "kernels.h"

namespace mplpp {

namespace {

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// What one group has in flight: the tables and messages of two steps, the
// records of those and the next ones, and the operand vectors of the update.
// The copies of turn k: table and messages of step k + 2, record of step k + 4.
template <int LM, typename Rec>
struct Stage {
    float tab[2][LM * LM];
    ulonglong2 msg[2][2 * LM];
    float vec[3 * LM];
    Rec rec[8];
};

template <int LM, typename Rec>
struct Walk {
    Stage<LM, Rec> &st;
    const float *tab;
    const ulonglong2 *msg;
    const Rec *recs;  // this group's first record
    int rec_step;     // records from one step to the next
    int n;            // steps per iteration
    int l;
    int next = 0;     // place of the next record to copy

    __device__ __forceinline__ void copy_rec(long long k)  // the record of step k, the steps in order
    {
        constexpr int kQ = static_cast<int>(sizeof(Rec) / 16);
        if (l < kQ)
            cp_async16(reinterpret_cast<char *>(&st.rec[k & 7]) + 16 * l,
                       reinterpret_cast<const char *>(recs + static_cast<long long>(next) * rec_step) + 16 * l);
        if (++next == n) next = 0;
    }
    __device__ __forceinline__ void copy_step(long long k)  // step k's table and messages (its record is there)
    {
        const Rec &r = st.rec[k & 7];
        const int Lu = r.Lu, Lv = r.Lv, chunks = Lu * (r.ld >> 2);
        float *dst = st.tab[k & 1];
        const float *src = tab + r.toff;
#pragma unroll
        for (int j = 0; j < LM / 4; ++j)
            if (l + j * LM < chunks) cp_async16(dst + 4 * (l + j * LM), src + 4 * (l + j * LM));
        if (n > 2) {  // phi_{v->u}, then phi_{u->v}: one run of entries
            const int entries = ((Lu + 3) & ~3) + ((Lv + 3) & ~3);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (l + j * LM < entries) cp_async16(&st.msg[k & 1][l + j * LM], msg + r.mu + l + j * LM);
        }
    }
    __device__ __forceinline__ void begin()
    {
        for (int k = 0; k < 4; ++k) copy_rec(k);
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
        copy_step(0);
        cp_async_commit();
        copy_step(1);
        cp_async_commit();
    }
    // Step k's record, table and messages (all of them before the copies of the turn overwrite them)
    __device__ __forceinline__ Rec take(long long k, float (&row)[LM], float (&col)[LM], float2 &mu, float2 &mv)
    {
        cp_async_wait<1>();
        __syncwarp();
        const Rec r = st.rec[k & 7];
        const float *th = st.tab[k & 1];
        if (r.Lu > 0) {
            const int s0 = min(l, r.Lu - 1), t0 = min(l, r.Lv - 1);
            const float4 *r4 = reinterpret_cast<const float4 *>(th + s0 * r.ld);
#pragma unroll
            for (int j = 0; j < LM / 4; ++j) {
                const float4 v = 4 * j < r.ld ? r4[j] : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                row[4 * j] = v.x;
                row[4 * j + 1] = v.y;
                row[4 * j + 2] = v.z;
                row[4 * j + 3] = v.w;
            }
#pragma unroll
            for (int s = 0; s < LM; ++s) col[s] = s < r.Lu ? th[s * r.ld + t0] : INFINITY;
        }
        ulonglong2 xu = make_ulonglong2(0ull, 0ull), xv = xu;
        if (n > 2) {
            if (l < r.Lu) xu = st.msg[k & 1][l];
            if (l < r.Lv) xv = st.msg[k & 1][((r.Lu + 3) & ~3) + l];
        } else {  // this edge's step came one or two before: its new messages, by the lanes that stored them
            if (l < r.Lu) xu = ld_se(msg + r.mu + l);
            if (l < r.Lv) xv = ld_se(msg + r.mv + l);
        }
        mu = se_df(xu);
        mv = se_df(xv);
        return r;
    }
    __device__ __forceinline__ void refill(long long k)  // the copies of turn k
    {
        copy_step(k + 2);
        copy_rec(k + 4);
        cp_async_commit();
    }
};

template <int LM>
__global__ void __launch_bounds__(32) hs_narrow_kernel(NarrowParams p)
{
    constexpr int EPW = 32 / LM;
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ __align__(16) Stage<LM, NarrowRec> stages[EPW];
    const int l = static_cast<int>(threadIdx.x) % LM, slot = static_cast<int>(threadIdx.x) / LM;
    const int begin = p.step_off[blockIdx.x], n = p.step_off[blockIdx.x + 1] - begin;
    const long long total = static_cast<long long>(n) * p.iterations;
    if (total == 0) return;
    Walk<LM, NarrowRec> walk{stages[slot], p.tab, p.msg, p.recs + static_cast<long long>(begin) * EPW + slot, EPW, n, l};
    walk.begin();
    bool drain = false;
    unsigned it = 0;
    int k_it = 0;  // steps of this iteration done
    for (long long k = 0; k < total; ++k) {
        float row[LM], col[LM];
        float2 mu, mv;
        const NarrowRec r = walk.take(k, row, col, mu, mv);
        const bool on_u = l < r.Lu, on_v = l < r.Lv;
        // update counts modulo 2^32 (only equality is tested)
        const unsigned vu = it * static_cast<unsigned>(r.deg_u) + static_cast<unsigned>(r.pos_u);
        const unsigned vv = it * static_cast<unsigned>(r.deg_v) + static_cast<unsigned>(r.pos_v);
        const unsigned want_u = vu + ((p.test_wait && k == 0 && blockIdx.x == 0) ? 1u : 0u);
        ulonglong2 *au = p.agg + r.au + l, *av = p.agg + r.av + l;
        ulonglong2 xu = make_ulonglong2(0ull, 0ull), xv = xu;
        if (on_u) xu = ld_se(au);
        if (on_v) xv = ld_se(av);
        for (long long spins = 1;; ++spins) {
            const bool ok_u = !on_u || se_ok(xu, want_u), ok_v = !on_v || se_ok(xv, vv);
            if (__all_sync(kAll, (ok_u && ok_v) || drain)) break;
            if (spins > p.spin_limit) {
                atomicCAS(p.err, 0, ERR_TIMEOUT);
                drain = true;
            } else if ((spins & 63) == 0 && *reinterpret_cast<volatile int *>(p.err) != 0) {
                drain = true;
            }
            if (spins > 64) __nanosleep(32);
            if (!ok_u) xu = ld_se(au);
            if (!ok_v) xv = ld_se(av);
        }
        group_update<LM>(
            row, col, se_df(xu), mu, se_df(xv), mv, stages[slot].vec, l,
            [&](float2 b, float2 m) {
                if (on_v) {
                    st_se(av, se_make(b, vv + 1u));
                    st_se(p.msg + r.mv + l, se_make(m, it + 1u));
                }
            },
            [&](float2 c, float2 m) {
                if (on_u) {
                    st_se(au, se_make(c, vu + 1u));
                    st_se(p.msg + r.mu + l, se_make(m, it + 1u));
                }
            });
        walk.refill(k);
        if (++k_it == n) {
            k_it = 0;
            ++it;
        }
    }
    cp_async_wait<0>();
}

template <int LM>
int max_warps()
{
    int per_sm = 0, dev = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hs_narrow_kernel<LM>, 32, 0) != cudaSuccess) return 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return per_sm * sms;
}

}  // namespace

int narrow_max_warps(int lmax)
{
    switch (res_lanes(lmax)) {
    case 8: return max_warps<8>();
    case 16: return max_warps<16>();
    default: return max_warps<32>();
    }
}

cudaError_t launch_narrow(const NarrowParams &p, int warps, int lmax, cudaStream_t st)
{
    if (warps <= 0) return cudaSuccess;
    switch (res_lanes(lmax)) {
    case 8: hs_narrow_kernel<8><<<warps, 32, 0, st>>>(p); break;
    case 16: hs_narrow_kernel<16><<<warps, 32, 0, st>>>(p); break;
    default: hs_narrow_kernel<32><<<warps, 32, 0, st>>>(p); break;
    }
    return cudaGetLastError();
}

}  // namespace mplpp
