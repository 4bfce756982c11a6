// ADAPTAHOP subhalos on HOP's chains (Parallel HOP Sec. 6, "Parallel HOP
// and Subhalos").
//
//  S1  symmetric boundary table: the directed chain-pair table (both
//      particles >= delta_outer, as in HOP's table), kept only for pairs
//      linked in both directions, each with the larger direction's sum
//      (link.cu, boundaries_table with symmetric = true);
//  S2  dense ids for the chain roots above delta_outer (scan) and, per
//      particle above delta_outer, its root's id;
//  S3  one pass over the particles gives every chain its densest member's
//      key and, for up to kLev thresholds at once, the number (and fp64
//      density sum, if needed) of its members with dens >= delta_s;
//  S4  per threshold, links with s < 2 delta_s are destroyed; the rest join
//      chains into connected components (hook the larger root under the
//      smaller with atomicMin, compress, repeat until no edge joins two
//      roots), all thresholds in the same launches;
//  S5  chains' counts, sums and keys are added up per component; a component
//      is a subhalo when count >= n_min and mean density >= delta_s (1 +
//      f_poisson / sqrt(count));
//  S6  subhalos are ranked by peak key: the chains are sorted by their key
//      once, and a subhalo's rank is the number of subhalos' peak chains
//      before its own in that order (one scan over all thresholds);
//  S7  one pass over the particles writes every threshold's labels from the
//      chain's label row.
//
// The two per-particle passes read 12 bytes per particle each, whatever the
// number of thresholds (a pass per threshold and purpose read them 2 L
// times), and write 4 bytes per threshold: HBM-bound.  What depends on the
// threshold works on chains, a hundred times fewer.
// Halo statistics and subhalos of 16.8M particles at five thresholds: 3309 us
// with a pass, a component search and a sort per threshold, 1996 us so.
#include "hop_internal.cuh"

#include <algorithm>
#include <vector>
#include <cmath>

namespace {

constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr int kMaxRounds = 64;

// S2: roots above delta_outer; chain labels must be roots of [0, n).
__global__ void sub_root_flag_kernel(const uint32_t *__restrict__ chain, const uint64_t *__restrict__ dkey,
                                 int64_t n, float d_o, uint32_t *__restrict__ flag, uint32_t *__restrict__ err)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = chain[i];
        if (c >= (uint64_t)n || chain[c] != c) atomicOr(err, kErrBadIndex);
        flag[i] = (c == (uint32_t)i && key_dens(dkey[i]) >= d_o) ? 1u : 0u;
    }
}

// Per particle above delta_outer: its root's dense id.  A particle above
// delta_outer has a root above it (hops go uphill); anything else is an
// inconsistent input.
__global__ void sub_particle_chain_kernel(const uint32_t *__restrict__ chain, const uint64_t *__restrict__ dkey,
                                      int64_t n, float d_o, const uint32_t *__restrict__ cid,
                                      uint32_t *__restrict__ pc, uint32_t *__restrict__ err)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t v = kNone;
        if (key_dens(dkey[i]) >= d_o) {
            const uint32_t r = chain[i];
            if (r >= (uint64_t)n || !(key_dens(dkey[r]) >= d_o)) atomicOr(err, kErrBadIndex);
            else v = cid[r];
        }
        pc[i] = v;
    }
}

// Every chain's key starts as its root's.
__global__ void sub_root_key_kernel(const uint32_t *__restrict__ chain, const uint64_t *__restrict__ dkey, int64_t n,
                                    const uint32_t *__restrict__ pc, unsigned long long *__restrict__ pkey)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        if (chain[i] == (uint32_t)i && pc[i] != kNone) pkey[pc[i]] = dkey[i];
}

__global__ void sub_edge_ids_kernel(const uint64_t *__restrict__ ekey, int64_t m, int64_t n,
                                const uint32_t *__restrict__ chain, const uint64_t *__restrict__ dkey, float d_o,
                                const uint32_t *__restrict__ cid, uint32_t *__restrict__ ea,
                                uint32_t *__restrict__ eb, uint32_t *__restrict__ err)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t lo = (uint32_t)(ekey[e] >> 32), hi = (uint32_t)ekey[e];
        if (lo >= (uint64_t)n || hi >= (uint64_t)n || chain[lo] != lo || chain[hi] != hi ||
            !(key_dens(dkey[lo]) >= d_o) || !(key_dens(dkey[hi]) >= d_o)) {
            atomicOr(err, kErrBadIndex);
            ea[e] = eb[e] = 0;
            continue;
        }
        ea[e] = cid[lo];
        eb[e] = cid[hi];
    }
}

constexpr int kLev = 8;   // thresholds handled together; a chain's row of kLev 4-byte values is one sector

struct Levels {
    float ds[kLev];
    int L;
};

// Sum of x over the lanes of `peers` (the lane's own set of a match), in its
// first lane: every round adds the next lane that is still in to each lane of
// even rank and drops the odd ones.
__device__ __forceinline__ double peer_sum(uint32_t peers, int lane, double x)
{
    uint32_t rank = __popc(peers & ((1u << lane) - 1u));
    uint32_t above = peers & (0xfffffffeu << lane);
    while (__any_sync(0xffffffffu, above != 0)) {
        const int next = __ffs(above);                     // 0: none
        const double y = __shfl_sync(0xffffffffu, x, next ? next - 1 : lane);
        if (next) x += y;
        above &= __ballot_sync(0xffffffffu, (rank & 1u) == 0);
        rank >>= 1;
    }
    return x;
}

// S3: count[c * kLev + l], sum (the same layout, or nullptr) and peak key of
// every chain.  The lanes of a warp that hold the same chain are found by a
// match, wherever they are (a halo's particles alternate between its chains),
// their counts are the set bits of a ballot per threshold, and one lane adds
// them.  pkey holds the root's key on entry, normally the chain's largest, so
// it is only read.
constexpr int kSubU = 4;

template <bool SUM>
__global__ void sub_chain_stats_kernel(const uint64_t *__restrict__ dkey, const uint32_t *__restrict__ pc, int64_t n,
                                       const Levels lev, uint32_t *__restrict__ cnt, double *__restrict__ sum,
                                       unsigned long long *pkey)
{
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * kSubU;
    for (int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) * kSubU; w0 < n; w0 += stride) {
        uint64_t k[kSubU];
        uint32_t c[kSubU];
        unsigned long long top[kSubU];
#pragma unroll
        for (int u = 0; u < kSubU; ++u) {
            const int64_t i = w0 + u * 32 + lane;
            k[u] = i < n ? dkey[i] : 0ull;
            c[u] = i < n ? pc[i] : kNone;
        }
#pragma unroll
        for (int u = 0; u < kSubU; ++u) top[u] = c[u] != kNone ? pkey[c[u]] : ~0ull;
#pragma unroll
        for (int u = 0; u < kSubU; ++u) {
            const uint32_t rr = c[u];
            if (!__any_sync(0xffffffffu, rr != kNone)) continue;
            if (k[u] > top[u]) atomicMax(&pkey[rr], (unsigned long long)k[u]);
            const float d = key_dens(k[u]);
            const uint32_t peers = __match_any_sync(0xffffffffu, rr);
            const bool head = rr != kNone && lane == __ffs(peers) - 1;
            for (int l = 0; l < lev.L; ++l) {
                const bool in = rr != kNone && d >= lev.ds[l];
                const uint32_t m = __popc(__ballot_sync(0xffffffffu, in) & peers);
                if (head && m) atomicAdd(&cnt[(int64_t)rr * kLev + l], m);
                if constexpr (SUM) {
                    const double x = peer_sum(peers, lane, in ? (double)d : 0.0);
                    if (head && m) atomicAdd(&sum[(int64_t)rr * kLev + l], x);
                }
            }
        }
    }
}

// S4, all levels at once: parent[l * C + c].
__global__ void sub_iota_kernel(uint32_t *p, int64_t C, int L)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * L; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = (uint32_t)(i % C);
}

__global__ void sub_hook_kernel(const uint32_t *__restrict__ ea, const uint32_t *__restrict__ eb,
                                const double *__restrict__ es, int64_t m, const Levels lev, int64_t C,
                                uint32_t *parent, uint32_t *changed)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const double s = es[e];
        const uint32_t a = ea[e], b = eb[e];
        for (int l = 0; l < lev.L; ++l) {
            if (!(s >= 2.0 * (double)lev.ds[l])) continue;
            uint32_t *p = parent + l * C;
            const uint32_t ra = find_root(p, a), rb = find_root(p, b);
            if (ra == rb) continue;
            atomicMin(&p[max(ra, rb)], min(ra, rb));
            *changed = 1u;
        }
    }
}

__global__ void sub_compress_kernel(uint32_t *parent, int64_t C, int L)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * L; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t *p = parent + i / C * C;
        parent[i] = find_root(p, (uint32_t)(i - i / C * C));
    }
}

// S5: the chains' shares of every component, index l * C + component.
__global__ void sub_component_kernel(const uint32_t *__restrict__ cnt, const double *__restrict__ sum,
                                     const unsigned long long *__restrict__ pkey, int64_t C, int L,
                                     const uint32_t *__restrict__ parent, unsigned long long *__restrict__ ccnt,
                                     double *__restrict__ csum, unsigned long long *__restrict__ cpk)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * L; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i / C, c = i - l * C;
        const uint32_t k = cnt[c * kLev + l];
        if (!k) continue;
        const int64_t r = l * C + parent[i];
        atomicAdd(&ccnt[r], (unsigned long long)k);
        if (csum) atomicAdd(&csum[r], sum[c * kLev + l]);
        atomicMax(&cpk[r], pkey[c]);
    }
}

// The significance cut, in the same fp64 operations as the definition.
// With f = 0 the cut is mean >= delta_s, which every set of members passes:
// each member is >= delta_s, and rounding is monotone, so a running fp64
// sum of N of them is >= N delta_s (exact for a float32 delta_s and
// N < 2^29) and the rounded mean is >= delta_s, in any summation order.
// Then (f = 0 and n < 2^29) sum is nullptr and only the count is tested.
__device__ __forceinline__ bool sub_accept(unsigned long long k, const double *sum, int64_t r, double ds, long long n_min,
                                           double f)
{
    if (k == 0 || (long long)k < n_min) return false;
    if (!sum) return true;
    const double N = (double)k;
    const double mean = __ddiv_rn(sum[r], N);
    const double thr = __dmul_rn(ds, __dadd_rn(1.0, __ddiv_rn(f, __dsqrt_rn(N))));
    return mean >= thr;
}

__global__ void sub_keys_kernel(const unsigned long long *__restrict__ pkey, int64_t C, uint64_t *__restrict__ gk,
                                uint32_t *__restrict__ gv)
{
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        gk[c] = ~(uint64_t)pkey[c];   // ascending = peak density desc, index asc
        gv[c] = (uint32_t)c;
    }
}

// S6: flag[l * C + position of chain c in key order] = c is the peak chain
// of a subhalo at level l.
__global__ void sub_flag_kernel(const uint32_t *__restrict__ order, const unsigned long long *__restrict__ pkey, int64_t C,
                                const Levels lev, const uint32_t *__restrict__ parent,
                                const unsigned long long *__restrict__ ccnt, const double *__restrict__ csum,
                                const unsigned long long *__restrict__ cpk, long long n_min, double f,
                                uint32_t *__restrict__ flag)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * lev.L;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i / C;
        const uint32_t c = order[i - l * C];
        const int64_t r = l * C + parent[l * C + c];
        flag[i] = cpk[r] == pkey[c] && sub_accept(ccnt[r], csum, r, (double)lev.ds[l], n_min, f) ? 1u : 0u;
    }
}

// rank[l * C + component], and the number of subhalos per level.
__global__ void sub_rank_kernel(const uint32_t *__restrict__ order, const uint32_t *__restrict__ flag,
                                const uint32_t *__restrict__ pos, int64_t C, int L, const uint32_t *__restrict__ parent,
                                int32_t *__restrict__ rank, uint32_t *__restrict__ n_lev)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * L; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i / C;
        const uint32_t at = pos[i] - pos[l * C];
        if (i - l * C == C - 1) n_lev[l] = at + flag[i];
        if (flag[i]) rank[l * C + parent[l * C + order[i - l * C]]] = (int32_t)at;
    }
}

// Every chain's row of labels: its component's rank at each level, or -1
// (rank holds -1 where there is no subhalo).
__global__ void sub_row_kernel(const int32_t *__restrict__ rank, const uint32_t *__restrict__ parent, int64_t C, int L,
                               int32_t *__restrict__ row)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C * L; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i / C, c = i - l * C;
        row[c * kLev + l] = rank[l * C + parent[i]];
    }
}

// S7
__global__ void sub_label_kernel(const uint64_t *__restrict__ dkey, const uint32_t *__restrict__ pc, int64_t n,
                                 const Levels lev, const int32_t *__restrict__ row, int32_t *__restrict__ sub)
{
    static_assert(kLev == 8, "a row is two 16-byte reads");
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t c = pc[i];
        int32_t v[kLev] = {-1, -1, -1, -1, -1, -1, -1, -1};
        if (c != kNone) {
            const float d = key_dens(dkey[i]);
            const int4 a = reinterpret_cast<const int4 *>(row + (int64_t)c * kLev)[0],
                       b = reinterpret_cast<const int4 *>(row + (int64_t)c * kLev)[1];
            const int32_t x[kLev] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int l = 0; l < kLev; ++l)
                if (l < lev.L && d >= lev.ds[l]) v[l] = x[l];
        }
#pragma unroll
        for (int l = 0; l < kLev; ++l)
            if (l < lev.L) sub[l * n + i] = v[l];
    }
}

int subhalos(hop_ctx *c, const uint32_t *chain, const float *dens, const uint64_t *dkey, const uint32_t *nbr, int ld, int64_t n,
             int n_merge, float d_o, const float *levels, int L, int64_t n_min, double f, int32_t *sub,
             int64_t *n_sub)
{
    // S1
    HOP_CUDA(c, cudaEventRecord(c->ev[2], c->stream));
    uint64_t *ek;
    double *es;
    int64_t m;
    int rc = boundaries_table(c, chain, dens, nbr, ld, n, n_merge, d_o, &ek, &es, &m, true);
    if (rc) return rc;
    HOP_CUDA(c, cudaEventRecord(c->ev[3], c->stream));
    // S2
    uint32_t *hp = (uint32_t *)c->h_pinned;
    // misc: total, then kMaxRounds round flags, then kLev subhalo counts
    uint32_t *misc = (uint32_t *)ctx_buf(c, S_MISC, (size_t)(2 + kMaxRounds + kLev) * sizeof(uint32_t));
    uint32_t *cid = (uint32_t *)ctx_buf(c, S_SUB, (size_t)(2 * n + 64) * sizeof(uint32_t));
    if (!misc || !cid) return HOP_ENOMEM;
    uint32_t *pc = cid + ((n + 1 + 63) & ~int64_t(63));
    uint32_t *d_total = misc, *d_flags = misc + 2, *d_lev = misc + 2 + kMaxRounds;
    HOP_CUDA(c, cudaMemsetAsync(misc, 0, (size_t)(2 + kMaxRounds + kLev) * sizeof(uint32_t), c->stream));
    sub_root_flag_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(chain, dkey, n, d_o, cid, c->d_err);
    HOP_LAUNCH(c);
    rc = scan_exclusive_u32(c, cid, cid, n, d_total);
    if (rc) return rc;
    sub_particle_chain_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(chain, dkey, n, d_o, cid, pc, c->d_err);
    HOP_LAUNCH(c);
    HOP_CUDA(c, cudaMemcpyAsync(hp, misc, 4, cudaMemcpyDeviceToHost, c->stream));
    HOP_CUDA(c, cudaStreamSynchronize(c->stream));
    const int64_t C = hp[0];
    // thresholds per batch: at most kLev, fewer where the arrays over (level,
    // chain) would grow past 2^28 entries, or past the memory that is left
    const int64_t Cp = std::max<int64_t>(C, 1), mp = std::max<int64_t>(m, 1);
    int LB = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(L, kLev), (int64_t(1) << 28) / Cp));
    const bool with_sum = f > 0.0 || n >= (int64_t(1) << 29);
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += align256(bytes); return o; };
    // what does not depend on LB first
    const size_t o_cnt = take(Cp * kLev * 4), o_sum = take(with_sum ? Cp * kLev * 8 : 8), o_pkey = take(Cp * 8),
                 o_row = take(Cp * kLev * 4), o_ea = take(mp * 4), o_eb = take(mp * 4), o_gk = take(Cp * 8),
                 o_gkb = take(Cp * 8), o_gv = take(Cp * 4), o_gvb = take(Cp * 4),
                 o_tmp = take(radix_sort_scratch_bytes(Cp)), fixed = off;
    size_t o_parent, o_ccnt, o_csum, o_cpk, o_flag, o_pos, o_rank;
    char *base = nullptr;
    for (;; LB = (LB + 1) / 2) {
        off = fixed;
        o_parent = take(Cp * LB * 4);
        o_ccnt = take(Cp * LB * 8);
        o_csum = take(with_sum ? Cp * LB * 8 : 8);
        o_cpk = take(Cp * LB * 8);
        o_flag = take((Cp * LB + 1) * 4);
        o_pos = take((Cp * LB + 1) * 4);
        o_rank = take(Cp * LB * 4);
        base = (char *)ctx_buf(c, S_SUB_C, off);
        if (base || LB == 1) break;
    }
    if (!base) return HOP_ENOMEM;
    c->err.clear();
    uint32_t *cnt = (uint32_t *)(base + o_cnt), *parent = (uint32_t *)(base + o_parent),
             *flag = (uint32_t *)(base + o_flag), *gpos = (uint32_t *)(base + o_pos), *ea = (uint32_t *)(base + o_ea),
             *eb = (uint32_t *)(base + o_eb);
    int32_t *row = (int32_t *)(base + o_row), *rank = (int32_t *)(base + o_rank);
    unsigned long long *pkey = (unsigned long long *)(base + o_pkey), *ccnt = (unsigned long long *)(base + o_ccnt),
                       *cpk = (unsigned long long *)(base + o_cpk);
    double *sum = with_sum ? (double *)(base + o_sum) : nullptr, *csum = with_sum ? (double *)(base + o_csum) : nullptr;
    uint64_t *gk = (uint64_t *)(base + o_gk), *gkb = (uint64_t *)(base + o_gkb);
    uint32_t *order = (uint32_t *)(base + o_gv), *gvb = (uint32_t *)(base + o_gvb);
    void *tmp = base + o_tmp;
    if (m > 0) {
        sub_edge_ids_kernel<<<grid_for(c, m), 256, 0, c->stream>>>(ek, m, n, chain, dkey, d_o, cid, ea, eb, c->d_err);
        HOP_LAUNCH(c);
    }
    rc = ctx_check_device_error(c);
    if (rc) return rc;
    c->stats.n_chains = C;
    c->stats.n_edges = m;
    if (C == 0) {
        HOP_CUDA(c, cudaMemsetAsync(sub, 0xFF, (size_t)L * n * sizeof(int32_t), c->stream));
        for (int l = 0; l < L; ++l) n_sub[l] = 0;
        return HOP_OK;
    }
    // Rounds run without host round trips except the convergence test, read
    // once per kRoundBatch rounds (rounds after convergence change nothing).
    constexpr int kRoundBatch = 4;
    for (int l0 = 0; l0 < L; l0 += LB) {
        Levels lev;
        lev.L = std::min(LB, L - l0);
        for (int l = 0; l < kLev; ++l) lev.ds[l] = l < lev.L ? levels[l0 + l] : INFINITY;
        const int64_t CL = C * lev.L;
        // S3 (the keys and their order are the same for every batch)
        HOP_CUDA(c, cudaMemsetAsync(cnt, 0, C * kLev * 4, c->stream));
        if (sum) HOP_CUDA(c, cudaMemsetAsync(sum, 0, C * kLev * 8, c->stream));
        if (l0 == 0) {
            sub_root_key_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(chain, dkey, n, pc, pkey);
            HOP_LAUNCH(c);
        }
        if (sum)
            sub_chain_stats_kernel<true><<<grid_for(c, n), 256, 0, c->stream>>>(dkey, pc, n, lev, cnt, sum, pkey);
        else
            sub_chain_stats_kernel<false><<<grid_for(c, n), 256, 0, c->stream>>>(dkey, pc, n, lev, cnt, sum, pkey);
        HOP_LAUNCH(c);
        if (l0 == 0) {
            uint64_t *k0 = gk, *k1 = gkb;
            sub_keys_kernel<<<grid_for(c, C), 256, 0, c->stream>>>(pkey, C, k0, order);
            HOP_LAUNCH(c);
            rc = radix_sort_u64(c, k0, k1, order, gvb, C, 0, 64, tmp);
            if (rc) return rc;
        }
        // S4
        sub_iota_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(parent, C, lev.L);
        HOP_LAUNCH(c);
        int rounds = 0;
        bool converged = m == 0;
        while (!converged) {
            if (rounds + kRoundBatch > kMaxRounds) return ctx_fail(c, HOP_ETIMEOUT, "subhalo components did not converge");
            HOP_CUDA(c, cudaMemsetAsync(d_flags + rounds, 0, kRoundBatch * sizeof(uint32_t), c->stream));
            for (int b = 0; b < kRoundBatch; ++b, ++rounds) {
                sub_hook_kernel<<<grid_for(c, m), 256, 0, c->stream>>>(ea, eb, es, m, lev, C, parent, d_flags + rounds);
                HOP_LAUNCH(c);
                sub_compress_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(parent, C, lev.L);
                HOP_LAUNCH(c);
            }
            HOP_CUDA(c, cudaMemcpyAsync(hp + 1, d_flags + rounds - 1, 4, cudaMemcpyDeviceToHost, c->stream));
            HOP_CUDA(c, cudaStreamSynchronize(c->stream));
            converged = hp[1] == 0;
        }
        // S5, S6, S7
        HOP_CUDA(c, cudaMemsetAsync(ccnt, 0, CL * 8, c->stream));
        if (csum) HOP_CUDA(c, cudaMemsetAsync(csum, 0, CL * 8, c->stream));
        HOP_CUDA(c, cudaMemsetAsync(cpk, 0, CL * 8, c->stream));
        HOP_CUDA(c, cudaMemsetAsync(rank, 0xFF, CL * 4, c->stream));
        sub_component_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(cnt, sum, pkey, C, lev.L, parent, ccnt, csum, cpk);
        HOP_LAUNCH(c);
        sub_flag_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(order, pkey, C, lev, parent, ccnt, csum, cpk,
                                                                (long long)n_min, f, flag);
        HOP_LAUNCH(c);
        rc = scan_exclusive_u32(c, flag, gpos, CL, nullptr);
        if (rc) return rc;
        sub_rank_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(order, flag, gpos, C, lev.L, parent, rank, d_lev);
        HOP_LAUNCH(c);
        sub_row_kernel<<<grid_for(c, CL), 256, 0, c->stream>>>(rank, parent, C, lev.L, row);
        HOP_LAUNCH(c);
        sub_label_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(dkey, pc, n, lev, row, sub + (int64_t)l0 * n);
        HOP_LAUNCH(c);
        HOP_CUDA(c, cudaMemcpyAsync(hp + 2, d_lev, lev.L * sizeof(uint32_t), cudaMemcpyDeviceToHost, c->stream));
        HOP_CUDA(c, cudaStreamSynchronize(c->stream));
        for (int l = 0; l < lev.L; ++l) n_sub[l0 + l] = (int64_t)hp[2 + l];
    }
    return HOP_OK;
}

}  // namespace

extern "C" int hop_subhalos(hop_ctx *c, const uint32_t *chain, const float *dens, const uint32_t *nbr,
                            int32_t ld_nbr, int64_t n, int32_t n_merge, float delta_outer, const float *levels,
                            int32_t n_levels, int64_t n_min, double f_poisson, int32_t *sub, int64_t *n_sub)
{
    if (!c) return HOP_EINVAL;
    c->err.clear();
    if (!chain || !dens || !nbr || !sub || !n_sub || !levels || n <= 0 || n_levels <= 0)
        return ctx_fail(c, HOP_EINVAL, "chain, dens, nbr, levels, sub, n_sub, n > 0 and n_levels > 0 are required");
    if (n >= (int64_t(1) << 31) - 1) return ctx_fail(c, HOP_EINVAL, "n must be < 2^31 - 1");
    if (n_merge < 1 || n_merge > ld_nbr) return ctx_fail(c, HOP_EINVAL, "n_merge must be in [1, ld_nbr]");
    if (n_min < 1) return ctx_fail(c, HOP_EINVAL, "n_min must be >= 1");
    if (!(f_poisson >= 0.0) || !std::isfinite(f_poisson)) return ctx_fail(c, HOP_EINVAL, "f_poisson must be >= 0");
    for (int l = 0; l < n_levels; ++l)
        if (!std::isfinite(levels[l]) || !(levels[l] >= delta_outer))
            return ctx_fail(c, HOP_EINVAL, "every level must be finite and >= delta_outer");
    HOP_CUDA(c, cudaSetDevice(c->device));
    const int64_t launches0 = c->launches;
    HOP_CUDA(c, cudaEventRecord(c->ev[0], c->stream));
    uint64_t *dkey = (uint64_t *)ctx_buf(c, S_DKEY, n * sizeof(uint64_t));
    if (!dkey) return HOP_ENOMEM;
    int rc = make_dkey(c, dens, nullptr, n, dkey);
    if (rc) return rc;
    rc = subhalos(c, chain, dens, dkey, nbr, ld_nbr, n, n_merge, delta_outer, levels, n_levels, n_min, f_poisson, sub,
                  n_sub);
    if (rc) return rc;
    HOP_CUDA(c, cudaEventRecord(c->ev[1], c->stream));
    const int e = ctx_check_device_error(c);
    float ms = 0.f, ms_b = 0.f;
    if (cudaEventElapsedTime(&ms, c->ev[0], c->ev[1]) != cudaSuccess) cudaGetLastError();
    if (cudaEventElapsedTime(&ms_b, c->ev[2], c->ev[3]) != cudaSuccess) cudaGetLastError();
    c->stats.ms_total = ms;
    c->stats.ms_boundaries = ms_b;
    c->stats.ms_merge = ms - ms_b;
    c->stats.launches = c->launches - launches0;
    return e;
}
