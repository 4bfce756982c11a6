// Certified cell-stencil kNN fused with the M4 cubic-spline density (HOP
// step 1, Parallel HOP Sec. 2) for float32 positions: four queries per warp,
// eight lanes per query.
//
// A warp takes four consecutive Morton-sorted particles.  Consecutive ones
// farther apart than the first radius (a jump of the Morton curve) are
// searched one after another, the others together:
//   1. Cells.  The cells (side about R / cpr) that meet the members' bounding
//      box grown by R are listed once for all of them; the Morton code and
//      the gap of each axis cell are computed by one lane each and combined
//      by shuffles.
//   2. Staging.  The lanes read the cells' particles, 128 per step (four
//      independent 16-byte loads per lane), and the ones within R of the box
//      go to a tile in shared memory.
//   3. Evaluation.  Lane p of a query takes every eighth staged particle; d^2
//      and sorted index of those within R go to the lane's own list, one
//      column of a [slot][lane] array, so that no two lanes meet in a bank
//      and no ballot is needed.  When a list is nearly full, the query's
//      limit drops to the upper edge of the bin holding its Ndens-th entry.
//   4. Selection.  A histogram of the query's lists (32 bins linear in d^2,
//      two 16-bit counts per word) places the entries up to the Ndens-th
//      bin, bin by bin, in one array (a counting sort).  The exact Ndens-th
//      d^2 is ranked within its bin, the density is a fixed-point sum over
//      the array, and an entry's place in the neighbour list is the start of
//      its bin plus its rank in it by (d^2, original index).
// A query is certified when at least Ndens particles lie within R; the
// others search again with a larger R.  What this kernel does not take -- a
// ball that wraps around the box, more cells than it lists, a crowd at the
// Ndens-th distance -- it hands over to the warp-per-query kernel
// (knn_cg.cu), which runs after it over the list of such queries.
//
// What bounds it: instruction issue and latency (2.0k warp instructions per
// particle, issue 43 % busy at 16 warps per SM; DRAM and tensor cores play no
// part).  Four queries share the cell listing and the reads that a warp per
// query repeats for each, and eight lanes per query keep private lists, which
// need no ballots.  Kernel time against a warp per query (3.7k instructions),
// learned first radius unless stated: 16.8M particles 82.1 -> 68.4 ms, 64
// subvolumes of 22M together 111.8 -> 86.2 ms, 3M with Ndens = Nhop = 65
// (closed form) 22.2 -> 15.3 ms, 4,913 particles 0.99 -> 0.40 ms.
//
// Results equal those of the other kNN kernels bit for bit: the same
// per-component minimum-image differences, the same fused d^2, the same
// exact Ndens-th distance, list order and fixed-point density sum.
#include "hop_internal.cuh"
#include "knn_common.cuh"

#include <algorithm>
#include <math.h>

namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr int kGqWarps = 4;            // warps per block
constexpr int kGqQ = 4;                // queries per warp (eight lanes each)
constexpr int kGqSlots = 32;           // list entries per lane
constexpr int kGqTile = 160;           // staged particles
constexpr int kGqCells = 128;          // cells held at once
constexpr int kGqAxis = 10;            // axis cells of a region, at most
constexpr int kGqBins = 32;            // histogram bins, linear in d^2
constexpr int kGqTries = 96;

struct GqDev {
    const float4 *spos;
    const uint64_t *keys;
    const uint32_t *cellT;
    int level_dense;
    int64_t n, n_groups;
    int gpc;                           // groups per radius chunk
    float box, norm, cells_per_box;
    int k, n_out, ld_out, capq;
    const float *chunk_r;
    float plain_r;
    const SegDesc *seg;
    int B;
    uint32_t *nbr_s;
    float *dens_s;
    float *rk_s;
    uint32_t *hand;                    // queries handed over ...
    unsigned long long *hand_n;        // ... and their number
    unsigned long long *group_counter, *counters;
    uint32_t *err;
};

// Shared memory of one warp, byte offsets.  The cells and the tile (search)
// share their space with the sorted arrays (selection).
struct GqSmem {
    static constexpr int ld = 0;                                    // [kGqSlots][32] d^2
    static constexpr int ls = ld + kGqSlots * 128;                  // [kGqSlots][32] sorted index
    static constexpr int hist = ls + kGqSlots * 128;                // [kGqBins / 2][32] two 16-bit counts
    static constexpr int bst = hist + kGqBins / 2 * 128;            // [kGqQ][kGqBins + 2] u16 bin starts
    static constexpr int cra = (bst + kGqQ * (kGqBins + 2) * 2 + 15) & ~15;   // kGqCells range starts
    static constexpr int cpre = cra + kGqCells * 4;                 // kGqCells + 4 prefix offsets
    static constexpr int tile = cpre + (kGqCells + 4) * 4;          // kGqTile float4
    static_assert(tile % 16 == 0, "the tile is read 16 bytes at a time");
    __host__ __device__ static int total(int capq)
    {
        const int search = tile + kGqTile * 16, sel = cra + kGqQ * capq * 8;
        return ((search > sel ? search : sel) + 15) & ~15;
    }
};

__device__ __forceinline__ float quad_min(float v)
{
    v = fminf(v, __shfl_xor_sync(kAll, v, 8));
    return fminf(v, __shfl_xor_sync(kAll, v, 16));
}
__device__ __forceinline__ float quad_max(float v)
{
    v = fmaxf(v, __shfl_xor_sync(kAll, v, 8));
    return fmaxf(v, __shfl_xor_sync(kAll, v, 16));
}
// Sum over the eight lanes of a query.
__device__ __forceinline__ int oct_sum(int v)
{
    v += __shfl_xor_sync(kAll, v, 1);
    v += __shfl_xor_sync(kAll, v, 2);
    return v + __shfl_xor_sync(kAll, v, 4);
}

__device__ __forceinline__ int gq_bin(float d2, float scale) { return min((int)(d2 * scale), kGqBins - 1); }

// Counts the lanes' lists into the histogram and finds, for each query, the
// bin of the rank-th entry: packed as bin << 20 | below << 10 | upto (0 when
// the lists hold fewer).  With `place` the histogram words become the
// positions at which each lane's entries of a bin go, and bst the bins'
// starts.
struct GqFound {
    uint32_t k, o;
};
template <bool PLACE>
__device__ __forceinline__ GqFound gq_count(const float *Ld, uint32_t *hist, uint16_t *bst, int cnt, int cmax,
                                            float scale, int k, int n_out, int lane)
{
    const int q = lane >> 3, p = lane & 7;
#pragma unroll
    for (int i = 0; i < kGqBins / 2 * 32 / 128; ++i)
        reinterpret_cast<uint4 *>(hist)[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    for (int i = 0; i < cmax; ++i) {
        if (i < cnt) {
            const int b = gq_bin(Ld[i * 32], scale);
            hist[(b >> 1) * 32 + lane] += 1u << ((b & 1) * 16);
        }
    }
    __syncwarp();
    // lane p holds bins 4p .. 4p + 3 (words 2p, 2p + 1) of its query; column
    // r of the query's eight is read in an order of each lane's own, so that
    // the lanes read distinct banks
    uint32_t *w0 = hist + 2 * p * 32 + q * 8, *w1 = w0 + 32;
    uint32_t s0 = 0, s1 = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int c = (r + p) & 7;
        s0 += w0[c];
        s1 += w1[c];
    }
    const int n0 = s0 & 0xffffu, n1 = s0 >> 16, n2 = s1 & 0xffffu, n3 = s1 >> 16;
    int incl = n0 + n1 + n2 + n3;
    const int tot = incl;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o, 8);
        if (p >= o) incl += y;
    }
    const int b0 = incl - tot, b1 = b0 + n0, b2 = b1 + n1, b3 = b2 + n2, b4 = incl;
    auto find = [&](int rank) {
        uint32_t v = 0;
        const bool has = b0 < rank && rank <= b4;
        if (has) {
            int bin = 4 * p, lo = b0, hi = b1;
            if (rank > b1) { bin = 4 * p + 1; lo = b1; hi = b2; }
            if (rank > b2) { bin = 4 * p + 2; lo = b2; hi = b3; }
            if (rank > b3) { bin = 4 * p + 3; lo = b3; hi = b4; }
            v = ((uint32_t)bin << 20) | ((uint32_t)lo << 10) | (uint32_t)hi;
        }
        const uint32_t m = (__ballot_sync(kAll, has) >> (q * 8)) & 0xffu;
        v = __shfl_sync(kAll, v, q * 8 + (m ? __ffs(m) - 1 : 0));
        return m ? v : 0u;
    };
    GqFound f;
    f.k = find(k);
    f.o = n_out > 0 ? find(n_out) : 0u;
    if constexpr (PLACE) {
        uint32_t r0 = (uint32_t)b0 | ((uint32_t)b1 << 16), r1 = (uint32_t)b2 | ((uint32_t)b3 << 16);
        uint16_t *t = bst + q * (kGqBins + 2) + 4 * p;
        t[0] = (uint16_t)b0;
        t[1] = (uint16_t)b1;
        t[2] = (uint16_t)b2;
        t[3] = (uint16_t)b3;
        if (p == 7) t[4] = (uint16_t)b4;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int c = (r + p) & 7;
            const uint32_t x0 = w0[c], x1 = w1[c];
            w0[c] = r0;
            w1[c] = r1;
            r0 += x0;
            r1 += x1;
        }
        __syncwarp();
    }
    return f;
}

// The largest d^2 of bin `bin`, rounded up: every value above it falls in a
// later bin.
__device__ __forceinline__ float gq_edge(int bin, float scale) { return (float)(bin + 1) / scale * 1.000001f; }

// Drops the limit of every query that holds at least k entries (and is in
// `which`) to the upper edge of the bin of its k-th, and its lists to the
// entries up to it.  Out of line: only lists that are nearly full, or a
// crowded k-th bin, need it.
__device__ __noinline__ void gq_tighten(float *Ld, uint32_t *Ls, uint32_t *hist, bool which, int &cnt, float &tau, int k,
                                        int lane)
{
    const int cmax = (int)__reduce_max_sync(kAll, (unsigned)cnt);
    const float scale = (float)kGqBins / tau;
    const GqFound f = gq_count<false>(Ld, hist, nullptr, which ? cnt : 0, cmax, scale, k, 0, lane);
    if (which && f.k) {
        const float e = fminf(tau, gq_edge((int)(f.k >> 20), scale));
        int m = 0;
        for (int i = 0; i < cnt; ++i) {
            const float v = Ld[i * 32];
            const uint32_t s = Ls[i * 32];
            if (v <= e) {
                Ld[m * 32] = v;
                Ls[m * 32] = s;
                ++m;
            }
        }
        cnt = m;
        tau = e;
    }
    __syncwarp();
}

// Lists the non-empty cells of level l that meet the box [fl, fh] grown by
// r; returns their count, or -1 if an axis or the list is too long.
__device__ __forceinline__ int gq_cells(float flx, float fhx, float fly, float fhy, float flz, float fhz, float r,
                                        float box, int l, const uint32_t *__restrict__ cellT,
                                        const uint64_t *__restrict__ keys, int level_dense, uint32_t *cra, uint32_t *cln,
                                        int lane, uint32_t lt)
{
    const int G = 1 << l;
    const float csz = box / (float)G, sc = (float)G / box;
    const float eps = box * 9.5367431640625e-7f;   // 2^-20 of the box: far above coordinate rounding
    const float r2c = r * r * 1.00001f + box * box * 1e-12f;
    // lane 10 a + i: cell i of axis a
    const int ax = lane < kGqAxis ? 0 : lane < 2 * kGqAxis ? 1 : 2;
    const float fl = ax == 0 ? flx : ax == 1 ? fly : flz, fh = ax == 0 ? fhx : ax == 1 ? fhy : fhz;
    const int c0 = (int)floorf((fl - r - eps) * sc), na = (int)floorf((fh + r + eps) * sc) - c0 + 1;
    const int nx = __shfl_sync(kAll, na, 0), ny = __shfl_sync(kAll, na, kGqAxis), nz = __shfl_sync(kAll, na, 2 * kGqAxis);
    if (max(nx, max(ny, nz)) > min(kGqAxis, G)) return -1;
    const int ca = c0 + (lane - kGqAxis * ax);
    const float gap = fmaxf(0.f, fmaxf(fl - (float)(ca + 1) * csz, (float)ca * csz - fh) - eps);
    const float gap2 = gap * gap;
    const uint32_t cw = (uint32_t)ca & (uint32_t)(G - 1);
    const uint32_t m0 = spread3_8(cw) << ax, m1 = spread3_8(cw >> 8) << ax;
    const int nxy = nx * ny, ncube = nxy * nz;
    // cell ci of the cube is (ci mod nx, (ci / nx) mod ny, ci / (nx ny)); the
    // quotients come from float reciprocals, exact for these small integers
    const float inx = 1.f / (float)nx, inxy = 1.f / (float)nxy;
    int nkeep = 0;
    for (int cb = 0; cb < ncube; cb += 32) {
        const int ci = cb + lane, cc = min(ci, ncube - 1);
        const int iz = (int)(((float)cc + 0.5f) * inxy);
        const int rxy = cc - iz * nxy;
        const int iy = (int)(((float)rxy + 0.5f) * inx);
        const int ix = rxy - iy * nx;
        const int jy = iy + kGqAxis, jz = iz + 2 * kGqAxis;
        const float g2 = __shfl_sync(kAll, gap2, ix) + __shfl_sync(kAll, gap2, jy) + __shfl_sync(kAll, gap2, jz);
        const uint32_t lo = __shfl_sync(kAll, m0, ix) | __shfl_sync(kAll, m0, jy) | __shfl_sync(kAll, m0, jz);
        const uint32_t hi = __shfl_sync(kAll, m1, ix) | __shfl_sync(kAll, m1, jy) | __shfl_sync(kAll, m1, jz);
        uint32_t ra = 0, rb = 0;
        if (ci < ncube && g2 <= r2c) cell_range(cellT, keys, level_dense, l, ((uint64_t)hi << 24) | lo, ra, rb);
        const uint32_t bal = __ballot_sync(kAll, rb > ra);
        const int pos = nkeep + __popc(bal & lt);
        if (rb > ra && pos < kGqCells) {
            cra[pos] = ra;
            cln[pos] = rb - ra;
        }
        nkeep += __popc(bal);
        if (nkeep > kGqCells) break;
    }
    __syncwarp();
    return nkeep <= kGqCells ? nkeep : -1;
}

// Turns the nc cell lengths in cpre into their exclusive prefix, cpre[nc] the
// total (returned); four cells per lane.
__device__ __forceinline__ uint32_t gq_prefix(uint32_t *cpre, int nc, int lane)
{
    static_assert(kGqCells == 128, "four cells per lane");
    const uint4 v = reinterpret_cast<const uint4 *>(cpre)[lane];
    const int j = 4 * lane;
    const uint32_t a = j < nc ? v.x : 0u, b = j + 1 < nc ? v.y : 0u, c = j + 2 < nc ? v.z : 0u, d = j + 3 < nc ? v.w : 0u;
    const uint32_t mine = a + b + c + d;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t e = incl - mine, total = __shfl_sync(kAll, incl, 31);
    __syncwarp();
    reinterpret_cast<uint4 *>(cpre)[lane] = make_uint4(e, e + a, e + a + b, e + a + b + c);
    if (lane == 0) cpre[kGqCells] = total;   // read as cpre[nc] when every cell is in use
    __syncwarp();
    return total;
}

template <bool SEG>
__global__ void __launch_bounds__(kGqWarps * 32, 4) knn_gq_kernel(GqDev a)
{
    using L = GqSmem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int q = lane >> 3, p = lane & 7;
    const uint32_t lt = (1u << lane) - 1u;
    unsigned char *wb = smem_raw + L::total(a.capq) * (threadIdx.x >> 5);
    float *Ld = (float *)(wb + L::ld) + lane;
    uint32_t *Ls = (uint32_t *)(wb + L::ls) + lane;
    uint32_t *hist = (uint32_t *)(wb + L::hist);
    uint16_t *bst = (uint16_t *)(wb + L::bst);
    uint32_t *cra = (uint32_t *)(wb + L::cra), *cpre = (uint32_t *)(wb + L::cpre);
    float4 *tile = (float4 *)(wb + L::tile);
    float *Dd = (float *)(wb + L::cra) + q * a.capq;
    uint32_t *Ds = (uint32_t *)(wb + L::cra) + (kGqQ + q) * a.capq;
    const int k = a.k, n_out = a.nbr_s ? a.n_out : 0;
    unsigned long long cand_acc = 0;
    uint32_t search_acc = 0, retry_acc = 0, warp_acc = 0;

    for (;;) {
        unsigned long long gr = 0;
        if (lane == 0) gr = atomicAdd(a.group_counter, 1ull);
        gr = __shfl_sync(kAll, gr, 0);
        if ((int64_t)gr >= a.n_groups) break;
        const int64_t ch = (int64_t)gr / a.gpc;
        int64_t s_first, n_end;
        float box, norm, R0;
        const uint32_t *cellT;
        int level_dense;
        if constexpr (SEG) {
            const SegDesc &sd = a.seg[seg_of_chunk(a.seg, a.B, ch)];
            n_end = sd.base + sd.n;
            s_first = sd.base + ((int64_t)gr - sd.chunk0 * a.gpc) * kGqQ;
            box = (float)sd.box;
            norm = (float)sd.norm;
            cellT = a.cellT + sd.cell0;
            level_dense = sd.level_dense;
            R0 = sd.plain_r;
        } else {
            n_end = a.n;
            s_first = (int64_t)gr * kGqQ;
            box = a.box;
            norm = a.norm;
            cellT = a.cellT;
            level_dense = a.level_dense;
            R0 = a.plain_r;
        }
        const int nq = (int)min((int64_t)kGqQ, n_end - s_first);
        if (nq <= 0) continue;   // the last chunk of a subvolume may hold fewer groups
        ++warp_acc;
        if (a.chunk_r) R0 = a.chunk_r[ch];
        if (!(R0 > 0.f)) R0 = box * 1e-6f;
        const float half = 0.5f * box;
        const float eps = box * 9.5367431640625e-7f;
        const int64_t sq = s_first + min(q, nq - 1);
        float qx, qy, qz;
        {
            const float4 v = a.spos[sq];
            qx = v.x;
            qy = v.y;
            qz = v.z;
        }
        // a query farther than R0 from the one before it starts a new search
        const float ex = qx - __shfl_up_sync(kAll, qx, 8), ey = qy - __shfl_up_sync(kAll, qy, 8),
                    ez = qz - __shfl_up_sync(kAll, qz, 8);
        const uint32_t cuts = __ballot_sync(kAll, p == 0 && q > 0 && q < nq && ex * ex + ey * ey + ez * ez > R0 * R0);
        int g0 = 0;
        while (g0 < nq) {
            const uint32_t rest = cuts & (kAll << (g0 * 8)) & ~(1u << (g0 * 8));
            const int g1 = rest ? (__ffs(rest) - 1) >> 3 : nq;
            bool member = q >= g0 && q < g1;   // still to be served
            g0 = g1;
            float R = R0;
            int tries = 0;
            for (;;) {
                // ------------- the region: the members' box, grown by R
                float flx = quad_min(member ? qx : INFINITY), fhx = quad_max(member ? qx : -INFINITY);
                float fly = quad_min(member ? qy : INFINITY), fhy = quad_max(member ? qy : -INFINITY);
                float flz = quad_min(member ? qz : INFINITY), fhz = quad_max(member ? qz : -INFINITY);
                // where it crosses a face, coordinates >= L/2 move by -L (exact)
                const bool wx = flx - R < 0.f || fhx + R >= box, wy = fly - R < 0.f || fhy + R >= box,
                           wz = flz - R < 0.f || fhz + R >= box;
                const bool mixed = (wx && flx - R < half && half <= fhx + R) || (wy && fly - R < half && half <= fhy + R) ||
                                   (wz && flz - R < half && half <= fhz + R);
                float fx = qx, fy = qy, fz = qz;
                const bool shifted = wx || wy || wz;
                if (shifted) {
                    if (wx && qx >= half) fx = qx - box;
                    if (wy && qy >= half) fy = qy - box;
                    if (wz && qz >= half) fz = qz - box;
                    flx = quad_min(member ? fx : INFINITY);
                    fhx = quad_max(member ? fx : -INFINITY);
                    fly = quad_min(member ? fy : INFINITY);
                    fhy = quad_max(member ? fy : -INFINITY);
                    flz = quad_min(member ? fz : INFINITY);
                    fhz = quad_max(member ? fz : -INFINITY);
                }
                bool give_up = 2.f * R >= half || mixed || tries >= kGqTries;
                uint32_t total = 0;
                int nc = 0;
                if (!give_up) {
                    // the finest level whose cells have a side of at least R / cells_per_box ...
                    const float cells = box * a.cells_per_box / R;
                    int l = min(max((int)((__float_as_uint(cells) >> 23) & 0xFFu) - 127, 1), kMaxLevel);
                    for (;;) {
                        nc = gq_cells(flx, fhx, fly, fhy, flz, fhz, R, box, l, cellT, a.keys, level_dense, cra, cpre,
                                      lane, lt);
                        if (nc >= 0 || l <= 1) break;
                        --l;   // too many cells meet the region: take coarser ones
                    }
                    give_up = nc < 0;
                }
                if (give_up) {
                    if (member && p == 0) a.hand[atomicAdd(a.hand_n, 1ull)] = (uint32_t)sq;
                    break;
                }
                total = gq_prefix(cpre, nc, lane);
                ++search_acc;
                // ------------- stage and evaluate
                int cnt = 0, m = 0;
                float tau = member ? R * R : -1.f;
                bool crowd = false;
                {
                    const float lx = flx - eps, hx = fhx + eps, ly = fly - eps, hy = fhy + eps, lz = flz - eps, hz = fhz + eps;
                    const float r2c = R * R * 1.00001f + box * box * 1e-12f;
                    const uint32_t upto_lane = lane == 31 ? kAll : ((2u << lane) - 1u);
                    const int nmem = __popc(__ballot_sync(kAll, member)) >> 3;
                    int cbase = -1;   // the cell holding particle g - 1
                    for (uint32_t g = 0; g < total; g += 128) {
                        uint32_t s[4];
                        float4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            // the cell of each lane's particle, from the cell
                            // starts inside the window (one bit each)
                            const uint32_t w0 = g + 32 * u;
                            const int j = cbase + 1 + lane;
                            const uint32_t st = j < nc ? cpre[j] : total;
                            const uint32_t bit = (st >= w0 && st < w0 + 32) ? 1u << (st - w0) : 0u;
                            const uint32_t starts = __reduce_or_sync(kAll, bit);
                            const int c = cbase + __popc(starts & upto_lane);
                            const uint32_t gi = w0 + (uint32_t)lane;
                            s[u] = gi < total ? cra[c] + (gi - cpre[c]) : 0xffffffffu;
                            cbase += __popc(starts);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            v[u] = s[u] != 0xffffffffu ? a.spos[s[u]] : make_float4(INFINITY, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            float4 c = v[u];
                            if (shifted) {
                                if (wx && c.x >= half) c.x -= box;   // the padding's INFINITY stays one
                                if (wy && c.y >= half) c.y -= box;
                                if (wz && c.z >= half) c.z -= box;
                            }
                            const float gx = fmaxf(fmaxf(lx - c.x, c.x - hx), 0.f);
                            const float gy = fmaxf(fmaxf(ly - c.y, c.y - hy), 0.f);
                            const float gz = fmaxf(fmaxf(lz - c.z, c.z - hz), 0.f);
                            const bool keep = gx * gx + gy * gy + gz * gz <= r2c;
                            const uint32_t bal = __ballot_sync(kAll, keep);
                            c.w = __uint_as_float(s[u]);
                            if (keep) tile[m + __popc(bal & lt)] = c;
                            m += __popc(bal);
                        }
                        const bool last = g + 128 >= total;
                        if (m <= kGqTile - 128 && !last) continue;
                        if (last) {
                            // pad to a multiple of 32 with entries no test accepts
                            const float nan = __int_as_float(0x7fc00000);
                            if (lane < ((32 - (m & 31)) & 31)) tile[m + lane] = make_float4(nan, nan, nan, 0.f);
                            cand_acc += (unsigned long long)m * (unsigned long long)nmem;
                            m = (m + 31) & ~31;
                        } else {
                            cand_acc += (unsigned long long)(m & ~31) * (unsigned long long)nmem;
                        }
                        __syncwarp();
                        int j0 = 0;
                        for (; j0 + 32 <= m; j0 += 32) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const float4 c = tile[j0 + u * 8 + p];
                                const float dx = c.x - fx, dy = c.y - fy, dz = c.z - fz;
                                const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                                if (d2 <= tau) {
                                    Ld[cnt * 32] = d2;
                                    Ls[cnt * 32] = __float_as_uint(c.w);
                                    ++cnt;
                                }
                            }
                            if (__any_sync(kAll, cnt > kGqSlots - 4)) {
                                gq_tighten(Ld, Ls, hist, member && !crowd, cnt, tau, k, lane);
                                // a list that stays full: a crowd at the limit
                                const uint32_t f = __ballot_sync(kAll, cnt > kGqSlots - 4);
                                if ((f >> (q * 8)) & 0xffu) {
                                    crowd = true;
                                    cnt = 0;
                                    tau = -1.f;
                                }
                            }
                        }
                        m -= j0;
                        if (!last) {
                            // the remainder moves to the front
                            float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (lane < m) c = tile[j0 + lane];
                            __syncwarp();
                            if (lane < m) tile[lane] = c;
                        }
                        __syncwarp();
                    }
                }
                // ------------- selection
                const int tot = oct_sum(cnt);
                bool ok = member && !crowd && tot >= k;
                if (__any_sync(kAll, ok)) {
                    int cmax = 0;
                    float scale = 0.f;
                    GqFound f;
                    for (int it = 0;; ++it) {
                        cmax = (int)__reduce_max_sync(kAll, ok ? (unsigned)cnt : 0u);
                        scale = (float)kGqBins / tau;
                        f = gq_count<true>(Ld, hist, bst, ok ? cnt : 0, cmax, scale, k, n_out, lane);
                        const bool full = ok && (int)(f.k & 1023u) > a.capq;
                        if (!__any_sync(kAll, full)) break;
                        if (it == 3) {
                            // the bin stays crowded
                            if (full) {
                                ok = false;
                                crowd = true;
                            }
                            break;
                        }
                        gq_tighten(Ld, Ls, hist, full, cnt, tau, k, lane);
                    }
                    const int bk = (int)(f.k >> 20), below = (int)((f.k >> 10) & 1023u), upto = ok ? (int)(f.k & 1023u) : 0;
                    for (int i = 0; i < cmax; ++i) {
                        if (ok && i < cnt) {
                            const float v = Ld[i * 32];
                            const int b = gq_bin(v, scale);
                            if (b <= bk) {
                                uint32_t *w = hist + (b >> 1) * 32 + lane;
                                const uint32_t x = *w;
                                const int pos = (int)((x >> ((b & 1) * 16)) & 0xffffu);
                                *w = x + (1u << ((b & 1) * 16));
                                Dd[pos] = v;
                                Ds[pos] = Ls[i * 32];
                            }
                        }
                    }
                    __syncwarp();
                    // the exact k-th d^2, within its bin
                    float vk = -1.f;
                    for (int e = below + p; e < upto; e += 8) {
                        const float v = Dd[e];
                        int l0 = below, le = below;
                        for (int h = below; h < upto; ++h) {
                            const float u = Dd[h];
                            l0 += u < v;
                            le += u <= v;
                        }
                        if (l0 < k && k <= le) vk = v;
                    }
                    __syncwarp();
                    vk = fmaxf(vk, __shfl_xor_sync(kAll, vk, 1));
                    vk = fmaxf(vk, __shfl_xor_sync(kAll, vk, 2));
                    vk = fmaxf(vk, __shfl_xor_sync(kAll, vk, 4));
                    // density: fixed-point sum of w(2 r / r_k) over entries with d^2 < r_k^2
                    const float rk = sqrtf(vk);
                    const float inv_h = vk > 0.f ? 2.f / rk : 0.f;
                    unsigned long long wsum = 0;
                    for (int e = p; e < upto; e += 8) {
                        const float v = Dd[e];
                        if (v < vk) {
                            const float w = m4<float>(sqrtf(v) * inv_h);
                            wsum += (unsigned long long)(w * 4294967296.0f + 0.5f);
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) wsum += __shfl_xor_sync(kAll, wsum, o);
                    if (ok && p == 0) {
                        float dens;
                        if (vk > 0.f) {
                            const float h = rk * 0.5f;
                            dens = (float)(norm * ((float)wsum * 2.3283064365386963e-10f) / (h * h * h));
                        } else {
                            dens = INFINITY;
                        }
                        a.dens_s[sq] = dens;
                        if (a.rk_s) a.rk_s[sq] = rk;
                    }
                    // the n_out nearest by (d^2, original index): the start of
                    // the entry's bin and its rank in it
                    if (n_out > 0) {
                        const int upto_o = ok ? (int)(f.o & 1023u) : 0;
                        const uint16_t *t = bst + q * (kGqBins + 2);
                        uint32_t *row = a.nbr_s + (size_t)sq * a.ld_out;
                        for (int e = p; e < upto_o; e += 8) {
                            const float v = Dd[e];
                            const uint32_t se = Ds[e];
                            const int b = gq_bin(v, scale);
                            const int h0 = t[b], h1 = t[b + 1];
                            int rank = h0;
                            for (int h = h0; h < h1; ++h) {
                                const float u = Dd[h];
                                rank += u < v;
                                if (u == v && h != e)
                                    rank += __float_as_uint(a.spos[Ds[h]].w) < __float_as_uint(a.spos[se].w);
                            }
                            if (rank < n_out) row[rank] = se;
                        }
                    }
                    __syncwarp();
                }
                if (member && crowd && p == 0) a.hand[atomicAdd(a.hand_n, 1ull)] = (uint32_t)sq;
                member = member && !ok && !crowd;
                if (!__any_sync(kAll, member)) break;
                // the others: too few within R
                ++retry_acc;
                ++tries;
                const float grow = member ? fmaxf(1.25f, 1.1f * cbrtf((float)k / (float)max(tot, 1))) : 1.25f;
                R *= fminf(quad_max(grow), 8.f);
                __syncwarp();
            }
        }
    }
    if (lane == 0) {
        atomicAdd(&a.counters[kCntCand], cand_acc);
        atomicAdd(&a.counters[kCntSearch], (unsigned long long)search_acc);
        atomicAdd(&a.counters[kCntRetry], (unsigned long long)retry_acc);
        atomicAdd(&a.counters[kCntWarps], (unsigned long long)warp_acc);
    }
}

template <bool SEG> int knn_gq_run(hop_ctx *c, const KnnArgs &ka, int qpw, int cpr)
{
    GqDev d;
    d.spos = (const float4 *)ka.spos;
    d.keys = ka.keys;
    d.cellT = ka.cellT;
    d.level_dense = ka.level_dense;
    d.n = ka.n;
    d.gpc = qpw / kGqQ;
    d.n_groups = SEG ? ka.n_chunks * d.gpc : (ka.n + kGqQ - 1) / kGqQ;
    d.box = (float)ka.box;
    d.norm = (float)(ka.box * ka.box * ka.box / ((double)(ka.n_norm > 0 ? ka.n_norm : ka.n) * 3.14159265358979323846));
    d.cells_per_box = (float)std::min(std::max(cpr, 1), 3);
    d.k = ka.k;
    d.n_out = ka.n_out;
    d.ld_out = ka.ld_out;
    d.capq = ((ka.k + 32 + 7) / 8) * 8;
    d.chunk_r = ka.chunk_r;
    d.plain_r = ka.plain_r;
    d.seg = ka.seg;
    d.B = ka.B;
    d.nbr_s = ka.nbr_s;
    d.dens_s = ka.dens_s;
    d.rk_s = ka.rk_s;
    d.counters = c->d_counters;
    d.group_counter = c->d_counters + kCntNum;
    d.hand_n = c->d_counters + kCntNum + 1;
    d.err = c->d_err;
    d.hand = (uint32_t *)ctx_buf(c, S_KNN_HAND, (size_t)ka.n * sizeof(uint32_t));
    if (!d.hand) return HOP_ENOMEM;
    HOP_CUDA(c, cudaMemsetAsync(d.group_counter, 0, 3 * sizeof(unsigned long long), c->stream));
    const size_t smem = (size_t)GqSmem::total(d.capq) * kGqWarps;
    auto kern = knn_gq_kernel<SEG>;
    HOP_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    HOP_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGqWarps * 32, smem));
    if (per_sm < 1) return ctx_fail(c, HOP_EINVAL, "kNN lists do not fit in shared memory");
    const int64_t need = (d.n_groups + kGqWarps - 1) / kGqWarps;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * c->num_sms, need));
    kern<<<(unsigned)blocks, kGqWarps * 32, smem, c->stream>>>(d);
    HOP_LAUNCH(c);
    return knn_wq_launch(c, ka, qpw, cpr, d.hand, d.hand_n, d.hand_n + 1);
}

}  // namespace

int knn_gq_launch(hop_ctx *c, const KnnArgs &a, int qpw, int cpr)
{
    if (qpw != 4 && qpw != 8 && qpw != 16)
        return ctx_fail(c, HOP_EINVAL, "the grouped kNN takes radius chunks of 4, 8 or 16 queries");
    return a.seg ? knn_gq_run<true>(c, a, qpw, cpr) : knn_gq_run<false>(c, a, qpw, cpr);
}
