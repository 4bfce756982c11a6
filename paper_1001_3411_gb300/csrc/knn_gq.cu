// Certified cell-stencil kNN fused with the M4 cubic-spline density (HOP
// step 1, Parallel HOP Sec. 2): four queries per warp, eight lanes per query.
// It serves float32 positions at 4, 8 and 16 queries per radius chunk and
// float64 positions at any number (searched in float32, decided in float64).
//
// A warp takes a unit of 16 consecutive Morton-sorted particles and serves
// them in four groups of four.  Consecutive ones farther apart than the
// first radius (a jump of the Morton curve) are searched one after another,
// the others of a group together:
//   1. Boxes, down to 512 particles.  The tree of bounding boxes over the
//      sorted particles (boxtree.cu) is walked once per unit, level by level,
//      32 boxes per step, to the 512-particle nodes that meet the unit's box
//      grown by its largest first radius.
//   2. Boxes, down to eight particles.  Of those, the nodes that meet the
//      group's box grown by R are opened, then the 64-particle nodes below
//      them; what is left is a list of runs of eight particles.
//   3. Evaluation.  The lanes read 16 runs at a time (four independent
//      16-byte loads each, the next 16 runs' in flight) and put the particles
//      within R of the group's box, fewer than half, in a tile in shared
//      memory.  Lane p of a query takes every eighth of the tile; d^2 and
//      sorted index of those within R go to the lane's own list, one column
//      of a [slot][lane] array: no two lanes meet in a bank and no ballot is
//      needed.  When a list is nearly full, the query's limit drops to the
//      upper edge of the bin holding its Ndens-th entry, divided again until
//      few others remain, and the reach of the box with it; where a region
//      meets many nodes the query's own comes first, so that this happens
//      early.
//   4. Selection.  A histogram of the query's lists (32 bins linear in d^2,
//      16-bit counts) places the entries up to the Ndens-th
//      bin, bin by bin, in one array (a counting sort).  The exact Ndens-th
//      d^2 is ranked within its bin, the density is a fixed-point sum over
//      the array, and an entry's place in the neighbour list is the start of
//      its bin plus its rank in it by (d^2, original index).
// A query is certified when at least Ndens particles lie within R; the
// others search again with a larger R.  A group whose region crosses both a
// face and L/2 is served one query at a time.  What this kernel does not take
// -- a ball that wraps around the box, a float32 box whose squares leave
// float32's range, more nodes than it lists at every radius that holds Ndens,
// more than 32 particles too many at the Ndens-th distance, float64 distances
// too close for float32 to bin -- it hands over to a warp-per-query kernel
// (knn_cg.cu; float64: knn.cu, and whole nodes of such particles four queries
// per warp), which runs after it over the list of such queries.  Such queries
// take 0.3 ms however few there are, and 2 to 8 ms where their radii are far
// too large, so radii reach the largest that does not wrap before one is
// handed over (4,913 particles: 0.37 -> 0.08 ms), and halve where a region
// meets too many nodes.  (Limits cut once instead, and no smaller radius:
// 4,200 of 16.8M queries handed over and 33.6 ms instead of 31.7, 14,700 of
// 2.1M with the plain radius and 19.1 ms instead of 7.4.)
//
// What bounds it: instruction issue and shared-memory wavefronts (58 % of
// issue slots and 66 % of wavefronts at 16 warps per SM, 1.35k warp
// instructions per particle); DRAM and tensor cores play no part.  Four
// queries share the walk and the reads that a warp per query repeats for
// each.  The code is kept small on purpose (loops not unrolled, one call site
// of what is long, rare parts out of line): at 55 KB instead of 42 KB
// instruction-cache misses were the largest stall and the 16.8M-particle kNN
// took 48.3 ms instead of 37.7.  Evaluating every particle of the runs (108
// per group) straight from cp.async buffers took 37.7 ms where the tile takes
// 33.6: a 16-byte read costs four wavefronts whether or not the four queries
// read the same words.
// Kernel time, with learned first radius unless stated (in brackets a warp
// per query): 16.8M particles 31.7 ms (82.1), 64 subvolumes of 22M together
// 43.6 ms (111.8), 3M with Ndens = Nhop = 65 (closed form) 7.0 ms (22.2), 2.1M
// with the plain radius 7.5 ms (59.2), 4,913 particles 0.08 ms (0.99), 32,768
// float64 particles 0.54 ms (5.2, the single-scan kernel).
//
// Results equal those of the other kNN kernels bit for bit: the same
// per-component minimum-image differences, the same fused d^2, the same
// exact Ndens-th distance, list order and fixed-point density sum.
#include "hop_internal.cuh"
#include "knn_common.cuh"

#include <algorithm>
#include <cmath>
#include <math.h>
#include <type_traits>

namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr int kGqWarps = 4;            // warps per block
constexpr int kGqQ = 4;                // queries per warp (eight lanes each)
constexpr int kGqSlots = 32;           // list entries per lane
constexpr int kGqUnit = 16;            // queries of a unit
constexpr int kGqN2 = 96;              // 512-particle nodes held
constexpr int kGqN1 = 192;             // 64-particle nodes held at once
constexpr int kGqN0 = 256;             // runs of eight particles held at once
constexpr int kGqBins = 32;            // histogram bins, linear in d^2
constexpr int kGqCutBins = 16;         // the same for a cut during the search
constexpr int kGqTile = 144;           // particles staged: 16 runs, and up to 15 left over
constexpr int kGqTries = 96;           // searches and halvings until some query of a group is done
// A region is grown by this much of the box whatever its radius: below it a
// smaller radius meets the same nodes.
constexpr float kGqFinest = 0x1p-20f;
// Float64 particles: within a ball of this radius the rounding's slack is more
// than a bin, whatever the limit.
constexpr float kGqFinest64 = 0x1p-15f;
// Box sides whose float32 squares stay in range: the largest square is 3 L^2
// (2^121.6), and the smallest margin of a box test, 1e-12 L^2, is still
// hundreds of denormal steps, far above the test's rounding.  Beyond them a
// limit could become infinite (and an infinite d^2 has no bin) or a neighbour
// be missed: float32 particles in such boxes go to the warp-per-query kernel,
// float64 ones are searched in units of the box.
constexpr float kGqBoxMin = 0x1p-50f, kGqBoxMax = 0x1p60f;

struct GqDev {
    const float4 *spos;
    const double4 *spos64;             // F64: the positions themselves
    BoxTree tree;
    uint32_t n, pad_run;               // pad_run: a run past the last particle
    int64_t n_tasks;                   // units of 16 queries, in `split` parts each
    int split;
    int qpw;                           // queries per radius chunk
    float box, norm;                   // F64: the box in the search's units, in [1, 2)
    double box64, norm64;
    float unit;                        // F64: the search's units per unit of the caller's
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
    uint32_t *runs;                    // F64: runs of four queries handed over ...
    unsigned long long *runs_n;        // ... and their number
    unsigned long long *task_counter, *counters;
};

// Shared memory of one warp, byte offsets.  The node lists (search) share
// their space with the sorted arrays (selection).
struct GqSmem {
    static constexpr int list = 0;                                  // [kGqSlots][32] d^2 and run
    static constexpr int hist = list + kGqSlots * 256;              // [kGqBins][32] u16 counts
    static constexpr int bst = hist + kGqBins * 64;                 // [kGqQ][kGqBins + 2] u16 bin starts
    static constexpr int u2 = (bst + kGqQ * (kGqBins + 2) * 2 + 15) & ~15;   // the unit's 512-particle nodes
    static constexpr int t0 = u2 + kGqN2 * 4;                       // a search's runs (read 16 bytes at a time) ...
    static constexpr int t1 = t0 + (kGqN0 + 16) * 4;                 // ... 64-particle nodes ...
    static constexpr int t2 = t1 + kGqN1 * 4;                       // ... and 512-particle nodes
    static constexpr int thist = t2 + kGqN2 * 4;                    // the histogram of a cut during the search
    static constexpr int search_end = thist + kGqCutBins * 64;
    // the particles in reach of a batch of runs share the space of hist and bst
    static constexpr int tile = hist;
    static_assert(kGqTile * 16 <= u2 - hist, "the tile fits");
    static_assert(t0 % 16 == 0, "runs are read 16 bytes at a time");
    // Row stride of the sorted arrays: 8 mod 32, so that the four queries'
    // lanes (eight consecutive words each) read distinct banks.
    __host__ __device__ static int stride(int capq) { return (capq + 23) / 32 * 32 + 8; }
    __host__ __device__ static int total(int capq, bool f64)
    {
        const int sel = t0 + kGqQ * stride(capq) * (f64 ? 12 : 8);
        return ((search_end > sel ? search_end : sel) + 15) & ~15;
    }
};

extern __shared__ __align__(16) unsigned char gq_smem[];

// Shared-memory byte address of an offset into gq_smem.
__device__ __forceinline__ uint32_t gq_addr(uint32_t o) { return (uint32_t)__cvta_generic_to_shared(gq_smem + o); }

// Appends (d2, sorted index) to the lane's list when d2 <= tau: one predicated store
// and one predicated add.
__device__ __forceinline__ void gq_keep(uint32_t &lp, float d2, float tau, uint32_t s)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.le.f32 p, %1, %2;\n\t@p st.shared.v2.b32 [%0], {%3, %4};\n\t"
                 "@p add.u32 %0, %0, 256;\n\t}"
                 : "+r"(lp)
                 : "f"(d2), "f"(tau), "r"(__float_as_uint(d2)), "r"(s)
                 : "memory");
}

__device__ __forceinline__ float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// A box grown by a radius: a node meets it when its distance from the box
// (made a little smaller, so that rounding never drops one) is within r.
// Where the grown box crosses a face, coordinates >= L/2 move by -L (exact),
// and a node is taken at both places.
struct Region {
    float lx, hx, ly, hy, lz, hz, r2c, box;
    bool wx, wy, wz, shifted;
    __device__ __forceinline__ static float gap(float lo, float hi, float l, float h)
    {
        return fmaxf(fmaxf(lo - h, l - hi), 0.f);
    }
    __device__ __forceinline__ bool meets(const float4 &lo, const float4 &hi) const
    {
        float gx = gap(lo.x, hi.x, lx, hx), gy = gap(lo.y, hi.y, ly, hy), gz = gap(lo.z, hi.z, lz, hz);
        if (shifted) {
            // (an axis that is not shifted takes the same place twice)
            const float bx = wx ? box : 0.f, by = wy ? box : 0.f, bz = wz ? box : 0.f;
            gx = fminf(gx, gap(lo.x - bx, hi.x - bx, lx, hx));
            gy = fminf(gy, gap(lo.y - by, hi.y - by, ly, hy));
            gz = fminf(gz, gap(lo.z - bz, hi.z - bz, lz, hz));
        }
        return gx * gx + gy * gy + gz * gz <= r2c;
    }
    // The region of the lanes' points (those with `in`) for radius r; false
    // when it wraps around the box or crosses both a face and L/2 on an
    // axis.  x, y, z become the points' coordinates in the region's frame.
    __device__ __forceinline__ bool build(bool in, float &x, float &y, float &z, float r, float box_)
    {
        box = box_;
        const float half = 0.5f * box, eps = box * kGqFinest;   // far above rounding
        lx = warp_min(in ? x : INFINITY);
        hx = warp_max(in ? x : -INFINITY);
        ly = warp_min(in ? y : INFINITY);
        hy = warp_max(in ? y : -INFINITY);
        lz = warp_min(in ? z : INFINITY);
        hz = warp_max(in ? z : -INFINITY);
        wx = lx - r < 0.f || hx + r >= box;
        wy = ly - r < 0.f || hy + r >= box;
        wz = lz - r < 0.f || hz + r >= box;
        shifted = wx || wy || wz;
        if (2.f * r >= half) return false;
        if (shifted) {
            if ((wx && lx - r < half && half <= hx + r) || (wy && ly - r < half && half <= hy + r) ||
                (wz && lz - r < half && half <= hz + r))
                return false;
            if (wx && x >= half) x -= box;
            if (wy && y >= half) y -= box;
            if (wz && z >= half) z -= box;
            lx = warp_min(in ? x : INFINITY);
            hx = warp_max(in ? x : -INFINITY);
            ly = warp_min(in ? y : INFINITY);
            hy = warp_max(in ? y : -INFINITY);
            lz = warp_min(in ? z : INFINITY);
            hz = warp_max(in ? z : -INFINITY);
        }
        lx -= eps;
        hx += eps;
        ly -= eps;
        hy += eps;
        lz -= eps;
        hz += eps;
        r2c = reach(r * r);
        return true;
    }
    __device__ __forceinline__ float reach(float d2) const { return d2 * 1.00001f + box * box * 1e-12f; }
    __device__ __forceinline__ void set_reach(float d2) { r2c = fminf(r2c, reach(fmaxf(d2, 0.f))); }
};

// Sum over the eight lanes of a query.
__device__ __forceinline__ int oct_sum(int v)
{
    v += __shfl_xor_sync(kAll, v, 1);
    v += __shfl_xor_sync(kAll, v, 2);
    return v + __shfl_xor_sync(kAll, v, 4);
}

// Bin of a d^2 <= tau: the integer part of d^2 * scale, left in the low bits
// of a float (one instruction, exact product, rounded towards zero); scale
// keeps it below BINS.
template <int BINS> __device__ __forceinline__ float gq_scale(float tau)
{
    return fminf(__fdividef(BINS - 0.01f, tau), 5e37f);
}
__device__ __forceinline__ uint32_t gq_bin_bits(float d2, float scale)   // 0x4b000000 + the bin
{
    return __float_as_uint(__fmaf_rz(d2, scale, 8388608.f));
}
__device__ __forceinline__ int gq_bin(float d2, float scale) { return (int)(gq_bin_bits(d2, scale) - 0x4b000000u); }
// The address of a lane's 16-bit histogram column, less what gq_bin_bits *
// 64 adds to the bin's row.
__device__ __forceinline__ uint32_t gq_column(const uint16_t *hist, int lane)
{
    return (uint32_t)__cvta_generic_to_shared(hist) + 2u * (uint32_t)lane - 0x4b000000u * 64u;
}
// With `on`, adds one to a lane's histogram entry; returns what it held.
__device__ __forceinline__ uint32_t gq_next(uint32_t addr, bool on)
{
    uint32_t v = 0;
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tsetp.ne.b32 p, %2, 0;\n\t@p ld.shared.u16 %0, [%1];\n\t"
                 "add.u32 t, %0, 1;\n\t@p st.shared.u16 [%1], t;\n\t}"
                 : "+r"(v)
                 : "r"(addr), "r"((int)on)
                 : "memory");
    return v;
}
// A value that only later bins exceed.
__device__ __forceinline__ float gq_edge(int bin, float scale) { return __fdividef((float)(bin + 1), scale) * 1.000002f; }

// Counts the lanes' lists (cnt entries) into the histogram and
// finds, for each query, the bin of its k-th and of its n_out-th entry:
// packed as bin << 20 | below << 10 | upto (0 when the lists hold fewer).
// With PLACE the histogram becomes the positions at which each lane's
// entries of a bin go, and bst the bins' starts.  Without it, entries outside
// [lo, hi] are not counted and the bins start at lo.
struct GqFound {
    uint32_t k, o;
};
template <int BINS, bool PLACE>
__device__ __forceinline__ GqFound gq_count(const float2 *list, int cnt, int cmax, uint16_t *hist,
                                            uint16_t *bst, float scale, int k, int n_out, int lane, float lo = 0.f,
                                            float hi = 0.f)
{
    const int q = lane >> 3, p = lane & 7;
#pragma unroll
    for (int i = 0; i < BINS * 64 / 512; ++i) reinterpret_cast<uint4 *>(hist)[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    const uint32_t col = gq_column(hist, lane);
#pragma unroll 1
    for (int i = 0; i < cmax; i += 2) {
        // (a column has an even number of slots)
        const float v0 = list[i * 32].x, v1 = list[(i + 1) * 32].x;
        if constexpr (PLACE) {
            gq_next(col + gq_bin_bits(v0, scale) * 64, i < cnt);
            gq_next(col + gq_bin_bits(v1, scale) * 64, i + 1 < cnt);
        } else {
            gq_next(col + gq_bin_bits(v0 - lo, scale) * 64, i < cnt && v0 >= lo && v0 <= hi);
            gq_next(col + gq_bin_bits(v1 - lo, scale) * 64, i + 1 < cnt && v1 >= lo && v1 <= hi);
        }
    }
    __syncwarp();
    // lane p holds bins p, p + 8 .. of its query, each one read of 16 bytes
    // (the query's eight lanes)
    constexpr int J = BINS / 8;
    uint4 w[J];
    int t[J], st[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        w[j] = *reinterpret_cast<const uint4 *>(hist + (p + 8 * j) * 32 + q * 8);
        const uint32_t s = w[j].x + w[j].y + w[j].z + w[j].w;
        t[j] = (int)((s & 0xffffu) + (s >> 16));
    }
    int all = 0;
#pragma unroll
    for (int j = 0; j < J; j += 2) {
        // two bins' prefixes over the lanes at once, 16 bits each
        uint32_t a = (uint32_t)t[j] | ((uint32_t)t[j + 1] << 16);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, a, o, 8);
            if (p >= o) a += y;
        }
        const uint32_t s = __shfl_sync(kAll, a, 7, 8);
        st[j] = all + (int)(a & 0xffffu) - t[j];
        all += (int)(s & 0xffffu);
        st[j + 1] = all + (int)(a >> 16) - t[j + 1];
        all += (int)(s >> 16);
    }
    if constexpr (PLACE)
        if (p == 7) bst[q * (BINS + 2) + BINS] = (uint16_t)all;
    auto find = [&](int rank) {
        uint32_t v = 0;
#pragma unroll
        for (int j = 0; j < J; ++j)
            if (st[j] < rank && rank <= st[j] + t[j])
                v = ((uint32_t)(p + 8 * j) << 20) | ((uint32_t)st[j] << 10) | (uint32_t)(st[j] + t[j]);
        const uint32_t m = (__ballot_sync(kAll, v != 0u) >> (q * 8)) & 0xffu;
        v = __shfl_sync(kAll, v, q * 8 + (m ? __ffs(m) - 1 : 0));
        return m ? v : 0u;
    };
    GqFound f;
    f.k = find(k);
    f.o = n_out > 0 ? find(n_out) : 0u;
    if constexpr (PLACE) {
#pragma unroll
        for (int j = 0; j < J; ++j) {
            uint32_t r = (uint32_t)st[j];
            auto next = [&](uint32_t x) {
                const uint32_t out = r * 0x10001u + (x << 16);
                r += (x & 0xffffu) + (x >> 16);
                return out;
            };
            uint4 o;
            o.x = next(w[j].x);
            o.y = next(w[j].y);
            o.z = next(w[j].z);
            o.w = next(w[j].w);
            *reinterpret_cast<uint4 *>(hist + (p + 8 * j) * 32 + q * 8) = o;
            bst[q * (BINS + 2) + p + 8 * j] = (uint16_t)st[j];
        }
        __syncwarp();
    }
    return f;
}

// Drops the limit of every query that holds at least k entries (and is in
// `which`) to the upper edge of the bin of its k-th (plus slack), and its
// lists to the entries up to it.  While more than `most` entries remain, the
// k-th's bin is divided again: a query in a void beside a halo has most of
// its entries in the outermost bin, one at a halo's cusp in the innermost.
// Out of line: only lists that are nearly full, or a crowded k-th bin, need it.
struct Tight {
    int cnt;
    float tau;
};
__device__ __noinline__ Tight gq_tighten(uint32_t wo, int cnt, bool which, float tau, float slack, int k, int most,
                                         int lane)
{
    float2 *list = (float2 *)(gq_smem + wo + GqSmem::list) + lane;
    uint16_t *hist = (uint16_t *)(gq_smem + wo + GqSmem::thist);
    const int cmax = (int)__reduce_max_sync(kAll, which ? (unsigned)cnt : 0u);
    float lo = 0.f, hi = tau;
    bool on = which;
    int below = 0;   // entries under lo
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
        const float scale = gq_scale<kGqCutBins>(hi - lo);
        const GqFound f =
            gq_count<kGqCutBins, false>(list, on ? cnt : 0, cmax, hist, nullptr, scale, k - below, 0, lane, lo, hi);
        on = on && f.k;
        if (on) {
            const int b = (int)(f.k >> 20);
            hi = fminf(hi, (lo + gq_edge(b, scale)) * 1.000001f);
            lo += __fdividef((float)b, scale);
            on = below + (int)(f.k & 1023u) > most && hi > lo;
        }
        if (!__any_sync(kAll, on)) break;
        int u = 0;
#pragma unroll 1
        for (int i = 0; on && i < cnt; ++i) u += list[i * 32].x < lo;
        below = oct_sum(u);
        on = on && below < k;
    }
    if (which && hi < tau) {
        tau = fminf(tau, hi + slack);
        int m = 0;
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            const float2 v = list[i * 32];
            if (v.x <= tau) {
                list[m * 32] = v;
                ++m;
            }
        }
        cnt = m;
    }
    __syncwarp();
    return {cnt, tau};
}

// The 512-particle nodes over sorted particles [base, end) that meet the
// region, at offset oa (ob: scratch of the same size); returns their count, or -1 if
// a level has more than kGqN2.  Out of line: once per unit, and for searches
// beyond the unit's radius.
__device__ __noinline__ int gq_descend(const BoxTree &t, const Region rg, uint32_t base, uint32_t end, uint32_t oa,
                                       uint32_t ob, int lane)
{
    uint32_t *A = (uint32_t *)(gq_smem + oa), *B = (uint32_t *)(gq_smem + ob);
    const uint32_t lt = (1u << lane) - 1u;
    int lv = 2;
    while (((end - 1) >> (3 * lv + 3)) - (base >> (3 * lv + 3)) >= (uint32_t)kBoxTop) ++lv;
    uint32_t *cur = (lv & 1) ? B : A, *nxt = (lv & 1) ? A : B;
    const uint32_t first = base >> (3 * lv + 3), cnt = ((end - 1) >> (3 * lv + 3)) - first + 1;
    int n;
    {
        const uint32_t node = first + (uint32_t)lane;
        bool in = (uint32_t)lane < cnt;
        if (in) in = rg.meets(t.lo[t.off[lv] + node], t.hi[t.off[lv] + node]);
        const uint32_t bal = __ballot_sync(kAll, in);
        if (in) cur[__popc(bal & lt)] = node;
        n = __popc(bal);
    }
    for (--lv; lv >= 2; --lv) {
        __syncwarp();
        int m = 0;
        for (int i = 0; i < n; i += 4) {
            const int j = i + (lane >> 3);
            bool in = j < n;
            uint32_t node = 0;
            if (in) {
                node = cur[j] * 8 + (lane & 7);
                in = rg.meets(t.lo[t.off[lv] + node], t.hi[t.off[lv] + node]);
            }
            const uint32_t bal = __ballot_sync(kAll, in);
            const int pos = m + __popc(bal & lt);
            if (in && pos < kGqN2) nxt[pos] = node;
            m += __popc(bal);
        }
        if (m > kGqN2) return -1;
        n = m;
        uint32_t *x = cur;
        cur = nxt;
        nxt = x;
    }
    __syncwarp();
    return n;
}

// Appends the children of up to 16 nodes of level lv + 1 (list[i ..  n)) that
// meet the region to out (m entries so far; room for 128 more); the four
// steps' loads are independent.
__device__ __forceinline__ int gq_open(const BoxTree &t, int lv, const Region &rg, const uint32_t *list, int i, int n,
                                       uint32_t *out, int m, int lane, uint32_t lt)
{
    const float4 *lo = t.lo + t.off[lv], *hi = t.hi + t.off[lv];
    uint32_t node[4];
    float4 l[4], h[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = i + 4 * u + (lane >> 3);
        node[u] = list[min(j, n - 1)] * 8 + (lane & 7);
        l[u] = lo[node[u]];
        h[u] = hi[node[u]];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (i + 4 * u >= n) break;
        const bool in = i + 4 * u + (lane >> 3) < n && rg.meets(l[u], h[u]);
        const uint32_t bal = __ballot_sync(kAll, in);
        if (in) out[m + __popc(bal & lt)] = node[u];
        m += __popc(bal);
    }
    return m;
}

// The first radius at particle s where the given one wraps: the mean-density
// distance, or where that is larger the distance to the farthest corner of
// the boxes that hold the particle's own 64 (more than 64 wanted: 128)
// neighbours in sort order, which is enough for k of them.
__device__ __noinline__ float gq_box_radius(const BoxTree &t, float4 v, uint32_t s, uint32_t base, uint32_t end, int k,
                                              float plain_r)
{
    const int nodes = k <= 64 ? 1 : 2;
    const uint32_t node = (s >> 6) & ~(uint32_t)(nodes - 1);
    if (node * 64 < base || (uint64_t)(node + nodes) * 64 > end) return plain_r;
    float dx = 0.f, dy = 0.f, dz = 0.f;
    for (int i = 0; i < nodes; ++i) {
        const float4 lo = t.lo[t.off[1] + node + i], hi = t.hi[t.off[1] + node + i];
        dx = fmaxf(dx, fmaxf(v.x - lo.x, hi.x - v.x));
        dy = fmaxf(dy, fmaxf(v.y - lo.y, hi.y - v.y));
        dz = fmaxf(dz, fmaxf(v.z - lo.z, hi.z - v.z));
    }
    return fminf(plain_r, sqrtf(dx * dx + dy * dy + dz * dz) * 1.0001f);
}

// Whether a full 512-particle node of double-precision particles is too tight
// for the float search.  That search is certain of an order only while the
// rounding's slack stays below a bin, which is so for limits above 2^-14.1 of
// the box; a node with a diagonal below 2^-17 lies within one bin of any such
// limit, with more particles than a query's list holds.
__device__ __noinline__ bool gq_tight_node(const BoxTree &t, uint32_t node, uint32_t end, float box)
{
    if (((uint64_t)node + 1) * 512 > end) return false;
    const float4 lo = t.lo[t.off[2] + node], hi = t.hi[t.off[2] + node];
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dx + dy * dy + dz * dz < box * box * 0x1p-34f;
}

// The factor by which a radius grows that held tot < k particles.
__device__ __noinline__ float gq_grow(int k, int tot)
{
    return fmaxf(1.25f, 1.1f * cbrtf((float)k / (float)max(tot, 1)));
}

// Exact squared minimum-image distance of two double-precision particles, as
// the single-scan kernel rounds it.
__device__ __forceinline__ double gq_d2_f64(const double4 &c, double x, double y, double z, double box)
{
    const double half = 0.5 * box;
    const double dx = wrapdiff(c.x, x, box, half), dy = wrapdiff(c.y, y, box, half), dz = wrapdiff(c.z, z, box, half);
    return fma(dx, dx, fma(dy, dy, dz * dz));
}

// F64: the search runs on positions rounded to float; a squared distance
// found that way is within `err` of the exact one (the bound is the two
// coordinates' rounding, the frame shift's, and the float arithmetic).  The
// entries up to the bin after the Ndens-th's therefore hold the exact Ndens
// nearest as long as a bin is wider than 2 err; their distances are computed
// again in double, and an entry's place is ranked over its own and the two
// neighbouring bins.
template <bool SEG, bool F64>
__global__ void __launch_bounds__(kGqWarps * 32, F64 ? 3 : 4) knn_gq_kernel(const GqDev a)
{
    using L = GqSmem;
    int lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));   // (kept in a register)
    const int q = lane >> 3, p = lane & 7;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t wo = (uint32_t)L::total(a.capq, F64) * (threadIdx.x >> 5);   // the warp's shared memory
    unsigned char *wb = gq_smem + wo;
    float2 *list = (float2 *)(wb + L::list) + lane;
    const uint32_t list0 = gq_addr(wo + L::list) + lane * 8;
    const uint32_t full = list0 + (kGqSlots - 2) * 256;   // a list beyond it has no room for two more
    float4 *tile = (float4 *)(wb + L::tile);
    uint16_t *hist = (uint16_t *)(wb + L::hist);
    uint16_t *bst = (uint16_t *)(wb + L::bst);
    uint32_t *U2 = (uint32_t *)(wb + L::u2), *T0 = (uint32_t *)(wb + L::t0), *T1 = (uint32_t *)(wb + L::t1),
             *T2 = (uint32_t *)(wb + L::t2);
    using D2 = std::conditional_t<F64, double, float>;
    D2 *Dd = (D2 *)(wb + L::t0) + q * L::stride(a.capq);                     // the query's entries, bin by bin
    uint32_t *Ds = (uint32_t *)(wb + L::t0) + (kGqQ * (int)sizeof(D2) / 4 + q) * L::stride(a.capq);
    const int k = a.k, n_out = a.nbr_s ? a.n_out : 0;
    unsigned long long cand_acc = 0;
    uint32_t search_acc = 0, retry_acc = 0, warp_acc = 0;

    for (;;) {
        unsigned long long task = 0;
        if (lane == 0) task = atomicAdd(a.task_counter, 1ull);
        task = __shfl_sync(kAll, task, 0);
        if ((int64_t)task >= a.n_tasks) break;
        const int per_task = kGqUnit / a.split;
        uint32_t base, end, s_unit, ch0;
        float box, norm, plain_r;
        if constexpr (SEG) {
            const SegDesc &sd = a.seg[seg_of_unit(a.seg, a.B, (int64_t)task / a.split)];
            base = (uint32_t)sd.base;
            end = (uint32_t)(sd.base + sd.n);
            s_unit = base + (uint32_t)((int64_t)task - sd.unit0 * a.split) * per_task;
            ch0 = (uint32_t)sd.chunk0;
            box = (float)sd.box;
            norm = (float)sd.norm;
            plain_r = sd.plain_r;
        } else {
            base = 0;
            end = a.n;
            s_unit = (uint32_t)task * per_task;
            ch0 = 0;
            box = a.box;
            norm = a.norm;
            plain_r = a.plain_r;
        }
        const int nu = (int)min((int64_t)per_task, (int64_t)end - (int64_t)s_unit);
        if (nu <= 0) continue;   // the last unit of a subvolume may hold fewer parts
        if constexpr (F64) {
            // (63,000 particles, 60,000 of them within 1e-6 of the box: 172 ms
            // where every query was searched and handed over by itself, 120 ms
            // so, 123 ms through the single-scan kernel alone)
            if (__any_sync(kAll, gq_tight_node(a.tree, s_unit >> 9, end, box))) {
                if (lane < nu && lane % 4 == 0) a.runs[atomicAdd(a.runs_n, 1ull)] = s_unit + (uint32_t)lane;
                warp_acc += (nu + 3) / 4;
                continue;
            }
        }
        // lane i (and i + 16) holds query i of the unit; r4: its group's radius
        float ux, uy, uz, r4, ru;
        {
            const uint32_t su = s_unit + min(lane & (kGqUnit - 1), nu - 1);
            const float4 v = a.spos[su];
            ux = v.x;
            uy = v.y;
            uz = v.z;
            // (a first radius whose ball wraps around the box, as of a chunk
            // across a jump of the Morton curve, gives way to the boxes')
            float r = a.chunk_r ? a.chunk_r[ch0 + (su - base) / (uint32_t)a.qpw] : plain_r;
            if constexpr (F64)
                if (a.chunk_r) r *= a.unit;
            if (2.f * r >= 0.5f * box) r = gq_box_radius(a.tree, v, su, base, end, k, plain_r);
            if (!(r > 0.f)) r = box * 1e-6f;
            // (a ball that wraps is handed over)
            if constexpr (!F64)
                if (!(box >= kGqBoxMin && box <= kGqBoxMax)) r = INFINITY;
            r = fmaxf(r, __shfl_xor_sync(kAll, r, 1));
            r4 = fmaxf(r, __shfl_xor_sync(kAll, r, 2));
            ru = warp_max(r4);
        }
        int n2u = -1;
        {
            Region rg;
            float x = ux, y = uy, z = uz;
            if (rg.build(true, x, y, z, ru, box)) n2u = gq_descend(a.tree, rg, base, end, wo + L::u2, wo + L::t2, lane);
        }
        for (int g = 0; g < nu; g += kGqQ) {
            const int nq = min(kGqQ, nu - g);
            ++warp_acc;
            const uint32_t sq = s_unit + g + min(q, nq - 1);
            const float R0 = __shfl_sync(kAll, r4, g);
            const float qx = __shfl_sync(kAll, ux, g + min(q, nq - 1)), qy = __shfl_sync(kAll, uy, g + min(q, nq - 1)),
                        qz = __shfl_sync(kAll, uz, g + min(q, nq - 1));
            // a query farther than R0 from the one before it starts a new search
            const float ex = qx - __shfl_up_sync(kAll, qx, 8), ey = qy - __shfl_up_sync(kAll, qy, 8),
                        ez = qz - __shfl_up_sync(kAll, qz, 8);
            const uint32_t cuts = __ballot_sync(kAll, p == 0 && q > 0 && q < nq && ex * ex + ey * ey + ez * ez > R0 * R0);
            uint32_t todo = (1u << (8 * nq - 1)) * 2u - 1u;   // the lanes of the queries still to be served
            // the query's radius; the largest that held too few
            float rq = R0, rfew = 0.f;
            bool alone = false;   // the first query left is searched by itself until it is done
            int tries = 0;
            while (todo) {
                // from the first one up to the next cut, or the first alone
                const int g0 = __ffs(todo) - 1;
                const uint32_t later = cuts & ~((2u << g0) - 1u);
                uint32_t set = todo & (later ? (later & (0u - later)) - 1u : kAll);
                if (alone) set = 0xffu << g0;
                const bool member = (set >> lane) & 1u;
                const float R = warp_max(member ? rq : 0.f);
                // ------------- the 512-particle nodes that meet the region
                Region rg;
                float fx = qx, fy = qy, fz = qz;
                int n2 = -1;
                const bool built = rg.build(member, fx, fy, fz, R, box) && tries < kGqTries;
                if (built) {
                    if (n2u >= 0 && R <= ru) {
                        n2 = 0;
                        for (int i = 0; i < n2u; i += 32) {
                            bool in = i + lane < n2u;
                            uint32_t node = 0;
                            if (in) {
                                node = U2[i + lane];
                                in = rg.meets(a.tree.lo[a.tree.off[2] + node], a.tree.hi[a.tree.off[2] + node]);
                            }
                            const uint32_t bal = __ballot_sync(kAll, in);
                            if (in) T2[n2 + __popc(bal & lt)] = node;
                            n2 += __popc(bal);
                        }
                        __syncwarp();
                    } else {
                        n2 = gq_descend(a.tree, rg, base, end, wo + L::t2, wo + L::t1, lane);
                    }
                }
                if (n2 < 0) {
                    // too many nodes: a smaller radius as long as that may
                    // hold enough: of the whole group with the plain radius
                    // (2.1M particles: 7.4 ms, 9.6 one by one), otherwise of
                    // one query at a time (64 subvolumes, learned radius:
                    // 43.6 ms, 48.2 together).  The radius is remembered only
                    // through the one that held too few, which grows with
                    // every search: a limit kept from a region that met too
                    // many nodes binds queries it was not measured on, and
                    // they crept up to it until the tries ran out (200
                    // particles in a void around a ball of 100,000, plain
                    // radius: 25.2 ms and 3,059 searches that held too few,
                    // now 3.6 ms and 257)
                    const float few = warp_max(member ? rfew : 0.f);
                    if (built && R > fmaxf(1.05f * few, (F64 ? kGqFinest64 : kGqFinest) * box) &&
                        (!a.chunk_r || alone || set == (0xffu << g0))) {
                        ++tries;
                        if (member) rq = few > 0.f ? sqrtf(R * few) : 0.5f * R;
                        continue;
                    }
                    // several queries' region that crosses both a face and
                    // L/2, or meets too many nodes: the first one alone
                    alone = !alone && set != (0xffu << g0);
                    if (!alone) {
                        if (member && p == 0) a.hand[atomicAdd(a.hand_n, 1ull)] = sq;
                        todo &= ~set;
                        tries = 0;
                    }
                    continue;
                }
                ++search_acc;
                if (n2 > 8) {
                    // a large region: the query's own node first, so that the
                    // limits drop before the others are opened
                    const uint32_t own = __shfl_sync(kAll, sq, g0) >> 9;
                    for (int i = lane; i < n2; i += 32)
                        if (i > 0 && T2[i] == own) {
                            T2[i] = T2[0];
                            T2[0] = own;
                        }
                    __syncwarp();
                }
                // ------------- open them and evaluate the runs
                uint32_t lp = list0;   // the end of the lane's list
                float tau = member ? R * R : -1.f;
                bool crowd = false;
                float slack = 0.f;   // F64: 2 err
                if constexpr (F64) {
                    const float d = box * 2.38418579e-7f;   // 2^-22 of the box per component
                    slack = 2.f * (3.47f * R * d + 3.f * d * d + R * R * 4.76837158e-7f);
                }
                int i2 = 0, i1 = 0, n1 = 0, cand = 0;
                for (;;) {
                    int n0 = 0;
                    // 16 nodes at a time: 512-particle ones while the list
                    // below has room, then 64-particle ones
                    bool fill = n1 == 0;
                    while (n0 <= kGqN0 - 128) {
                        if (fill && (i2 >= n2 || n1 > kGqN1 - 128)) {
                            fill = false;
                            __syncwarp();
                        }
                        if (!fill && i1 >= n1) {
                            if (i2 >= n2) break;
                            fill = true;
                            i1 = n1 = 0;
                            __syncwarp();
                        }
                        const int m = gq_open(a.tree, fill ? 1 : 0, rg, fill ? T2 : T1, fill ? i2 : i1, fill ? n2 : n1,
                                              fill ? T1 : T0, fill ? n1 : n0, lane, lt);
                        if (fill) {
                            n1 = m;
                            i2 += 16;
                        } else {
                            n0 = m;
                            i1 += 16;
                        }
                    }
                    if (n0 == 0) break;
                    // up to a multiple of 16 with runs past the last particle
                    if (lane < 16) T0[n0 + lane] = a.pad_run;
                    __syncwarp();
                    const float4 *sp = a.spos + p;
                    float4 v[4];
                    uint32_t run[4];
                    auto load = [&](int j) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            run[u] = T0[j + 4 * u + q] * 8;
                            v[u] = sp[run[u]];
                        }
                    };
                    cand += n0 * 8;   // every particle read, by the box's distance or its own
                    load(0);
                    int m = 0;
#pragma unroll 1
                    for (int j = 0; j < n0; j += 16) {
                        if (rg.shifted) {
                            const float half = 0.5f * box, bx = rg.wx ? box : 0.f, by = rg.wy ? box : 0.f,
                                        bz = rg.wz ? box : 0.f;
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (v[u].x >= half) v[u].x -= bx;
                                if (v[u].y >= half) v[u].y -= by;
                                if (v[u].z >= half) v[u].z -= bz;
                            }
                        }
                        // a lane's particles in reach of the box go to the tile
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            float4 c = v[u];
                            const float gx = Region::gap(c.x, c.x, rg.lx, rg.hx), gy = Region::gap(c.y, c.y, rg.ly, rg.hy),
                                        gz = Region::gap(c.z, c.z, rg.lz, rg.hz);
                            bool in = gx * gx + gy * gy + gz * gz <= rg.r2c;
                            // a run at the end of a subvolume also holds particles of the next
                            if constexpr (SEG) in = in && run[u] + p - base < end - base;
                            const uint32_t bal = __ballot_sync(kAll, in);
                            c.w = __uint_as_float(run[u] + p);
                            if (in) tile[m + __popc(bal & lt)] = c;
                            m += __popc(bal);
                        }
                        const bool last = j + 16 >= n0;
                        if (!last) load(j + 16);
                        if (last) {
                            // up to a multiple of 16 with entries no test accepts
                            const float nan = __int_as_float(0x7fc00000);
                            if (lane < ((16 - (m & 15)) & 15)) tile[m + lane] = make_float4(nan, nan, nan, 0.f);
                            m = (m + 15) & ~15;
                        }
                        __syncwarp();
                        int r = 0;
                        while (r + 16 <= m) {
                            bool over = false;
#pragma unroll 1
                            for (; r + 16 <= m && !over; r += 16) {
                                const float4 c = tile[r + p], d = tile[r + 8 + p];
                                const float cx = c.x - fx, cy = c.y - fy, cz = c.z - fz;
                                const float dx = d.x - fx, dy = d.y - fy, dz = d.z - fz;
                                gq_keep(lp, fmaf(cx, cx, fmaf(cy, cy, cz * cz)), tau, __float_as_uint(c.w));
                                gq_keep(lp, fmaf(dx, dx, fmaf(dy, dy, dz * dz)), tau, __float_as_uint(d.w));
                                over = __any_sync(kAll, lp > full);
                            }
                            if (over) {
                                __syncwarp();
                                const Tight t = gq_tighten(wo, (int)(lp - list0) >> 8, member && !crowd, tau, slack, k,
                                                           a.capq, lane);
                                lp = list0 + t.cnt * 256;
                                tau = t.tau;
                                // a list that stays full: a crowd at the limit
                                if ((__ballot_sync(kAll, lp > full) >> (q * 8)) & 0xffu) {
                                    crowd = true;
                                    lp = list0;
                                    tau = -1.f;
                                }
                                // no more than the largest limit needs be read
                                rg.set_reach(warp_max(tau));
                            }
                        }
                        // what is left (fewer than 16) moves to the front
                        m -= r;
                        float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (lane < m) c = tile[r + lane];
                        __syncwarp();
                        if (lane < m) tile[lane] = c;
                    }
                    __syncwarp();
                }
                cand_acc += (unsigned long long)cand * (unsigned long long)(__popc(__ballot_sync(kAll, member)) >> 3);
                int cnt = (int)(lp - list0) >> 8;
                // ------------- selection
                const int tot = oct_sum(cnt);
                bool ok = member && !crowd && tot >= k;
                if (__any_sync(kAll, ok)) {
                    int cmax = 0;
                    float scale = 0.f;
                    GqFound f;
                    int upto = 0, upto_o = 0;
                    const uint16_t *t = bst + q * (kGqBins + 2);
                    for (int it = 0;; ++it) {
                        cmax = (int)__reduce_max_sync(kAll, ok ? (unsigned)cnt : 0u);
                        scale = gq_scale<kGqBins>(tau);
                        f = gq_count<kGqBins, true>(list, ok ? cnt : 0, cmax, hist, bst, scale, k, n_out, lane);
                        upto = (int)(f.k & 1023u);
                        upto_o = (int)(f.o & 1023u);
                        if constexpr (F64) {
                            upto = t[min((int)(f.k >> 20) + 2, kGqBins)];
                            upto_o = t[min((int)(f.o >> 20) + 2, kGqBins)];
                            if (ok && slack > 0.9f * tau * (1.f / kGqBins)) {
                                // bins too narrow for float distances
                                ok = false;
                                crowd = true;
                            } else if (ok && (int)(f.k >> 20) == kGqBins - 1 && tau >= R * R) {
                                ok = false;   // not certain that R reaches the exact Ndens-th: a larger one
                            }
                        }
                        const bool over = ok && upto > a.capq;
                        if (!__any_sync(kAll, over)) break;
                        if (it == 3) {
                            // the bin stays crowded
                            if (over) {
                                ok = false;
                                crowd = true;
                            }
                            break;
                        }
                        const Tight c = gq_tighten(wo, cnt, over, tau, slack, k, a.capq, lane);
                        cnt = c.cnt;
                        tau = c.tau;
                    }
                    const int bk = (int)(f.k >> 20);
                    const int below = F64 ? t[max(bk - 1, 0)] : (int)((f.k >> 10) & 1023u);
                    if (!ok) upto = upto_o = 0;
                    const uint32_t col = gq_column(hist, lane), last_bin = 0x4b000000u + (uint32_t)bk + (F64 ? 1u : 0u);
                    double q64x = 0.0, q64y = 0.0, q64z = 0.0;
                    if constexpr (F64) {
                        const double4 v = a.spos64[sq];
                        q64x = v.x;
                        q64y = v.y;
                        q64z = v.z;
                    }
                    const int cnt_ok = ok ? cnt : 0;
#pragma unroll 2
                    for (int i = 0; i < cmax; ++i) {
                        const float2 v = list[i * 32];
                        const uint32_t b = gq_bin_bits(v.x, scale);
                        const bool on = i < cnt_ok && b <= last_bin;
                        const uint32_t pos = gq_next(col + b * 64, on);
                        if (on) {
                            if constexpr (F64)
                                Dd[pos] = gq_d2_f64(a.spos64[__float_as_uint(v.y)], q64x, q64y, q64z, a.box64);
                            else
                                Dd[pos] = v.x;
                            Ds[pos] = __float_as_uint(v.y);
                        }
                    }
                    __syncwarp();
                    // the exact k-th d^2: the largest of its bin with fewer
                    // than k smaller entries
                    D2 vk = D2(-1);
#pragma unroll 1
                    for (int e = below + p; e < upto; e += 8) {
                        const D2 v = Dd[e];
                        int l = below;
#pragma unroll 2
                        for (int h = below; h < upto; ++h) l += Dd[h] < v;
                        if (l < k) vk = max(vk, v);
                    }
                    __syncwarp();
                    vk = max(vk, __shfl_xor_sync(kAll, vk, 1));
                    vk = max(vk, __shfl_xor_sync(kAll, vk, 2));
                    vk = max(vk, __shfl_xor_sync(kAll, vk, 4));
                    // density: fixed-point (2^-32) sum of w(2 r / r_k) over
                    // entries with d^2 < r_k^2; a weight of 1 is one more
                    // than the conversion's largest value
                    const D2 rk = sqrt(vk);
                    const D2 inv_h = vk > D2(0) ? D2(2) / rk : D2(0);
                    unsigned long long wsum = 0;
#pragma unroll 1
                    for (int e = p; e < upto; e += 8) {
                        const D2 v = Dd[e];
                        if constexpr (F64) {
                            if (v < vk) wsum += (unsigned long long)(m4<double>(sqrt(v) * inv_h) * 4294967296.0 + 0.5);
                            continue;
                        }
                        // m4(), both of its pieces computed
                        const float x = sqrtf((float)v) * (float)inv_h, y = 2.f - x;
                        const float wi = 1.f - 1.5f * x * x + 0.75f * x * x * x, wo_ = 0.25f * y * y * y;
                        const float w = (x < 1.f ? wi : wo_) * 4294967296.0f + 0.5f;
                        if (v < vk) wsum += (unsigned long long)__float2uint_rz(w) + (w >= 4294967296.0f ? 1u : 0u);
                    }
                    __syncwarp();
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) wsum += __shfl_xor_sync(kAll, wsum, o);
                    if (ok && p == 0) {
                        float dens;
                        if (vk > D2(0)) {
                            const D2 h = rk * D2(0.5);
                            if constexpr (F64)
                                dens = (float)(a.norm64 * ((double)wsum * 2.3283064365386963e-10) / (h * h * h));
                            else
                                dens = (float)(norm * ((float)wsum * 2.3283064365386963e-10f) / (h * h * h));
                        } else {
                            dens = INFINITY;
                        }
                        a.dens_s[sq] = dens;
                        if (a.rk_s) a.rk_s[sq] = (float)rk;
                    }
                    // the n_out nearest by (d^2, original index): the start of
                    // the entry's bin and its rank in it
                    if (n_out > 0) {
                        uint32_t *row = a.nbr_s + (size_t)sq * a.ld_out;
                        // the entries that may come before or after entry e
                        auto around = [&](int e, D2 v, int &h0, int &h1) {
                            if constexpr (F64) {
                                // its bin from its place, then one bin either way
                                int b = 0;
                                while (b < kGqBins - 1 && t[b + 1] <= e) ++b;
                                h0 = t[max(b - 1, 0)];
                                h1 = min((int)t[min(b + 2, kGqBins)], upto_o);
                            } else {
                                const int b = gq_bin(v, scale);
                                h0 = t[b];
                                h1 = t[b + 1];
                            }
                        };
                        int sum = 0;
#pragma unroll 1
                        for (int e = p; e < upto_o; e += 8) {
                            const D2 v = Dd[e];
                            int h0, h1;
                            around(e, v, h0, h1);
                            int rank = h0;
#pragma unroll 2
                            for (int h = h0; h < h1; ++h) rank += Dd[h] < v;
                            if (rank < n_out) row[rank] = Ds[e];
                            sum += rank;
                        }
                        __syncwarp();
                        // the ranks are 0 .. upto_o - 1 unless two distances
                        // are equal; only then rank again, equal ones by index
                        const bool ties = oct_sum(sum) != upto_o * (upto_o - 1) / 2;
                        if (__any_sync(kAll, ties)) {
#pragma unroll 1
                            for (int e = p; ties && e < upto_o; e += 8) {
                                const D2 v = Dd[e];
                                const uint32_t se = Ds[e], oe = __float_as_uint(a.spos[se].w);
                                int h0, h1;
                                around(e, v, h0, h1);
                                int rank = h0;
#pragma unroll 1
                                for (int h = h0; h < h1; ++h) {
                                    const D2 u = Dd[h];
                                    rank += u < v;
                                    if (u == v) rank += __float_as_uint(a.spos[Ds[h]].w) < oe;
                                }
                                if (rank < n_out) row[rank] = se;
                            }
                        }
                    }
                    __syncwarp();
                }
                if (member && crowd && p == 0) a.hand[atomicAdd(a.hand_n, 1ull)] = (uint32_t)sq;
                todo &= ~__ballot_sync(kAll, ok || (member && crowd));
                if (!(todo & set)) {
                    alone = false;
                    tries = 0;
                }
                // the others of the set hold too few within R: a larger one, at
                // first not beyond the largest this kernel takes
                if (todo & set) {
                    ++retry_acc;
                    ++tries;
                    if (member && !ok && !crowd) {
                        const float most = 0.2499f * box;
                        rq = R * fminf(gq_grow(k, tot), 8.f);
                        if (R < 0.99f * most) rq = fminf(rq, most);
                        rfew = R;
                    }
                }
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

// Rounded copies of double-precision particles, the padding included, times
// `unit`, a power of two (exact): a box side of any size becomes one in
// [1, 2), so that neither the search's squares nor its error bounds leave
// float32's range.
__global__ void to_float4_kernel(const double4 *__restrict__ in, int64_t n, double unit, float4 *__restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double4 v = in[i];
        out[i] = make_float4((float)(v.x * unit), (float)(v.y * unit), (float)(v.z * unit),
                             __uint_as_float((uint32_t)__double_as_longlong(v.w)));
    }
}

template <bool SEG, bool F64> int knn_gq_run(hop_ctx *c, const KnnArgs &ka, int qpw, int cpr)
{
    GqDev d;
    d.spos64 = nullptr;
    d.spos = (const float4 *)ka.spos;
    d.box = (float)ka.box;
    d.plain_r = ka.plain_r;
    d.unit = 1.f;
    if constexpr (F64) {
        const double unit = std::scalbn(1.0, -std::ilogb(ka.box)), side = ka.box * unit;
        d.box = (float)side;
        d.plain_r = plain_radius_for(ka.n, side, ka.k);
        d.unit = (float)unit;   // (0 or inf where the caller's radii are inf or 0: the boxes' radius then)
        const int64_t m = ka.n + kSposPad;
        float4 *f = (float4 *)ctx_buf(c, S_SPOS_F, (size_t)m * sizeof(float4));
        if (!f) return HOP_ENOMEM;
        to_float4_kernel<<<grid_for(c, m), 256, 0, c->stream>>>((const double4 *)ka.spos, m, unit, f);
        HOP_LAUNCH(c);
        d.spos = f;
        d.spos64 = (const double4 *)ka.spos;
    }
    const int rc = box_tree_build(c, d.spos, ka.n, &d.tree);
    if (rc) return rc;
    d.n = (uint32_t)ka.n;
    d.pad_run = (uint32_t)((ka.n + 7) / 8);
    // a warp takes a whole unit, except where that leaves warps idle or a long
    // last wave: then a half or a quarter of one.  kNN of NFW boxes in us,
    // learned radius, whole / half / quarter: 4,913 particles 164 / 104 / 82;
    // 32,768 238 / 176 / 154; 65,537 301 / 260 / 250; 131,071 391 / 373 / 354;
    // 262,147 637 / 586 / 604; 524,287 1110 / 1137 / 1196; 2.1M 4048 / 4269 /
    // 4677 (each part walks the unit's boxes again).  The lines, at 39,000 and
    // 78,000 particles, lie lower than these times would put them.
    const int64_t units = SEG ? ka.n_units : (ka.n + kGqUnit - 1) / kGqUnit;
    const int64_t warps = (int64_t)c->num_sms * 16;
    d.split = units >= 2 * warps ? 1 : units >= warps ? 2 : 4;
    d.n_tasks = units * d.split;
    d.qpw = qpw;
    d.norm = (float)(ka.box * ka.box * ka.box / ((double)(ka.n_norm > 0 ? ka.n_norm : ka.n) * 3.14159265358979323846));
    d.box64 = ka.box;
    d.norm64 = ka.box * ka.box * ka.box / ((double)(ka.n_norm > 0 ? ka.n_norm : ka.n) * 3.14159265358979323846);
    d.k = ka.k;
    d.n_out = ka.n_out;
    d.ld_out = ka.ld_out;
    d.capq = ((ka.k + 32 + 7) / 8) * 8;
    d.chunk_r = ka.chunk_r;
    d.seg = ka.seg;
    d.B = ka.B;
    d.nbr_s = ka.nbr_s;
    d.dens_s = ka.dens_s;
    d.rk_s = ka.rk_s;
    d.counters = c->d_counters;
    // (the words after the counters are zero: a pass clears them at its start)
    d.task_counter = c->d_counters + kCntNum;
    d.hand_n = c->d_counters + kCntNum + 1;
    d.runs_n = d.hand_n + 2;
    d.hand = (uint32_t *)ctx_buf(c, S_KNN_HAND, (size_t)(ka.n + (F64 ? ka.n / 4 + 4 : 0)) * sizeof(uint32_t));
    if (!d.hand) return HOP_ENOMEM;
    d.runs = d.hand + ka.n;
    const size_t smem = (size_t)GqSmem::total(d.capq, F64) * kGqWarps;
    auto kern = knn_gq_kernel<SEG, F64>;
    HOP_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    HOP_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGqWarps * 32, smem));
    if (per_sm < 1) return ctx_fail(c, HOP_EINVAL, "kNN lists do not fit in shared memory");
    const int64_t need = (d.n_tasks + kGqWarps - 1) / kGqWarps;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * c->num_sms, need));
    kern<<<(unsigned)blocks, kGqWarps * 32, smem, c->stream>>>(d);
    HOP_LAUNCH(c);
    if constexpr (F64) {
        const int rr = knn_runs_f64_launch(c, ka, qpw, cpr, d.runs, d.runs_n, d.runs_n + 1);
        return rr ? rr : knn_hand_f64_launch(c, ka, qpw, cpr, d.hand, d.hand_n, d.hand_n + 1);
    }
    return knn_wq_launch(c, ka, qpw, cpr, d.hand, d.hand_n, d.hand_n + 1);
}

}  // namespace

int knn_gq_launch(hop_ctx *c, const KnnArgs &a, bool f64, int qpw, int cpr)
{
    if (qpw < 1) return ctx_fail(c, HOP_EINVAL, "radius chunks hold at least one query");
    if (f64) return knn_gq_run<false, true>(c, a, qpw, cpr);
    return a.seg ? knn_gq_run<true, false>(c, a, qpw, cpr) : knn_gq_run<false, false>(c, a, qpw, cpr);
}
