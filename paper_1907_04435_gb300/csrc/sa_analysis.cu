// sa_analysis.cu -- analysis measures over a polygonal region of a ground grid (Sec. 7.2).
//
// Shadow area: the sum over the region's cells of shadow(p) x area(p), where shadow(p) is
// the fraction of the interval's steps the cell spends in shadow (gross counts give the
// gross fraction, continuous counts the continuous one) and area(p) = dx^2.  A cell is in
// the region when its centre is, by the even-odd rule.  The shadow score over several
// intervals is the weighted sum of their areas (weights w_t in [-1, 1]):
// sum over the region's cells of sum_t w_t x shadow_t(p) x area(p), one pass over the
// cells that reads every interval's counts of a cell together.
//
// The centres are rounded exactly as the receivers' (FP32), then tested in FP64 with
// explicit roundings, so the decision for a centre does not depend on the compiler's
// contraction of multiply-adds.
#include <math.h>
#include <stdio.h>

#include <string.h>

#include <algorithm>
#include <vector>

#include "sa_handles.cuh"
#include "sa_light.cuh"

namespace sa {

namespace {

constexpr int kAreaThreads = 256;

// even-odd rule: count the polygon edges crossed by the ray from (x, y) toward +x
__device__ bool inside_polygon(const double2* __restrict__ poly, int n, double x, double y) {
    bool in = false;
    for (int i = 0; i < n; ++i) {
        const double2 a = poly[i], b = poly[i + 1 == n ? 0 : i + 1];
        if ((a.y > y) != (b.y > y)) {
            const double t = __ddiv_rn(__dsub_rn(y, a.y), __dsub_rn(b.y, a.y));
            const double xc = __dadd_rn(a.x, __dmul_rn(t, __dsub_rn(b.x, a.x)));
            if (x < xc) in = !in;
        }
    }
    return in;
}

__global__ void k_shadow_area(const int* __restrict__ steps, float x0, float y0, float dx, int nx,
                              long long R, const double2* __restrict__ poly, int n,
                              double inv_total, double* __restrict__ out) {
    __shared__ double s_part[kAreaThreads / 32];
    double s = 0.0;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < R;
         c += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(c % nx), iy = (int)(c / nx);
        const float cx = __fadd_rn(x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), dx));
        const float cy = __fadd_rn(y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), dx));
        if (steps[c] != 0 && inside_polygon(poly, n, (double)cx, (double)cy))
            s += (double)steps[c] * inv_total;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kAreaThreads / 32; ++w) t += s_part[w];
        atomicAdd(out, t);
    }
}

// Shadow score over intervals: coef[t] = w_t / total_steps_t; counts are [n_t][R].
__global__ void k_shadow_score(const int* __restrict__ steps, long long R, int n_t,
                               const double* __restrict__ coef, float x0, float y0, float dx,
                               int nx, const double2* __restrict__ poly, int n,
                               double* __restrict__ out) {
    __shared__ double s_part[kAreaThreads / 32];
    double s = 0.0;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < R;
         c += (long long)gridDim.x * blockDim.x) {
        double v = 0.0;
        bool any = false;
        for (int t = 0; t < n_t; ++t) {
            const int k = __ldcs(&steps[(long long)t * R + c]);
            if (k != 0) {
                v = fma((double)k, coef[t], v);
                any = true;
            }
        }
        if (!any) continue;
        const int ix = (int)(c % nx), iy = (int)(c / nx);
        const float cx = __fadd_rn(x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), dx));
        const float cy = __fadd_rn(y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), dx));
        if (inside_polygon(poly, n, (double)cx, (double)cy)) s += v;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kAreaThreads / 32; ++w) t += s_part[w];
        atomicAdd(out, t);
    }
}

// Building contribution (Sec. 7.2).  For every cell of the region and every step the
// accrual raster marks as shadowed, the buildings the ray toward the sun meets beyond
// t_min are found, and each is credited one cell-step: "casting" counts, per building,
// the cell-steps whose ray meets it (a ray meeting several buildings credits each once);
// "nearest" counts, per building, the cell-steps whose nearest hit lies on it, so that
// these partition the region's shadowed cell-steps -- except the ones the raster marks
// shadowed whose FP32 ray grazes past every triangle (shadow edges), counted apart.
//
// A first pass lists, per run of <= 16 consecutive steps of a block, the region's cells
// with a shadowed step in it.  A CTA then takes 128 listed cells of one run (each warp alone
// where the cells are far apart: contrib_by_fan) and walks the BVH once for all of them
// (walk_group, as the ray-traced accrual does): the pairs of a cell and a triangle that the
// run's rays may reach are tested exactly at each of the cell's shadowed steps (Plucker
// form, with the distance).  Per cell and step the nearest
// hit is kept in shared memory -- distance and triangle in one 64-bit key, so the minimum
// does not depend on the order; equal distances go to the lower triangle index, as a walk
// of the node list in its order gives -- and per cell and run a short list of kCastList
// (building, steps met) pairs.  Where a cell's run meets more buildings than the list holds,
// the CTA walks again for those cells, once per class of building ids modulo kCastSplit,
// and where a class does not fit either, modulo the next power of it.  Counts are integers,
// credited by atomics on per-building totals (runs of equal nearest buildings are credited
// at once).
constexpr int kCastList = 12;               // buildings per cell and run: what five CTAs per SM leave
constexpr unsigned kCastSplit = 4;          // classes per level when the list runs out
constexpr int kCastLevels = 16;             // 4^15 classes of 2^31 ids: none holds more than the list
constexpr unsigned kRayMost = 64;           // buildings a ray may meet: more are reported
constexpr int kContribChunk = 64;           // triangles staged per pass
constexpr int kContribCtas = 5;             // resident CTAs per SM

struct ContribArgs {
    DevScene sc;
    const StepConst* steps;
    const BlockConst* runs;           // runs of <= kContribRun steps; mask_block / mask_bit locate them
    const RunLight* lights;           // their light-space constants
    int n_runs;
    const unsigned long long* masks;  // the raster's step masks [blocks][R]
    long long R;
    float x0, y0, dx;
    int nx;
    int bx0, by0, bnx, bny;           // the region's bounding box, in cells
    const double2* poly;
    int n;
    unsigned long long* cast_cnt;     // [B]
    unsigned long long* near_cnt;     // [B]
    unsigned long long* stats;        // [2]
    int n_b;                          // buildings (length of the counters)
    // compacted work: per run, the cells with a shadowed step in it (global cell index)
    const int* items;                 // run r's cells at item0[r] .. item0[r] + n_items[r]
    const unsigned* item0;            // [n_runs]
    const unsigned* n_items;          // [n_runs]
    const int* cta_base;              // [n_runs + 1] first CTA of each run
    const unsigned* by_fan;           // [n_runs] not 0: the run's cells go to k_contribution_fan
};

// What a CTA's walks leave for its threads' cells.
struct ContribLists {
    unsigned long long key[kContribRun][kTileThreads];   // nearest hit: distance bits, triangle + 1
    int cb[kCastList][kTileThreads];          // casting list: building, -1 when free
    unsigned cm[kCastList][kTileThreads];     //               steps whose ray meets it
    unsigned over[kCastLevels][kTileThreads / 32];   // per level, the cells whose list ran out
};

// A CTA's shared memory: of the grouped walk, and of the walk by warps.
struct ContribSmem {
    ContribLists c;
    LightSmem<kContribChunk> l;               // l.m: the cells' shadowed steps
    GroupSmem<kContribChunk, 512> g;
};
struct ContribFanSmem {
    union {
        ContribLists c;
        int ids[kRayMost][kTileThreads];      // of the recount: the buildings a ray has met
    };
    BlockConst bc;
    float4 d[kContribRun], r[kContribRun];    // the run's directions and their reciprocals
};
static_assert(sizeof(ContribSmem) <= 227 * 1024 / kContribCtas - 1024, "resident CTAs per SM");

// Work list of the traversal: per run, the region's cells with at least one shadowed
// step in it, in patch order (8 x 4 cells per patch; strips of kStrip patch rows, column by column), so
// that the 128 cells a CTA takes stay close together.  Cells shadowed at no step of a run
// cost nothing there.  Two passes over the patches: counts per (run, patch), then -- after
// an exclusive scan of the counts into offsets -- the cells themselves.
constexpr int kStrip = 8;

__host__ __device__ inline long long contrib_patches(int bnx, int bny) {
    return (long long)((bnx + 7) / 8) * (((bny + 3) / 4 + kStrip - 1) / kStrip * kStrip);
}

__global__ void k_contrib_items(ContribArgs a, bool fill, unsigned* __restrict__ counts,
                                const unsigned* __restrict__ offsets, int* __restrict__ items) {
    const int lane = threadIdx.x & 31;
    const int tiles_x = (a.bnx + 7) >> 3;
    const long long n_patches = contrib_patches(a.bnx, a.bny);
    const long long warp_id = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp_id >= n_patches) return;                                  // whole warps
    const int strip = (int)(warp_id / (tiles_x * kStrip)), at = (int)(warp_id - (long long)strip * tiles_x * kStrip);
    const int tx = at / kStrip, ty = strip * kStrip + at % kStrip;
    const int lx = tx * 8 + (lane & 7), ly = ty * 4 + (lane >> 3);
    const int ix = a.bx0 + lx, iy = a.by0 + ly;
    const float x = __fadd_rn(a.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), a.dx));
    const float y = __fadd_rn(a.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), a.dx));
    const bool in_region = lx < a.bnx && ly < a.bny && inside_polygon(a.poly, a.n, (double)x, (double)y);
    const long long cell = (long long)iy * a.nx + ix;
    for (int r = 0; r < a.n_runs; ++r) {
        const BlockConst& bc = a.runs[r];
        const unsigned run_bits = bc.K >= 32 ? 0xffffffffu : ((1u << bc.K) - 1u);
        const bool want = in_region &&
                          ((unsigned)(a.masks[(long long)bc.mask_block * a.R + cell] >> bc.mask_bit) & run_bits) != 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, want);
        const long long slot = (long long)r * n_patches + warp_id;
        if (!fill) {
            if (lane == 0) counts[slot] = (unsigned)__popc(bal);
        } else if (want) {
            items[offsets[slot] + __popc(bal & ((1u << lane) - 1u))] = (int)cell;
        }
    }
}

// The thread's cell of a run.
struct ContribCell {
    int r;                // the CTA's run
    bool live;
    unsigned m;           // the run's steps at which the cell is shadowed
    float4 p;             // its ray's origin and t_min
};

__device__ __forceinline__ ContribCell contrib_cell(const ContribArgs& a) {
    ContribCell c;
    // the first run whose CTAs end past this one (runs without cells have none)
    c.r = 0;
    for (int end = a.n_runs - 1; c.r < end;) {
        const int mid = (c.r + end) >> 1;
        if (a.cta_base[mid + 1] <= (int)blockIdx.x) c.r = mid + 1;
        else end = mid;
    }
    const unsigned slot = (unsigned)((int)blockIdx.x - a.cta_base[c.r]) * (unsigned)kTileThreads + threadIdx.x;
    c.live = slot < a.n_items[c.r];
    const long long cell = c.live ? (long long)SA_CHK(a.items[(long long)a.item0[c.r] + slot], a.R, sa::CK_CONTRIB_CELL) : 0;
    const int ix = (int)(cell % a.nx), iy = (int)(cell / a.nx);
    const BlockConst& bc = a.runs[c.r];
    const unsigned run_bits = bc.K >= 32 ? 0xffffffffu : ((1u << bc.K) - 1u);
    c.m = c.live ? (unsigned)(a.masks[(long long)bc.mask_block * a.R + cell] >> bc.mask_bit) & run_bits : 0u;
    c.p = make_float4(__fadd_rn(a.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), a.dx)),
                      __fadd_rn(a.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), a.dx)), 0.f, kGroundTmin);
    return c;
}

// A walk's pass over the buildings with id = rem modulo mod = kCastSplit^level, for the cells
// whose list ran out a level above.
struct ContribPass {
    int level = 0;
    unsigned mod = 1, rem = 0;
    // the pass after this one, whose lists ran out for some cell if `split`; false: none
    __device__ __forceinline__ bool next(bool split) {
        if (split) {
            ++level;
            mod *= kCastSplit;
            return true;
        }
        while (level > 0 && rem >= mod - mod / kCastSplit) {     // the last class of its level
            rem -= mod - mod / kCastSplit;
            mod /= kCastSplit;
            --level;
        }
        rem += mod / kCastSplit;
        return level > 0;
    }
};

__device__ __forceinline__ bool starts_pass(ContribLists& s, const ContribPass& ps, bool live) {
    const int tid = threadIdx.x, lane = tid & 31;
    const bool mine = ps.level == 0 ? live : ((s.over[ps.level - 1][tid >> 5] >> lane) & 1u) != 0u;
#pragma unroll
    for (int e = 0; e < kCastList; ++e) {
        s.cb[e][tid] = -1;
        s.cm[e][tid] = 0u;
    }
    if (lane == 0) s.over[ps.level][tid >> 5] = 0u;
    return mine;
}

// Building bid is met at the steps `hits` of cell `who`.
__device__ __forceinline__ void put_casting(ContribLists& s, int who, int bid, unsigned hits, unsigned* over) {
    int i = 0;
    for (; i < kCastList; ++i) {
        int cur = *(volatile int*)&s.cb[i][who];
        if (cur < 0) {
            cur = atomicCAS(&s.cb[i][who], -1, bid);
            if (cur < 0) cur = bid;
        }
        if (cur == bid) break;
    }
    if (i < kCastList) atomicOr(&s.cm[i][who], hits);
    else atomicOr(&over[who >> 5], 1u << (who & 31));
}

// Adds the warp's credits, n of building bid per lane (0: none).  The totals of a small city
// are few words, which an atomic per cell and run queues at: one per warp and building then
// (16 buildings, 328^2 cells, 481 steps: whole call 3.88 -> 1.16 ms).  Where a warp's cells
// meet many buildings, in an order of their own, that costs more than it saves (2,000
// buildings, 512^2 cells: 1.94 -> 1.97).
constexpr int kFewBuildings = 256;

__device__ __forceinline__ void credit_warp(unsigned long long* cnt, int n_b, int bid, unsigned n) {
    if (n_b > kFewBuildings) {
        if (n) atomicAdd(&cnt[bid], (unsigned long long)n);
        return;
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, n != 0u); todo;) {
        const int lead = __ffs(todo) - 1, b = __shfl_sync(0xffffffffu, bid, lead);
        const bool same = n != 0u && bid == b;
        const unsigned sum = __reduce_add_sync(0xffffffffu, same ? n : 0u);
        if ((int)(threadIdx.x & 31) == lead) atomicAdd(&cnt[b], (unsigned long long)sum);
        todo &= ~__ballot_sync(0xffffffffu, same);
    }
}

// Credits what a pass found for the thread's cell (steps m; mine, and its list not run out:
// the casting); returns, from the first pass, the steps at which a building was met.  Whole
// warps.
__device__ __forceinline__ unsigned credit_pass(const ContribArgs& a, ContribLists& s, const ContribPass& ps, bool mine,
                                                bool ovf, unsigned m) {
    const int tid = threadIdx.x;
    unsigned found = 0u;
    if (ps.level == 0) {
        // nearest: a stretch of steps with the same building at a time
        int last = -1, at = -1;                       // a triangle, and its building
        for (unsigned rest = m; __any_sync(0xffffffffu, rest != 0u);) {
            int bid = -1;
            unsigned n = 0;
            while (rest) {
                const int k = __ffs(rest) - 1;
                const unsigned long long key = s.key[k][tid];
                if (key != ~0ull) {
                    const int tri = (int)((unsigned)key - 1u);
                    if (tri != last) {
                        last = tri;
                        at = (int)SA_CHK(__float_as_int(__ldg(&a.sc.tris[3 * tri]).w), a.n_b, sa::CK_CONTRIB_BUILDING);
                    }
                    if (n != 0u && at != bid) break;
                    bid = at;
                    ++n;
                    found |= 1u << k;
                }
                s.key[k][tid] = 0ull;                 // from here on: buildings met at the step
                rest &= rest - 1u;
            }
            credit_warp(a.near_cnt, a.n_b, bid, n);
        }
    }
    const bool credit = mine && !ovf;
    for (int e = 0; e < kCastList; ++e) {
        const int bid = credit ? s.cb[e][tid] : -1;
        if (!__any_sync(0xffffffffu, bid >= 0)) break;
        unsigned met = bid >= 0 ? s.cm[e][tid] : 0u;
        if (ps.level > 0)                         // a ray's first kRayMost buildings are credited
            for (unsigned w = met; w; w &= w - 1u)
                if (s.key[__ffs(w) - 1][tid]++ >= kRayMost) met &= ~(w & (0u - w));
        credit_warp(a.cast_cnt, a.n_b, bid, (unsigned)__popc(met));
    }
    return found;
}

// The cell-steps that met no building (`grazed`), and the rays past kRayMost of them.
__device__ __forceinline__ void credit_stats(const ContribArgs& a, unsigned grazed, unsigned long long n_over) {
    unsigned long long n_graze = (unsigned long long)__popc(grazed);
    for (int q = 16; q > 0; q >>= 1) {
        n_graze += __shfl_down_sync(0xffffffffu, n_graze, q);
        n_over += __shfl_down_sync(0xffffffffu, n_over, q);
    }
    if ((threadIdx.x & 31) == 0) {
        if (n_over) atomicAdd(&a.stats[0], n_over);
        if (n_graze) atomicAdd(&a.stats[1], n_graze);
    }
}

// Tests n <= 32 queued pairs of a warp, one per lane: the hits of a pair's wanted steps go
// into its cell's keys (nearest) and casting list.
__device__ __forceinline__ void drain_contrib(ContribSmem& s, const unsigned short* q, int n, int kn, int n_b,
                                              bool nearest, unsigned* over) {
    const int lane = threadIdx.x & 31;
    if (lane >= n) return;
    const unsigned e = q[lane];
    const int who = (int)(e >> 8), t = (int)(e & 0xffu);
    LightSmem<kContribChunk>& l = s.l;
    const float4 p = l.o[who];
    const float4 a = l.tri[3 * t], b = l.tri[3 * t + 1], c = l.tri[3 * t + 2], nv = l.n[t];
    const PluckerTri pt = plucker_setup_n(make_float3(p.x, p.y, p.z), a, b, c, make_float3(nv.x, nv.y, nv.z));
    unsigned long long M[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[i][j] = f2_pack(pt.m[i][j], pt.m[i][j]);
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < kContribRun; k += 2) {
        if (k >= kn) break;
        const unsigned long long dx = l.d2[k >> 1][0], dy = l.d2[k >> 1][1], dz = l.d2[k >> 1][2];
        float sv[3][2];
#pragma unroll
        for (int i = 0; i < 3; ++i)
            f2_unpack(f2_fma(dz, M[i][2], f2_fma(dy, M[i][1], f2_mul(dx, M[i][0]))), sv[i][0], sv[i][1]);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (min3f(sv[0][h], sv[1][h], sv[2][h]) >= 0.f || max3f(sv[0][h], sv[1][h], sv[2][h]) <= 0.f)
                m |= 1u << (k + h);
    }
    m &= l.m[who];
    // inside the edges at a wanted step: the distance decides (plucker_hit's roundings)
    unsigned hits = 0;
    const unsigned tri = l.front[t];                  // its index + 1
    while (m) {
        const int k = __ffs(m) - 1;
        m &= m - 1u;
        float dx[2], dy[2], dz[2];
        f2_unpack(l.d2[k >> 1][0], dx[0], dx[1]);
        f2_unpack(l.d2[k >> 1][1], dy[0], dy[1]);
        f2_unpack(l.d2[k >> 1][2], dz[0], dz[1]);
        const bool odd = k & 1;
        const float nd = fmaf(odd ? dz[1] : dz[0], pt.nz,
                              fmaf(odd ? dy[1] : dy[0], pt.ny, __fmul_rn(odd ? dx[1] : dx[0], pt.nx)));
        const float lim = __fmul_rn(p.w, nd);
        if ((nd > 0.f && pt.aon > lim) || (nd < 0.f && pt.aon < lim)) {
            hits |= 1u << k;
            const unsigned long long key =
                ((unsigned long long)__float_as_uint(pt.aon / nd) << 32) | tri;   // distance > 0
            if (nearest && key < *(volatile unsigned long long*)&s.c.key[k][who]) atomicMin(&s.c.key[k][who], key);
        }
    }
    if (hits) put_casting(s.c, who, (int)SA_CHK(__float_as_int(a.w), n_b, sa::CK_CONTRIB_BUILDING), hits, over);
}

// Bound by the latency of the pairs' culls and tests at 20 warps per SM (the keys and lists
// fill its shared memory).  512 x 512 cells, 2000 buildings, 481 steps in June, the whole
// call: 3.49 ms with a warp walking the node list with 32 cells' fans, 1.86 ms grouped (2.21
// in runs of 32 steps with eight list entries, which leave 16 warps per SM, and patches row
// by row; patches in strips of 8 rows 1.86, of 4 1.95, row by row 2.41).  A December day,
// where a run meets more buildings than a list holds: 1000 buildings, 300 x 200 cells 24.9
// -> 6.4 ms (a recount ray by ray for those cells: 16.6; classes of 8 and lists of 8: 7.0).
__global__ void __launch_bounds__(kTileThreads, kContribCtas)
k_building_contribution(ContribArgs a) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    ContribSmem& s = *reinterpret_cast<ContribSmem*>(s_raw);
    const int tid = threadIdx.x, lane = tid & 31;
    const ContribCell c = contrib_cell(a);
    if (a.by_fan[c.r]) return;
    const RunLight& rl = a.lights[c.r];
    const int K = a.runs[c.r].K;
    for (int k = 0; k < K; ++k) s.c.key[k][tid] = ~0ull;
    s.l.o[tid] = c.p;
    stage_directions(s.l, a.steps, rl);
    unsigned long long n_box = 0;
    unsigned found = 0u;
    ContribPass ps;
    bool ovf;
    do {
        const bool mine = starts_pass(s.c, ps, c.live);
        s.l.m[tid] = mine ? c.m : 0u;
        walk_group<false>(
            s.l, s.g, a.sc, rl, mine, c.p,
            [&](int tri) {
                const bool in = ps.mod == 1u || (unsigned)__float_as_int(__ldg(&a.sc.tris[3 * tri]).w) % ps.mod == ps.rem;
                return in ? (unsigned)tri + 1u : 0u;
            },
            n_box, [&](int nt, float la, float lb) {
                light_pass(s.l, rl, nt, mine, c.p, la, lb, 0u, [&](const unsigned short* q, int n) {
                    drain_contrib(s, q, n, K, a.n_b, ps.level == 0, s.c.over[ps.level]);
                });
                return false;
            });
        ovf = (s.c.over[ps.level][tid >> 5] >> lane) & 1u;
        found |= credit_pass(a, s.c, ps, mine, ovf, c.m);
    } while (ps.next(__syncthreads_or(ovf)));
    unsigned lost = 0u;
    for (unsigned rest = found; rest; rest &= rest - 1u)
        if (s.c.key[__ffs(rest) - 1][tid] > kRayMost) ++lost;
    credit_stats(a, c.m & ~found, lost);
}

// The same by warps: each walks the node list for its 32 cells, a node entered when any
// cell's own fan of the run's rays overlaps it, and every lane tests its cell.  A cell whose
// run meets more buildings than its list holds counts them again ray by ray, each lane
// alone.  For the runs of contrib_by_fan.
__global__ void __launch_bounds__(kTileThreads, 6)
k_contribution_fan(ContribArgs a) {
    __shared__ ContribFanSmem s;
    const int tid = threadIdx.x, lane = tid & 31;
    const ContribCell c = contrib_cell(a);
    if (!a.by_fan[c.r]) return;
    const float3 o = make_float3(c.p.x, c.p.y, c.p.z);
    for (int w = tid; w < (int)(sizeof(BlockConst) / 4); w += kTileThreads)
        reinterpret_cast<int*>(&s.bc)[w] = reinterpret_cast<const int*>(&a.runs[c.r])[w];
    __syncthreads();
    const BlockConst& bc = s.bc;
    const int K = bc.K;
    if (tid < K) {
        const StepConst& st = a.steps[bc.j0 + tid];
        s.d[tid] = make_float4(st.dx, st.dy, st.dz, 0.f);
        s.r[tid] = make_float4(st.ix, st.iy, st.iz, 0.f);
    }
    for (int k = 0; k < K; ++k) s.c.key[k][tid] = ~0ull;
    const ContribPass ps;                          // one pass
    starts_pass(s.c, ps, c.live);
    __syncthreads();
    const bool wedge = bc.wedge_ok != 0.f;
    for (int i = __any_sync(0xffffffffu, c.m != 0u) ? 0 : a.sc.n_nodes; i < a.sc.n_nodes;) {
        const float4 lo = __ldg(&a.sc.nodes[2 * i]);
        const float4 hi = __ldg(&a.sc.nodes[2 * i + 1]);
        const int esc = SA_ESC(__float_as_int(lo.w), i, a.sc.n_nodes, sa::CK_TRACE_ESCAPE);
        const int tri = SA_LEAF(__float_as_int(hi.w), a.sc.T, sa::CK_TRACE_LEAF);
        const bool in = c.m != 0u && (wedge ? fan_box(o, bc, lo, hi) : slope_box(o, bc, lo, hi));
        if (tri < 0) {
            i = __any_sync(0xffffffffu, in) ? i + 1 : esc;
            continue;
        }
        i = esc;
        unsigned cand = 0u;
        float4 ta, tb, tc;
        if (in) {
            ta = __ldg(&a.sc.tris[3 * tri]);
            tb = __ldg(&a.sc.tris[3 * tri + 1]);
            tc = __ldg(&a.sc.tris[3 * tri + 2]);
            if (plane_reachable(o, ta, tb, tc, bc)) {
                int ka, kb;
                candidate_steps(o, bc, bc.psi, ta, tb, tc, &ka, &kb);
                if (ka <= kb) cand = c.m & ((2u << kb) - 1u) & ~((1u << ka) - 1u);
            }
        }
        const int wa = __reduce_min_sync(0xffffffffu, cand ? __ffs(cand) - 1 : 32);
        const int wb = __reduce_max_sync(0xffffffffu, cand ? 31 - __clz(cand) : -1);
        if (wa > wb) continue;
        unsigned hits = 0u;
        PluckerTri pt;
        if (cand) pt = plucker_setup(o, ta, tb, tc);
        for (int k = wa; k <= wb; ++k) {
            if (!((cand >> k) & 1u)) continue;
            const float4 d = s.d[k];
            if (!plucker_hit(pt, d.x, d.y, d.z, kGroundTmin)) continue;
            hits |= 1u << k;
            const float nd = fmaf(d.z, pt.nz, fmaf(d.y, pt.ny, __fmul_rn(d.x, pt.nx)));
            const unsigned long long key =
                ((unsigned long long)__float_as_uint(pt.aon / nd) << 32) | ((unsigned)tri + 1u);
            if (key < s.c.key[k][tid]) s.c.key[k][tid] = key;
        }
        if (hits) put_casting(s.c, tid, (int)SA_CHK(__float_as_int(ta.w), a.n_b, sa::CK_CONTRIB_BUILDING), hits, s.c.over[0]);
    }
    __syncwarp();
    const bool ovf = (s.c.over[0][tid >> 5] >> lane) & 1u;
    const unsigned found = credit_pass(a, s.c, ps, c.live, ovf, c.m);
    __syncthreads();                               // the lists of all lanes are done with
    unsigned lost = 0u;
    for (unsigned todo = ovf ? found : 0u; todo; todo &= todo - 1u) {
        const int k = __ffs(todo) - 1;
        const float4 d = s.d[k], r = s.r[k];
        int n = 0;
        bool more = false;
        for (int i = 0; i < a.sc.n_nodes;) {
            const float4 lo = __ldg(&a.sc.nodes[2 * i]), hi = __ldg(&a.sc.nodes[2 * i + 1]);
            const int esc = SA_ESC(__float_as_int(lo.w), i, a.sc.n_nodes, sa::CK_TRACE_ESCAPE);
            const int tri = SA_LEAF(__float_as_int(hi.w), a.sc.T, sa::CK_TRACE_LEAF);
            if (!hit_box_before(o, r.x, r.y, r.z, lo, hi, 3.4e38f)) {
                i = esc;
                continue;
            }
            if (tri < 0) {
                i = i + 1;
                continue;
            }
            i = esc;
            const float4 ta = __ldg(&a.sc.tris[3 * tri]);
            if (!plucker_hit(plucker_setup(o, ta, __ldg(&a.sc.tris[3 * tri + 1]), __ldg(&a.sc.tris[3 * tri + 2])), d.x, d.y,
                             d.z, kGroundTmin))
                continue;
            const int bid = (int)SA_CHK(__float_as_int(ta.w), a.n_b, sa::CK_CONTRIB_BUILDING);
            int e = 0;
            while (e < n && s.ids[e][tid] != bid) ++e;
            if (e < n) continue;
            if (n < (int)kRayMost) s.ids[n++][tid] = bid;
            else more = true;
        }
        for (int e = 0; e < n; ++e) atomicAdd(&a.cast_cnt[s.ids[e][tid]], 1ull);
        lost += more;
    }
    credit_stats(a, c.m & ~found, lost);
}

// Whether the cells of a run take the walk by warps.  `held`: the scene's triangles over the
// ground of a group's 128 cells, as far apart as the grid's.  A group stages and culls every
// triangle that its box reaches, so on a coarse grid over a large dense city it works for
// few cells at a time; a warp's cells enter only what their own fans meet, but pay for long
// fans, with a low sun (many buildings met, and counted ray by ray past the list) or hours
// between the steps.  Both, whole call, ms by groups / by warps, 200^2 cells over 122k
// triangles: held 17 in June 1.7 / 2.7, 67 5.9 / 4.2, 186 18 / 6.2, 1,073 37 / 5.0; 17 at
// 5-minute steps 1.2 / 1.2, 67 4.7 / 1.8; 67 on a December day 25 / 35, 186 43 / 49, 477
// 104 / 57; 186 for its last half hour of sun (slopes to 20) 6.3 / 16, 477 45 / 20; 67 at hour
// steps in December 13 / 115, 477 43 / 180.  Over 7,400 triangles groups take 2.2 ms at the
// most.
bool contrib_by_fan(const BlockConst& run, const std::vector<StepConst>& steps, int T, double held) {
    if (T < 12000 || (run.K > 1 && run.wedge_ok == 0.f)) return false;
    const StepConst &a = steps[(size_t)run.j0], &b = steps[(size_t)(run.j0 + run.K - 1)];
    const double turn = (double)a.dx * b.dx + (double)a.dy * b.dy + (double)a.dz * b.dz;   // cosine
    const double slope = std::max({fabsf(run.uxlo), fabsf(run.uxhi), fabsf(run.uylo), fabsf(run.uyhi)});
    if (slope <= 5.0) return held > (turn > 0.989 ? 28.0 : 17.0);                          // 0.15
    return turn > 0.36 && held > std::min(350.0, 28.0 * (slope / 5.0) * (slope / 5.0));    // 1.2
}

}  // namespace

cudaError_t launch_building_contribution(const DevScene& sc, const float* scene_box, const DevRecv& rc, const DevSun& sun,
                                         const std::vector<BlockConst>& runs,
                                         const std::vector<StepConst>& h_steps, int n_buildings,
                                         const float* poly_xy, int n, double* casting_out,
                                         double* nearest_out, unsigned long long* stats_out,
                                         cudaStream_t st) {
    const long long R = (long long)rc.nx * rc.ny;
    const int B = n_buildings > 0 ? n_buildings : 1;
    const size_t n_cnt = 2 * (size_t)B + 2;
    cudaError_t e = cudaSuccess;
    unsigned long long *masks = nullptr, *cnt = nullptr;
    int *items = nullptr, *cbase = nullptr;
    RunLight* lights = nullptr;
    unsigned *pcnt = nullptr, *poff = nullptr, *runinfo = nullptr;
    double2* dp = nullptr;
    BlockConst* druns = nullptr;
    std::vector<double2> hp((size_t)n);
    double xmin = 1e300, xmax = -1e300, ymin = 1e300, ymax = -1e300;
    for (int i = 0; i < n; ++i) {
        hp[(size_t)i] = make_double2((double)poly_xy[2 * i], (double)poly_xy[2 * i + 1]);
        xmin = std::min(xmin, hp[(size_t)i].x); xmax = std::max(xmax, hp[(size_t)i].x);
        ymin = std::min(ymin, hp[(size_t)i].y); ymax = std::max(ymax, hp[(size_t)i].y);
    }
    // cells whose centre may lie in the polygon (one cell of margin for rounding)
    const double dx = rc.dx;
    const double fx0 = std::max(0.0, std::floor((xmin - rc.x0) / dx - 0.5) - 1.0);
    const double fx1 = std::min((double)rc.nx - 1.0, std::ceil((xmax - rc.x0) / dx - 0.5) + 1.0);
    const double fy0 = std::max(0.0, std::floor((ymin - rc.y0) / dx - 0.5) - 1.0);
    const double fy1 = std::min((double)rc.ny - 1.0, std::ceil((ymax - rc.y0) / dx - 0.5) + 1.0);
    std::vector<unsigned long long> h_cnt(n_cnt, 0ull);
#define TRY(x) do { e = (x); if (e != cudaSuccess) goto done; } while (0)
    TRY(sa::scratch_alloc(&cnt, sizeof(unsigned long long) * n_cnt, st));
    TRY(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * n_cnt, st));
    if (R > 0 && sun.n_blocks > 0 && sc.T > 0 && !runs.empty() && fx0 <= fx1 && fy0 <= fy1) {
        TRY(sa::scratch_alloc(&dp, sizeof(double2) * (size_t)n, st));
        TRY(cudaMemcpyAsync(dp, hp.data(), sizeof(double2) * (size_t)n, cudaMemcpyHostToDevice, st));
        TRY(sa::scratch_alloc(&druns, sizeof(BlockConst) * runs.size(), st));
        TRY(cudaMemcpyAsync(druns, runs.data(), sizeof(BlockConst) * runs.size(), cudaMemcpyHostToDevice, st));
        // the accrual raster's per-block step masks mark the shadowed steps
        TRY(sa::scratch_alloc(&masks, sizeof(unsigned long long) * (size_t)R * sun.n_blocks, st));
        TRY(cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)R * sun.n_blocks, st));
        {
            DevOut out;
            memset(&out, 0, sizeof(out));
            out.masks = reinterpret_cast<uint64_t*>(masks);
            TRY(launch_raster_ground(sc, rc, sun, out, st));
        }
        TRY(sa::scratch_alloc(&lights, sizeof(RunLight) * runs.size(), st));
        TRY(launch_run_lights(sun.steps, druns, (int)runs.size(), 1, lights, st));
        ContribArgs ca;
        ca.sc = sc; ca.steps = sun.steps; ca.runs = druns; ca.lights = lights; ca.n_runs = (int)runs.size();
        ca.masks = masks; ca.R = R;
        ca.x0 = rc.x0; ca.y0 = rc.y0; ca.dx = rc.dx; ca.nx = rc.nx;
        ca.bx0 = (int)fx0; ca.by0 = (int)fy0;
        ca.bnx = (int)fx1 - (int)fx0 + 1; ca.bny = (int)fy1 - (int)fy0 + 1;
        ca.poly = dp; ca.n = n;
        ca.cast_cnt = cnt; ca.near_cnt = cnt + B; ca.stats = cnt + 2 * B; ca.n_b = B;
        // the work lists: per run, the cells with a shadowed step in it, in patch order
        const int nr = (int)runs.size();
        const long long patches = contrib_patches(ca.bnx, ca.bny);
        const long long nslots = patches * nr;
        TRY(sa::scratch_alloc(&pcnt, sizeof(unsigned) * (size_t)(nslots + 1), st));
        TRY(sa::scratch_alloc(&poff, sizeof(unsigned) * (size_t)(nslots + 1), st));
        TRY(sa::scratch_alloc(&cbase, sizeof(int) * (size_t)(nr + 1), st));
        TRY(sa::scratch_alloc(&runinfo, sizeof(unsigned) * 3 * (size_t)nr, st));
        const unsigned pblocks = (unsigned)((patches + 3) / 4);
        k_contrib_items<<<pblocks, 128, 0, st>>>(ca, false, pcnt, nullptr, nullptr);
        TRY(cudaGetLastError());
        TRY(cudaMemsetAsync(pcnt + nslots, 0, sizeof(unsigned), st));
        TRY(cudaMemcpyAsync(poff, pcnt, sizeof(unsigned) * (size_t)(nslots + 1), cudaMemcpyDeviceToDevice, st));
        TRY(exclusive_scan_u32(poff, nslots + 1, nullptr, st));
        // per run: its first item and its count (run r's offsets start at slot r x patches)
        std::vector<unsigned> h_off((size_t)nr + 1);
        TRY(cudaMemcpy2DAsync(h_off.data(), sizeof(unsigned), poff, sizeof(unsigned) * (size_t)patches,
                              sizeof(unsigned), (size_t)nr + 1, cudaMemcpyDeviceToHost, st));
        TRY(cudaStreamSynchronize(st));
        const unsigned total = h_off[(size_t)nr];
        TRY(sa::scratch_alloc(&items, sizeof(int) * ((size_t)total + 1), st));
        k_contrib_items<<<pblocks, 128, 0, st>>>(ca, true, nullptr, poff, items);
        TRY(cudaGetLastError());
        std::vector<unsigned> h_run(3 * (size_t)nr);
        const double area = ((double)scene_box[3] - scene_box[0]) * ((double)scene_box[4] - scene_box[1]);
        const double held = area > 0.0 ? (double)sc.T * kTileThreads * (double)ca.dx * ca.dx / area : 0.0;
        std::vector<int> h_base((size_t)nr + 1, 0);
        for (int r = 0; r < nr; ++r) {
            h_run[(size_t)r] = h_off[(size_t)r];
            h_run[(size_t)nr + r] = h_off[(size_t)r + 1] - h_off[(size_t)r];
            h_run[2 * (size_t)nr + r] = contrib_by_fan(runs[(size_t)r], h_steps, sc.T, held) ? 1u : 0u;
            h_base[(size_t)r + 1] = h_base[(size_t)r] + (int)((h_run[(size_t)nr + r] + kTileThreads - 1u) / kTileThreads);
        }
        TRY(cudaMemcpyAsync(runinfo, h_run.data(), sizeof(unsigned) * 3 * (size_t)nr, cudaMemcpyHostToDevice, st));
        TRY(cudaMemcpyAsync(cbase, h_base.data(), sizeof(int) * (size_t)(nr + 1), cudaMemcpyHostToDevice, st));
        ca.items = items; ca.item0 = runinfo; ca.n_items = runinfo + nr; ca.by_fan = runinfo + 2 * (size_t)nr;
        ca.cta_base = cbase;
        const long long n_fan = std::count(h_run.begin() + 2 * (long long)nr, h_run.end(), 1u);
        const int ctas = h_base[(size_t)nr];
        if (ctas > 0) {
            KernelTimer kt(KT_CONTRIB, st);
            if (n_fan > 0) k_contribution_fan<<<(unsigned)ctas, kTileThreads, 0, st>>>(ca);
            if (n_fan < nr) {
                TRY(cudaFuncSetAttribute(k_building_contribution, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(ContribSmem)));
                k_building_contribution<<<(unsigned)ctas, kTileThreads, sizeof(ContribSmem), st>>>(ca);
            }
        }
        TRY(cudaGetLastError());
    }
    TRY(cudaMemcpyAsync(h_cnt.data(), cnt, sizeof(unsigned long long) * n_cnt, cudaMemcpyDeviceToHost, st));
    TRY(cudaStreamSynchronize(st));
    {
        const double wgt = sun.S > 0 ? (double)rc.dx * (double)rc.dx / (double)sun.S : 0.0;
        for (int b = 0; b < n_buildings; ++b) {
            casting_out[b] = (double)h_cnt[(size_t)b] * wgt;
            nearest_out[b] = (double)h_cnt[(size_t)B + b] * wgt;
        }
        stats_out[0] = h_cnt[2 * (size_t)B];
        stats_out[1] = h_cnt[2 * (size_t)B + 1];
    }
done:
    for (void* p : {(void*)masks, (void*)cnt, (void*)lights, (void*)dp, (void*)druns,
                    (void*)items, (void*)pcnt, (void*)poff, (void*)runinfo, (void*)cbase})
        if (p) cudaFreeAsync(p, st);
    return e;
#undef TRY
}

}  // namespace sa

extern "C" {

sa_status sa_shadow_area(const sa_receivers* grid, const int32_t* steps, int32_t total_steps,
                         const float* poly_xy, int32_t n, void* stream, double* area) {
    const char* who = "sa_shadow_area";
    if (!grid || !steps || !poly_xy || !area)
        return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_area: NULL argument");
    if (!grid->is_grid) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_area: receivers must be a ground grid");
    if (n < 3) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_area: a polygon needs 3 vertices");
    if (total_steps <= 0) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_area: total_steps <= 0");
    std::vector<double2> hp((size_t)n);
    for (int i = 0; i < n; ++i) {
        const float x = poly_xy[2 * i], y = poly_xy[2 * i + 1];
        if (!isfinite(x) || !isfinite(y))
            return sa::report_error(SA_ERR_DEGENERATE, "sa_shadow_area: non-finite polygon vertex");
        hp[(size_t)i] = make_double2((double)x, (double)y);
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    double2* dp = nullptr;
    double* dsum = nullptr;
    double result = 0.0;
    cudaError_t e = sa::scratch_alloc(&dp, sizeof(double2) * (size_t)n, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&dsum, sizeof(double), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dp, hp.data(), sizeof(double2) * (size_t)n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dsum, 0, sizeof(double), st);
    if (e == cudaSuccess && grid->R > 0) {
        const long long blocks = std::min<long long>((grid->R + sa::kAreaThreads - 1) / sa::kAreaThreads, 152ll * 16);
        sa::k_shadow_area<<<(unsigned)blocks, sa::kAreaThreads, 0, st>>>(
            steps, grid->x0, grid->y0, grid->dx, grid->nx, grid->R, dp, n,
            1.0 / (double)total_steps, dsum);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&result, dsum, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (dp) cudaFreeAsync(dp, st);
    if (dsum) cudaFreeAsync(dsum, st);
    if (e != cudaSuccess) {
        char msg[256];
        snprintf(msg, sizeof(msg), "%s: %s", who, cudaGetErrorString(e));
        return sa::report_error(SA_ERR_CUDA, msg);
    }
    *area = result * (double)grid->dx * (double)grid->dx;
    return SA_OK;
}

sa_status sa_shadow_score(const sa_receivers* grid, const int32_t* steps, int32_t n_intervals,
                          const int32_t* total_steps, const float* weights, const float* poly_xy,
                          int32_t n, void* stream, double* score) {
    const char* who = "sa_shadow_score";
    if (!grid || !poly_xy || !score || !total_steps || !weights || (n_intervals > 0 && !steps))
        return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: NULL argument");
    if (!grid->is_grid) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: receivers must be a ground grid");
    if (n < 3) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: a polygon needs 3 vertices");
    if (n_intervals < 1) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: n_intervals < 1");
    std::vector<double> coef((size_t)n_intervals);
    for (int t = 0; t < n_intervals; ++t) {
        if (total_steps[t] <= 0) return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: total_steps <= 0");
        if (!(weights[t] >= -1.f && weights[t] <= 1.f))
            return sa::report_error(SA_ERR_INVALID_ARG, "sa_shadow_score: a weight outside [-1, 1]");
        coef[(size_t)t] = (double)weights[t] / (double)total_steps[t];
    }
    std::vector<double2> hp((size_t)n);
    for (int i = 0; i < n; ++i) {
        const float x = poly_xy[2 * i], y = poly_xy[2 * i + 1];
        if (!isfinite(x) || !isfinite(y))
            return sa::report_error(SA_ERR_DEGENERATE, "sa_shadow_score: non-finite polygon vertex");
        hp[(size_t)i] = make_double2((double)x, (double)y);
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    double2* dp = nullptr;
    double* dcoef = nullptr;
    double* dsum = nullptr;
    double result = 0.0;
    cudaError_t e = sa::scratch_alloc(&dp, sizeof(double2) * (size_t)n, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&dcoef, sizeof(double) * (size_t)n_intervals, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&dsum, sizeof(double), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dp, hp.data(), sizeof(double2) * (size_t)n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dcoef, coef.data(), sizeof(double) * (size_t)n_intervals, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dsum, 0, sizeof(double), st);
    if (e == cudaSuccess && grid->R > 0) {
        const long long blocks = std::min<long long>((grid->R + sa::kAreaThreads - 1) / sa::kAreaThreads, 152ll * 16);
        sa::k_shadow_score<<<(unsigned)blocks, sa::kAreaThreads, 0, st>>>(
            steps, grid->R, n_intervals, dcoef, grid->x0, grid->y0, grid->dx, grid->nx, dp, n, dsum);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&result, dsum, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (dp) cudaFreeAsync(dp, st);
    if (dcoef) cudaFreeAsync(dcoef, st);
    if (dsum) cudaFreeAsync(dsum, st);
    if (e != cudaSuccess) {
        char msg[256];
        snprintf(msg, sizeof(msg), "%s: %s", who, cudaGetErrorString(e));
        return sa::report_error(SA_ERR_CUDA, msg);
    }
    *score = result * (double)grid->dx * (double)grid->dx;
    return SA_OK;
}

}  // extern "C"
