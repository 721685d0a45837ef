// sa_raster.cu -- shadow accrual map of a ground receiver grid (Sec. 4).
//
// The paper's shadow accrual map projects every occluder point s along the block's sun
// directions onto a shadow plane and writes one depth slice per step in a single pass over
// the geometry (Sec. 4, Step 1; Theorem 1 shows the slices equal one shadow map per step).
// For receivers on the ground the shadow plane can be the ground itself: every occluder
// lies above z = 0, so a ground point is shadowed at step j exactly when it lies inside
// the projection of some triangle along d_j onto z = 0 (no depth test is needed, Step 2
// reduces to a coverage test).  The map is therefore kept in receiver space, at the
// receivers themselves, as one bit per step: no texel resampling, no aliasing, no bias.
//
// Per block of <= 64 steps:
//   k_reach           with many (triangle, block) pairs, lists the triangles that can reach
//                     the grid at some step
//   k_bin             one pass over the triangles bins each into the 32 x 32-cell tiles its
//                     projection can reach during the block (the triangle swept along the
//                     block's slope box)
//   k_raster_items    one CTA per tile and block keeps the tile's 1024 x 64-bit slices in
//                     shared memory, projects each binned triangle for every step of the
//                     block, sets bit k of each covered cell and leaves each cell's run
//                     summary
//   k_items_fold      stitches the summaries into the gross / continuous counts
//   k_raster          one CTA per tile, its blocks in series, the reduction fused (the raster
//                     in fixed scratch, and the per-step raster of a large grid)
// With one step per block the same kernels form the per-step shadow raster baseline.
// Batched scenarios: k_batch_base and k_batch_delta change the base city's masks where a
// variant does; k_batch rasters every block of an affected tile (no room for the masks).
//
// Coverage is decided with edge functions evaluated from canonically ordered endpoints,
// so an edge shared by two projected triangles yields exactly negated values in the two
// and a cell centre on it is covered by at least one (watertight).
#include <algorithm>

#include "sa_internal.cuh"

namespace sa {

namespace {

constexpr int kTile = 32;               // cells per tile side
constexpr int kRasterThreads = 256;     // 8 warps x 4 rows each
// triangles staged per batch (<= 64: a unit packs its triangle in 6 bits)
#ifndef SA_RASTER_BATCH
#define SA_RASTER_BATCH 64
#endif
constexpr int kTriBatch = SA_RASTER_BATCH;
static_assert(kTriBatch <= 64, "a unit packs its triangle in 6 bits");
// work units (triangle, run of steps) of a batch: one per thread
constexpr int kMaxUnits = kRasterThreads;
constexpr int kChangeList = 256;        // k_batch_delta: changed triangles picked per round
// resident CTAs per SM the raster kernels are compiled for (registers: 65536 / (256 x this));
// 6 is also what the item kernels' 32 KB of shared memory allow, and 5 what it leaves the
// kernels that hold a tile's running counts beside it (k_raster, k_batch: 44 KB)
#ifndef SA_RASTER_CTAS
#define SA_RASTER_CTAS 6
#endif
constexpr int kStateCtas = 5;

struct TileGeom {
    float x0, y0, dx;
    int nx, ny, tiles_x, tiles_y;
};

__device__ __forceinline__ bool tri_above_ground(const float4& a, const float4& b, const float4& c) {
    return fmaxf(a.z, fmaxf(b.z, c.z)) > 0.f;
}

// Conservative tile range of a triangle swept over a slope box.
__device__ __forceinline__ bool swept_tiles(const float4& a, const float4& b, const float4& c,
                                            float uxlo, float uxhi, float uylo, float uyhi,
                                            const TileGeom& g, int* tx0, int* tx1, int* ty0, int* ty1) {
    float xmin = 3.4e38f, xmax = -3.4e38f, ymin = 3.4e38f, ymax = -3.4e38f;
    const float4* v[3] = {&a, &b, &c};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float z = fmaxf(v[q]->z, 0.f);
        xmin = fminf(xmin, v[q]->x - z * uxhi);
        xmax = fmaxf(xmax, v[q]->x - z * uxlo);
        ymin = fminf(ymin, v[q]->y - z * uyhi);
        ymax = fmaxf(ymax, v[q]->y - z * uylo);
    }
    const float inv = 1.f / (kTile * g.dx);
    // one cell of margin on every side absorbs rounding of the projections
    const float fx0 = floorf((xmin - g.x0 - g.dx) * inv), fx1 = floorf((xmax - g.x0 + g.dx) * inv);
    const float fy0 = floorf((ymin - g.y0 - g.dx) * inv), fy1 = floorf((ymax - g.y0 + g.dx) * inv);
    if (fx1 < 0.f || fy1 < 0.f || fx0 >= (float)g.tiles_x || fy0 >= (float)g.tiles_y) return false;
    *tx0 = (int)fmaxf(fx0, 0.f);
    *tx1 = (int)fminf(fx1, (float)(g.tiles_x - 1));
    *ty0 = (int)fmaxf(fy0, 0.f);
    *ty1 = (int)fminf(fy1, (float)(g.tiles_y - 1));
    return true;
}

// For a closed scene only triangles facing the sun at some step of the block cast the
// shadow's coverage (the projection of a closed solid is covered by its sun-facing faces).
// n: the triangle's unnormalised normal.  The bounds of n . d over the block's direction
// box decide most triangles without the loop over its steps; 1e-5 |n|_1 is far more than
// the rounding of either (3 ulp), so the answer is the loop's.
__device__ __forceinline__ bool faces_sun(const float3& n, const StepConst* steps, const BlockConst& bc) {
    const float hi = fmaxf(n.x * bc.dlo[0], n.x * bc.dhi[0]) + fmaxf(n.y * bc.dlo[1], n.y * bc.dhi[1]) +
                     fmaxf(n.z * bc.dlo[2], n.z * bc.dhi[2]);
    const float lo = fminf(n.x * bc.dlo[0], n.x * bc.dhi[0]) + fminf(n.y * bc.dlo[1], n.y * bc.dhi[1]) +
                     fminf(n.z * bc.dlo[2], n.z * bc.dhi[2]);
    const float tol = 1e-5f * (fabsf(n.x) + fabsf(n.y) + fabsf(n.z));
    if (hi < -tol) return false;
    if (lo > tol) return true;
    for (int k = 0; k < bc.K; ++k) {
        const StepConst& s = steps[bc.j0 + k];
        if (n.x * s.dx + n.y * s.dy + n.z * s.dz > 0.f) return true;
    }
    return false;
}

// The triangles whose shadow may reach the grid at some step of blocks [0, n_blocks): the
// tile range swept over the union of the blocks' slope boxes, with swept_tiles's own margin
// (so a triangle it drops has no tile in any block).  A grid in the middle of a city is
// reached by few: 1024^2 cells among 1.3M triangles, 132 blocks, 3 chunks of k_bin 1.25 ms
// -> 0.27 in 2 and 16 us here, the whole call 8.43 -> 7.47; 231 x 187 cells among 60k, 92 days
// 4.13 -> 3.79 ms.
constexpr int kReachThreads = 256;
__global__ void __launch_bounds__(kReachThreads)
k_reach(DevScene sc, const BlockConst* __restrict__ blocks, int n_blocks, TileGeom g, unsigned* __restrict__ n,
        int* __restrict__ list) {
    __shared__ float s_box[kReachThreads / 32][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float x0 = 3.4e38f, x1 = -3.4e38f, y0 = 3.4e38f, y1 = -3.4e38f;
    for (int b = threadIdx.x; b < n_blocks; b += kReachThreads) {
        x0 = fminf(x0, blocks[b].uxlo);
        x1 = fmaxf(x1, blocks[b].uxhi);
        y0 = fminf(y0, blocks[b].uylo);
        y1 = fmaxf(y1, blocks[b].uyhi);
    }
    for (int o = 16; o > 0; o >>= 1) {
        x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
        y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
    }
    if (lane == 0) { s_box[warp][0] = x0; s_box[warp][1] = x1; s_box[warp][2] = y0; s_box[warp][3] = y1; }
    __syncthreads();
    for (int w = 0; w < kReachThreads / 32; ++w) {
        x0 = fminf(x0, s_box[w][0]);
        x1 = fmaxf(x1, s_box[w][1]);
        y0 = fminf(y0, s_box[w][2]);
        y1 = fmaxf(y1, s_box[w][3]);
    }
    for (long long base = (long long)blockIdx.x * kReachThreads; base < sc.T; base += (long long)gridDim.x * kReachThreads) {
        const long long t = base + threadIdx.x;
        bool in = false;
        if (t < sc.T) {
            const float4 a = __ldg(&sc.tris[3 * t]), b = __ldg(&sc.tris[3 * t + 1]), c = __ldg(&sc.tris[3 * t + 2]);
            int tx0, tx1, ty0, ty1;
            in = tri_above_ground(a, b, c) && swept_tiles(a, b, c, x0, x1, y0, y1, g, &tx0, &tx1, &ty0, &ty1);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        unsigned at = 0u;
        if (lane == 0 && bal) at = atomicAdd(n, (unsigned)__popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) list[at + __popc(bal & ((1u << lane) - 1u))] = (int)t;
    }
}

// Bins of blocks [b0, b0 + nbc), of the n triangles of `list` (null: of all): a thread loads
// its triangle once and takes `per` of the
// blocks (blockIdx.y picks which), so a season's blocks do not read the mesh again each.
// Counting (FILL false) adds to counts[block][tile]; filling writes the triangle at
// offsets[block][tile], or at a fixed place of `cap` triangles per bin when offsets is
// null (a mesh so small that every bin can hold all of it: one pass, nothing to size).
template <bool FILL>
__global__ void k_bin(DevScene sc, const int* __restrict__ list, int n_list, const StepConst* __restrict__ steps,
                      const BlockConst* __restrict__ blocks, int b0, int nbc, int per, TileGeom g,
                      const unsigned* __restrict__ offsets, unsigned cap,
                      unsigned* __restrict__ counts, int* __restrict__ bins) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_list) return;
    const int t = list ? __ldg(&list[i]) : i;
    const float4 a = __ldg(&sc.tris[3 * t]), b = __ldg(&sc.tris[3 * t + 1]),
                 c = __ldg(&sc.tris[3 * t + 2]);
    if (!tri_above_ground(a, b, c)) return;
    const float ux = b.x - a.x, uy = b.y - a.y, uz = b.z - a.z;
    const float vx = c.x - a.x, vy = c.y - a.y, vz = c.z - a.z;
    const float3 n = make_float3(uy * vz - uz * vy, uz * vx - ux * vz, ux * vy - uy * vx);
    const int bl0 = blockIdx.y * per, bl1 = min(nbc, bl0 + per);
    for (int bl = bl0; bl < bl1; ++bl) {
        const BlockConst& bc = blocks[b0 + bl];
        // the tile range first: it culls the triangles whose shadow misses the grid before
        // the facing test (both are conservative, so the order leaves the bins unchanged)
        int tx0, tx1, ty0, ty1;
        if (!swept_tiles(a, b, c, bc.uxlo, bc.uxhi, bc.uylo, bc.uyhi, g, &tx0, &tx1, &ty0, &ty1)) continue;
        if (sc.closed && !faces_sun(n, steps, bc)) continue;
        const size_t row = (size_t)bl * g.tiles_x * g.tiles_y;
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) {
                const size_t cell = row + ty * g.tiles_x + tx;
                const unsigned slot = atomicAdd(&counts[cell], 1u);
                if (FILL) bins[(offsets ? (size_t)offsets[cell] : cell * cap) + slot] = t;
            }
    }
}

constexpr int kBinThreads = 128;

// Grid of k_bin: up to 8 blocks a thread.  More would read the mesh less often still, but a
// triangle inside the grid then makes its atomics for all of them in series (64 blocks a
// thread, 1.5M triangles, a 1024^2 grid in the middle: 2.76 ms, 8 a thread 1.25); fewer where the triangles alone do not fill the chip.
dim3 bin_grid(int T, int nbc, int* per) {
    const int gx = (T + kBinThreads - 1) / kBinThreads;
    *per = std::max(1, std::min(8, (int)((long long)gx * nbc / (152 * 16))));
    if ((nbc + *per - 1) / *per > 65535) *per = (nbc + 65534) / 65535;
    return dim3((unsigned)gx, (unsigned)((nbc + *per - 1) / *per));
}

struct RasterArgs {
    DevScene sc;
    DevSun sun;
    TileGeom g;
    int b0, nbc;                     // first block and number of blocks of this chunk
    const unsigned* offsets;         // [nbc][tiles] bin offsets
    const unsigned* counts;          // [nbc][tiles] bin sizes
    const int* bins;
    DevOut out;
    int* best;                       // continuous state (== out.continuous or scratch)
    int load_state;                  // 0: start from zero, 1: from out.gross / best / run
    int final_chunk;
    int cull;                        // closed scene: only faces toward the sun
    int run;                         // steps per work unit
    long long R;
    const int* order;                // tile (item) of each CTA (null: CTA i takes i)
    unsigned cap;                    // items: triangles per bin when offsets is null
    int parts;                       // items: parts a block's steps are cut into
    unsigned* summary;               // items: run summaries [nbc][parts][R] (nullable)
};

constexpr int kWarpsRaster = kRasterThreads / 32;

struct BatchArgs {
    TileGeom g;
    const float4* base_tris;
    const BatchInterval* intervals;
    const BatchVariant* variants;
    const int4* items;                // (interval, variant, tile, 0)
    int n_items;
    unsigned* counter;                // work queue head, zeroed before the launch
    const int* removed;               // removed base building ids of all variants
    const float4* tower_tris;         // tower triangles of all variants (3 float4 each)
    int* counts_out;
    int* impact_out;                  // nullable
    int cull;
    int run;                          // steps per work unit
    unsigned long long* stats;        // nullable
};
// steps per work unit (run length); a process-wide option, 24 by default
int g_raster_run = 24;

// Edge function of a triangle edge (3D endpoints v -> v') projected along step k, at a
// ground point p (all xy tile-local).  With c = p - v.xy and e = v' - v,
//   E_k(p) = cross(q' - q, p - q),  q = v.xy - v.z u_k,  u_k = d_xy / d_z,
// expands to  E_k(p) = P + Qx u_k.x + Qy u_k.y  with
//   P = e.x c.y - e.y c.x,  Qx = -v.z e.y - e.z c.y,  Qy = v.z e.x + e.z c.x,
// so a cell sets (P, Qx, Qy) up once and tests a run of steps with two FMAs per edge.
// The endpoints are taken in a canonical order (the other order only flips the sign), so
// an edge shared by two triangles gives the same value in both up to an exact negation:
// a cell on it is covered by at least one (watertight).
struct EdgeRef {
    float vx, vy, vz, ex, ey, ez;   // canonical start point, and the edge vector times the
                                    // sign of the triangle's own orientation of the edge
};

// The sign is folded into the edge vector: P, Qx and Qy are then the canonical values
// times +-1, and since rounding to nearest is symmetric under negation every step's edge
// value is the canonical one times +-1 exactly, up to the sign of a zero.  The front test
// takes +0 as inside and -0 as outside; where the two triangles of an edge both get a
// zero, at least one of them gets +0 (a rounded sum of zeros is -0 only when both terms
// are -0, and the other triangle's terms are then +0), so a cell on the edge is covered.
// The back test takes both zeros as inside.
__device__ __forceinline__ EdgeRef edge_ref(const float4& a, const float4& b) {
    const bool keep = a.x < b.x || (a.x == b.x && (a.y < b.y || (a.y == b.y && a.z < b.z)));
    const float4& v = keep ? a : b;
    const float4& w = keep ? b : a;
    const float s = keep ? 1.f : -1.f;
    return EdgeRef{v.x, v.y, v.z, s * (w.x - v.x), s * (w.y - v.y), s * (w.z - v.z)};
}

// The edge's step-test terms as affine functions of the cell centre (x, y): with c = (x, y)
// - v, P = e_x c_y - e_y c_x = pa y + pb x + pc, Q_x = -(v_z e_y + e_z c_y) = -ra y + qc and
// Q_y = v_z e_x + e_z c_x = ra x + rc.  The constants are rounded once per staged triangle,
// each from the edge vector in a way that an exactly negated edge vector negates exactly,
// so the triangles sharing an edge still compute exactly negated values.
struct EdgeLin {
    float pa, pb, pc, ra, qc, rc;
};

__device__ __forceinline__ EdgeLin edge_lin(const EdgeRef& e) {
    EdgeLin l;
    l.pa = e.ex;
    l.pb = -e.ey;
    l.pc = -fmaf(l.pa, e.vy, l.pb * e.vx);
    l.ra = e.ez;
    l.qc = -fmaf(e.vz, e.ey, -(e.ez * e.vy));
    l.rc = fmaf(e.vz, e.ex, -(e.ez * e.vx));
    return l;
}

// Shared memory of one tile: staged triangles (xy tile-local), the block's directions, ground
// slopes and per-run slope boxes, the batch's work units, the tile's step masks and its
// cell centres.
struct TileSmem {
    float4 tri[kTriBatch * 3];
    // the staged triangles' edge functions (EdgeLin, 6 floats each), 20 floats apart so
    // that a cell's test reads them as five float4
    float edges[kTriBatch * 20];
    float4 d[kMaxBlock];                     // step directions
    // slopes (u.x of two steps, u.y of the same two) for the paired step tests: [0][i] starts
    // at step 2i, [1][i] at step 2i + 1 (the last pair of a block repeats its last step)
    float4 up[2][kMaxBlock / 2];
    float2 u[kMaxBlock];
    float4 ubox[kMaxBlock];                  // per run: (min u.x, max u.x, min u.y, max u.y)
    float4 uend[kMaxBlock];                  // per run: slopes of its first and last step
    float2 udev[kMaxBlock];                  // per run: largest |u - chord| over its steps
    // step masks of the cells, steps 0..31 and 32..63 apart: 32-bit shared atomics are one
    // instruction, 64-bit ones a compare-and-swap loop
    unsigned lo[kTile * kTile], hi[kTile * kTile];
    unsigned long long row_full[kTile];      // steps at which every cell of a row is shadowed
    // the batch's units that reach the tile: columns and rows (unit_box) | triangle << 20 |
    // run << 26, the run's facing steps (front; back, open scenes only), and the unit's
    // first row in the list of all units' rows; first[g] is the unit of row 32 g
    unsigned unit[kMaxUnits], fr[kMaxUnits], bk[kMaxUnits];
    unsigned short start[kMaxUnits];
    unsigned char first[kMaxUnits + 1];
    unsigned made;                           // rows << 9 | units
    int next_row;                            // next rows to hand out
    // per warp: the covered rows of a claim, (first cell - first position, unit, steps it can
    // set), and cells waiting for their step tests, unit << 22 | triangle << 16 | first step of
    // its run << 10 | cell, drained 32 at a time so that every lane tests a cell whichever
    // unit it comes from
    int4 row[kRasterThreads / 32][32];
    unsigned queue[kRasterThreads / 32][64];
    float xl[kTile], yl[kTile];
    unsigned char valid[kTriBatch];
    unsigned char run_k0[kMaxBlock + 1];     // first step of each run, and K

    __device__ __forceinline__ unsigned long long mask(int cell) const {
        return ((unsigned long long)hi[cell] << 32) | lo[cell];
    }
    __device__ __forceinline__ void set_mask(int cell, unsigned long long m) {
        lo[cell] = (unsigned)m;
        hi[cell] = (unsigned)(m >> 32);
    }
};

// an SM's 228 KB hold the CTAs that the kernels are compiled for, with 1 KB each of the system's
constexpr int kSmShared = 228 * 1024, kCtaShared = 1024;
static_assert(SA_RASTER_CTAS * (sizeof(TileSmem) + sizeof(int) * (kChangeList + 2) + kCtaShared) <= kSmShared, "items");
static_assert(kStateCtas * (sizeof(TileSmem) + sizeof(RunState) * kTile * kTile + kCtaShared) <= kSmShared, "by tile");

// Tile origin and cell centres in tile-local coordinates; the centres are rounded exactly
// as the receivers' world coordinates, then shifted.
__device__ __forceinline__ void tile_setup(TileSmem& sm, const TileGeom& g, int tx, int ty,
                                           float* tox, float* toy) {
    *tox = __fadd_rn(g.x0, __fmul_rn((float)(tx * kTile), g.dx));
    *toy = __fadd_rn(g.y0, __fmul_rn((float)(ty * kTile), g.dx));
    if (threadIdx.x < kTile) {
        sm.xl[threadIdx.x] = __fadd_rn(g.x0, __fmul_rn(__fadd_rn((float)(tx * kTile + threadIdx.x), 0.5f), g.dx)) - *tox;
    } else if (threadIdx.x < 2 * kTile) {
        const int q = threadIdx.x - kTile;
        sm.yl[q] = __fadd_rn(g.y0, __fmul_rn(__fadd_rn((float)(ty * kTile + q), 0.5f), g.dx)) - *toy;
    }
    for (int c = threadIdx.x; c < kTile * kTile; c += kRasterThreads) sm.set_mask(c, 0ull);
}


// The steps of one run (from k0) that cover cell (x, y): bit k of the result is step k0 + k.
// kmax: steps of the block's longest run, the same for every lane; fr and bk drop the steps
// beyond a shorter run.  CULL: closed scene, only front faces count.
template <bool CULL>
__device__ __forceinline__ unsigned cell_steps(const TileSmem& sm, const EdgeLin& E0,
                                               const EdgeLin& E1, const EdgeLin& E2, float x,
                                               float y, int k0, int kmax, unsigned fr, unsigned bk) {
    float P[3], QX[3], QY[3];
    const EdgeLin* ee[3] = {&E0, &E1, &E2};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const EdgeLin& e = *ee[q];
        P[q] = fmaf(e.pa, y, fmaf(e.pb, x, e.pc));
        QX[q] = fmaf(-e.ra, y, e.qc);
        QY[q] = fmaf(e.ra, x, e.rc);
    }
    // steps in pairs: E = P + Qx u_x + Qy u_y for two steps per packed instruction
    unsigned long long P2[3], QX2[3], QY2[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        P2[q] = f2_pack(P[q], P[q]);
        QX2[q] = f2_pack(QX[q], QX[q]);
        QY2[q] = f2_pack(QY[q], QY[q]);
    }
    const ulonglong2* up = reinterpret_cast<const ulonglong2*>(sm.up[k0 & 1]) + (k0 >> 1);
    // Fully unrolled over the longest run.  A step covers the cell from the front when no
    // edge value has its sign bit set (+0 counts as inside, -0 as outside): that bit is
    // shifted in from the sign word, so the front mask comes out in reverse step order.
    // From the back (open scenes) all three values are <= 0, zeros of either sign
    // included: two back faces sharing an edge may both get +0 there.
    unsigned hf = 0, hb = 0;
#pragma unroll
    for (int k = 0; k < 32; k += 2) {
        if (k >= kmax) break;
        const ulonglong2 u = up[k >> 1];
        float f[3][2];
#pragma unroll
        for (int q = 0; q < 3; ++q) f2_unpack(f2_fma(QY2[q], u.y, f2_fma(QX2[q], u.x, P2[q])), f[q][0], f[q][1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned a = __float_as_uint(f[0][h]), b = __float_as_uint(f[1][h]), c = __float_as_uint(f[2][h]);
            hf = __funnelshift_l(~(a | b | c), hf, 1);
            if (!CULL && max3f(f[0][h], f[1][h], f[2][h]) <= 0.f) hb |= 1u << (k + h);
        }
    }
    // steps 0 .. K2 - 1 (an odd run's last pair repeats a step beyond it, which the masks
    // drop) back in order: step k at bit k
    const int K2 = (kmax + 1) & ~1;
    hf = __brev(hf) >> (32 - K2);
    return CULL ? (hf & fr) : ((hf & fr) | (hb & bk));
}

// Step tests of up to 32 queued cells (n >= 1), one per lane: each item names its work unit
// and its cell; the unit's run, its facing steps and the triangle's canonical edges are
// read back from shared memory.
template <bool COUNT, bool CULL>
__device__ __forceinline__ void drain_cells(TileSmem& sm, const unsigned* q, int n, int kmax,
                                            unsigned long long& n_cell,
                                            unsigned long long& n_test) {
    const int lane = threadIdx.x & 31;
    const unsigned item = q[lane < n ? lane : 0];
    const int j = (int)(item >> 22), cell = (int)SA_CHK(item & 1023u, kTile * kTile, sa::CK_RASTER_CELL);
    const int t = (int)((item >> 16) & 63u), k0 = (int)((item >> 10) & 63u);
    const unsigned fr = sm.fr[j], bk = CULL ? 0u : sm.bk[j];
    const float4* ef = reinterpret_cast<const float4*>(&sm.edges[20 * t]);
    const float4 f0 = ef[0], f1 = ef[1], f2 = ef[2], f3 = ef[3], f4 = ef[4];
    const EdgeLin E0{f0.x, f0.y, f0.z, f0.w, f1.x, f1.y};
    const EdgeLin E1{f1.z, f1.w, f2.x, f2.y, f2.z, f2.w};
    const EdgeLin E2{f3.x, f3.y, f3.z, f3.w, f4.x, f4.y};
    if (COUNT && lane < n) {
        const int sub = (int)(sm.unit[j] >> 26);
        ++n_cell;
        n_test += sm.run_k0[sub + 1] - k0;
    }
    const unsigned hit = cell_steps<CULL>(sm, E0, E1, E2, sm.xl[cell & (kTile - 1)],
                                          sm.yl[cell >> 5], k0, kmax, fr, bk);
    const unsigned long long m = (unsigned long long)hit << k0;
    if (lane < n) {
        if ((unsigned)m) atomicOr(&sm.lo[cell], (unsigned)m);
        if ((unsigned)(m >> 32)) atomicOr(&sm.hi[cell], (unsigned)(m >> 32));
    }
}

// The cells of the tile whose centres (k + 0.5) dx fall in the swept bounding box of the
// projections of triangle t over run `sub`, with 0.01 cell of slack, as columns c0..c1 and
// rows r0..r1 packed 5 bits each (c0 | c1 << 5 | r0 << 10 | r1 << 15); -1 when it reaches no
// cell.
__device__ __forceinline__ int unit_box(const TileSmem& sm, int t, int sub, float inv_dx) {
    const float4 a = sm.tri[3 * t], b = sm.tri[3 * t + 1], c = sm.tri[3 * t + 2];
    const float4 ub = sm.ubox[sub];
    const float uxlo = ub.x, uxhi = ub.y, uylo = ub.z, uyhi = ub.w;
    const float az = fmaxf(a.z, 0.f), bz = fmaxf(b.z, 0.f), cz = fmaxf(c.z, 0.f);
    const float xmin = fminf(a.x - az * uxhi, fminf(b.x - bz * uxhi, c.x - cz * uxhi));
    const float xmax = fmaxf(a.x - az * uxlo, fmaxf(b.x - bz * uxlo, c.x - cz * uxlo));
    const float ymin = fminf(a.y - az * uyhi, fminf(b.y - bz * uyhi, c.y - cz * uyhi));
    const float ymax = fmaxf(a.y - az * uylo, fmaxf(b.y - bz * uylo, c.y - cz * uylo));
    const float fc0 = ceilf(xmin * inv_dx - 0.51f), fc1 = floorf(xmax * inv_dx - 0.49f);
    const float fr0 = ceilf(ymin * inv_dx - 0.51f), fr1 = floorf(ymax * inv_dx - 0.49f);
    if (fc1 < 0.f || fr1 < 0.f || fc0 > (float)(kTile - 1) || fr0 > (float)(kTile - 1) ||
        fc0 > fc1 || fr0 > fr1) return -1;
    const int c0 = (int)fmaxf(fc0, 0.f), c1 = (int)fminf(fc1, (float)(kTile - 1));
    const int r0 = (int)fmaxf(fr0, 0.f), r1 = (int)fminf(fr1, (float)(kTile - 1));
    return c0 | (c1 << 5) | (r0 << 10) | (r1 << 15);
}

// Row span of a unit in tile row `row` (within its box): the cells cs .. cs + w - 1.
// A vertex at height z projects to v.xy - z u_k, and the run's slopes lie within udev of the
// chord between its first and last.  The projections therefore lie in the hull of the two
// end steps' triangles, widened by z_max udev; as the vertices move along one direction,
// the hull's edges are among the two triangles' edges and the three vertices' paths (two
// paths span a trapezoid, whose diagonals are inside).  The hull's x-range over the band
// [y - sy, y + sy], widened by sx, bounds the row's covered cells (0.15 cell and 2 mm of
// slack absorb rounding).  Against the middle step's triangle widened by half of z_max
// times the run's slope box, which a tall triangle or a low sun made far too wide (24 % of
// the district's cell set-ups met no step, 88 % in December): district ground 2.16 -> 2.10
// ms, 1024^2 cells on 16 December 15.6 -> 5.03 ms, 231 x 187 cells, 92 days 4.21 -> 4.09 ms.
__device__ __forceinline__ void row_span(const TileSmem& sm, int t, int sub, int box, int row,
                                         float inv_dx, int* cs, int* w) {
    *cs = 0;
    *w = 0;
    const int c0 = box & 31, c1 = (box >> 5) & 31;
    const float4 a = sm.tri[3 * t], b = sm.tri[3 * t + 1], c = sm.tri[3 * t + 2];
    const float4 ue = sm.uend[sub];
    const float2 dv = sm.udev[sub];
    const float az = fmaxf(a.z, 0.f), bz = fmaxf(b.z, 0.f), cz = fmaxf(c.z, 0.f);
    const float zm = fmaxf(az, fmaxf(bz, cz));
    const float slack = 0.15f + 2e-3f * inv_dx;                 // in cells
    const float y = sm.yl[row];
    const float band = fmaf(zm, dv.y, slack / inv_dx);
    const float ya = y - band, yb = y + band;
    float lo = 3.4e38f, hi = -3.4e38f;
    // the part of segment p - q within the band
    auto clip = [&](float px, float py, float qx, float qy) {
        const float e0 = fminf(py, qy), e1 = fmaxf(py, qy), dy = qy - py;
        if (e1 < ya || e0 > yb) return;
        float xa = px, xb = qx;
        if (e1 - e0 > 1e-4f) {
            // the spans carry slack, so an approximate quotient suffices
            const float slope = __fdividef(qx - px, dy);
            xa = fmaf(fmaxf(ya, e0) - py, slope, px);
            xb = fmaf(fminf(yb, e1) - py, slope, px);
        }
        lo = fminf(lo, fminf(xa, xb));
        hi = fmaxf(hi, fmaxf(xa, xb));
    };
    const float ax = fmaf(-az, ue.x, a.x), ay = fmaf(-az, ue.y, a.y), bx = fmaf(-bz, ue.x, b.x),
                by = fmaf(-bz, ue.y, b.y), cx = fmaf(-cz, ue.x, c.x), cy = fmaf(-cz, ue.y, c.y);
    const float Ax = fmaf(-az, ue.z, a.x), Ay = fmaf(-az, ue.w, a.y), Bx = fmaf(-bz, ue.z, b.x),
                By = fmaf(-bz, ue.w, b.y), Cx = fmaf(-cz, ue.z, c.x), Cy = fmaf(-cz, ue.w, c.y);
    clip(ax, ay, bx, by);
    clip(bx, by, cx, cy);
    clip(cx, cy, ax, ay);
    clip(Ax, Ay, Bx, By);
    clip(Bx, By, Cx, Cy);
    clip(Cx, Cy, Ax, Ay);
    clip(ax, ay, Ax, Ay);
    clip(bx, by, Bx, By);
    clip(cx, cy, Cx, Cy);
    if (lo <= hi) {
        const float sx = zm * dv.x;
        const float f0 = fmaxf(ceilf((lo - sx) * inv_dx - 0.5f - slack), (float)c0);
        const float f1 = fminf(floorf((hi + sx) * inv_dx - 0.5f + slack), (float)c1);
        if (f0 <= f1) {
            *cs = (int)f0;
            *w = (int)f1 - *cs + 1;
        }
    }
}

__device__ __forceinline__ int lane_prefix(int x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += v;
    }
    return x;
}

// Rows rb .. rb + 31 of the batch's units: one lane per row finds its unit and its span; one
// lane per covered cell checks whether the cell is already shadowed at every step its unit
// could set (a stale read only skips less) and queues the others for the step tests, 32
// at a time whichever unit they come from.
template <bool COUNT, bool CULL>
__device__ __forceinline__ void raster_rows(TileSmem& sm, int rb, int rows, int n_units, int kmax, float inv_dx,
                                            int& qn, unsigned long long& n_cell,
                                            unsigned long long& n_test, unsigned long long& n_span) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned upto = 0xffffffffu >> (31 - lane);           // this lane and the ones below
    unsigned* q = sm.queue[warp];
    // the units that start within these rows follow the one that holds row rb: their starts
    // are distinct, so a lane's unit is the count of starts up to it
    const int j0 = sm.first[rb >> 5];
    const int jn = j0 + 1 + lane, at = jn < n_units ? (int)sm.start[jn] - rb : 32;
    const unsigned starts = __reduce_or_sync(0xffffffffu, at < 32 ? 1u << at : 0u);
    const int j = j0 + __popc(starts & upto), ridx = rb + lane;
    int cs = 0, w = 0, what = 0;
    unsigned long long can = 0ull;
    if (ridx < rows) {
        const unsigned un = sm.unit[j];
        const int row = (int)((un >> 10) & 31u) + (ridx - sm.start[j]), sub = (int)(un >> 26);
        const int k0 = sm.run_k0[sub];
        can = (unsigned long long)(CULL ? sm.fr[j] : (sm.fr[j] | sm.bk[j])) << k0;
        what = (j << 22) | (int)((un >> 4) & 0x3f0000u) | (k0 << 10);
        if ((sm.row_full[row] & can) != can)
            row_span(sm, (int)((un >> 20) & 63u), sub, (int)(un & 0xfffffu), row, inv_dx, &cs, &w);
        cs += row * kTile;                                      // the row's first cell
    }
    const int cincl = lane_prefix(w);
    const int total = __shfl_sync(0xffffffffu, cincl, 31);
    if (COUNT && lane == 0) n_span += (unsigned long long)total;
    const int cex = cincl - w;
    const unsigned some = __ballot_sync(0xffffffffu, w > 0);
    // the rows with cells, in order
    if (w > 0)
        sm.row[warp][__popc(some & (upto >> 1))] = make_int4(cs - cex, what, (int)(unsigned)can, (int)(unsigned)(can >> 32));
    __syncwarp();
    int before = -1;                                            // rows that started before this window, less one
    for (int base = 0; base < total; base += 32) {
        const int from = cex - base;
        const unsigned begun = __reduce_or_sync(0xffffffffu, w > 0 && (unsigned)from < 32u ? 1u << from : 0u);
        const int idx = base + lane;
        const bool in = idx < total;
        const int4 info = sm.row[warp][in ? before + __popc(begun & upto) : 0];
        before += __popc(begun);
        const int cell = in ? (int)SA_CHK(info.x + idx, kTile * kTile, sa::CK_RASTER_CELL) : 0;
        const bool need = in && (((unsigned)info.z & ~sm.lo[cell]) | ((unsigned)info.w & ~sm.hi[cell])) != 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, need);
        if (need) q[qn + __popc(bal & (upto >> 1))] = (unsigned)info.y | (unsigned)cell;
        qn += __popc(bal);
        if (qn >= 32) {
            __syncwarp();
            drain_cells<COUNT, CULL>(sm, q + (qn - 32), 32, kmax, n_cell, n_test);
            qn -= 32;
            __syncwarp();
        }
    }
    __syncwarp();
}

// One block of steps of one tile: the n triangles given by fetch(i, vertex, &v) (false =
// skip the triangle) are staged in batches.  A work unit is a triangle and a run of <= 32
// steps; one thread per unit finds its facing steps and swept box, the units that reach
// the tile list their rows, and warps take 32 rows at a time (raster_rows); step bits are
// ORed into the masks.  Leaves the masks complete for the block.
// prefilled: the masks hold bits from the start, whose full rows are skipped at once.
// Bound by issue slots (77 % busy, 26 of 32 lanes active).  Against warps that claimed four
// units at a time and expanded them lane by lane (a binary search in shuffles for every row
// and cell, 64-bit shared atomics, step loops of differing lengths): district ground 2.10 ->
// 1.65 ms, 231 x 187 cells x 92 days 4.09 -> 3.38 ms, 16 scenarios 4.43 -> 3.38 ms.  48
// triangles a batch measure the same, 32 2 % more, 5 and 4 CTAs per SM 3 and 9 % more.
template <bool COUNT, bool CULL, class Fetch>
__device__ void raster_block(TileSmem& sm, const Fetch& fetch, int n, const StepConst* steps,
                             int j0, int K, float tox, float toy, float inv_dx, int kSub,
                             unsigned long long& n_cell, unsigned long long& n_test,
                             unsigned long long& n_unit, unsigned long long& n_span,
                             bool prefilled = false) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nsub = (K + kSub - 1) / kSub, kmax = (K + nsub - 1) / nsub;
    const int batch = min(kTriBatch, kMaxUnits / nsub);
    __syncthreads();
    if (threadIdx.x < K) {
        const StepConst& s = steps[j0 + threadIdx.x];
        sm.u[threadIdx.x] = make_float2(s.ux, s.uy);
        sm.d[threadIdx.x] = make_float4(s.dx, s.dy, s.dz, 0.f);
    }
    __syncthreads();
    if (threadIdx.x < K) {
        const int k = threadIdx.x, k1 = min(k + 1, K - 1);
        sm.up[k & 1][k >> 1] = make_float4(sm.u[k].x, sm.u[k1].x, sm.u[k].y, sm.u[k1].y);
    }
    if (threadIdx.x <= nsub) sm.run_k0[threadIdx.x] = (unsigned char)(threadIdx.x * K / nsub);
    if (threadIdx.x < kTile) sm.row_full[threadIdx.x] = 0ull;
    // per run, a warp with a step per lane: the slope box, the end steps, and the largest
    // deviation from the chord between them
    for (int run = warp; run < nsub; run += kWarpsRaster) {
        const int k0 = run * K / nsub, kn = (run + 1) * K / nsub - k0;
        const float2 p = sm.u[k0], q = sm.u[k0 + kn - 1], u = sm.u[k0 + min(lane, kn - 1)];
        const float ex = q.x - p.x, ey = q.y - p.y, e2 = ex * ex + ey * ey;
        const float t = e2 > 0.f ? fminf(fmaxf(((u.x - p.x) * ex + (u.y - p.y) * ey) / e2, 0.f), 1.f) : 0.f;
        float x0 = u.x, x1 = u.x, y0 = u.y, y1 = u.y;
        float dx = fabsf(fmaf(-t, ex, u.x - p.x)), dy = fabsf(fmaf(-t, ey, u.y - p.y));
        for (int o = 16; o > 0; o >>= 1) {
            x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
            x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
            y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
            y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
            dx = fmaxf(dx, __shfl_xor_sync(0xffffffffu, dx, o));
            dy = fmaxf(dy, __shfl_xor_sync(0xffffffffu, dy, o));
        }
        if (lane == 0) {
            sm.ubox[run] = make_float4(x0, x1, y0, y1);
            sm.uend[run] = make_float4(p.x, p.y, q.x, q.y);
            // (rounding of u and of the deviation itself: a few ulp of |u|)
            const float ulp = 1e-6f * (fabsf(p.x) + fabsf(p.y) + fabsf(q.x) + fabsf(q.y));
            sm.udev[run] = make_float2(dx + ulp, dy + ulp);
        }
    }
    for (int base = 0; base < n; base += batch) {
        const int nt = min(batch, n - base);
        __syncthreads();
        for (int i = threadIdx.x; i < nt * 3; i += kRasterThreads) {
            float4 v;
            const bool ok = fetch(base + i / 3, i % 3, &v);
            v.x -= tox;
            v.y -= toy;
            sm.tri[i] = v;
            if (i % 3 == 0) sm.valid[i / 3] = ok ? 1 : 0;
        }
        // the steps at which a whole row is shadowed already, and (below) the whole tile:
        // no later triangle can change them there, so its units lose those steps and rows
        // before their spans are found, and a tile shadowed at every step is done.  A low
        // sun bins thousands of triangles to a tile that the first few hundred fill
        // (1024^2 cells, 16 December: 25.0 -> 16.4 ms; the June district is unchanged).
        if (base > 0 || prefilled) {
            for (int row = warp; row < kTile; row += kWarpsRaster) {
                const unsigned lo = __reduce_and_sync(0xffffffffu, sm.lo[row * kTile + lane]);
                const unsigned hi = __reduce_and_sync(0xffffffffu, sm.hi[row * kTile + lane]);
                if (lane == 0) sm.row_full[row] = ((unsigned long long)hi << 32) | lo;
            }
        }
        if (threadIdx.x == 0) {
            sm.next_row = kWarpsRaster * 32;
            sm.made = 0u;
        }
        __syncthreads();
        unsigned long long tile_full = 0ull;
        if (base > 0 || prefilled) {
            const unsigned long long m = sm.row_full[lane];
            tile_full = ((unsigned long long)__reduce_and_sync(0xffffffffu, (unsigned)(m >> 32)) << 32) |
                        __reduce_and_sync(0xffffffffu, (unsigned)m);
            const unsigned long long all = K >= 64 ? ~0ull : (1ull << K) - 1ull;
            if ((tile_full & all) == all) break;
        }
        if (threadIdx.x < nt * 3) {
            const int t = threadIdx.x / 3, e = threadIdx.x - 3 * t;
            const EdgeLin l = edge_lin(edge_ref(sm.tri[threadIdx.x], sm.tri[e == 2 ? 3 * t : threadIdx.x + 1]));
            float* o = &sm.edges[20 * t + 6 * e];
            o[0] = l.pa; o[1] = l.pb; o[2] = l.pc; o[3] = l.ra; o[4] = l.qc; o[5] = l.rc;
        }
        // this thread's unit: triangle t, run sub (neighbouring lanes share the run)
        int box = -1, t = 0, sub = 0;
        unsigned fr = 0u, bk = 0u;
        if (threadIdx.x < nt * nsub) {
            sub = threadIdx.x / nt;
            t = threadIdx.x - sub * nt;
            if (sm.valid[t]) {
                const float4 a = sm.tri[3 * t], b = sm.tri[3 * t + 1], c = sm.tri[3 * t + 2];
                const float ux = b.x - a.x, uy = b.y - a.y, uz = b.z - a.z;
                const float vx = c.x - a.x, vy = c.y - a.y, vz = c.z - a.z;
                const float nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
                const int k0 = sm.run_k0[sub], kn = sm.run_k0[sub + 1] - k0;
                for (int k = 0; k < kn; ++k) {
                    const float4 d = sm.d[k0 + k];
                    const float nd = nx * d.x + ny * d.y + nz * d.z;
                    if (nd > 0.f) fr |= 1u << k;
                    if (!CULL && nd < 0.f) bk |= 1u << k;
                }
                const unsigned open = ~(unsigned)(tile_full >> k0);
                fr &= open;
                bk &= open;
                if (fr | bk) box = unit_box(sm, t, sub, inv_dx);
            }
        }
        const int rows = box < 0 ? 0 : ((box >> 15) & 31) - ((box >> 10) & 31) + 1;
        const unsigned live = __ballot_sync(0xffffffffu, rows > 0);
        const int rincl = lane_prefix(rows);
        unsigned slot = 0u;
        if (lane == 31 && live) slot = atomicAdd(&sm.made, ((unsigned)rincl << 9) | (unsigned)__popc(live));
        slot = __shfl_sync(0xffffffffu, slot, 31);
        if (rows > 0) {
            const int j = (int)(slot & 511u) + __popc(live & ((1u << lane) - 1u)), start = (int)(slot >> 9) + rincl - rows;
            sm.unit[j] = (unsigned)box | ((unsigned)t << 20) | ((unsigned)sub << 26);
            sm.fr[j] = fr;
            if (!CULL) sm.bk[j] = bk;
            sm.start[j] = (unsigned short)start;
            const int g = (start + 31) >> 5;                    // at most one multiple of 32 in its rows
            if (32 * g < start + rows) sm.first[g] = (unsigned char)j;
        }
        if (COUNT && lane == 0) n_unit += (unsigned long long)__popc(live);
        __syncthreads();
        const int n_units = (int)(sm.made & 511u), n_rows = (int)(sm.made >> 9);
        // warps take 32 rows at a time from a shared counter, so an expensive group does not
        // hold the warps that would otherwise wait for its warp at the next barrier (the
        // next group is claimed before this one is worked, hiding the atomic's latency)
        int rb = warp * 32, qn = 0;
        while (rb < n_rows) {
            int nx = 0;
            if (lane == 0) nx = atomicAdd(&sm.next_row, 32);
            raster_rows<COUNT, CULL>(sm, rb, n_rows, n_units, kmax, inv_dx, qn, n_cell, n_test, n_span);
            rb = __shfl_sync(0xffffffffu, nx, 0);
        }
        // the queue's last cells, before the batch's triangles are replaced
        if (qn > 0) drain_cells<COUNT, CULL>(sm, sm.queue[warp], qn, kmax, n_cell, n_test);
        __syncwarp();
    }
    __syncthreads();
}

__device__ __forceinline__ void flush_raster_counts(unsigned long long* stats, unsigned long long n_cell,
                                                    unsigned long long n_test,
                                                    unsigned long long n_unit,
                                                    unsigned long long n_span) {
    for (int o = 16; o > 0; o >>= 1) {
        n_cell += __shfl_down_sync(0xffffffffu, n_cell, o);
        n_test += __shfl_down_sync(0xffffffffu, n_test, o);
        n_unit += __shfl_down_sync(0xffffffffu, n_unit, o);
        n_span += __shfl_down_sync(0xffffffffu, n_span, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&stats[0], n_unit);
        atomicAdd(&stats[1], n_span);
        atomicAdd(&stats[2], n_cell);
        atomicAdd(&stats[3], n_test);
    }
}

// One CTA per 32 x 32-cell tile, every block of the chunk in order; the gross /
// continuous state of the tile's cells stays in shared memory between blocks.  It needs no
// memory per block, so the raster in fixed scratch (launch_raster_ground_in) takes it, and
// the per-step raster of a large grid; k_raster_items is faster on the rest (below).
template <bool CULL, int CTAS>
__global__ void __launch_bounds__(kRasterThreads, CTAS)
k_raster(RasterArgs ra) {
    __shared__ TileSmem sm;
    __shared__ RunState s_st[kTile * kTile];       // gross / run / best of the tile's cells
    unsigned long long n_cell = 0, n_test = 0, n_unit = 0, n_span = 0;
    const TileGeom& g = ra.g;
    const int tile = ra.order ? ra.order[blockIdx.x] : (int)blockIdx.x;
    const int tx = tile % g.tiles_x, ty = tile / g.tiles_x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = warp * 4;
    float tox, toy;
    tile_setup(sm, g, tx, ty, &tox, &toy);
    const int ix = tx * kTile + lane;
    // each thread owns the cells (row0 + q, lane), q < 4, and alone touches their state
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int iy = ty * kTile + row0 + q;
        const long long o = (long long)iy * g.nx + ix;
        RunState st{0, 0, 0};
        if (ix < g.nx && iy < g.ny && ra.load_state) {
            st.gross = ra.out.gross[o];
            st.best = ra.best[o];
            st.run = ra.out.run[o];
        }
        s_st[(row0 + q) * kTile + lane] = st;
    }
    const int n_tiles = g.tiles_x * g.tiles_y;
    const float inv_dx = 1.f / g.dx;
    for (int bl = 0; bl < ra.nbc; ++bl) {
        const BlockConst* bcp = &ra.sun.blocks[ra.b0 + bl];
        const size_t bin = (size_t)bl * n_tiles + tile;
        const unsigned cnt = ra.counts[bin];
        const int* bins = ra.bins + ra.offsets[bin];
        const float4* tris = ra.sc.tris;
        const int T = ra.sc.T;
        auto fetch = [bins, tris, T](int i, int v, float4* out) {
            *out = __ldg(&tris[3 * SA_CHK(bins[i], T, sa::CK_RASTER_BIN) + v]);
            (void)T;
            return true;
        };
        raster_block<false, CULL>(sm, fetch, (int)cnt, ra.sun.steps, bcp->j0, bcp->K, tox, toy,
                                  inv_dx, ra.run, n_cell, n_test, n_unit, n_span);
        const int K = bcp->K, new_day = bcp->new_day;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int cell = (row0 + q) * kTile + lane;
            const unsigned long long m = sm.mask(cell);
            sm.set_mask(cell, 0ull);
            RunState st = s_st[cell];
            stitch(st, m, K, new_day);
            s_st[cell] = st;
            const int iy = ty * kTile + row0 + q;
            if (ra.out.masks && ix < g.nx && iy < g.ny)
                ra.out.masks[(size_t)bcp->mask_block * ra.R + (long long)iy * g.nx + ix] |= m << bcp->mask_bit;
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int iy = ty * kTile + row0 + q;
        if (ix >= g.nx || iy >= g.ny) continue;
        const long long o = (long long)iy * g.nx + ix;
        const RunState st = s_st[(row0 + q) * kTile + lane];
        ra.out.gross[o] = st.gross;
        ra.best[o] = st.best;
        ra.out.run[o] = st.run;
        if (ra.final_chunk && ra.out.minutes) ra.out.minutes[o] = (float)st.gross * ra.out.step_minutes;
    }
}

// One CTA per item, (block, tile) and one of `parts` consecutive pieces of the block's steps:
// the items of a small grid's long interval fill the chip where its tiles alone cannot.
// Each item leaves its cells' run summaries (run_summary, 4 bytes per block and cell), which
// k_items_fold stitches in time order, and its step masks where they are asked for.
// Against one CTA per tile with the blocks in series (k_raster), same inputs and bits:
// 231 x 187 cells, 92 days (56 tiles, 828 blocks) 54.1 -> 4.54 ms; 64^2 cells, one day
// 216 -> 57 us; 512^2 604 -> 286 us; 2048^2 2.43 -> 2.21 ms (heavy items start first,
// 23.9 KB of shared memory instead of 35.9); 1024^2 in December 27.5 -> 25.2 ms.
template <bool COUNT, bool CULL>
__global__ void __launch_bounds__(kRasterThreads, SA_RASTER_CTAS)
k_raster_items(RasterArgs ra) {
    __shared__ TileSmem sm;
    unsigned long long n_cell = 0, n_test = 0, n_unit = 0, n_span = 0;
    const TileGeom& g = ra.g;
    const int n_tiles = g.tiles_x * g.tiles_y;
    const int item = ra.order ? ra.order[blockIdx.x] : (int)blockIdx.x;
    const int bl = item / n_tiles, tile = item - bl * n_tiles;
    const int tx = tile % g.tiles_x, ty = tile / g.tiles_x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = blockIdx.y;
    const BlockConst* bcp = &ra.sun.blocks[ra.b0 + bl];
    const int k0 = part * bcp->K / ra.parts, K = (part + 1) * bcp->K / ra.parts - k0;
    const unsigned cnt = ra.counts[item];
    const int ix = tx * kTile + lane, row0 = warp * 4;
    if (cnt > 0 && K > 0) {
        float tox, toy;
        tile_setup(sm, g, tx, ty, &tox, &toy);
        const int* bins = ra.bins + (ra.offsets ? (size_t)ra.offsets[item] : (size_t)item * ra.cap);
        const float4* tris = ra.sc.tris;
        const int T = ra.sc.T;
        auto fetch = [bins, tris, T](int i, int v, float4* out) {
            *out = __ldg(&tris[3 * SA_CHK(bins[i], T, sa::CK_RASTER_BIN) + v]);
            (void)T;
            return true;
        };
        raster_block<COUNT, CULL>(sm, fetch, (int)cnt, ra.sun.steps, bcp->j0 + k0, K, tox, toy, 1.f / g.dx,
                                  ra.run, n_cell, n_test, n_unit, n_span);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int iy = ty * kTile + row0 + q;
        if (ix >= g.nx || iy >= g.ny) continue;
        const unsigned long long m = (cnt > 0 && K > 0) ? sm.mask((row0 + q) * kTile + lane) : 0ull;
        const size_t cell = (size_t)iy * g.nx + ix;
        if (ra.summary) ra.summary[((size_t)bl * ra.parts + part) * ra.R + cell] = run_summary(m, K);
        // pieces and one-step blocks share a mask word
        if (ra.out.masks && m)
            atomicOr(reinterpret_cast<unsigned long long*>(&ra.out.masks[(size_t)bcp->mask_block * ra.R + cell]),
                     m << (bcp->mask_bit + k0));
    }
    if (COUNT) flush_raster_counts(ra.out.stats, n_cell, n_test, n_unit, n_span);
}

constexpr int kFoldThreads = 128;
constexpr int kFoldTile = 1024;      // steps-and-day codes staged in shared memory at a time
constexpr int kFoldAhead = 8;        // summaries a thread loads ahead of their use

// Stitches the chunk's run summaries, in time order, into each cell's gross / continuous
// state (as stitch does with the masks themselves), VEC cells per thread.  Bound by memory
// on a large grid (4 bytes in per block, 12 out; four cells per thread: 16-byte loads, 2048^2
// cells x 9 blocks 79 -> 37 us); a small one keeps a cell per thread for the parallelism.
template <int VEC>
__global__ void __launch_bounds__(kFoldThreads)
k_items_fold(const unsigned* __restrict__ summary, long long R, const BlockConst* __restrict__ blocks,
             int nbc, int parts, DevOut out, int* __restrict__ best, int load_state, int final_chunk) {
    __shared__ int s_code[kFoldTile];
    const long long r = ((long long)blockIdx.x * kFoldThreads + threadIdx.x) * VEC;
    const int n_all = nbc * parts;
    RunState st[VEC];
#pragma unroll
    for (int c = 0; c < VEC; ++c) {
        st[c] = RunState{0, 0, 0};
        if (r < R && load_state) st[c] = RunState{out.gross[r + c], out.run[r + c], best[r + c]};
    }
    for (int p0 = 0; p0 < n_all; p0 += kFoldTile) {
        const int n = min(kFoldTile, n_all - p0);
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kFoldThreads) {
            const int b = (p0 + i) / parts, q = (p0 + i) - b * parts;
            const int K = blocks[b].K;
            s_code[i] = ((q + 1) * K / parts - q * K / parts) | (q == 0 && blocks[b].new_day ? 128 : 0);
        }
        __syncthreads();
        if (r >= R) continue;
        for (int i = 0; i < n; i += kFoldAhead) {
            unsigned v[kFoldAhead][VEC];
#pragma unroll
            for (int q = 0; q < kFoldAhead; ++q) {
                const unsigned* at = summary + (size_t)(p0 + i + q) * R + r;
                if (i + q >= n) {
#pragma unroll
                    for (int c = 0; c < VEC; ++c) v[q][c] = 0u;
                } else if (VEC == 4) {
                    const uint4 x = __ldcs(reinterpret_cast<const uint4*>(at));
                    v[q][0] = x.x; v[q][VEC > 1 ? 1 : 0] = x.y; v[q][VEC > 2 ? 2 : 0] = x.z; v[q][VEC > 3 ? 3 : 0] = x.w;
                } else {
                    v[q][0] = __ldcs(at);
                }
            }
#pragma unroll
            for (int q = 0; q < kFoldAhead; ++q) {
                if (i + q >= n) break;
                const int code = s_code[i + q], K = code & 127;
#pragma unroll
                for (int c = 0; c < VEC; ++c) {
                    RunState& s = st[c];
                    const unsigned x = v[q][c];
                    if (code & 128) s.run = 0;
                    const int pop = (int)(x & 255u);
                    s.gross += pop;
                    if (pop == K) {
                        s.run += K;
                        s.best = max(s.best, s.run);
                    } else {
                        s.best = max(s.best, max(s.run + (int)((x >> 8) & 255u), (int)(x >> 24)));
                        s.run = (int)((x >> 16) & 255u);
                    }
                }
            }
        }
    }
    if (r >= R) return;
    const float dt = out.step_minutes;
    if (VEC == 4) {
        const RunState &a = st[0], &b = st[VEC > 1 ? 1 : 0], &c = st[VEC > 2 ? 2 : 0], &d = st[VEC > 3 ? 3 : 0];
        *reinterpret_cast<int4*>(out.gross + r) = make_int4(a.gross, b.gross, c.gross, d.gross);
        *reinterpret_cast<int4*>(best + r) = make_int4(a.best, b.best, c.best, d.best);
        if (!final_chunk) *reinterpret_cast<int4*>(out.run + r) = make_int4(a.run, b.run, c.run, d.run);
        else if (out.minutes)
            *reinterpret_cast<float4*>(out.minutes + r) =
                make_float4((float)a.gross * dt, (float)b.gross * dt, (float)c.gross * dt, (float)d.gross * dt);
    } else {
        out.gross[r] = st[0].gross;
        best[r] = st[0].best;
        if (!final_chunk) out.run[r] = st[0].run;
        else if (out.minutes) out.minutes[r] = (float)st[0].gross * dt;
    }
}

// --------------------------------------------------------------- batched scenarios
// A persistent launch over work items (interval, variant, tile of the variant's region).
// Each item rasters every block of its interval for one tile: the base city's binned
// triangles minus the variant's removed buildings, plus the variant's tower triangles.
// It writes the counts of the tile's cells inside the region and, where the base counts
// are given, the impact (variant minus base).
template <bool COUNT, bool CULL>
__global__ void __launch_bounds__(kRasterThreads, kStateCtas)
k_batch(BatchArgs ba) {
    __shared__ TileSmem sm;
    __shared__ RunState s_st[kTile * kTile];       // gross / run / best of the tile's cells
    __shared__ int s_item;
    unsigned long long n_cell = 0, n_test = 0, n_unit = 0, n_span = 0;
    const TileGeom& g = ba.g;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = warp * 4;
    const float inv_dx = 1.f / g.dx;
    const int n_tiles = g.tiles_x * g.tiles_y;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (int)atomicAdd(ba.counter, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= ba.n_items) break;
        const int4 it = ba.items[item];                  // interval, variant, tile, affected
        const BatchInterval& iv = ba.intervals[it.x];
        const BatchVariant& var = ba.variants[it.y];
        const int tile = it.z;
        const int tx = tile % g.tiles_x, ty = tile / g.tiles_x;
        if (!it.w) {
            // neither a removed building's nor a tower's shadow can reach this tile during
            // the interval: the variant's counts are the base counts
            for (int c = threadIdx.x; c < kTile * kTile; c += kRasterThreads) {
                const int ix = tx * kTile + (c & (kTile - 1)), iy = ty * kTile + c / kTile;
                const int lx = ix - var.ix0, ly = iy - var.iy0;
                if (ix >= g.nx || iy >= g.ny || lx < 0 || ly < 0 || lx >= var.nx || ly >= var.ny) continue;
                const long long o = iv.out_base + var.out_off + (long long)ly * var.nx + lx;
                ba.counts_out[o] = iv.base_counts[(long long)iy * g.nx + ix];
                if (ba.impact_out) ba.impact_out[o] = 0;
            }
            continue;
        }
        float tox, toy;
        tile_setup(sm, g, tx, ty, &tox, &toy);
#pragma unroll
        for (int q = 0; q < 4; ++q) s_st[(row0 + q) * kTile + lane] = RunState{0, 0, 0};
        const int* rem = ba.removed + var.rem_off;
        const int n_rem = var.n_rem;
        const float4* towers = ba.tower_tris + 3ll * var.tower_off;
        const int n_tow = var.n_tower;
        for (int bl = 0; bl < iv.n_blocks; ++bl) {
            const BlockConst& bc = iv.blocks[bl];
            const unsigned off = iv.offsets[(size_t)bl * n_tiles + tile];
            const int cnt = (int)iv.counts[(size_t)bl * n_tiles + tile];
            const int* bins = iv.bins + off;
            const float4* tris = ba.base_tris;
            auto fetch = [=](int i, int v, float4* out) {
                if (i >= cnt) {
                    *out = __ldg(&towers[3 * (i - cnt) + v]);
                    return true;
                }
                const float4 x = __ldg(&tris[3 * bins[i] + v]);
                *out = x;
                if (v != 0) return true;
                const int bid = __float_as_int(__ldg(&tris[3 * bins[i]]).w);
                for (int q = 0; q < n_rem; ++q)
                    if (rem[q] == bid) return false;
                return true;
            };
            raster_block<COUNT, CULL>(sm, fetch, cnt + n_tow, iv.steps, bc.j0, bc.K, tox, toy,
                                      inv_dx, ba.run, n_cell, n_test, n_unit, n_span);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int cell = (row0 + q) * kTile + lane;
                const unsigned long long m = sm.mask(cell);
                sm.set_mask(cell, 0ull);
                RunState st = s_st[cell];
                stitch(st, m, bc.K, bc.new_day);
                s_st[cell] = st;
            }
        }
        const int ix = tx * kTile + lane;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int iy = ty * kTile + row0 + q;
            const int lx = ix - var.ix0, ly = iy - var.iy0;
            if (ix >= g.nx || iy >= g.ny || lx < 0 || ly < 0 || lx >= var.nx || ly >= var.ny) continue;
            const long long o = iv.out_base + var.out_off + (long long)ly * var.nx + lx;
            const int gross = s_st[(row0 + q) * kTile + lane].gross;
            ba.counts_out[o] = gross;
            if (ba.impact_out && iv.base_counts)
                ba.impact_out[o] = gross - iv.base_counts[(long long)iy * g.nx + ix];
        }
    }
    if (COUNT) flush_raster_counts(ba.stats, n_cell, n_test, n_unit, n_span);
}

// Batched scenarios from the base city's step masks.  A variant's mask of a tile and block
// differs from the base mask only where its removed buildings or its towers cast shadow, and
// every decision is the OR of the same exact tests, so it is put together from them:
//   - a block no changed box's swept shadow reaches keeps the base counts;
//   - bits no removed triangle covers stay as they are; the others are decided again by the
//     base bins without the removed buildings, everything else counting as filled so that
//     the raster passes over it;
//   - the towers' triangles are ORed in on top.
// An item is one (interval, variant, tile, block) that k_batch_pick found changed; its change
// of the gross counts is added to the outputs, which k_batch_base has set to the base
// counts.  Against k_batch (every block of an affected tile rastered whole): 16 variants x 2
// intervals x 3 days over 1024^2 cells 18.2 -> 3.05 ms (bound by issue, in the towers' rasters
// and in the units that set up the few triangles of an item).

// Triangles of k_batch_delta's rasters: item i is tris[map[list[i]]] (either index may be
// absent); one of the removed buildings' triangles is skipped.
struct DeltaFetch {
    const float4* tris;
    const int* map;
    const int* list;
    const int* rem;
    int n_rem;
    __device__ __forceinline__ bool operator()(int i, int v, float4* out) const {
        int t = list ? list[i] : i;
        if (map) t = map[t];
        const float4 x = __ldg(&tris[3ll * t + v]);
        *out = x;
        if (v != 0 || n_rem == 0) return true;
        const int bid = __float_as_int(x.w);
        for (int q = 0; q < n_rem; ++q)
            if (rem[q] == bid) return false;
        return true;
    }
};

// One copy of the unrolled step tests for the three rasters of a block.
template <bool COUNT, bool CULL>
__device__ __noinline__ void raster_block_call(TileSmem& sm, const DeltaFetch& fetch, int n, const StepConst* steps,
                                               const BlockConst& bc, float tox, float toy, float inv_dx, int kSub,
                                               bool prefilled, unsigned long long* cnt) {
    raster_block<COUNT, CULL>(sm, fetch, n, steps, bc.j0, bc.K, tox, toy, inv_dx, kSub, cnt[0], cnt[1], cnt[2], cnt[3],
                              prefilled);
}

// Can the shadow of the box [x0, x1] x [y0, y1] x [z0, z1], swept over the block, reach tile
// (tx, ty)?  A point f at height z shadows f - z u, u in the block's slope box, so some
// height must have z u within the box's plan minus the tile: four half-lines of z.  One
// cell of margin on every side absorbs rounding, as in swept_tiles, and a millimetre in z
// the quotients'.  (The bounding box of the sweep takes in several times the tiles of a
// high tower's shadow that falls across the grid's axes: 16 variants x 2 intervals x 3 days
// 3.37 -> 3.05 ms with this test for the items and their triangles.)
__device__ __forceinline__ bool box_reaches(float x0, float x1, float y0, float y1, float z0, float z1,
                                            const BlockConst& bc, const TileGeom& g, int tx, int ty) {
    const float side = kTile * g.dx, X = fmaf((float)tx, side, g.x0), Y = fmaf((float)ty, side, g.y0);
    float lo = fmaxf(z0, 0.f), hi = fmaxf(z1, 0.f);
    auto half_line = [&](float u, float d) {                       // z u <= d
        if (u > 0.f) hi = fminf(hi, __fdividef(d, u));
        else if (u < 0.f) lo = fmaxf(lo, __fdividef(d, u));
        else if (d < 0.f) hi = -3.4e38f;
    };
    half_line(bc.uxlo, x1 - (X - g.dx));
    half_line(-bc.uxhi, X + side + g.dx - x0);
    half_line(bc.uylo, y1 - (Y - g.dx));
    half_line(-bc.uyhi, Y + side + g.dx - y0);
    return lo <= fmaf(fabsf(hi), 1e-5f, hi + 1e-3f);
}

template <bool COUNT, bool CULL>
__global__ void __launch_bounds__(kRasterThreads, SA_RASTER_CTAS)
k_batch_delta(BatchArgs ba, BatchDelta bd) {
    __shared__ TileSmem sm;
    __shared__ int s_list[kChangeList];
    __shared__ int s_item, s_n;
    unsigned long long cnt[4] = {0ull, 0ull, 0ull, 0ull};       // cell set-ups, step tests, units, spans
    const TileGeom& g = ba.g;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = warp * 4;
    const float inv_dx = 1.f / g.dx;
    const int n_tiles = g.tiles_x * g.tiles_y;
    while (true) {
        __syncthreads();
        if (tid == 0) s_item = (int)atomicAdd(ba.counter, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= ba.n_items) break;
        // interval, variant, tile, block * 4 + (removed buildings reach it) * 2 + (towers do)
        const int4 it = ba.items[bd.order[item]];
        const BatchInterval& iv = ba.intervals[it.x];
        const BatchVariant& var = ba.variants[it.y];
        const int tile = it.z, bl = it.w >> 2;
        const bool remv = it.w & 2, tow = it.w & 1;
        const int tx = tile % g.tiles_x, ty = tile / g.tiles_x;
        const int ix = tx * kTile + lane;
        const float4* towers = ba.tower_tris + 3ll * var.tower_off;
        const int* rem = ba.removed + var.rem_off;
        const int n_rem = var.n_rem;
        const int* rem_tri = bd.rem_tri + var.remtri_off;
        const float4* tris = ba.base_tris;
        const BlockConst& bc = iv.blocks[bl];
        float tox, toy;
        tile_setup(sm, g, tx, ty, &tox, &toy);
        unsigned long long base[4], now[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int iy = ty * kTile + row0 + q;
            base[q] = (ix < g.nx && iy < g.ny)
                          ? __ldg(&bd.masks[(size_t)bl * bd.R + iv.mask_off + (size_t)iy * g.nx + ix]) : 0ull;
            now[q] = base[q];
            if (remv) sm.set_mask((row0 + q) * kTile + lane, 0ull);
        }
        // rasters the changed triangles pick(i) < n that reach the tile, kChangeList at a time
        auto raster_changed = [&](DeltaFetch f, int n, bool prefilled) {
            for (int i0 = 0; i0 < n; i0 += kChangeList) {
                __syncthreads();
                if (tid == 0) s_n = 0;
                __syncthreads();
                const int i = i0 + tid;
                bool pick = false;
                if (i < n) {
                    const float4* t = f.tris + 3ll * (f.map ? f.map[i] : i);
                    const float4 a = __ldg(t), b = __ldg(t + 1), c = __ldg(t + 2);
                    pick = tri_above_ground(a, b, c) &&
                           box_reaches(fminf(a.x, fminf(b.x, c.x)), fmaxf(a.x, fmaxf(b.x, c.x)),
                                       fminf(a.y, fminf(b.y, c.y)), fmaxf(a.y, fmaxf(b.y, c.y)),
                                       fminf(a.z, fminf(b.z, c.z)), fmaxf(a.z, fmaxf(b.z, c.z)), bc, g, tx, ty);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, pick);
                int at = 0;
                if (lane == 0 && bal) at = atomicAdd(&s_n, __popc(bal));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (pick) s_list[at + __popc(bal & ((1u << lane) - 1u))] = i;
                __syncthreads();
                const int m = s_n;
                f.list = s_list;
                if (m > 0)
                    raster_block_call<COUNT, CULL>(sm, f, m, iv.steps, bc, tox, toy, inv_dx, ba.run, prefilled, cnt);
            }
        };
        if (remv) {
            raster_changed(DeltaFetch{tris, rem_tri, nullptr, nullptr, 0}, var.n_remtri, false);
            __syncthreads();
            bool any = false;
            unsigned long long open[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int cell = (row0 + q) * kTile + lane;
                open[q] = base[q] & sm.mask(cell);         // bits to decide again
                now[q] = base[q] & ~open[q];
                any |= open[q] != 0ull;
                sm.set_mask(cell, ~open[q]);
            }
            if (__syncthreads_or(any)) {
                const size_t bin = (size_t)bl * n_tiles + tile;
                raster_block_call<COUNT, CULL>(sm, DeltaFetch{tris, iv.bins + iv.offsets[bin], nullptr, rem, n_rem},
                                               (int)iv.counts[bin], iv.steps, bc, tox, toy, inv_dx, ba.run, true, cnt);
                __syncthreads();
#pragma unroll
                for (int q = 0; q < 4; ++q) now[q] |= sm.mask((row0 + q) * kTile + lane) & open[q];
            }
        }
        if (tow) {
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.set_mask((row0 + q) * kTile + lane, now[q]);
            raster_changed(DeltaFetch{towers, nullptr, nullptr, nullptr, 0}, var.n_tower, true);
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) now[q] = sm.mask((row0 + q) * kTile + lane);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int iy = ty * kTile + row0 + q;
            const int lx = ix - var.ix0, ly = iy - var.iy0;
            const int delta = __popcll(now[q]) - __popcll(base[q]);
            if (delta == 0 || ix >= g.nx || iy >= g.ny || lx < 0 || ly < 0 || lx >= var.nx || ly >= var.ny) continue;
            const long long o = iv.out_base + var.out_off + (long long)ly * var.nx + lx;
            atomicAdd(&ba.counts_out[o], delta);
            if (ba.impact_out) atomicAdd(&ba.impact_out[o], delta);
        }
    }
    if (COUNT) flush_raster_counts(ba.stats, cnt[0], cnt[1], cnt[2], cnt[3]);
}

// The work items of k_batch_delta: for every affected (interval, variant, tile) and block,
// whether a changed box's shadow, swept over the block, can reach the tile.  Counts them
// (items null; a count, unlike the items that are then made of it, may pass 32 bits), or
// appends them with their weights: the base triangles to raster again, and the boxes.
__global__ void k_batch_pick(TileGeom g, const BatchInterval* __restrict__ intervals,
                             const BatchVariant* __restrict__ variants, const float4* __restrict__ boxes,
                             const int4* __restrict__ tiles, long long n, int max_blocks,
                             unsigned long long* __restrict__ total, int4* __restrict__ items,
                             unsigned* __restrict__ weights) {
    unsigned long long found = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n * max_blocks;
         i += (long long)gridDim.x * blockDim.x) {
        const int4 t = tiles[i / max_blocks];
        const int bl = (int)(i % max_blocks);
        const BatchInterval& iv = intervals[t.x];
        if (bl >= iv.n_blocks) continue;
        const BatchVariant& var = variants[t.y];
        const int tx = t.z % g.tiles_x, ty = t.z / g.tiles_x;
        bool remv = false;
        unsigned n_rem = 0, n_tow = 0;
        for (int q = 0; q < var.n_box; ++q) {
            const float4 lo = __ldg(&boxes[2 * (var.box_off + q)]), hi = __ldg(&boxes[2 * (var.box_off + q) + 1]);
            if (!box_reaches(lo.x, hi.x, lo.y, hi.y, 0.f, hi.z, iv.blocks[bl], g, tx, ty)) continue;
            if (lo.w != 0.f) { remv = true; ++n_rem; }
            else ++n_tow;
        }
        if (!n_rem && !n_tow) continue;
        if (!items) {
            ++found;
            continue;
        }
        const unsigned long long at = atomicAdd(total, 1ull);
        items[at] = make_int4(t.x, t.y, t.z, bl * 4 + (remv ? 2 : 0) + (n_tow ? 1 : 0));
        weights[at] = 1u + 4u * n_tow + (remv ? 16u * n_rem + iv.counts[(size_t)bl * g.tiles_x * g.tiles_y + t.z] : 0u);
    }
    if (found) atomicAdd(total, found);
}

// The base counts, and no impact, for every cell of every region.
__global__ void k_batch_base(BatchArgs ba, int V, int I) {
    for (int iv = blockIdx.y; iv < V * I; iv += gridDim.y) {
        const BatchInterval& bi = ba.intervals[iv / V];
        const BatchVariant& var = ba.variants[iv % V];
        const long long n = (long long)var.nx * var.ny, o0 = bi.out_base + var.out_off;
        for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
            const long long ly = c / var.nx, lx = c - ly * var.nx;
            ba.counts_out[o0 + c] = bi.base_counts[(var.iy0 + ly) * ba.g.nx + var.ix0 + lx];
            if (ba.impact_out) ba.impact_out[o0 + c] = 0;
        }
    }
}

// Launch order of the tiles when a CTA takes all blocks of a tile: as launch_work_order, by
// the triangles binned to the tile over the chunk's blocks.
__global__ void k_tile_sums(const unsigned* __restrict__ counts, int nbc, int n_tiles, unsigned* __restrict__ sums) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tiles) return;
    unsigned c = 0;
    for (int b = 0; b < nbc; ++b) c += counts[(size_t)b * n_tiles + t];
    sums[t] = c;
}

// A launch of more tiles than 4 CTAs per SM hold takes the build for kStateCtas
// resident CTAs per SM (fewer registers, more warps to hide latency); a smaller one, all of
// whose tiles are resident at once anyway, takes the build for 4 (more registers, no
// spills).
void launch_k_raster(const RasterArgs& ra, int n_tiles, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 0;
    if (n_tiles > 4 * sms) {
        if (ra.cull) k_raster<true, kStateCtas><<<n_tiles, kRasterThreads, 0, st>>>(ra);
        else k_raster<false, kStateCtas><<<n_tiles, kRasterThreads, 0, st>>>(ra);
    } else {
        if (ra.cull) k_raster<true, 4><<<n_tiles, kRasterThreads, 0, st>>>(ra);
        else k_raster<false, 4><<<n_tiles, kRasterThreads, 0, st>>>(ra);
    }
}

void launch_k_items(const RasterArgs& ra, int n_items, bool stats, cudaStream_t st) {
    const dim3 grid((unsigned)n_items, (unsigned)ra.parts);
    if (ra.cull) {
        if (stats) k_raster_items<true, true><<<grid, kRasterThreads, 0, st>>>(ra);
        else k_raster_items<false, true><<<grid, kRasterThreads, 0, st>>>(ra);
    } else {
        if (stats) k_raster_items<true, false><<<grid, kRasterThreads, 0, st>>>(ra);
        else k_raster_items<false, false><<<grid, kRasterThreads, 0, st>>>(ra);
    }
}

}  // namespace

// Four cells per thread from a million cells up, where every row of summaries and every
// output starts on 16 bytes.
void launch_fold(const unsigned* summary, long long R, const BlockConst* blocks, int nbc, int parts,
                 const DevOut& out, int* best, int load_state, int final_chunk, cudaStream_t st) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(out.gross) | reinterpret_cast<uintptr_t>(best) |
                         reinterpret_cast<uintptr_t>(out.run) | reinterpret_cast<uintptr_t>(out.minutes) |
                         reinterpret_cast<uintptr_t>(summary);
    if (R >= (1 << 20) && R % 4 == 0 && (at & 15) == 0) {
        const unsigned g = (unsigned)((R / 4 + kFoldThreads - 1) / kFoldThreads);
        k_items_fold<4><<<g, kFoldThreads, 0, st>>>(summary, R, blocks, nbc, parts, out, best, load_state, final_chunk);
    } else {
        const unsigned g = (unsigned)((R + kFoldThreads - 1) / kFoldThreads);
        k_items_fold<1><<<g, kFoldThreads, 0, st>>>(summary, R, blocks, nbc, parts, out, best, load_state, final_chunk);
    }
}

// Pieces each block's steps are cut into: one from 1,824 items (two waves of
// SA_RASTER_CTAS CTAs on 152 SMs) up, where the items alone fill the chip and a piece only
// repeats the staging (512^2 cells, 9 blocks, 2,304 items: 0.29 ms in one piece, 0.33 in
// two), more below it, up to 4 (64^2 cells, 5 blocks, 20 items: 84 us in one, 57 us in four,
// 54 us in six; 300^2 cells, 900 items: 255 us in one, 232 us in two, 226 us in three).
static int raster_parts(int n_tiles, int n_blocks) {
    const long long items = (long long)n_tiles * n_blocks, fill = 152ll * SA_RASTER_CTAS * 2;
    return (int)std::max(1ll, std::min(4ll, (fill + items - 1) / items));
}

static TileGeom tile_geom(const DevRecv& rc) {
    TileGeom g;
    g.x0 = rc.x0; g.y0 = rc.y0; g.dx = rc.dx; g.nx = rc.nx; g.ny = rc.ny;
    g.tiles_x = (rc.nx + kTile - 1) / kTile;
    g.tiles_y = (rc.ny + kTile - 1) / kTile;
    return g;
}

// Runs every block of `sun` through the accrual raster, in chunks of blocks whose bins
// fit a bounded scratch budget.  out.run must be scratch [R]; out.continuous may be NULL,
// and out.gross too when only the masks are wanted.  With `summaries`
// ([n_blocks][R]) the run summary of every block goes there and out is not touched.
static cudaError_t raster_ground(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                                 const DevOut& out, unsigned* summaries, cudaStream_t st) {
    const TileGeom g = tile_geom(rc);
    const int n_tiles = g.tiles_x * g.tiles_y;
    const long long R = (long long)rc.nx * rc.ny;
    if (R == 0 || sun.n_blocks == 0) return cudaSuccess;
    // One-step blocks (the per-step raster) of a grid whose tiles fill the chip go by tile: a
    // summary per step is as much memory as the raster's own work (2048^2 cells, 481 steps:
    // 30.9 ms by tile, 32.3 by item; 300 x 200 cells, 70 tiles, 241 steps: 4.07 and 0.50 ms).
    bool by_tile = !summaries && out.gross && !out.stats && n_tiles >= 4 * 152 &&
                   sun.S < 8ll * sun.n_blocks;
    int parts = summaries || by_tile ? 1 : raster_parts(n_tiles, sun.n_blocks);
    bool fold = !summaries && out.gross && !by_tile;
    cudaError_t e = cudaSuccess;
    // blocks per chunk: 64, and more where a small grid's counters, bins (every triangle in
    // every tile at the most: the sums stay below 2^31) and run summaries (1 GiB) allow it
    auto chunk_blocks = [&](int T) {
        long long chunk = by_tile ? 64ll : std::max(64ll, std::min((1ll << 20) / n_tiles, (1ll << 31) / ((long long)std::max(T, 1) * n_tiles)));
        if (fold) chunk = std::min(chunk, std::max(1ll, (1ll << 30) / (4ll * parts * R)));
        return (int)std::min<long long>(sun.n_blocks, chunk);
    };
    // a mesh so small that every bin may hold all of it needs no counting pass, no scan and
    // no read-back of the bins' size
    auto is_direct = [&](int chunk, int T) {
        return !by_tile && T > 0 && (double)chunk * n_tiles * T <= (double)(4 << 20);
    };
    // Many blocks or a large mesh: the triangles that reach the grid at all are listed first
    // (k_reach and a read-back, 20 us), and where they are the lesser part, only they go
    // on.  4M (triangle, block) pairs are about as much in the two passes of k_bin.
    int T = sc.T, chunk = chunk_blocks(T);
    int* list = nullptr;
    unsigned* d_reach = nullptr;
    if (!is_direct(chunk, T) && (long long)T * sun.n_blocks >= (4ll << 20)) {
        unsigned n = 0;
        e = sa::scratch_alloc(&d_reach, sizeof(unsigned), st);
        if (e == cudaSuccess) e = sa::scratch_alloc(&list, sizeof(int) * (size_t)T, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(d_reach, 0, sizeof(unsigned), st);
        if (e == cudaSuccess) {
            KernelTimer kt(KT_RASTER_BIN, st);
            k_reach<<<(unsigned)std::min(152 * 8, (T + kReachThreads - 1) / kReachThreads), kReachThreads, 0, st>>>(
                sc, sun.blocks, sun.n_blocks, g, d_reach, list);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&n, d_reach, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess && n <= (unsigned)T / 2) {
            T = (int)n;
            chunk = chunk_blocks(T);
        } else if (list) {
            cudaFreeAsync(list, st);
            list = nullptr;
        }
    }
    unsigned* summary = summaries;
    if (e == cudaSuccess && fold) {
        // without memory for the summaries of one block, by tile, which needs none
        e = sa::scratch_alloc_blocks(&summary, sizeof(unsigned) * (size_t)parts * (size_t)R, &chunk, st);
        if (e == cudaErrorMemoryAllocation && !out.stats) {
            e = cudaSuccess;
            by_tile = true;
            fold = false;
            parts = 1;
            chunk = chunk_blocks(T);
        }
    }
    const size_t nc = (size_t)chunk * n_tiles;
    const bool direct = is_direct(chunk, T);
    // one block of words: counts | cursor (zeroed together) | offsets | order | total | buckets
    unsigned* words = nullptr;
    int* bins = nullptr;
    int* best = out.continuous;
    int* best_scratch = nullptr;
    size_t bins_cap = 0;
    if (e == cudaSuccess) e = sa::scratch_alloc(&words, sizeof(unsigned) * (4 * nc + 1 + kOrderBuckets), st);
    unsigned *counts = words, *cursor = words + nc, *offsets = words + 2 * nc, *d_total = words + 4 * nc,
             *hist = d_total + 1;
    int* order = reinterpret_cast<int*>(words + 3 * nc);
    if (e == cudaSuccess && !best && out.gross) {
        e = sa::scratch_alloc(&best_scratch, sizeof(int) * (size_t)R, st);
        best = best_scratch;
    }
    if (e == cudaSuccess && direct) {
        bins_cap = nc * (size_t)T;
        e = sa::scratch_alloc(&bins, sizeof(int) * bins_cap, st);
    }
    if (e == cudaSuccess && out.gross && out.accumulate_into) {
        // run lengths never cross calls (calls cover whole days)
        e = cudaMemsetAsync(out.run, 0, sizeof(int) * (size_t)R, st);
        if (e == cudaSuccess && !out.continuous) e = cudaMemsetAsync(best, 0, sizeof(int) * (size_t)R, st);
    }
    for (int b0 = 0, nbc = 0; b0 < sun.n_blocks && e == cudaSuccess; b0 += nbc) {
        nbc = std::min(sun.n_blocks - b0, chunk);
        const size_t ncc = (size_t)nbc * n_tiles;
        int per = 1;
        const dim3 grid = bin_grid(std::max(T, 1), nbc, &per);
        e = cudaMemsetAsync(words, 0, sizeof(unsigned) * (direct ? ncc : nc + ncc), st);
        if (e != cudaSuccess) break;
        unsigned total = 0;
        if (direct) {
            KernelTimer kt(KT_RASTER_BIN, st);
            k_bin<true><<<grid, kBinThreads, 0, st>>>(sc, list, T, sun.steps, sun.blocks, b0, nbc, per, g, nullptr,
                                                      (unsigned)T, counts, bins);
        } else if (T > 0) {
            {
                KernelTimer kt(KT_RASTER_BIN, st);
                k_bin<false><<<grid, kBinThreads, 0, st>>>(sc, list, T, sun.steps, sun.blocks, b0, nbc, per, g, nullptr, 0u,
                                                           counts, nullptr);
            }
            if (by_tile) {       // the sums borrow the offsets, which are written below
                k_tile_sums<<<(n_tiles + 255) / 256, 256, 0, st>>>(counts, nbc, n_tiles, offsets);
                e = launch_work_order(offsets, nullptr, n_tiles, hist, order, nullptr, st);
            } else {
                e = launch_work_order(counts, nullptr, (long long)ncc, hist, order, nullptr, st);
            }
            if (e != cudaSuccess) break;
            e = cudaMemcpyAsync(offsets, counts, sizeof(unsigned) * ncc, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) break;
            e = exclusive_scan_u32(offsets, (long long)ncc, d_total, st);
            if (e != cudaSuccess) break;
            e = cudaMemcpyAsync(&total, d_total, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
            if (e != cudaSuccess) break;
            e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) break;
            if (total > bins_cap) {
                if (bins) cudaFreeAsync(bins, st);
                bins_cap = (size_t)total + total / 4 + 1024;
                e = sa::scratch_alloc(&bins, sizeof(int) * bins_cap, st);
                if (e == cudaErrorMemoryAllocation && nbc > 1) {      // again, with half the blocks
                    e = cudaSuccess;
                    bins_cap = 0;
                    chunk = (nbc + 1) / 2;
                    nbc = 0;
                    continue;
                }
                if (e != cudaSuccess) break;
            }
            if (total > 0) {
                KernelTimer kt(KT_RASTER_BIN, st);
                k_bin<true><<<grid, kBinThreads, 0, st>>>(sc, list, T, sun.steps, sun.blocks, b0, nbc, per, g, offsets, 0u,
                                                          cursor, bins);
            }
        } else {
            e = cudaMemsetAsync(offsets, 0, sizeof(unsigned) * ncc, st);
            if (e != cudaSuccess) break;
        }
        RasterArgs ra;
        ra.sc = sc; ra.sun = sun; ra.g = g; ra.b0 = b0; ra.nbc = nbc;
        ra.offsets = direct ? nullptr : offsets; ra.counts = counts; ra.bins = bins;
        ra.out = out; ra.best = best;
        ra.load_state = (b0 > 0) || out.accumulate_into;
        ra.final_chunk = (b0 + nbc >= sun.n_blocks);
        ra.R = R;
        ra.cull = sc.closed;
        ra.run = g_raster_run;
        ra.order = T > 0 && !direct ? order : nullptr;
        ra.cap = direct ? (unsigned)T : 0u;
        ra.parts = parts;
        ra.summary = summaries ? summaries + (size_t)b0 * (size_t)R : summary;
        {
            KernelTimer kt(KT_RASTER, st);
            if (by_tile) launch_k_raster(ra, n_tiles, st);
            else launch_k_items(ra, (int)ncc, out.stats != nullptr, st);
        }
        if (fold)
            launch_fold(summary, R, sun.blocks + b0, nbc, parts, out, best, ra.load_state, ra.final_chunk, st);
        e = cudaGetLastError();
    }
    for (void* p : {(void*)words, (void*)bins, (void*)best_scratch, (void*)list, (void*)d_reach, fold ? (void*)summary : nullptr})
        if (p) cudaFreeAsync(p, st);
    return e;
}

cudaError_t launch_raster_ground(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                                 const DevOut& out, cudaStream_t st) {
    return raster_ground(sc, rc, sun, out, nullptr, st);
}

cudaError_t launch_raster_summaries(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                                    unsigned* summaries, cudaStream_t st) {
    DevOut out{};
    return raster_ground(sc, rc, sun, out, summaries, st);
}

namespace {
inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
}  // namespace

cudaError_t launch_raster_ground_in(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                                    const DevOut& out, cudaStream_t st, unsigned char* scratch,
                                    size_t bytes, int* capacity_error) {
    *capacity_error = 0;
    TileGeom g;
    g.x0 = rc.x0; g.y0 = rc.y0; g.dx = rc.dx; g.nx = rc.nx; g.ny = rc.ny;
    g.tiles_x = (rc.nx + kTile - 1) / kTile;
    g.tiles_y = (rc.ny + kTile - 1) / kTile;
    const int n_tiles = g.tiles_x * g.tiles_y;
    const long long R = (long long)rc.nx * rc.ny;
    if (R == 0) return cudaSuccess;
    const int max_chunk = 16;
    const size_t nc = (size_t)max_chunk * n_tiles;
    // carve: run [R], best [R] (when the caller passes no continuous buffer), total,
    // counts / offsets / cursor [max_chunk * tiles], scan partials, bins (the rest)
    size_t off = 0;
    int* run = reinterpret_cast<int*>(scratch + off);
    off += align256(sizeof(int) * (size_t)R);
    int* best = out.continuous;
    if (!best) {
        best = reinterpret_cast<int*>(scratch + off);
        off += align256(sizeof(int) * (size_t)R);
    }
    unsigned* d_total = reinterpret_cast<unsigned*>(scratch + off);
    off += 256;
    unsigned* counts = reinterpret_cast<unsigned*>(scratch + off);
    off += align256(sizeof(unsigned) * nc);
    unsigned* offsets = reinterpret_cast<unsigned*>(scratch + off);
    off += align256(sizeof(unsigned) * nc);
    unsigned* cursor = reinterpret_cast<unsigned*>(scratch + off);
    off += align256(sizeof(unsigned) * nc);
    unsigned* partial = reinterpret_cast<unsigned*>(scratch + off);
    off += align256(sizeof(unsigned) * (size_t)scan_partials((long long)nc));
    if (off >= bytes) { *capacity_error = 1; return cudaSuccess; }
    int* bins = reinterpret_cast<int*>(scratch + off);
    const size_t bins_cap = (bytes - off) / sizeof(int);
    DevOut o = out;
    o.run = run;
    // Bins of blocks [b0, b0 + nbc): counts, their exclusive scan into offsets, and the
    // total, read back to the host.
    auto count_chunk = [&](int b0, int nbc, unsigned* total) -> cudaError_t {
        const size_t ncc = (size_t)nbc * n_tiles;
        *total = 0;
        cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(unsigned) * ncc, st);
        if (e != cudaSuccess) return e;
        if (sc.T == 0) return cudaMemsetAsync(offsets, 0, sizeof(unsigned) * ncc, st);
        int per = 1;
        const dim3 grid = bin_grid(sc.T, nbc, &per);
        k_bin<false><<<grid, kBinThreads, 0, st>>>(sc, nullptr, sc.T, sun.steps, sun.blocks, b0, nbc, per, g, nullptr, 0u, counts, nullptr);
        e = cudaMemcpyAsync(offsets, counts, sizeof(unsigned) * ncc, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = exclusive_scan_u32_with(offsets, (long long)ncc, partial, d_total, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(total, d_total, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        return e;
    };
    // Sizing pass, before any output is written: cut the blocks into chunks whose bins fit
    // the scratch (halving a chunk that does not), or report that one block alone does not.
    std::vector<int2> plan;
    int b0 = 0;
    int nbc = sun.n_blocks < max_chunk ? sun.n_blocks : max_chunk;
    while (b0 < sun.n_blocks) {
        if (b0 + nbc > sun.n_blocks) nbc = sun.n_blocks - b0;
        unsigned total = 0;
        cudaError_t e = count_chunk(b0, nbc, &total);
        if (e != cudaSuccess) return e;
        if ((size_t)total > bins_cap) {
            if (nbc == 1) { *capacity_error = 1; return cudaSuccess; }
            nbc = (nbc + 1) / 2;          // retry this chunk with fewer blocks
            continue;
        }
        plan.push_back(make_int2(b0, nbc));
        b0 += nbc;
    }
    cudaError_t e = cudaSuccess;
    if (out.accumulate_into) {
        e = cudaMemsetAsync(run, 0, sizeof(int) * (size_t)R, st);
        if (e == cudaSuccess && !out.continuous) e = cudaMemsetAsync(best, 0, sizeof(int) * (size_t)R, st);
        if (e != cudaSuccess) return e;
    }
    for (const int2& c : plan) {
        unsigned total = 0;
        e = count_chunk(c.x, c.y, &total);
        if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, sizeof(unsigned) * (size_t)c.y * n_tiles, st);
        if (e != cudaSuccess) return e;
        if (total > 0) {
            int per = 1;
            const dim3 grid = bin_grid(sc.T, c.y, &per);
            k_bin<true><<<grid, kBinThreads, 0, st>>>(sc, nullptr, sc.T, sun.steps, sun.blocks, c.x, c.y, per, g, offsets, 0u, cursor, bins);
        }
        RasterArgs ra;
        ra.sc = sc; ra.sun = sun; ra.g = g; ra.b0 = c.x; ra.nbc = c.y;
        ra.offsets = offsets; ra.counts = counts; ra.bins = bins;
        ra.out = o; ra.best = best;
        ra.load_state = (c.x > 0) || out.accumulate_into;
        ra.final_chunk = (c.x + c.y >= sun.n_blocks);
        ra.R = R;
        ra.cull = sc.closed;
        ra.run = g_raster_run;
        ra.order = nullptr;
        ra.cap = 0u;
        ra.parts = 1;
        ra.summary = nullptr;
        launch_k_raster(ra, n_tiles, st);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void set_raster_run(int run) { g_raster_run = run; }
int get_raster_run() { return g_raster_run; }

cudaError_t build_bins(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                       unsigned** offsets, unsigned** counts, int** bins, cudaStream_t st) {
    *offsets = nullptr; *counts = nullptr; *bins = nullptr;
    TileGeom g;
    g.x0 = rc.x0; g.y0 = rc.y0; g.dx = rc.dx; g.nx = rc.nx; g.ny = rc.ny;
    g.tiles_x = (rc.nx + kTile - 1) / kTile;
    g.tiles_y = (rc.ny + kTile - 1) / kTile;
    const size_t nc = (size_t)sun.n_blocks * g.tiles_x * g.tiles_y;
    if (nc == 0) return cudaSuccess;
    cudaError_t e = device_alloc(counts, sizeof(unsigned) * nc);
    if (e == cudaSuccess) e = device_alloc(offsets, sizeof(unsigned) * nc);
    unsigned* cursor = nullptr;
    unsigned* d_total = nullptr;
    if (e == cudaSuccess) e = sa::scratch_alloc(&cursor, sizeof(unsigned) * nc, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&d_total, sizeof(unsigned), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(*counts, 0, sizeof(unsigned) * nc, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, sizeof(unsigned) * nc, st);
    unsigned total = 0;
    int per = 1;
    const dim3 grid = bin_grid(sc.T > 0 ? sc.T : 1, sun.n_blocks, &per);
    if (e == cudaSuccess && sc.T > 0) {
        k_bin<false><<<grid, kBinThreads, 0, st>>>(sc, nullptr, sc.T, sun.steps, sun.blocks, 0, sun.n_blocks, per, g, nullptr, 0u,
                                                   *counts, nullptr);
        e = cudaMemcpyAsync(*offsets, *counts, sizeof(unsigned) * nc, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = exclusive_scan_u32(*offsets, (long long)nc, d_total, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&total, d_total, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    } else if (e == cudaSuccess) {
        e = cudaMemsetAsync(*offsets, 0, sizeof(unsigned) * nc, st);
    }
    if (e == cudaSuccess) e = device_alloc(bins, sizeof(int) * ((size_t)total + 1));
    if (e == cudaSuccess && total > 0)
        k_bin<true><<<grid, kBinThreads, 0, st>>>(sc, nullptr, sc.T, sun.steps, sun.blocks, 0, sun.n_blocks, per, g, *offsets, 0u,
                                                  cursor, *bins);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (cursor) cudaFreeAsync(cursor, st);
    if (d_total) cudaFreeAsync(d_total, st);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);
        if (*counts) cudaFree(*counts);
        if (*offsets) cudaFree(*offsets);
        if (*bins) cudaFree(*bins);
        *counts = nullptr; *offsets = nullptr; *bins = nullptr;
    }
    return e;
}

int batch_ctas_per_sm(bool by_delta) { return by_delta ? SA_RASTER_CTAS : kStateCtas; }

cudaError_t pick_batch_items(const BatchLaunch& bl, const int4* d_tiles, long long n, int max_blocks,
                             unsigned max_items, unsigned long long* n_items, int4** items, int** order, cudaStream_t st) {
    *n_items = 0;
    *items = nullptr;
    *order = nullptr;
    if (n == 0 || max_blocks == 0) return cudaSuccess;
    const TileGeom g = tile_geom(bl.grid);
    unsigned long long* totals = nullptr;        // of the two passes; the buckets of the order
    unsigned* weights = nullptr;
    cudaError_t e = sa::scratch_alloc(&totals, sizeof(unsigned long long) * 2 + sizeof(unsigned) * kOrderBuckets, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(totals, 0, sizeof(unsigned long long) * 2, st);
    const unsigned ctas = (unsigned)std::min(152ll * 32, (n * max_blocks + 127) / 128);
    unsigned long long total = 0;
    if (e == cudaSuccess) {
        k_batch_pick<<<ctas, 128, 0, st>>>(g, bl.intervals, bl.variants, bl.delta->boxes, d_tiles, n, max_blocks,
                                           totals, nullptr, nullptr);
        e = cudaMemcpyAsync(&total, totals, sizeof(total), cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && total > 0 && total <= max_items) {
        e = device_alloc(items, sizeof(int4) * (size_t)total);
        if (e == cudaSuccess) e = device_alloc(order, sizeof(int) * (size_t)total);
        if (e == cudaSuccess) e = sa::scratch_alloc(&weights, sizeof(unsigned) * (size_t)total, st);
        if (e == cudaSuccess) {
            k_batch_pick<<<ctas, 128, 0, st>>>(g, bl.intervals, bl.variants, bl.delta->boxes, d_tiles, n, max_blocks,
                                               totals + 1, *items, weights);
            e = launch_work_order(weights, nullptr, (long long)total, reinterpret_cast<unsigned*>(totals + 2), *order,
                                  nullptr, st);
        }
    }
    if (totals) cudaFreeAsync(totals, st);
    if (weights) cudaFreeAsync(weights, st);
    *n_items = total;
    return e;
}

cudaError_t launch_batch(const BatchLaunch& bl, cudaStream_t st) {
    BatchArgs ba;
    ba.g.x0 = bl.grid.x0; ba.g.y0 = bl.grid.y0; ba.g.dx = bl.grid.dx;
    ba.g.nx = bl.grid.nx; ba.g.ny = bl.grid.ny;
    ba.g.tiles_x = (bl.grid.nx + kTile - 1) / kTile;
    ba.g.tiles_y = (bl.grid.ny + kTile - 1) / kTile;
    ba.base_tris = bl.base.tris;
    ba.intervals = bl.intervals;
    ba.variants = bl.variants;
    ba.items = bl.items;
    ba.n_items = bl.n_items;
    ba.counter = bl.counter;
    ba.removed = bl.removed;
    ba.tower_tris = bl.tower_tris;
    ba.counts_out = bl.counts_out;
    ba.impact_out = bl.impact_out;
    ba.cull = bl.base.closed;
    ba.run = bl.run;
    ba.stats = bl.stats;
    cudaError_t e = cudaMemsetAsync(bl.counter, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    if (bl.delta) {
        const int VI = bl.V * bl.I;
        if (VI > 0 && bl.max_cells > 0) {
            const dim3 grid((unsigned)std::min(1024ll, (bl.max_cells + 255) / 256), (unsigned)std::min(VI, 65535));
            k_batch_base<<<grid, 256, 0, st>>>(ba, bl.V, bl.I);
        }
        if (bl.n_items == 0) return cudaGetLastError();
        if (ba.cull) {
            if (bl.stats) k_batch_delta<true, true><<<bl.ctas, kRasterThreads, 0, st>>>(ba, *bl.delta);
            else k_batch_delta<false, true><<<bl.ctas, kRasterThreads, 0, st>>>(ba, *bl.delta);
        } else {
            if (bl.stats) k_batch_delta<true, false><<<bl.ctas, kRasterThreads, 0, st>>>(ba, *bl.delta);
            else k_batch_delta<false, false><<<bl.ctas, kRasterThreads, 0, st>>>(ba, *bl.delta);
        }
        return cudaGetLastError();
    }
    if (bl.n_items == 0) return cudaSuccess;
    if (ba.cull) {
        if (bl.stats) k_batch<true, true><<<bl.ctas, kRasterThreads, 0, st>>>(ba);
        else k_batch<false, true><<<bl.ctas, kRasterThreads, 0, st>>>(ba);
    } else {
        if (bl.stats) k_batch<true, false><<<bl.ctas, kRasterThreads, 0, st>>>(ba);
        else k_batch<false, false><<<bl.ctas, kRasterThreads, 0, st>>>(ba);
    }
    return cudaGetLastError();
}

}  // namespace sa
