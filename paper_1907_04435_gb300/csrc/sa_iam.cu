// sa_iam.cu -- inverse accrual map (Sec. 5) of a ground receiver grid.
//
// Per block of K steps:
//   k_iam_sources  every cell centre p traces toward the sun at the block's first step and
//               keeps the L nearest intersections farther than 1 m (the paper's source
//               levels and its 100 cm acne rule); k_iam_sources_warp for very coarse grids.
//   k_iam_draw  each source s casts its shadow at step
//               k at q_k, the projection of s along d_k onto the ground; the shadow line
//               q_0 -> q_{K-1} is cut into K - 1 pieces and piece [q_k, q_{k+1}] sets bit
//               k of every grid cell it touches (closed cells), bit K-1 being set at
//               q_{K-1}.  The same is done from the block's last step with the pieces
//               running backwards (the paper's t_n -> t_1 map), which catches stretching
//               shadows and sources missed by the first map.
//   k_iam_fold  folds the blocks' 64-bit vectors of each cell into its gross / continuous
//               state.
// The bit vectors live in one uint64 per cell and block; drawing gathers a line's bits in a
// cell and uses one atomicOr.  All blocks go in one launch: one launch per block left
// the chip waiting for the longest warps of each (4.81 -> 3.20 ms; 64^2 cells 2.95 ms ->
// 0.29 with the gathered marks).  This is the paper's approximate method: it is compared with its
// own FP64 restatement and with the exact result (the paper's area-error bar).
#include <algorithm>

#include "sa_internal.cuh"
#include "sa_light.cuh"

namespace sa {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = 4;
constexpr int kMaxLevels = 8;
constexpr float kSourceTmin = 1.0f;     // sources closer than 100 cm are ignored (Sec. 5)

// Watertight test returning the distance of the hit (see hit_tri).
template <int KZ>
__device__ __forceinline__ bool hit_tri_t(const float3& o, const float4& a, const float4& b,
                                          const float4& c, float Sx, float Sy, float Sz,
                                          float tmin, float* t_out) {
    constexpr int KX = (KZ + 1) % 3, KY = (KZ + 2) % 3;
    const float az = comp<KZ>(a) - comp3<KZ>(o);
    const float bz = comp<KZ>(b) - comp3<KZ>(o);
    const float cz = comp<KZ>(c) - comp3<KZ>(o);
    const float ax = fmaf(-Sx, az, comp<KX>(a) - comp3<KX>(o));
    const float ay = fmaf(-Sy, az, comp<KY>(a) - comp3<KY>(o));
    const float bx = fmaf(-Sx, bz, comp<KX>(b) - comp3<KX>(o));
    const float by = fmaf(-Sy, bz, comp<KY>(b) - comp3<KY>(o));
    const float cx = fmaf(-Sx, cz, comp<KX>(c) - comp3<KX>(o));
    const float cy = fmaf(-Sy, cz, comp<KY>(c) - comp3<KY>(o));
    const float U = __fsub_rn(__fmul_rn(cx, by), __fmul_rn(cy, bx));
    const float V = __fsub_rn(__fmul_rn(ax, cy), __fmul_rn(ay, cx));
    const float W = __fsub_rn(__fmul_rn(bx, ay), __fmul_rn(by, ax));
    if ((U < 0.f || V < 0.f || W < 0.f) && (U > 0.f || V > 0.f || W > 0.f)) return false;
    const float det = U + V + W;
    if (det == 0.f) return false;
    const float T = U * (Sz * az) + V * (Sz * bz) + W * (Sz * cz);
    const float t = T / det;
    if (!(t > tmin)) return false;
    *t_out = t;
    return true;
}

struct Grid {
    float x0, y0, dx;
    int nx, ny;
};

// Marks of a thread's shadow line: consecutive pieces mostly stay in one cell, so its bits are
// gathered and ORed into memory once, when the line leaves it.  (Reading the word first to
// skip bits that are set made every lane of the warp wait: 3.20 ms against 2.76 for 613 x 457
// cells x 481 steps.)
template <class Cell>
struct Marker {
    unsigned long long* masks;
    Cell cell;
    unsigned long long bits;
    __device__ __forceinline__ void flush() {
        if (bits) atomicOr(&masks[cell], bits);
    }
    __device__ __forceinline__ void mark(Cell c, unsigned long long bit) {
        if (c != cell) {
            flush();
            cell = c;
            bits = 0ull;
        }
        bits |= bit;
    }
};

// Every closed grid cell touched by the segment P -> Q gets `bit`.
template <class Cell>
__device__ void draw_segment(const Grid& g, float px, float py, float qx, float qy,
                             Marker<Cell>& mk, unsigned long long bit) {
    const float inv = 1.f / g.dx;
    const float ymin = fminf(py, qy), ymax = fmaxf(py, qy);
    int iy0 = (int)ceilf((ymin - g.y0) * inv) - 1;
    int iy1 = (int)floorf((ymax - g.y0) * inv);
    iy0 = max(iy0, 0);
    iy1 = min(iy1, g.ny - 1);
    for (int iy = iy0; iy <= iy1; ++iy) {
        const float b0 = g.y0 + (float)iy * g.dx, b1 = b0 + g.dx;
        float xa, xb;
        if (py == qy) {
            if (py < b0 || py > b1) continue;
            xa = fminf(px, qx); xb = fmaxf(px, qx);
        } else {
            const float rdy = 1.f / (qy - py);
            const float ta = (b0 - py) * rdy, tb = (b1 - py) * rdy;
            const float lo = fmaxf(fminf(ta, tb), 0.f), hi = fminf(fmaxf(ta, tb), 1.f);
            if (lo > hi) continue;
            const float x1 = fmaf(lo, qx - px, px), x2 = fmaf(hi, qx - px, px);
            xa = fminf(x1, x2); xb = fmaxf(x1, x2);
        }
        int ix0 = (int)ceilf((xa - g.x0) * inv) - 1;
        int ix1 = (int)floorf((xb - g.x0) * inv);
        ix0 = max(ix0, 0);
        ix1 = min(ix1, g.nx - 1);
        const Cell row = (Cell)iy * (Cell)g.nx;
        for (int ix = ix0; ix <= ix1; ++ix) mk.mark(row + (Cell)ix, bit);
    }
}

// A walk of the BVH for the sources of one or two ends of blocks (end 2 b: block b's first
// step, 2 b + 1: its last): a block's last step and the next one's first are neighbours
// within a day, and their rays share a walk.
struct IamWalk {
    int step, n;          // the walk's steps: step, and step + 1 where n is 2; none where n is 0
    int end;              // the first step's end; a second step's is the next
};

// The walk of every end of the n blocks (none for an end that shares the one before).
__global__ void k_iam_walks(const StepConst* __restrict__ steps, const BlockConst* __restrict__ blocks, int n,
                            IamWalk* __restrict__ walks, RunLight* __restrict__ runs) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x), b = i >> 1;
    if (b >= n) return;
    auto joins = [&](int q) {       // block q's first step shares the walk of the one before
        return q > 0 && q < n && !blocks[q].new_day && blocks[q - 1].j0 + blocks[q - 1].K == blocks[q].j0;
    };
    const int j = i & 1 ? blocks[b].j0 + blocks[b].K - 1 : blocks[b].j0;
    const int m = i & 1 ? (joins(b + 1) ? 2 : 1) : (joins(b) ? 0 : 1);
    walks[i] = IamWalk{j, m, i};
    if (m == 0) return;
    const int k = j + m - 1;
    const LightBasis L = light_basis(steps[k], steps[j], steps[k]);
    LightStep ls = light_drift(L, steps[j]);         // (the bounds on d . n are not used)
    light_merge(ls, light_drift(L, steps[k]));
    light_finish(L, ls, &runs[i]);
    runs[i].k0 = 0;
    runs[i].kn = m;
    runs[i].j0 = j;
    runs[i].blk = b;
}

// Tests n <= 32 queued pairs of a warp, one per lane, and puts the hits into their cells'
// lists: the distance's bits order as the distance does, and what a slot's minimum pushes
// out goes on to the next slot, so the L slots end with the L least in order, whichever
// order the hits came in.
template <int KZ, class Smem>
__device__ __forceinline__ void drain_sources(Smem& sm, unsigned (*near)[kTileThreads], const unsigned short* q, int n,
                                              const StepConst& s, int L) {
    const int lane = threadIdx.x & 31;
    if (lane >= n) return;
    const unsigned e = q[lane];
    const int who = (int)(e >> 8), i = (int)(e & 0xffu);
    const float4 p = sm.o[who];
    float t;
    if (!hit_tri_t<KZ>(make_float3(p.x, p.y, p.z), sm.tri[3 * i], sm.tri[3 * i + 1], sm.tri[3 * i + 2], s.Sx, s.Sy, s.Sz,
                       kSourceTmin, &t)) return;
    unsigned v = __float_as_uint(t);
    for (int l = 0; l < L && v != 0xffffffffu; ++l) v = max(v, atomicMin(&near[l][who], v));
}

constexpr int kIamChunk = 64;
constexpr int kPatchX = 16, kPatchY = 8;       // a group's cells: 8 x 4 per warp

// The sources of a group of 128 cells at the ends of blocks of one walk: the CTA walks the BVH
// once for all of its rays (walk_group) and tests the pairs that their common direction lets
// through.  src [2 blocks][L][R]: distances, ascending, 0 past the last.  Bound by the latency
// of the walk's steps.  613 x 457 cells, 18 ends: 403 us, 630 with a walk per end, some 800
// with a node-list walk per 32 cells and end, whose lanes tested a ray each.
__global__ void __launch_bounds__(kTileThreads, 8)
k_iam_sources(DevScene sc, Grid g, const StepConst* __restrict__ steps, const IamWalk* __restrict__ walks,
              const RunLight* __restrict__ runs, int L, float* __restrict__ src) {
    __shared__ LightSmem<kIamChunk> sm;
    __shared__ GroupSmem<kIamChunk, 512> gs;
    __shared__ unsigned near[2][kMaxLevels][kTileThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int groups_x = (g.nx + kPatchX - 1) / kPatchX;
    const int gy = (int)(blockIdx.x / (unsigned)groups_x), gx = (int)(blockIdx.x - (unsigned)gy * (unsigned)groups_x);
    const int ix = gx * kPatchX + (warp & 1) * 8 + (lane & 7), iy = gy * kPatchY + (warp >> 1) * 4 + (lane >> 3);
    const bool active = ix < g.nx && iy < g.ny;
    const RunLight& rl = runs[blockIdx.y];
    const IamWalk walk = walks[blockIdx.y];
    if (walk.n == 0) return;
    const float4 p = make_float4(__fadd_rn(g.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), g.dx)),
                                 __fadd_rn(g.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), g.dx)), 0.f, 0.f);
    sm.o[tid] = p;
    sm.m[tid] = 0u;
    for (int h = 0; h < walk.n; ++h)
        for (int l = 0; l < L; ++l) near[h][l][tid] = 0xffffffffu;
    unsigned long long n_box = 0;
    walk_group<false>(sm, gs, sc, rl, active, p, [](int) { return 1u; }, n_box, [&](int nt, float la, float lb) {
        light_pass<false>(sm, rl, nt, active, p, la, lb, 1u, [&](const unsigned short* q, int n) {
            for (int h = 0; h < walk.n; ++h) {
                const StepConst& s = steps[walk.step + h];
                if (s.kz == 2) drain_sources<2>(sm, near[h], q, n, s, L);
                else if (s.kz == 0) drain_sources<0>(sm, near[h], q, n, s, L);
                else drain_sources<1>(sm, near[h], q, n, s, L);
            }
        });
        return false;
    });
    if (!active) return;
    const long long R = (long long)g.nx * g.ny;
    for (int h = 0; h < walk.n; ++h) {
        float* out = src + (long long)(walk.end + h) * L * R + (long long)iy * g.nx + ix;
        for (int l = 0; l < L; ++l) {
            const unsigned v = near[h][l][tid];
            out[(long long)l * R] = v == 0xffffffffu ? 0.f : __uint_as_float(v);
        }
    }
}

// The L nearest hits of the warp's rays toward step s, in order (bits of the distances, past the
// last 0xffffffff), by one walk of the node list: a node is entered when any ray meets it
// before its L-th hit so far.
template <int KZ>
__device__ __forceinline__ void nearest_by_warp(const DevScene& sc, const float3& o, const StepConst& s, bool active, int L,
                                                unsigned* best) {
#pragma unroll
    for (int l = 0; l < kMaxLevels; ++l) best[l] = 0xffffffffu;
    float last = 3.4e38f;
    for (int i = __any_sync(kFull, active) ? 0 : sc.n_nodes; i < sc.n_nodes;) {
        const float4 lo = __ldg(&sc.nodes[2 * i]);
        const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
        const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_TRACE_ESCAPE);
        const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_TRACE_LEAF);
        const bool in = active && hit_box_before(o, s.ix, s.iy, s.iz, lo, hi, last);
        if (tri < 0) {
            i = __any_sync(kFull, in) ? i + 1 : esc;
            continue;
        }
        i = esc;
        float t;
        if (!in || !hit_tri_t<KZ>(o, __ldg(&sc.tris[3 * tri]), __ldg(&sc.tris[3 * tri + 1]), __ldg(&sc.tris[3 * tri + 2]), s.Sx,
                                  s.Sy, s.Sz, kSourceTmin, &t)) continue;
        unsigned v = __float_as_uint(t);
#pragma unroll
        for (int l = 0; l < kMaxLevels; ++l) {
            if (l >= L) break;
            const unsigned b = best[l];
            best[l] = min(b, v);
            v = max(b, v);
            if (l == L - 1 && best[l] != 0xffffffffu) last = __uint_as_float(best[l]);
        }
    }
}

// The scene's triangles over the ground of a group's 128 cells from which its box holds too many
// of them against what its rays meet, and the sources are found by warps.  Whole call, ms
// by groups / by warps, 122k triangles, 481 steps in June: 268 triangles 0.77 / 1.05, 1,677
// 0.94 / 0.68, 6,708 4.1 / 0.79, 47,702 34 / 1.1; in December 745 2.2 / 3.0, 3,773 3.3 / 3.9,
// 11,925 8.8 / 5.6; hour steps 745 0.73 / 0.85, 3,773 2.5 / 1.3.
constexpr double kGroupHeld = 1600.0;

// The same sources by warps of 8 x 4 cells and end, for cells far apart (kGroupHeld).
__global__ void __launch_bounds__(32 * kWarps)
k_iam_sources_warp(DevScene sc, Grid g, const StepConst* __restrict__ steps, const BlockConst* __restrict__ blocks, int L,
                   float* __restrict__ src) {
    const int lane = threadIdx.x & 31;
    const long long warp_id = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    const int tiles_x = (g.nx + 7) >> 3, end = blockIdx.y;
    const long long ty = warp_id / tiles_x;
    const int tx = (int)(warp_id - ty * tiles_x);
    const int ix = tx * 8 + (lane & 7);
    const long long iy = ty * 4 + (lane >> 3);
    const bool active = ix < g.nx && iy < g.ny;
    const BlockConst& bc = blocks[end >> 1];
    const StepConst s = steps[end & 1 ? bc.j0 + bc.K - 1 : bc.j0];
    const float3 o = make_float3(__fadd_rn(g.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), g.dx)),
                                 __fadd_rn(g.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), g.dx)), 0.f);
    unsigned best[kMaxLevels];
    if (s.kz == 2) nearest_by_warp<2>(sc, o, s, active, L, best);
    else if (s.kz == 0) nearest_by_warp<0>(sc, o, s, active, L, best);
    else nearest_by_warp<1>(sc, o, s, active, L, best);
    if (!active) return;
    const long long R = (long long)g.nx * g.ny;
    float* out = src + (long long)end * L * R + iy * g.nx + ix;
#pragma unroll
    for (int l = 0; l < kMaxLevels; ++l)
        if (l < L) out[(long long)l * R] = best[l] == 0xffffffffu ? 0.f : __uint_as_float(best[l]);
}

// A CTA lists the sources of its 128 cells, 32 in a patch of 8 x 4 per warp; then its threads
// draw them, one line per thread whichever cell it comes from: most cells are lit or have two
// sources where their neighbours have four, and a warp that drew its own cells' sources
// waited for the longest list.  Bound by issue: the pieces of the lines, one after the other.
template <class Cell>
__global__ void __launch_bounds__(32 * kWarps, 12)
k_iam_draw(Grid g, const StepConst* __restrict__ steps, const BlockConst* __restrict__ blocks,
           int L, const float* __restrict__ src, unsigned long long* __restrict__ all_masks) {
    __shared__ float s_t[32 * kWarps * kMaxLevels * 2];               // the sources' distances,
    __shared__ unsigned short s_from[32 * kWarps * kMaxLevels * 2];   // thread | direction << 15
    __shared__ float2 s_o[32 * kWarps], s_u[kMaxBlock];
    __shared__ int s_n;
    const int tid = threadIdx.x, lane = tid & 31;
    const int j0 = blocks[blockIdx.y].j0, K = blocks[blockIdx.y].K;
    const long long R = (long long)g.nx * g.ny;
    const long long warp_id = (long long)blockIdx.x * kWarps + (tid >> 5);
    const int tiles_x = (g.nx + 7) >> 3;
    const long long ty = warp_id / tiles_x;
    const int tx = (int)(warp_id - ty * tiles_x);
    const int ix = tx * 8 + (lane & 7);
    const long long iy = ty * 4 + (lane >> 3);
    const bool active = ix < g.nx && iy < g.ny;
    s_o[tid] = make_float2(__fadd_rn(g.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), g.dx)),
                           __fadd_rn(g.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), g.dx)));
    if (tid < K) s_u[tid] = make_float2(steps[j0 + tid].ux, steps[j0 + tid].uy);
    if (tid == 0) s_n = 0;
    __syncthreads();
    for (int dir = 0; dir < 2; ++dir) {
        // level by level, so that neighbours' lines of one source surface stay together
        const float* in = src + ((long long)blockIdx.y * 2 + dir) * L * R + iy * g.nx + ix;
        for (int l = 0; l < L; ++l) {
            const float t = active ? __ldcs(&in[(long long)l * R]) : 0.f;
            const unsigned has = __ballot_sync(kFull, t > 0.f);
            if (!has) break;
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_n, __popc(has));
            at = __shfl_sync(kFull, at, 0) + __popc(has & ((1u << lane) - 1u));
            if (t > 0.f) {
                s_t[at] = t;
                s_from[at] = (unsigned short)(tid | (dir << 15));
            }
        }
    }
    __syncthreads();
    Marker<Cell> mk{all_masks + (long long)blockIdx.y * g.nx * g.ny, (Cell)-1, 0ull};
    for (int e = tid; e < s_n; e += 32 * kWarps) {
        const float t = s_t[e];
        const int from = s_from[e], dir = from >> 15;
        const float2 p0 = s_o[from & 0x7fff];
        // q_k for the block's steps; the pieces run forward (dir 0) or backward (dir 1)
        int k = dir == 0 ? 0 : K - 1;
        const int dk = dir == 0 ? 1 : -1;
        const StepConst& s = steps[j0 + k];
        const float sx = fmaf(t, s.dx, p0.x), sy = fmaf(t, s.dy, p0.y), sz = t * s.dz;
        float px = fmaf(-sz, s_u[k].x, sx), py = fmaf(-sz, s_u[k].y, sy);
        for (int i = 0; i + 1 < K; ++i) {
            const float2 u = s_u[k + dk];
            const float qx = fmaf(-sz, u.x, sx), qy = fmaf(-sz, u.y, sy);
            draw_segment(g, px, py, qx, qy, mk, 1ull << k);
            px = qx; py = qy;
            k += dk;
        }
        draw_segment(g, px, py, px, py, mk, 1ull << k);
    }
    mk.flush();
}

__global__ void k_iam_fold(long long R, const BlockConst* __restrict__ blocks, int nbc,
                           const unsigned long long* __restrict__ masks, DevOut out, int first,
                           int last) {
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    RunState st{0, 0, 0};
    if (!first || out.accumulate_into) {
        st.gross = out.gross[r];
        st.best = out.continuous ? out.continuous[r] : 0;
        st.run = (first) ? 0 : out.run[r];
    }
    for (int b = 0; b < nbc; ++b) {
        const unsigned long long m = masks[(long long)b * R + r];
        stitch(st, m, blocks[b].K, blocks[b].new_day);
        if (out.masks && m) out.masks[(long long)blocks[b].mask_block * R + r] |= m;
    }
    out.gross[r] = st.gross;
    if (out.continuous) out.continuous[r] = st.best;
    out.run[r] = st.run;
    if (last && out.minutes) out.minutes[r] = (float)st.gross * out.step_minutes;
}

}  // namespace

cudaError_t launch_iam(const DevScene& sc, const float* scene_box, const DevRecv& rc, const DevSun& sun,
                       int L, const DevOut& out, cudaStream_t st) {
    const long long R = (long long)rc.nx * rc.ny;
    if (R == 0) return cudaSuccess;
    if (L < 1 || L > kMaxLevels) return cudaErrorInvalidValue;
    const double area = ((double)scene_box[3] - scene_box[0]) * ((double)scene_box[4] - scene_box[1]);
    const double held = area > 0.0 ? (double)sc.T * kTileThreads * (double)rc.dx * rc.dx / area : 0.0;
    const bool by_warps = held > kGroupHeld;
    // the blocks go in one launch, as many as 1 GiB of masks and sources holds, or the memory
    // there is
    int chunk = (int)std::max(1ll, std::min({(long long)sun.n_blocks, 32767ll, (1ll << 30) / ((8ll + 8ll * L) * R)}));
    unsigned long long* masks = nullptr;
    float* src = nullptr;
    RunLight* runs = nullptr;
    IamWalk* d_walks = nullptr;
    cudaError_t e = sa::scratch_alloc_blocks(&src, sizeof(float) * 2 * (size_t)L * (size_t)R, &chunk, st);
    if (e == cudaSuccess) e = sa::scratch_alloc_blocks(&masks, sizeof(unsigned long long) * (size_t)R, &chunk, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&runs, sizeof(RunLight) * 2 * (size_t)chunk, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&d_walks, sizeof(IamWalk) * 2 * (size_t)chunk, st);
    Grid g{rc.x0, rc.y0, rc.dx, rc.nx, rc.ny};
    const long long warps = (long long)((rc.nx + 7) / 8) * ((rc.ny + 3) / 4);
    const unsigned ctas = (unsigned)((warps + kWarps - 1) / kWarps);
    for (int b0 = 0; b0 < sun.n_blocks && e == cudaSuccess; b0 += chunk) {
        const int nbc = std::min(chunk, sun.n_blocks - b0);
        e = cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)R * nbc, st);
        if (e != cudaSuccess) break;
        {
            KernelTimer kt(KT_IAM, st);
            const dim3 groups((unsigned)((rc.nx + kPatchX - 1) / kPatchX) * (unsigned)((rc.ny + kPatchY - 1) / kPatchY),
                              2u * (unsigned)nbc);
            if (by_warps) {
                k_iam_sources_warp<<<dim3(ctas, 2u * (unsigned)nbc), 32 * kWarps, 0, st>>>(sc, g, sun.steps, sun.blocks + b0, L, src);
            } else {
                k_iam_walks<<<(2 * nbc + 63) / 64, 64, 0, st>>>(sun.steps, sun.blocks + b0, nbc, d_walks, runs);
                k_iam_sources<<<groups, kTileThreads, 0, st>>>(sc, g, sun.steps, d_walks, runs, L, src);
            }
            const dim3 grid(ctas, (unsigned)nbc);
            if (R < (1ll << 31)) k_iam_draw<unsigned><<<grid, 32 * kWarps, 0, st>>>(g, sun.steps, sun.blocks + b0, L, src, masks);
            else k_iam_draw<long long><<<grid, 32 * kWarps, 0, st>>>(g, sun.steps, sun.blocks + b0, L, src, masks);
        }
        k_iam_fold<<<(unsigned)((R + 255) / 256), 256, 0, st>>>(R, sun.blocks + b0, nbc, masks, out, b0 == 0,
                                                               b0 + nbc == sun.n_blocks);
        e = cudaGetLastError();
    }
    for (void* p : {(void*)masks, (void*)src, (void*)runs, (void*)d_walks})
        if (p) cudaFreeAsync(p, st);
    return e;
}

}  // namespace sa
