// sa_sam_points.cu -- shadow accrual map for point receivers (facades), in light space.
//
// Sec. 4 renders the scene once per interval into a map on a plane orthogonal to the sun
// direction and tests every receiver against its n slices.  Here each run of <= 32
// consecutive steps of a block gets such a light-space map.  Coordinates are taken in a
// basis (e1, e2) orthogonal to the run's middle direction d_m, around a reference point.
// The map is a grid of light-space tiles:
//   - every triangle that faces the sun at some step of the run is binned into the tiles
//     its projection covers, widened by the drift of the run's rays up to the triangle's
//     top: a ray of step k from a receiver leaves the receiver's light-space point by
//     h x delta_k at height h above it (delta_k = (d_k . e1, d_k . e2) / d_k.z), and the
//     run's delta_k lie in a box that is long along the sun's motion and thin across it;
//   - every receiver goes into the single tile holding its own projection.
// A receiver and a triangle its rays can meet during the run therefore share a tile.
// One pass over the geometry per run thus serves all of the run's steps.  The test
// itself is exact: per (receiver, triangle) the Plücker edge moments are set up once,
// then each of the run's steps costs three dot products and a distance check
// (watertight with canonically ordered edges, as in the ray-traced accrual).  For a
// closed scene only sun-facing triangles are binned: any ray that meets a closed solid
// crosses one of its sun-facing faces.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "sa_handles.cuh"
#include "sa_light.cuh"

namespace sa {

namespace {

// side (m) of the light-space tiles
#ifndef SA_LIGHT_TILE
#define SA_LIGHT_TILE 32.f
#endif
// resident CTAs per SM k_sam_tile is compiled for: 9 gives 56 registers, 16 bytes of spills
#ifndef SA_TILE_CTAS
#define SA_TILE_CTAS 9
#endif

// Steps of the run at which the triangle faces the sun (cull) or is not edge-on to it.  Its
// normal's bounds over the run settle most triangles without the loop.
__device__ __forceinline__ unsigned run_front(const float4& a, const float4& b, const float4& c,
                                              const StepConst* steps, const RunLight& rl, bool cull) {
    const float ux = b.x - a.x, uy = b.y - a.y, uz = b.z - a.z;
    const float vx = c.x - a.x, vy = c.y - a.y, vz = c.z - a.z;
    const float nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
    const unsigned full = rl.kn >= 32 ? 0xffffffffu : ((1u << rl.kn) - 1u);
    const float2 nb = run_dot_bounds(rl, nx, ny, nz);
    if (nb.x > 0.f || nb.y < 0.f) return cull && nb.y < 0.f ? 0u : full;   // one sign at every step
    unsigned m = 0;
    for (int k = 0; k < rl.kn; ++k) {
        const StepConst& s = steps[rl.j0 + rl.k0 + k];
        const float nd = nx * s.dx + ny * s.dy + nz * s.dz;
        if (cull ? nd > 0.f : nd != 0.f) m |= 1u << k;
    }
    return m;
}

// tile range of a triangle's widened light-space box; false if outside the grid
__device__ __forceinline__ bool tri_tiles(const float4& a, const float4& b, const float4& c,
                                          const RunLight& rl, int* ta0, int* ta1, int* tb0, int* tb1) {
    float pa[3], pb[3];
    light_ab(rl, rl.c, a.x, a.y, a.z, &pa[0], &pb[0]);
    light_ab(rl, rl.c, b.x, b.y, b.z, &pa[1], &pb[1]);
    light_ab(rl, rl.c, c.x, c.y, c.z, &pa[2], &pb[2]);
    // receivers that a ray rising at most H to the triangle's top can reach it from
    const float H = fmaxf(fmaxf(a.z, fmaxf(b.z, c.z)) - rl.zr, 0.f);
    const float amin = fminf(pa[0], fminf(pa[1], pa[2])) - fmaf(H, rl.da_hi, kLightSlack);
    const float amax = fmaxf(pa[0], fmaxf(pa[1], pa[2])) + fmaf(H, rl.da_lo, kLightSlack);
    const float bmin = fminf(pb[0], fminf(pb[1], pb[2])) - fmaf(H, rl.db_hi, kLightSlack);
    const float bmax = fmaxf(pb[0], fmaxf(pb[1], pb[2])) + fmaf(H, rl.db_lo, kLightSlack);
    const float inv = 1.f / rl.tile;
    const float fa0 = floorf((amin - rl.a0) * inv), fa1 = floorf((amax - rl.a0) * inv);
    const float fb0 = floorf((bmin - rl.b0) * inv), fb1 = floorf((bmax - rl.b0) * inv);
    if (fa1 < 0.f || fb1 < 0.f || fa0 >= (float)rl.nta || fb0 >= (float)rl.ntb) return false;
    *ta0 = (int)fmaxf(fa0, 0.f);
    *ta1 = (int)fminf(fa1, (float)(rl.nta - 1));
    *tb0 = (int)fmaxf(fb0, 0.f);
    *tb1 = (int)fminf(fb1, (float)(rl.ntb - 1));
    return true;
}

__device__ __forceinline__ int recv_tile(const float4& o, const RunLight& rl) {
    float a, b;
    light_ab(rl, rl.c, o.x, o.y, o.z, &a, &b);
    const float inv = 1.f / rl.tile;
    const int ta = min(max((int)floorf((a - rl.a0) * inv), 0), rl.nta - 1);
    const int tb = min(max((int)floorf((b - rl.b0) * inv), 0), rl.ntb - 1);
    return rl.tile_base + tb * rl.nta + ta;
}

__global__ void k_lt_bin(DevScene sc, const StepConst* __restrict__ steps,
                         const RunLight* __restrict__ runs, int n_runs, bool fill,
                         unsigned* __restrict__ counts, const unsigned* __restrict__ offsets,
                         unsigned* __restrict__ cursor, int* __restrict__ bins) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (t >= sc.T || r >= n_runs) return;
    const RunLight& rl = runs[r];
    const float4 a = __ldg(&sc.tris[3 * t]), b = __ldg(&sc.tris[3 * t + 1]), c = __ldg(&sc.tris[3 * t + 2]);
    if (run_front(a, b, c, steps, rl, sc.closed != 0) == 0u) return;
    int ta0, ta1, tb0, tb1;
    if (!tri_tiles(a, b, c, rl, &ta0, &ta1, &tb0, &tb1)) return;
    for (int tb = tb0; tb <= tb1; ++tb)
        for (int ta = ta0; ta <= ta1; ++ta) {
            const int cell = rl.tile_base + tb * rl.nta + ta;
            if (fill) bins[offsets[cell] + atomicAdd(&cursor[cell], 1u)] = t;
            else atomicAdd(&counts[cell], 1u);
        }
}

// Receivers are Morton-ordered, so neighbouring lanes usually share a tile: lanes with the
// same tile are grouped (match_any) and their leader makes one atomic for the group.
__global__ void k_lr_bin(const float4* __restrict__ orig, long long R,
                         const RunLight* __restrict__ runs, int n_runs, bool fill,
                         unsigned* __restrict__ counts, const unsigned* __restrict__ offsets,
                         unsigned* __restrict__ cursor, int* __restrict__ bins) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const bool valid = s < R && r < n_runs;
    const int cell = valid ? recv_tile(orig[s], runs[r]) : -1 - lane;   // unique when invalid
    const unsigned peers = __match_any_sync(0xffffffffu, cell);
    const int leader = __ffs(peers) - 1;
    const unsigned rank = __popc(peers & ((1u << lane) - 1u));
    unsigned base = 0;
    if (valid && lane == leader) {
        if (fill) base = atomicAdd(&cursor[cell], (unsigned)__popc(peers));
        else atomicAdd(&counts[cell], (unsigned)__popc(peers));
    }
    if (fill) {
        base = __shfl_sync(0xffffffffu, base, leader);
        if (valid) bins[offsets[cell] + base + rank] = (int)s;
    }
}

struct TileArgs {
    DevScene sc;
    const StepConst* steps;
    const RunLight* runs;
    int n_runs;
    const int* tile_run;           // run of each global tile
    const int* order;              // tile of each CTA, most work first, empty tiles left out
    const unsigned* t_off; const unsigned* t_cnt; const int* t_bins;
    const unsigned* r_off; const unsigned* r_cnt; const int* r_bins;
    const float4* orig;
    unsigned long long* masks;     // [blocks of the chunk][R] block masks (sorted order)
    long long R;
    unsigned long long* stats;
};

// One CTA per light-space tile.  The tile's triangles are staged in shared memory with
// their light boxes, top heights and sun-facing step bits.  Each warp then takes 32 of the
// tile's receivers at a time, one per lane, and runs over the staged triangles in step:
//   - a cheap per-pair cull (the triangle is not wholly below the receiver, and the
//     receiver's light-space point lies inside the triangle's box widened by the drift a
//     ray of the run can make before it rises to the triangle's top);
//   - the pairs that survive (a few in a hundred) are appended to a per-warp queue;
//   - whenever the queue holds 32 pairs, every lane takes one and runs the exact test, so
//     the expensive set-up is never paid by idle lanes;
//   - a receiver shadowed at every step of the run, by this chunk or by earlier ones of the
//     tile, is dropped, and a pass ends when all 32 are.
// Bound by issue (76 % of the slots busy at 36 warps per SM).  Dropping the receivers that
// are done: 300,000 points x 2000 buildings, 20 January at 2-minute steps 21.0 -> 12.0 ms;
// 100,000 points x 500 buildings, 16 December 6.80 -> 3.49; a million points in June, where
// few triangles reach a receiver, 2.01 -> 1.94.
// Results are OR-ed into per-receiver masks in shared memory, then into the block masks.
template <bool COUNT>
__global__ void __launch_bounds__(kTileThreads, SA_TILE_CTAS)
k_sam_tile(TileArgs ta) {
    __shared__ LightSmem<kTriChunk> sm;
    unsigned long long n_pair = 0, n_test = 0;
    const int tile = ta.order[blockIdx.x];
    const unsigned tcnt = ta.t_cnt[tile], rcnt = ta.r_cnt[tile];
    if (tcnt == 0 || rcnt == 0) return;
    const RunLight& rl = ta.runs[ta.tile_run[tile]];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    stage_directions(sm, ta.steps, rl);
    const bool cull = ta.sc.closed != 0;
    const unsigned full = rl.kn >= 32 ? 0xffffffffu : ((1u << rl.kn) - 1u);
    for (unsigned base = 0; base < tcnt; base += kTriChunk) {
        const int nt = (int)min((unsigned)kTriChunk, tcnt - base);
        __syncthreads();
        for (int i = threadIdx.x; i < nt; i += kTileThreads) {
            const int t = (int)SA_CHK(ta.t_bins[ta.t_off[tile] + base + i], ta.sc.T, sa::CK_POINTS_TRI);
            stage_triangle(sm, i, ta.sc.tris, t, rl, rl.c);
            sm.front[i] = run_front(sm.tri[3 * i], sm.tri[3 * i + 1], sm.tri[3 * i + 2], ta.steps, rl, cull);
        }
        __syncthreads();
        // every warp runs the same number of passes, so the loop below stays warp-uniform
        for (unsigned r0 = (unsigned)warp * 32u; r0 < rcnt; r0 += kTileThreads) {
            const unsigned i = r0 + lane;
            const bool valid = i < rcnt;
            const int s = valid ? (int)SA_CHK(ta.r_bins[ta.r_off[tile] + i], ta.R, sa::CK_POINTS_RECV) : -1;
            // the steps that earlier chunks of the tile's triangles have shadowed already
            unsigned had = 0u;
            if (valid && base > 0) had = (unsigned)(__ldcg(&ta.masks[(long long)rl.blk * ta.R + s]) >> rl.k0) & full;
            const bool live = valid && had != full;
            if (!__any_sync(0xffffffffu, live)) continue;
            const float4 p = live ? ta.orig[s] : make_float4(0.f, 0.f, 0.f, 0.f);
            sm.o[threadIdx.x] = p;
            sm.m[threadIdx.x] = had;
            float la = 0.f, lb = 0.f;
            light_ab(rl, rl.c, p.x, p.y, p.z, &la, &lb);
            light_pass(sm, rl, nt, live, p, la, lb, full, [&](const unsigned short* q, int n) {
                drain_pairs<COUNT>(sm, q, n, lane, rl.kn, n_pair, n_test);
            });
            __syncwarp();
            const unsigned m = sm.m[threadIdx.x];
            if (live && m != had) atomicOr(&ta.masks[(long long)rl.blk * ta.R + s], (unsigned long long)m << rl.k0);
            __syncwarp();
        }
    }
    if (COUNT) {
        for (int off = 16; off > 0; off >>= 1) {
            n_pair += __shfl_down_sync(0xffffffffu, n_pair, off);
            n_test += __shfl_down_sync(0xffffffffu, n_test, off);
        }
        if (lane == 0) {
            atomicAdd(&ta.stats[0], n_pair);
            atomicAdd(&ta.stats[1], n_test);
        }
    }
}

// Stitch the chunk's blocks, in order, into each receiver's gross / continuous state.
__global__ void k_points_fold(long long R, const int* __restrict__ perm,
                              const BlockConst* __restrict__ blocks, int nbc,
                              unsigned long long* __restrict__ masks, DevOut out,
                              int* __restrict__ run, int* __restrict__ best, int first, int last) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= R) return;
    const long long r = SA_CHK(perm[s], R, sa::CK_POINTS_PERM);
    RunState st{0, 0, 0};
    if (!first || out.accumulate_into) {
        st.gross = out.gross[r];
        st.best = best[r];
        st.run = first ? 0 : run[r];
    }
    for (int b = 0; b < nbc; ++b) {
        const BlockConst& bc = blocks[b];
        const unsigned long long m = masks[(long long)b * R + s];
        stitch(st, m, bc.K, bc.new_day);
        if (out.masks) out.masks[(long long)bc.mask_block * R + r] |= m;
    }
    out.gross[r] = st.gross;
    best[r] = st.best;
    run[r] = st.run;
    if (last && out.minutes) out.minutes[r] = (float)st.gross * out.step_minutes;
}

int g_point_run = 27;

}  // namespace

void set_point_run(int run) { g_point_run = run; }
int get_point_run() { return g_point_run; }

cudaError_t launch_sam_points(const DevScene& sc, const float* scene_box, const DevRecv& rc,
                              const float* recv_box, const DevSun& sun,
                              const std::vector<BlockConst>& h_blocks,
                              const std::vector<StepConst>& h_steps, const DevOut& out,
                              cudaStream_t st) {
    const long long R = rc.R;
    if (R == 0 || h_blocks.empty()) return cudaSuccess;
    const int run_len = std::max(1, std::min(kRunMax, get_point_run()));
    const float tile = SA_LIGHT_TILE;
    // blocks per chunk: the receiver bins hold every receiver once per run (4 bytes), the
    // masks 8 bytes per receiver and block; keep both within ~1 GiB and <= 64 blocks
    const int runs_per_block = (kMaxBlock + run_len - 1) / run_len;
    const long long per_block = (long long)R * (4ll * runs_per_block + 8ll);
    const int chunk = (int)std::max(1ll, std::min(64ll, (1ll << 30) / std::max(1ll, per_block)));
    const int nbc_max = std::min(chunk, (int)h_blocks.size());
    cudaError_t e = cudaSuccess;
    unsigned long long* masks = nullptr;
    int *run = nullptr, *best = nullptr;
    e = sa::scratch_alloc(&masks, sizeof(unsigned long long) * (size_t)R * nbc_max, st);
    if (e == cudaSuccess) e = sa::scratch_alloc(&run, sizeof(int) * (size_t)R, st);
    if (e == cudaSuccess && !out.continuous) e = sa::scratch_alloc(&best, sizeof(int) * (size_t)R, st);
    if (e == cudaSuccess && out.accumulate_into && !out.continuous)
        e = cudaMemsetAsync(best, 0, sizeof(int) * (size_t)R, st);
    int* bestp = out.continuous ? out.continuous : best;
    const double c[3] = {0.5 * (recv_box[0] + recv_box[3]), 0.5 * (recv_box[1] + recv_box[4]),
                         0.5 * (recv_box[2] + recv_box[5])};
    const double zmin_r = recv_box[2];
    std::vector<RunLight> hr;
    std::vector<int> tile_run;
    const int n_blocks = (int)h_blocks.size();
    // a chunk also ends once its runs hold kMaxTiles light-space tiles
    constexpr long long kMaxTiles = 1ll << 24;
    for (int b0 = 0, nbc = 0; b0 < n_blocks && e == cudaSuccess; b0 += nbc) {
        hr.clear();
        tile_run.clear();
        int tiles = 0;
        for (nbc = 0; nbc < chunk && b0 + nbc < n_blocks && (nbc == 0 || tiles < kMaxTiles); ++nbc) {
            const int bl = nbc;
            const BlockConst& bc = h_blocks[b0 + bl];
            // the block's steps in nr runs of balanced lengths (<= run_len)
            const int nr = (bc.K + run_len - 1) / run_len;
            for (int ri = 0; ri < nr; ++ri) {
                const int k0 = ri * bc.K / nr;
                RunLight rl;
                memset(&rl, 0, sizeof(rl));
                rl.k0 = k0;
                rl.kn = (ri + 1) * bc.K / nr - k0;
                rl.j0 = bc.j0;
                rl.blk = bl;
                const int j = bc.j0 + k0;
                const LightBasis lb = light_basis(h_steps[j + rl.kn / 2], h_steps[j], h_steps[j + rl.kn - 1]);
                LightStep ls = light_step(lb, h_steps[j]);
                for (int k = 1; k < rl.kn; ++k) light_merge(ls, light_step(lb, h_steps[j + k]));
                light_finish(lb, ls, &rl);
                const double *e1 = lb.e1, *e2 = lb.e2;
                rl.zr = (float)zmin_r - 0.01f;
                for (int q = 0; q < 3; ++q) rl.c[q] = (float)c[q];
                // tile grid over the light-space box of the receivers
                double amin = 1e30, amax = -1e30, bmin = 1e30, bmax = -1e30;
                for (int corner = 0; corner < 8; ++corner) {
                    const double x = (corner & 1 ? recv_box[3] : recv_box[0]) - c[0];
                    const double y = (corner & 2 ? recv_box[4] : recv_box[1]) - c[1];
                    const double z = (corner & 4 ? recv_box[5] : recv_box[2]) - c[2];
                    const double a = e1[0] * x + e1[1] * y + e1[2] * z, b = e2[0] * x + e2[1] * y + e2[2] * z;
                    amin = std::min(amin, a); amax = std::max(amax, a);
                    bmin = std::min(bmin, b); bmax = std::max(bmax, b);
                }
                double ts = tile;
                while ((amax - amin) / ts * (bmax - bmin) / ts > 4.0e6) ts *= 2.0;
                rl.tile = (float)ts;
                rl.a0 = (float)(amin - 1.0);
                rl.b0 = (float)(bmin - 1.0);
                rl.nta = std::max(1, (int)std::ceil((amax - amin + 2.0) / ts));
                rl.ntb = std::max(1, (int)std::ceil((bmax - bmin + 2.0) / ts));
                rl.tile_base = tiles;
                tiles += rl.nta * rl.ntb;
                for (int q = 0; q < rl.nta * rl.ntb; ++q) tile_run.push_back((int)hr.size());
                hr.push_back(rl);
            }
        }
        const int n_runs = (int)hr.size();
        RunLight* d_runs = nullptr;
        int* d_tile_run = nullptr;
        unsigned *tc = nullptr, *toff = nullptr, *tcur = nullptr, *rcn = nullptr, *roff = nullptr,
                 *rcur = nullptr, *d_total = nullptr, *hist = nullptr;
        int *tbins = nullptr, *rbins = nullptr, *order = nullptr;
        const size_t nt = (size_t)tiles;
#define TRYB(x) do { if (e == cudaSuccess) e = (x); } while (0)
        TRYB(cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)R * nbc, st));
        TRYB(sa::scratch_alloc(&d_runs, sizeof(RunLight) * hr.size(), st));
        TRYB(sa::scratch_alloc(&d_tile_run, sizeof(int) * nt, st));
        TRYB(sa::scratch_alloc(&tc, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&toff, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&tcur, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&rcn, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&roff, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&rcur, sizeof(unsigned) * nt, st));
        TRYB(sa::scratch_alloc(&d_total, 2 * sizeof(unsigned), st));   // bin total, tiles with work
        TRYB(sa::scratch_alloc(&hist, sizeof(unsigned) * kOrderBuckets, st));   // zeroed by the launch
        TRYB(sa::scratch_alloc(&order, sizeof(int) * nt, st));
        TRYB(sa::scratch_alloc(&rbins, sizeof(int) * (size_t)R * n_runs, st));
        TRYB(cudaMemcpyAsync(d_runs, hr.data(), sizeof(RunLight) * hr.size(), cudaMemcpyHostToDevice, st));
        TRYB(cudaMemcpyAsync(d_tile_run, tile_run.data(), sizeof(int) * nt, cudaMemcpyHostToDevice, st));
        TRYB(cudaMemsetAsync(tc, 0, sizeof(unsigned) * nt, st));
        TRYB(cudaMemsetAsync(tcur, 0, sizeof(unsigned) * nt, st));
        TRYB(cudaMemsetAsync(rcn, 0, sizeof(unsigned) * nt, st));
        TRYB(cudaMemsetAsync(rcur, 0, sizeof(unsigned) * nt, st));
        const dim3 gt((unsigned)std::max(1, (sc.T + 127) / 128), n_runs);
        const dim3 gr((unsigned)((R + 255) / 256), n_runs);
        unsigned totals[2] = {0u, 0u};
        if (e == cudaSuccess) {
            if (sc.T > 0) k_lt_bin<<<gt, 128, 0, st>>>(sc, sun.steps, d_runs, n_runs, false, tc, nullptr, nullptr, nullptr);
            k_lr_bin<<<gr, 256, 0, st>>>(rc.orig, R, d_runs, n_runs, false, rcn, nullptr, nullptr, nullptr);
            e = launch_work_order(tc, rcn, (long long)nt, hist, order, d_total + 1, st);
        }
        TRYB(cudaMemcpyAsync(toff, tc, sizeof(unsigned) * nt, cudaMemcpyDeviceToDevice, st));
        TRYB(cudaMemcpyAsync(roff, rcn, sizeof(unsigned) * nt, cudaMemcpyDeviceToDevice, st));
        TRYB(exclusive_scan_u32(roff, (long long)nt, nullptr, st));
        TRYB(exclusive_scan_u32(toff, (long long)nt, d_total, st));
        TRYB(cudaMemcpyAsync(totals, d_total, 2 * sizeof(unsigned), cudaMemcpyDeviceToHost, st));
        TRYB(cudaStreamSynchronize(st));
        const unsigned total = totals[0], work_tiles = totals[1];
        TRYB(sa::scratch_alloc(&tbins, sizeof(int) * ((size_t)total + 1), st));
        if (e == cudaSuccess) {
            if (sc.T > 0 && total > 0)
                k_lt_bin<<<gt, 128, 0, st>>>(sc, sun.steps, d_runs, n_runs, true, nullptr, toff, tcur, tbins);
            k_lr_bin<<<gr, 256, 0, st>>>(rc.orig, R, d_runs, n_runs, true, nullptr, roff, rcur, rbins);
            TileArgs ta;
            ta.sc = sc; ta.steps = sun.steps; ta.runs = d_runs; ta.n_runs = n_runs;
            ta.tile_run = d_tile_run;
            ta.order = order;
            ta.t_off = toff; ta.t_cnt = tc; ta.t_bins = tbins;
            ta.r_off = roff; ta.r_cnt = rcn; ta.r_bins = rbins;
            ta.orig = rc.orig; ta.masks = masks; ta.R = R; ta.stats = out.stats;
            if (work_tiles > 0) {
                KernelTimer kt(KT_SAM_POINTS, st);
                if (out.stats) k_sam_tile<true><<<work_tiles, kTileThreads, 0, st>>>(ta);
                else k_sam_tile<false><<<work_tiles, kTileThreads, 0, st>>>(ta);
            }
            k_points_fold<<<(unsigned)((R + 255) / 256), 256, 0, st>>>(
                R, rc.perm, sun.blocks + b0, nbc, masks, out, run, bestp, b0 == 0,
                b0 + nbc == n_blocks);
            e = cudaGetLastError();
        }
        for (void* p : {(void*)d_runs, (void*)d_tile_run, (void*)tc, (void*)toff, (void*)tcur,
                        (void*)rcn, (void*)roff, (void*)rcur, (void*)d_total, (void*)tbins, (void*)rbins,
                        (void*)hist, (void*)order})
            if (p) cudaFreeAsync(p, st);
#undef TRYB
    }
    if (masks) cudaFreeAsync(masks, st);
    if (run) cudaFreeAsync(run, st);
    if (best) cudaFreeAsync(best, st);
    return e;
}

}  // namespace sa
