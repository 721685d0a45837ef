// sa_trace.cu -- ray-traced shadow accumulation on the linear BVH.
//
//   k_sweep    plain per-step sweep: one any-hit ray per receiver and sun step (the
//              per-minute ray-tracing baseline of Sec. 8.1).
//   k_accrual  ray-traced accrual: one traversal per group of 128 receivers and run of
//              <= 27 steps, whose query is the fan of the run's rays from all of them.
//              The shadow of an occluder point sweeps a line while the sun moves (Sec.
//              3.2); seen from the receiver, the run's rays sweep a thin wedge, and only
//              geometry inside that wedge can shadow it in the run.  Each candidate
//              triangle is tested exactly, per step (Plucker form).
//   k_accrual_fan  the same with a warp's 32 receivers and whole blocks, a node entered when
//              any receiver's own wedge overlaps it: for points so few for the triangles
//              that a group's box holds far more than its rays (accrual_by_warps).
//
// The work is cut into items (TraceItems) that leave run summaries for launch_fold.
// k_sweep (an option) and k_accrual_fan are warp-coherent: the 32 lanes of a warp hold
// neighbouring receivers (an 8 x 4 patch of a ground grid or 32 consecutive points) and
// walk the depth-first node list together -- a node is entered when any lane's query
// overlaps it -- so node loads are warp-uniform broadcasts.
#include <algorithm>

#include "sa_internal.cuh"
#include "sa_light.cuh"

namespace sa {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarpsPerCta = 4;

// Morton order of point receivers for the ray-traced accrual, 16 bits in cubic cells: facade
// points come sorted by wall orientation first, which spreads a group over the city; next
// to one another their rays share nodes (1M points: 19.5 -> 6.6 ms with the sort's 0.06).
__global__ void k_regroup_keys(const float4* __restrict__ orig, long long R, float x0, float y0, float z0, float inv,
                               unsigned* __restrict__ keys, unsigned* __restrict__ vals) {
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= R) return;
    const float4 p = orig[s];
    keys[s] = morton30((p.x - x0) * inv, (p.y - y0) * inv, (p.z - z0) * inv) >> 14;
    vals[s] = (unsigned)s;
}

// 192 triangles, 60,000 points by 29 to 481 steps: 0.21 to 0.30 ms sorted, 0.15 to 0.23 as they come.
constexpr int kRegroupTris = 1000;

struct Receiver {
    float3 o;
    float tmin;
    float3 n;        // facade normal (zero for ground receivers)
    long long out;   // output index
    bool active;
};

__device__ __forceinline__ Receiver load_receiver(const DevRecv& rc, long long warp_id, int lane) {
    Receiver r;
    if (rc.is_grid) {
        const int tiles_x = (rc.nx + 7) >> 3;
        const long long ty = warp_id / tiles_x;
        const int tx = (int)(warp_id - ty * tiles_x);
        const int ix = tx * 8 + (lane & 7);
        const long long iy = ty * 4 + (lane >> 3);
        r.active = ix < rc.nx && iy < rc.ny;
        // cell centre, rounded exactly as x0 + (ix + 0.5) * dx in FP32 without contraction
        r.o.x = __fadd_rn(rc.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), rc.dx));
        r.o.y = __fadd_rn(rc.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), rc.dx));
        r.o.z = 0.f;
        r.tmin = kGroundTmin;
        r.n = make_float3(0.f, 0.f, 0.f);
        r.out = iy * rc.nx + ix;
    } else {
        long long s = warp_id * 32 + lane;
        r.active = s < rc.R;
        if (r.active && rc.order) s = SA_CHK(rc.order[s], rc.R, sa::CK_POINTS_RECV);
        const float4 p = r.active ? rc.orig[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        r.o = make_float3(p.x, p.y, p.z);
        r.tmin = p.w;
        const float4 nn = (r.active && rc.nrm) ? rc.nrm[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        r.n = make_float3(nn.x, nn.y, nn.z);
        r.out = r.active ? rc.perm[s] : 0;
    }
    return r;
}

__device__ __forceinline__ long long warp_count(const DevRecv& rc) {
    if (rc.is_grid) return (long long)((rc.nx + 7) >> 3) * ((rc.ny + 3) >> 2);
    return (rc.R + 31) / 32;
}

__device__ __forceinline__ RunState load_state(const DevOut& out, const Receiver& r) {
    RunState s{0, 0, 0};
    if (out.accumulate_into && r.active) {
        s.gross = out.gross[r.out];
        s.best = out.continuous ? out.continuous[r.out] : 0;
    }
    return s;
}

__device__ __forceinline__ void store_state(const DevOut& out, const Receiver& r,
                                            const RunState& s) {
    if (!r.active) return;
    out.gross[r.out] = s.gross;
    if (out.continuous) out.continuous[r.out] = s.best;
    if (out.minutes) out.minutes[r.out] = (float)s.gross * out.step_minutes;
}

// Few receivers over a long interval leave most of the chip idle when a warp takes every
// block of its 32 receivers in turn.  The work is then cut into items, one per warp of
// receivers, block and one of `parts` pieces of its steps, which leave run summaries
// ([blocks][parts][R]) for the fold to stitch.
struct TraceItems {
    int b0, parts;
    unsigned* summary;
};

__device__ __forceinline__ void store_item(const DevOut& out, const DevRecv& rc, const Receiver& r,
                                           const TraceItems& it, uint64_t m, int K, int mask_block,
                                           int mask_bit) {
    if (!r.active) return;
    if (it.summary) it.summary[(size_t)blockIdx.y * rc.R + r.out] = run_summary(m, K);
    if (out.masks && m)
        atomicOr(reinterpret_cast<unsigned long long*>(&out.masks[(long long)mask_block * rc.R + r.out]),
                 (unsigned long long)m << mask_bit);
}

// Warp-coherent any-hit query of one step for the whole warp.
template <int KZ, bool COUNT>
__device__ __forceinline__ bool any_hit_packet(const DevScene& sc, const float3& o, float tmin,
                                               const StepConst& s, bool want,
                                               unsigned long long& n_box,
                                               unsigned long long& n_tri) {
    bool hit = false;
    int i = 0;
    unsigned live = __ballot_sync(kFull, want);
    while (live != 0u && i < sc.n_nodes) {
        const float4 lo = __ldg(&sc.nodes[2 * i]);
        const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
        const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_TRACE_ESCAPE);
        const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_TRACE_LEAF);
        const bool in = want && !hit && hit_box(o, s.ix, s.iy, s.iz, lo, hi);
        if (COUNT && want && !hit) ++n_box;
        if (tri >= 0) {
            if (in) {
                if (COUNT) ++n_tri;
                const float4 a = __ldg(&sc.tris[3 * tri]);
                const float4 b = __ldg(&sc.tris[3 * tri + 1]);
                const float4 c = __ldg(&sc.tris[3 * tri + 2]);
                hit = hit_tri<KZ>(o, a, b, c, s.Sx, s.Sy, s.Sz, tmin);
            }
            i = esc;
            live = __ballot_sync(kFull, want && !hit);
        } else {
            i = __any_sync(kFull, in) ? i + 1 : esc;
        }
    }
    return hit;
}

__device__ __forceinline__ void flush_counts(const DevOut& out, unsigned long long n_box,
                                             unsigned long long n_tri) {
    for (int o = 16; o > 0; o >>= 1) {
        n_box += __shfl_down_sync(kFull, n_box, o);
        n_tri += __shfl_down_sync(kFull, n_tri, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&out.stats[0], n_box);
        atomicAdd(&out.stats[1], n_tri);
    }
}

template <bool COUNT>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_sweep(DevScene sc, DevRecv rc, DevSun sun, DevOut out) {
    unsigned long long n_box = 0, n_tri = 0;
    const int lane = threadIdx.x & 31;
    const long long warp_id = (long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (warp_id >= warp_count(rc)) return;
    const Receiver r = load_receiver(rc, warp_id, lane);
    RunState st = load_state(out, r);
    for (int b = 0; b < sun.n_blocks; ++b) {
        const int j0 = sun.blocks[b].j0, K = sun.blocks[b].K;
        uint64_t m = 0;
        for (int k = 0; k < K; ++k) {
            const StepConst s = sun.steps[j0 + k];
            bool h;
            if (s.kz == 2) h = any_hit_packet<2, COUNT>(sc, r.o, r.tmin, s, r.active, n_box, n_tri);
            else if (s.kz == 0) h = any_hit_packet<0, COUNT>(sc, r.o, r.tmin, s, r.active, n_box, n_tri);
            else h = any_hit_packet<1, COUNT>(sc, r.o, r.tmin, s, r.active, n_box, n_tri);
            if (h) m |= 1ull << k;
        }
        stitch(st, m, K, sun.blocks[b].new_day);
        if (out.masks && r.active)
            out.masks[(long long)sun.blocks[b].mask_block * rc.R + r.out] |= m << sun.blocks[b].mask_bit;
    }
    store_state(out, r, st);
    if (COUNT) flush_counts(out, n_box, n_tri);
}

// ------------------------------------------------------------------- accrual trace
constexpr int kAccrualRun = 27;   // steps per run, at the most (<= kRunMax)

__global__ void k_run_lights(const StepConst* __restrict__ steps, const BlockConst* __restrict__ blocks, int n,
                             int parts, RunLight* __restrict__ runs) {
    const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;                                              // whole warps
    const BlockConst& bc = blocks[i / parts];
    const int part = i % parts;
    const int k0 = part * bc.K / parts, kn = (part + 1) * bc.K / parts - k0, j = bc.j0 + k0;
    RunLight* rl = &runs[i];
    if (kn > 0) {
        const LightBasis L = light_basis(steps[j + kn / 2], steps[j], steps[j + kn - 1]);
        LightStep s = light_step(L, steps[j + min(lane, kn - 1)]);
        for (int o = 16; o > 0; o >>= 1) {
            LightStep t;
            t.da_lo = __shfl_xor_sync(kFull, s.da_lo, o); t.da_hi = __shfl_xor_sync(kFull, s.da_hi, o);
            t.db_lo = __shfl_xor_sync(kFull, s.db_lo, o); t.db_hi = __shfl_xor_sync(kFull, s.db_hi, o);
            for (int q = 0; q < 3; ++q) t.mx[q] = __shfl_xor_sync(kFull, s.mx[q], o);
            light_merge(s, t);
        }
        if (lane == 0) light_finish(L, s, rl);
    }
    if (lane == 0) {
        rl->k0 = k0;
        rl->kn = kn;
        rl->j0 = bc.j0;
        rl->blk = i / parts;
    }
}

// Receiver of a thread: 128 Morton-consecutive points, or a 16 x 8 patch of a ground grid
// (an 8 x 4 patch per warp).
__device__ __forceinline__ Receiver load_group_receiver(const DevRecv& rc, long long group) {
    if (!rc.is_grid) return load_receiver(rc, group * (kTileThreads / 32) + (threadIdx.x >> 5), threadIdx.x & 31);
    Receiver r;
    const int gx = (rc.nx + 15) >> 4, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long gy = group / gx;
    const int ix = (int)(group - gy * gx) * 16 + (warp & 1) * 8 + (lane & 7);
    const long long iy = gy * 8 + (warp >> 1) * 4 + (lane >> 3);
    r.active = ix < rc.nx && iy < rc.ny;
    r.o.x = __fadd_rn(rc.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), rc.dx));
    r.o.y = __fadd_rn(rc.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), rc.dx));
    r.o.z = 0.f;
    r.tmin = kGroundTmin;
    r.n = make_float3(0.f, 0.f, 0.f);
    r.out = iy * rc.nx + ix;
    return r;
}

// Ray-traced accrual of one run of steps for 128 neighbouring receivers: the CTA walks the
// BVH once for all of them (walk_group), and each warp culls and tests the pairs of its
// receivers with the leaves' triangles, exactly and per step, as the light-space map does;
// a group shadowed at every step stops.  Bound by issue in the pair culls and tests.  The
// traversal by one warp's 32 fans (k_accrual_fan, 80 instructions a node for every warp of
// receivers and block in series) took 3.43 ms on 517 x 389 cells x 481 steps, 2.35 ms as
// items; the grouped one 0.76 ms.  1024^2 cells: 13.8 -> 4.03 ms; 1M facade points: 16.5 ->
// 6.7 ms.
template <bool COUNT>
__global__ void __launch_bounds__(kTileThreads, 8)
k_accrual(DevScene sc, DevRecv rc, DevSun sun, DevOut out, TraceItems it, const RunLight* __restrict__ runs) {
    __shared__ LightSmem<kTriChunk> sm;
    __shared__ GroupSmem<kTriChunk, 1024> gs;
    unsigned long long n_box = 0, n_pair = 0, n_test = 0;
    const int tid = threadIdx.x, lane = tid & 31;
    const RunLight& rl = runs[blockIdx.y];
    const BlockConst& bc = sun.blocks[it.b0 + (int)blockIdx.y / it.parts];
    const Receiver r = load_group_receiver(rc, blockIdx.x);
    const int kn = rl.kn;
    const unsigned full = kn >= 32 ? 0xffffffffu : ((1u << kn) - 1u);
    sm.m[tid] = 0u;
    if (kn > 0) {
        const float4 p = make_float4(r.o.x, r.o.y, r.o.z, r.tmin);
        sm.o[tid] = p;
        stage_directions(sm, sun.steps, rl);
        walk_group<COUNT>(sm, gs, sc, rl, r.active, p, [full](int) { return full; }, n_box, [&](int nt, float la, float lb) {
            light_pass(sm, rl, nt, r.active && sm.m[tid] != full, p, la, lb, full, [&](const unsigned short* q, int n) {
                drain_pairs<COUNT>(sm, q, n, lane, kn, n_pair, n_test);
            });
            __syncwarp();
            return !r.active || sm.m[tid] == full;
        });
    }
    store_item(out, rc, r, it, sm.m[tid], kn, bc.mask_block, bc.mask_bit + rl.k0);
    if (COUNT) flush_counts(out, n_box, n_test);
}

// ------------------------------------------------------------ per-lane traversal
// Watertight test with the major axis chosen at run time (component selects instead of
// the template), so lanes of a warp can test different steps at once.
__device__ __forceinline__ float pick(const float4& v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }
__device__ __forceinline__ float pick3(const float3& v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }

__device__ __forceinline__ bool hit_tri_rt(const float3& o, const float4& a, const float4& b,
                                           const float4& c, const StepConst& s, float tmin) {
    const int kz = s.kz, kx = kz == 2 ? 0 : kz + 1, ky = kz == 0 ? 2 : kz - 1;
    const float oz = pick3(o, kz), ox = pick3(o, kx), oy = pick3(o, ky);
    const float az = pick(a, kz) - oz, bz = pick(b, kz) - oz, cz = pick(c, kz) - oz;
    const float ax = fmaf(-s.Sx, az, pick(a, kx) - ox), ay = fmaf(-s.Sy, az, pick(a, ky) - oy);
    const float bx = fmaf(-s.Sx, bz, pick(b, kx) - ox), by = fmaf(-s.Sy, bz, pick(b, ky) - oy);
    const float cx = fmaf(-s.Sx, cz, pick(c, kx) - ox), cy = fmaf(-s.Sy, cz, pick(c, ky) - oy);
    const float U = __fsub_rn(__fmul_rn(cx, by), __fmul_rn(cy, bx));
    const float V = __fsub_rn(__fmul_rn(ax, cy), __fmul_rn(ay, cx));
    const float W = __fsub_rn(__fmul_rn(bx, ay), __fmul_rn(by, ax));
    if ((U < 0.f || V < 0.f || W < 0.f) && (U > 0.f || V > 0.f || W > 0.f)) return false;
    const float det = U + V + W;
    if (det == 0.f) return false;
    const float T = U * (s.Sz * az) + V * (s.Sz * bz) + W * (s.Sz * cz);
    return det > 0.f ? (T > tmin * det) : (T < tmin * det);
}

template <bool COUNT>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_accrual_fan(DevScene sc, DevRecv rc, DevSun sun, DevOut out, TraceItems it) {
    // block and step constants are copied per warp, so warps never wait for one another
    __shared__ BlockConst s_bc[kWarpsPerCta];
    __shared__ StepConst s_st[kWarpsPerCta][kMaxBlock];
    unsigned long long n_box = 0, n_tri = 0;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long warp_id = (long long)blockIdx.x * kWarpsPerCta + wib;
    if (warp_id >= warp_count(rc)) return;
    const Receiver r = load_receiver(rc, warp_id, lane);
    BlockConst& bc = s_bc[wib];
    StepConst* ss = s_st[wib];
    __syncwarp();
    for (int w = lane; w < (int)(sizeof(BlockConst) / 4); w += 32)
        reinterpret_cast<int*>(&bc)[w] = reinterpret_cast<const int*>(&sun.blocks[it.b0 + blockIdx.y])[w];
    __syncwarp();
    {
        const int K = bc.K;
        for (int w = lane; w < K * (int)(sizeof(StepConst) / 4); w += 32)
            reinterpret_cast<int*>(ss)[w] = reinterpret_cast<const int*>(&sun.steps[bc.j0])[w];
        __syncwarp();
        const uint64_t full = (K >= 64) ? ~0ull : ((1ull << K) - 1ull);
        uint64_t m = 0;
        const bool wedge = bc.wedge_ok != 0.f;
        // lower bound of n . d over the block's direction box
        const float nd_lo = fminf(r.n.x * bc.dlo[0], r.n.x * bc.dhi[0]) +
                            fminf(r.n.y * bc.dlo[1], r.n.y * bc.dhi[1]) +
                            fminf(r.n.z * bc.dlo[2], r.n.z * bc.dhi[2]);
        const bool front = nd_lo > 1e-6f;
        int i = 0;
        unsigned live = __ballot_sync(kFull, r.active && m != full);
        while (live != 0u && i < sc.n_nodes) {
            const float4 lo = __ldg(&sc.nodes[2 * i]);
            const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
            const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_TRACE_ESCAPE);
            const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_TRACE_LEAF);
            const bool want = r.active && m != full;
            const bool in = want && (wedge ? fan_box(r.o, bc, lo, hi, front, r.n) : slope_box(r.o, bc, lo, hi));
            if (COUNT && want) ++n_box;
            if (tri >= 0) {
                int ka = K, kb = -1;
                float4 ta, tb, tc;
                if (in) {
                    ta = __ldg(&sc.tris[3 * tri]);
                    tb = __ldg(&sc.tris[3 * tri + 1]);
                    tc = __ldg(&sc.tris[3 * tri + 2]);
                    if (plane_reachable(r.o, ta, tb, tc, bc))
                        candidate_steps(r.o, bc, bc.psi, ta, tb, tc, &ka, &kb);
                }
                const int wa = __reduce_min_sync(kFull, ka);
                const int wb = __reduce_max_sync(kFull, kb);
                if (wa <= wb) {
                    PluckerTri pt;
                    if (ka <= kb) pt = plucker_setup(r.o, ta, tb, tc);
                    for (int k = wa; k <= wb; ++k) {
                        const bool test = k >= ka && k <= kb && !((m >> k) & 1ull);
                        if (test) {
                            if (COUNT) ++n_tri;
                            if (plucker_hit(pt, ss[k].dx, ss[k].dy, ss[k].dz, r.tmin)) {
                                m |= 1ull << k;
                            }
                        }
                    }
                }
                i = esc;
                live = __ballot_sync(kFull, r.active && m != full);
            } else {
                i = __any_sync(kFull, in) ? i + 1 : esc;
            }
        }
        store_item(out, rc, r, it, m, K, bc.mask_block, bc.mask_bit);
    }
    if (COUNT) flush_counts(out, n_box, n_tri);
}

// Ray-traced accrual with one independent traversal per lane ("while-while": each lane
// descends internal nodes until it reaches a leaf its fan overlaps, then the lanes process
// their leaves together).  Block and step constants are copied per warp into shared
// memory, so warps of a CTA never wait for one another.
template <bool COUNT>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_accrual_lane(DevScene sc, DevRecv rc, DevSun sun, DevOut out) {
    __shared__ BlockConst s_bc[kWarpsPerCta];
    __shared__ StepConst s_st[kWarpsPerCta][kMaxBlock];
    unsigned long long n_box = 0, n_tri = 0;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long warp_id = (long long)blockIdx.x * kWarpsPerCta + wib;
    if (warp_id >= warp_count(rc)) return;
    const Receiver r = load_receiver(rc, warp_id, lane);
    RunState st = load_state(out, r);
    BlockConst& bc = s_bc[wib];
    StepConst* ss = s_st[wib];
    for (int b = 0; b < sun.n_blocks; ++b) {
        __syncwarp();
        for (int w = lane; w < (int)(sizeof(BlockConst) / 4); w += 32)
            reinterpret_cast<int*>(&bc)[w] = reinterpret_cast<const int*>(&sun.blocks[b])[w];
        __syncwarp();
        const int K = bc.K;
        for (int w = lane; w < K * (int)(sizeof(StepConst) / 4); w += 32)
            reinterpret_cast<int*>(ss)[w] = reinterpret_cast<const int*>(&sun.steps[bc.j0])[w];
        __syncwarp();
        const uint64_t full = (K >= 64) ? ~0ull : ((1ull << K) - 1ull);
        const bool wedge = bc.wedge_ok != 0.f;
        uint64_t m = 0;
        int i = r.active ? 0 : sc.n_nodes;
        while (i < sc.n_nodes && m != full) {
            int tri = -1;
            float4 lo, hi;
            while (i < sc.n_nodes) {
                lo = __ldg(&sc.nodes[2 * i]);
                hi = __ldg(&sc.nodes[2 * i + 1]);
                const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_TRACE_ESCAPE);
                const bool in = wedge ? fan_box(r.o, bc, lo, hi) : slope_box(r.o, bc, lo, hi);
                if (COUNT) ++n_box;
                if (!in) { i = esc; continue; }
                tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_TRACE_LEAF);
                if (tri >= 0) { i = esc; break; }
                i = i + 1;
            }
            if (tri < 0) break;
            const float4 ta = __ldg(&sc.tris[3 * tri]);
            const float4 tb = __ldg(&sc.tris[3 * tri + 1]);
            const float4 tc = __ldg(&sc.tris[3 * tri + 2]);
            int ka = 0, kb = -1;
            if (plane_reachable(r.o, ta, tb, tc, bc)) candidate_steps(r.o, bc, bc.psi, ta, tb, tc, &ka, &kb);
            for (int k = ka; k <= kb; ++k) {
                if ((m >> k) & 1ull) continue;
                if (COUNT) ++n_tri;
                if (hit_tri_rt(r.o, ta, tb, tc, ss[k], r.tmin)) m |= 1ull << k;
            }
        }
        stitch(st, m, K, bc.new_day);
        if (out.masks && r.active) out.masks[(long long)bc.mask_block * rc.R + r.out] |= m << bc.mask_bit;
    }
    store_state(out, r, st);
    if (COUNT) flush_counts(out, n_box, n_tri);
}

// Per-step sweep with one independent traversal per lane, an item per warp.
template <bool COUNT>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_sweep_lane(DevScene sc, DevRecv rc, DevSun sun, DevOut out, TraceItems it) {
    unsigned long long n_box = 0, n_tri = 0;
    const int lane = threadIdx.x & 31;
    const long long warp_id = (long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (warp_id >= warp_count(rc)) return;
    const Receiver r = load_receiver(rc, warp_id, lane);
    const BlockConst& bc = sun.blocks[it.b0 + (int)blockIdx.y / it.parts];
    const int part = (int)blockIdx.y % it.parts;
    const int k0 = part * bc.K / it.parts, K = (part + 1) * bc.K / it.parts - k0;
    const int j0 = bc.j0 + k0;
    uint64_t m = 0;
    for (int k = 0; k < K; ++k) {
        const StepConst s = sun.steps[j0 + k];
        bool hit = false;
        int i = r.active ? 0 : sc.n_nodes;
        while (i < sc.n_nodes && !hit) {
            const float4 lo = __ldg(&sc.nodes[2 * i]);
            const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
            const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_TRACE_ESCAPE);
            const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_TRACE_LEAF);
            if (COUNT) ++n_box;
            if (!hit_box(r.o, s.ix, s.iy, s.iz, lo, hi)) { i = esc; continue; }
            if (tri < 0) { i = i + 1; continue; }
            if (COUNT) ++n_tri;
            hit = hit_tri_rt(r.o, __ldg(&sc.tris[3 * tri]), __ldg(&sc.tris[3 * tri + 1]),
                             __ldg(&sc.tris[3 * tri + 2]), s, r.tmin);
            i = esc;
        }
        if (hit) m |= 1ull << k;
    }
    store_item(out, rc, r, it, m, K, bc.mask_block, bc.mask_bit + k0);
    if (COUNT) flush_counts(out, n_box, n_tri);
}

long long host_warps(const DevRecv& rc) {
    if (rc.is_grid) return (long long)((rc.nx + 7) / 8) * ((rc.ny + 3) / 4);
    return (rc.R + 31) / 32;
}

}  // namespace

// Traversal mode: 1 = warp-coherent (packet), 2 = per lane, 0 = the measured default: per lane
// for the per-step sweep (single rays: lanes rarely wait on each other); for the accrual a
// walk per group of 128 receivers, or the packet's for thin point sets (launch_accrual_trace).
int g_trace_mode[2] = {0, 0};   // [0] sweep, [1] accrual

static bool use_lane(int which, const DevRecv& rc) {
    const int mode = g_trace_mode[which];
    (void)rc;
    return mode == 2 || (mode == 0 && which == 0);
}

// Runs launch(items, grid.y) over every block in chunks whose summaries fit 1 GiB (and the
// memory there is), folding each chunk into the receivers' state.  Without memory for one
// block's summaries nothing has been launched.
template <class Launch>
static cudaError_t by_items(const DevRecv& rc, const DevSun& sun, const DevOut& out, int parts, cudaStream_t st,
                            Launch launch) {
    const long long R = rc.R;
    int chunk = (int)std::max(1ll, std::min({(long long)sun.n_blocks, 65535ll / parts, (1ll << 30) / (4ll * parts * R)}));
    unsigned* summary = nullptr;
    int *run = nullptr, *best = out.continuous, *best_scratch = nullptr;
    cudaError_t e = sa::scratch_alloc(&run, sizeof(int) * (size_t)R, st);
    if (e == cudaSuccess && !best) {
        e = sa::scratch_alloc(&best_scratch, sizeof(int) * (size_t)R, st);
        best = best_scratch;
        if (e == cudaSuccess && out.accumulate_into) e = cudaMemsetAsync(best, 0, sizeof(int) * (size_t)R, st);
    }
    if (e == cudaSuccess)
        e = sa::scratch_alloc_blocks(&summary, sizeof(unsigned) * (size_t)parts * (size_t)R, &chunk, st);
    if (e == cudaSuccess && out.accumulate_into) e = cudaMemsetAsync(run, 0, sizeof(int) * (size_t)R, st);
    DevOut o = out;
    o.run = run;
    for (int b0 = 0; b0 < sun.n_blocks && e == cudaSuccess; b0 += chunk) {
        const int nbc = std::min(chunk, sun.n_blocks - b0);
        e = launch(TraceItems{b0, parts, summary}, (unsigned)(nbc * parts));
        if (e != cudaSuccess) break;
        launch_fold(summary, R, sun.blocks + b0, nbc, parts, o, best, b0 > 0 || out.accumulate_into,
                    b0 + nbc >= sun.n_blocks, st);
        e = cudaGetLastError();
    }
    for (void* p : {(void*)summary, (void*)run, (void*)best_scratch})
        if (p) cudaFreeAsync(p, st);
    return e;
}

// Pieces of a sweep's blocks: 16 of an hour's 60 steps (4 each) where the warps are few, 4
// from 311,296 items up, never more than a block has steps on average.  64^2 cells, 241
// steps: 1,124 us with the blocks in series, 298 in one piece each, 72 in 16; 300^2 cells:
// 5.34 -> 2.41 ms in 15; 1000 x 800 cells: 11.7 -> 10.7 ms in 4, 10.9 in 15.
static int trace_parts(long long warps, const DevSun& sun) {
    const long long items = warps * sun.n_blocks, fill = 152ll * 2048;
    const long long p = std::max(4ll, std::min(16ll, (fill + items - 1) / items));
    return (int)std::max(1ll, std::min(p, (long long)sun.S / sun.n_blocks));
}

cudaError_t launch_sweep_trace(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                               const DevOut& out, cudaStream_t st) {
    const long long warps = host_warps(rc);
    if (warps == 0) return cudaSuccess;
    const unsigned ctas = (unsigned)((warps + kWarpsPerCta - 1) / kWarpsPerCta);
    const int T = 32 * kWarpsPerCta;
    KernelTimer kt(KT_SWEEP, st);
    if (use_lane(0, rc)) {
        const int parts = trace_parts(warps, sun);
        const cudaError_t e = by_items(rc, sun, out, parts, st, [&](const TraceItems& it, unsigned ny) {
            if (out.stats) k_sweep_lane<true><<<dim3(ctas, ny), T, 0, st>>>(sc, rc, sun, out, it);
            else k_sweep_lane<false><<<dim3(ctas, ny), T, 0, st>>>(sc, rc, sun, out, it);
            return cudaGetLastError();
        });
        if (e != cudaErrorMemoryAllocation) return e;      // else the walk that needs no memory
    }
    if (out.stats) k_sweep<true><<<ctas, T, 0, st>>>(sc, rc, sun, out);
    else k_sweep<false><<<ctas, T, 0, st>>>(sc, rc, sun, out);
    return cudaGetLastError();
}

cudaError_t launch_run_lights(const StepConst* steps, const BlockConst* blocks, int n_blocks, int parts,
                              RunLight* runs, cudaStream_t st) {
    const int n = n_blocks * parts;
    if (n > 0) k_run_lights<<<(n + 3) / 4, 128, 0, st>>>(steps, blocks, n, parts, runs);
    return cudaGetLastError();
}

// Whether point receivers walk by warps, each with its own fan, rather than by groups.  A
// group's box must not hold far more than its rays do, and where 128 consecutive points
// straddle a bisection of the plan it holds a good part of the scene: that group's CTA
// takes time in proportion to the scene, 80 to 120 us per 1,000 triangles whatever the
// points, while the walks by warps take about as much per point and block.  So points that
// are few for the triangles go by warps, unless the sun is low (long fans: their cost grows
// with the slope), the scene small, the blocks many (a group's cost grows less with them,
// and less still where each spans hours) or a block's rays too far apart for a wedge.
// Points spread over the scene, ms by warps / by groups, 481 steps in June if not said:
// 122k triangles, 32k points 5.0 / 14, 147k 14 / 17, 294k 24 / 19; 365k, 95k 13 / 46; 2,340,
// 600 1.4 / 0.4; 122k and 73k points: 29 steps 3.7 / 12, 7 days of 2 minutes 32 / 34, 30
// days of 10 minutes 92 / 42, March to a slope of 4.9 11 / 16, February to 23 26 / 18,
// December 57 / 28.  Where the two are close the line errs to the warps.
static bool accrual_by_warps(const DevScene& sc, const float* box, const DevRecv& rc, const float* recv_box,
                             const DevSun& sun) {
    if (g_trace_mode[1] == 1) return true;
    if (rc.is_grid || !sun.thin) return false;
    // the scene's triangles under the points' plan
    auto area = [](const float* b) { return ((double)b[3] - b[0]) * ((double)b[4] - b[1]); };
    const double share = area(box) > 0.0 ? std::min(1.0, area(recv_box) / area(box)) : 1.0;
    const double slope = std::max(2.0, (double)sun.max_slope);
    double f = 9.0 / sun.n_blocks;
    if (f < 1.0) f *= std::min(1.0, 0.5 / std::max(1e-3, (double)sun.max_angle));
    if (slope > 5.0) f = std::min(1.0, f) * 5.0 / slope;
    return (double)rc.R < 2.2 * f * (share * sc.T - 6000.0 * slope);
}

int drift_parts(const BlockConst& b, const std::vector<StepConst>& steps, int parts, int most, double limit) {
    // the drift is the ground slopes' spread, foreshortened: no side passes their box's diagonal
    const double ux = (double)b.uxhi - b.uxlo, uy = (double)b.uyhi - b.uylo;
    if (ux * ux + uy * uy <= limit) return parts;
    const int base = parts;
    while (parts < most) {
        bool wide = false;
        for (int q = 0; q < parts && !wide; ++q) {
            const int k0 = q * b.K / parts, kn = (q + 1) * b.K / parts - k0, j = b.j0 + k0;
            if (kn < 2) continue;
            const LightBasis L = light_basis(steps[(size_t)(j + kn / 2)], steps[(size_t)j], steps[(size_t)(j + kn - 1)]);
            LightStep s = light_drift(L, steps[(size_t)j]);
            for (int k = 1; k < kn; ++k) light_merge(s, light_drift(L, steps[(size_t)(j + k)]));
            wide = (s.da_hi - s.da_lo) * (s.db_hi - s.db_lo) > limit;
        }
        if (!wide) break;
        parts += base;
    }
    return std::min(parts, most);
}

// A run's box is widened by its rays' drift, so a run whose rays spread far -- a low sun, or
// hours between its first step and last -- reaches most of a city, and its groups work for
// all of it: shorter runs then, by the largest drift box of any (area per square metre of
// rise; 0.02 of a June day's 27-minute runs, 9 of a December day's, 225 where a 2-hour run
// takes in sunrise).  400^2 cells at 0.5 m over 61,676 triangles, ms for a largest box of
// 225 / 50 / 9 / 1.8: 26 / 6.7 / 1.4 / 0.93; 15 minutes a step until sunset 19 / 6.6 / 2 / 0.5: 7.8 /
// 3.1 / 1.4 / 0.67; December 9 / 2.4 / 0.7 / 0.2: 4.1 / 2.3 / 2.9 / 4.9.  The groups of points are
// wide themselves (60,000 facade points: December 7.5 / 10 / 15 / 25, sunrise 18 / 8.7 / 6.1 /
// 6.3).
constexpr double kDriftGrid = 4.0, kDriftPoints = 12.0;

cudaError_t launch_accrual_trace(const DevScene& sc, const float* scene_box, const DevRecv& rc, const float* recv_box,
                                 const DevSun& sun, const std::vector<BlockConst>& h_blocks,
                                 const std::vector<StepConst>& h_steps, const DevOut& out, cudaStream_t st) {
    const long long warps = host_warps(rc);
    if (warps == 0) return cudaSuccess;
    const unsigned ctas = (unsigned)((warps + kWarpsPerCta - 1) / kWarpsPerCta);
    const int T = 32 * kWarpsPerCta;
    KernelTimer kt(KT_ACCRUAL, st);
    if (use_lane(1, rc)) {
        if (out.stats) k_accrual_lane<true><<<ctas, T, 0, st>>>(sc, rc, sun, out);
        else k_accrual_lane<false><<<ctas, T, 0, st>>>(sc, rc, sun, out);
    } else {
        DevRecv rg = rc;
        unsigned *keys = nullptr, *order = nullptr;
        cudaError_t e = cudaSuccess;
        // (a small scene's few triangles are all staged by any group)
        if (!rc.is_grid && rc.nrm && sc.T >= kRegroupTris) {
            e = sa::scratch_alloc(&keys, sizeof(unsigned) * (size_t)rc.R, st);
            if (e == cudaSuccess) e = sa::scratch_alloc(&order, sizeof(unsigned) * (size_t)rc.R, st);
            const float ext = std::max({recv_box[3] - recv_box[0], recv_box[4] - recv_box[1], recv_box[5] - recv_box[2]});
            if (e == cudaSuccess)
                k_regroup_keys<<<(unsigned)((rc.R + 255) / 256), 256, 0, st>>>(
                    rc.orig, rc.R, recv_box[0], recv_box[1], recv_box[2], ext > 0.f ? 1.f / ext : 0.f, keys, order);
            if (e == cudaSuccess) e = radix_sort_pairs(keys, order, rc.R, st, 16);
            if (e == cudaSuccess) rg.order = order;
            if (e == cudaErrorMemoryAllocation) e = cudaSuccess;      // the points in their own order
        }
        if (e == cudaSuccess && accrual_by_warps(sc, scene_box, rc, recv_box, sun)) {
            e = by_items(rg, sun, out, 1, st, [&](const TraceItems& it, unsigned ny) {
                if (out.stats) k_accrual_fan<true><<<dim3(ctas, ny), T, 0, st>>>(sc, rg, sun, out, it);
                else k_accrual_fan<false><<<dim3(ctas, ny), T, 0, st>>>(sc, rg, sun, out, it);
                return cudaGetLastError();
            });
        } else if (e == cudaSuccess) {
            // runs of balanced lengths: every block in as many pieces as any needs
            const int base = (sun.max_K + kAccrualRun - 1) / kAccrualRun;
            int parts = base;
            for (const BlockConst& b : h_blocks)
                parts = std::max(parts, drift_parts(b, h_steps, base, std::min(16 * base, sun.max_K),
                                                    rc.is_grid ? kDriftGrid : kDriftPoints));
            const unsigned groups = (unsigned)(rc.is_grid ? (long long)((rc.nx + 15) / 16) * ((rc.ny + 7) / 8)
                                                          : (rc.R + kTileThreads - 1) / kTileThreads);
            RunLight* runs = nullptr;
            e = sa::scratch_alloc(&runs, sizeof(RunLight) * (size_t)sun.n_blocks * parts, st);
            if (e == cudaSuccess)
                e = by_items(rg, sun, out, parts, st, [&](const TraceItems& it, unsigned ny) {
                    const cudaError_t el = launch_run_lights(sun.steps, sun.blocks + it.b0, (int)ny / parts, parts, runs, st);
                    if (el != cudaSuccess) return el;
                    if (out.stats) k_accrual<true><<<dim3(groups, ny), kTileThreads, 0, st>>>(sc, rg, sun, out, it, runs);
                    else k_accrual<false><<<dim3(groups, ny), kTileThreads, 0, st>>>(sc, rg, sun, out, it, runs);
                    return cudaGetLastError();
                });
            if (runs) cudaFreeAsync(runs, st);
        }
        if (keys) cudaFreeAsync(keys, st);
        if (order) cudaFreeAsync(order, st);
        return e;
    }
    return cudaGetLastError();
}

void set_trace_mode(int which, int mode) { g_trace_mode[which] = mode; }
int get_trace_mode(int which) { return g_trace_mode[which]; }

}  // namespace sa
