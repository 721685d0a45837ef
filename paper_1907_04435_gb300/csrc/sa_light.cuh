// sa_light.cuh -- the light-space map of a run of steps (Sec. 4): a CTA's triangles staged with
// their light boxes, edge lines and distance bounds, the culls of (receiver, triangle)
// pairs, and the exact test of the pairs that survive.  Shared by the map of point
// receivers (triangles from light-space bins) and the ray-traced accrual (triangles from a
// traversal of the BVH with the fan of the run's rays).
#pragma once

#include <math.h>

#include "sa_internal.cuh"

namespace sa {

constexpr int kRunMax = 32;
constexpr float kLightSlack = 0.05f;    // absolute slack (m) of the light-space culls (rounding)
// threads per CTA, one receiver each (a multiple of 32), and triangles staged per chunk (<= 256)
#ifndef SA_TILE_THREADS
#define SA_TILE_THREADS 128
#endif
#ifndef SA_TILE_CHUNK
#define SA_TILE_CHUNK 128
#endif
constexpr int kTileThreads = SA_TILE_THREADS;
constexpr int kTriChunk = SA_TILE_CHUNK;
constexpr int kQueue = 64;

struct RunLight {
    float e1[3], e2[3];          // light-space basis (orthogonal to the run's middle direction)
    float c[3];                  // reference point
    float a0, b0, tile;          // tile grid origin and tile side (m)
    float zr;                    // lowest receiver height
    int nta, ntb;                // tiles along e1, e2
    int tile_base;               // first global tile index of this run
    int k0, kn;                  // steps of the run within the block
    int j0;                      // first step of the block
    int blk;                     // block within the chunk (row of the chunk's masks)
    // light-space drift per metre of height over the run's steps, as the margins it
    // implies on each side: a ray point at height h above the receiver lies within
    // [-h da_hi, h da_lo] of it along e1 and [-h db_hi, h db_lo] along e2 (all >= 0)
    float da_hi, da_lo, db_hi, db_lo;
    // every step direction of the run is d_m + alpha t + beta b + nu n (t, b, n: an FP32
    // basis around d_m), with |alpha| <= ba, |beta| <= bb, |nu| <= bn
    float dm[3], tv[3], bv[3], ba, bb, bn;
};

// light-space coordinates relative to the reference point c
__device__ __forceinline__ void light_ab(const RunLight& rl, const float* c, float x, float y, float z,
                                         float* a, float* b) {
    const float dx = x - c[0], dy = y - c[1], dz = z - c[2];
    *a = rl.e1[0] * dx + rl.e1[1] * dy + rl.e1[2] * dz;
    *b = rl.e2[0] * dx + rl.e2[1] * dy + rl.e2[2] * dz;
}

// Light-space basis of a run and an FP32 orthonormal basis around its middle direction d_m (as
// stored, FP32): t along the run's motion, b = n x t, n = d_m / |d_m|.
struct LightBasis {
    double e1[3], e2[3];
    float dm[3], t[3], b[3], n[3];
};

__host__ __device__ inline void light_normalize(double* v) {
    const double n = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    v[0] /= n; v[1] /= n; v[2] /= n;
}

__host__ __device__ inline double light_det(const double A[3][3]) {
    return A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) -
           A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
           A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
}

__host__ __device__ inline LightBasis light_basis(const StepConst& mid, const StepConst& first, const StepConst& last) {
    LightBasis L;
    double dm[3] = {mid.dx, mid.dy, mid.dz};
    light_normalize(dm);
    L.e1[0] = dm[1]; L.e1[1] = -dm[0]; L.e1[2] = 0.0;            // horizontal, orthogonal to dm
    if (L.e1[0] * L.e1[0] + L.e1[1] * L.e1[1] < 1e-12) { L.e1[0] = 1.0; L.e1[1] = 0.0; }
    light_normalize(L.e1);
    L.e2[0] = dm[1] * L.e1[2] - dm[2] * L.e1[1];
    L.e2[1] = dm[2] * L.e1[0] - dm[0] * L.e1[2];
    L.e2[2] = dm[0] * L.e1[1] - dm[1] * L.e1[0];
    light_normalize(L.e2);
    double t3[3] = {(double)last.dx - first.dx, (double)last.dy - first.dy, (double)last.dz - first.dz};
    const double tn = t3[0] * dm[0] + t3[1] * dm[1] + t3[2] * dm[2];
    for (int q = 0; q < 3; ++q) t3[q] -= tn * dm[q];
    if (t3[0] * t3[0] + t3[1] * t3[1] + t3[2] * t3[2] < 1e-24)
        for (int q = 0; q < 3; ++q) t3[q] = L.e1[q];
    light_normalize(t3);
    double b3[3] = {dm[1] * t3[2] - dm[2] * t3[1], dm[2] * t3[0] - dm[0] * t3[2], dm[0] * t3[1] - dm[1] * t3[0]};
    light_normalize(b3);
    L.dm[0] = mid.dx; L.dm[1] = mid.dy; L.dm[2] = mid.dz;
    for (int q = 0; q < 3; ++q) {
        L.t[q] = (float)t3[q];
        L.b[q] = (float)b3[q];
        L.n[q] = (float)dm[q];
    }
    return L;
}

// One step's share of a run's bounds: its drift per metre of height in light space, and the
// |coefficients| of d - d_m in the FP32 basis (Cramer's rule); light_drift: the drift alone.
struct LightStep {
    double da_lo, da_hi, db_lo, db_hi, mx[3];
};

__host__ __device__ inline LightStep light_drift(const LightBasis& L, const StepConst& s) {
    LightStep r;
    const double dz = s.dz > 1e-12f ? (double)s.dz : 1e-12;
    const double da = (L.e1[0] * s.dx + L.e1[1] * s.dy + L.e1[2] * s.dz) / dz;
    const double db = (L.e2[0] * s.dx + L.e2[1] * s.dy + L.e2[2] * s.dz) / dz;
    r.da_lo = fmin(0.0, da); r.da_hi = fmax(0.0, da);
    r.db_lo = fmin(0.0, db); r.db_hi = fmax(0.0, db);
    r.mx[0] = r.mx[1] = r.mx[2] = 0.0;
    return r;
}

__host__ __device__ inline LightStep light_step(const LightBasis& L, const StepConst& s) {
    LightStep r = light_drift(L, s);
    const double M[3][3] = {{L.t[0], L.b[0], L.n[0]}, {L.t[1], L.b[1], L.n[1]}, {L.t[2], L.b[2], L.n[2]}};
    const double D = light_det(M);
    const double dl[3] = {(double)s.dx - L.dm[0], (double)s.dy - L.dm[1], (double)s.dz - L.dm[2]};
    for (int col = 0; col < 3; ++col) {
        double Mc[3][3];
        for (int i = 0; i < 3; ++i)
            for (int c = 0; c < 3; ++c) Mc[i][c] = c == col ? dl[i] : M[i][c];
        r.mx[col] = fabs(light_det(Mc) / D);
    }
    return r;
}

__host__ __device__ inline void light_merge(LightStep& a, const LightStep& b) {
    a.da_lo = fmin(a.da_lo, b.da_lo); a.da_hi = fmax(a.da_hi, b.da_hi);
    a.db_lo = fmin(a.db_lo, b.db_lo); a.db_hi = fmax(a.db_hi, b.db_hi);
    for (int q = 0; q < 3; ++q) a.mx[q] = fmax(a.mx[q], b.mx[q]);
}

// The basis, drift box and direction bounds into rl, padded for rounding.
__host__ __device__ inline void light_finish(const LightBasis& L, const LightStep& s, RunLight* rl) {
    const double pad = 1e-6 + 1e-4 * fmax(s.da_hi - s.da_lo, s.db_hi - s.db_lo);
    rl->da_hi = (float)(s.da_hi * 1.0001 + pad);
    rl->da_lo = (float)(-s.da_lo * 1.0001 + pad);
    rl->db_hi = (float)(s.db_hi * 1.0001 + pad);
    rl->db_lo = (float)(-s.db_lo * 1.0001 + pad);
    for (int q = 0; q < 3; ++q) {
        rl->e1[q] = (float)L.e1[q];
        rl->e2[q] = (float)L.e2[q];
        rl->dm[q] = L.dm[q];
        rl->tv[q] = L.t[q];
        rl->bv[q] = L.b[q];
    }
    rl->ba = (float)(s.mx[0] * (1.0 + 1e-6) + 1e-12);
    rl->bb = (float)(s.mx[1] * (1.0 + 1e-6) + 1e-12);
    rl->bn = (float)(s.mx[2] * (1.0 + 1e-6) + 1e-12);
}

// Shared memory of a CTA that stages CHUNK triangles at a time.
template <int CHUNK>
struct LightSmem {
    // staged triangles: vertices in .xyz; .w of the second and third vertex hold the
    // bounds of d . n over the run's steps (run_dot_bounds)
    float4 tri[CHUNK * 3];
    float4 n[CHUNK];              // normals (origin-independent set-up), highest vertex z in .w
    float4 box[CHUNK];            // light box (amin, amax, bmin, bmax), widened by the slack
    float4 edge[3][CHUNK];        // light-space edge lines (nx, ny, c + slack, drift)
    unsigned front[CHUNK];        // steps to test
    unsigned long long d2[kRunMax / 2][3];   // directions of steps (k, k + 1), k even
    float4 o[kTileThreads];           // receiver origins (and t_min) of the pass
    unsigned m[kTileThreads];         // their step bits
    unsigned short q[kTileThreads / 32][kQueue];         // pair queues: receiver slot << 8 | triangle
    unsigned char list[kTileThreads / 32][CHUNK];    // triangles near the warp's receivers
};

template <class Smem>
__device__ __forceinline__ void stage_directions(Smem& sm, const StepConst* steps, const RunLight& rl) {
    if (2 * threadIdx.x < rl.kn) {
        const int k = 2 * threadIdx.x, k1 = min(k + 1, rl.kn - 1);
        const StepConst& s = steps[rl.j0 + rl.k0 + k];
        const StepConst& t = steps[rl.j0 + rl.k0 + k1];
        sm.d2[threadIdx.x][0] = f2_pack(s.dx, t.dx);
        sm.d2[threadIdx.x][1] = f2_pack(s.dy, t.dy);
        sm.d2[threadIdx.x][2] = f2_pack(s.dz, t.dz);
    }
}

// Bounds [lo, hi] on the FP32 value of d . v (in the rounding of the step tests) at every
// step d of the run, for a vector v of the triangle: d . v = d_m . v + alpha (t . v) +
// beta (b . v) + nu (n . v) exactly, n . v is within 2e-7 |v|_1 of d_m . v, and 2^-20 |v|_1
// covers the roundings of the step test's value and of these bounds (each below 8 ulp of
// |v|_1: every direction component is at most 1 in magnitude).
__device__ __forceinline__ float2 run_dot_bounds(const RunLight& rl, float vx, float vy, float vz) {
    const float c = fmaf(rl.dm[2], vz, fmaf(rl.dm[1], vy, rl.dm[0] * vx));
    const float tv = fmaf(rl.tv[2], vz, fmaf(rl.tv[1], vy, rl.tv[0] * vx));
    const float bv = fmaf(rl.bv[2], vz, fmaf(rl.bv[1], vy, rl.bv[0] * vx));
    const float l1 = fabsf(vx) + fabsf(vy) + fabsf(vz);
    const float r = fmaf(rl.ba, fabsf(tv), fmaf(rl.bb, fabsf(bv), fmaf(rl.bn, fabsf(c), 0x1p-20f * l1)));
    return make_float2(c - r, c + r);
}

// Lines of a triangle's light-space projection, as unit inward normals and offsets: a point
// x is inside iff n . x + c >= 0 for all three.  A ray of the run that meets the triangle at
// height h above the receiver passes x = r + h delta, so r can be shadowed by it only if
// n . r + c >= -h max(0, n . delta) for every line; .w holds max(0, max of n . delta over
// the run's drift box), so the cull is n . r + c >= -(rise x .w + slack).  A projection
// too thin to orient passes every point (the light box still applies).
__device__ __forceinline__ void light_edges(const float* pa, const float* pb, const RunLight& rl,
                                            float4& e0, float4& e1, float4& e2) {
    float4* e[3] = {&e0, &e1, &e2};
    const float ax = pa[1] - pa[0], ay = pb[1] - pb[0];
    const float bx = pa[2] - pa[0], by = pb[2] - pb[0];
    const float area2 = ax * by - ay * bx;
    const float l0 = sqrtf(ax * ax + ay * ay), l1 = sqrtf(bx * bx + by * by);
    const bool thin = !(fabsf(area2) > 1e-4f * l0 * l1);
    const float sg = area2 > 0.f ? 1.f : -1.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int j = i == 2 ? 0 : i + 1;
        const float ex = pa[j] - pa[i], ey = pb[j] - pb[i];
        const float len = sqrtf(ex * ex + ey * ey);
        if (thin || !(len > 1e-6f)) {
            *e[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        const float nx = -sg * ey / len, ny = sg * ex / len;
        // largest n . delta over the drift box [-da_lo, da_hi] x [-db_lo, db_hi]
        const float sup = fmaxf(nx * rl.da_hi, -nx * rl.da_lo) + fmaxf(ny * rl.db_hi, -ny * rl.db_lo);
        *e[i] = make_float4(nx, ny, -(nx * pa[i] + ny * pb[i]), fmaxf(sup, 0.f) * 1.0001f);
    }
}

// Stages triangle (a, b, c) of the scene in slot i; the caller sets sm.front[i].
template <class Smem>
__device__ __forceinline__ void stage_triangle(Smem& sm, int i, const float4* tris, int t,
                                               const RunLight& rl, const float* ref) {
                const float4 a = __ldg(&tris[3 * t]), b = __ldg(&tris[3 * t + 1]),
                             c = __ldg(&tris[3 * t + 2]);
                sm.tri[3 * i] = a; sm.tri[3 * i + 1] = b; sm.tri[3 * i + 2] = c;
                const float3 nrm = plucker_normal(a, b, c);
                sm.n[i] = make_float4(nrm.x, nrm.y, nrm.z, fmaxf(a.z, fmaxf(b.z, c.z)));
                float pa[3], pb[3];
                light_ab(rl, ref, a.x, a.y, a.z, &pa[0], &pb[0]);
                light_ab(rl, ref, b.x, b.y, b.z, &pa[1], &pb[1]);
                light_ab(rl, ref, c.x, c.y, c.z, &pa[2], &pb[2]);
                // the box and the edge lines carry the culls' slack already
                sm.box[i] = make_float4(fminf(pa[0], fminf(pa[1], pa[2])) - kLightSlack,
                                       fmaxf(pa[0], fmaxf(pa[1], pa[2])) + kLightSlack,
                                       fminf(pb[0], fminf(pb[1], pb[2])) - kLightSlack,
                                       fmaxf(pb[0], fmaxf(pb[1], pb[2])) + kLightSlack);
                light_edges(pa, pb, rl, sm.edge[0][i], sm.edge[1][i], sm.edge[2][i]);
    #pragma unroll
                for (int q3 = 0; q3 < 3; ++q3) sm.edge[q3][i].z += kLightSlack;
                const float2 ndb = run_dot_bounds(rl, nrm.x, nrm.y, nrm.z);
                sm.tri[3 * i + 1].w = ndb.x;
                sm.tri[3 * i + 2].w = ndb.y;
}

template <bool COUNT, class Smem>
__device__ __forceinline__ void drain_pairs(Smem& sm, const unsigned short* q, int n, int lane,
                                            int kn, unsigned long long& n_pair,
                                            unsigned long long& n_test) {
    const bool live = lane < n;
    const unsigned e = live ? q[lane] : 0u;
    const int who = (int)(e >> 8), t = (int)(e & 0xffu);
    const float4 p = sm.o[who];
    const float2 ndb = make_float2(sm.tri[3 * t + 1].w, sm.tri[3 * t + 2].w);
    // A receiver whose rays start at distance 0 (t_min = 0: the facade samples) with d . n
    // of one sign at every step of the run: its pair passed the plane-side cull, so the
    // distance check (a . n against 0 x d . n) holds at every step and only the inside
    // test varies.  A warp whose pairs all are so skips the distance check.
    const bool const_ahead = !live || (p.w == 0.f && (ndb.x > 0.f || ndb.y < 0.f));
    const bool all_const = __all_sync(0xffffffffu, const_ahead);
    if (!live) return;
    const float3 o = make_float3(p.x, p.y, p.z);
    const float4 a = sm.tri[3 * t], b = sm.tri[3 * t + 1], c = sm.tri[3 * t + 2];
    const unsigned want = sm.front[t];
    if (COUNT) ++n_pair;
    const float4 nv = sm.n[t];
    const PluckerTri pt = plucker_setup_n(o, a, b, c, make_float3(nv.x, nv.y, nv.z));
    // every step of the run is tested without branches, two steps per packed instruction
    // (the same roundings as plucker_hit); steps the triangle turns away from, and the
    // repeated step of an odd run's last pair, are masked off afterwards
    unsigned long long M[3][3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int c = 0; c < 3; ++c) M[e][c] = f2_pack(pt.m[e][c], pt.m[e][c]);
    unsigned m = 0;
    if (all_const) {
#pragma unroll
        for (int k = 0; k < kRunMax; k += 2) {
            if (k >= kn) break;
            const unsigned long long dx = sm.d2[k >> 1][0], dy = sm.d2[k >> 1][1], dz = sm.d2[k >> 1][2];
            float sv[3][2];
#pragma unroll
            for (int e = 0; e < 3; ++e)
                f2_unpack(f2_fma(dz, M[e][2], f2_fma(dy, M[e][1], f2_mul(dx, M[e][0]))), sv[e][0], sv[e][1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool inside = min3f(sv[0][h], sv[1][h], sv[2][h]) >= 0.f ||
                                    max3f(sv[0][h], sv[1][h], sv[2][h]) <= 0.f;
                if (inside) m |= 1u << (k + h);
            }
        }
    } else {
        unsigned long long N[3];
        N[0] = f2_pack(pt.nx, pt.nx); N[1] = f2_pack(pt.ny, pt.ny); N[2] = f2_pack(pt.nz, pt.nz);
#pragma unroll
        for (int k = 0; k < kRunMax; k += 2) {
            if (k >= kn) break;
            const unsigned long long dx = sm.d2[k >> 1][0], dy = sm.d2[k >> 1][1], dz = sm.d2[k >> 1][2];
            float sv[3][2], nd[2];
#pragma unroll
            for (int e = 0; e < 3; ++e)
                f2_unpack(f2_fma(dz, M[e][2], f2_fma(dy, M[e][1], f2_mul(dx, M[e][0]))), sv[e][0], sv[e][1]);
            f2_unpack(f2_fma(dz, N[2], f2_fma(dy, N[1], f2_mul(dx, N[0]))), nd[0], nd[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool inside = min3f(sv[0][h], sv[1][h], sv[2][h]) >= 0.f ||
                                    max3f(sv[0][h], sv[1][h], sv[2][h]) <= 0.f;
                const float lim = __fmul_rn(p.w, nd[h]);
                const bool ahead = (nd[h] > 0.f && pt.aon > lim) || (nd[h] < 0.f && pt.aon < lim);
                if (inside && ahead) m |= 1u << (k + h);
            }
        }
    }
    m &= want;
    if (COUNT) n_test += (unsigned)__popc(want);
    if (m) atomicOr(&sm.m[who], m);
}

// One pass of a warp's 32 receivers (sm.o, sm.m; light coordinates la, lb) over the nt staged
// triangles: the triangles no ray of any of them can reach are dropped for the whole warp
// at once, the other pairs are culled per lane, queued, and tested 32 at a time.
// drain(queue, n) tests n <= 32 pairs, receiver slot << 8 | triangle each, one per lane.  A
// receiver whose sm.m has come to `full` needs no more, and the pass ends when none does.
// SIDE: also drops the pairs whose receiver lies on the side of the triangle's plane that no ray
// leaves toward it, by the Pluecker test's own distance check (p.w: t_min).
template <bool SIDE = true, class Smem, class Drain>
__device__ __forceinline__ void light_pass(Smem& sm, const RunLight& rl, int nt, bool live, const float4& p,
                                           float la, float lb, unsigned full, Drain drain) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned short* q = sm.q[warp];
    // the warp's receivers' light-space box and lowest height
    float wa0 = live ? la : 3.4e38f, wa1 = live ? la : -3.4e38f;
    float wb0 = live ? lb : 3.4e38f, wb1 = live ? lb : -3.4e38f;
    float wz = live ? p.z : 3.4e38f;
    for (int off = 16; off > 0; off >>= 1) {
        wa0 = fminf(wa0, __shfl_xor_sync(0xffffffffu, wa0, off));
        wa1 = fmaxf(wa1, __shfl_xor_sync(0xffffffffu, wa1, off));
        wb0 = fminf(wb0, __shfl_xor_sync(0xffffffffu, wb0, off));
        wb1 = fmaxf(wb1, __shfl_xor_sync(0xffffffffu, wb1, off));
        wz = fminf(wz, __shfl_xor_sync(0xffffffffu, wz, off));
    }
    int nl = 0;
    for (int t0 = 0; t0 < nt; t0 += 32) {
        const int t = t0 + lane;           // < the chunk: the arrays are read in bounds
        const float rise = sm.n[t].w - wz;
        const float h = fmaxf(rise, 0.f);
        const float4 bx = sm.box[t];
        bool near = (t < nt) & (sm.front[t] != 0u) & (rise >= -0.01f);
        near &= (fmaf(h, rl.da_hi, wa1) >= bx.x) & (fmaf(-h, rl.da_lo, wa0) <= bx.y) &
                (fmaf(h, rl.db_hi, wb1) >= bx.z) & (fmaf(-h, rl.db_lo, wb0) <= bx.w);
#pragma unroll
        for (int q3 = 0; q3 < 3; ++q3) {
            const float4 e = sm.edge[q3][t];
            near &= fmaf(h, e.w, fmaxf(e.x * wa0, e.x * wa1) + fmaxf(e.y * wb0, e.y * wb1) + e.z) >= 0.f;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, near);
        if (near) sm.list[warp][nl + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)t;
        nl += __popc(bal);
    }
    int n = 0;
    __syncwarp();
    // a lane without a receiver, or done, rises below every triangle
    float pz = live ? p.z : 3.4e38f;
    const float da_hi = rl.da_hi, da_lo = rl.da_lo, db_hi = rl.db_hi, db_lo = rl.db_lo;
    // j == nl drains the queue's last pairs: one call site keeps the unrolled step
    // tests in the instruction cache once
    for (int j = 0; j <= nl; ++j) {
        const int t = j < nl ? (int)sm.list[warp][j] : 0;    // j == nl: nothing passes
        const float rise = j < nl ? sm.n[t].w - pz : -3.4e38f;
        const float h = fmaxf(rise, 0.f);
        const float4 bx = sm.box[t];
        bool pass = (rise >= -0.01f) & (fmaf(h, da_hi, la) >= bx.x) & (fmaf(-h, da_lo, la) <= bx.y) &
                    (fmaf(h, db_hi, lb) >= bx.z) & (fmaf(-h, db_lo, lb) <= bx.w);
        if (pass) {
#pragma unroll
            for (int q3 = 0; q3 < 3; ++q3) {
                const float4 e = sm.edge[q3][t];
                pass &= fmaf(h, e.w, fmaf(e.x, la, fmaf(e.y, lb, e.z))) >= 0.f;
            }
            if (SIDE) {
                // the receiver on the side of the triangle's plane that no ray of the run
                // leaves toward it: the step test's own distance check (a . n against
                // t_min d . n, same roundings) fails at every step
                const float4 v0 = sm.tri[3 * t];
                const float4 nv = sm.n[t];
                const float aon = fmaf(nv.z, __fsub_rn(v0.z, p.z),
                                       fmaf(nv.y, __fsub_rn(v0.y, p.y), __fmul_rn(nv.x, __fsub_rn(v0.x, p.x))));
                const float2 nd = make_float2(sm.tri[3 * t + 1].w, sm.tri[3 * t + 2].w);
                if (nd.x > 0.f) pass &= aon > __fmul_rn(p.w, nd.x);
                else if (nd.y < 0.f) pass &= aon < __fmul_rn(p.w, nd.y);
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, pass);
        if (pass) q[n + __popc(bal & ((1u << lane) - 1u))] =
            (unsigned short)(((unsigned)threadIdx.x << 8) | (unsigned)t);
        n += __popc(bal);
        if (n >= 32 || (j == nl && n > 0)) {
            const int cnt = min(n, 32);
            __syncwarp();
            drain(q + (n - cnt), cnt);
            n -= cnt;
            __syncwarp();
            if (sm.m[threadIdx.x] == full) pz = 3.4e38f;
            if (__all_sync(0xffffffffu, pz == 3.4e38f)) break;   // and the queued pairs are theirs
        }
    }
}

// ------------------------------------------------------------------- grouped traversal
// CHUNK triangles staged at a time, a node stack of STACK entries
template <int CHUNK, int STACK>
struct GroupSmem {
    int stack[STACK];
    int leaf[CHUNK + kTileThreads];
    int nst, nleaf;
    float box[kTileThreads / 32][6];
};

// Walks the BVH once for a CTA's group of receivers (one per thread: origin and t_min p) with
// all of their fans of a run as the query, kTileThreads nodes at a time from a shared
// stack: in the run's light space a ray at height h above its receiver lies within the
// receiver's coordinates widened by h times the run's drift box, so a node is entered when
// its projected box reaches the group's, widened by the rise to the node's top.  The
// leaves' triangles are staged CHUNK at a time (sm.front: front(tri), not 0), and
// pass(nt, la, lb) takes them; it returns whether the thread's receiver needs no more, and the walk ends when
// none does.  sm.o must be set, sm.m too if pass uses it.
template <bool COUNT, int CHUNK, int STACK, class Front, class Pass>
__device__ __forceinline__ void walk_group(LightSmem<CHUNK>& sm, GroupSmem<CHUNK, STACK>& gs, const DevScene& sc,
                                           const RunLight& rl, bool active, const float4& p, Front front,
                                           unsigned long long& n_box, Pass pass) {
    constexpr unsigned kAll = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the group's box, and its centre as the reference point
    float lo[3] = {p.x, p.y, p.z}, hi[3] = {p.x, p.y, p.z};
    for (int q = 0; q < 3; ++q) {
        if (!active) { lo[q] = 3.4e38f; hi[q] = -3.4e38f; }
        for (int o = 16; o > 0; o >>= 1) {
            lo[q] = fminf(lo[q], __shfl_xor_sync(kAll, lo[q], o));
            hi[q] = fmaxf(hi[q], __shfl_xor_sync(kAll, hi[q], o));
        }
        if (lane == 0) { gs.box[warp][q] = lo[q]; gs.box[warp][3 + q] = hi[q]; }
    }
    if (tid == 0) {
        gs.stack[0] = 0;
        gs.nst = sc.n_nodes > 0 ? 1 : 0;
        gs.nleaf = 0;
    }
    __syncthreads();
    float ref[3], half[3];
    for (int q = 0; q < 3; ++q) {
        float a = gs.box[0][q], b = gs.box[0][3 + q];
        for (int w = 1; w < kTileThreads / 32; ++w) {
            a = fminf(a, gs.box[w][q]);
            b = fmaxf(b, gs.box[w][3 + q]);
        }
        ref[q] = 0.5f * (a + b);
        half[q] = 0.5f * (b - a);
    }
    const float zlow = ref[2] - half[2] - 0.01f;
    // half extents of the group in light space, with the culls' slack
    const float ga = fabsf(rl.e1[0]) * half[0] + fabsf(rl.e1[1]) * half[1] + fabsf(rl.e1[2]) * half[2] + kLightSlack;
    const float gb = fabsf(rl.e2[0]) * half[0] + fabsf(rl.e2[1]) * half[1] + fabsf(rl.e2[2]) * half[2] + kLightSlack;
    float la, lb;
    light_ab(rl, ref, p.x, p.y, p.z, &la, &lb);
    while (true) {
        __syncthreads();
        int nst = SA_AT_MOST(gs.nst, STACK), nleaf = gs.nleaf;
        while (nst > 0 && nleaf < CHUNK) {
            // A wave of w nodes leaves at most w more, so waves end at STACK - 96; from there it
            // goes node by node, depth first, which adds one per level of the tree.  The tree
            // is at most 62 deep (30 bits of Morton code, then the index's), so 96 are enough.
            const int take = min(kTileThreads, min(nst, max(1, STACK - 96 - nst)));
            const int i = tid < take ? gs.stack[nst - 1 - tid] : -1;
            __syncthreads();
            if (tid == 0) gs.nst = nst - take;
            __syncthreads();
            bool in = false;
            int tri = -1;
            if (i >= 0) {
                const float4 nlo = __ldg(&sc.nodes[2 * i]);
                const float4 nhi = __ldg(&sc.nodes[2 * i + 1]);
                tri = SA_LEAF(__float_as_int(nhi.w), sc.T, sa::CK_WALK_LEAF);
                if (COUNT) ++n_box;
                const float hx = 0.5f * (nhi.x - nlo.x), hy = 0.5f * (nhi.y - nlo.y), hz = 0.5f * (nhi.z - nlo.z);
                float a, b;
                light_ab(rl, ref, nlo.x + hx, nlo.y + hy, nlo.z + hz, &a, &b);
                const float ra = fmaf(fabsf(rl.e1[2]), hz, fmaf(fabsf(rl.e1[1]), hy, fabsf(rl.e1[0]) * hx));
                const float rb = fmaf(fabsf(rl.e2[2]), hz, fmaf(fabsf(rl.e2[1]), hy, fabsf(rl.e2[0]) * hx));
                const float rise = nhi.z - zlow;
                in = (rise >= 0.f) & (fmaf(rise, rl.da_hi, ga) >= a - ra) & (fmaf(-rise, rl.da_lo, -ga) <= a + ra) &
                     (fmaf(rise, rl.db_hi, gb) >= b - rb) & (fmaf(-rise, rl.db_lo, -gb) <= b + rb);
            }
            const bool leaf = in && tri >= 0, node = in && tri < 0 && SA_CHILDREN(sc.nodes, i, sc.n_nodes, sa::CK_WALK_CHILD);
            const unsigned bn = __ballot_sync(kAll, node), bl = __ballot_sync(kAll, leaf);
            int pn = 0, pl = 0;
            if (lane == 0) {
                if (bn) pn = atomicAdd(&gs.nst, 2 * __popc(bn));
                if (bl) pl = atomicAdd(&gs.nleaf, __popc(bl));
            }
            pn = __shfl_sync(kAll, pn, 0);
            pl = __shfl_sync(kAll, pl, 0);
            const unsigned below = (1u << lane) - 1u;
            if (node) {
                // in depth-first order the left child follows, and the right one follows it
                const int left = i + 1, right = __float_as_int(__ldg(&sc.nodes[2 * left]).w);
                const int at = pn + 2 * __popc(bn & below);
                if (SA_ROOM(at, STACK, sa::CK_WALK_STACK)) gs.stack[at] = right;
                if (SA_ROOM(at + 1, STACK, sa::CK_WALK_STACK)) gs.stack[at + 1] = left;
            }
            if (leaf) gs.leaf[pl + __popc(bl & below)] = tri;
            __syncthreads();
            nst = SA_AT_MOST(gs.nst, STACK);
            nleaf = gs.nleaf;
        }
        const int nt = min(nleaf, CHUNK), left = nleaf - nt;
        if (nt == 0) break;
        if (tid < nt) {
            const int tri = gs.leaf[tid];
            stage_triangle(sm, tid, sc.tris, tri, rl, ref);
            sm.front[tid] = front(tri);
        }
        const int carry = tid < left ? gs.leaf[nt + tid] : 0;
        __syncthreads();
        if (tid < left) gs.leaf[tid] = carry;
        if (tid == 0) gs.nleaf = left;
        const bool done = pass(nt, la, lb);
        __syncwarp();
        if (__syncthreads_and(done)) break;
    }
}

// Light-space constants of the runs that n blocks are cut into (piece q of K steps runs from
// q K / parts): one warp per run, a lane per step.
cudaError_t launch_run_lights(const StepConst* steps, const BlockConst* blocks, int n_blocks, int parts,
                              RunLight* runs, cudaStream_t st);

}  // namespace sa
