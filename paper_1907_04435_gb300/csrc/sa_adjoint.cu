// sa_adjoint.cu -- derivative of the region's shadow-minutes with respect to building heights.
//
// Objective (continuous time between the sun steps): between steps j and j+1 of a day the
// sun follows the great circle d(a) = slerp(d_j, d_{j+1}, a), a in [0, 1], over one step
// length dt.  A ground receiver contributes dt * chi where the status does not change over
// the interval and dt * a* (shadow -> lit) or dt * (1 - a*) (lit -> shadow) where it flips
// at a*.  S = sum_r w_r * (those contributions).  Heights only move flip times, so
//     dS/dh_b = sum over flips f caused by building b of  w_r * dt * s_f * da*/dh_b,
// s_f = +1 for shadow -> lit and -1 for lit -> shadow.
//
// Kernels:
//   k_flip_count / k_flip_fill  walk each receiver's forward step masks (from the accrual
//                               raster) and list the intervals whose end statuses differ;
//                               intervals without a flip add dt * chi to S directly.
//   k_arcs                      the FP64 constants of every interval's arc.
//   k_flip_solve                per flip: find the buildings that shadow the receiver at the
//                               shadowed end (FP32 BVH traversal), locate each one's flip
//                               a*_b on the exact prism test, in a projective parameter of
//                               the same arc in which every prism constraint is linear: the
//                               pair of constraints that close the entry interval at the
//                               flip is found in FP32, with margins that certify it, and
//                               gives the flip in closed form in FP64 (without the margins,
//                               an FP64 search finds it); then take the first (lit ->
//                               shadow) or last (shadow -> lit), and if the flip is the
//                               shadow of a roof edge e of building b crossing the
//                               receiver, differentiate the grazing condition
//                                  G(a, h) = A_e + h B_e(a) = 0,  B_e(a) = c_e x u(a),
//                               u = d_xy / d_z:  da*/dh = -B_e / (h dB_e/da).  A flip caused
//                               by a vertical edge does not depend on h.
#include <float.h>
#include <string.h>

#include <algorithm>

#include "sa_internal.cuh"

namespace sa {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxCand = 8;
constexpr int kBisect = 40;   // halvings of [0, 1]: the flip to 1e-12 of a step
constexpr int kLinEdges = 8;  // footprints up to this many edges take the linear form
constexpr int kBisectF = 22;  // FP32 halvings that bracket a flip before its closed form
constexpr int kSolveThreads = 128;
constexpr int kSumCtas = 512;
constexpr double kSide = 1e-10;   // FP64 status checks this far on both sides of a root

// Step mask of a block for receiver r, and the status of the step before it in the same day
// (none: the block's own first step, which makes no interval and no flip).
struct BlockBits {
    unsigned long long m;       // bit k: shadowed at step j0 + k
    unsigned long long before;  // bit k: shadowed at the step before it
    unsigned long long pairs;   // bit k: step k ends an interval (the first of a day ends none)
};

__device__ __forceinline__ BlockBits block_bits(const unsigned long long* masks, long long R,
                                                const BlockConst& bc, long long r, bool& carry) {
    BlockBits b;
    const unsigned long long full = bc.K >= 64 ? ~0ull : ((1ull << bc.K) - 1ull);
    b.m = (masks[(long long)bc.mask_block * R + r] >> bc.mask_bit) & full;
    b.before = ((b.m << 1) | (carry ? 1ull : 0ull)) & full;
    b.pairs = bc.new_day ? full & ~1ull : full;
    carry = (b.m >> (bc.K - 1)) & 1ull;
    return b;
}

// Sum of s over the CTA's threads in a fixed order (at thread 0; at most 1,024 threads).
__device__ __forceinline__ double cta_sum(double s) {
    __shared__ double s_part[32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(kFull, s, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0)
        for (unsigned w = 1; w < blockDim.x / 32; ++w) s += s_part[w];
    return s;
}

// Sums whose order depends on n alone, so that S repeats to the last bit.
__global__ void k_sum(const double* __restrict__ x, long long n, double* __restrict__ part) {
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s += x[i];
    s = cta_sum(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void k_sum_pair(const double* __restrict__ x, const double* __restrict__ y, double* __restrict__ S) {
    double s = 0.0;
    for (int i = threadIdx.x; i < kSumCtas; i += blockDim.x) s += x[i] + y[i];
    s = cta_sum(s);
    if (threadIdx.x == 0) *S = s;
}

// The list's order: groups of consecutive blocks, in each the grid's 8 x 4-cell patches, one
// warp each.  Flips that neighbours see at nearly the same time, mostly of one edge, then
// share a warp in k_flip_solve: their rays visit the same nodes and their derivatives go to
// the same building (k_flip_solve 8.9 -> 6.9 ms before the
// certified search).
struct FlipOrder {
    int nx, ny, tiles_x;
    long long n;          // threads: 32 per patch
    int per;              // blocks per group
};

__device__ __forceinline__ long long patch_cell(const FlipOrder& g, long long t) {
    const long long p = t >> 5;
    const int lane = (int)(t & 31), tx = (int)(p % g.tiles_x);
    const long long ix = tx * 8 + (lane & 7), iy = (p / g.tiles_x) * 4 + (lane >> 3);
    return ix < g.nx && iy < g.ny ? iy * g.nx + ix : -1;
}

// Flips per group and receiver (counts [groups][n]), and the minutes of the intervals
// without one: both are counts of bits (481 steps one by one took 1.10 ms on 600k cells,
// whose masks are 43 MB).
__global__ void k_flip_count(const unsigned long long* __restrict__ masks, long long R, FlipOrder g,
                             const BlockConst* __restrict__ blocks, int n_blocks,
                             const float* __restrict__ weights, double dt,
                             unsigned* __restrict__ counts, double* __restrict__ part) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long r = t < g.n ? patch_cell(g, t) : -1;
    double s = 0.0;
    if (t < g.n) {
        unsigned n = 0, steady = 0;
        bool carry = false;
        for (int b = 0; b < n_blocks; ++b) {
            if (r >= 0) {
                const BlockBits w = block_bits(masks, R, blocks[b], r, carry);
                n += __popcll((w.m ^ w.before) & w.pairs);
                steady += __popcll(w.m & w.before & w.pairs);
            }
            if ((b + 1) % g.per == 0 || b + 1 == n_blocks) {
                counts[(long long)(b / g.per) * g.n + t] = n;
                n = 0;
            }
        }
        if (r >= 0) s = (double)steady * dt * (weights ? (double)weights[r] : 1.0);
    }
    s = cta_sum(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void k_flip_fill(const unsigned long long* __restrict__ masks, long long R, FlipOrder g,
                            const BlockConst* __restrict__ blocks, int n_blocks,
                            const unsigned* __restrict__ offsets, int4* __restrict__ flips) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long r = t < g.n ? patch_cell(g, t) : -1;
    if (r < 0) return;
    unsigned w = 0;
    bool carry = false;
    for (int b = 0; b < n_blocks; ++b) {
        if (b % g.per == 0) w = offsets[(long long)(b / g.per) * g.n + t];
        const BlockBits q = block_bits(masks, R, blocks[b], r, carry);
        unsigned long long f = (q.m ^ q.before) & q.pairs;
        while (f) {
            const int k = __ffsll((long long)f) - 1;
            f &= f - 1ull;
            flips[w++] = make_int4((int)(r & 0x7fffffff), (int)(r >> 31), blocks[b].j0 + k - 1,
                                   (int)((q.before >> k) & 1ull));
        }
    }
}

struct Vec3 { double x, y, z; };

__device__ __forceinline__ Vec3 unit(const StepConst& s) {
    const double x = s.dx, y = s.dy, z = s.dz;
    const double n = sqrt(x * x + y * y + z * z);
    return Vec3{x / n, y / n, z / n};
}

struct Arc {
    Vec3 a, b;
    double theta, sin_theta;
};

// The arc from step j to step j + 1, one per interval: unit end a, chord e = b - a, angle.
struct ArcConst {
    double ax, ay, az, ex, ey, ez;
    double theta, sin_theta, omc;     // omc = 1 - cos theta = |e|^2 / 2
    double inv_theta;                 // 1 / theta (0 for a degenerate arc)
};

__global__ void k_arcs(const StepConst* __restrict__ steps, int n, ArcConst* __restrict__ arcs) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const Vec3 a = unit(steps[j]), b = unit(steps[j + 1]);
    ArcConst c;
    c.ax = a.x; c.ay = a.y; c.az = a.z;
    c.ex = b.x - a.x; c.ey = b.y - a.y; c.ez = b.z - a.z;
    const double nx = a.y * b.z - a.z * b.y, ny = a.z * b.x - a.x * b.z, nz = a.x * b.y - a.y * b.x;
    c.sin_theta = sqrt(nx * nx + ny * ny + nz * nz);
    c.omc = 0.5 * (c.ex * c.ex + c.ey * c.ey + c.ez * c.ez);
    c.theta = atan2(c.sin_theta, 1.0 - c.omc);
    c.inv_theta = c.theta < 1e-12 ? 0.0 : 1.0 / c.theta;
    arcs[j] = c;
}

__device__ __forceinline__ Arc arc_of(const ArcConst& c) {
    return Arc{Vec3{c.ax, c.ay, c.az}, Vec3{c.ax + c.ex, c.ay + c.ey, c.az + c.ez}, c.theta, c.sin_theta};
}

__device__ __forceinline__ Vec3 arc_dir(const Arc& c, double al) {
    if (c.theta < 1e-12) {
        Vec3 d{c.a.x + al * (c.b.x - c.a.x), c.a.y + al * (c.b.y - c.a.y), c.a.z + al * (c.b.z - c.a.z)};
        const double n = sqrt(d.x * d.x + d.y * d.y + d.z * d.z);
        return Vec3{d.x / n, d.y / n, d.z / n};
    }
    const double wa = sin((1.0 - al) * c.theta) / c.sin_theta, wb = sin(al * c.theta) / c.sin_theta;
    Vec3 d{wa * c.a.x + wb * c.b.x, wa * c.a.y + wb * c.b.y, wa * c.a.z + wb * c.b.z};
    const double n = sqrt(d.x * d.x + d.y * d.y + d.z * d.z);
    return Vec3{d.x / n, d.y / n, d.z / n};
}

__device__ __forceinline__ Vec3 arc_ddir(const Arc& c, double al) {
    if (c.theta < 1e-12) return Vec3{c.b.x - c.a.x, c.b.y - c.a.y, c.b.z - c.a.z};
    const double ka = -c.theta * cos((1.0 - al) * c.theta) / c.sin_theta;
    const double kb = c.theta * cos(al * c.theta) / c.sin_theta;
    return Vec3{ka * c.a.x + kb * c.b.x, ka * c.a.y + kb * c.b.y, ka * c.a.z + kb * c.b.z};
}

// Exact prism test: does the ray from ground point (px, py) toward d cross the convex CCW
// footprint between heights 0 and h?  Returns the entry height interval and the edge that
// bounds it from below (-1: the ground).
struct Entry {
    bool inside;
    double zlo, zhi;
    int elo;
};

__device__ Entry prism(const float2* xy, int a, int v, double h, double px, double py,
                       double ux, double uy) {
    double zlo = 0.0, zhi = h;
    int elo = -1;
    for (int i = 0; i < v; ++i) {
        const float2 p0 = xy[a + i], p1 = xy[a + (i + 1 == v ? 0 : i + 1)];
        const double cx = (double)p1.x - (double)p0.x, cy = (double)p1.y - (double)p0.y;
        const double A = cx * (py - (double)p0.y) - cy * (px - (double)p0.x);
        const double Bc = cx * uy - cy * ux;     // left-of-edge constraint: A + z Bc >= 0
        if (Bc > 0.0) {
            const double z = -A / Bc;
            if (z > zlo) { zlo = z; elo = i; }
        } else if (Bc < 0.0) {
            const double z = -A / Bc;
            if (z < zhi) zhi = z;
        } else if (A < 0.0) {
            return Entry{false, 1.0, 0.0, -1};
        }
    }
    return Entry{zlo <= zhi, zlo, zhi, elo};
}

// The same decision as prism(...).inside, without divisions: each bound z = -A / B of the
// entry interval is kept as a fraction with a positive denominator and compared by cross
// multiplication.
__device__ bool prism_inside(const float2* xy, int a, int v, double h, double px, double py,
                             double ux, double uy) {
    double nlo = 0.0, dlo = 1.0;     // lower bound nlo / dlo
    double nhi = h, dhi = 1.0;       // upper bound nhi / dhi
    for (int i = 0; i < v; ++i) {
        const float2 p0 = xy[a + i], p1 = xy[a + (i + 1 == v ? 0 : i + 1)];
        const double cx = (double)p1.x - (double)p0.x, cy = (double)p1.y - (double)p0.y;
        const double A = cx * (py - (double)p0.y) - cy * (px - (double)p0.x);
        const double Bc = cx * uy - cy * ux;
        if (Bc > 0.0) {
            if (-A * dlo > nlo * Bc) { nlo = -A; dlo = Bc; }
        } else if (Bc < 0.0) {
            if (A * dhi < nhi * -Bc) { nhi = A; dhi = -Bc; }
        } else if (A < 0.0) {
            return false;
        }
    }
    return nlo * dhi <= nhi * dlo;
}

// Status of building b along the arc in the projective parameter be: the direction
// a + be (b - a) (not normalised: the slopes u = d_xy / d_z do not depend on its length)
// runs over the same great-circle arc as slerp, monotonically, so a flip found in be is
// the same physical flip; its slerp parameter follows from the angle to a.
__device__ __forceinline__ bool prism_along(const FootprintSet& fs, const float* heights, int b,
                                            double px, double py, const Arc& arc, double be) {
    const double dx = fma(be, arc.b.x - arc.a.x, arc.a.x);
    const double dy = fma(be, arc.b.y - arc.a.y, arc.a.y);
    const double dz = fma(be, arc.b.z - arc.a.z, arc.a.z);
    const double iz = 1.0 / dz;
    return prism_inside(fs.xy, fs.fp_off[b], fs.fp_off[b + 1] - fs.fp_off[b], (double)heights[b],
                        px, py, dx * iz, dy * iz);
}

// Along the arc d(be) = a + be (b - a) every edge constraint of the prism is linear in be
// once multiplied by d_z(be) > 0: the bound z = -A / B_c becomes (-A d_z) / (B_c d_z) with
// B_c d_z = c x d_xy = E0 + be E1.  Set up once per (flip, building), each bisection step
// then costs a few FP64 multiply-adds per edge and no division.
struct PrismLin {
    int v;
    double h, az, ez;
    double A[kLinEdges], E0[kLinEdges], E1[kLinEdges];
};

__device__ void prism_lin_setup(PrismLin& P, const float2* xy, int a, int v, double h, double px,
                                double py, const Arc& arc) {
    P.v = v;
    P.h = h;
    P.az = arc.a.z;
    P.ez = arc.b.z - arc.a.z;
    const double ex = arc.b.x - arc.a.x, ey = arc.b.y - arc.a.y;
    for (int i = 0; i < v; ++i) {
        const float2 p0 = xy[a + i], p1 = xy[a + (i + 1 == v ? 0 : i + 1)];
        const double cx = (double)p1.x - (double)p0.x, cy = (double)p1.y - (double)p0.y;
        P.A[i] = cx * (py - (double)p0.y) - cy * (px - (double)p0.x);
        P.E0[i] = cx * arc.a.y - cy * arc.a.x;
        P.E1[i] = cx * ey - cy * ex;
    }
}

__device__ bool prism_lin_inside(const PrismLin& P, double be) {
    const double dz = fma(be, P.ez, P.az);
    double nlo = 0.0, dlo = 1.0, nhi = P.h, dhi = 1.0;
    for (int i = 0; i < P.v; ++i) {
        const double den = fma(be, P.E1[i], P.E0[i]);
        const double num = -P.A[i] * dz;
        if (den > 0.0) {
            if (num * dlo > nlo * den) { nlo = num; dlo = den; }
        } else if (den < 0.0) {
            if (-num * dhi < nhi * -den) { nhi = -num; dhi = -den; }
        } else if (P.A[i] < 0.0) {
            return false;
        }
    }
    return nlo * dhi <= nhi * dlo;
}

// The same test with FP32 coefficients: used only to bracket the flip coarsely (the
// bracket is confirmed in FP64 below).
struct PrismLinF {
    int v;
    float h, az, ez;
    float A[kLinEdges], E0[kLinEdges], E1[kLinEdges];
};

__device__ void prism_lin_to_f(const PrismLin& P, PrismLinF& F) {
    F.v = P.v; F.h = (float)P.h; F.az = (float)P.az; F.ez = (float)P.ez;
    for (int i = 0; i < P.v; ++i) { F.A[i] = (float)P.A[i]; F.E0[i] = (float)P.E0[i]; F.E1[i] = (float)P.E1[i]; }
}

__device__ bool prism_lin_inside_f(const PrismLinF& P, float be) {
    const float dz = fmaf(be, P.ez, P.az);
    float nlo = 0.f, dlo = 1.f, nhi = P.h, dhi = 1.f;
    for (int i = 0; i < P.v; ++i) {
        const float den = fmaf(be, P.E1[i], P.E0[i]);
        const float num = -P.A[i] * dz;
        if (den > 0.f) {
            if (num * dlo > nlo * den) { nlo = num; dlo = den; }
        } else if (den < 0.f) {
            if (-num * dhi < nhi * -den) { nhi = -num; dhi = -den; }
        } else if (P.A[i] < 0.f) {
            return false;
        }
    }
    return nlo * dhi <= nhi * dlo;
}

// The constraints that bound the entry interval at be: il the lower bound (-1: the ground),
// iu the upper bound (-1: the roof height h).
__device__ void prism_lin_active(const PrismLin& P, double be, int* il, int* iu) {
    const double dz = fma(be, P.ez, P.az);
    double nlo = 0.0, dlo = 1.0, nhi = P.h, dhi = 1.0;
    *il = -1;
    *iu = -1;
    for (int i = 0; i < P.v; ++i) {
        const double den = fma(be, P.E1[i], P.E0[i]);
        const double num = -P.A[i] * dz;
        if (den > 0.0 && num * dlo > nlo * den) { nlo = num; dlo = den; *il = i; }
        if (den < 0.0 && -num * dhi < nhi * -den) { nhi = -num; dhi = -den; *iu = i; }
    }
}

// The flip where the interval closes between lower bound il and upper bound iu, in closed
// form: both bounds are ratios of functions linear in be, so their equality is linear.
//   edge il against the roof:  -A_i d_z(be) = h (E0_i + be E1_i)
//   edge il against edge iu:    A_i (E0_j + be E1_j) = A_j (E0_i + be E1_i)
__device__ bool pair_root(const PrismLin& P, int il, int iu, double* be) {
    if (il < 0) return false;
    const double Ai = P.A[il];
    if (iu < 0) {
        const double den = fma(Ai, P.ez, P.h * P.E1[il]);
        if (den == 0.0) return false;
        *be = -fma(Ai, P.az, P.h * P.E0[il]) / den;
        return true;
    }
    const double Aj = P.A[iu];
    const double den = Ai * P.E1[iu] - Aj * P.E1[il];
    if (den == 0.0) return false;
    *be = (Aj * P.E0[il] - Ai * P.E0[iu]) / den;
    return true;
}

// slerp parameter of the projective parameter be (see prism_along): the angle from a to
// d = a + be e has |a x d| = be sin theta and a . d = 1 - be (1 - cos theta).
__device__ __forceinline__ double slerp_param(const ArcConst& c, double be) {
    if (c.inv_theta == 0.0) return be;
    double ang;
    if (c.theta < 0.1) {
        // steps up to about 20 minutes: the arctangent's power series (the next term, t^16 / 17
        // of the first, is 6e-18 of it at t = 0.1)
        const double t = be * c.sin_theta / (1.0 - be * c.omc), q = t * t;
        double p = -1.0 / 15.0;
        p = fma(p, q, 1.0 / 13.0);
        p = fma(p, q, -1.0 / 11.0);
        p = fma(p, q, 1.0 / 9.0);
        p = fma(p, q, -1.0 / 7.0);
        p = fma(p, q, 0.2);
        p = fma(p, q, -1.0 / 3.0);
        ang = fma(t * q, p, t);
    } else {
        ang = atan2(be * c.sin_theta, 1.0 - be * c.omc);
    }
    return fmin(1.0, fmax(0.0, ang * c.inv_theta));
}

// Flip of one building along the arc, searched in FP64: s0 is its status at be = 0.  False
// when the statuses at the ends are not those of a flip.
__device__ __noinline__ bool solve_fp64(const FootprintSet& fs, const float* heights, int b, double px,
                                        double py, const Arc& arc, bool s0, double* be_star) {
    const int fa = fs.fp_off[b], v = fs.fp_off[b + 1] - fa;
    if (v <= kLinEdges) {
        PrismLin P;
        prism_lin_setup(P, fs.xy, fa, v, (double)heights[b], px, py, arc);
        if (prism_lin_inside(P, 0.0) != s0 || prism_lin_inside(P, 1.0) == s0) return false;
        // bracket in FP32, then the closed form of the pair of constraints that close the
        // interval, confirmed by FP64 statuses on both sides of it
        PrismLinF F;
        prism_lin_to_f(P, F);
        float flo = 0.f, fhi = 1.f;
        for (int it = 0; it < kBisectF; ++it) {
            const float mid = 0.5f * (flo + fhi);
            if (prism_lin_inside_f(F, mid) == s0) flo = mid; else fhi = mid;
        }
        int il, iu;
        prism_lin_active(P, s0 ? (double)flo : (double)fhi, &il, &iu);
        double r;
        if (pair_root(P, il, iu, &r) && r > kSide && r < 1.0 - kSide &&
            fabs(r - 0.5 * ((double)flo + (double)fhi)) < 1e-4 &&
            prism_lin_inside(P, r - kSide) == s0 && prism_lin_inside(P, r + kSide) != s0) {
            *be_star = r;
            return true;
        }
        double lo = 0.0, hi = 1.0;   // invariant: status(lo) == status at the start
        for (int it = 0; it < kBisect; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (prism_lin_inside(P, mid) == s0) lo = mid; else hi = mid;
        }
        *be_star = 0.5 * (lo + hi);
        return true;
    }
    if (prism_along(fs, heights, b, px, py, arc, 0.0) != s0) return false;
    if (prism_along(fs, heights, b, px, py, arc, 1.0) == s0) return false;
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < kBisect; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (prism_along(fs, heights, b, px, py, arc, mid) == s0) lo = mid; else hi = mid;
    }
    *be_star = 0.5 * (lo + hi);
    return true;
}

// The same flip with FP64 only where it counts.  The statuses inside(be) form an interval of
// the arc (the prism is convex), so the flip is where one pair of bounds -- lower edge il,
// upper edge or roof iu -- closes the entry interval.  The pair is found in FP32 from the
// lit end: the pair that is closed there has its root nearer to the flip, and the pair closed
// at that root replaces it until none is.  It is accepted only with margins far above the
// FP32 errors (1e-4 of the point's own distance, against 2e-5): every other constraint is
// slack at the root and at the shadowed end.  The root itself, and its derivative with respect to h, are FP64 from the two
// constraints' exact coefficients.  FP64 runs at 1/64 of the FP32 rate here, and the search
// in it kept that pipe 83 % busy (park of 600k cells, 200 buildings: 12.2 ms for all flips,
// now 1.06, and 0.46 for the 5 % that are left to it; 0.67
// and 9 % with the pair's middle alone as the point inside at the shadowed end, and a park
// on 16 December 1.29 -> 0.41).
// Returns 1 with the root, 0 when undecided.  *dbe_dh: derivative of a roof-edge flip.
__device__ __forceinline__ int solve_fast(const FootprintSet& fs, int fa, int v, float h, float px, float py,
                                          const ArcConst& arc, bool c0, double* be_star, double* dbe_dh) {
    const float ax = (float)arc.ax, ay = (float)arc.ay, az = (float)arc.az;
    const float ex = (float)arc.ex, ey = (float)arc.ey, ez = (float)arc.ez;
    // constraint i: A_i d_z(be) + z (E0_i + be E1_i) >= 0 for the heights z inside; its margin is
    // T_i (reach + z), T_i = 1e-4 |c_i| (padding: i >= v is never read)
    float A[kLinEdges], E0[kLinEdges], E1[kLinEdges], T[kLinEdges];
    const float2* xy = fs.xy + fa;
    float reach = 1.f;
    float2 p0 = xy[0];
    const float2 first = p0;
#pragma unroll
    for (int i = 0; i < kLinEdges; ++i) {
        if (i < v) {
            const float2 p1 = i + 1 < v ? xy[i + 1] : first;
            const float cx = p1.x - p0.x, cy = p1.y - p0.y, dx = px - p0.x, dy = py - p0.y;
            A[i] = cx * dy - cy * dx;
            E0[i] = cx * ay - cy * ax;
            E1[i] = cx * ey - cy * ex;
            T[i] = (fabsf(cx) + fabsf(cy)) * 1e-4f;
            reach = fmaxf(reach, fabsf(dx) + fabsf(dy));
            p0 = p1;
        } else {
            A[i] = E0[i] = E1[i] = T[i] = 0.f;
        }
    }
    auto bounds = [&](float be, float& L, float& U, int& il, int& iu) {
        const float dz = fmaf(be, ez, az);
        L = 0.f; U = h; il = -1; iu = -1;
#pragma unroll
        for (int i = 0; i < kLinEdges; ++i) {
            const float den = fmaf(be, E1[i], E0[i]);
            const float z = __fdividef(-A[i] * dz, den);
            if (i < v && den > 0.f && z > L) { L = z; il = i; }
            if (i < v && den < 0.f && z < U) { U = z; iu = i; }
        }
    };
    // every constraint but il and iu holds with its margin at height z
    auto slack = [&](float be, float z, int il, int iu) {
        const float dz = fmaf(be, ez, az);
        bool ok = true;
#pragma unroll
        for (int i = 0; i < kLinEdges; ++i)
            ok &= i >= v || i == il || i == iu ||
                  fmaf(z, fmaf(be, E1[i], E0[i]), A[i] * dz) > T[i] * (reach + z);
        return ok;
    };
    const float sh = c0 ? 0.f : 1.f, lit = 1.f - sh;
    const float zm = 1e-4f * (h + reach);          // margin of heights
    float L, U;
    int il, iu;
    int pl = -2, pu = -2;
    float be = lit;
    bool done = false;
    for (int it = 0; it < 6 && !done; ++it) {
        bounds(be, L, U, il, iu);
        if ((il == pl && iu == pu) || (it > 0 && L <= U)) { done = true; break; }
        if (il < 0 || L <= U) return 0;
        pl = il; pu = iu;
        float Ai = 0.f, E0i = 0.f, E1i = 0.f, Aj = 0.f, E0j = 0.f, E1j = 0.f;
#pragma unroll
        for (int i = 0; i < kLinEdges; ++i) {
            if (i == il) { Ai = A[i]; E0i = E0[i]; E1i = E1[i]; }
            if (i == iu) { Aj = A[i]; E0j = E0[i]; E1j = E1[i]; }
        }
        be = iu < 0 ? __fdividef(-fmaf(Ai, az, h * E0i), fmaf(Ai, ez, h * E1i))
                    : __fdividef(Aj * E0i - Ai * E0j, Ai * E1j - Aj * E1i);
        if (!(be > 0.f && be < 1.f)) return 0;
    }
    if (!done) return 0;
    // FP64: the pair's exact coefficients, and its root
    auto coef = [&](int i, double* a, double* e0, double* e1) {
        const float2 p = xy[i], q = i + 1 == v ? first : xy[i + 1];
        const double cx = (double)q.x - (double)p.x, cy = (double)q.y - (double)p.y;
        *a = cx * ((double)py - (double)p.y) - cy * ((double)px - (double)p.x);
        *e0 = cx * arc.ay - cy * arc.ax;
        *e1 = cx * arc.ey - cy * arc.ex;
    };
    double ai, e0i, e1i, r;
    coef(pl, &ai, &e0i, &e1i);
    *dbe_dh = 0.0;
    double num, den;
    if (pu < 0) {
        den = fma(ai, arc.ez, (double)h * e1i);
        num = -fma(ai, arc.az, (double)h * e0i);
    } else {
        double aj, e0j, e1j;
        coef(pu, &aj, &e0j, &e1j);
        den = ai * e1j - aj * e1i;
        num = aj * e0i - ai * e0j;
    }
    if (den == 0.0) return 0;
    const double inv = 1.0 / den;
    r = num * inv;
    if (!(r > 1e-6 && r < 1.0 - 1e-6)) return 0;
    // closed toward the lit end
    const double side = fma((double)lit, den, -num);
    if (!(pu < 0 ? side < 0.0 : side > 0.0)) return 0;
    const double dl = fma(r, e1i, e0i);
    if (pu < 0) *dbe_dh = -dl * inv;
    // certificates at the root and at the lit end
    const float rf = (float)r;
    float Al = 0.f, E0l = 0.f, E1l = 0.f, Au = 0.f, E0u = -1.f, E1u = 0.f, Tl = 0.f, Tu = 0.f;
#pragma unroll
    for (int i = 0; i < kLinEdges; ++i) {
        if (i == pl) { Al = A[i]; E0l = E0[i]; E1l = E1[i]; Tl = T[i]; }
        if (i == pu) { Au = A[i]; E0u = E0[i]; E1u = E1[i]; Tu = T[i]; }
    }
    // at be: the pair's denominators above a hundredth of their edge (z then errs by 2e-5 of
    // reach + z at the most), its mean height within the prism, every other constraint slack
    // there.  The two bounds meet at the root and the others hold around it, so the arc
    // leaves the prism there toward the lit end.  At the shadowed end any height inside will
    // do: the pair's middle (the pair is open there, since the root lies between it and the
    // lit end), or, where another edge is nearer there, the middle of all constraints' bounds
    // with every constraint slack.
    auto holds = [&](float at) {
        const float dz = fmaf(at, ez, az), denl = fmaf(at, E1l, E0l), denu = fmaf(at, E1u, E0u);
        const float zl = __fdividef(-Al * dz, denl);
        const float z = 0.5f * (zl + (pu < 0 ? h : __fdividef(-Au * dz, denu)));
        return denl > 100.f * Tl && denu < -100.f * Tu && z > zm && (pu < 0 || z < h - zm) && slack(at, z, pl, pu);
    };
    auto inside = [&](float at) {
        float l, u;
        int i, j;
        bounds(at, l, u, i, j);
        const float z = 0.5f * (l + u);
        return z > zm && z < h - zm && slack(at, z, -1, -1);
    };
    const bool ok = fmaf(lit, E1l, E0l) > 100.f * Tl && fmaf(lit, E1u, E0u) < -100.f * Tu && holds(rf) && (holds(sh) || inside(sh));
    if (!ok) return 0;
    *be_star = r;
    return 1;
}

// Buildings hit by the FP32 ray from o toward step s (all hits, not only the first).
__device__ int hit_buildings(const DevScene& sc, const float3& o, const StepConst& s, int* ids) {
    int n = 0;
    int i = 0;
    while (i < sc.n_nodes) {
        const float4 lo = __ldg(&sc.nodes[2 * i]);
        const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
        const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_ADJ_ESCAPE);
        const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_ADJ_LEAF);
        const bool in = hit_box(o, s.ix, s.iy, s.iz, lo, hi);
        if (tri >= 0) {
            if (in) {
                const float4 a = __ldg(&sc.tris[3 * tri]);
                const float4 b = __ldg(&sc.tris[3 * tri + 1]);
                const float4 c = __ldg(&sc.tris[3 * tri + 2]);
                if (hit_tri_any(s.kz, o, a, b, c, s, kGroundTmin)) {
                    const int bid = __float_as_int(a.w);
                    bool seen = false;
                    for (int q = 0; q < n; ++q) seen |= (ids[q] == bid);
                    if (!seen && n < kMaxCand) ids[n++] = bid;
                }
            }
            i = esc;
        } else {
            i = in ? i + 1 : esc;
        }
    }
    return n;
}

struct SolveArgs {
    DevScene sc;
    FootprintSet fs;
    const float* heights;
    const StepConst* steps;
    const ArcConst* arcs;
    float x0, y0, dx;
    int nx;
    const float* weights;
    double dt;
    const int4* flips;
    long long n_flips;
    unsigned* later;         // flips left to the FP64 search, and how many
    unsigned* n_later;
    double* minutes;         // each flip's part of S
    double* dSdh;
};

// The flip of one list entry: adds its minutes to s; returns the building whose roof edge
// casts it and the contribution to that building's derivative, or -1; -2 (FAST) when a
// building's flip is not certified and the whole entry is left to the FP64 search.
template <bool FAST>
__device__ __forceinline__ int solve_flip(const SolveArgs& a, const int4& fl, double& s, double& grad) {
    const long long r = (long long)(unsigned)fl.x | ((long long)fl.y << 31);
    const int j = fl.z, c0 = fl.w;
    const int ix = (int)(r % a.nx), iy = (int)(r / a.nx);
    float3 o;
    o.x = __fadd_rn(a.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), a.dx));
    o.y = __fadd_rn(a.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), a.dx));
    o.z = 0.f;
    const double w = a.weights ? (double)a.weights[r] : 1.0;
    // candidates: buildings hit at the shadowed end
    int ids[kMaxCand];
    const int n = hit_buildings(a.sc, o, a.steps[c0 ? j : j + 1], ids);
    const ArcConst arc = a.arcs[j];
    double best = c0 ? -1.0 : 2.0, best_dh = 0.0;
    int bbest = -1;
    for (int q = 0; q < n; ++q) {
        const int b = ids[q];
        const int fa = a.fs.fp_off[b], v = a.fs.fp_off[b + 1] - fa;
        double be = -1.0, dh = 0.0;
        if (FAST) {
            if (v > kLinEdges || !solve_fast(a.fs, fa, v, a.heights[b], o.x, o.y, arc, c0 != 0, &be, &dh)) return -2;
        } else if (!solve_fp64(a.fs, a.heights, b, (double)o.x, (double)o.y, arc_of(arc), c0 != 0, &be)) {
            continue;
        }
        // the slerp parameter grows with be
        if (c0 ? (be > best) : (be < best)) { best = be; best_dh = dh; bbest = b; }
    }
    if (bbest < 0) {
        // No single building explains the flip in FP64 (a step status decided within FP32
        // rounding of a boundary): the flip time is unknown, count half the interval and
        // no derivative.
        s += 0.5 * a.dt * w;
        return -1;
    }
    const double al = slerp_param(arc, best);
    s += a.dt * w * (c0 ? al : 1.0 - al);
    const double sf = c0 ? 1.0 : -1.0;
    if (FAST) {
        if (best_dh == 0.0) return -1;                            // vertical-edge event
        // d alpha / d be = |d x d'| / (|d|^2 theta) on the arc d = a + be e
        const double dal = arc.inv_theta == 0.0
                               ? 1.0
                               : arc.sin_theta * arc.inv_theta / (1.0 - 2.0 * arc.omc * best * (1.0 - best));
        grad = w * a.dt * sf * best_dh * dal;
        return bbest;
    }
    // is the flip the shadow of a roof edge?  (entry through edge e exactly at height h)
    const int fa = a.fs.fp_off[bbest], v = a.fs.fp_off[bbest + 1] - fa;
    const double h = (double)a.heights[bbest], px = o.x, py = o.y;
    const Arc ac = arc_of(arc);
    const Vec3 d = arc_dir(ac, al);
    const Vec3 dd = arc_ddir(ac, al);
    const double ux = d.x / d.z, uy = d.y / d.z;
    const double dux = (dd.x * d.z - d.x * dd.z) / (d.z * d.z);
    const double duy = (dd.y * d.z - d.y * dd.z) / (d.z * d.z);
    const Entry e = prism(a.fs.xy, fa, v, h, px, py, ux, uy);
    const double tol = 1e-6 * (h + 1.0);
    if (e.elo < 0 || fabs(e.zlo - h) > tol || e.zhi < h - tol) return -1;   // vertical-edge event
    const float2 p0 = a.fs.xy[fa + e.elo], p1 = a.fs.xy[fa + (e.elo + 1 == v ? 0 : e.elo + 1)];
    const double cx = (double)p1.x - (double)p0.x, cy = (double)p1.y - (double)p0.y;
    const double Bc = cx * uy - cy * ux;
    const double dB = cx * duy - cy * dux;
    if (dB == 0.0) return -1;
    grad = w * a.dt * sf * (-Bc / (h * dB));
    return bbest;
}

// One flip per thread: first every flip by the certified search (FAST), then the ones it left
// over, packed so that no warp runs the FP64 search for one lane.  The minutes go to a list
// that is summed in a fixed order (an atomic per flip on S alone serialised at the L2), the
// derivatives are summed per warp and building before their atomics.
template <bool FAST>
__global__ void __launch_bounds__(kSolveThreads) k_flip_solve(SolveArgs a) {
    const int lane = threadIdx.x & 31;
    const long long n = FAST ? a.n_flips : (long long)*a.n_later;
    for (long long f0 = (long long)blockIdx.x * kSolveThreads; f0 < n; f0 += (long long)gridDim.x * kSolveThreads) {
        const long long f = f0 + threadIdx.x;
        double s = 0.0, grad = 0.0;
        int b = -1;
        if (f < n) {
            const long long i = FAST ? f : (long long)a.later[f];
            b = solve_flip<FAST>(a, a.flips[i], s, grad);
            a.minutes[i] = s;
        }
        __syncwarp();
        if (FAST) {
            const unsigned left = __ballot_sync(kFull, b == -2);
            unsigned at = 0;
            if (lane == 0 && left) at = atomicAdd(a.n_later, (unsigned)__popc(left));
            at = __shfl_sync(kFull, at, 0);
            if (b == -2) a.later[at + __popc(left & ((1u << lane) - 1u))] = (unsigned)f;
        }
        // sum over the lanes of the same building (pairs of peers first, then pairs of pairs), and
        // one atomic by its first lane
        const unsigned same = __match_any_sync(kFull, b);
        const int leader = __ffs(same) - 1;
        unsigned above = same & (0xfffffffeu << lane);
        unsigned rank = __popc(same & ((1u << lane) - 1u));
        while (__any_sync(kFull, above != 0u)) {
            const int next = __ffs(above) - 1;
            const double t = __shfl_sync(kFull, grad, next < 0 ? lane : next);
            if (next >= 0) grad += t;
            above &= ~__ballot_sync(kFull, rank & 1u);
            rank >>= 1;
        }
        if (b >= 0 && lane == leader) atomicAdd(&a.dSdh[b], grad);
    }
}

__global__ void k_to_float(const double* __restrict__ in, float* __restrict__ out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)in[i];
}

}  // namespace

cudaError_t launch_height_grad(const DevScene& sc, const FootprintSet& fs, const float* d_heights,
                               const DevRecv& rc, const DevSun& sun, float step_minutes,
                               const float* weights, float* dS_dh, double* d_S, cudaStream_t st) {
    const long long R = (long long)rc.nx * rc.ny;
    cudaError_t e = cudaSuccess;
    double* dsdh = nullptr;
    double* S = nullptr;
    unsigned long long* masks = nullptr;
    unsigned* counts = nullptr;
    unsigned* d_total = nullptr;
    int4* flips = nullptr;
    ArcConst* arcs = nullptr;
    double *steady = nullptr, *minutes = nullptr;
    unsigned* later = nullptr;
    const int B = fs.B;
#define TRY(x) do { e = (x); if (e != cudaSuccess) goto done; } while (0)
    TRY(sa::scratch_alloc(&dsdh, sizeof(double) * (B > 0 ? B : 1), st));
    TRY(sa::scratch_alloc(&S, sizeof(double) * (1 + kSumCtas), st));      // S and its flips' partial sums
    TRY(cudaMemsetAsync(dsdh, 0, sizeof(double) * (B > 0 ? B : 1), st));
    TRY(cudaMemsetAsync(S, 0, sizeof(double) * (1 + kSumCtas), st));
    if (R > 0 && sun.n_blocks > 0) {
        TRY(sa::scratch_alloc(&masks, sizeof(unsigned long long) * (size_t)R * sun.n_blocks, st));
        TRY(cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)R * sun.n_blocks, st));
        {
            DevOut out;
            memset(&out, 0, sizeof(out));                  // only the masks are wanted
            out.masks = reinterpret_cast<uint64_t*>(masks);
            TRY(launch_raster_ground(sc, rc, sun, out, st));
        }
        constexpr int kGroups = 32;         // of blocks, at the most
        FlipOrder go;
        go.nx = rc.nx; go.ny = rc.ny; go.tiles_x = (rc.nx + 7) / 8;
        go.n = 32ll * go.tiles_x * ((rc.ny + 3) / 4);
        go.per = (sun.n_blocks + kGroups - 1) / kGroups;
        long long slots = go.n * ((sun.n_blocks + go.per - 1) / go.per);
        e = sa::scratch_alloc(&counts, sizeof(unsigned) * (size_t)slots, st);
        if (e == cudaErrorMemoryAllocation) {          // no room for the groups' counts: one group
            go.per = sun.n_blocks;
            slots = go.n;
            e = sa::scratch_alloc(&counts, sizeof(unsigned) * (size_t)slots, st);
        }
        if (e != cudaSuccess) goto done;
        TRY(sa::scratch_alloc(&d_total, sizeof(unsigned), st));
        const double dt = step_minutes;
        const unsigned grid = (unsigned)((go.n + 255) / 256);
        TRY(sa::scratch_alloc(&steady, sizeof(double) * (kSumCtas + (size_t)grid), st));
        k_flip_count<<<grid, 256, 0, st>>>(masks, R, go, sun.blocks, sun.n_blocks, weights, dt, counts,
                                           steady + kSumCtas);
        TRY(cudaGetLastError());
        TRY(exclusive_scan_u32(counts, slots, d_total, st));
        unsigned total = 0;
        TRY(cudaMemcpyAsync(&total, d_total, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
        TRY(cudaStreamSynchronize(st));
        if (total > 0) {
            TRY(sa::scratch_alloc(&flips, sizeof(int4) * (size_t)total, st));
            k_flip_fill<<<grid, 256, 0, st>>>(masks, R, go, sun.blocks, sun.n_blocks, counts, flips);
            // the list replaces the masks and counts, whose memory serves what follows
            cudaFreeAsync(masks, st);
            cudaFreeAsync(counts, st);
            masks = nullptr;
            counts = nullptr;
            TRY(sa::scratch_alloc(&arcs, sizeof(ArcConst) * (size_t)sun.S, st));
            k_arcs<<<(sun.S + 127) / 128, 128, 0, st>>>(sun.steps, sun.S - 1, arcs);
            SolveArgs sa;
            sa.arcs = arcs;
            sa.sc = sc; sa.fs = fs; sa.heights = d_heights; sa.steps = sun.steps;
            sa.x0 = rc.x0; sa.y0 = rc.y0; sa.dx = rc.dx; sa.nx = rc.nx;
            sa.weights = weights; sa.dt = dt; sa.flips = flips; sa.n_flips = total;
            TRY(sa::scratch_alloc(&minutes, sizeof(double) * (size_t)total, st));
            sa.minutes = minutes; sa.dSdh = dsdh;
            TRY(sa::scratch_alloc(&later, sizeof(unsigned) * ((size_t)total + 1), st));
            TRY(cudaMemsetAsync(later, 0, sizeof(unsigned), st));
            sa.n_later = later;
            sa.later = later + 1;
            const unsigned ctas = (unsigned)(((long long)total + kSolveThreads - 1) / kSolveThreads);
            k_flip_solve<true><<<ctas, kSolveThreads, 0, st>>>(sa);
            k_flip_solve<false><<<std::min(ctas, 152u * 16u), kSolveThreads, 0, st>>>(sa);
            k_sum<<<kSumCtas, 256, 0, st>>>(minutes, total, S + 1);
            TRY(cudaGetLastError());
        }
        // S: the steady intervals, then the flips
        k_sum<<<kSumCtas, 256, 0, st>>>(steady + kSumCtas, grid, steady);
        k_sum_pair<<<1, 256, 0, st>>>(steady, S + 1, S);
        TRY(cudaGetLastError());
    }
    if (B > 0) k_to_float<<<(B + 255) / 256, 256, 0, st>>>(dsdh, dS_dh, B);
    TRY(cudaGetLastError());
    if (d_S) TRY(cudaMemcpyAsync(d_S, S, sizeof(double), cudaMemcpyDeviceToDevice, st));
done:
    if (dsdh) cudaFreeAsync(dsdh, st);
    if (S) cudaFreeAsync(S, st);
    if (masks) cudaFreeAsync(masks, st);
    if (counts) cudaFreeAsync(counts, st);
    if (d_total) cudaFreeAsync(d_total, st);
    if (flips) cudaFreeAsync(flips, st);
    if (arcs) cudaFreeAsync(arcs, st);
    if (later) cudaFreeAsync(later, st);
    if (steady) cudaFreeAsync(steady, st);
    if (minutes) cudaFreeAsync(minutes, st);
    return e;
#undef TRY
}

}  // namespace sa
