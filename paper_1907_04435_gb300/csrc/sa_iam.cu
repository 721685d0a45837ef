// sa_iam.cu -- inverse accrual map (Sec. 5) of a ground receiver grid.
//
// Per block of K steps:
//   k_iam_draw  every cell centre p traces toward the sun at the block's first step and
//               keeps the L nearest intersections farther than 1 m (the paper's source
//               levels and its 100 cm acne rule).  Each source s casts its shadow at step
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

// Slab test with an upper bound on the entry distance.
__device__ __forceinline__ bool hit_box_before(const float3& o, const StepConst& s, const float4& lo,
                                               const float4& hi, float tmax) {
    float tx0 = (lo.x - o.x) * s.ix, tx1 = (hi.x - o.x) * s.ix;
    float ty0 = (lo.y - o.y) * s.iy, ty1 = (hi.y - o.y) * s.iy;
    float tz0 = (lo.z - o.z) * s.iz, tz1 = (hi.z - o.z) * s.iz;
    float tn = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.f));
    float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fmaxf(tz0, tz1));
    return tn <= tf * 1.0000005f && tn <= tmax;
}

// The L nearest hits (ascending) of the ray from o along step s; warp-coherent traversal.
template <int KZ>
__device__ int nearest_sources(const DevScene& sc, const float3& o, const StepConst& s,
                               bool active, int L, float* best) {
    int n = 0;
    int i = 0;
    while (i < sc.n_nodes && __any_sync(kFull, active)) {
        const float4 lo = __ldg(&sc.nodes[2 * i]);
        const float4 hi = __ldg(&sc.nodes[2 * i + 1]);
        const int esc = SA_ESC(__float_as_int(lo.w), i, sc.n_nodes, sa::CK_IAM_ESCAPE);
        const int tri = SA_LEAF(__float_as_int(hi.w), sc.T, sa::CK_IAM_LEAF);
        const float bound = n < L ? 3.4e38f : best[L - 1];
        const bool in = active && hit_box_before(o, s, lo, hi, bound);
        if (tri >= 0) {
            if (in) {
                const float4 a = __ldg(&sc.tris[3 * tri]);
                const float4 b = __ldg(&sc.tris[3 * tri + 1]);
                const float4 c = __ldg(&sc.tris[3 * tri + 2]);
                float t;
                if (hit_tri_t<KZ>(o, a, b, c, s.Sx, s.Sy, s.Sz, kSourceTmin, &t) && t < bound) {
                    int k = n < L ? n++ : L - 1;
                    while (k > 0 && best[k - 1] > t) { best[k] = best[k - 1]; --k; }
                    best[k] = t;
                }
            }
            i = esc;
        } else {
            i = __any_sync(kFull, in) ? i + 1 : esc;
        }
    }
    return n;
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

// A CTA finds the sources of its 128 cells, 32 in a patch of 8 x 4 per warp, and lists them;
// then its threads draw them, one line per thread whichever cell it comes from: most cells
// are lit or have two sources where their neighbours have four, and a warp that drew its own
// cells' sources waited for the longest list.  Bound by issue: the pieces of the lines, one
// after the other (12 CTAs per SM: 2.17 ms the call, 2.21 at 10, 2.24 at 14).  613 x 457
// cells x 481 steps: 2.76 ms with each thread's own sources, 2.17; 1024^2 9.84 -> 7.79; 400 x
// 300 on 21 December, when most cells have all four, 3.23 -> 3.13.
template <class Cell>
__global__ void __launch_bounds__(32 * kWarps, 12)
k_iam_draw(DevScene sc, Grid g, const StepConst* __restrict__ steps, const BlockConst* __restrict__ blocks,
           int L, unsigned long long* __restrict__ all_masks) {
    __shared__ float s_t[32 * kWarps * kMaxLevels * 2];               // the sources' distances,
    __shared__ unsigned short s_from[32 * kWarps * kMaxLevels * 2];   // thread | direction << 15
    __shared__ float2 s_o[32 * kWarps], s_u[kMaxBlock];
    __shared__ int s_n;
    const int tid = threadIdx.x, lane = tid & 31;
    const int j0 = blocks[blockIdx.y].j0, K = blocks[blockIdx.y].K;
    const long long warp_id = (long long)blockIdx.x * kWarps + (tid >> 5);
    const int tiles_x = (g.nx + 7) >> 3;
    const long long ty = warp_id / tiles_x;
    const int tx = (int)(warp_id - ty * tiles_x);
    const int ix = tx * 8 + (lane & 7);
    const long long iy = ty * 4 + (lane >> 3);
    const bool active = ix < g.nx && iy < g.ny;
    float3 o;
    o.x = __fadd_rn(g.x0, __fmul_rn(__fadd_rn((float)ix, 0.5f), g.dx));
    o.y = __fadd_rn(g.y0, __fmul_rn(__fadd_rn((float)iy, 0.5f), g.dx));
    o.z = 0.f;
    s_o[tid] = make_float2(o.x, o.y);
    if (tid < K) s_u[tid] = make_float2(steps[j0 + tid].ux, steps[j0 + tid].uy);
    if (tid == 0) s_n = 0;
    __syncthreads();
    for (int dir = 0; dir < 2; ++dir) {
        const StepConst s = steps[dir == 0 ? j0 : j0 + K - 1];
        float best[kMaxLevels];
        int n;
        if (s.kz == 2) n = nearest_sources<2>(sc, o, s, active, L, best);
        else if (s.kz == 0) n = nearest_sources<0>(sc, o, s, active, L, best);
        else n = nearest_sources<1>(sc, o, s, active, L, best);
        // level by level, so that neighbours' lines of one source surface stay together
        for (int l = 0; l < L; ++l) {
            const unsigned has = __ballot_sync(kFull, l < n);
            if (!has) break;
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_n, __popc(has));
            at = __shfl_sync(kFull, at, 0) + __popc(has & ((1u << lane) - 1u));
            if (l < n) {
                s_t[at] = best[l];
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

cudaError_t launch_iam(const DevScene& sc, const DevRecv& rc, const DevSun& sun,
                       int L, const DevOut& out, cudaStream_t st) {
    const long long R = (long long)rc.nx * rc.ny;
    if (R == 0) return cudaSuccess;
    if (L < 1 || L > kMaxLevels) return cudaErrorInvalidValue;
    // the blocks go in one launch, as many as 1 GiB of masks holds
    const int chunk = (int)std::max(1ll, std::min({(long long)sun.n_blocks, 65535ll, (1ll << 30) / (8ll * R)}));
    const size_t words = (size_t)R * chunk;
    unsigned long long* masks = nullptr;
    cudaError_t e = sa::scratch_alloc(&masks, sizeof(unsigned long long) * words, st);
    if (e != cudaSuccess) return e;
    Grid g{rc.x0, rc.y0, rc.dx, rc.nx, rc.ny};
    const long long warps = (long long)((rc.nx + 7) / 8) * ((rc.ny + 3) / 4);
    const unsigned ctas = (unsigned)((warps + kWarps - 1) / kWarps);
    for (int b0 = 0; b0 < sun.n_blocks && e == cudaSuccess; b0 += chunk) {
        const int nbc = std::min(chunk, sun.n_blocks - b0);
        e = cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)R * nbc, st);
        if (e != cudaSuccess) break;
        {
            KernelTimer kt(KT_IAM, st);
            const dim3 grid(ctas, (unsigned)nbc);
            if (R < (1ll << 31)) k_iam_draw<unsigned><<<grid, 32 * kWarps, 0, st>>>(sc, g, sun.steps, sun.blocks + b0, L, masks);
            else k_iam_draw<long long><<<grid, 32 * kWarps, 0, st>>>(sc, g, sun.steps, sun.blocks + b0, L, masks);
        }
        k_iam_fold<<<(unsigned)((R + 255) / 256), 256, 0, st>>>(R, sun.blocks + b0, nbc, masks, out, b0 == 0,
                                                               b0 + nbc == sun.n_blocks);
        e = cudaGetLastError();
    }
    cudaError_t e2 = cudaFreeAsync(masks, st);
    return e != cudaSuccess ? e : e2;
}

}  // namespace sa
