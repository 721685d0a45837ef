// A CTA's grouped walk (walk_group) over a made-up node list: a flat sun straight above, so that
// a node is entered when its box meets the group's.  Counts how often each triangle is
// staged and how many nodes are visited.  Built with -DSA_CHECKED by the test that loads it.
#include <string.h>

#include <vector>

#include "sa_light.cuh"

namespace sa {
int register_check_reader(CheckReader) { return 0; }

template <int CHUNK, int STACK>
__global__ void __launch_bounds__(kTileThreads) k_walk(DevScene sc, RunLight rl, unsigned* staged, unsigned long long* visits) {
    __shared__ LightSmem<CHUNK> sm;
    __shared__ GroupSmem<CHUNK, STACK> gs;
    const float4 p = make_float4((float)threadIdx.x, 0.f, 0.f, 0.f);
    sm.o[threadIdx.x] = p;
    sm.m[threadIdx.x] = 0u;
    unsigned long long n_box = 0;
    walk_group<true>(sm, gs, sc, rl, true, p, [staged](int tri) { atomicAdd(&staged[tri], 1u); return 1u; }, n_box,
                     [](int, float, float) { return false; });
    atomicAdd(visits, n_box);
}
}  // namespace sa

// nodes: float [n][8] (lo.xyz, escape link's bits, hi.xyz, triangle's bits); word: the check's
// [site, index, bound].  Returns the CUDA error.
extern "C" int run_walk(const float* nodes, int n, int T, int small, unsigned* staged, unsigned long long* visits,
                        unsigned long long* word) {
    using namespace sa;
    float4 *dn = nullptr, *dt = nullptr;
    unsigned* ds = nullptr;
    unsigned long long* dv = nullptr;
    const float up[3] = {0.f, 0.f, 1.f};
    RunLight rl;
    memset(&rl, 0, sizeof(rl));
    rl.e1[0] = rl.e2[1] = 1.f;
    memcpy(rl.dm, up, sizeof(up));
    rl.kn = 1;
    cudaError_t e = cudaMalloc(&dn, sizeof(float) * 8 * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dt, sizeof(float4) * 3 * (size_t)T);
    if (e == cudaSuccess) e = cudaMalloc(&ds, sizeof(unsigned) * (size_t)T);
    if (e == cudaSuccess) e = cudaMalloc(&dv, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemcpy(dn, nodes, sizeof(float) * 8 * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(dt, 0, sizeof(float4) * 3 * (size_t)T);
    if (e == cudaSuccess) e = cudaMemset(ds, 0, sizeof(unsigned) * (size_t)T);
    if (e == cudaSuccess) e = cudaMemset(dv, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) {
        DevScene sc{};
        sc.nodes = dn;
        sc.tris = dt;
        sc.n_nodes = n;
        sc.T = T;
        if (small) k_walk<64, 512><<<1, kTileThreads>>>(sc, rl, ds, dv);
        else k_walk<128, 1024><<<1, kTileThreads>>>(sc, rl, ds, dv);
        e = cudaDeviceSynchronize();
    }
    if (e == cudaSuccess) e = cudaMemcpy(staged, ds, sizeof(unsigned) * (size_t)T, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(visits, dv, sizeof(unsigned long long), cudaMemcpyDeviceToHost);
    word[0] = word[1] = word[2] = 0ull;
    if (e == cudaSuccess) e = sa_read_check_tu(word, 1);
    for (void* p : {(void*)dn, (void*)dt, (void*)ds, (void*)dv})
        if (p) cudaFree(p);
    return (int)e;
}
