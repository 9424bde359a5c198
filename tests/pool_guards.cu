// Pooled walks over trees given by the caller, for tests/test_gpu_pool_guards.py: trees that the scene builder refuses.
#include <cuda_runtime.h>

#include "pt_pool.cuh"

namespace {

using namespace pt;

struct Io {
    const DevScene& s;
    float* t;
    uint32_t* tri;
    __device__ DevScene scene() const { return s; }
    // every slot's ray starts at the origin and goes up the x axis; slots with kAnySlot look for an occluder before 5000
    __device__ void fetch(uint32_t slot, float3& o, float3& d, float& tbest, uint32_t& best, const float4*&,
                          const float4*&) const {
        o = f3(0.f, 0.f, 0.f);
        d = f3(1.f, 0.f, 0.f);
        tbest = (slot & kAnySlot) ? 5000.f : __int_as_float(0x7f800000);
        best = kMiss;
    }
    __device__ void emit(uint32_t slot, float th, uint32_t hit, uint32_t) const {
        const uint32_t i = (slot & ~kAnySlot) * 2u + (slot >> 31);
        t[i] = th;
        tri[i] = hit;
    }
};

template <bool INST, bool SHARE>
__global__ void __launch_bounds__(32) k_walk(const __grid_constant__ DevScene s, uint32_t n, uint32_t* counter, float* t,
                                             uint32_t* tri) {
    SlotPool q(counter, 2u * n);          // n closest-hit slots, then n any-hit slots
    pool_walk<INST, SHARE>(s, q, n, Io{s, t, tri});
}

}  // namespace

// One warp walks n closest-hit and n any-hit rays; t and tri hold both results of ray i at 2 i and 2 i + 1.  All pointers
// are host memory.  inst (and with it tlas) may be null: a single-level scene.
extern "C" int pool_guards_run(const float* nodes, uint32_t n_nodes, const float* tris, uint32_t n_tris, const float* tlas,
                               uint32_t n_tlas, const float* inst, uint32_t n_inst, uint32_t n, int share, float* t,
                               uint32_t* tri, uint32_t* status) {
    float4 *dn, *dt, *da = nullptr, *di = nullptr;
    uint32_t* words;
    float* dth;
    uint32_t* dtri;
    cudaMalloc(&dn, n_nodes * 64);
    cudaMalloc(&dt, n_tris * 48);
    cudaMalloc(&words, 256);
    cudaMalloc(&dth, 8 * n);
    cudaMalloc(&dtri, 8 * n);
    cudaMemcpy(dn, nodes, n_nodes * 64, cudaMemcpyHostToDevice);
    cudaMemcpy(dt, tris, n_tris * 48, cudaMemcpyHostToDevice);
    cudaMemset(words, 0, 256);
    if (inst) {
        cudaMalloc(&da, n_tlas * 64);
        cudaMalloc(&di, n_inst * 128);
        cudaMemcpy(da, tlas, n_tlas * 64, cudaMemcpyHostToDevice);
        cudaMemcpy(di, inst, n_inst * 128, cudaMemcpyHostToDevice);
    }
    DevScene s{};
    s.nodes = dn;
    s.tris = dt;
    s.status = words + 32;
    s.tlas = da;
    s.inst = di;
    if (inst) k_walk<true, false><<<1, 32>>>(s, n, words, dth, dtri);
    else if (share) k_walk<false, true><<<1, 32>>>(s, n, words, dth, dtri);
    else k_walk<false, false><<<1, 32>>>(s, n, words, dth, dtri);
    const cudaError_t e = cudaDeviceSynchronize();
    cudaMemcpy(t, dth, 8 * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(tri, dtri, 8 * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(status, words + 32, 4, cudaMemcpyDeviceToHost);
    cudaFree(dn);
    cudaFree(dt);
    cudaFree(da);
    cudaFree(di);
    cudaFree(words);
    cudaFree(dth);
    cudaFree(dtri);
    return (int)e;
}
