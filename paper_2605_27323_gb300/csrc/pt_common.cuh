// pt_common.cuh -- device helpers shared by the kernel translation units: warp-aggregated
// atomics, the per-path event recorders, the megakernel's path and bounce functions (also the
// body of the wavefront's hybrid continuation kernel), the wavefront's scene sources and the
// adjoint's record type and warp-aggregated gradient accumulation.
#pragma once
#include <cstdio>

#include "pt_device.cuh"
#include "pt_launch.h"
#include "pt_trace.cuh"

namespace pt {

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Programmatic dependent launch (sm_90+): a stage kernel that the host launches with the
// programmatic-serialization attribute may begin while the previous kernel of its stream drains.
// It first waits until that kernel has finished and its writes are visible (a no-op when launched
// normally), then lets the next kernel of the stream begin its own launch, whose blocks become
// resident as this kernel's blocks exit and wait in the same way.
__device__ __forceinline__ void stage_prologue() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch through cudaLaunchKernelEx with the programmatic-serialization attribute when l.pdl is set
// (the kernel must begin with stage_prologue()), else as an ordinary launch.
template <class... KArgs, class... Args>
cudaError_t launch_k(const Launch& l, size_t smem, void (*k)(KArgs...), Args... args) {
    if (!l.pdl) {
        k<<<l.grid, l.block, smem, l.st>>>(args...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)l.grid);
    cfg.blockDim = dim3((unsigned)l.block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = l.st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Warp-aggregated append to the shadow queue and the ray queue (stream compaction, Sec. 3.1): every lane
// of the warp calls it; lanes with `shadow` / `ray` receive consecutive slots of each from a single 64-bit
// atomic on the pair of counts (neither carries: they stay below the queue capacity < 2^32).  Atomics on
// one address complete about every 1.5 ns, which bounds the shading of a dense queue: with one atomic
// per warp and queue 2 M camera hits took 135 us, with one for both 101 us.  (One per block of 256 needs
// barriers that cost more than they save: 111 us.)
__device__ __forceinline__ void warp_append2(BounceCounts* next, bool shadow, bool ray, uint32_t& k, uint32_t& q) {
    const uint32_t ms = __ballot_sync(0xFFFFFFFFu, shadow), mr = __ballot_sync(0xFFFFFFFFu, ray);
    unsigned long long base = 0ull;
    if (lane_id() == 0u && (ms | mr))
        base = atomicAdd(reinterpret_cast<unsigned long long*>(next),
                         (unsigned long long)__popc(ms) | (unsigned long long)__popc(mr) << 32);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    const uint32_t below = (1u << lane_id()) - 1u;
    k = (uint32_t)base + (uint32_t)__popc(ms & below);
    q = (uint32_t)(base >> 32) + (uint32_t)__popc(mr & below);
}

// Warp-granular dynamic work: the queue is cut into chunks (32 slots, one per lane; 32 / G when groups
// of G lanes share a ray).  A warp's first chunk is its own index in the grid; it claims every further
// one with one atomic, so warps that drew cheap rays take more chunks and the grid ends together (a
// static grid-stride split leaves the SMs waiting on the warps that drew the longest rays).
// `counter` is zero at launch.
__device__ __forceinline__ uint32_t first_chunk() { return (blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ uint32_t next_chunk(uint32_t* counter) {
    uint32_t b = 0u;
    if (lane_id() == 0u) b = atomicAdd(counter, 1u);
    return ((gridDim.x * blockDim.x) >> 5) + __shfl_sync(0xFFFFFFFFu, b, 0);
}

// Slots [0, total) taken by the warps of a grid (the pooled walks).  A warp's first slots, up to one per
// lane, are its own by its place in the grid; after those it claims, with one atomic, exactly what its idle
// lanes need when they need it, so that no warp sits on slots while others run dry: with runs of 32 held and
// the next run claimed ahead, warps ran dry 190 to 300 us into the 320 us walk of 2 M camera rays (1080p frame
// 1.77 -> 1.67 ms, its two-level form 1.77 -> 1.65, 128 x 128 box 283 -> 256 us; claiming ahead except for the
// last 32, 64, 96, 128, 192 slots per warp: 1.744, 1.712, 1.697, 1.685, 1.676).  `counter` is zero at launch.
struct SlotPool {
    uint32_t* counter;
    uint32_t total, first;               // slots, and those that need no claim
    uint32_t own, own_end;               // the warp's first slots
    uint32_t seen;                       // slots up to here are taken for certain
    __device__ __forceinline__ SlotPool(uint32_t* ctr, uint32_t n) : counter(ctr), total(n), seen(0u) {
        const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
        const uint32_t size = min(32u, (n + n_warps - 1u) / n_warps);
        own = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * size;
        own_end = own + size;
        first = n_warps * size;
    }
    __device__ __forceinline__ bool more() const { return seen < total; }
    // This lane's slot of those handed to the lanes of `idle` (all 32 lanes call it), or >= total.
    __device__ __forceinline__ uint32_t take(uint32_t idle) {
        const uint32_t k = (uint32_t)__popc(idle), rank = (uint32_t)__popc(idle & ((1u << lane_id()) - 1u));
        uint32_t j;
        if (seen == 0u) {                // the first call finds every lane idle
            j = own + rank < own_end ? own + rank : total;
            seen = first;
        } else {
            uint32_t b = 0u;
            if (lane_id() == 0u) b = atomicAdd(counter, k);
            b = first + __shfl_sync(0xFFFFFFFFu, b, 0);
            j = b + rank;
            seen = b + k;
        }
        return ((idle >> lane_id()) & 1u) ? j : total;
    }
};

// The same slots dealt out without a counter, runs of 32 to the warps in turn (closest-hit queries, which keep no
// state between calls: calls on one scene may overlap on several streams).
struct DealtPool {
    uint32_t total, n_warps, warp;
    uint32_t used = 0u;                  // of the warp's own sequence
    __device__ __forceinline__ explicit DealtPool(uint32_t n) : total(n) {
        n_warps = (gridDim.x * blockDim.x) >> 5;
        warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    }
    __device__ __forceinline__ uint32_t slot(uint32_t i) const {
        const uint64_t j = ((uint64_t)(i >> 5) * n_warps + warp) * 32u + (i & 31u);
        return j < total ? (uint32_t)j : total;
    }
    __device__ __forceinline__ bool more() const { return slot(used) < total; }
    __device__ __forceinline__ uint32_t take(uint32_t idle) {
        const uint32_t rank = (uint32_t)__popc(idle & ((1u << lane_id()) - 1u));
        const uint32_t j = slot(used + rank);
        used += (uint32_t)__popc(idle);
        return ((idle >> lane_id()) & 1u) ? j : total;
    }
};

__device__ __forceinline__ void warp_add_u64(unsigned long long* dst, unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    if (lane_id() == 0 && v) atomicAdd(dst, v);
}

__device__ __forceinline__ float4 f4(float3 a, float w) { return make_float4(a.x, a.y, a.z, w); }

// ================================================================== megakernel
// Event recorders of one path (compile-time: the production kernel records nothing).
struct NoRec {
    __device__ __forceinline__ void ev(uint32_t, uint32_t, uint32_t, float, float) {}
};
struct SigRec {   // order-free branch signature
    uint32_t sg = 0;
    __device__ __forceinline__ void ev(uint32_t b, uint32_t k, uint32_t v, float, float) { sg ^= sig_event(b, k, v); }
};
struct LogRec {   // event list with two diagnostic numbers per event (testing aid)
    uint32_t* ev_u;
    float* ev_f;
    uint32_t n = 0;
    __device__ __forceinline__ void ev(uint32_t b, uint32_t k, uint32_t v, float f0, float f1) {
        if (n >= kMaxEvents) return;
        ev_u[2 * n] = (b << 4) | k;
        ev_u[2 * n + 1] = v;
        ev_f[2 * n] = f0;
        ev_f[2 * n + 1] = f1;
        ++n;
    }
};

// One whole path (Sec. 2.2 steps 1-5) in registers: the body of the megakernel.
template <class Rec, bool MIS, bool INST>
__device__ __forceinline__ float3 mk_path(const DevScene& s, const DevCamera& c, const RenderParams& p, uint64_t path,
                                          Rec& rec, uint32_t& n_ext, uint32_t& n_shd) {
    const float3 env = f3(s.env_r, s.env_g, s.env_b);
    const uint32_t pixel = (uint32_t)(path / p.spp);
    const uint32_t sample = p.sample_offset + (uint32_t)(path - (uint64_t)pixel * p.spp);
    const uint32_t key = path_key(p.seed, pixel, sample);
    float3 o, d;
    float u0, u1;
    pixel_jitter(p.sampler, p.seed, pixel, sample, key, u0, u1);
    camera_ray(c, pixel, u0, u1, o, d);                        // step 1
    float3 tp = f3(1.f, 1.f, 1.f), L = f3(0.f, 0.f, 0.f);
    bool prev_delta = true;
    float prev_pdf = 0.f;
    for (uint32_t b = 0; b < p.max_depth; ++b) {
        ++n_ext;
        Hit h;                                                 // step 2
        if constexpr (INST) h = trace_closest_inst<false, false>(s, o, d);
        else h = trace_closest(s, o, d);
        if (h.tri == kMiss) {
            L = add_rn(L, mul_rn(tp, env));
            rec.ev(b, 0, kMiss, __int_as_float(0x7f800000), tp.x);
            break;
        }
        Vertex V = shade_vertex<MIS, INST>(s, p, key, b, o, d, tp, prev_delta, prev_pdf, h.t, h.tri, h.inst);
        rec.ev(b, 0, V.prim, h.t, tp.x);
        if (V.emit_counted) L = add_rn(L, V.emit);             // step 3
        if (V.last) break;
        if (V.nee) {                                           // shadow evaluation
            uint32_t vis = 0;
            if (V.cast) {
                ++n_shd;
                bool occluded;
                if constexpr (INST) occluded = trace_any_inst<false, false>(s, V.s_o, V.s_d, V.s_tmax);
                else occluded = trace_any(s, V.s_o, V.s_d, V.s_tmax);
                vis = occluded ? 0u : 1u;
                if (vis) L = add_rn(L, V.contrib);
            }
            rec.ev(b, 1, (V.light_j << 2) | ((uint32_t)V.cast << 1) | vis, V.nee_cx, V.nee_cl);
        }
        rec.ev(b, 2, V.bsdf_code, V.w.x, V.nd.x);
        if (V.rr >= 0) rec.ev(b, 3, (uint32_t)V.rr, V.rr_q, u01(key, b, D_RR));
        if (!V.cont) break;                                    // step 4 done; step 5: repeat
        o = V.no;
        d = V.nd;
        tp = V.ntp;
        prev_delta = V.delta;
        prev_pdf = V.pdf;
    }
    return L;
}

// One bounce of a path held in registers (extend, shade, shadow evaluation), the loop body of the
// regenerating megakernel and of the wavefront's continuation kernel.  Returns true when the path
// ends; otherwise the state has moved to bounce b + 1.
// SK: shared-memory short-stack entries of the walks (0: local stack; see trace_closest).  cc, ca:
// traversal counters of the closest-hit and any-hit walks (NoCount: none).
template <bool SIG, bool MIS, bool INST, int SK = 0, class C = NoCount>
__device__ __forceinline__ bool mk_bounce(const DevScene& s, const RenderParams& p, float3 env, uint32_t key,
                                          uint32_t& b, float3& o, float3& d, float3& tp, bool& prev_delta,
                                          float& prev_pdf, float3& L, uint32_t& sg, uint32_t& n_ext,
                                          uint32_t& n_shd, C& cc, C& ca) {
    ++n_ext;
    Hit h = trace_closest<INST, SK, !INST>(s, o, d, cc);
    if (h.tri == kMiss) {
        L = add_rn(L, mul_rn(tp, env));
        if (SIG) sg ^= sig_event(b, 0, kMiss);
        return true;
    }
    Vertex V = shade_vertex<MIS, INST>(s, p, key, b, o, d, tp, prev_delta, prev_pdf, h.t, h.tri, h.inst);
    if (SIG) sg ^= sig_event(b, 0, V.prim);
    if (V.emit_counted) L = add_rn(L, V.emit);
    if (V.last) return true;
    if (V.nee) {
        uint32_t vis = 0;
        if (V.cast) {
            ++n_shd;
            vis = trace_any<INST, SK, !INST>(s, V.s_o, V.s_d, V.s_tmax, ca) ? 0u : 1u;
            if (vis) L = add_rn(L, V.contrib);
        }
        if (SIG) sg ^= sig_event(b, 1, (V.light_j << 2) | ((uint32_t)V.cast << 1) | vis);
    }
    if (SIG) {
        sg ^= sig_event(b, 2, V.bsdf_code);
        if (V.rr >= 0) sg ^= sig_event(b, 3, (uint32_t)V.rr);
    }
    if (!V.cont) return true;
    o = V.no;
    d = V.nd;
    tp = V.ntp;
    prev_delta = V.delta;
    prev_pdf = V.pdf;
    ++b;
    return false;
}
template <bool SIG, bool MIS, bool INST, int SK = 0>
__device__ __forceinline__ bool mk_bounce(const DevScene& s, const RenderParams& p, float3 env, uint32_t key,
                                          uint32_t& b, float3& o, float3& d, float3& tp, bool& prev_delta,
                                          float& prev_pdf, float3& L, uint32_t& sg, uint32_t& n_ext,
                                          uint32_t& n_shd) {
    NoCount cc, ca;
    return mk_bounce<SIG, MIS, INST, SK>(s, p, env, key, b, o, d, tp, prev_delta, prev_pdf, L, sg, n_ext, n_shd, cc,
                                         ca);
}

// Counting instantiations: the warp's node and triangle counts added to s.trav[k], s.trav[k + 1]
// (all 32 lanes call it, converged).
template <class C>
__device__ __forceinline__ void flush_count(const DevScene& s, const C& c, int k);
template <>
__device__ __forceinline__ void flush_count<NoCount>(const DevScene&, const NoCount&, int) {}
template <>
__device__ __forceinline__ void flush_count<TravCount>(const DevScene& s, const TravCount& c, int k) {
    warp_add_u64(s.trav + k, c.nodes);
    warp_add_u64(s.trav + k + 1, c.tris);
}

// ================================================================== wavefront stages
// Scene sources: where a wavefront kernel finds the scene, camera and path numbering of a queue
// entry.  SingleSrc: one scene passed by value (pt_render).  TableSrc: many scenes in device
// tables, the scene found from the global path id by binary search over the scenes' first path ids
// (pt_render_batch).  The per-path arithmetic is the same shared device code either way.
struct PathLoc {
    uint64_t path;     // global path id (signature index)
    uint32_t pixel, sample, sid;
};

struct SingleSrc {
    DevScene s;
    DevCamera c;
    RenderParams p;
    __device__ __forceinline__ uint64_t base() const { return p.path_begin; }
    __device__ __forceinline__ uint32_t sid_of(uint64_t, uint32_t) const { return 0; }
    __device__ __forceinline__ PathLoc locate(uint64_t base, uint32_t pid) const {
        PathLoc l;
        l.path = base + pid;
        l.pixel = (uint32_t)(l.path / p.spp);
        l.sample = p.sample_offset + (uint32_t)(l.path - (uint64_t)l.pixel * p.spp);
        l.sid = 0;
        return l;
    }
    __device__ __forceinline__ DevScene scene(uint32_t) const { return s; }
    __device__ __forceinline__ DevCamera camera(uint32_t) const { return c; }
    __device__ __forceinline__ RenderParams params(uint32_t) const { return p; }
    // scene id carried in the queue records: none needed for one scene
    __device__ __forceinline__ uint32_t ray_tag(uint32_t, uint32_t flags) const { return flags; }
    __device__ __forceinline__ uint32_t sid_from_ray(float) const { return 0; }
    __device__ __forceinline__ float3 eye(uint32_t) const { return f3(p.ex, p.ey, p.ez); }
    __device__ __forceinline__ uint32_t shadow_tag(uint32_t light_j, uint32_t) const { return light_j; }
    __device__ __forceinline__ uint32_t sid_from_shadow(float, uint64_t, uint32_t) const { return 0; }
    __device__ __forceinline__ PathLoc locate_in(uint64_t base, uint32_t pid, uint32_t) const { return locate(base, pid); }
};

struct TableSrc {
    BatchTables t;
    RenderParams p;    // depth and roulette (spp per scene and the seed from the tables)
    __device__ __forceinline__ uint64_t base() const { return *t.wave_base; }
    __device__ __forceinline__ uint32_t sid_of(uint64_t base, uint32_t pid) const {
        const uint64_t g = base + pid;
        uint32_t lo = 0, hi = t.n - 1;                  // last scene with off[s] <= g
        while (lo < hi) {
            uint32_t mid = (lo + hi + 1) >> 1;
            if (__ldg(t.off + mid) <= g) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }
    __device__ __forceinline__ PathLoc locate(uint64_t base, uint32_t pid) const {
        PathLoc l;
        l.sid = sid_of(base, pid);
        l.path = base + pid;
        const uint64_t local = l.path - __ldg(t.off + l.sid);
        const uint32_t spp = __ldg(t.spp + l.sid);
        l.pixel = (uint32_t)(local / spp);
        l.sample = (uint32_t)(local - (uint64_t)l.pixel * spp);
        return l;
    }
    __device__ __forceinline__ DevScene scene(uint32_t sid) const { return t.scenes[sid]; }
    __device__ __forceinline__ DevCamera camera(uint32_t sid) const { return t.cams[sid]; }
    __device__ __forceinline__ RenderParams params(uint32_t sid) const {
        RenderParams q = p;
        q.spp = __ldg(t.spp + sid);
        q.seed = __ldg(t.seed);
        return q;
    }
    // the scene id rides in the records' spare bits: ray d.w = flags | sid << 8; shadow c.w = sid
    __device__ __forceinline__ uint32_t ray_tag(uint32_t sid, uint32_t flags) const { return flags | (sid << 8); }
    __device__ __forceinline__ uint32_t sid_from_ray(float dw) const { return __float_as_uint(dw) >> 8; }
    __device__ __forceinline__ float3 eye(uint32_t sid) const {
        return f3(t.cams[sid].ex, t.cams[sid].ey, t.cams[sid].ez);
    }
    __device__ __forceinline__ uint32_t shadow_tag(uint32_t, uint32_t sid) const { return sid; }
    __device__ __forceinline__ uint32_t sid_from_shadow(float cw, uint64_t, uint32_t) const {
        return __float_as_uint(cw);
    }
    __device__ __forceinline__ PathLoc locate_in(uint64_t base, uint32_t pid, uint32_t sid) const {
        PathLoc l;
        l.sid = sid;
        l.path = base + pid;
        const uint64_t local = l.path - __ldg(t.off + sid);
        const uint32_t spp = __ldg(t.spp + sid);
        l.pixel = (uint32_t)(local / spp);
        l.sample = (uint32_t)(local - (uint64_t)l.pixel * spp);
        return l;
    }
};

// ================================================================== adjoint (path replay)
struct AdjRec {
    float3 tp;       // throughput arriving at the vertex
    float3 w;        // throughput multiplier of the continuation (BSDF weight / q)
    float3 dwa;      // d w / d albedo
    float3 nee_g;    // f G A of a visible NEE sample (0 otherwise)
    float3 nee_dfa;  // d(f G A Le_light) / d albedo
    float Le;        // emission of the hit material times its weight when its term is counted
    float we;        // that weight (1, or the MIS weight of a BSDF-sampled light hit)
    float Lj;        // emission of the sampled light's material
    uint32_t mat, lmat;
    uint32_t flags;  // 1: continues, 2: NEE visible, 4: emission counted
};

constexpr uint32_t kNoKey = 0xFFFFFFFFu;

// Warp-aggregated accumulation into per-material gradients: lanes holding the same key add their
// values once (one atomic per distinct key per warp).  All 32 lanes call it; key == kNoKey means
// nothing to add.  v = (d/d albedo rgb, d/d emission).
__device__ __forceinline__ void warp_accumulate(float* acc, float* g_alb, float* g_em, bool smem, uint32_t key,
                                                float4 v) {
    uint32_t pending = __ballot_sync(0xFFFFFFFFu, key != kNoKey);
    while (pending) {
        const uint32_t leader = __ffs(pending) - 1u;
        const uint32_t k = __shfl_sync(0xFFFFFFFFu, key, leader);
        const bool mine = key == k;
        const uint32_t grp = __ballot_sync(0xFFFFFFFFu, mine);
        float4 sum = mine ? v : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int o = 16; o > 0; o >>= 1) {
            sum.x += __shfl_xor_sync(0xFFFFFFFFu, sum.x, o);
            sum.y += __shfl_xor_sync(0xFFFFFFFFu, sum.y, o);
            sum.z += __shfl_xor_sync(0xFFFFFFFFu, sum.z, o);
            sum.w += __shfl_xor_sync(0xFFFFFFFFu, sum.w, o);
        }
        if (lane_id() == leader) {
            if (smem) {
                if (sum.x != 0.f) atomicAdd(&acc[4 * k], sum.x);
                if (sum.y != 0.f) atomicAdd(&acc[4 * k + 1], sum.y);
                if (sum.z != 0.f) atomicAdd(&acc[4 * k + 2], sum.z);
                if (sum.w != 0.f) atomicAdd(&acc[4 * k + 3], sum.w);
            } else {
                if (sum.x != 0.f) atomicAdd(&g_alb[3 * k], sum.x);
                if (sum.y != 0.f) atomicAdd(&g_alb[3 * k + 1], sum.y);
                if (sum.z != 0.f) atomicAdd(&g_alb[3 * k + 2], sum.z);
                if (sum.w != 0.f) atomicAdd(&g_em[k], sum.w);
            }
        }
        pending &= ~grp;
    }
}

}  // namespace pt
