// pt_k_wave.cu -- the wavefront pipeline (Sec. 2.3, 3, 3.1): raygen -> per bounce { extend ->
// (key sort) -> shade -> shadow } -> accumulate.  Stages are linked by structure-of-arrays
// queues of 16-byte records (128-bit coalesced loads and stores); compaction is a warp-aggregated
// atomic append into the next queues (one atomic per warp instead of one per path and queue).  Every
// bounce has counters of its own (BounceCounts), so nothing rotates them between two stages and there is
// no host round trip.  Grids are persistent (a multiple of the SM count) and stride over the device-side
// count, so no host read-back or indirect launch is needed.  Also the batched variants (many scenes, one
// wavefront).
#include <type_traits>

#include "pt_common.cuh"
#include "pt_pool.cuh"

namespace pt {

// Ray generation: the direction of every path of the wave, active count = n.  What is the same for all
// camera rays is not stored: slot j is path j, the origin is the eye, the throughput 1 and the radiance 0,
// which extend and shade know at bounce 0 (16 bytes written and 2 x 16 read per path instead of 64 and
// 32 + 64: shading the 2 M camera hits of a 1080p frame 101 -> 86 us, the frame 1.770 -> 1.753 ms).  The
// wave's first path id is a launch argument here and is published to device memory (wave_base_dev) for the
// kernels of the bounce loop.  clear: the call's first wave also zeroes the call's totals and status word (a memset
// of their own cost a small image 3 us).
template <class Src>
__global__ void __launch_bounds__(256) k_raygen(Src src, uint64_t base, uint32_t n, WfBuffers w,
                                                unsigned long long* wave_base_dev, bool clear) {
    stage_prologue();
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const PathLoc l = src.locate(base, i);
        const RenderParams p = src.params(l.sid);
        const uint32_t key = path_key(p.seed, l.pixel, l.sample);
        float3 o, d;
        float u0, u1;
        pixel_jitter(p.sampler, p.seed, l.pixel, l.sample, key, u0, u1);
        camera_ray(src.camera(l.sid), l.pixel, u0, u1, o, d);
        w.q_d[0][i] = f4(d, __uint_as_float(src.ray_tag(l.sid, 1u)));   // previous vertex "delta": the camera
        if (w.sig) w.sig[l.path] = 0u;
    }
    if (blockIdx.x == 0) {
        if (clear) {
            uint32_t* words = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(w.hist) - kHistOffset);
            for (uint32_t k = threadIdx.x; k < (uint32_t)(kBounceOffset / 4); k += blockDim.x) words[k] = 0u;
        }
        for (uint32_t k = threadIdx.x; k < (uint32_t)kBounceSlots; k += blockDim.x)
            w.bc[k] = BounceCounts{0u, k == 0u ? n : 0u, 0u, 0u};
        if (threadIdx.x == 0 && wave_base_dev) *wave_base_dev = base;
    }
}

// Extension rays as the pooled walks take them: a queue slot's ray (and its scene's tree), its hit record.
template <class Src, bool INST>
struct ExtendIo {
    const Src& src;
    const float4* __restrict__ qo;      // null at bounce 0: camera rays
    const float4* __restrict__ qd;
    float2* __restrict__ hit;
    uint32_t* __restrict__ hit_inst;
    uint64_t base;
    __device__ __forceinline__ DevScene scene() const { return src.scene(0u); }
    __device__ __forceinline__ void fetch(uint32_t j, float3& o, float3& d, float& tbest, uint32_t& best,
                                          const float4*& nodes, const float4*& tris) const {
        const float4 d4 = __ldcs(&qd[j]);
        const uint32_t sid = src.sid_from_ray(d4.w);
        o = qo ? xyz(__ldcs(&qo[j])) : src.eye(sid);
        d = xyz(d4);
        tbest = __int_as_float(0x7f800000);
        best = kMiss;
        if constexpr (!std::is_same<Src, SingleSrc>::value) {
            const DevScene s = src.scene(sid);
            nodes = s.nodes;
            tris = s.tris;
        }
    }
    __device__ __forceinline__ void emit(uint32_t j, float t, uint32_t tri, uint32_t inst) const {
        hit[j] = make_float2(t, __uint_as_float(tri));
        if (INST) hit_inst[j] = inst;
    }
};

// Extension rays and shadow rays (slots with kAnySlot; `best` carries their path, tbest < 0: occluded).
template <class Src, bool SIG, bool INST, bool ADJ>
struct TraceIo {
    ExtendIo<Src, INST> ext;
    const WfBuffers& w;
    const AdjBuffers& a;
    uint32_t b;
    __device__ __forceinline__ DevScene scene() const { return ext.scene(); }
    __device__ __forceinline__ void fetch(uint32_t slot, float3& o, float3& d, float& tbest, uint32_t& best,
                                          const float4*& nodes, const float4*& tris) const {
        if (!(slot & kAnySlot)) {
            ext.fetch(slot, o, d, tbest, best, nodes, tris);
            return;
        }
        const uint32_t k = slot & ~kAnySlot;
        const float4 so = __ldcs(&w.s_o[k]), sd = __ldcs(&w.s_d[k]);
        o = xyz(so);
        d = xyz(sd);
        tbest = so.w;
        best = __float_as_uint(sd.w);
        if constexpr (!ADJ && !std::is_same<Src, SingleSrc>::value) {
            const DevScene s = ext.src.scene(ext.src.sid_from_shadow(__ldcs(&w.s_c[k].w), ext.base, best));
            nodes = s.nodes;
            tris = s.tris;
        }
    }
    __device__ __forceinline__ void emit(uint32_t slot, float t, uint32_t tri, uint32_t inst) const {
        if (!(slot & kAnySlot)) {
            ext.emit(slot, t, tri, inst);
            return;
        }
        const bool occ = t < 0.0f;
        if constexpr (ADJ) {
            if (!occ) {
                float* fl = reinterpret_cast<float*>(a.rec + 4 * ((size_t)(b - 1u) * w.capacity + tri) + 3) + 3;
                *fl = __uint_as_float(__float_as_uint(*fl) | 2u);
            }
        } else {
            if (occ && !SIG) return;
            const float4 sc = __ldcs(&w.s_c[slot & ~kAnySlot]);
            if (!occ) w.L[tri] = f4(add_rn(xyz(w.L[tri]), xyz(sc)), 0.f);
            if (SIG) {
                const uint32_t lj = __float_as_uint(sc.w);
                w.sig[ext.base + tri] ^= sig_event(b - 1u, 1, (lj << 2) | 2u | (occ ? 0u : 1u));
            }
        }
    }
};

// Resident blocks of 256 of the traversal kernels, which cap their registers.  Pooled walks: 5 (48 registers; no spills
// in the loop without shared ends, up to 16 bytes with them and 92 in the shared end itself, 44 in the batch's form;
// against 6 blocks with 80 bytes of spills 1.94 -> 1.91 ms per 1080p frame, against 4 blocks 1.96 -> 1.91).  Lockstep walks (short stack, counting): 6 single-level (40 registers), 4 two-level (64
// registers; 6 blocks measured slower, and without a bound ptxas takes 78 registers, leaving 3 blocks:
// 2.89 -> 3.00 ms per two-level frame).
constexpr int trace_blocks(bool inst, bool pooled) { return inst ? 4 : pooled ? 5 : 6; }

// Extend: closest hit of every active ray (scene-intersection stage); hit records per queue slot.
// SK > 0: the walks keep their top SK stack entries in dynamic shared memory (single-level only).
// CNT: count the walks' node visits and triangle tests into the scene's traversal counters.
template <class Src, bool INST, int SK = 0, bool CNT = false, bool SHARE = false>
__global__ void __launch_bounds__(256, trace_blocks(INST, SK == 0 && !CNT)) k_extend(
    const __grid_constant__ Src src, const __grid_constant__ WfBuffers w, int in, uint32_t b) {
    stage_prologue();
    const uint32_t n = min(w.bc[b].active, w.capacity);
    if (n == 0u) return;       // an emptied queue: no claims (the same for every thread)
    const uint64_t base = src.base();
    const float4* __restrict__ qo = b == 0u ? nullptr : w.q_o[in];
    const float4* __restrict__ qd = w.q_d[in];
    float2* __restrict__ hit = w.hit;
    if constexpr (SK == 0 && !CNT) {
        SlotPool q(&w.bc[b].claim, n);
        pool_walk<INST, SHARE>(src.scene(0), q, n, ExtendIo<Src, INST>{src, qo, qd, hit, w.hit_inst, base});
    } else {       // single-level, in lockstep
        typename std::conditional<CNT, TravCount, NoCount>::type cnt;
        const uint32_t chunks = (n + 31u) / 32u;
        for (uint32_t c = first_chunk(); c < chunks; c = next_chunk(&w.bc[b].claim)) {
            const uint32_t j = c * 32u + lane_id();
            if (j >= n) continue;
            const float4 d4 = __ldcs(&qd[j]);
            const uint32_t sid = src.sid_from_ray(d4.w);
            const float3 o = qo ? xyz(__ldcs(&qo[j])) : src.eye(sid);
            const Hit h = trace_closest<false, SK>(src.scene(sid), o, xyz(d4), cnt);
            hit[j] = make_float2(h.t, __uint_as_float(h.tri));
        }
        flush_count(src.scene(0), cnt, 0);
    }
}

// Key sort before shading (counting sort): keys + block histograms, scan, scatter into `perm`.
template <class Src, bool INST>
__global__ void __launch_bounds__(256) k_sort_keys(Src src, WfBuffers w, int in, uint32_t b, uint32_t mode,
                                                   uint32_t n_keys) {
    extern __shared__ uint32_t hist_s[];
    for (uint32_t k = threadIdx.x; k < n_keys; k += blockDim.x) hist_s[k] = 0u;
    __syncthreads();
    const uint32_t n = min(w.bc[b].active, w.capacity);
    const uint64_t base = src.base();
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        uint32_t tri = __float_as_uint(w.hit[j].y);
        uint32_t key = n_keys - 1u;                          // misses last
        if (tri != kMiss) {
            const DevScene s = src.scene(src.sid_from_ray(w.q_d[in][j].w));
            uint32_t m = __float_as_uint(__ldg(s.tris + 3 * (size_t)tri + 1).w);
            if (INST) {        // an instance may replace the mesh's material
                const uint32_t mw = __float_as_uint(__ldg(s.inst + 8 * (size_t)w.hit_inst[j] + 3).z);
                if (mw != 0u) m = (mw & 0x7FFFFFFFu) - 1u;
            }
            key = mode == 1u ? __float_as_uint(__ldg(reinterpret_cast<const float*>(s.mats + m))) : m;
            key = min(key, n_keys - 2u);
        }
        w.keys[j] = key;
        atomicAdd(&hist_s[key], 1u);
    }
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < n_keys; k += blockDim.x)
        if (hist_s[k]) atomicAdd(&w.bucket[k], hist_s[k]);
}

// Exclusive scan of the bucket counts (one block of 1024 threads, n_keys <= 4096).
__global__ void __launch_bounds__(1024) k_sort_scan(WfBuffers w, uint32_t n_keys) {
    __shared__ uint32_t part[1024];
    const uint32_t t = threadIdx.x;
    uint32_t v[4], sum = 0;
    for (int k = 0; k < 4; ++k) {
        uint32_t idx = 4 * t + k;
        v[k] = idx < n_keys ? w.bucket[idx] : 0u;
        sum += v[k];
    }
    part[t] = sum;
    __syncthreads();
    for (uint32_t off = 1; off < 1024; off <<= 1) {          // Hillis-Steele inclusive scan
        uint32_t x = t >= off ? part[t - off] : 0u;
        __syncthreads();
        part[t] += x;
        __syncthreads();
    }
    uint32_t run = part[t] - sum;
    for (int k = 0; k < 4; ++k) {
        uint32_t idx = 4 * t + k;
        if (idx < n_keys) w.bucket[idx] = run;
        run += v[k];
    }
}

__global__ void __launch_bounds__(256) k_sort_scatter(WfBuffers w, uint32_t b) {
    const uint32_t n = min(w.bc[b].active, w.capacity);
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t base = warp * 32u; base < n; base += n_warps * 32u) {
        uint32_t j = base + lane_id();
        bool valid = j < n;
        uint32_t key = valid ? w.keys[j] : 0xFFFFFFFFu;
        uint32_t peers = __match_any_sync(0xFFFFFFFFu, key);
        uint32_t leader = __ffs(peers) - 1u;
        uint32_t rank = __popc(peers & ((1u << lane_id()) - 1u));
        uint32_t off = 0u;
        if (valid && lane_id() == leader) off = atomicAdd(&w.bucket[key], (uint32_t)__popc(peers));
        off = __shfl_sync(0xFFFFFFFFu, off, leader);
        if (valid) w.perm[off + rank] = j;
    }
}

// Queue records (rays, hits, shadow rays) are loaded and stored with the streaming cache hint
// (__ldcs / __stcs: evict first from L2).  A bounce's queues (about 100 MB at 1080p) would otherwise
// push the scene (39 MB of nodes, 55 MB of triangles) out of the 126 MB L2, and deep-bounce walks then
// wait on DRAM for every node: with the hint the wavefront frame runs 1-1.5% faster at every depth.

// Shading of one queue entry (emission, NEE sample, BSDF sample, roulette): the records of its
// continuation ray and shadow ray, if any.
struct ShadeOut {
    bool want_ray = false, want_shadow = false;
    float4 ro, rd, rtp, so, sd, sc;
};

template <class Src, bool SIG, bool INST>
__device__ __forceinline__ ShadeOut shade_entry(const Src& src, const WfBuffers& w, int in, uint32_t b, bool sorted,
                                                uint64_t base, uint32_t j) {
    ShadeOut r;
    const uint32_t slot = sorted ? w.perm[j] : j;
    const float4 d4 = __ldcs(&w.q_d[in][slot]);
    const float2 hh = __ldcs(&w.hit[slot]);
    const uint32_t sid = src.sid_from_ray(d4.w);
    float4 o4, tp4;
    if (b == 0u) {       // a camera ray (see k_raygen)
        o4 = f4(src.eye(sid), __uint_as_float(slot));
        tp4 = make_float4(1.f, 1.f, 1.f, 0.f);
    } else {
        o4 = __ldcs(&w.q_o[in][slot]);
        tp4 = __ldcs(&w.q_tp[in][slot]);
    }
    const uint32_t pid = __float_as_uint(o4.w);
    const PathLoc l = src.locate_in(base, pid, sid);
    const DevScene s = src.scene(l.sid);
    const float3 tp = xyz(tp4);
    const uint32_t tri = __float_as_uint(hh.y);
    if (tri == kMiss) {
        const float3 L0 = b == 0u ? f3(0.f, 0.f, 0.f) : xyz(w.L[pid]);
        w.L[pid] = f4(add_rn(L0, mul_rn(tp, f3(s.env_r, s.env_g, s.env_b))), 0.f);
        if (SIG) w.sig[l.path] ^= sig_event(b, 0, kMiss);
        return r;
    }
    const RenderParams p = src.params(l.sid);
    const uint32_t key = path_key(p.seed, l.pixel, l.sample);
    Vertex V = shade_vertex<true, INST>(s, p, key, b, xyz(o4), xyz(d4), tp, (__float_as_uint(d4.w) & 1u) != 0u, tp4.w,
                                        hh.x, tri, INST ? w.hit_inst[slot] : kMiss);
    if (b == 0u) {
        w.L[pid] = f4(V.emit_counted ? add_rn(f3(0.f, 0.f, 0.f), V.emit) : f3(0.f, 0.f, 0.f), 0.f);
    } else if (V.emit_counted) {
        w.L[pid] = f4(add_rn(xyz(w.L[pid]), V.emit), 0.f);
    }
    uint32_t sg = 0;
    if (SIG) sg = sig_event(b, 0, V.prim);
    if (!V.last) {
        if (V.nee) {
            if (V.cast) {
                r.want_shadow = true;
                r.so = f4(V.s_o, V.s_tmax);
                r.sd = f4(V.s_d, __uint_as_float(pid));
                r.sc = f4(V.contrib, __uint_as_float(src.shadow_tag(V.light_j, l.sid)));
            } else if (SIG) {
                sg ^= sig_event(b, 1, V.light_j << 2);
            }
        }
        if (SIG) {
            sg ^= sig_event(b, 2, V.bsdf_code);
            if (V.rr >= 0) sg ^= sig_event(b, 3, (uint32_t)V.rr);
        }
        if (V.cont) {
            r.want_ray = true;
            r.ro = f4(V.no, __uint_as_float(pid));
            r.rd = f4(V.nd, __uint_as_float(src.ray_tag(l.sid, V.delta ? 1u : 0u)));
            r.rtp = f4(V.ntp, V.pdf);
        }
    }
    if (SIG) w.sig[l.path] ^= sg;
    return r;
}

template <class Src>
__device__ __forceinline__ void put_shadow(const Src& src, const WfBuffers& w, uint32_t k, const ShadeOut& r) {
    if (k < w.capacity) {
        __stcs(&w.s_o[k], r.so);
        __stcs(&w.s_d[k], r.sd);
        __stcs(&w.s_c[k], r.sc);
    } else {
        atomicOr(src.scene(0).status, ST_QUEUE);
    }
}

template <class Src>
__device__ __forceinline__ void put_ray(const Src& src, const WfBuffers& w, int out, uint32_t q, const ShadeOut& r) {
    if (q < w.capacity) {
        __stcs(&w.q_o[out][q], r.ro);
        __stcs(&w.q_d[out][q], r.rd);
        __stcs(&w.q_tp[out][q], r.rtp);
    } else {
        atomicOr(src.scene(0).status, ST_QUEUE);
    }
}

// Shade: emission, NEE sample (-> shadow queue), BSDF sample, roulette, compaction of survivors: each
// warp appends its survivors with one atomic for both queues (warp-aggregated).
template <class Src, bool SIG, bool INST>
__global__ void __launch_bounds__(256, 3) k_shade(Src src, WfBuffers w, int in, uint32_t b, bool sorted) {
    stage_prologue();
    const uint32_t n = min(w.bc[b].active, w.capacity);
    const uint64_t base = src.base();
    const int out = in ^ 1;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t wb = warp * 32u; wb < n; wb += n_warps * 32u) {
        const uint32_t j = wb + lane_id();
        ShadeOut r;
        if (j < n) r = shade_entry<Src, SIG, INST>(src, w, in, b, sorted, base, j);
        uint32_t k, q;
        warp_append2(&w.bc[b + 1], r.want_shadow, r.want_ray, k, q);
        if (r.want_shadow) put_shadow(src, w, k, r);
        if (r.want_ray) put_ray(src, w, out, q, r);
    }
}

// Shadow: any-hit test of each queued shadow ray; unoccluded contributions are added to the path.
// At most one shadow ray per path per bounce, so the read-modify-write of L needs no atomics.
template <class Src, bool SIG, bool INST, int SK = 0, bool CNT = false>
__global__ void __launch_bounds__(256) k_shadow(Src src, WfBuffers w, uint32_t b) {
    const uint32_t n = min(w.bc[b + 1].shadow, w.capacity);
    if (n == 0u) return;
    const uint64_t base = src.base();
    typename std::conditional<CNT, TravCount, NoCount>::type cnt;
    const uint32_t chunks = (n + 31u) / 32u;
    for (uint32_t c = first_chunk(); c < chunks; c = next_chunk(&w.bc[b].claim_shadow)) {
        const uint32_t j = c * 32u + lane_id();
        if (j >= n) continue;
        const float4 so = __ldcs(&w.s_o[j]), sd = __ldcs(&w.s_d[j]), sc = __ldcs(&w.s_c[j]);
        const uint32_t pid = __float_as_uint(sd.w);
        const bool occ =
            trace_any<INST, SK>(src.scene(src.sid_from_shadow(sc.w, base, pid)), xyz(so), xyz(sd), so.w, cnt);
        if (!occ) {
            float3 L = add_rn(xyz(w.L[pid]), xyz(sc));
            w.L[pid] = f4(L, 0.f);
        }
        if (SIG) {
            const uint32_t lj = __float_as_uint(sc.w);
            w.sig[base + pid] ^= sig_event(b, 1, (lj << 2) | 2u | (occ ? 0u : 1u));
        }
    }
    flush_count(src.scene(0), cnt, 2);
}

// The cooperative form of the fused trace stage: each group of G lanes takes one extension ray, then
// one shadow ray, per claim (trace_closest_group / trace_any_group, or their two-level forms); the
// group's first lane writes the result exactly as the one-lane form does.
constexpr uint32_t kCoopMinLanes = 2u;
// Groups of two lanes only below this many walks: from there on the pooled walk is the faster one (the launch of
// 56 k walks at bounce 4 of a 1080p frame: 1.547 -> 1.510 ms for the frame, its two-level form 1.608 -> 1.585, four 720p
// frames 2.242 -> 2.187); in the grids of small images, sized to their queues, groups of two are.  Where between
// those the two measure alike is not known.
constexpr uint32_t kPairMaxWalks = 1u << 15;

// SHARE only sets the two kernels' copies apart: ptxas 13.0 crashes on one function called by both.
template <class Src, bool SIG, bool INST, bool ADJ, bool SHARE>
__device__ __noinline__ void trace_groups(const Src& src, const WfBuffers& w, const AdjBuffers& a, int in,
                                             uint32_t b, uint32_t n_ext, uint32_t n_shd, uint32_t G) {
    const uint64_t base = src.base();
    const uint32_t per = 32u / G, sub = lane_id() / G;
    const bool lead = (lane_id() & (G - 1u)) == 0u;
    unsigned long long led = 0;      // walks this lane's group traced, counted once per group
    const float4* __restrict__ qo = w.q_o[in];
    const float4* __restrict__ qd = w.q_d[in];
    // one chunk sequence over both sets: the extension rays' chunks, then the shadow rays'
    const uint32_t c_ext = (n_ext + per - 1u) / per, c_all = c_ext + (n_shd + per - 1u) / per;
    uint32_t c = first_chunk();
    for (; c < c_ext; c = next_chunk(&w.bc[b].claim)) {
        const uint32_t j = c * per + sub;
        const bool valid = j < n_ext;
        float4 o4 = make_float4(0.f, 0.f, 0.f, 0.f), d4 = make_float4(0.f, 0.f, 1.f, 0.f);
        if (valid) {
            o4 = __ldcs(&qo[j]);
            d4 = __ldcs(&qd[j]);
        }
        const uint32_t sid = valid ? src.sid_from_ray(d4.w) : 0u;
        const Hit h = INST ? trace_closest_group_inst(src.scene(sid), xyz(o4), xyz(d4), valid, G)
                           : trace_closest_group(src.scene(sid), xyz(o4), xyz(d4), valid, G);
        if (valid && lead) {
            w.hit[j] = make_float2(h.t, __uint_as_float(h.tri));
            if (INST) w.hit_inst[j] = h.inst;
            ++led;
        }
    }
    for (; c < c_all; c = next_chunk(&w.bc[b].claim)) {
        const uint32_t k = (c - c_ext) * per + sub;
        const bool valid = k < n_shd;
        float4 so = make_float4(0.f, 0.f, 0.f, 0.f), sd = make_float4(0.f, 0.f, 1.f, 0.f);
        float4 sc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
            so = __ldcs(&w.s_o[k]);
            sd = __ldcs(&w.s_d[k]);
            if (!ADJ) sc = __ldcs(&w.s_c[k]);
        }
        const uint32_t pid = __float_as_uint(sd.w);
        const uint32_t sid = (valid && !ADJ) ? src.sid_from_shadow(sc.w, base, pid) : 0u;
        const bool occ = INST ? trace_any_group_inst(src.scene(sid), xyz(so), xyz(sd), so.w, valid, G)
                              : trace_any_group(src.scene(sid), xyz(so), xyz(sd), so.w, valid, G);
        if (!valid || !lead) continue;
        ++led;
        if constexpr (ADJ) {
            if (!occ) {
                float* fl = reinterpret_cast<float*>(a.rec + 4 * ((size_t)(b - 1u) * w.capacity + pid) + 3) + 3;
                *fl = __uint_as_float(__float_as_uint(*fl) | 2u);
            }
        } else {
            if (!occ) {
                float3 L = add_rn(xyz(w.L[pid]), xyz(sc));
                w.L[pid] = f4(L, 0.f);
            }
            if (SIG) {
                const uint32_t lj = __float_as_uint(sc.w);
                w.sig[base + pid] ^= sig_event(b - 1u, 1, (lj << 2) | 2u | (occ ? 0u : 1u));
            }
        }
    }
    warp_add_u64(&w.hist[kHistGroupWalks + __ffs((int)G) - 2], led);
}

// Trace (the extend stage of bounce b fused with the shadow stage of bounce b - 1): one launch walks
// the BVH for the continuation rays of bounce b (closest hit, queue `in`, bc[b].active entries) and for
// the shadow rays that shading cast at bounce b - 1 (any hit, the shadow queue, bc[b].shadow entries).
// The two sets are independent -- a shadow ray only adds its contribution to its path's radiance, and
// only the next shading reads that radiance -- so each path still adds its terms in the order
// emission(b - 1), NEE(b - 1), emission(b), as in the megakernel.  Launches walk both sets
// through one pool (pool_walk): the continuation rays first, then the shadow rays; the counting launches
// take 32 continuation rays at a time until none is left and then 32 shadow rays at a time.
// A launch therefore ends when both sets are done, and the shadow walks fill the extension walks' tail
// instead of running after a stage boundary.
// ADJ: the adjoint replay's variant, whose shadow walks mark the vertex record's NEE sample visible
// (flag 2 of record 3 of bounce b - 1) instead of adding a contribution.
template <class Src, bool SIG, bool INST, bool CNT = false, bool ADJ = false, bool SHARE = false>
__global__ void __launch_bounds__(256, trace_blocks(INST, !CNT)) k_trace(
    const __grid_constant__ Src src, const __grid_constant__ WfBuffers w, const __grid_constant__ AdjBuffers a, int in, uint32_t b) {
    stage_prologue();
    const uint32_t n_ext = min(w.bc[b].active, w.capacity), n_shd = min(w.bc[b].shadow, w.capacity);
    if (n_ext + n_shd == 0u) return;       // the same for every thread
    const uint64_t base = src.base();
    // Lanes per walk: 1 while the walks fill the grid; once they are few (the sparse late bounces),
    // the largest power of two G <= 32 with walks x G <= the grid's threads (cooperative walks, see kPairMaxWalks; the
    // counting instantiations keep the one-lane walk their counts describe).
    // The same for every thread: the counts are fixed during the launch.
    uint32_t G = 1u;
    if constexpr (!CNT) {
        const uint64_t threads = (uint64_t)gridDim.x * blockDim.x;
        while (G < 32u && (uint64_t)(n_ext + n_shd) * (2u * G) <= threads) G *= 2u;
        if (G < kCoopMinLanes || (G < 4u && n_ext + n_shd >= kPairMaxWalks)) G = 1u;
    }
    if (G > 1u) {
        trace_groups<Src, SIG, INST, ADJ, SHARE>(src, w, a, in, b, n_ext, n_shd, G);
        return;
    }
    if constexpr (!CNT) {
        SlotPool q(&w.bc[b].claim, n_ext + n_shd);
        pool_walk<INST, SHARE>(src.scene(0), q, n_ext,
                               TraceIo<Src, SIG, INST, ADJ>{{src, w.q_o[in], w.q_d[in], w.hit, w.hit_inst, base}, w, a, b});
    } else {       // counting (single-level, no signatures), in lockstep
        TravCount cc, ca;
        const uint32_t c_ext = (n_ext + 31u) / 32u, c_all = c_ext + (n_shd + 31u) / 32u;
        uint32_t c = first_chunk();
        for (; c < c_ext; c = next_chunk(&w.bc[b].claim)) {
            const uint32_t j = c * 32u + lane_id();
            if (j >= n_ext) continue;
            const float4 o4 = __ldcs(&w.q_o[in][j]), d4 = __ldcs(&w.q_d[in][j]);
            const Hit h = trace_closest<false, 0>(src.scene(src.sid_from_ray(d4.w)), xyz(o4), xyz(d4), cc);
            w.hit[j] = make_float2(h.t, __uint_as_float(h.tri));
        }
        for (; c < c_all; c = next_chunk(&w.bc[b].claim)) {
            const uint32_t k = (c - c_ext) * 32u + lane_id();
            if (k >= n_shd) continue;
            const float4 so = __ldcs(&w.s_o[k]), sd = __ldcs(&w.s_d[k]), sc = __ldcs(&w.s_c[k]);
            const uint32_t pid = __float_as_uint(sd.w);
            if (!trace_any<false, 0>(src.scene(src.sid_from_shadow(sc.w, base, pid)), xyz(so), xyz(sd), so.w, ca))
                w.L[pid] = f4(add_rn(xyz(w.L[pid]), xyz(sc)), 0.f);
        }
        flush_count(src.scene(0), cc, 0);
        flush_count(src.scene(0), ca, 2);
    }
}

// ================================================================== accumulation
// The end of a wave adds its bounces' counts to the call's totals (block 0 of the accumulation).
__device__ __forceinline__ void fold_counts(const BounceCounts* bc, unsigned long long* hist) {
    if (bc == nullptr || blockIdx.x != 0) return;
    for (uint32_t b = threadIdx.x; b < 64u; b += blockDim.x) {
        hist[b] += bc[b].active;
        hist[64u + b] += bc[b + 1u].shadow;
    }
}
// A pixel's samples added to (r, g, b) in sample order.  Records of four floats (a wave's L, 16-byte aligned) take one
// load each: with several samples a pixel, neighbouring lanes are 16 * spp bytes apart, so that a request is a line
// a lane, and three loads of 4 bytes cost three of them.  16 samples: the 128 x 128 box 244.3 -> 240.3 us, a 512 x
// 512 training step 3.837 -> 3.807 ms; 1 and 3 samples: no change.  The megakernel's records have three floats.
__device__ __forceinline__ void add_samples(const float* __restrict__ L, uint32_t stride_f, uint64_t px, uint32_t spp,
                                            float& r, float& g, float& b) {
    if (stride_f == 4u) {
        const float4* q = reinterpret_cast<const float4*>(L) + px * spp;
#pragma unroll 4
        for (uint32_t smp = 0; smp < spp; ++smp) {
            const float4 v = q[smp];
            r = __fadd_rn(r, v.x);
            g = __fadd_rn(g, v.y);
            b = __fadd_rn(b, v.z);
        }
    } else {
        const float* q = L + px * spp * stride_f;
        for (uint32_t smp = 0; smp < spp; ++smp) {
            r = __fadd_rn(r, q[smp * stride_f]);
            g = __fadd_rn(g, q[smp * stride_f + 1]);
            b = __fadd_rn(b, q[smp * stride_f + 2]);
        }
    }
}

__global__ void __launch_bounds__(256) k_reduce(const float* __restrict__ L, uint32_t stride_f, uint64_t pixel_begin,
                                                uint64_t n_pixels, uint32_t spp, float* __restrict__ img,
                                                const BounceCounts* bc, unsigned long long* hist) {
    stage_prologue();
    fold_counts(bc, hist);
    const float inv = 1.0f / (float)spp;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t px = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; px < n_pixels; px += stride) {
        float r = 0.f, g = 0.f, bl = 0.f;
        add_samples(L, stride_f, px, spp, r, g, bl);
        float* o = img + 3 * (pixel_begin + px);
        o[0] = __fmul_rn(r, inv);
        o[1] = __fmul_rn(g, inv);
        o[2] = __fmul_rn(bl, inv);
    }
}

// Progressive accumulation (the running average of Sec. 2.3): add this call's samples of each
// pixel, in sample order, to the pixel's FP32 running sum and write sum / count (img may be null).
// Continuing the sum is exactly what the one-call reduce does, so frames of k1, k2, ... samples end
// at the image of one call with k1 + k2 + ... samples, bit for bit.
__global__ void __launch_bounds__(256) k_accumulate(const float* __restrict__ L, uint32_t stride_f,
                                                    uint64_t pixel_begin, uint64_t n_pixels, uint32_t spp,
                                                    float* __restrict__ sum, uint32_t count, float* __restrict__ img,
                                                    const BounceCounts* bc, unsigned long long* hist) {
    stage_prologue();
    fold_counts(bc, hist);
    const float inv = 1.0f / (float)count;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t px = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; px < n_pixels; px += stride) {
        float* a = sum + 3 * (pixel_begin + px);
        float r = a[0], g = a[1], bl = a[2];
        add_samples(L, stride_f, px, spp, r, g, bl);
        a[0] = r;
        a[1] = g;
        a[2] = bl;
        if (img) {
            float* o = img + 3 * (pixel_begin + px);
            o[0] = __fmul_rn(r, inv);
            o[1] = __fmul_rn(g, inv);
            o[2] = __fmul_rn(bl, inv);
        }
    }
}

__global__ void k_copy_L(const float4* __restrict__ L4, uint64_t n, float* __restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float4 v = L4[i];
        out[3 * i] = v.x;
        out[3 * i + 1] = v.y;
        out[3 * i + 2] = v.z;
    }
}

// Batched accumulation: add this wave's samples of each pixel, in sample order, to the pixel's
// running FP32 sum in its scene's output image (zeroed before the first wave).  A pixel split
// between two waves continues from the stored partial sum, so the additions are exactly those of
// the single-scene reduce.
__global__ void __launch_bounds__(256) k_reduce_batch(BatchTables t, const float4* __restrict__ L,
                                                      const BatchSegment* __restrict__ seg, uint32_t n_seg,
                                                      unsigned long long w0, unsigned long long w1,
                                                      unsigned long long n_flat) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t f = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; f < n_flat; f += stride) {
        uint32_t lo = 0, hi = n_seg - 1;
        while (lo < hi) {
            uint32_t mid = (lo + hi + 1) >> 1;
            if (seg[mid].flat_begin <= f) lo = mid;
            else hi = mid - 1;
        }
        const BatchSegment sg = seg[lo];
        const uint64_t px = sg.px_begin + (f - sg.flat_begin);
        const uint32_t spp = t.spp[sg.scene];
        const uint64_t first = t.off[sg.scene] + px * spp;
        const uint64_t a = first > w0 ? first : w0;
        const uint64_t e = first + spp < w1 ? first + spp : w1;
        float* o = t.out[sg.scene] + 3 * px;
        float r = o[0], g = o[1], bl = o[2];
        for (uint64_t q = a; q < e; ++q) {
            const float4 v = L[q - w0];
            r = __fadd_rn(r, v.x);
            g = __fadd_rn(g, v.y);
            bl = __fadd_rn(bl, v.z);
        }
        o[0] = r;
        o[1] = g;
        o[2] = bl;
    }
}

// Batched accumulation, last step: sums -> means (the single-scene reduce's final multiply).
__global__ void k_scale_batch(BatchTables t, const unsigned long long* __restrict__ px_off, unsigned long long total) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t f = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; f < total; f += stride) {
        uint32_t lo = 0, hi = t.n - 1;
        while (lo < hi) {
            uint32_t mid = (lo + hi + 1) >> 1;
            if (px_off[mid] <= f) lo = mid;
            else hi = mid - 1;
        }
        const float inv = 1.0f / (float)t.spp[lo];
        float* o = t.out[lo] + 3 * (f - px_off[lo]);
        o[0] = __fmul_rn(o[0], inv);
        o[1] = __fmul_rn(o[1], inv);
        o[2] = __fmul_rn(o[2], inv);
    }
}


// ------------------------------------------------------------------ launchers

cudaError_t launch_raygen(const Launch& l, const DevCamera& c, const RenderParams& p, uint32_t n, const WfBuffers& w,
                          bool clear) {
    SingleSrc src{DevScene{}, c, p};
    return launch_k(l, 0, k_raygen<SingleSrc>, src, p.path_begin, n, w, (unsigned long long*)nullptr, clear);
}

cudaError_t launch_extend(const Launch& l, const DevScene& s, const WfBuffers& w, int in, uint32_t bounce,
                          const RenderParams& p) {
    SingleSrc src{s, DevCamera{}, p};
    if (s.tlas) return launch_k(l, 0, k_extend<SingleSrc, true>, src, w, in, bounce);
    if (p.count_trav) return launch_k(l, 0, k_extend<SingleSrc, false, 0, true>, src, w, in, bounce);
    if (p.short_stack)
        return launch_k(l, stack_smem_bytes(kShortStack, l.block), k_extend<SingleSrc, false, kShortStack>, src, w, in, bounce);
    if (p.share) return launch_k(l, 0, k_extend<SingleSrc, false, 0, false, true>, src, w, in, bounce);
    return launch_k(l, 0, k_extend<SingleSrc, false>, src, w, in, bounce);
}

cudaError_t launch_sort(const Launch& l, const DevScene& s, const WfBuffers& w, int in, uint32_t bounce, uint32_t mode,
                        uint32_t n_keys, const RenderParams& p) {
    cudaError_t e = cudaMemsetAsync(w.bucket, 0, sizeof(uint32_t) * n_keys, l.st);
    if (e != cudaSuccess) return e;
    SingleSrc src{s, DevCamera{}, p};
    if (s.tlas) k_sort_keys<SingleSrc, true><<<l.grid, l.block, sizeof(uint32_t) * n_keys, l.st>>>(src, w, in, bounce, mode, n_keys);
    else k_sort_keys<SingleSrc, false><<<l.grid, l.block, sizeof(uint32_t) * n_keys, l.st>>>(src, w, in, bounce, mode, n_keys);
    k_sort_scan<<<1, 1024, 0, l.st>>>(w, n_keys);
    k_sort_scatter<<<l.grid, l.block, 0, l.st>>>(w, bounce);
    return cudaGetLastError();
}

cudaError_t launch_shade(const Launch& l, const DevScene& s, const RenderParams& p, const WfBuffers& w, int in,
                         uint32_t bounce, bool sorted) {
    SingleSrc src{s, DevCamera{}, p};
    if (s.tlas) {
        if (w.sig) return launch_k(l, 0, k_shade<SingleSrc, true, true>, src, w, in, bounce, sorted);
        return launch_k(l, 0, k_shade<SingleSrc, false, true>, src, w, in, bounce, sorted);
    }
    if (w.sig) return launch_k(l, 0, k_shade<SingleSrc, true, false>, src, w, in, bounce, sorted);
    return launch_k(l, 0, k_shade<SingleSrc, false, false>, src, w, in, bounce, sorted);
}

cudaError_t launch_shadow(const Launch& l, const DevScene& s, const RenderParams& p, const WfBuffers& w,
                          uint32_t bounce) {
    SingleSrc src{s, DevCamera{}, p};
    if (s.tlas) {
        if (w.sig) k_shadow<SingleSrc, true, true><<<l.grid, l.block, 0, l.st>>>(src, w, bounce);
        else k_shadow<SingleSrc, false, true><<<l.grid, l.block, 0, l.st>>>(src, w, bounce);
    } else {
        const size_t sm = stack_smem_bytes(kShortStack, l.block);
        if (p.count_trav && !w.sig) {
            k_shadow<SingleSrc, false, false, 0, true><<<l.grid, l.block, 0, l.st>>>(src, w, bounce);
        } else if (p.short_stack) {
            if (w.sig) k_shadow<SingleSrc, true, false, kShortStack><<<l.grid, l.block, sm, l.st>>>(src, w, bounce);
            else k_shadow<SingleSrc, false, false, kShortStack><<<l.grid, l.block, sm, l.st>>>(src, w, bounce);
        } else {
            if (w.sig) k_shadow<SingleSrc, true, false><<<l.grid, l.block, 0, l.st>>>(src, w, bounce);
            else k_shadow<SingleSrc, false, false><<<l.grid, l.block, 0, l.st>>>(src, w, bounce);
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_raygen_batch(const Launch& l, const BatchTables& t, const RenderParams& p, uint64_t base, uint32_t n,
                                const WfBuffers& w) {
    TableSrc src{t, p};
    k_raygen<TableSrc><<<l.grid, l.block, 0, l.st>>>(src, base, n, w, t.wave_base, false);
    return cudaGetLastError();
}

cudaError_t launch_bounce_batch(const Launch& le, const Launch& ls, const Launch& lw, const Launch& lk,
                                const BatchTables& t, const RenderParams& p, const WfBuffers& w, uint32_t b,
                                uint32_t sort_mode, uint32_t n_keys, bool fused) {
    TableSrc src{t, p};
    const int in = (int)(b & 1u);
    // fused and unsorted: the stage kernels are programmatic dependents of the kernel before them
    // (programmatic edges of the captured bounce graph; bounce 0's first launch opens the graph)
    const bool pdl = fused && n_keys == 0;
    Launch lt = lw, lsh = ls;
    lt.pdl = pdl;
    lsh.pdl = pdl;
    cudaError_t e;
    if (fused && b > 0)   // lw: the fused launch (this bounce's extension and the last bounce's shadow walks)
        e = launch_k(lt, 0, k_trace<TableSrc, false, false>, src, w, AdjBuffers{}, in, b);
    else
        e = launch_k(le, 0, k_extend<TableSrc, false>, src, w, in, b);
    if (e != cudaSuccess) return e;
    if (n_keys) {
        if ((e = cudaMemsetAsync(w.bucket, 0, sizeof(uint32_t) * n_keys, lk.st)) != cudaSuccess) return e;
        k_sort_keys<TableSrc, false><<<lk.grid, lk.block, sizeof(uint32_t) * n_keys, lk.st>>>(src, w, in, b, sort_mode, n_keys);
        k_sort_scan<<<1, 1024, 0, lk.st>>>(w, n_keys);
        k_sort_scatter<<<lk.grid, lk.block, 0, lk.st>>>(w, b);
    }
    if ((e = launch_k(lsh, 0, k_shade<TableSrc, false, false>, src, w, in, b, n_keys > 0)) != cudaSuccess) return e;
    if (!fused) k_shadow<TableSrc, false, false><<<lw.grid, lw.block, 0, lw.st>>>(src, w, b);
    return cudaGetLastError();
}

cudaError_t launch_reduce_batch(const Launch& l, const BatchTables& t, const float4* L, const BatchSegment* seg,
                                uint32_t n_seg, uint64_t w0, uint64_t w1, uint64_t n_flat) {
    if (n_flat == 0) return cudaSuccess;
    k_reduce_batch<<<l.grid, l.block, 0, l.st>>>(t, L, seg, n_seg, w0, w1, n_flat);
    return cudaGetLastError();
}

cudaError_t launch_scale_batch(const Launch& l, const BatchTables& t, const unsigned long long* px_off, uint64_t total) {
    if (total == 0) return cudaSuccess;
    k_scale_batch<<<l.grid, l.block, 0, l.st>>>(t, px_off, total);
    return cudaGetLastError();
}

cudaError_t launch_trace(const Launch& l, const DevScene& s, const RenderParams& p, const WfBuffers& w, int in,
                         uint32_t bounce) {
    SingleSrc src{s, DevCamera{}, p};
    const AdjBuffers a{};
    if (s.tlas) {
        if (w.sig) return launch_k(l, 0, k_trace<SingleSrc, true, true>, src, w, a, in, bounce);
        return launch_k(l, 0, k_trace<SingleSrc, false, true>, src, w, a, in, bounce);
    }
    if (p.count_trav && !w.sig) return launch_k(l, 0, k_trace<SingleSrc, false, false, true>, src, w, a, in, bounce);
    if (w.sig) return launch_k(l, 0, k_trace<SingleSrc, true, false>, src, w, a, in, bounce);
    if (p.share) return launch_k(l, 0, k_trace<SingleSrc, false, false, false, false, true>, src, w, a, in, bounce);
    return launch_k(l, 0, k_trace<SingleSrc, false, false>, src, w, a, in, bounce);
}

cudaError_t launch_trace_adj(const Launch& l, const DevScene& s, const RenderParams& p, const WfBuffers& w,
                             const AdjBuffers& a, int in, uint32_t bounce) {
    SingleSrc src{s, DevCamera{}, p};
    if (s.tlas) return launch_k(l, 0, k_trace<SingleSrc, false, true, false, true>, src, w, a, in, bounce);
    if (p.share) return launch_k(l, 0, k_trace<SingleSrc, false, false, false, true, true>, src, w, a, in, bounce);
    return launch_k(l, 0, k_trace<SingleSrc, false, false, false, true>, src, w, a, in, bounce);
}

cudaError_t launch_reduce(const Launch& l, const float* L, uint32_t stride, uint64_t pixel_begin, uint64_t n_pixels,
                          uint32_t spp, float* img, const WfBuffers* w) {
    return launch_k(l, 0, k_reduce, L, stride, pixel_begin, n_pixels, spp, img,
                    w ? (const BounceCounts*)w->bc : nullptr, w ? w->hist : nullptr);
}

cudaError_t launch_accumulate(const Launch& l, const float* L, uint32_t stride, uint64_t pixel_begin, uint64_t n_pixels,
                              uint32_t spp, float* sum, uint32_t count, float* img, const WfBuffers* w) {
    return launch_k(l, 0, k_accumulate, L, stride, pixel_begin, n_pixels, spp, sum, count, img,
                    w ? (const BounceCounts*)w->bc : nullptr, w ? w->hist : nullptr);
}

cudaError_t launch_copy_L(const Launch& l, const float4* L4, uint64_t n, float* out_L3) {
    k_copy_L<<<l.grid, l.block, 0, l.st>>>(L4, n, out_L3);
    return cudaGetLastError();
}

// Resident blocks per SM of this unit's kernels (0: not one of them).
int occupancy_wave(int which, int block) {
    int nb = 0;
    cudaError_t e = cudaErrorInvalidValue;
    const size_t sm = stack_smem_bytes(kShortStack, block);   // the short-stack instantiations' shared stacks
    switch (which) {
        case K_EXTEND: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extend<SingleSrc, false>, block, 0); break;
        case K_SHADE: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shade<SingleSrc, false, false>), block, 0); break;
        case K_SHADOW: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shadow<SingleSrc, false, false>), block, 0); break;
        case K_EXTEND_SS:
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extend<SingleSrc, false, kShortStack>, block, sm);
            break;
        case K_SHADOW_SS:
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shadow<SingleSrc, false, false, kShortStack>), block, sm);
            break;
        case K_TRACE: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_trace<SingleSrc, false, false>), block, 0); break;
        case K_TRACE_INST: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_trace<SingleSrc, false, true>), block, 0); break;
        case K_TRACE_BATCH: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_trace<TableSrc, false, false>), block, 0); break;
        case K_EXTEND_BATCH: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extend<TableSrc, false>, block, 0); break;
        case K_SHADE_BATCH: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shade<TableSrc, false, false>), block, 0); break;
        case K_SHADOW_BATCH: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shadow<TableSrc, false, false>), block, 0); break;
        case K_EXTEND_INST: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_extend<SingleSrc, true>, block, 0); break;
        case K_SHADE_INST: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shade<SingleSrc, false, true>), block, 0); break;
        case K_SHADOW_INST: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (k_shadow<SingleSrc, false, true>), block, 0); break;
        default: return 0;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb > 0 ? nb : 1;
}

}  // namespace pt
