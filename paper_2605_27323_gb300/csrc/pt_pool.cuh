// pt_pool.cuh -- pooled walks: the traversal loop of the wavefront's trace stages, of the regenerating megakernel
// and of the closest-hit queries.
//
// A lockstep walk of 32 rays (each lane its own ray, the warp takes 32 new ones when the last has
// finished) issues every instruction for 9 lanes of 32 on average after the first bounce: lanes whose
// walk ended wait for the longest one, and a leaf step runs for the one or two lanes that hold a leaf
// while the others wait.  Here a warp keeps its lanes supplied from a pool of queue slots:
//   - node steps repeat while at least kNodeLanes lanes hold an inner node;
//   - then all lanes that hold a leaf test it together;
//   - once kIdleLanes lanes have finished, they write their results and take the next slots.
// (Persistent warps that refill idle lanes from a pool of rays: Aila and Laine, "Understanding the Efficiency of Ray
// Traversal on GPUs", HPG 2009.)  Extension (closest-hit) and shadow (any-hit) rays share the loop, so a launch drains
// its warps once and not once per kind.  Each ray visits the nodes and triangles of the lockstep walk in the same
// order, so hits are the same bit for bit.  (The shared ends below, and the groups of lanes of launches with few walks,
// visit some more: subtrees walked before another lane's hit culls them.  Their hits are the same too.)
//
// What bounds it, in the launch of bounce 1 at 1080p on 1.15 M triangles: the L1 data path, busy 82% of the time with
// divergent node requests (issue 61%, long-scoreboard stalls for the rest).  Requests fill it, not bytes: a node as
// two 256-bit loads beats four of 128 bits by 1%, and reading its 56 used bytes in three loads costs 2% on the
// terrain.  Against the lockstep walk: 168 -> 115 warp instructions per walk, 9.5 -> 19 lanes per instruction, 683
// -> 524 us; camera rays 117 -> 92, 15 -> 23, 360 -> 275 us.
#pragma once
#include "pt_common.cuh"

namespace pt {

constexpr uint32_t kDone = 0xFFFFFFFFu;    // no subtree left (never a leaf reference: triangles < 2^28)
constexpr uint32_t kNoSlot = 0xFFFFFFFFu;
// 8 and 20 measured best over the frames of {8, 10, 12} x {8, 12, 16, 20} lanes; they are the lowest and the highest
// tried, and were tried before the last walks were shared (1080p 1.600 ms against 1.648 at 12 and 12, 1.658 at 12 and
// 8; the terrain 9.61 against 9.87 and 10.18): fewer node lanes waste L1 cycles, more make the loop leave its node steps
// too often; a refill costs some 150 instructions and a claim for the whole warp, however few lanes it serves.
constexpr uint32_t kNodeLanes = 8;
constexpr uint32_t kIdleLanes = 20;
// Fault guards against trees that the builder refuses (deeper than the stack) or never makes (cycles).  A phase takes at
// most kPhaseSteps node steps and the stack has room for as many entries beyond its depth; once a turn -- a node phase
// and a leaf phase -- a walk that stands above the depth is given up, and so are all walks of a warp that has counted
// kMaxWarpSteps since its lanes last took slots.  A turn takes every walking lane a step on and a repeated node step at
// least kNodeLanes of them, so walks of up to kMaxSteps steps never meet that count.  A look at the stack at every push
// instead costs 2% of the 1080p frame and 3% of its two-level form, a count at every node step 1%.  With the stack looked
// at once a turn and every other step counted: the frame 1.485 -> 1.490 ms, the megakernel's 1.900 -> 1.922, the terrain
// 9.49 -> 9.53.  Two levels count every step, where a second copy of the step costs more than the count: the frame
// 1.580 -> 1.594 ms (1.597 by twos), the megakernel's 2.217 -> 2.261 (2.334).
constexpr uint32_t kPhaseSteps = 64;
constexpr uint32_t kMaxWarpSteps = (32u / kNodeLanes + 1u) * kMaxSteps;

__device__ __forceinline__ float3 shfl3(float3 v, uint32_t from) {
    return f3(__shfl_sync(0xFFFFFFFFu, v.x, from), __shfl_sync(0xFFFFFFFFu, v.y, from),
              __shfl_sync(0xFFFFFFFFu, v.z, from));
}

// Original id of a hit, looked up only to decide ties: the triangle's, in a two-level scene offset by the
// instance's first id.
__device__ __forceinline__ uint32_t pool_prim(const DevScene& s, uint32_t inst, uint32_t prim) {
    return __float_as_uint(__ldg(s.inst + 8 * (size_t)inst + 3).y) + prim;
}
template <bool INST>
__device__ __forceinline__ uint32_t pool_id(const DevScene& s, const float4* tris, uint32_t best, uint32_t inst) {
    if (best == kMiss) return kMiss;
    const uint32_t prim = __float_as_uint(__ldg(tris + 3 * (size_t)best).w);
    return INST ? pool_prim(s, inst, prim) : prim;
}

// One lane's walk, stepped in the phases above by all 32 lanes together.  A closest-hit walk starts with
// tbest = infinity and ends with the hit in (tbest, best, binst); an any-hit walk starts with its end distance in
// tbest, which turns negative when an occluder is found (`best` is the caller's).
// INST: a two-level scene.  A lane at a top-level leaf takes its ray into the leaf's instance (in the leaf
// phase) and walks the mesh's tree with the same stack, above the top-level entries (`floor` marks them);
// when the mesh's part of the stack is empty it returns to the world ray, kept in wo / wd.  Visits and tests
// are those of trace_closest_inst / trace_any_inst, in the same order.  Against those nested lockstep loops,
// on the 1080p frame of 200 placed spheres: bounce 1 879 -> 556 us, the frame 2.29 -> 1.76 ms (1.90 ms at 5
// blocks an SM with 144 bytes of spills).
template <bool INST>
struct Walker {
    // (reference, entry distance); each tree is shallower than kStack.  An array of its own beside the
    // walker, whose other members then stay in registers.
    static constexpr int kDepth = INST ? 2 * kStack : kStack;
    using Stack = uint2[kDepth + kPhaseSteps + 1];
    int sp = 0, floor = 0;
    uint32_t ref = kDone, best = kMiss;
    uint32_t cur = kMiss, binst = kMiss;       // INST: the instance the lane is in (kMiss: top level), the hit's
    float3 o, d, id, wo, wd;
    float tbest = 0.f;
    const float4 *nodes, *tris;

    __device__ __forceinline__ explicit Walker(const DevScene& s)
        : nodes(INST ? s.tlas : s.nodes), tris(s.tris) {
        o = d = id = wo = wd = f3(0.f, 0.f, 0.f);
    }
    // Begin at the root; the caller has set o, d, tbest and best.
    __device__ __forceinline__ void begin(const DevScene& s) {
        id = ray_rcp(d);
        ref = 0u;
        sp = 0;
        if (INST) {
            wo = o;
            wd = d;
            nodes = s.tlas;
            cur = binst = kMiss;
            floor = 0;
        }
    }
    // The next deferred subtree whose entry is not beyond the best hit.
    __device__ __forceinline__ void pop(const DevScene& s, Stack& stk) {
        ref = kDone;
        if constexpr (!INST) {
            while (sp > 0) {
                const uint2 v = stk[--sp];
                if (__uint_as_float(v.y) <= tbest * 1.0000005f) {
                    ref = v.x;
                    return;
                }
            }
        } else {
            while (true) {
                if (sp == floor) {
                    if (cur == kMiss) return;
                    cur = kMiss;               // the mesh is done: back to the top level
                    floor = 0;
                    nodes = s.tlas;
                    o = wo;
                    d = wd;
                    id = ray_rcp(d);
                    continue;
                }
                const uint2 v = stk[--sp];
                if (__uint_as_float(v.y) <= tbest * 1.0000005f) {
                    ref = v.x;
                    return;
                }
            }
        }
    }
    // Node steps while at least kNodeLanes lanes hold an inner node, kPhaseSteps at most; counted in `steps`.
    __device__ __forceinline__ void node_phase(const DevScene& s, Stack& stk, uint32_t& steps) {
        const auto step = [&]() -> bool {
            if (!(ref & kLeafBit)) {
                float4 n0, n1, n2;
                uint2 r;
                load_node(nodes, ref, n0, n1, n2, r);
                float t0, t1;
                bool h0, h1;
                box_test2(n0, n1, n2, o, id, tbest, t0, t1, h0, h1);
                // the child to walk next (the nearer one when both boxes are hit) and the one deferred
                const bool first0 = h0 && (t0 <= t1 || !h1);
                ref = first0 ? r.x : r.y;
                if (h0 && h1) stk[sp++] = make_uint2(first0 ? r.y : r.x, __float_as_uint(first0 ? t1 : t0));
                else if (!(h0 || h1)) pop(s, stk);
            }
            return (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, !(ref & kLeafBit))) >= kNodeLanes;
        };
        uint32_t i = 0;
        if constexpr (INST) {
            while (step() && ++i < kPhaseSteps) {
            }
            steps += i;
        } else {
            while (step() && step() && ++i < kPhaseSteps / 2u) {
            }
            steps += 2u * i;
        }
    }
    // One leaf step of the lanes that hold a leaf; `any`: the lane's walk is an any-hit one.
    __device__ __forceinline__ void leaf_phase(const DevScene& s, Stack& stk, bool any) {
        if (!(ref & kLeafBit) || ref == kDone) return;
        const uint32_t first = (ref & 0x7FFFFFFFu) >> 3, n_leaf = (ref & 7u) + 1u;
        if (INST && cur == kMiss) {
            // the leaf's instances one after the other (the builder makes leaves of one)
            if (n_leaf > 1u) stk[sp++] = make_uint2(kLeafBit | (first + 1u) << 3 | (n_leaf - 2u), 0u);
            const InstRay r = instance_ray(s, first, wo, wd);
            cur = first;
            floor = sp;
            nodes = s.nodes;
            o = r.o;
            d = r.d;
            id = ray_rcp(d);
            ref = r.root;
            return;
        }
        bool over = false;
        for (uint32_t k = 0; k < n_leaf && !over; ++k) {
            float t;
            uint32_t prim;
            if (!tri_test(tris, first + k, o, d, t, prim) || !(t > 0.0f)) continue;
            if (any) {
                over = t < tbest;
            } else if (t < tbest || (t == tbest && pool_id<INST>(s, tris, best, binst) >
                                                       (INST ? pool_prim(s, cur, prim) : prim))) {
                tbest = t;
                best = first + k;
                if (INST) binst = cur;
            }
        }
        if (over) {
            tbest = -1.0f;       // occluded
            ref = kDone;
        } else {
            pop(s, stk);
        }
    }
    // The end of a turn.
    __device__ __forceinline__ void guard(const DevScene& s, uint32_t& steps) {
        if (++steps >= kMaxWarpSteps || sp > kDepth) {
            if (ref != kDone) atomicOr(s.status, ST_TRAVERSAL);
            ref = kDone;
            sp = 0;
        }
    }
};

// A slot of the pool: an extension ray's queue index, or a shadow ray's with kAnySlot set (capacities stay
// far below 2^31: a path's records take 180 bytes).
constexpr uint32_t kAnySlot = 0x80000000u;

// The end of a pool.  With no slot left, lanes run dry while the longest walks -- chains of several hundred
// dependent node loads -- keep the launch alive.  Here the walks that are left belong to the warp: a lane
// without work takes the oldest deferred subtree (the one nearest the root; as in work stealing, Blumofe and Leiserson,
// "Scheduling Multithreaded Computations by Work Stealing", 1999) of a lane that holds one, with
// that lane's ray, and walks it.  A ray's best hit so far, the smallest (t, original id), lies in shared memory under
// its first lane's number; it culls every lane that works on the ray, and is the hit at the end: the closest-hit
// rule makes it independent of the order of the walk (as in trace_closest_group).  When the slots ran out the
// launches of a 1080p frame lasted another 70 to 80 us, the length of one walk: 1.601 -> 1.547 ms with this, its
// adjoint 1.700 -> 1.654 ms.  It goes in phases too: kDrainSteps node steps, a leaf step, then subtrees change hands.
// 1, 2, 3, 4 steps: the frame 1.485, 1.484, 1.483, 1.489 ms, four 720p frames 2.091, 2.053, 2.037, 2.044 (1.494 and
// 2.111 with a node or leaf step of each lane in turn).  6, 12 or 20 idle lanes before it starts measure the same.
constexpr uint32_t kDrainLanes = 12;
constexpr int kDrainSteps = 3;
struct DrainShared {
    unsigned long long key[32];       // t | original id of the ray's best hit
    uint32_t tri[32];                 // its triangle (any-hit rays: the caller's `best`)
    uint32_t lane[32];                // donors, in lane order
};
constexpr uint32_t kAnyRec = 32u;     // flag of a record number: an any-hit ray

// Not inlined, and given the lane's walk as plain values, so that the loop above keeps its registers; the
// rays are read again.
template <class Io>
__device__ __noinline__ void pool_drain(const Io& io, DrainShared& sh, uint32_t slot, Walker<false>::Stack& stk, int sp,
                                        uint32_t ref, float tbest, uint32_t best) {
    const uint32_t lane = lane_id(), below = (1u << lane) - 1u;
    const DevScene s = io.scene();
    Walker<false> k(s);
    if (slot != kNoSlot) {
        io.fetch(slot, k.o, k.d, k.tbest, k.best, k.nodes, k.tris);
        k.id = ray_rcp(k.d);
        k.tbest = tbest;
        k.best = best;
    }
    k.ref = ref;
    k.sp = sp;
    uint32_t rec = lane | ((slot & kAnySlot) ? kAnyRec : 0u), occluded = 0u;
    if (slot != kNoSlot) {
        sh.key[lane] = (unsigned long long)__float_as_uint(k.tbest) << 32 |
                       ((rec & kAnyRec) ? kMiss : pool_id<false>(s, k.tris, k.best, kMiss));
        sh.tri[lane] = k.best;
    }
    __syncwarp();
    int bot = 0;                      // the lane's deferred subtrees: stk[bot .. k.sp)
    for (uint32_t steps = 0;; ++steps) {
        const uint32_t r = rec & 31u;
        bool hit = false;
        unsigned long long cand = 0ull;
        uint32_t cand_tri = 0u;
        const auto pop = [&] {
            k.ref = kDone;
            while (k.sp > bot) {
                const uint2 v = stk[--k.sp];
                if (__uint_as_float(v.y) <= k.tbest * 1.0000005f) {
                    k.ref = v.x;
                    break;
                }
            }
        };
        if (k.ref != kDone) k.tbest = __uint_as_float((uint32_t)(sh.key[r] >> 32));
#pragma unroll 1
        for (int rep = 0; rep < kDrainSteps; ++rep) {
            if (!(k.ref & kLeafBit)) {
                float4 n0, n1, n2;
                uint2 c;
                load_node(k.nodes, k.ref, n0, n1, n2, c);
                float t0, t1;
                bool h0, h1;
                box_test2(n0, n1, n2, k.o, k.id, k.tbest, t0, t1, h0, h1);
                const bool first0 = h0 && (t0 <= t1 || !h1);
                k.ref = first0 ? c.x : c.y;
                if (h0 && h1) stk[k.sp++] = make_uint2(first0 ? c.y : c.x, __float_as_uint(first0 ? t1 : t0));
                else if (!(h0 || h1)) pop();
            }
            __syncwarp();
        }
        if (k.ref != kDone && (k.ref & kLeafBit)) {
            const uint32_t first = (k.ref & 0x7FFFFFFFu) >> 3, n_leaf = (k.ref & 7u) + 1u;
            cand = sh.key[r];
            for (uint32_t i = 0; i < n_leaf; ++i) {
                float t;
                uint32_t prim;
                if (!tri_test(k.tris, first + i, k.o, k.d, t, prim) || !(t > 0.0f)) continue;
                if (rec & kAnyRec) {
                    hit = hit || t < k.tbest;
                } else {
                    const unsigned long long v = (unsigned long long)__float_as_uint(t) << 32 | prim;
                    if (v < cand) {
                        cand = v;
                        cand_tri = first + i;
                        hit = true;
                    }
                }
            }
            if (hit && !(rec & kAnyRec)) {
                atomicMin(&sh.key[r], cand);
                k.tbest = __uint_as_float((uint32_t)(cand >> 32));
            }
            pop();
        }
        __syncwarp();
        if (hit && !(rec & kAnyRec) && sh.key[r] == cand) sh.tri[r] = cand_tri;
        occluded |= __reduce_or_sync(0xFFFFFFFFu, hit && (rec & kAnyRec) ? 1u << r : 0u);
        if ((rec & kAnyRec) && ((occluded >> r) & 1u)) {
            k.ref = kDone;
            k.sp = bot;
        }
        if (k.sp > Walker<false>::kDepth) {
            atomicOr(s.status, ST_TRAVERSAL);
            k.ref = kDone;
            k.sp = bot;
        }
        const uint32_t idle = __ballot_sync(0xFFFFFFFFu, k.ref == kDone);
        if (idle == 0xFFFFFFFFu) break;
        const uint32_t donors = __ballot_sync(0xFFFFFFFFu, k.ref != kDone && k.sp > bot);
        if (idle && donors) {
            const uint32_t pairs = min((uint32_t)__popc(idle), (uint32_t)__popc(donors));
            const uint32_t rd = (uint32_t)__popc(donors & below), ri = (uint32_t)__popc(idle & below);
            uint2 give = make_uint2(kDone, 0u);
            if (((donors >> lane) & 1u) && rd < pairs) {
                give = stk[bot++];
                sh.lane[rd] = lane;
            }
            __syncwarp();
            const bool takes = ((idle >> lane) & 1u) && ri < pairs;
            const uint32_t from = takes ? sh.lane[ri] : lane;
            const uint2 got = make_uint2(__shfl_sync(0xFFFFFFFFu, give.x, from), __shfl_sync(0xFFFFFFFFu, give.y, from));
            const uint32_t rec2 = __shfl_sync(0xFFFFFFFFu, rec, from);
            const float3 o2 = shfl3(k.o, from), d2 = shfl3(k.d, from), id2 = shfl3(k.id, from);
            if (takes) {
                rec = rec2;
                k.o = o2;
                k.d = d2;
                k.id = id2;
                k.sp = bot = 0;
                if (__uint_as_float(got.y) <= __uint_as_float((uint32_t)(sh.key[rec & 31u] >> 32)) * 1.0000005f)
                    k.ref = got.x;
            }
        }
        if (steps >= kMaxSteps) {
            if (k.ref != kDone) atomicOr(s.status, ST_TRAVERSAL);
            break;
        }
    }
    __syncwarp();
    if (slot != kNoSlot)
        io.emit(slot, ((occluded >> lane) & 1u) ? -1.0f : __uint_as_float((uint32_t)(sh.key[lane] >> 32)), sh.tri[lane],
                kMiss);
}

// The pool's slots [0, n_ext) are the extension rays, [n_ext, q.total) the shadow rays.
// SHARE: the end of the pool is walked by pool_drain.
template <bool INST, bool SHARE, class Pool, class Io>
__device__ __forceinline__ void pool_walk(const DevScene& s, Pool& q, uint32_t n_ext, const Io& io) {
    __shared__ DrainShared sh[SHARE ? 8 : 1];
    Walker<INST> k(s);
    typename Walker<INST>::Stack stk;
    uint32_t slot = kNoSlot, steps = 0;
    while (true) {
        const uint32_t idle = __ballot_sync(0xFFFFFFFFu, k.ref == kDone);
        const bool all = idle == 0xFFFFFFFFu;
        if constexpr (SHARE) {
            static_assert(!INST, "single-level scenes");
            if (!all && !q.more() && (uint32_t)__popc(idle) >= kDrainLanes) {
                if (k.ref == kDone && slot != kNoSlot) {
                    io.emit(slot, k.tbest, k.best, k.binst);
                    slot = kNoSlot;
                }
                pool_drain(io, sh[threadIdx.x >> 5], slot, stk, k.sp, k.ref, k.tbest, k.best);
                break;
            }
        }
        if (all || ((uint32_t)__popc(idle) >= kIdleLanes && q.more())) {
            if (k.ref == kDone && slot != kNoSlot) {
                io.emit(slot, k.tbest, k.best, k.binst);
                slot = kNoSlot;
            }
            if (!q.more()) break;
            const uint32_t j = q.take(idle);
            if (j < q.total) {
                slot = j < n_ext ? j : ((j - n_ext) | kAnySlot);
                io.fetch(slot, k.o, k.d, k.tbest, k.best, k.nodes, k.tris);
                k.begin(s);
            }
            steps = 0;
        }
        k.node_phase(s, stk, steps);
        k.leaf_phase(s, stk, (slot & kAnySlot) != 0u);
        k.guard(s, steps);
    }
}

}  // namespace pt
