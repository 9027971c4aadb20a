// Warp-cooperative tracing: 32 rays per warp, each lane walking the BVH for its own ray, the
// surfel tests of all lanes pooled.
//
// A lane that reaches a leaf does not test the surfel: it appends (ray, surfel) to a queue of
// the warp in shared memory, and whenever 32 candidates are waiting the warp tests all of
// them at once, one per lane.  With the test inside the traversal loop nearly every iteration
// ran it for the one or two lanes at a leaf (11 of 32 lanes active per instruction, two test
// bodies per node); pooled, a warp of the 50,000-surfel bowl makes about 52 full tests
// instead of some 250 thin ones, and 27 of 32 lanes are active.  The tree is four wide for
// the same reason: a step costs votes, queue and stack beside the boxes.  These kernels are
// bound by instruction issue (73 % of the slots used; L1 50 %, L2 20 %, DRAM 5 %).  Measured,
// thread per ray before and warp per 32 rays now: hemisphere rays of the 50,000-surfel bowl
// (12.8 M) 40.6 -> 25.0 ms, its shadow backward 0.85 -> 0.39 ms; a 1920 x 1080 image of it
// 7.4 -> 3.1 ms; the pair backward of 4,000 surfels 46.4 -> 19.7 ms (with the blocks of rgs_pairs.cu).
#pragma once
#include <algorithm>

#include "rgs_internal.cuh"

constexpr unsigned WT_FULL = 0xffffffffu;
constexpr int WT_QUEUE = 32 + 4 * 32; // up to 31 candidates left over plus four per lane

// The lanes' traversal stacks: the first WT_SMEM_STACK entries (node, bits of its entry
// distance) in shared memory, entry s of lane l at [s][l]; deeper entries in local memory.
constexpr int WT_SMEM_STACK = 12;

struct __align__(16) WarpQueue {
    int2 stack[WT_SMEM_STACK][32];
    int2 cand[WT_QUEUE]; // (surfel, ray)
};

// Traversal of every lane's ray o + t d, 0 < t < tmax (lanes with active == false take part in
// the pooled tests only).  ORDERED: nearer children first all the way, which is what makes a
// limit found on the way cut anything off (with the waiting children in any order, half of the
// camera directions traced an image 2-4 times slower); otherwise only the nearest is first.
// test(j, ray, valid) is called by the whole warp, each lane with one candidate (valid: it has
// one), and followed by a warp barrier; after every pooled test limit(tmax) returns the lane's
// current tmax, so that what the tests found may cut the traversal short (no hit up to tmax is
// lost to it: slab4 is conservative).  FAR: the origin may lie outside the scene.  Returns false
// if this lane's stack overflowed (part of the tree was then skipped).
template <bool ORDERED, bool FAR, class Test, class Limit>
__device__ __forceinline__ bool warp_traverse(const SceneDev &sc, float3 o, float3 d, float tmax, bool active,
                                              WarpQueue &q, Test &&test, Limit &&limit) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const SlabRay ray = slab_ray(o, d);
    int2 deep[RGS_STACK - WT_SMEM_STACK];
    int sp = 0, qn = 0;
    int node = active ? 0 : -1;
    bool ok = true;
    if (sc.n == 1) { // no inner node: the one surfel is everybody's candidate
        const unsigned m = __ballot_sync(WT_FULL, active);
        if (active) q.cand[__popc(m & below)] = make_int2(0, lane);
        qn = __popc(m);
        node = -1;
    }
    while (true) {
        const bool walking = __any_sync(WT_FULL, node >= 0);
        if (!walking && qn == 0) break;
        unsigned hit = 0u;
        float t[4];
        int kid[4];
        if (node >= 0) {
            const BvhNode nd = ld_node(sc, node);
            hit = slab4<FAR>(nd, ray, tmax, t);
#pragma unroll
            for (int c = 0; c < 4; ++c) kid[c] = nd.kid[c];
        }
        if (walking) {
#pragma unroll
            for (int c = 0; c < 4; ++c) { // surfels to the queue
                const bool leaf = (hit >> (4 + c)) & 1u;
                const unsigned m = __ballot_sync(WT_FULL, leaf);
                if (leaf) q.cand[qn + __popc(m & below)] = make_int2(kid[c], lane);
                qn += __popc(m);
            }
        }
        // the nearest crossed node is next, the others wait on the stack, nearest on top (depths
        // are positive, so their bits order them; the child's number takes the lowest two bits)
        unsigned key[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) key[c] = (hit >> c) & 1u ? (__float_as_uint(t[c]) & ~3u) | c : 0xffffffffu;
        auto order = [&](int a, int b) {
            const unsigned lo = min(key[a], key[b]);
            key[b] = max(key[a], key[b]);
            key[a] = lo;
        };
        order(0, 1);
        order(2, 3);
        order(0, 2);
        if constexpr (ORDERED) {
            order(1, 3);
            order(1, 2);
        }
        auto child = [&](unsigned k) {
            const int a = k & 1u ? kid[1] : kid[0], b = k & 1u ? kid[3] : kid[2];
            return k & 2u ? b : a;
        };
        int next = (int)key[0] >= 0 ? child(key[0]) : -1;
        if (sp <= WT_SMEM_STACK - 3) {
#pragma unroll
            for (int c = 3; c >= 1; --c)
                if ((int)key[c] >= 0) {
                    q.stack[sp][lane] = make_int2(child(key[c]), (int)key[c]);
                    ++sp;
                }
        } else {
            for (int c = 3; c >= 1; --c)
                if ((int)key[c] >= 0) {
                    const int2 e = make_int2(child(key[c]), (int)key[c]);
                    if (sp < WT_SMEM_STACK) q.stack[sp][lane] = e;
                    else if (sp < RGS_STACK) deep[sp - WT_SMEM_STACK] = e;
                    else ok = false, --sp;
                    ++sp;
                }
        }
        // the pooled test of the last 32 candidates (one place in the code: the kernels that
        // inline all this are near the size of the instruction cache)
        while (qn >= 32 || (!walking && qn > 0)) {
            __syncwarp();
            const int m = min(qn, 32);
            qn -= m;
            const int2 e = lane < m ? q.cand[qn + lane] : make_int2(0, 0);
            test(e.x, e.y, lane < m);
            __syncwarp();
            tmax = limit(tmax);
        }
        while (next < 0 && sp > 0) { // the last waiting node that the limit has not passed
            --sp;
            const int2 e = sp < WT_SMEM_STACK ? q.stack[sp][lane] : deep[sp - WT_SMEM_STACK];
            if (__int_as_float(e.y & ~3) <= tmax) next = e.x; // (the lowest bits are the child's number)
        }
        node = next;
    }
    return ok;
}

// Hands the hits of a pooled test to the lanes that own their rays: every lane calls f(b) for
// the lanes b, in increasing order, whose candidate is a hit on this lane's ray.  What f reads of
// lane b has to be in shared memory before the call; a barrier separates the two.
struct WarpOwners {
    unsigned who[32]; // zero between calls
};
template <class F> __device__ __forceinline__ void warp_owner_loop(WarpOwners &w, bool hit, int ray, F &&f) {
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(WT_FULL, hit ? ray : 32 + lane);
    if (hit && !(peers & ((1u << lane) - 1u))) w.who[ray] = peers;
    __syncwarp();
    unsigned mine = w.who[lane];
    if (mine) w.who[lane] = 0u;
    for (; mine; mine &= mine - 1u) f(__ffs(mine) - 1);
}

// Shadow rays and segments, one per lane: what a pooled test needs of them, and the transmittance
// of each as its lane multiplies it up.
struct __align__(16) WarpOcclusion {
    WarpQueue q;
    float4 o[32], d[32]; // origin and own surfel; direction and length
    float om[32];
    WarpOwners own;
};
// (surfel, light) pairs that a warp takes: a warp lasts as long as its longest shadow ray, and
// up to 100,000 pairs are less than a wave of warps (8,000 surfels and a light, direct term and
// shadow backward with 32 pairs a warp, 16 and 8: 0.54, 0.38, 0.32 ms; 50,000: 0.65, 0.58, 0.66).
constexpr long long SHADOW_FEW = 100000;
inline int shadow_pairs(long long pairs) { return pairs <= SHADOW_FEW ? 16 : 32; }
// T = prod (1 - alpha_k) over the surfels k that the lane's ray (o, d, t < tmax, not `self`)
// meets, the factors that are exactly 0 counted in nzero instead; occluder(surfel, its record,
// lane of the ray) may reject a hit.  ONE: all rays have this origin and own surfel.  All lanes call.
template <bool ONE, class Occ>
__device__ __forceinline__ bool warp_transmittance(const SceneDev &sc, WarpOcclusion &s, float3 o, float3 d, float tmax,
                                                   int self, bool active, float eps, float &T, int &nzero,
                                                   Occ &&occluder) {
    const int lane = threadIdx.x & 31;
    if constexpr (!ONE) s.o[lane] = make_float4(o.x, o.y, o.z, __int_as_float(self));
    s.d[lane] = make_float4(d.x, d.y, d.z, tmax);
    s.own.who[lane] = 0u;
    T = 1.f;
    nzero = 0;
    __syncwarp();
    auto test = [&](int k, int ray, bool valid) {
        bool hit = false;
        const float4 ro = ONE ? make_float4(o.x, o.y, o.z, __int_as_float(self)) : s.o[ray];
        if (valid && k != __float_as_int(ro.w)) {
            const float4 rd = s.d[ray];
            const SurfelRec rec = ld_surfel(sc, k);
            float t, r2;
            hit = hit_rec(sc, rec, f3(ro), f3(rd), rd.w, eps, t, r2) && occluder(k, rec, ray);
            if (hit) s.om[lane] = 1.f - alpha_of(sc, rec.P.w, surfel_G(sc, r2));
        }
        warp_owner_loop(s.own, hit, ray, [&](int b) {
            const float om = s.om[b];
            if (om == 0.f) ++nzero;
            else T *= om;
        });
    };
    return warp_traverse<false, false>(sc, o, d, tmax, active, s.q, test, [](float m) { return m; });
}

// ------------------------------------------------------------------ ordered compositing
// log2(1 - alpha) in steps of 2^-16, for the early-out bound only (a fast approximation; whole
// numbers, because shared memory adds those in one instruction and floats in a
// compare-and-swap loop).  An opaque hit counts as 2^-24, and so does an alpha above 1: the
// transmittance behind it is below the cut.  A NaN counts as 2^24, no bound.
__device__ __forceinline__ int log_transmit(float alpha) {
    return (int)(65536.f * (alpha > 1.f ? -24.f : fmaxf(fminf(__log2f(1.f - alpha), 24.f), -24.f)));
}
// Once the hits found so far on a ray multiply to a transmittance below RGS_T_EPS, no hit
// behind the farthest of them is composited, so the ray may end there.  -20.2 leaves a
// quarter of a unit below log2(1e-6) = -19.93 for the approximations.  The margin behind
// that hit covers the depth-tie rule: a run of near-equal depths (gaps up to
// 1e-6 max(1, t)) is ordered by caller index, so a hit behind may still belong to a run that
// starts in front; a chain of gaps crossing 1e-4 max(1, t) takes more than RGS_HMAX hits.
constexpr int WT_LOG_CUT = (int)(-20.2 * 65536);
__device__ __forceinline__ float wt_limit(float far_hit) { return far_hit + 1.05e-4f * fmaxf(1.f, far_hit); }

constexpr int WT_LIST = RGS_HMAX + 32; // a ray's list: RGS_HMAX hits and one pooled test's more

struct __align__(16) WarpSort {
    float t[WT_LIST];
    int j[WT_LIST];
};

// A ray's list while its hits are collected: (surfel, depth bits, alpha bits, unused) a hit.
// A list that has outgrown RGS_HMAX (H <= WT_LIST hits): keeps the RGS_HMAX nearest (equal
// depths: the lower internal index) and returns the depth of the farthest of them.
__device__ __forceinline__ float warp_truncate(int H, int4 *list, WarpSort &s) {
    constexpr int K = WT_LIST / 32;
    const int lane = threadIdx.x & 31;
    int4 h[K];
    int rank[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = lane + 32 * k;
        rank[k] = 0;
        h[k] = make_int4(0, 0x7f800000, 0, 0);
        if (e < H) {
            h[k] = list[e];
            s.t[e] = __int_as_float(h[k].y);
            s.j[e] = h[k].x;
        }
    }
    __syncwarp();
    for (int m = 0; m < H; ++m) {
        const int tm = __float_as_int(s.t[m]), jm = s.j[m];
#pragma unroll
        for (int k = 0; k < K; ++k) rank[k] += (tm < h[k].y || (tm == h[k].y && jm < h[k].x)) ? 1 : 0;
    }
    int far = 0;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (lane + 32 * k < H && rank[k] < RGS_HMAX) {
            list[rank[k]] = h[k];
            far = max(far, h[k].y);
        }
    far = __reduce_max_sync(WT_FULL, far);
    __syncwarp();
    return __int_as_float(far);
}

// What a warp keeps of its 32 rays while their hits are collected.
struct WarpHits {
    WarpQueue q;
    float4 rd[32]; // direction and current depth limit of every ray
    int cnt[32];   // hits in its list
    int lg[32];    // sum of log2(1 - alpha) over them (log_transmit)
    int far[32];   // bits of the farthest one's depth
    unsigned long long lower[32]; // key (depth bits, surfel) that hits have to lie behind
    WarpSort sort;
};
// The nearest RGS_HMAX hits of every active lane's ray (o common to the warp's rays, hits
// behind the ray's `lower` key, not `self`), unordered, in lists [32][WT_LIST]; counts in
// s.cnt.  lg0: log2 of the transmittance in front (log_transmit's steps).  A ray's traversal
// ends once the hits found make the rest invisible.  full: this lane's ray had more than
// RGS_HMAX (in front of that end).  Returns false if this lane's stack overflowed.
// LOWER: `lower` is looked at; FAR: o may lie outside the scene (a camera).
template <bool LOWER, bool FAR>
__device__ __forceinline__ bool warp_collect(const SceneDev &sc, float3 o, float3 d, int self, bool active, float eps,
                                             int lg0, WarpHits &s, int4 *lists, bool &full) {
    const int lane = threadIdx.x & 31;
    s.rd[lane] = make_float4(d.x, d.y, d.z, INFINITY);
    s.cnt[lane] = 0;
    s.lg[lane] = lg0;
    s.far[lane] = 0;
    full = false;
    __syncwarp();
    auto test = [&](int j, int ray, bool valid) {
        if (!valid) return;
        const float4 dr = s.rd[ray];
        float t, r2, op;
        if (!hit_surfel_t(sc, j, self, o, f3(dr), INFINITY, eps, t, r2, op) || t > dr.w) return;
        if (LOWER && (((unsigned long long)__float_as_uint(t) << 32) | (unsigned)j) <= s.lower[ray]) return;
        const int at = atomicAdd(&s.cnt[ray], 1);
        const float alpha = alpha_of(sc, op, surfel_G(sc, r2));
        lists[ray * WT_LIST + at] = make_int4(j, __float_as_int(t), __float_as_int(alpha), 0);
        atomicAdd(&s.lg[ray], log_transmit(alpha));
        atomicMax(&s.far[ray], __float_as_int(t));
    };
    auto limit = [&](float tmax) {
        const unsigned big = __ballot_sync(WT_FULL, s.cnt[lane] > RGS_HMAX);
        if (s.lg[lane] < WT_LOG_CUT) tmax = fminf(tmax, wt_limit(__int_as_float(s.far[lane])));
        for (unsigned m = big; m; m &= m - 1) { // keep the RGS_HMAX nearest
            const int x = __ffs(m) - 1;
            const float far = warp_truncate(s.cnt[x], lists + x * WT_LIST, s.sort);
            if (lane == x) {
                s.cnt[x] = RGS_HMAX;
                tmax = fminf(tmax, far);
                full = true;
            }
        }
        s.rd[lane].w = tmax;
        __syncwarp();
        return tmax;
    };
    return warp_traverse<true, FAR>(sc, o, d, INFINITY, active, s.q, test, limit);
}

// One ray's H <= 32 K collected hits, put in depth order (ascending t; runs of near-equal depth
// by caller index) and composited by the whole warp: (j, a_h) to the first half of
// list[0 .. kept).  Returns kept, the hits up to the first whose transmittance in front is below
// the cut (an alpha above 1 makes the product negative, and a second one positive again); T: the
// transmittance in front of the ray's first hit, and then behind its last (0 where the list ended
// before).  nan_ends: whether a NaN transmittance ends the list.  cut: the last
// run of near-equal depths may go on behind the list, so it is left out (unless it is the whole
// list); H becomes the hits that count and last the largest key (depth bits, surfel) among them.
// K hits per lane; all lanes call.  sa, su: RGS_HMAX more words of shared memory each (the
// traversal's stack, which is empty by now).
template <int K>
__device__ __forceinline__ int warp_composite(const SceneDev &sc, int &H, int4 *list, WarpSort &s, float *sa, int *su,
                                              bool cut, bool nan_ends, float &T, unsigned long long &last) {
    const int lane = threadIdx.x & 31;
    float t[K], al[K];
    int j[K], rank[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = lane + 32 * k;
        const int4 h = e < H ? list[e] : make_int4(0, 0x7f800000, 0, 0);
        j[k] = h.x;
        t[k] = __int_as_float(h.y);
        al[k] = __int_as_float(h.z);
        rank[k] = 0;
        s.t[e] = t[k];
    }
    __syncwarp();
    for (int m = 0; m < H; m += 4) { // strictly nearer hits (the list is padded with infinities)
        const float4 tm = *reinterpret_cast<const float4 *>(&s.t[m]);
#pragma unroll
        for (int k = 0; k < K; ++k)
            rank[k] += (tm.x < t[k] ? 1 : 0) + (tm.y < t[k] ? 1 : 0) + (tm.z < t[k] ? 1 : 0) + (tm.w < t[k] ? 1 : 0);
    }
    // equal depths (always of one run, whose order follows below): by place in the list
    if constexpr (K == 1) {
        rank[0] += __popc(__match_any_sync(WT_FULL, __float_as_uint(t[0])) & ((1u << lane) - 1u));
    } else {
        for (int m = 0; m < H; ++m) {
            const float tm = s.t[m];
#pragma unroll
            for (int k = 0; k < K; ++k) rank[k] += (tm == t[k] && m < lane + 32 * k) ? 1 : 0;
        }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (lane + 32 * k < H) {
            s.t[rank[k]] = t[k];
            s.j[rank[k]] = j[k];
            sa[rank[k]] = al[k];
        }
    __syncwarp();
    unsigned starts[K];
    bool runs = false;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = lane + 32 * k;
        bool st = true;
        if (e < H && e > 0) {
            const float tp = s.t[e - 1];
            st = s.t[e] - tp > 1e-6f * fmaxf(1.f, tp);
        }
        starts[k] = __ballot_sync(WT_FULL, st);
        runs |= starts[k] != WT_FULL;
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (lane + 32 * k < H) {
            j[k] = s.j[lane + 32 * k];
            al[k] = sa[lane + 32 * k];
        }
    if (cut) {
        int b = 0; // the last run's first hit
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const int left = H - 32 * q;
            const unsigned m = left <= 0 ? 0u : starts[q] & (left >= 32 ? WT_FULL : (1u << left) - 1u);
            if (m) b = 32 * q + 31 - __clz(m);
        }
        if (b > 0) H = b;
        const unsigned tb = __float_as_uint(s.t[H - 1]);
        unsigned mj = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int e = lane + 32 * k;
            if (e < H && __float_as_uint(s.t[e]) == tb) mj = max(mj, (unsigned)j[k]);
        }
        last = ((unsigned long long)tb << 32) | __reduce_max_sync(WT_FULL, mj);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k >= H) al[k] = 0.f;
    }
    if (runs) { // each run by caller index
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k < H) su[lane + 32 * k] = __ldg(&sc.uid[j[k]]);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int e = lane + 32 * k;
            if (e < H) {
                int b = 0, f = H; // e's run: the last start up to e, the next one after it
#pragma unroll
                for (int q = 0; q <= k; ++q) {
                    const unsigned m = starts[q] & (q == k ? (2u << lane) - 1u : WT_FULL);
                    if (m) b = 32 * q + 31 - __clz(m);
                }
#pragma unroll
                for (int q = K - 1; q >= k; --q) {
                    const unsigned m = starts[q] & (q == k ? ~((2u << lane) - 1u) : WT_FULL);
                    if (m) f = min(H, 32 * q + __ffs(m) - 1);
                }
                const int u = su[e];
                int at = b;
                for (int m = b; m < f; ++m) at += su[m] < u ? 1 : 0;
                rank[k] = at;
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k < H) {
                s.j[rank[k]] = j[k];
                sa[rank[k]] = al[k];
            }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k < H) {
                j[k] = s.j[lane + 32 * k];
                al[k] = sa[lane + 32 * k];
            }
    }
    // a_h = alpha_h prod_{k<h} (1 - alpha_k), a product scan over the lanes
    int kept = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = lane + 32 * k;
        float inc = 1.f - al[k];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float v = __shfl_up_sync(WT_FULL, inc, off);
            if (lane >= off) inc *= v;
        }
        float exc = __shfl_up_sync(WT_FULL, inc, 1);
        exc = T * (lane == 0 ? 1.f : exc);
        const unsigned ends = __ballot_sync(WT_FULL, e >= H || (nan_ends ? !(exc >= RGS_T_EPS) : exc < RGS_T_EPS));
        const int here = kept == 32 * k ? (ends ? __ffs(ends) - 1 : 32) : 0; // (nothing behind an end)
        if (lane < here) *reinterpret_cast<int2 *>(&list[e]) = make_int2(j[k], __float_as_int(al[k] * exc));
        kept += here;
        T *= __shfl_sync(WT_FULL, inc, 31);
    }
    if (kept < H) T = 0.f;
    return kept;
}

__device__ __forceinline__ int warp_composite_any(const SceneDev &sc, int &H, int4 *list, WarpHits &s, bool cut,
                                                  bool nan_ends, float &T, unsigned long long &last) {
    float *sa = reinterpret_cast<float *>(&s.q.stack[0][0]);
    int *su = reinterpret_cast<int *>(sa + RGS_HMAX);
    if (H <= 32) return warp_composite<1>(sc, H, list, s.sort, sa, su, false, nan_ends, T, last); // (cut lists are full)
    if (H <= 64) return warp_composite<2>(sc, H, list, s.sort, sa, su, false, nan_ends, T, last);
    return warp_composite<3>(sc, H, list, s.sort, sa, su, cut, nan_ends, T, last);
}
// the composited hit e of a list
__device__ __forceinline__ int2 wt_hit(const int4 *list, int e) { return *reinterpret_cast<const int2 *>(&list[e]); }
static_assert(WT_SMEM_STACK * 64 >= 2 * RGS_HMAX, "the compositing borrows the stack");

// Warps of a persistent tracing grid: their scratch lists (2 KB a ray, 319 MB for the 4,864
// warps GB300 holds; where that is not to be had, fewer warps) and their work counter, pooled.
// room: bytes that a memory budget leaves for the lists (negative: no budget); under a budget the grid
// shrinks to what fits, but not below a block per SM (40 MB): fewer would idle the chip.
struct WarpLists {
    cudaStream_t st;
    int4 *lists = nullptr;
    unsigned *work = nullptr;
    int blocks = 0;
    ~WarpLists() {
        pool_release(lists, st);
        pool_release(work, st);
    }
    rgs_status get(const void *kernel, int threads, long long jobs, long long room) {
        int dev = 0, sms = 0, per_sm = 0;
        RGS_CUDA(cudaGetDevice(&dev));
        RGS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        RGS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0));
        const int warps = threads / 32;
        const size_t per_block = (size_t)warps * 32 * WT_LIST;
        const long long want = (jobs + warps - 1) / warps;
        long long fit = (long long)sms * (per_sm > 0 ? per_sm : 1);
        if (room >= 0) fit = std::min(fit, std::max((long long)sms, room / (long long)(per_block * sizeof(int4))));
        blocks = (int)(want < fit ? want : fit);
        if (blocks < 1) blocks = 1;
        rgs_status r;
        while ((r = pool_alloc(&lists, blocks * per_block, st)) == RGS_ERR_OOM && blocks > 1)
            blocks = (blocks + 1) / 2;
        if (r != RGS_OK) return r;
        return pool_alloc(&work, 1, st);
    }
};
