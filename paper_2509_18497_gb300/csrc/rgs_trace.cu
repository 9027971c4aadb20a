// Transport tracing (rgs_trace_transport).
//
//  k_trace_hemi : a warp per 32 hemisphere rays (App. B) of one surfel.  Hits are collected
//                 during BVH traversal, put in depth order (near-equal depths by caller
//                 index), alpha-composited (Eq. L_I) and stored contiguously per ray.
//  k_direct     : a lane per (surfel, light) shadow ray; transmittance product and
//                 the direct term D (Sec. 5.2) for every column of that light.
//  k_src_*      : the same records grouped by source surfel (transposed index) for the
//                 adjoint's gather form of K^T.
#include <algorithm>

#include "rgs_warp_trace.cuh"

#ifndef RGS_TRACE_PATCH_A
#define RGS_TRACE_PATCH_A 8
#endif
#ifndef RGS_TRACE_MINB
#define RGS_TRACE_MINB 8 // resident 128-thread blocks per SM the register budget is sized for (measured best)
#endif
constexpr int HEMI_THREADS = 128, DIRECT_THREADS = 128;

namespace {

// A warp per patch of 32 rays of one surfel (or a part of it), patches handed out by a counter.  The lanes walk
// the tree for their own rays and pool the surfel tests (rgs_warp_trace.cuh); accepted hits
// go to per-ray lists in this warp's scratch (rewritten for every patch; all warps' 319 MB are
// more than the L2 holds, and what of them reaches DRAM is four times the records' bytes, a
// twentieth of the time at the copy rate), each ray's traversal ends once the hits found make the
// rest invisible, and the warp then orders and composites one ray after the other, a lane per hit.  It allocates exactly
// its rays' kept hits with one atomic and stores every ray's records contiguously.
__global__ void __launch_bounds__(HEMI_THREADS, RGS_TRACE_MINB) k_trace_hemi(SceneDev sc, RaysDev rays, long long jobs, int split, long long cap_slots,
                                                       unsigned long long *slot_ctr, unsigned *work, int2 *rec_ja,
                                                       long long *off_out, int *cnt_out, float4 *dir_out,
                                                       int *src_cnt, int *flags, int pa, int4 *lists) {
    __shared__ WarpHits sm_all[HEMI_THREADS / 32];
    const int lane = threadIdx.x & 31;
    WarpHits &sm = sm_all[threadIdx.x >> 5];
    int4 *list = lists + (size_t)(blockIdx.x * (HEMI_THREADS / 32) + (threadIdx.x >> 5)) * (32 * WT_LIST);
    const float eps = *sc.eps_plane;
    const int per = rays.nd >> 5; // patches of a surfel
    while (true) {
        unsigned job = 0;
        if (lane == 0) job = atomicAdd(work, 1u);
        job = __shfl_sync(WT_FULL, job, 0);
        if (job >= jobs) return;
        // a patch of 32 rays, or one of its `split` parts
        const unsigned w = job / (unsigned)split;
        const bool active = lane / (32 / split) == (int)(job - w * (unsigned)split);
        // the warps of surfel i take patches of pa x (32 / pa) strata (elevation x azimuth) of its
        // na x nbs grid, so that a warp's rays leave in similar directions; pa = 0: 32 consecutive rays
        const int i = (int)(w / (unsigned)per), pt = (int)(w - (unsigned)i * (unsigned)per);
        int q = pt * 32 + lane;
        if (pa > 0) {
            const int pb = 32 / pa, per_row = rays.nbs / pb;
            const int a = (pt / per_row) * pa + lane / pb, b = (pt % per_row) * pb + lane % pb;
            q = a * rays.nbs + b;
        }
        const int r = i * rays.nd + q; // this lane's ray (outputs are indexed by ray)
        const float3 o = f3(sc.P[i]);
        const float3 d = ray_dir(rays.seed, sc.uid[i], q, rays.na, rays.nbs, f3(sc.FU[i]), f3(sc.FV[i]), f3(sc.N4[i]));
        if (active) dir_out[r] = make_float4(d.x, d.y, d.z, 0.f);
        bool full;
        if (!warp_collect<false, false>(sc, o, d, i, active, eps, 0, sm, list, full)) atomicAdd(&flags[FLAG_STACK], 1);
        int kept = 0; // of this lane's ray
        for (int x = 0; x < 32; ++x) {
            int H = sm.cnt[x];
            if (H == 0) continue;
            float T = 1.f;
            unsigned long long last;
            const int k = warp_composite_any(sc, H, list + x * WT_LIST, sm, false, false, T, last);
            __syncwarp();
            if (lane == x) {
                kept = k;
                // a full list only loses something if the transmittance is still above the cut
                if (full && k == H && T >= RGS_T_EPS) atomicAdd(&flags[FLAG_FULL_RAYS], 1);
            }
        }
        // warp-aggregated, exactly sized record allocation
        int incl = kept;
#pragma unroll
        for (int offs = 1; offs < 32; offs <<= 1) {
            const int v = __shfl_up_sync(WT_FULL, incl, offs);
            if (lane >= offs) incl += v;
        }
        const int total = __shfl_sync(WT_FULL, incl, 31);
        unsigned long long sbase = 0;
        if (lane == 31 && total > 0) sbase = atomicAdd(slot_ctr, (unsigned long long)total);
        sbase = __shfl_sync(WT_FULL, sbase, 31);
        const unsigned long long mine = sbase + (unsigned long long)(incl - kept);
        const bool fits = mine + (unsigned long long)kept <= (unsigned long long)cap_slots;
        if (active) {
            off_out[r] = (long long)mine;
            cnt_out[r] = fits ? kept : 0;
        }
        if (!fits && active) atomicAdd(&flags[FLAG_CAPACITY], 1);
        const unsigned store = __ballot_sync(WT_FULL, fits && kept > 0);
        for (unsigned m = store; m; m &= m - 1) {
            const int x = __ffs(m) - 1;
            const int k = __shfl_sync(WT_FULL, kept, x);
            int2 *out = rec_ja + sbase + (unsigned)__shfl_sync(WT_FULL, incl - kept, x);
            for (int e = lane; e < k; e += 32) {
                const int2 ja = wt_hit(list + x * WT_LIST, e);
                out[e] = ja;
                atomicAdd(&src_cnt[ja.x], 1); // transposed-index histogram
            }
        }
        __syncwarp(); // the lists are rewritten by the next patch
    }
}

// Direct term (Sec. 5.2): D_i[L*3+ch][k] = o_i c_{i,l(k),ch} Y_k(R_i w) I_{L,ch} (n_i.w)/r^2 T
// (no 1/r^2 and a shadow ray to infinity for a directional light)
// A warp per 32 or 16 (surfel, light) pairs, their shadow rays traced together (rgs_warp_trace.cuh).
template <int NC>
__global__ void __launch_bounds__(DIRECT_THREADS) k_direct(SceneDev sc, int nl, int per, int ldir, const float *__restrict__ lpos,
                                                          const float *__restrict__ lint, int C, float *D, int *flags) {
    __shared__ WarpOcclusion sm[DIRECT_THREADS / 32];
    const int tid = (blockIdx.x * (DIRECT_THREADS / 32) + (threadIdx.x >> 5)) * per + (threadIdx.x & 31);
    const bool live = (threadIdx.x & 31) < per && tid < sc.n * nl;
    const int i = live ? tid / nl : 0, lt = live ? tid - i * nl : 0;
    const float4 Pi = sc.P[i];
    const float3 o = f3(Pi), n = f3(sc.N4[i]);
    float r, fall;
    const float3 w = light_dir(lpos, lt, o, ldir, r, fall);
    const float cs = dot3(n, w);
    const bool lit = live && cs > 0.f;
    float T;
    int nzero;
    if (!warp_transmittance<false>(sc, sm[threadIdx.x >> 5], o, w, r, i, lit, *sc.eps_plane, T, nzero,
                            [](int, const SurfelRec &, int) { return true; }))
        atomicAdd(&flags[FLAG_STACK], 1);
    if (!live) return;
    float *Dout = D + ((size_t)i * C + lt * 3) * NC;
    if (!lit) {
        for (int q = 0; q < 3 * NC; ++q) Dout[q] = 0.f;
        return;
    }
    if (nzero) T = 0.f;
    float Y[NC];
    sh_eval<NC>(reflect_n(n, w), Y);
    const float pre = alpha_center(sc, i) * cs * fall * T;
    for (int ch = 0; ch < 3; ++ch) {
        const float I = lint[3 * lt + ch];
        for (int k = 0; k < NC; ++k) Dout[ch * NC + k] = sc.cl[(size_t)i * 12 + band_of(k) * 3 + ch] * Y[k] * I * pre;
    }
}

} // namespace

static int strata_a(int nd) {
    int na = 1;
    while ((2 * na) * (2 * na) <= nd) na *= 2;
    return na;
}

// Shared by both transports: the light copies, the per-surfel buffers (flags, D, the
// per-source counts and offsets of the transposed index) sized for the scene.
rgs_status rgs_transport_common(rgs_transport *t, const rgs_lights *L, cudaStream_t st) {
    rgs_scene *sc = t->sc;
    const int n = sc->n;
    t->n = n;
    t->L = sc->L;
    t->nc = sc->nc;
    t->nl = L ? L->n_lights : 0;
    t->ldir = (L && L->directional) ? 1 : 0;
    t->C = 3 * (t->nl > 0 ? t->nl : 1);
    t->nb_last = -1;
    rgs_status r;
    if (t->nl > t->lcap) {
        if ((r = dev_alloc(&t->lpos, 3 * (size_t)t->nl, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->lint, 3 * (size_t)t->nl, &t->device_bytes)) != RGS_OK) return r;
        t->lcap = t->nl;
    }
    if (t->nl > 0) {
        RGS_CUDA(cudaMemcpyAsync(t->lpos, L->pos, sizeof(float) * 3 * t->nl, cudaMemcpyDeviceToDevice, st));
        RGS_CUDA(cudaMemcpyAsync(t->lint, L->intensity, sizeof(float) * 3 * t->nl, cudaMemcpyDeviceToDevice, st));
    }
    if (!t->counter && (r = dev_alloc(&t->counter, 1, &t->device_bytes)) != RGS_OK) return r;
    if (!t->flags && (r = dev_alloc(&t->flags, FLAG_COUNT, &t->device_bytes)) != RGS_OK) return r;
    const long long arr = (long long)n * t->C * t->nc;
    if (arr > t->nc_cap) {
        if ((r = dev_alloc(&t->D, (size_t)arr, &t->device_bytes)) != RGS_OK) return r;
        t->nc_cap = arr;
        t->iters_cap = 0; // iterate buffers are sized by the array size: force regrowth
        t->q_cap = 0;
        t->iters16_cap = 0;
    }
    if (n > t->src_cap) {
        if ((r = dev_alloc(&t->src_off, (size_t)n + 1, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->src_cnt, (size_t)n, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->cursor, (size_t)n, &t->device_bytes)) != RGS_OK) return r;
        t->scan_tmp_cap = rgs_scan_tmp_size(n);
        if ((r = dev_alloc(&t->scan_tmp, (size_t)t->scan_tmp_cap, &t->device_bytes)) != RGS_OK) return r;
        t->src_cap = n;
    }
    return RGS_OK;
}

// D = o c (x) Y(R w) I cos / r^2 T for every (surfel, light), or 0 without lights
rgs_status rgs_direct_term(rgs_transport *t, cudaStream_t st) {
    SceneDev sd = t->sc->dev();
    if (t->nl > 0) {
        const int per = shadow_pairs((long long)t->n * t->nl), pb = DIRECT_THREADS / 32 * per; // pairs of a warp, a block
        const int blocks = (t->n * t->nl + pb - 1) / pb;
        switch (t->nc) {
        case 1: { ProfScope ps_("k_direct", st); k_direct<1><<<blocks, DIRECT_THREADS, 0, st>>>(sd, t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->D, t->flags); } break;
        case 4: { ProfScope ps_("k_direct", st); k_direct<4><<<blocks, DIRECT_THREADS, 0, st>>>(sd, t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->D, t->flags); } break;
        case 9: { ProfScope ps_("k_direct", st); k_direct<9><<<blocks, DIRECT_THREADS, 0, st>>>(sd, t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->D, t->flags); } break;
        default: { ProfScope ps_("k_direct", st); k_direct<16><<<blocks, DIRECT_THREADS, 0, st>>>(sd, t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->D, t->flags); }
        }
        RGS_LAUNCH("direct");
    } else {
        RGS_CUDA(cudaMemsetAsync(t->D, 0, sizeof(float) * t->arr(), st));
    }
    return RGS_OK;
}

rgs_status rgs_trace_impl(rgs_transport *t, const rgs_lights *L, const rgs_trace_opts *o, cudaStream_t st) {
    rgs_scene *sc = t->sc;
    const int n = sc->n;
    rgs_status r;
    t->kind = RGS_KIND_HEMISPHERE;
    rgs_tc_invalidate(t);
    rgs_mc_free(t);
    t->tc_used = false;
    t->nd = o->nd;
    t->na = strata_a(o->nd);
    t->nbs = o->nd / t->na;
    t->seed = o->seed;
    if ((r = rgs_transport_common(t, L, st)) != RGS_OK) return r;
    const long long n_rays = (long long)n * o->nd;
    // per-ray arrays
    if (n_rays > t->rays_cap) {
        if ((r = dev_alloc(&t->cnt, (size_t)n_rays, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->dir, (size_t)n_rays, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->off, (size_t)n_rays, &t->device_bytes)) != RGS_OK) return r;
        t->rays_cap = n_rays;
    }

    long long want = o->hit_capacity > 0 ? o->hit_capacity : (t->cap_slots > 0 ? t->cap_slots : n_rays * 24);
    if (o->hit_capacity <= 0 && t->cap_slots == 0) {
        // first trace of a large transport: rather than reserve a guess of 24 slots per ray,
        // let the first pass only count (no slots: every warp's store is refused, the
        // counter still adds up) and reserve what it needs
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) cudaGetLastError();
        if ((double)want * sizeof(int2) > 0.25 * (double)free_b) want = 0;
    }
    SceneDev sd = sc->dev();
    // warp patch of the strata grid: the largest pa <= RGS_TRACE_PATCH_A dividing na with
    // 32 / pa dividing nbs; none (0) keeps 32 consecutive rays per warp
    int pa = 0;
    for (int c = RGS_TRACE_PATCH_A; c >= 1 && !pa; c >>= 1)
        if (t->na % c == 0 && 32 % c == 0 && t->nbs % (32 / c) == 0) pa = c;
    // A warp lasts as long as its slowest ray: few patches are traced in 2 or 4 parts (500
    // patches: 0.26, 0.19, 0.16 ms in 1, 2, 4 parts; 2,000: 0.33, 0.28, 0.31; 4,000: 0.46, 0.45, 0.59).
    const int split = n_rays < 750 * 32 ? 4 : (n_rays < 1500 * 32 ? 2 : 1);
    const long long jobs = n_rays / 32 * split;
    WarpLists warps{st};
    const long long records = 8 * std::max(want - t->cap_slots, 0ll); // still to be allocated
    if ((r = warps.get((const void *)k_trace_hemi, HEMI_THREADS, jobs, t->budget_room(records))) != RGS_OK) return r;
    for (int attempt = 0; attempt < 2; ++attempt) {
        if (want > t->cap_slots) {
            if ((r = dev_alloc(&t->rec_ja, (size_t)want, &t->device_bytes)) != RGS_OK) return r;
            t->cap_slots = want;
        }
        RGS_CUDA(cudaMemsetAsync(t->counter, 0, sizeof(unsigned long long), st));
        RGS_CUDA(cudaMemsetAsync(t->flags, 0, sizeof(int) * FLAG_COUNT, st));
        RGS_CUDA(cudaMemsetAsync(t->src_cnt, 0, sizeof(int) * n, st));
        RaysDev rd = t->rays();
        RGS_CUDA(cudaMemsetAsync(warps.work, 0, sizeof(unsigned), st));
        { ProfScope ps_("k_trace_hemi", st); k_trace_hemi<<<warps.blocks, HEMI_THREADS, 0, st>>>(sd, rd, jobs, split, t->cap_slots, t->counter, warps.work, t->rec_ja, t->off, t->cnt, t->dir, t->src_cnt, t->flags, pa, warps.lists); }
        RGS_LAUNCH("trace_hemi");
        unsigned long long used = 0;
        int flags[FLAG_COUNT];
        RGS_CUDA(cudaMemcpyAsync(&used, t->counter, sizeof used, cudaMemcpyDeviceToHost, st));
        RGS_CUDA(cudaMemcpyAsync(flags, t->flags, sizeof flags, cudaMemcpyDeviceToHost, st));
        RGS_CUDA(cudaStreamSynchronize(st));
        t->n_slots = (long long)used;
        t->n_full = flags[FLAG_FULL_RAYS];
        if (flags[FLAG_STACK]) {
            rgs_set_error("BVH traversal stack overflow on %d rays", flags[FLAG_STACK]);
            return RGS_ERR_CAPACITY;
        }
        if (!flags[FLAG_CAPACITY]) break;
        if (o->hit_capacity > 0 || attempt == 1) {
            rgs_set_error("hit-record capacity %lld slots too small (%llu needed)", t->cap_slots, used);
            return RGS_ERR_CAPACITY;
        }
        const unsigned long long slack = used > (1ull << 30) ? used / 32 : used / 8; // for later re-traces
        want = (long long)(used + slack + 1024);
    }

    if ((r = rgs_direct_term(t, st)) != RGS_OK) return r;

    // per-source hit counts -> offsets of the transposed index (filled by rgs_adjoint)
    if ((r = rgs_scan_counts(t->src_cnt, t->src_off, n, t->scan_tmp, t->scan_tmp_cap, st)) != RGS_OK) return r;
    long long total = 0;
    RGS_CUDA(cudaMemcpyAsync(&total, t->src_off + n, sizeof total, cudaMemcpyDeviceToHost, st));
    RGS_CUDA(cudaStreamSynchronize(st));
    t->n_hits = total;
    return RGS_OK;
}
