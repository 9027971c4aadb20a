// Many right-hand sides (many lights): kernels with one lane per column.
//
// With C columns the per-hit work of the gather is a row of C x nc coefficients of the
// source surfel.  The 3-column kernels (rgs_solve.cu, rgs_adjoint.cu) would re-read every
// hit record once per 3-column tile; here a warp takes one ray at
// a time and its 32 lanes take 32 consecutive columns, so each hit is read once per
// 32-column tile and every row load is one contiguous 512-byte (BF16) or 1-KiB (FP32)
// warp access.  Which layout a launch uses is decided per kernel family by wide_bounce and
// wide_opacity (rgs_internal.cuh).
#include "rgs_bounce_body.cuh"

namespace {

// ------------------------------------------------------------------ forward bounce
template <int NC, class T>
__global__ void RGS_MCB_LB k_bounce_mc(SceneDev sc, RaysDev rays, int C, const T *__restrict__ Bg,
                                                         const float *__restrict__ Bprev, const float *__restrict__ S,
                                                         float *__restrict__ Qout, float *__restrict__ Bout,
                                                         __nv_bfloat16 *__restrict__ Bout16, double *norm2) {
    __shared__ float red[MC_WARPS * NC * 32];
    bounce_receiver_mc<NC, T>(sc, rays, C, Bg, Bprev, S, Qout, Bout, Bout16, norm2, blockIdx.x, blockIdx.y, red);
}

// ------------------------------------------------------------------ adjoint
// opacity backward, ray by ray: per hit g_h (partial over this column tile and iterate chunk)
// accumulated into gh[slot]; a warp per ray, lanes over columns.  The lanes hold 32 of the ray's
// records at a time, four hits' rows are requested together, and their four sums over the
// columns share one reduction: with a hit, its row and a five-step reduction at a time every
// hit waited for the last, and lane 0's stores took a request each (60,000 surfels, 128 rays, 48
// columns, two launches: 103 -> 85 ms).  HALF: a tile of up to 16 columns, the upper 16 lanes
// take every other hit (85 -> 75 ms).
template <int NC, int NA, class T, bool HALF>
__global__ void RGS_MC_LB k_opacity_g_mc(SceneDev sc, RaysDev rays, int C, int ct, int na,
                                                            OpaSet<T, NA> it, float *gh, bool first) {
    constexpr int RS = row_stride<NC, T>();
    constexpr bool COOP = sizeof(T) == 4 && NC == 16 && !HALF; // whole-tile reads (TileDot)
    const int warp_g = (int)((blockIdx.x * (size_t)MC_THREADS + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    const int n_rays = sc.n * rays.nd;
    if (warp_g >= n_rays) return; // whole warps
    const int r = warp_g;
    const int cnt = rays.cnt[r];
    if (cnt == 0) return;
    int own = HALF ? lane & 15 : lane; // the tile column whose terms this lane forms
    if constexpr (COOP) own = TileDot<T, NC>::own(lane);
    const int col = ct * 32 + own;
    const bool live = col < C;
    const int colc = live ? col : C - 1;
    const int ncols = min(32, C - ct * 32);
    const int i = r / rays.nd;
    const float3 n = f3(sc.N4[i]);
    const float3 d = f3(rays.dir[r]);
    float Yo[NC], y[NA];
    {
        float Yi[NC];
        sh_eval<NC>(neg3(d), Yo);
        sh_eval<NC>(reflect_n(n, d), Yi);
        const float oi = alpha_center(sc, i) * (3.14159265358979f / (float)rays.nd);
#pragma unroll
        for (int aa = 0; aa < NA; ++aa) {
            float s = 0.f;
            if (aa < na && live) {
                float v[NC];
                load_col<NC>(it.v[aa] + ((size_t)i * C + col) * NC, v);
#pragma unroll
                for (int k = 0; k < NC; ++k) s += __ldg(&sc.cl[(size_t)i * 12 + band_of(k) * 3 + col % 3]) * Yi[k] * v[k];
            }
            y[aa] = oi * s;
        }
    }
    const long long base = rays.off[r];
    [[maybe_unused]] float ys[8]; // this lane's half of Y(-d) (TileDot)
    if constexpr (COOP) TileDot<T, NC>::pick(Yo, lane, ys);
    constexpr int U = 4;
    for (int h0 = 0; h0 < cnt; h0 += 32) {
        const int m = min(32, cnt - h0);
        const int jl = lane < m ? __ldg(&rays.rec_ja[base + h0 + lane]).x : 0;
        float mine = 0.f; // g of hit h0 + lane
        const int half = HALF ? lane >> 4 : 0;
        for (int q = 0; q < m; q += HALF ? 2 * U : U) {
            int j[U];
            float acc[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                j[u] = __shfl_sync(0xffffffffu, jl, min(HALF ? q + 2 * u + half : q + u, m - 1));
                acc[u] = 0.f;
            }
#pragma unroll
            for (int aa = 0; aa < NA; ++aa) {
                if (aa < na) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        float s = 0.f;
                        if constexpr (COOP) {
                            s = TileDot<T, NC>::dot(it.b[aa] + ((size_t)j[u] * C + ct * 32) * RS, ncols, lane, ys);
                        } else {
                            float v[NC];
                            load_col<NC>(it.b[aa] + ((size_t)j[u] * C + colc) * RS, v);
#pragma unroll
                            for (int k = 0; k < NC; ++k) s += Yo[k] * v[k];
                        }
                        acc[u] += y[aa] * s;
                    }
                }
            }
            // the four sums over the (half) warp at once: its two top lane bits come to select the hit
            constexpr int B1 = HALF ? 8 : 16, B2 = B1 / 2;
            const bool b1 = lane & B1, b2 = lane & B2;
            const float s01 = (b1 ? acc[1] : acc[0]) + __shfl_xor_sync(0xffffffffu, b1 ? acc[0] : acc[1], B1);
            const float s23 = (b1 ? acc[3] : acc[2]) + __shfl_xor_sync(0xffffffffu, b1 ? acc[2] : acc[3], B1);
            float s = (b2 ? s23 : s01) + __shfl_xor_sync(0xffffffffu, b2 ? s01 : s23, B2);
#pragma unroll
            for (int off = B2 / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            const int d = lane - q, u = HALF ? d >> 1 : d;
            const int from = (u & 1 ? B1 : 0) | (u & 2 ? B2 : 0) | (HALF && (d & 1) ? 16 : 0);
            s = __shfl_sync(0xffffffffu, s, from);
            if (d >= 0 && u < U) mine = s;
        }
        if (lane < m) {
            const long long slot = base + h0 + lane;
            gh[slot] = first ? mine : gh[slot] + mine;
        }
    }
}

} // namespace

// ------------------------------------------------------------------ launchers
template <int NC>
rgs_status mc_bounce(const rgs_transport *t, SceneDev sd, RaysDev rd, bool rows16, const float *Bprev,
                     const __nv_bfloat16 *Bprev16, const float *S, float *Q, float *Bout, __nv_bfloat16 *Bout16,
                     double *norm2, cudaStream_t st) {
    dim3 grid(t->n, (t->C + 31) / 32);
    if (rows16) {
        ProfScope ps_("k_bounce_mc", st);
        k_bounce_mc<NC, __nv_bfloat16><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, Bprev16, Bprev, S, Q, Bout, Bout16, norm2);
    } else {
        ProfScope ps_("k_bounce_mc", st);
        k_bounce_mc<NC, float><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, Bprev, Bprev, S, Q, Bout, Bout16, norm2);
    }
    RGS_LAUNCH("bounce_mc");
    return RGS_OK;
}

template <int NC>
rgs_status mc_opacity(rgs_transport *t, SceneDev sd, RaysDev rd, int na, const float *const *v, const float *const *Bf,
                      const __nv_bfloat16 *const *Bh, bool first, cudaStream_t st) {
    constexpr int NA = 4;
    const long long n_rays = (long long)t->n * t->nd;
    const unsigned grid = (unsigned)((n_rays * 32 + MC_THREADS - 1) / MC_THREADS);
    OpaSet<float, NA> sf = {};
    OpaSet<__nv_bfloat16, NA> sh = {};
    for (int a = 0; a < na; ++a) {
        sf.v[a] = sh.v[a] = v[a];
        sf.b[a] = Bf[a];
        sh.b[a] = Bh ? Bh[a] : nullptr;
    }
    for (int ct = 0; ct * 32 < t->C; ++ct) {
        if (Bh) {
            ProfScope ps_("k_opacity_g_mc", st);
            if (half_tile(NC, t->C - ct * 32, true))
                k_opacity_g_mc<NC, NA, __nv_bfloat16, true><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, ct, na, sh, t->gh, first && ct == 0);
            else
                k_opacity_g_mc<NC, NA, __nv_bfloat16, false><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, ct, na, sh, t->gh, first && ct == 0);
        } else {
            ProfScope ps_("k_opacity_g_mc", st);
            if (half_tile(NC, t->C - ct * 32, false))
                k_opacity_g_mc<NC, NA, float, true><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, ct, na, sf, t->gh, first && ct == 0);
            else
                k_opacity_g_mc<NC, NA, float, false><<<grid, MC_THREADS, 0, st>>>(sd, rd, t->C, ct, na, sf, t->gh, first && ct == 0);
        }
    }
    RGS_LAUNCH("opacity mc");
    return RGS_OK;
}

#define RGS_MC_INSTANTIATE(NC)                                                                                         \
    template rgs_status mc_bounce<NC>(const rgs_transport *, SceneDev, RaysDev, bool, const float *,                   \
                                      const __nv_bfloat16 *, const float *, float *, float *, __nv_bfloat16 *,         \
                                      double *, cudaStream_t);                                                         \
    template rgs_status mc_opacity<NC>(rgs_transport *, SceneDev, RaysDev, int, const float *const *,                 \
                                       const float *const *, const __nv_bfloat16 *const *, bool, cudaStream_t);
RGS_MC_INSTANTIATE(1)
RGS_MC_INSTANTIATE(4)
RGS_MC_INSTANTIATE(9)
RGS_MC_INSTANTIATE(16)
