// Image formation (rgs_render / rgs_render_adjoint): Eq. L_I for the rays of a pinhole camera
// over a solved radiance B -- what the paper's tile rasterizer draws from the surfels'
// outgoing SH radiance (Sec. 5.3, end) -- and its transpose, the dL/dB a loss on the image
// hands to rgs_adjoint (Sec. 6, opening).
//
//  k_render : a warp per tile of 8 x 1 to 8 x 4 pixels.  The pixel rays o + t d meet the surfels in depth
//             order under the transport's hit rules (eps_plane, the cutoff, tie runs; no surfel
//             excluded), composited a_h = alpha_h prod_{k<h} (1 - alpha_k) until the
//             transmittance is below RGS_T_EPS, and the warp shades each pixel's hits at
//             once: I[c] = sum_h a_h Y(-d)^T B_j[c], or adds their a_h Y_k(-d) dI[c] to dB_j[c][k].
#include "rgs_bounce_body.cuh"
#include "rgs_warp_trace.cuh"

namespace {

constexpr int RN_THREADS = 128;
constexpr int RN_MINB = 7;   // resident blocks per SM the register budget is sized for
constexpr int RN_NARROW = 8; // up to this many columns a lane shades a hit, beyond it a column

// pixel (x, y) (y down) of a W x H pinhole camera cam = {o, forward, up} with vertical field
// of view fov: right = forward x up, the true up = right x forward, the pixel's centre
__device__ __forceinline__ float3 pixel_dir(const float *cam, int W, int H, float fov, int x, int y) {
    const float3 f = make_float3(cam[3], cam[4], cam[5]), u0 = make_float3(cam[6], cam[7], cam[8]);
    const float lf = sqrtf(dot3(f, f));
    const float3 fn = (1.f / lf) * f;
    float3 r = make_float3(fn.y * u0.z - fn.z * u0.y, fn.z * u0.x - fn.x * u0.z, fn.x * u0.y - fn.y * u0.x);
    r = (1.f / sqrtf(dot3(r, r))) * r;
    const float3 u = make_float3(r.y * fn.z - r.z * fn.y, r.z * fn.x - r.x * fn.z, r.x * fn.y - r.y * fn.x);
    const float th = tanf(0.5f * fov);
    const float sx = (2.f * (x + 0.5f) / (float)W - 1.f) * th * (float)W / (float)H;
    const float sy = (1.f - 2.f * (y + 0.5f) / (float)H) * th;
    float3 d = fn + sx * r + sy * u;
    return (1.f / sqrtf(dot3(d, d))) * d;
}

struct Cam {
    float v[9];
};

// internal [N][C][NC] <- user [N][nc][C]
template <int NC>
__global__ void k_render_from_user(int n, int C, const int *__restrict__ uid, const float *__restrict__ X, float *Y) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n * C * NC) return;
    const int k = (int)(idx % NC);
    const size_t ic = idx / NC;
    const int c = (int)(ic % C);
    const int i = (int)(ic / C);
    Y[idx] = X[((size_t)uid[i] * NC + k) * C + c];
}
// user [N][nc][C] <- internal [N][C][NC]
template <int NC>
__global__ void k_render_to_user(int n, int C, const int *__restrict__ uid, const float *__restrict__ X, float *Y) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n * C * NC) return;
    const int k = (int)(idx % NC);
    const size_t ic = idx / NC;
    const int c = (int)(ic % C);
    const int i = (int)(ic / C);
    Y[((size_t)uid[i] * NC + k) * C + c] = X[idx];
}

// I[c] (+)= sum over a pixel's composited hits (j, a_h) of a_h Y(-d)^T B_j[c], by a warp
template <int NC>
__device__ __forceinline__ void shade_pixel(const int4 *hits, int n, float3 d, int C, const float *__restrict__ B,
                                            float *out, bool first) {
    const int lane = threadIdx.x & 31;
    float Yo[NC];
    sh_eval<NC>(neg3(d), Yo);
    if (C <= RN_NARROW) {
        // few columns: a lane per hit (with a lane per column all but C lanes would idle)
        for (int c = 0; c < C; ++c) {
            float acc = 0.f;
            for (int h = lane; h < n; h += 32) {
                const int2 ja = wt_hit(hits, h);
                float v[NC];
                load_col<NC>(B + ((size_t)ja.x * C + c) * NC, v);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < NC; ++k) s += Yo[k] * v[k];
                acc += __int_as_float(ja.y) * s;
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(WT_FULL, acc, off);
            if (lane == 0) out[c] = first ? acc : out[c] + acc;
        }
        return;
    }
    if constexpr (NC == 16) {
        // 32-column tiles of each source row read as two contiguous 1-KB warp requests, every
        // lane ending with the dot product of one tile column (TileDot)
        float ys[8];
        TileDot<float, 16>::pick(Yo, lane, ys);
        const int own = TileDot<float, 16>::own(lane);
        for (int c0 = 0; c0 < C; c0 += 32) {
            const int ncols = min(32, C - c0);
            float acc = 0.f;
            for (int h = 0; h < n; ++h) {
                const int2 ja = wt_hit(hits, h);
                acc += __int_as_float(ja.y) * TileDot<float, 16>::dot(B + ((size_t)ja.x * C + c0) * 16, ncols, lane, ys);
            }
            if (own < ncols) out[c0 + own] = first ? acc : out[c0 + own] + acc;
        }
    } else {
        for (int c = lane; c < C; c += 32) {
            float acc = 0.f;
            for (int h = 0; h < n; ++h) {
                const int2 ja = wt_hit(hits, h);
                const float *row = B + ((size_t)ja.x * C + c) * NC;
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < NC; ++k) s += Yo[k] * __ldg(row + k);
                acc += __int_as_float(ja.y) * s;
            }
            out[c] = first ? acc : out[c] + acc;
        }
    }
}

// dB_j[c][k] += a_h Y_k(-d) dI[c] over a pixel's composited hits, by a warp
template <int NC>
__device__ __forceinline__ void scatter_pixel(const int4 *hits, int n, float3 d, int C, const float *__restrict__ dI,
                                              float *dB) {
    const int lane = threadIdx.x & 31;
    float Yo[NC];
    sh_eval<NC>(neg3(d), Yo);
    for (int e = lane; e < n * C; e += 32) { // (hit, column) pairs over the lanes
        const int h = e / C, c = e - h * C;
        const float g = __ldg(&dI[c]);
        if (g == 0.f) continue;
        const int2 ja = wt_hit(hits, h);
        const float ga = __int_as_float(ja.y) * g;
        float *row = dB + ((size_t)ja.x * C + c) * NC;
        if constexpr (NC % 4 == 0) { // rows of NC floats start on 16-byte boundaries
#pragma unroll
            for (int q = 0; q < NC / 4; ++q)
                atomicAdd(reinterpret_cast<float4 *>(row) + q,
                          make_float4(ga * Yo[4 * q], ga * Yo[4 * q + 1], ga * Yo[4 * q + 2], ga * Yo[4 * q + 3]));
        } else {
#pragma unroll
            for (int k = 0; k < NC; ++k) atomicAdd(row + k, ga * Yo[k]);
        }
    }
}

// Persistent warps take tiles of 8 x rows pixels from a counter; the lanes trace their pixels'
// rays together (rgs_warp_trace.cuh), then the warp composites and shades one pixel after the
// other from its scratch lists: no record leaves the SM's neighbourhood, and every ray is
// traced once.  A ray with more than RGS_HMAX hits in front of the transmittance cut takes
// further passes, each behind the last composited hit, so any number is composited.
// ADJ: in = dL/dimg, out = dL/dB (zeroed); else in = B, out = the image.
template <int NC, bool ADJ>
__global__ void __launch_bounds__(RN_THREADS, RN_MINB) k_render(SceneDev sc, Cam cam, int W, int H, int rows, float fov, int C,
                                                               const float *__restrict__ in, float *out, unsigned *work,
                                                               int4 *lists, int *flags) {
    __shared__ WarpHits sm_all[RN_THREADS / 32];
    const int lane = threadIdx.x & 31;
    WarpHits &sm = sm_all[threadIdx.x >> 5];
    int4 *list = lists + (size_t)(blockIdx.x * (RN_THREADS / 32) + (threadIdx.x >> 5)) * (32 * WT_LIST);
    const float eps = *sc.eps_plane;
    const int tx = (W + 7) / 8, ty = (H + rows - 1) / rows;
    const float3 o = make_float3(cam.v[0], cam.v[1], cam.v[2]);
    while (true) {
        unsigned w = 0;
        if (lane == 0) w = atomicAdd(work, 1u);
        w = __shfl_sync(WT_FULL, w, 0);
        if (w >= (unsigned)tx * (unsigned)ty) return;
        const int x = (int)(w % (unsigned)tx) * 8 + (lane & 7), y = (int)(w / (unsigned)tx) * rows + (lane >> 3);
        const bool live = x < W && y < H && (lane >> 3) < rows;
        const float3 d = pixel_dir(cam.v, W, H, fov, x, y);
        const size_t pix = (size_t)y * W + x;
        float T = 1.f;
        sm.lower[lane] = 0ull;
        bool more = live;
        for (bool first = true; __any_sync(WT_FULL, more); first = false) {
            bool full;
            const int lg0 = first ? 0 : (int)(65536.f * __log2f(fmaxf(T, 1e-30f)));
            if (!warp_collect<true, true>(sc, o, d, -1, more, eps, lg0, sm, list, full)) atomicAdd(&flags[FLAG_STACK], 1);
            const unsigned rays = __ballot_sync(WT_FULL, more), fulls = __ballot_sync(WT_FULL, full);
            more = false;
            for (unsigned m = rays; m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                int n = sm.cnt[q];
                const bool cut = (fulls >> q) & 1u;
                const float3 dq = f3(sm.rd[q]);
                float Tq = __shfl_sync(WT_FULL, T, q);
                unsigned long long last = 0ull;
                int kept = 0;
                if (n > 0) kept = warp_composite_any(sc, n, list + q * WT_LIST, sm, cut, true, Tq, last);
                __syncwarp();
                if (lane == q) {
                    T = Tq;
                    more = cut && Tq >= RGS_T_EPS;
                    sm.lower[q] = last;
                }
                const size_t px = __shfl_sync(WT_FULL, pix, q);
                if constexpr (ADJ) scatter_pixel<NC>(list + q * WT_LIST, kept, dq, C, in + px * C, out);
                else shade_pixel<NC>(list + q * WT_LIST, kept, dq, C, in, out + px * C, first);
                __syncwarp();
            }
        }
    }
}

struct RenderScratch {
    cudaStream_t st;
    float *X = nullptr;
    int *flag = nullptr;
    ~RenderScratch() {
        pool_release(flag, st);
        pool_release(X, st);
    }
};

rgs_status check_args(const rgs_transport *t, const float *in, const float *cam, int W, int H, float fov,
                      const float *out, const char *what) {
    if (!t || !in || !cam || !out) {
        rgs_set_error("%s: NULL argument", what);
        return RGS_ERR_ARG;
    }
    if (t->kind == RGS_KIND_NONE) {
        rgs_set_error("%s: the transport has not been traced", what);
        return RGS_ERR_STATE;
    }
    if (W <= 0 || H <= 0 || (long long)W * H > (1ll << 26) || !(fov > 0.f && fov < 3.14159f)) {
        rgs_set_error("%s: image %d x %d or field of view %g out of range", what, W, H, (double)fov);
        return RGS_ERR_ARG;
    }
    for (int q = 0; q < 9; ++q)
        if (!isfinite(cam[q])) {
            rgs_set_error("%s: non-finite camera", what);
            return RGS_ERR_NONFINITE;
        }
    return RGS_OK;
}

// Rows of a warp's tile. A warp lasts as long as its slowest pixels (grazing rays meet hundreds
// of surfels, some take several passes), so an image with few tiles for the 4,256 warps in
// flight is traced 8 or 16 pixels to a warp: less is shared, but the last warp ends sooner.
// 200,000 pixels: 4 rows 0.8 to 4.2 ms, 2 rows 0.6 to 2.2, 1 row 0.5 to 1.4 (thread per pixel
// before: 1.7 to 4.7); 532,000: 1.3 to 3.5, 1.3 to 2.2, 1.6 to 1.9; 2,074,000: 3.3, 3.3, 4.3.
int tile_rows(int W, int H) {
    const long long px = (long long)W * H;
    return px < 500000 ? 1 : (px < 1200000 ? 2 : 4);
}

// the tiles' launch, and the check that no traversal stack overflowed
template <int NC, bool ADJ>
rgs_status run_tiles(rgs_transport *t, const float *in, const float *cam, int W, int H, float fov, float *out,
                     RenderScratch &s) {
    rgs_status r;
    if ((r = pool_alloc(&s.flag, (size_t)FLAG_COUNT, s.st)) != RGS_OK) return r;
    RGS_CUDA(cudaMemsetAsync(s.flag, 0, sizeof(int) * FLAG_COUNT, s.st));
    Cam c;
    for (int q = 0; q < 9; ++q) c.v[q] = cam[q];
    WarpLists warps{s.st};
    const int rows = tile_rows(W, H);
    const long long tiles = (long long)((W + 7) / 8) * ((H + rows - 1) / rows);
    if ((r = warps.get((const void *)k_render<NC, ADJ>, RN_THREADS, tiles, t->budget_room(4 * (long long)t->arr()))) != RGS_OK) return r;
    RGS_CUDA(cudaMemsetAsync(warps.work, 0, sizeof(unsigned), s.st));
    {
        ProfScope ps_(ADJ ? "k_render_adj" : "k_render", s.st);
        k_render<NC, ADJ><<<warps.blocks, RN_THREADS, 0, s.st>>>(t->sc->dev(), c, W, H, rows, fov, t->C, in, out, warps.work,
                                                                warps.lists, s.flag);
    }
    RGS_LAUNCH("render");
    return RGS_OK;
}

rgs_status check_stack(RenderScratch &s) {
    int stack_overflows = 0;
    RGS_CUDA(cudaMemcpyAsync(&stack_overflows, s.flag + FLAG_STACK, sizeof(int), cudaMemcpyDeviceToHost, s.st));
    RGS_CUDA(cudaStreamSynchronize(s.st));
    if (stack_overflows) {
        rgs_set_error("render: BVH traversal stack overflow on %d pixel rays", stack_overflows);
        return RGS_ERR_CAPACITY;
    }
    return RGS_OK;
}

template <int NC>
rgs_status render_nc(rgs_transport *t, const float *B, const float *cam, int W, int H, float fov, float *img,
                     cudaStream_t st) {
    rgs_status r;
    RenderScratch s{st};
    const size_t A = (size_t)t->n * t->C * NC;
    if ((r = pool_alloc(&s.X, A, st)) != RGS_OK) return r;
    {
        ProfScope ps_("k_render_from_user", st);
        k_render_from_user<NC><<<(unsigned)((A + 255) / 256), 256, 0, st>>>(t->n, t->C, t->sc->uid, B, s.X);
    }
    RGS_LAUNCH("render from user");
    if ((r = run_tiles<NC, false>(t, s.X, cam, W, H, fov, img, s)) != RGS_OK) return r;
    return check_stack(s);
}

template <int NC>
rgs_status render_adjoint_nc(rgs_transport *t, const float *dimg, const float *cam, int W, int H, float fov,
                             float *dB, cudaStream_t st) {
    rgs_status r;
    RenderScratch s{st};
    const size_t A = (size_t)t->n * t->C * NC;
    if ((r = pool_alloc(&s.X, A, st)) != RGS_OK) return r;
    RGS_CUDA(cudaMemsetAsync(s.X, 0, sizeof(float) * A, st));
    if ((r = run_tiles<NC, true>(t, dimg, cam, W, H, fov, s.X, s)) != RGS_OK) return r;
    {
        ProfScope ps_("k_render_to_user", st);
        k_render_to_user<NC><<<(unsigned)((A + 255) / 256), 256, 0, st>>>(t->n, t->C, t->sc->uid, s.X, dB);
    }
    RGS_LAUNCH("render to user");
    return check_stack(s);
}

} // namespace

extern "C" rgs_status rgs_render(rgs_transport *t, const float *B, const float *cam, int32_t W, int32_t H, float fov,
                                 float *img, void *stream) {
    rgs_status r = check_args(t, B, cam, W, H, fov, img, "rgs_render");
    if (r != RGS_OK) return r;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    switch (t->nc) {
    case 1: return render_nc<1>(t, B, cam, W, H, fov, img, st);
    case 4: return render_nc<4>(t, B, cam, W, H, fov, img, st);
    case 9: return render_nc<9>(t, B, cam, W, H, fov, img, st);
    default: return render_nc<16>(t, B, cam, W, H, fov, img, st);
    }
}

extern "C" rgs_status rgs_render_adjoint(rgs_transport *t, const float *dL_dimg, const float *cam, int32_t W,
                                         int32_t H, float fov, float *dL_dB, void *stream) {
    rgs_status r = check_args(t, dL_dimg, cam, W, H, fov, dL_dB, "rgs_render_adjoint");
    if (r != RGS_OK) return r;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    switch (t->nc) {
    case 1: return render_adjoint_nc<1>(t, dL_dimg, cam, W, H, fov, dL_dB, st);
    case 4: return render_adjoint_nc<4>(t, dL_dimg, cam, W, H, fov, dL_dB, st);
    case 9: return render_adjoint_nc<9>(t, dL_dimg, cam, W, H, fov, dL_dB, st);
    default: return render_adjoint_nc<16>(t, dL_dimg, cam, W, H, fov, dL_dB, st);
    }
}
