// Bounce gather/projection for one receiver and one column tile (the body of k_bounce and
// of the persistent batch kernel): CTA-wide, up to BOUNCE_THREADS threads, red = shared scratch
// of (BOUNCE_THREADS/32) * G * KPL * CT floats.
#pragma once
#include "rgs_internal.cuh"

#define BOUNCE_THREADS 256

// many-column (lane-per-column) layout: a warp takes one ray at a time and its 32 lanes take
// 32 consecutive columns of one tile
constexpr int MC_WARPS = 8;
constexpr int MC_THREADS = MC_WARPS * 32;
static_assert(MC_THREADS == BOUNCE_THREADS, "the batch kernel runs both bodies in one block");
static_assert(BOUNCE_THREADS == 256, "RGS_BOUNCE_LB and RGS_MC_LB assume 256 threads");

// the NC coefficients of one column of a row (FP32 rows of NC floats, BF16 rows padded)
template <int NC> __device__ __forceinline__ void load_col(const float *__restrict__ p, float *v) {
    if constexpr (NC % 4 == 0) {
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) {
            const float4 f = __ldg(reinterpret_cast<const float4 *>(p) + q);
            v[4 * q] = f.x;
            v[4 * q + 1] = f.y;
            v[4 * q + 2] = f.z;
            v[4 * q + 3] = f.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = __ldg(p + k);
    }
}
// (BF16 rows of 9 or 16 coefficients are padded to 32 bytes: one request a lane.  As two
// 16-byte requests at a 32-byte stride a warp's kilobyte took the L1 twice the wavefronts.)
template <int NC> __device__ __forceinline__ void load_col(const __nv_bfloat16 *__restrict__ p, float *v) {
    if constexpr (NC >= 9) {
        float4 a, b;
        ld_rec32(p, a, b);
        const float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const unsigned u = __float_as_uint(f[m]);
            if (2 * m < NC) v[2 * m] = __uint_as_float(u << 16);
            if (2 * m + 1 < NC) v[2 * m + 1] = __uint_as_float(u & 0xffff0000u);
        }
    } else {
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = __bfloat162float(p[k]);
    }
}
template <int NC, class T> constexpr int row_stride() {
    return sizeof(T) == 2 ? ((NC >= 9) ? 16 : NC) : NC;
}

// Dot products of Y with the 32 columns of one FP32 source row tile (nc = 16: 64 B per
// column, 2 KB per tile), read as two contiguous 1-KB warp requests, a lane taking 32 B (half
// of one column).  Each lane forms its partial dot products with its half of Y, and one
// exchange between the 2 lanes holding each column leaves lane l with the whole dot product
// of tile column own(l).  A 64-B column row per lane at a 64-B stride costs the L1 about
// twice the wavefronts for the same bytes.
// Columns past the tile's `ncols` live ones read the last live column (their results are
// not used).  All 32 lanes take part (the shuffles use the full mask).
template <class T, int NC> struct TileDot;

template <int NC> struct TileDot<float, NC> {
    static_assert(NC == 16, "FP32 tiles of 16 coefficients per column");
    static constexpr int KPL = 8;
    __device__ static int own(int lane) { return 16 * (lane & 1) + (lane >> 1); }
    __device__ static void pick(const float *Y, int lane, float (&y)[KPL]) {
#pragma unroll
        for (int m = 0; m < KPL; ++m) y[m] = lane & 1 ? Y[8 + m] : Y[m];
    }
    // tile: the tile's first column in source row j; ncols: its live columns (1..32)
    __device__ static float dot(const float *__restrict__ tile, int ncols, int lane, const float (&y)[KPL]) {
        const int g = lane & 1, a = lane >> 1;
        float p[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int c = min(16 * q + a, ncols - 1);
            float4 f, h;
            ld_rec32(tile + c * 16 + 8 * g, f, h);
            p[q] = y[0] * f.x + y[1] * f.y + y[2] * f.z + y[3] * f.w;
            p[q] += y[4] * h.x + y[5] * h.y + y[6] * h.z + y[7] * h.w;
        }
        const float r = __shfl_xor_sync(0xffffffffu, g ? p[0] : p[1], 1);
        return (g ? p[1] : p[0]) + r;
    }
};

template <int NC, int CT, class SL>
__device__ __forceinline__ void bounce_epilogue(const SceneDev &sc, int C, const float (&acc)[SL::KPL][CT], float w,
                                                const float *__restrict__ Bprev, const float *__restrict__ S,
                                                float *__restrict__ Qout, float *__restrict__ Bout,
                                                __nv_bfloat16 *__restrict__ Bout16, double *norm2, int i, int col0,
                                                float *red);

template <int NC, int CT, class SL>
__device__ __forceinline__ void bounce_receiver(const SceneDev &sc, const RaysDev &rays, int C,
                                                const typename SL::T *__restrict__ Bg, const float *__restrict__ Bprev,
                                                const float *__restrict__ S, float *__restrict__ Qout,
                                                float *__restrict__ Bout, __nv_bfloat16 *__restrict__ Bout16,
                                                double *norm2, int i, int col0, float *red) {

    constexpr int G = SL::G, KPL = SL::KPL, RS = SL::STRIDE;
    const int nd = rays.nd, groups = blockDim.x / G;
    const int grp = threadIdx.x / G, g = threadIdx.x % G;
    const float3 n = f3(sc.N4[i]);
    float acc[KPL][CT];
#pragma unroll
    for (int m = 0; m < KPL; ++m)
#pragma unroll
        for (int c = 0; c < CT; ++c) acc[m][c] = 0.f;

    for (int q = grp; q < nd; q += groups) {
        const long long r = (long long)i * nd + q;
        const float3 d = f3(rays.dir[r]);
        float yo[KPL], yi[KPL];
        {
            float Y[NC];
            sh_eval<NC>(neg3(d), Y);
            SL::pick(Y, g, yo);
            sh_eval<NC>(reflect_n(n, d), Y);
            SL::pick(Y, g, yi);
        }
        const int cnt = rays.cnt[r];
        const long long base = rays.off[r];
        float x[CT];
#pragma unroll
        for (int c = 0; c < CT; ++c) x[c] = 0.f;
#pragma unroll (NC == 16 ? 3 : 4)
        for (int h = 0; h < cnt; ++h) {
            const int2 ja = __ldg(&rays.rec_ja[base + h]);
            const float a = __int_as_float(ja.y);
            const typename SL::T *Bj = Bg + ((size_t)ja.x * C + col0) * RS;
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                float v[KPL];
                SL::load(Bj + c * RS, g, v);
                float s = 0.f;
#pragma unroll
                for (int m = 0; m < KPL; ++m) s += yo[m] * v[m];
                x[c] += a * s;
            }
        }
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            const float xc = SL::group_sum(x[c]);
#pragma unroll
            for (int m = 0; m < KPL; ++m) acc[m][c] += yi[m] * xc;
        }
    }
    bounce_epilogue<NC, CT, SL>(sc, C, acc, 3.14159265358979f / (float)nd, Bprev, S, Qout, Bout, Bout16, norm2, i, col0,
                                red);
}

// Reduction of the per-thread projections acc over the CTA and the bounce update of one
// (receiver, column tile): Q = w * sum, B = S + o_i c_i (x) Q, its BF16 copy, and the FP64
// partial of ||B - Bprev||^2.  Ends with __syncthreads (red is reused).
template <int NC, int CT, class SL>
__device__ __forceinline__ void bounce_epilogue(const SceneDev &sc, int C, const float (&acc)[SL::KPL][CT], float w,
                                                const float *__restrict__ Bprev, const float *__restrict__ S,
                                                float *__restrict__ Qout, float *__restrict__ Bout,
                                                __nv_bfloat16 *__restrict__ Bout16, double *norm2, int i, int col0,
                                                float *red) {
    constexpr int G = SL::G, KPL = SL::KPL;
    // reduce over the groups: lanes with equal g within the warp, then across warps
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 0; m < KPL; ++m)
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            float v = acc[m][c];
#pragma unroll
            for (int off = G; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane < G) red[(warp * G + lane) * (KPL * CT) + m * CT + c] = v;
        }
    __syncthreads();
    double dsq = 0.0;
    for (int e = threadIdx.x; e < NC * CT; e += blockDim.x) {
        const int k = e / CT, c = e - k * CT;
        int gg = 0, mm = 0;
#pragma unroll
        for (int g2 = 0; g2 < G; ++g2)
#pragma unroll
            for (int m2 = 0; m2 < KPL; ++m2)
                if (SL::k(g2, m2) == k) {
                    gg = g2;
                    mm = m2;
                }
        float v = 0.f;
        for (int q = 0; q < blockDim.x / 32; ++q) v += red[(q * G + gg) * (KPL * CT) + mm * CT + c];
        const int col = col0 + c;
        const float Q = w * v;
        const size_t idx = ((size_t)i * C + col) * NC + k;
        Qout[idx] = Q;
        const float oc = alpha_center(sc, i) * sc.cl[(size_t)i * 12 + band_of(k) * 3 + (col % 3)];
        const float b = S[idx] + oc * Q;
        Bout[idx] = b;
        if (Bout16) Bout16[((size_t)i * C + col) * bf16_stride<NC>() + k] = __float2bfloat16_rn(b);
        const double df = (double)b - (double)Bprev[idx];
        dsq += df * df;
    }
    // FP64 residual norm: warp reduce, one atomic per warp with work
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dsq += __shfl_xor_sync(0xffffffffu, dsq, off);
    if (lane == 0 && warp * 32 < NC * CT) atomicAdd(norm2, dsq);
    __syncthreads(); // red is reused by the caller's next receiver
}

// Lane-per-column bounce for one receiver and one 32-column tile (the body of k_bounce_mc and
// of the persistent batch kernel's wide items); red = shared scratch of MC_WARPS * NC * 32 floats.
template <int NC, class T, bool HALF>
__device__ __forceinline__ void bounce_receiver_mc(const SceneDev &sc, const RaysDev &rays, int C,
                                                   const T *__restrict__ Bg, const float *__restrict__ Bprev,
                                                   const float *__restrict__ S, float *__restrict__ Qout,
                                                   float *__restrict__ Bout, __nv_bfloat16 *__restrict__ Bout16,
                                                   double *norm2, int i, int tile, float *red) {
    constexpr int RS = row_stride<NC, T>();
    constexpr bool COOP = sizeof(T) == 4 && NC == 16 && !HALF; // whole-tile reads (TileDot)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int own = HALF ? lane & 15 : lane; // the tile column whose sums this lane keeps
    if constexpr (COOP) own = TileDot<T, NC>::own(lane);
    const int col = tile * 32 + own;
    const bool live = col < C;
    const int colc = live ? col : C - 1;
    const int ncols = min(32, C - tile * 32);
    const int nd = rays.nd;
    const float3 n = f3(sc.N4[i]);
    float acc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) acc[k] = 0.f;
    for (int rq = warp; rq < nd; rq += MC_WARPS) {
        const long long r = (long long)i * nd + rq;
        const float3 d = f3(rays.dir[r]);
        float Yo[NC];
        sh_eval<NC>(neg3(d), Yo);
        const int cnt = rays.cnt[r];
        const long long base = rays.off[r];
        float x = 0.f;
        [[maybe_unused]] float ys[8]; // this lane's half of Y(-d) (TileDot)
        if constexpr (COOP) TileDot<T, NC>::pick(Yo, lane, ys);
        for (int h0 = 0; h0 < cnt; h0 += 32) { // the lanes hold 32 records; four rows are requested together
            const int m = min(32, cnt - h0);
            const int2 rec = lane < m ? __ldg(&rays.rec_ja[base + h0 + lane]) : make_int2(0, 0);
#pragma unroll 4
            for (int q = 0; q < m; q += HALF ? 2 : 1) { // HALF: the upper 16 lanes take the next hit
                const int h = HALF ? q + (lane >> 4) : q, hc = HALF ? min(h, m - 1) : h;
                const int j = __shfl_sync(0xffffffffu, rec.x, hc);
                const float a = __int_as_float(__shfl_sync(0xffffffffu, rec.y, hc));
                if constexpr (COOP) {
                    x += a * TileDot<T, NC>::dot(Bg + ((size_t)j * C + tile * 32) * RS, ncols, lane, ys);
                } else {
                    float v[NC];
                    load_col<NC>(Bg + ((size_t)j * C + colc) * RS, v);
                    float s = 0.f;
#pragma unroll
                    for (int k = 0; k < NC; ++k) s += Yo[k] * v[k];
                    if (!HALF || h < m) x += a * s; // (no weight of 0: the row may hold an infinity)
                }
            }
        }
        if constexpr (HALF) x += __shfl_xor_sync(0xffffffffu, x, 16);
        float Yi[NC];
        sh_eval<NC>(reflect_n(n, d), Yi);
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[k] += Yi[k] * x;
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) red[(warp * NC + k) * 32 + own] = acc[k]; // (HALF: both halves the same)
    __syncthreads();
    double dsq = 0.0;
    const float w = 3.14159265358979f / (float)nd;
    for (int e = threadIdx.x; e < NC * 32; e += MC_THREADS) {
        const int k = e >> 5, c = e & 31;
        const int cc = tile * 32 + c;
        if (cc >= C) continue;
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < MC_WARPS; ++q) v += red[(q * NC + k) * 32 + c];
        const float Q = w * v;
        const size_t idx = ((size_t)i * C + cc) * NC + k;
        Qout[idx] = Q;
        const float b = S[idx] + alpha_center(sc, i) * sc.cl[(size_t)i * 12 + band_of(k) * 3 + (cc % 3)] * Q;
        Bout[idx] = b;
        if (Bout16) Bout16[((size_t)i * C + cc) * ((NC >= 9) ? 16 : NC) + k] = __float2bfloat16_rn(b);
        const double df = (double)b - (double)Bprev[idx];
        dsq += df * df;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dsq += __shfl_xor_sync(0xffffffffu, dsq, off);
    if (lane == 0) atomicAdd(norm2, dsq);
    __syncthreads(); // red is reused by the caller's next receiver
}
// the same, a tile of up to 16 columns taken two hits at a time
template <int NC, class T>
__device__ __forceinline__ void bounce_receiver_mc(const SceneDev &sc, const RaysDev &rays, int C,
                                                   const T *__restrict__ Bg, const float *__restrict__ Bprev,
                                                   const float *__restrict__ S, float *__restrict__ Qout,
                                                   float *__restrict__ Bout, __nv_bfloat16 *__restrict__ Bout16,
                                                   double *norm2, int i, int tile, float *red) {
    if (half_tile(NC, C - tile * 32, sizeof(T) == 2))
        bounce_receiver_mc<NC, T, true>(sc, rays, C, Bg, Bprev, S, Qout, Bout, Bout16, norm2, i, tile, red);
    else
        bounce_receiver_mc<NC, T, false>(sc, rays, C, Bg, Bprev, S, Qout, Bout, Bout16, norm2, i, tile, red);
}
