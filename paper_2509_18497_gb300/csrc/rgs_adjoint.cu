// Adjoint (rgs_adjoint): exact gradients of L(B^(n)) for the truncated bounce series.
//
//   v^(0) = dL/dB^(n),  v^(a) = K^T v^(a-1)   (Eq. final_dL_dE: the same paths with the
//                                              decay reversed, propagating gradients)
//   u = sum_a v^(a) = dL/dS,   P_i[l][ch] = sum_{k in l, light} (sum_{a<n} v^(a) Q^(n-1-a) + u Dgeo)
//
// K^T v is a gather over the records grouped by source surfel j:
//   (K^T v)_j[c][k] = sum_{hits e on j} a_e Y_k(-d_e) y_e[c],
//   y_e[c] = (pi/nd) o_i sum_k' c_{i,l(k'),ch} Y_k'(R_i d_e) v_i[c][k']      (i = receiver of e)
// k_adj_ray forms y per ray once (one record with the ray's direction) and k_adj_src gathers
// (d, y) per entry, 32 bytes, instead of a 192-byte row of v_i per entry (k_adj_src_tile: 12
// columns, 64 bytes).  With it go the hits' opacity sums g_e = sum_a y_e^(a) . (Y(-d_e) B_j^(n-1-a));
// k_opacity_g forms them ray by ray where the index comes in parts.
// k_opacity_rec and k_shadow_bwd run the compositing backward of every
// hemisphere and shadow ray (dL/dalpha_h = T_h (g_h - R_h), dL/dT = -prod of the other (1 - alpha)).
#include <algorithm>
#include <vector>

#include "rgs_warp_trace.cuh"

namespace {

constexpr int SHADOW_THREADS = 128;
constexpr int ADJ_THREADS = 128;
static_assert(ADJ_THREADS == 128, "RGS_ADJ_LB assumes 128 threads");

// user [N][nc][C] -> internal [N][C][NC]
template <int NC>
__global__ void k_from_user(int n, int C, const int *__restrict__ uid, const float *__restrict__ X, float *Y) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n * C * NC) return;
    const int k = (int)(idx % NC);
    const size_t ic = idx / NC;
    const int c = (int)(ic % C);
    const int i = (int)(ic / C);
    Y[idx] = X[((size_t)uid[i] * NC + k) * C + c];
}

// Sums over a surfel's columns of one channel, by a warp: lane o holds value o = ch NC + k of
// three consecutive columns (and o + 32), so that every step of three columns reads one
// contiguous row piece and each sum is formed in column order by one lane.  A thread per
// surfel walked its row alone: with 1,536 columns 3.5 ms per launch on 3,000 surfels.
constexpr int ROW_WARPS = 4;
template <int NC, class F> __device__ __forceinline__ void column_sums(int C, float (&acc)[2], F &&value) {
    constexpr int W = 3 * NC;
    const int lane = threadIdx.x & 31;
    acc[0] = acc[1] = 0.f;
#pragma unroll 4
    for (int q = 0; q < C / 3; ++q) {
        if (lane < W) acc[0] += value(q * W + lane);
        if (lane + 32 < W) acc[1] += value(q * W + lane + 32);
    }
}

// P_i[l][ch] += sum_{c, k in l} X[i][c][k] * Y[i][c][k]   (a warp per surfel)
template <int NC>
__global__ void __launch_bounds__(32 * ROW_WARPS) k_pair_accum(int n, int C, const float *__restrict__ X,
                                                              const float *__restrict__ Y, float *P) {
    __shared__ float part[ROW_WARPS][64];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, i = blockIdx.x * ROW_WARPS + w;
    if (i >= n) return;
    const size_t row = (size_t)i * C * NC;
    float acc[2];
    column_sums<NC>(C, acc, [&](int e) { return __ldg(&X[row + e]) * __ldg(&Y[row + e]); });
    part[w][lane] = acc[0];
    part[w][lane + 32] = acc[1];
    __syncwarp();
    if (lane < 12) {
        const int l = lane / 3, ch = lane - 3 * l;
        float s = 0.f;
        for (int k = l * l; k < (l + 1) * (l + 1) && k < NC; ++k) s += part[w][ch * NC + k];
        P[(size_t)i * 12 + lane] += s;
    }
}

// Per ray r of receiver i, for a tile of CT columns:
//   y_r[c] = (pi/nd) o_i sum_k' c_{i,l(k'),ch} Y_k'(R_i d_r) v_i[c][k']
// in one record with the ray's direction for the by-source gather: 8 floats (d, 0, y[0..2], 0)
// for 3 columns, 16 (d, 0, y[0..11]) for 12 (columns past C are zero).  With d and y in arrays of
// their own each entry touched two cache lines, and at 3 columns a tile 48 columns took 16
// passes: the gather held the L1 data pipe at 80 % of peak with lookups.  60,000 surfels, 128
// rays, 48 columns, four bounces: the gather 71 -> 28.5 ms.
template <int CT> constexpr int adj_rec() { return CT == 3 ? 8 : 16; }
template <int NC, int CT>
__global__ void __launch_bounds__(256) k_adj_ray(SceneDev sc, RaysDev rays, int C, int col0,
                                                 const float *__restrict__ vin, float *__restrict__ rec) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= sc.n * rays.nd) return;
    const int i = r / rays.nd;
    const float3 n = f3(sc.N4[i]);
    const float3 d = f3(rays.dir[r]);
    float Yi[NC], cy[NC]; // cy: c_{i,l(k),ch} Y_k of one channel
    sh_eval<NC>(reflect_n(n, d), Yi);
    const float oi = alpha_center(sc, i) * (3.14159265358979f / (float)rays.nd);
    const float *vi = vin + ((size_t)i * C + col0) * NC;
    float y[CT];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
#pragma unroll
        for (int k = 0; k < NC; ++k) cy[k] = __ldg(&sc.cl[(size_t)i * 12 + band_of(k) * 3 + ch]) * Yi[k];
#pragma unroll
        for (int c = ch; c < CT; c += 3) { // (col0 is a multiple of 3)
            float s = 0.f;
            if (CT == 3 || col0 + c < C) {
#pragma unroll
                for (int k = 0; k < NC; ++k) s += cy[k] * __ldg(&vi[c * NC + k]);
            }
            y[c] = oi * s;
        }
    }
    float4 *out = reinterpret_cast<float4 *>(rec + (size_t)r * adj_rec<CT>());
    out[0] = make_float4(d.x, d.y, d.z, 0.f);
#pragma unroll
    for (int q = 0; q < adj_rec<CT>() / 4 - 1; ++q)
        out[q + 1] = make_float4(y[(4 * q) % CT], y[(4 * q + 1) % CT], y[(4 * q + 2) % CT],
                                 4 * q + 3 < CT ? y[(4 * q + 3) % CT] : 0.f);
}

// (K^T v)_j[c][k] = sum_{entries e on j} a_e Y_k(-d_e) y_e[c]; one CTA per source j.
// 3 columns: a thread per entry.
// OPA: the opacity backward's per-hit sums as well, which need the same two things of an entry,
//   g_e (+)= sum_c y_e[c] Y(-d_e) . B_j[c],
// B the iterate paired with v.  By source its row is read once per CTA; the ray-wise gather
// reads a row per hit, at the ~10 TB/s the L2 gives (192 bytes a hit and iterate for 3 FP32
// columns, 1.5 KB for 48 BF16 ones).  Both passes, 20,000 surfels, 128 rays, 16 coefficients,
// three pairings: 3 columns 4.2 -> 1.7 ms, 12 columns 15.3 -> 4.4; 60,000 surfels, 48 BF16
// columns, four pairings: 104 -> 56 ms.
struct AdjOpa {
    const float *Bf;         // B^(b), FP32 rows
    const __nv_bfloat16 *Bh; // its BF16 rows (the batched modes), or NULL
    float *gt;               // per entry of the index
    bool first;              // write instead of add
};
template <int NC> __device__ __forceinline__ float adj_opa_row(const AdjOpa &o, size_t jc, int k) {
    return o.Bh ? __bfloat162float(o.Bh[jc * bf16_stride<NC>() + k]) : __ldg(&o.Bf[jc * NC + k]);
}
template <int NC, bool OPA>
__global__ void RGS_ADJ_LB k_adj_src(int C, int col0, const long long *__restrict__ src_off,
                                                        const int2 *__restrict__ tr, const float *__restrict__ rec,
                                                        float *__restrict__ vout, float *__restrict__ u, int j0,
                                                        long long ebase, AdjOpa opa) {
    constexpr int CT = 3, RS = adj_rec<CT>();
    const int j = j0 + blockIdx.x; // sources j0 .. of this index part; its entries start at ebase
    constexpr int NQ = (NC + 3) / 4;
    __shared__ float4 Bj[OPA ? CT * NQ : 1];
    if constexpr (OPA) {
        if (threadIdx.x < CT * NQ * 4) {
            const int c = threadIdx.x / (NQ * 4), k = threadIdx.x % (NQ * 4);
            reinterpret_cast<float *>(Bj)[threadIdx.x] = k < NC ? adj_opa_row<NC>(opa, (size_t)j * C + col0 + c, k) : 0.f;
        }
        __syncthreads();
    }
    float acc[NC][CT];
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int c = 0; c < CT; ++c) acc[k][c] = 0.f;
    const long long e0 = src_off[j] - ebase, e1 = src_off[j + 1] - ebase;
    // the next entry's record and sum are requested before this one is worked on, the entry
    // after it before that
    auto entry = [&](long long e) { return e < e1 ? __ldg(&tr[e]) : make_int2(0, 0); };
    long long e = e0 + threadIdx.x;
    int2 ent = entry(e), ent1 = entry(e + ADJ_THREADS);
    float4 d4 = make_float4(0.f, 0.f, 0.f, 0.f), y4 = d4;
    float old = 0.f, old1 = 0.f;
    if (e < e1) {
        ld_rec32(rec + (size_t)ent.x * RS, d4, y4);
        if (OPA && !opa.first) old = opa.gt[e];
    }
    for (; e < e1; e += ADJ_THREADS) {
        const float a = __int_as_float(ent.y);
        const long long en = e + ADJ_THREADS;
        float4 d41 = d4, y41 = y4;
        if (en < e1) {
            ld_rec32(rec + (size_t)ent1.x * RS, d41, y41);
            if (OPA && !opa.first) old1 = opa.gt[en];
        }
        const int2 ent2 = entry(en + ADJ_THREADS);
        float Yo[NC];
        sh_eval<NC>(make_float3(-d4.x, -d4.y, -d4.z), Yo);
        if constexpr (OPA) {
            const float yc[3] = {y4.x, y4.y, y4.z};
            float g = old;
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                float t = 0.f;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 b = Bj[c * NQ + q];
                    const float bk[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (4 * q + k < NC) t += Yo[4 * q + k < NC ? 4 * q + k : 0] * bk[k];
                }
                g += yc[c] * t;
            }
            opa.gt[e] = g;
        }
        const float y[3] = {a * y4.x, a * y4.y, a * y4.z};
#pragma unroll
        for (int k = 0; k < NC; ++k)
#pragma unroll
            for (int c = 0; c < CT; ++c) acc[k][c] += Yo[k] * y[c];
        ent = ent1;
        ent1 = ent2;
        d4 = d41;
        y4 = y41;
        old = old1;
    }
    __shared__ float red[ADJ_THREADS / 32][NC * CT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            float v = acc[k][c];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0) red[warp][k * CT + c] = v;
        }
    __syncthreads();
    for (int e = threadIdx.x; e < NC * CT; e += ADJ_THREADS) {
        float v = 0.f;
        for (int q = 0; q < ADJ_THREADS / 32; ++q) v += red[q][e];
        const int k = e / CT, c = e - k * CT;
        const size_t idx = ((size_t)j * C + col0 + c) * NC + k;
        vout[idx] = v;
        u[idx] += v;
    }
}

// 12 columns: the entries' records are copied into shared memory 128 at a time (asynchronously,
// the next batch while this one is used: their latency, not the arithmetic, is what bounds
// the gather), a thread evaluates the SH of one entry, and G lanes per entry, each CL
// columns, multiply: 48 FMAs (two coefficients to an instruction), 96 with the opacity sums
// (OPA), whose partial results are copied ahead with the records (read where they are
// added to, the pass took a third longer).  A lane takes whole columns, so that the pairs of
// Y come from shared memory as they are; with a quarter of the coefficients of all 12 each, the
// duplicated factors were a fifth of the instructions (66 -> 56 ms for the 16 launches of four
// bounces on 60,000 surfels, 128 rays, 48 columns, opacity sums included).
constexpr int ADJ_STRIDE = 20; // floats of a record in shared memory (16-byte rows without conflicts)
template <int NC> struct AdjLanes {
    static constexpr int G = NC >= 9 ? 4 : 1, CL = 12 / G; // lanes per entry, columns per lane
};
template <int NC> struct AdjTile {
    __align__(16) float rec[2][ADJ_THREADS][ADJ_STRIDE];
    __align__(16) float Y[ADJ_THREADS][ADJ_STRIDE]; // Y(-d)
    float a[2][ADJ_THREADS], g[2][ADJ_THREADS]; // weights; opacity sums so far
};
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
template <int NC, bool OPA>
__global__ void __launch_bounds__(ADJ_THREADS, OPA ? 4 : 6) k_adj_src_tile(int C, int col0, const long long *__restrict__ src_off,
                                                               const int2 *__restrict__ tr, const float *__restrict__ rec,
                                                               float *__restrict__ vout, float *__restrict__ u, int j0,
                                                               long long ebase, AdjOpa opa) {
    constexpr int CT = 12, RS = adj_rec<CT>(), G = AdjLanes<NC>::G, CL = AdjLanes<NC>::CL;
    constexpr int NP = (NC + 1) / 2, NY = (NC + 3) / 4; // pairs of coefficients; 16-byte pieces of Y
    __shared__ AdjTile<NC> s;
    const int j = j0 + blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, g = tid % G;
    uint64_t acc[CL][NP];
#pragma unroll
    for (int c = 0; c < CL; ++c)
#pragma unroll
        for (int k = 0; k < NP; ++k) acc[c][k] = 0ull;
    uint64_t Bj[OPA ? CL : 1][OPA ? NP : 1]; // this lane's columns of the source's paired row
    if constexpr (OPA) {
        auto el = [&](int c, int k) {
            return c < C && k < NC ? adj_opa_row<NC>(opa, (size_t)j * C + c, k) : 0.f;
        };
#pragma unroll
        for (int c = 0; c < CL; ++c)
#pragma unroll
            for (int k = 0; k < NP; ++k) Bj[c][k] = pack2(el(col0 + CL * g + c, 2 * k), el(col0 + CL * g + c, 2 * k + 1));
    }
    const long long e0 = src_off[j] - ebase, e1 = src_off[j + 1] - ebase;
    const int batches = (int)((e1 - e0 + ADJ_THREADS - 1) / ADJ_THREADS);
    auto entry = [&](int b) { // this thread's entry of batch b (ray -1: none)
        const long long e = e0 + (long long)b * ADJ_THREADS + tid;
        return e < e1 ? __ldg(&tr[e]) : make_int2(-1, 0);
    };
    auto fetch = [&](int b, int2 ent) { // batch b: four lanes copy a record
        const int st = b & 1;
        s.a[st][tid] = __int_as_float(ent.y);
        if (OPA && !opa.first && ent.x >= 0) cp_async4(&s.g[st][tid], opa.gt + e0 + (long long)b * ADJ_THREADS + tid);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int from = 8 * q + (lane >> 2), ray = __shfl_sync(0xffffffffu, ent.x, from);
            if (ray >= 0)
                cp_async16(&s.rec[st][(tid & ~31) + from][4 * (lane & 3)], rec + (size_t)ray * RS + 4 * (lane & 3));
        }
        asm volatile("cp.async.commit_group;");
    };
    int2 ent = entry(0);
    if (batches > 0) fetch(0, ent);
    ent = entry(1);
    for (int b = 0; b < batches; ++b) {
        const int st = b & 1;
        if (b + 1 < batches) {
            fetch(b + 1, ent);
            ent = entry(b + 2);
            asm volatile("cp.async.wait_group 1;");
        } else {
            asm volatile("cp.async.wait_group 0;");
        }
        __syncthreads();
        const int m = (int)min((long long)ADJ_THREADS, e1 - e0 - (long long)b * ADJ_THREADS);
        if (tid < m) {
            const float4 d = *reinterpret_cast<const float4 *>(s.rec[st][tid]);
            float Yo[NC];
            sh_eval<NC>(make_float3(-d.x, -d.y, -d.z), Yo);
#pragma unroll
            for (int k = 0; k < 4 * NY; ++k) s.Y[tid][k] = k < NC ? Yo[k < NC ? k : 0] : 0.f;
        }
        __syncthreads();
        const int rounds = (m + ADJ_THREADS / G - 1) / (ADJ_THREADS / G); // (all lanes: OPA sums over a group's)
#pragma unroll 1
        for (int q0 = 0; q0 < rounds; ++q0) {
            const int at = q0 * (ADJ_THREADS / G) + tid / G, x = min(at, m - 1);
            if (!OPA && at >= m) break;
            uint64_t Y[2 * NY];
            float y[CL];
#pragma unroll
            for (int q = 0; q < NY; ++q) {
                const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(&s.Y[x][4 * q]);
                Y[2 * q] = f.x;
                Y[2 * q + 1] = f.y;
            }
#pragma unroll
            for (int c = 0; c < CL; ++c) y[c] = s.rec[st][x][4 + CL * g + c];
            if constexpr (OPA) {
                float t = 0.f;
#pragma unroll
                for (int c = 0; c < CL; ++c) {
                    uint64_t two = 0ull;
#pragma unroll
                    for (int k = 0; k < NP; ++k) two = fma2(Y[k], Bj[c][k], two);
                    const float2 sc = unpack2(two);
                    t += y[c] * (sc.x + sc.y);
                }
#pragma unroll
                for (int off = 1; off < G; off <<= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
                if (g == 0 && at < m)
                    opa.gt[e0 + (long long)b * ADJ_THREADS + x] = opa.first ? t : s.g[st][x] + t;
                if (at >= m) break;
            }
            const float a = s.a[st][x];
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                const uint64_t ay = pack2(a * y[c], a * y[c]);
#pragma unroll
                for (int k = 0; k < NP; ++k) acc[c][k] = fma2(ay, Y[k], acc[c][k]);
            }
        }
        __syncthreads(); // the tables are rewritten
    }
    float *red = &s.rec[0][0][0]; // [warp][NC CT]
    constexpr int OUT = NC * CT;
    static_assert(ADJ_THREADS / 32 * OUT <= 2 * ADJ_THREADS * ADJ_STRIDE, "the sums fit the records' place");
#pragma unroll
    for (int c = 0; c < CL; ++c)
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const float2 two = unpack2(acc[c][k / 2]);
            float v = k & 1 ? two.y : two.x;
#pragma unroll
            for (int off = 16; off >= G; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane < G) red[(tid >> 5) * OUT + k * CT + CL * lane + c] = v;
        }
    __syncthreads();
    for (int e = tid; e < NC * CT; e += ADJ_THREADS) {
        const int c = e / NC, k = e - c * NC;
        if (col0 + c >= C) continue;
        float v = 0.f;
        for (int q = 0; q < ADJ_THREADS / 32; ++q) v += red[q * OUT + k * CT + c];
        const size_t idx = ((size_t)j * C + col0 + c) * NC + k;
        vout[idx] = v;
        u[idx] += v;
    }
}

// Shadow rays: dL/dT_L = q = sum_{k,ch} u_i[L,ch][k] o_i c_{i,l,ch} Y_k(R_i w) I cos/r^2,
// dT/dalpha_m = -prod_{m' != m} (1 - alpha_m'); also adds u (x) Dgeo to P.  With dp (and
// ds) the geometry gradients of the direct term as well (Eq. dl-dgeo-1 for the light's
// direction): with h_k = sum_ch u_i[L,ch][k] o_i c_{i,l(k),ch} I_ch and H = h . Y(R_i w), the
// term H (n_i.w) fall T moves with w (through Y(R_i w) and n_i.w), with fall = 1/r^2 and with
// each shadow occluder's crossing point; a directional light has a fixed w and fall = 1.
// gF (with dp): the frame gradients, through n_i (cos and R_i) and the occluders' frames.
// A warp per 32 or 16 (surfel, light) pairs (shadow_pairs), their shadow rays traced together twice
// (rgs_warp_trace.cuh):
// for the transmittances, then for the occluders' terms.
struct ShadowWarp {
    WarpOcclusion w;
    float q[32], T[32]; // dL/dT and the product of the factors that are not 0
    int nz[32];         // how many are 0
    float gp[32][3], gw[32][3];
};
template <int NC, bool GEO>
__global__ void __launch_bounds__(SHADOW_THREADS) k_shadow_bwd(SceneDev sc, int nl, int per, int ldir, const float *__restrict__ lpos, const float *__restrict__ lint,
                             int C, const float *__restrict__ u, float *P, float *dop, float *dp, float *ds, float *gF) {
    extern __shared__ __align__(16) unsigned char shadow_smem[];
    ShadowWarp &sm = reinterpret_cast<ShadowWarp *>(shadow_smem)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int tid = (blockIdx.x * (SHADOW_THREADS / 32) + (threadIdx.x >> 5)) * per + lane;
    const bool live = lane < per && tid < sc.n * nl;
    const int i = live ? tid / nl : 0, lt = live ? tid - i * nl : 0;
    const float4 Pi = sc.P[i];
    const float3 o = f3(Pi), n = f3(sc.N4[i]);
    float r, fall;
    const float3 w = light_dir(lpos, lt, o, ldir, r, fall);
    const float cs = dot3(n, w);
    const bool lit = live && cs > 0.f;
    const float eps = *sc.eps_plane;
    float Tnz;
    int nzero;
    warp_transmittance<false>(sc, sm.w, o, w, r, i, lit, eps, Tnz, nzero, [](int, const SurfelRec &, int) { return true; });
    float qv = 0.f, H = 0.f;
    const float T = nzero ? 0.f : Tnz;
    float3 gw = make_float3(0.f, 0.f, 0.f), gpi = make_float3(0.f, 0.f, 0.f);
    if (lit) {
        float Y[NC], h[NC];
        const float3 rw = reflect_n(n, w);
        sh_eval<NC>(rw, Y);
        const float pre = cs * fall;
        const float *ui = u + ((size_t)i * C + lt * 3) * NC;
        const float ai = alpha_center(sc, i);
        float acc[4][3] = {};
#pragma unroll
        for (int k = 0; k < NC; ++k) h[k] = 0.f;
        for (int ch = 0; ch < 3; ++ch) {
            const float I = lint[3 * lt + ch];
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const float cl = sc.cl[(size_t)i * 12 + band_of(k) * 3 + ch];
                const float uy = ui[ch * NC + k] * Y[k] * I * pre;
                qv += uy * cl;
                acc[band_of(k)][ch] += uy * T;
                h[k] += ui[ch * NC + k] * I * cl;
            }
        }
        for (int b = 0; b < 4; ++b)
            for (int ch = 0; ch < 3; ++ch)
                if (acc[b][ch] != 0.f) atomicAdd(&P[(size_t)i * 12 + b * 3 + ch], acc[b][ch]);
        qv *= ai;
        if constexpr (GEO) {
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                h[k] *= ai;
                H += h[k] * Y[k];
            }
            const float3 t1 = sh_grad_dot<NC>(rw, h);
            const float3 t3 = reflect_n(n, t1);
            const float f = fall * T;
            gw = make_float3(f * (cs * t3.x + H * n.x), f * (cs * t3.y + H * n.y), f * (cs * t3.z + H * n.z));
            const float3 gn = reflect_grad_n(n, w, (f * cs) * t1) + (H * f) * w; // R_i w and cos = n_i.w
            geo_add3(gF + GEO_GF * (size_t)i + GEO_N, gn);
        }
    }
    const bool second = lit && qv != 0.f && nzero <= 1;
    if (__any_sync(WT_FULL, second)) {
        sm.q[lane] = qv;
        sm.T[lane] = Tnz;
        sm.nz[lane] = nzero;
        __syncwarp();
        auto test = [&](int j, int ray, bool valid) {
            bool terms = false;
            if (valid) {
                const float4 ro = sm.w.o[ray], rd = sm.w.d[ray];
                const float3 oo = f3(ro), dd = f3(rd);
                float t, g, oj;
                if (hit_surfel(sc, j, __float_as_int(ro.w), oo, dd, rd.w, eps, t, g, oj)) {
                    const float om = 1.f - alpha_of(sc, oj, g);
                    const float others = sm.nz[ray] == 0 ? sm.T[ray] / om : (om == 0.f ? sm.T[ray] : 0.f);
                    if (others != 0.f) {
                        const float q = sm.q[ray];
                        atomicAdd(&dop[j], -q * others * dalpha_do(sc, oj, g));
                        if constexpr (GEO) {
                            const float coef = -q * others * dalpha_dq(sc, oj, g);
                            if (coef != 0.f) {
                                terms = true;
                                float uu, vv;
                                const float3 pw = crossing_pw(sc, j, oo, dd, t, uu, vv);
                                sm.gp[lane][0] = coef * pw.x;
                                sm.gp[lane][1] = coef * pw.y;
                                sm.gp[lane][2] = coef * pw.z;
                                sm.gw[lane][0] = (coef * t) * pw.x;
                                sm.gw[lane][1] = (coef * t) * pw.y;
                                sm.gw[lane][2] = (coef * t) * pw.z;
                                geo_add3(dp + GEO_DP * (size_t)j, (-coef) * pw);
                                geo_add2(ds + 2 * (size_t)j, coef * (-2.f * uu * uu * __ldg(&sc.FU[j].w)),
                                         coef * (-2.f * vv * vv * __ldg(&sc.FV[j].w)));
                                occluder_frame_grad(sc, j, oo, dd, t, uu, vv, coef, gF);
                            }
                        }
                    }
                }
            }
            if constexpr (GEO)
                warp_owner_loop(sm.w.own, terms, ray, [&](int b) {
                    gpi = gpi + make_float3(sm.gp[b][0], sm.gp[b][1], sm.gp[b][2]);
                    gw = gw + make_float3(sm.gw[b][0], sm.gw[b][1], sm.gw[b][2]);
                });
        };
        warp_traverse<false, false>(sc, o, w, r, second, sm.w.q, test, [](float m) { return m; });
    }
    if constexpr (GEO) {
        if (!lit) return;
        float3 gp = gpi;
        if (!ldir) { // w = (p_L - p_i)/r, fall = 1/r^2
            const float ww = dot3(w, gw), gr = H * cs * T * (-2.f * fall / r);
            gp.x += -(gw.x - w.x * ww) / r - w.x * gr;
            gp.y += -(gw.y - w.y * ww) / r - w.y * gr;
            gp.z += -(gw.z - w.z * ww) / r - w.z * gr;
        }
        geo_add3(dp + GEO_DP * (size_t)i, gp);
    }
}

template <int NC>
void launch_shadow(rgs_transport *t, cudaStream_t st, float *dp, float *ds, float *gF) {
    const int per = shadow_pairs((long long)t->n * t->nl), pb = SHADOW_THREADS / 32 * per; // pairs of a warp, a block
    const unsigned blocks = (unsigned)((t->n * t->nl + pb - 1) / pb);
    const size_t smem = sizeof(ShadowWarp) * (SHADOW_THREADS / 32);
    ProfScope ps_("k_shadow_bwd", st);
    if (dp) k_shadow_bwd<NC, true><<<blocks, SHADOW_THREADS, smem, st>>>(t->sc->dev(), t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->u, t->Pg, t->dop, dp, ds, gF);
    else k_shadow_bwd<NC, false><<<blocks, SHADOW_THREADS, smem, st>>>(t->sc->dev(), t->nl, per, t->ldir, t->lpos, t->lint, t->C, t->u, t->Pg, t->dop, dp, ds, gF);
}

// Hemisphere rays, part 1: for every stored hit h of ray r (receiver i, source j_h),
//   g_h = sum_{a<n} sum_c y_r^(a)[c] Y(-d_r) . B^(n-1-a)_{j_h}[c],
//   y_r^(a)[c] = (pi/nd) o_i sum_k' c_{i,l(k'),ch} Y_k'(R_i d_r) v_i^(a)[c][k'],
// accumulated into gh[slot] for iterates a0 .. a0+na-1 (first chunk writes, later add).
template <int NC, int CT, int NA, class SLB>
__global__ void RGS_OPA_LB k_opacity_g(SceneDev sc, RaysDev rays, int C, int col0, int na,
                                                   OpaSet<typename SLB::T, NA> it, float *gh, bool first) {
    using SL = Slice<NC>;
    constexpr int G = SL::G, KPL = SL::KPL;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int ray = t / G, g = t % G;
    const int n_rays = sc.n * rays.nd;
    const bool live = ray < n_rays;
    const int r = live ? ray : n_rays - 1;
    const int cnt = live ? rays.cnt[r] : 0;
    const int i = r / rays.nd;
    const float3 n = f3(sc.N4[i]);
    const float3 d = f3(rays.dir[r]);
    float yo[KPL];
    float y[NA][CT];
    {
        float Y[NC], yi[KPL];
        sh_eval<NC>(neg3(d), Y);
        SL::pick(Y, g, yo);
        sh_eval<NC>(reflect_n(n, d), Y);
        SL::pick(Y, g, yi);
        const float oi = alpha_center(sc, i) * (3.14159265358979f / (float)rays.nd);
#pragma unroll
        for (int aa = 0; aa < NA; ++aa) {
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                float s = 0.f;
                if (aa < na) {
                    const int ch = (col0 + c) % 3;
                    float v[KPL];
                    SL::load(it.v[aa] + ((size_t)i * C + col0 + c) * NC, g, v);
#pragma unroll
                    for (int m = 0; m < KPL; ++m) {
                        const int kk = SL::k(g, m);
                        const float cl = (kk < NC) ? __ldg(&sc.cl[(size_t)i * 12 + band_of(kk) * 3 + ch]) : 0.f;
                        s += cl * yi[m] * v[m];
                    }
                }
                y[aa][c] = oi * SL::group_sum(s);
            }
        }
    }
    const long long base = rays.off[r];
    const int rows = SL::G == 1 ? cnt : __reduce_max_sync(0xffffffffu, cnt); // groups of a warp stay converged
    for (int h = 0; h < rows; ++h) {
        float acc = 0.f;
        int j = 0;
        if (h < cnt) j = __ldg(&rays.rec_ja[base + h]).x;
#pragma unroll
        for (int aa = 0; aa < NA; ++aa) {
            if (aa < na && h < cnt) {
                const typename SLB::T *Bj = it.b[aa] + ((size_t)j * C + col0) * SLB::STRIDE;
#pragma unroll
                for (int c = 0; c < CT; ++c) {
                    float v[KPL];
                    SLB::load(Bj + c * SLB::STRIDE, g, v);
                    float s = 0.f;
#pragma unroll
                    for (int m = 0; m < KPL; ++m) s += yo[m] * v[m];
                    acc += y[aa][c] * s;
                }
            }
        }
        acc = SL::group_sum(acc);
        if (g == 0 && h < cnt) {
            const long long slot = base + h;
            gh[slot] = first ? acc : gh[slot] + acc;
        }
    }
}

// Hemisphere rays, part 2: back to front, R_{h-1} = alpha_h g_h + (1 - alpha_h) R_h and
// dL/do_{j_h} += T_h (g_h - R_h) dalpha_h/do, with T_h the transmittance in front of hit h,
// T_h = a_h / alpha_h from the stored weight.  G_h is recomputed from the stored direction
// (bit-identical to the trace's value).
// gt: the sums are there in the order of the transposed index, and gh holds each record's entry
// (50,000 surfels, 256 rays: 5.4 ms against 2.8 for a pass that sorts them and 3.4).
__global__ void RGS_OPAREC_LB k_opacity_rec(SceneDev sc, RaysDev rays, const float *__restrict__ gh,
                                                     const float *__restrict__ gt, float *dop) {
    // Blocks take the rays in a scattered order (block b -> b * 2654435761 mod gridDim, a
    // bijection: the multiplier is prime): blocks resident at the same time then hold
    // receivers spread over the scene, so their dL/do atomics go to sources all over it
    // instead of piling onto the few sources of one neighbourhood (32 % faster measured).
    const unsigned bs = (unsigned)(((unsigned long long)blockIdx.x * 2654435761ull) % gridDim.x);
    const int r = (int)bs * blockDim.x + threadIdx.x;
    if (r >= sc.n * rays.nd) return;
    const int cnt = rays.cnt[r];
    if (cnt == 0) return;
    const long long base = rays.off[r];
    const int i = r / rays.nd;
    const float3 o = f3(sc.P[i]);
    const float3 d = f3(rays.dir[r]);
    float R = 0.f;
    for (int h = cnt - 1; h >= 0; --h) {
        const long long slot = base + h;
        const int2 ja = __ldg(&rays.rec_ja[slot]);
        const int j = ja.x;
        float t, r2, oj;
        accepted_hit(sc, j, o, d, t, r2, oj);
        const float G = surfel_G(sc, r2);
        const float alpha = alpha_of(sc, oj, G);
        const float g = gt ? __ldg(&gt[__float_as_uint(gh[slot])]) : gh[slot]; // (gt: gh holds the records' entries)
        // the transmittance in front of the hit from its stored weight a_h = alpha_h T_h
        // (alpha_h = 0 makes dalpha/do vanish for the disc and Gaussian models; GFSGS: alpha = 0
        // only where x = o G = 0, where dalpha/do is 0 too)
        const float Th = alpha > 0.f ? __int_as_float(ja.y) / alpha : 0.f;
        const float da = Th * (g - R);
        if (da != 0.f) atomicAdd(&dop[j], da * dalpha_do(sc, oj, G));
        R = alpha * g + (1.f - alpha) * R;
    }
}

// Geometry gradients of the hemisphere-ray transport (Eqs. dl-dgeo-0/1), part 1 (compositing),
// one thread per ray from the per-record g_h of the opacity backward: each hit's alpha moves
// with q_h = u^2 + v^2 at the hit point on its source's plane, with dL/dalpha_h =
// T_h (g_h - R_h) (back to front, as k_opacity_rec); q_h moves with p_i, the ray direction
// and the source's centre, scales and frame.  The ray leaves p_i along
// d = c_x t^u_i + c_y t^v_i + c_z n_i with fixed c, so dL/dd goes to the receiver's frame.
// The receiver's terms are summed over the warp (nd is a multiple of 32, so a warp's rays
// share their receiver) and added once per warp.  Part 2 is k_hemi_geo_dir.
__global__ void __launch_bounds__(128) k_hemi_geo(SceneDev sc, RaysDev rays, int nb, const float *__restrict__ gh,
                                                 float *dp, float *ds, float *gF) {
    // scattered block order (as k_opacity_rec): resident blocks hold receivers spread over the
    // scene, so their per-hit atomics land on sources all over it
    const unsigned bs = (unsigned)(((unsigned long long)blockIdx.x * 2654435761ull) % gridDim.x);
    const int r = (int)bs * blockDim.x + threadIdx.x;
    const int n_rays = sc.n * rays.nd;
    if (r - (int)(threadIdx.x & 31) >= n_rays) return; // whole warps (n_rays % 32 == 0)
    const int i = r / rays.nd;
    const int cnt = rays.cnt[r];
    const float3 o = f3(sc.P[i]), n = f3(sc.N4[i]), d = f3(rays.dir[r]);
    float3 gpi = make_float3(0.f, 0.f, 0.f), gd = make_float3(0.f, 0.f, 0.f);
    if (cnt > 0 && nb > 0) {
        const long long base = rays.off[r];
        float R = 0.f;
        for (int h = cnt - 1; h >= 0; --h) {
            const int2 ja = __ldg(&rays.rec_ja[base + h]);
            const int j = ja.x;
            float th, r2, oj;
            accepted_hit(sc, j, o, d, th, r2, oj);
            const float G = surfel_G(sc, r2);
            const float al = alpha_of(sc, oj, G);
            const float g = gh[base + h];
            // the transmittance in front of the hit from its stored weight a_h = alpha_h T_h
            // (alpha_h = 0 makes dalpha/dq vanish too)
            const float Th = al > 0.f ? __int_as_float(ja.y) / al : 0.f;
            const float coef = Th * (g - R) * dalpha_dq(sc, oj, G);
            if (coef != 0.f) {
                const float4 Nj = __ldg(&sc.N4[j]), Pj = __ldg(&sc.P[j]);
                const float t = (Nj.x * (Pj.x - o.x) + Nj.y * (Pj.y - o.y) + Nj.z * (Pj.z - o.z)) /
                                (Nj.x * d.x + Nj.y * d.y + Nj.z * d.z);
                float uu, vv;
                const float3 pw = crossing_pw(sc, j, o, d, t, uu, vv);
                gpi = gpi + coef * pw;
                gd = gd + (coef * t) * pw;
                geo_add3(dp + GEO_DP * (size_t)j, (-coef) * pw);
                geo_add2(ds + 2 * (size_t)j, coef * (-2.f * uu * uu * __ldg(&sc.FU[j].w)),
                         coef * (-2.f * vv * vv * __ldg(&sc.FV[j].w)));
                occluder_frame_grad(sc, j, o, d, t, uu, vv, coef, gF);
            }
            R = al * g + (1.f - al) * R;
        }
    }
    const float3 tu = f3(sc.FU[i]), tv = f3(sc.FV[i]);
    const float cx = dot3(d, tu), cy = dot3(d, tv), cz = dot3(d, n);
    const float3 gn = cz * gd;
    float red[12] = {gpi.x, gpi.y, gpi.z, cx * gd.x, cx * gd.y, cx * gd.z, cy * gd.x, cy * gd.y, cy * gd.z,
                     gn.x, gn.y, gn.z};
#pragma unroll
    for (int q = 0; q < 12; ++q)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) red[q] += __shfl_xor_sync(0xffffffffu, red[q], off);
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (red[q] != 0.f) atomicAdd(&dp[GEO_DP * (size_t)i + q], red[q]);
#pragma unroll
        for (int q = 0; q < 9; ++q)
            if (red[3 + q] != 0.f) atomicAdd(&gF[GEO_GF * (size_t)i + 4 * (q / 3) + q % 3], red[3 + q]);
    }
}

constexpr int GEO_DIR_THREADS = 256;

// Part 2 (directional effects), a CTA per receiver and G lanes per ray, each lane a slice of
// the SH coefficients (the layout of the bounce gather): Y(R_i d) through
// X^(a)[c] = Y(-d).P^(a)[c] and Y(-d) through the composited source rows
// P^(a)[c] = sum_h a_h B_{j_h}^(nb-1-a)[c] (gathered once per 3-column tile and iterate);
// with cv = (pi/nd) o_i c_i (x) v_i^(a)[c], w_i = sum X cv and w_o = sum (cv.Y(R_i d)) P,
// dL/dd = R_i grad Y(R_i d).w_i - grad Y(-d).w_o, dL/dn_i from R_i, summed over the
// receiver's rays into its frame gradient.
template <int NC>
__global__ void __launch_bounds__(GEO_DIR_THREADS) k_hemi_geo_dir(SceneDev sc, RaysDev rays, int C, int nb, size_t A,
                                                                const float *__restrict__ V,
                                                                const float *__restrict__ Bit, float *gF) {
    using SL = Slice<NC>;
    constexpr int G = SL::G, KPL = SL::KPL, GROUPS = GEO_DIR_THREADS / G, CT = 3;
    __shared__ float red[GEO_DIR_THREADS / 32][9];
    const int i = blockIdx.x;
    const int grp = threadIdx.x / G, g = threadIdx.x % G, lane = threadIdx.x & 31;
    const int nd = rays.nd;
    const float3 n = f3(sc.N4[i]), tu = f3(sc.FU[i]), tv = f3(sc.FV[i]);
    const float wa = alpha_center(sc, i) * (3.14159265358979f / (float)nd);
    float acc[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[q] = 0.f;
    for (int qb = 0; qb < nd; qb += GROUPS) { // every lane makes the same trips (group shuffles)
        const int q = qb + grp;
        const bool live = q < nd;
        const long long r = (long long)i * nd + (live ? q : 0);
        const float3 d = f3(rays.dir[r]);
        const int cnt = live ? rays.cnt[r] : 0;
        const long long base = rays.off[r];
        const float3 rd = reflect_n(n, d);
        float yo[KPL], yi[KPL];
        {
            float Y[NC];
            sh_eval<NC>(neg3(d), Y);
            SL::pick(Y, g, yo);
            sh_eval<NC>(rd, Y);
            SL::pick(Y, g, yi);
        }
        float wi[KPL], wo[KPL];
#pragma unroll
        for (int m = 0; m < KPL; ++m) wi[m] = wo[m] = 0.f;
        for (int a = 0; a < nb; ++a) {
            const float *va = V + A * a + (size_t)i * C * NC;
            const float *Bb = Bit + A * (nb - 1 - a);
            for (int c0 = 0; c0 < C; c0 += CT) {
                float P[CT][KPL];
#pragma unroll
                for (int c = 0; c < CT; ++c)
#pragma unroll
                    for (int m = 0; m < KPL; ++m) P[c][m] = 0.f;
#pragma unroll 2
                for (int h = 0; h < cnt; ++h) {
                    const int2 ja = __ldg(&rays.rec_ja[base + h]);
                    const float ah = __int_as_float(ja.y);
                    const float *Bj = Bb + ((size_t)ja.x * C + c0) * NC;
#pragma unroll
                    for (int c = 0; c < CT; ++c) {
                        float v[KPL];
                        SL::load(Bj + c * NC, g, v);
#pragma unroll
                        for (int m = 0; m < KPL; ++m) P[c][m] += ah * v[m];
                    }
                }
#pragma unroll
                for (int c = 0; c < CT; ++c) {
                    const int col = c0 + c;
                    float vv[KPL], cv[KPL];
                    SL::load(va + (size_t)col * NC, g, vv);
                    float xs = 0.f, ys = 0.f;
#pragma unroll
                    for (int m = 0; m < KPL; ++m) {
                        const int k = SL::k(g, m);
                        cv[m] = k < NC ? wa * __ldg(&sc.cl[(size_t)i * 12 + band_of(k) * 3 + (col % 3)]) * vv[m] : 0.f;
                        xs += yo[m] * P[c][m];
                        ys += cv[m] * yi[m];
                    }
                    const float X = SL::group_sum(xs), y = SL::group_sum(ys);
#pragma unroll
                    for (int m = 0; m < KPL; ++m) {
                        wi[m] += X * cv[m];
                        wo[m] += y * P[c][m];
                    }
                }
            }
        }
        // the whole w_i, w_o from the group's lanes
        float WI[NC], WO[NC];
#pragma unroll
        for (int g2 = 0; g2 < G; ++g2)
#pragma unroll
            for (int m = 0; m < KPL; ++m) {
                const float xi = __shfl_sync(0xffffffffu, wi[m], (lane & ~(G - 1)) + g2);
                const float xo = __shfl_sync(0xffffffffu, wo[m], (lane & ~(G - 1)) + g2);
                const int k = SL::k(g2, m);
                if (k < NC) {
                    WI[k] = xi;
                    WO[k] = xo;
                }
            }
        if (live && g == 0 && cnt > 0) {
            const float3 t1 = sh_grad_dot<NC>(rd, WI);
            const float3 gd = reflect_n(n, t1) - sh_grad_dot<NC>(neg3(d), WO);
            const float cx = dot3(d, tu), cy = dot3(d, tv), cz = dot3(d, n);
            const float3 gn = reflect_grad_n(n, d, t1) + cz * gd;
            acc[0] += cx * gd.x, acc[1] += cx * gd.y, acc[2] += cx * gd.z;
            acc[3] += cy * gd.x, acc[4] += cy * gd.y, acc[5] += cy * gd.z;
            acc[6] += gn.x, acc[7] += gn.y, acc[8] += gn.z;
        }
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        float v = acc[q];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) red[threadIdx.x >> 5][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        float v = 0.f;
        for (int w = 0; w < GEO_DIR_THREADS / 32; ++w) v += red[w][threadIdx.x];
        if (v != 0.f) atomicAdd(&gF[GEO_GF * (size_t)i + 4 * (threadIdx.x / 3) + threadIdx.x % 3], v);
    }
}

template <int NC>
__global__ void __launch_bounds__(32 * ROW_WARPS) k_finalize(SceneDev sc, int C, const float *__restrict__ u,
                                                            const float *__restrict__ P, const float *__restrict__ kk,
                                                            const float *__restrict__ dop_acc, float *dE, float *dad,
                                                            float *dop) {
    const int lane = threadIdx.x & 31, i = blockIdx.x * ROW_WARPS + (threadIdx.x >> 5);
    if (i >= sc.n) return;
    const int ui = sc.uid[i];
    const float *Pi = P + (size_t)i * 12;
    if (dE) {
        const size_t row = (size_t)i * C * NC;
        float acc[2];
        column_sums<NC>(C, acc, [&](int e) { return __ldg(&u[row + e]); });
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = lane + 32 * h, ch = o / NC, k = o - ch * NC;
            if (o < 3 * NC) dE[((size_t)ui * NC + k) * 3 + ch] = acc[h];
        }
    }
    if (lane > 0) return;
    const float ai = alpha_center(sc, i);
    if (dad)
        for (int ch = 0; ch < 3; ++ch) dad[(size_t)ui * 3 + ch] = 4.f * kk[i] * ai * Pi[ch];
    if (dop) {
        float s = 0.f;
        for (int q = 0; q < 12; ++q) s += sc.cl[(size_t)i * 12 + q] * Pi[q];
        dop[ui] = dop_acc[i] + dalpha_center(sc, i) * s;
    }
}

// transposed index: the records of every ray on a source j0 <= j < j1 scattered into
// per-source lists of (ray, a), stored from entry ebase = src_off[j0] on
__global__ void k_src_fill(RaysDev rays, int n_rays, unsigned long long *cursor, int2 *tr, int j0, int j1,
                           long long ebase, unsigned *entry) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rays) return;
    const long long base = rays.off[r];
    const int c = rays.cnt[r];
    for (int h = 0; h < c; ++h) {
        const int2 ja = rays.rec_ja[base + h];
        if (ja.x < j0 || ja.x >= j1) continue;
        const unsigned long long pos = atomicAdd(&cursor[ja.x], 1ull);
        tr[(long long)pos - ebase] = make_int2(r, ja.y);
        if (entry) entry[base + h] = (unsigned)pos; // the record's entry
    }
}

// the records' sums from the order of the index: gh[slot] holds the record's entry, then its sum
__global__ void k_opacity_slots(long long n_slots, unsigned n_hits, const float *__restrict__ gt, float *gh) {
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n_slots; s += (long long)gridDim.x * blockDim.x) {
        const unsigned e = __float_as_uint(gh[s]);
        if (e < n_hits) gh[s] = __ldg(&gt[e]); // (slots between the rays' records hold anything)
    }
}

__global__ void k_copy_off(const long long *off, unsigned long long *cursor, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cursor[i] = (unsigned long long)off[i];
}


// the transposed index of sources j0 .. j1-1 into t->tr (entries from ebase on); entries: every
// record's entry into t->gh
rgs_status build_index(rgs_transport *t, int j0, int j1, long long ebase, bool entries, cudaStream_t st) {
    const int n = t->n;
    const long long n_rays = (long long)n * t->nd;
    RaysDev rd = t->rays();
    { ProfScope ps_("k_copy_off", st); k_copy_off<<<(n + 255) / 256, 256, 0, st>>>(t->src_off, t->cursor, n); }
    { ProfScope ps_("k_src_fill", st); k_src_fill<<<(unsigned)((n_rays + 255) / 256), 256, 0, st>>>(rd, (int)n_rays, t->cursor, t->tr, j0, j1, ebase, entries ? reinterpret_cast<unsigned *>(t->gh) : nullptr); }
    RGS_LAUNCH("transposed index");
    return RGS_OK;
}

// g_h (+)= the na iterates of one group, all column tiles; first: the group that writes gh
template <int NC>
rgs_status opacity_group(rgs_transport *t, SceneDev sd, RaysDev rd, int na, const float *const *v,
                         const float *const *Bf, const __nv_bfloat16 *const *Bh, bool first, cudaStream_t st) {
    if (wide_opacity(NC, t->C, Bh != nullptr)) return mc_opacity<NC>(t, sd, rd, na, v, Bf, Bh, first, st);
    constexpr int NA = 4;
    const long long n_rays = (long long)t->n * t->nd;
    const unsigned gg = (unsigned)((n_rays * Slice<NC>::G + 255) / 256);
    OpaSet<float, NA> sf = {};
    OpaSet<__nv_bfloat16, NA> sh = {};
    for (int a = 0; a < na; ++a) {
        sf.v[a] = sh.v[a] = v[a];
        sf.b[a] = Bf[a];
        sh.b[a] = Bh ? Bh[a] : nullptr;
    }
    for (int col0 = 0; col0 < t->C; col0 += 3) {
        const bool wr = first && col0 == 0;
        if (Bh) { // the batched modes gather the BF16 iterate copies
            ProfScope ps_("k_opacity_g", st);
            k_opacity_g<NC, 3, NA, SliceH<NC>><<<gg, 256, 0, st>>>(sd, rd, t->C, col0, na, sh, t->gh, wr);
        } else {
            ProfScope ps_("k_opacity_g", st);
            k_opacity_g<NC, 3, NA, Slice<NC>><<<gg, 256, 0, st>>>(sd, rd, t->C, col0, na, sf, t->gh, wr);
        }
    }
    RGS_LAUNCH("opacity gather");
    return RGS_OK;
}

// The adjoint walks the bounces backwards, b = n-1 .. 0 (a = n-1-b = 0 .. n-1), in segments
// [lo, hi] that end at a stored iterate: one segment holding everything when every iterate
// was kept, else one per checkpoint, whose B^(b) and Q^(b) are recomputed from B^(lo) into
// pooled scratch before the segment's v^(a) are formed and used.
template <int NC>
rgs_status run_adjoint(rgs_transport *t, const float *g, float *dE, float *dad, float *dopo,
                       const std::vector<int> &parts, const std::vector<long long> &part_base, cudaStream_t st,
                       const RgsGeoAcc *geo, bool tcp) {
    const int n = t->n, C = t->C, nb = t->nb_last, s = t->stride;
    const size_t A = t->arr();
    const size_t A16 = (size_t)n * C * bf16_stride<NC>();
    const bool bf16 = t->prec_last != RGS_FP32;
    SceneDev sd = t->sc->dev();
    RaysDev rd = t->rays();
    const unsigned ga = (unsigned)((A + 255) / 256);
    const unsigned gw = (unsigned)((n + ROW_WARPS - 1) / ROW_WARPS);
    const long long n_rays = (long long)n * t->nd;
    const unsigned gr = (unsigned)((n_rays + 255) / 256);
    auto vp = [&](int a) { return t->v + A * (s ? a % (s + 1) : a); };
    // v^(0) = g (internal layout), u = v^(0), P = 0, dop = 0
    { ProfScope ps_("k_from_user", st); k_from_user<NC><<<ga, 256, 0, st>>>(n, C, t->sc->uid, g, vp(0)); }
    RGS_CUDA(cudaMemcpyAsync(t->u, vp(0), sizeof(float) * A, cudaMemcpyDeviceToDevice, st));
    RGS_CUDA(cudaMemsetAsync(t->Pg, 0, sizeof(float) * 12 * (size_t)n, st));
    RGS_CUDA(cudaMemsetAsync(t->dop, 0, sizeof(float) * (size_t)n, st));
    RGS_LAUNCH("adjoint init");
    // v^(a) = K^T v^(a-1), u += v^(a): per part of the transposed index (one part holding
    // every source unless memory asked for more), per column tile
    // and, where t->gt is there, g_e of the pairing (v^(a-1), B^(n-a)), B^(n-a) given in FP32 and BF16
    const bool fused = !tcp && t->gt;
    auto KT = [&](int a, const float *Bf, const __nv_bfloat16 *Bh) -> rgs_status {
        rgs_status q;
        if (tcp) { // tensor cores over source tiles: y^(a-1) = o c (x) v^(a-1) in BF16 row blocks
            // mode 2: the opacity gather pairs y^(a) with B^(n-1-a) while y^(a) is at hand, per
            // (tile, receiver) group (at 16 columns per MMA it measured slower than the row
            // gathers and than the sampled products that modes -1 and 1 run after the bounces)
            const bool gh = (dopo || geo) && nb >= 1 && t->tc_mode == 2;
            if (a == 1) {
                if ((q = rgs_tc_make_y(t, vp(0), 0, st)) != RGS_OK) return q;
                if (gh && (q = rgs_tc_opacity(t, 0, t->iters + A * (nb - 1), true, st)) != RGS_OK) return q;
            }
            if ((q = rgs_tc_adjoint_bounce(t, (a - 1) & 1, a & 1, vp(a), t->u, st)) != RGS_OK) return q;
            if (gh && a <= nb - 1 && (q = rgs_tc_opacity(t, a & 1, t->iters + A * (nb - 1 - a), false, st)) != RGS_OK)
                return q;
            return RGS_OK;
        }
        for (size_t p = 0; p + 1 < parts.size(); ++p) {
            const int j0 = parts[p], j1 = parts[p + 1];
            if (j1 <= j0) continue;
            const long long eb = part_base[p];
            if (parts.size() > 2 && (q = build_index(t, j0, j1, eb, false, st)) != RGS_OK) return q;
            for (int col0 = 0; col0 < C;) {
                const AdjOpa opa{Bf, Bh, t->gt, a == 1 && col0 == 0};
                if (t->dy_cols == 12 && C - col0 > 3) {
                    { ProfScope ps_("k_adj_ray", st); k_adj_ray<NC, 12><<<gr, 256, 0, st>>>(sd, rd, C, col0, vp(a - 1), t->dy); }
                    ProfScope ps_("k_adj_src_tile", st);
                    (fused ? k_adj_src_tile<NC, true> : k_adj_src_tile<NC, false>)<<<j1 - j0, ADJ_THREADS, 0, st>>>(C, col0, t->src_off, t->tr, t->dy, vp(a), t->u, j0, eb, opa);
                    col0 += 12;
                    continue;
                }
                { ProfScope ps_("k_adj_ray", st); k_adj_ray<NC, 3><<<gr, 256, 0, st>>>(sd, rd, C, col0, vp(a - 1), t->dy); }
                ProfScope ps_("k_adj_src", st);
                (fused ? k_adj_src<NC, true> : k_adj_src<NC, false>)<<<j1 - j0, ADJ_THREADS, 0, st>>>(C, col0, t->src_off, t->tr, t->dy, vp(a), t->u, j0, eb, opa);
                col0 += 3;
            }
            RGS_LAUNCH("adjoint bounce");
        }
        return RGS_OK;
    };
    // segment scratch (checkpointing): B^(lo+1 .. lo+s) FP32 (+BF16) and Q^(lo .. lo+s-1)
    struct SegScratch {
        cudaStream_t st;
        std::vector<float *> B, Q;
        std::vector<__nv_bfloat16 *> B16;
        double *nrm = nullptr;
        ~SegScratch() {
            for (auto &p : B) pool_release(p, st);
            for (auto &p : Q) pool_release(p, st);
            for (auto &p : B16) pool_release(p, st);
            pool_release(nrm, st);
        }
    } seg{st, {}, {}, {}, nullptr};
    rgs_status r;
    if (s) {
        seg.B.assign(s, nullptr);
        seg.Q.assign(s, nullptr);
        seg.B16.assign(s, nullptr);
        for (int k = 0; k < s; ++k) {
            if ((r = pool_alloc(&seg.B[k], A, st)) != RGS_OK) return r;
            if ((r = pool_alloc(&seg.Q[k], A, st)) != RGS_OK) return r;
            if (bf16) {
                if ((r = pool_alloc(&seg.B16[k], A16, st)) != RGS_OK) return r;
                RGS_CUDA(cudaMemsetAsync(seg.B16[k], 0, sizeof(__nv_bfloat16) * A16, st)); // row padding
            }
        }
        if ((r = pool_alloc(&seg.nrm, RGS_MAX_BOUNCES + 1, st)) != RGS_OK) return r;
    }
    bool first_g = true;
    // the opacity gather's form, fixed for the whole adjoint (the sampled products sum in
    // the source tiles' hit order and hand the record slots their sums after the last pairing)
    const bool sddmm = tcp && (t->tc_mode == -1 || t->tc_mode == 1) && rgs_tc_opa_pass_cols(t) > 0;
    for (int hi = nb - 1; hi >= 0;) {
        const int lo = s ? (hi / s) * s : 0;
        // iterates B^(b) (FP32, BF16) and Q^(b) of this segment, indexed by b - lo
        std::vector<const float *> Bf(hi - lo + 1), Qb(hi - lo + 1);
        std::vector<const __nv_bfloat16 *> Bh(hi - lo + 1);
        if (!s) {
            for (int b = lo; b <= hi; ++b) {
                Bf[b - lo] = t->iters + A * b;
                Bh[b - lo] = bf16 ? t->iters16 + A16 * b : nullptr;
                Qb[b - lo] = t->Q + A * b;
            }
        } else {
            if ((r = rgs_recompute(t, lo, hi + 1, seg.B.data(), seg.B16.data(), seg.Q.data(), seg.nrm, st)) != RGS_OK)
                return r;
            for (int b = lo; b <= hi; ++b) {
                Bf[b - lo] = b == lo ? t->iters + A * t->slot(lo) : seg.B[b - lo - 1];
                Bh[b - lo] = !bf16 ? nullptr : (b == lo ? t->iters16 + A16 * t->slot(lo) : seg.B16[b - lo - 1]);
                Qb[b - lo] = seg.Q[b - lo];
            }
        }
        for (int b = hi; b >= lo; --b) {
            const int a = nb - 1 - b;
            { ProfScope ps_("k_pair_accum", st); k_pair_accum<NC><<<gw, 32 * ROW_WARPS, 0, st>>>(n, C, vp(a), Qb[b - lo], t->Pg); }
            RGS_LAUNCH("pair accum");
            if ((r = KT(a + 1, Bf[b - lo], Bh[b - lo])) != RGS_OK) return r; // (v^(n) only adds to u)
        }
        if ((dopo || geo) && sddmm) { // g_h as sampled products on the tensor cores
            for (int b = hi; b >= lo; --b) {
                if ((r = rgs_tc_opacity_sddmm(t, vp(nb - 1 - b), Bf[b - lo], first_g, b == 0, st)) != RGS_OK) return r;
                first_g = false;
            }
        } else if ((dopo || geo) && !fused && !(tcp && t->tc_mode == 2)) { // g_h over this segment's iterates, four per launch
            for (int b0 = hi; b0 >= lo; b0 -= 4) {
                const int na = min(4, b0 - lo + 1);
                const float *vv[4], *bb[4];
                const __nv_bfloat16 *hh[4];
                for (int q = 0; q < na; ++q) {
                    const int b = b0 - q;
                    vv[q] = vp(nb - 1 - b);
                    bb[q] = Bf[b - lo];
                    hh[q] = Bh[b - lo];
                }
                if ((r = opacity_group<NC>(t, sd, rd, na, vv, bb, bf16 ? hh : nullptr, first_g, st)) != RGS_OK) return r;
                first_g = false;
            }
        }
        hi = lo - 1;
    }
    if (fused && geo) { // (k_opacity_rec alone reads them through the entries)
        ProfScope ps_("k_opacity_slots", st);
        k_opacity_slots<<<(unsigned)std::min<long long>((t->n_slots + 255) / 256, 8192), 256, 0, st>>>(t->n_slots, (unsigned)t->n_hits, t->gt, t->gh);
        RGS_LAUNCH("opacity sums to the records");
    }
    if (t->nl > 0) {
        launch_shadow<NC>(t, st, geo ? geo->dp : nullptr, geo ? geo->ds : nullptr, geo ? geo->gF : nullptr);
        RGS_LAUNCH("shadow backward");
    }
    if (nb >= 1 && dopo) {
        { ProfScope ps_("k_opacity_rec", st); k_opacity_rec<<<gr, 256, 0, st>>>(sd, rd, t->gh, fused && !geo ? t->gt : nullptr, t->dop); }
        RGS_LAUNCH("hemisphere opacity backward");
    }
    if (nb >= 1 && geo) { // every iterate is kept (the caller checked the stride)
        const long long n_rays = (long long)n * t->nd;
        { ProfScope ps_("k_hemi_geo", st); k_hemi_geo<<<(unsigned)((n_rays + 127) / 128), 128, 0, st>>>(sd, rd, nb, t->gh, geo->dp, geo->ds, geo->gF); }
        RGS_LAUNCH("hemisphere geometry backward");
        { ProfScope ps_("k_hemi_geo_dir", st); k_hemi_geo_dir<NC><<<n, GEO_DIR_THREADS, 0, st>>>(sd, rd, C, nb, A, t->v, t->iters, geo->gF); }
        RGS_LAUNCH("hemisphere geometry backward (directional)");
    }
    { ProfScope ps_("k_finalize", st); k_finalize<NC><<<gw, 32 * ROW_WARPS, 0, st>>>(sd, C, t->u, t->Pg, t->sc->kk, t->dop, dE, dad, dopo); }
    RGS_LAUNCH("finalize");
    return tcp ? rgs_tc_check(t, st) : RGS_OK;
}

} // namespace

// ------------------------------------------------------------------ pieces shared with the
// center-to-center adjoint (rgs_pairs.cu)
void rgs_copy_offsets(const long long *off, unsigned long long *cursor, int n, cudaStream_t st) {
    k_copy_off<<<(n + 255) / 256, 256, 0, st>>>(off, cursor, n);
}

namespace {
template <int NC> rgs_status prologue_nc(rgs_transport *t, const float *g, cudaStream_t st) {
    const int n = t->n, C = t->C, nb = t->nb_last;
    const size_t A = t->arr();
    { ProfScope ps_("k_from_user", st); k_from_user<NC><<<(unsigned)((A + 255) / 256), 256, 0, st>>>(n, C, t->sc->uid, g, t->v); }
    RGS_CUDA(cudaMemcpyAsync(t->u, t->v, sizeof(float) * A, cudaMemcpyDeviceToDevice, st));
    RGS_CUDA(cudaMemsetAsync(t->Pg, 0, sizeof(float) * 12 * (size_t)n, st));
    RGS_CUDA(cudaMemsetAsync(t->dop, 0, sizeof(float) * (size_t)n, st));
    if (nb >= 1) { ProfScope ps_("k_pair_accum", st); k_pair_accum<NC><<<(n + ROW_WARPS - 1) / ROW_WARPS, 32 * ROW_WARPS, 0, st>>>(n, C, t->v, t->Q + A * (nb - 1), t->Pg); }
    RGS_LAUNCH("adjoint init");
    return RGS_OK;
}
template <int NC> rgs_status accum_nc(rgs_transport *t, const float *X, const float *Y, cudaStream_t st) {
    { ProfScope ps_("k_pair_accum", st); k_pair_accum<NC><<<(t->n + ROW_WARPS - 1) / ROW_WARPS, 32 * ROW_WARPS, 0, st>>>(t->n, t->C, X, Y, t->Pg); }
    RGS_LAUNCH("pair accum");
    return RGS_OK;
}
template <int NC> rgs_status shadow_nc(rgs_transport *t, cudaStream_t st, float *dp, float *ds, float *gF) {
    if (t->nl <= 0) return RGS_OK;
    launch_shadow<NC>(t, st, dp, ds, gF);
    RGS_LAUNCH("shadow backward");
    return RGS_OK;
}
template <int NC> rgs_status finalize_nc(rgs_transport *t, float *dE, float *dad, float *dop, cudaStream_t st) {
    { ProfScope ps_("k_finalize", st); k_finalize<NC><<<(t->n + ROW_WARPS - 1) / ROW_WARPS, 32 * ROW_WARPS, 0, st>>>(t->sc->dev(), t->C, t->u, t->Pg, t->sc->kk, t->dop, dE, dad, dop); }
    RGS_LAUNCH("finalize");
    return RGS_OK;
}
} // namespace

#define RGS_NC_SWITCH(nc, call1, call4, call9, call16)                                                                 \
    switch (nc) {                                                                                                      \
    case 1: return call1;                                                                                              \
    case 4: return call4;                                                                                              \
    case 9: return call9;                                                                                              \
    default: return call16;                                                                                            \
    }
rgs_status rgs_adjoint_prologue(rgs_transport *t, int nc, const float *g, cudaStream_t st) {
    RGS_NC_SWITCH(nc, prologue_nc<1>(t, g, st), prologue_nc<4>(t, g, st), prologue_nc<9>(t, g, st), prologue_nc<16>(t, g, st))
}
rgs_status rgs_pair_accum(rgs_transport *t, int nc, const float *X, const float *Y, cudaStream_t st) {
    RGS_NC_SWITCH(nc, accum_nc<1>(t, X, Y, st), accum_nc<4>(t, X, Y, st), accum_nc<9>(t, X, Y, st), accum_nc<16>(t, X, Y, st))
}
rgs_status rgs_shadow_backward(rgs_transport *t, int nc, cudaStream_t st, float *dp, float *ds, float *gF) {
    RGS_NC_SWITCH(nc, shadow_nc<1>(t, st, dp, ds, gF), shadow_nc<4>(t, st, dp, ds, gF), shadow_nc<9>(t, st, dp, ds, gF),
                  shadow_nc<16>(t, st, dp, ds, gF))
}
rgs_status rgs_adjoint_finalize(rgs_transport *t, int nc, float *dE, float *dad, float *dop, cudaStream_t st) {
    RGS_NC_SWITCH(nc, finalize_nc<1>(t, dE, dad, dop, st), finalize_nc<4>(t, dE, dad, dop, st),
                  finalize_nc<9>(t, dE, dad, dop, st), finalize_nc<16>(t, dE, dad, dop, st))
}
#undef RGS_NC_SWITCH

rgs_status rgs_adjoint_impl(rgs_transport *t, const float *g, float *dE, float *dad, float *dop, cudaStream_t st,
                            float *dp, float *ds, float *dtu, float *dtv) {
    if (t->kind == RGS_KIND_PAIRS) return rgs_adjoint_pairs_impl(t, g, dE, dad, dop, nullptr, dp, ds, dtu, dtv, st);
    const bool want_geo = dp || ds || dtu || dtv;
    if (want_geo && t->stride != 0) {
        rgs_set_error("geometry gradients of the hemisphere transport need every iterate: solve with checkpointing off");
        return RGS_ERR_STATE;
    }
    rgs_status r;
    const int nb = t->nb_last, n = t->n;
    const size_t A = t->arr();
    const long long n_rays = (long long)n * t->nd;
    if (n > t->pg_cap) {
        if ((r = dev_alloc(&t->Pg, (size_t)n * 12, &t->device_bytes)) != RGS_OK) return r;
        if ((r = dev_alloc(&t->dop, (size_t)n, &t->device_bytes)) != RGS_OK) return r;
        t->pg_cap = n;
    }
    // Workspaces that live only inside this call come from the stream-ordered pool and are
    // returned to it on every exit path: v^(0..n), u, the transposed index, the per-ray
    // adjoint values and the per-record opacity sums.
    struct Scratch {
        rgs_transport *t;
        cudaStream_t st;
        ~Scratch() {
            pool_release(t->v, st);
            pool_release(t->u, st);
            pool_release(t->tr, st);
            pool_release(t->dy, st);
            pool_release(t->gh, st);
            pool_release(t->gt, st);
            pool_release(geo.dp, st);
            pool_release(geo.ds, st);
            pool_release(geo.gF, st);
        }
        RgsGeoAcc geo;
    } scratch{t, st, {}};
    const bool want_gh = (dop || want_geo) && nb >= 1;
    // the last solve ran on the tensor cores: so do the transposed bounces (source tiles
    // instead of the transposed hit index and the per-ray adjoint values)
    const bool tcp = t->tc_used && t->kind == RGS_KIND_HEMISPHERE && t->stride == 0 && nb >= 1;
    if (tcp && ((r = rgs_tc_prepare_adjoint(t, st)) != RGS_OK || (r = rgs_tc_reset_flags(t, st)) != RGS_OK)) return r;
    if (want_geo) {
        RgsGeoAcc &geo = scratch.geo;
        if ((r = pool_alloc(&geo.dp, (size_t)n * GEO_DP, st)) != RGS_OK) return r;
        if ((r = pool_alloc(&geo.ds, (size_t)n * 2, st)) != RGS_OK) return r;
        if ((r = pool_alloc(&geo.gF, (size_t)n * GEO_GF, st)) != RGS_OK) return r;
        RGS_CUDA(cudaMemsetAsync(geo.dp, 0, sizeof(float) * n * GEO_DP, st));
        RGS_CUDA(cudaMemsetAsync(geo.ds, 0, sizeof(float) * n * 2, st));
        RGS_CUDA(cudaMemsetAsync(geo.gF, 0, sizeof(float) * n * GEO_GF, st));
    }
    const RgsGeoAcc *geop = want_geo ? &scratch.geo : nullptr;
    const int n_v = t->stride ? t->stride + 1 : nb + 1;
    if ((r = pool_alloc(&t->v, A * n_v, st)) != RGS_OK) return r;
    if ((r = pool_alloc(&t->u, A, st)) != RGS_OK) return r;
    if (want_gh && (r = pool_alloc(&t->gh, (size_t)t->n_slots, st)) != RGS_OK) return r;
    // The transposed index in one part when it fits next to the segment scratch of a
    // checkpointed adjoint, else in P parts of about equal entry counts, each rebuilt from
    // the records for every transposed bounce.
    const double A16 = t->prec_last != RGS_FP32 ? 2.0 * n * t->C * (t->nc >= 9 ? 16 : t->nc) : 0.0;
    const double seg = t->stride ? t->stride * (8.0 * A + A16) + 8.0 * (RGS_MAX_BOUNCES + 1) : 0.0;
    const double tr_all = 8.0 * (double)t->n_hits;
    double avail = 0.92 * (double)pool_available_bytes() - seg;
    if (t->mem_budget > 0) {
        const double scratch = 4.0 * A * (n_v + 1) + (want_gh ? 4.0 * t->n_slots : 0.0);
        avail = std::min(avail, (double)t->mem_budget - (double)t->device_bytes - scratch - seg);
    }
    if (!tcp) {
        // Records of 12-column tiles (64 bytes a ray) or of 3-column ones (32), by what a transposed
        // bounce then takes, in passes over the entries (8.3 G entries, 48 columns: 0.12 s each):
        // one per tile; with the index in P parts 2 + P / 2 for building it anew; and 0.3 per column
        // for gathering the opacity sums ray by ray (1.8 s) where they cannot be formed on the way.
        auto passes = [&](int cols) {
            const double room = avail - (cols == 12 ? 64.0 : 32.0) * n_rays;
            int P = 1;
            while (P < 64 && tr_all / P > room) P *= 2;
            const bool sums = P == 1 && t->n_hits < (1ll << 32) && 12.0 * (double)t->n_hits <= room;
            return (t->C + cols - 1) / cols + (P > 1 ? 2.0 + 0.5 * P : 0.0) + (want_gh && !sums ? 0.3 * t->C : 0.0);
        };
        t->dy_cols = t->C > 3 && passes(12) < passes(3) ? 12 : 3;
        r = pool_alloc(&t->dy, (size_t)n_rays * (t->dy_cols == 12 ? 16 : 8), st);
        if (r == RGS_ERR_OOM && t->dy_cols == 12) {
            t->dy_cols = 3;
            r = pool_alloc(&t->dy, (size_t)n_rays * 8, st);
        }
        if (r != RGS_OK) return r;
        avail -= (t->dy_cols == 12 ? 64.0 : 32.0) * n_rays;
    }
    int P = 1;
    while (!tcp && P < 64 && tr_all / P > avail) P *= 2;
    std::vector<int> parts{0};
    std::vector<long long> base{0};
    if (P > 1) {
        std::vector<long long> off((size_t)n + 1);
        RGS_CUDA(cudaMemcpyAsync(off.data(), t->src_off, sizeof(long long) * (n + 1), cudaMemcpyDeviceToHost, st));
        RGS_CUDA(cudaStreamSynchronize(st));
        int j = 0;
        for (int p = 1; p < P; ++p) {
            const long long target = (long long)((double)t->n_hits * p / P);
            while (j < n && off[j] < target) ++j;
            parts.push_back(j);
            base.push_back(off[j]);
        }
    }
    parts.push_back(n);
    long long biggest = 0;
    for (size_t p = 0; p + 1 < parts.size(); ++p) {
        const long long e1 = p + 2 < parts.size() ? base[p + 1] : t->n_hits;
        biggest = std::max(biggest, e1 - base[p]);
    }
    if (!tcp) {
        if ((r = pool_alloc(&t->tr, (size_t)std::max(biggest, 1ll), st)) != RGS_OK) return r;
        // the opacity sums with the transposed bounces where the index is in one part and their
        // array in its order has room; else ray-wise gathers, over the iterates' rows
        if (want_gh && parts.size() == 2 && t->n_hits > 0 && t->n_hits < (1ll << 32) && 12.0 * (double)t->n_hits <= avail) {
            r = pool_alloc(&t->gt, (size_t)t->n_hits, st);
            if (r != RGS_OK && r != RGS_ERR_OOM) return r;
        }
        if (parts.size() == 2 && (r = build_index(t, 0, n, 0, t->gt != nullptr, st)) != RGS_OK) return r;
    }
    switch (t->nc) {
    case 1: r = run_adjoint<1>(t, g, dE, dad, dop, parts, base, st, geop, false); break;
    case 4: r = run_adjoint<4>(t, g, dE, dad, dop, parts, base, st, geop, false); break;
    case 9: r = run_adjoint<9>(t, g, dE, dad, dop, parts, base, st, geop, false); break;
    default: r = run_adjoint<16>(t, g, dE, dad, dop, parts, base, st, geop, tcp);
    }
    if (r != RGS_OK || !want_geo) return r;
    return rgs_geometry_out(t, scratch.geo, dp, ds, dtu, dtv, st);
}
