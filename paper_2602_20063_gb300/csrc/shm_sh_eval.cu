// Direct evaluation of real spherical-harmonic glyphs (no table): value, S^2 gradient and normal of
// r(w) = sum_lm c_lm Y_lm(w), the ground truth and the fit targets of the Hermite maps (§4.2).
//
// Y_lm in the polynomial form of shm_build.cu: Y_lm = n_m P_l^m(z) Re or Im (x + iy)^m, n_0 = 1, else
// sqrt2, with dP_l^m/dz = f_lm P_l^{m+1}, f_lm = sqrt((l-m)(l+m+1)).  Summed by order m:
//   r   = sum_m C_m U_m + S_m V_m            U_m, V_m   = sum_l c_{l,+-m} n_m P_l^m
//   r_z = sum_m C_m U'_m + S_m V'_m          U'_m, V'_m = sum_l c_{l,+-m} n_m f_lm P_l^{m+1}
//   r_x = sum_m m (C_{m-1} U_m + S_{m-1} V_m),  r_y = sum_m m (C_{m-1} V_m - S_{m-1} U_m)
// and grad_{S^2} r is the tangential part of (r_x, r_y, r_z).
// The Legendre functions come from the monic three-term recurrence p_l = z p_{l-1} - beta_l p_{l-2},
// P_l^m = kappa_lm p_l^m, with the scale kappa folded into the coefficients: two operations per (l, m)
// instead of a normalised recurrence with its square roots.  Running the family of order M serves
// U_M, V_M (coefficients of order M) and U'_{M-1}, V'_{M-1} (order M-1), so one term (l, M) is a float4
// of scaled coefficients and six multiply-adds.
//
// Bound: FP32 issue (6 FMA per term; 40 B of I/O per query).  k_sh_eval_seg: all queries of a warp's
// slab belong to one glyph (segments or a single glyph); the warp scales that glyph's coefficients
// into its own shared memory once and every lane runs four queries as two float2 pairs, so a term is
// one broadcast 16-byte read for 128 queries (one pair per lane 289 us, three 254 us).  1,024 glyphs of
// L = 16, 2^22 queries: 3,777 -> 236 us (a thread per query with its Legendre table in local memory and
// about 60 instructions per term before), about half of the FP32 rate of its 1,160 multiply-adds per
// query; the error against 64 bits fell from 6.2e-7 to 5.0e-7 of the gradient.
// Where fewer than EV_SHORT queries of a glyph are left, scaling its coefficients and a slab of mostly idle
// lanes cost more than the queries: 32 queries then go a lane each (ev_one), lanes on glyphs of their own, and
// runs of empty segments are searched over.  100,000 glyphs of L = 8, 1 / 2 / 4 queries each: 304 / 232 / 233 -> 26 /
// 25 / 41 us (a thread per query before 45 / 83 / 123); 50,000 of 8: 120 -> 41; two segments among 200,000 empty ones
// 16.4 ms -> 15 us.  With 16 queries each a slab takes 109 us for 800,000 queries, the lanes no less.
// k_sh_eval_ids: per-query glyphs; ev_one for every query: the coefficients are gathered, each once (the
// derivative by its own recurrence).
#include <math.h>

#include "shm_internal.h"

namespace shm {

namespace {

constexpr int EV_LMAX = 20;
constexpr int EV_TERMS = (EV_LMAX + 1) * (EV_LMAX + 2) / 2;
constexpr int EV_BLOCK = 128;
constexpr int EV_WARPS = EV_BLOCK / 32;
constexpr int EV_SHORT = 16;  // fewer queries of a glyph than this go a thread each
constexpr int EV_RES = 4;  // CTAs per SM: 121 registers, no spills (five with 96 registers spill: 264 us)

// Constants of the terms (M, l), l = M..L, in the order the families run.
struct EvTable {
    float nbeta[EV_TERMS];  // -beta_l of order M (0 for the first two degrees of a family)
    float kc[EV_TERMS];     // n_M kappa_{l,M}
    float kd[EV_TERMS];     // n_{M-1} f_{l,M-1} kappa_{l,M}
};

EvTable make_table(int L)
{
    EvTable T;
    double kmm = sqrt(1.0 / (4.0 * 3.14159265358979323846));
    int t = 0;
    for (int m = 0; m <= L; ++m) {
        if (m > 0) kmm *= sqrt((2.0 * m + 1.0) / (2.0 * m));
        double kappa = kmm, a_prev = 0.0;
        for (int l = m; l <= L; ++l, ++t) {
            double beta = 0.0;
            if (l > m) {
                const double l2 = (double)l * l, m2 = (double)m * m, lm = (double)(l - 1) * (l - 1);
                const double a = sqrt((4.0 * l2 - 1.0) / (l2 - m2));
                if (l > m + 1) beta = sqrt((lm - m2) / (4.0 * lm - 1.0)) / a_prev;
                kappa *= a;
                a_prev = a;
            }
            T.nbeta[t] = (float)-beta;
            T.kc[t] = (float)(kappa * (m == 0 ? 1.0 : sqrt(2.0)));
            T.kd[t] = m == 0 ? 0.0f
                             : (float)(kappa * sqrt((double)(l - m + 1) * (l + m)) * (m == 1 ? 1.0 : sqrt(2.0)));
        }
    }
    return T;
}

struct EvArgs {
    int L, G;
    const float* coeffs;
    int64_t Q;
    const float* dirs;
    const int32_t* glyph;
    const int64_t* seg;
    float *R, *grad, *normal;
    int32_t* dev_status;
};

__device__ __forceinline__ void ev_store(const EvArgs& a, int64_t q, float r, const Vec3& g, const Vec3& n)
{
    if (a.R) __stcs(a.R + q, r);
    if (a.grad) { __stcs(a.grad + 3 * q, g.x); __stcs(a.grad + 3 * q + 1, g.y); __stcs(a.grad + 3 * q + 2, g.z); }
    if (a.normal) { __stcs(a.normal + 3 * q, n.x); __stcs(a.normal + 3 * q + 1, n.y); __stcs(a.normal + 3 * q + 2, n.z); }
}

__device__ __forceinline__ void ev_store_nan(const EvArgs& a, int64_t q)
{
    const float v = __int_as_float(0x7fc00000);
    ev_store(a, q, v, Vec3{v, v, v}, Vec3{v, v, v});
}

__device__ __forceinline__ bool ev_valid(float n2) { return n2 > 0.0f && n2 <= 3.0e38f; }

// Tangential part of the polynomial gradient, the normal, and the stores of one query.
__device__ __forceinline__ void ev_finish(const EvArgs& a, int64_t q, float d0, float d1, float d2, const Vec3& w, float r,
                                          float gx, float gy, float gz)
{
    const float wg = w.x * gx + w.y * gy + w.z * gz;
    const Vec3 gs{gx - w.x * wg, gy - w.y * wg, gz - w.z * wg};
    ev_store(a, q, r, gs, surface_normal(d0, d1, d2, r, gs));
}

// Up to 64 NP queries q0 + lane + 32 k < q1 of one glyph, two per pair of lanes; co: the glyph's scaled
// terms in shared memory, nb: the recurrence constants.
template <int NP>
__device__ __forceinline__ void ev_slab(const EvArgs& a, const float4* co, const float* nb, int64_t q0, int64_t q1,
                                        int lane, uint32_t& status)
{
    float2 x[NP], y[NP], z[NP], C[NP], S[NP], R[NP], gx[NP], gy[NP], gz[NP];
    bool ok[2 * NP];
    auto load = [&](int k, float& d0, float& d1, float& d2) {
        const int64_t q = q0 + lane + 32 * k;
        d0 = d1 = d2 = 0.0f;
        if (q < q1) { d0 = __ldg(a.dirs + 3 * q); d1 = __ldg(a.dirs + 3 * q + 1); d2 = __ldg(a.dirs + 3 * q + 2); }
    };
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float wx[2], wy[2], wz[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float d0, d1, d2;
            load(2 * p + h, d0, d1, d2);
            const float n2 = d0 * d0 + d1 * d1 + d2 * d2;
            ok[2 * p + h] = ev_valid(n2);
            const float il = ok[2 * p + h] ? rsqrtf(n2) : 0.0f;
            wx[h] = d0 * il; wy[h] = d1 * il; wz[h] = d2 * il;
        }
        x[p] = make_float2(wx[0], wx[1]); y[p] = make_float2(wy[0], wy[1]); z[p] = make_float2(wz[0], wz[1]);
        C[p] = bc(1.0f);
        S[p] = R[p] = gx[p] = gy[p] = gz[p] = bc(0.0f);
    }
    const int L = a.L;
    int t = 0;
    for (int M = 0; M <= L; ++M) {
        float2 p1[NP], p2[NP], U[NP], V[NP], Uz[NP], Vz[NP];
        {
            const float4 c = co[t++];  // l = M: p = 1
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                p2[p] = bc(0.0f); p1[p] = bc(1.0f);
                U[p] = bc(c.x); V[p] = bc(c.y); Uz[p] = bc(c.z); Vz[p] = bc(c.w);
            }
        }
#pragma unroll 4
        for (int l = M + 1; l <= L; ++l, ++t) {
            const float4 c = co[t];
            const float b = nb[t];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 pl = pfma(z[p], p1[p], pmul(bc(b), p2[p]));
                p2[p] = p1[p];
                p1[p] = pl;
                U[p] = pfma(bc(c.x), pl, U[p]);
                V[p] = pfma(bc(c.y), pl, V[p]);
                Uz[p] = pfma(bc(c.z), pl, Uz[p]);
                Vz[p] = pfma(bc(c.w), pl, Vz[p]);
            }
        }
        const float fm = (float)M;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (M > 0) {
                gz[p] = pfma(C[p], Uz[p], pfma(S[p], Vz[p], gz[p]));
                const float2 mU = pmul(bc(fm), U[p]), mV = pmul(bc(fm), V[p]);
                gx[p] = pfma(C[p], mU, pfma(S[p], mV, gx[p]));
                gy[p] = pfma(C[p], mV, pfma(pmul(S[p], bc(-1.0f)), mU, gy[p]));
                const float2 Cn = pfma(x[p], C[p], pmul(pmul(y[p], bc(-1.0f)), S[p]));
                S[p] = pfma(x[p], S[p], pmul(y[p], C[p]));
                C[p] = Cn;
            }
            R[p] = pfma(C[p], U[p], pfma(S[p], V[p], R[p]));
        }
    }
#pragma unroll
    for (int k = 0; k < 2 * NP; ++k) {
        const int p = k >> 1;
        const int64_t q = q0 + lane + 32 * k;
        if (q >= q1) continue;
        if (!ok[k]) {
            status |= SHM_DEV_NONFINITE;
            ev_store_nan(a, q);
            continue;
        }
        float d0, d1, d2;
        load(k, d0, d1, d2);
        const bool hi = (k & 1) != 0;
        ev_finish(a, q, d0, d1, d2, hi ? Vec3{x[p].y, y[p].y, z[p].y} : Vec3{x[p].x, y[p].x, z[p].x}, hi ? R[p].y : R[p].x,
                  hi ? gx[p].y : gx[p].x, hi ? gy[p].y : gy[p].x, hi ? gz[p].y : gz[p].x);
    }
}

// One query on glyph g (any int), a thread by itself: the coefficients are gathered, each once, and the
// derivative runs by its own recurrence.  Lanes of a warp may be on different glyphs.
__device__ __forceinline__ void ev_one(const EvArgs& a, const EvTable& T, int64_t q, int g, uint32_t& status)
{
    const int L = a.L, K = (L + 1) * (L + 1);
    const float d0 = __ldg(a.dirs + 3 * q), d1 = __ldg(a.dirs + 3 * q + 1), d2 = __ldg(a.dirs + 3 * q + 2);
    const float n2 = d0 * d0 + d1 * d1 + d2 * d2;
    bool ok = (g >= 0 && g < a.G);
    if (!ok) status |= SHM_DEV_BOUNDS;
    if (ok && !ev_valid(n2)) { ok = false; status |= SHM_DEV_NONFINITE; }
    if (!ok) {
        ev_store_nan(a, q);
        return;
    }
    const float il = rsqrtf(n2);
    const Vec3 w{d0 * il, d1 * il, d2 * il};
    const float* c = a.coeffs + (int64_t)g * K;
    float C = 1.0f, S = 0.0f, R = 0.0f, gx = 0.0f, gy = 0.0f, gz = 0.0f;
    int t = 0;
    for (int M = 0; M <= L; ++M) {
        float p1 = 1.0f, p2 = 0.0f, e1 = 0.0f, e2 = 0.0f;  // p and dp/dz of degrees l-1 and l-2
        float U = 0.0f, V = 0.0f, Uz = 0.0f, Vz = 0.0f;
        for (int l = M; l <= L; ++l, ++t) {
            float p = 1.0f, e = 0.0f;
            if (l > M) {
                const float nbt = T.nbeta[t];
                p = fmaf(w.z, p1, nbt * p2);
                e = fmaf(w.z, e1, fmaf(nbt, e2, p1));
                p2 = p1; e2 = e1;
                p1 = p; e1 = e;
            }
            const float kc = T.kc[t];
            const float cc = kc * __ldg(c + l * l + l + M), cs = kc * __ldg(c + l * l + l - M);
            U = fmaf(cc, p, U);
            V = fmaf(cs, p, V);
            Uz = fmaf(cc, e, Uz);
            Vz = fmaf(cs, e, Vz);
        }
        const float fm = (float)M;
        if (M > 0) {
            gx = fmaf(fm, C * U + S * V, gx);
            gy = fmaf(fm, C * V - S * U, gy);
            const float Cn = w.x * C - w.y * S;
            S = w.x * S + w.y * C;
            C = Cn;
        }
        R += C * U + S * V;
        gz += C * Uz + S * Vz;
    }
    ev_finish(a, q, d0, d1, d2, w, R, gx, gy, gz);
}

// Glyph of each lane's query q0 + lane, given the glyph g of q0 (0 <= g < G, seg[g] <= q0): the number of
// segment ends at or before it, counted over the next 32 ends held one per lane; a lane whose query lies
// past all 32 (runs of empty segments) searches by itself.  Every lane calls it.
__device__ __forceinline__ int ev_lane_glyph(const int64_t* seg, int G, int g, int64_t q0, int lane)
{
    const int64_t q = q0 + lane;
    const int64_t end = g + 1 + lane <= G ? __ldg(seg + g + 1 + lane) : INT64_MAX;
    int k = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
        if (__shfl_sync(0xffffffffu, end, k + s - 1) <= q) k += s;
    if (__shfl_sync(0xffffffffu, end, k) > q) return g + k;
    int lo = g + k + 1, hi = G + 1;  // seg[lo] <= q
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(seg + mid) <= q) lo = mid; else hi = mid;
    }
    return lo;
}

// Warp w of W takes queries [Q w / W, Q (w + 1) / W) and walks the glyphs they belong to.  SHORT: segments may be short
// on average.
template <bool SHORT>
__global__ void __launch_bounds__(EV_BLOCK, EV_RES) k_sh_eval_seg(EvArgs a, const __grid_constant__ EvTable T)
{
    extern __shared__ __align__(16) float4 ev_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = a.L, nt = (L + 1) * (L + 2) / 2, K = (L + 1) * (L + 1);
    float4* co = ev_smem + warp * nt;
    float* nb = reinterpret_cast<float*>(ev_smem + EV_WARPS * nt);
    for (int t = threadIdx.x; t < nt; t += EV_BLOCK) nb[t] = T.nbeta[t];
    __syncthreads();
    const int64_t W = (int64_t)gridDim.x * EV_WARPS, w = (int64_t)blockIdx.x * EV_WARPS + warp;
    const int64_t per = ((a.Q + W - 1) / W + 31) & ~(int64_t)31;
    int64_t q = w * per;
    const int64_t qe = min(a.Q, q + per);
    uint32_t status = 0;
    int g = 0;
    if (a.seg && q < qe) g = (q < __ldg(a.seg)) ? -1 : seg_find_warp(a.seg, a.G, q);
    while (q < qe) {
        int64_t e = qe;  // end of glyph g's queries within the warp's range
        if (a.seg) {
            // past empty segments to the one that holds q: by a search, or 32 ends at a time where segments are not short
            if (SHORT) {
                if (g >= 0 && g < a.G && q >= __ldg(a.seg + g + 1) && (++g < a.G) && q >= __ldg(a.seg + g + 1))
                    g = seg_find_warp(a.seg, a.G, q);
            } else if (g >= 0) {
                for (unsigned m = ~0u; m == ~0u && g < a.G; g += __popc(m))
                    m = __ballot_sync(0xffffffffu, g + 1 + lane <= a.G && __ldg(a.seg + min(g + 1 + lane, a.G)) <= q);
            }
            e = g >= a.G ? qe : min(qe, __ldg(a.seg + g + 1));
        }
        if (g < 0 || g >= a.G) {
            status |= SHM_DEV_BOUNDS;
            for (; q < e; q += 32)
                if (q + lane < e) ev_store_nan(a, q + lane);
            q = e;
            g = g < 0 ? 0 : g;
            continue;
        }
        if (SHORT && e - q < EV_SHORT) {
            // 32 queries, each lane on its own glyph
            const int gl = a.seg ? ev_lane_glyph(a.seg, a.G, g, q, lane) : g;
            if (q + lane < qe) ev_one(a, T, q + lane, gl, status);
            g = __shfl_sync(0xffffffffu, gl, 31);
            q += 32;
            continue;
        }
        const float* c = a.coeffs + (int64_t)g * K;
        __syncwarp();
        for (int t = lane, M = 0, first = 0; t < nt; t += 32) {
            while (t >= first + (L + 1 - M)) { first += L + 1 - M; ++M; }
            const int l = M + t - first, k0 = l * l + l;
            const float kc = T.kc[t], kd = T.kd[t];
            float4 v;
            v.x = kc * __ldg(c + k0 + M);
            v.y = M > 0 ? kc * __ldg(c + k0 - M) : 0.0f;
            v.z = M > 0 ? kd * __ldg(c + k0 + M - 1) : 0.0f;
            v.w = M > 1 ? kd * __ldg(c + k0 - M + 1) : 0.0f;
            co[t] = v;
        }
        __syncwarp();
        while (q < e) {
            if (e - q > 64) {
                ev_slab<2>(a, co, nb, q, e, lane, status);
                q += 128;
            } else {
                ev_slab<1>(a, co, nb, q, e, lane, status);
                q += 64;
            }
        }
        q = e;
    }
    report_status(a.dev_status, status);
}

__global__ void __launch_bounds__(EV_BLOCK) k_sh_eval_ids(EvArgs a, const __grid_constant__ EvTable T)
{
    uint32_t status = 0;
    for (int64_t q = (int64_t)blockIdx.x * EV_BLOCK + threadIdx.x; q < a.Q; q += (int64_t)gridDim.x * EV_BLOCK)
        ev_one(a, T, q, __ldg(a.glyph + q), status);
    report_status(a.dev_status, status);
}

}  // namespace

cudaError_t launch_sh_eval(int L, int G, const float* coeffs, int64_t Q, const float* dirs, const int32_t* glyph,
                           const int64_t* seg, float* R, float* grad, float* normal, int32_t* dev_status,
                           cudaStream_t s)
{
    if (Q == 0) return cudaSuccess;
    const EvTable T = make_table(L);
    const EvArgs a{L, G, coeffs, Q, dirs, glyph, seg, R, grad, normal, dev_status};
    if (glyph) {
        int64_t blocks = (Q + EV_BLOCK - 1) / EV_BLOCK;
        const int64_t cap = (int64_t)sm_count() * 16;
        if (blocks > cap) blocks = cap;
        k_sh_eval_ids<<<(unsigned)blocks, EV_BLOCK, 0, s>>>(a, T);
        return cudaGetLastError();
    }
    const int nt = (L + 1) * (L + 2) / 2;
    const int smem = EV_WARPS * nt * 16 + nt * 4;
    // at least 32 queries per warp, at most one resident wave of warps
    int64_t blocks = (Q + 32 * EV_WARPS - 1) / (32 * EV_WARPS);
    const int64_t cap = (int64_t)sm_count() * EV_RES;
    if (blocks > cap) blocks = cap;
    // (the lanes' path costs the other 1.7 %, in registers and scheduling, where it is not taken)
    if (seg && Q < 64LL * G) k_sh_eval_seg<true><<<(unsigned)blocks, EV_BLOCK, smem, s>>>(a, T);
    else k_sh_eval_seg<false><<<(unsigned)blocks, EV_BLOCK, smem, s>>>(a, T);
    return cudaGetLastError();
}

}  // namespace shm
