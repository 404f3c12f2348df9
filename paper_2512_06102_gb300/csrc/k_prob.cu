// k_prob.cu -- per-(cell, direction) ignition tables (Section 3, Eqs. 1-4)
// and their parameter gradient.
//
// k_prob_table: for a target cell v and the 8 incoming directions d (source u =
// v - Delta_d),
//   r[v][d] = gamma(v) * phi(u, d),   q[v][d] = 1 - exp(-r[v][d])
// with phi from Eq. 3 (wind Eq. 1 and slope Eq. 2 taken at the source) and
// gamma the target's susceptibility.  A CTA takes a tile of cells: the slope part
// once for each edge between two cells, then a thread a cell.  Bound by FP32
// issue (75% active), not by the 32 B of q (and 32 B of r) a cell.
//
// k_rates_bwd: dL/dtheta = sum_t sum_{v,d} glam_t(v) pb_t(v - Delta_d) dr[v][d]/dtheta,
// every derivative written without division so that classes with no fuel
// (mu_den = -1) are exact.  Deterministic: per-block FP64 partials, summed in
// a fixed order by the last block to finish.
#include <math.h>

#include <algorithm>
#include <cmath>

#include "jwf_internal.cuh"
#include "rate_model.cuh"

namespace {

struct DirConst {
    float cphi[8], sphi[8], inv_len[8];
};

__device__ __forceinline__ DirConst dir_const() {
    const float h = 0.70710678118654752f;   // sqrt(2)/2
    DirConst k = {{1.f, h, 0.f, -h, -1.f, -h, 0.f, h},
                  {0.f, h, 1.f, h, 0.f, -h, -1.f, -h},
                  {1.f, h, 1.f, h, 1.f, h, 1.f, h}};
    return k;
}

// Shape of one directional factor: E = alpha_w1 V + alpha_w2 V (cos - 1) + alpha_s S.
struct RateTerms {
    float S;        // slope in degrees (Eq. 2)
    float cosm1;    // cos(phi_d - Theta) - 1
    float V;        // wind speed at the source
    float K;        // exp(E)
};

__device__ __forceinline__ RateTerms rate_terms(const JwfDevParams& P, float z_src, float z_dst,
                                                float V, float cth, float sth, float cphi,
                                                float sphi, float inv_len, float slope_scale) {
    RateTerms t;
    const float x = (z_dst - z_src) * inv_len;              // rise over run
    t.S = atanf(x) * slope_scale;                           // degrees
    const float cosd = cphi * cth + sphi * sth;             // cos(phi_d - Theta)
    t.cosm1 = cosd - 1.0f;
    t.V = V;
    const float E = P.alpha_w1 * V + P.alpha_w2 * V * t.cosm1 + P.alpha_s * t.S;
    t.K = expf(E);
    return t;
}

// sin and cos of d pi/8, d = 0..7, in double (made on the host)
struct WindTrig {
    double s[8], c[8];
};

__global__ void k_wind_exponent(int32_t N, const float* __restrict__ ws, const float* __restrict__ wd,
                                double alpha_w1, double alpha_w2, const WindTrig T, float2* __restrict__ wexp) {
    // alpha_w1 V + alpha_w2 V (cos(d pi/4 - Theta) - 1) per env and direction, in
    // double (cos - 1 written as -2 sin^2 to avoid cancellation), split hi + lo.
    // One thread an env: sin(d pi/8 - Theta/2) = sin(d pi/8) cos(Theta/2) -
    // cos(d pi/8) sin(Theta/2), so one sincos serves the eight directions.
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N) return;
    const double V = (double)ws[e];
    double sh, ch;
    sincos(0.5 * (double)wd[e], &sh, &ch);
    float2* out = wexp + (int64_t)e * 8;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const double s = T.s[d] * ch - T.c[d] * sh;
        const double w = alpha_w1 * V + alpha_w2 * V * (-2.0 * s * s);
        const float hi = (float)w;
        out[d] = make_float2(hi, (float)(w - (double)hi));
    }
}

static WindTrig wind_trig() {
    WindTrig T;
    const double pi = 3.14159265358979323846;
    for (int d = 0; d < 8; ++d) {
        T.s[d] = std::sin(d * pi / 8.0);
        T.c[d] = std::cos(d * pi / 8.0);
    }
    T.c[4] = 0.0;       // cos(pi/2) exactly
    return T;
}

// Table tiles: up to kPtCells target cells, rows x columns by the grid's shape
// (jwf_table_tiles), staged with a one-cell ring.  An edge between two cells is met twice, once from each side, with
// opposite signs of the elevation difference; every step of the slope's
// exponent (difference, product, atan, product) is odd bit for bit, so it is
// evaluated once per edge (directions 0..3 of the cells of the tile, of the
// row above and of the columns left and right) and read negated from the
// other side.
constexpr int kPtT = 256;
constexpr int kPtRing = JWF_PT_RING;                       // most cells of a tile with its ring
constexpr int kPtNone = 255;                               // class of a ring cell outside the grid
struct ProbSmem {
    RateConsts K;
    df wexp[8];                                            // the env's wind exponents
    float z[kPtRing];
    df S[4][kPtRing];                                      // slope part of the exponent, [direction][edge target]
    uint8_t cl[kPtRing];
};
// per-cell wind: sin and cos of half the wind direction at the source as
// double-floats, and its speed
struct ProbWindSmem {
    df sh[kPtRing], ch[kPtRing];
    float V[kPtRing];
};
// sin and cos of d pi/8 and the wind coefficients as double-floats (made on the host)
struct WindTrigF {
    df s[8], c[8];
    df a1, m2a2;                                           // alpha_w1, -2 alpha_w2
};

// alpha_w1 V + alpha_w2 V (cos(d pi/4 - Theta) - 1) at a source with its own
// wind, in double-floats: cos - 1 = -2 s^2, s = sin(d pi/8 - Theta/2) by the
// addition theorem (absolute error of s below 1e-13, as much in the exponent;
// the rates' error against 64 bits, 5.8e-8 to 6.2e-8 over grids of 20 x 33 to 512
// x 400, is the one with a double sine a direction, which took 50 FP64
// operations each on two FP64 lanes an SM)
__device__ __forceinline__ df wind_exponent_cell(df sh, df ch, float V, int d, const WindTrigF& T) {
    const df s = df_add(df_mul(T.s[d], ch), df_neg(df_mul(T.c[d], sh)));
    return df_mul({V, 0.f}, df_add(T.a1, df_mul(T.m2a2, df_mul(s, s))));
}

// Floor: 5 B in and 64 B out a cell (table with rates).  Instruction bound:
// the double-float slope and the two exponentials of eight directions.  1024
// grids of 128 x 128 with rates: one thread a cell, every edge from both sides,
// indices and terrain from global memory 1036 us; an edge once 867; and without
// branches between the directions (40 -> 63 registers) 703 us, 1.5 TB/s.
template <bool CELL_WIND>
__global__ void __launch_bounds__(kPtT, CELL_WIND ? 3 : 4)
k_prob_table(const int4* __restrict__ tiles, int64_t n_tiles, const int32_t* __restrict__ Hs,
             const int32_t* __restrict__ Ws, const int64_t* __restrict__ offs,
             const uint8_t* __restrict__ cls, const float* __restrict__ dem,
             const float* __restrict__ ws, const float* __restrict__ wd,
             const float2* __restrict__ wexp, const RateConsts K, const WindTrigF T, float* __restrict__ q,
             float* __restrict__ r) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ProbSmem& S = *reinterpret_cast<ProbSmem*>(smem_raw);
    ProbWindSmem& Sw = *reinterpret_cast<ProbWindSmem*>(smem_raw + (sizeof(ProbSmem) + 15) / 16 * 16);
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(sizeof(RateConsts) / 4); i += kPtT)
        reinterpret_cast<float*>(&S.K)[i] = reinterpret_cast<const float*>(&K)[i];
    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const int4 tl = tiles[ti];
        const int e = tl.x, y0 = tl.y, x0 = tl.z;
        const int H = Hs[e], W = Ws[e];
        const int64_t off = offs[e];
        const int th = min(tl.w >> 16, H - y0), tw = min(tl.w & 0xffff, W - x0);
        const int P = tw + 2;
        // i / n for the row lengths of this tile, by a multiply-high with the rounded-up reciprocal
        const uint32_t m_ring = 0xffffffffu / (uint32_t)(tw + 2) + 1u;
        __syncthreads();                                   // the previous tile has been read
        for (int i = tid; i < (th + 2) * (tw + 2); i += kPtT) {
            const int ry = (int)__umulhi((uint32_t)i, m_ring), rx = i - ry * (tw + 2);
            const int y = y0 - 1 + ry, x = x0 - 1 + rx;
            const int j = i;
            if (y < 0 || y >= H || x < 0 || x >= W) {
                S.cl[j] = kPtNone;
                continue;
            }
            const int64_t u = off + (int64_t)y * W + x;
            S.cl[j] = cls[u];
            S.z[j] = dem[u];
            if constexpr (CELL_WIND) {
                double sh, ch;
                sincos(0.5 * (double)wd[u], &sh, &ch);
                const float shh = (float)sh, chh = (float)ch;
                Sw.sh[j] = {shh, (float)(sh - (double)shh)};
                Sw.ch[j] = {chh, (float)(ch - (double)chh)};
                Sw.V[j] = ws[u];
            }
        }
        if (!CELL_WIND && tid < 8) {
            const float2 w2 = wexp[(int64_t)e * 8 + tid];
            S.wexp[tid] = {w2.x, w2.y};
        }
        __syncthreads();
        // edges: target (row ry of the ring's rows 0..th, any ring column), source at target - Delta_d
        for (int i = tid; i < (th + 1) * (tw + 2); i += kPtT) {
            const int ry = (int)__umulhi((uint32_t)i, m_ring), rx = i - ry * (tw + 2);
            const int j = i;
            const int cv = S.cl[j];
            const float zv = S.z[j];
            if (cv == kPtNone) continue;
            // without a branch between the four, so that their chains overlap:
            // an edge that is not there takes the cell itself for its source
            // (its entry is never read)
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const int sx = rx - jwf_dx(d);
                const bool in = sx >= 0 && sx < tw + 2;
                const int u = in ? (ry - jwf_dr(d)) * P + sx : j;
                const df slope = atan_df(df_mul(two_sum(zv, -S.z[u]), S.K.inv_run[d]), S.K);
                S.S[d][j] = df_mul(S.K.slope_coef, slope);
            }
        }
        __syncthreads();
        const uint32_t m_tile = tw == 1 ? 0u : 0xffffffffu / (uint32_t)tw + 1u;
        for (int i = tid; i < th * tw; i += kPtT) {
            const int ty = tw == 1 ? i : (int)__umulhi((uint32_t)i, m_tile), tx = i - ty * tw;
            const int j = (ty + 1) * P + tx + 1;
            const int cv = S.cl[j];
            float rr[8], qq[8];
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                // (no branch: a warp's cells seldom agree on one, and the
                // directions' chains overlap without)
                const int u = j - jwf_dr(d) * P - jwf_dx(d);
                const int cu = S.cl[u];
                const float G = cu != kPtNone ? S.K.G[cv][cu] : 0.f;
                const df sl = d < 4 ? S.S[d][j] : df_neg(S.S[d & 3][u]);
                df wx;
                if constexpr (CELL_WIND)
                    wx = wind_exponent_cell(Sw.sh[u], Sw.ch[u], Sw.V[u], d, T);
                else
                    wx = S.wexp[d];
                const float rate = rate_from(G, df_add(wx, sl));
                rr[d] = G != 0.f ? rate : 0.f;             // no fuel at the source or the target
                qq[d] = G != 0.f ? prob_of(rate) : 0.f;
            }
            const int64_t v = off + (int64_t)(y0 + ty) * W + x0 + tx;
            float4* q4 = reinterpret_cast<float4*>(q + v * 8);
            q4[0] = make_float4(qq[0], qq[1], qq[2], qq[3]);
            q4[1] = make_float4(qq[4], qq[5], qq[6], qq[7]);
            if (r != nullptr) {
                float4* r4 = reinterpret_cast<float4*>(r + v * 8);
                r4[0] = make_float4(rr[0], rr[1], rr[2], rr[3]);
                r4[1] = make_float4(rr[4], rr[5], rr[6], rr[7]);
            }
        }
    }
}

// Diagnostics of the step kernels' two-level probability (below_prob): for
// each tuple i (target and source class, elevations, wind part of the
// exponent as hi + lo, direction), out[3i .. 3i+2] = p_f, its bound B and the
// double-float probability.
__global__ void k_prob_check(int64_t n, const uint8_t* __restrict__ cv, const uint8_t* __restrict__ cu,
                             const float* __restrict__ zv, const float* __restrict__ zu,
                             const float2* __restrict__ wexp, const int32_t* __restrict__ dir, const RateConsts K,
                             float* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int d = dir[i] & 7;
        const float G = K.G[cv[i] & 15][cu[i] & 15];
        const float2 w2 = wexp[i];
        float B = 0.f;
        const float pf = prob_fast(G, zv[i], zu[i], w2.x, d, rate_view(K, K), &B);
        out[3 * i] = pf;
        out[3 * i + 1] = B;
        out[3 * i + 2] = G == 0.f ? 0.f : prob_of(rate_of(G, zv[i], zu[i], {w2.x, w2.y}, d, K));
    }
}

constexpr int kRbThreads = 256;
constexpr int kRbScalars = 5;   // p_base, alpha_w1, alpha_w2, alpha_s, alpha_gamma

// Rate adjoint of a block of steps, on 2-D tiles:
//   gr[v][d] += sum_t glam_t(v) pb_t(v - Delta_d),  pb = (1 - m) p_burn,
// each thread summing four rows of a column over the steps in registers (in
// step order; a cell without a burning neighbour would add exact zeros and is
// passed over) and updating gr once, unless all its sums are zero.  The p_burn
// and mask (tile and a one-cell halo, zero outside the grid) and glam (tile) of
// the next two steps are copied to shared memory while a step is summed.
//
// With ab (the incoming dL/dp_burn of the steps, only read where pb is not 0)
// also gpc += sum_t sum_v ab_t(v) pb_t(v): the warps first take a pass of the
// column sweeps each (two steps, or an odd count's last), a lane a column of 32
// rows, adding in float in the sweeps' order (the later step a row ahead of the
// earlier), the columns in double.  Tiles are 32 x 32 then, else the relaxed
// step's 16 x 64 (whose rows take fewer sectors).
constexpr int kAccT = 256;
constexpr int kAccCPT = 4;                                     // rows a thread
constexpr int kAccStages = 3;
template <bool GPC>
struct AccTile {
    static constexpr int Rows = GPC ? JWF_AT_ROWS : JWF_RT_ROWS, Cols = GPC ? JWF_AT_COLS : JWF_RT_COLS;
    static constexpr int W = Cols + 2, N = (Rows + 2) * W;     // tile + 1: p_burn
    static constexpr int PbPT = (N + kAccT - 1) / kAccT;       // of which a thread copies
};
static_assert(JWF_AT_ROWS * JWF_AT_COLS == kAccT * kAccCPT && JWF_RT_ROWS * JWF_RT_COLS == kAccT * kAccCPT, "tile size");
static_assert(JWF_AT_ROWS == JWF_SW_ROWS && JWF_AT_ROWS == JWF_SW2_ROWS && JWF_AT_COLS == 32,
              "a warp's chain is a sweep's strip");
// a step's staged planes; the mask's only when the accumulation has masks
template <bool MASKED, bool GPC>
struct AccStage {
    float pb[AccTile<GPC>::N], m[MASKED ? AccTile<GPC>::N : 1];
    float gl[kAccT * kAccCPT];
};

// A thread's share of a step's copies, the same every step: its elements of
// the p_burn window (tile + one-cell halo) and of the glam tile, as offsets
// from the tile's first cell (halo offsets are negative; kAccOut outside the
// grid).
constexpr int32_t kAccOut = INT32_MIN;
template <bool GPC>
struct AccPlan {
    int32_t pb[AccTile<GPC>::PbPT];
    int32_t gl[kAccCPT];
};

template <bool GPC>
__device__ __forceinline__ void acc_plan(AccPlan<GPC>& pl, int y0, int x0, int H, int W) {
    using A = AccTile<GPC>;
#pragma unroll
    for (int k = 0; k < A::PbPT; ++k) {
        const int i = (int)threadIdx.x + k * kAccT;
        const int y = y0 - 1 + i / A::W, x = x0 - 1 + i % A::W;
        pl.pb[k] = (i < A::N && y >= 0 && y < H && x >= 0 && x < W) ? (y - y0) * W + (x - x0) : kAccOut;
    }
#pragma unroll
    for (int k = 0; k < kAccCPT; ++k) {
        const int i = (int)threadIdx.x + k * kAccT;
        const int y = y0 + i / A::Cols, x = x0 + i % A::Cols;
        pl.gl[k] = (y < H && x < W) ? (y - y0) * W + (x - x0) : kAccOut;
    }
}

// copies of one step: t0 = the global index of the tile's first cell in that step's planes
template <bool MASKED, bool GPC>
__device__ __forceinline__ void acc_stage(AccStage<MASKED, GPC>& b, const AccPlan<GPC>& pl, int64_t t0,
                                          const float* __restrict__ glam, const float* __restrict__ pburn,
                                          const float* __restrict__ mask) {
    using A = AccTile<GPC>;
#pragma unroll
    for (int k = 0; k < A::PbPT; ++k) {
        const int i = (int)threadIdx.x + k * kAccT;
        if (i >= A::N) break;
        if (pl.pb[k] == kAccOut) {
            b.pb[i] = 0.f;
            if constexpr (MASKED) b.m[i] = 0.f;
            continue;
        }
        const int64_t u = t0 + pl.pb[k];
        jwf_cp_async4(&b.pb[i], pburn + u);
        if constexpr (MASKED) {
            if (mask != nullptr)
                jwf_cp_async4(&b.m[i], mask + u);
            else
                b.m[i] = 0.f;
        }
    }
#pragma unroll
    for (int k = 0; k < kAccCPT; ++k)
        if (pl.gl[k] != kAccOut) jwf_cp_async4(&b.gl[(int)threadIdx.x + k * kAccT], glam + t0 + pl.gl[k]);
}

constexpr int kGpcRows = 4;                                    // rows of a chain loaded at once

// sum of ab pb over column x0 + lane of the tile and the steps of pass ps
template <bool MASKED>
__device__ __forceinline__ float gpc_chain(int ps, int n_steps, int64_t cells, int64_t tile0, int rows, int W,
                                           const float* __restrict__ pburn, const float* __restrict__ mask,
                                           const float* __restrict__ ab, int lane) {
    const int t0 = 2 * ps;
    const bool two = t0 + 1 < n_steps;
    const int64_t ou = (int64_t)(two ? t0 + 1 : t0) * cells + tile0 + lane;       // the later step
    const int64_t ow = (int64_t)t0 * cells + tile0 + lane;                        // the earlier one
    float s = 0.f, pw = 0.f, aw = 0.f;
    for (int y = 0; y < rows; y += kGpcRows) {
        float pu[kGpcRows], au[kGpcRows], pv[kGpcRows], av[kGpcRows];
#pragma unroll
        for (int k = 0; k < kGpcRows; ++k) {
            const int64_t o = (int64_t)(y + k) * W;
            pu[k] = pv[k] = 0.f;
            if (y + k < rows) {
                pu[k] = pburn[ou + o];
                if (MASKED) pu[k] *= 1.0f - mask[ou + o];
                if (two) {
                    pv[k] = pburn[ow + o];
                    if (MASKED) pv[k] *= 1.0f - mask[ow + o];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kGpcRows; ++k) {
            const int64_t o = (int64_t)(y + k) * W;
            au[k] = pu[k] != 0.f ? ab[ou + o] : 0.f;
            av[k] = pv[k] != 0.f ? ab[ow + o] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kGpcRows; ++k) {
            if (pu[k] != 0.f) s = __fmaf_rn(au[k], pu[k], s);
            if (pw != 0.f) s = __fmaf_rn(aw, pw, s);
            pw = pv[k];
            aw = av[k];
        }
    }
    if (pw != 0.f) s = __fmaf_rn(aw, pw, s);
    return s;
}

template <bool MASKED, bool GPC>
__global__ void __launch_bounds__(kAccT, MASKED ? 3 : 4)
k_rates_accumulate(const int4* __restrict__ tiles, int64_t n_tiles, const int32_t* __restrict__ Hs,
                   const int32_t* __restrict__ Ws, const int64_t* __restrict__ offs, int64_t cells, int32_t n_steps,
                   const float* __restrict__ glam, const float* __restrict__ pburn,
                   const float* __restrict__ mask, float* __restrict__ gr, const float* __restrict__ ab,
                   double* __restrict__ partials, uint32_t* __restrict__ counter, double* __restrict__ gpc) {
    using A = AccTile<GPC>;
    __shared__ __align__(16) AccStage<MASKED, GPC> st[kAccStages];
    const int tx = (int)threadIdx.x % A::Cols, ty = (int)threadIdx.x / A::Cols;
    double acc = 0.0;
    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const int4 tl = tiles[ti];
        const int e = tl.x, y0 = tl.y, x0 = tl.z;
        const int H = Hs[e], W = Ws[e];
        const int64_t off = offs[e];
        AccPlan<GPC> pl;
        acc_plan(pl, y0, x0, H, W);
        const int64_t tile0 = off + (int64_t)y0 * W + x0;
        __syncthreads();                   // the previous tile has been read
        for (int t = 0; t < kAccStages - 1; ++t) {
            if (t < n_steps) acc_stage(st[t], pl, (int64_t)t * cells + tile0, glam, pburn, mask);
            jwf_cp_async_commit();
        }
        if constexpr (GPC) {
            if (x0 + tx < W)
                for (int ps = ty; ps < (n_steps + 1) / 2; ps += kAccT / 32)
                    acc += (double)gpc_chain<MASKED>(ps, n_steps, cells, tile0, min(A::Rows, H - y0), W, pburn, mask,
                                                     ab, tx);
        }
        float w[kAccCPT][8];
#pragma unroll
        for (int k = 0; k < kAccCPT; ++k)
#pragma unroll
            for (int d = 0; d < 8; ++d) w[k][d] = 0.f;
        int cur = 0;
        for (int t = 0; t < n_steps; ++t) {
            jwf_cp_async_wait_prev();      // step t has landed (the next one may be in flight)
            if constexpr (MASKED) {
                // each thread masks the elements it fetched
                AccStage<MASKED, GPC>& m = st[cur];
                if (mask != nullptr) {
#pragma unroll
                    for (int k = 0; k < A::PbPT; ++k) {
                        const int i = (int)threadIdx.x + k * kAccT;
                        if (i < A::N) m.pb[i] *= 1.0f - m.m[i];
                    }
                }
            }
            __syncthreads();               // and every thread is past step t - 1, whose stage is free
            const int nxt = cur == 0 ? kAccStages - 1 : cur - 1;
            if (t + kAccStages - 1 < n_steps)
                acc_stage(st[nxt], pl, (int64_t)(t + kAccStages - 1) * cells + tile0, glam, pburn, mask);
            jwf_cp_async_commit();
            const AccStage<MASKED, GPC>& b = st[cur];
            cur = cur + 1 == kAccStages ? 0 : cur + 1;
            const float* c = &b.pb[(ty * kAccCPT + 1) * A::W + tx + 1];
            float a0 = c[-A::W - 1], a1 = c[-A::W], a2 = c[-A::W + 1], b0 = c[-1], b1 = c[0], b2 = c[1];
#pragma unroll
            for (int k = 0; k < kAccCPT; ++k) {
                const float c0 = c[(k + 1) * A::W - 1], c1 = c[(k + 1) * A::W], c2 = c[(k + 1) * A::W + 1];
                const float src[8] = {b0, c0, c1, c2, b2, a2, a1, a0};
                uint32_t bits = __float_as_uint(b0) | __float_as_uint(c0) | __float_as_uint(c1) | __float_as_uint(c2) |
                                __float_as_uint(b2) | __float_as_uint(a2) | __float_as_uint(a1) | __float_as_uint(a0);
                const float* gl = &b.gl[(ty * kAccCPT + k) * A::Cols + tx];
                // (a caller's glam may be infinite or NaN, whose product with 0 is
                // not 0; the on-chip adjoint's is saturated)
                if constexpr (!GPC) bits |= (__float_as_uint(*gl) & 0x7f800000u) == 0x7f800000u ? 1u : 0u;
                if (bits != 0u) {
                    const float g = *gl;
#pragma unroll
                    for (int d = 0; d < 8; ++d) w[k][d] += g * src[d];
                }
                a0 = b0; a1 = b1; a2 = b2;
                b0 = c0; b1 = c1; b2 = c2;
            }
        }
        bool any = false;
#pragma unroll
        for (int k = 0; k < kAccCPT; ++k)
#pragma unroll
            for (int d = 0; d < 8; ++d) any = any || w[k][d] != 0.f;
        if (!any) continue;
#pragma unroll
        for (int k = 0; k < kAccCPT; ++k) {
            const int y = y0 + ty * kAccCPT + k, x = x0 + tx;
            if (y >= H || x >= W) continue;
            float4* g4 = reinterpret_cast<float4*>(gr + (off + (int64_t)y * W + x) * 8);
            float4 a = g4[0], c = g4[1];
            a.x += w[k][0]; a.y += w[k][1]; a.z += w[k][2]; a.w += w[k][3];
            c.x += w[k][4]; c.y += w[k][5]; c.z += w[k][6]; c.w += w[k][7];
            g4[0] = a;
            g4[1] = c;
        }
    }
    if constexpr (GPC) {
        // deterministic reduction: per-CTA sums, added in order by the last CTA
        __shared__ double red[kAccT / 32];
        __shared__ bool am_last;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (tx == 0) red[ty] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int i = 0; i < kAccT / 32; ++i) s += red[i];
            partials[blockIdx.x] = s;
            __threadfence();
            am_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
        }
        __syncthreads();
        if (!am_last) return;
        __threadfence();
        double s = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += kAccT) s += __ldcg(&partials[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (tx == 0) red[ty] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double tot = 0.0;
            for (int i = 0; i < kAccT / 32; ++i) tot += red[i];
            *gpc += tot;
            *counter = 0u;
        }
    }
}

// a + b as float plus the rounding errors of the sum (|lo| stays far below
// |hi|'s last bit times the number of terms: about 2^-46 relative)
__device__ __forceinline__ df sum_add(df a, df b) {
    const df t = two_sum(a.hi, b.hi);
    return {t.hi, __fadd_rn(t.lo, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ df warp_sum(df s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s = sum_add(s, {__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)});
    return s;
}

// Parameter gradient through the rates.  Per target cell v and direction d
// (source u = v - Delta_d), w = gr[v][d] is the adjoint of r(v, d); with
// r = gamma(v) phi(u, d),
//   dr/dp_base = gamma A_u K,   dr/dalpha_gamma = A_v phi,
//   dr/dalpha_w1 = r V,  dr/dalpha_w2 = r V (cos - 1),  dr/dalpha_s = r S,
//   dr/dmu_veg[k] = (1 + mu_den[k]) B_k,  dr/dmu_den[k] = (1 + mu_veg[k]) B_k,
// where B_k gathers alpha_gamma phi (target of class k) and gamma p_base K
// (source of class k); no division, so classes without fuel are exact.
// Each thread sums its cells in float (a few dozen terms); the class bins sit
// in shared memory, one column per thread (class-major, conflict-free); the
// block and the grid are reduced in a fixed order (the last block to finish
// adds the per-block partials in double), so the result is deterministic.  A warp
// sums a value, in double-floats: in double, one value after the other with a
// barrier a level of a tree, the reduction was most of the kernel's time (two
// FP64 lanes an SM, and a chain of 27 x 4 loads in the last block: relaxed rollout
// of 64 grids of 150 x 117, 12 steps, 1156 us, now 1024; the gradient differs by
// 1e-15 of its norm).
template <int C>
__global__ void __launch_bounds__(kRbThreads)
k_rates_bwd(const int2* __restrict__ tiles, int64_t n_tiles, const int32_t* __restrict__ Hs,
            const int32_t* __restrict__ Ws, const int64_t* __restrict__ offs, int64_t cells,
            const float* __restrict__ gr, const uint8_t* __restrict__ cls,
            const float* __restrict__ dem, const float* __restrict__ ws,
            const float* __restrict__ wd, int per_cell_wind, const JwfDevParams P,
            double* __restrict__ partials, uint32_t* __restrict__ counter,
            double* __restrict__ gparams) {
    constexpr int NV = kRbScalars + 2 * C;
    __shared__ float bins[C * kRbThreads];
    __shared__ float scal[kRbScalars * kRbThreads];
    __shared__ bool am_last;
    const int tid = threadIdx.x;
    for (int k = 0; k < C; ++k) bins[k * kRbThreads + tid] = 0.f;
    float g_pb = 0.f, g_w1 = 0.f, g_w2 = 0.f, g_s = 0.f, g_gam = 0.f;
    const DirConst dc = dir_const();
    const float slope_scale = 57.295779513082320876f;
    const float inv_cell = 1.0f / P.cell_size;

    for (int64_t ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
        const int2 tile = tiles[ti];
        const int e = tile.x;
        const int W = Ws[e], H = Hs[e];
        const int local = tile.y + tid;
        if (local >= H * W) continue;
        const int64_t off = offs[e];
        const int y = local / W, x = local - (local / W) * W;
        const int64_t v = off + local;
        const float4* g4 = reinterpret_cast<const float4*>(gr + v * 8);
        const float4 ga = __ldg(g4), gb = __ldg(g4 + 1);
        const float w[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
        const int cv = cls[v];
        const float zv = dem[v];
        const float Av = (1.0f + P.mu_veg[cv]) * (1.0f + P.mu_den[cv]);
        const float gamma = P.alpha_gamma * Av;
        float cth = 0.f, sth = 0.f, Venv = 0.f;
        if (!per_cell_wind) {
            Venv = ws[e];
            sincosf(wd[e], &sth, &cth);
        }
        float tgt = 0.f;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            if (w[d] == 0.f) continue;
            const int uy = y - jwf_dr(d), ux = x - jwf_dx(d);
            if (uy < 0 || uy >= H || ux < 0 || ux >= W) continue;
            const int64_t u = off + (int64_t)uy * W + ux;
            const int cu = cls[u];
            float V = Venv, c = cth, s = sth;
            if (per_cell_wind) {
                V = ws[u];
                sincosf(wd[u], &s, &c);
            }
            const RateTerms t = rate_terms(P, dem[u], zv, V, c, s, dc.cphi[d], dc.sphi[d],
                                           dc.inv_len[d] * inv_cell, slope_scale);
            const float Au = (1.0f + P.mu_veg[cu]) * (1.0f + P.mu_den[cu]);
            const float phi = P.p_base * Au * t.K;
            const float wr = w[d] * gamma * phi;
            g_pb += w[d] * gamma * Au * t.K;
            g_w1 += wr * t.V;
            g_w2 += wr * t.V * t.cosm1;
            g_s += wr * t.S;
            g_gam += w[d] * Av * phi;
            tgt += w[d] * phi;
            bins[cu * kRbThreads + tid] += w[d] * gamma * P.p_base * t.K;   // source of class cu
        }
        if (tgt != 0.f) bins[cv * kRbThreads + tid] += P.alpha_gamma * tgt;  // target of class cv
    }
    // block reduction: warp w sums the threads' values i = w, w + 8, ..
    scal[tid] = g_pb;
    scal[kRbThreads + tid] = g_w1;
    scal[2 * kRbThreads + tid] = g_w2;
    scal[3 * kRbThreads + tid] = g_s;
    scal[4 * kRbThreads + tid] = g_gam;
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll 1
    for (int i = warp; i < NV; i += kRbThreads / 32) {
        // i < 5: a scalar; then mu_veg and mu_den of class k
        const int k = i < kRbScalars ? 0 : (i - kRbScalars) % C;
        const float* src = i < kRbScalars ? &scal[i * kRbThreads] : &bins[k * kRbThreads];
        const float f = i < kRbScalars ? 1.0f : 1.0f + (i - kRbScalars < C ? P.mu_den[k] : P.mu_veg[k]);
        df s = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < kRbThreads / 32; ++j) s = sum_add(s, {__fmul_rn(src[j * 32 + lane], f), 0.f});
        s = warp_sum(s);
        double g = (double)s.hi + (double)s.lo;
        if (!isfinite(s.hi)) {                     // out of float's range: once more in double
            g = 0.0;
            for (int j = 0; j < kRbThreads / 32; ++j) g += (double)__fmul_rn(src[j * 32 + lane], f);
            for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        }
        if (lane == 0) partials[(int64_t)blockIdx.x * NV + i] = g;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) am_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    // the last block sums the block partials in a fixed order
    const int nC = P.n_classes;
#pragma unroll 1
    for (int i = warp; i < NV; i += kRbThreads / 32) {
        double g = 0.0;
#pragma unroll 4
        for (int b = lane; b < (int)gridDim.x; b += 32) g += __ldcg(&partials[(int64_t)b * NV + i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (lane == 0) {
            // layout [p_base, alpha_w1, alpha_w2, alpha_s, alpha_gamma, mu_veg[nC], mu_den[nC]]
            if (i < kRbScalars) {
                gparams[i] += g;
            } else if (i < kRbScalars + C) {
                if (i - kRbScalars < nC) gparams[i] += g;
            } else {
                const int k = i - kRbScalars - C;
                if (k < nC) gparams[kRbScalars + nC + k] += g;
            }
        }
    }
    if (tid == 0) *counter = 0u;
}

template <int C>
cudaError_t launch_rates_contract_c(jwf_ctx* c, const float* gr, const uint8_t* cls, const float* dem,
                                    const float* ws, const float* wd, double* gparams, cudaStream_t s) {
    constexpr int NV = kRbScalars + 2 * C;
    int64_t grid = (int64_t)c->num_sms * 6;
    if (grid > c->n_tiles) grid = c->n_tiles;
    if (grid * NV > c->partial_cap) grid = c->partial_cap / NV;
    if (grid < 1) return cudaErrorInvalidValue;
    k_rates_bwd<C><<<(unsigned)grid, kRbThreads, 0, s>>>(
        c->d_tiles, c->n_tiles, c->d_H, c->d_W, c->d_off, c->cells, gr, cls, dem, ws, wd,
        (c->flags & JWF_WIND_PER_CELL) ? 1 : 0, c->P, c->d_partials, c->d_red_counter, gparams);
    return cudaGetLastError();
}

}  // namespace

static df split_df(double v) {
    const float hi = (float)v;
    return {hi, (float)(v - (double)hi)};
}

void jwf_make_rate_consts(jwf_ctx* c) {
    const double pi = 3.14159265358979323846;
    RateConsts* K = &c->K;
    *K = RateConsts{};
    for (int k = 0; k <= 64; ++k) {
        const double th = k * pi / 256.0;
        K->atan_th[k] = split_df(th);
        K->atan_tan[k] = split_df(std::tan(th));
    }
    K->half_pi = split_df(pi / 2.0);
    K->slope_coef = split_df((double)c->P.alpha_s * 180.0 / pi);
    for (int d = 0; d < 8; ++d)
        K->inv_run[d] = split_df(1.0 / ((double)c->P.cell_size * ((d & 1) ? std::sqrt(2.0) : 1.0)));
    for (int a = 0; a < 16; ++a)
        for (int b = 0; b < 16; ++b) {
            if (a >= c->n_classes || b >= c->n_classes) {
                K->G[a][b] = 0.f;
                continue;
            }
            const double gamma = (double)c->P.alpha_gamma * (1.0 + (double)c->P.mu_veg[a]) *
                                 (1.0 + (double)c->P.mu_den[a]);
            const double base = (double)c->P.p_base * (1.0 + (double)c->P.mu_veg[b]) *
                                (1.0 + (double)c->P.mu_den[b]);
            K->G[a][b] = (float)(gamma * base);
        }
}

cudaError_t jwf_launch_prob_check(const jwf_ctx* c, int64_t n, const uint8_t* cv, const uint8_t* cu,
                                  const float* zv, const float* zu, const float* wexp, const int32_t* dir,
                                  float* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const RateConsts& K = c->K;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)c->num_sms * 8);
    k_prob_check<<<(unsigned)blocks, 256, 0, s>>>(n, cv, cu, zv, zu, reinterpret_cast<const float2*>(wexp), dir, K,
                                                   out);
    return cudaGetLastError();
}

cudaError_t jwf_launch_wind_exponent(const jwf_ctx* c, const float* ws, const float* wd, cudaStream_t s) {
    k_wind_exponent<<<(c->N + 127) / 128, 128, 0, s>>>(c->N, ws, wd, (double)c->P.alpha_w1,
                                                         (double)c->P.alpha_w2, wind_trig(), c->d_wexp);
    return cudaGetLastError();
}

cudaError_t jwf_launch_wind_series(jwf_ctx* c, cudaStream_t s) {
    // the series is [steps][N]: the same kernel over steps x N "envs"
    const int64_t n = (int64_t)c->wser_n * c->N;
    if (n == 0) return cudaSuccess;
    k_wind_exponent<<<(unsigned)((n + 127) / 128), 128, 0, s>>>((int32_t)n, c->s_ws, c->s_wd,
                                                               (double)c->P.alpha_w1, (double)c->P.alpha_w2,
                                                               wind_trig(), c->d_wser);
    return cudaGetLastError();
}

// Tile shape (rows << 16 | columns) of an H x W grid: of the ways to split the
// columns evenly, the one with the fewest rounds of 256 threads (a round of edges
// costs about as much as one of cells).  A fixed 16 x 64 left a 74-column grid
// tiles of 10 columns (226 grids of 418 x 74: 426 us before, 522 with them).
// `most`: cells a tile, fewer in small batches so that every SM has tiles.
int32_t jwf_table_tile_shape(int32_t H, int32_t W, int32_t most) {
    int64_t best = INT64_MAX;
    int32_t shape = 1 << 16 | 1;
    for (int32_t parts = 1; parts <= W; ++parts) {
        const int32_t cols = (W + parts - 1) / parts;
        if (cols > 128) continue;
        if (cols < 16 && best != INT64_MAX) break;
        int32_t rows = std::min(most / cols, JWF_PT_RING / (cols + 2) - 2);
        if (rows < 1) continue;
        rows = std::min(rows, H);
        const int32_t bands = (H + rows - 1) / rows;
        rows = (H + bands - 1) / bands;
        const int64_t rounds = (rows * cols + 255) / 256 + ((rows + 1) * (cols + 2) + 255) / 256;
        const int64_t cost = (rounds * 4 + 1) * bands * parts;
        if (cost < best) {
            best = cost;
            shape = rows << 16 | cols;
        }
    }
    return shape;
}

cudaError_t jwf_launch_prob_table(const jwf_ctx* c, const uint8_t* cls, const float* dem,
                                  const float* ws, const float* wd, cudaStream_t s) {
    const RateConsts& K = c->K;
    const bool per_cell = (c->flags & JWF_WIND_PER_CELL) != 0u;
    if (!per_cell) {
        const cudaError_t err = jwf_launch_wind_exponent(c, ws, wd, s);
        if (err != cudaSuccess) return err;
    }
    const size_t smem = (sizeof(ProbSmem) + 15) / 16 * 16 + (per_cell ? sizeof(ProbWindSmem) : 0);
    WindTrigF T{};
    if (per_cell) {
        const WindTrig t = wind_trig();
        for (int d = 0; d < 8; ++d) {
            T.s[d] = split_df(t.s[d]);
            T.c[d] = split_df(t.c[d]);
        }
        T.a1 = split_df((double)c->P.alpha_w1);
        T.m2a2 = split_df(-2.0 * (double)c->P.alpha_w2);
    }
    static int smem_set[2][64] = {};
    if (c->device < 0 || c->device >= 64) return cudaErrorInvalidDevice;
    if (!smem_set[per_cell ? 1 : 0][c->device]) {
        const cudaError_t err = cudaFuncSetAttribute(per_cell ? k_prob_table<true> : k_prob_table<false>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err != cudaSuccess) return err;
        smem_set[per_cell ? 1 : 0][c->device] = 1;
    }
    int64_t grid = (int64_t)c->num_sms * (per_cell ? 3 : 4);
    if (grid > c->n_pttiles) grid = c->n_pttiles;
    float* rates = (c->flags & JWF_KEEP_RATES) ? c->d_r : nullptr;
    if (per_cell)
        k_prob_table<true><<<(unsigned)grid, kPtT, smem, s>>>(c->d_pttiles, c->n_pttiles, c->d_H, c->d_W, c->d_off,
                                                             cls, dem, ws, wd, c->d_wexp, K, T, c->d_q, rates);
    else
        k_prob_table<false><<<(unsigned)grid, kPtT, smem, s>>>(c->d_pttiles, c->n_pttiles, c->d_H, c->d_W, c->d_off,
                                                              cls, dem, ws, wd, c->d_wexp, K, T, c->d_q, rates);
    return cudaGetLastError();
}

cudaError_t jwf_launch_rates_accumulate(const jwf_ctx* c, int32_t n_steps, const float* glam,
                                        const float* pburn, const float* mask, float* gr, const float* ab,
                                        double* gpc, cudaStream_t s) {
    auto k = gpc != nullptr ? (mask != nullptr ? k_rates_accumulate<true, true> : k_rates_accumulate<false, true>)
                            : (mask != nullptr ? k_rates_accumulate<true, false> : k_rates_accumulate<false, false>);
    const int64_t n = gpc != nullptr ? c->n_atiles : c->n_rtiles;
    const int64_t grid = gpc != nullptr ? std::min(n, c->partial_cap) : n;
    k<<<(unsigned)grid, kAccT, 0, s>>>(gpc != nullptr ? c->d_atiles : c->d_rtiles, n, c->d_H, c->d_W, c->d_off,
                                       c->cells, n_steps, glam, pburn, mask, gr, ab, c->d_partials, c->d_red_counter,
                                       gpc);
    return cudaGetLastError();
}

cudaError_t jwf_launch_rates_contract(jwf_ctx* c, const float* gr, const uint8_t* cls, const float* dem,
                                      const float* ws, const float* wd, double* gparams, cudaStream_t s) {
    // class-count specialisations keep the per-class bins sized to the table
    const int C = c->n_classes;
    if (C <= 1) return launch_rates_contract_c<1>(c, gr, cls, dem, ws, wd, gparams, s);
    if (C <= 4) return launch_rates_contract_c<4>(c, gr, cls, dem, ws, wd, gparams, s);
    if (C <= 11) return launch_rates_contract_c<11>(c, gr, cls, dem, ws, wd, gparams, s);
    if (C <= 16) return launch_rates_contract_c<16>(c, gr, cls, dem, ws, wd, gparams, s);
    return cudaErrorNotSupported;
}

cudaError_t jwf_launch_rates_bwd(jwf_ctx* c, int32_t n_steps, const float* glam,
                                 const float* pburn, const float* mask, const uint8_t* cls,
                                 const float* dem, const float* ws, const float* wd,
                                 double* gparams, cudaStream_t s) {
    cudaError_t err = cudaMemsetAsync(c->d_gr, 0, (size_t)c->cells * 8 * sizeof(float), s);
    if (err == cudaSuccess) err = jwf_launch_rates_accumulate(c, n_steps, glam, pburn, mask, c->d_gr, nullptr, nullptr, s);
    if (err == cudaSuccess) err = jwf_launch_rates_contract(c, c->d_gr, cls, dem, ws, wd, gparams, s);
    return err;
}
