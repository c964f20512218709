// Inside the atom spheres (Section 3, Eq. 3.4-3.7): the density's spherical-harmonic
// components on a logarithmic radial mesh, and the inner Dirichlet problem whose boundary
// values are the sphere-surface coefficients V_LM(R) of the interstitial solve.
//
// Radial mesh of sphere a: r_j = R_a exp((j - (n-1)) dx), dx = ln(R_a / r_min) / (n - 1); the
// paper uses a logarithmic mesh of 429 points.  rho_LM(r_j) is Eq. 3.7's surface projection
// taken on the sphere of radius r_j (the projection's Gauss-Legendre x uniform rule).  The
// inner solve is the Green's-function form of Eq. 3.5 with the overall sign that satisfies
// Eq. 3.4 (d2/dr2 + 2/r d/dr - L(L+1)/r^2) V_LM = 4pi (rho_LM - delta_L0 Z delta):
//   V_LM(r) = V_LM(R) (r/R)^L - 4pi/(2L+1) [ r^-(L+1) I1(r) + r^L I2(r) - r^L R^-(2L+1) I1(R) ]
//           + delta_L0 sqrt(4pi) Z (1/r - 1/R),
// I1(r) = int_0^r rho_LM r'^(L+2) dr', I2(r) = int_r^R rho_LM r'^(1-L) dr', integrated in
// x = ln r with the cubic through the four nearest samples per interval.  The density
// projection runs its Slater sums in FP32 pairs; the radial solve is one block per (atom, LM)
// with the interval integrals summed as block-wide prefix (I1) and suffix (I2) scans.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "df.cuh"
#include "internal.cuh"
#include "rule.cuh"

namespace lasto {

namespace {

constexpr int SD_NT = 128;
constexpr int SD_MAXQ = 2048;      // quadrature points per sphere
constexpr double SD_EXP_CUT = 40.0;
constexpr float SD_FAR = 20.0f;   // Slater terms beyond zeta r = 20 in plain FP32

using dfa::df;

struct SdExp {
    float h[64], l[64];   // 2^(-j/64) as double-floats
};

// The neighbours' share of rho_LM is smooth in r: at every quadrature direction the sum
// f(r) = sum_t W e^{-zeta |r u - D_t|} is analytic up to the branch points r = D e^{+-i theta} of
// the distances, which lie outside the sphere (D >= R_a + R_t), and |f| <= sum W inside the
// ellipse through the nearest of them.  So K Chebyshev points on (0, R_a) carry it: with s =
// 2 D_min / R_a - 1 and rho = s + sqrt(s^2 - 1) the interpolation error is at most 4 sum W
// rho^-K / (rho - 1) (Trefethen, Approximation Theory and Approximation Practice, theorem 8.2),
// and K is taken for 2^-66 sum W: 26 points at D_min = 2.1 R_a, whatever the number of radii.
// Beyond SD_KMAX points (a neighbour's small sphere close to a large one), or when the mesh has
// fewer radii, every radius is evaluated.
constexpr int SD_KMAX = 48;
constexpr int SD_BLOCKS = 32;      // blocks per sphere of the evaluation, looping over the points

__device__ __forceinline__ int sd_points(float dmin, double Ra, double r_min, int n_rad)
{
    const float R = (float)Ra;
    const float s = 2.0f * dmin / R - 1.0f, rho = s + sqrtf(s * s - 1.0f);
    const float k = ceilf((45.8f + logf(4.0f / (rho - 1.0f))) / logf(rho));
    // 0: every radius (so too for radii outside the sphere, for overlaps and for NaN)
    if (!(r_min < Ra) || !(k <= (float)SD_KMAX) || k >= (float)n_rad) return 0;
    return k < 2.0f ? 2 : (int)k;
}

// the neighbours' sum projected at point `i` of sphere a: Chebyshev point i (K > 0) or radius i
__device__ __forceinline__ double sd_radius(int i, int K, double Ra, double dx, int n_rad)
{
    if (K > 0) return 0.5 * Ra * (1.0 + cospi((2 * i + 1) / (2.0 * K)));
    return i == n_rad - 1 ? Ra : Ra * exp((i - (n_rad - 1)) * dx);
}

// Neighbours' Slater sums of sphere a = blockIdx.y at its K Chebyshev points (or at every
// radius), projected: out[a][lm][i], i < K.  rec: sphere records (position, radius, Slater
// weights and exponents per atom).  The sums run in FP32 pairs (about 44 bits: Tang's
// table-driven exp), with positions taken relative to the sphere's centre so that the pairs stay
// small; terms beyond zeta r = 20 (below e^-20 of their weight) in plain FP32; the projection
// sums over the quadrature points are FP64.  Bound: FP32 issue.  Pd55, 429 radii: 4.73 ms with
// every radius evaluated -> 0.35 ms.
__global__ void __launch_bounds__(SD_NT) k_sphere_neighbours(int na, const double* __restrict__ rec, int n_rad,
                                                             double r_min, const __grid_constant__ SphereRule rule,
                                                             SdExp tab, double* __restrict__ out)
{
    extern __shared__ float sd_sm[];   // per atom: D = pos_t - pos_a (3 pairs), W (3 pairs)
    __shared__ double rq[SD_MAXQ];     // the sum at the quadrature points
    __shared__ double F[9 * RULE_NT], trig[2 * RULE_NP];
    __shared__ float wmin[SD_NT / 32];
    const int a = blockIdx.y, tid = threadIdx.x;
    const int np = rule.np, nq = rule.nt * np;
    const double* ra = rec + (size_t)SPHERE_REC_DOUBLES * a;
    const double Ra = ra[3];
    const double dx = log(Ra / r_min) / (n_rad - 1);
    float dmin2 = 1e30f;
    for (int t = tid; t < na; t += SD_NT) {
        const double* rt = rec + (size_t)SPHERE_REC_DOUBLES * t;
        float* o = sd_sm + 12 * t;
        for (int c = 0; c < 3; c++) {
            const df D = dfa::from_double(rt[c] - ra[c]);
            o[2 * c] = D.h;
            o[2 * c + 1] = D.l;
            const df W = dfa::from_double(rt[4 + c]);
            o[6 + 2 * c] = W.h;
            o[7 + 2 * c] = W.l;
        }
        if (t != a) dmin2 = fminf(dmin2, fmaf(o[0], o[0], fmaf(o[2], o[2], o[4] * o[4])));
    }
    for (int t = tid; t < 2 * np; t += SD_NT) trig[t] = rule.trig[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmin2 = fminf(dmin2, __shfl_xor_sync(0xffffffffu, dmin2, o));
    if ((tid & 31) == 0) wmin[tid >> 5] = dmin2;
    __syncthreads();
    for (int w = 0; w < SD_NT / 32; w++) dmin2 = fminf(dmin2, wmin[w]);
    const int K = sd_points(sqrtf(dmin2) * (1.0f - 1e-5f), Ra, r_min, n_rad);
    // the exponents are the same on every atom (checked by the sphere kernel)
    df zt[3];
    float zmin = 1e30f;
    for (int c = 0; c < 3; c++) {
        zt[c] = dfa::from_double(ra[7 + c]);
        zmin = fminf(zmin, zt[c].h);
    }
    const float cut = (float)SD_EXP_CUT / zmin, cut2 = cut * cut * (1.0f + 1e-5f);
    bool twice[3];   // zeta_c exactly twice zeta_0
#pragma unroll
    for (int c = 0; c < 3; c++) twice[c] = c > 0 && zt[c].h == 2.0f * zt[0].h && zt[c].l == 2.0f * zt[0].l;
    const float far = SD_FAR / zmin, far2 = far * far * (1.0f + 1e-4f);
    for (int i = blockIdx.x; i < (K > 0 ? K : n_rad); i += gridDim.x) {
        const double r = sd_radius(i, K, Ra, dx, n_rad);
        for (int q = tid; q < nq; q += SD_NT) {
            const int row = q / np, b = q - row * np;
            const double rs = r * rule.st[row];
            const df px = dfa::from_double(rs * trig[2 * b]), py = dfa::from_double(rs * trig[2 * b + 1]),
                     pz = dfa::from_double(r * rule.ct[row]);
            df rho = {0.0f, 0.0f};
            float rfar = 0.0f;   // the terms beyond zeta d = SD_FAR in plain FP32, added once below
            for (int t = 0; t < na; t++) {
                if (t == a) continue;
                const float* o = sd_sm + 12 * t;
                const float fx = (px.h - o[0]) + (px.l - o[1]), fy = (py.h - o[2]) + (py.l - o[3]);
                const float fz = (pz.h - o[4]) + (pz.l - o[5]);
                const float r2f = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
                if (r2f > cut2) continue;
                if (r2f > far2) {
                    const float rf = sqrtf(r2f);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const float e = zt[c].h * rf;
                        if (e < (float)SD_EXP_CUT) rfar = fmaf(o[6 + 2 * c], expf(-e), rfar);
                    }
                    continue;
                }
                const df ex = dfa::add(px, df{-o[0], -o[1]});
                const df ey = dfa::add(py, df{-o[2], -o[3]});
                const df ez = dfa::add(pz, df{-o[4], -o[5]});
                const df d2 = dfa::add(dfa::add(dfa::sqr(ex), dfa::sqr(ey)), dfa::sqr(ez));
                const df d = dfa::sqrt_df(d2);
                df e0 = {0.0f, 0.0f};
                bool have0 = false;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const df e = dfa::mul(d, zt[c]);
                    if (e.h >= (float)SD_EXP_CUT) continue;
                    if (e.h > SD_FAR) {
                        rfar = fmaf(o[6 + 2 * c], expf(-e.h), rfar);
                    } else {
                        // zeta_c = 2 zeta_0: e^{-zeta_c d} = (e^{-zeta_0 d})^2
                        const df ec = (c > 0 && twice[c] && have0) ? dfa::sqr(e0) : dfa::exp_neg(e, tab.h, tab.l);
                        if (c == 0) {
                            e0 = ec;
                            have0 = true;
                        }
                        rho = dfa::add(rho, dfa::mul(df{o[6 + 2 * c], o[7 + 2 * c]}, ec));
                    }
                }
            }
            rq[q] = dfa::to_double(dfa::add_f(rho, rfar));
        }
        __syncthreads();
        rule_rings<SD_NT>(rq, rule.nt, np, trig, F);
        __syncthreads();
        if (tid < NLM) out[((size_t)a * NLM + tid) * n_rad + i] = rule_lm(rule, F, 0, rule.nt, tid);
        __syncthreads();   // rq and F are free again
    }
}

// Sums of the harmonics over the rule: g[lm] = sum_q w_q y_lm and the Gram matrix G[lm][l'm'] =
// sum_q w_q y_lm y_l'm' (what the projection makes of a constant and of the sphere's own y_l'm').
// A rule that is exact to degree 8 gives sqrt(4 pi) delta and the identity.
struct RuleGram {
    int exact;
    double g[NLM], G[NLM][NLM];
};

RuleGram rule_gram(const SphereRule& q)
{
    RuleGram r;
    std::memset(&r, 0, sizeof(r));
    r.exact = q.nt >= 5 && q.np >= 9;
    if (r.exact) {
        r.g[0] = std::sqrt(4.0 * PI);
        for (int lm = 0; lm < NLM; lm++) r.G[lm][lm] = 1.0;
        return r;
    }
    const double y00 = 0.5 / std::sqrt(PI);
    auto factor = [&](int lm, int b) {   // g_c(phi_b)
        const int l = l_of_lm(lm), ms = lm - l * l - l, p = (int)(((long long)std::abs(ms) * b) % q.np);
        return ms == 0 ? 1.0 : ms > 0 ? q.trig[2 * p] : q.trig[2 * p + 1];
    };
    for (int a = 0; a < q.nt; a++) {
        const double w = q.wf[a][0] / y00;   // the ring's weight
        for (int b = 0; b < q.np; b++) {
            double wy[NLM];
            for (int lm = 0; lm < NLM; lm++) {
                const int l = l_of_lm(lm);
                wy[lm] = q.wf[a][rule_slot(l, std::abs(lm - l * l - l))] * factor(lm, b);
                r.g[lm] += wy[lm];
            }
            for (int s = 0; s < NLM; s++)
                for (int t = 0; t < NLM; t++) r.G[s][t] += wy[s] * (wy[t] / w);
        }
    }
    return r;
}

// rho_LM(r_j) of sphere a = blockIdx.y, lm = SD_LM blockIdx.x ..: the neighbours' Chebyshev
// interpolant at r_j (Clenshaw's recurrence on the coefficients formed from out's first K
// entries; every radius holds its own value when K = 0), the sphere's own Slater terms through
// g, and the own nonspherical part zeta_1^3/(8 pi) e^{-zeta_1 r} (1 - r^2/R^2)^2 c_lm (r/R)^l
// (zero on the surface) through G.  FP64; a thread per radius.  Bound: FP64 issue (Pd55, 429 radii: 99 us).
constexpr int SD_LM = 5;
__global__ void __launch_bounds__(SD_NT) k_sphere_expand(int na, const double* __restrict__ rec,
                                                         const double* __restrict__ clm, int n_rad, double r_min,
                                                         const __grid_constant__ RuleGram gram, double* __restrict__ out)
{
    __shared__ double F[SD_LM][SD_KMAX], C[SD_LM][SD_KMAX], ct[4 * SD_KMAX];
    __shared__ float wmin[SD_NT / 32];
    const int a = blockIdx.y, lm0 = blockIdx.x * SD_LM, tid = threadIdx.x;
    const double* ra = rec + (size_t)SPHERE_REC_DOUBLES * a;
    const double Ra = ra[3];
    const double dx = log(Ra / r_min) / (n_rad - 1);
    float dmin2 = 1e30f;   // as in k_sphere_neighbours
    for (int t = tid; t < na; t += SD_NT) {
        const double* rt = rec + (size_t)SPHERE_REC_DOUBLES * t;
        const float ex = (float)(rt[0] - ra[0]), ey = (float)(rt[1] - ra[1]), ez = (float)(rt[2] - ra[2]);
        if (t != a) dmin2 = fminf(dmin2, fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmin2 = fminf(dmin2, __shfl_xor_sync(0xffffffffu, dmin2, o));
    if ((tid & 31) == 0) wmin[tid >> 5] = dmin2;
    __syncthreads();
    for (int w = 0; w < SD_NT / 32; w++) dmin2 = fminf(dmin2, wmin[w]);
    const int K = sd_points(sqrtf(dmin2) * (1.0f - 1e-5f), Ra, r_min, n_rad);
    double* o = out + ((size_t)a * NLM + lm0) * n_rad;
    if (K > 0) {
        for (int t = tid; t < SD_LM * K; t += SD_NT) F[t / K][t % K] = o[(size_t)(t / K) * n_rad + t % K];
        for (int t = tid; t < 4 * K; t += SD_NT) ct[t] = cospi(t / (2.0 * K));
        __syncthreads();
        for (int t = tid; t < SD_LM * K; t += SD_NT) {
            const int s = t / K, k = t % K;
            double acc = 0.0;
            for (int i = 0, p = k; i < K; i++) {   // p = k (2 i + 1) mod 4 K
                acc = fma(F[s][i], ct[p], acc);
                p += 2 * k;
                while (p >= 4 * K) p -= 4 * K;
            }
            C[s][k] = acc * (k == 0 ? 1.0 : 2.0) / K;
        }
        __syncthreads();
    }
    const double z1 = ra[7], pre = z1 * z1 * z1 / (8.0 * PI);
    for (int j = tid; j < n_rad; j += SD_NT) {
        const bool last = j == n_rad - 1;
        const double r = last ? Ra : Ra * exp((j - (n_rad - 1)) * dx);
        double b1[SD_LM], b2[SD_LM];
        if (K > 0) {
            const double x2 = 4.0 * r / Ra - 2.0;
#pragma unroll
            for (int s = 0; s < SD_LM; s++) b1[s] = b2[s] = 0.0;
            for (int k = K - 1; k > 0; k--)
#pragma unroll
                for (int s = 0; s < SD_LM; s++) {
                    const double b0 = fma(x2, b1[s], C[s][k] - b2[s]);
                    b2[s] = b1[s];
                    b1[s] = b0;
                }
#pragma unroll
            for (int s = 0; s < SD_LM; s++) b1[s] = fma(0.5 * x2, b1[s], C[s][0] - b2[s]);
        } else {
#pragma unroll
            for (int s = 0; s < SD_LM; s++) b1[s] = o[(size_t)s * n_rad + j];
        }
        const double e1 = exp(-z1 * r), sr = r / Ra, tt = 1.0 - sr * sr, nsr = r < Ra ? pre * e1 * tt * tt : 0.0;
        double pw[5];
        pw[0] = 0.0;
        pw[1] = nsr * sr;
        for (int l = 2; l < 5; l++) pw[l] = pw[l - 1] * sr;
        const bool own = lm0 == 0 || !gram.exact;
        const double sl = own ? fma(ra[4], e1, fma(ra[5], exp(-ra[8] * r), ra[6] * exp(-ra[9] * r))) : 0.0;
#pragma unroll
        for (int s = 0; s < SD_LM; s++) {
            const int lm = lm0 + s;
            double v = b1[s];
            if (own) v = fma(gram.g[lm], sl, v);
            if (gram.exact) {
                if (lm > 0) v = fma(clm[24 * (size_t)a + lm - 1], pw[l_of_lm(lm)], v);
            } else {
                for (int t = 1; t < NLM; t++)
                    v = fma(gram.G[lm][t] * clm[24 * (size_t)a + t - 1], pw[l_of_lm(t)], v);
            }
            o[(size_t)s * n_rad + j] = v;
        }
    }
}

__device__ __forceinline__ double seg_integral(double g0, double g1, double g2, double g3, int kind, double h)
{
    // kind 0: first interval (samples j..j+3), 1: interior (j-1..j+2), 2: last (j-2..j+1)
    if (kind == 0) return h / 24.0 * (9.0 * g0 + 19.0 * g1 - 5.0 * g2 + g3);
    if (kind == 2) return h / 24.0 * (g0 - 5.0 * g1 + 19.0 * g2 + 9.0 * g3);
    return h / 24.0 * (-g0 + 13.0 * g1 + 13.0 * g2 - g3);
}

constexpr int IS_NT = 128;
constexpr int IS_MAX = 4096;   // radial points per sphere

// inclusive scan of one double per thread over the block (warp shuffles, then the warps' totals)
__device__ __forceinline__ double block_incl_scan(double v, double* wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    __syncthreads();
    if (lane == 31) wsum[w] = v;
    __syncthreads();
    for (int q = 0; q < w; q++) v += wsum[q];
    return v;
}

// One block per (atom, LMS harmonics).  The radii and their reciprocals once, then per harmonic
// the integrands at the mesh points, the cubic-rule integral over each interval, I1 as a prefix
// sum and I2 as a suffix sum of the intervals (each thread a contiguous run of intervals, the
// runs' totals scanned across the block), and V_LM.  Bound: FP64 issue, or for few atoms a block's own
// chain.  The exponential of a radius costs more than its share of a harmonic, so five harmonics share
// it where the atoms fill the SMs, and no division is left per point; up to IS_ONE atoms a block takes
// one harmonic (bitwise the same).  429 radii, a block per harmonic with divisions, then with
// one and with five harmonics per block: 1 atom 24, 23, 74 us; 13 atoms 53, 47, 74; 40 atoms 119,
// 105, 115; 55 atoms 166, 137, 115 us.
constexpr int IS_LM = 5;
constexpr int IS_ONE = 40;
template <int LMS>
__global__ void __launch_bounds__(IS_NT) k_inner_solve(const double* __restrict__ R,
                                                       const double* __restrict__ Z, int n, double r_min,
                                                       const double* __restrict__ rho_lm,
                                                       const double* __restrict__ vR, double* __restrict__ v)
{
    extern __shared__ double is_sm[];   // x[n], 1/x[n], g1[n], g2[n], seg1[n], seg2[n]
    __shared__ double wsum[IS_NT / 32];
    double* xs = is_sm;
    double* ix = xs + n;
    double* g1 = ix + n;
    double* g2 = g1 + n;
    double* s1 = g2 + n;
    double* s2 = s1 + n;
    const int a = blockIdx.x / (NLM / LMS), lm0 = (blockIdx.x % (NLM / LMS)) * LMS;
    const double Ra = R[a];
    const double h = log(Ra / r_min) / (n - 1);
    for (int j = threadIdx.x; j < n; j += IS_NT) {
        const double x = j == n - 1 ? Ra : Ra * exp((j - (n - 1)) * h);
        xs[j] = x;
        ix[j] = 1.0 / x;
    }
    const double iRa = 1.0 / Ra, sq4piZ = 3.5449077018110318 * Z[a];
    // contiguous runs of intervals per thread: [c0, c1)
    const int m = n - 1, per = (m + IS_NT - 1) / IS_NT;
    const int c0 = min(m, (int)threadIdx.x * per), c1 = min(m, c0 + per);
    for (int lm = lm0; lm < lm0 + LMS; lm++) {
        const int L = l_of_lm(lm);
        const double* rho = rho_lm + ((size_t)a * NLM + lm) * n;
        double* out = v + ((size_t)a * NLM + lm) * n;
        for (int j = threadIdx.x; j < n; j += IS_NT) {
            const double x = xs[j], i1 = ix[j], f = rho[j] * x * x;
            double xl = 1.0, il = 1.0;
            for (int e = 0; e < L; e++) {
                xl *= x;
                il *= i1;
            }
            g1[j] = f * x * xl;   // rho r^(L+2) dr = rho r^(L+3) d(ln r)
            g2[j] = f * il;       // rho r^(1-L) dr = rho r^(2-L) d(ln r)
        }
        __syncthreads();
        for (int j = threadIdx.x; j < n - 1; j += IS_NT) {
            const int b = j == 0 ? 0 : (j == n - 2 ? n - 4 : j - 1);
            const int kind = j == 0 ? 0 : (j == n - 2 ? 2 : 1);
            s1[j] = seg_integral(g1[b], g1[b + 1], g1[b + 2], g1[b + 3], kind, h);
            s2[j] = seg_integral(g2[b], g2[b + 1], g2[b + 2], g2[b + 3], kind, h);
        }
        const double I1_0 = g1[0] / (L + 3);   // rho taken constant on [0, r_0]: rho_0 r_0^(L+3) / (L+3)
        __syncthreads();
        double run1 = 0.0, run2 = 0.0;
        for (int j = c0; j < c1; j++) {
            run1 += s1[j];
            run2 += s2[j];
        }
        const double inc1 = block_incl_scan(run1, wsum);
        __syncthreads();
        const double inc2 = block_incl_scan(run2, wsum);
        __syncthreads();
        if (threadIdx.x == IS_NT - 1) {
            wsum[0] = inc1;   // I1 over all intervals
            wsum[1] = inc2;   // I2 over all intervals
        }
        __syncthreads();
        const double tot1 = wsum[0], tot2 = wsum[1];
        const double c = 4.0 * 3.14159265358979323846 / (2 * L + 1);
        double iRaL = 1.0;
        for (int e = 0; e < L; e++) iRaL *= iRa;
        // V = x^L (V(R) / R^L + c I1(R) / R^(2L+1) - c I2) - c I1 / x^(L+1)
        const double head = fma(c * (I1_0 + tot1), iRaL * iRaL * iRa, vR[(size_t)a * NLM + lm] * iRaL);
        // points [c0, c1) of this thread's run, and the last point m with the run that ends there:
        // I1 at point j = I1_0 + intervals [0, j), I2 = intervals [j, m)
        if (c0 < c1) {
            double p1 = inc1 - run1, p2 = tot2 - (inc2 - run2);
            const int last = c1 == m ? m : c1 - 1;
            for (int j = c0; j <= last; j++) {
                if (j > c0) {
                    p1 += s1[j - 1];
                    p2 -= s2[j - 1];
                }
                const double x = xs[j], i1 = ix[j];
                double xl = 1.0, il = i1;
                for (int e = 0; e < L; e++) {
                    xl *= x;
                    il *= i1;
                }
                const double I2 = j == m ? 0.0 : p2;
                double val = xl * (head - c * I2) - c * (I1_0 + p1) * il;
                if (L == 0) val += sq4piZ * (i1 - iRa);
                out[j] = val;
            }
        }
        __syncthreads();   // the integrands' arrays are free again
    }
}

}  // namespace

cudaError_t launch_sphere_density(int na, const double* rec, const double* clm, const SphereRule& q, int n_rad,
                                  double r_min, double* out, cudaStream_t s)
{
    SdExp tab;
    for (int t = 0; t < 64; t++) {
        const double v = std::exp2(-t / 64.0);
        tab.h[t] = (float)v;
        tab.l[t] = (float)(v - (double)tab.h[t]);
    }
    const size_t smem = sizeof(float) * 12 * (size_t)na;
    if (smem > 160 * 1024 || q.nt * q.np > SD_MAXQ) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_sphere_neighbours, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    k_sphere_neighbours<<<dim3((unsigned)std::min(n_rad, SD_BLOCKS), (unsigned)na), SD_NT, smem, s>>>(na, rec, n_rad, r_min, q,
                                                                                          tab, out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    static_assert(NLM % SD_LM == 0, "groups of harmonics");
    k_sphere_expand<<<dim3(NLM / SD_LM, (unsigned)na), SD_NT, 0, s>>>(na, rec, clm, n_rad, r_min, rule_gram(q), out);
    return cudaGetLastError();
}

cudaError_t launch_inner_solve(int na, const double* R, const double* Z, int n_rad, double r_min,
                               const double* rho_lm, const double* vR, double* v, cudaStream_t s)
{
    if (n_rad > IS_MAX) return cudaErrorInvalidValue;
    const size_t smem = sizeof(double) * 6 * (size_t)n_rad;
    static_assert(NLM % IS_LM == 0, "groups of harmonics");
    const int lms = na <= IS_ONE ? 1 : IS_LM;
    auto* kernel = lms == 1 ? k_inner_solve<1> : k_inner_solve<IS_LM>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(sizeof(double) * 6 * IS_MAX));
    if (e != cudaSuccess) return e;
    kernel<<<(unsigned)(na * (NLM / lms)), IS_NT, smem, s>>>(R, Z, n_rad, r_min, rho_lm, vR, v);
    return cudaGetLastError();
}

}  // namespace lasto
