// Right-hand side of the interstitial Poisson problem: per-sphere pseudo-density,
// deposit on the mesh, boundary multipoles and Dirichlet face values.
//
// Section 1 of the paper: the rapidly varying density inside each sphere is replaced
// by a smooth pseudo-density with the same multipole moments (nucleus included); only
// the monopole is replaced, the nonspherical terms go on the grid as they are.
// Section 3 (constraints beside Eq. 3.2-3.3): same charge inside the sphere, same
// value and slope at R.  Reading of the shape: rho_tilde = a + b r^2 + c r^4.
//
// GPU formulation.  With the same three Slater exponents on every atom, the spherical
// average of the neighbours' Slater terms about sphere i factorises into
//   N_i(r) = sum_k [ 2 A_ik sinh(zeta_k r)/r - 2 B_ik cosh(zeta_k r) ],
//   A_ik = sum_{j != i} W_jk e^{-zeta_k D_ij} (1 + zeta_k D_ij) / (2 D_ij zeta_k^2),
//   B_ik = sum_{j != i} W_jk e^{-zeta_k D_ij} / (2 D_ij zeta_k),
// (W = w zeta^3 / 8 pi), so a node inside sphere i costs three exponentials instead
// of one average per neighbour, and the sphere charge integrals are closed forms.
// Inside sphere i the deposit evaluates n_e - rho0_i + rho_tilde_i as
//   (neighbours' Slater terms at the node) - N_i(r) + rho_ns,i(x) + rho_tilde_i(r),
// the atom's own spherical terms cancelling exactly rather than numerically.
#include <cmath>

#include "df.cuh"
#include <mutex>

#include "internal.cuh"

namespace lasto {

// ---------------------------------------------------------------- harmonics table
static __constant__ Mono c_mono[N_MONO_TERMS];

constexpr int EXP_N = 2048;   // entries of the exponential's table: a power of two
// ln 2 / EXP_N, also as a double-float
constexpr double LN2_N = 0.69314718055994530942 / EXP_N;
constexpr float LN2_H = (float)LN2_N, LN2_L = (float)(LN2_N - (double)LN2_H);
static __device__ double g_exp_tab64[EXP_N];
static __device__ float2 g_exp_tab[EXP_N];   // 2^(-j/EXP_N) as double-floats

void host_monomials(Mono* o)
{
    const double pi = PI;
    const double c0 = 0.5 / std::sqrt(pi), c1 = std::sqrt(3.0 / (4 * pi));
    const double c2a = 0.5 * std::sqrt(15 / pi), c2b = 0.25 * std::sqrt(5 / pi), c2c = 0.25 * std::sqrt(15 / pi);
    const double c3a = 0.25 * std::sqrt(35 / (2 * pi)), c3b = 0.5 * std::sqrt(105 / pi), c3c = 0.25 * std::sqrt(21 / (2 * pi));
    const double c3d = 0.25 * std::sqrt(7 / pi), c3e = 0.25 * std::sqrt(105 / pi);
    const double c4a = 0.75 * std::sqrt(35 / pi), c4b = 0.75 * std::sqrt(35 / (2 * pi)), c4c = 0.75 * std::sqrt(5 / pi);
    const double c4d = 0.75 * std::sqrt(5 / (2 * pi)), c4e = (3.0 / 16) / std::sqrt(pi), c4f = 0.375 * std::sqrt(5 / pi);
    const double c4g = (3.0 / 16) * std::sqrt(35 / pi);
    const Mono t[N_MONO_TERMS] = {
        {0, 0, 0, 0, c0},
        {1, 0, 1, 0, c1}, {2, 0, 0, 1, c1}, {3, 1, 0, 0, c1},
        {4, 1, 1, 0, c2a}, {5, 0, 1, 1, c2a},
        {6, 0, 0, 2, 2 * c2b}, {6, 2, 0, 0, -c2b}, {6, 0, 2, 0, -c2b},
        {7, 1, 0, 1, c2a}, {8, 2, 0, 0, c2c}, {8, 0, 2, 0, -c2c},
        {9, 2, 1, 0, 3 * c3a}, {9, 0, 3, 0, -c3a},
        {10, 1, 1, 1, c3b},
        {11, 0, 1, 2, 4 * c3c}, {11, 2, 1, 0, -c3c}, {11, 0, 3, 0, -c3c},
        {12, 0, 0, 3, 2 * c3d}, {12, 2, 0, 1, -3 * c3d}, {12, 0, 2, 1, -3 * c3d},
        {13, 1, 0, 2, 4 * c3c}, {13, 3, 0, 0, -c3c}, {13, 1, 2, 0, -c3c},
        {14, 2, 0, 1, c3e}, {14, 0, 2, 1, -c3e},
        {15, 3, 0, 0, c3a}, {15, 1, 2, 0, -3 * c3a},
        {16, 3, 1, 0, c4a}, {16, 1, 3, 0, -c4a},
        {17, 2, 1, 1, 3 * c4b}, {17, 0, 3, 1, -c4b},
        {18, 1, 1, 2, 6 * c4c}, {18, 3, 1, 0, -c4c}, {18, 1, 3, 0, -c4c},
        {19, 0, 1, 3, 4 * c4d}, {19, 2, 1, 1, -3 * c4d}, {19, 0, 3, 1, -3 * c4d},
        {20, 0, 0, 4, 8 * c4e}, {20, 4, 0, 0, 3 * c4e}, {20, 0, 4, 0, 3 * c4e},
        {20, 2, 2, 0, 6 * c4e}, {20, 2, 0, 2, -24 * c4e}, {20, 0, 2, 2, -24 * c4e},
        {21, 1, 0, 3, 4 * c4d}, {21, 3, 0, 1, -3 * c4d}, {21, 1, 2, 1, -3 * c4d},
        {22, 2, 0, 2, 6 * c4f}, {22, 0, 2, 2, -6 * c4f}, {22, 4, 0, 0, -c4f}, {22, 0, 4, 0, c4f},
        {23, 3, 0, 1, c4b}, {23, 1, 2, 1, -3 * c4b},
        {24, 4, 0, 0, c4g}, {24, 2, 2, 0, -6 * c4g}, {24, 0, 4, 0, c4g},
    };
    for (int i = 0; i < N_MONO_TERMS; i++) o[i] = t[i];
}

void host_solid_harmonics(double x, double y, double z, double* S)
{
    Mono t[N_MONO_TERMS];
    host_monomials(t);
    double px[5] = {1, x, x * x, x * x * x, x * x * x * x}, py[5] = {1, y, y * y, y * y * y, y * y * y * y},
           pz[5] = {1, z, z * z, z * z * z, z * z * z * z};
    for (int q = 0; q < NLM; q++) S[q] = 0.0;
    for (int i = 0; i < N_MONO_TERMS; i++) S[t[i].lm] += t[i].coef * px[t[i].a] * py[t[i].b] * pz[t[i].c];
}

// ---------------------------------------------------------------- sphere records
// rec[i][*]: 0-2 pos, 3 R, 4-6 W_k, 7-9 zeta_k, 10-12 A_k, 13-15 B_k, 16-18 (a, b, c),
// 19 q, 20 rho0(R), 21 rho0'(R), 22-23: x y z R^2 as four floats, 24-78 float forms for the
// FP32-pair deposit (pairs are double-floats): the position as three floats per axis (exact), W
// pairs, zeta, EXP_N zeta / ln 2 pairs, which zeta are twice zeta_0, 2 A and 2 B pairs, 1/R^2,
// zeta_1^3 / (8 pi), and the nonspherical polynomial sum_lm c_lm / R^l S_lm: a pair per monomial
// x^a y^b z^c of degree 0 to 4 (the constant is 0) in the order of its Horner evaluation, a = 4..0,
// b = 4-a..0, c = 4-a-b..0; from 80 the same coefficients in FP64
enum { RX = 0, RR = 3, RW = 4, RZ = 7, RA = 10, RB = 13, RC = 16, RQ = 19, RRHO = 20, RDRHO = 21, RXF = 22, RF = 24, RP = 80 };
enum { FP = 0, FW = 9, FZ = 15, FC = 18, F2 = 24, FA = 26, FB = 32, FR = 38, FN = 40, FH = 42 };   // floats from RF
constexpr int POLY_N = 35;
static_assert(RF + (FH + 2 * POLY_N + 1) / 2 <= RP && RP + POLY_N <= SPHERE_REC_DOUBLES, "sphere record");

// place of x^a y^b z^c in the Horner order
__host__ __device__ constexpr int poly_slot(int a, int b, int c)
{
    int s = 0;
    for (int q = 4; q > a; q--) s += (5 - q) * (6 - q) / 2;
    for (int q = 4 - a; q > b; q--) s += 5 - a - q;
    return s + (4 - a - b) - c;
}

// the monomials of each place: S_lm's coefficients there (lm 0: none; the constant is left out)
constexpr int POLY_TERMS = 4;
struct PolyTerm {
    int lm;
    double coef;
};
static __device__ PolyTerm g_poly[POLY_N][POLY_TERMS];

// Constant tables are per device: each device gets its own upload, once, with that device
// current (a flag per device, so alternating devices uploads nothing again).
constexpr int MAX_DEVICES = 64;
static bool g_mono_uploaded[MAX_DEVICES] = {};
static bool g_constants_done[MAX_DEVICES] = {};
static std::mutex g_constants_mutex;

static cudaError_t ensure_monomials()
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_constants_mutex);
    if (g_mono_uploaded[dev]) return cudaSuccess;
    Mono t[N_MONO_TERMS];
    host_monomials(t);
    e = cudaMemcpyToSymbol(c_mono, t, sizeof(t));
    if (e != cudaSuccess) return e;
    PolyTerm pt[POLY_N][POLY_TERMS] = {};
    for (int q = 1; q < N_MONO_TERMS; q++) {
        PolyTerm* o = pt[poly_slot(t[q].a, t[q].b, t[q].c)];
        int k = 0;
        while (k < POLY_TERMS && o[k].lm != 0) k++;
        if (k == POLY_TERMS) return cudaErrorInvalidValue;
        o[k].lm = t[q].lm;
        o[k].coef = t[q].coef;
    }
    e = cudaMemcpyToSymbol(g_poly, pt, sizeof(pt));
    if (e != cudaSuccess) return e;
    static float2 ex[EXP_N];   // (under the lock)
    static double ex64[EXP_N];
    for (int j = 0; j < EXP_N; j++) {
        const double v = std::exp2(-j / (double)EXP_N);
        ex64[j] = v;
        ex[j].x = (float)v;
        ex[j].y = (float)(v - (double)ex[j].x);
    }
    e = cudaMemcpyToSymbol(g_exp_tab64, ex64, sizeof(ex64));
    if (e != cudaSuccess) return e;
    e = cudaMemcpyToSymbol(g_exp_tab, ex, sizeof(ex));
    if (e == cudaSuccess) g_mono_uploaded[dev] = true;
    return e;
}

struct SphArgs {
    int na;
    const double *pos, *Z, *R, *w, *zeta, *clm;
    const double* ax[3];
    int n[3];
    double* rec;
    double *q, *rhoR, *drhoR, *coef;
    int* status;
};

using dfa::df;

// x as the sum of three floats (72 bits: exact over any range of exponents that matters here)
__device__ __forceinline__ void three_floats(double x, float* o)
{
    o[0] = (float)x;
    x -= (double)o[0];
    o[1] = (float)x;
    o[2] = (float)(x - (double)o[1]);
}

constexpr int SPH_NT = 128;

// One block per sphere.  The neighbour sums run over the block; then one lane per Slater term
// forms the term's share of rho, rho' and the charge, 24 threads the nonspherical coefficients
// over R^l.  Latency bound (a serial chain of FP64 exponentials and divisions on one thread
// before): 55 spheres 47.8 -> 22.6 us, 147 spheres 54.3 -> 29.0 us.
__global__ void __launch_bounds__(SPH_NT) k_sphere_params(SphArgs a)
{
    __shared__ double red[6], own[3][3];
    __shared__ int bad_geom, bad_zeta;
    const int i = blockIdx.x, tid = threadIdx.x;
    if (tid == 0) bad_geom = bad_zeta = 0;
    __syncthreads();
    const double xi = a.pos[3 * i], yi = a.pos[3 * i + 1], zi = a.pos[3 * i + 2], Ri = a.R[i];
    double zt[3], c8[3], iz[3];   // zeta, zeta^3 / (8 pi), 1 / (2 zeta)
    for (int k = 0; k < 3; k++) {
        zt[k] = a.zeta[3 * i + k];
        c8[k] = zt[k] * zt[k] * zt[k] / (8.0 * PI);
        iz[k] = 0.5 / zt[k];
    }
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int j = tid; j < a.na; j += SPH_NT) {
        if (j == i) continue;
        const double dx = a.pos[3 * j] - xi, dy = a.pos[3 * j + 1] - yi, dz = a.pos[3 * j + 2] - zi;
        const double D = sqrt(dx * dx + dy * dy + dz * dz);
        if (!(D >= Ri + a.R[j])) bad_geom = 1;
        const double iD = 1.0 / D;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const double z = a.zeta[3 * j + k];
            double c = c8[k], hz = iz[k];
            if (z != zt[k]) {
                bad_zeta = 1;
                c = z * z * z / (8.0 * PI);
                hz = 0.5 / z;
            }
            // B's term W e^{-zeta D} / (2 D zeta); A's is (D + 1 / zeta) times it
            const double t = a.w[3 * j + k] * c * exp(-z * D) * iD * hz;
            acc[3 + k] += t;
            acc[k] = fma(t, D + 2.0 * hz, acc[k]);
        }
    }
    for (int v = 0; v < 6; v++) {
        const double s = block_sum<SPH_NT>(acc[v]);
        if (tid == 0) red[v] = s;
    }
    __syncthreads();
    double* r = a.rec + (size_t)SPHERE_REC_DOUBLES * i;
    if (tid < 3) {
        // the sphere must sit two nodes inside every face
        const double c = a.pos[3 * i + tid];
        if (!(c - Ri >= a.ax[tid][2] && c + Ri <= a.ax[tid][a.n[tid] - 3])) bad_geom = 1;
        const int k = tid;
        const double z = a.zeta[3 * i + k], wk = a.w[3 * i + k];
        const double W = wk * z * z * z / (8.0 * PI);
        const double A = red[k], B = red[3 + k];
        r[RW + k] = W;
        r[RZ + k] = z;
        r[RA + k] = A;
        r[RB + k] = B;
        float* f = reinterpret_cast<float*>(r + RF);
        const df Wf = dfa::from_double(W), cf = dfa::from_double(z * (1.0 / LN2_N));
        f[FW + 2 * k] = Wf.h;
        f[FW + 2 * k + 1] = Wf.l;
        f[FZ + k] = (float)z;
        f[FC + 2 * k] = cf.h;
        f[FC + 2 * k + 1] = cf.l;
        if (k == 0)
            f[F2] = __int_as_float((a.zeta[3 * i + 1] == 2.0 * z ? 1 : 0) | (a.zeta[3 * i + 2] == 2.0 * z ? 2 : 0));
        const double zR = z * Ri, eR = exp(-zR), sh = sinh(zR), ch = cosh(zR);
        own[0][k] = W * eR + 2.0 * A * sh / Ri - 2.0 * B * ch;
        own[1][k] = -z * W * eR + 2.0 * A * (z * ch / Ri - sh / (Ri * Ri)) - 2.0 * B * z * sh;
        // electrons inside the sphere: own normalised Slater term + neighbour averages
        const double in = wk * (1.0 - eR * (1.0 + zR + 0.5 * zR * zR));
        const double I1 = Ri * ch / z - sh / (z * z);                                   // int r sinh
        const double I2 = Ri * Ri * sh / z - 2.0 * Ri * ch / (z * z) + 2.0 * sh / (z * z * z);  // int r^2 cosh
        own[2][k] = in + 4.0 * PI * (2.0 * A * I1 - 2.0 * B * I2);
        const df A2 = dfa::from_double(2.0 * A), B2 = dfa::from_double(2.0 * B);
        f[FA + 2 * k] = A2.h;
        f[FA + 2 * k + 1] = A2.l;
        f[FB + 2 * k] = B2.h;
        f[FB + 2 * k + 1] = B2.l;
        if (k == 0) {
            const df n1 = dfa::from_double(z * z * z / (8.0 * PI));
            f[FN] = n1.h;
            f[FN + 1] = n1.l;
        }
    } else if (tid >= 32 && tid < 64) {
        // the nonspherical polynomial's coefficients, two per thread
        const double iR = 1.0 / Ri;
        for (int slot = tid - 32; slot < POLY_N; slot += 32) {
            double v = 0.0;
#pragma unroll
            for (int t = 0; t < POLY_TERMS; t++) {
                const int lm = g_poly[slot][t].lm;
                const double iR2 = iR * iR;
                const double iRl = lm >= 16 ? iR2 * iR2 : lm >= 9 ? iR2 * iR : lm >= 4 ? iR2 : iR;
                if (lm > 0) v = fma(g_poly[slot][t].coef * iRl, a.clm[24 * (size_t)i + lm - 1], v);
            }
            const df c = dfa::from_double(v);
            float* f = reinterpret_cast<float*>(r + RF) + FH + 2 * slot;
            f[0] = c.h;
            f[1] = c.l;
            r[RP + slot] = v;
        }
    } else if (tid == 64) {
        r[RX] = xi;
        r[RX + 1] = yi;
        r[RX + 2] = zi;
        r[RR] = Ri;
        float* xf = reinterpret_cast<float*>(r + RXF);
        xf[0] = (float)xi;
        xf[1] = (float)yi;
        xf[2] = (float)zi;
        xf[3] = (float)(Ri * Ri);
        const df iR2 = dfa::from_double(1.0 / (Ri * Ri));
        float* f = reinterpret_cast<float*>(r + RF) + FR;
        f[0] = iR2.h;
        f[1] = iR2.l;
    } else if (tid >= 96 && tid < 99) {
        three_floats(a.pos[3 * i + tid - 96], reinterpret_cast<float*>(r + RF) + FP + 3 * (tid - 96));
    }
    __syncthreads();
    if (tid != 0) return;
    const double rho = own[0][0] + own[0][1] + own[0][2], drho = own[1][0] + own[1][1] + own[1][2];
    const double q = own[2][0] + own[2][1] + own[2][2] - a.Z[i];
    const double Qr = q / (4.0 * PI);
    const double R2 = Ri * Ri, R3 = R2 * Ri, R4 = R2 * R2, R7 = R4 * R3;
    const double cc = (Qr - rho * R3 / 3.0 + drho * R4 / 15.0) * (105.0 / (8.0 * R7));
    const double bb = drho / (2.0 * Ri) - 2.0 * cc * R2;
    const double aa = rho - 0.5 * drho * Ri + cc * R4;
    r[RC] = aa;
    r[RC + 1] = bb;
    r[RC + 2] = cc;
    r[RQ] = q;
    r[RRHO] = rho;
    r[RDRHO] = drho;
    if (a.q) a.q[i] = q;
    if (a.rhoR) a.rhoR[i] = rho;
    if (a.drhoR) a.drhoR[i] = drho;
    if (a.coef) {
        a.coef[3 * i] = aa;
        a.coef[3 * i + 1] = bb;
        a.coef[3 * i + 2] = cc;
    }
    if (a.status) {
        if (bad_zeta) atomicMax(a.status, (int)LASTO_ERR_INVALID_ARG);
        if (bad_geom) atomicMax(a.status, (int)LASTO_ERR_GEOMETRY);
    }
}

cudaError_t launch_sphere_params(const lasto_cluster& cl, const double* ax0, const double* ax1, const double* ax2,
                                 double* rec, double* q, double* rhoR, double* drhoR, double* coef, int* status,
                                 cudaStream_t s)
{
    const cudaError_t em = ensure_monomials();
    if (em != cudaSuccess) return em;
    SphArgs a;
    a.na = cl.n_atoms;
    a.pos = cl.pos;
    a.Z = cl.Z;
    a.R = cl.R;
    a.w = cl.slater_w;
    a.zeta = cl.slater_zeta;
    a.clm = cl.c_lm;
    a.ax[0] = ax0;
    a.ax[1] = ax1;
    a.ax[2] = ax2;
    for (int d = 0; d < 3; d++) a.n[d] = cl.n[d];
    a.rec = rec;
    a.q = q;
    a.rhoR = rhoR;
    a.drhoR = drhoR;
    a.coef = coef;
    a.status = status;
    k_sphere_params<<<cl.n_atoms, SPH_NT, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- deposit
struct DepArgs {
    int na;
    int n[3];
    const double* ax[3];
    const double* rec;
    double* b;
    int* owner;
    int* status;
};

__global__ void k_deposit_df(DepArgs a);

constexpr int DEP_NT = 256;
constexpr double EXP_CUT = 40.0;   // e^{-40} * max W < 1e-14 absolute; skipped terms are below FP64 rounding of n_e
// FP32-pair deposit: where a pair's precision changes, in units of 1/zeta_min.  A Slater term is
// summed with an absolute error far below that of the density it adds to, so a term that is small
// at its distance needs fewer bits: from NEAR_T on (e^-9 of its weight) about 35 relative bits
// do, from MID_T on an FP32 exponential of an accurate exponent (relative error 3e-7), from FAR_T
// on plain FP32 (a few 1e-6 in e^{-zeta r}: the FP32 distance and exponent).  The far limit was 20
// with no class before it but the double-float one: an error four times as large, where three
// equal exponents add up (1.1e-10 of the density node by node), at 2.6 times the time.
constexpr float NEAR_T = 9.0f;
constexpr float MID_T = 18.0f;
constexpr float FAR_T = 22.0f;
// Slater terms with zeta r > DF_EXP_CUT are dropped, and atoms beyond DF_EXP_CUT / zeta_min of a
// tile's bounding box for the whole tile.  Measured against the oracle on the small test clusters
// (Pd13 graded 33^3 and uniform 65^3, Pd2): the largest node-wise error where the density exceeds
// 1e-3 of its maximum is 2e-11 to 6e-11 of the local density at 37; at 34 it was 3.6e-10.
constexpr float DF_EXP_CUT = 37.0f;

// one 8 x 8 x 8 tile of nodes per block, two nodes (four planes apart) per thread
__global__ void k_deposit64(DepArgs a);
constexpr int DEP64_MAX_ATOMS = 1828;   // most atoms the FP64 form takes (its two index lists: 14 KiB)
constexpr int DT_X = 8, DT_Y = 8, DT_Z = 8;
static_assert(DT_X * DT_Y * DT_Z == 2 * DEP_NT, "deposit tile = one block");
constexpr int DF_MAX_ATOMS = 2432;      // most atoms the FP32-pair form takes (its four index lists: 38 KiB)

// bytes of a launch's index lists
static size_t deposit_smem(bool mixed, int na) { return sizeof(int) * (mixed ? 4 : 2) * (size_t)na; }

cudaError_t launch_deposit(const lasto_cluster& cl, const double* rec, int precision, double* b, int* owner, int* status,
                           cudaStream_t s)
{
    cudaError_t e = ensure_monomials();
    if (e != cudaSuccess) return e;
    DepArgs a;
    a.na = cl.n_atoms;
    for (int d = 0; d < 3; d++) a.n[d] = cl.n[d];
    a.ax[0] = cl.x;
    a.ax[1] = cl.y;
    a.ax[2] = cl.z;
    a.rec = rec;
    a.b = b;
    a.owner = owner;
    a.status = status;
    const bool mixed = precision == LASTO_PREC_MIXED;
    if (cl.n_atoms > (mixed ? DF_MAX_ATOMS : DEP64_MAX_ATOMS)) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)((cl.n[0] + DT_X - 1) / DT_X), (unsigned)((cl.n[1] + DT_Y - 1) / DT_Y),
                    (unsigned)((cl.n[2] + DT_Z - 1) / DT_Z));
    if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidValue;
    if (mixed)
        k_deposit_df<<<grid, DEP_NT, deposit_smem(true, a.na), s>>>(a);
    else
        k_deposit64<<<grid, DEP_NT, deposit_smem(false, a.na), s>>>(a);
    return cudaGetLastError();
}

__device__ __forceinline__ bool inside_fp64(const DepArgs& a, double x, double y, double z, int t)
{
    const double* r = a.rec + (size_t)SPHERE_REC_DOUBLES * t;
    const double dx = x - r[RX], dy = y - r[RX + 1], dz = z - r[RX + 2];
    return fma(dx, dx, fma(dy, dy, dz * dz)) < r[RR] * r[RR];
}

// ---------------------------------------------------------------- deposit (FP64)
constexpr double ROUND_MAGIC64 = 6755399441055744.0;   // 1.5 * 2^52

// r of a squared distance: the hardware's approximate reciprocal square root (about 20 bits, not
// on the FP64 pipe) and one third-order step, t (1 - h)^(-1/2) = t (1 + h/2 + 3 h^2/8 + O(h^3))
__device__ __forceinline__ double root64(double r2)
{
    double s;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(s) : "d"(r2));
    const double t = r2 * s, h = fma(-t, s, 1.0);
    return fma(t * h, fma(h, 0.375, 0.5), t);
}

// e^{-zeta r}, c = EXP_N zeta / ln 2: k = round(c r), 2^(-k/EXP_N) from the table times 1 + p,
// p = e^x - 1 to third order (|x| <= 1.7e-4: the fourth is 3.5e-17): seven FP64 operations.  k at
// least kmax: returns false without the last four.
__device__ __forceinline__ bool exp64(double r, double c, int kmax, const double* __restrict__ T, double* e)
{
    constexpr double C1 = -LN2_N, C2 = 0.5 * LN2_N * LN2_N, C3 = -LN2_N * LN2_N * LN2_N / 6.0;
    const double y = fma(r, c, ROUND_MAGIC64);
    // (the bits of y grow with it, also beyond the range of a 32-bit k)
    if (__double_as_longlong(y) - 0x4338000000000000ll >= kmax) return false;
    const int k = __double2loint(y);
    const double f = fma(r, c, -(y - ROUND_MAGIC64));
    const double t = T[k & (EXP_N - 1)];
    const double v = fma(t, f * fma(f, fma(f, C3, C2), C1), t);
    *e = __hiloint2double(__double2hiint(v) - (k & ~(EXP_N - 1)) * ((1 << 20) / EXP_N), __double2loint(v));
    return true;
}

// FP64 form of inside_value below: s - N_i(r) + rho_ns + pseudo-density at the offset d
__device__ __noinline__ double inside_value64(double s, const double* __restrict__ rc, double dx, double dy, double dz,
                                              const double* __restrict__ T)
{
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const double r = r2 > 0.0 ? root64(r2) : 0.0, ir = r > 0.0 ? 1.0 / r : 0.0;
    double nbr = 0.0, e1 = 1.0;
#pragma unroll 1
    for (int q = 0; q < 3; q++) {
        const double z = rc[RZ + q], c = z * (1.0 / LN2_N), zr = z * r;
        double em = 0.0, ep = 0.0;
        exp64(r, c, 0x7fffffff, T, &em);
        exp64(r, -c, 0x7fffffff, T, &ep);
        if (q == 0) e1 = em;
        double shr;   // sinh(zeta r) / r
        if (zr > 0.3) {
            shr = 0.5 * (ep - em) * ir;
        } else {      // its series to (zeta r)^10
            const double x2 = zr * zr;
            shr = z * fma(x2, fma(x2, fma(x2, fma(x2, fma(x2, 1.0 / 39916800.0, 1.0 / 362880.0), 1.0 / 5040.0), 1.0 / 120.0),
                                  1.0 / 6.0), 1.0);
        }
        nbr += fma(2.0 * rc[RA + q], shr, -rc[RB + q] * (ep + em));
    }
    double ang = 0.0;
#pragma unroll
    for (int a = 4; a >= 0; a--) {
        double qy = 0.0;
#pragma unroll
        for (int b = 4 - a; b >= 0; b--) {
            double qz = rc[RP + poly_slot(a, b, 4 - a - b)];
#pragma unroll
            for (int c = 3 - a - b; c >= 0; c--) qz = fma(qz, dz, rc[RP + poly_slot(a, b, c)]);
            qy = b == 4 - a ? qz : fma(qy, dy, qz);
        }
        ang = a == 4 ? qy : fma(ang, dx, qy);
    }
    const double iR = 1.0 / rc[RR], tt = fma(-r2 * iR, iR, 1.0), z1 = rc[RZ];
    const double ns = z1 * z1 * z1 / (8.0 * PI) * e1 * tt * tt * ang;
    return s - nbr + ns + fma(fma(rc[RC + 2], r2, rc[RC + 1]), r2, rc[RC]);
}

// The FP64 deposit on the tiles of the FP32-pair form: atoms beyond the cut-off of a tile's
// bounding box dropped, the others sorted into those close enough for every term and for the test
// of the node inside the sphere (within 40 / the largest zeta, or their own radius), and the rest,
// whose largest-zeta terms are all dropped; the squares of the coordinate differences staged.  A
// pair takes 16 FP64 operations (two additions, five for the root, seven for e^{-zeta_0 r}, two
// for (W0 + W1 e) e) where a distance, a correctly rounded root and a library exponential per
// term took about 50; nodes inside spheres are queued for full warps.  Bound: FP64 issue (0.595 T
// per second here): Pd55 129^3 9912 -> 3356 us, Pd13 65^3 463 -> 210 us.
constexpr int D64_CH = 32;
__global__ void __launch_bounds__(DEP_NT) k_deposit64(DepArgs a)
{
    extern __shared__ int lists[];                  // [2][na]
    constexpr int ROWS = DT_X + DT_Y + DT_Z;
    __shared__ unsigned s_cnt[DEP_NT / 32];
    __shared__ int s_queued;
    __shared__ double s_x[ROWS];                    // node coordinates
    __shared__ double s_T[EXP_N];
    __shared__ __align__(16) double s_sq[D64_CH][ROWS];
    __shared__ __align__(16) double s_w[D64_CH][4];  // W, R^2
    const int tid = threadIdx.x, na = a.na;
    const int i0 = blockIdx.x * DT_X, j0 = blockIdx.y * DT_Y, k0 = blockIdx.z * DT_Z;
    const int li = tid & 7, lj = (tid >> 3) & 7, lk = tid >> 6;
    if (tid == 0) s_queued = 0;
    for (int t = tid; t < EXP_N; t += DEP_NT) s_T[t] = g_exp_tab64[t];
    if (tid < ROWS) {
        const int d = tid >> 3, first = d == 0 ? i0 : d == 1 ? j0 : k0;
        s_x[tid] = a.ax[d][min(first + (tid & 7), a.n[d] - 1)];
    }
    // the exponents are the same on every atom (checked by the sphere kernel)
    const float* f0 = reinterpret_cast<const float*>(a.rec + RF);
    const bool twice1 = __float_as_int(f0[F2]) & 1, twice2 = __float_as_int(f0[F2]) & 2;
    const float zf[3] = {f0[FZ], f0[FZ + 1], f0[FZ + 2]};
    const float zmin = fminf(fminf(zf[0], zf[1]), zf[2]), zmax = fmaxf(fmaxf(zf[0], zf[1]), zf[2]);
    const double c[3] = {a.rec[RZ] * (1.0 / LN2_N), a.rec[RZ + 1] * (1.0 / LN2_N), a.rec[RZ + 2] * (1.0 / LN2_N)};
    const int kcut = (int)(EXP_CUT / LN2_N);
    __syncthreads();
    // margins 1e-3 on the squared distances cover the rounding of the FP32 tests
    int count[2] = {0, 0};
    {
        const float cut = (float)EXP_CUT * (1.0f + 1e-3f);
        const float lim = (cut / zmin) * (cut / zmin), near2 = (cut / zmax) * (cut / zmax);
        const int w = tid >> 5, l = tid & 31;
        for (int base = 0; base < na; base += DEP_NT) {
            const int t = base + tid;
            int cls = 2;
            if (t < na) {
                const float4 p = *reinterpret_cast<const float4*>(a.rec + (size_t)SPHERE_REC_DOUBLES * t + RXF);
                const float dx = fmaxf(fmaxf((float)s_x[0] - p.x, p.x - (float)s_x[DT_X - 1]), 0.0f);
                const float dy = fmaxf(fmaxf((float)s_x[DT_X] - p.y, p.y - (float)s_x[DT_X + DT_Y - 1]), 0.0f);
                const float dz = fmaxf(fmaxf((float)s_x[DT_X + DT_Y] - p.z, p.z - (float)s_x[ROWS - 1]), 0.0f);
                const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                // (comparisons that a NaN position or exponent fails: such an atom is near)
                cls = !(d2 > p.w * (1.0f + 1e-3f)) || !(d2 > near2) ? 0 : d2 > lim ? 2 : 1;
            }
            const unsigned m0 = __ballot_sync(0xffffffffu, cls == 0), m1 = __ballot_sync(0xffffffffu, cls == 1);
            if (l == 0) s_cnt[w] = __popc(m0) | __popc(m1) << 16;
            __syncthreads();
            unsigned before = 0, all = 0;
            for (int v = 0; v < DEP_NT / 32; v++) {
                if (v == w) before = all;
                all += s_cnt[v];
            }
            if (cls < 2)
                lists[cls * na + (cls ? count[1] + (int)(before >> 16) : count[0] + (int)(before & 0xffff)) +
                      __popc((cls ? m1 : m0) & ((1u << l) - 1u))] = t;
            __syncthreads();
            count[0] += (int)(all & 0xffff);
            count[1] += (int)(all >> 16);
        }
    }
    const int i = i0 + li, j = j0 + lj, kA = k0 + lk, kB = kA + 4;
    const bool okA = i < a.n[0] && j < a.n[1] && kA < a.n[2], okB = okA && kB < a.n[2];
    double sA = 0.0, sB = 0.0;
    int ownA = -1, ownB = -1;
    // terms that a distant atom keeps: zeta_q below the largest
    const bool on0 = zf[0] < zmax, on1 = zf[1] < zmax, on2 = zf[2] < zmax;
    for (int pass = 0; pass < 2; pass++) {
        const int cnt = count[pass];
        const int* list = lists + pass * na;
        for (int c0 = 0; c0 < cnt; c0 += D64_CH) {
            const int ch = min(D64_CH, cnt - c0);
            __syncthreads();
            for (int t = tid; t < ch * ROWS; t += DEP_NT) {
                const int q = t / ROWS, r = t - q * ROWS;
                const double d = s_x[r] - a.rec[(size_t)SPHERE_REC_DOUBLES * list[c0 + q] + RX + (r >> 3)];
                s_sq[q][r] = d * d;
            }
            for (int t = tid; t < ch * 4; t += DEP_NT) {
                const double* r = a.rec + (size_t)SPHERE_REC_DOUBLES * list[c0 + (t >> 2)];
                s_w[t >> 2][t & 3] = (t & 3) < 3 ? r[RW + (t & 3)] : r[RR] * r[RR];
            }
            __syncthreads();
            if (pass == 0) {
                for (int q = 0; q < ch; q++) {
                    const double xy = s_sq[q][li] + s_sq[q][DT_X + lj];
                    const double w0 = s_w[q][0], w1 = s_w[q][1], w2 = s_w[q][2], R2 = s_w[q][3];
#pragma unroll
                    for (int n = 0; n < 2; n++) {
                        const double r2 = xy + s_sq[q][DT_X + DT_Y + lk + 4 * n];
                        if (r2 < R2 * (1.0 + 1e-14)) {   // decided on the unrounded differences near the surface
                            const int t = list[c0 + q];
                            if (r2 < R2 * (1.0 - 1e-14) ||
                                inside_fp64(a, s_x[li], s_x[DT_X + lj], s_x[DT_X + DT_Y + lk + 4 * n], t)) {
                                if (n) ownB = t;
                                else ownA = t;
                                continue;
                            }
                        }
                        const double r = r2 > 0.0 ? root64(r2) : 0.0;
                        double& s = n ? sB : sA;
                        double e0 = 0.0, e = 0.0;
                        const bool in0 = exp64(r, c[0], kcut, s_T, &e0);
                        if (in0) s = fma(w0, e0, s);
                        if (twice1) s = fma(w1, e0 * e0, s);
                        else if (exp64(r, c[1], kcut, s_T, &e)) s = fma(w1, e, s);
                        if (twice2) s = fma(w2, e0 * e0, s);
                        else if (exp64(r, c[2], kcut, s_T, &e)) s = fma(w2, e, s);
                    }
                }
            } else if (on0 && on1 && twice1 && !on2) {
                for (int q = 0; q < ch; q++) {
                    const double xy = s_sq[q][li] + s_sq[q][DT_X + lj];
                    const double w0 = s_w[q][0], w1 = s_w[q][1];
#pragma unroll
                    for (int n = 0; n < 2; n++) {
                        double e;
                        if (exp64(root64(xy + s_sq[q][DT_X + DT_Y + lk + 4 * n]), c[0], kcut, s_T, &e)) {
                            double& s = n ? sB : sA;
                            s = fma(fma(w1, e, w0), e, s);
                        }
                    }
                }
            } else {
                for (int q = 0; q < ch; q++) {
                    const double xy = s_sq[q][li] + s_sq[q][DT_X + lj];
#pragma unroll
                    for (int n = 0; n < 2; n++) {
                        const double r = root64(xy + s_sq[q][DT_X + DT_Y + lk + 4 * n]);
                        double& s = n ? sB : sA;
                        double e;
                        if (on0 && exp64(r, c[0], kcut, s_T, &e)) s = fma(s_w[q][0], e, s);
                        if (on1 && exp64(r, c[1], kcut, s_T, &e)) s = fma(s_w[q][1], e, s);
                        if (on2 && exp64(r, c[2], kcut, s_T, &e)) s = fma(s_w[q][2], e, s);
                    }
                }
            }
        }
    }
    auto store = [&](int P, double bv) {
        a.b[P] = bv;
        if ((__double2hiint(bv) & 0x7ff00000) == 0x7ff00000 && a.status) atomicMax(a.status, (int)LASTO_ERR_NONFINITE);
    };
    __syncthreads();   // the staged squares are not needed any more: their memory holds the queue
    double* q_sum = &s_sq[0][0];
    __shared__ int q_node[2 * DEP_NT][2];
    static_assert(sizeof(s_sq) >= 2 * DEP_NT * sizeof(double), "queue");
#pragma unroll
    for (int n = 0; n < 2; n++) {
        if (!(n ? okB : okA)) continue;
        const int own = n ? ownB : ownA, P = ((n ? kB : kA) * a.n[1] + j) * a.n[0] + i;   // (fewer than 2^31 nodes)
        if (a.owner) a.owner[P] = own;
        if (own < 0) {
            store(P, 4.0 * PI * (n ? sB : sA));
        } else {
            const int e = atomicAdd(&s_queued, 1);
            q_sum[e] = n ? sB : sA;
            q_node[e][0] = tid | n << 8;
            q_node[e][1] = own;
        }
    }
    __syncthreads();
    for (int e = tid; e < s_queued; e += DEP_NT) {
        const int node = q_node[e][0];
        const int ni = node & 7, nj = node >> 3 & 7, nk = (node >> 6 & 3) + 4 * (node >> 8);
        const double* rc = a.rec + (size_t)SPHERE_REC_DOUBLES * q_node[e][1];
        const double v = inside_value64(q_sum[e], rc, s_x[ni] - rc[RX], s_x[DT_X + nj] - rc[RX + 1],
                                        s_x[DT_X + DT_Y + nk] - rc[RX + 2], s_T);
        store(((k0 + nk) * a.n[1] + j0 + nj) * a.n[0] + i0 + ni, 4.0 * PI * v);
    }
}

// ---------------------------------------------------------------- deposit (FP32 pairs)
constexpr float ROUND_MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer in the low bits

// the power of two 2^-floor(k / EXP_N) from the bits of k + ROUND_MAGIC
__device__ __forceinline__ float pow2_of(int ki)
{
    return __int_as_float(0x3f800000 - (ki & ~(EXP_N - 1)) * ((1 << 23) / EXP_N));
}

// r = r0 + r1 of a squared distance h + l (h >= 0): the FP32 root by the approximate reciprocal
// square root and one Newton correction, relative error about 2^-46
__device__ __forceinline__ df root(float h, float l)
{
    const float s = h > 0.0f ? rsqrtf(h) : 0.0f;
    const float r0 = h * s;
    return {r0, (fmaf(-r0, r0, h) + l) * (0.5f * s)};
}

// y = c r in units of ln 2 / EXP_N (c = EXP_N zeta / ln 2 as a double-float), unevaluated
__device__ __forceinline__ df exponent(df r, float ch, float cl)
{
    const float y0 = r.h * ch;
    return {y0, fmaf(r.l, ch, fmaf(r.h, cl, fmaf(r.h, ch, -y0)))};
}

// e^{-y ln2/EXP_N} to double-float accuracy: k = round(y), 2^(-k/EXP_N) from the table (Tang's
// table-driven reduction) times 1 + g, |g| <= 1.7e-4: g's linear term as a double-float, its
// quadratic and cubic terms in FP32
__device__ __forceinline__ df exp_pair(df y, const float2* __restrict__ T)
{
    const float km = y.h + ROUND_MAGIC;
    const df f = dfa::fast_two_sum(y.h - (km - ROUND_MAGIC), y.l);
    const int ki = __float_as_int(km);
    const float2 t = T[ki & (EXP_N - 1)];
    const float gh = -LN2_H * f.h;
    float gl = fmaf(-LN2_H, f.h, -gh);
    gl = fmaf(-LN2_L, f.h, gl);
    gl = fmaf(-LN2_H, f.l, gl);
    gl = fmaf(gh * gh, fmaf(gh, 1.0f / 6.0f, 0.5f), gl);
    const float p = t.x * gh;
    const float lo = fmaf(t.x, gh, -p) + fmaf(t.x, gl, fmaf(t.y, gh, t.y));
    const float e = t.x + p;
    const float sc = pow2_of(ki);
    return {e * sc, (((t.x - e) + p) + lo) * sc};
}

// the same to about 35 bits (an error below 4e-11; four times that with 512 entries): 1 + g with g in FP32, the pair left unevaluated
__device__ __forceinline__ df exp_mid(df y, const float2* __restrict__ T)
{
    constexpr float C1 = -LN2_H, C2 = 0.5f * LN2_H * LN2_H, C3 = -LN2_H * LN2_H * LN2_H / 6.0f;
    const float km = y.h + ROUND_MAGIC;
    const float f = (y.h - (km - ROUND_MAGIC)) + y.l;
    const int ki = __float_as_int(km);
    const float2 t = T[ki & (EXP_N - 1)];
    const float g = f * fmaf(f, fmaf(f, C3, C2), C1);
    const float sc = pow2_of(ki);
    return {t.x * sc, fmaf(t.x, g, t.y) * sc};
}

// s += w e, the sum left as an unevaluated pair
__device__ __forceinline__ void add_product(df& s, float wh, float wl, df e)
{
    const float p = wh * e.h;
    const float l = fmaf(wh, e.h, -p) + fmaf(wh, e.l, wl * e.h);
    const df t = dfa::two_sum(s.h, p);
    s.h = t.h;
    s.l += t.l + l;
}

// e^{-x ln 2}
__device__ __forceinline__ float ex2_neg(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(-x));
    return r;
}

// p - o of two three-float numbers, to double-float accuracy of the difference
__device__ __forceinline__ df diff3(const float* p, const float* o)
{
    const df s = dfa::two_sum(p[0], -o[0]), t = dfa::two_sum(p[1], -o[1]);
    df u = dfa::two_sum(s.l, t.h);
    u.l += t.l + (p[2] - o[2]);
    df w = dfa::two_sum(s.h, u.h);
    w.l += u.l;
    return dfa::fast_two_sum(w.h, w.l);
}

struct DfExps {
    float ch[3], cl[3];   // EXP_N zeta / ln 2
    bool twice[3];        // zeta_q exactly twice zeta_0
};

// s = s x + c in double-floats
__device__ __forceinline__ df mul_add(df s, df x, df c)
{
    const float p = s.h * x.h;
    const float e = fmaf(s.h, x.h, -p) + fmaf(s.h, x.l, s.l * x.h);
    df t = dfa::two_sum(p, c.h);
    t.l += e + c.l;
    return dfa::fast_two_sum(t.h, t.l);
}

// n_e's monopole swap and nonspherical part at a node inside its sphere, added to the neighbours'
// Slater sum s: s - N_i(r) + rho_ns + pseudo-density.  d: node - centre.  The nonspherical part is
// its polynomial in d by nested Horner steps (34 multiply-adds where the sum over the harmonics'
// 55 monomials took four products each); the pseudo-density, ten times the result in places, is
// FP64.
__device__ __noinline__ double inside_value(df s, const double* __restrict__ rc, df dx, df dy, df dz, DfExps ex,
                                            const float2* __restrict__ T)
{
    const float2* f2 = reinterpret_cast<const float2*>(reinterpret_cast<const float*>(rc + RF));
    auto pair = [&](int o) {
        const float2 v = f2[o >> 1];
        return df{v.x, v.y};
    };
    const df r2 = dfa::add(dfa::add(dfa::sqr(dx), dfa::sqr(dy)), dfa::sqr(dz));
    const df rr = root(r2.h, r2.l), r = dfa::fast_two_sum(rr.h, rr.l);
    df nbr = {0.0f, 0.0f}, e1 = {1.0f, 0.0f};
#pragma unroll 1
    for (int q = 0; q < 3; q++) {
        const float ch = q == 0 ? ex.ch[0] : q == 1 ? ex.ch[1] : ex.ch[2];
        const float cl = q == 0 ? ex.cl[0] : q == 1 ? ex.cl[1] : ex.cl[2];
        const df y = exponent(r, ch, cl);
        const df em = exp_pair(y, T), ep = exp_pair(dfa::neg(y), T);
        if (q == 0) e1 = em;
        const df A2 = pair(FA + 2 * q), B2 = pair(FB + 2 * q);
        df shr;   // 2 sinh(zeta r) / r
        if (y.h > 1e-3f / LN2_H) {
            shr = dfa::div(dfa::add(ep, dfa::neg(em)), r);
        } else {
            const df zt = dfa::from_double(rc[RZ + q]);
            const float zr = zt.h * r.h;
            shr = dfa::mul(df{2.0f * zt.h, 2.0f * zt.l}, dfa::add_f(df{1.0f, 0.0f}, zr * zr * (1.0f / 6.0f)));
        }
        const df t = dfa::add(dfa::mul(A2, shr), dfa::neg(dfa::mul(B2, dfa::add(ep, em))));
        nbr = dfa::add(nbr, df{0.5f * t.h, 0.5f * t.l});
    }
    // nonspherical part: slater(zeta_1, r) (1 - r^2/R^2)^2 sum c_lm (r/R)^l y_lm
    df ang = {0.0f, 0.0f};
#pragma unroll
    for (int a = 4; a >= 0; a--) {
        df qy = {0.0f, 0.0f};
#pragma unroll
        for (int b = 4 - a; b >= 0; b--) {
            df qz = pair(FH + 2 * poly_slot(a, b, 4 - a - b));
#pragma unroll
            for (int c = 3 - a - b; c >= 0; c--) qz = mul_add(qz, dz, pair(FH + 2 * poly_slot(a, b, c)));
            qy = b == 4 - a ? qz : mul_add(qy, dy, qz);
        }
        ang = a == 4 ? qy : mul_add(ang, dx, qy);
    }
    const df tt = dfa::add_f(dfa::neg(dfa::mul(r2, pair(FR))), 1.0f);
    const df radial = dfa::mul(dfa::mul(pair(FN), e1), dfa::sqr(tt));
    s = dfa::add(dfa::add(s, dfa::neg(nbr)), dfa::mul(radial, ang));
    const double rsq = dfa::to_double(r2);
    return dfa::to_double(s) + fma(fma(rc[RC + 2], rsq, rc[RC + 1]), rsq, rc[RC]);
}

// The FP32-pair deposit works on 8 x 8 x 8 tiles of nodes (a warp covers 8 x 4 x 1, each thread
// two nodes four planes apart).  Once per block, every atom is dropped (beyond the cut-off of the
// tile's bounding box) or sorted by its distance from that box into four lists, each taken
// through a loop of its own in which every lane does the same work:
//   near    the double-float sum, with the test for the node inside the atom's sphere;
//   mid     every node beyond NEAR_T / zeta_min of the atom: e^{-zeta r} to about 35 bits;
//   outer   every node beyond MID_T / zeta_min: the FP32 exponential of the accurate exponent;
//   far     every node beyond FAR_T / zeta_min: plain FP32.
// Near, mid and outer atoms are staged as the squares of the 24 coordinate differences of the tile's
// planes, so that a pair's squared distance costs two or four additions per node instead of three
// double-float subtractions, squares and sums: near as double-floats, the others as a multiple of a
// common power of two plus a remainder, whose high parts add exactly.  Bound: instruction issue.
// Before this form (three branches inside one loop over the atoms, 8 x 8 x 4 tiles): Pd147 161^3
// 1308 us, Pd561 385^3 29.7 ms, Pd55 129^3 461 us; now 479 us, 10.8 ms and 175 us (0.81 of the issue
// rate), with a quarter of the error (Pd147: 5.8e-13 -> 1.6e-13 of the 2-norm).
constexpr int DF_CH = 32;    // near or mid atoms staged at a time
constexpr int DF_FCH = 128;  // far atoms staged at a time
constexpr int DF_ROWS = DT_X + DT_Y + DT_Z;

__global__ void __launch_bounds__(DEP_NT, 3) k_deposit_df(DepArgs a)
{
    extern __shared__ int lists[];                 // near, mid, outer, far atom indices [4][na]
    __shared__ unsigned long long s_cnt[DEP_NT / 32];   // four 16-bit counts
    __shared__ float2 s_off[DF_ROWS];              // node coordinate - tile origin, double-float
    __shared__ float2 s_T[EXP_N];
    __shared__ float2 s_D[DF_CH][3];               // atom - tile origin
    __shared__ __align__(16) float2 s_sq[DF_CH][DF_ROWS];
    __shared__ __align__(16) float s_w[DF_CH][8];  // W pairs, R^2, -
    __shared__ __align__(16) float s_far[DF_FCH][8];
    __shared__ int s_queued;
    __shared__ float s_org[3][3], s_box[3][2];     // the tile origin as three floats, the tile's bounds
    const int tid = threadIdx.x, na = a.na;
    const int i0 = blockIdx.x * DT_X, j0 = blockIdx.y * DT_Y, k0 = blockIdx.z * DT_Z;
    const int li = tid & 7, lj = (tid >> 3) & 7, lk = tid >> 6;
    if (tid == 0) s_queued = 0;
    for (int t = tid; t < EXP_N; t += DEP_NT) s_T[t] = g_exp_tab[t];
    // tile origin: its first node; offsets from it keep the pairs' magnitudes small.  (FP64 work
    // is kept to these two warps and to what a node's own sphere needs: the pipe is narrow enough
    // that conversions and differences per atom in every tile kept it 46 % busy and cost a third
    // of the kernel's time; the sphere records hold float forms instead.)
    if (tid < DF_ROWS) {
        const int d = tid >> 3, o = tid & 7, first = d == 0 ? i0 : d == 1 ? j0 : k0;
        const df v = dfa::from_double(a.ax[d][min(first + o, a.n[d] - 1)] - a.ax[d][first]);
        s_off[tid] = make_float2(v.h, v.l);
    } else if (tid >= 32 && tid < 35) {
        const int d = tid - 32, first = d == 0 ? i0 : d == 1 ? j0 : k0;
        three_floats(a.ax[d][first], s_org[d]);
        s_box[d][0] = s_org[d][0];
        s_box[d][1] = (float)a.ax[d][min(first + 7, a.n[d] - 1)];
    }
    // the exponents are the same on every atom (checked by the sphere kernel)
    const float* f0 = reinterpret_cast<const float*>(a.rec + RF);
    const int twice = __float_as_int(f0[F2]);
    float zt[3], zmin = 1e30f;
    DfExps ex;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        zt[q] = f0[FZ + q];
        zmin = fminf(zmin, zt[q]);
        ex.ch[q] = f0[FC + 2 * q];
        ex.cl[q] = f0[FC + 2 * q + 1];
        ex.twice[q] = q > 0 && (twice >> (q - 1) & 1);
    }
    __syncthreads();
    const float cut = DF_EXP_CUT / zmin, cut2 = cut * cut * (1.0f + 1e-5f);
    // Sort the atoms in ascending order, tested in FP32 on the records' float copies of the
    // positions.  The margins 1e-3 on the squared distances cover the rounding of these tests
    // (~1e-6 relative): an atom dropped here is beyond the cut-off at every node of the tile, and
    // a mid or far atom is beyond its limit, and beyond its own sphere, at every node.
    int count[4] = {0, 0, 0, 0};
    {
        const float lim = cut2 * (1.0f + 1e-3f);
        const float near2 = (NEAR_T / zmin) * (NEAR_T / zmin) * (1.0f + 1e-3f);
        const float mid2 = (MID_T / zmin) * (MID_T / zmin) * (1.0f + 1e-3f);
        const float far2 = (FAR_T / zmin) * (FAR_T / zmin) * (1.0f + 1e-3f);
        const float bx0 = s_box[0][0], bx1 = s_box[0][1], by0 = s_box[1][0], by1 = s_box[1][1];
        const float bz0 = s_box[2][0], bz1 = s_box[2][1];
        const int w = tid >> 5, l = tid & 31;
        for (int base = 0; base < na; base += DEP_NT) {
            const int t = base + tid;
            int cls = 4;
            if (t < na) {
                const float4 c = *reinterpret_cast<const float4*>(a.rec + (size_t)SPHERE_REC_DOUBLES * t + RXF);
                const float dx = fmaxf(fmaxf(bx0 - c.x, c.x - bx1), 0.0f);
                const float dy = fmaxf(fmaxf(by0 - c.y, c.y - by1), 0.0f);
                const float dz = fmaxf(fmaxf(bz0 - c.z, c.z - bz1), 0.0f);
                const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                // (comparisons that a NaN position or exponent fails: such an atom is near)
                cls = !(d2 > c.w * (1.0f + 1e-3f)) ? 0
                      : d2 > lim                   ? 4
                      : d2 > far2                  ? 3
                      : d2 > mid2                  ? 2
                      : d2 > near2                 ? 1
                                                   : 0;
            }
            unsigned mine = 0;   // lanes of this lane's class
            unsigned long long cnt = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const unsigned m = __ballot_sync(0xffffffffu, cls == q);
                if (cls == q) mine = m;
                cnt |= (unsigned long long)__popc(m) << (16 * q);
            }
            if (l == 0) s_cnt[w] = cnt;
            __syncthreads();
            unsigned long long before = 0, all = 0;
            for (int v = 0; v < DEP_NT / 32; v++) {
                if (v == w) before = all;
                all += s_cnt[v];
            }
            if (cls < 4) {
                const int c0 = cls == 0 ? count[0] : cls == 1 ? count[1] : cls == 2 ? count[2] : count[3];
                lists[cls * na + c0 + (int)(before >> (16 * cls) & 0xffff) + __popc(mine & ((1u << l) - 1u))] = t;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; q++) count[q] += (int)(all >> (16 * q) & 0xffff);
        }
    }
    const int i = i0 + li, j = j0 + lj, kA = k0 + lk, kB = kA + 4;
    const bool okA = i < a.n[0] && j < a.n[1] && kA < a.n[2], okB = okA && kB < a.n[2];
    df sA = {0.0f, 0.0f}, sB = {0.0f, 0.0f};   // the double-float sums
    float fA = 0.0f, fB = 0.0f;                // the outer and far atoms' FP32 sums
    int ownA = -1, ownB = -1;

    // ---- near, mid and outer atoms, DF_CH at a time
    // high parts of the mid and outer squares: multiples of g = 2^(e - 23) with 2^e >= 4 cut^2, rounded by
    // adding 1.5 * 2^23 g; three of them add exactly for distances up to twice the cut-off
    const float grid_magic = __int_as_float(((__float_as_int(4.0f * cut2) >> 23) + 1) << 23) * 1.5f;
    for (int pass = 0; pass < 3; pass++) {
        const int cnt = pass == 0 ? count[0] : pass == 1 ? count[1] : count[2];
        const int* list = lists + pass * na;
        for (int c0 = 0; c0 < cnt; c0 += DF_CH) {
            const int ch = min(DF_CH, cnt - c0);
            __syncthreads();
            for (int t = tid; t < ch * 8; t += DEP_NT) {
                const int q = t >> 3, f = t & 7;
                const double* r = a.rec + (size_t)SPHERE_REC_DOUBLES * list[c0 + q];
                const float* fr = reinterpret_cast<const float*>(r + RF);
                if (f < 3) {
                    const df D = diff3(fr + FP + 3 * f, s_org[f]);
                    s_D[q][f] = make_float2(D.h, D.l);
                } else if (f < 6) {
                    s_w[q][2 * (f - 3)] = fr[FW + 2 * (f - 3)];
                    s_w[q][2 * (f - 3) + 1] = fr[FW + 2 * (f - 3) + 1];
                } else if (f == 6) {
                    s_w[q][6] = reinterpret_cast<const float*>(r + RXF)[3];
                }
            }
            __syncthreads();
            for (int t = tid; t < ch * DF_ROWS; t += DEP_NT) {
                const int q = t / DF_ROWS, c = t - q * DF_ROWS;
                const float2 o = s_off[c], D = s_D[q][c >> 3];
                df d = dfa::sqr(dfa::add(df{o.x, o.y}, df{-D.x, -D.y}));
                if (pass > 0) {
                    const float hi = (d.h + grid_magic) - grid_magic;
                    d.l += d.h - hi;
                    d.h = hi;
                }
                s_sq[q][c] = make_float2(d.h, d.l);
            }
            __syncthreads();
            if (pass == 0) {
                for (int q = 0; q < ch; q++) {
                    const float2 X = s_sq[q][li], Y = s_sq[q][DT_X + lj];
                    const float4 W01 = *reinterpret_cast<const float4*>(&s_w[q][0]);
                    const float4 W2R = *reinterpret_cast<const float4*>(&s_w[q][4]);
                    const df xy = dfa::add(df{X.x, X.y}, df{Y.x, Y.y});
#pragma unroll
                    for (int n = 0; n < 2; n++) {
                        const float2 Z = s_sq[q][DT_X + DT_Y + lk + 4 * n];
                        const df r2 = dfa::add(xy, df{Z.x, Z.y});
                        if (r2.h > cut2) continue;
                        if (r2.h < W2R.z * (1.0f + 2e-6f)) {
                            const int t = list[c0 + q];
                            const bool in = (r2.h < W2R.z * (1.0f - 2e-6f)) ||
                                            inside_fp64(a, a.ax[0][min(i, a.n[0] - 1)], a.ax[1][min(j, a.n[1] - 1)],
                                                        a.ax[2][min(n ? kB : kA, a.n[2] - 1)], t);
                            if (in) {
                                if (n) ownB = t;
                                else ownA = t;
                                continue;
                            }
                        }
                        const df r = root(r2.h, r2.l);
                        df& s = n ? sB : sA;
                        df e0 = {0.0f, 0.0f};
#pragma unroll
                        for (int v = 0; v < 3; v++) {
                            if (zt[v] * r.h >= DF_EXP_CUT) continue;
                            df e;
                            if (v > 0 && ex.twice[v] && zt[0] * r.h < DF_EXP_CUT) {
                                e = dfa::sqr(e0);   // e^{-2 zeta_0 r}
                            } else {
                                e = exp_pair(exponent(r, ex.ch[v], ex.cl[v]), s_T);
                            }
                            if (v == 0) e0 = e;
                            add_product(s, v == 0 ? W01.x : v == 1 ? W01.z : W2R.x,
                                        v == 0 ? W01.y : v == 1 ? W01.w : W2R.y, e);
                        }
                    }
                }
            } else if (pass == 1) {
                // a term that is beyond the cut-off at every mid distance is dropped for all of
                // them; nodes of a mid atom beyond 2^-120 are held there (the exponent's range)
                const float rmin = NEAR_T / zmin, ymax = 120.0f * EXP_N;
                const bool on0 = zt[0] * rmin < DF_EXP_CUT, on1 = zt[1] * rmin < DF_EXP_CUT,
                           on2 = zt[2] * rmin < DF_EXP_CUT;
                if (on0 && on1 && ex.twice[1] && !on2) {
                    // (W0 + W1 e) e, e = e^{-zeta_0 r}
                    for (int q = 0; q < ch; q++) {
                        const float2 X = s_sq[q][li], Y = s_sq[q][DT_X + lj];
                        const float4 W = *reinterpret_cast<const float4*>(&s_w[q][0]);
                        const float xh = X.x + Y.x, xl = X.y + Y.y;
#pragma unroll
                        for (int n = 0; n < 2; n++) {
                            const float2 Z = s_sq[q][DT_X + DT_Y + lk + 4 * n];
                            df y = exponent(root(xh + Z.x, xl + Z.y), ex.ch[0], ex.cl[0]);
                            y.h = fminf(y.h, ymax);
                            const df e = exp_mid(y, s_T);
                            const float p = W.z * e.h;
                            df v = dfa::two_sum(W.x, p);
                            v.l += W.y + (fmaf(W.z, e.h, -p) + fmaf(W.z, e.l, W.w * e.h));
                            add_product(n ? sB : sA, v.h, v.l, e);
                        }
                    }
                } else {
                    for (int q = 0; q < ch; q++) {
                        const float2 X = s_sq[q][li], Y = s_sq[q][DT_X + lj];
                        const float xh = X.x + Y.x, xl = X.y + Y.y;
#pragma unroll
                        for (int n = 0; n < 2; n++) {
                            const float2 Z = s_sq[q][DT_X + DT_Y + lk + 4 * n];
                            const df r = root(xh + Z.x, xl + Z.y);
#pragma unroll
                            for (int v = 0; v < 3; v++) {
                                if (!(v == 0 ? on0 : v == 1 ? on1 : on2)) continue;
                                df y = exponent(r, ex.ch[v], ex.cl[v]);
                                y.h = fminf(y.h, ymax);
                                add_product(n ? sB : sA, s_w[q][2 * v], s_w[q][2 * v + 1], exp_mid(y, s_T));
                            }
                        }
                    }
                }
            } else {
                // e^{-zeta r} = 2^-y0 (1 - y1 ln 2), y0 + y1 = zeta r / ln 2
                const float rmin = MID_T / zmin;
                const bool on0 = zt[0] * rmin < DF_EXP_CUT, on1 = zt[1] * rmin < DF_EXP_CUT,
                           on2 = zt[2] * rmin < DF_EXP_CUT;
                constexpr float LN2 = 0.693147181f, S = 1.0f / EXP_N;
                if (on0 && (!on1 || ex.twice[1]) && !on2) {
                    const float ch0 = ex.ch[0] * S, cl0 = ex.cl[0] * S;
                    for (int q = 0; q < ch; q++) {
                        const float2 X = s_sq[q][li], Y = s_sq[q][DT_X + lj];
                        const float4 W = *reinterpret_cast<const float4*>(&s_w[q][0]);
                        const float xh = X.x + Y.x, xl = X.y + Y.y, w1 = on1 ? W.z : 0.0f;
#pragma unroll
                        for (int n = 0; n < 2; n++) {
                            const float2 Z = s_sq[q][DT_X + DT_Y + lk + 4 * n];
                            const df y = exponent(root(xh + Z.x, xl + Z.y), ch0, cl0);
                            const float e0 = ex2_neg(y.h), e = fmaf(-LN2 * y.l, e0, e0);
                            float& f = n ? fB : fA;
                            f = fmaf(fmaf(w1, e, W.x), e, f);
                        }
                    }
                } else {
                    for (int q = 0; q < ch; q++) {
                        const float2 X = s_sq[q][li], Y = s_sq[q][DT_X + lj];
                        const float xh = X.x + Y.x, xl = X.y + Y.y;
#pragma unroll
                        for (int n = 0; n < 2; n++) {
                            const float2 Z = s_sq[q][DT_X + DT_Y + lk + 4 * n];
                            const df r = root(xh + Z.x, xl + Z.y);
#pragma unroll
                            for (int v = 0; v < 3; v++) {
                                if (!(v == 0 ? on0 : v == 1 ? on1 : on2)) continue;
                                const df y = exponent(r, ex.ch[v] * S, ex.cl[v] * S);
                                const float e0 = ex2_neg(y.h);
                                float& f = n ? fB : fA;
                                f = fmaf(s_w[q][2 * v], fmaf(-LN2 * y.l, e0, e0), f);
                            }
                        }
                    }
                }
            }
            // the low parts gather the terms below the high parts' last place: kept small, as their own
            // rounding is FP32
            sA = dfa::fast_two_sum(sA.h, sA.l);
            sB = dfa::fast_two_sum(sB.h, sB.l);
        }
    }

    // ---- far atoms: their terms, each below e^-FAR_T of its weight, in plain FP32 and added to
    // the double-float sum once.  The distance comes from the FP32 roundings of the two offsets
    // (one subtraction per axis): the atom's offset is at most r plus the tile's extent, so r
    // carries a relative error of ~1.5e-7.  A term that is beyond the cut-off at every far
    // distance is dropped for all of them.
    {
        const bool on0 = zt[0] * (FAR_T / zmin) < DF_EXP_CUT, on1 = zt[1] * (FAR_T / zmin) < DF_EXP_CUT,
                   on2 = zt[2] * (FAR_T / zmin) < DF_EXP_CUT;
        const float l2e = 1.44269504f;
        const float c0f = zt[0] * l2e, c1f = zt[1] * l2e, c2f = zt[2] * l2e;
        const float pxf = s_off[li].x, pyf = s_off[DT_X + lj].x;
        const float pzA = s_off[DT_X + DT_Y + lk].x, pzB = s_off[DT_X + DT_Y + lk + 4].x;
        for (int c0 = 0; c0 < count[3]; c0 += DF_FCH) {
            const int ch = min(DF_FCH, count[3] - c0);
            __syncthreads();
            for (int t = tid; t < ch; t += DEP_NT) {
                const float* fr = reinterpret_cast<const float*>(
                    a.rec + (size_t)SPHERE_REC_DOUBLES * lists[3 * na + c0 + t] + RF);
                float D[3];
#pragma unroll
                for (int d = 0; d < 3; d++)
                    D[d] = (fr[FP + 3 * d] - s_org[d][0]) + (fr[FP + 3 * d + 1] - s_org[d][1]);
                *reinterpret_cast<float4*>(&s_far[t][0]) = make_float4(D[0], D[1], D[2], fr[FW]);
                s_far[t][4] = fr[FW + 2];
                s_far[t][5] = fr[FW + 4];
            }
            __syncthreads();
            if (on0 && !on1 && !on2) {
#pragma unroll 4
                for (int q = 0; q < ch; q++) {
                    const float4 A = *reinterpret_cast<const float4*>(&s_far[q][0]);
                    const float fx = pxf - A.x, fy = pyf - A.y, za = pzA - A.z, zb = pzB - A.z;
                    const float xy = fmaf(fx, fx, fy * fy);
                    const float ra = fmaf(za, za, xy), rb = fmaf(zb, zb, xy);
                    fA = fmaf(A.w, ex2_neg(c0f * (ra * rsqrtf(ra))), fA);
                    fB = fmaf(A.w, ex2_neg(c0f * (rb * rsqrtf(rb))), fB);
                }
            } else {
                for (int q = 0; q < ch; q++) {
                    const float4 A = *reinterpret_cast<const float4*>(&s_far[q][0]);
                    const float fx = pxf - A.x, fy = pyf - A.y, za = pzA - A.z, zb = pzB - A.z;
                    const float xy = fmaf(fx, fx, fy * fy);
                    const float ra2 = fmaf(za, za, xy), rb2 = fmaf(zb, zb, xy);
                    const float ra = ra2 * rsqrtf(ra2), rb = rb2 * rsqrtf(rb2);
                    if (on0) {
                        fA = fmaf(A.w, ex2_neg(c0f * ra), fA);
                        fB = fmaf(A.w, ex2_neg(c0f * rb), fB);
                    }
                    if (on1) {
                        fA = fmaf(s_far[q][4], ex2_neg(c1f * ra), fA);
                        fB = fmaf(s_far[q][4], ex2_neg(c1f * rb), fB);
                    }
                    if (on2) {
                        fA = fmaf(s_far[q][5], ex2_neg(c2f * ra), fA);
                        fB = fmaf(s_far[q][5], ex2_neg(c2f * rb), fB);
                    }
                }
            }
        }
    }

    // nodes outside every sphere are done; the others' sums go to a queue that full warps take
    // (one to ten lanes of a warp are inside a sphere where any are)
    auto store = [&](int P, double bv) {
        a.b[P] = bv;
        // (infinities and NaN by the exponent's bits)
        if ((__double2hiint(bv) & 0x7ff00000) == 0x7ff00000 && a.status) atomicMax(a.status, (int)LASTO_ERR_NONFINITE);
    };
    const df fourpi = dfa::from_double(4.0 * PI);
    __syncthreads();   // the staged atoms are not needed any more: their memory holds the queue
    float2* q_sum = &s_sq[0][0];
    int* q_node = reinterpret_cast<int*>(&s_far[0][0]);   // place in the tile, then the atom
    static_assert(sizeof(s_sq) >= 2 * DEP_NT * sizeof(float2) && sizeof(s_far) >= 4 * DEP_NT * sizeof(int), "queue");
#pragma unroll
    for (int n = 0; n < 2; n++) {
        if (!(n ? okB : okA)) continue;
        const int own = n ? ownB : ownA;
        df s = n ? sB : sA;
        s = dfa::add_f(dfa::fast_two_sum(s.h, s.l), n ? fB : fA);
        const int P = ((n ? kB : kA) * a.n[1] + j) * a.n[0] + i;   // (grids hold fewer than 2^31 nodes)
        if (a.owner) a.owner[P] = own;
        if (own < 0) {
            store(P, dfa::to_double(dfa::mul(fourpi, s)));
        } else {
            const int e = atomicAdd(&s_queued, 1);
            q_sum[e] = make_float2(s.h, s.l);
            q_node[2 * e] = tid | n << 8;
            q_node[2 * e + 1] = own;
        }
    }
    __syncthreads();
    for (int e = tid; e < s_queued; e += DEP_NT) {
        const int node = q_node[2 * e];
        const int ni = node & 7, nj = node >> 3 & 7, nk = (node >> 6 & 3) + 4 * (node >> 8);
        const double* rc = a.rec + (size_t)SPHERE_REC_DOUBLES * q_node[2 * e + 1];
        const float* fr = reinterpret_cast<const float*>(rc + RF) + FP;
        df d[3];
#pragma unroll
        for (int v = 0; v < 3; v++) {
            const df D = diff3(fr + 3 * v, s_org[v]);
            const float2 o = s_off[v == 0 ? ni : v == 1 ? DT_X + nj : DT_X + DT_Y + nk];
            d[v] = dfa::add(df{o.x, o.y}, dfa::neg(D));
        }
        const double v = inside_value(df{q_sum[e].x, q_sum[e].y}, rc, d[0], d[1], d[2], ex, s_T);
        store(((k0 + nk) * a.n[1] + j0 + nj) * a.n[0] + i0 + ni, 4.0 * PI * v);
    }
}

void init_device_constants()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return;
    {
        std::lock_guard<std::mutex> lock(g_constants_mutex);
        if (g_constants_done[dev]) return;
    }
    // the index lists of the largest cluster.  (Dynamic and static memory share one limit: a request beyond
    // it is refused, and the kernel keeps the default, 48 KiB for both.)
    bool ok = ensure_monomials() == cudaSuccess;
    ok = cudaFuncSetAttribute(k_deposit64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)deposit_smem(false, DEP64_MAX_ATOMS)) ==
             cudaSuccess && ok;
    ok = cudaFuncSetAttribute(k_deposit_df, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)deposit_smem(true, DF_MAX_ATOMS)) ==
             cudaSuccess && ok;
    init_mg_attributes();
    init_direct_attributes();
    init_slab_attributes();
    init_wave_attributes();
    std::lock_guard<std::mutex> lock(g_constants_mutex);
    g_constants_done[dev] = ok;   // (else the next call tries again)
}

// ---------------------------------------------------------------- boundary multipoles
// Q_lm = sum (b/4pi) vol S_lm(node - centre).  S_lm is a polynomial of degree l in
// (x, y, z) and vol a product of per-axis dual lengths, so the sum factorises:
// per-column y-moments (5 FMAs per node), then x and z contractions, then the monomial
// expansion of each S_lm.

// tab[axis][a][i] = (x_i - c)^a * dual_i, a = 0..4 (blockIdx.y: the axis)
__global__ void k_moment_tables(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                                int nx, int ny, int nz, double cx, double cy, double cz, double* __restrict__ tab)
{
    const int d = blockIdx.y, n = d == 0 ? nx : d == 1 ? ny : nz;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* a = d == 0 ? x : d == 1 ? y : z;
    const double c = d == 0 ? cx : d == 1 ? cy : cz;
    double* out = tab + 5 * (size_t)(d == 0 ? 0 : d == 1 ? nx : nx + ny);
    double p = (i == 0) ? 0.5 * (a[1] - a[0]) : (i == n - 1) ? 0.5 * (a[n - 1] - a[n - 2]) : 0.5 * (a[i + 1] - a[i - 1]);
    const double e = a[i] - c;
    for (int q = 0; q < 5; q++) {
        out[(size_t)q * n + i] = p;
        p *= e;
    }
}

// pairs (a, b) with a + b <= 4, in a fixed order
__constant__ int c_ab[15][2] = {{0, 0}, {0, 1}, {0, 2}, {0, 3}, {0, 4}, {1, 0}, {1, 1}, {1, 2}, {1, 3},
                                {2, 0}, {2, 1}, {2, 2}, {3, 0}, {3, 1}, {4, 0}};

// plane[ab][k] = sum_ij xm[a][i] ym[b][j] b[k, j, i]: one block per plane.  A thread sums the five
// y-moments of a column i over one of JG ranges of j (consecutive lanes read consecutive nodes; a
// sum along x would need a shuffle tree per row, and FP64 additions are scarce on this GPU), the
// block adds the ranges and contracts the columns.  Columns in tiles of MOM_T.  Bound: 5 FP64
// operations per node (129^3: 18 us).  With the tables and the z contraction 129^3 100 -> 41 us (before:
// a thread per row, uncoalesced, then a thread per plane and pair), 385^3 710 -> 624 us.
constexpr int MOM_T = 1024;

__global__ void __launch_bounds__(MOM_T) k_plane_moments(const double* __restrict__ b, int nx, int ny, int nz, int JG,
                                                        const double* __restrict__ xm, const double* __restrict__ ym,
                                                        double* __restrict__ plane)
{
    extern __shared__ double s_col[];   // [5][JG][columns of a tile]
    __shared__ double s_ab[15];
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int jl = (ny + JG - 1) / JG;
    if (tid < 15) s_ab[tid] = 0.0;
    for (int i0 = 0; i0 < nx; i0 += MOM_T) {
        const int ni = min(MOM_T, nx - i0);
        for (int e = tid; e < ni * JG; e += blockDim.x) {
            const int g = e / ni, i = e - g * ni, j1 = min(ny, (g + 1) * jl);
            const double* col = b + (size_t)k * ny * nx + i0 + i;
            double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
            for (int j = g * jl; j < j1; j++) {
                const double v = col[(size_t)j * nx];
#pragma unroll
                for (int q = 0; q < 5; q++) acc[q] = fma(__ldg(ym + (size_t)q * ny + j), v, acc[q]);
            }
#pragma unroll
            for (int q = 0; q < 5; q++) s_col[(q * JG + g) * ni + i] = acc[q];
        }
        __syncthreads();
        for (int e = tid; e < 5 * ni; e += blockDim.x) {   // the ranges' sums into the first one's place
            const int q = e / ni, i = e - q * ni;
            double v = s_col[q * JG * ni + i];
            for (int g = 1; g < JG; g++) v += s_col[(q * JG + g) * ni + i];
            s_col[q * JG * ni + i] = v;
        }
        __syncthreads();
        for (int ab = warp; ab < 15; ab += nw) {
            const double* xa = xm + (size_t)c_ab[ab][0] * nx + i0;
            const double* cb = s_col + c_ab[ab][1] * JG * ni;
            double acc = 0.0;
            for (int i = lane; i < ni; i += 32) acc = fma(xa[i], cb[i], acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
            if (lane == 0) s_ab[ab] += acc;
        }
        __syncthreads();
    }
    if (tid < 15) plane[(size_t)tid * nz + k] = s_ab[tid];
}

// M[a][b][c] = sum_k zm[c][k] plane[ab][k] (a warp per monomial); Q_lm = sum_terms coef M / (4 pi)
__global__ void __launch_bounds__(1024) k_final_moments(const double* __restrict__ plane, int nz,
                                                       const double* __restrict__ zm, double* __restrict__ Q)
{
    __shared__ double M[5][5][5];
    const int t = threadIdx.x, lane = t & 31;
    for (int mono = t >> 5; mono < 35; mono += 32) {
        // the monomial -> (ab, c) in the order of c_ab with c = 0 .. 4 - a - b
        int idx = 0, ab = 0;
        while (mono >= idx + 5 - c_ab[ab][0] - c_ab[ab][1]) idx += 5 - c_ab[ab][0] - c_ab[ab][1], ab++;
        const int C = mono - idx;
        const double* pl = plane + (size_t)ab * nz;
        const double* zc = zm + (size_t)C * nz;
        double acc = 0.0;
        for (int k = lane; k < nz; k += 32) acc = fma(zc[k], pl[k], acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) M[c_ab[ab][0]][c_ab[ab][1]][C] = acc;
    }
    __syncthreads();
    // a term per thread, then a harmonic's sum per thread (in the terms' order)
    __shared__ double s_term[N_MONO_TERMS];
    __shared__ int s_lm[N_MONO_TERMS];
    if (t < N_MONO_TERMS) {
        const Mono mo = c_mono[t];
        s_lm[t] = mo.lm;
        s_term[t] = mo.coef * M[mo.a][mo.b][mo.c];
    }
    __syncthreads();
    if (t < NLM) {
        double q = 0.0;
#pragma unroll 8
        for (int m = 0; m < N_MONO_TERMS; m++)
            if (s_lm[m] == t) q += s_term[m];
        Q[t] = q / (4.0 * PI);
    }
}

cudaError_t launch_multipoles(const int n[3], const double* x, const double* y, const double* z, const double* b,
                              const double centre[3], double* tabs, double* plane, double* Q, cudaStream_t s)
{
    cudaError_t e = ensure_monomials();
    if (e != cudaSuccess) return e;
    const int nm = std::max(n[0], std::max(n[1], n[2])), ni = std::min(n[0], MOM_T), JG = std::min(n[1], MOM_T / ni);
    const unsigned nt = (unsigned)(ni * JG + 31) / 32 * 32;
    const double *xm = tabs, *ym = xm + 5 * (size_t)n[0], *zm = ym + 5 * (size_t)n[1];
    k_moment_tables<<<dim3((nm + 127) / 128, 3), 128, 0, s>>>(x, y, z, n[0], n[1], n[2], centre[0], centre[1], centre[2],
                                                              tabs);
    k_plane_moments<<<(unsigned)n[2], nt, sizeof(double) * 5 * ni * JG, s>>>(b, n[0], n[1], n[2], JG, xm, ym, plane);
    k_final_moments<<<1, 1024, 0, s>>>(plane, n[2], zm, Q);
    return cudaGetLastError();
}

size_t multipole_scratch_doubles(const int n[3]) { return 5 * ((size_t)n[0] + n[1] + n[2]) + 15 * (size_t)n[2]; }

// ---------------------------------------------------------------- Dirichlet faces
// slot of x^a y^b z^c (a + b + c = l, 1 <= l <= 4): degree offset + s(s+1)/2 + c, s = b + c
__host__ __device__ constexpr int ex_slot(int l, int b, int c)
{
    return (l == 1 ? 0 : l == 2 ? 3 : l == 3 ? 9 : 19) + (b + c) * (b + c + 1) / 2 + c;
}

// u = -sum_lm 4 pi/(2l+1) Q_lm S_lm(d) / r^(2l+1), d = node - centre (Eq. 2.7 decay).  S_lm is
// homogeneous of degree l, so with e = d / r^2 this is P(e) / r, one polynomial of degree 4 whose 35
// coefficients each block forms first: about 55 FP64 operations per node where the harmonics one by
// one take 300.  129^3 63.6 -> 18.1 us, 385^3 465 -> 109 us.
__global__ void k_boundary_fill(int nx, int ny, int nz, const double* __restrict__ x, const double* __restrict__ y,
                                const double* __restrict__ z, double cx, double cy, double cz,
                                const double* __restrict__ Q, double* __restrict__ u)
{
    // the coefficients: a term of a harmonic per thread, then a coefficient's sum per thread
    __shared__ double s_cf[35], s_term[N_MONO_TERMS];
    __shared__ int s_slot[N_MONO_TERMS];
    if (threadIdx.x < N_MONO_TERMS) {
        const Mono mo = c_mono[threadIdx.x];
        const int l = mo.a + mo.b + mo.c;
        s_slot[threadIdx.x] = l == 0 ? 0 : 1 + ex_slot(l, mo.b, mo.c);
        s_term[threadIdx.x] = -4.0 * PI / (2.0 * l + 1.0) * Q[mo.lm] * mo.coef;
    }
    __syncthreads();
    if (threadIdx.x < 35) {
        double cf = 0.0;
#pragma unroll 8
        for (int m = 0; m < N_MONO_TERMS; m++)
            if (s_slot[m] == (int)threadIdx.x) cf += s_term[m];
        s_cf[threadIdx.x] = cf;
    }
    __syncthreads();
    const size_t fx = (size_t)ny * nz, fy = (size_t)nx * nz, fz = (size_t)nx * ny;
    const size_t total = 2 * (fx + fy + fz);
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= total) return;
    int i, j, k;
    size_t r = t;
    if (r < 2 * fx) {
        const int side = (int)(r / fx);
        r %= fx;
        i = side ? nx - 1 : 0;
        j = (int)(r % ny);
        k = (int)(r / ny);
    } else if ((r -= 2 * fx) < 2 * fy) {
        const int side = (int)(r / fy);
        r %= fy;
        j = side ? ny - 1 : 0;
        i = (int)(r % nx);
        k = (int)(r / nx);
    } else {
        r -= 2 * fy;
        const int side = (int)(r / fz);
        r %= fz;
        k = side ? nz - 1 : 0;
        i = (int)(r % nx);
        j = (int)(r / nx);
    }
    const double dx = x[i] - cx, dy = y[j] - cy, dz = z[k] - cz;
    const double ir = rsqrt(fma(dz, dz, fma(dy, dy, dx * dx))), ir2 = ir * ir;
    const double X = dx * ir2, Y = dy * ir2, Z = dz * ir2;
    double px = 0.0;   // Horner in x of Horner in y of Horner in z
#pragma unroll
    for (int a = 4; a >= 0; a--) {
        double py = 0.0;
#pragma unroll
        for (int b = 4 - a; b >= 0; b--) {
            double pz = 0.0;
#pragma unroll
            for (int c = 4 - a - b; c >= 0; c--) {
                const double cf = s_cf[a + b + c == 0 ? 0 : 1 + ex_slot(a + b + c, b, c)];
                pz = c == 4 - a - b ? cf : fma(pz, Z, cf);
            }
            py = b == 4 - a ? pz : fma(py, Y, pz);
        }
        px = a == 4 ? py : fma(px, X, py);
    }
    u[((size_t)k * ny + j) * nx + i] = px * ir;
}

cudaError_t launch_boundary_fill(const int n[3], const double* x, const double* y, const double* z, double cx,
                                 double cy, double cz, const double* Q, double* u, cudaStream_t s)
{
    cudaError_t e = ensure_monomials();
    if (e != cudaSuccess) return e;
    const size_t total = 2 * ((size_t)n[1] * n[2] + (size_t)n[0] * n[2] + (size_t)n[0] * n[1]);
    k_boundary_fill<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(n[0], n[1], n[2], x, y, z, cx, cy, cz, Q, u);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- exact superposition faces
// M_l = int_0^R zeta_1^3/(8pi) e^{-zeta_1 r} (1 - r^2/R^2)^2 (r/R)^l r^(l+2) dr, l = 0..4, by a
// 64-point Gauss-Legendre rule: block = atom, thread = node (found by Newton's method on the
// Legendre recurrence).
__global__ void k_nonsph_moments(int na, const double* __restrict__ R, const double* __restrict__ zeta,
                                 double* __restrict__ M)
{
    __shared__ double part[5][64];
    const int a = blockIdx.x, q = threadIdx.x;
    // node q of the 64-point rule (ascending cos), initial guess from the Chebyshev nodes
    double t = -cos(PI * (q + 0.75) / (64 + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; it++) {
        double p0 = 1.0, p1 = t;
        for (int k = 2; k <= 64; k++) {
            const double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = 64 * (t * p1 - p0) / (t * t - 1.0);
        const double dt = p1 / dp;
        t -= dt;
        if (fabs(dt) < 1e-16) break;
    }
    const double wq = 2.0 / ((1.0 - t * t) * dp * dp);
    const double Ra = R[a], z1 = zeta[3 * a];
    const double r = 0.5 * Ra * (t + 1.0), tt = 1.0 - r * r / (Ra * Ra);
    const double f = 0.5 * Ra * wq * z1 * z1 * z1 / (8.0 * PI) * exp(-z1 * r) * tt * tt * r * r;
    double pl = 1.0;
    for (int l = 0; l < 5; l++) {
        part[l][q] = f * pl;
        pl *= (r / Ra) * r;
    }
    __syncthreads();
    for (int st = 32; st > 0; st >>= 1) {
        if (q < st)
            for (int l = 0; l < 5; l++) part[l][q] += part[l][q + st];
        __syncthreads();
    }
    if (q < 5) M[5 * (size_t)a + q] = part[q][0];
}

// u on the faces = sum over atoms of Z/r - sum_k w_k [1/r - e^{-zeta_k r}(1/r + zeta_k/2)]
// - sum_{l>=1,m} 4pi/(2l+1) c_lm M_l S_lm(d) / r^(2l+1), evaluated per atom as
// (Z - sum_k w_k)/r + sum_k w_k e^{-zeta_k r}(1/r + zeta_k/2) - sum_l r^-(2l+1) P_l(d), where
// P_l = sum_m 4pi/(2l+1) c_lm M_l S_lm is a homogeneous polynomial of degree l whose monomial
// coefficients each block forms once per atom (34 for l = 1..4).  Terms with zeta_k r >= 40
// (below e^-40 of w_k) are dropped, as in the deposit.
constexpr int EX_NT = 128;
constexpr int EX_CH = 64;        // atoms staged per pass
constexpr int EX_NC = 34;        // monomials of degree 1..4
constexpr int EX_REC = 10 + EX_NC;  // x y z q w0 w1 w2 zeta0 zeta1 zeta2 | coefficients

__global__ void __launch_bounds__(EX_NT) k_boundary_exact(int nx, int ny, int nz, const double* __restrict__ x,
                                                          const double* __restrict__ y, const double* __restrict__ z,
                                                          int na, const double* __restrict__ pos,
                                                          const double* __restrict__ Zn, const double* __restrict__ w,
                                                          const double* __restrict__ zeta,
                                                          const double* __restrict__ clm,
                                                          const double* __restrict__ M, double* __restrict__ u)
{
    __shared__ double rec[EX_CH][EX_REC];
    const size_t fx = (size_t)ny * nz, fy = (size_t)nx * nz, fz = (size_t)nx * ny;
    const size_t total = 2 * (fx + fy + fz);
    const size_t t = blockIdx.x * (size_t)EX_NT + threadIdx.x;
    const bool valid = t < total;
    int i = 0, j = 0, k = 0;
    if (valid) {
        size_t r = t;
        if (r < 2 * fx) {
            const int side = (int)(r / fx);
            r %= fx;
            i = side ? nx - 1 : 0;
            j = (int)(r % ny);
            k = (int)(r / ny);
        } else if ((r -= 2 * fx) < 2 * fy) {
            const int side = (int)(r / fy);
            r %= fy;
            j = side ? ny - 1 : 0;
            i = (int)(r % nx);
            k = (int)(r / nx);
        } else {
            r -= 2 * fy;
            const int side = (int)(r / fz);
            r %= fz;
            k = side ? nz - 1 : 0;
            i = (int)(r % nx);
            j = (int)(r / nx);
        }
    }
    const double px = x[i], py = y[j], pz = z[k];
    double v = 0.0;
    for (int base = 0; base < na; base += EX_CH) {
        const int nch = min(EX_CH, na - base);
        __syncthreads();
        for (int q = threadIdx.x; q < nch; q += EX_NT) {
            const int at = base + q;
            double* o = rec[q];
            o[0] = pos[3 * at];
            o[1] = pos[3 * at + 1];
            o[2] = pos[3 * at + 2];
            o[3] = Zn[at] - (w[3 * at] + w[3 * at + 1] + w[3 * at + 2]);
            o[4] = w[3 * at];
            o[5] = w[3 * at + 1];
            o[6] = w[3 * at + 2];
            o[7] = zeta[3 * at];
            o[8] = zeta[3 * at + 1];
            o[9] = zeta[3 * at + 2];
            for (int c = 0; c < EX_NC; c++) o[10 + c] = 0.0;
            for (int tm = 1; tm < N_MONO_TERMS; tm++) {
                const Mono mo = c_mono[tm];
                const int l = l_of_lm(mo.lm);
                const double K = 4.0 * PI / (2 * l + 1) * clm[24 * (size_t)at + mo.lm - 1] * M[5 * (size_t)at + l];
                o[10 + ex_slot(l, mo.b, mo.c)] += K * mo.coef;
            }
        }
        __syncthreads();
        if (!valid) continue;
        for (int q = 0; q < nch; q++) {
            const double* o = rec[q];
            const double dx = px - o[0], dy = py - o[1], dz = pz - o[2];
            const double d = sqrt(fma(dx, dx, fma(dy, dy, dz * dz))), id = 1.0 / d, id2 = id * id;
            double e = o[3] * id;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const double zc = o[7 + c];
                if (zc * d < EXP_CUT) e = fma(o[4 + c] * exp(-zc * d), id + 0.5 * zc, e);
            }
            double xp[5], yp[5], zp[5];
            xp[0] = yp[0] = zp[0] = 1.0;
#pragma unroll
            for (int p = 1; p < 5; p++) {
                xp[p] = xp[p - 1] * dx;
                yp[p] = yp[p - 1] * dy;
                zp[p] = zp[p - 1] * dz;
            }
            double P[5];
#pragma unroll
            for (int l = 1; l <= 4; l++) {
                double acc = 0.0;
#pragma unroll
                for (int sb = 0; sb <= l; sb++)
#pragma unroll
                    for (int c = 0; c <= sb; c++)
                        acc = fma(o[10 + ex_slot(l, sb - c, c)], xp[l - sb] * yp[sb - c] * zp[c], acc);
                P[l] = acc;
            }
            const double multi = id2 * id * fma(id2, fma(id2, fma(id2, P[4], P[3]), P[2]), P[1]);
            v += e - multi;
        }
    }
    if (valid) u[((size_t)k * ny + j) * nx + i] = v;
}

cudaError_t launch_boundary_exact(const lasto_cluster& cl, double* M, double* u, cudaStream_t s)
{
    cudaError_t e = ensure_monomials();
    if (e != cudaSuccess) return e;
    k_nonsph_moments<<<cl.n_atoms, 64, 0, s>>>(cl.n_atoms, cl.R, cl.slater_zeta, M);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int* n = cl.n;
    const size_t total = 2 * ((size_t)n[1] * n[2] + (size_t)n[0] * n[2] + (size_t)n[0] * n[1]);
    k_boundary_exact<<<(unsigned)((total + EX_NT - 1) / EX_NT), EX_NT, 0, s>>>(n[0], n[1], n[2], cl.x, cl.y, cl.z, cl.n_atoms,
                                                                     cl.pos, cl.Z, cl.slater_w, cl.slater_zeta,
                                                                     cl.c_lm, M, u);
    return cudaGetLastError();
}

}  // namespace lasto
