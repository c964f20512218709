// The raw-density entry point (Eq. 3.1's representation of the density: values on the grid,
// and inside each sphere its spherical-harmonic components on the logarithmic radial mesh).
// The caller gives the electron density at every node and each sphere's spherical component
// rho_00(r_j); the pseudo-density of Section 3 is built from the table, and the deposit
// replaces the spherical part inside each sphere by it (Section 1's monopole swap).
#include "internal.cuh"

namespace lasto {

namespace {

constexpr double RAW_PI = 3.14159265358979323846;

// weight of sample j (of n >= 5, in units of h / 24) in the sum of the cubic rule over all intervals
__device__ __forceinline__ double cubic_weight(int j, int n)
{
    int w = 0;
    if (j < 4) w += j == 0 ? 9 : j == 1 ? 19 : j == 2 ? -5 : 1;
    const int e = n - 1 - j;
    if (e < 4) w += e == 0 ? 9 : e == 1 ? 19 : e == 2 ? -5 : 1;
#pragma unroll
    for (int t = 0; t < 4; t++) {   // sample j is the t-th of the interior interval q
        const int q = j + 1 - t;
        if (q >= 1 && q <= n - 3) w += (t == 0 || t == 3) ? -1 : 13;
    }
    return (double)w;
}

// One block per sphere: q = sqrt(4pi) int_0^R rho_00 r^2 dr - Z (rule in ln r, rho_00
// constant on [0, r_min]), rho(R) = rho_00(R)/sqrt(4pi), rho'(R) from the one-sided fourth-
// order difference in ln r, and the quartic a + b r^2 + c r^4 meeting the three constraints
// (written out: c = (Q - rho R^3/3 + rho' R^4/15) 105/(8 R^7), b = rho'/(2R) - 2 c R^2,
// a = rho - rho' R/2 + c R^4 with Q = q/(4pi)).  Record: x y z R a b c h.  Also the
// geometry check: the sphere two nodes inside every face and disjoint from the others.
// The integral is one weighted sum over the samples, taken by the block: latency bound (a few
// FP64 exponentials deep), 55 spheres of 429 samples 1451 us (one thread per sphere, four
// exponentials per interval) -> 16.4 us.
constexpr int RSP_NT = 128;
__global__ void __launch_bounds__(RSP_NT) k_raw_sphere_params(RawArgs a, double* __restrict__ rec,
                                                              int* __restrict__ status)
{
    const int i = blockIdx.x;
    const double Ri = a.R[i], rm = a.r_min;
    const int n = a.n_rad;
    const double h = log(Ri / rm) / (n - 1);
    const double* f = a.rho00 + (size_t)i * n;
    double part = 0.0;
    for (int j = threadIdx.x; j < n; j += RSP_NT) {
        const double x = j == n - 1 ? Ri : Ri * exp((j - (n - 1)) * h);
        part = fma(cubic_weight(j, n) * f[j], x * x * x, part);
    }
    bool bad = false;
    for (int j = threadIdx.x; j < a.na; j += RSP_NT) {
        if (j == i) continue;
        const double dx = a.pos[3 * i] - a.pos[3 * j], dy = a.pos[3 * i + 1] - a.pos[3 * j + 1],
                     dz = a.pos[3 * i + 2] - a.pos[3 * j + 2];
        if (sqrt(dx * dx + dy * dy + dz * dz) < Ri + a.R[j]) bad = true;
    }
    if (threadIdx.x < 3) {
        const int d = threadIdx.x;
        const double cc = a.pos[3 * i + d];
        if (!(cc - Ri >= a.ax[d][2] && cc + Ri <= a.ax[d][a.n[d] - 3])) bad = true;
    }
    if (bad && status) atomicMax(status, (int)LASTO_ERR_GEOMETRY);
    const double sum = block_sum<RSP_NT>(part);
    if (threadIdx.x != 0) return;
    const double s4 = sqrt(4.0 * RAW_PI);
    const double q = s4 * fma(h / 24.0, sum, f[0] * rm * rm * rm / 3.0) - a.Z[i];
    const int m = n - 1;
    const double rho = f[m] / s4;
    const double drho = (25.0 * f[m] - 48.0 * f[m - 1] + 36.0 * f[m - 2] - 16.0 * f[m - 3] + 3.0 * f[m - 4]) /
                        (12.0 * h) / (Ri * s4);
    const double Q = q / (4.0 * RAW_PI), R2 = Ri * Ri, R4 = R2 * R2;
    const double c = (Q - rho * Ri * R2 / 3.0 + drho * R4 / 15.0) * 105.0 / (8.0 * R4 * R2 * Ri);
    const double b = drho / (2.0 * Ri) - 2.0 * c * R2;
    const double aa = rho - drho * Ri / 2.0 + c * R4;
    double* o = rec + (size_t)RAW_REC * i;
    o[0] = a.pos[3 * i];
    o[1] = a.pos[3 * i + 1];
    o[2] = a.pos[3 * i + 2];
    o[3] = Ri;
    o[4] = aa;
    o[5] = b;
    o[6] = c;
    o[7] = h;
    if (!isfinite(q) || !isfinite(aa) || !isfinite(b) || !isfinite(c))
        if (status) atomicMax(status, (int)LASTO_ERR_NONFINITE);
}

// rho_00(r)/sqrt(4pi) of sphere i: cubic Lagrange in ln r on the four nearest samples; below
// r_min the straight line through the first two
__device__ __forceinline__ double monopole_at(const double* __restrict__ f, int n, double rm, double h, double r)
{
    if (r <= rm) {
        const double r1 = rm * exp(h);
        return f[0] + (f[1] - f[0]) * (r - rm) / (r1 - rm);
    }
    const double t = log(r / rm) / h;
    int j = (int)floor(t);
    j = j < 1 ? 1 : (j > n - 3 ? n - 3 : j);
    const double s = t - j;
    const double l0 = -s * (s - 1.0) * (s - 2.0) / 6.0, l1 = (s + 1.0) * (s - 1.0) * (s - 2.0) / 2.0;
    const double l2 = -(s + 1.0) * s * (s - 2.0) / 2.0, l3 = (s + 1.0) * s * (s - 1.0) / 6.0;
    return l0 * f[j - 1] + l1 * f[j] + l2 * f[j + 1] + l3 * f[j + 2];
}

// b = 4pi (ne - rho_00(r)/sqrt(4pi) + quartic(r)) inside sphere i (|x - X_i| < R_i), 4pi ne
// outside.  Ownership: an FP32 distance test decides all nodes farther than 1e-4 R^2 from
// a sphere surface; the rest are decided in FP64.  A block takes 32 x 8 x 4 nodes (lanes along x) and
// first lists, in the atoms' order, the spheres that reach its nodes' box by that FP32 test (with room
// for its rounding): most boxes meet none.  Nodes that pass the FP32 test of some sphere are queued
// and finished together, so that the FP64 of the exact test and of the table (a logarithm, divisions)
// runs in whole warps: it is the bound, 10 % of the nodes of Pd55 129^3.  167 us with every sphere
// tested at every node and the inside nodes in place (214 with the lists alone) -> 119 us.
constexpr int RD_X = 32, RD_Y = 8, RD_Z = 4;
constexpr int RD_MAX_ATOMS = 12800;   // most atoms it takes (their list: 50 KiB)

__global__ void __launch_bounds__(RD_X * RD_Y) k_raw_deposit(RawArgs a, const double* __restrict__ rec,
                                                            double* __restrict__ b, int* __restrict__ owner,
                                                            int* __restrict__ status)
{
    extern __shared__ int near_at[];   // [na]: atoms whose spheres reach the box
    __shared__ int s_cnt[RD_Y], s_queued;
    __shared__ unsigned s_queue[RD_X * RD_Y * RD_Z];   // node of the box | place in the list << 10
    static_assert(RD_X * RD_Y * RD_Z == 1 << 10 && RD_X == 32 && RD_Y == 8, "queue entries and decoding");
    const int gx = (a.n[0] + RD_X - 1) / RD_X, gy = (a.n[1] + RD_Y - 1) / RD_Y;
    const int bz = (int)blockIdx.x / (gx * gy), rem = (int)blockIdx.x - bz * gx * gy;
    const int lane = threadIdx.x % RD_X, wp = threadIdx.x / RD_X;
    const int i0 = (rem % gx) * RD_X, j0 = (rem / gx) * RD_Y, k0 = bz * RD_Z;
    // the box of the block's nodes, in FP32 as the test below sees them
    float lo[3], hi[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const int first = d == 0 ? i0 : d == 1 ? j0 : k0, len = d == 0 ? RD_X : d == 1 ? RD_Y : RD_Z;
        const float c = (float)a.ax[d][min(first + min(lane, len - 1), a.n[d] - 1)];
        lo[d] = hi[d] = c;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    }
    int count = 0;
    for (int base = 0; base < a.na; base += RD_X * RD_Y) {
        const int t = base + (int)threadIdx.x;
        bool in = false;
        if (t < a.na) {
            const double* o = rec + (size_t)RAW_REC * t;
            float r2 = 0.0f;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const float c = (float)o[d], e = fmaxf(fmaxf(lo[d] - c, c - hi[d]), 0.0f);
                r2 += e * e;
            }
            in = !(r2 > (float)(o[3] * o[3]) * (1.0f + 1e-4f) * (1.0f + 1e-5f));
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        __syncthreads();
        if (lane == 0) s_cnt[wp] = __popc(m);
        __syncthreads();
        int at = count;
        for (int q = 0; q < RD_Y; q++) {
            at += q < wp ? s_cnt[q] : 0;
            count += s_cnt[q];
        }
        if (in) near_at[at + __popc(m & ((1u << lane) - 1u))] = t;
    }
    if (threadIdx.x == 0) s_queued = 0;
    __syncthreads();
    auto finish = [&](size_t P, double v, int own) {
        const double bv = 4.0 * RAW_PI * v;
        b[P] = bv;
        if (owner) owner[P] = own;
        if (!isfinite(bv) && status) atomicMax(status, (int)LASTO_ERR_NONFINITE);
    };
    const int i = i0 + lane, j = j0 + wp;
    if (i < a.n[0] && j < a.n[1]) {
        const float xf = (float)a.ax[0][i], yf = (float)a.ax[1][j];
        for (int kk = 0; kk < min(RD_Z, a.n[2] - k0); kk++) {
            const size_t P = ((size_t)(k0 + kk) * a.n[1] + j) * a.n[0] + i;
            const float zf = (float)a.ax[2][k0 + kk];
            int q = 0;
            for (; q < count; q++) {
                const double* o = rec + (size_t)RAW_REC * near_at[q];
                const float dx = xf - (float)o[0], dy = yf - (float)o[1], dz = zf - (float)o[2];
                if (!(dx * dx + dy * dy + dz * dz > (float)(o[3] * o[3]) * (1.0f + 1e-4f))) break;
            }
            if (q < count)
                s_queue[atomicAdd(&s_queued, 1)] = (unsigned)(kk * 256 + (int)threadIdx.x) | (unsigned)q << 10;
            else
                finish(P, a.ne[P], -1);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < s_queued; e += RD_X * RD_Y) {
        const int node = (int)(s_queue[e] & 1023u), ni = i0 + (node & 31), nj = j0 + ((node >> 5) & 7), nk = k0 + (node >> 8);
        const size_t P = ((size_t)nk * a.n[1] + nj) * a.n[0] + ni;
        const double x = a.ax[0][ni], y = a.ax[1][nj], z = a.ax[2][nk];
        double v = a.ne[P];
        int own = -1;
        for (int q = (int)(s_queue[e] >> 10); q < count && own < 0; q++) {
            const double* o = rec + (size_t)RAW_REC * near_at[q];
            const double ex = x - o[0], ey = y - o[1], ez = z - o[2];
            const double r = sqrt(ex * ex + ey * ey + ez * ez);
            if (!(r < o[3])) continue;
            own = near_at[q];
            const double rho0 = monopole_at(a.rho00 + (size_t)own * a.n_rad, a.n_rad, a.r_min, o[7], r) /
                                sqrt(4.0 * RAW_PI);
            v = v - rho0 + (o[4] + o[5] * r * r + o[6] * r * r * r * r);
        }
        finish(P, v, own);
    }
}

}  // namespace

cudaError_t launch_raw_sphere_params(const RawArgs& a, double* rec, int* status, cudaStream_t s)
{
    k_raw_sphere_params<<<a.na, RSP_NT, 0, s>>>(a, rec, status);
    return cudaGetLastError();
}

cudaError_t launch_raw_deposit(const RawArgs& a, const double* rec, double* b, int* owner, int* status, cudaStream_t s)
{
    const size_t N = (size_t)a.n[0] * a.n[1] * a.n[2];
    if (a.na > RD_MAX_ATOMS || N >= (size_t(1) << 31)) return cudaErrorInvalidValue;
    const size_t smem = sizeof(int) * (size_t)a.na;
    // (the default 48 KiB holds the static memory, 4 KiB, too; always the same request, whatever other
    // threads ask for)
    if (smem > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_raw_deposit, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(int) * RD_MAX_ATOMS));
        if (e != cudaSuccess) return e;
    }
    const size_t g = (size_t)((a.n[0] + RD_X - 1) / RD_X) * ((a.n[1] + RD_Y - 1) / RD_Y) * ((a.n[2] + RD_Z - 1) / RD_Z);
    k_raw_deposit<<<(unsigned)g, RD_X * RD_Y, smem, s>>>(a, rec, b, owner, status);
    return cudaGetLastError();
}

}  // namespace lasto
