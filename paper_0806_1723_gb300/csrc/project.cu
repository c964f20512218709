// Sphere-surface projection V_LM(R_i) = int y_LM V dOmega (Eq. 3.6), with V from
// trilinear interpolation of the grid potential ("interpolates onto the sphere
// boundaries", Section 1).  Reading of the measure: the unit-sphere solid angle, so
// that V = sum_LM V_LM y_LM on the surface (Eq. 3.5).  The quadrature is
// Gauss-Legendre in cos(theta) times uniform phi; its rings and factors (SphereRule, 5 KB) are
// mesh independent, built on the host and passed as a kernel parameter.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"
#include "rule.cuh"

namespace cg = cooperative_groups;

namespace lasto {

// Gauss-Legendre nodes on [-1, 1]: Newton's method on P_n from the asymptotic guess
// cos(pi (i - 1/4) / (n + 1/2)), P_n and P_n' from the three-term recurrence.  Convergence is
// quadratic, so a step below 1e-12 leaves x exact to rounding; P_n' is then taken there.
static void gauss_legendre(int n, std::vector<double>& t, std::vector<double>& w)
{
    t.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 1; i <= n; i++) {
        double x = std::cos(PI * (i - 0.25) / (n + 0.5));
        double dpn = 1.0;
        bool done = false;
        for (int it = 0; it < 60; it++) {
            double pm = 1.0, pc = x;
            for (int k = 1; k < n; k++) {
                const double pn = ((2 * k + 1) * x * pc - k * pm) / (k + 1);
                pm = pc;
                pc = pn;
            }
            if (n == 1) pm = 1.0;
            dpn = n * (pm - x * pc) / (1.0 - x * x);
            if (done) break;
            const double dx = pc / dpn;
            x -= dx;
            done = std::fabs(dx) < 1e-12;
        }
        t[n - i] = x;
        w[n - i] = 2.0 / ((1.0 - x * x) * dpn * dpn);
    }
}

// y_lm(theta, phi) = f_lm(theta) cos(m phi) for m >= 0 and f_l|m|(theta) sin(|m| phi) for m < 0,
// with f_lm(theta) = y_lm(theta, 0): the rule keeps w_theta f_lm per ring of the quadrature.
static void make_sphere_rule(int n_theta, int n_phi, SphereRule* q)
{
    std::vector<double> ct, wt;
    gauss_legendre(n_theta, ct, wt);
    std::memset(q, 0, sizeof(*q));
    q->nt = n_theta;
    q->np = n_phi;
    for (int a = 0; a < n_theta; a++) {
        const double st = std::sqrt(std::max(0.0, 1.0 - ct[a] * ct[a]));
        q->ct[a] = ct[a];
        q->st[a] = st;
        double S[NLM];
        host_solid_harmonics(st, 0.0, ct[a], S);
        const double wq = wt[a] * 2.0 * PI / n_phi;
        for (int l = 0; l < 5; l++)
            for (int m = 0; m <= l; m++) q->wf[a][rule_slot(l, m)] = wq * S[l * l + l + m];
    }
    for (int b = 0; b < n_phi; b++) {
        const double ph = 2.0 * PI * b / n_phi;
        q->trig[2 * b] = std::cos(ph);
        q->trig[2 * b + 1] = std::sin(ph);
    }
}

// The rule of n_theta x n_phi points: a constant table of the two numbers, kept per host thread
// (about 15 us to build, more than the projection of a small cluster takes on the device).
const SphereRule& sphere_rule(int n_theta, int n_phi)
{
    thread_local SphereRule q = {};
    if (q.nt != n_theta || q.np != n_phi) make_sphere_rule(n_theta, n_phi, &q);
    return q;
}

// The order of a double as an integer (both zeros equal, NaN beyond the infinities): the cell
// search compares on the integer units, as FP64 compares run at 1/64 of their rate here.
__device__ __forceinline__ long long order_key(double v)
{
    const long long b = __double_as_longlong(v);
    return b < 0 ? -(b & 0x7fffffffffffffffll) : b;
}

// largest i with c[i] <= p, clamped to [0, n-2] (kp = order_key(p))
__device__ __forceinline__ int cell_of(const double* c, int n, long long kp)
{
    int lo = 0, hi = n - 1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (order_key(c[mid]) <= kp) lo = mid;
        else hi = mid;
    }
    if (order_key(c[hi]) <= kp) lo = hi;
    return lo > n - 2 ? n - 2 : lo;
}

constexpr int PRJ_NT = 128;
constexpr int PRJ_STAGE = 2800;   // axis nodes (three axes together) staged in shared memory
constexpr int PRJ_BLOCKS = 4 * 152;

// One sphere per cluster of gridDim.x blocks, each block a run of the quadrature's rings.  The
// potential at a block's points goes to shared memory, then each ring's sums over phi with the
// nine factors cos m phi, sin m phi (m <= 4), then the 25 sums over the rings: 9 FMAs per point
// where 25 stored harmonics per point took 25 and their table (115 KB, built and copied by the
// host in every call of the single operation).  Bound: FP64 issue and the latency of one sphere's
// chain, so the rings are split over up to eight blocks while the spheres alone leave SMs idle
// (13 spheres on 65^3: 37.4 -> 13.2 us; 55 on 129^3: 41 -> 16.6 us).  The blocks' partial
// sums meet in rank order in the first block's shared memory, so the result is reproducible.
__global__ void __launch_bounds__(PRJ_NT) k_project(int nx, int ny, int nz, const double* __restrict__ x,
                                                   const double* __restrict__ y, const double* __restrict__ z,
                                                   const double* __restrict__ u, const double* __restrict__ pos,
                                                   const double* __restrict__ R, const __grid_constant__ SphereRule q,
                                                   int staged, double* __restrict__ vlm, int* status)
{
    extern __shared__ double sm[];
    __shared__ double part[NLM];
    const int split = (int)gridDim.x, rank = (int)blockIdx.x, a = (int)blockIdx.y, tid = (int)threadIdx.x;
    const int np = q.np, r0 = q.nt * rank / split, rows = q.nt * (rank + 1) / split - r0;
    const int rows_max = (q.nt + split - 1) / split;
    double* V = sm;                        // [rows][np]
    double* trig = V + rows_max * np;      // [np][2]
    double* F = trig + 2 * np;             // [rows][9]
    const double *xs = x, *ys = y, *zs = z;
    if (staged) {
        double* c = F + 9 * rows_max;
        for (int t = tid; t < nx + ny + nz; t += PRJ_NT)
            c[t] = t < nx ? x[t] : t < nx + ny ? y[t - nx] : z[t - nx - ny];
        xs = c;
        ys = c + nx;
        zs = ys + ny;
    }
    for (int t = tid; t < 2 * np; t += PRJ_NT) trig[t] = q.trig[t];
    const double cx = pos[3 * a], cy = pos[3 * a + 1], cz = pos[3 * a + 2], Ra = R[a];
    __syncthreads();
    int bad = 0;
    for (int t = tid; t < rows * np; t += PRJ_NT) {
        const int row = t / np, b = t - row * np;
        const double st = q.st[r0 + row];
        // + 0.0: a negative zero becomes the positive one
        const double px = fma(Ra, st * trig[2 * b], cx) + 0.0, py = fma(Ra, st * trig[2 * b + 1], cy) + 0.0,
                     pz = fma(Ra, q.ct[r0 + row], cz) + 0.0;
        const long long kx = order_key(px), ky = order_key(py), kz = order_key(pz);
        double v = 0.0;
        if (kx >= order_key(xs[0]) && kx <= order_key(xs[nx - 1]) && ky >= order_key(ys[0]) &&
            ky <= order_key(ys[ny - 1]) && kz >= order_key(zs[0]) && kz <= order_key(zs[nz - 1])) {
            const int i = cell_of(xs, nx, kx), j = cell_of(ys, ny, ky), k = cell_of(zs, nz, kz);
            const size_t sy = nx, sz = (size_t)nx * ny;
            const double* c0 = u + (size_t)k * sz + (size_t)j * sy + i;
            const double a0 = c0[0], a1 = c0[1], a2 = c0[sy], a3 = c0[sy + 1];
            const double a4 = c0[sz], a5 = c0[sz + 1], a6 = c0[sz + sy], a7 = c0[sz + sy + 1];
            const double tx = (px - xs[i]) / (xs[i + 1] - xs[i]);
            const double ty = (py - ys[j]) / (ys[j + 1] - ys[j]);
            const double tz = (pz - zs[k]) / (zs[k + 1] - zs[k]);
            const double v00 = fma(tx, a1 - a0, a0), v10 = fma(tx, a3 - a2, a2);
            const double v01 = fma(tx, a5 - a4, a4), v11 = fma(tx, a7 - a6, a6);
            const double v0 = fma(ty, v10 - v00, v00), v1 = fma(ty, v11 - v01, v01);
            v = fma(tz, v1 - v0, v0);
        } else {
            bad = 1;
        }
        V[t] = v;
    }
    __syncthreads();
    rule_rings<PRJ_NT>(V, rows, np, trig, F);
    __syncthreads();
    if (tid < NLM) part[tid] = rule_lm(q, F, r0, rows, tid);
    if (split == 1) {
        if (tid < NLM) vlm[(size_t)NLM * a + tid] = part[tid];
    } else {
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        if (rank == 0 && tid < NLM) {
            double s = part[tid];
            for (int r = 1; r < split; r++) s += cl.map_shared_rank(part, r)[tid];
            vlm[(size_t)NLM * a + tid] = s;
        }
        cl.sync();   // the first block has read this block's sums
    }
    if (bad && status) atomicMax(status, (int)LASTO_ERR_GEOMETRY);
}

cudaError_t launch_project(const int n[3], const double* x, const double* y, const double* z, const double* u,
                           int n_atoms, const double* pos, const double* R, const SphereRule& q, double* vlm,
                           int* status, cudaStream_t s)
{
    if (n_atoms <= 0) return cudaSuccess;
    int split = 1;
    while (split < 8 && 2 * split <= q.nt && (long long)n_atoms * 2 * split <= PRJ_BLOCKS) split *= 2;
    const size_t axes = (size_t)n[0] + n[1] + n[2];
    const int staged = axes <= PRJ_STAGE ? 1 : 0, rows = (q.nt + split - 1) / split;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(PRJ_NT);
    cfg.dynamicSmemBytes = sizeof(double) * ((size_t)rows * q.np + 2 * q.np + 9 * rows + (staged ? axes : 0));
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)split;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = split > 1 ? 1 : 0;
    cudaError_t e = cudaSuccess;
    for (int a0 = 0; a0 < n_atoms && e == cudaSuccess; a0 += 65535) {   // the grid's y limit
        cfg.gridDim = dim3((unsigned)split, (unsigned)std::min(65535, n_atoms - a0));
        e = cudaLaunchKernelEx(&cfg, k_project, n[0], n[1], n[2], x, y, z, u, pos + 3 * (size_t)a0, R + a0, q, staged,
                               vlm + (size_t)NLM * a0, status);
    }
    return e;
}

}  // namespace lasto
