// Exact solve of a coarse level by fast diagonalisation: the operator is the sum of three 1-D
// operators, so in their eigenvectors A e = b is a division,
//   e = (Bz x By x Bx) (lam_x + lam_y + lam_z)^-1 (Fz x Fy x Fx) b,
// with F = Q^T sqrt(V), B = V^{-1/2} Q for the symmetrised tridiagonal operator S = Q Lam Q^T (V the
// dual-cell lengths).  The paper's coarse solve ("exact", Section 3) at more than its nine nodes:
// the levels below would be swept by short launches whose latency, not work, sets the cycle's
// time, where six small matrix products per node line are three launches.
//
// Measured on GB300 (whole solves, sweeps and the one-block kernel below the same level before):
// Pd55 129^3 mixed 5760 -> 3680 us (14 -> 13 iterations), Pd561 385^3 SCF step 47.7 -> 41.5 ms (14
// -> 11 iterations), Pd55 129^3 FP64 13.9 -> 12.6 ms, Pd13 65^3 FP64 2.07 -> 1.71 ms.
#include <algorithm>

#include "ctl.cuh"
#include "internal.cuh"

namespace lasto {

// ---------------------------------------------------------------- eigenvectors
// One block per axis: the implicit QL algorithm for symmetric tridiagonal matrices (Dubrulle,
// Martin and Wilkinson, 1968) on S scaled by its largest element, in the precision of the
// cycle it serves.  Q is a product of plane rotations, so it is orthogonal whatever the axis --
// also for the near-degenerate pairs of an axis with two refined regions -- and e = Q D Q^T b stays
// symmetric whatever the rounding.  Definite, which the conjugate gradients also ask of their
// preconditioner, it is because every eigenvalue is held at or below -8 / length^2: the operator is
// exact for quadratics, so its inverse of -1 is (x - x_0)(x_1 - x) / 2 <= length^2 / 8, which bounds the
// norm of the inverse.  QL's errors are a small multiple (0.2 to 2.5 seen) of eps times the largest
// element, so a strongly graded axis, whose smallest eigenvalues FP32 would lose, is done in FP64
// also for the FP32 cycle (EIG_WIDE; such solves take 100 iterations and more).
// One lane runs the scalar chain (a rotation is about ten dependent operations)
// and the other warps apply the rotations of the QL step before to Q, a component per thread.
// Bound: that chain's latency; it runs beside the deposit.  Parallel cyclic Jacobi in the same
// place took 697 us at m = 63; this 253 us (m = 95: 510 us; FP64: 282 us at m = 15, 900 us at m = 31).
constexpr int EIG_NT = 128;
// FP64 where FP32's eps times the largest element passes this part of the bound on the smallest
// eigenvalue: below it that eigenvalue is right to about a seventh.  On 129 nodes over 80 bohr that is at a
// ratio of spacings of 200, where both take 140 iterations (23.9 ms in FP32, 26.3 in FP64: 2.4 ms at
// m = 63, 5.5 at 95); one axis with four cells 1000 times finer than the rest: FP32 diverges, FP64
// 139 iterations (the smoothed hierarchy without this level: 148).
constexpr double EIG_WIDE = 1.0 / 16;
static_assert(DIRECT_MAX <= EIG_NT - 32, "a component of Q per applying thread");

// the hardware's approximate reciprocal square root; FP64: about 20 bits of it and one third-order
// step, s (1 - h)^(-1/2) = s (1 + h/2 + 3 h^2/8 + O(h^3)), h = 1 - v s^2
__device__ __forceinline__ float inv_sqrt(float v)
{
    float s;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(v));
    return s;
}
__device__ __forceinline__ double inv_sqrt(double v)
{
    double s;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(s) : "d"(v));
    const double h = fma(-v * s, s, 1.0);
    return fma(s * h, fma(h, 0.375, 0.5), s);
}

// T: the precision of the iteration; big: S's largest element, low: the bound on its smallest
template <typename T, typename O>
__device__ __forceinline__ void direct_eig_axis(const AxisStore& A, T* Q, const DirectMats<O>& out, int dim, int mp, double big,
                                                double low)
{
    __shared__ T d[DIRECT_MAX + 1], e[DIRECT_MAX + 1], rc[2][DIRECT_MAX + 1], rs[2][DIRECT_MAX + 1];
    // per turn, in two buffers: rotations of columns (i, i + 1), i = hi - 1 .. lo, and whether it was the last
    __shared__ int r_hi[2], r_lo[2], s_done[2];
    const int tid = threadIdx.x, lane = tid & 31;
    const int m = A.n - 2, ld = m + 1 - (m & 1);
    __shared__ T s_scale;
    if (tid == 0) s_scale = (T)big;
    for (int t = tid; t < m * ld; t += EIG_NT) Q[t] = t / ld == t % ld ? (T)1 : (T)0;   // [m][ld]: row i holds eigenvector i
    if (tid == 0) r_hi[0] = r_hi[1] = r_lo[0] = r_lo[1] = 0;
    __syncthreads();
    for (int i = tid; i < m; i += EIG_NT) {
        d[i] = (T)(-A.dg[i + 1] / (double)s_scale);
        e[i] = i + 1 < m ? (T)(sqrt(A.cp[i + 1] * A.cm[i + 2]) / (double)s_scale) : (T)0;
    }
    __syncthreads();
    const T eps = sizeof(T) == 4 ? (T)6e-8 : (T)1.1e-16;
    int l = 0, iter = 0;   // warp 0: the eigenvalue being isolated, its QL steps so far
    for (int turn = 0;; turn++) {
        const int buf = turn & 1;
        if (tid < 32) {
            // the unreduced block l .. hi
            int hi = m - 1;
            for (; l < m; l++, iter = 0) {
                hi = m - 1;
                for (int base = l; base < m - 1; base += 32) {
                    const int i = base + lane;
                    const bool small = i < m - 1 && abs(e[i]) <= eps * (abs(d[i]) + abs(d[i + 1]));
                    const unsigned b = __ballot_sync(0xffffffffu, small);
                    if (b) {
                        hi = base + __ffs(b) - 1;
                        break;
                    }
                }
                if (hi > l && iter < 60) break;
            }
            if (lane == 0) {
                s_done[buf] = l >= m;
                if (l < m) {
                    // shift: the eigenvalue of the leading 2 x 2 block nearer d[l]
                    const T e0 = e[l];
                    T g = (d[l + 1] - d[l]) / (2 * e0);
                    const T h = sqrt(g * g + 1);
                    g = d[hi] - d[l] + e0 / (g + (g >= 0 ? h : -h));
                    T s = 1, c = 1, p = 0;
                    int i = hi - 1;
                    T ei = e[i], di = d[i], dn = d[i + 1];
                    for (; i >= l; i--) {
                        const T en = e[max(i - 1, 0)], dm = d[max(i - 1, 0)];   // for the next rotation
                        const T f = s * ei, b = c * ei;
                        const T r2 = f * f + g * g;
                        if (!(r2 > (sizeof(T) == 4 ? (T)1e-36 : (T)1e-290))) {   // the block splits here
                            e[i + 1] = 0;
                            d[i + 1] = dn - p;
                            break;
                        }
                        const T ir = inv_sqrt(r2);
                        e[i + 1] = r2 * ir;
                        s = f * ir;
                        c = g * ir;
                        const T q = dn - p;
                        const T r = (di - q) * s + 2 * c * b;
                        p = s * r;
                        d[i + 1] = q + p;
                        g = c * r - b;
                        rc[buf][i] = c;
                        rs[buf][i] = s;
                        dn = di;
                        di = dm;
                        ei = en;
                    }
                    r_hi[buf] = hi;
                    r_lo[buf] = i + 1;
                    if (i < l) {
                        d[l] -= p;
                        e[l] = g;
                    }
                    e[hi] = 0;
                }
            }
            iter++;
        } else if (tid - 32 < m) {
            T* q = Q + (tid - 32);
            const int hi = r_hi[buf ^ 1], lo = r_lo[buf ^ 1];
            T up = q[hi * ld];
            for (int i = hi - 1; i >= lo; i--) {
                const T c = rc[buf ^ 1][i], s = rs[buf ^ 1][i], v = q[i * ld];
                q[(i + 1) * ld] = s * v + c * up;
                up = c * v - s * up;
            }
            q[lo * ld] = up;
        }
        __syncthreads();
        if (s_done[buf]) break;   // (the turn before, whose rotations were applied in this one, was the last)
    }
    // transposed, padded with zeros to mp: Ft[i][p] = Q[p][i] sqrt(V_i), Bt[p][i] = Q[p][i] / sqrt(V_i)
    for (int t = tid; t < mp * mp; t += EIG_NT) {
        const int p = t / mp, i = t - p * mp;
        const bool in = p < m && i < m;
        const T sv = in ? (T)sqrt(A.dual[i + 1]) : (T)1, v = in ? Q[p * ld + i] : (T)0;
        out.Bt[dim][p * mp + i] = (O)(v / sv);
        out.Ft[dim][i * mp + p] = (O)(v * sv);
    }
    for (int p = tid; p < m; p += EIG_NT) {
        const O v = (O)(d[p] * s_scale), most = (O)-low;
        out.lam[dim][p] = v > most ? most : v;   // (a NaN stays one)
    }
}

template <typename T>
__global__ void __launch_bounds__(EIG_NT) k_direct_eig(AxisStore ax0, AxisStore ax1, AxisStore ax2, DirectMats<T> out, int mp)
{
    extern __shared__ __align__(16) unsigned char eig_sm[];
    __shared__ double s_big;
    const int dim = blockIdx.x;
    const AxisStore& A = dim == 0 ? ax0 : dim == 1 ? ax1 : ax2;
    const double length = A.c[A.n - 1] - A.c[0], low = 8.0 / (length * length);
    if (threadIdx.x == 0) {
        double big = 0.0;
        for (int i = 1; i <= A.n - 2; i++) big = fmax(big, A.dg[i]);
        s_big = big;
    }
    __syncthreads();
    const double big = s_big;
    if (sizeof(T) == 4 && 6e-8 * big > EIG_WIDE * low)
        direct_eig_axis(A, reinterpret_cast<double*>(eig_sm), out, dim, mp, big, low);
    else
        direct_eig_axis(A, reinterpret_cast<T*>(eig_sm), out, dim, mp, big, low);
}

// padded size of the transform matrices
static int direct_pad(const int n[3])
{
    const int m = std::max(n[0], std::max(n[1], n[2])) - 2;
    return m <= 32 ? 32 : m <= 64 ? 64 : 96;
}

template <typename T>
cudaError_t launch_direct_eig(const LevelStore& L, const DirectMats<T>& out, cudaStream_t s)
{
    const size_t m = (size_t)std::max(L.n[0], std::max(L.n[1], L.n[2])) - 2;
    k_direct_eig<T><<<3, EIG_NT, sizeof(double) * m * (m + 1), s>>>(L.ax[0], L.ax[1], L.ax[2], out, direct_pad(L.n));
    return cudaGetLastError();
}
template cudaError_t launch_direct_eig<float>(const LevelStore&, const DirectMats<float>&, cudaStream_t);
template cudaError_t launch_direct_eig<double>(const LevelStore&, const DirectMats<double>&, cudaStream_t);

// ---------------------------------------------------------------- the transforms
// A block of (RB / RM) x (MP / RN) threads forms C[r][c] = sum_k At[k][r] B[k][c], RB rows by MP
// columns, both operands in shared memory k-major, so that a thread's RM rows and RN columns are one
// vector load each per k (7.4 to 9.4 us a launch at m = 63, 21 to 24 us at
// m = 95, cold caches; scalar loads from row-major operands took 13 us at m = 63).  Rows and columns beyond the level's modes are padding (zero matrices, or columns
// that are never stored).
template <typename T, int N>
struct alignas(sizeof(T) * N) Vec {
    T v[N];
};

template <typename T, int MP, int RB, int RM, int RN>
struct Tile {
    static constexpr int CX = MP / RN, NT = CX * (RB / RM);
    static __device__ __forceinline__ int col() { return (int)(threadIdx.x % CX) * RN; }
    static __device__ __forceinline__ int row() { return (int)(threadIdx.x / CX) * RM; }
    // lda, ldb: RB and MP
    static __device__ __forceinline__ void multiply(const T* __restrict__ At, const T* __restrict__ B, int K, T (&acc)[RM][RN])
    {
        const T* pa = At + row();
        const T* pb = B + col();
#pragma unroll
        for (int r = 0; r < RM; r++)
#pragma unroll
            for (int c = 0; c < RN; c++) acc[r][c] = 0;
#pragma unroll 8
        for (int k = 0; k < K; k++) {
            const Vec<T, RM> a = *reinterpret_cast<const Vec<T, RM>*>(pa + k * RB);
            const Vec<T, RN> b = *reinterpret_cast<const Vec<T, RN>*>(pb + k * MP);
#pragma unroll
            for (int r = 0; r < RM; r++)
#pragma unroll
                for (int c = 0; c < RN; c++) acc[r][c] = fma(a.v[r], b.v[c], acc[r][c]);
        }
    }
};

template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copies_done()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// rows x (columns c0 .. c0 + N - 1) of a matrix padded to MP columns, 16 bytes at a time
template <typename T, int MP, int N, int NT>
__device__ __forceinline__ void stage_matrix(T* dst, const T* src, int rows, int c0)
{
    constexpr int V = 16 / sizeof(T), PER = N / V;
    for (int t = threadIdx.x; t < rows * PER; t += NT) {
        const int r = t / PER, c = (t - r * PER) * V;
        copy_async<16>(dst + r * N + c, src + r * MP + c0 + c);
    }
}

// Forward y then x: plane k, y modes b0 .. b0 + RB - 1:
// w[k][b][a] = sum_i Fx[a][i] (sum_j Fy[b][j] rhs[j][i])
template <typename T, int MP, int RB, int RM, int RN>
__device__ __forceinline__ void direct_fwd(const DirectArgs<T>& a, T* sm)
{
    using W = Tile<T, MP, RB, RM, RN>;
    const int mx = a.n[0] - 2, my = a.n[1] - 2;
    const int k = blockIdx.x, b0 = blockIdx.y * RB;
    T* P = sm;                 // [my][MP] the plane
    T* FX = P + my * MP;       // [mx][MP]
    T* FY = FX + mx * MP;      // [my][RB]
    T* T1 = FY + my * RB;      // [mx][RB]
    const T* src = a.b + ((size_t)(k + 1) * a.n[1] + 1) * a.n[0] + 1;
    for (int t = threadIdx.x; t < my * MP; t += W::NT) {
        const int j = t / MP, i = t - j * MP;
        if (i < mx) copy_async<sizeof(T)>(P + t, src + (size_t)j * a.n[0] + i);
    }
    stage_matrix<T, MP, MP, W::NT>(FX, a.M.Ft[0], mx, 0);
    stage_matrix<T, MP, RB, W::NT>(FY, a.M.Ft[1], my, b0);
    copies_done();
    T acc[RM][RN];
    const int r0 = W::row(), c0 = W::col();
    W::multiply(FY, P, my, acc);
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (c0 + c < mx) T1[(c0 + c) * RB + r0 + r] = acc[r][c];
    __syncthreads();
    W::multiply(T1, FX, mx, acc);
    T* w = a.w + (size_t)k * my * mx;
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (b0 + r0 + r < my && c0 + c < mx) w[(size_t)(b0 + r0 + r) * mx + c0 + c] = acc[r][c];
}

// z forward, division by the eigenvalue sums, z backward, in place: y mode b; a block's RB rows are
// the x modes a0 .. a0 + RB - 1, its columns the z modes (then planes)
template <typename T, int MP, int RB, int RM, int RN>
__device__ __forceinline__ void direct_z(const DirectArgs<T>& a, T* sm)
{
    using W = Tile<T, MP, RB, RM, RN>;
    const int mx = a.n[0] - 2, my = a.n[1] - 2, mz = a.n[2] - 2;
    const int b = blockIdx.x, a0 = blockIdx.y * RB;
    T* FZ = sm;                // [mz][MP]
    T* BZ = FZ + mz * MP;      // [mz][MP]
    T* S = BZ + mz * MP;       // [mz][RB]
    T* U = S + mz * RB;        // [mz][RB]
    T* w = a.w + (size_t)b * mx + a0;
    const size_t sk = (size_t)my * mx;
    for (int t = threadIdx.x; t < mz * RB; t += W::NT) {
        const int k = t / RB, c = t - k * RB;
        if (a0 + c < mx) copy_async<sizeof(T)>(S + t, w + k * sk + c);
    }
    stage_matrix<T, MP, MP, W::NT>(FZ, a.M.Ft[2], mz, 0);
    stage_matrix<T, MP, MP, W::NT>(BZ, a.M.Bt[2], mz, 0);
    copies_done();
    T acc[RM][RN];
    const int r0 = W::row(), c0 = W::col();
    W::multiply(S, FZ, mz, acc);
    const T ly = a.M.lam[1][b];
#pragma unroll
    for (int r = 0; r < RM; r++) {
        const T lxy = ly + a.M.lam[0][min(a0 + r0 + r, mx - 1)];
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (c0 + c < mz) U[(c0 + c) * RB + r0 + r] = acc[r][c] / (lxy + a.M.lam[2][c0 + c]);
    }
    __syncthreads();
    W::multiply(U, BZ, mz, acc);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (c0 + c < mz) S[(c0 + c) * RB + r0 + r] = acc[r][c];
    __syncthreads();
    for (int t = threadIdx.x; t < mz * RB; t += W::NT) {
        const int k = t / RB, c = t - k * RB;
        if (a0 + c < mx) w[k * sk + c] = S[t];
    }
}

// Backward y then x: plane k, rows j0 .. j0 + RB - 1 of the solution's interior
template <typename T, int MP, int RB, int RM, int RN>
__device__ __forceinline__ void direct_back(const DirectArgs<T>& a, T* sm)
{
    using W = Tile<T, MP, RB, RM, RN>;
    const int mx = a.n[0] - 2, my = a.n[1] - 2;
    const int k = blockIdx.x, j0 = blockIdx.y * RB;
    T* P = sm;                 // [my][MP] the plane's modes
    T* BX = P + my * MP;       // [mx][MP]
    T* BY = BX + mx * MP;      // [my][RB]
    T* T1 = BY + my * RB;      // [mx][RB]
    const T* w = a.w + (size_t)k * my * mx;
    for (int t = threadIdx.x; t < my * MP; t += W::NT) {
        const int b = t / MP, i = t - b * MP;
        if (i < mx) copy_async<sizeof(T)>(P + t, w + (size_t)b * mx + i);
    }
    stage_matrix<T, MP, MP, W::NT>(BX, a.M.Bt[0], mx, 0);
    stage_matrix<T, MP, RB, W::NT>(BY, a.M.Bt[1], my, j0);
    copies_done();
    T acc[RM][RN];
    const int r0 = W::row(), c0 = W::col();
    W::multiply(BY, P, my, acc);
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (c0 + c < mx) T1[(c0 + c) * RB + r0 + r] = acc[r][c];
    __syncthreads();
    W::multiply(T1, BX, mx, acc);
    T* u = a.u + ((size_t)(k + 1) * a.n[1] + 1) * a.n[0] + 1;
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++)
            if (j0 + r0 + r < my && c0 + c < mx) u[(size_t)(j0 + r0 + r) * a.n[0] + c0 + c] = acc[r][c];
}

template <typename T, int MP, int RB, int RM, int RN, int STAGE>
__global__ void __launch_bounds__((Tile<T, MP, RB, RM, RN>::NT)) k_direct(const __grid_constant__ DirectArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char dir_sm[];
    T* sm = reinterpret_cast<T*>(dir_sm);
    if (STAGE == 0) direct_fwd<T, MP, RB, RM, RN>(a, sm);
    else if (STAGE == 1) direct_z<T, MP, RB, RM, RN>(a, sm);
    else direct_back<T, MP, RB, RM, RN>(a, sm);
}

// lockstep batches: member = blockIdx.z
template <int MP, int RB, int RM, int RN, int STAGE>
__global__ void __launch_bounds__((Tile<float, MP, RB, RM, RN>::NT)) k_direct_bat(const __grid_constant__ BatPack<BatDirect> m)
{
    extern __shared__ __align__(16) unsigned char dir_sm[];
    float* sm = reinterpret_cast<float*>(dir_sm);
    const BatDirect& M = m.m[blockIdx.z];
    if (M.ctl->go_in == 0) return;   // this member's inner loop has ended
    if (STAGE == 0) direct_fwd<float, MP, RB, RM, RN>(M.a, sm);
    else if (STAGE == 1) direct_z<float, MP, RB, RM, RN>(M.a, sm);
    else direct_back<float, MP, RB, RM, RN>(M.a, sm);
}

template <typename T, int MP, int RB, int RM, int RN>
struct Direct {
    static size_t smem(const int n[3])
    {
        const size_t mx = n[0] - 2, my = n[1] - 2, mz = n[2] - 2;
        return sizeof(T) * std::max((mx + my) * (size_t)(MP + RB), 2 * mz * (size_t)(MP + RB));
    }
    static cudaError_t launch(const DirectArgs<T>& a, cudaStream_t s)
    {
        const unsigned mx = a.n[0] - 2, my = a.n[1] - 2, mz = a.n[2] - 2;
        constexpr int NT = Tile<T, MP, RB, RM, RN>::NT;
        k_direct<T, MP, RB, RM, RN, 0><<<dim3(mz, (my + RB - 1) / RB), NT, smem(a.n), s>>>(a);
        k_direct<T, MP, RB, RM, RN, 1><<<dim3(my, (mx + RB - 1) / RB), NT, smem(a.n), s>>>(a);
        k_direct<T, MP, RB, RM, RN, 2><<<dim3(mz, (my + RB - 1) / RB), NT, smem(a.n), s>>>(a);
        return cudaGetLastError();
    }
    static cudaError_t launch_bat(const int n[3], const BatPack<BatDirect>& m, int nm, cudaStream_t s)
    {
        const unsigned mx = n[0] - 2, my = n[1] - 2, mz = n[2] - 2;
        constexpr int NT = Tile<float, MP, RB, RM, RN>::NT;
        k_direct_bat<MP, RB, RM, RN, 0><<<dim3(mz, (my + RB - 1) / RB, nm), NT, smem(n), s>>>(m);
        k_direct_bat<MP, RB, RM, RN, 1><<<dim3(my, (mx + RB - 1) / RB, nm), NT, smem(n), s>>>(m);
        k_direct_bat<MP, RB, RM, RN, 2><<<dim3(mz, (my + RB - 1) / RB, nm), NT, smem(n), s>>>(m);
        return cudaGetLastError();
    }
    static void attributes()
    {
        constexpr int MOST = 160 * 1024;
        cudaFuncSetAttribute(k_direct<T, MP, RB, RM, RN, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
        cudaFuncSetAttribute(k_direct<T, MP, RB, RM, RN, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
        cudaFuncSetAttribute(k_direct<T, MP, RB, RM, RN, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
        if constexpr (sizeof(T) == 4) {
            cudaFuncSetAttribute(k_direct_bat<MP, RB, RM, RN, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
            cudaFuncSetAttribute(k_direct_bat<MP, RB, RM, RN, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
            cudaFuncSetAttribute(k_direct_bat<MP, RB, RM, RN, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
        }
    }
};

// FP32: a plane split over two blocks (63 planes alone leave 89 SMs idle); FP64: 4 or 8 rows per
// block, as each SM's FP64 pipe bounds it.
using D32 = Direct<float, 32, 16, 2, 2>;
using D64 = Direct<float, 64, 32, 4, 2>;
using D96 = Direct<float, 96, 48, 4, 4>;
using D32d = Direct<double, 32, 4, 1, 1>;
using D64d = Direct<double, 64, 8, 2, 1>;

template <>
cudaError_t launch_direct<float>(const DirectArgs<float>& a, cudaStream_t s)
{
    switch (direct_pad(a.n)) {
    case 32: return D32::launch(a, s);
    case 64: return D64::launch(a, s);
    default: return D96::launch(a, s);
    }
}

template <>
cudaError_t launch_direct<double>(const DirectArgs<double>& a, cudaStream_t s)
{
    switch (direct_pad(a.n)) {
    case 32: return D32d::launch(a, s);
    case 64: return D64d::launch(a, s);
    default: return cudaErrorInvalidValue;   // (DIRECT_MAX64)
    }
}

cudaError_t launch_direct_bat(const int n[3], const BatPack<BatDirect>& m, int nm, cudaStream_t s)
{
    switch (direct_pad(n)) {
    case 32: return D32::launch_bat(n, m, nm, s);
    case 64: return D64::launch_bat(n, m, nm, s);
    default: return D96::launch_bat(n, m, nm, s);
    }
}

void init_direct_attributes()
{
    D32::attributes();
    D64::attributes();
    D96::attributes();
    D32d::attributes();
    D64d::attributes();
    cudaFuncSetAttribute(k_direct_eig<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    cudaFuncSetAttribute(k_direct_eig<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
}

}  // namespace lasto
