// 3x3x3 convolution of the learned-guess network on the fifth-generation tensor cores
// (tcgen05): an implicit GEMM, M = 128 nodes per CTA, N = cout, K = 27 taps x cin, issued as
// K = 16 steps (one tap, 16 input channels) of tcgen05.mma kind::f16 (BF16 x BF16 -> FP32)
// with the accumulator in tensor memory.  Two forms: over the grids as one padded sequence
// (k_conv_seq, nearly all calls), and with gathered rows (k_conv_tc: tap groups split over CTAs,
// and rows too long for the first).
//
// In the second, A (128 x 16 per step) is gathered by the CTA's 128 threads, one node row each (the
// neighbour's 16 channels, zero outside the grid), into shared memory in the no-swizzle
// K-major core-matrix layout: 8 rows x 16 bytes per core matrix, the two K halves 128 bytes
// apart (leading byte offset), consecutive 8-row groups 256 bytes apart (stride byte
// offset).  B (cout x 16 per step) is stored in global memory already in that layout (packed
// once per weight set) and copied in.  Both arrive by cp.async (16-byte copies, zero-filled
// outside the grid) three steps ahead of their MMA, in a ring of five shared stages: one
// thread issues the MMA of a stage and commits it to the stage's mbarrier, which releases the
// stage for the copies of the step five later.  After the last step every thread reads its node's row of the
// accumulator (tcgen05.ld 32x32b: warp w owns tensor-memory lanes 32w .. 32w+31) and applies
// bias, ReLU and the output conversions.  Every mbarrier wait is bounded: on a timeout the kernel records an error, stops issuing, waits (again bounded) for its
// copies and for the last MMA it issued, which may still read its shared memory and write its
// tensor memory, frees the latter and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "internal.cuh"

namespace lasto {
namespace tc {

typedef __nv_bfloat16 bf16;

constexpr int TC_M = 128;        // nodes per CTA (MMA M), one per thread
constexpr int TC_STAGES = 5;
constexpr int TC_AHEAD = 3;      // steps whose operand copies are in flight
constexpr long long TC_SPIN_LIMIT = 1LL << 20;

struct Grid {
    int nb, D, H, W;
    __host__ __device__ size_t nodes() const { return (size_t)nb * D * H * W; }
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: no swizzle, K-major, LBO 128 B, SBO 256 B, version 1
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)(128 >> 4) << 16;
    d |= (uint64_t)(256 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M = 128, N
__host__ __device__ constexpr uint32_t make_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

// QUIT: gives up at once (the self-test; a limit that the kernels take as an argument costs their loops
// 2 to 5 %)
template <bool QUIT = false>
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    if (QUIT) return false;
    for (long long it = 0; it < TC_SPIN_LIMIT; it++) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// y = act(conv(x, w) + bias) for one 128-node tile; with part != null the raw sums of tap
// group blockIdx.y go to part[blockIdx.y][node][COUT] instead.
template <int COUT, bool QUIT>
__global__ void __launch_bounds__(TC_M) k_conv_tc(Grid g, int cin, const bf16* __restrict__ x,
                                                 const uint4* __restrict__ wpk, const float* __restrict__ bias,
                                                 int relu, float* __restrict__ y32, int ldy32, int off32,
                                                 bf16* __restrict__ y16, int ldy16, int off16,
                                                 float* __restrict__ part, int* __restrict__ err)
{
    constexpr int A_BYTES = TC_M * 32;
    constexpr int B_BYTES = COUT * 32;
    constexpr int NCOL = COUT <= 32 ? 32 : (COUT <= 64 ? 64 : 128);
    __shared__ __align__(1024) unsigned char sA[TC_STAGES][A_BYTES];
    __shared__ __align__(1024) unsigned char sB[TC_STAGES][B_BYTES];
    __shared__ __align__(8) unsigned long long mbar[TC_STAGES];
    __shared__ uint32_t tmem_slot;
    // the first step in whose iteration a wait ran out.  Threads compare it with their own step behind
    // that step's barrier, so that they leave at the same one, also where a faster thread has set it for
    // the next already.  (A barrier that carries the flag itself costs 6 % of the kernel.)
    __shared__ volatile int give_up;
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t N = g.nodes();
    const size_t node0 = (size_t)blockIdx.x * TC_M;

    if (tid == 0) {
        give_up = INT_MAX;
        for (int s = 0; s < TC_STAGES; s++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[s])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NCOL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;

    // this thread's node
    const size_t node = node0 + tid;
    const bool live = node < N;
    int b = 0, z = 0, yy = 0, xx = 0;
    if (live) {
        size_t r = node;
        xx = (int)(r % g.W);
        r /= g.W;
        yy = (int)(r % g.H);
        r /= g.H;
        z = (int)(r % g.D);
        b = (int)(r / g.D);
    }
    const int cpt = cin / 16;                       // K steps per tap
    const int tpg = 27 / gridDim.y, tap_a = blockIdx.y * tpg;
    const int nk = tpg * cpt;
    const uint32_t idesc = make_idesc(COUT);
    // canonical placement of this thread's row: 8-row group m8, row rr
    const int m8 = tid >> 3, rr = tid & 7;
    const int offA0 = (m8 * 2 + 0) * 128 + rr * 16, offA1 = (m8 * 2 + 1) * 128 + rr * 16;

    // issue the copies of step k into its stage (after the MMA that last read the stage)
    auto prefetch = [&](int k) {
        const int st = k % TC_STAGES;
        if (k >= TC_STAGES) {
            if (!mbar_wait<QUIT>(smem_u32(&mbar[st]), (uint32_t)((k / TC_STAGES - 1) & 1))) give_up = k - TC_AHEAD;
        }
        const int tap = tap_a + k / cpt, c0 = (k % cpt) * 16;
        const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
        const int zz = z + dz, y2 = yy + dy, x2 = xx + dx;
        const bool in = live && zz >= 0 && zz < g.D && y2 >= 0 && y2 < g.H && x2 >= 0 && x2 < g.W;
        const size_t nbn = in ? (((size_t)b * g.D + zz) * g.H + y2) * g.W + x2 : 0;
        const bf16* src = x + nbn * cin + c0;
        const uint32_t n = in ? 16u : 0u;   // 0: the 16 bytes are zero-filled, nothing is read
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(&sA[st][offA0])), "l"(src),
                     "r"(n)
                     : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(&sA[st][offA1])), "l"(src + 8),
                     "r"(n)
                     : "memory");
        const uint4* wsrc = wpk + ((size_t)(tap * cpt + c0 / 16)) * (B_BYTES / 16);
        for (int t = tid; t < B_BYTES / 16; t += TC_M)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(sB[st] + 16 * t)), "l"(wsrc + t)
                         : "memory");
    };
    for (int k = 0; k < TC_AHEAD; k++) {
        if (k < nk) prefetch(k);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    int issued = 0;   // steps
    bool bad = false;
    for (int kc = 0; kc < nk; kc++) {
        const int s = kc % TC_STAGES;
        if (kc + TC_AHEAD < nk) prefetch(kc + TC_AHEAD);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        asm volatile("cp.async.wait_group %0;\n" ::"n"(TC_AHEAD) : "memory");   // step kc's copies have landed
        // make the shared-memory writes visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (give_up <= kc) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint64_t ad = make_desc(smem_u32(sA[s])), bd = make_desc(smem_u32(sB[s]));
            asm volatile(
                "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                    tmem),
                "l"(ad), "l"(bd), "r"(idesc), "r"(kc > 0 ? 1 : 0)
                : "memory");
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             smem_u32(&mbar[s]))
                         : "memory");
        }
        issued = kc + 1;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    // wait for the last MMA (commits complete in issue order), also in a block that gives up
    if (issued > 0) {
        const int s = (issued - 1) % TC_STAGES;
        if (!mbar_wait(smem_u32(&mbar[s]), (uint32_t)(((issued - 1) / TC_STAGES) & 1))) bad = true;
    }
    bad = __syncthreads_or(bad || issued < nk);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (!bad) {
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        float acc[COUT];
#pragma unroll
        for (int c = 0; c < COUT; c += 16) tmem_ld16(lane_base + (uint32_t)c, acc + c);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        // the accumulator rows leave through shared memory, 16 channels at a time, so that
        // consecutive threads store consecutive addresses (the A ring is idle now)
        float* stage = reinterpret_cast<float*>(&sA[0][0]);   // [TC_M][17]
#pragma unroll
        for (int c0 = 0; c0 < COUT; c0 += 16) {
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 16; j++) stage[tid * 17 + j] = acc[c0 + j];
            __syncthreads();
            for (int e = tid; e < TC_M * 16; e += TC_M) {
                const int r = e >> 4, j = e & 15, c = c0 + j;
                const size_t nd = node0 + r;
                if (nd >= N) continue;
                const float a = stage[r * 17 + j];
                if (part) {
                    part[((size_t)blockIdx.y * N + nd) * COUT + c] = a;
                } else {
                    float v = a + (bias ? bias[c] : 0.0f);
                    if (relu) v = fmaxf(v, 0.0f);
                    if (y32) y32[nd * ldy32 + off32 + c] = v;
                    if (y16) y16[nd * ldy16 + off16 + c] = __float2bfloat16(v);
                }
            }
        }
    } else if (tid == 0 && err) {
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOL) : "memory");
}

// ---------------------------------------------------------------- grids as one padded sequence
// The nodes of all grids in one sequence of positions with a zero column after every row, a zero
// row after every plane and a zero plane after every grid: position ((b (D+1) + z)(H+1) + y)(W+1) +
// x.  Every neighbour of a node is then at a constant distance (a pad where the grid ends), so a
// tap's operand for 128 consecutive positions is the staged sequence read from another start: 16
// bytes (8 channels) per position, 8 positions to a core matrix, whatever the shift.  A tile reads
// its input from L2 once per z neighbour instead of once per tap.
struct Seq {
    int W, H, D;
    int pitch, plane;       // W + 1, (W + 1)(H + 1)
    int total;              // positions
    DivMagic dp, dh, dd;    // division by W + 1, H + 1, D + 1
};

inline bool make_seq(const Grid& g, Seq* q)
{
    const size_t total = (size_t)g.nb * (g.D + 1) * (g.H + 1) * (g.W + 1);
    if (total >= (size_t(1) << 30)) return false;
    q->W = g.W;
    q->H = g.H;
    q->D = g.D;
    q->pitch = g.W + 1;
    q->plane = (g.W + 1) * (g.H + 1);
    q->total = (int)total;
    q->dp = div_magic((unsigned)g.W + 1);
    q->dh = div_magic((unsigned)g.H + 1);
    q->dd = div_magic((unsigned)g.D + 1);
    return true;
}

// node at position p, or -1 (a pad, or outside the sequence)
__device__ __forceinline__ int seq_node(const Seq& q, int p)
{
    if ((unsigned)p >= (unsigned)q.total) return -1;
    const int q1 = (int)div_by((unsigned)p, q.dp), x = p - q1 * q.pitch;
    const int q2 = (int)div_by((unsigned)q1, q.dh), y = q1 - q2 * (q.H + 1);
    const int b = (int)div_by((unsigned)q2, q.dd), z = q2 - b * (q.D + 1);
    return x == q.W || y == q.H || z == q.D ? -1 : ((b * q.D + z) * q.H + y) * q.W + x;
}

// shared-memory matrix descriptor without swizzle, byte offsets lbo and sbo
__device__ __forceinline__ uint64_t make_desc_any(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(sbo >> 4) << 32 | (uint64_t)1 << 46;
}

// Issued by a whole warp in uniform control flow, one elected lane executing: 21 cycles per MMA at
// M = 64, N = 16 and 36 at M = 128, against 44 and more from a branch on the thread's index, where
// every descriptor has to be moved to the uniform registers.
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, int accumulate)
{
    asm volatile(
        "{\n.reg .pred p, q;\nelect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile(
        "{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar)
        : "memory");
}

__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(in ? 16u : 0u) : "memory");
}

// y = act(conv(x, w) + bias) for 256 positions per CTA: two M = 128 accumulators.  The channels go
// through shared memory 16 at a time (two buffers where there are more): the three z neighbours'
// segments of 256 + 2 (W + 2) positions and the 27 taps' weight tiles; then 2 x 27 MMAs, K = 16,
// issued by a ninth warp while the other eight load.  Bound: 3 TB/s of 32-byte pieces from L2, the
// weights a third to a half of them (a sixth of the time is MMAs; more warps, one buffer and more
// CTAs per SM, or an x neighbour triple per MMA change nothing).  8 grids of 33^3, against the kernel
// above, which gathers every tap's neighbour rows from L2 (745 MB at 48 channels), a K step per
// barrier: 48 -> 16 channels 204 -> 53 us, 16 -> 48 87 -> 33 us, 64 -> 64 336 -> 108 us.
constexpr int SQ_NT = 256, SQ_M = 256;
__host__ __device__ constexpr int sq_seg(int W) { return SQ_M + 2 * (W + 2); }
inline size_t sq_smem(int W, int cin, int cout)
{
    return (cin > 16 ? 2 : 1) * ((size_t)6 * sq_seg(W) * 16 + (size_t)27 * 32 * cout);
}

template <int COUT, bool QUIT>
__global__ void __launch_bounds__(SQ_NT + 32) k_conv_seq(Seq q, int cin, int cout, const bf16* __restrict__ x, const uint4* __restrict__ wpk,
                                                    const float* __restrict__ bias, int relu, float* __restrict__ y32,
                                                    int ldy32, int off32, bf16* __restrict__ y16, int ldy16, int off16,
                                                    int* __restrict__ err)
{
    constexpr int NCOL = 2 * COUT <= 32 ? 32 : 2 * COUT <= 64 ? 64 : 2 * COUT <= 128 ? 128 : 256;
    extern __shared__ __align__(1024) unsigned char sq_raw[];
    __shared__ __align__(8) unsigned long long mbar[2];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5;
    bool bad = false;   // a wait ran out
    const int seg = sq_seg(q.W), p0 = blockIdx.x * SQ_M, cpt = cin / 16;
    const int n0 = blockIdx.y * COUT;   // the CTA's output channels n0 .. n0 + COUT - 1
    const uint32_t a_bytes = 6 * seg * 16, buf_bytes = a_bytes + 27 * 32 * COUT, base = smem_u32(sq_raw);
    if (tid == 0) {
        for (int s = 0; s < 2; s++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[s])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NCOL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t idesc = make_idesc(COUT);

    // channels 16 c .. 16 c + 15 into buffer c & 1 (after the MMAs that last read it): a lane pair
    // per position, 32 contiguous bytes
    auto load = [&](int c) {
        if (c >= 2 && !mbar_wait<QUIT>(smem_u32(&mbar[c % 2]), (uint32_t)((c / 2 - 1) & 1))) {
            bad = true;
            return;
        }
        const uint32_t buf = base + (c % 2) * buf_bytes;
        const int h = tid & 1;
        for (int t = tid >> 1; t < 3 * seg; t += SQ_NT / 2) {
            const int dz = t >= 2 * seg ? 2 : t >= seg ? 1 : 0;
            const int nd = seq_node(q, p0 + (dz - 1) * q.plane - (q.pitch + 1) + t - dz * seg);
            copy16(buf + (h * 3 * seg + t) * 16, x + (size_t)(nd < 0 ? 0 : nd) * cin + c * 16 + h * 8, nd >= 0);
        }
        for (int t = tid; t < 27 * 2 * COUT; t += SQ_NT) {
            const int tap = t / (2 * COUT), r = t - tap * 2 * COUT;
            copy16(buf + a_bytes + t * 16, wpk + (size_t)(tap * cpt + c) * 2 * cout + 2 * n0 + r, true);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (tid < SQ_NT) load(0);
    int issued = 0;   // channel chunks
    for (int c = 0; c < cpt; c++) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // visible to the tensor core
        bad = __syncthreads_or(bad);
        if (bad) break;
        if (__shfl_sync(0xffffffffu, warp, 0) == SQ_NT / 32) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t buf = base + (c % 2) * buf_bytes;
            const uint64_t a0 = make_desc_any(buf, 3 * seg * 16, 128);
            const uint64_t b0 = make_desc(buf + a_bytes);
#pragma unroll
            for (int dz = 0; dz < 3; dz++) {
#pragma unroll
                for (int t = 0; t < 9; t++) {
                    // (positions from -(pitch + 1) on; addresses in units of 16 bytes)
                    const uint64_t ad = a0 + (uint32_t)(dz * seg + (t / 3) * q.pitch + t % 3);
                    const uint64_t bd = b0 + (dz * 9 + t) * 2 * COUT;
#pragma unroll
                    for (int m = 0; m < 2; m++) mma_f16(tmem + m * COUT, ad + m * 128, bd, idesc, c > 0 || dz > 0 || t > 0);
                }
            }
            mma_commit(smem_u32(&mbar[c % 2]));
        }
        issued = c + 1;
        if (tid < SQ_NT && c + 1 < cpt) load(c + 1);   // while these are issued
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (issued > 0) {   // the last commit (they complete in issue order), also in a block that gives up
        const int c = issued - 1;
        if (!mbar_wait(smem_u32(&mbar[c % 2]), (uint32_t)((c / 2) & 1))) bad = true;
    }
    bad = __syncthreads_or(bad);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (!bad) {
        // warp w: accumulator w / 4, tensor-memory lanes 32 (w % 4) ..; the rows leave through shared
        // memory (idle now), so that a warp stores consecutive channels of consecutive nodes
        if (tid < SQ_NT) {
            constexpr int LD = COUT + 4, Q = COUT / 4;
            const int nd = seq_node(q, p0 + tid), lane = tid & 31;
            const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * COUT);
            float* stage = reinterpret_cast<float*>(sq_raw) + warp * 32 * LD;
#pragma unroll
            for (int c0 = 0; c0 < COUT; c0 += 16) {
                float v[16];
                tmem_ld16(lane_base + (uint32_t)c0, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    v[j] += bias ? bias[n0 + c0 + j] : 0.0f;
                    if (relu) v[j] = fmaxf(v[j], 0.0f);
                }
#pragma unroll
                for (int j = 0; j < 16; j += 4)
                    *reinterpret_cast<float4*>(stage + lane * LD + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
            __syncwarp();
            const bool v32 = ((ldy32 | off32) & 3) == 0 && ((uintptr_t)y32 & 15) == 0;
            const bool v16 = ((ldy16 | off16) & 3) == 0 && ((uintptr_t)y16 & 7) == 0;
            for (int e = lane; e < 32 * Q; e += 32) {
                const int r = e / Q, c = (e - r * Q) * 4, node = __shfl_sync(0xffffffffu, nd, r);
                const float4 v = *reinterpret_cast<const float4*>(stage + r * LD + c);
                if (node < 0) continue;
                if (y32) {
                    float* o = y32 + (size_t)node * ldy32 + off32 + n0 + c;
                    if (v32) {
                        *reinterpret_cast<float4*>(o) = v;
                    } else {
                        o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
                    }
                }
                if (y16) {
                    bf16* o = y16 + (size_t)node * ldy16 + off16 + n0 + c;
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
                    if (v16) {
                        *reinterpret_cast<uint2*>(o) =
                            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                    } else {
                        o[0] = lo.x, o[1] = lo.y, o[2] = hi.x, o[3] = hi.y;
                    }
                }
            }
        }
    } else if (tid == 0 && err) {
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOL) : "memory");
}

// Pack w [27][cin][cout] into the per-step B tiles: step k = tap * (cin/16) + c0/16 holds
// element (n = output channel, kk = input channel c0 + kk) at byte
// ((n/8)*2 + kk/8)*128 + (n%8)*16 + (kk%8)*2 of its cout*32-byte tile.
__global__ void k_pack_weights(int cin, int cout, const bf16* __restrict__ w, bf16* __restrict__ wpk)
{
    const size_t total = (size_t)27 * cin * cout;
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int co = (int)(t % cout);
    const int ci = (int)((t / cout) % cin);
    const int tap = (int)(t / ((size_t)cout * cin));
    const int step = tap * (cin / 16) + ci / 16, kk = ci % 16;
    const size_t byte = (size_t)step * cout * 32 + ((co / 8) * 2 + kk / 8) * 128 + (co % 8) * 16 + (kk % 8) * 2;
    wpk[byte / 2] = w[t];
}

__global__ void k_tc_epilogue(size_t N, int cout, int groups, const float* __restrict__ part,
                              const float* __restrict__ bias, int relu, float* __restrict__ y32, int ldy32, int off32,
                              bf16* __restrict__ y16, int ldy16, int off16)
{
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= N * cout) return;
    const size_t nd = t / cout;
    const int co = (int)(t % cout);
    float v = part[t];
    for (int k = 1; k < groups; k++) v += part[(size_t)k * N * cout + t];
    v += bias ? bias[co] : 0.0f;
    if (relu) v = fmaxf(v, 0.0f);
    if (y32) y32[nd * ldy32 + off32 + co] = v;
    if (y16) y16[nd * ldy16 + off16 + co] = __float2bfloat16(v);
}

// ---------------------------------------------------------------- weight gradient
// dw[tap][ci][co] += sum over nodes of x[node + tap][ci] dy[node][co]: a GEMM with M = the
// (tap, ci) rows of a tile of taps (TPT = floor(128 / cin) taps, 128 rows, rows past TPT cin
// zero), N = cout, K = nodes, one CTA per (node chunk, tile).  Both operands are read
// MN-major from channels-last rows: a stage holds 64 nodes, for each node the TPT neighbour
// rows of cin channels (16-byte pieces; zero outside the grid) in A and its cout channels of
// dy in B, and is consumed by four K = 16 MMAs.  Core matrices (8 nodes x 8 channels, 128
// contiguous bytes) sit 128 bytes apart along the channels and 16 * rows bytes apart along
// the nodes; for these MN-major operands the descriptor's leading byte offset is the step
// along K (nodes) and its stride byte offset the step along M / N (channels) -- the other
// assignment reads outside the tiles (measured: wrong sums).  The accumulator (128 lanes x
// cout columns of tensor memory) is added to dw with FP32 atomics at the end.
constexpr int WG_STAGES = 3;
constexpr int WG_AHEAD = 2;
constexpr int WG_STEP = 64;                          // nodes per stage (four MMAs)
constexpr int WG_CHUNK = 2048;                       // nodes per CTA
constexpr int WG_A_BYTES = TC_M * 2 * WG_STEP;       // 128 rows x 64 nodes
__host__ __device__ constexpr int wg_smem(int cout) { return WG_STAGES * (WG_A_BYTES + cout * 2 * WG_STEP); }

__device__ __forceinline__ uint64_t make_desc_mn(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(sbo >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// node index -> (b, z, y, x) by multiply-high division by the invariant W, H, D (nodes < 2^31)
struct GridDiv {
    DivMagic w, h, d;
};
// div_by for divisors from 1 on (l = 0: m = 2^31, a shift by 31)
__device__ __forceinline__ unsigned div_any(unsigned n, DivMagic q)
{
    return (unsigned)(((unsigned long long)n * q.m) >> (32 + q.s));
}

template <int COUT, bool QUIT>
__global__ void __launch_bounds__(TC_M) k_conv_wgrad_tc(Grid g, GridDiv gd, int cin, const bf16* __restrict__ x,
                                                       const bf16* __restrict__ dy, float* __restrict__ dw,
                                                       int* __restrict__ err)
{
    constexpr int B_BYTES = COUT * 2 * WG_STEP;
    constexpr int NCOL = COUT <= 32 ? 32 : (COUT <= 64 ? 64 : 128);
    extern __shared__ __align__(1024) unsigned char wg_smem_raw[];
    unsigned char* sA = wg_smem_raw;                               // [WG_STAGES][WG_A_BYTES]
    unsigned char* sB = wg_smem_raw + WG_STAGES * WG_A_BYTES;      // [WG_STAGES][B_BYTES]
    __shared__ __align__(8) unsigned long long mbar[WG_STAGES];
    __shared__ uint32_t tmem_slot;
    // the first step in whose iteration a wait ran out.  Threads compare it with their own step behind
    // that step's barrier, so that they leave at the same one, also where a faster thread has set it for
    // the next already.  (A barrier that carries the flag itself costs 6 % of the kernel.)
    __shared__ volatile int give_up;
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t N = g.nodes();
    const size_t node0 = (size_t)blockIdx.x * WG_CHUNK;
    const int tpt = TC_M / cin, tap0 = blockIdx.y * tpt;
    const int ntap = min(tpt, 27 - tap0);
    const int rows = ntap * cin;                                   // live rows of the tile
    const int r8n = rows / 8;                                      // 16-byte pieces per node in A

    // zero the ring (padding rows stay zero; no copy ever writes them)
    for (int t = tid; t < WG_STAGES * (WG_A_BYTES + B_BYTES) / 16; t += TC_M)
        reinterpret_cast<uint4*>(wg_smem_raw)[t] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        give_up = INT_MAX;
        for (int st = 0; st < WG_STAGES; st++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[st])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NCOL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const size_t nodes = N > node0 ? min((size_t)WG_CHUNK, N - node0) : 0;
    const int nk = (int)((nodes + WG_STEP - 1) / WG_STEP);
    // core-matrix steps: along the channels (M / N) and along the nodes (K)
    constexpr uint32_t A_CH = 128, A_ND = 16 * 128, B_CH = 128, B_ND = (COUT / 8) * 128;
    const uint32_t idesc = make_idesc(COUT) | (1u << 15) | (1u << 16);   // A and B MN-major

    auto prefetch = [&](int k) {
        const int st = k % WG_STAGES;
        if (k >= WG_STAGES) {
            if (!mbar_wait<QUIT>(smem_u32(&mbar[st]), (uint32_t)((k / WG_STAGES - 1) & 1))) give_up = k - WG_AHEAD;
        }
        // A: piece p = (node kk, row group r8), r8 fastest (one node's row read contiguously)
        for (int p = tid; p < WG_STEP * r8n; p += TC_M) {
            const int kk = p / r8n, r8 = p - kk * r8n;
            const int m = r8 * 8, tl = m / cin, c0 = m - tl * cin;
            const size_t node = node0 + (size_t)k * WG_STEP + kk;
            bool in = node < N;
            size_t nbn = 0;
            if (in) {
                const unsigned r = (unsigned)node, q1 = div_any(r, gd.w), q2 = div_any(q1, gd.h), b = div_any(q2, gd.d);
                const int xx = (int)(r - q1 * (unsigned)g.W), yy = (int)(q1 - q2 * (unsigned)g.H);
                const int z = (int)(q2 - b * (unsigned)g.D);
                const int tap = tap0 + tl;
                const int zz = z + tap / 9 - 1, y2 = yy + (tap / 3) % 3 - 1, x2 = xx + tap % 3 - 1;
                in = zz >= 0 && zz < g.D && y2 >= 0 && y2 < g.H && x2 >= 0 && x2 < g.W;
                nbn = in ? (((size_t)b * g.D + zz) * g.H + y2) * g.W + x2 : 0;
            }
            const uint32_t dst = smem_u32(sA + st * WG_A_BYTES + r8 * A_CH + (kk >> 3) * A_ND + (kk & 7) * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(x + nbn * cin + c0),
                         "r"(in ? 16u : 0u)
                         : "memory");
        }
        for (int p = tid; p < WG_STEP * (COUT / 8); p += TC_M) {
            const int kk = p / (COUT / 8), c8 = p - kk * (COUT / 8);
            const size_t node = node0 + (size_t)k * WG_STEP + kk;
            const bool in = node < N;
            const uint32_t dst = smem_u32(sB + st * B_BYTES + c8 * B_CH + (kk >> 3) * B_ND + (kk & 7) * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst),
                         "l"(dy + (in ? node : 0) * COUT + c8 * 8), "r"(in ? 16u : 0u)
                         : "memory");
        }
    };
    for (int k = 0; k < WG_AHEAD; k++) {
        if (k < nk) prefetch(k);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    int issued = 0;   // steps
    bool bad = false;
    for (int kc = 0; kc < nk; kc++) {
        const int st = kc % WG_STAGES;
        if (kc + WG_AHEAD < nk) prefetch(kc + WG_AHEAD);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        asm volatile("cp.async.wait_group %0;\n" ::"n"(WG_AHEAD) : "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (give_up <= kc) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int j = 0; j < WG_STEP / 16; j++) {   // 16 nodes = two core matrices along K
                const uint64_t ad = make_desc_mn(smem_u32(sA + st * WG_A_BYTES + j * 2 * A_ND), A_ND, A_CH);
                const uint64_t bd = make_desc_mn(smem_u32(sB + st * B_BYTES + j * 2 * B_ND), B_ND, B_CH);
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                        tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"((kc > 0 || j > 0) ? 1 : 0)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             smem_u32(&mbar[st]))
                         : "memory");
        }
        issued = kc + 1;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (issued > 0) {   // the last MMA, also in a block that gives up
        const int st = (issued - 1) % WG_STAGES;
        if (!mbar_wait(smem_u32(&mbar[st]), (uint32_t)(((issued - 1) / WG_STAGES) & 1))) bad = true;
    }
    bad = __syncthreads_or(bad || issued < nk);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (!bad && nk > 0) {
        // thread tid owns accumulator row m = tid (tensor-memory lane tid)
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        float acc[COUT];
#pragma unroll
        for (int c = 0; c < COUT; c += 16) tmem_ld16(lane_base + (uint32_t)c, acc + c);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        const int m = tid;
        if (m < rows) {
            const int tl = m / cin, ci = m - tl * cin;
            float* dst = dw + ((size_t)(tap0 + tl) * cin + ci) * COUT;
#pragma unroll
            for (int c = 0; c < COUT; c++) atomicAdd(dst + c, acc[c]);
        }
    } else if (bad && tid == 0 && err) {
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOL) : "memory");
}

// The same GEMM over the padded sequence: per stage 128 positions of dy and the three z neighbours'
// segments of x (CG channels), both channel group by channel group, 16 bytes per position, which is
// the MN-major operand layout (8 positions x 8 channels to a core matrix) for every shift.  One
// M = 64 MMA (64 channel rows, those beyond CG unused) per tap and 16 positions.  Up to 16 output
// channels the three x neighbours share one: dw[dz, dy, dx] = sum_p x[p + dz, dy] dy[p - dx], with dy
// staged at the three shifts (an MMA costs 21 cycles at 16 columns, 26 at 48, 43 at 96: at 16
// channels 62 against 79 us, at 48 140 against 131).  Every tap has its own columns of tensor memory,
// so the input is staged once for all taps of the CTA.  Stages alternate between two buffers, filled
// by eight warps while a ninth issues; a CTA takes every gridDim.x-th one, and adds its sums to dw
// with vector reductions, at the latest after `most` stages: the tensor core's FP32 accumulation
// truncates, so its error grows with the length of a sum (positive values, 64 x 64 channels on 8 grids
// of 33^3: 1.7e-5 of the largest and 245 us with one sum per CTA, 3.6e-6 and 258 us so; 3.8e-6 in the
// gathered form).  Bound: 32-byte pieces from L2 (3 to 4 TB/s; three or four
// buffers, or 16 loading warps, change nothing).  8 grids of 33^3, against the kernel above (27
// gathered rows per node): 48 x 16 channels 330 -> 57 us.
constexpr int WS_K = 128, WS_NT = 256;
__host__ __device__ constexpr int ws_dx(int cout) { return cout <= 16 ? 3 : 1; }
__host__ __device__ constexpr int ws_seg(int W) { return WS_K + 2 * (W + 2); }
// groups of ws_dx taps whose columns fit in tensor memory
__host__ __device__ constexpr int ws_groups(int cout) { return cout <= 16 ? 9 : cout <= 32 ? 14 : cout <= 48 ? 9 : cout <= 64 ? 7 : cout <= 96 ? 5 : 4; }
inline size_t ws_smem(int W, int cg, int cout)
{
    // two buffers, and what the unused rows of the second one's operand read beyond it
    return 2 * ((size_t)cg / 8 * 3 * ws_seg(W) * 16 + (size_t)ws_dx(cout) * cout / 8 * WS_K * 16) + (size_t)(64 - cg) / 8 * 3 * ws_seg(W) * 16;
}

// One element's sum over the stages k0 .. k1 - 1 of a CTA from the nodes themselves: output node at
// position p - e, input node one tap away.
__device__ __noinline__ float ws_node_sum(const Seq& q, int k0, int k1, int e, int tap, const bf16* __restrict__ x, int cin,
                                          const bf16* __restrict__ dy, int cout)
{
    const int shift = (tap / 9 - 1) * q.plane + (tap / 3 % 3 - 1) * q.pitch + tap % 3 - 1;
    float s = 0.0f;
    for (int k = k0; k < k1; k++)
        for (int i = 0; i < WS_K; i++) {
            const int p = ((int)blockIdx.x + k * (int)gridDim.x) * WS_K + i - e;
            const int out = seq_node(q, p), in = seq_node(q, p + shift);
            if (out >= 0 && in >= 0) s = fmaf(__bfloat162float(x[(size_t)in * cin]), __bfloat162float(dy[(size_t)out * cout]), s);
        }
    return s;
}

template <int COUT, bool QUIT>
__global__ void __launch_bounds__(WS_NT + 32) k_conv_wgrad_seq(Seq q, int cin, int cg, int most, const bf16* __restrict__ x,
                                                          const bf16* __restrict__ dy, float* __restrict__ dw,
                                                          int* __restrict__ err)
{
    constexpr int DX = ws_dx(COUT), N = DX * COUT, TAPS = ws_groups(COUT), USED = TAPS * N;   // a group: DX taps
    constexpr int NCOL = USED <= 128 ? 128 : USED <= 256 ? 256 : 512;
    extern __shared__ __align__(1024) unsigned char ws_raw[];
    __shared__ __align__(8) unsigned long long mbar[2];
    __shared__ uint32_t tmem_slot;
    bool bad = false;   // a wait ran out
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int seg = ws_seg(q.W), groups = cin / cg;
    const int tap0 = (int)blockIdx.y / groups * TAPS, c0 = (int)blockIdx.y % groups * cg, ntap = min(TAPS, 27 / DX - tap0);
    const int nchunk = (q.total + WS_K - 1) / WS_K;
    const int nk = ((int)blockIdx.x < nchunk) ? (nchunk - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int runs = (nk + most - 1) / most, run = nk > 0 ? (nk + runs - 1) / runs : 1;   // stages per accumulation
    const uint32_t a_bytes = (uint32_t)cg / 8 * 3 * seg * 16, b_bytes = N / 8 * WS_K * 16;
    // both B buffers, then both A buffers
    const uint32_t baseA = smem_u32(ws_raw) + 2 * b_bytes, baseB = smem_u32(ws_raw);
    if (tid == 0) {
        for (int s = 0; s < 2; s++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[s])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(NCOL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // M = 64, A and B MN-major
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | (4u << 24);

    auto load = [&](int k) {
        const int s = k & 1, p0 = ((int)blockIdx.x + k * (int)gridDim.x) * WS_K;
        if (k >= 2 && !mbar_wait<QUIT>(smem_u32(&mbar[s]), (uint32_t)((k / 2 - 1) & 1))) {
            bad = true;
            return;
        }
        const int h = tid & 1;
        for (int t = tid >> 1; t < 3 * seg; t += WS_NT / 2) {
            const int dz = t >= 2 * seg ? 2 : t >= seg ? 1 : 0;
            const int nd = seq_node(q, p0 + (dz - 1) * q.plane - (q.pitch + 1) + t - dz * seg);
            const bf16* src = x + (size_t)(nd < 0 ? 0 : nd) * cin + c0;
            for (int c = h; c < cg / 8; c += 2) copy16(baseA + s * a_bytes + (c * 3 * seg + t) * 16, src + c * 8, nd >= 0);
        }
        for (int t = tid >> 1; t < DX * WS_K; t += WS_NT / 2) {
            const int dx = t / WS_K, i = t - dx * WS_K;   // dy at p0 + i - (dx - 1)
            const int nd = seq_node(q, p0 + i - (DX == 3 ? dx - 1 : 0));
            const bf16* src = dy + (size_t)(nd < 0 ? 0 : nd) * COUT;
#pragma unroll
            for (int c = 0; c < COUT / 16; c++)
                copy16(baseB + s * b_bytes + ((dx * (COUT / 8) + 2 * c + h) * WS_K + i) * 16, src + (2 * c + h) * 8, nd >= 0);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // the sums of a run into dw.  An M = 64 accumulator: row r in tensor-memory lane 32 (r / 16) + r % 16
    // A NaN may come from a pad alone (its 0 times an infinity at the grid's edge): such elements are formed
    // again without the pads.
    auto drain = [&](int k0, int k1) {
        const int row = (warp & 3) * 16 + (lane & 15);
        const bool live = lane < 16 && row < cg, vec = ((uintptr_t)dw & 15) == 0;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int t = tid < WS_NT ? warp >> 2 : ntap * DX; t < ntap * DX; t += WS_NT / 128) {
            float* dst = dw + ((size_t)(tap0 * DX + t) * cin + c0 + row) * COUT;
#pragma unroll
            for (int c = 0; c < COUT; c += 16) {
                float v[16];
                __syncwarp();
                tmem_ld16(lane_base + (uint32_t)(t * COUT + c), v);
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                if (!live) continue;
                bool nan = false;
#pragma unroll
                for (int j = 0; j < 16; j++) nan |= v[j] != v[j];
                if (nan) {
#pragma unroll 1
                    for (int j = 0; j < 16; j++)
                        atomicAdd(dst + c + j, ws_node_sum(q, k0, k1, DX == 3 ? t % 3 - 1 : 0, tap0 * DX + t, x + c0 + row, cin,
                                                           dy + c + j, COUT));
                } else if (vec) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(dst + c + j), "f"(v[j]),
                                     "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3])
                                     : "memory");
                } else {
                    for (int j = 0; j < 16; j++) atomicAdd(dst + c + j, v[j]);
                }
            }
        }
    };
    if (nk > 0 && tid < WS_NT) load(0);
    int issued = 0;   // stages
    for (int k = 0, first = 0; k < nk; k++) {   // first: of the run
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        bad = __syncthreads_or(bad);
        if (bad) break;
        if (__shfl_sync(0xffffffffu, warp, 0) == WS_NT / 32) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint64_t a0 = make_desc_any(baseA + (k & 1) * a_bytes, 128, 3 * seg * 16);
            const uint64_t b0 = make_desc_any(baseB + (k & 1) * b_bytes, 128, WS_K * 16);
#pragma unroll
            for (int t = 0; t < TAPS; t++) {
                const int tap = (tap0 + t) * DX;   // its start in a segment set, in positions
                const uint64_t ad = a0 + (uint32_t)(tap / 9 * seg + (tap / 3) % 3 * q.pitch + (DX == 3 ? 1 : tap % 3));
                if (t < ntap) {
#pragma unroll
                    for (int j = 0; j < WS_K / 16; j++) mma_f16(tmem + t * N, ad + j * 16, b0 + j * 16, idesc, k > first || j > 0);
                }
            }
            mma_commit(smem_u32(&mbar[k & 1]));
        }
        issued = k + 1;
        if (tid < WS_NT && k + 1 < nk) load(k + 1);   // while these are issued
        if (k + 1 == nk || k + 1 == first + run) {
            // (commits complete in issue order)
            if (!mbar_wait<QUIT>(smem_u32(&mbar[k & 1]), (uint32_t)((k / 2) & 1))) bad = true;
            bad = __syncthreads_or(bad);
            if (bad) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            drain(first, k + 1);
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");   // (the next stage's barrier)
            first = k + 1;
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (bad && issued > 0) mbar_wait(smem_u32(&mbar[(issued - 1) & 1]), (uint32_t)(((issued - 1) / 2) & 1));
    if (bad && tid == 0 && err) {
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOL) : "memory");
}

}  // namespace tc

cudaError_t launch_pack_weights(int cin, int cout, const void* w, void* wpk, cudaStream_t s)
{
    const size_t total = (size_t)27 * cin * cout;
    tc::k_pack_weights<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(cin, cout, (const tc::bf16*)w, (tc::bf16*)wpk);
    return cudaGetLastError();
}

int conv_fwd_tc(int nb, const int dims[3], int cin, int cout, const void* x, const void* wpk, const float* bias,
                int relu, float* y32, int ldy32, int off32, void* y16, int ldy16, int off16, float* scratch,
                size_t scratch_floats, int* err, void* stream, bool give_up)
{
    using namespace tc;
    if (give_up && cout != 16 && cout != 32 && cout != 64) return LASTO_ERR_INVALID_ARG;   // the self-test's sizes
    if (nb < 1 || !dims || cin % 16 || cin < 16 || !x || !wpk ||
        !(cout == 16 || cout == 32 || cout == 48 || cout == 64 || cout == 96 || cout == 128))
        return LASTO_ERR_INVALID_ARG;
    Grid g{nb, dims[2], dims[1], dims[0]};
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned nbk = (unsigned)((g.nodes() + TC_M - 1) / TC_M);
    int groups = 1;
    if (scratch)
        for (int cand : {3, 9, 27})
            if ((size_t)nbk * cand <= 2432 && (size_t)cand * g.nodes() * cout <= scratch_floats) groups = cand;
    float* part = groups > 1 ? scratch : nullptr;
    const dim3 grid(nbk, groups);
    const bf16* X = (const bf16*)x;
    const uint4* W = (const uint4*)wpk;
    bf16* Y16 = (bf16*)y16;
    // the padded sequence where a tile's segments fit in shared memory (rows of up to about 800
    // nodes).  Many channels on few tiles are better
    // split over CTAs by taps (128 -> 64 channels: 6 tiles 23.3 against 18.8 us, 16 tiles 23.8
    // against 25.4; 64 -> 64 on 3 tiles 15.1 against 14.8, 16 -> 16 7.1 against 12.6), if there is
    // room for their sums (without: 97 us).
    Seq q;
    const int half = cout > 64 ? 2 : 1;   // 96 and 128 output channels as two CTAs' work
    const size_t sm = sq_smem(g.W, cin, cout / half);
    if (make_seq(g, &q) && (!scratch || cin <= 64 || q.total / SQ_M >= cin / 8) && sm <= 200 * 1024) {
        const dim3 tiles((unsigned)((q.total + SQ_M - 1) / SQ_M), (unsigned)half);
#define LASTO_SQ_CASE(C, Q)                                                                                           \
    case C + Q:                                                                                                       \
        if (cudaFuncSetAttribute(k_conv_seq<C, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) !=        \
            cudaSuccess)                                                                                              \
            return LASTO_ERR_CUDA;                                                                                    \
        k_conv_seq<C, Q><<<tiles, SQ_NT + 32, sm, s>>>(q, cin, cout, X, W, bias, relu, y32, ldy32, off32, Y16, ldy16, off16, \
                                                    err);                                                             \
        break;
        switch (cout / half + (give_up ? 1 : 0)) {
            LASTO_SQ_CASE(16, 0)
            LASTO_SQ_CASE(32, 0)
            LASTO_SQ_CASE(48, 0)
            LASTO_SQ_CASE(64, 0)
            LASTO_SQ_CASE(16, 1)
            LASTO_SQ_CASE(32, 1)
            LASTO_SQ_CASE(64, 1)
        }
#undef LASTO_SQ_CASE
        return cudaGetLastError() == cudaSuccess ? LASTO_OK : LASTO_ERR_CUDA;
    }
#define LASTO_TC_CASE(C, Q)                                                                                           \
    case C + Q:                                                                                                       \
        k_conv_tc<C, Q><<<grid, TC_M, 0, s>>>(g, cin, X, W, bias, relu, y32, ldy32, off32, Y16, ldy16, off16, part,   \
                                           err);                                                                      \
        break;
    switch (cout + (give_up ? 1 : 0)) {
        LASTO_TC_CASE(16, 0)
        LASTO_TC_CASE(32, 0)
        LASTO_TC_CASE(48, 0)
        LASTO_TC_CASE(64, 0)
        LASTO_TC_CASE(96, 0)
        LASTO_TC_CASE(128, 0)
        LASTO_TC_CASE(16, 1)
        LASTO_TC_CASE(32, 1)
        LASTO_TC_CASE(64, 1)
        default: return LASTO_ERR_INVALID_ARG;
    }
#undef LASTO_TC_CASE
    if (part) {
        const size_t n = g.nodes() * cout;
        k_tc_epilogue<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g.nodes(), cout, groups, part, bias, relu, y32,
                                                                  ldy32, off32, Y16, ldy16, off16);
    }
    return cudaGetLastError() == cudaSuccess ? LASTO_OK : LASTO_ERR_CUDA;
}

int conv_wgrad_tc(int nb, const int dims[3], int cin, int cout, const void* x, const void* dy16, float* dw,
                  int* err, void* stream, bool give_up)
{
    using namespace tc;
    if (give_up && cout != 16 && cout != 32 && cout != 64) return LASTO_ERR_INVALID_ARG;   // the self-test's sizes
    if (nb < 1 || !dims || cin % 16 || cin < 16 || cin > 128 || !x || !dy16 || !dw ||
        !(cout == 16 || cout == 32 || cout == 48 || cout == 64 || cout == 96 || cout == 128))
        return LASTO_ERR_INVALID_ARG;
    Grid g{nb, dims[2], dims[1], dims[0]};
    if (g.nodes() == 0) return LASTO_OK;
    if (g.nodes() >= (size_t(1) << 31)) return LASTO_ERR_INVALID_ARG;
    const GridDiv gd{div_magic((unsigned)g.W), div_magic((unsigned)g.H), div_magic((unsigned)g.D)};
    cudaStream_t s = (cudaStream_t)stream;
    const int tpt = TC_M / cin;
    const dim3 grid((unsigned)((g.nodes() + WG_CHUNK - 1) / WG_CHUNK), (unsigned)((27 + tpt - 1) / tpt));
    const bf16* X = (const bf16*)x;
    const bf16* DY = (const bf16*)dy16;
    // the padded sequence with the largest group of channels whose buffers fit (rows of up to about
    // 450 nodes); one CTA per SM: its accumulators fill the tensor memory
    Seq q;
    int cg = 64;
    while (cg > 16 && (cin % cg || ws_smem(g.W, cg, cout) > 220 * 1024)) cg -= 16;
    if (make_seq(g, &q) && cin % cg == 0 && ws_smem(g.W, cg, cout) <= 220 * 1024) {
        const size_t sm = std::max(ws_smem(g.W, cg, cout), (size_t)116 * 1024);
        const int per = ws_groups(cout) * ws_dx(cout);
        const int ny = (27 + per - 1) / per * (cin / cg), nchunk = (q.total + WS_K - 1) / WS_K;
        const dim3 grid((unsigned)std::min(nchunk, std::max(1, 152 / ny)), (unsigned)ny);
        // a sum of at most WG_CHUNK nodes, as in the gathered form (the pads add nothing)
        const int most = (int)((size_t)WG_CHUNK * (size_t)q.total / g.nodes() / WS_K);
#define LASTO_WS_CASE(C, Q)                                                                                           \
    case C + Q:                                                                                                       \
        if (cudaFuncSetAttribute(k_conv_wgrad_seq<C, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) !=  \
            cudaSuccess)                                                                                              \
            return LASTO_ERR_CUDA;                                                                                    \
        k_conv_wgrad_seq<C, Q><<<grid, WS_NT + 32, sm, s>>>(q, cin, cg, most, X, DY, dw, err);                        \
        break;
        switch (cout + (give_up ? 1 : 0)) {
            LASTO_WS_CASE(16, 0)
            LASTO_WS_CASE(32, 0)
            LASTO_WS_CASE(48, 0)
            LASTO_WS_CASE(64, 0)
            LASTO_WS_CASE(96, 0)
            LASTO_WS_CASE(128, 0)
            LASTO_WS_CASE(16, 1)
            LASTO_WS_CASE(32, 1)
            LASTO_WS_CASE(64, 1)
        }
#undef LASTO_WS_CASE
        return cudaGetLastError() == cudaSuccess ? LASTO_OK : LASTO_ERR_CUDA;
    }
#define LASTO_WG_CASE(C, Q)                                                                                           \
    case C + Q:                                                                                                       \
        if (cudaFuncSetAttribute(k_conv_wgrad_tc<C, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, wg_smem(C)) !=   \
            cudaSuccess)                                                                                              \
            return LASTO_ERR_CUDA;                                                                                    \
        k_conv_wgrad_tc<C, Q><<<grid, TC_M, wg_smem(C), s>>>(g, gd, cin, X, DY, dw, err);                             \
        break;
    switch (cout + (give_up ? 1 : 0)) {
        LASTO_WG_CASE(16, 0)
        LASTO_WG_CASE(32, 0)
        LASTO_WG_CASE(48, 0)
        LASTO_WG_CASE(64, 0)
        LASTO_WG_CASE(96, 0)
        LASTO_WG_CASE(128, 0)
        LASTO_WG_CASE(16, 1)
        LASTO_WG_CASE(32, 1)
        LASTO_WG_CASE(64, 1)
        default: return LASTO_ERR_INVALID_ARG;
    }
#undef LASTO_WG_CASE
    return cudaGetLastError() == cudaSuccess ? LASTO_OK : LASTO_ERR_CUDA;
}

}  // namespace lasto
