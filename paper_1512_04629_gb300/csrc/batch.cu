// batch.cu -- multi-right-hand-side (SpMM) V-cycle kernels and batched PCG.
//
// SpMM layout: the K right-hand sides of a row are contiguous (row-major
// n x K).  A group of G = K / W lanes owns a row, and lane t owns the W
// consecutive columns W t .. W t + W - 1, moved as one 16-byte vector (W = 4
// floats or 2 doubles).  Every lane of the group reads the row's (column,
// value) pairs itself -- the same address across the group, served as one
// broadcast -- kAhead entries at a time, their vector loads in flight
// together; each column sums its entries in row order.  The matrix is read
// once per block of K right-hand sides instead of K times.  A block takes a
// contiguous range of rows: what a row gathers of the grid lines beside its
// own is then still in L1 from the block's last steps, and L2 -- whose
// bandwidth bounds these kernels, a 7-point row at K = 32 gathers 7 x 128
// bytes -- serves it about once instead of per row (how long a range:
// spmm_grid).  Lognormal 112^3, K = 32, FP32, finest level: residual 165 ->
// 113 us (it no longer writes x = D^-1 b either), prolongation 124 -> 97,
// post-smoothing 170 -> 121 (it writes the correction in FP32, not widened).
// Forming r.z in the post-smoothing too was slower (340 us against 121 + 179):
// its registers leave half the warps.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "batch_ops.cuh"
#include "common.cuh"
#include "fp_convert.cuh"

namespace amg {
namespace bat {

namespace {

constexpr int kThreads = 256;

template <typename VT, typename XT> __device__ __forceinline__ XT cvt(VT v) { return (XT)v; }

template <> __device__ __forceinline__ float cvt<__nv_bfloat16, float>(__nv_bfloat16 v) { return __bfloat162float(v); }

// 16-byte vectors of a row block (the block's base is 16-byte aligned: K is a
// multiple of 8 and every n x K buffer starts on an allocation boundary)
__device__ __forceinline__ void vload(const float *p, float (&x)[4]) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
}
__device__ __forceinline__ void vload(const double *p, double (&x)[2]) {
    const double2 q = __ldg(reinterpret_cast<const double2 *>(p));
    x[0] = q.x; x[1] = q.y;
}
// for a buffer the same kernel writes (its own row only)
__device__ __forceinline__ void vload_rw(const float *p, float (&x)[4]) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
}
__device__ __forceinline__ void vload_rw(const double *p, double (&x)[2]) {
    const double2 q = *reinterpret_cast<const double2 *>(p);
    x[0] = q.x; x[1] = q.y;
}
__device__ __forceinline__ void vstore(float *p, const float (&x)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void vstore(double *p, const double (&x)[2]) {
    *reinterpret_cast<double2 *>(p) = make_double2(x[0], x[1]);
}

constexpr int kSpmmThreads = 512;  // largest block of an SpMM pass
constexpr int kAhead = 4;          // entries whose vector loads are in flight together
// resident blocks the passes are compiled for: FP32 three (42 registers) --
// with two its passes at 112^3, K = 32 take 8% longer, with four or with two
// entries ahead 4-9% -- and FP64, whose operands fill 64 registers, two
template <typename XT> constexpr int kSpmmBlocks = sizeof(XT) == 8 ? 2 : 3;

// entries e .. e + C - 1 of a row: their columns and values, then their
// vectors, are in flight together
template <int C, typename VT, typename XT, int K, bool SCALE, bool SUB>
__device__ __forceinline__ void entries(int32_t e, const int32_t *__restrict__ ci, const VT *__restrict__ v,
                                        const XT *__restrict__ src, const XT *__restrict__ dinv, int c0,
                                        XT (&acc)[16 / sizeof(XT)]) {
    constexpr int W = 16 / sizeof(XT);
    int32_t j[C];
    XT a[C], x[C][W], m[C];
#pragma unroll
    for (int q = 0; q < C; ++q) {
        j[q] = __ldg(ci + e + q);
        a[q] = cvt<VT, XT>(__ldg(v + e + q));
    }
#pragma unroll
    for (int q = 0; q < C; ++q) {
        vload(src + (int64_t)j[q] * K + c0, x[q]);
        if (SCALE) m[q] = __ldg(dinv + j[q]);
    }
#pragma unroll
    for (int q = 0; q < C; ++q) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const XT y = SCALE ? x[q][w] * m[q] : x[q][w];
            if (SUB) acc[w] -= a[q] * y;
            else acc[w] += a[q] * y;
        }
    }
}

// acc += sum over the row's entries, in entry order, of a_ij * src_j[c0 ..]
// (SCALE: times dinv_j, for x_j = dinv_j b_j that was never written); SUB:
// subtracted, for residuals whose accumulator starts at b.  kAhead entries
// at a time, then the rest.  In FP64 the rest must be branches: as plain
// conditions (entries<2>, entries<1>) the compiler predicates it, and a
// predicated-off FMA holds the FP64 pipe like a real one -- in A p over rows of
// five entries (4 + 1) the two absent ones took 501 us instead of 399 at 2D
// 2048^2, K = 8.  A switch with all of the rest in flight (SWITCH, A p) and
// loops of two and one (the FP64 cycle's passes, whose registers the switch
// spills) compile to branches: lognormal 160^3, K = 64, FP32 cycle 485 ms with
// loops in A p, 477 with the switch; 128^3, K = 32, FP64 250 with loops in the
// passes, 254 with the switch, 259 with conditions.  In FP32 conditions are
// the fastest form (lognormal 112^3, K = 32: by 0.8% of the solve).
template <typename VT, typename XT, int K, bool SCALE, bool SUB, bool SWITCH = false>
__device__ __forceinline__ void row_block_sum(int32_t p0, int32_t p1, const int32_t *__restrict__ ci,
                                              const VT *__restrict__ v, const XT *__restrict__ src,
                                              const XT *__restrict__ dinv, int c0, XT (&acc)[16 / sizeof(XT)]) {
    int32_t e = p0;
    for (; e + kAhead <= p1; e += kAhead) entries<kAhead, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc);
    if constexpr (SWITCH) {
        switch (p1 - e) {
            case 3: entries<3, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc); break;
            case 2: entries<2, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc); break;
            case 1: entries<1, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc); break;
            default: break;
        }
    } else if constexpr (sizeof(XT) == 8) {
#pragma unroll 1
        for (; e + 2 <= p1; e += 2) entries<2, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc);
#pragma unroll 1
        for (; e < p1; ++e) entries<1, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc);
    } else {
        if (e + 2 <= p1) {
            entries<2, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc);
            e += 2;
        }
        if (e < p1) entries<1, VT, XT, K, SCALE, SUB>(e, ci, v, src, dinv, c0, acc);
    }
}

// operands of an SpMM pass (unused ones null)
template <typename XT> struct SpmmArgs {
    const XT *B = nullptr;     // right-hand sides of this level
    const XT *X = nullptr;     // the gathered block
    const XT *dinv = nullptr;  // this level's inverse ell1 diagonal (restriction: the coarse level's)
    XT *O1 = nullptr, *O2 = nullptr;
};

// kResB: O1 = B - A (dinv .* B), the residual of a pre-smooth x = dinv .* B
//        that is not written (kProlB forms it again); kRes: O1 = B - A X
// kPost: O1 = X + dinv .* (B - A X)
// kRest: O1 = R X; kRestX: also O2 = dinv .* O1, the coarse pre-smooth
// kProl: O1 += P X; kProlB: O1 = dinv .* B + P X
enum Op { kResB, kRes, kPost, kRest, kRestX, kProl, kProlB };

template <typename VT, typename XT, int K, int OP>
__global__ void __launch_bounds__(kSpmmThreads, kSpmmBlocks<XT>)
spmm_kernel(int32_t n, int32_t chunk, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
            const VT *__restrict__ v, SpmmArgs<XT> g) {
    constexpr int W = 16 / sizeof(XT), G = K / W;
    constexpr bool kResid = OP == kResB || OP == kRes || OP == kPost;
    const int c0 = (int)(threadIdx.x % G) * W, step = blockDim.x / G;
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = min((int64_t)n, lo + chunk);
    int64_t i = lo + threadIdx.x / G;
    int32_t p0 = 0, p1 = 0;
    if (i < hi) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
    for (; i < hi; i += step) {
        const int32_t q0 = p0, q1 = p1;
        if (i + step < hi) { p0 = __ldg(rp + i + step); p1 = __ldg(rp + i + step + 1); }
        const int64_t base = i * K + c0;
        XT acc[W], o[W];
        if constexpr (kResid) vload(g.B + base, acc);
        else {
#pragma unroll
            for (int w = 0; w < W; ++w) acc[w] = XT(0);
        }
        if constexpr (OP == kProlB) vload(g.B + base, o);
        if constexpr (OP == kProl) vload_rw(g.O1 + base, o);
        if constexpr (OP == kPost) vload(g.X + base, o);
        XT d = XT(0);
        if constexpr (OP == kPost || OP == kRestX || OP == kProlB) d = __ldg(g.dinv + i);
        row_block_sum<VT, XT, K, OP == kResB, kResid>(q0, q1, ci, v, OP == kResB ? g.B : g.X, g.dinv, c0, acc);
        if constexpr (OP == kResB || OP == kRes || OP == kRest || OP == kRestX) {
            vstore(g.O1 + base, acc);
            if constexpr (OP == kRestX) {
#pragma unroll
                for (int w = 0; w < W; ++w) o[w] = acc[w] * d;
                vstore(g.O2 + base, o);
            }
        } else {
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if constexpr (OP == kProl) o[w] += acc[w];
                else if constexpr (OP == kProlB) o[w] = o[w] * d + acc[w];
                else o[w] += d * acc[w];
            }
            vstore(g.O1 + base, o);
        }
    }
}

// A block's threads and rows.  Blocks take ranges of about kSpmmSteps steps
// (64 KB of the gathered block), in as many even waves as that makes: blocks
// start in order, so the rows at work at one time are a front that moves
// through the matrix, and what a row gathers a grid plane away is in L2 from
// the front's last pass or about to serve its next.  With one range per
// resident block over the whole matrix that neighbour lies in another block's
// range, and above the L2's size it comes from HBM again; such a pass also
// holds the whole device for its time, and the short passes of other
// hierarchies wait.  Solves in ms, whole-matrix ranges -> these: lognormal,
// K = 64, 96^3 86.3 -> 83.0, 112^3 136.7 -> 137.1, 128^3 242 -> 228, 160^3
// 535 -> 485; K = 32, 112^3 73.0 -> 74.0, 128^3 124.3 -> 118.6, 160^3 270 ->
// 251; 2D 2048^2, K = 8 109.5 -> 104.7.  Ranges of 4 or 6 steps are within 1%
// of 8, of 16 and 32 up to 6% slower, of 1 (rows in launch order) 7-10%.
// Serving eight hierarchies, p50 / p99: 99 / 299 -> 88 / 235 ms.  Levels
// that fill the device less than once get smaller blocks, down to one warp's
// rows each.
constexpr int kSpmmSteps = 8;
struct SpmmGrid {
    int threads, blocks;
    int32_t chunk;
};
SpmmGrid spmm_grid(int64_t n, int G, int resident) {
    const int64_t sms = ::amg::resident_blocks(2048);
    int threads = kSpmmThreads;
    while (threads > 64 && div_up(n * G, threads) < sms * resident) threads >>= 1;
    const int64_t rows = threads / G;  // per step
    const int64_t want = (n + rows - 1) / rows;
    const int64_t cap = sms * resident * (kSpmmThreads / threads);
    const int64_t waves = std::max<int64_t>(1, (want + cap - 1) / cap / kSpmmSteps);
    const int64_t steps = (want + cap * waves - 1) / (cap * waves);
    SpmmGrid g;
    g.threads = threads;
    g.chunk = (int32_t)(steps * rows);
    g.blocks = (int)((n + g.chunk - 1) / g.chunk);
    return g;
}

template <typename VT, typename XT, int OP>
void dispatch(const CycMat<VT> &A, int K, const SpmmArgs<XT> &g, cudaStream_t s) {
    const int32_t n = A.nrows;
    if (n == 0) return;
    auto launch = [&](auto kc) {
        constexpr int KK = decltype(kc)::value;
        const SpmmGrid gr = spmm_grid(n, KK / (16 / (int)sizeof(XT)), kSpmmBlocks<XT>);
        spmm_kernel<VT, XT, KK, OP><<<gr.blocks, gr.threads, 0, s>>>(n, gr.chunk, A.rp, A.ci, A.v, g);
        ::amg::count_launch();
    };
    switch (K) {
        case 8: launch(std::integral_constant<int, 8>{}); break;
        case 16: launch(std::integral_constant<int, 16>{}); break;
        case 32: launch(std::integral_constant<int, 32>{}); break;
        case 64: launch(std::integral_constant<int, 64>{}); break;
        default: throw Error(AMG_ERR_INVALID, "batch width must be 8, 16, 32 or 64");
    }
    AMG_CHECK_LAUNCH();
}

// one block per row of the dense inverse: thread groups of K lanes take every
// (256 / K)-th entry, and the groups' sums are added in order (one thread per
// column walking the row alone took 10 us at 62 unknowns)
template <typename XT>
__global__ void __launch_bounds__(kThreads)
coarse_kernel(int32_t n, int K, const double *__restrict__ inv, const XT *__restrict__ B, XT *__restrict__ X) {
    __shared__ double sh[kThreads];
    const int32_t row = blockIdx.x;
    const int c = threadIdx.x % K, g = threadIdx.x / K, ng = kThreads / K;
    double s = 0.0;
#pragma unroll 4
    for (int32_t j = g; j < n; j += ng) s += inv[(size_t)row * n + j] * (double)B[(int64_t)j * K + c];
    sh[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x >= K) return;
    for (int q = 1; q < ng; ++q) s += sh[q * K + threadIdx.x];
    X[(int64_t)row * K + c] = (XT)s;
}

// ---------------------------------------------------------------------------
// per-column deterministic reductions.  Each block sums its threads' values of
// a column in thread order and stores one partial per column; a finisher
// kernel (one block per column) sums the partials in block order and updates
// that column's scalars.  No atomics, no fences.
enum ColFin { kColRz = 0, kColAp = 1, kColXr = 2, kColTt = 3 };

template <int NV, int FIN>
__global__ void __launch_bounds__(kThreads)
col_finish_kernel(int nblocks, const double *partials, ColScalars sc, int flexible) {
    const int c = blockIdx.x;
    __shared__ double sh[NV][kThreads / 32];
    double t[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        t[k] = 0.0;
        const double *p = partials + ((size_t)k * kMaxCols + c) * kBatchReduceBlocks;
        for (int b = threadIdx.x; b < nblocks; b += kThreads) t[k] += p[b];
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = t[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sh[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double out[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        out[k] = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) out[k] += sh[k][i];
    }
    if (FIN == kColRz) {
        if (sc.active[c]) {
            double rho_new = out[0];
            if (sc.start[c]) sc.beta[c] = 0.0;
            else sc.beta[c] = flexible ? (-sc.alpha[c] * out[NV - 1]) / sc.rho[c] : rho_new / sc.rho[c];
            if (NV > 1) sc.zq[c] = out[NV - 1];
            sc.rho[c] = rho_new;
            sc.start[c] = 0;
        }
    } else if (FIN == kColAp) {
        sc.pq[c] = out[0];
        sc.alpha[c] = (sc.active[c] && out[0] > 0.0) ? sc.rho[c] / out[0] : 0.0;
    } else if (FIN == kColXr) {
        sc.rr[c] = out[0];
    } else {
        sc.tt[c] = out[0];
    }
}

// Blocks of a reducing kernel that gives each row G lanes: one resident wave,
// at least four rows per lane group.  The wave is asked of the runtime: with
// eight blocks per SM assumed, r.z of FP32 cycles, whose 42 registers let five
// stay, ran in two waves, the second three fifths full (2D 2048^2, K = 8: 178
// us, 129 as one wave).
template <auto KERN> int reduce_grid(int32_t n, int G) {
    static std::atomic<int> per_sm{0};
    int b = per_sm.load(std::memory_order_relaxed);
    if (b == 0) {
        AMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, KERN, kThreads, 0));
        b = std::max(b, 1);
        per_sm.store(b, std::memory_order_relaxed);
    }
    const int64_t rows = kThreads / G;
    const int64_t want = ((n + rows - 1) / rows + 3) / 4;
    const int64_t cap = std::min<int64_t>(kBatchReduceBlocks, (int64_t)b * ::amg::resident_blocks(2048));
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
}

__device__ __forceinline__ void zload(const double *p, double (&z)[2]) { vload(p, z); }
__device__ __forceinline__ void zload(const float *p, double (&z)[2]) {
    const float2 q = __ldg(reinterpret_cast<const float2 *>(p));
    z[0] = widen(q.x);
    z[1] = widen(q.y);
}

// per-column sums of a block whose threads hold two adjacent columns each
// (lane t of a group of K / 2: columns 2 t, 2 t + 1), threads in order
template <int K, int NV>
__device__ __forceinline__ void pair_partials(const double (&part)[NV][2], double *partials) {
    constexpr int G = K / 2;
    __shared__ double sh[NV][2][kThreads];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        sh[k][0][threadIdx.x] = part[k][0];
        sh[k][1][threadIdx.x] = part[k][1];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NV * K; e += kThreads) {
        const int k = e / K, c = e % K;
        double sum = 0.0;
        for (int t = c / 2; t < kThreads; t += G) sum += sh[k][c & 1][t];
        partials[((size_t)k * kMaxCols + c) * kBatchReduceBlocks + blockIdx.x] = sum;
    }
}

// r.z and (NV = 2) z.q: two columns of a row per thread, rows grid-stride
template <int K, int NV, typename ZT>
__global__ void __launch_bounds__(kThreads)
rz_kernel(int32_t n, const double *__restrict__ R, const ZT *__restrict__ Z, const double *__restrict__ Q,
          double *partials) {
    constexpr int G = K / 2, RPB = kThreads / G;
    double part[NV][2] = {};
    const int c = (int)(threadIdx.x % G) * 2;
#pragma unroll 2
    for (int64_t i = (int64_t)blockIdx.x * RPB + threadIdx.x / G; i < n; i += (int64_t)gridDim.x * RPB) {
        const int64_t e = i * K + c;
        double z[2], r[2];
        zload(Z + e, z);
        vload(R + e, r);
        part[0][0] += r[0] * z[0];
        part[0][1] += r[1] * z[1];
        if constexpr (NV == 2) {
            double q[2];
            vload(Q + e, q);
            part[1][0] += q[0] * z[0];
            part[1][1] += q[1] * z[1];
        }
    }
    pair_partials<K, NV>(part, partials);
}

// P = Z + beta P on the active columns, two per thread
template <int K, typename ZT>
__global__ void __launch_bounds__(kThreads)
p_update_kernel(int64_t pairs, const ZT *__restrict__ Z, double *__restrict__ P, ColScalars sc) {
    const int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (e >= pairs) return;
    const int c = (int)(e % (K / 2)) * 2;
    const bool a0 = sc.active[c] != 0, a1 = sc.active[c + 1] != 0;
    if (!a0 && !a1) return;
    double z[2], p[2];
    zload(Z + 2 * e, z);
    vload_rw(P + 2 * e, p);
    if (a0) p[0] = z[0] + sc.beta[c] * p[0];
    if (a1) p[1] = z[1] + sc.beta[c + 1] * p[1];
    vstore(P + 2 * e, p);
}

// x = dinv .* R on an n x K block (the FP64 cycle's finest pre-smooth)
template <int K>
__global__ void __launch_bounds__(kThreads)
scale_kernel(int64_t pairs, const double *__restrict__ R, const double *__restrict__ dinv, double *__restrict__ X) {
    const int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (e >= pairs) return;
    const double d = __ldg(dinv + e / (K / 2));
    double r[2];
    vload(R + 2 * e, r);
    r[0] *= d;
    r[1] *= d;
    vstore(X + 2 * e, r);
}

// Q = A P (or T = B - A X when RESID) on the FP64 n x K blocks, with the
// per-column partials of p . Ap (or ||t||^2); the row-block mapping of
// spmm_kernel with W = 2, rows taken grid-stride
template <int K, bool RESID>
__global__ void __launch_bounds__(kThreads)
ap_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ v,
          const double *__restrict__ Pin, const double *__restrict__ Bin, double *__restrict__ Qout,
          double *partials) {
    constexpr int W = 2, G = K / W, RPB = kThreads / G;
    const int t = threadIdx.x % G, c0 = t * W;
    double part[W] = {0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * RPB + threadIdx.x / G; i < n; i += (int64_t)gridDim.x * RPB) {
        double acc[W] = {0.0, 0.0};
        const int64_t base = i * K + c0;
        if (RESID) vload(Bin + base, acc);
        row_block_sum<double, double, K, false, RESID, true>(__ldg(rp + i), __ldg(rp + i + 1), ci, v, Pin, nullptr, c0, acc);
        if (RESID) {
#pragma unroll
            for (int w = 0; w < W; ++w) part[w] += acc[w] * acc[w];
            vstore(Qout + base, acc);
        } else {
            double p[W];
            vload(Pin + base, p);
            vstore(Qout + base, acc);
#pragma unroll
            for (int w = 0; w < W; ++w) part[w] += p[w] * acc[w];
        }
    }
    // per-column partial: column W t + w sums slot w of the threads with lane t, in thread order
    __shared__ double sh[W][kThreads];
#pragma unroll
    for (int w = 0; w < W; ++w) sh[w][threadIdx.x] = part[w];
    __syncthreads();
    if (threadIdx.x < K) {
        const int col = threadIdx.x, tt = col / W, w = col % W;
        double sum = 0.0;
        for (int r = tt; r < kThreads; r += G) sum += sh[w][r];
        partials[(size_t)col * kBatchReduceBlocks + blockIdx.x] = sum;
    }
}

// two columns of a row per thread, rows grid-stride.  At 112^3, K = 32 it
// moves 2.34 GB in 433 us, 80% of the copy rate; streaming load and store
// policies change nothing
template <int K>
__global__ void __launch_bounds__(kThreads)
xr_kernel(int32_t n, const double *__restrict__ P, const double *__restrict__ Q, double *__restrict__ X,
          double *__restrict__ R, float *__restrict__ R32, ColScalars sc, double *partials) {
    constexpr int G = K / 2, RPB = kThreads / G;
    const int c = (int)(threadIdx.x % G) * 2;
    const double a0 = sc.active[c] ? sc.alpha[c] : 0.0, a1 = sc.active[c + 1] ? sc.alpha[c + 1] : 0.0;
    // tested as integers: a comparison of doubles would sit in the loop on the FP64 pipe
    const bool s0 = __double_as_longlong(a0) << 1 != 0, s1 = __double_as_longlong(a1) << 1 != 0;
    double part[1][2] = {};
#pragma unroll 2
    for (int64_t i = (int64_t)blockIdx.x * RPB + threadIdx.x / G; i < n; i += (int64_t)gridDim.x * RPB) {
        const int64_t e = i * K + c;
        double r[2];
        vload_rw(R + e, r);
        if (s0 || s1) {
            double x[2], p[2], q[2];
            vload_rw(X + e, x);
            vload(P + e, p);
            vload(Q + e, q);
            if (s0) {
                x[0] += a0 * p[0];
                r[0] -= a0 * q[0];
            }
            if (s1) {
                x[1] += a1 * p[1];
                r[1] -= a1 * q[1];
            }
            vstore(X + e, x);
            vstore(R + e, r);
        }
        // the next FP32 cycle's input, every column
        if (R32) *reinterpret_cast<float2 *>(R32 + e) = make_float2(narrow(r[0]), narrow(r[1]));
        part[0][0] += r[0] * r[0];
        part[0][1] += r[1] * r[1];
    }
    pair_partials<K, 1>(part, partials);
}

// a request's right-hand side into column c of B, R (and R32); X, P, Q zeroed
__global__ void __launch_bounds__(kThreads)
admit_kernel(int32_t n, int K, int c, const double *__restrict__ b, double *__restrict__ B, double *__restrict__ R,
             float *__restrict__ R32, double *__restrict__ X, double *__restrict__ P, double *__restrict__ Q) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const int64_t e = i * K + c;
    const double v = b[i];
    B[e] = v;
    R[e] = v;
    if (R32) R32[e] = (float)v;
    X[e] = 0.0;
    P[e] = 0.0;
    Q[e] = 0.0;
}

__global__ void gather_kernel(int32_t n, int K, int c, const double *M, double *v) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] = M[i * K + c];
}
__global__ void copy_masked_kernel(int64_t total, int K, const double *T, double *R, float *R32, const int *mask) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total || !mask[e % K]) return;
    R[e] = T[e];
    if (R32) R32[e] = (float)T[e];
}

template <typename XT> __global__ void to_cycle_kernel(const double *src, XT *dst, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (XT)src[i];
}
}  // namespace

int batch_width(int k) {
    if (k <= 8) return 8;
    if (k <= 16) return 16;
    if (k <= 32) return 32;
    if (k <= 64) return 64;
    throw Error(AMG_ERR_INVALID, "at most 64 right-hand sides per batch");
}

namespace {
// f(std::integral_constant<int, K>) for a compiled width
template <class F> void with_width(int K, F &&f) {
    switch (K) {
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 16: f(std::integral_constant<int, 16>{}); break;
        case 32: f(std::integral_constant<int, 32>{}); break;
        case 64: f(std::integral_constant<int, 64>{}); break;
        default: throw Error(AMG_ERR_INVALID, "batch width must be 8, 16, 32 or 64");
    }
    AMG_CHECK_LAUNCH();
}
}  // namespace

template <typename VT, typename XT>
void residual_of_scaled(const CycMat<VT> &A, int K, const XT *B, const XT *dinv, XT *R, cudaStream_t s) {
    SpmmArgs<XT> g;
    g.B = B; g.dinv = dinv; g.O1 = R;
    dispatch<VT, XT, kResB>(A, K, g, s);
}
template <typename VT, typename XT>
void residual_from_x(const CycMat<VT> &A, int K, const XT *B, const XT *X, XT *R, cudaStream_t s) {
    SpmmArgs<XT> g;
    g.B = B; g.X = X; g.O1 = R;
    dispatch<VT, XT, kRes>(A, K, g, s);
}
template <typename VT, typename XT>
void post_smooth(const CycMat<VT> &A, int K, const XT *X, const XT *B, const XT *dinv, XT *XO, cudaStream_t s) {
    SpmmArgs<XT> g;
    g.B = B; g.X = X; g.dinv = dinv; g.O1 = XO;
    dispatch<VT, XT, kPost>(A, K, g, s);
}
template <typename XT>
void restrict_to(const CycMat<XT> &R, int K, const XT *X, XT *BC, const XT *dinv_c, XT *XC, cudaStream_t s) {
    SpmmArgs<XT> g;
    g.X = X; g.O1 = BC; g.dinv = dinv_c; g.O2 = XC;
    if (XC) dispatch<XT, XT, kRestX>(R, K, g, s);
    else dispatch<XT, XT, kRest>(R, K, g, s);
}
template <typename XT>
void prolong_add(const CycMat<XT> &P, int K, const XT *XC, XT *X, const XT *B, const XT *dinv, cudaStream_t s) {
    SpmmArgs<XT> g;
    g.X = XC; g.O1 = X; g.B = B; g.dinv = dinv;
    if (B) dispatch<XT, XT, kProlB>(P, K, g, s);
    else dispatch<XT, XT, kProl>(P, K, g, s);
}
template <typename XT>
void coarse_solve(int32_t n, int K, const double *inv, const XT *B, XT *X, cudaStream_t s) {
    if (n == 0) return;
    { coarse_kernel<XT><<<n, kThreads, 0, s>>>(n, K, inv, B, X); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
void scale(int32_t n, int K, const double *R, const double *dinv, double *X, cudaStream_t s) {
    const int64_t pairs = (int64_t)n * K / 2;
    with_width(K, [&](auto kc) {
        scale_kernel<decltype(kc)::value><<<div_up(pairs, kThreads), kThreads, 0, s>>>(pairs, R, dinv, X);
        ::amg::count_launch();
    });
}

template <typename ZT>
void rz(int32_t n, int K, const double *R, const ZT *Z, const double *Q, ColScalars sc, double *partials,
        cudaStream_t s) {
    constexpr int NV = sizeof(ZT) == 8 ? 1 : 2;  // FP32 cycles: flexible CG, whose beta needs z.q
    int blocks = 0;
    with_width(K, [&](auto kc) {
        blocks = reduce_grid<rz_kernel<decltype(kc)::value, NV, ZT>>(n, K / 2);
        rz_kernel<decltype(kc)::value, NV, ZT><<<blocks, kThreads, 0, s>>>(n, R, Z, Q, partials);
        ::amg::count_launch();
    });
    { col_finish_kernel<NV, kColRz><<<K, kThreads, 0, s>>>(blocks, partials, sc, NV == 2); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

template <typename ZT> void p_update(int32_t n, int K, const ZT *Z, double *P, ColScalars sc, cudaStream_t s) {
    const int64_t pairs = (int64_t)n * K / 2;
    with_width(K, [&](auto kc) {
        p_update_kernel<decltype(kc)::value, ZT><<<div_up(pairs, kThreads), kThreads, 0, s>>>(pairs, Z, P, sc);
        ::amg::count_launch();
    });
}

template <int K, bool RESID>
static void launch_ap_k(const CycMat<double> &A, const double *P, const double *B, double *Q, ColScalars sc,
                        double *partials, cudaStream_t s) {
    const int blocks = reduce_grid<ap_kernel<K, RESID>>(A.nrows, K / 2);
    { ap_kernel<K, RESID><<<blocks, kThreads, 0, s>>>(A.nrows, A.rp, A.ci, A.v, P, B, Q, partials); ::amg::count_launch(); }
    if (RESID) { col_finish_kernel<1, kColTt><<<K, kThreads, 0, s>>>(blocks, partials, sc, 0); ::amg::count_launch(); }
    else { col_finish_kernel<1, kColAp><<<K, kThreads, 0, s>>>(blocks, partials, sc, 0); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

template <bool RESID>
static void launch_ap(const CycMat<double> &A, int K, const double *P, const double *B, double *Q, ColScalars sc,
                      double *partials, cudaStream_t s) {
    switch (K) {
        case 8: launch_ap_k<8, RESID>(A, P, B, Q, sc, partials, s); break;
        case 16: launch_ap_k<16, RESID>(A, P, B, Q, sc, partials, s); break;
        case 32: launch_ap_k<32, RESID>(A, P, B, Q, sc, partials, s); break;
        case 64: launch_ap_k<64, RESID>(A, P, B, Q, sc, partials, s); break;
        default: throw Error(AMG_ERR_INVALID, "batch width must be 8, 16, 32 or 64");
    }
}

void ap(const CycMat<double> &A, int K, const double *P, double *Q, ColScalars sc, double *partials,
        cudaStream_t s) {
    launch_ap<false>(A, K, P, nullptr, Q, sc, partials, s);
}

void residual(const CycMat<double> &A, int K, const double *B, const double *X, double *T, ColScalars sc,
              double *partials, cudaStream_t s) {
    launch_ap<true>(A, K, X, B, T, sc, partials, s);
}

void xr_update(int32_t n, int K, const double *P, const double *Q, double *X, double *R, float *R32, ColScalars sc,
               double *partials, cudaStream_t s) {
    int blocks = 0;
    with_width(K, [&](auto kc) {
        blocks = reduce_grid<xr_kernel<decltype(kc)::value>>(n, K / 2);
        xr_kernel<decltype(kc)::value><<<blocks, kThreads, 0, s>>>(n, P, Q, X, R, R32, sc, partials);
        ::amg::count_launch();
    });
    { col_finish_kernel<1, kColXr><<<K, kThreads, 0, s>>>(blocks, partials, sc, 0); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

void admit_column(int32_t n, int K, int c, const double *b, double *B, double *R, float *R32, double *X, double *P,
                  double *Q, cudaStream_t s) {
    { admit_kernel<<<div_up(n, kThreads), kThreads, 0, s>>>(n, K, c, b, B, R, R32, X, P, Q); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
void gather_column(int32_t n, int K, int c, const double *M, double *v, cudaStream_t s) {
    { gather_kernel<<<div_up(n, kThreads), kThreads, 0, s>>>(n, K, c, M, v); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
void copy_masked_columns(int32_t n, int K, const double *T, double *R, const int *mask, cudaStream_t s, float *R32) {
    int64_t total = (int64_t)n * K;
    { copy_masked_kernel<<<div_up(total, kThreads), kThreads, 0, s>>>(total, K, T, R, R32, mask); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

template <typename XT> void to_cycle(const double *src, XT *dst, int64_t n, cudaStream_t s) {
    { to_cycle_kernel<XT><<<div_up(n, kThreads), kThreads, 0, s>>>(src, dst, n); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
#define AMG_PINST(VT, XT)                                                                                          \
    template void residual_of_scaled<VT, XT>(const CycMat<VT> &, int, const XT *, const XT *, XT *, cudaStream_t); \
    template void post_smooth<VT, XT>(const CycMat<VT> &, int, const XT *, const XT *, const XT *, XT *, cudaStream_t);
AMG_PINST(float, float)
AMG_PINST(__nv_bfloat16, float)
#undef AMG_PINST
template void residual_from_x<double, double>(const CycMat<double> &, int, const double *, const double *, double *,
                                              cudaStream_t);
template void post_smooth<double, double>(const CycMat<double> &, int, const double *, const double *, const double *,
                                          double *, cudaStream_t);
#define AMG_SINST(XT)                                                                                               \
    template void restrict_to<XT>(const CycMat<XT> &, int, const XT *, XT *, const XT *, XT *, cudaStream_t);       \
    template void prolong_add<XT>(const CycMat<XT> &, int, const XT *, XT *, const XT *, const XT *, cudaStream_t); \
    template void coarse_solve<XT>(int32_t, int, const double *, const XT *, XT *, cudaStream_t);                   \
    template void rz<XT>(int32_t, int, const double *, const XT *, const double *, ColScalars, double *,            \
                         cudaStream_t);                                                                             \
    template void p_update<XT>(int32_t, int, const XT *, double *, ColScalars, cudaStream_t);
AMG_SINST(double)
AMG_SINST(float)
#undef AMG_SINST
template void to_cycle<float>(const double *, float *, int64_t, cudaStream_t);

}  // namespace bat
}  // namespace amg
