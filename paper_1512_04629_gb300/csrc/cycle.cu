// cycle.cu -- V-cycle and PCG kernels.
//
// Every kernel here is a streaming pass over a sparse matrix or a few
// vectors: HBM bandwidth and the FP64 pipe (one warp instruction in 16 clocks
// per SM) bound the large levels, a chain of dependent loads the small ones.
// Three SpMV layouts serve all of them:
//  * vector-CSR: a group of T lanes (T = 2..32) owns a row; each lane loads
//    16-byte vectors of values and column indices (2 FP64 / 4 FP32 / 8 BF16
//    entries) read through the non-coherent path, masks the entries outside
//    its row, gathers x, and the group reduces with xor shuffles;
//  * SELL-C (C = 32, 16, 8): C-row slices stored column-major, read by one
//    warp with T = 32 / C lanes per row -- lane l takes row l % C and every
//    T-th entry from l / C -- so each warp load is one contiguous
//    128/256-byte segment whatever C; a shorter C splits long rows over more
//    lanes (shorter dependent chains per thread) and pads less;
//  * row patterns (patterns.cu), for a finest operator of few distinct rows:
//    one byte a row, the rows themselves in shared memory.
// Reductions for PCG are deterministic: fixed grid, per-block partials,
// summed in block order by the last block to finish (small grids) or by a
// one-block finisher kernel.
#include <cuda_bf16.h>

#include <cstdlib>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "cycle_ops.cuh"
#include "fp_convert.cuh"
#include "pdl.cuh"

namespace amg {
namespace cyc {

namespace {

constexpr int kThreads = 256;


template <typename VT, typename XT> __device__ __forceinline__ XT cvt(VT v) { return (XT)v; }
template <> __device__ __forceinline__ float cvt<__nv_bfloat16, float>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}

// 16-byte vector loads of V consecutive entries
template <typename VT> struct Vec;
template <> struct Vec<double> {
    static constexpr int V = 2;
    __device__ __forceinline__ static void load(const double *v, const int32_t *c, int64_t q, double (&vv)[2], int32_t (&cc)[2]) {
        double2 a = __ldg(reinterpret_cast<const double2 *>(v + q));
        int2 b = __ldg(reinterpret_cast<const int2 *>(c + q));
        vv[0] = a.x; vv[1] = a.y; cc[0] = b.x; cc[1] = b.y;
    }
};
template <> struct Vec<float> {
    static constexpr int V = 4;
    __device__ __forceinline__ static void load(const float *v, const int32_t *c, int64_t q, float (&vv)[4], int32_t (&cc)[4]) {
        float4 a = __ldg(reinterpret_cast<const float4 *>(v + q));
        int4 b = __ldg(reinterpret_cast<const int4 *>(c + q));
        vv[0] = a.x; vv[1] = a.y; vv[2] = a.z; vv[3] = a.w;
        cc[0] = b.x; cc[1] = b.y; cc[2] = b.z; cc[3] = b.w;
    }
};
template <> struct Vec<__nv_bfloat16> {
    static constexpr int V = 8;
    __device__ __forceinline__ static void load(const __nv_bfloat16 *v, const int32_t *c, int64_t q,
                                                __nv_bfloat16 (&vv)[8], int32_t (&cc)[8]) {
        uint4 a = __ldg(reinterpret_cast<const uint4 *>(v + q));
        int4 b0 = __ldg(reinterpret_cast<const int4 *>(c + q));
        int4 b1 = __ldg(reinterpret_cast<const int4 *>(c + q + 4));
        const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&a);
#pragma unroll
        for (int u = 0; u < 8; ++u) vv[u] = h[u];
        cc[0] = b0.x; cc[1] = b0.y; cc[2] = b0.z; cc[3] = b0.w;
        cc[4] = b1.x; cc[5] = b1.y; cc[6] = b1.z; cc[7] = b1.w;
    }
};

// acc + a x, or acc - a x (SUB): one fused multiply-add either way.  The
// residuals b - sum a x start their accumulator at b, so the subtraction of
// the finished sum is not an operation of its own -- on this part an FP64
// warp instruction holds its pipe for 16 clocks, and a 7-entry row's residual
// is then 7 of them instead of 8.
template <bool SUB, typename XT> __device__ __forceinline__ XT mac(XT acc, XT a, XT x) {
    return SUB ? acc - a * x : acc + a * x;
}

// init + sum (SUB: init - sum) over one CSR row by a group of T lanes (all
// lanes get the result; init is the group's first lane's)
template <typename VT, typename XT, int T, bool SUB = false, class G>
__device__ __forceinline__ XT csr_row_sum(int32_t p0, int32_t p1, int t, const int32_t *__restrict__ ci,
                                          const VT *__restrict__ v, G gather, XT init = XT(0)) {
    constexpr int V = Vec<VT>::V;
    XT acc = t == 0 ? init : XT(0);
    for (int32_t q = (p0 & ~(V - 1)) + t * V; q < p1; q += T * V) {
        VT vv[V];
        int32_t cc[V];
        Vec<VT>::load(v, ci, q, vv, cc);
#pragma unroll
        for (int u = 0; u < V; ++u) {
            int32_t e = q + u;
            if (e >= p0 && e < p1) acc = mac<SUB>(acc, cvt<VT, XT>(vv[u]), gather(cc[u]));
        }
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, T);
    return acc;
}

// SELL column indices: int32 columns, or int16 offsets from the row (when
// every |column - row| of the operator fits; 2 bytes less per stored entry)
struct SellIdx {
    const int32_t *col;
    const int16_t *delta;
};
// a read-only load; CS: with the evict-first (streaming) policy, for
// operators much larger than L2 (the finest level's, always, and any whose
// stored entries pass kStreamBytes): read once per pass, they would only
// push the gathered vectors and the smaller levels out of L1 and L2
template <bool CS, typename T> __device__ __forceinline__ T ld_ro(const T *p) {
    if constexpr (CS && (std::is_same<T, double>::value || std::is_same<T, float>::value ||
                         std::is_same<T, int32_t>::value || std::is_same<T, int16_t>::value))
        return __ldcs(p);
    else
        return __ldg(p);
}
template <bool D16, bool CS = false>
__device__ __forceinline__ int32_t sell_col(const SellIdx &ix, int32_t p, int32_t row) {
    if constexpr (D16) return row + (int32_t)ld_ro<CS>(ix.delta + p);
    else return ld_ro<CS>(ix.col + p);
}

constexpr int kShortMax = 8;  // widest slice of the load-first path

// a slice of width W (W <= 8): every value and column load first, then every
// gather, then the products in k order -- short rows (interpolation P,
// coarse operators) otherwise pay a load -> gather round trip per entry
template <int W, typename VT, typename XT, bool D16, bool CS, bool SUB, class G>
__device__ __forceinline__ XT sell_short_sum(XT acc, int32_t off, int32_t row, const SellIdx &ix,
                                             const VT *__restrict__ sv, G gather) {
    VT v[W];
    int32_t c[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        v[k] = ld_ro<CS>(sv + off + k * 32);
        c[k] = sell_col<D16, CS>(ix, off + k * 32, row);
    }
    XT g[W];
#pragma unroll
    for (int k = 0; k < W; ++k) g[k] = gather(c[k]);
#pragma unroll
    for (int k = 0; k < W; ++k) acc = mac<SUB>(acc, cvt<VT, XT>(v[k]), g[k]);
    return acc;
}

// the same for a width known at run time (1..8; the same for the whole warp)
template <typename VT, typename XT, bool D16, bool CS, bool SUB, class G>
__device__ __forceinline__ XT sell_short_any(XT acc, int32_t w, int32_t off, int32_t row, const SellIdx &ix,
                                             const VT *__restrict__ sv, G gather) {
    switch (w) {
        case 1: return sell_short_sum<1, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 2: return sell_short_sum<2, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 3: return sell_short_sum<3, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 4: return sell_short_sum<4, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 5: return sell_short_sum<5, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 6: return sell_short_sum<6, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 7: return sell_short_sum<7, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        case 8: return sell_short_sum<8, VT, XT, D16, CS, SUB>(acc, off, row, ix, sv, gather);
        default: return acc;
    }
}

// init + sum (SUB: init - sum) over the row stored at SELL position pos
// (slice pos / 32, lane pos % 32), entries in k order whatever the path;
// SHORT: slices of width <= 8 take the load-everything-first path (the
// transfer operators P and R, whose rows are short; the relaxation kernels
// measured slower with it)
template <typename VT, typename XT, bool D16, bool SHORT, bool CS, bool SUB, class G>
__device__ __forceinline__ XT sell_row_sum(int32_t pos, int32_t row, const int32_t *__restrict__ soff,
                                           const int32_t *__restrict__ sw, const SellIdx &ix,
                                           const VT *__restrict__ sv, G gather, XT init = XT(0)) {
    int32_t s = pos >> 5, lane = pos & 31;
    int32_t off = __ldg(soff + s) + lane, w = __ldg(sw + s);
    if constexpr (SHORT) {  // w: uniform over the warp (one slice)
        if (w <= kShortMax) return sell_short_any<VT, XT, D16, CS, SUB>(init, w, off, row, ix, sv, gather);
    }
    XT acc = init;
#pragma unroll 4
    for (int32_t k = 0; k < w; ++k) {
        int32_t p = off + k * 32;
        acc = mac<SUB>(acc, cvt<VT, XT>(ld_ro<CS>(sv + p)), gather(sell_col<D16, CS>(ix, p, row)));
    }
    return acc;
}

// ---------------------------------------------------------------------------
// Operators stored by row patterns (patterns.cu): the table in shared memory,
// one lane per row.  What is left to stream is the vectors and one byte per
// row, so FP64 kernels run at the FP64 pipe and FP32 ones near the bandwidth
// of the vectors.  A block keeps its table over the rows it takes with the
// grid's stride, and reads the next row's pattern number while it works on
// this one.  Against SELL-32 with int16 offsets: 3D 7-point 128^3 in FP64,
// residual 35.7 -> 29 us (FP64 pipe: 23), post-smoothing with r.z 45.7 -> 38
// (30), A p 40.4 -> 32 (27); 27-point 192^3, FP32 residual 268 -> 70, FP64
// A p 391 -> 327 (304).  Six resident blocks per SM: with five the 27-point
// solve takes 25.2 ms instead of 23.6, with eight (32 registers) 23.8.
// ---------------------------------------------------------------------------
constexpr int kPatBlocks = 6;  // resident blocks per SM the kernels are compiled for

// The table as the kernels hold it.  FP32 keeps an entry's value and offset
// side by side, one 8-byte shared load per entry: two loads made the 27-point
// residual load/store-bound (192^3: 94 -> 72 us).  FP64 keeps two arrays:
// its kernels are bound by the FP64 pipe, and 16-byte entries cost them more
// bank conflicts than the second load does (128^3 solve 10.8 vs 10.5 ms).
template <typename VT> struct PatSmem {
    const VT *val;         // FP64
    const int32_t *delta;  // FP64
    const float2 *ent;     // FP32: value, offset bits
    const VT *dinv;
    const int32_t *len;
    int32_t width;
    __device__ __forceinline__ void entry(int32_t e, VT &a, int32_t &d) const {
        if constexpr (sizeof(VT) == 4) {
            const float2 q = ent[e];
            a = q.x;
            d = __float_as_int(q.y);
        } else {
            a = val[e];
            d = delta[e];
        }
    }
};

// copies the table and lets the next kernel launch; returns after this
// kernel's own predecessor has finished (the table does not depend on it)
template <typename VT> __device__ __forceinline__ PatSmem<VT> pat_begin(const PatView<VT> &pt) {
    extern __shared__ __align__(16) unsigned char pat_raw[];
    pdl_launch_next();
    const int32_t ne = pt.npat * pt.width;
    VT *val = reinterpret_cast<VT *>(pat_raw);
    float2 *ent = reinterpret_cast<float2 *>(pat_raw);
    VT *dinv = sizeof(VT) == 4 ? reinterpret_cast<VT *>(ent + ne) : val + ne;
    int32_t *len = reinterpret_cast<int32_t *>(dinv + pt.npat), *delta = len + pt.npat;
    for (int32_t e = threadIdx.x; e < ne; e += kThreads) {
        const VT a = __ldg(pt.val + e);
        const int32_t d = __ldg(pt.delta + e);
        if constexpr (sizeof(VT) == 4) {
            ent[e] = make_float2(a, __int_as_float(d));
        } else {
            val[e] = a;
            delta[e] = d;
        }
    }
    for (int32_t e = threadIdx.x; e < pt.npat; e += kThreads) {
        dinv[e] = __ldg(pt.dinv + e);
        len[e] = __ldg(pt.len + e);
    }
    __syncthreads();
    pdl_wait();
    return PatSmem<VT>{val, delta, ent, dinv, len, pt.width};
}

template <int W, bool SUB, typename XT>
__device__ __forceinline__ XT pat_chunk(XT acc, const PatSmem<XT> &t, int32_t e, const XT *xr) {
    XT g[W], a[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        int32_t d;
        t.entry(e + k, a[k], d);
        g[k] = ld_dyn(xr + d);
    }
#pragma unroll
    for (int k = 0; k < W; ++k) acc = mac<SUB>(acc, a[k], g[k]);
    return acc;
}

// acc +/- the row's sum, entries in order; the whole warp takes the longest of
// its rows (the shorter ones add 0 times their own diagonal's x)
template <bool SUB, typename XT>
__device__ __forceinline__ XT pat_row_sum(XT acc, const PatSmem<XT> &t, int32_t p, const XT *xr) {
    const int32_t w = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)t.len[p]);
    const int32_t e = p * t.width;
    int32_t k = 0;
    for (; k + 8 <= w; k += 8) acc = pat_chunk<8, SUB>(acc, t, e + k, xr);
    switch (w - k) {
        case 1: return pat_chunk<1, SUB>(acc, t, e + k, xr);
        case 2: return pat_chunk<2, SUB>(acc, t, e + k, xr);
        case 3: return pat_chunk<3, SUB>(acc, t, e + k, xr);
        case 4: return pat_chunk<4, SUB>(acc, t, e + k, xr);
        case 5: return pat_chunk<5, SUB>(acc, t, e + k, xr);
        case 6: return pat_chunk<6, SUB>(acc, t, e + k, xr);
        case 7: return pat_chunk<7, SUB>(acc, t, e + k, xr);
        default: return acc;
    }
}

// f(i, p, live) for every row i of the grid-strided loop, p its pattern; a
// warp's lanes past the last row repeat it with live = false
template <typename VT, class F> __device__ __forceinline__ void pat_rows(int32_t n, const PatView<VT> &pt, F f) {
    const uint32_t stride = gridDim.x * kThreads, last = (uint32_t)n - 1u;  // r + stride < 2^32
    const uint32_t lane = threadIdx.x & 31;
    uint32_t r = blockIdx.x * kThreads + threadIdx.x;
    int32_t p = __ldg(pt.pid + min(r, last));
    for (; r - lane <= last; r += stride) {
        const int32_t pc = p;
        p = __ldg(pt.pid + min(r + stride, last));
        f((int32_t)min(r, last), pc, r <= last);
    }
}

enum Op { kPost = 1, kSpmv = 2, kSpmvAdd = 3, kSpmvScale = 4, kResX = 5 };

// the operations that form b - A x: their row accumulators start at b
template <int OP> constexpr bool kIsResid = OP == kPost || OP == kResX;

// what an operation does with its row's sum s (b - A x for the residual forms)
template <typename XT, int OP>
__device__ __forceinline__ void row_store(int32_t i, XT s, const XT *__restrict__ dinv, const XT *__restrict__ x,
                                          XT *__restrict__ o1, XT *__restrict__ o2) {
    if (OP == kPost) {
        o1[i] = x[i] + dinv[i] * s;
    } else if (OP == kSpmv) {
        o1[i] = s;
    } else if (OP == kSpmvScale) {
        o1[i] = s;
        o2[i] = s * dinv[i];
    } else if (OP == kResX) {
        o2[i] = s;
    } else {
        o1[i] += s;
    }
}

// the row's own operands of an operation, loaded before its sum is known
template <typename XT> struct RowOwn {
    XT b, d, x, o;
};
// what the kernel before may have written
template <typename XT, int OP>
__device__ __forceinline__ void own_dynamic(RowOwn<XT> &w, int32_t i, const XT *b, const XT *x, const XT *o1) {
    if (kIsResid<OP>) w.b = ld_dyn(b + i);
    if (OP == kPost) w.x = ld_dyn(x + i);
    if (OP == kSpmvAdd) w.o = ld_dyn(o1 + i);
}
template <typename XT, int OP>
__device__ __forceinline__ void own_store(const RowOwn<XT> &w, int32_t i, XT s, XT *o1, XT *o2) {
    if (OP == kPost) {
        o1[i] = w.x + w.d * s;
    } else if (OP == kSpmv) {
        o1[i] = s;
    } else if (OP == kSpmvScale) {
        o1[i] = s;
        o2[i] = s * w.d;
    } else if (OP == kResX) {
        o2[i] = s;
    } else {
        o1[i] = w.o + s;
    }
}

// Grids of at most kPreBlocks blocks per SM -- the small levels, whose kernels
// are a chain of dependent loads and not work -- take a form that loads the
// operator before it waits for the kernel before: the row bounds, the first
// entries and the diagonal are then in registers when the vectors are ready,
// and the chain that is left is one gather.  Larger grids run in several
// waves, of which only the first could use it, and the registers would cost
// them resident warps.
constexpr int kPreBlocks = 4;
static bool preload_grid(int blocks) { return blocks <= ::amg::resident_blocks(2048) * kPreBlocks; }

template <typename VT, typename XT, int T, int OP, bool PRE>
__global__ void __launch_bounds__(kThreads)
csr_op_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const VT *__restrict__ v,
              const XT *b, const XT *dinv, const XT *x, XT *o1, XT *o2) {
    constexpr bool SUB = kIsResid<OP>;
    if constexpr (!PRE) pdl_begin();
    else pdl_launch_next();
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t i = (int32_t)(g / T);
    int t = (int)(g % T);
    int32_t p0 = 0, p1 = 0;
    if (i < n) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
    const bool own = i < n && t == 0;
    RowOwn<XT> w{};
    if constexpr (!PRE) {
        if (own && SUB) w.b = b[i];
        const XT s = csr_row_sum<VT, XT, T, SUB>(p0, p1, t, ci, v, [&](int32_t j) { return __ldg(x + j); }, w.b);
        if (!own) return;
        if (OP == kPost || OP == kSpmvScale) w.d = dinv[i];
        if (OP == kPost) w.x = x[i];
        if (OP == kSpmvAdd) w.o = o1[i];
        own_store<XT, OP>(w, i, s, o1, o2);
    } else {
        constexpr int V = Vec<VT>::V, NC = 2;  // chunks of the row held in registers
        VT vv[NC][V];
        int32_t cc[NC][V];
        int32_t q = (p0 & ~(V - 1)) + t * V;
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (q + c * T * V < p1) Vec<VT>::load(v, ci, q + c * T * V, vv[c], cc[c]);
        if (own && (OP == kPost || OP == kSpmvScale)) w.d = __ldg(dinv + i);
        pdl_wait();
        if (own) own_dynamic<XT, OP>(w, i, b, x, o1);
        XT xv[NC][V];
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const int32_t e = q + c * T * V + u;
                if (e >= p0 && e < p1) xv[c][u] = ld_dyn(x + cc[c][u]);
            }
        XT acc = own ? w.b : XT(0);
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const int32_t e = q + c * T * V + u;
                if (e >= p0 && e < p1) acc = mac<SUB>(acc, cvt<VT, XT>(vv[c][u]), xv[c][u]);
            }
        for (q += NC * T * V; q < p1; q += T * V) {
            Vec<VT>::load(v, ci, q, vv[0], cc[0]);
#pragma unroll
            for (int u = 0; u < V; ++u)
                if (q + u < p1) acc = mac<SUB>(acc, cvt<VT, XT>(vv[0][u]), ld_dyn(x + cc[0][u]));
        }
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, T);
        if (own) own_store<XT, OP>(w, i, acc, o1, o2);
    }
}

// One lane per row of a SELL-32 operator; SHORT: every slice fits the
// load-first path; CS: the operator's entries load with the evict-first
// policy (CycMat::stream)
template <typename VT, typename XT, int OP, bool D16, bool SHORT, bool CS>
__global__ void __launch_bounds__(kThreads)
sell_op_kernel(int32_t n, const int32_t *__restrict__ perm, const int32_t *__restrict__ soff, const int32_t *__restrict__ sw,
               SellIdx ix, const VT *__restrict__ sv, const XT *__restrict__ b,
               const XT *__restrict__ dinv, const XT *__restrict__ x, XT *__restrict__ o1, XT *__restrict__ o2) {
    pdl_begin();
    int32_t pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= n) return;
    const int32_t i = perm ? __ldg(perm + pos) : pos;
    // transfers (P, R: short rows, latency-bound): the row's own operand is
    // loaded before the row sum so its latency overlaps the gathers
    constexpr bool kTransfer = OP == kSpmvAdd || OP == kSpmvScale;
    XT own = XT(0);
    if (OP == kSpmvAdd) own = o1[i];
    if (OP == kSpmvScale) own = dinv[i];
    const XT init = kIsResid<OP> ? b[i] : XT(0);
    const XT s = sell_row_sum<VT, XT, D16, SHORT || kTransfer, CS, kIsResid<OP>>(pos, i, soff, sw, ix, sv, [&](int32_t j) { return __ldg(x + j); }, init);
    if (OP == kSpmvScale) {
        o1[i] = s;
        o2[i] = s * own;
    } else if (OP == kSpmvAdd) {
        o1[i] = own + s;
    } else {
        row_store<XT, OP>(i, s, dinv, x, o1, o2);
    }
}

template <typename XT, int OP>
__global__ void __launch_bounds__(kThreads, kPatBlocks)
pat_op_kernel(int32_t n, PatView<XT> pt, const XT *b, const XT *x, XT *o1, XT *o2) {
    const PatSmem<XT> t = pat_begin(pt);
    pat_rows(n, pt, [&](int32_t i, int32_t p, bool live) {
        const XT xi = OP == kPost ? ld_dyn(x + i) : XT(0);
        const XT s = pat_row_sum<kIsResid<OP>>(kIsResid<OP> ? ld_dyn(b + i) : XT(0), t, p, x + i);
        if (!live) return;
        if (OP == kPost) o1[i] = xi + t.dinv[p] * s;
        else if (OP == kSpmv) o1[i] = s;
        else o2[i] = s;
    });
}

// rows in rounds of one resident wave, the blocks spread evenly over them
static int pat_grid(int32_t n) {
    const int64_t need = div_up((int64_t)n, (int64_t)kThreads), res = ::amg::resident_blocks(2048) * (int64_t)kPatBlocks;
    return (int)div_up(need, div_up(need, res));
}

template <typename XT, int OP>
static void launch_pat_op(const CycMat<XT> &A, const XT *b, const XT *x, XT *o1, XT *o2, cudaStream_t s) {
    const size_t smem = pat_smem_bytes<XT>(A.pat.npat, A.pat.width);
    pdl_launch(pat_op_kernel<XT, OP>, pat_grid(A.nrows), kThreads, smem, s, A.nrows, A.pat, b, x, o1, o2);
    ::amg::count_launch();
    AMG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// Row-partitioned execution (amg_partition): before each product every block
// gathers its ghost values from the global vector -- the exchange that a
// distributed run performs by messages -- then the same CSR kernels run with
// a gather that reads owned columns from the block's slice of the vector and
// ghosts from its part of the ghost buffer.  The loops, grids and sums are the
// unpartitioned kernels', so the results are the same bits.
// ---------------------------------------------------------------------------
__global__ void part_exchange_kernel(int64_t nghost, const int32_t *__restrict__ gcol, const double *__restrict__ src,
                                     double *__restrict__ gbuf) {
    pdl_begin();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nghost) return;
    gbuf[k] = __ldg(src + __ldg(gcol + k));
}

// block of row i (rows past the end, which gather nothing, get block 0)
__device__ __forceinline__ int part_of(const PartView &pv, int32_t i) {
    int p = 0;
    while (p + 1 < pv.parts && __ldg(pv.row0 + p + 1) <= i) ++p;
    return p;
}

// where row i's gathers read: owned columns from src + col0[p], ghosts from
// gbuf + goff[p]
struct PartRow {
    const double *xl, *g;
    int32_t nloc;
    __device__ __forceinline__ double operator()(int32_t c) const { return c < nloc ? __ldg(xl + c) : __ldg(g + (c - nloc)); }
};
__device__ __forceinline__ PartRow part_row(const PartView &pv, int32_t i, int32_t n, const double *src) {
    const int p = i < n ? part_of(pv, i) : 0;
    const int32_t c0 = __ldg(pv.col0 + p);
    return PartRow{src + c0, pv.gbuf + __ldg(pv.goff + p), __ldg(pv.col0 + p + 1) - c0};
}

template <int T, int OP>
__global__ void __launch_bounds__(kThreads)
part_op_kernel(int32_t n, const int32_t *__restrict__ rp, PartView pv, const double *__restrict__ v,
               const double *__restrict__ b, const double *__restrict__ dinv, const double *__restrict__ x,
               double *__restrict__ o1, double *__restrict__ o2) {
    pdl_begin();
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t i = (int32_t)(g / T);
    int t = (int)(g % T);
    int32_t p0 = 0, p1 = 0;
    if (i < n) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
    const double init = kIsResid<OP> && i < n && t == 0 ? b[i] : 0.0;
    const double s = csr_row_sum<double, double, T, kIsResid<OP>>(p0, p1, t, pv.cext, v, part_row(pv, i, n, x), init);
    if (i >= n || t != 0) return;
    row_store<double, OP>(i, s, dinv, x, o1, o2);
}

// the exchange for an operator whose products gather src
void part_exchange(const PartView &pv, const double *src, cudaStream_t s) {
    if (pv.nghost == 0) return;
    { pdl_launch(part_exchange_kernel, (int)div_up(pv.nghost, (int64_t)kThreads), kThreads, 0, s, pv.nghost, pv.gcol, src, pv.gbuf); ::amg::count_launch(); }
}

template <int OP>
void part_op(const CycMat<double> &A, const double *b, const double *dinv, const double *x, double *o1, double *o2,
             cudaStream_t s) {
    const int32_t n = A.nrows;
    part_exchange(A.part, x, s);
    // one lane per row: the order of the unpartitioned one-lane kernels
    { pdl_launch(part_op_kernel<1, OP>, (int)div_up((int64_t)n, (int64_t)kThreads), kThreads, 0, s, n, A.rp, A.part, A.v, b, dinv, x, o1, o2); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

// SELL-C with C < 32: one warp per slice of C rows, T = 32 / C lanes per
// row.  Lane l holds row l % C and the entries k = l / C, l / C + T, ... (the
// slice width is a multiple of T); its part of the row is loaded U entries
// at a time -- all values and columns, then all gathers, then the products
// -- and the T parts are added by xor shuffles.  The row's sum therefore
// runs in another order than a sequential one (not bit-equal to CSR).
// CS: the operator's entries load with the evict-first policy.
template <typename VT, typename XT, int OP, bool D16, int C, bool CS, bool PRE>
__global__ void __launch_bounds__(kThreads)
sell_lanes_op_kernel(int32_t n, const int32_t *__restrict__ perm, const int32_t *__restrict__ soff,
                     const int32_t *__restrict__ sw, SellIdx ix, const VT *__restrict__ sv, const XT *b,
                     const XT *dinv, const XT *x, XT *o1, XT *o2) {
    if constexpr (!PRE) pdl_begin();
    else pdl_launch_next();
    constexpr int T = 32 / C, U = 4;
    const int32_t slice = (int32_t)(((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31, r = lane % C, t = lane / C;
    if (slice * C >= n) return;  // whole warp: slices are warp-uniform
    const int32_t pos = slice * C + r;
    const bool valid = pos < n;
    const int32_t i = valid ? (perm ? __ldg(perm + pos) : pos) : 0;
    const int32_t off = __ldg(soff + slice) + lane, w = __ldg(sw + slice);
    constexpr bool SUB = kIsResid<OP>;
    if constexpr (PRE) {  // see kPreBlocks: the lane's first H entries before the wait
        constexpr int H = 8;
        const int32_t nk = valid ? w / T : 0;
        const bool own = valid && t == 0;
        VT v[H];
        int32_t c[H];
#pragma unroll
        for (int k = 0; k < H; ++k)
            if (k < nk) {
                v[k] = ld_ro<CS>(sv + off + k * 32);
                c[k] = sell_col<D16, CS>(ix, off + k * 32, i);
            }
        RowOwn<XT> ro{};
        if (own && (OP == kPost || OP == kSpmvScale)) ro.d = __ldg(dinv + i);
        pdl_wait();
        if (own) own_dynamic<XT, OP>(ro, i, b, x, o1);
        XT acc = ro.b, xv[H];
#pragma unroll
        for (int k = 0; k < H; ++k)
            if (k < nk) xv[k] = ld_dyn(x + c[k]);
#pragma unroll
        for (int k = 0; k < H; ++k)
            if (k < nk) acc = mac<SUB>(acc, cvt<VT, XT>(v[k]), xv[k]);
        auto dyn = [&](int32_t j) { return ld_dyn(x + j); };
        int32_t k = H;
        for (; k + U <= nk; k += U) acc = sell_short_sum<U, VT, XT, D16, CS, SUB>(acc, off + k * 32, i, ix, sv, dyn);
        if (k < nk) acc = sell_short_any<VT, XT, D16, CS, SUB>(acc, nk - k, off + k * 32, i, ix, sv, dyn);
#pragma unroll
        for (int o = 16; o >= C; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (own) own_store<XT, OP>(ro, i, acc, o1, o2);
        return;
    }
    auto gather = [&](int32_t j) { return __ldg(x + j); };
    XT acc = XT(0);
    if (valid) {
        if (SUB && t == 0) acc = b[i];
        const int32_t nk = w / T;  // entries of this lane
        int32_t k = 0;
        if ((OP == kSpmvAdd || OP == kSpmvScale) && nk <= kShortMax) {
            // transfers: a lane's part of a row is short, so all of it loads
            // first (nk is the same for the whole warp), rather than one
            // load -> gather round trip per entry in the tail loop
            acc = sell_short_any<VT, XT, D16, CS, SUB>(acc, nk, off, i, ix, sv, gather);
            k = nk;
        }
        for (; k + U <= nk; k += U) acc = sell_short_sum<U, VT, XT, D16, CS, SUB>(acc, off + k * 32, i, ix, sv, gather);
        // the last nk - k < U entries, loaded together (a warp-uniform count)
        switch (nk - k) {
            case 1: acc = sell_short_sum<1, VT, XT, D16, CS, SUB>(acc, off + k * 32, i, ix, sv, gather); break;
            case 2: acc = sell_short_sum<2, VT, XT, D16, CS, SUB>(acc, off + k * 32, i, ix, sv, gather); break;
            case 3: acc = sell_short_sum<3, VT, XT, D16, CS, SUB>(acc, off + k * 32, i, ix, sv, gather); break;
            default: break;
        }
    }
#pragma unroll
    for (int o = 16; o >= C; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (!valid || t != 0) return;
    row_store<XT, OP>(i, acc, dinv, x, o1, o2);
}

template <typename VT, typename XT, int OP, int C>
void launch_sell_lanes(const CycMat<VT> &A, const XT *b, const XT *dinv, const XT *x, XT *o1, XT *o2,
                       cudaStream_t s) {
    const int32_t n = A.nrows;
    const SellIdx ix{A.sci, A.sd};
    const int64_t warps = div_up((int64_t)n, (int64_t)C);
    const int g = (int)div_up(warps * 32, (int64_t)kThreads);
    auto launch = [&](auto cs, auto pre) {
        constexpr bool CS = decltype(cs)::value, PRE = decltype(pre)::value;
        if (A.sd)
            { pdl_launch(sell_lanes_op_kernel<VT, XT, OP, true, C, CS, PRE>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
        else
            { pdl_launch(sell_lanes_op_kernel<VT, XT, OP, false, C, CS, PRE>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
    };
    if (preload_grid(g)) {
        launch(std::false_type(), std::true_type());
        return;
    }
    if constexpr (std::is_same<VT, double>::value && std::is_same<XT, double>::value) {
        if (A.stream) launch(std::true_type(), std::false_type());
        else launch(std::false_type(), std::false_type());
    } else {
        launch(std::false_type(), std::false_type());
    }
}

template <typename VT, typename XT, int OP>
void dispatch_op(const CycMat<VT> &A, const XT *b, const XT *dinv, const XT *x, XT *o1, XT *o2, cudaStream_t s) {
    int32_t n = A.nrows;
    if (n == 0) return;
    if constexpr (std::is_same<VT, double>::value && std::is_same<XT, double>::value) {
        if (A.part.parts) {
            part_op<OP>(A, b, dinv, x, o1, o2, s);
            return;
        }
    }
    if constexpr (std::is_same<VT, XT>::value && (kIsResid<OP> || OP == kSpmv)) {
        if (A.pat.pid) {
            launch_pat_op<XT, OP>(A, b, x, o1, o2, s);
            return;
        }
    }
    if ((A.variant == AMG_SPMV_SELL16 || A.variant == AMG_SPMV_SELL8) && A.sv && A.sell_c == sell_height(A.variant)) {
        if (A.sell_c == 16) launch_sell_lanes<VT, XT, OP, 16>(A, b, dinv, x, o1, o2, s);
        else launch_sell_lanes<VT, XT, OP, 8>(A, b, dinv, x, o1, o2, s);
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.variant == AMG_SPMV_SELL32 && A.sv && A.sell_c == 32) {
        const SellIdx ix{A.sci, A.sd};
        // the load-first path for operators whose rows all fit it (measured:
        // faster at level 0, slower on the longer, irregular coarse rows)
        const bool sh = A.max_row > 0 && A.max_row <= kShortMax;
        const int g = div_up(n, kThreads);
        auto launch = [&](auto cs) {
            constexpr bool CS = decltype(cs)::value;
            if (A.sd && sh)
                { pdl_launch(sell_op_kernel<VT, XT, OP, true, true, CS>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
            else if (A.sd)
                { pdl_launch(sell_op_kernel<VT, XT, OP, true, false, CS>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
            else if (sh)
                { pdl_launch(sell_op_kernel<VT, XT, OP, false, true, CS>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
            else
                { pdl_launch(sell_op_kernel<VT, XT, OP, false, false, CS>, g, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, b, dinv, x, o1, o2); ::amg::count_launch(); }
        };
        // the streaming loads only in FP64 (the reduced-precision copies are half the size or less)
        if constexpr (std::is_same<VT, double>::value && std::is_same<XT, double>::value) {
            if (A.stream) launch(std::true_type());
            else launch(std::false_type());
        } else {
            launch(std::false_type());
        }
    } else {
        int T = threads_per_row(A.variant);
        int blocks = div_up((int64_t)n * T, kThreads);
        auto launch = [&](auto tc) {
            constexpr int L = decltype(tc)::value;
            if (preload_grid(blocks)) pdl_launch(csr_op_kernel<VT, XT, L, OP, true>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, b, dinv, x, o1, o2);
            else pdl_launch(csr_op_kernel<VT, XT, L, OP, false>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, b, dinv, x, o1, o2);
            ::amg::count_launch();
        };
        switch (T) {
            case 1: launch(std::integral_constant<int, 1>{}); break;
            case 2: launch(std::integral_constant<int, 2>{}); break;
            case 4: launch(std::integral_constant<int, 4>{}); break;
            case 8: launch(std::integral_constant<int, 8>{}); break;
            case 16: launch(std::integral_constant<int, 16>{}); break;
            default: launch(std::integral_constant<int, 32>{}); break;
        }
    }
    AMG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// deterministic block reduction with last-block finish
// ---------------------------------------------------------------------------
enum Fin { kFinAp = 0, kFinXr = 1, kFinRz = 2, kFinTt = 3 };

constexpr int kFinThreads = 1024;

// what the last step of a reduction needs besides the sums: the WHILE
// condition of the captured loop for the x, r update, and whether the reducing
// kernel finishes itself
struct FinCtl {
    cudaGraphConditionalHandle handle{};
    int use_handle = 0;
    int fused = 0;
};

// finish of r.z / z.q: beta and rho (start: beta = 0)
__device__ __forceinline__ void finish_rz(PcgScalars *sc, double rz, double zq) {
    if (!sc->start) {
        sc->zq = zq;
        sc->beta = sc->flexible ? (-sc->alpha * zq) / sc->rho : rz / sc->rho;
    } else {
        sc->beta = 0.0;
    }
    sc->rho = rz;
    sc->start = 0;
}

// the CG scalars from the finished sums (one thread)
template <int NV, int FIN>
__device__ __forceinline__ void finish_scalars(const double (&t)[NV], PcgScalars *sc, const FinCtl &ctl) {
    if (FIN == kFinAp) {
        sc->pq = t[0];
        bool ok = t[0] > 0.0 && sc->rho > 0.0;
        if (!ok) sc->breakdown = 1;
        sc->alpha = ok ? sc->rho / t[0] : 0.0;
    } else if (FIN == kFinXr) {
        sc->rr = t[0];
        int its = sc->its + 1;
        sc->its = its;
        if (sc->divf > 0.0 && !sc->breakdown) {
            // the window test, in the oracle's form: norms, not squares
            const double rn = sqrt(t[0]);
            const bool end = its % sc->kwin == 0;
            if (!isfinite(rn) || (end && rn > sc->divf * sc->rn_ws)) sc->diverged = 1;
            else if (end) sc->rn_ws = rn;
        }
        if (ctl.use_handle) {
            bool go = t[0] > sc->thresh2 && its < sc->max_its && !sc->breakdown && !sc->diverged && isfinite(t[0]);
            cudaGraphSetConditional(ctl.handle, go ? 1u : 0u);
        }
    } else if (FIN == kFinRz) {
        finish_rz(sc, t[0], NV > 1 ? t[NV - 1] : 0.0);
    } else {
        sc->tt = t[0];
    }
}

// Reductions without a block-wide barrier at the end: every thread parks its
// values in shared memory; the last warp of the block to arrive (a shared
// arrival counter, zeroed when the kernel starts) adds them, lane l the
// values l, l + 32, ... in warp order and then the 32 sums by shuffles, and
// stores the block partial.  Warps that finish early leave at once instead of
// waiting for the block's slowest gathers.  A shuffle tree in every warp
// would issue 40 FP64 warp instructions a block where this issues 12; with
// eight resident blocks per SM, all ending together, that is 2 us of the FP64
// pipe at the end of each reducing kernel.
//
// The block partials are summed in a fixed order -- no atomics on floating-
// point values, a deterministic result -- by the last block to finish on
// grids of at most kFuseBlocks blocks (one warp, a few partials a lane; the
// order does not depend on which block it is), and by a one-block finisher
// kernel launched next on larger ones: there the single warp's rounds of
// loads and the fence of every block cost what the launch saves.
__device__ __forceinline__ unsigned *arrival_counter() {
    __shared__ unsigned c;
    return &c;
}

// every kernel that calls block_partials calls this first (all threads)
__device__ __forceinline__ void block_partials_begin() {
    if (threadIdx.x == 0) *arrival_counter() = 0u;
    __syncthreads();
}

template <int NV, int FIN>
__device__ __forceinline__ void block_partials(double (&v)[NV], Reduce red, PcgScalars *sc, const FinCtl &ctl) {
    __shared__ double sh[NV][kThreads];
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] = v[k];
    __threadfence_block();
    __syncwarp();
    unsigned ticket = 0;
    if (lane == 0) ticket = atomicAdd(arrival_counter(), 1u);
    if (__shfl_sync(0xffffffffu, ticket, 0) != kThreads / 32 - 1) return;
    __threadfence_block();
    double t[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        t[k] = ((volatile double *)sh[k])[lane];
#pragma unroll
        for (int w = 1; w < kThreads / 32; ++w) t[k] += ((volatile double *)sh[k])[lane + 32 * w];
        for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
        if (lane == 0) red.partials[k * kMaxReduceBlocks + blockIdx.x] = t[k];
    }
    if (!ctl.fused) return;
    if (gridDim.x > 1) {
        if (lane == 0) {
            __threadfence();
            ticket = atomicAdd(red.counter, 1u);
        }
        if (__shfl_sync(0xffffffffu, ticket, 0) != gridDim.x - 1) return;
        __threadfence();
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            t[k] = 0.0;
#pragma unroll 8
            for (unsigned b = lane; b < gridDim.x; b += 32) t[k] += __ldcg(red.partials + k * kMaxReduceBlocks + b);
            for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
        }
        if (lane == 0) *red.counter = 0u;
    }
    if (lane == 0) finish_scalars<NV, FIN>(t, sc, ctl);
}

template <int NV, int FIN>
__global__ void __launch_bounds__(kFinThreads)
finish_kernel(int nblocks, Reduce red, PcgScalars *sc, FinCtl ctl) {
    pdl_begin();
    __shared__ double sh[NV][kFinThreads / 32];
    double t[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) t[k] = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x; b < nblocks; b += kFinThreads) {
#pragma unroll
        for (int k = 0; k < NV; ++k) t[k] += red.partials[k * kMaxReduceBlocks + b];
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = t[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sh[k][w] = x;
    }
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = sh[k][lane];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        t[k] = x;
    }
    if (lane == 0) finish_scalars<NV, FIN>(t, sc, ctl);
}

// 16 blocks (64 x 64): the solve 974 -> 948 us with its three reductions a step
// finishing themselves; 400 to 600 blocks measure the same either way, and at
// 900 to 1200 (all of 101^3 and 128^3) the finisher kernel is 1-5% of the
// solve faster.
constexpr int kFuseBlocks = 128;

// how a reducing kernel of `blocks` blocks finishes
FinCtl fin_ctl(int blocks, cudaGraphConditionalHandle handle = cudaGraphConditionalHandle{}, bool use_handle = false) {
    FinCtl c;
    c.handle = handle;
    c.use_handle = use_handle ? 1 : 0;
    c.fused = blocks <= kFuseBlocks;
    return c;
}

// after the reducing kernel: the finisher where it does not finish itself
template <int NV, int FIN>
void launch_finish(int nblocks, Reduce red, PcgScalars *sc, cudaStream_t s, const FinCtl &ctl) {
    if (ctl.fused) return;
    { pdl_launch(finish_kernel<NV, FIN>, 1, kFinThreads, 0, s, nblocks, red, sc, ctl); ::amg::count_launch(); }
}

// Grid of a reducing kernel: at most one resident wave, so every thread
// loops over several rows and the block's reduction (FP64 adds, the scarce
// pipe on this part) runs once per thread, not once per row.
int reduce_blocks(int64_t threads_needed) {
    int64_t b = (threads_needed + kThreads - 1) / kThreads;
    int64_t cap = ::amg::resident_blocks(kThreads);
    if (b > cap) b = cap;
    if (b > kMaxReduceBlocks) b = kMaxReduceBlocks;
    if (b < 1) b = 1;
    return (int)b;
}

// ---------------------------------------------------------------------------
// PCG kernels (FP64)
// ---------------------------------------------------------------------------
template <typename ZT>
__global__ void p_update_kernel(int32_t n, const ZT *__restrict__ z, double *__restrict__ p, const PcgScalars *sc) {
    pdl_begin();
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    p[i] = widen(z[i]) + sc->beta * p[i];
}

// q = A p (SELL-32, one thread per row) and p . q; each warp walks slices
// with a stride of the grid's warp count.  RESID: q = b - A p and q . q (the
// true residual of p = x)
template <bool D16, bool SHORT, bool RESID>
__global__ void __launch_bounds__(kThreads)
ap_sell_kernel(int32_t n, const int32_t *__restrict__ perm, const int32_t *__restrict__ soff, const int32_t *__restrict__ sw,
               SellIdx ix, const double *__restrict__ sv, const double *__restrict__ p, const double *__restrict__ b,
               double *__restrict__ q, PcgScalars *sc, Reduce red, FinCtl ctl) {
    pdl_begin();
    block_partials_begin();
    double part[1] = {0.0};
    const int lane = threadIdx.x & 31;
    const int32_t nsl = (n + 31) >> 5, nwarps = (int32_t)((gridDim.x * kThreads) >> 5);
    for (int32_t sl = (int32_t)((blockIdx.x * kThreads + threadIdx.x) >> 5); sl < nsl; sl += nwarps) {
        const int32_t pos = sl * 32 + lane;
        if (pos >= n) continue;
        const int32_t i = perm ? __ldg(perm + pos) : pos;
        const double s = sell_row_sum<double, double, D16, SHORT, true, RESID>(pos, i, soff, sw, ix, sv, [&](int32_t j) { return __ldg(p + j); }, RESID ? b[i] : 0.0);
        if (RESID) {
            q[i] = s;
            part[0] += s * s;
        } else {
            q[i] = s;
            part[0] += p[i] * s;
        }
    }
    block_partials<1, RESID ? kFinTt : kFinAp>(part, red, sc, ctl);
}

// the same with the operator stored by row patterns
template <bool RESID>
__global__ void __launch_bounds__(kThreads, kPatBlocks)
ap_pat_kernel(int32_t n, PatView<double> pt, const double *p, const double *b, double *q, PcgScalars *sc, Reduce red,
              FinCtl ctl) {
    block_partials_begin();
    const PatSmem<double> t = pat_begin(pt);
    double part[1] = {0.0};
    pat_rows(n, pt, [&](int32_t i, int32_t pat, bool live) {
        const double pi = RESID ? 0.0 : ld_dyn(p + i);
        const double s = pat_row_sum<RESID>(RESID ? ld_dyn(b + i) : 0.0, t, pat, p + i);
        if (!live) return;
        q[i] = s;
        part[0] += RESID ? s * s : pi * s;
    });
    block_partials<1, RESID ? kFinTt : kFinAp>(part, red, sc, ctl);
}

// q = A p (vector-CSR, T lanes per row) and p . q
template <int T, bool PART = false>
__global__ void __launch_bounds__(kThreads)
ap_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ v,
          const double *__restrict__ p, double *__restrict__ q, PcgScalars *sc, Reduce red, FinCtl ctl,
          PartView pv = PartView()) {
    pdl_begin();
    block_partials_begin();
    double part[1] = {0.0};
    int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < (int64_t)((n + (kThreads / T) - 1) / (kThreads / T)) * (kThreads / T) * T; g += stride) {
        int32_t i = (int32_t)(g / T);
        int t = (int)(g % T);
        int32_t p0 = 0, p1 = 0;
        if (i < n) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
        double s;
        if constexpr (PART) {  // ci: block-local columns
            s = csr_row_sum<double, double, T>(p0, p1, t, ci, v, part_row(pv, i, n, p));
        } else {
            s = csr_row_sum<double, double, T>(p0, p1, t, ci, v, [&](int32_t j) { return __ldg(p + j); });
        }
        if (i < n && t == 0) {
            q[i] = s;
            part[0] += p[i] * s;
        }
    }
    block_partials<1, kFinAp>(part, red, sc, ctl);
}

__global__ void __launch_bounds__(kThreads)
xr_update_kernel(int32_t n, const double *__restrict__ p, const double *__restrict__ q, double *__restrict__ x,
                 double *__restrict__ r, PcgScalars *sc, Reduce red, CycleInput next, double *__restrict__ xs, FinCtl ctl) {
    pdl_begin();
    block_partials_begin();
    const double alpha = sc->alpha;
    const bool step = alpha != 0.0;  // 0: breakdown -- x and r stay as they are
    // this step starts a divergence-test window: keep x as it was
    const bool ckpt = xs != nullptr && sc->divf > 0.0 && sc->its % sc->kwin == 0;
    double part[1] = {0.0};
    for (int32_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
        double ri = r[i];
        if (ckpt) xs[i] = x[i];
        if (step) {
            x[i] += alpha * p[i];
            ri -= alpha * q[i];
            r[i] = ri;
        }
        // the next cycle's input and its level-0 pre-smooth from zero
        if (next.x64) {
            next.x64[i] = ri * __ldg(next.dinv64 + i);
        } else if (next.x32) {
            const float r32 = narrow(ri);
            next.r32[i] = r32;
            next.x32[i] = r32 * __ldg(next.dinv32 + i);
        }
        part[0] += ri * ri;
    }
    block_partials<1, kFinXr>(part, red, sc, ctl);
}

__global__ void __launch_bounds__(kThreads)
rz_kernel(int32_t n, const double *__restrict__ r, const double *__restrict__ z, const double *__restrict__ q,
          PcgScalars *sc, Reduce red, FinCtl ctl) {
    pdl_begin();
    block_partials_begin();
    int first = sc->start;
    double part[2] = {0.0, 0.0};
    for (int32_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
        double zi = z[i];
        part[0] += r[i] * zi;
        if (!first) part[1] += zi * q[i];
    }
    block_partials<2, kFinRz>(part, red, sc, ctl);
}

template <int T, bool PART = false>
__global__ void __launch_bounds__(kThreads)
resid_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ v,
             const double *__restrict__ b, const double *__restrict__ x, double *__restrict__ t_out,
             PcgScalars *sc, Reduce red, FinCtl ctl, PartView pv = PartView()) {
    pdl_begin();
    block_partials_begin();
    double part[1] = {0.0};
    int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < (int64_t)((n + (kThreads / T) - 1) / (kThreads / T)) * (kThreads / T) * T; g += stride) {
        int32_t i = (int32_t)(g / T);
        int t = (int)(g % T);
        int32_t p0 = 0, p1 = 0;
        if (i < n) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
        const double init = i < n && t == 0 ? b[i] : 0.0;
        double e;
        if constexpr (PART) e = csr_row_sum<double, double, T, true>(p0, p1, t, ci, v, part_row(pv, i, n, x), init);
        else e = csr_row_sum<double, double, T, true>(p0, p1, t, ci, v, [&](int32_t j) { return __ldg(x + j); }, init);
        if (i < n && t == 0) {
            t_out[i] = e;
            part[0] += e * e;
        }
    }
    block_partials<1, kFinTt>(part, red, sc, ctl);
}

// level-0 post-smoothing z = x + d (b - A x) with r.z (r = b) and, for
// flexible CG only (ZQ), z.q -- plain CG's beta needs no z.q, so the FP64
// cycle reads no q and issues one FMA less per row
template <int T, bool ZQ, bool PART = false>
__global__ void __launch_bounds__(kThreads)
post_rz_csr_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ v,
                   const double *__restrict__ x, const double *__restrict__ b, const double *__restrict__ dinv,
                   double *__restrict__ z, const double *__restrict__ q, PcgScalars *sc, Reduce red, FinCtl ctl,
                   PartView pv = PartView()) {
    pdl_begin();
    block_partials_begin();
    double part[ZQ ? 2 : 1];
#pragma unroll
    for (int k = 0; k < (ZQ ? 2 : 1); ++k) part[k] = 0.0;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    const int64_t gend = (int64_t)((n + (kThreads / T) - 1) / (kThreads / T)) * (kThreads / T) * T;
    for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < gend; g += stride) {
        const int32_t i = (int32_t)(g / T);
        const int t = (int)(g % T);
        int32_t p0 = 0, p1 = 0;
        if (i < n) { p0 = __ldg(rp + i); p1 = __ldg(rp + i + 1); }
        const double bi = i < n && t == 0 ? b[i] : 0.0;
        double e;
        if constexpr (PART) e = csr_row_sum<double, double, T, true>(p0, p1, t, ci, v, part_row(pv, i, n, x), bi);
        else e = csr_row_sum<double, double, T, true>(p0, p1, t, ci, v, [&](int32_t j) { return __ldg(x + j); }, bi);
        if (i < n && t == 0) {
            const double zi = x[i] + dinv[i] * e;
            z[i] = zi;
            part[0] += bi * zi;
            if (ZQ) part[ZQ ? 1 : 0] += zi * q[i];
        }
    }
    block_partials<ZQ ? 2 : 1, kFinRz>(part, red, sc, ctl);
}

template <bool D16, bool ZQ>
__global__ void __launch_bounds__(kThreads)
post_rz_sell_kernel(int32_t n, const int32_t *__restrict__ perm, const int32_t *__restrict__ soff,
                    const int32_t *__restrict__ sw, SellIdx ix, const double *__restrict__ sv,
                    const double *__restrict__ x, const double *__restrict__ b, const double *__restrict__ dinv,
                    double *__restrict__ z, const double *__restrict__ q, PcgScalars *sc, Reduce red, FinCtl ctl) {
    pdl_begin();
    block_partials_begin();
    double part[ZQ ? 2 : 1];
#pragma unroll
    for (int k = 0; k < (ZQ ? 2 : 1); ++k) part[k] = 0.0;
    const int lane = threadIdx.x & 31;
    const int32_t nsl = (n + 31) >> 5, nwarps = (int32_t)((gridDim.x * kThreads) >> 5);
    for (int32_t sl = (int32_t)((blockIdx.x * kThreads + threadIdx.x) >> 5); sl < nsl; sl += nwarps) {
        const int32_t pos = sl * 32 + lane;
        if (pos >= n) continue;
        const int32_t i = perm ? __ldg(perm + pos) : pos;
        const double bi = b[i];
        const double e = sell_row_sum<double, double, D16, false, true, true>(pos, i, soff, sw, ix, sv, [&](int32_t j) { return __ldg(x + j); }, bi);
        const double zi = x[i] + dinv[i] * e;
        z[i] = zi;
        part[0] += bi * zi;
        if (ZQ) part[ZQ ? 1 : 0] += zi * q[i];
    }
    block_partials<ZQ ? 2 : 1, kFinRz>(part, red, sc, ctl);
}

template <bool ZQ>
__global__ void __launch_bounds__(kThreads, kPatBlocks)
post_rz_pat_kernel(int32_t n, PatView<double> pt, const double *x, const double *b, double *z, const double *q,
                   PcgScalars *sc, Reduce red, FinCtl ctl) {
    block_partials_begin();
    const PatSmem<double> t = pat_begin(pt);
    double part[ZQ ? 2 : 1];
#pragma unroll
    for (int k = 0; k < (ZQ ? 2 : 1); ++k) part[k] = 0.0;
    pat_rows(n, pt, [&](int32_t i, int32_t p, bool live) {
        const double bi = ld_dyn(b + i), xi = ld_dyn(x + i);
        const double e = pat_row_sum<true>(bi, t, p, x + i);
        if (!live) return;
        const double zi = xi + t.dinv[p] * e;
        z[i] = zi;
        part[0] += bi * zi;
        if (ZQ) part[ZQ ? 1 : 0] += zi * q[i];
    });
    block_partials<ZQ ? 2 : 1, kFinRz>(part, red, sc, ctl);
}

// r.z and z.q of the FP32 cycle's output, which stays in FP32 (the search
// direction's update widens it again: 4 bytes a value instead of 8 written
// and read)
__global__ void __launch_bounds__(kThreads)
rz32_kernel(int32_t n, const float *__restrict__ z32, const double *__restrict__ r, const double *__restrict__ q,
            PcgScalars *sc, Reduce red, FinCtl ctl) {
    pdl_begin();
    block_partials_begin();
    double part[2] = {0.0, 0.0};
    for (int32_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
        const double zi = widen(z32[i]);
        part[0] += r[i] * zi;
        part[1] += zi * q[i];
    }
    block_partials<2, kFinRz>(part, red, sc, ctl);
}

template <typename XT>
__global__ void scale_kernel(int64_t n, const XT *__restrict__ a, const XT *__restrict__ d, XT *__restrict__ out) {
    pdl_begin();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a[i] * d[i];
}

__global__ void to_f32_scaled_kernel(int64_t n, const double *__restrict__ src, const float *__restrict__ d,
                                     float *__restrict__ dst, float *__restrict__ xdst) {
    pdl_begin();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = narrow(src[i]);
    dst[i] = v;
    xdst[i] = v * d[i];
}

// ---------------------------------------------------------------------------
// coarse solve: x = inv b, one warp per row
// ---------------------------------------------------------------------------
template <typename XT>
__global__ void coarse_kernel(int32_t n, const double *__restrict__ inv, const XT *b, XT *x) {
    constexpr int H = 4;  // entries a lane loads before the wait: the whole row up to 128 unknowns
    pdl_launch_next();
    int lane = threadIdx.x & 31;
    int32_t row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (row >= n) return;
    const double *a = inv + (size_t)row * n;
    double av[H];
#pragma unroll
    for (int k = 0; k < H; ++k) av[k] = lane + 32 * k < n ? __ldg(a + lane + 32 * k) : 0.0;
    pdl_wait();
    double s = 0.0;
    XT bv[H];
#pragma unroll
    for (int k = 0; k < H; ++k) bv[k] = lane + 32 * k < n ? ld_dyn(b + lane + 32 * k) : XT(0);
#pragma unroll
    for (int k = 0; k < H; ++k)
        if (32 * k < n) s += av[k] * (double)bv[k];
    for (int32_t j = lane + 32 * H; j < n; j += 32) s += __ldg(a + j) * (double)ld_dyn(b + j);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) x[row] = (XT)s;
}

// ---------------------------------------------------------------------------
// conversions and SELL construction
// ---------------------------------------------------------------------------
template <typename VT>
__global__ void convert_kernel(const double *src, VT *dst, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (VT)src[i];
}
template <>
__global__ void convert_kernel<__nv_bfloat16>(const double *src, __nv_bfloat16 *dst, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = __double2bfloat16(src[i]);
}

template <typename XT>
__global__ void to_f64_kernel(const XT *src, double *dst, int64_t n) {
    pdl_begin();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (double)src[i];
}

// rows sorted by length (descending, then index) inside windows of
// kSellSigma rows: one block sorts one window with a bitonic network
__global__ void __launch_bounds__(512) sell_sort_kernel(int32_t n, const int32_t *rp, int32_t *perm) {
    __shared__ unsigned long long key[kSellSigma];
    int32_t w0 = blockIdx.x * kSellSigma;
    for (int t = threadIdx.x; t < kSellSigma; t += blockDim.x) {
        int32_t i = w0 + t;
        key[t] = i < n ? ((unsigned long long)(0x7fffffff - (rp[i + 1] - rp[i])) << 32) | (unsigned)i : ~0ull;
    }
    __syncthreads();
    for (int size = 2; size <= kSellSigma; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < kSellSigma; t += blockDim.x) {
                int partner = t ^ stride;
                if (partner > t) {
                    bool up = (t & size) == 0;
                    unsigned long long a = key[t], c = key[partner];
                    if ((a > c) == up) { key[t] = c; key[partner] = a; }
                }
            }
            __syncthreads();
        }
    }
    for (int t = threadIdx.x; t < kSellSigma; t += blockDim.x) {
        int32_t i = w0 + t;
        if (i < n) perm[i] = (int32_t)(key[t] & 0xffffffffu);
    }
}

// width of each slice of C rows: its longest row, rounded up to a multiple
// of the 32 / C lanes that share a row
__global__ void slice_width_kernel(int32_t n, const int32_t *rp, const int32_t *perm, int32_t *sw, int C) {
    int32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t nsl = (n + C - 1) / C;
    if (s >= nsl) return;
    int32_t w = 0;
    for (int32_t pos = s * C; pos < min(n, s * C + C); ++pos) {
        int32_t i = perm ? perm[pos] : pos;
        w = max(w, rp[i + 1] - rp[i]);
    }
    const int32_t T = 32 / C;
    sw[s] = (w + T - 1) / T * T;
}

__global__ void slice_size_kernel(int32_t nsl, const int32_t *sw, int32_t *sz, int C) {
    int32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nsl) sz[s] = sw[s] * C;
}

template <typename VT>
__global__ void sell_fill_kernel(int32_t n, const int32_t *rp, const int32_t *ci, const VT *v, const int32_t *perm,
                                 const int32_t *soff, const int32_t *sw, int32_t *sci, VT *sv, int16_t *sd, int C) {
    int32_t pos = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t nsl = (n + C - 1) / C;
    if (pos >= nsl * C) return;
    int32_t s = pos / C, lane = pos % C;
    int32_t off = soff[s] + lane, w = sw[s];
    int32_t i = pos < n ? (perm ? perm[pos] : pos) : -1;
    int32_t p0 = i >= 0 ? rp[i] : 0, len = i >= 0 ? rp[i + 1] - p0 : 0;
    // padding: value 0 at a column the row itself holds (its last one), or
    // column 0 for an empty row -- always inside x, also for rectangular
    // operators (P is n x n_c); with int16 offsets an empty row pads with
    // its own index (offset 0; those operators are square)
    const int32_t pad_col = len > 0 ? ci[p0 + len - 1] : (sd ? (i >= 0 ? i : 0) : 0);
    for (int32_t k = 0; k < w; ++k) {
        int32_t p = off + k * C;
        const int32_t c = k < len ? ci[p0 + k] : pad_col;
        if (sd) sd[p] = (int16_t)(i >= 0 ? c - i : 0);
        else sci[p] = c;
        sv[p] = k < len ? v[p0 + k] : VT(0);
    }
}

// out[0] = max |column - row|, out[1] = max stored entries of a row
__global__ void max_col_offset_kernel(int32_t n, const int32_t *rp, const int32_t *ci, int *out) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    int m = 0, len = 0;
    if (i < n) {
        for (int32_t p = rp[i]; p < rp[i + 1]; ++p) m = max(m, abs(ci[p] - i));
        len = rp[i + 1] - rp[i];
    }
    m = __reduce_max_sync(0xffffffffu, (unsigned)m);
    len = __reduce_max_sync(0xffffffffu, (unsigned)len);
    // one atomic per block: atomics of every warp on one address serialise
    __shared__ int sm[kThreads / 32], sl[kThreads / 32];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { sm[w] = m; sl[w] = len; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { m = max(m, sm[k]); len = max(len, sl[k]); }
        if (m) atomicMax(out, m);
        if (len) atomicMax(out + 1, len);
    }
}

}  // namespace

int threads_per_row(int variant) {
    switch (variant) {
        case AMG_SPMV_CSR1: return 1;
        case AMG_SPMV_CSR2: return 2;
        case AMG_SPMV_CSR4: return 4;
        case AMG_SPMV_CSR8: return 8;
        case AMG_SPMV_CSR16: return 16;
        case AMG_SPMV_CSR32: return 32;
        default: return 4;
    }
}

template <typename VT, typename XT>
void post_smooth(const CycMat<VT> &A, const XT *x, const XT *b, const XT *dinv, XT *xo, cudaStream_t s) {
    dispatch_op<VT, XT, kPost>(A, b, dinv, x, xo, nullptr, s);
}
template <typename VT, typename XT>
void spmv(const CycMat<VT> &A, const XT *x, XT *y, bool accumulate, cudaStream_t s) {
    if (accumulate) dispatch_op<VT, XT, kSpmvAdd>(A, nullptr, nullptr, x, y, nullptr, s);
    else dispatch_op<VT, XT, kSpmv>(A, nullptr, nullptr, x, y, nullptr, s);
}
template <typename VT, typename XT>
void spmv_scaled(const CycMat<VT> &A, const XT *x, const XT *d, XT *y, XT *xs, cudaStream_t s) {
    dispatch_op<VT, XT, kSpmvScale>(A, nullptr, d, x, y, xs, s);
}
template <typename VT, typename XT>
void residual_from_x(const CycMat<VT> &A, const XT *b, const XT *x, XT *r, cudaStream_t s) {
    dispatch_op<VT, XT, kResX>(A, b, nullptr, x, nullptr, r, s);
}

template <typename XT>
void coarse_solve(int32_t n, const double *inv, const XT *b, XT *x, cudaStream_t s) {
    if (n == 0) return;
    { pdl_launch(coarse_kernel<XT>, div_up(n, 8), 256, 0, s, n, inv, b, x); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

template <typename ZT> void pcg_p_update(int32_t n, const ZT *z, double *p, const PcgScalars *sc, cudaStream_t s) {
    { pdl_launch(p_update_kernel<ZT>, div_up(n, kThreads), kThreads, 0, s, n, z, p, sc); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

template void pcg_p_update<double>(int32_t, const double *, double *, const PcgScalars *, cudaStream_t);
template void pcg_p_update<float>(int32_t, const float *, double *, const PcgScalars *, cudaStream_t);

template <int T>
static void launch_ap(const CycMat<double> &A, const double *p, double *q, PcgScalars *sc, Reduce red, cudaStream_t s) {
    int blocks = reduce_blocks((int64_t)A.nrows * T);
    { pdl_launch(ap_kernel<T>, blocks, kThreads, 0, s, A.nrows, A.rp, A.ci, A.v, p, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); }
    launch_finish<1, kFinAp>(blocks, red, sc, s, fin_ctl(blocks));
}

// the SELL forms of A p and of the true residual; returns the block count
template <bool RESID>
static int launch_ap_sell(const CycMat<double> &A, const double *p, const double *b, double *q, PcgScalars *sc,
                          Reduce red, cudaStream_t s) {
    const int blocks = reduce_blocks(A.nrows);
    const FinCtl ctl = fin_ctl(blocks);
    const SellIdx ix{A.sci, A.sd};
    const bool sh = A.max_row > 0 && A.max_row <= kShortMax;
    if (A.sd && sh)
        { pdl_launch(ap_sell_kernel<true, true, RESID>, blocks, kThreads, 0, s, A.nrows, A.perm, A.soff, A.sw, ix, A.sv, p, b, q, sc, red, ctl); ::amg::count_launch(); }
    else if (A.sd)
        { pdl_launch(ap_sell_kernel<true, false, RESID>, blocks, kThreads, 0, s, A.nrows, A.perm, A.soff, A.sw, ix, A.sv, p, b, q, sc, red, ctl); ::amg::count_launch(); }
    else if (sh)
        { pdl_launch(ap_sell_kernel<false, true, RESID>, blocks, kThreads, 0, s, A.nrows, A.perm, A.soff, A.sw, ix, A.sv, p, b, q, sc, red, ctl); ::amg::count_launch(); }
    else
        { pdl_launch(ap_sell_kernel<false, false, RESID>, blocks, kThreads, 0, s, A.nrows, A.perm, A.soff, A.sw, ix, A.sv, p, b, q, sc, red, ctl); ::amg::count_launch(); }
    return blocks;
}

void pcg_ap(const CycMat<double> &A, const double *p, double *q, PcgScalars *sc, Reduce red, cudaStream_t s) {
    if (A.part.parts) {  // row-partitioned: exchange, then the one-lane kernel's loop
        part_exchange(A.part, p, s);
        const int blocks = reduce_blocks(A.nrows);
        { pdl_launch(ap_kernel<1, true>, blocks, kThreads, 0, s, A.nrows, A.rp, A.part.cext, A.v, p, q, sc, red, fin_ctl(blocks), A.part); ::amg::count_launch(); }
        launch_finish<1, kFinAp>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.pat.pid) {
        const int blocks = pat_grid(A.nrows);
        { pdl_launch(ap_pat_kernel<false>, blocks, kThreads, pat_smem_bytes<double>(A.pat.npat, A.pat.width), s, A.nrows, A.pat, p, (const double *)nullptr, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
        launch_finish<1, kFinAp>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.variant == AMG_SPMV_SELL32 && A.sv && A.sell_c == 32) {
        const int blocks = launch_ap_sell<false>(A, p, nullptr, q, sc, red, s);
        launch_finish<1, kFinAp>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    switch (threads_per_row(A.variant == AMG_SPMV_SELL32 ? AMG_SPMV_CSR4 : A.variant)) {
        case 1: launch_ap<1>(A, p, q, sc, red, s); break;
        case 2: launch_ap<2>(A, p, q, sc, red, s); break;
        case 4: launch_ap<4>(A, p, q, sc, red, s); break;
        case 8: launch_ap<8>(A, p, q, sc, red, s); break;
        case 16: launch_ap<16>(A, p, q, sc, red, s); break;
        default: launch_ap<32>(A, p, q, sc, red, s); break;
    }
    AMG_CHECK_LAUNCH();
}

void pcg_xr_update(int32_t n, const double *p, const double *q, double *x, double *r, PcgScalars *sc,
                   Reduce red, cudaGraphConditionalHandle handle, bool use_handle, const CycleInput &next,
                   double *xs, cudaStream_t s) {
    int blocks = reduce_blocks(n);
    const FinCtl ctl = fin_ctl(blocks, handle, use_handle);
    { pdl_launch(xr_update_kernel, blocks, kThreads, 0, s, n, p, q, x, r, sc, red, next, xs, ctl); ::amg::count_launch(); }
    launch_finish<1, kFinXr>(blocks, red, sc, s, ctl);
    AMG_CHECK_LAUNCH();
}

template <bool ZQ>
static void post_smooth_rz_launch(const CycMat<double> &A, const double *x, const double *b, const double *dinv,
                                  double *z, const double *q, PcgScalars *sc, Reduce red, cudaStream_t s) {
    const int32_t n = A.nrows;
    constexpr int NV = ZQ ? 2 : 1;
    if (A.part.parts) {
        part_exchange(A.part, x, s);
        const int blocks = reduce_blocks(n);
        { pdl_launch(post_rz_csr_kernel<1, ZQ, true>, blocks, kThreads, 0, s, n, A.rp, A.part.cext, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), A.part); ::amg::count_launch(); }
        launch_finish<NV, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.pat.pid) {
        const int blocks = pat_grid(n);
        { pdl_launch(post_rz_pat_kernel<ZQ>, blocks, kThreads, pat_smem_bytes<double>(A.pat.npat, A.pat.width), s, n, A.pat, x, b, z, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
        launch_finish<NV, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.variant == AMG_SPMV_SELL32 && A.sv && A.sell_c == 32) {
        int blocks = reduce_blocks(n);
        const SellIdx ix{A.sci, A.sd};
        if (A.sd)
            { pdl_launch(post_rz_sell_kernel<true, ZQ>, blocks, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, x, b, dinv, z, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
        else
            { pdl_launch(post_rz_sell_kernel<false, ZQ>, blocks, kThreads, 0, s, n, A.perm, A.soff, A.sw, ix, A.sv, x, b, dinv, z, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
        launch_finish<NV, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    int T = threads_per_row(A.variant);
    int blocks = reduce_blocks((int64_t)n * T);
    switch (T) {
        case 1: { pdl_launch(post_rz_csr_kernel<1, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
        case 2: { pdl_launch(post_rz_csr_kernel<2, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
        case 4: { pdl_launch(post_rz_csr_kernel<4, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
        case 8: { pdl_launch(post_rz_csr_kernel<8, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
        case 16: { pdl_launch(post_rz_csr_kernel<16, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
        default: { pdl_launch(post_rz_csr_kernel<32, ZQ>, blocks, kThreads, 0, s, n, A.rp, A.ci, A.v, x, b, dinv, z, q, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); } break;
    }
    launch_finish<NV, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
    AMG_CHECK_LAUNCH();
}

bool post_smooth_rz(const CycMat<double> &A, const double *x, const double *b, const double *dinv, double *z,
                    const double *q, PcgScalars *sc, Reduce red, cudaStream_t s) {
    if (A.nrows == 0) return false;
    if (q) post_smooth_rz_launch<true>(A, x, b, dinv, z, q, sc, red, s);
    else post_smooth_rz_launch<false>(A, x, b, dinv, z, q, sc, red, s);
    return true;
}

void pcg_rz32(int32_t n, const float *z32, const double *r, const double *q, PcgScalars *sc, Reduce red,
              cudaStream_t s) {
    int blocks = reduce_blocks(n);
    { pdl_launch(rz32_kernel, blocks, kThreads, 0, s, n, z32, r, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
    launch_finish<2, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
    AMG_CHECK_LAUNCH();
}

template <typename XT> void scale(int64_t n, const XT *a, const XT *d, XT *out, cudaStream_t s) {
    if (n <= 0) return;
    { pdl_launch(scale_kernel<XT>, div_up(n, kThreads), kThreads, 0, s, n, a, d, out); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
template void scale<double>(int64_t, const double *, const double *, double *, cudaStream_t);
template void scale<float>(int64_t, const float *, const float *, float *, cudaStream_t);

void to_f32_scaled(int64_t n, const double *src, const float *d, float *dst, float *xdst, cudaStream_t s) {
    if (n <= 0) return;
    { pdl_launch(to_f32_scaled_kernel, div_up(n, kThreads), kThreads, 0, s, n, src, d, dst, xdst); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

void pcg_rz(int32_t n, const double *r, const double *z, const double *q, PcgScalars *sc, Reduce red,
            cudaStream_t s) {
    int blocks = reduce_blocks(n);
    { pdl_launch(rz_kernel, blocks, kThreads, 0, s, n, r, z, q, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
    launch_finish<2, kFinRz>(blocks, red, sc, s, fin_ctl(blocks));
    AMG_CHECK_LAUNCH();
}

void true_residual(const CycMat<double> &A, const double *b, const double *x, double *t, PcgScalars *sc,
                   Reduce red, cudaStream_t s) {
    if (A.part.parts) {  // row-partitioned: the four-lane kernel's loop, as below
        part_exchange(A.part, x, s);
        const int blocks = reduce_blocks((int64_t)A.nrows * 4);
        { pdl_launch(resid_kernel<4, true>, blocks, kThreads, 0, s, A.nrows, A.rp, A.part.cext, A.v, b, x, t, sc, red, fin_ctl(blocks), A.part); ::amg::count_launch(); }
        launch_finish<1, kFinTt>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.pat.pid) {
        const int blocks = pat_grid(A.nrows);
        { pdl_launch(ap_pat_kernel<true>, blocks, kThreads, pat_smem_bytes<double>(A.pat.npat, A.pat.width), s, A.nrows, A.pat, x, b, t, sc, red, fin_ctl(blocks)); ::amg::count_launch(); }
        launch_finish<1, kFinTt>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    if (A.variant == AMG_SPMV_SELL32 && A.sv && A.sell_c == 32) {  // the operator's tuned SELL copy, as A p uses
        const int blocks = launch_ap_sell<true>(A, x, b, t, sc, red, s);
        launch_finish<1, kFinTt>(blocks, red, sc, s, fin_ctl(blocks));
        AMG_CHECK_LAUNCH();
        return;
    }
    int blocks = reduce_blocks((int64_t)A.nrows * 4);
    { pdl_launch(resid_kernel<4>, blocks, kThreads, 0, s, A.nrows, A.rp, A.ci, A.v, b, x, t, sc, red, fin_ctl(blocks), PartView()); ::amg::count_launch(); }
    launch_finish<1, kFinTt>(blocks, red, sc, s, fin_ctl(blocks));
    AMG_CHECK_LAUNCH();
}

template <typename VT> void convert_values(const double *src, VT *dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    { convert_kernel<VT><<<div_up(n, kThreads), kThreads, 0, s>>>(src, dst, n); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}
template <typename XT> void convert_vec_from_f64(const double *src, XT *dst, int64_t n, cudaStream_t s) {
    convert_values<XT>(src, dst, n, s);
}
template <typename XT> void convert_vec_to_f64(const XT *src, double *dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    { pdl_launch(to_f64_kernel<XT>, div_up(n, kThreads), kThreads, 0, s, src, dst, n); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

int64_t sell_layout(int32_t n, const int32_t *rp, int32_t *perm, int32_t *soff, int32_t *sw, cudaStream_t s, int C) {
    if (C != 32 && C != 16 && C != 8) throw Error(AMG_ERR_INVALID, "SELL slice height must be 32, 16 or 8");
    int32_t nsl = (n + C - 1) / C;
    if (nsl == 0) return 0;
    TmpBuf sz(sizeof(int32_t) * (nsl + 1), s);
    if (perm) { sell_sort_kernel<<<div_up(n, kSellSigma), 512, 0, s>>>(n, rp, perm); ::amg::count_launch(); }
    { slice_width_kernel<<<div_up(nsl, kThreads), kThreads, 0, s>>>(n, rp, perm, sw, C); ::amg::count_launch(); }
    { slice_size_kernel<<<div_up(nsl, kThreads), kThreads, 0, s>>>(nsl, sw, sz.as<int32_t>(), C); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
    return exclusive_scan_i32(sz.as<int32_t>(), soff, nsl, s);
}

template <typename VT>
void sell_fill(int32_t n, const int32_t *rp, const int32_t *ci, const VT *v, const int32_t *perm, const int32_t *soff,
               const int32_t *sw, int32_t *sci, VT *sv, cudaStream_t s, int16_t *sd, int C) {
    int32_t nsl = (n + C - 1) / C;
    if (nsl == 0) return;
    { sell_fill_kernel<VT><<<div_up((int64_t)nsl * C, kThreads), kThreads, 0, s>>>(n, rp, ci, v, perm, soff, sw, sci, sv, sd, C); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
}

int32_t max_col_offset(int32_t n, const int32_t *rp, const int32_t *ci, cudaStream_t s, int32_t *max_row) {
    if (max_row) *max_row = 0;
    if (n == 0) return 0;
    TmpBuf out(sizeof(int) * 2, s);
    AMG_CUDA(cudaMemsetAsync(out.ptr, 0, sizeof(int) * 2, s));
    { max_col_offset_kernel<<<div_up(n, kThreads), kThreads, 0, s>>>(n, rp, ci, out.as<int>()); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
    int h[2];
    read_back(h, out.ptr, sizeof(h), s);
    if (max_row) *max_row = h[1];
    return h[0];
}

// explicit instantiations
#define AMG_INST(VT, XT)                                                                                  \
    template void post_smooth<VT, XT>(const CycMat<VT> &, const XT *, const XT *, const XT *, XT *, cudaStream_t); \
    template void spmv<VT, XT>(const CycMat<VT> &, const XT *, XT *, bool, cudaStream_t); \
    template void spmv_scaled<VT, XT>(const CycMat<VT> &, const XT *, const XT *, XT *, XT *, cudaStream_t); \
    template void residual_from_x<VT, XT>(const CycMat<VT> &, const XT *, const XT *, XT *, cudaStream_t);
AMG_INST(double, double)
AMG_INST(float, float)
AMG_INST(__nv_bfloat16, float)
#undef AMG_INST
template void coarse_solve<double>(int32_t, const double *, const double *, double *, cudaStream_t);
template void coarse_solve<float>(int32_t, const double *, const float *, float *, cudaStream_t);
template void convert_values<float>(const double *, float *, int64_t, cudaStream_t);
template void convert_values<__nv_bfloat16>(const double *, __nv_bfloat16 *, int64_t, cudaStream_t);
template void convert_vec_from_f64<float>(const double *, float *, int64_t, cudaStream_t);
template void convert_vec_to_f64<float>(const float *, double *, int64_t, cudaStream_t);
template void sell_fill<double>(int32_t, const int32_t *, const int32_t *, const double *, const int32_t *,
                                const int32_t *, const int32_t *, int32_t *, double *, cudaStream_t, int16_t *, int);
template void sell_fill<float>(int32_t, const int32_t *, const int32_t *, const float *, const int32_t *,
                               const int32_t *, const int32_t *, int32_t *, float *, cudaStream_t, int16_t *, int);
template void sell_fill<__nv_bfloat16>(int32_t, const int32_t *, const int32_t *, const __nv_bfloat16 *,
                                       const int32_t *, const int32_t *, const int32_t *, int32_t *, __nv_bfloat16 *,
                                       cudaStream_t, int16_t *, int);

}  // namespace cyc
}  // namespace amg
