// patterns.cu -- operators with few distinct rows.
//
// A constant-coefficient stencil on a uniform grid (the 5-, 7-, 9- and
// 27-point operators of the finest level) stores the same row -- the same
// column offsets from the diagonal, the same values -- millions of times: 27
// distinct rows in 3D, nine in 2D.  Such an operator is kept as one byte per
// row, the number of its pattern, and a small table of the patterns, which
// the cycle kernels hold in shared memory: a 27-point row moves 1 byte
// instead of 162 (FP32 SELL with int16 offsets) or 270 (FP64).  Nothing is
// rounded or assumed: rows are matched by a hash first and then compared
// entry by entry, bit for bit, with their pattern, and a row's sum runs over
// the same entries in the same order as in CSR or SELL-32.
//
// Three passes on the stream, one read-back: hash every row into a table of
// at most kPatMax keys (given up at once when it overflows: coefficients that
// vary leave after the first blocks), number the patterns and write their
// table from one representative row each, compare every row with its pattern.
#include <algorithm>

#include "common.cuh"
#include "cycle_ops.cuh"

namespace amg {
namespace cyc {

namespace {

constexpr int kThreads = 256;
constexpr int kSlots = 1024;  // hash slots, at most a quarter of them for an operator that is kept
constexpr int kProbes = 64;   // longest probe sequence followed (longer: given up)

struct PatHead {
    int fail, npat, width, count;
};
// the passes' workspace, cleared as one block: a slot's representative is
// kept as kNoRow - row, so that clearing it means "none"
struct PatWork {
    PatHead head;
    unsigned long long keys[kSlots];
    int32_t rep[kSlots], map[kSlots];
};
constexpr int32_t kNoRow = 0x7fffffff;

__device__ __forceinline__ unsigned long long mix(unsigned long long z) {
    // the finaliser of SplitMix64 (Steele, Lea, Flood 2014)
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// One thread per row of [first, n): its hash finds or takes a slot; the slot's
// representative is the lowest row that hashed there.  The first kSample rows
// go in a launch of their own: rows that all differ overflow the table there,
// and the rest leaves at once -- in one launch the first wave's 300 thousand
// threads fight for the table's slots (0.56 ms at 128^3 lognormal).
constexpr int kSample = 4096;
__global__ void __launch_bounds__(kThreads)
pat_hash_kernel(int32_t first, int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                const double *__restrict__ v, PatHead *hd, unsigned long long *keys, int32_t *rep, uint16_t *slot) {
    const int64_t i = (int64_t)first + blockIdx.x * kThreads + threadIdx.x;
    if (i >= n || *(volatile int *)&hd->fail) return;
    const int32_t p0 = rp[i], len = rp[i + 1] - p0;
    if (len < 1 || len > kPatWidth) {
        hd->fail = 1;
        return;
    }
    if (len > *(volatile int *)&hd->width) atomicMax(&hd->width, len);
    unsigned long long h = mix((unsigned long long)len + 0x9E3779B97F4A7C15ull);
    for (int32_t k = 0; k < len; ++k) {
        h = mix(h + (unsigned long long)(uint32_t)(ci[p0 + k] - (int32_t)i));
        h = mix(h ^ (unsigned long long)__double_as_longlong(v[p0 + k]));
    }
    if (h == 0) h = 1;  // 0 marks an empty slot
    uint32_t s = (uint32_t)h & (kSlots - 1);
    for (int probe = 0; probe < kProbes && !*(volatile int *)&hd->fail; ++probe, s = (s + 1) & (kSlots - 1)) {
        unsigned long long k = *(volatile unsigned long long *)&keys[s];
        if (k == 0) {
            k = atomicCAS(&keys[s], 0ull, h);
            if (k == 0) {
                if (atomicAdd(&hd->count, 1) >= kPatMax) hd->fail = 1;
                k = h;
            }
        }
        if (k == h) {
            const int32_t key = kNoRow - (int32_t)i;
            if (key > *(volatile int32_t *)&rep[s]) atomicMax(&rep[s], key);
            slot[i] = (uint16_t)s;
            return;
        }
    }
    hd->fail = 1;
}

// One block: pattern numbers by slot order, the table from the representative
// rows (entries past a row's length: value 0 on the diagonal).
__global__ void __launch_bounds__(kSlots)
pat_table_kernel(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, const double *__restrict__ v,
                 const double *__restrict__ dinv, PatHead *hd, const unsigned long long *keys, const int32_t *rep,
                 int32_t *map, PatTable t) {
    __shared__ int32_t rows[kSlots];
    __shared__ int warp_cnt[kSlots / 32];
    if (hd->fail) return;  // uniform: written by the kernel before
    const int s = threadIdx.x, lane = s & 31, w = s >> 5;
    const bool used = keys[s] != 0ull;
    const unsigned m = __ballot_sync(0xffffffffu, used);
    if (lane == 0) warp_cnt[w] = __popc(m);
    __syncthreads();
    int id = __popc(m & ((1u << lane) - 1u)), total = 0;
    for (int k = 0; k < kSlots / 32; ++k) {
        if (k < w) id += warp_cnt[k];
        total += warp_cnt[k];
    }
    if (total > kPatMax) {
        if (s == 0) hd->fail = 1;
        return;
    }
    if (used) {
        map[s] = id;
        rows[id] = kNoRow - rep[s];
    }
    __syncthreads();
    const int W = hd->width;
    for (int e = s; e < total * W; e += kSlots) {
        const int p = e / W, k = e % W;
        const int32_t i = rows[p], p0 = rp[i], len = rp[i + 1] - p0;
        const double a = k < len ? v[p0 + k] : 0.0;
        t.val64[e] = a;
        t.val32[e] = (float)a;
        t.delta[e] = k < len ? ci[p0 + k] - i : 0;
        if (k == 0) {
            t.len[p] = len;
            t.dinv64[p] = dinv[i];
            t.dinv32[p] = (float)dinv[i];
        }
    }
    if (s == 0) hd->npat = total;
}

// Every row against its pattern, entry by entry.
__global__ void __launch_bounds__(kThreads)
pat_check_kernel(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                 const double *__restrict__ v, PatHead *hd, const uint16_t *__restrict__ slot,
                 const int32_t *__restrict__ map, PatTable t, uint8_t *pid) {
    const int32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n || *(volatile int *)&hd->fail) return;
    const int W = hd->width, p = map[slot[i]];
    const int32_t p0 = rp[i], len = rp[i + 1] - p0;
    bool same = len == t.len[p];
    if (same)
        for (int32_t k = 0; k < len; ++k)
            same = same && ci[p0 + k] - i == t.delta[p * W + k] &&
                   __double_as_longlong(v[p0 + k]) == __double_as_longlong(t.val64[p * W + k]);
    if (!same) hd->fail = 1;
    pid[i] = (uint8_t)p;
}

}  // namespace

size_t pat_table_bytes() { return (size_t)kPatMax * ((kPatWidth + 1) * (sizeof(double) + sizeof(float)) + (kPatWidth + 1) * sizeof(int32_t)); }

PatTable pat_table(void *base) {
    PatTable t;
    const size_t e = (size_t)kPatMax * kPatWidth;
    t.val64 = static_cast<double *>(base);
    t.dinv64 = t.val64 + e;
    t.val32 = reinterpret_cast<float *>(t.dinv64 + kPatMax);
    t.dinv32 = t.val32 + e;
    t.delta = reinterpret_cast<int32_t *>(t.dinv32 + kPatMax);
    t.len = t.delta + e;
    return t;
}

bool build_patterns(const DevCSR &M, const double *dinv, uint8_t *pid, void *table, int32_t *npat, int32_t *width,
                    cudaStream_t s) {
    const int32_t n = M.nrows;
    *npat = *width = 0;
    if (n == 0 || M.nrows != M.ncols || M.nnz > (int64_t)n * kPatWidth) return false;
    TmpBuf work(sizeof(PatWork), s), slots(sizeof(uint16_t) * (size_t)n, s);
    AMG_CUDA(cudaMemsetAsync(work.ptr, 0, sizeof(PatWork), s));
    PatWork *w = work.as<PatWork>();
    PatHead *hd = &w->head;
    uint16_t *slot = slots.as<uint16_t>();
    const PatTable t = pat_table(table);
    const int g = div_up(n, kThreads);
    const int32_t head_rows = std::min(n, (int32_t)kSample);
    { pat_hash_kernel<<<div_up(head_rows, kThreads), kThreads, 0, s>>>(0, head_rows, M.rp(), M.ci(), M.v(), hd, w->keys, w->rep, slot); ::amg::count_launch(); }
    if (n > head_rows) { pat_hash_kernel<<<div_up(n - head_rows, kThreads), kThreads, 0, s>>>(head_rows, n, M.rp(), M.ci(), M.v(), hd, w->keys, w->rep, slot); ::amg::count_launch(); }
    { pat_table_kernel<<<1, kSlots, 0, s>>>(M.rp(), M.ci(), M.v(), dinv, hd, w->keys, w->rep, w->map, t); ::amg::count_launch(); }
    { pat_check_kernel<<<g, kThreads, 0, s>>>(n, M.rp(), M.ci(), M.v(), hd, slot, w->map, t, pid); ::amg::count_launch(); }
    AMG_CHECK_LAUNCH();
    PatHead h;
    read_back(&h, hd, sizeof(h), s);
    if (h.fail || pat_smem_bytes<double>(h.npat, h.width) > kPatSmem) return false;
    *npat = h.npat;
    *width = h.width;
    return true;
}

}  // namespace cyc
}  // namespace amg
