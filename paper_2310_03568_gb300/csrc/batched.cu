// Batched reduce_by_index -> +-scan -> sum over many independent instances,
// forward and vjp, in a few persistent launches.
//
// Forward (per instance i, op ADD or MAX, initial histogram all zero):
//   hist_i  = reduce_by_index (replicate m_i 0) op keys_i vals_i     (Sec. 4)
//   scan_i  = scan (+) hist_i                                        (Sec. 5.1)
//   loss    = sum_i sum_j scan_i[j]                                  (Sec. 3)
// vjp: ybar of the sum is a broadcast (Sec. 3.2.1), the +-scan's adjoint a
// reverse +-scan (Sec. 5.3.1) -- of a constant, so (m - j) lossbar without a
// pass over memory -- then the gather of Sec. 4.2.1 (ADD) or the
// argmax scatter of Fig. 5 (MAX; the zero initial value wins ties).
//
// Launches: init (one block per instance) -> histogram (persistent blocks
// pulling (instance, element range) work items from an atomic counter; a
// shared-memory table when the instance's bins fit and the item is long
// enough to amortise it, global atomics otherwise) -> scan + loss (one block
// per instance, deterministic loss from per-instance partials combined in
// instance order by the last block).  Backward: per-item gather / zero-fill ->
// per-instance histogram adjoints and argmax scatter.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "hist_common.cuh"
#include "internal.h"

namespace adc {

constexpr int kBHistThreads = 512;
constexpr int kBScanThreads = 512;
constexpr int kBBinThreads = 1024;  // init and scatter: one element per thread and step
constexpr int32_t kDefaultSmemBins = 12288;  // 96 KB of table: two blocks per SM

// Packed max key: order-preserving value bits above the inverted index, so a
// 64-bit atomicMax keeps the largest value and, among equal values, the
// smallest index (Fig. 5's lifted operator).
__device__ __forceinline__ unsigned long long bmax_key(float v, int64_t i) {
    return ((unsigned long long)ordered_key(v) << 32) | (0xffffffffu - (uint32_t)i);
}
__device__ __forceinline__ int64_t bmax_index(unsigned long long k) { return (int64_t)(0xffffffffu - (uint32_t)k); }

// Elements per thread and step of the histogram launch (1, 4 or 8; tuning hook).
static int g_batched_ipt = 8;

// Elements before `p` and `q` (both at the same element offset) reach a 16-byte
// boundary together, or -1 when they never do.
__device__ __forceinline__ int64_t quad_head(const void *p, const void *q) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
    return ((a ^ b) & 15) ? -1 : (int64_t)(((16 - (a & 15)) & 15) / 4);
}

__global__ void k_b_init(const adc_instance *__restrict__ desc, float *__restrict__ hist,
                         unsigned long long *__restrict__ tab) {
    const adc_instance d = desc[blockIdx.x];
    if (d.op == ADC_OP_ADD) {
#pragma unroll 4
        for (int64_t j = threadIdx.x; j < d.m; j += blockDim.x) hist[d.bin_off + j] = 0.f;
    } else {
#pragma unroll 4
        for (int64_t j = threadIdx.x; j < d.m; j += blockDim.x) tab[d.bin_off + j] = 0ull;
    }
}

// Every element of an item, in groups: update(key[4], value[4], element of the
// first, use[4]), use[c] set for keys in [0, m), so that an update which reads
// before it writes can have the group's reads in flight together.
// IPT = 4 or 8: 16-byte loads, IPT elements per thread and step, the next
// step's loads issued before this step's updates; the elements before the
// first 16-byte boundary and the last few one by one.  IPT = 1: one by one.
template <int IPT, class F>
__device__ __forceinline__ void b_elements(const int32_t *__restrict__ k, const float *__restrict__ v, int64_t len,
                                           int64_t m, F &&update) {
    const auto one = [&](int64_t e) {
        const int32_t kk[4] = {__ldcs(k + e), -1, -1, -1};
        const float vv[4] = {__ldcs(v + e), 0.f, 0.f, 0.f};
        const bool use[4] = {(uint32_t)kk[0] < (uint64_t)m, false, false, false};
        update(kk, vv, e, use);
    };
    int64_t head = IPT == 1 ? -1 : quad_head(k, v);
    if (head < 0 || head >= len) {
        for (int64_t e = threadIdx.x; e < len; e += blockDim.x) one(e);
        return;
    }
    constexpr int U = IPT < 4 ? 1 : IPT / 4;  // quads per thread and step
    const int64_t quads = (len - head) / 4;
    if (threadIdx.x < head) one(threadIdx.x);
    const int64_t tail = head + 4 * quads + threadIdx.x;
    if (tail < len) one(tail);  // fewer than 4
    const int4 *k4 = reinterpret_cast<const int4 *>(k + head);
    const float4 *v4 = reinterpret_cast<const float4 *>(v + head);
    int4 kq[U], kn[U];
    float4 vq[U], vn[U];
    const auto fetch = [&](int64_t q0, int4 (&kd)[U], float4 (&vd)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t q = q0 + (int64_t)u * blockDim.x;
            kd[u] = q < quads ? __ldcs(k4 + q) : make_int4(-1, -1, -1, -1);
            vd[u] = q < quads ? __ldcs(v4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    int64_t q0 = threadIdx.x;
    fetch(q0, kq, vq);
    while (q0 < quads) {
        const int64_t qn = q0 + (int64_t)U * blockDim.x;
        fetch(qn, kn, vn);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t e = head + 4 * (q0 + (int64_t)u * blockDim.x);
            const int32_t kk[4] = {kq[u].x, kq[u].y, kq[u].z, kq[u].w};
            const float vv[4] = {vq[u].x, vq[u].y, vq[u].z, vq[u].w};
            bool use[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) use[c] = (uint32_t)kk[c] < (uint64_t)m;
            update(kk, vv, e, use);
            kq[u] = kn[u];
            vq[u] = vn[u];
        }
        q0 = qn;
    }
}

using Key4 = const int32_t (&)[4];
using Val4 = const float (&)[4];
using Use4 = const bool (&)[4];

// The packed max of a group into t[key]: the current keys are read first, all
// four in flight, and only values that can still win go to the atomic.
template <bool GLOBAL>
__device__ __forceinline__ void bmax_update(unsigned long long *t, Key4 kk, Val4 vv, int64_t e, Use4 use) {
    unsigned long long key[4], cur[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        key[c] = bmax_key(vv[c], e + c);
        cur[c] = ~0ull;
        if (use[c]) cur[c] = GLOBAL ? __ldcg(t + kk[c]) : *reinterpret_cast<volatile unsigned long long *>(t + kk[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (key[c] > cur[c]) atomicMax(t + kk[c], key[c]);
}
__device__ __forceinline__ void badd_update(float *t, Key4 kk, Val4 vv, Use4 use) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (use[c]) atomicAdd(t + kk[c], vv[c]);
}

// Persistent blocks pull items.  An item whose bins fit the block's shared
// memory (`smem_bytes`; 4 bytes a bin for +, 8 for max) and are few enough to
// be worth flushing is built there, in up to one copy of the table per warp
// (fewer warps on one address; as many copies as fit and as the item's length
// pays for), and flushed with one atomic per bin and item -- consecutive
// addresses, so far cheaper than one scattered atomic per element.
template <int IPT>
__global__ void __launch_bounds__(kBHistThreads, 2)
k_b_hist(const adc_instance *__restrict__ desc, const adc_work *__restrict__ items, const int64_t n_items,
         const int32_t *__restrict__ keys, const float *__restrict__ vals, float *__restrict__ hist,
         unsigned long long *__restrict__ tab, const int32_t smem_bytes, unsigned *__restrict__ counter) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *sf = reinterpret_cast<float *>(smem_raw);
    unsigned long long *su = reinterpret_cast<unsigned long long *>(smem_raw);
    __shared__ unsigned s_item;
    while (true) {
        __syncthreads();  // the previous item's flush is done before smem is reused
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
        __syncthreads();
        const int64_t w = s_item;
        if (w >= n_items) return;
        const adc_work it = items[w];
        const adc_instance d = desc[it.inst];
        const int32_t *k = keys + d.val_off + it.start;
        const float *v = vals + d.val_off + it.start;
        const int64_t len = it.len, m = d.m;
        const bool add = d.op == ADC_OP_ADD;
        const int64_t cap = smem_bytes / (add ? 4 : 8);
        const bool use_smem = m <= cap && 2 * len >= m;
        int R = 1;
        if (use_smem) {
            const int64_t fit = cap / m, pay = len / (8 * m);
            const int64_t r = fit < pay ? fit : pay;
            R = r < 1 ? 1 : (r < kBHistThreads / kWarp ? (int)r : kBHistThreads / kWarp);
        }
        const int copy = (int)(threadIdx.x >> 5) % R;
        if (add) {
            float *g = hist + d.bin_off;
            if (use_smem) {
                for (int64_t j = threadIdx.x; j < m * R; j += blockDim.x) sf[j] = 0.f;
                __syncthreads();
                float *mine = sf + copy * m;
                b_elements<IPT>(k, v, len, m, [&](Key4 kk, Val4 vv, int64_t, Use4 use) { badd_update(mine, kk, vv, use); });
                __syncthreads();
                for (int64_t j = threadIdx.x; j < m; j += blockDim.x) {
                    float a = sf[j];
                    for (int r = 1; r < R; ++r) a += sf[r * m + j];
                    if (a != 0.f) atomicAdd(g + j, a);
                }
            } else {
                b_elements<IPT>(k, v, len, m, [&](Key4 kk, Val4 vv, int64_t, Use4 use) { badd_update(g, kk, vv, use); });
            }
        } else {
            unsigned long long *g = tab + d.bin_off;
            if (use_smem) {
                for (int64_t j = threadIdx.x; j < m * R; j += blockDim.x) su[j] = 0ull;
                __syncthreads();
                unsigned long long *mine = su + copy * m;
                b_elements<IPT>(k, v, len, m, [&](Key4 kk, Val4 vv, int64_t e, Use4 use) {
                    bmax_update<false>(mine, kk, vv, it.start + e, use);
                });
                __syncthreads();
                for (int64_t j = threadIdx.x; j < m; j += blockDim.x) {
                    unsigned long long a = su[j];
                    for (int r = 1; r < R; ++r) a = su[r * m + j] > a ? su[r * m + j] : a;
                    if (a > __ldcg(g + j)) atomicMax(g + j, a);
                }
            } else {
                b_elements<IPT>(k, v, len, m, [&](Key4 kk, Val4 vv, int64_t e, Use4 use) {
                    bmax_update<true>(g, kk, vv, it.start + e, use);
                });
            }
        }
    }
}

// Block-wide inclusive +-scan of one float per thread (kBScanThreads threads).
__device__ __forceinline__ float block_incl_sum(float x, float *tmp, float *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        float w = lane < kBScanThreads / kWarp ? tmp[lane] : 0.f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        tmp[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    *total = tmp[31];
    return x + (warp > 0 ? tmp[warp - 1] : 0.f);
}

// s += x; returns what the addition rounded off (two-sum; Knuth, TAOCP 2, 4.2.2).
__device__ __forceinline__ float two_sum(float &s, float x) {
    const float a = s;
    s = __fadd_rn(a, x);
    const float t = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(x, t));
}

// A thread's sum of floats, no less precise than a double's, without this part's
// slow FP64 pipe: hi + mid + lo, where mid takes what the additions to hi round
// off and lo what those to mid do, so that only lo rounds, at 2^-72 of the
// largest partial sum, and one conversion at the end (groups of eight in hi and
// mid alone, converted and added in double, were 2^-48, and one instance of 1e6
// bins and 1e7 values took 0.608 ms forward, 0.512 this way).  A group with which
// hi is not finite is added in double, as it stands.
struct LongSum {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    double rest = 0.0;
    __device__ __forceinline__ double value() const {
        if (hi == 0.f && mid == 0.f && lo == 0.f) return rest;  // the warps without bins skip the conversions
        return rest + ((double)hi + ((double)mid + (double)lo));
    }
    template <int I> __device__ __forceinline__ void add(const float (&x)[I]) {
        LongSum s = *this;
#pragma unroll
        for (int c = 0; c < I; ++c) s.lo = __fadd_rn(s.lo, two_sum(s.mid, two_sum(s.hi, x[c])));
        if (fabsf(s.hi) <= 3.0e38f) {
            *this = s;
        } else {
            rest = value();
            for (int c = 0; c < I; ++c) rest += (double)x[c];
            hi = mid = lo = 0.f;
        }
    }
};

// Block-wide sum, valid in thread 0: one warp adds the warps' sums (every
// thread adding all of them is 32 times the FP64 work: 8 us per block here).
__device__ __forceinline__ double block_sum_d(double x, double *tmp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    __syncthreads();
    if (lane == 0) tmp[warp] = x;
    __syncthreads();
    double s = 0.0;
    if (warp == 0) {
        if (lane < (int)(blockDim.x >> 5)) s = tmp[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    return s;
}

constexpr int kBScanItems = 8;  // consecutive bins per thread and step

// One block per instance, kBScanThreads * kBScanItems bins per step: every
// thread folds its consecutive bins, one block scan per step.
__global__ void __launch_bounds__(kBScanThreads, 3)
k_b_scan_loss(const adc_instance *__restrict__ desc, const int32_t count, float *__restrict__ hist,
              const unsigned long long *__restrict__ tab, float *__restrict__ scan, int32_t *__restrict__ is,
              float *__restrict__ loss_parts, float *__restrict__ loss, unsigned *__restrict__ ticket) {
    constexpr int I = kBScanItems;
    __shared__ float tmp[32];
    __shared__ double tmpd[32];
    __shared__ bool last;
    const adc_instance d = desc[blockIdx.x];
    const bool add = d.op == ADC_OP_ADD;
    float *h = hist + d.bin_off, *sc = scan + d.bin_off;
    int32_t *ix = is + d.bin_off;
    const unsigned long long *tb = tab + d.bin_off;
    const auto aligned16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    const bool vec = aligned16(h) && aligned16(sc) && aligned16(ix) && aligned16(tb);
    float carry = 0.f;
    LongSum sum_of_scan;
    for (int64_t base = 0; base < d.m; base += kBScanThreads * I) {
        const int64_t j0 = base + (int64_t)threadIdx.x * I;
        const bool whole = vec && j0 + I <= d.m;
        float x[I];
        if (add) {
            if (whole) {
#pragma unroll
                for (int q = 0; q < I / 4; ++q) {
                    const float4 t = *reinterpret_cast<const float4 *>(h + j0 + 4 * q);
                    x[4 * q] = t.x;
                    x[4 * q + 1] = t.y;
                    x[4 * q + 2] = t.z;
                    x[4 * q + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int c = 0; c < I; ++c) x[c] = j0 + c < d.m ? h[j0 + c] : 0.f;
            }
        } else {
            unsigned long long key[I];
            int32_t at[I];
            if (whole) {
#pragma unroll
                for (int q = 0; q < I / 2; ++q) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(tb + j0 + 2 * q);
                    key[2 * q] = t.x;
                    key[2 * q + 1] = t.y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < I; ++c) key[c] = j0 + c < d.m ? tb[j0 + c] : 0ull;
            }
#pragma unroll
            for (int c = 0; c < I; ++c) {
                // the key holds the value; the zero initial value wins ties
                const float val = key[c] != 0ull ? from_ordered((uint32_t)(key[c] >> 32)) : 0.f;
                const bool won = !(0.f >= val);
                x[c] = won ? val : 0.f;
                at[c] = won ? (int32_t)bmax_index(key[c]) : (int32_t)d.n;
            }
            if (whole) {
#pragma unroll
                for (int q = 0; q < I / 4; ++q) {
                    *reinterpret_cast<float4 *>(h + j0 + 4 * q) =
                        make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
                    *reinterpret_cast<int4 *>(ix + j0 + 4 * q) =
                        make_int4(at[4 * q], at[4 * q + 1], at[4 * q + 2], at[4 * q + 3]);
                }
            } else {
#pragma unroll
                for (int c = 0; c < I; ++c)
                    if (j0 + c < d.m) {
                        h[j0 + c] = x[c];
                        ix[j0 + c] = at[c];
                    }
            }
        }
        // A thread's bins are summed from zero and what lies before them is added to
        // each sum: one rounding at the prefix's magnitude per bin, however many bins
        // a thread has.
        float sum = 0.f;
#pragma unroll
        for (int c = 0; c < I; ++c) {
            sum += x[c];
            x[c] = sum;
        }
        float total;
        const float inc = block_incl_sum(sum, tmp, &total);
        float before = carry + __shfl_up_sync(0xffffffffu, inc, 1);
        if ((threadIdx.x & 31) == 0) before = carry + (threadIdx.x > 0 ? tmp[(threadIdx.x >> 5) - 1] : 0.f);
#pragma unroll
        for (int c = 0; c < I; ++c) x[c] = j0 + c < d.m ? before + x[c] : 0.f;
        sum_of_scan.add(x);
        if (whole) {
#pragma unroll
            for (int q = 0; q < I / 4; ++q)
                *reinterpret_cast<float4 *>(sc + j0 + 4 * q) =
                    make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
        } else {
#pragma unroll
            for (int c = 0; c < I; ++c)
                if (j0 + c < d.m) sc[j0 + c] = x[c];
        }
        carry += total;
    }
    const double part = block_sum_d(sum_of_scan.value(), tmpd);
    if (threadIdx.x == 0) {
        loss_parts[blockIdx.x] = (float)part;
        __threadfence();
        last = atomicAdd(ticket, 1u) == (unsigned)count - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < count; i += blockDim.x) acc += (double)__ldcg(loss_parts + i);
    const double s = block_sum_d(acc, tmpd);
    if (threadIdx.x == 0) *loss = (float)s;
}

// histbar[j] = sum_{k >= j} lbar: the reverse +-scan of a broadcast adjoint is
// (m - j) lbar, one rounding instead of a scan's.
__device__ __forceinline__ float b_hbar(int64_t m, int64_t j, float lb) { return (float)(m - j) * lb; }

// ADD: valsbar_e = histbar[k_e], which needs no table; MAX: zero-fill (the
// scatter follows).  16-byte accesses where the item's keys and adjoints reach
// a 16-byte boundary together.
__global__ void __launch_bounds__(kBHistThreads)
k_b_vjp_items(const adc_instance *__restrict__ desc, const adc_work *__restrict__ items, const int64_t n_items,
              const int32_t *__restrict__ keys, const float *__restrict__ loss_bar, float *__restrict__ valsbar,
              unsigned *__restrict__ counter) {
    __shared__ unsigned s_item;
    const float lb = *loss_bar;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
        __syncthreads();
        const int64_t w = s_item;
        if (w >= n_items) return;
        const adc_work it = items[w];
        const adc_instance d = desc[it.inst];
        const bool add = d.op == ADC_OP_ADD;
        const int32_t *k = keys + d.val_off + it.start;
        float *o = valsbar + d.val_off + it.start;
        const int64_t len = it.len, m = d.m;
        const auto grad = [&](int32_t kk) { return (uint32_t)kk < (uint64_t)m ? b_hbar(m, kk, lb) : 0.f; };
        const auto one = [&](int64_t e) { o[e] = add ? grad(__ldcs(k + e)) : 0.f; };
        const int64_t head = quad_head(k, o);
        if (head < 0 || head >= len) {
            for (int64_t e = threadIdx.x; e < len; e += blockDim.x) one(e);
            continue;
        }
        const int64_t quads = (len - head) / 4;
        if (threadIdx.x < head) one(threadIdx.x);
        if (head + 4 * quads + threadIdx.x < len) one(head + 4 * quads + threadIdx.x);
        const int4 *k4 = reinterpret_cast<const int4 *>(k + head);
        float4 *o4 = reinterpret_cast<float4 *>(o + head);
        if (!add) {
#pragma unroll 4
            for (int64_t q = threadIdx.x; q < quads; q += blockDim.x) __stcs(o4 + q, make_float4(0.f, 0.f, 0.f, 0.f));
            continue;
        }
        constexpr int U = 4;
        for (int64_t q0 = threadIdx.x; q0 < quads; q0 += (int64_t)U * blockDim.x) {
            int4 kq[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t q = q0 + (int64_t)u * blockDim.x;
                kq[u] = q < quads ? __ldcs(k4 + q) : make_int4(-1, -1, -1, -1);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t q = q0 + (int64_t)u * blockDim.x;
                if (q < quads) __stcs(o4 + q, make_float4(grad(kq[u].x), grad(kq[u].y), grad(kq[u].z), grad(kq[u].w)));
            }
        }
    }
}

// The histogram adjoints, and for MAX their scatter to the selected elements.
__global__ void __launch_bounds__(kBBinThreads)
k_b_hbar_scatter(const adc_instance *__restrict__ desc, const int32_t *__restrict__ is,
                 const float *__restrict__ loss_bar, float *__restrict__ histbar, float *__restrict__ valsbar) {
    const adc_instance d = desc[blockIdx.x];
    const float lb = *loss_bar;
    if (d.op != ADC_OP_MAX) {
#pragma unroll 4
        for (int64_t j = threadIdx.x; j < d.m; j += blockDim.x) histbar[d.bin_off + j] = b_hbar(d.m, j, lb);
        return;
    }
    constexpr int U = 4;
    for (int64_t j0 = threadIdx.x; j0 < d.m; j0 += (int64_t)U * blockDim.x) {
        int32_t i[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + (int64_t)u * blockDim.x;
            i[u] = j < d.m ? is[d.bin_off + j] : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t j = j0 + (int64_t)u * blockDim.x;
            if (j >= d.m) break;
            const float g = b_hbar(d.m, j, lb);
            histbar[d.bin_off + j] = g;
            if (i[u] >= 0 && i[u] < d.n) valsbar[d.val_off + i[u]] = g;
        }
    }
}

}  // namespace adc

using namespace adc;

namespace {
inline bool al(const void *p, size_t a) { return p != nullptr && reinterpret_cast<uintptr_t>(p) % a == 0; }
size_t ws_need(int64_t total_bins) { return kWsHeader + align_up((size_t)total_bins * 8, 256); }
}  // namespace

extern "C" {

int64_t adc_batched_plan(const adc_instance *desc, int32_t count, int64_t chunk, adc_work *items, int64_t capacity) {
    if (desc == nullptr || count < 1 || chunk < 1) return -1;
    // largest instances first: long items start early and small ones fill the tail
    std::vector<int32_t> order(count);
    for (int32_t i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return desc[a].n > desc[b].n; });
    int64_t k = 0;
    for (int32_t r = 0; r < count; ++r) {
        const adc_instance &d = desc[order[r]];
        if (d.n < 0 || d.m < 1) return -1;
        for (int64_t s = 0; s < d.n; s += chunk) {
            if (items != nullptr && k < capacity) {
                items[k].inst = order[r];
                items[k].pad = 0;
                items[k].start = s;
                items[k].len = (d.n - s < chunk) ? d.n - s : chunk;
            }
            ++k;
        }
    }
    return k;
}

size_t adc_batched_workspace_bytes(int32_t count, int64_t total_bins) {
    if (count < 1 || total_bins < 1) return 0;
    return ws_need(total_bins);
}

adc_status adc_batched_hist_scan_fwd(const adc_instance *desc, int32_t count, const adc_work *items, int64_t n_items,
                                     int64_t total_bins, const int32_t *keys, const float *vals, float *hist,
                                     float *scan, int32_t *is, float *loss_parts, float *loss, int32_t smem_bins,
                                     void *ws, size_t ws_bytes, void *stream) {
    if (count < 1 || n_items < 0 || total_bins < 1 || smem_bins < 0) return ADC_ERR_INVALID_ARG;
    if (!al(desc, 8) || (n_items > 0 && (!al(items, 8) || !al(keys, 4) || !al(vals, 4))) || !al(hist, 4) ||
        !al(scan, 4) || !al(is, 4) || !al(loss_parts, 4) || !al(loss, 4))
        return ADC_ERR_INVALID_ARG;
    if (!al(ws, 256)) return ADC_ERR_INVALID_ARG;
    if (ws_bytes < ws_need(total_bins)) return ADC_ERR_WORKSPACE;
    if (smem_bins == 0) smem_bins = kDefaultSmemBins;
    const size_t smem = (size_t)smem_bins * 8;
    if (smem > 200 * 1024) return ADC_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char *w = static_cast<char *>(ws);
    auto *tab = reinterpret_cast<unsigned long long *>(w + kWsHeader);
    if (cudaMemsetAsync(ws, 0, kWsHeader, s) != cudaSuccess) return ADC_ERR_CUDA;
    k_b_init<<<count, kBBinThreads, 0, s>>>(desc, hist, tab);
    if (n_items > 0) {
        int per_sm = (int)((224 * 1024) / (smem + 1024));
        per_sm = per_sm < 1 ? 1 : (per_sm > 4 ? 4 : per_sm);
        const unsigned grid = (unsigned)(num_sms() * per_sm);
        unsigned *ctr = counter_slot(ws, 0);
        auto run = [&](auto kern) -> bool {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
                return false;
            kern<<<grid, kBHistThreads, smem, s>>>(desc, items, n_items, keys, vals, hist, tab, (int32_t)smem, ctr);
            return true;
        };
        const bool ok = g_batched_ipt == 1 ? run(k_b_hist<1>) : g_batched_ipt == 8 ? run(k_b_hist<8>) : run(k_b_hist<4>);
        if (!ok) return ADC_ERR_CUDA;
    }
    k_b_scan_loss<<<count, kBScanThreads, 0, s>>>(desc, count, hist, tab, scan, is, loss_parts, loss, counter_slot(ws, 1));
    return check_launch();
}

adc_status adc_batched_hist_scan_vjp(const adc_instance *desc, int32_t count, const adc_work *items, int64_t n_items,
                                     int64_t total_bins, const int32_t *keys, const int32_t *is, const float *loss_bar,
                                     float *histbar, float *valsbar, void *ws, size_t ws_bytes, void *stream) {
    if (count < 1 || n_items < 0 || total_bins < 1) return ADC_ERR_INVALID_ARG;
    if (!al(desc, 8) || (n_items > 0 && (!al(items, 8) || !al(keys, 4) || !al(valsbar, 4))) || !al(is, 4) ||
        !al(loss_bar, 4) || !al(histbar, 4))
        return ADC_ERR_INVALID_ARG;
    if (!al(ws, 256)) return ADC_ERR_INVALID_ARG;
    if (ws_bytes < kWsHeader) return ADC_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(ws, 0, kWsHeader, s) != cudaSuccess) return ADC_ERR_CUDA;
    if (n_items > 0)
        k_b_vjp_items<<<num_sms() * 4, kBHistThreads, 0, s>>>(desc, items, n_items, keys, loss_bar, valsbar,
                                                              counter_slot(ws, 2));
    k_b_hbar_scatter<<<count, kBBinThreads, 0, s>>>(desc, is, loss_bar, histbar, valsbar);
    return check_launch();
}

}  // extern "C"

extern "C" void adc_debug_set_batched_items(int items) {
    g_batched_ipt = (items == 1 || items == 4) ? items : 8;
}
