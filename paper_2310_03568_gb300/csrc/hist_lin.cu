// General reduce_by_index for the non-commutative linFnComp operator with up
// to a few thousand bins (Sec. 4.1, Fig. 4).  The paper sorts the elements by
// bin (stable) and runs segmented scans over the sorted values; what those
// scans compute per element is the fold of its bin's values before it (l_i)
// and after it (r_i), in index order.  Here no element is moved:
//   1. per chunk of kLThreads * R elements (one block; warp w owns the w-th
//      run of 32 * R consecutive elements, R rounds of 32): every warp walks
//      its run in index order and folds each element into its bin's entry of
//      a warp-private table in shared memory.  Within a round, lanes holding
//      the same bin update one after another in lane order, so every bin's
//      entry is the ordered fold of the run's values; the block then composes
//      the warp tables per bin in warp order -> P[chunk][bin] (identity where
//      the bin is absent);
//   2. per bin, its column of P in chunk order: the exclusive prefix
//      L[c][bin] = hist0 . P[0..c-1][bin], the c's product of the exclusive
//      suffix Rc[c][bin], hist and the bin total A (for hist0bar);
//   3. vjp, per chunk: the forward walk again, keeping each element's
//      exclusive prefix p_i within its warp run, and a backward walk (the
//      forward one's lane ranks, reversed) keeping the product s_i of the c's
//      after it; per bin and warp the block forms what lies before the run
//      (L . earlier runs) and the product of the c's after it (later runs,
//      Rc), and every element gets
//      vbar_i = d(l_i . v_i . r_i)/dv_i ^T histbar[k_i] with l_i = before . p_i
//      and r_i.c = s_i * after.c.
// Within every bin the values meet in index order, as the sequential
// definition requires; only the bracketing differs (associativity).
// Traffic: the forward reads keys and values once (12 B per fp32 element) and
// moves the [chunks][m] matrices (P and L 8 B, Rc 4 B per bin and chunk); the
// vjp reads keys, values, L and Rc and writes the adjoints once.  Bound by the
// latency of the walks' shared-memory steps, at 16 to 24 warps per SM (the
// tables fill the shared memory).  n = 1e7, m = 1000, fp32: fold 0.074 -> 0.049
// ms (ranks found by ballots a round ahead instead of a match in the update's
// way), columns 0.037 -> 0.029 ms and vjp 0.189 -> 0.111 ms (ranks reused
// backwards, chunk-major matrices, no votes in the walks).
#include "common.cuh"
#include "hist_common.cuh"
#include "internal.h"

namespace adc {

constexpr int kLThreads = 256;
constexpr int kLWarps = kLThreads / kWarp;
// The vjp's shared memory (per-warp tables of (b, c) and of c, histbar) fits
// one block up to 2047 bins (fp32) / 1023 bins (fp64).
template <typename T> constexpr int64_t lmax_bins() { return sizeof(T) == 4 ? 2047 : 1023; }
template <typename T> struct LChunk {
    static constexpr int kRounds = sizeof(T) == 4 ? 16 : 8;  // rounds of 32 elements per warp
    static constexpr int kRun = kWarp * kRounds;             // elements per warp
    static constexpr int kSize = kLThreads * kRounds;        // elements per chunk (block)
};

template <typename T> __device__ __forceinline__ Pair<T> lf(const Pair<T> &a, const Pair<T> &b) {
    return {b.b + b.c * a.b, b.c * a.c};  // (b1,c1) . (b2,c2) = (b2 + c2*b1, c2*c1)
}
template <typename T> __device__ __forceinline__ Pair<T> lf_id() { return {T(0), T(1)}; }
// d(l . v . r)/dv ^T g for linFnComp
template <typename T> __device__ __forceinline__ Pair<T> lf_adj(const Pair<T> &l, const Pair<T> &r, const Pair<T> &g) {
    return {r.c * g.b, r.c * (l.b * g.b + l.c * g.c)};
}

// One (b, c) element as one 8- or 16-byte streaming load (the array is
// 16-byte aligned, so every element is aligned to its size).
__device__ __forceinline__ Pair<float> ld_pair(const Pair<float> *p) {
    const float2 t = __ldcs(reinterpret_cast<const float2 *>(p));
    return {t.x, t.y};
}
__device__ __forceinline__ Pair<double> ld_pair(const Pair<double> *p) {
    const double2 t = __ldcs(reinterpret_cast<const double2 *>(p));
    return {t.x, t.y};
}

// One warp run of a chunk: keys (-1 past n) and values, round r at element
// base + r * 32 + lane, every load issued before the first use.
template <typename T, int R>
__device__ __forceinline__ void load_run(const int32_t *__restrict__ keys, const Pair<T> *__restrict__ vals,
                                         int64_t base, int64_t n, int m, int32_t (&k)[R], Pair<T> (&v)[R]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = base + r * kWarp + lane;
        k[r] = i < n ? __ldcs(keys + i) : -1;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = base + r * kWarp + lane;
        v[r] = in_range(k[r], m) ? ld_pair(vals + i) : lf_id<T>();
    }
}

// Which lanes of a round share a bin, found one round ahead of the walk so that
// the table update of one round and the search of the next overlap.  Every
// lane with an in-range key writes its lane number to its key's byte in `tag`
// (one byte per bin and warp); the lanes that do not read their own number
// back share a bin with another lane.  Few of them (the usual case: about two
// rounds in five at m = 1000 have one pair): each such key is broadcast and
// balloted; many: __match_any_sync, whose cost does not grow with them but is
// several times one ballot's.  Warp-wide: all lanes call tag_write / ranks.
struct LRank {
    uint8_t rank, cnt;  // the lane's place among the lanes with its bin (lane order), and their number
};
__device__ __forceinline__ void tag_write(int32_t key, bool ok, uint8_t *tag) {
    if (ok) tag[key] = (uint8_t)(threadIdx.x & 31);
}
// After a __syncwarp() that follows tag_write(); the lanes of the fullest bin
// (1: no two share one), found here once rather than by a vote before every step.
__device__ __forceinline__ int ranks(int32_t key, bool ok, const uint8_t *tag, LRank &r) {
    const int lane = threadIdx.x & 31;
    unsigned lost = __ballot_sync(0xffffffffu, ok && tag[key] != (uint8_t)lane);
    r = {0, 1};
    if (lost == 0u) return 1;
    int steps = 1;
    unsigned peers = 1u << lane;
    if (__popc(lost) <= 4) {
        while (lost) {
            const int32_t k = __shfl_sync(0xffffffffu, key, __ffs(lost) - 1);
            const unsigned same = __ballot_sync(0xffffffffu, ok && key == k);
            if (ok && key == k) peers = same;
            steps = __popc(same) > steps ? __popc(same) : steps;
            lost &= ~same;
        }
    } else {
        peers = __match_any_sync(0xffffffffu, ok ? key : -1);
        if (!ok) peers = 1u << lane;
        steps = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(peers));
    }
    r.rank = (uint8_t)__popc(peers & ((1u << lane) - 1u));
    r.cnt = (uint8_t)__popc(peers);
    return steps;
}
// One round's updates: upd() runs for every lane with an in-range key, at once
// when no two share a bin, else in rank order, in as many steps as the fullest
// bin has lanes.  Two steps are the usual case and stand outside the loop; with
// one bin there are 32, where a vote before each step was what the walk did
// (n = 1e7: m = 1 forward 0.195 -> 0.134 ms, vjp 0.442 -> 0.310; m = 400 vjp
// 0.105 -> 0.096; m = 1000 0.122 -> 0.111).  The loop is unrolled by two: by four,
// 32 copies of it in the vjp are too much code (m = 31 to 1000 5% to 9% slower),
// and rolled, m = 1 takes 0.152 and 0.386 ms.
template <class F> __device__ __forceinline__ void ranked_update(int steps, bool ok, int rank, F &&upd) {
    if (steps == 1) {
        if (ok) upd();
        return;
    }
    if (ok && rank == 0) upd();
    __syncwarp();
    if (ok && rank == 1) upd();
    __syncwarp();
#pragma unroll 2
    for (int q = 2; q < steps; ++q) {
        if (ok && rank == q) upd();
        __syncwarp();
    }
}

// ------------------------------------------------------------ chunk fold --
// P[chunk * m + bin] = ordered fold of the chunk's values of that bin.
template <typename T>
__global__ void __launch_bounds__(kLThreads)
k_linh_fold(const int32_t *__restrict__ keys, const Pair<T> *__restrict__ vals, const int64_t n, const int m,
            Pair<T> *__restrict__ P) {
    using C = LChunk<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Pair<T> *s_tab = reinterpret_cast<Pair<T> *>(smem_raw);              // [kLWarps][m]
    uint8_t *s_tag = reinterpret_cast<uint8_t *>(s_tab + (size_t)kLWarps * m);  // [kLWarps][m]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t c = blockIdx.x;
    Pair<T> *tab = s_tab + (size_t)warp * m;
    uint8_t *tag = s_tag + (size_t)warp * m;
    int32_t k[C::kRounds];
    Pair<T> v[C::kRounds];
    load_run<T, C::kRounds>(keys, vals, c * C::kSize + (int64_t)warp * C::kRun, n, m, k, v);
    for (int j = lane; j < m; j += kWarp) tab[j] = lf_id<T>();
    __syncwarp();
    LRank rk;
    tag_write(k[0], in_range(k[0], m), tag);
    __syncwarp();
    int steps = ranks(k[0], in_range(k[0], m), tag, rk);
#pragma unroll
    for (int r = 0; r < C::kRounds; ++r) {
        const int32_t key = k[r];
        const Pair<T> x = v[r];
        const int nx = r + 1 < C::kRounds ? r + 1 : r;
        if (r + 1 < C::kRounds) tag_write(k[nx], in_range(k[nx], m), tag);
        ranked_update(steps, in_range(key, m), rk.rank, [&] { tab[key] = lf(tab[key], x); });
        __syncwarp();
        if (r + 1 < C::kRounds) steps = ranks(k[nx], in_range(k[nx], m), tag, rk);
    }
    __syncthreads();
    for (int j = tid; j < m; j += kLThreads) {
        Pair<T> acc = s_tab[j];
#pragma unroll
        for (int w = 1; w < kLWarps; ++w) acc = lf(acc, s_tab[(size_t)w * m + j]);
        P[c * m + j] = acc;
    }
}

// ---------------------------------------------------------- bin columns --
// L[c][j] (what lies before chunk c in bin j: hist0 . P[0..c-1][j]), Rc[c][j]
// (the product of the c's after it; the vjp needs no more of the suffix),
// hist[j] and the bin total A[j], from the columns P[.][j].  The matrices are
// chunk-major, so that the chunk kernels read and write them in order
// (bin-major, each of a chunk's 8-byte cells was a sector of its own).  A block
// takes kColBins bins -- 64 contiguous bytes of a row -- and cuts their columns
// into kColSegs segments, one thread each: fold the segment, scan the segments
// (one warp per bin), walk it again forwards for L and backwards for Rc (both
// walks read from L2).  Bound by the latency of the loads, kColRows rows at a
// time, so with few bins and many chunks, where the bins alone are a handful of
// blocks, the rows are split over further blocks too (grid.y), behind a pass
// that folds each block's rows: col_splits().  Forward at n = 1e8: m = 4 0.838 ->
// 0.529 ms, m = 31 0.690 -> 0.512, m = 100 0.598 -> 0.404 (together with the
// walks' counted steps); m = 1000 has blocks enough.
constexpr int kColBins = 8;
constexpr int kColSegs = kLThreads / kColBins;
constexpr int kColRows = 8;  // loads in flight
static_assert(kColSegs == kWarp && kColBins == kLWarps, "a warp scans one bin's segments");

// One thread's segment: rows [c0, c1) of the block's rows [r0, r1), and its fold.
template <typename T> struct ColSegment {
    int64_t c0, c1;
    Pair<T> fold;
    __device__ ColSegment(const Pair<T> *col, int64_t m, int64_t r0, int64_t r1, int sg, bool live) {
        int64_t per = (r1 - r0 + kColSegs - 1) / kColSegs;
        if (per < kColRows) per = kColRows;
        c0 = r0 + sg * per < r1 ? r0 + sg * per : r1;
        c1 = c0 + per < r1 ? c0 + per : r1;
        fold = lf_id<T>();
        if (!live) return;
        for (int64_t c = c0; c < c1; c += kColRows) {
            Pair<T> x[kColRows];
#pragma unroll
            for (int u = 0; u < kColRows; ++u) x[u] = c + u < c1 ? col[(c + u) * m] : lf_id<T>();
#pragma unroll
            for (int u = 0; u < kColRows; ++u) fold = lf(fold, x[u]);
        }
    }
};

// Inclusive scan of a warp's states in lane order.
template <typename T> __device__ __forceinline__ Pair<T> lf_warp_scan(Pair<T> v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const Pair<T> up = shfl_up(v, o);
        if (lane >= o) v = lf(up, v);
    }
    return v;
}

// F[split][j]: the fold of the split's rows of bin j.
template <typename T>
__global__ void __launch_bounds__(kLThreads)
k_linh_colfold(const Pair<T> *__restrict__ P, const int64_t nc, const int64_t m, const int64_t rows,
               Pair<T> *__restrict__ F) {
    __shared__ Pair<T> s_fold[kColBins][kColSegs + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = threadIdx.x % kColBins, sg = threadIdx.x / kColBins;
    const int64_t j0 = (int64_t)blockIdx.x * kColBins, r0 = blockIdx.y * rows, r1 = r0 + rows < nc ? r0 + rows : nc;
    const ColSegment<T> seg(P + j0 + b, m, r0, r1, sg, j0 + b < m);
    s_fold[b][sg] = seg.fold;
    __syncthreads();
    const Pair<T> all = lf_warp_scan(s_fold[warp][lane]);
    if (lane == kWarp - 1 && j0 + warp < m) F[blockIdx.y * m + j0 + warp] = all;
}

template <typename T>
__global__ void __launch_bounds__(kLThreads)
k_linh_cols(const Pair<T> *__restrict__ P, const Pair<T> *__restrict__ h0, const int64_t nc, const int64_t m,
            const int64_t rows, const Pair<T> *__restrict__ F, Pair<T> *__restrict__ L, T *__restrict__ Rc,
            Pair<T> *__restrict__ hist, Pair<T> *__restrict__ A) {
    __shared__ Pair<T> s_fold[kColBins][kColSegs + 1];  // the segments' folds, then what lies before them
    __shared__ T s_after[kColBins][kColSegs + 1];       // the product of the c's after them
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = threadIdx.x % kColBins, sg = threadIdx.x / kColBins;
    const int64_t j0 = (int64_t)blockIdx.x * kColBins, j = j0 + b;
    const bool live = j < m;
    const int64_t r0 = blockIdx.y * rows, r1 = r0 + rows < nc ? r0 + rows : nc;
    const Pair<T> *col = P + j;
    const ColSegment<T> seg(col, m, r0, r1, sg, live);
    s_fold[b][sg] = seg.fold;
    __syncthreads();
    {
        const int64_t jw = j0 + warp;  // the warp's bin
        // the rows of the other splits: the fold of the earlier ones, the c's of the later ones
        Pair<T> pre = lf_id<T>();
        T post = T(1);
        for (int q0 = 0; q0 < (int)gridDim.y && gridDim.y > 1; q0 += kWarp) {
            const int q = q0 + lane;
            const Pair<T> x = q < (int)gridDim.y && jw < m ? F[q * m + jw] : lf_id<T>();
            const Pair<T> inc = lf_warp_scan(q < (int)blockIdx.y ? x : lf_id<T>());
            pre = lf(pre, shfl_idx(inc, kWarp - 1));
            T c = q > (int)blockIdx.y ? x.c : T(1);
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) c *= __shfl_xor_sync(0xffffffffu, c, o);
            post *= c;
        }
        const Pair<T> own = s_fold[warp][lane], inc = lf_warp_scan(own);
        Pair<T> ex = shfl_up(inc, 1);
        T suf = own.c;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const T dn = __shfl_down_sync(0xffffffffu, suf, o);
            if (lane + o < kWarp) suf = dn * suf;
        }
        T after = __shfl_down_sync(0xffffffffu, suf, 1);
        if (lane == 0) ex = lf_id<T>();
        if (lane == kWarp - 1) after = T(1);
        s_fold[warp][lane] = lf(pre, ex);
        s_after[warp][lane] = post * after;
        if (lane == kWarp - 1 && blockIdx.y == gridDim.y - 1 && jw < m) {
            const Pair<T> all = lf(pre, inc);
            A[jw] = all;
            hist[jw] = h0 ? lf(h0[jw], all) : all;
        }
    }
    __syncthreads();
    if (!live) return;
    Pair<T> run = h0 ? lf(h0[j], s_fold[b][sg]) : s_fold[b][sg];
    T after = s_after[b][sg];
    for (int64_t c = seg.c0; c < seg.c1; c += kColRows) {
        Pair<T> x[kColRows];
#pragma unroll
        for (int u = 0; u < kColRows; ++u) x[u] = c + u < seg.c1 ? col[(c + u) * m] : lf_id<T>();
#pragma unroll
        for (int u = 0; u < kColRows; ++u)
            if (c + u < seg.c1) {
                L[(c + u) * m + j] = run;
                run = lf(run, x[u]);
            }
    }
    for (int64_t c = seg.c1; c > seg.c0; c -= kColRows) {
        T x[kColRows];
#pragma unroll
        for (int u = 0; u < kColRows; ++u) x[u] = c - 1 - u >= seg.c0 ? col[(c - 1 - u) * m].c : T(1);
#pragma unroll
        for (int u = 0; u < kColRows; ++u)
            if (c - 1 - u >= seg.c0) {
                Rc[(c - 1 - u) * m + j] = after;
                after = x[u] * after;
            }
    }
}

// Splits of the rows: so many that the blocks fill the SMs once, each with a
// full step of every thread's loads at least, and none where the bins alone are
// a block for every second SM.
static int64_t col_splits(int64_t nc, int64_t m) {
    const int64_t blocks = (m + kColBins - 1) / kColBins, want = num_sms() / blocks;
    const int64_t most = nc / (kColSegs * kColRows);
    return want < 2 || most < 2 ? 1 : want < most ? want : most;
}

// ------------------------------------------------------------------- vjp --
template <typename T>
__global__ void __launch_bounds__(kLThreads, 2)
k_linh_vjp(const int32_t *__restrict__ keys, const Pair<T> *__restrict__ vals, const int64_t n, const int m,
           const Pair<T> *__restrict__ L, const T *__restrict__ Rc, const Pair<T> *__restrict__ hb,
           Pair<T> *__restrict__ vbar, const int accumulate) {
    using C = LChunk<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Pair<T> *s_tab = reinterpret_cast<Pair<T> *>(smem_raw);  // [kLWarps][m]: folds, then (before . g, after.c)
    Pair<T> *s_g = s_tab + (size_t)kLWarps * m;              // [m] histbar
    T *s_q = reinterpret_cast<T *>(s_g + m);                  // [kLWarps][m] products of c (backward walk)
    uint8_t *s_tag = reinterpret_cast<uint8_t *>(s_q + (size_t)kLWarps * m);  // [kLWarps][m]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t c = blockIdx.x;
    const int64_t base = c * C::kSize + (int64_t)warp * C::kRun;
    Pair<T> *tab = s_tab + (size_t)warp * m;
    T *qt = s_q + (size_t)warp * m;
    uint8_t *tag = s_tag + (size_t)warp * m;
    int32_t k[C::kRounds];
    Pair<T> v[C::kRounds];
    load_run<T, C::kRounds>(keys, vals, base, n, m, k, v);
    for (int j = lane; j < m; j += kWarp) {
        tab[j] = lf_id<T>();
        qt[j] = T(1);
    }
    for (int j = tid; j < m; j += kLThreads) s_g[j] = hb[j];
    __syncwarp();
    // forward walk: p_i = the run's fold of i's bin before i; the ranks are kept
    // for the backward walk, where the order is reversed
    Pair<T> p[C::kRounds];
    LRank rk[C::kRounds];
    uint32_t steps[C::kRounds / 4] = {};  // a byte for each round (uniform)
    tag_write(k[0], in_range(k[0], m), tag);
    __syncwarp();
    steps[0] = (uint32_t)ranks(k[0], in_range(k[0], m), tag, rk[0]);
#pragma unroll
    for (int r = 0; r < C::kRounds; ++r) {
        const int32_t key = k[r];
        const Pair<T> x = v[r];
        const int nx = r + 1 < C::kRounds ? r + 1 : r;
        if (r + 1 < C::kRounds) tag_write(k[nx], in_range(k[nx], m), tag);
        Pair<T> pr = lf_id<T>();
        ranked_update((int)((steps[r / 4] >> (8 * (r % 4))) & 255u), in_range(key, m), rk[r].rank, [&] {
            pr = tab[key];
            tab[key] = lf(pr, x);
        });
        p[r] = pr;
        __syncwarp();
        if (r + 1 < C::kRounds)
            steps[nx / 4] |= (uint32_t)ranks(k[nx], in_range(k[nx], m), tag, rk[nx]) << (8 * (nx % 4));
    }
    // backward walk: s_i = product of the c's of i's bin after i in the run
    T sv[C::kRounds];
#pragma unroll
    for (int r = C::kRounds - 1; r >= 0; --r) {
        const int32_t key = k[r];
        const T xc = v[r].c;
        T sr = T(1);
        ranked_update((int)((steps[r / 4] >> (8 * (r % 4))) & 255u), in_range(key, m), rk[r].cnt - 1 - rk[r].rank, [&] {
            sr = qt[key];
            qt[key] = xc * sr;
        });
        sv[r] = sr;
        __syncwarp();
    }
    __syncthreads();
    // per bin and warp run: u = <L . earlier runs, g> and the product of the
    // c's after the run (later runs, then R)
    for (int j = tid; j < m; j += kLThreads) {
        const Pair<T> g = s_g[j];
        Pair<T> before = L[c * m + j];
        T fc[kLWarps], u[kLWarps];
#pragma unroll
        for (int w = 0; w < kLWarps; ++w) {
            const Pair<T> f = s_tab[(size_t)w * m + j];
            u[w] = g.b * before.b + g.c * before.c;
            fc[w] = f.c;
            before = lf(before, f);
        }
        T after = Rc[c * m + j];
#pragma unroll
        for (int w = kLWarps - 1; w >= 0; --w) {
            s_tab[(size_t)w * m + j] = Pair<T>{u[w], after};
            after = fc[w] * after;
        }
    }
    __syncthreads();
    // vbar_i = (rc g.b, rc <l_i, g>) with l_i = before . p_i, rc = s_i * after
#pragma unroll
    for (int r = 0; r < C::kRounds; ++r) {
        const int64_t i = base + r * kWarp + lane;
        if (i >= n) continue;
        Pair<T> out{T(0), T(0)};
        if (in_range(k[r], m)) {
            const Pair<T> ua = tab[k[r]];
            const Pair<T> g = s_g[k[r]];
            const T rc = sv[r] * ua.c;
            out = Pair<T>{rc * g.b, rc * (g.b * p[r].b + p[r].c * ua.b)};
        }
        if (accumulate) {
            const Pair<T> o = vbar[i];
            out = Pair<T>{o.b + out.b, o.c + out.c};
        }
        vbar[i] = out;
    }
}

// hist0bar[j] (+)= d(hist0 . A)/d hist0 ^T histbar[j] = A.c * histbar[j]
template <typename T>
__global__ void k_linh_h0bar(const Pair<T> *__restrict__ A, const Pair<T> *__restrict__ hb, Pair<T> *__restrict__ h0b,
                             const int64_t m, const int accumulate) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const Pair<T> g = lf_adj(lf_id<T>(), A[j], hb[j]);
        h0b[j] = accumulate ? Pair<T>{h0b[j].b + g.b, h0b[j].c + g.c} : g;
    }
}

// -------------------------------------------------------------------- host --
template <typename T> static int64_t num_chunks(int64_t n) {
    const int64_t c = (n + LChunk<T>::kSize - 1) / LChunk<T>::kSize;
    return c > 0 ? c : 1;
}

struct LinLayout {
    size_t P, ws_bytes;                  // workspace
    size_t L, R, A, saved_bytes;         // residuals
};

template <typename T> static LinLayout lin_layout(int64_t n, int64_t m) {
    LinLayout o;
    const int64_t nc = num_chunks<T>(n);
    const size_t cells = (size_t)m * (size_t)nc * sizeof(Pair<T>);
    o.P = kWsHeader;
    o.ws_bytes = align_up(kWsHeader + cells, 256);
    o.L = 0;
    o.R = align_up(cells, 256);
    o.A = 2 * align_up(cells, 256);
    o.saved_bytes = o.A + align_up((size_t)m * sizeof(Pair<T>), 256);
    return o;
}

bool linh_applicable(adc_dtype dt, int64_t m) {
    return m >= 1 && m <= (dt == ADC_F64 ? lmax_bins<double>() : lmax_bins<float>());
}

size_t linh_ws_bytes(adc_dtype dt, int64_t n, int64_t m) {
    return dt == ADC_F64 ? lin_layout<double>(n, m).ws_bytes : lin_layout<float>(n, m).ws_bytes;
}
size_t linh_saved_bytes(adc_dtype dt, int64_t n, int64_t m) {
    return dt == ADC_F64 ? lin_layout<double>(n, m).saved_bytes : lin_layout<float>(n, m).saved_bytes;
}

template <typename T> static size_t fold_smem(int64_t m) { return (size_t)kLWarps * m * (sizeof(Pair<T>) + 1); }
template <typename T> static size_t vjp_smem(int64_t m) {
    return (size_t)(kLWarps + 1) * m * sizeof(Pair<T>) + (size_t)kLWarps * m * (sizeof(T) + 1);
}

template <typename T>
static adc_status linh_fwd_t(int64_t n, int64_t m, const int32_t *keys, const Pair<T> *vals, const Pair<T> *h0,
                             Pair<T> *hist, void *saved, void *ws, cudaStream_t s) {
    const LinLayout Lo = lin_layout<T>(n, m);
    const int64_t nc = num_chunks<T>(n);
    char *sv = static_cast<char *>(saved);
    Pair<T> *P = reinterpret_cast<Pair<T> *>(static_cast<char *>(ws) + Lo.P);
    const size_t smem = fold_smem<T>(m);
    if (cudaFuncSetAttribute(k_linh_fold<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return ADC_ERR_CUDA;
    k_linh_fold<T><<<(unsigned)nc, kLThreads, smem, s>>>(keys, vals, n, (int)m, P);
    const int64_t blocks = (m + kColBins - 1) / kColBins, want = col_splits(nc, m);
    const int64_t rows = (nc + want - 1) / want, splits = (nc + rows - 1) / rows;
    const dim3 grid((unsigned)blocks, (unsigned)splits);
    T *Rc = reinterpret_cast<T *>(sv + Lo.R);
    // (the upper half of the residuals' Rc is free, and a split has at least two rows)
    Pair<T> *F = reinterpret_cast<Pair<T> *>(sv + Lo.R + align_up((size_t)m * nc * sizeof(T), 16));
    if (splits > 1) k_linh_colfold<T><<<grid, kLThreads, 0, s>>>(P, nc, m, rows, F);
    k_linh_cols<T><<<grid, kLThreads, 0, s>>>(P, h0, nc, m, rows, F, reinterpret_cast<Pair<T> *>(sv + Lo.L), Rc, hist,
                                              reinterpret_cast<Pair<T> *>(sv + Lo.A));
    return check_launch();
}

template <typename T>
static adc_status linh_vjp_t(int64_t n, int64_t m, const int32_t *keys, const Pair<T> *vals, const void *saved,
                             const Pair<T> *hb, Pair<T> *vb, Pair<T> *h0b, int acc, cudaStream_t s) {
    const LinLayout Lo = lin_layout<T>(n, m);
    const int64_t nc = num_chunks<T>(n);
    const char *sv = static_cast<const char *>(saved);
    const Pair<T> *L = reinterpret_cast<const Pair<T> *>(sv + Lo.L);
    const T *R = reinterpret_cast<const T *>(sv + Lo.R);
    const Pair<T> *A = reinterpret_cast<const Pair<T> *>(sv + Lo.A);
    if (n > 0) {
        const size_t smem = vjp_smem<T>(m);
        if (cudaFuncSetAttribute(k_linh_vjp<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return ADC_ERR_CUDA;
        k_linh_vjp<T><<<(unsigned)nc, kLThreads, smem, s>>>(keys, vals, n, (int)m, L, R, hb, vb, acc);
    }
    if (h0b) {
        const int64_t g = (m + 255) / 256;
        k_linh_h0bar<T><<<(unsigned)(g < 1024 ? g : 1024), 256, 0, s>>>(A, hb, h0b, m, acc);
    }
    return check_launch();
}

adc_status linh_fwd(adc_dtype dt, int64_t n, int64_t m, const int32_t *keys, const void *vals, const void *hist0,
                    void *hist, void *saved, void *ws, cudaStream_t s) {
    if (dt == ADC_F64)
        return linh_fwd_t<double>(n, m, keys, static_cast<const Pair<double> *>(vals),
                                  static_cast<const Pair<double> *>(hist0), static_cast<Pair<double> *>(hist), saved,
                                  ws, s);
    return linh_fwd_t<float>(n, m, keys, static_cast<const Pair<float> *>(vals), static_cast<const Pair<float> *>(hist0),
                             static_cast<Pair<float> *>(hist), saved, ws, s);
}

adc_status linh_vjp(adc_dtype dt, int64_t n, int64_t m, const int32_t *keys, const void *vals, const void *saved,
                    const void *histbar, void *valsbar, void *hist0bar, int accumulate, cudaStream_t s) {
    if (dt == ADC_F64)
        return linh_vjp_t<double>(n, m, keys, static_cast<const Pair<double> *>(vals), saved,
                                  static_cast<const Pair<double> *>(histbar), static_cast<Pair<double> *>(valsbar),
                                  static_cast<Pair<double> *>(hist0bar), accumulate, s);
    return linh_vjp_t<float>(n, m, keys, static_cast<const Pair<float> *>(vals), saved,
                             static_cast<const Pair<float> *>(histbar), static_cast<Pair<float> *>(valsbar),
                             static_cast<Pair<float> *>(hist0bar), accumulate, s);
}

}  // namespace adc
