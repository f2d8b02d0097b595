// Streaming single-pass scan: persistent blocks, one per SM, every input byte
// read from DRAM once, every output byte written once.
//
// Tiles are claimed one at a time from an atomic counter (claim order = logical
// order, so a tile only ever waits on tiles of running blocks) and travel
// through a ring of STAGES shared-memory buffers:
//   load      cp.async, 16 bytes per lane; every warp copies its own segment,
//             so a load needs no block barrier; AHEAD tiles in flight;
//   fold      every thread folds its row of RB contiguous bytes, one warp scan
//             gives its exclusive prefix in the warp, and the warps' totals go
//             to the publishing warp, which publishes the tile's aggregate
//             (tagged words) and claims the next tile;
//   look-back a warp of its own extends the block's running prefix -- the
//             exclusive prefix of its previous tile -- by the aggregates of that
//             tile and of the tiles that other blocks claimed in between.  No
//             inclusive prefixes are published: the aggregates of a round are
//             published at about the same time, so one poll finds most of them,
//             and there is no chain from block to block;
//   store     every thread rescans its row from its prefix, writes the results
//             over the stage, and the warp writes its segment out in 512-byte
//             runs.
// What bounds it: the time from a tile's fold to its prefix, about 4 us at full
// bandwidth, during which its inputs wait in shared memory.  With one input
// array six 32 KB stages cover it (n = 1e8 fp32 + forward 0.136 ms, 0.87 of the
// 6.8 TB/s copy rate; the range engine, which reads the input twice, 0.215);
// with three arrays four 48 KB stages do not (lin vjp 0.633 ms, 0.74; 0.764).
// Hence: four copies of the aggregates, so that fewer blocks poll the same
// lines (lin vjp 0.90 -> 0.72 ms before the roles were split); claims at the
// pace of the folds (claimed in bursts, a block folds neighbouring tiles a
// round apart and everything behind them waits); one reader that scans the
// aggregates for everyone, two hops instead of one, took 0.150 ms, and more
// look-back warps or pauses between polls were slower too.  Waits between warps
// are mbarriers; all waits are bounded.
//
// Rows are RB = 64 or 128 bytes; 16-byte chunk c of row r sits at chunk
// c ^ swz(r), so that the row walks (one row per lane) and the copies (one
// 512-byte run per warp) are both free of bank conflicts.
//
// Besides the scan interface of scan_engine.cuh an Op provides
//   Elem, kStreams, stream(s)   the input arrays;  dst()  the output array
//   Scalar, accumulating()      out += results, per scalar
//   pad(s)                      element s beyond the ends (its item is the identity)
//   kWalk 0: item(v)            state of element i;     out(run, i)
//   kWalk 1: item(a, xn)        a = stream 0 at i, xn = stream 1 at i + 1;
//            out(run, yp)       yp = stream 2 at i - 1
//   kWalk 2: item(a, y, yn, i, n), out(run, y, yp, i)   a = stream 0, y = stream 1
//   kExact (0 if absent)        which fp32 roundings are carried along, below
#pragma once

#include <cfloat>
#include <string.h>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "scan_engine.cuh"
#include "tma.cuh"

namespace adc {

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <class Op, int NWC, int RB, int STAGES> struct StreamShape {
    using E = typename Op::Elem;
    static_assert(sizeof(E) <= 16 && (RB == 64 || RB == 128), "a unit holds whole elements; row_swizzle()");
    static constexpr int U = 16;                                    // bytes loaded at once by a row walk
    static constexpr int NPU = U / (int)sizeof(E);                  // elements in them
    static constexpr int UR = RB / U;                               // and how many to a row
    static constexpr int C = RB / 16;                               // 16-byte chunks per row
    static constexpr int EPR = RB / (int)sizeof(E);                 // elements per row (thread)
    static constexpr int SEG = 32 * RB;                             // a warp's bytes of one stream
    static constexpr int SEGP = SEG + 2 * U;                        // and one unit on each side (halos)
    static constexpr int NS = Op::kStreams;
    static constexpr int TILE = NWC * 32 * EPR;                     // elements
    static constexpr size_t kData = (size_t)NWC * NS * SEGP;               // one stage's streams
    static constexpr size_t kEx = (size_t)NWC * 32 * sizeof(typename Op::State);  // its rows' in-warp prefixes
    static constexpr size_t kSmem = STAGES * (kData + kEx);
    static int64_t tiles(int64_t n) { return (n + TILE - 1) / TILE; }
};

template <int RB> __device__ __forceinline__ int row_swizzle(int row) {
    return RB == 128 ? (row & 7) : ((row >> 1) & 3);
}

// One warp's segment of one stream in a stage.
template <class Sh, int RB> struct Segment {
    using E = typename Sh::E;
    unsigned char *p;
    __device__ __forceinline__ unsigned char *chunk(int row, int c) const {
        return p + row * RB + ((c ^ row_swizzle<RB>(row)) << 4);
    }
    __device__ __forceinline__ void load(int row, int u, E (&v)[Sh::NPU]) const {
        const uint4 t = *reinterpret_cast<const uint4 *>(chunk(row, u));
        memcpy(v, &t, 16);
    }
    __device__ __forceinline__ void store(int row, int u, const E (&v)[Sh::NPU]) const {
        uint4 t;
        memcpy(&t, v, 16);
        *reinterpret_cast<uint4 *>(chunk(row, u)) = t;
    }
    // first element of the row after `row`, last element of the row before it
    __device__ __forceinline__ E after(int row) const {
        E v[Sh::NPU];
        if (row == 31) memcpy(v, p + Sh::SEG, Sh::U);
        else load(row + 1, 0, v);
        return v[0];
    }
    __device__ __forceinline__ E before(int row) const {
        E v[Sh::NPU];
        if (row == 0) memcpy(v, p + Sh::SEG + Sh::U, Sh::U);
        else load(row - 1, Sh::UR - 1, v);
        return v[Sh::NPU - 1];
    }
};

// Copies the 16 bytes at byte offset b of an array of nb bytes into shared
// memory: asynchronously when they lie inside it, else element by element
// with `pad` outside.
template <typename E>
__device__ __forceinline__ void copy16(unsigned char *dst, const E *src, int64_t b, int64_t nb, const E &pad) {
    if (b >= 0 && b + 16 <= nb) {
        cp_async16(dst, reinterpret_cast<const unsigned char *>(src) + b);
        return;
    }
    E v[16 / sizeof(E)];
#pragma unroll
    for (int k = 0; k < (int)(16 / sizeof(E)); ++k) {
        const int64_t at = b + k * (int64_t)sizeof(E);
        v[k] = (at >= 0 && at < nb) ? src[at / (int64_t)sizeof(E)] : pad;
    }
    uint4 t;
    memcpy(&t, v, 16);
    *reinterpret_cast<uint4 *>(dst) = t;
}

// fp32 roundings that are carried along (Op::kExact).
// kExactProduct: the state's coefficient coef(s) is the product of the elements'
// coefficients.  The relative error of a product is the sum of the roundings of
// all its multiplications, in whatever order they are done, so where a linear
// recurrence grows over tens of thousands of elements, 1e-6 to 6e-6 of the result
// was rounding.  A tile's fold keeps each multiplication's error (an FMA gives it)
// beside the coefficient, two FMAs per element, and rounds once per tile: 1e-7 to
// 8e-7 (lin, n = 1e6 to 1e8), for 3% to 10% of the vjps' time (n = 1e8 lin 0.612 ->
// 0.633 ms, * 0.293 -> 0.321; the range engine 0.764 and 0.41).  Without bringing
// the coefficient to the nearest after every combine, lin took 0.619 ms, but with
// errors up to 1.2e-6.
// kExactSum: the block's running prefix is extended once per round of tiles, at
// its own magnitude: 160 roundings over n = 1e8.  extend(hi, lo, d) sums up
// their errors beside it (sumOfProd n = 5e7: 5.7e-7 -> 2.4e-7, as without tiles).
// A coefficient or prefix that is not finite carries no error: NaN and
// infinities come out as without it.
enum { kExactNone = 0, kExactProduct = 1, kExactSum = 2 };
template <class Op, class = void> struct ExactOf : std::integral_constant<int, kExactNone> {};
template <class Op> struct ExactOf<Op, std::void_t<decltype(Op::kExact)>> : std::integral_constant<int, Op::kExact> {};

// hi += d, the rounding error added to lo (two-sum; Knuth, TAOCP 2, 4.2.2).
template <typename T> __device__ __forceinline__ void add_carry(T &hi, T &lo, T d) {
    const T a = hi, s = a + d, b = s - a;
    lo += (a - (s - b)) + (d - b);
    hi = s;
}

// A product that is rounded before it is used, never contracted into an FMA.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// What a tile's fold carries: the state, and its coefficient's error.
template <class Op, bool PRODUCT = ExactOf<Op>::value == kExactProduct> struct TileFold {
    using S = typename Op::State;
    using X = S;
    const Op &op;
    __device__ X identity() const { return op.identity(); }
    __device__ X step(const X &a, const S &x) const { return op.combine(a, x); }  // one more element
    __device__ X sealed(const X &a) const { return a; }                           // after the last one
    __device__ X combine(const X &a, const X &b) const { return op.combine(a, b); }
    __device__ static const S &state(const X &a) { return a; }
};
template <class Op> struct TileFold<Op, true> {
    using S = typename Op::State;
    struct X {
        S s;
        float e;
    };
    const Op &op;
    __device__ X identity() const { return {op.identity(), 0.f}; }
    __device__ X step(const X &a, const S &x) const {
        const float ac = Op::coef(a.s), xc = Op::coef(x), c = __fmul_rn(xc, ac);
        X r{op.combine(a.s, x), fmaf(xc, a.e, fmaf(xc, ac, -c))};
        Op::coef(r.s) = c;
        return r;
    }
    __device__ X sealed(X r) const {  // the coefficient to the nearest, what is left in e
        const float c = Op::coef(r.s), t = __fadd_rn(c, r.e);
        if (r.e != 0.f && fabsf(t) <= FLT_MAX) {
            Op::coef(r.s) = t;
            r.e = __fsub_rn(r.e, __fsub_rn(t, c));
        } else {
            r.e = 0.f;
        }
        return r;
    }
    __device__ X combine(const X &a, const X &b) const {
        X r = step(a, b.s);
        r.e = fmaf(b.e, Op::coef(a.s), r.e);
        return sealed(r);
    }
    __device__ static const S &state(const X &a) { return a.s; }
};

// The block's running prefix.
template <class Op, bool SUM = ExactOf<Op>::value == kExactSum> struct RunningPrefix {
    using S = typename Op::State;
    S run;
    __device__ explicit RunningPrefix(const Op &op) : run(op.identity()) {}
    __device__ void extend(const Op &op, const S &d) { run = op.combine(run, d); }
    __device__ S value() const { return run; }
};
template <class Op> struct RunningPrefix<Op, true> {
    using S = typename Op::State;
    S run, lo;
    __device__ explicit RunningPrefix(const Op &op) : run(op.identity()) { memset(&lo, 0, sizeof(S)); }
    __device__ void extend(const Op &op, const S &d) { op.extend(run, lo, d); }
    __device__ S value() const {
        S out;
        const float *h = reinterpret_cast<const float *>(&run), *l = reinterpret_cast<const float *>(&lo);
        float *o = reinterpret_cast<float *>(&out);
#pragma unroll
        for (int k = 0; k < (int)(sizeof(S) / 4); ++k) {
            const float t = __fadd_rn(h[k], l[k]);
            o[k] = fabsf(t) <= FLT_MAX ? t : h[k];
        }
        return out;
    }
};

// Folds the aggregates of tiles [from, to) in order onto *run (a whole warp;
// uniform result); false, alike in every lane, if a bounded wait ran out.
// Word k of tile t is aggw[k * stride + t].  Every lane polls its own words
// until they are there.  kLaneMajor = false: 32 consecutive tiles per load
// (256 contiguous bytes) and one ordered warp reduction for each of the Q
// loads, all in flight together; true: Q consecutive tiles per lane and one
// reduction in all -- for states whose combine is what costs (fp64 on this
// part's FP64 pipe: 0.090 -> 0.069 ms for the n = 1e7 * forward).  Handing the
// tiles over through shared memory to have both was slower for fp32 (0.148 ->
// 0.160 ms, n = 1e8 +): it lengthens the one chain that everything waits for.
template <class Op>
__device__ __forceinline__ bool stream_lookback(const Op &op, const unsigned long long *__restrict__ aggw,
                                                unsigned stride, unsigned from, unsigned to,
                                                RunningPrefix<Op> *run, long long limit) {
    using S = typename Op::State;
    constexpr int K = Tagged<S>::K;
    constexpr int Q = 5;  // 160 tiles: one per SM, so one step as a rule
    constexpr bool kLaneMajor = sizeof(typename Op::Scalar) == 8;
    const unsigned lane = threadIdx.x & 31;
    for (unsigned base = from; base < to; base += 32 * Q) {
        unsigned long long w[Q][K];
        unsigned todo = 0;
        const auto tile = [&](int q) { return base + (kLaneMajor ? lane * Q + q : 32 * q + lane); };
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (tile(q) < to) todo |= 1u << q;
        long long it = 0;
        while (__any_sync(0xffffffffu, todo != 0u)) {
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if ((todo >> q) & 1u) {
#pragma unroll
                    for (int k = 0; k < K; ++k) w[q][k] = ld_relaxed_u64(aggw + (size_t)k * stride + tile(q));
                }
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if ((todo >> q) & 1u) {
                    bool ok = true;
#pragma unroll
                    for (int k = 0; k < K; ++k) ok &= (unsigned)(w[q][k] >> 32) == kFlagAgg;
                    if (ok) todo &= ~(1u << q);
                }
            if (++it > limit) break;
        }
        if (__any_sync(0xffffffffu, todo != 0u)) return false;
        S v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            v[q] = op.identity();
            if (tile(q) < to) {
                unsigned *dst = reinterpret_cast<unsigned *>(&v[q]);
#pragma unroll
                for (int k = 0; k < K; ++k) dst[k] = (unsigned)w[q][k];
            }
        }
        if constexpr (kLaneMajor) {
#pragma unroll
            for (int q = 1; q < Q; ++q) v[0] = op.combine(v[0], v[q]);
        }
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {  // lane 0 ends with lanes 0..31 in order
#pragma unroll
            for (int q = 0; q < (kLaneMajor ? 1 : Q); ++q) {
                const S other = shfl_down(v[q], o);
                if (lane + o < kWarp) v[q] = op.combine(v[q], other);
            }
        }
#pragma unroll
        for (int q = 0; q < (kLaneMajor ? 1 : Q); ++q) v[q] = shfl_idx(v[q], 0);
        if constexpr (!kLaneMajor) {
#pragma unroll
            for (int q = 1; q < Q; ++q) v[0] = op.combine(v[0], v[q]);
        }
        run->extend(op, v[0]);
    }
    return true;
}

constexpr int stream_threads(int nwc, bool split) { return (nwc * (split ? 2 : 1) + 2) * 32; }

template <class Op, int NWC, int RB, int STAGES, int AHEAD, bool SPLIT, bool REVERSE>
__global__ void __launch_bounds__(stream_threads(NWC, SPLIT), 1)
k_scan_stream(const Op op, const int64_t n, const int64_t num_tiles, unsigned long long *__restrict__ aggw,
              const int reps, const DevCtl ctl) {
    using S = typename Op::State;
    using E = typename Op::Elem;
    using T = typename Op::Scalar;
    using Sh = StreamShape<Op, NWC, RB, STAGES>;
    using Seg = Segment<Sh, RB>;
    using X = typename TileFold<Op>::X;
    const TileFold<Op> tf{op};
    constexpr int K = Tagged<S>::K;
    constexpr int RING = 2 * STAGES;  // claimed tiles remembered
    static_assert(AHEAD >= 1 && AHEAD < STAGES && NWC <= 32, "loads in flight, and a stage for the tile being folded");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long s_bar_agg[STAGES], s_bar_pre[STAGES], s_bar_free[STAGES],
        s_bar_claim[RING];
    __shared__ X s_agg[STAGES][NWC];
    __shared__ S s_wex[STAGES][NWC], s_pre[STAGES];
    __shared__ unsigned s_tile[RING];
    __shared__ volatile int s_abort;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Tiles and slots are 32-bit: the rings' quotients and remainders are in every
    // role's serial path, the look-back's above all.
    const unsigned T_ = (unsigned)num_tiles;
    // the waits on other blocks (ctl.spin_limit) end before those inside the block
    const long long wait_limit = ctl.spin_limit < (1ll << 40) ? ctl.spin_limit * 16 : ctl.spin_limit;
    if (threadIdx.x == 0) {
        for (int b = 0; b < STAGES; ++b) {
            mbar_init(&s_bar_agg[b], NWC);
            mbar_init(&s_bar_pre[b], 2);
            mbar_init(&s_bar_free[b], NWC);
        }
        for (int b = 0; b < RING; ++b) mbar_init(&s_bar_claim[b], 1);
        mbar_init_fence();
        s_abort = 0;
    }
    __syncthreads();
    // A whole warp's wait inside the block for use `slot` of a ring of barriers;
    // false, alike in every lane, if the block gave up or the limit ran out.
    const auto wait_ring = [&](unsigned long long *bars, unsigned slot, unsigned ring) -> bool {
        unsigned long long *bar = bars + slot % ring;
        const unsigned parity = (slot / ring) & 1u;
        bool ok = false;
        for (long long it = 0; it <= wait_limit && !s_abort; ++it)
            if ((ok = mbar_try_wait(bar, parity))) break;
        return __all_sync(0xffffffffu, ok);
    };
    const auto give_up = [&] {
        s_abort = 1;
        set_error(ctl.err, kErrTimeout);
    };

    constexpr int kWorkers = SPLIT ? 2 * NWC : NWC;
    if (warp == kWorkers + 1) {  // -------------------------------------- look-back --
        const unsigned long long *mine = aggw + (size_t)(blockIdx.x % reps) * T_ * K;
        RunningPrefix<Op> run(op);  // the exclusive prefix of tile `from`
        unsigned from = 0;
        for (unsigned i = 0;; ++i) {
            if (!wait_ring(s_bar_claim, i, RING)) return;
            const unsigned t = s_tile[i % RING];
            if (t >= T_) return;
            const bool ok = stream_lookback(op, mine, T_, from, t, &run, ctl.spin_limit);
            if (!ok && lane == 0) give_up();
            // once the tile itself is folded, the previous use of its slots is over
            if (!ok || !wait_ring(s_bar_agg, i, STAGES)) return;
            if (lane == 0) {
                s_pre[i % STAGES] = run.value();
                mbar_arrive(&s_bar_pre[i % STAGES]);
            }
            from = t;
        }
    }
    if (warp == kWorkers) {  // ------------------- claims tiles, publishes aggregates --
        // Tiles are claimed at the pace of the folds: claims in bursts would give a
        // block neighbouring tiles that it folds a whole round apart, and every
        // tile behind them would wait for that round.
        const auto claimed = [&](unsigned slot, unsigned t) {  // lane 0
            s_tile[slot % RING] = t;
            mbar_arrive(&s_bar_claim[slot % RING]);
        };
        unsigned next = 0;
        if (lane == 0) {
            for (int j = 0; j <= AHEAD; ++j) claimed(j, atomicAdd(ctl.counter, 1u));
            next = atomicAdd(ctl.counter, 1u);
        }
        for (unsigned i = 0;; ++i) {
            if (!wait_ring(s_bar_claim, i, RING)) return;
            const unsigned t = s_tile[i % RING];
            if (t >= T_ || !wait_ring(s_bar_agg, i, STAGES)) return;
            X incx = lane < NWC ? s_agg[i % STAGES][lane] : tf.identity();
#pragma unroll
            for (int o = 1; o < NWC; o <<= 1) shfl_combine(tf, incx, o, false, lane >= o);
            const S inc = tf.state(incx), total = shfl_idx(inc, NWC - 1);
            if (lane < reps && (long long)t != ctl.stall_tile) {
                const unsigned *w = reinterpret_cast<const unsigned *>(&total);
#pragma unroll
                for (int k = 0; k < K; ++k)
                    st_relaxed_u64(aggw + ((size_t)lane * K + k) * T_ + t, ((unsigned long long)kFlagAgg << 32) | w[k]);
            }
            S wex = shfl_up(inc, 1);
            if (lane == 0) wex = op.identity();
            if (lane < NWC) s_wex[i % STAGES][lane] = wex;
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&s_bar_pre[i % STAGES]);
                claimed(i + AHEAD + 1, next);
                next = atomicAdd(ctl.counter, 1u);
            }
            __syncwarp();
        }
    }

    // ---------------------------------------------------- fold and store warps --
    // SPLIT: warps 0..NWC-1 load and fold, the next NWC store, so that neither waits
    // for the other; else the same warps do both, tile i's store STAGES - AHEAD
    // iterations after its fold.
    const int w = warp < NWC ? warp : warp - NWC;
    const int seg = REVERSE ? NWC - 1 - w : w;  // the warp's segment of the tile, its lanes' rows
    const int row = REVERSE ? 31 - lane : lane;
    const int64_t nb = n * (int64_t)sizeof(E);
    const auto segment = [&](unsigned slot, int s) -> Seg {
        return Seg{smem_raw + (slot % STAGES) * (unsigned)Sh::kData + (unsigned)(w * Sh::NS + s) * Sh::SEGP};
    };
    S *const s_ex = reinterpret_cast<S *>(smem_raw + STAGES * Sh::kData) + w * 32 + lane;  // + stage * NWC * 32
    const auto first_byte = [&](unsigned t) -> int64_t {
        const int64_t p = REVERSE ? T_ - 1 - t : t;
        return (p * NWC + seg) * (int64_t)Sh::SEG;
    };

    bool alive = true;
    const auto load = [&](unsigned slot) {
        if (!wait_ring(s_bar_claim, slot, RING)) {
            alive = false;
            return;
        }
        const unsigned t = s_tile[slot % RING];
        if (t < T_) {
            if (SPLIT && slot >= STAGES && !wait_ring(s_bar_free, slot - STAGES, STAGES)) {
                alive = false;
                return;
            }
            const int64_t b0 = first_byte(t);
#pragma unroll
            for (int s = 0; s < Sh::NS; ++s) {
                const Seg d = segment(slot, s);
                const E *src = op.stream(s);
                if (b0 + Sh::SEG <= nb) {
#pragma unroll
                    for (int j = 0; j < Sh::C; ++j) {
                        const int q = j * 32 + lane;
                        cp_async16(d.chunk(q / Sh::C, q % Sh::C),
                                   reinterpret_cast<const unsigned char *>(src) + b0 + q * 16);
                    }
                } else {
                    const E pad = op.pad(s);
                    for (int j = 0; j < Sh::C; ++j) {
                        const int q = j * 32 + lane;
                        copy16(d.chunk(q / Sh::C, q % Sh::C), src, b0 + q * 16, nb, pad);
                    }
                }
                if constexpr (Op::kWalk != 0) {  // one unit after the segment, one before it
                    if (s > 0 && lane < 2)
                        copy16(d.p + Sh::SEG + 16 * lane, src, lane ? b0 - Sh::U : b0 + Sh::SEG, nb, op.pad(s));
                }
            }
        }
        cp_async_commit();
    };
    const auto fold = [&](unsigned i, unsigned t) {
        cp_async_wait<AHEAD - 1>();
        __syncwarp();
        const int64_t e0 = first_byte(t) / (int64_t)sizeof(E) + (int64_t)row * Sh::EPR;
        X a = tf.identity();
        const Seg s0 = segment(i, 0);
        if constexpr (Op::kWalk == 0) {
#pragma unroll
            for (int uu = 0; uu < Sh::UR; ++uu) {
                E v[Sh::NPU];
                s0.load(row, REVERSE ? Sh::UR - 1 - uu : uu, v);
#pragma unroll
                for (int kk = 0; kk < Sh::NPU; ++kk) a = tf.step(a, op.item(v[REVERSE ? Sh::NPU - 1 - kk : kk]));
            }
        } else {
            static_assert(Op::kWalk == 0 || REVERSE, "the vjp walks run in descending order");
            const Seg s1 = segment(i, 1);
            E xn = s1.after(row);
#pragma unroll
            for (int u = Sh::UR - 1; u >= 0; --u) {
                E v[Sh::NPU], x[Sh::NPU];
                s0.load(row, u, v);
                s1.load(row, u, x);
#pragma unroll
                for (int k = Sh::NPU - 1; k >= 0; --k) {
                    const E nx = k + 1 < Sh::NPU ? x[k + 1 < Sh::NPU ? k + 1 : 0] : xn;
                    if constexpr (Op::kWalk == 1) a = tf.step(a, op.item(v[k], nx));
                    else a = tf.step(a, op.item(v[k], x[k], nx, e0 + u * Sh::NPU + k, n));
                }
                xn = x[0];
            }
        }
        const X inc = warp_inclusive_scan(tf, tf.sealed(a));
        S ex = shfl_up(tf.state(inc), 1);
        if (lane == 0) ex = op.identity();
        if (lane == kWarp - 1) s_agg[i % STAGES][w] = inc;
        s_ex[(i % STAGES) * NWC * 32] = ex;
        __syncwarp();
        if (lane == kWarp - 1) mbar_arrive(&s_bar_agg[i % STAGES]);
    };
    // fp32 sums: a row's elements are summed from zero and the row's prefix is
    // added to each partial sum.  Added to the prefix one by one, each of a row's 32
    // elements rounds at the prefix's magnitude: 1.1e-7 of the results for values
    // in (-1, 1) at n = 2^24 (16-element rows 8e-8), from zero 3.7e-8.  The pass is
    // bound by memory: n = 1e8 forward + vjp 0.267 ms before, 0.268 with it.
    constexpr bool kFromBase = Op::kWalk == 0 && ExactOf<Op>::value == kExactSum && std::is_same<S, float>::value;
    const auto store = [&](unsigned j) {
        const S pre = s_pre[j % STAGES], wex = s_wex[j % STAGES][w], ex = s_ex[(j % STAGES) * NWC * 32];
        S run = kFromBase ? op.combine(pre, op.combine(wex, ex)) : op.combine(op.combine(pre, wex), ex);
        S loc = op.identity();
        const int64_t b0 = first_byte(s_tile[j % RING]);
        const int64_t e0 = b0 / (int64_t)sizeof(E) + (int64_t)row * Sh::EPR;
        const Seg s0 = segment(j, 0);
        if constexpr (Op::kWalk == 0) {
#pragma unroll
            for (int uu = 0; uu < Sh::UR; ++uu) {
                const int u = REVERSE ? Sh::UR - 1 - uu : uu;
                E v[Sh::NPU];
                s0.load(row, u, v);
#pragma unroll
                for (int kk = 0; kk < Sh::NPU; ++kk) {
                    const int k = REVERSE ? Sh::NPU - 1 - kk : kk;
                    if constexpr (kFromBase) {
                        loc = op.combine(loc, op.item(v[k]));
                        v[k] = op.out(op.combine(run, loc), e0 + u * Sh::NPU + k);
                    } else {
                        run = op.combine(run, op.item(v[k]));
                        v[k] = op.out(run, e0 + u * Sh::NPU + k);
                    }
                }
                s0.store(row, u, v);
            }
        } else {
            const Seg s1 = segment(j, 1), sy = segment(j, Op::kWalk == 1 ? 2 : 1);
            E xn = s1.after(row);
            E y[Sh::NPU];
            sy.load(row, Sh::UR - 1, y);
#pragma unroll
            for (int u = Sh::UR - 1; u >= 0; --u) {
                E v[Sh::NPU], x[Sh::NPU], yl[Sh::NPU];  // yl: the unit before y
                s0.load(row, u, v);
                if constexpr (Op::kWalk == 1) {
                    s1.load(row, u, x);
                } else {
#pragma unroll
                    for (int k = 0; k < Sh::NPU; ++k) x[k] = y[k];
                }
                if (u > 0) sy.load(row, u > 0 ? u - 1 : 0, yl);
                else yl[Sh::NPU - 1] = sy.before(row);
#pragma unroll
                for (int k = Sh::NPU - 1; k >= 0; --k) {
                    const E nx = k + 1 < Sh::NPU ? x[k + 1 < Sh::NPU ? k + 1 : 0] : xn;
                    const E yp = k > 0 ? y[k > 0 ? k - 1 : 0] : yl[Sh::NPU - 1];
                    if constexpr (Op::kWalk == 1) {
                        run = op.combine(run, op.item(v[k], nx));
                        v[k] = op.out(run, yp);
                    } else {
                        const int64_t e = e0 + u * Sh::NPU + k;
                        run = op.combine(run, op.item(v[k], x[k], nx, e, n));
                        v[k] = op.out(run, x[k], yp, e);
                    }
                }
                xn = x[0];
                s0.store(row, u, v);
#pragma unroll
                for (int k = 0; k < Sh::NPU; ++k) y[k] = yl[k];
            }
        }
        __syncwarp();
        // the segment out, 512 contiguous bytes per step
        unsigned char *dst = reinterpret_cast<unsigned char *>(op.dst());
        constexpr int VT = 16 / (int)sizeof(T);
#pragma unroll
        for (int c = 0; c < Sh::C; ++c) {
            const int q = c * 32 + lane;
            const int64_t b = b0 + q * 16;
            uint4 t = *reinterpret_cast<const uint4 *>(s0.chunk(q / Sh::C, q % Sh::C));
            T r[VT];
            memcpy(r, &t, 16);
            if (b + 16 <= nb) {
                if (op.accumulating()) {
                    const uint4 o = *reinterpret_cast<const uint4 *>(dst + b);
                    T old[VT];
                    memcpy(old, &o, 16);
#pragma unroll
                    for (int k = 0; k < VT; ++k) r[k] = old[k] + r[k];
                    memcpy(&t, r, 16);
                }
                __stcs(reinterpret_cast<uint4 *>(dst + b), t);
            } else {
#pragma unroll
                for (int k = 0; k < VT; ++k) {
                    const int64_t at = b + k * (int64_t)sizeof(T);
                    T *d = reinterpret_cast<T *>(dst + at);
                    if (at < nb) *d = op.accumulating() ? *d + r[k] : r[k];
                }
            }
        }
        __syncwarp();  // every lane has read the stage: it may be refilled
    };

    if (SPLIT && warp >= NWC) {
        for (unsigned j = 0;; ++j) {
            if (!wait_ring(s_bar_claim, j, RING)) return;
            if (s_tile[j % RING] >= T_) return;
            if (!wait_ring(s_bar_pre, j, STAGES)) {
                if (lane == 0) give_up();
                return;
            }
            store(j);
            if (lane == 0) mbar_arrive(&s_bar_free[j % STAGES]);
        }
    }
    for (int j = 0; j < AHEAD && alive; ++j) load(j);
    constexpr unsigned D = STAGES - AHEAD, kNone = 0xffffffffu;
    unsigned end = kNone;  // first slot without a tile
    for (unsigned i = 0; alive; ++i) {
        if (end == kNone) {
            const unsigned t = s_tile[i % RING];
            if (t >= T_) end = i;
            else fold(i, t);
        }
        if constexpr (SPLIT) {
            if (end != kNone) break;
        } else {
            if (end != kNone && i >= D && i - D >= end) break;
            if (i >= D) {
                if (!wait_ring(s_bar_pre, i - D, STAGES)) {
                    alive = false;
                    break;
                }
                store(i - D);
            }
        }
        if (end == kNone) load(i + AHEAD);
    }
    cp_async_wait<0>();
    if (!alive && lane == 0) give_up();
}

// Whether one instantiation fits an SM, its dynamic shared memory allowed;
// cached per device (atomics: every writer stores the same value).
template <class Op, int NWC, int RB, int STAGES, int AHEAD, bool SPLIT, bool REVERSE> bool stream_ready() {
    using Sh = StreamShape<Op, NWC, RB, STAGES>;
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    int ok = cache[dev].load(std::memory_order_relaxed);
    if (ok == 0) {
        auto *k = k_scan_stream<Op, NWC, RB, STAGES, AHEAD, SPLIT, REVERSE>;
        int b = 0;
        ok = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem) == cudaSuccess &&
                     cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k, stream_threads(NWC, SPLIT),
                                                                   Sh::kSmem) == cudaSuccess &&
                     b >= 1
                 ? 1
                 : 0;
        if (ok) cache[dev].store(1, std::memory_order_relaxed);
    }
    return ok != 0;
}

// Copies of the published aggregates: each block reads the copy of its number
// modulo kStreamReps, so that fewer blocks poll the same lines.
constexpr int kStreamReps = 4;

// Queue one streaming scan of the whole call: the workspace's header, not zeroed
// yet, and the region after it, whose `avail` bytes bound the copies.
template <class Op, int NWC, int RB, int STAGES, int AHEAD, bool SPLIT, bool REVERSE>
adc_status run_scan_stream(const Op &op, int64_t n, void *ws, size_t avail, cudaStream_t s) {
    if (n == 0) return ADC_OK;
    using Sh = StreamShape<Op, NWC, RB, STAGES>;
    if (!stream_ready<Op, NWC, RB, STAGES, AHEAD, SPLIT, REVERSE>()) return ADC_ERR_CUDA;
    const int64_t T = Sh::tiles(n);
    const size_t one = (size_t)T * Tagged<typename Op::State>::K * 8;
    int reps = (int)(avail / one < (size_t)kStreamReps ? avail / one : (size_t)kStreamReps);
    if (reps < 1) return ADC_ERR_WORKSPACE;
    void *region = static_cast<char *>(ws) + kWsHeader;
    if (cudaMemsetAsync(ws, 0, kWsHeader + one * reps, s) != cudaSuccess) return ADC_ERR_CUDA;
    const int64_t G = num_sms();
    k_scan_stream<Op, NWC, RB, STAGES, AHEAD, SPLIT, REVERSE><<<(unsigned)(T < G ? T : G), stream_threads(NWC, SPLIT), Sh::kSmem, s>>>(
        op, n, T, static_cast<unsigned long long *>(region), reps, make_ctl(ws, 0));
    return check_launch();
}

}  // namespace adc
