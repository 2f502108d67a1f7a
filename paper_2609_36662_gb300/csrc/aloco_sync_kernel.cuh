// Fused outer-synchronisation pass (one launch per round).
//
// Each thread walks the parameter vector with a grid stride.  Per 16-byte
// pack it loads theta, v and the M replicas once, forms the pseudo-gradients
// Delta_m = theta - x_m (Algorithm 1), their sum S, the drift-energy and
// ||sum||^2 partials (Eq. adaptive-h-core-diagnostics), applies the
// corrected Nesterov step (Eq. autoloco-corrected-nesterov, with the
// normalisation of Eq. normalized-pseudo-gradient folded into c_avg), and
// stores theta', v' and the replica reset from the same registers.
//
// Reductions are deterministic: per-thread fp32 partials are promoted to
// fp64 every kFlush packs, threads are combined in a fixed order within the
// warp and across warps into one fp64 partial per block, and the last block
// to finish (atomic ticket, no spinning) sums the block partials in a fixed
// order.  The grid depends only on (M, dtype, n, device), so a round
// on the same inputs reproduces its statistics bit for bit.
#pragma once

#include <cuda_bf16.h>
#include <float.h>

#include "aloco_internal.h"

namespace aloco {

// Packs accumulated in fp32 before promotion to fp64: at most 64 (fp32) or
// 128 (bf16) squared terms per fp32 partial.
constexpr int kFlush = 16;

// Tuning knobs (compile-time): packs loaded per thread before any is used,
// minimum resident blocks per SM requested from the register allocator, and
// the cache policy of the streaming loads and stores.
#ifndef ALOCO_UNROLL
#define ALOCO_UNROLL 1
#endif
#ifndef ALOCO_MINB
#define ALOCO_MINB 0  // 0: the per-instance table below
#endif
#ifndef ALOCO_LD
#define ALOCO_LD 0  // 0 ld.global.cs, 1 ld.global.lu, 2 plain, 3 ld.global.cg
#endif
#ifndef ALOCO_ST
#define ALOCO_ST 0  // 0 st.global.cs, 1 plain, 2 st.global.cg
#endif

template <typename T>
__device__ __forceinline__ T ld_stream(const T *p) {
#if ALOCO_LD == 0
    return __ldcs(p);
#elif ALOCO_LD == 1
    return __ldlu(p);
#elif ALOCO_LD == 2
    return *p;
#else
    return __ldcg(p);
#endif
}
template <typename T>
__device__ __forceinline__ void st_stream(T *p, T v) {
#if ALOCO_ST == 0
    __stcs(p, v);
#elif ALOCO_ST == 1
    *p = v;
#else
    __stcg(p, v);
#endif
}

__device__ __forceinline__ float4 ldcs4(const void *base, int64_t i) {
    return ld_stream(reinterpret_cast<const float4 *>(base) + i);
}
__device__ __forceinline__ uint4 ldcs4u(const void *base, int64_t i) {
    return ld_stream(reinterpret_cast<const uint4 *>(base) + i);
}
__device__ __forceinline__ void stcs4(void *base, int64_t i, float4 val) {
    st_stream(reinterpret_cast<float4 *>(base) + i, val);
}
__device__ __forceinline__ void stcs4u(void *base, int64_t i, uint4 val) {
    st_stream(reinterpret_cast<uint4 *>(base) + i, val);
}

// Exact widening of the two bf16 values packed in a 32-bit word (element
// 2k in the low half, 2k+1 in the high half).
__device__ __forceinline__ float bf16_lo(uint32_t w) {
    return __uint_as_float(w << 16);
}
__device__ __forceinline__ float bf16_hi(uint32_t w) {
    return __uint_as_float(w & 0xFFFF0000u);
}
// Round two fp32 values to bf16 (nearest even) and pack them.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

__device__ __forceinline__ unsigned not_finite(float a, float b) {
    return (fabsf(a) <= FLT_MAX && fabsf(b) <= FLT_MAX) ? 0u : 1u;
}

// Outer step for one element given S = sum_m Delta_m:
//   Dtil = c S ; v' = mu v + Dtil ; d = Dtil + mu v' ; g' = g - eta d
// Each coefficient is applied as hi + lo: the small lo term enters the
// addend of the FMA that carries the hi product, so the coefficient's own
// fp32 rounding does not bias every element the same way.
struct Coef {
    float c_hi, c_lo, mu_hi, mu_lo, ne_hi, ne_lo;
};
__device__ __forceinline__ void outer_step(const Coef &k, float s, float g,
                                           float v, float &gp, float &vp) {
    const float dt = fmaf(s, k.c_hi, s * k.c_lo);
    vp = fmaf(k.mu_hi, v, fmaf(k.mu_lo, v, dt));
    const float d = fmaf(k.mu_hi, vp, fmaf(k.mu_lo, vp, dt));
    gp = g + fmaf(k.ne_hi, d, k.ne_lo * d);
}

// One 16-byte replica access ("pack") and the matching theta / v elements.
// fp32 replicas: 4 elements, one float4 of each stream.  bf16 replicas: 8
// elements, one uint4 of each replica and two float4 of theta and v.
template <bool BF16>
struct Pack;

template <>
struct Pack<false> {
    static constexpr int E = 4;
    using Raw = float4;
    __device__ static void load(const float *p, int64_t i, float (&o)[E]) {
        const float4 t = ldcs4(p, i);
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    }
    __device__ static void store(float *p, int64_t i, const float (&o)[E]) {
        stcs4(p, i, make_float4(o[0], o[1], o[2], o[3]));
    }
    __device__ static Raw load_x(const void *p, int64_t i) { return ldcs4(p, i); }
    __device__ static void widen(const Raw &r, float (&o)[E]) {
        o[0] = r.x; o[1] = r.y; o[2] = r.z; o[3] = r.w;
    }
    __device__ static Raw narrow(const float (&o)[E]) {
        return make_float4(o[0], o[1], o[2], o[3]);
    }
    __device__ static void store_x(void *p, int64_t i, const Raw &r) {
        stcs4(p, i, r);
    }
};

template <>
struct Pack<true> {
    static constexpr int E = 8;
    using Raw = uint4;
    __device__ static void load(const float *p, int64_t i, float (&o)[E]) {
        const float4 a = ldcs4(p, 2 * i), b = ldcs4(p, 2 * i + 1);
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
        o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    }
    __device__ static void store(float *p, int64_t i, const float (&o)[E]) {
        stcs4(p, 2 * i, make_float4(o[0], o[1], o[2], o[3]));
        stcs4(p, 2 * i + 1, make_float4(o[4], o[5], o[6], o[7]));
    }
    __device__ static Raw load_x(const void *p, int64_t i) { return ldcs4u(p, i); }
    __device__ static void widen(const Raw &r, float (&o)[E]) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            o[2 * j] = bf16_lo(w[j]);
            o[2 * j + 1] = bf16_hi(w[j]);
        }
    }
    __device__ static Raw narrow(const float (&o)[E]) {
        return make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]),
                          pack_bf16x2(o[4], o[5]), pack_bf16x2(o[6], o[7]));
    }
    __device__ static void store_x(void *p, int64_t i, const Raw &r) {
        stcs4u(p, i, r);
    }
};

template <bool BF16>
__device__ __forceinline__ float load_replica(const void *p, int64_t j) {
    if constexpr (BF16)
        return __uint_as_float((uint32_t)(reinterpret_cast<const uint16_t *>(p)[j]) << 16);
    else
        return reinterpret_cast<const float *>(p)[j];
}

__device__ __forceinline__ float from_lane_xor(float v, int mask) {
    return __shfl_xor_sync(0xffffffffu, v, mask);
}
__device__ __forceinline__ double from_lane_xor(double v, int mask) {
    return __shfl_xor_sync(0xffffffffu, v, mask);
}
__device__ __forceinline__ unsigned long long from_lane_xor(unsigned long long v, int mask) {
    return __shfl_xor_sync(0xffffffffu, v, mask);
}

// Warp sums of the P values each lane holds (P a power of two, at most 32)
// by recursive halving: at each step a lane keeps the half of its values
// that its lane bit selects and adds the partner's copy of that half; the
// last steps add across the lanes that share a value.  Lane L returns the
// warp sum of value L >> (5 - log2 P).  The order is fixed (and a + b = b + a
// exactly), so every lane holding a value has the same bits.
template <int P, typename T>
__device__ __forceinline__ T warp_sum_scatter(T (&v)[P]) {
    static_assert(P >= 1 && P <= 32 && (P & (P - 1)) == 0, "P: a power of two");
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int mask = 16 >> st;
        const int n = P >> st;  // values still held
        if (n > 1) {
            const bool up = (lane & mask) != 0;
#pragma unroll
            for (int i = 0; i < n / 2; ++i) {
                const T send = up ? v[i] : v[i + n / 2];
                const T keep = up ? v[i + n / 2] : v[i];
                v[i] = keep + from_lane_xor(send, mask);
            }
        } else {
            v[0] = v[0] + from_lane_xor(v[0], mask);
        }
    }
    return v[0];
}
__host__ __device__ constexpr int pow2_at_least(int n) {
    return n <= 1 ? 1 : 2 * pow2_at_least((n + 1) / 2);
}
// Of the P values each lane holds, the one whose warp sum warp_sum_scatter
// returns there.
template <int P, typename T>
__device__ __forceinline__ T lane_value(T (&v)[P]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = P, mask = 16; n > 1; n >>= 1, mask >>= 1) {
        const bool up = (lane & mask) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) v[i] = up ? v[i + n / 2] : v[i];
    }
    return v[0];
}

// Warp sums of non-negative floats as 64-bit integers: a value's mantissa in
// units of 2^-34 of the last place of the warp's largest value (`top`, its
// bits), so that 32 of them fit and add without rounding.  A value below 2^-34
// of the largest loses less than a unit, 2^-57 of the largest, and the
// conversion at the end rounds once: at most 31 x 2^-57 + 2^-53 of the sum, where
// the five roundings of a sum of doubles leave up to 5 x 2^-53.  An addition is two
// integer ones, where an fp64 one holds the SM's fp64 pipe for 16 clocks.
// An infinity or NaN comes back from `top` itself.
__device__ __forceinline__ unsigned warp_top(float e) {
    return __reduce_max_sync(0xffffffffu, __float_as_uint(e));
}
__device__ __forceinline__ unsigned long long to_fixed(float e, unsigned top) {
    // biased exponents; a subnormal has the smallest normal one
    const int ee = max((int)(__float_as_uint(e) >> 23), 1);
    const int et = max((int)(top >> 23), 1);
    const unsigned mant = __float_as_uint(e) - ((unsigned)(ee - 1) << 23);
    return ((unsigned long long)mant << 34) >> min(et - ee, 63);
}
__device__ __forceinline__ double from_fixed(unsigned long long sum, unsigned top) {
    if (top >= 0x7f800000u) return (double)__uint_as_float(top);
    const int et = max((int)(top >> 23), 1);
    // times 2^(et - 184)
    return __ull2double_rn(sum) * __hiloint2double((1023 + et - 184) << 20, 0);
}
// Lane L returns the sum over the warp of value L >> (5 - log2 P); values
// from `used` on are 0 (`used` is the same in every lane).
template <int P>
__device__ __forceinline__ double warp_sum_scatter_exact(const float (&e)[P], int used = P) {
    unsigned top[P];
    unsigned long long v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        top[i] = 0;
        v[i] = 0;
        if (i >= used) continue;
        top[i] = warp_top(e[i]);
        v[i] = to_fixed(e[i], top[i]);
    }
    const unsigned long long sum = warp_sum_scatter<P>(v);
    return from_fixed(sum, lane_value<P>(top));
}
__device__ __forceinline__ double warp_sum_exact(float e) {
    const unsigned top = warp_top(e);
    unsigned long long v = to_fixed(e, top);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += from_lane_xor(v, off);
    return from_fixed(v, top);
}
// The sum of column `col` over rows 0..n - 1 (n <= 32), in every lane.
template <int COLS>
__device__ __forceinline__ double column_sum(const double (*rows)[COLS], int n, int col) {
    const int lane = threadIdx.x & 31;
    double v = lane < n ? rows[lane][col] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Grid reduction of the block's fp64 rows: warp w wrote rows[w][m] for m < M
// and rows[w][MM] (sum S^2); the block's NW warps all call it.  Each block
// writes one row of M + 1 partials; the last block to finish (atomic ticket,
// no spinning) adds the rows in a fixed order, resets the ticket and
// publishes the totals.  The order of every addition is fixed by the grid.
// Latency-bound, on a part whose SM adds two doubles a clock: a warp-wide
// fp64 add holds the pipe for 16 clocks, so the work is laid out for few of
// them.  One warp folds a column (five adds); the grid's rows are read as k
// interleaved slices, one thread per slice and column, which keeps many
// loads in flight and the additions of different columns in one instruction.
// The host page is written by the threads that hold the totals, together.
template <int MM, int NW, int S>
__device__ __forceinline__ void finish_rows(const SyncArgs &a, int M, double (&rows)[S][MM + 1],
                                            unsigned nf) {
    static_assert(S >= NW && S <= 32, "a warp folds a column of rows");
    constexpr int kThreads = NW * 32;
    __shared__ unsigned long long shnf[NW];
    __shared__ bool s_last;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int np = M + 1;  // values per block: M energies + sum S^2
    auto slot = [&](int p) { return p < M ? p : MM; };
    auto warp_sum = [](unsigned long long v) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        return v;
    };

    const unsigned long long nfl = warp_sum(nf);
    if (lane == 0) shnf[warp] = nfl;
    __syncthreads();
    // the NW rows of 32 / R columns in one warp at a time
    constexpr int R = pow2_at_least(NW), C = 32 / R;
    for (int p0 = warp * C; p0 < np; p0 += NW * C) {
        const int p = p0 + lane / R, w = lane % R;
        double v = w < NW && p < np ? rows[w][slot(p)] : 0.0;
#pragma unroll
        for (int off = R / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (w == 0 && p < np) a.partials[(int64_t)blockIdx.x * np + p] = v;
    }
    if (t == kThreads - 1) {
        unsigned long long n = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) n += shnf[w];
        a.nf_partials[blockIdx.x] = n;
    }
    // thread 0's fence after the barrier orders the whole block's writes
    // (the outputs too) before its ticket
    __syncthreads();
    if (t == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(a.ticket, 1u);
        s_last = (prev == gridDim.x - 1);
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;

    const int grid = (int)gridDim.x;
    const int k = kThreads / np < S ? kThreads / np : S;  // slices of rows
    const int r = t / np, p = t - r * np;
    unsigned long long nacc = 0;
    for (int b = t; b < grid; b += kThreads) nacc += __ldcg(a.nf_partials + b);
    if (r < k) {
        // loads in flight: enough for one pass over a slice where the
        // registers allow (43 rows of 32 workers in batches of eight took 6 us)
        constexpr int U = NW >= 16 ? 8 : MM > 16 ? 22 : 12;
        double acc = 0.0;
        for (int b0 = r; b0 < grid; b0 += U * k) {
            double q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int b = b0 + u * k;
                q[u] = b < grid ? __ldcg(a.partials + (int64_t)b * np + p) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) acc += q[u];
        }
        rows[r][slot(p)] = acc;
    }
    nacc = warp_sum(nacc);
    if (lane == 0) shnf[warp] = nacc;
    __syncthreads();
    volatile double *out = a.stats_out;
    for (int c = warp; c < np; c += NW) {
        const double v = column_sum(rows, k, slot(c));
        if (lane == 0) {
            a.totals[c] = v;
            if (out) out[c] = v;
        }
    }
    if (t == kThreads - 1) {
        unsigned long long n = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) n += shnf[w];
        *a.nf_total = n;
        *a.ticket = 0u;  // ready for the next launch
        if (out) {
            out[kNfSlot] = __longlong_as_double((long long)n);
            out[kErrorSlot] = __ldcg(a.totals + kErrorSlot);
        }
    }
    if (out) {
        // the totals are written: the round's number follows, behind a fence
        // that orders the block's writes to the page before it
        __syncthreads();
        if (t == 0) {
            __threadfence_system();
            reinterpret_cast<volatile unsigned long long *>(a.stats_out)[kSeqSlot] = a.seq;
        }
    }
}

// A warp's row from its threads' partials: energies by recursive halving
// (about MM additions a warp instead of 5 MM), in doubles or, from fp32
// partials, in fixed point.
template <int MM>
__device__ __forceinline__ void store_row(double (&row)[MM + 1], double energy, double b) {
    constexpr int P = pow2_at_least(MM);
    const int lane = threadIdx.x & 31, m = lane / (32 / P);
    if (lane % (32 / P) == 0 && m < MM) row[m] = energy;
    if (lane == 0) row[MM] = b;
}
template <int MM>
__device__ __forceinline__ void fold_warp(double (&row)[MM + 1], const double (&e)[MM], double b) {
    constexpr int P = pow2_at_least(MM);
    double v[P];
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = m < MM ? e[m < MM ? m : 0] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) b += from_lane_xor(b, off);
    store_row<MM>(row, warp_sum_scatter<P>(v), b);
}
template <int MM>
__device__ __forceinline__ void fold_warp(double (&row)[MM + 1], const float (&e)[MM], float b) {
    constexpr int P = pow2_at_least(MM);
    float v[P];
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = m < MM ? e[m < MM ? m : 0] : 0.f;
    store_row<MM>(row, warp_sum_scatter_exact<P>(v), warp_sum_exact(b));
}

// finish_rows from per-thread fp64 partials.  Against shuffle trees over
// every value in every thread, serial folds in one thread and a serial
// publish: 2^20 parameters x 4 fp32 workers 20.0 -> 15.1 us (the kernel, ncu),
// 6e6 x 32 bf16 190 -> 166 us; the fused INT8 kernel, 1024 threads a block,
// 2e7 x 16 bf16 385 -> 300 us, 2e7 x 8 fp32 330 -> 283 us.  S bounds the rows
// where shared memory is short.
template <int MM, int NW, int S = 32>
__device__ __forceinline__ void reduce_and_finish(const SyncArgs &a, int M,
                                                  double (&e64)[MM], double b64,
                                                  unsigned nf) {
    __shared__ double rows[S][MM + 1];
    fold_warp<MM>(rows[threadIdx.x >> 5], e64, b64);
    finish_rows<MM, NW>(a, M, rows, nf);
}

// Minimum resident blocks per SM the register allocator must allow (it
// bounds registers per thread to 65536 / (kBlock * value)); 0 leaves the
// choice to the compiler, which measured as good as any fixed budget.
template <int MT, bool BF16>
constexpr int min_blocks() {
    return ALOCO_MINB > 0 ? ALOCO_MINB : 0;
}

template <int MT, bool BF16>
__global__ void __launch_bounds__(kBlock, (min_blocks<MT, BF16>()))
    sync_kernel(const __grid_constant__ SyncArgs a) {
    constexpr int MM = MT > 0 ? MT : ALOCO_MAX_WORKERS;
    const int M = MT > 0 ? MT : a.M;

    float e32[MM];
    double e64[MM];
#pragma unroll
    for (int m = 0; m < MM; ++m) {
        e32[m] = 0.f;
        e64[m] = 0.0;
    }
    float b32 = 0.f;
    double b64 = 0.0;
    unsigned nf = 0;
    int cnt = 0;

    const Coef k{a.c_hi, a.c_lo, a.mu_hi, a.mu_lo, a.neg_eta_hi, a.neg_eta_lo};
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;

    auto flush = [&]() {
#pragma unroll
        for (int m = 0; m < MM; ++m) {
            e64[m] += (double)e32[m];
            e32[m] = 0.f;
        }
        b64 += (double)b32;
        b32 = 0.f;
    };

    // ---------------------------------------------------- vector body
    using P = Pack<BF16>;
    constexpr int E = P::E;

    // Pseudo-gradients of one replica pack: S += Delta, ||Delta_m||^2 += Delta^2.
    auto accumulate = [&](const float (&gg)[E], const typename P::Raw &raw,
                          float (&s)[E], float &e) {
        float xx[E];
        P::widen(raw, xx);
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const float d = gg[j] - xx[j];
            s[j] += d;
            e = fmaf(d, d, e);
        }
    };
    // Outer step of the pack and its stores: theta', v', replica reset.
    auto finish = [&](int64_t i, const float (&gg)[E], const float (&vv)[E],
                      const float (&s)[E]) {
        float gp[E], vp[E];
#pragma unroll
        for (int j = 0; j < E; ++j) {
            b32 = fmaf(s[j], s[j], b32);
            outer_step(k, s[j], gg[j], vv[j], gp[j], vp[j]);
            nf += not_finite(gp[j], vp[j]);
        }
        P::store(a.g, i, gp);
        P::store(a.v, i, vp);
        if (!a.keep_x) {
            const typename P::Raw xo = P::narrow(gp);
#pragma unroll
            for (int m = 0; m < MM; ++m) {
                if (MT == 0 && m >= M) continue;
                P::store_x(a.x[m], i, xo);
            }
        }
        if (++cnt == kFlush) {
            flush();
            cnt = 0;
        }
    };

    if constexpr (MT > 0) {
        // Compile-time M: every load of the U packs is issued before any is
        // used, so (M + 2) U 16-byte loads (bf16: (M + 4) U) are in flight.
        constexpr int U = ALOCO_UNROLL;
        for (int64_t i0 = tid; i0 < a.nvec; i0 += stride * U) {
            float G[U][E], V[U][E];
            typename P::Raw X[U][MT];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t i = i0 + u * stride;
                if (i >= a.nvec) continue;
                P::load(a.g, i, G[u]);
                P::load(a.v, i, V[u]);
#pragma unroll
                for (int m = 0; m < MT; ++m) X[u][m] = P::load_x(a.x[m], i);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t i = i0 + u * stride;
                if (i >= a.nvec) continue;
                float s[E];
#pragma unroll
                for (int j = 0; j < E; ++j) s[j] = 0.f;
#pragma unroll
                for (int m = 0; m < MT; ++m) accumulate(G[u], X[u][m], s, e32[m]);
                finish(i, G[u], V[u], s);
            }
        }
    } else {
        // Any M up to 32: replicas are loaded in groups of 8 (independent
        // loads in flight) and consumed group by group, which bounds the
        // registers that hold loaded packs.
        constexpr int kGroup = 8;
        for (int64_t i = tid; i < a.nvec; i += stride) {
            float gg[E], vv[E], s[E];
            P::load(a.g, i, gg);
            P::load(a.v, i, vv);
#pragma unroll
            for (int j = 0; j < E; ++j) s[j] = 0.f;
#pragma unroll
            for (int m0 = 0; m0 < MM; m0 += kGroup) {
                if (m0 >= M) break;
                typename P::Raw X[kGroup];
#pragma unroll
                for (int q = 0; q < kGroup; ++q)
                    if (m0 + q < M) X[q] = P::load_x(a.x[m0 + q], i);
#pragma unroll
                for (int q = 0; q < kGroup; ++q)
                    if (m0 + q < M) accumulate(gg, X[q], s, e32[m0 + q]);
            }
            finish(i, gg, vv, s);
        }
    }

    // ------------------- scalar head and remainder, or the whole vector
    // where the buffers share no 16-byte boundary.  A call on one of three
    // shards of 5e7 x 6 bf16, cut off a boundary, took 267 us element by
    // element and takes 144 us with its packs behind a head.
    // With the worker count known only at run time the loads go out 16 at a
    // time and whatever the count (replica 0 again beyond it): behind a test of
    // the count each waits for the one before.  Whole vectors element by
    // element (kernel), tested one by one, tested in groups of 16, and this: 1.6e7
    // x 17 bf16 1010, 1359 and 644 us, x 32 1076, 1942 and 723; fp32 x 17 935, 1100
    // and 689, x 32 1109, 1326 and 930.  A known count takes one group: of its own
    // size for bf16 (1.6e7 x 1: 169 us, 178 in one of 16), of 16 for fp32 (133 and 140).
    constexpr int PACK = BF16 ? 8 : 4;
    for (int64_t r = tid; r < a.head + a.n - a.nvec * PACK; r += stride) {
        const int64_t j = r < a.head ? r - a.head : a.nvec * PACK + r - a.head;
        const float g = a.g[j];
        const float v = a.v[j];
        float s = 0.f;
        constexpr int kElemGroup = BF16 && MT > 0 ? MT : 16;
#pragma unroll
        for (int m0 = 0; m0 < MM; m0 += kElemGroup) {
            float x[kElemGroup];
#pragma unroll
            for (int q = 0; q < kElemGroup; ++q)
                if (MT == 0 || m0 + q < M)
                    x[q] = load_replica<BF16>(a.x[m0 + q < M ? m0 + q : 0], j);
#pragma unroll
            for (int q = 0; q < kElemGroup; ++q) {
                if (MT > 0 && m0 + q >= M) continue;
                const float d = m0 + q < M ? g - x[q] : 0.f;
                s += d;
                e32[m0 + q] = fmaf(d, d, e32[m0 + q]);
            }
        }
        b32 = fmaf(s, s, b32);
        float gp, vp;
        outer_step(k, s, g, v, gp, vp);
        nf += not_finite(gp, vp);
        a.g[j] = gp;
        a.v[j] = vp;
#pragma unroll
        for (int m = 0; m < MM; ++m) {
            if ((MT == 0 && m >= M) || a.keep_x) continue;
            if constexpr (BF16)
                reinterpret_cast<__nv_bfloat16 *>(a.x[m])[j] =
                    __float2bfloat16_rn(gp);
            else
                reinterpret_cast<float *>(a.x[m])[j] = gp;
        }
        if (++cnt == kFlush) {
            flush();
            cnt = 0;
        }
    }
    // A small round: no thread has come to a flush, so its sums are the fp32
    // partials, and a warp adds them in fixed point instead of doubles, whose
    // flush and sums wait for the SM's fp64 pipe (two additions a clock).  The
    // kernel at 2^20 parameters, doubles against fixed point, L2 flushed: 4 fp32
    // workers 21.0 and 20.0 us, 8 28.2 and 25.9, 16 bf16 30.7 and 28.5, 32 52.0
    // and 46.6; 2e5 x 8 fp32 19.1 and 15.8.
    const int64_t loose = a.head + a.n - a.nvec * PACK;
    const bool small = (a.nvec + stride - 1) / stride + (loose + stride - 1) / stride < kFlush;
    __shared__ double rows[32][MM + 1];
    if (small) {
        fold_warp<MM>(rows[threadIdx.x >> 5], e32, b32);
    } else {
        flush();
        fold_warp<MM>(rows[threadIdx.x >> 5], e64, b64);
    }
    finish_rows<MM, kBlock / 32>(a, M, rows, nf);
}

// Tuned residency (blocks of kBlock threads per SM) of the fused pass for
// M workers, measured on GB300 over M = 1..32 and both replica types on a
// 2^28-parameter round: fewer resident warps streaming more arrays keep
// HBM busier once M + 2 streams are in flight.  Capped by occupancy.
template <bool BF16>
constexpr int tuned_blocks_per_sm(int M) {
    if (BF16) return M <= 7 ? 2 : 1;
    return M == 1 ? 4 : M == 2 ? 3 : M <= 8 ? 2 : 1;
}

// Persistent grid for one instance: SMs x resident blocks.
template <int MT, bool BF16>
cudaError_t plan_one(int64_t work_items, int sm_count, int M, int request,
                     LaunchPlan *plan) {
    static PerDevice cache;  // per instance and device, computed once
    const void *fn = reinterpret_cast<const void *>(&sync_kernel<MT, BF16>);
    const int dev = PerDevice::device();
    int occupancy = cache.get(dev);
    if (occupancy == 0) {
        int b = 0;
        cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, sync_kernel<MT, BF16>,
                                                          kBlock, 0);
        if (e != cudaSuccess) return e;
        occupancy = b > 0 ? b : 1;
        cache.set(dev, occupancy);
    }
    int blocks_per_sm = request > 0 ? request : tuned_blocks_per_sm<BF16>(M);
    if (blocks_per_sm <= 0 || blocks_per_sm > occupancy) blocks_per_sm = occupancy;
    int64_t want = (work_items + kBlock - 1) / kBlock;
    int64_t full = (int64_t)sm_count * blocks_per_sm;
    int64_t grid = want < full ? want : full;
    if (grid < 1) grid = 1;
    plan->kernel = fn;
    plan->grid = (int)grid;
    plan->block = kBlock;
    return cudaSuccess;
}

template <bool BF16>
cudaError_t plan_dispatch(int M, int64_t work_items, int sm_count,
                          int blocks_per_sm, LaunchPlan *plan) {
    switch (M) {
#define ALOCO_CASE(K) \
    case K:           \
        return plan_one<K, BF16>(work_items, sm_count, M, blocks_per_sm, plan);
        ALOCO_CASE(1) ALOCO_CASE(2) ALOCO_CASE(3) ALOCO_CASE(4)
        ALOCO_CASE(5) ALOCO_CASE(6) ALOCO_CASE(7) ALOCO_CASE(8)
        ALOCO_CASE(9) ALOCO_CASE(10) ALOCO_CASE(11) ALOCO_CASE(12)
        ALOCO_CASE(13) ALOCO_CASE(14) ALOCO_CASE(15) ALOCO_CASE(16)
#undef ALOCO_CASE
        default:
            return plan_one<0, BF16>(work_items, sm_count, M, blocks_per_sm,
                                     plan);
    }
}

}  // namespace aloco
