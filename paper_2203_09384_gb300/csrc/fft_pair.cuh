// complex32 transforms of N = 64..2048, two signals per thread (sm_103a).
//
// A complex32 element is 4 bytes in HBM but the same FP32 work as a complex64
// one, so with one signal per thread these lengths were bound by instruction
// issue and by the shared-memory/L1 data path, not by HBM.  Here every thread
// carries the same elements of two signals, as register pairs (first signal,
// second signal), and
//   * all butterfly and twiddle arithmetic is the packed two-wide FP32 form
//     (add/sub/mul/fma .f32x2): the same FLOP rate at half the issue slots, and
//     packing across signals needs no shuffling of components;
//   * one twiddle load, one swizzled address and one 128-bit shared-memory
//     access serve both signals.
// Every operation is the scalar kernels' own, rounding for rounding (the
// products that nvcc contracts into FMAs there are explicit FMAs here), so the
// stored values and exponents do not depend on which kernel ran.
#pragma once

#include "fft_device.cuh"

namespace gbfft {

// ---------------------------------------------------------------------------
// packed arithmetic: .x belongs to the first signal, .y to the second
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

struct C2 {  // one complex element of each of the two signals
    float2 re, im;
};
__device__ __forceinline__ C2 add2(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 sub2(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a + (-i) b and a - (-i) b
__device__ __forceinline__ C2 add_neg_i(C2 a, C2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
__device__ __forceinline__ C2 sub_neg_i(C2 a, C2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }
// twiddle product, contracted as nvcc contracts cmul()
__device__ __forceinline__ C2 cmul2(C2 a, float2 w) {
    const float2 wr = both(w.x), wi = both(w.y);
    return {fma2(a.re, wr, neg2(mul2(a.im, wi))), fma2(a.re, wi, mul2(a.im, wr))};
}
// c a' + s b' forms of the constant products inside the radix-16 butterfly
// (nvcc folds the constants' signs before it contracts):
// omega_16^1 = (c, -s) and ^3 = (s, -c) with the pair passed as (c, s)
__device__ __forceinline__ C2 cmul_conj2(C2 a, float c, float s) {
    return {fma2(a.re, both(c), mul2(a.im, both(s))), fma2(a.im, both(c), mul2(a.re, both(-s)))};
}
// omega_16^9 = (-cos(pi/8), sin(pi/8))
__device__ __forceinline__ C2 cmul_w9_2(C2 a) {
    return {fma2(a.re, both(-kCos8), mul2(a.im, both(-kSin8))), fma2(a.re, both(kSin8), mul2(a.im, both(-kCos8)))};
}

template <int R>
struct PairDft;

// the two outer additions of a radix-4 butterfly: sums and differences of
// (0, 2) and (1, 3) in, outputs in natural order
__device__ __forceinline__ void dft4_outer(C2 s02, C2 d02, C2 s13, C2 d13, C2& o0, C2& o1, C2& o2, C2& o3) {
    o0 = add2(s02, s13);
    o2 = sub2(s02, s13);
    o1 = add_neg_i(d02, d13);
    o3 = sub_neg_i(d02, d13);
}

template <>
struct PairDft<4> {
    static __device__ __forceinline__ void run(C2* v) {
        dft4_outer(add2(v[0], v[2]), sub2(v[0], v[2]), add2(v[1], v[3]), sub2(v[1], v[3]), v[0], v[1], v[2], v[3]);
    }
};

// omega_8 a = sqrt(1/2) t with t = (re + im, im - re), and
// omega_8^3 a = sqrt(1/2) (t.re, -t.im) with t = (im - re, re + im): the
// factor sqrt(1/2) goes into the FMA of the addition that follows
__device__ __forceinline__ C2 w8_1_sum(C2 a) { return {add2(a.re, a.im), sub2(a.im, a.re)}; }
__device__ __forceinline__ C2 w8_3_sum(C2 a) { return {sub2(a.im, a.re), add2(a.re, a.im)}; }
__device__ __forceinline__ C2 fma_c2(C2 t, float kr, float ki, C2 e) {
    return {fma2(t.re, both(kr), e.re), fma2(t.im, both(ki), e.im)};
}

template <>
struct PairDft<8> {
    static __device__ __forceinline__ void run(C2* v) {
        C2 e[4] = {v[0], v[2], v[4], v[6]};
        C2 o[4] = {v[1], v[3], v[5], v[7]};
        PairDft<4>::run(e);
        PairDft<4>::run(o);
        const C2 t1 = w8_1_sum(o[1]), t3 = w8_3_sum(o[3]);
        v[0] = add2(e[0], o[0]);
        v[4] = sub2(e[0], o[0]);
        v[1] = fma_c2(t1, kSqrtHalf, kSqrtHalf, e[1]);
        v[5] = fma_c2(t1, -kSqrtHalf, -kSqrtHalf, e[1]);
        v[2] = add_neg_i(e[2], o[2]);
        v[6] = sub_neg_i(e[2], o[2]);
        v[3] = fma_c2(t3, kSqrtHalf, -kSqrtHalf, e[3]);
        v[7] = fma_c2(t3, -kSqrtHalf, kSqrtHalf, e[3]);
    }
};

template <>
struct PairDft<16> {
    // 4 x 4, as Dft<16>: input index r1 + 4 r2, output index k2 + 4 k1
    static __device__ __forceinline__ void run(C2* v) {
        C2 y[4][4];
#pragma unroll
        for (int r1 = 0; r1 < 4; ++r1) {
            y[r1][0] = v[r1];
            y[r1][1] = v[r1 + 4];
            y[r1][2] = v[r1 + 8];
            y[r1][3] = v[r1 + 12];
            PairDft<4>::run(y[r1]);
        }
        {
            C2 z[4] = {y[0][0], y[1][0], y[2][0], y[3][0]};
            PairDft<4>::run(z);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[4 * k] = z[k];
        }
        {
            const C2 a = cmul_conj2(y[1][1], kCos8, kSin8);  // ^1
            const C2 t = w8_1_sum(y[2][1]);                  // ^2
            const C2 b = cmul_conj2(y[3][1], kSin8, kCos8);  // ^3
            dft4_outer(fma_c2(t, kSqrtHalf, kSqrtHalf, y[0][1]), fma_c2(t, -kSqrtHalf, -kSqrtHalf, y[0][1]),
                       add2(a, b), sub2(a, b), v[1], v[5], v[9], v[13]);
        }
        {
            const C2 t1 = w8_1_sum(y[1][2]);  // ^2
            const C2 t3 = w8_3_sum(y[3][2]);  // ^6
            const C2 p = {mul2(t3.re, both(kSqrtHalf)), mul2(t3.im, both(-kSqrtHalf))};
            const C2 m = {neg2(p.re), neg2(p.im)};
            dft4_outer(add_neg_i(y[0][2], y[2][2]), sub_neg_i(y[0][2], y[2][2]),  // ^4
                       fma_c2(t1, kSqrtHalf, kSqrtHalf, p), fma_c2(t1, kSqrtHalf, kSqrtHalf, m), v[2], v[6], v[10],
                       v[14]);
        }
        {
            const C2 a = cmul_conj2(y[1][3], kSin8, kCos8);  // ^3
            const C2 t = w8_3_sum(y[2][3]);                  // ^6
            const C2 b = cmul_w9_2(y[3][3]);                 // ^9
            dft4_outer(fma_c2(t, kSqrtHalf, -kSqrtHalf, y[0][3]), fma_c2(t, -kSqrtHalf, kSqrtHalf, y[0][3]),
                       add2(a, b), sub2(a, b), v[3], v[7], v[11], v[15]);
        }
    }
};

// ---------------------------------------------------------------------------
// schedule of a pair kernel: P = S / 2 signal pairs per block, T = N / E
// threads per pair, a ring of D tiles filled by bulk copies (per warp when a
// pair lives in one warp, per block when it spans warps)
// ---------------------------------------------------------------------------
template <int LOG2N_, int E_, int S_, int R0, int R1, int R2, int R3, int MINB_, int D_, bool STEAL_>
struct PairCfg {
    // one block per tile is launched, and a running block takes the tiles of
    // blocks that have not started (TileTaker)
    static constexpr bool kSteal = STEAL_;
    static constexpr int LOG2N = LOG2N_;
    static constexpr int N = 1 << LOG2N_;
    static constexpr int E = E_;
    static constexpr int T = N / E;
    static constexpr int S = S_;
    static constexpr int P = S / 2;
    static constexpr int NT = P * T;
    static constexpr int MINB = MINB_;
    static constexpr int D = D_;
    static constexpr int M = (R0 > 0) + (R1 > 0) + (R2 > 0) + (R3 > 0);
    static constexpr bool kWarpLocal = T <= 32;
    static constexpr int radix(int s) { return s == 0 ? R0 : s == 1 ? R1 : s == 2 ? R2 : R3; }
    static constexpr int ns(int s) {
        int p = 1;
        for (int i = 0; i < s; ++i) p *= radix(i);
        return p;
    }
    static constexpr int tw_off(int s) {
        int o = 0;
        for (int i = 1; i < s; ++i) o += (radix(i) - 1) * ns(i);
        return o;
    }
    static constexpr int kTwiddles = tw_off(M);
    // A unit owns one tile at a time: a warp, or the block when pairs span warps.
    static constexpr int kUnits = kWarpLocal ? NT / 32 : 1;
    static constexpr int SU = S / kUnits;               // signals per unit tile
    static constexpr int kExchangeBytes = SU * N * 8;   // 16 bytes per element of a pair
    static constexpr int kTileBytes = SU * N * 4;       // binary16 pairs
    static constexpr int kSlotBytes = kTileBytes + (kWarpLocal ? 128 : 0);  // + the group gaps
    static constexpr int kUnitBytes = kExchangeBytes + D * kSlotBytes;
    static constexpr int kBarOffset = kUnits * kUnitBytes;
    static constexpr int kRedOffset = kBarOffset + kUnits * D * 8;
    // tile stealing: the answer, its mbarrier, the tile in the slot (-1: no more)
    static constexpr int kStealOffset = (kRedOffset + (kWarpLocal ? 0 : 2 * (NT / 32) * 4) + 15) / 16 * 16;
    static constexpr int kSmemBytes = kSteal ? kStealOffset + 32 : kStealOffset;
    // A tile in shared memory is split into groups of consecutive signals
    // placed 128 / groups bytes apart, and neighbouring pairs of a warp take
    // their signals from different groups: one access of the warp (stage s:
    // T lanes of 8 bytes, or of 4 where a thread has one butterfly) then
    // covers all banks once.  Packed, signals start on the same bank.
    static constexpr int groups(int s) {
        return !kWarpLocal ? 1 : E / radix(s) >= 2 ? (16 / T > 1 ? 16 / T : 1) : (32 / T > 1 ? 32 / T : 1);
    }
    static_assert(ns(M) == N && S % 2 == 0 && NT % 32 == 0 && D >= 1, "whole pairs, whole warps");
    static_assert(!kSteal || (kUnits == 1 && D == 1), "tile stealing: one tile at a time per block, one slot");
    static_assert(E % R0 == 0 && E % (R1 ? R1 : 1) == 0 && E % (R2 ? R2 : 1) == 0 && E % (R3 ? R3 : 1) == 0,
                  "every radix must divide E");
};

// Element (4-byte) offset of signal `sig` in a tile of G groups, and the first
// signal of pair p of a warp whose stage-0 access wants G groups.
template <class C, int G>
__device__ __forceinline__ int pair_place(int sig) {
    return sig * C::N + (G > 1 ? sig / (C::SU / G) * (32 / G) : 0);
}
template <class C, int G>
__device__ __forceinline__ int pair_signal(int p) {
    return (p % G) * (C::SU / G) + (p / G) * 2;
}

// Butterfly of thread t in slot c: the first and the last stage give a thread
// neighbouring butterflies (64-bit HBM accesses), the middle ones interleave.
template <class C, int s>
__device__ __forceinline__ int pair_bfly(int t, int c) {
    constexpr int K = C::E / C::radix(s);
    return (s == 0 || s == C::M - 1) ? K * t + c : t + C::T * c;
}

// Exchange slots are 16 bytes; the 8 slots of row `row = a >> 3` (128 B) are
// XOR-permuted by row ^ (row >> 3): conflict free at every length here
// (128-bit accesses resolve per quarter-warp).  The swizzle is linear over
// XOR, so for a thread's base and a compile-time offset `k` on bits the base
// leaves zero it is pair_swz(base) ^ pair_swz(k): the low three bits are one
// XOR per distinct value, the rest an immediate offset.
__host__ __device__ constexpr int pair_swz(int a) { return a ^ (((a >> 3) ^ (a >> 6)) & 7); }
__device__ __forceinline__ float4* pair_slot(float4* buf, int swz_base, int k) {
    return buf + (swz_base ^ (pair_swz(k) & 7)) + (pair_swz(k) & ~7);
}

template <class C, int s>
__device__ __forceinline__ void pair_scatter(const C2 (&v)[C::E], float4* buf, int sb, int t) {
    constexpr int R = C::radix(s), K = C::E / R, Ns = C::ns(s);
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const int j = pair_bfly<C, s>(t, c);
        const int base = pair_swz(sb + (j / Ns) * (Ns * R) + (j & (Ns - 1)));
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const C2 x = v[c * R + q];
            float4* p = pair_slot(buf, base, q * Ns);
            if (!dbg_ok(p >= buf && p < buf + C::P * C::N)) continue;
            *p = make_float4(x.re.x, x.re.y, x.im.x, x.im.y);
        }
    }
}

template <class C, int s>
__device__ __forceinline__ void pair_gather(C2 (&v)[C::E], float4* buf, int sb, int t) {
    constexpr int R = C::radix(s), K = C::E / R, stride = C::N / R;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const int base = pair_swz(sb + pair_bfly<C, s>(t, c));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float4* p = pair_slot(buf, base, r * stride);
            if (!dbg_ok(p >= buf && p < buf + C::P * C::N)) continue;
            const float4 f = *p;
            v[c * R + r] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
            GBFFT_DBG_ONLY(*p = make_float4(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000),
                                            __int_as_float(0x7fc00000), __int_as_float(0x7fc00000));)
        }
    }
}

template <class C, int s>
__device__ __forceinline__ void pair_twist_dft(C2 (&v)[C::E], int t, const float2* __restrict__ tw) {
    constexpr int R = C::radix(s), K = C::E / R, Ns = C::ns(s);
    if constexpr (s > 0) {
        const float2* twp = tw + C::tw_off(s) + (pair_bfly<C, s>(t, 0) & (Ns - 1));
#pragma unroll
        for (int r = 1; r < R; ++r) {
            if constexpr (K == 2 && s == C::M - 1) {
                // neighbouring butterflies read neighbouring twiddles: one 128-bit load
                const float4 w = __ldg(reinterpret_cast<const float4*>(twp + (r - 1) * Ns));
                v[r] = cmul2(v[r], make_float2(w.x, w.y));
                v[R + r] = cmul2(v[R + r], make_float2(w.z, w.w));
            } else {
                // T is a multiple of Ns in the middle stages: the thread's butterflies share the twiddle
                static_assert(K == 1 || C::T % Ns == 0, "one twiddle for the butterflies of a thread");
                const float2 w = __ldg(twp + (r - 1) * Ns);
#pragma unroll
                for (int c = 0; c < K; ++c) v[c * R + r] = cmul2(v[c * R + r], w);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < K; ++c) PairDft<R>::run(&v[c * R]);
}

// one binary16 element of each signal (32-bit words) to FP32
template <bool INV>
__device__ __forceinline__ C2 pair_from_half(uint32_t a, uint32_t b) {
    const float2 fa = __half22float2(bits_h2(__uint_as_float(a)));
    const float2 fb = __half22float2(bits_h2(__uint_as_float(b)));
    return {make_float2(fa.x, fb.x), INV ? make_float2(-fa.y, -fb.y) : make_float2(fa.y, fb.y)};
}

// stage 0 inputs of two signals from their ring slot (past the end of the
// batch: whatever the slot holds; such a signal's results are not stored, and
// the packed arithmetic keeps them apart from the other signal's)
template <class C, bool INV>
__device__ __forceinline__ void pair_load(C2 (&v)[C::E], const uint32_t* a, int t) {
    constexpr int R = C::radix(0), K = C::E / R, stride = C::N / R;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if constexpr (K >= 2) {
#pragma unroll
            for (int c = 0; c < K; c += 2) {
                const uint32_t* p = a + K * t + c + r * stride;
                const uint2 x = *reinterpret_cast<const uint2*>(p);
                const uint2 y = *reinterpret_cast<const uint2*>(p + C::N);
                v[c * R + r] = pair_from_half<INV>(x.x, y.x);
                v[(c + 1) * R + r] = pair_from_half<INV>(x.y, y.y);
            }
        } else {
            const uint32_t* p = a + t + r * stride;
            v[r] = pair_from_half<INV>(p[0], p[C::N]);
        }
    }
}

// Largest |component| of each of the thread's two signals.  Non-negative
// floats order like their bit patterns, and fmaxf has dropped any NaN.
template <class C>
__device__ __forceinline__ float2 pair_max(const C2 (&v)[C::E]) {
    float2 m = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < C::E; ++i) {
        m.x = fmaxf(m.x, fmaxf(fabsf(v[i].re.x), fabsf(v[i].im.x)));
        m.y = fmaxf(m.y, fmaxf(fabsf(v[i].re.y), fabsf(v[i].im.y)));
    }
    if constexpr (C::T >= 32) {
        m.x = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m.x)));
        m.y = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m.y)));
    } else {
#pragma unroll
        for (int o = 1; o < C::T; o <<= 1) {
            m.x = fmaxf(m.x, __shfl_xor_sync(0xffffffffu, m.x, o));
            m.y = fmaxf(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
        }
    }
    return m;
}

// last-stage outputs as binary16 pairs, in natural order from `a` (the first
// signal) and `a` + N (the second): HBM, or a tile in shared memory
template <class C, bool INV, bool GLOBAL>
__device__ __forceinline__ void pair_store(const C2 (&v)[C::E], uint32_t* a, int t, bool act_a, bool act_b, float ma,
                                           float mb) {
    constexpr int R = C::radix(C::M - 1), K = C::E / R, stride = C::N / R;
    const float2 mr = make_float2(ma, mb), mi = INV ? make_float2(-ma, -mb) : mr;
    uint32_t wa[C::E], wb[C::E];
#pragma unroll
    for (int i = 0; i < C::E; ++i) {
        const float2 re = mul2(v[i].re, mr), im = mul2(v[i].im, mi);
        wa[i] = __float_as_uint(h2_bits(__floats2half2_rn(re.x, im.x)));
        wb[i] = __float_as_uint(h2_bits(__floats2half2_rn(re.y, im.y)));
    }
    auto store = [&](const uint32_t (&w)[C::E], uint32_t* dst) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if constexpr (K >= 2) {
#pragma unroll
                for (int c = 0; c < K; c += 2) {
                    uint2* p = reinterpret_cast<uint2*>(dst + K * t + c + q * stride);
                    const uint2 x = make_uint2(w[c * R + q], w[(c + 1) * R + q]);
                    if constexpr (GLOBAL) __stcs(p, x); else *p = x;
                }
            } else {
                dst[t + q * stride] = w[q];
            }
        }
    };
    if (act_a) store(wa, a);
    if (act_b) store(wb, a + C::N);
}

template <class C, int s>
__device__ __forceinline__ void pair_stages(C2 (&v)[C::E], float4* buf, int sb, int t, const float2* __restrict__ tw) {
    if constexpr (s < C::M) {
        if constexpr (C::kWarpLocal) __syncwarp(); else __syncthreads();  // earlier readers of buf are done
        pair_scatter<C, s - 1>(v, buf, sb, t);
        if constexpr (C::kWarpLocal) __syncwarp(); else __syncthreads();
        pair_gather<C, s>(v, buf, sb, t);
        pair_twist_dft<C, s>(v, t, tw);
        pair_stages<C, s + 1>(v, buf, sb, t, tw);
    }
}

// global <- shared bulk copies of one thread: all committed ones have read
// their source / have completed
__device__ __forceinline__ void bulk_copy_s2g(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// N = 64..512: a pair lives in one warp, and every warp walks tiles of its
// own without any block barrier.  Bulk copies bring a tile in (ring of D
// slots, refilled once stage 0 has read one) and take the result out of the
// exchange buffer, so HBM traffic costs the LSU data path one conflict-free
// shared-memory access each way.  Bounded waits, error word and stall test
// mode as in fft_stockham_ring_kernel, per warp.
template <class C, bool INV>
__global__ void __launch_bounds__(C::NT, C::MINB)
    fft_pair_c32_warp_kernel(const uint32_t* in, const int8_t* in_exp, uint32_t* out, int8_t* out_exp, int64_t batch,
                             const float2* __restrict__ tw, float scale, int* err, uint64_t wait_ns, int stall) {
    pdl_enter();
    constexpr int D = C::D, GI = C::groups(0), GO = C::groups(C::M - 1);
    extern __shared__ __align__(16) float4 smem4[];
    unsigned char* base8 = reinterpret_cast<unsigned char*>(smem4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pr = lane / C::T;
    const int t = lane % C::T;
    const int ls = log2_pow2(scale);
    unsigned char* unit = base8 + warp * C::kUnitBytes;
    float4* xbuf = reinterpret_cast<float4*>(unit);
    uint32_t* otile = reinterpret_cast<uint32_t*>(unit);  // the outgoing tile reuses the exchange buffer
    unsigned char* ring = unit + C::kExchangeBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(base8 + C::kBarOffset) + warp * D;
    const int64_t ntiles = (batch + C::SU - 1) / C::SU;
    const int64_t first_tile = (int64_t)blockIdx.x * C::kUnits + warp, step = (int64_t)gridDim.x * C::kUnits;
    dbg_set_err(err);

    RingInFlight inflight;  // lane 0's copies in flight
    TileTaker taker;        // lane 0's requests (kSteal)
    // lane 0: tile `tile` into `slot`; the tile of the warp's iteration j goes to slot j mod D
    auto issue = [&](int slot, int64_t tile, uint32_t parity) {
        const int64_t first = tile * C::SU;
        const uint32_t* src = in + first * C::N;
        unsigned char* dst = ring + slot * C::kSlotBytes;
        constexpr int kG = C::SU / GI;  // signals per group
        const int64_t left = batch - first;
        const int nsig = left < C::SU ? (int)left : C::SU;
        mbar_arrive_expect_tx(&bars[slot], (uint32_t)(nsig * C::N * 4));
#pragma unroll
        for (int g = 0; g < GI; ++g) {
            const int n = min(nsig - g * kG, kG);
            if (n > 0)
                bulk_copy_g2s(dst + 4 * pair_place<C, GI>(g * kG), src + g * kG * C::N, (uint32_t)(n * C::N * 4),
                              &bars[slot]);
        }
        inflight.issued(slot, parity);
    };
    if (lane == 0) {
        for (int d = 0; d < D; ++d) mbar_init(&bars[d], 1);
        if constexpr (C::kSteal) {
            taker.resp = base8 + C::kStealOffset;
            taker.bar = reinterpret_cast<uint64_t*>(base8 + C::kStealOffset + 16);
            mbar_init(taker.bar, 1);
        }
        fence_mbar_init();
    }
    __syncwarp();
    if (lane == 0 && !stall) {
        for (int d = 0; d < D; ++d)
            if (first_tile + d * step < ntiles) issue(d, first_tile + d * step, 0);
    }
    if (C::kSteal && lane == 0) taker.request();
    bool dead = false;
    if (stall) {  // failure-detection test mode: a phase nothing will complete
        if (!mbar_wait_bounded(&bars[0], 0, wait_ns)) atomicCAS(err, 0, kErrTimeout);
        dead = true;
    }
    const int own = pair_signal<C, GI>(pr);  // the thread's first signal in the tile
    int slot = 0;
    uint32_t parity = 0;  // of the slot's current use
    int64_t next = 0;  // kSteal: the tile after this one, or -1
    for (int64_t tile = first_tile; tile >= 0 && tile < ntiles; tile = C::kSteal ? next : tile + step) {
        const int64_t first = tile * C::SU;
        const int64_t sig = first + own;
        const bool in_a = sig < batch, in_b = sig + 1 < batch;
        const int ea = in_a ? (int)in_exp[sig] : 0, eb = in_b ? (int)in_exp[sig + 1] : 0;
        if (!dead) {
            if (mbar_wait_bounded(&bars[slot], parity, wait_ns)) {
                inflight.completed(slot);
            } else {
                dead = true;
                atomicCAS(err, 0, kErrTimeout);
            }
        }
        if (C::kSteal && __any_sync(0xffffffffu, dead)) break;
        C2 v[C::E];
        pair_load<C, INV>(v, reinterpret_cast<const uint32_t*>(ring + slot * C::kSlotBytes) + pair_place<C, GI>(own), t);
        // the slot has been read: refill it; and the previous tile's copy out
        // of the exchange buffer has to be done before the exchange writes it
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            if constexpr (C::kSteal) {
                bool late = false;
                next = taker.take(wait_ns, late);
                if (late) atomicCAS(err, 0, kErrTimeout);
                if (next >= 0) {
                    issue(slot, next, parity ^ 1);
                    taker.request();
                }
            } else {
                if (!dead && !stall && tile + D * step < ntiles) issue(slot, tile + D * step, parity ^ 1);
            }
            bulk_wait_read();
        }
        if constexpr (C::kSteal) next = __shfl_sync(0xffffffffu, next, 0);
        if (++slot == D) {
            slot = 0;
            parity ^= 1;
        }
        pair_twist_dft<C, 0>(v, t, tw);
        pair_stages<C, 1>(v, xbuf, pr * C::N, t, tw);
        if (tile == first_tile) pdl_release();
        const float2 m = pair_max<C>(v);
        const C32Out oa = c32_out_scale<C::N>(m.x, ea, ls), ob = c32_out_scale<C::N>(m.y, eb, ls);
        const bool warp_dead = __any_sync(0xffffffffu, dead);
        if (t == 0 && in_a && !warp_dead) out_exp[sig] = (int8_t)oa.e;
        if (t == 0 && in_b && !warp_dead) out_exp[sig + 1] = (int8_t)ob.e;
        if constexpr (GO == 1) {  // whole 128-byte lines per access: straight to HBM
            pair_store<C, INV, true>(v, out + sig * C::N, t, in_a && !warp_dead, in_b && !warp_dead, oa.mult, ob.mult);
        } else {
            __syncwarp();  // the last exchange has been read
            pair_store<C, INV, false>(v, otile + pair_place<C, GO>(own), t, true, true, oa.mult, ob.mult);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && !warp_dead) {
                constexpr int kG = C::SU / GO;
                const int64_t left = batch - first;
                const int nsig = left < C::SU ? (int)left : C::SU;
                uint32_t* dst = out + first * C::N;
#pragma unroll
                for (int g = 0; g < GO; ++g) {
                    const int n = min(nsig - g * kG, kG);
                    if (n > 0)
                        bulk_copy_s2g(dst + g * kG * C::N, otile + pair_place<C, GO>(g * kG), (uint32_t)(n * C::N * 4));
                }
                bulk_commit();
            }
        }
    }
    if (lane == 0) {
        bulk_wait_all();
        if constexpr (C::kSteal) taker.drain(wait_ns);
        inflight.drain(bars, wait_ns);  // copies in flight after a wait gave up
    }
}

// N = 1024, 2048: thread 0 keeps the next D tiles of binary16 signals in
// flight into the ring (bounded waits, error word and stall test mode as in
// fft_stockham_ring_kernel); a slot is refilled at the barrier after stage 0
// has read it, so with D = 1 the copy runs behind the later stages.
template <class C, bool INV>
__global__ void __launch_bounds__(C::NT, C::MINB)
    fft_pair_c32_ring_kernel(const uint32_t* in, const int8_t* in_exp, uint32_t* out, int8_t* out_exp, int64_t batch,
                             const float2* __restrict__ tw, float scale, int* err, uint64_t wait_ns, int stall) {
    pdl_enter();
    pdl_release();
    constexpr int D = C::D;
    extern __shared__ __align__(16) float4 smem4[];
    unsigned char* base8 = reinterpret_cast<unsigned char*>(smem4);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base8 + C::kBarOffset);
    float* red = reinterpret_cast<float*>(base8 + C::kRedOffset);
    const int tid = threadIdx.x;
    const int pr = tid / C::T;
    const int t = tid % C::T;
    const int ls = log2_pow2(scale);
    const int64_t ntiles = (batch + C::S - 1) / C::S;
    dbg_set_err(err);

    RingInFlight inflight;  // thread 0's copies in flight
    TileTaker taker;        // thread 0's requests (kSteal)
    volatile int64_t* slot_tile = reinterpret_cast<volatile int64_t*>(base8 + C::kStealOffset + 24);  // kSteal
    // thread 0: `tile` into `slot`, for its use with phase parity `parity`
    auto issue = [&](int slot, int64_t tile, uint32_t parity) {
        const int64_t first = tile * C::S;
        const int64_t left = batch - first;
        const uint32_t bytes = (uint32_t)((left < C::S ? left : C::S) * C::N * 4);
        if constexpr (C::kSteal) *slot_tile = tile;
        mbar_arrive_expect_tx(&bars[slot], bytes);
        bulk_copy_g2s(base8 + C::kExchangeBytes + slot * C::kSlotBytes, in + first * C::N, bytes, &bars[slot]);
        inflight.issued(slot, parity);
    };
    if (tid == 0) {
        for (int d = 0; d < D; ++d) mbar_init(&bars[d], 1);
        if constexpr (C::kSteal) {
            taker.resp = base8 + C::kStealOffset;
            taker.bar = reinterpret_cast<uint64_t*>(base8 + C::kStealOffset + 16);
            mbar_init(taker.bar, 1);
        }
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0 && !stall) {
        for (int d = 0; d < D; ++d)
            if (blockIdx.x + (int64_t)d * gridDim.x < ntiles) issue(d, blockIdx.x + (int64_t)d * gridDim.x, 0);
    }
    if (C::kSteal && tid == 0) taker.request();
    bool dead = false;
    if (stall) {  // failure-detection test mode: a phase nothing will complete
        if (!mbar_wait_bounded(&bars[0], 0, wait_ns)) atomicCAS(err, 0, kErrTimeout);
        dead = true;
    }
    int64_t it = 0;
    for (int64_t tile = blockIdx.x; C::kSteal || tile < ntiles; tile += gridDim.x, ++it) {
        const int slot = (int)(it % D);
        if (!dead) {
            if (mbar_wait_bounded(&bars[slot], (uint32_t)((it / D) & 1), wait_ns)) {
                inflight.completed(slot);
            } else {
                dead = true;
                atomicCAS(err, 0, kErrTimeout);
            }
        }
        if constexpr (C::kSteal) tile = dead ? -1 : *slot_tile;
        const int64_t sig = tile * C::S + 2 * pr;
        bool in_a = false, in_b = false;
        int ea = 0, eb = 0;
        C2 v[C::E];
        // (a thread without a tile skips what no other thread waits for)
        if (!C::kSteal || tile >= 0) {
            in_a = sig < batch, in_b = sig + 1 < batch;
            ea = in_a ? (int)in_exp[sig] : 0, eb = in_b ? (int)in_exp[sig + 1] : 0;
            const uint32_t* src =
                reinterpret_cast<const uint32_t*>(base8 + C::kExchangeBytes + slot * C::kSlotBytes) + 2 * pr * C::N;
            pair_load<C, INV>(v, src, t);
            pair_twist_dft<C, 0>(v, t, tw);
            // (the previous tile's barrier before its store: the exchange buffer has been read)
            pair_scatter<C, 0>(v, smem4, pr * C::N, t);
        }
        fence_proxy_async_smem();
        // ... and every thread has read the slot: refill it
        if constexpr (C::kSteal) {
            // every thread leaves in the same iteration, also when one gave up
            if (__syncthreads_or(dead) || tile < 0) break;
            if (tid == 0) {
                bool late = false;
                const int64_t next = taker.take(wait_ns, late);
                if (late) atomicCAS(err, 0, kErrTimeout);
                if (next >= 0) {
                    issue(slot, next, (uint32_t)((it + 1) & 1));
                    taker.request();
                } else {
                    *slot_tile = -1;
                    mbar_arrive(&bars[slot]);
                }
            }
        } else {
            __syncthreads();
            if (tid == 0 && !dead && !stall && tile + (int64_t)D * gridDim.x < ntiles)
                issue(slot, tile + (int64_t)D * gridDim.x, (uint32_t)((it / D + 1) & 1));
        }
        pair_gather<C, 1>(v, smem4, pr * C::N, t);
        pair_twist_dft<C, 1>(v, t, tw);
        pair_stages<C, 2>(v, smem4, pr * C::N, t, tw);
        float2 m = pair_max<C>(v);
        const int warp = tid >> 5;
        if ((tid & 31) == 0) *reinterpret_cast<float2*>(red + 2 * warp) = m;
        __syncthreads();
        constexpr int W = C::T / 32;  // warps per pair
        m = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const float2 x = *reinterpret_cast<const float2*>(red + 2 * (warp / W * W + w));
            m = make_float2(fmaxf(m.x, x.x), fmaxf(m.y, x.y));
        }
        const C32Out oa = c32_out_scale<C::N>(m.x, ea, ls), ob = c32_out_scale<C::N>(m.y, eb, ls);
        const bool act_a = in_a && !dead, act_b = in_b && !dead;
        if (t == 0 && act_a) out_exp[sig] = (int8_t)oa.e;
        if (t == 0 && act_b) out_exp[sig + 1] = (int8_t)ob.e;
        pair_store<C, INV, true>(v, out + sig * C::N, t, act_a, act_b, oa.mult, ob.mult);
    }
    if (tid == 0) {
        if constexpr (C::kSteal) taker.drain(wait_ns);
        inflight.drain(bars, wait_ns);  // copies in flight after a wait gave up
    }
}

}  // namespace gbfft
