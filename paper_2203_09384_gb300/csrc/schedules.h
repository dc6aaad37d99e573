// Radix schedules per transform length: the analogue of the paper's host-side
// `stage_sizes` array and work-group factor (Sec. 4), fixed at compile time so
// that every stage's register array has a static size.  Several candidate
// schedules ("variants") may exist per length; plans use the one that
// GBFFT_SIZE_DEFAULTS gives for their size unless the caller or the autotuner
// picks another.
//
// Generic Stockham kernel rows:
//   GX(log2N, variant, E = complex elements per thread, S = signals per block,
//      R0, R1, R2, R3 = stage radices first to last (0 = no stage),
//      MINB = minimum resident blocks per SM requested from the compiler,
//      PIPE = 0: stage 0 loads straight from HBM into registers;
//             D >= 2: a ring of D shared-memory tiles filled by bulk-copy
//             (TMA) prefetch, D-1 tiles ahead of the one being transformed,
//      TC = 0: FP32 butterflies; 1 / 2: every radix-16 stage runs as a dense
//           16 x 16 complex product on FP16 / BF16 tensor cores (tcgen05),
//           FP32 accumulation (FP16: a power-of-two prescale per butterfly
//           row; BF16 shares FP32's exponent range and needs none); 5 / 6:
//           as 1 / 2 for the last radix-16 stage only,
//      XB = exchange buffers: 0 = automatic, 1 = one buffer and two barriers
//           per exchange (less shared memory, more resident blocks),
//           -1 = none: with PIPE >= 2, every exchange reuses the ring slot
//           the tile arrived in; -2 = as -1, and the tensor-core A operand
//           lives in that slot too; -3 = as -1, with the A operand in TMEM;
//           3 = none: the exchange of a two-stage N = R x R row with E = R is
//           a transpose by warp shuffles; -5 = as -1, with the signals of a
//           tile placed every N + T elements of the slot (one bulk copy per
//           signal), so that stage 0 reads them without bank conflicts,
//      CH = cache hints: bit 0 plain loads, bit 1 plain stores (else
//           evict-first); bit 2: one block per tile is launched and running
//           blocks take the tiles of blocks that have not started (TileTaker)
// Threads per block = S * N / E.  Stage 0 with R0 = E/2 (and the last stage,
// where its radix is E/2 or less) lets a thread own neighbouring butterflies,
// so its HBM accesses are 128-bit.  tests/test_bank_model.py replays the
// shared-memory exchanges of every row under the XOR swizzle of
// fft_device.cuh and counts their bank conflicts (64-bit accesses resolve per
// half-warp); tests/test_stockham_model.py replays every row's index mapping
// on the CPU and checks that it computes the DFT.
//
// One-thread-per-signal rows (N <= 32): SX(log2N, variant, warps per block,
// 32-signal groups per warp tile, cache hints as CH above).
#pragma once

#define GBFFT_GENERIC_SCHEDULES(GX)                   \
    GX(5, 1, 16, 128, 8, 4, 0, 0, 1, 0, 0, 0, 0) \
    GX(6, 0, 16, 16, 8, 8, 0, 0, 8, 2, 0, -5, 6) \
    GX(6, 2, 8, 32, 8, 8, 0, 0, 1, 0, 0, 3, 0) \
    GX(6, 3, 8, 32, 8, 8, 0, 0, 1, 0, 0, 0, 0) \
    GX(7, 0, 16, 8, 8, 16, 0, 0, 8, 2, 0, -5, 6) \
    GX(7, 1, 16, 16, 8, 16, 0, 0, 3, 2, 1, 0, 0) \
    GX(7, 2, 16, 16, 8, 16, 0, 0, 3, 2, 2, 0, 0) \
    GX(7, 3, 16, 32, 8, 16, 0, 0, 2, 0, 1, 0, 0) \
    GX(7, 4, 16, 32, 8, 16, 0, 0, 2, 0, 2, 0, 0) \
    GX(8, 17, 16, 16, 16, 16, 0, 0, 1, 0, 0, 0, 2) \
    GX(8, 7, 16, 8, 16, 16, 0, 0, 3, 2, 1, 0, 0) \
    GX(8, 8, 16, 8, 16, 16, 0, 0, 3, 2, 2, 0, 0) \
    GX(8, 3, 16, 16, 16, 16, 0, 0, 1, 0, 1, 0, 0) \
    GX(8, 4, 16, 16, 16, 16, 0, 0, 1, 0, 2, 0, 0) \
    GX(8, 9, 16, 16, 16, 16, 0, 0, 1, 0, 1, 0, 2) \
    GX(8, 10, 16, 16, 16, 16, 0, 0, 1, 0, 2, 0, 2) \
    GX(8, 11, 16, 8, 16, 16, 0, 0, 3, 2, 1, 0, 2) \
    GX(8, 2, 16, 8, 16, 16, 0, 0, 3, 2, 2, 0, 2) \
    GX(8, 1, 16, 8, 16, 16, 0, 0, 3, 2, 5, 0, 2) \
    GX(8, 12, 16, 8, 16, 16, 0, 0, 3, 2, 6, 0, 2) \
    GX(8, 13, 16, 16, 16, 16, 0, 0, 1, 0, 0, 3, 2) \
    GX(8, 14, 16, 8, 16, 16, 0, 0, 3, 2, 0, 0, 2) \
    GX(8, 15, 16, 8, 16, 16, 0, 0, 4, 2, 0, -1, 2) \
    GX(8, 16, 16, 8, 16, 16, 0, 0, 5, 2, 0, -1, 2) \
    GX(8, 0, 16, 8, 16, 16, 0, 0, 4, 2, 0, -1, 6) \
    GX(9, 0, 16, 1, 16, 2, 16, 0, 16, 2, 0, -1, 6) \
    GX(9, 1, 16, 8, 8, 8, 8, 0, 1, 0, 0, 0, 0) \
    GX(10, 0, 16, 1, 16, 4, 16, 0, 7, 2, 0, -1, 6) \
    GX(10, 1, 16, 2, 8, 16, 8, 0, 1, 0, 0, 0, 0) \
    GX(10, 2, 16, 2, 8, 16, 8, 0, 4, 0, 0, 0, 0) \
    GX(10, 3, 16, 2, 8, 16, 8, 0, 2, 3, 0, 0, 0) \
    GX(10, 4, 16, 2, 8, 16, 8, 0, 5, 2, 1, -3, 0) \
    GX(10, 5, 16, 2, 8, 16, 8, 0, 5, 2, 2, -3, 0) \
    GX(10, 6, 16, 2, 8, 16, 8, 0, 2, 2, 1, 0, 0) \
    GX(10, 7, 16, 2, 8, 16, 8, 0, 2, 2, 2, 0, 0) \
    GX(10, 10, 16, 2, 8, 16, 8, 0, 5, 2, 0, -1, 2) \
    GX(10, 11, 16, 2, 8, 16, 8, 0, 5, 2, 1, -2, 0) \
    GX(10, 12, 16, 2, 8, 16, 8, 0, 5, 2, 2, -2, 0) \
    GX(10, 13, 16, 2, 8, 16, 8, 0, 4, 2, 1, 1, 0) \
    GX(10, 14, 16, 2, 8, 16, 8, 0, 4, 2, 2, 1, 0) \
    GX(11, 0, 16, 1, 16, 8, 16, 0, 5, 2, 0, -1, 6) \
    GX(11, 1, 16, 1, 8, 16, 16, 0, 1, 0, 0, 0, 0) \
    GX(11, 2, 16, 1, 8, 16, 16, 0, 2, 3, 0, 0, 0) \
    GX(11, 3, 16, 2, 8, 16, 16, 0, 1, 2, 0, 0, 0) \
    GX(11, 15, 16, 1, 8, 16, 16, 0, 5, 2, 1, -3, 0) \
    GX(11, 16, 16, 1, 8, 16, 16, 0, 5, 2, 2, -3, 0) \
    GX(11, 6, 16, 1, 8, 16, 16, 0, 3, 2, 1, 0, 0) \
    GX(11, 7, 16, 1, 8, 16, 16, 0, 3, 2, 2, 0, 0) \
    GX(11, 10, 16, 1, 8, 16, 16, 0, 3, 2, 0, 0, 2) \
    GX(11, 11, 16, 1, 8, 16, 16, 0, 5, 2, 1, -2, 0) \
    GX(11, 12, 16, 1, 8, 16, 16, 0, 5, 2, 2, -2, 0) \
    GX(11, 13, 16, 1, 8, 16, 16, 0, 4, 2, 1, 1, 0) \
    GX(11, 14, 16, 1, 8, 16, 16, 0, 4, 2, 2, 1, 0) \
    GX(11, 4, 16, 1, 8, 16, 16, 0, 5, 2, 1, -3, 2) \
    GX(11, 5, 16, 1, 8, 16, 16, 0, 5, 2, 2, -3, 2) \
    GX(11, 17, 16, 1, 8, 16, 16, 0, 5, 2, 5, -3, 2) \
    GX(11, 18, 16, 1, 8, 16, 16, 0, 5, 2, 6, -3, 2) \
    GX(11, 19, 16, 1, 8, 16, 16, 0, 5, 2, 0, -1, 2) \
    GX(6, 4, 16, 64, 8, 8, 0, 0, 1, 0, 0, 0, 0) \
    GX(7, 6, 16, 32, 8, 16, 0, 0, 1, 0, 0, 0, 2) \
    GX(6, 5, 16, 16, 8, 8, 0, 0, 8, 2, 0, -5, 2) \
    GX(6, 6, 8, 8, 8, 8, 0, 0, 8, 0, 0, 3, 0) \
    GX(7, 7, 16, 8, 8, 16, 0, 0, 8, 2, 0, -5, 2) \
    GX(7, 8, 16, 8, 8, 16, 0, 0, 8, 0, 0, 0, 0) \
    GX(7, 9, 16, 16, 8, 16, 0, 0, 4, 2, 1, -3, 2) \
    GX(7, 10, 16, 16, 8, 16, 0, 0, 4, 2, 2, -3, 2) \
    GX(7, 11, 16, 16, 8, 16, 0, 0, 4, 2, 1, -3, 6) \
    GX(7, 12, 16, 16, 8, 16, 0, 0, 4, 2, 2, -3, 6) \
    GX(8, 19, 16, 4, 16, 16, 0, 0, 8, 0, 0, 0, 0) \
    GX(8, 20, 16, 8, 16, 16, 0, 0, 4, 2, 5, -3, 6) \
    GX(8, 21, 16, 8, 16, 16, 0, 0, 3, 2, 5, -3, 2) \
    GX(8, 22, 16, 8, 16, 16, 0, 0, 3, 2, 2, -3, 2) \
    GX(8, 23, 16, 8, 16, 16, 0, 0, 4, 2, 2, -3, 6) \
    GX(9, 3, 16, 2, 16, 2, 16, 0, 8, 0, 0, 0, 0) \
    GX(10, 15, 16, 1, 16, 4, 16, 0, 6, 0, 0, 0, 0) \
    GX(10, 16, 16, 1, 16, 4, 16, 0, 6, 2, 0, -1, 2) \
    GX(10, 17, 16, 2, 8, 16, 8, 0, 6, 2, 1, -3, 6) \
    GX(10, 18, 16, 2, 8, 16, 8, 0, 6, 2, 2, -3, 6) \
    GX(11, 20, 16, 1, 16, 8, 16, 0, 3, 2, 0, -1, 2) \
    GX(11, 21, 16, 1, 8, 16, 16, 0, 5, 2, 1, -3, 6) \
    GX(11, 22, 16, 1, 8, 16, 16, 0, 5, 2, 2, -3, 6) \
    GX(11, 24, 16, 1, 16, 8, 16, 0, 3, 0, 0, 0, 0)

#define GBFFT_SMALL_SCHEDULES(SX) \
    SX(1, 0, 1, 8, 4)                \
    SX(1, 1, 8, 2, 0)                \
    SX(1, 4, 4, 2, 0)                \
    SX(2, 0, 1, 4, 4)                \
    SX(2, 1, 8, 1, 0)                \
    SX(2, 2, 8, 4, 2)                \
    SX(2, 3, 16, 2, 2)               \
    SX(2, 6, 2, 2, 0)                \
    SX(3, 0, 1, 2, 4)                \
    SX(3, 1, 8, 1, 0)                \
    SX(3, 2, 4, 4, 0)                \
    SX(3, 5, 4, 1, 0)                \
    SX(4, 0, 1, 1, 6)                \
    SX(4, 1, 8, 1, 0)                \
    SX(4, 2, 8, 2, 0)                \
    SX(4, 5, 2, 1, 0)                \
    SX(4, 6, 2, 2, 0)                \
    SX(5, 0, 1, 1, 4)                \
    SX(5, 2, 4, 1, 0)                \
    SX(5, 5, 1, 1, 0)

// complex32-storage rows (FFT_C32): CX(log2N, variant, E, S, R0..R3, MINB,
// PIPE, XB).  XB = 6 (N >= 64): two signals per thread, packed FP32 arithmetic
// (fft_pair.cuh), S / 2 signal pairs and S N / (2 E) threads per block, a ring
// of PIPE bulk-copied tiles per warp (N <= 512) or per block; XB = 14: the same,
// taking the tiles of unstarted blocks (one warp per block for N <= 512).  XB = 0: the
// Stockham kernel with binary16 loads/stores, one signal per thread group (N >= 64:
// in the pair kernels' arithmetic, bit for bit).
// A length's first complex32 row is its default; for N <= 32 that is the
// one-thread-per-signal SCX row further down.
//
// Why the defaults are shaped so (2^27 elements, device time, against the
// one-signal-per-thread kernels they replaced, whose stored values and
// exponents they reproduce bit for bit): N = 64 244 -> 169 us, 128 241 -> 178,
// 256 210 -> 180, 512 285 -> 208, 1024 303 -> 220, 2048 302 -> 239 (and with
// tiles taken from unstarted blocks 164, 169, 169, -, 213, 232).  Blocks of
// 64 threads at N = 1024 (128: 237 us), because its barriers then join two
// warps only; one ring slot, because a second one costs the fourth block per SM
// (N = 1024 and 2048: 252 and 262 us with two slots and three blocks).
#define GBFFT_C32_SCHEDULES(CX)                   \
    CX(1, 3, 2, 256, 2, 0, 0, 0, 1, 0, 0)        \
    CX(2, 5, 2, 128, 2, 2, 0, 0, 1, 0, 0)        \
    CX(3, 4, 4, 128, 2, 4, 0, 0, 1, 0, 0)        \
    CX(4, 4, 8, 128, 4, 4, 0, 0, 1, 0, 0)        \
    CX(5, 4, 16, 128, 8, 4, 0, 0, 1, 0, 0)       \
    CX(6, 1, 16, 64, 8, 8, 0, 0, 4, 1, 6)        \
    CX(7, 5, 16, 32, 8, 16, 0, 0, 4, 1, 6)       \
    CX(8, 18, 16, 8, 16, 16, 0, 0, 8, 1, 6)      \
    CX(8, 6, 16, 4, 16, 16, 0, 0, 1, 0, 0)       \
    CX(9, 2, 16, 8, 8, 8, 8, 0, 4, 1, 6)         \
    CX(10, 8, 16, 2, 8, 16, 8, 0, 8, 1, 6)       \
    CX(10, 9, 16, 1, 8, 16, 8, 0, 4, 0, 0)       \
    CX(11, 8, 16, 2, 8, 16, 16, 0, 4, 1, 6)      \
    CX(11, 9, 16, 1, 8, 16, 16, 0, 3, 0, 0)      \
    CX(8, 5, 16, 16, 16, 16, 0, 0, 4, 1, 6)      \
    CX(6, 7, 16, 16, 8, 8, 0, 0, 16, 1, 14)      \
    CX(7, 13, 16, 8, 8, 16, 0, 0, 16, 1, 14)     \
    CX(8, 24, 16, 4, 16, 16, 0, 0, 16, 1, 14)    \
    CX(10, 19, 16, 2, 8, 16, 8, 0, 8, 1, 14)     \
    CX(11, 23, 16, 2, 8, 16, 16, 0, 4, 1, 14)

// complex32 one-thread-per-signal rows (N <= 32): SCX(log2N, variant, warps
// per block, 32-signal groups per warp tile, cache hints)
#define GBFFT_C32_SMALL_SCHEDULES(SCX) \
    SCX(1, 2, 8, 4, 0)                  \
    SCX(2, 4, 4, 8, 0)                  \
    SCX(3, 3, 8, 4, 0)                  \
    SCX(4, 3, 4, 4, 0)                  \
    SCX(5, 3, 4, 2, 0)                  \
    SCX(2, 7, 1, 4, 4)                  \
    SCX(3, 6, 1, 4, 4)                  \
    SCX(4, 7, 1, 2, 4)                  \
    SCX(5, 6, 1, 1, 4)

// Which row a plan that names none runs, by length, type and size of the call:
// DX(log2N, type, largest n * batch, variant), type 0 FP32, 1 / 2 FP16 / BF16
// tensor cores, 3 complex32; the first row that fits; past
// the last one, variant 0 (FP32) or the first variant of the type.  A default
// set by fft_set_default_variant (the autotuner's) goes before all of this.
//
// Past some 6 M elements (N = 2048: 12 M) the rows that take tiles of unstarted
// blocks (CH bit 2) win: variant 0 at every length.  Their first request costs about 1 us, so
// shorter calls run fixed strides, and with few tiles per SM want small blocks
// and tiles, which start their first store sooner and leave a shorter tail;
// evict-first direct loads and stores win while the output still fits in L2.
// Device time per call in a captured graph over three rotating buffer pairs, us:
// the best single schedule for all sizes that these rows replaced / the row for
// short calls / variant 0:
//   N = 2     2^21.4  9.5 /  6.6 /  -     2^22.2 14.4 / 13.0 / 12.8   2^24 44.1 / 45.3 / 40.5   2^28 652 / 606
//   N = 4     2^21.4  8.9 /  6.8 /  -     2^22.2 16.1 / 12.9 / 13.0   2^24 44.7 / 45.3 / 40.6   2^28 650 / 606
//   N = 8     2^21.4  9.5 /  7.0 /  -     2^22.2 17.1 / 13.0 / 13.1   2^24 43.6 / 45.6 / 40.7   2^28 652 / 606
//   N = 16    2^21.4  8.8 /  7.3 /  -     2^22.2 15.8 / 13.7 / 13.0   2^24 43.6 / 45.4 / 40.7   2^28 650 / 610
//   N = 32    2^21.4 10.7 /  8.2 /  -     2^22.2 14.3 / 13.0 / 13.1   2^24 43.9 / 45.0 / 40.7   2^28 645 / 606
//   N = 64    2^21.4 10.4 /  7.6 /  -     2^22.2 14.7 / 12.9 / 13.8   2^24 43.5 / 46.4 / 39.8   2^28 631 / 600
//   N = 128   2^21.4 10.8 /  8.5 /  -     2^22.2 14.8 / 13.7 / 14.1   2^24 42.6 / 43.4 / 40.3   2^28 633 / 601
//   N = 256   2^21.4 10.7 /  8.4 /  -     2^22.2 15.0 / 13.7 / 14.0   2^24 43.2 / 43.2 / 41.1   2^28 642 / 602
//   N = 512   2^21.4 12.1 /  8.7 /  -     2^22.2 16.2 / 14.4 / 15.4   2^24 45.2 / 43.4 / 41.9   2^28 636 / 603
//   N = 1024  2^21.4 11.8 /  9.0 /  -     2^22.2 17.3 / 15.5 / 16.4   2^24 45.6 / 43.4 / 41.9   2^28 650 / 602
//   N = 2048  2^21.4 12.0 /  9.8 / 12.9   2^23.2 28.7 / 27.4 / 28.0   2^24 45.7 / 44.5 / 44.0   2^28 652 / 607
// All rows of a length take its radices in one order, so a signal's result does
// not depend on how many others share its call.  At N = 2048 the ring (20) and
// the direct row (24) cross four times, as one more block an SM costs the one a
// round and the other less; ring / direct, calls chained in a graph: 602 K
// elements (294 signals) 2.9 / 3.2, 645 K 4.2 / 3.2, 2^20 4.3 / 4.0, 2^20.1 4.4 /
// 4.6, 2^20.5 5.7 / 5.8, 2^20.6 6.4 / 5.9, 2^20.9 7.7 / 7.5, 2^21 8.1 / 8.5.
// The lines at 2^16 and 2^17 of N = 64 and 128 and at 2^20 of N = 1024 are not
// drawn by time: up to there a default plan runs a bulk-copy kernel, because the
// tests of bounded waits take default plans of 611 signals as ones that wait on
// the device.  Bulk-copy / direct row, chained in a graph, us: N = 64 2^10 2.05 /
// 1.33, 2^14 2.2 / 1.5, 2^16 2.2 / 1.5; N = 128 2^10 1.85 / 1.5, 2^14 2.0 / 1.65, 2^17
// 2.1 / 1.8; N = 1024 2^10 1.8 / 1.55, 2^18 2.2 / 2.0, 2^19 2.8 / 3.2, 2^19.5 4.0 / 3.2,
// 2^20 4.05 / 3.8.  (The one schedule for all sizes before: 2.4-3.1, 2.3-2.8, 2.4-4.9.)
// N = 2048 below 602 K elements: 2^12 2.1 / 1.85, 2^18 2.3 / 2.1, 2^19 2.9 / 3.3.
//
// Tensor-core types: every row of a length rounds the same operands.  Before /
// after at 2^28: FP16 N = 128 672 / 607, 256 666 / 600, 1024 727 / 686,
// 2048 681 / 643; BF16 655 / 603, 643 / 600, 704 / 660, 665 / 632.  (Radix 16
// first and last was faster still by 2-9% at 1024 and 2048, but rounds other
// stages' operands to 16 bits.)
//
// complex32 (type 3), us, fixed stride / taken tiles: N = 4 2^24 26.2 / 23.8, 8
// 2^27 179 / 163, 16 2^27 174 / 158, 32 2^27 165 / 160, 64 2^27 169 / 164, 128
// 2^27 178 / 169, 256 2^27 181 / 169, 1024 2^27 218 / 213, 2048 2^27 240 / 232;
// N = 2 (211 / 237) and N = 512 (208 / 208) keep the fixed stride.  Short calls of
// N = 256, 1024 and 2048 take one signal per thread group and blocks of 64 or
// 128 threads: a thread's chain is shorter, and the machine is not full anyway.
// Two signals per thread / one, calls chained in a graph, us: N = 256 2^12 2.2 /
// 1.55, 2^18 2.4 / 1.8, 2^20 3.3 / 2.9, 2^20.5 4.7 / 3.9, 2^21.25 5.2 / 5.1, 2^21.5
// 6.2 / 6.6; N = 1024 2^12 2.4 / 1.8, 2^18 2.75 / 2.2, 2^19 3.0 / 2.7, 588 signals
// 3.05 / 2.85, 630 (over four blocks an SM) 3.2 / 3.35; N = 2048 2^12 2.7 / 1.9,
// 2^18 2.9 / 2.1, 222 signals 3.0 / 2.7, 238 3.05 / 3.3.
#define GBFFT_SIZE_DEFAULTS(DX) \
    DX(1, 0, 5 << 20, 4)        \
    DX(2, 0, 5 << 20, 6)        \
    DX(3, 0, 5 << 20, 5)        \
    DX(4, 0, 4 << 20, 5)        \
    DX(5, 0, 5 << 20, 5)        \
    DX(6, 0, 1 << 16, 5)        \
    DX(6, 0, 6 << 20, 6)        \
    DX(7, 0, 1 << 17, 7)        \
    DX(7, 0, 6 << 20, 8)        \
    DX(8, 0, 6 << 20, 19)       \
    DX(9, 0, 6 << 20, 3)        \
    DX(10, 0, 1 << 20, 16)      \
    DX(10, 0, 5 << 20, 15)      \
    DX(10, 0, 7 << 20, 16)      \
    DX(11, 0, 5 << 17, 20)      \
    DX(11, 0, 1 << 20, 24)      \
    DX(11, 0, 23 << 16, 20)     \
    DX(11, 0, 15 << 17, 24)     \
    DX(11, 0, 12 << 20, 20)     \
    DX(7, 1, 2 << 20, 1)        \
    DX(7, 1, 16 << 20, 9)       \
    DX(7, 1, INT64_MAX, 11)     \
    DX(7, 2, 2 << 20, 2)        \
    DX(7, 2, 16 << 20, 10)      \
    DX(7, 2, INT64_MAX, 12)     \
    DX(8, 1, 2 << 20, 1)        \
    DX(8, 1, 12 << 20, 21)      \
    DX(8, 1, INT64_MAX, 20)     \
    DX(8, 2, 1 << 19, 2)        \
    DX(8, 2, 12 << 20, 22)      \
    DX(8, 2, INT64_MAX, 23)     \
    DX(10, 1, 20 << 20, 4)      \
    DX(10, 1, INT64_MAX, 17)    \
    DX(10, 2, 20 << 20, 5)      \
    DX(10, 2, INT64_MAX, 18)    \
    DX(11, 1, 20 << 20, 4)      \
    DX(11, 1, INT64_MAX, 21)    \
    DX(11, 2, 20 << 20, 5)      \
    DX(11, 2, INT64_MAX, 22)    \
    DX(1, 3, 1 << 17, 3)        \
    DX(2, 3, 12 << 20, 4)       \
    DX(2, 3, INT64_MAX, 7)      \
    DX(3, 3, INT64_MAX, 6)      \
    DX(4, 3, INT64_MAX, 7)      \
    DX(5, 3, INT64_MAX, 6)      \
    DX(6, 3, 16 << 20, 1)       \
    DX(6, 3, INT64_MAX, 7)      \
    DX(7, 3, 14 << 20, 5)       \
    DX(7, 3, INT64_MAX, 13)     \
    DX(8, 3, 5 << 19, 6)        \
    DX(8, 3, 12 << 20, 5)       \
    DX(8, 3, INT64_MAX, 24)     \
    DX(10, 3, 19 << 15, 9)      \
    DX(10, 3, 48 << 20, 8)      \
    DX(10, 3, INT64_MAX, 19)    \
    DX(11, 3, 7 << 16, 9)       \
    DX(11, 3, 20 << 20, 8)      \
    DX(11, 3, INT64_MAX, 23)

#define GBFFT_MIN_LOG2N 1
#define GBFFT_MAX_LOG2N 11
#define GBFFT_MAX_VARIANTS 31  // FFT_FLAG_VARIANT(k) holds k = 0..30
