// das_attention.cu -- depth-asynchronous attention (Eqs. 2-3, Sec. 3.2) and
// the full-depth verify attention (Sec. 3.4) on the 5th-generation tensor
// cores of sm_103a (tcgen05, accumulators in tensor memory).
//
// Work decomposition: every (sequence, kv head) pair owns ceil(P/64) prefix
// tiles plus one block tile; all pairs' tiles form one list of N tiles, and
// CTA c of a persistent grid of C CTAs (one per SM) takes the c-th of C
// equal ranges of that list (block tiles weighted for their extra cost, see
// kBlockBytes), cut into segments at pair boundaries.  A segment that covers
// its pair writes the output.  The others write a partial (O / l and the
// log-sum-exp of their keys) to the workspace, and merge_kernel, launched
// right after as a programmatic dependent, combines each split pair's
// partials by log-sum-exp (8, 4 or 2 segments' loads in flight, chosen per
// launch).
//
// The products are formed transposed: keys and head dimensions are the rows
// (M = 128) of the MMAs and the pair's query rows (G * max_block of them, ordered
// i * G + g as a {64, G, max_block} box lands, rounded up to N = 16, 32 or 64)
// their columns:
//     S^T = K Q^T    two 64-key tiles (a step) at a time, K from shared memory
//     O^T += V^T P^T V as it lies in shared memory (MN-major)
//     l   += 1 P^T   the sums of P as rounded
// so that MMAs and softmax shrink with the number of query rows, the MMAs run
// at the full M = 128 rate, and a softmax thread owns one key: no exchange
// between threads is needed in a step but one barrier (with rows in the lanes,
// a 64-key tile cost a softmax warp about 1000 cycles of dependent latency, and
// its exchanges; D = 64 and e4m3 tiles, 16 KB, could not be consumed faster).
//
// One CTA = four softmax warps (eight for N = 64, two groups of 32 columns) +
// a producer, a P V and an S warp (+ four conversion warps for e4m3).
//   S warp: loads K, a slot per step, and issues S^T (and, of a segment's first
//     step, the scores of a few keys the other way round, from which each row's
//     first reference is taken).  e4m3 keys: two e4m3 or three e5m2 passes over
//     the query rows split into that many parts, see split_q.
//   producer warp: loads the query rows and V; the first steps' K too.
//   P V warp: O^T += V^T P^T and the row sums, once P is in shared memory.
//   conversion warps: the query split, and e4m3 V widened to f16 tiles.
//   softmax warps: thread j takes key j's scores of its group's query rows from
//     tensor memory, subtracts the rows' references (base 2; a reference only
//     moves when a score exceeds it by 2^8, or 2^12 for f16 P: then O and the sums
//     are rescaled in tensor memory), and writes P = 2^(s - m) as bf16 (f16
//     for widened values) into the swizzled, MN-major P buffer.  The sums of the
//     fp32 weights (for the lse) stay per thread, in tensor memory, and are added
//     up at a segment's end; the sum of the rounded weights normalises O, so that
//     the output is a convex combination of the values with exactly the
//     weights the tensor core used.
// It serves 64-wide heads and e4m3 operands over long ranges; bf16 calls with 128-wide
// heads, and short ranges, take the kernel of das_rows.cu (attn_short_ranges).
// Measured (us per call with its merge, das_rows.cu's kernel -> this one): ragged B8
// D64 29.6 -> 27.9, e4m3 keys B4 P16384 43.6 -> 42.3, e4m3 keys and values B8 ragged
// 51.1 -> 40.6.  Bound by the softmax step (about 2000 cycles) where keys and values
// are e4m3, and everywhere by how well the roles' code fits the instruction caches:
// warps stand for want of an instruction as long as they wait for anything else.
//
// The kernel is launched as a programmatic dependent of the previous kernel
// in the stream: barrier set-up, the tensor-memory allocation, the work plan
// (from lengths read before the wait, checked again after it) and an L2
// prefetch of the first tiles overlap the previous kernel's tail; nothing
// global is written, and nothing read is used unchecked, before
// griddepcontrol.wait.  Every wait is bounded (2 s); a time-out sets the
// status word and stops the CTA's waits.  Tensor memory is freed before the CTA
// exits.
#include <algorithm>
#include <atomic>

#include "das_tc.h"

namespace das {
namespace tc {
namespace {

constexpr int kPBufs = 2;            // P buffers
// P = 2^(s - m + shift).  A row's reference m moves only when log2 P would pass kTop:
// as in das_rows.cu by 2^8 for bf16 P, so that the fp32 sums of P V hold values up to
// about 2^(127 - 8) over the number of keys, and a row's largest weights mostly sit at
// or just below a reference (bf16 holds 1 exactly, and its relative error is half as
// large just below 1 as just above).  Moving at 2^60 instead cost both: infinities
// for values above about 2^60, and more error against 64 bits (batched 1.99e-3
// against 1.95e-3, e4m3 keys B4 P16384 1.88e-3 against 1.84e-3).  f16 P (widened values)
// holds 2^-25 to 2^16: kTop of 2^15, and a shift so that a long flat tail under one
// strong key vanishes from O only below 2^-28 of it (e4m3 keys and values, two calls
// of B8 ragged: shift 0 87.9 us, 3 89.6, 5 93.2, 7 98.5).
// When a row moves, all rows of the group move up to their maximum over the step:
// fewer moves, each of which costs a CTA about 1 us (ragged B8 D64 56.7 instead of
// 61.4 us, e4m3 keys B4 P16384 86.0 instead of 89.5).
// A segment's first reference is the maximum over its first kRefKeys keys.
constexpr float kTopBf16 = 8.f, kTopF16 = 15.f, kShiftF16 = 3.f;
constexpr int kRefKeys = 32;
constexpr float kNoRef = 3e38f;      // -reference of a row without a finite score yet

// Shared memory of one CTA.  A step is one or two consecutive 64-key tiles of
// a pair (two unless the pair or the range ends, or the second would be a
// block tile of another element type); its keys are the M = 128 rows of the
// S^T MMA.
//   K ring: one slot per step, [128 keys][D] (tile h at key rows 64 h).
//   V ring: one slot per tile, [64 keys][D]; with e4m3 values only prefix
//     tiles use it, and the conversion warps widen each into a slot of the W
//     ring, from which the P V MMAs then read every tile.
//   bf16 tiles are D / 64 panels of 128-byte rows, 128-byte swizzled; e4m3 key
//   tiles are rows of D bytes, swizzled over the row (128 or 64 bytes), e4m3
//   value tiles plain rows.
// Ring depths: V 4 tiles at D = 128 (5 were 0.4 % slower: more loads in flight than
// needed delay the ones needed first); K 3 slots or, for wide bf16 steps, as many as
// fit; S buffers: as many as tensor memory holds, a K slot is free once S is.
template <int D, bool KF8, bool VF8, int N>
struct Layout {
    static_assert(N == 16 || N == 32 || N == 64, "query columns: 16, 32 or 64");
    static constexpr bool kConv = KF8 || VF8;
    static constexpr int kGroups = N == 16 ? 1 : 2;  // softmax groups of four warps
    static constexpr int kCols = N / kGroups;        // query columns of a group
    static constexpr int kSoftWarps = 4 * kGroups;
    static constexpr int kThreads = (kSoftWarps + 3 + (kConv ? kConvWarps : 0)) * 32;
    static constexpr int kPanels = D / 64;
    static constexpr int kTileBytes = kTileKeys * D * 2;                // a bf16 K or V tile
    static constexpr int kKBytes = 2 * kTileKeys * D * (KF8 ? 1 : 2);   // a K slot
    static constexpr int kVBytes = kTileKeys * D * (VF8 ? 1 : 2);       // a V slot
    static constexpr int kKSlots = KF8 || N == 16 ? 3 : D == 64 ? 4 : 2;
    static constexpr int kVSlots = VF8 ? 4 : D == 64 ? 8 : 4;
    static constexpr int kWSlots = VF8 ? (D == 64 ? 4 : 3) : 0;
    static constexpr int kSBufs = KF8 && D == 128 && N == 64 ? 2 : 3;  // S buffers in tensor memory
    static constexpr int kQBytes = N * D * 2;    // one bf16 query buffer
    static constexpr int kQ8Bytes = N * D;       // one 8-bit query part
    // (e4m3 keys) parts of the query split (split_q)
    static constexpr int kParts = VF8 || D == 64 ? 3 : 2;
    static constexpr int kPBytes = 2 * kTileKeys * N * 2;
    static constexpr int kVOff = kKSlots * kKBytes;
    static constexpr int kWOff = kVOff + kVSlots * kVBytes;
    static constexpr int kQOff = kWOff + kWSlots * kTileBytes;
    static constexpr int kQ8Off = kQOff + 2 * kQBytes;  // the parts
    static constexpr int kPOff = kQ8Off + (KF8 ? kParts * kQ8Bytes : 0);
    // (D = 64) 16 keys x 64 ones (bf16, then f16): the second half of the P V A operand
    static constexpr int kOnesOff = kPOff + kPBufs * kPBytes;
    static constexpr int kBarOff = kOnesOff + (D == 128 ? 0 : VF8 ? 4096 : 2048);
    // barriers: kfull / kempty[kKSlots], vfull / vempty[kVSlots], wready /
    // wfree[kWSlots], qfull[2], qempty[2], qsplit[2], sready / sfree[kSBufs],
    // pready[2], pvdone[2], drain[2], rready
    static constexpr int kNumBars = 2 * (kKSlots + kVSlots + kWSlots) + 13 + 2 * kSBufs;
    static constexpr int kMiscOff = kBarOff + (kNumBars + 1) / 2 * 16;  // tensor memory base, abort flag
    static constexpr int kLenOff = kMiscOff + 16;  // lengths read before the dependency wait
    static constexpr int kNmOff = kLenOff + 64 * 4;       // -reference of each query row
    static constexpr int kAlphaOff = kNmOff + N * 4;      // rescale factors
    static constexpr int kRedOff = kAlphaOff + N * 4;     // [4 warps][N]
    static constexpr int kLrOff = kRedOff + 4 * N * 4;    // rounded row sums
    static constexpr int kQscOff = kLrOff + N * 4;        // score scale of each row, per buffer
    static constexpr int kBytes = kQscOff + (KF8 ? 2 * N * 4 : 0) + 1024;  // + alignment slack
    // tensor memory columns: S buffers, O, row sums (D = 128), then what every
    // lane needs of each query row -- minus its reference and (e4m3 keys) its
    // score scale, kept here because shared memory is what the kernel runs out
    // of -- the lanes' parts of the sums of the fp32 weights (registers: 32 more
    // would spill), and 8 columns of bf16 ones (and 8 of f16 ones), the A operand whose
    // products are row sums
    static constexpr int kOCol = kSBufs * N;
    static constexpr int kLCol = kOCol + N;
    static constexpr int kNmCol = kLCol + (D == 128 ? N : 0);
    static constexpr int kScCol = kNmCol + N;
    static constexpr int kSumCol = kScCol + (KF8 ? N : 0);
    static constexpr int kRefCol = kSumCol + N;  // scores of a segment's first keys, rows in lanes
    static constexpr int kOnesCol = kRefCol + kRefKeys;
    static constexpr int kTmemCols = N == 16 ? 256 : 512;
    static_assert(kOnesCol + (VF8 ? 16 : 8) <= kTmemCols, "tensor memory");
    static_assert(kKBytes % 1024 == 0 && kVBytes % 1024 == 0 && kQ8Bytes % 1024 == 0 &&
                      kPBytes % 1024 == 0 && kNmOff % 16 == 0,
                  "swizzled tiles need 1024-byte alignment");
    static_assert(kBytes <= 232448, "shared memory per CTA");
};

// Segment at walk position w: the pair's tiles of the range, `left` tiles of
// which remain.
struct Seg {
    int tiles;   // tiles of the segment
    int pairs;   // tiles that go two to a step (all but a block tile of another element type)
    int steps;
    int nfull;   // leading steps of two full prefix tiles
    bool blk;    // the segment ends with the pair's block tile
};
template <bool kConv>
__device__ __forceinline__ Seg segment(const Walk &w, int left) {
    Seg s;
    s.tiles = min(w.nt - w.t, left);
    s.blk = w.t + s.tiles == w.nt;
    s.pairs = s.tiles - (kConv && s.blk ? 1 : 0);
    s.steps = ((s.pairs + 1) >> 1) + s.tiles - s.pairs;
    s.nfull = max(0, min(w.t + s.tiles, w.P >> 6) - w.t) >> 1;
    return s;
}
// Tiles of step i.
__device__ __forceinline__ int step_tiles(const Seg &s, int i) {
    return 2 * i + 2 <= s.pairs ? 2 : 1;
}
__device__ __forceinline__ void walk_segment(const AttnParams &p, Walk &w, const Seg &s) {
    w.t += s.tiles - 1;
    walk_next(p, w);
}
// Valid keys of tile t of the walk's pair.
__device__ __forceinline__ int tile_keys(const Walk &w, int t) {
    return t == w.nt - 1 ? w.T : min(kTileKeys, w.P - t * kTileKeys);
}
// Ring position: slot and the parity of the phase being waited for.
template <int SLOTS>
struct Ring {
    int slot = 0;
    uint32_t parity = 0;
    __device__ __forceinline__ void next() {
        if (++slot == SLOTS) {
            slot = 0;
            parity ^= 1;
        }
    }
};

// Split of the query rows for e4m3 keys.  Row r of the bf16 query buffer q
// (128-byte-swizzled panels of [N rows][64 dims]) becomes PARTS 8-bit rows
// ([N rows][D] bytes, swizzled over the row): 2^e q rounded, the remainder
// rounded, and so on, with e the largest that keeps 2^e max_d |q_d| within the
// type (e clamped to +-120).
//   PARTS = 2: e4m3 (4 significant bits, largest 448, smallest 2^-9).  A bf16 value
//     has 8 significant bits, so the parts are exact where the last of them is 2^-9
//     or more: elements from 2^-9 of the row's largest on (which scales into
//     (224, 448]).  Below, an element is off by at most 2^-10, 2^-17 of the largest.
//   PARTS = 3: e5m2 (3 significant bits, largest 57344, smallest 2^-16): exact from
//     2^-23 of the largest on, below off by at most 2^-31 of it.  Taken where the
//     alternative was to widen the keys, which is exact.  (hi and lo as e4m3 and
//     e5m2 for the third part alone was exact to 2^-14 only.)
// 128 / N threads share a row; qsc[row] becomes the scale of the row's scores,
// scale_log2 2^-e (NaN for a row with an infinity or NaN).
template <int D, int N, int PARTS>
__device__ __forceinline__ void split_q(uint32_t q, uint32_t parts, float *qsc, float scale_log2,
                                        int ct) {
    constexpr int kTpr = kConvWarps * 32 / N;  // threads per row
    constexpr int kCh = D / 8 / kTpr;          // 8-element chunks per thread
    const int row = ct / kTpr, c0 = (ct % kTpr) * kCh;
    uint32_t w[kCh][4];
    uint32_t mb = 0;  // largest magnitude, as bits
#pragma unroll
    for (int i = 0; i < kCh; ++i) {
        const int c = c0 + i;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[i][0]), "=r"(w[i][1]), "=r"(w[i][2]), "=r"(w[i][3])
                     : "r"(q + (c >> 3) * (N * 128) + row * 128 + (((c & 7) ^ (row & 7)) << 4)));
#pragma unroll
        for (int u = 0; u < 4; ++u)
            mb = max(mb, max((w[i][u] << 16) & 0x7fff0000u, w[i][u] & 0x7fff0000u));
    }
#pragma unroll
    for (int d = 1; d < kTpr; d <<= 1) mb = max(mb, __shfl_xor_sync(kFull, mb, d));
    int e = 0;
    if (mb != 0u) {
        constexpr int kTopExp = PARTS == 3 ? 15 : 8;  // the largest value is 1.75 2^kTopExp
        e = ((mb & 0x7fffffu) <= 0x600000u ? kTopExp : kTopExp - 1) - ((int)(mb >> 23) - 127);
        e = e < -120 ? -120 : (e > 120 ? 120 : e);
    }
    const float sc = __uint_as_float((uint32_t)(127 + e) << 23);
#pragma unroll
    for (int i = 0; i < kCh; ++i) {
        uint32_t y[PARTS][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float xa = __uint_as_float(w[i][u] << 16) * sc;
            float xb = __uint_as_float(w[i][u] & 0xffff0000u) * sc;
#pragma unroll
            for (int z = 0; z < PARTS; ++z) {  // the next part of what is left
                uint32_t c2, f2;
                if (PARTS == 2)
                    asm("{\n .reg .b16 t;\n cvt.rn.satfinite.e4m3x2.f32 t, %2, %3;\n"
                        " cvt.u32.u16 %0, t;\n cvt.rn.f16x2.e4m3x2 %1, t;\n}"
                        : "=r"(c2), "=r"(f2)
                        : "f"(xb), "f"(xa));
                else
                    asm("{\n .reg .b16 t;\n cvt.rn.satfinite.e5m2x2.f32 t, %2, %3;\n"
                        " cvt.u32.u16 %0, t;\n cvt.rn.f16x2.e5m2x2 %1, t;\n}"
                        : "=r"(c2), "=r"(f2)
                        : "f"(xb), "f"(xa));
                float fa, fb;
                asm("{\n .reg .b16 a, b;\n mov.b32 {a, b}, %2;\n cvt.f32.f16 %0, a;\n"
                    " cvt.f32.f16 %1, b;\n}"
                    : "=f"(fa), "=f"(fb)
                    : "r"(f2));
                xa -= fa;
                xb -= fb;
                y[z][u >> 1] = (u & 1) ? y[z][u >> 1] | c2 << 16 : c2;
            }
        }
        // 8 bytes at byte 8 c of the row
        const int c = c0 + i, x = D == 128 ? row & 7 : (row >> 1) & 3;
        const uint32_t off = row * D + (((c >> 1) ^ x) << 4) + (c & 1) * 8;
#pragma unroll
        for (int z = 0; z < PARTS; ++z)
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(parts + z * (N * D) + off),
                         "r"(y[z][0]), "r"(y[z][1])
                         : "memory");
    }
    if (ct % kTpr == 0)
        qsc[row] = mb >= 0x7f800000u ? __uint_as_float(0x7fc00000u)
                                     : scale_log2 * __uint_as_float((uint32_t)(127 - e) << 23);
}

// N consecutive 32-bit columns of the calling thread's tensor-memory lane
// (taddr holds the warp's first lane); the loads and their wait form one
// statement, so no use of the registers can be scheduled before the data is
// there.
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[N]);
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, float (&v)[32]) {
    tmem_ld32(taddr, v);
}

// 16 columns of scores, of the rows' -reference and of their scale in one
// round trip.
__device__ __forceinline__ void tmem_ld_scores(uint32_t sa, uint32_t ma, uint32_t ca, float *v,
                                               float (&m)[16], float (&c)[16]) {
    uint32_t a[16], b[16], d[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%48];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,"
        "%28,%29,%30,%31}, [%49];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,"
        "%44,%45,%46,%47}, [%50];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
          "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]),
          "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]),
          "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]),
          "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]), "=r"(d[0]),
          "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]),
          "=r"(d[8]), "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]),
          "=r"(d[14]), "=r"(d[15])
        : "r"(sa), "r"(ma), "r"(ca)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        v[j] = __uint_as_float(a[j]);
        m[j] = __uint_as_float(b[j]);
        c[j] = __uint_as_float(d[j]);
    }
}
// N columns from each of two places, in one round trip.
template <int N>
__device__ __forceinline__ void tmem_ld_two(uint32_t xa, uint32_t ya, float *x, float (&y)[N]);
template <>
__device__ __forceinline__ void tmem_ld_two<16>(uint32_t xa, uint32_t ya, float *x, float (&y)[16]) {
    uint32_t a[16], b[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,"
        "%28,%29,%30,%31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
          "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]),
          "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]),
          "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]),
          "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15])
        : "r"(xa), "r"(ya)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        x[j] = __uint_as_float(a[j]);
        y[j] = __uint_as_float(b[j]);
    }
}

template <>
__device__ __forceinline__ void tmem_ld_two<32>(uint32_t xa, uint32_t ya, float *x, float (&y)[32]) {
    uint32_t a[32], b[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%64];\n"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,"
        "%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%65];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
          "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]),
          "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(a[16]), "=r"(a[17]), "=r"(a[18]),
          "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]), "=r"(a[24]),
          "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]),
          "=r"(a[31]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]),
          "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]),
          "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]), "=r"(b[16]), "=r"(b[17]),
          "=r"(b[18]), "=r"(b[19]), "=r"(b[20]), "=r"(b[21]), "=r"(b[22]), "=r"(b[23]),
          "=r"(b[24]), "=r"(b[25]), "=r"(b[26]), "=r"(b[27]), "=r"(b[28]), "=r"(b[29]),
          "=r"(b[30]), "=r"(b[31])
        : "r"(xa), "r"(ya)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        x[j] = __uint_as_float(a[j]);
        y[j] = __uint_as_float(b[j]);
    }
}

// The barrier of softmax group 0 or 1, and whether any of its threads says so.
template <int ID>
__device__ __forceinline__ bool bar_any(bool x) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n barrier.cta.red.or.pred p, %2, 128, q;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)x), "n"(ID)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ bool soft_any(int group, bool x) {
    return group == 0 ? bar_any<1>(x) : bar_any<2>(x);
}
__device__ __forceinline__ void soft_sync(int group) {
    if (group == 0)
        asm volatile("bar.sync 1, 128;" ::: "memory");
    else
        asm volatile("bar.sync 2, 128;" ::: "memory");
}

template <int NC>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const float (&x)[NC]) {
#pragma unroll
    for (int c = 0; c < NC; c += 16) {
        float o[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = x[c + j];
        tmem_st16(taddr + c, o);
    }
}

// The lane's columns from taddr: x, or what they hold plus x.  The stores are
// waited for by the next call, or by whoever reads them.
template <int NC>
__device__ __forceinline__ void tmem_accumulate(uint32_t taddr, float (&x)[NC], bool first) {
    if (!first) {
        float o[NC];
        tmem_wait_st();
        tmem_ld<NC>(taddr, o);
#pragma unroll
        for (int j = 0; j < NC; j += 2) add2(x[j], x[j + 1], x[j], x[j + 1], o[j], o[j + 1]);
    }
    tmem_st<NC>(taddr, x);
}

// NC values from shared memory into every lane's columns of tensor memory.
template <int NC>
__device__ __forceinline__ void row_values_to_tmem(uint32_t src, uint32_t dst) {
#pragma unroll
    for (int c = 0; c < NC; c += 16) {
        float x[16];
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            const float4 y = lds4(src + 4 * (c + j));
            x[j] = y.x;
            x[j + 1] = y.y;
            x[j + 2] = y.z;
            x[j + 3] = y.w;
        }
        tmem_st16(dst + c, x);
    }
    tmem_wait_st();
}

// A softmax group's slice of a P buffer: the 2 NC bytes of row `key` that hold
// its columns.  With two groups the swizzle of P puts them in the row's other
// half for keys with bit 2 set (128-byte rows at N = 64, 64-byte rows at N = 32).
template <int N>
__device__ __forceinline__ uint32_t slice_at(uint32_t pbuf, int group, int key) {
    return pbuf + key * (2 * N) + (N == 16 ? 0 : (group ^ ((key >> 2) & 1)) * N);
}

// The maximum (MAX; NaN ignored) or sum of x[r] over the warp's 32 lanes, for
// each of the NC query rows of its group, into red[r] (shared memory).  The
// values cross through the warp's rows of the group's slice of a P buffer, half
// of the rows at a time as fp32: 16 bytes out, 4 bytes in, 16 lanes a thread
// (31 shuffles or 32 redux instead took 870 and 2900 cycles at NC = 32).
template <bool MAX, int NC, int N>
__device__ __forceinline__ void lane_reduce(const float (&x)[NC], uint32_t pbuf, uint32_t red,
                                            int group, int key) {
    constexpr int H = NC / 2;  // rows a round: 4 H = 2 NC bytes a lane
    constexpr int C = H / 4;   // 16-byte chunks a lane
    const int lane = key & 31, row = lane & (H - 1), k0 = (key & 96) + lane / H * H;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h) __syncwarp();
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float *y = x + h * H + 4 * c;
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(
                             slice_at<N>(pbuf, group, key) + ((c ^ (key & (C - 1))) << 4)),
                         "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3])
                         : "memory");
        }
        __syncwarp();
        float y[H];  // all loads first: one latency
#pragma unroll
        for (int i = 0; i < H; ++i)
            y[i] = lds(slice_at<N>(pbuf, group, k0 + i) + (((row >> 2) ^ (i & (C - 1))) << 4) +
                       (row & 3) * 4);
#pragma unroll
        for (int d = H / 2; d > 0; d >>= 1)
#pragma unroll
            for (int i = 0; i < d; ++i) y[i] = MAX ? fmaxf(y[i], y[i + d]) : y[i] + y[i + d];
        float r = y[0];
#pragma unroll
        for (int d = H; d < 32; d <<= 1) {
            const float o = __shfl_xor_sync(kFull, r, d);
            r = MAX ? fmaxf(r, o) : r + o;
        }
        if (lane < H) sts(red + (h * H + row) * 4, r);
    }
}

// Registers a thread may use, so that a merge CTA (one warp in each of the SM's
// four register files of 512 x 32) fits beside the attention CTA: 192 with 7
// warps (two a file) leave 128, 128 with 11 (three a file) too.  bf16 with N = 64 takes
// 144 (44 bytes spilled; at 128 more), which leave 80, enough for all merge variants but
// the largest.  15 warps (four a file) leave no room at 128, and fewer would spill.
template <int D, bool KF8, bool VF8, int N>
constexpr int kRegCap = Layout<D, KF8, VF8, N>::kThreads <= 224 ? 192
                        : Layout<D, KF8, VF8, N>::kConv || N < 64 ? 128
                                                                  : 144;

// KF8 / VF8: prefix keys / values are e4m3 (tm_k / tm_v are 8-bit maps).
// N: query columns of the MMAs (16, 32 or 64; G * max_block rows rounded up).
template <int D, bool KF8, bool VF8, int N>
__global__ void __launch_bounds__(Layout<D, KF8, VF8, N>::kThreads, 1)
    __maxnreg__((kRegCap<D, KF8, VF8, N>))
    attn_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_k2,
                const __grid_constant__ CUtensorMap tm_v,
                const __grid_constant__ CUtensorMap tm_kb, const __grid_constant__ CUtensorMap tm_vb,
                const __grid_constant__ CUtensorMap tm_q, const AttnParams p) {
    using Lt = Layout<D, KF8, VF8, N>;
    constexpr bool kConv = Lt::kConv;
    constexpr int KS = Lt::kKSlots, VS = Lt::kVSlots, WS = VF8 ? Lt::kWSlots : 1;
    constexpr int kSBufs = Lt::kSBufs, kSoftWarps = Lt::kSoftWarps;
    constexpr int kProducerWarp = kSoftWarps;   // TMA loads
    constexpr int kMmaWarp = kSoftWarps + 1;    // MMAs of P V
    constexpr int kSWarp = kSoftWarps + 2;      // MMAs of S
    constexpr int kConvWarp0 = kSoftWarps + 3;  // (e4m3) query split, widening
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(sm);
    const uint32_t b_kfull = sbase + Lt::kBarOff, b_kempty = b_kfull + 8 * KS,
                   b_vfull = b_kempty + 8 * KS, b_vempty = b_vfull + 8 * VS,
                   b_wready = b_vempty + 8 * VS, b_wfree = b_wready + 8 * Lt::kWSlots,
                   b_qfull = b_wfree + 8 * Lt::kWSlots, b_qempty = b_qfull + 16,
                   b_qsplit = b_qempty + 16, b_sready = b_qsplit + 16, b_sfree = b_sready + 8 * Lt::kSBufs,
                   b_pready = b_sfree + 8 * Lt::kSBufs,
                   b_pvdone = b_pready + 16, b_drain = b_pvdone + 16, b_rready = b_drain + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sm + Lt::kMiscOff);
    const uint32_t abort_flag = sbase + Lt::kMiscOff + 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // barrier i's wait for a phase of that parity: exact, because every waiter
    // is at most one phase behind
    auto await = [&](uint32_t bar, int i, uint32_t parity) {
        return wait(bar + 8 * i, parity & 1u, abort_flag, p.status);
    };

    // set-up that touches no global memory: it may overlap the previous
    // kernel in the stream (programmatic dependent launch)
    auto init_bars = [&]() {  // one thread
        for (int s = 0; s < KS; ++s) {
            mbar_init(b_kfull + 8 * s, 1);
            mbar_init(b_kempty + 8 * s, 1);
        }
        for (int s = 0; s < VS; ++s) {
            mbar_init(b_vfull + 8 * s, 1);
            mbar_init(b_vempty + 8 * s, VF8 ? kConvWarps : 1);
        }
        for (int s = 0; s < Lt::kWSlots; ++s) {
            mbar_init(b_wready + 8 * s, kConvWarps);
            mbar_init(b_wfree + 8 * s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(b_qfull + 8 * i, 1);
            // e4m3 keys: the segment's last S, and every softmax warp once it
            // has read the row scales
            mbar_init(b_qempty + 8 * i, KF8 ? 1 + kSoftWarps : 1);
            mbar_init(b_qsplit + 8 * i, kConvWarps);
            mbar_init(b_pready + 8 * i, kSoftWarps);
            mbar_init(b_pvdone + 8 * i, 1);
            mbar_init(b_drain + 8 * i, 1);
        }
        mbar_init(b_rready, 1);
        for (int i = 0; i < kSBufs; ++i) {
            mbar_init(b_sready + 8 * i, 1);
            mbar_init(b_sfree + 8 * i, kSoftWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    };
    int *len_sm = reinterpret_cast<int *>(sm + Lt::kLenOff);  // [0, 32) P, [32, 64) T
    const int lane0 = threadIdx.x & 31;
    const bool spec = p.B <= 32;
    if (threadIdx.x == 0) {
        init_bars();
        sts(abort_flag, 0.f);
    }
    if (warp == 0) {
        asm volatile(
            "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                smem_u32(const_cast<uint32_t *>(tmem_slot))),
            "n"(Lt::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // The lengths as they read before the dependency wait (a kernel before
    // this one may still change them), one copy for the whole CTA: every
    // warp plans from the same values, and the check after the wait is the
    // same in every warp.
    if (spec && warp == kProducerWarp) {
        len_sm[lane0] = lane0 < p.B ? len_cg(p.prefix_len, lane0, p.capacity) : 0;
        len_sm[32 + lane0] = lane0 < p.B ? len_cg(p.block_len, lane0, p.max_block) : 0;
    }
    if (D == 64 && threadIdx.x < 128) {  // 2 KB of bf16 ones (and 2 KB of f16 ones)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                         sbase + Lt::kOnesOff + threadIdx.x * 16),
                     "r"(0x3F803F80u)
                     : "memory");
        if (VF8)
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                             sbase + Lt::kOnesOff + 2048 + threadIdx.x * 16),
                         "r"(0x3C003C00u)
                         : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kProducerWarp && elect_one()) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k2)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_v)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_q)) : "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    if (D == 128 && warp < 4) {  // (their readers wait for P, which these warps hand on)
        const uint32_t at = tmem + ((uint32_t)(warp * 32) << 16) + Lt::kOnesCol;
        tmem_fill8(at, 0x3F803F80u);
        if (VF8) tmem_fill8(at + 8, 0x3C003C00u);
    }

    // The plan from the lengths as they read before the dependency wait;
    // after the wait they are read again and the plan is kept only if every
    // length is unchanged.
    long long lo = 0, hi = 0;
    int ntiles = 0;
    Walk w0 = {0, 0, 0, 1, 0, 0};
    int sP = 0, sT = 0;
    if (spec) {
        sP = len_sm[lane0];
        sT = len_sm[32 + lane0];
        ntiles = plan(p, sP, sT, lo, hi, w0) ? (int)(hi - lo) : 0;
        // While the kernels before this one finish, pull the range's first
        // prefix tiles into L2 (the cache is L2-coherent: if a kernel before
        // this one writes them, the loads after the wait still see its data).
        if (warp == kProducerWarp && elect_one()) {
            Walk wp = w0;
            // the first segment's query rows (the kernel before this one may
            // be the one writing them: a prefetch only warms L2)
            if (ntiles > 0)
#pragma unroll
                for (int dp = 0; dp < Lt::kPanels; ++dp)
                    tma_prefetch_4d(&tm_q, dp * 64, wp.h * p.G, 0, wp.b);
            const int prefetch = ntiles > kLongRange ? 0 : kPrefetchTiles;
            for (int j = 0; j < ntiles && j < prefetch && wp.t < wp.nt - 1; ++j) {
                const int tok = wp.t * kTileKeys;
                if (KF8) {
                    tma_prefetch_5d(&tm_k, 0, wp.h, tok, wp.b, p.key_slab);
                } else if (j == 0) {  // (bf16: the step's two tiles at once)
                    tma_prefetch_5d(&tm_k2, 0, tok, 0, wp.h, p.key_slab * p.B + wp.b);
                }
                if (VF8)
                    tma_prefetch_5d(&tm_v, 0, wp.h, tok, wp.b, p.value_slab);
                else
                    tma_prefetch_5d(&tm_v, 0, tok, 0, wp.h, p.value_slab * p.B + wp.b);
                ++wp.t;  // stays inside the pair: its last (block) tile ends the loop
            }
        }
    }

    // Loads, issued by two warps, each walking the range on its own: the S warp
    // those of K (a slot is refilled as soon as the S that read it is done,
    // whatever V waits for), the producer warp the query rows and V.  The
    // first kFirstSteps steps' loads are all the producer's, in the order in
    // which they are needed (an SM takes about 64 bytes a cycle from L2: issued
    // by two warps at once, the first K came 0.6 us later), and may go out
    // before the lengths are checked (below).
    constexpr int kFirstSteps = 2;
    static_assert(KS >= kFirstSteps && VS >= 2 * kFirstSteps, "first loads never wait");
    Walk wl = w0;
    Seg sg = {0, 0, 0, 0, false};
    int qseg = -1, si = 0;         // segment, step of the segment
    int done = 0, loads = 0, kloads = 0;  // tiles of past segments; V and K slots filled
    Ring<KS> rk;
    Ring<VS> rv;
    bool ok = true;
    uint64_t policy = 0;
    if (warp == kProducerWarp || warp == kSWarp)
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    auto next_step = [&]() {
        if (++si == sg.steps) {
            si = 0;
            done += sg.tiles;
            walk_segment(p, wl, sg);
        }
    };
    auto step_tile0 = [&]() {
        return kConv && 2 * si >= sg.pairs ? wl.nt - 1 : wl.t + 2 * si;
    };
    // K of the current step, into a free slot
    auto load_k = [&]() {
        const int n = step_tiles(sg, si), t0 = step_tile0();
        if (elect_one()) {
            const uint32_t full = b_kfull + 8 * rk.slot;
            const uint32_t dst = sbase + rk.slot * Lt::kKBytes;
            const bool blk_last = t0 + n == wl.nt;  // the step's last tile is the block tile
            mbar_arrive_expect_tx(full, KF8 ? (blk_last ? Lt::kTileBytes : n * (Lt::kKBytes / 2))
                                            : n * Lt::kTileBytes);
            if (t0 + 1 < wl.nt - 1 && n == 2) {  // two prefix tiles
                if (KF8)
                    tma_5d(dst, &tm_k2, full, 0, wl.h, t0 * kTileKeys, wl.b, p.key_slab, policy);
                else
                    tma_5d(dst, &tm_k2, full, 0, t0 * kTileKeys, 0, wl.h, p.key_slab * p.B + wl.b,
                           policy);
            } else {
                for (int h = 0; h < n; ++h) {
                    const int t = t0 + h;
                    if (KF8 && t < wl.nt - 1) {
                        tma_5d(dst + h * (Lt::kKBytes / 2), &tm_k, full, 0, wl.h, t * kTileKeys,
                               wl.b, p.key_slab, policy);
                        continue;
                    }
#pragma unroll
                    for (int dp = 0; dp < Lt::kPanels; ++dp) {
                        // (e4m3 keys: the bf16 block tile, of 64-key panels)
                        const uint32_t at = dst + dp * (KF8 ? 8192 : 16384) + h * 8192;
                        if (t < wl.nt - 1)
                            tma_5d(at, &tm_k, full, 0, t * kTileKeys, dp, wl.h,
                                   p.key_slab * p.B + wl.b, policy);
                        else
                            tma_4d(at, &tm_kb, full, dp * 64, wl.h, 0, wl.b);
                    }
                }
            }
        }
        __syncwarp();
        ++kloads;
        rk.next();
    };
    // the current step's V and, with its segment's first, the query rows
    // (first = true: and its K, between the two)
    auto load_qv = [&](bool first) {
        if (si == 0) {
            sg = segment<kConv>(wl, ntiles - done);
            ++qseg;
            const int qb = qseg & 1;
            if (qseg >= 2) ok = ok && await(b_qempty, qb, (qseg - 2) >> 1);
            if (ok && elect_one()) {
                const uint32_t full = b_qfull + 8 * qb;
                const uint32_t dst = sbase + Lt::kQOff + qb * Lt::kQBytes;
                mbar_arrive_expect_tx(full, Lt::kPanels * p.rows_max * 128);
#pragma unroll
                for (int dp = 0; dp < Lt::kPanels; ++dp)
                    tma_4d(dst + dp * (N * 128), &tm_q, full, dp * 64, wl.h * p.G, 0, wl.b);
            }
        }
        if (first) load_k();
        const int n = step_tiles(sg, si), t0 = step_tile0();
        for (int h = 0; h < n; ++h) {
            const int t = t0 + h;
            // (e4m3 values) the conversion warps load a block tile's V
            if (VF8 && t == wl.nt - 1) break;
            if (loads >= VS) ok = ok && await(b_vempty, rv.slot, rv.parity ^ 1);
            if (ok && elect_one()) {
                const uint32_t full = b_vfull + 8 * rv.slot;
                const uint32_t dst = sbase + Lt::kVOff + rv.slot * Lt::kVBytes;
                mbar_arrive_expect_tx(full, Lt::kVBytes);
                if (VF8) {
                    tma_5d(dst, &tm_v, full, 0, wl.h, t * kTileKeys, wl.b, p.value_slab, policy);
                } else if (t < wl.nt - 1) {
                    tma_5d(dst, &tm_v, full, 0, t * kTileKeys, 0, wl.h, p.value_slab * p.B + wl.b,
                           policy);
                } else {
#pragma unroll
                    for (int dp = 0; dp < Lt::kPanels; ++dp)
                        tma_4d(dst + dp * 8192, &tm_vb, full, dp * 64, wl.h, 0, wl.b);
                }
            }
            __syncwarp();
            if (!ok) break;
            ++loads;
            rv.next();
        }
        next_step();
    };

    // every input (and the workspace) may be written by the previous kernel
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the first loads of the speculative plan go out while the lengths are
    // checked (no step here waits: fresh slots and query buffers only)
    auto first_loads = [&]() {
        for (int u = 0; u < kFirstSteps && done < ntiles; ++u) load_qv(true);
    };
    if (spec && warp == kProducerWarp) first_loads();
    {
        const int P1 = lane0 < p.B ? len_cg(p.prefix_len, lane0, p.capacity) : 0;
        const int T1 = lane0 < p.B ? len_cg(p.block_len, lane0, p.max_block) : 0;
        if (!(spec && __all_sync(kFull, P1 == sP && T1 == sT))) {  // the same in every warp
            if (spec) {  // loads issued under the stale plan land, then the barriers restart
                if (warp == kProducerWarp) {
                    for (int s = 0; s < kloads; ++s) await(b_kfull, s, 0);
                    for (int s = 0; s < loads; ++s) await(b_vfull, s, 0);
                    for (int q = 0; q <= qseg; ++q) await(b_qfull, q, 0);
                }
                __syncthreads();
                if (threadIdx.x == 0) init_bars();
                __syncthreads();
            }
            lo = hi = 0;
            w0 = {0, 0, 0, 1, 0, 0};
            ntiles = plan(p, P1, T1, lo, hi, w0) ? (int)(hi - lo) : 0;
            wl = w0;
            qseg = -1;
            si = done = loads = kloads = 0;
            rk = Ring<KS>();
            rv = Ring<VS>();
            ok = true;
        }
    }

    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (int b = 0; b < p.B; ++b)
            if (p.prefix_len[b] != clamp_prefix(p, b) || p.block_len[b] != clamp_block(p, b))
                atomicOr(p.status, kStatusClamped);
    // an empty range (only when N < C) runs no loop below

    int drain_copy = -1;  // the last copy a conversion warp started, for the abort path's drain
    if (warp == kProducerWarp) {
        // ================================ producer ===============================
        // Warp-uniform loop; one elected lane issues.  A V slot is reused once
        // the P V (or the widening) that read it has completed, a query buffer
        // once the last S of the segment before last has (and the softmax
        // warps have read its scales).
        if (kloads == 0) first_loads();  // (not spec, or the lengths had changed)
        while (done < ntiles && ok) load_qv(false);
    } else if (warp == kSWarp) {
        // =============================== S^T = K Q^T =============================
        const uint32_t id_s = idesc(128, N, 0, 0);
        constexpr uint32_t kE5 = Lt::kParts == 3 ? 1u : 0u;  // the query parts are e5m2
        const uint32_t id_s8 = idesc_e4m3(128, N) | kE5 << 10;
        const uint32_t id_r = idesc(64, kRefKeys, 0, 0), id_r8 = idesc_e4m3(64, kRefKeys) | kE5 << 7;
        // descriptors are affine in the address: build each base once and add
        // (byte offset >> 4) for slots, panels and k-steps
        const uint64_t dk = sdesc(sbase, 16, 1024, kSw128);
        const uint64_t dq = sdesc(sbase + Lt::kQOff, 16, 1024, kSw128);
        const uint64_t dk8 = sdesc(sbase, 16, 8 * D, D == 128 ? kSw128 : kSw64);
        const uint64_t dq8 = sdesc(sbase + Lt::kQ8Off, 16, 8 * D, D == 128 ? kSw128 : kSw64);
        // Of a segment's first step, the scores of its first keys are also formed the
        // other way round (rows in lanes: M = 64), where each row's maximum, the
        // first reference, is one thread's.
        // The walk over the steps that the producer loaded, then K of the slots
        // left.  e4m3 keys: while the query rows are split; else the first S first.
        auto start_loads = [&]() {
            for (int u = 0; done < ntiles && u < KS; ++u) {
                if (si == 0) sg = segment<kConv>(wl, ntiles - done);
                if (u < kFirstSteps) {
                    ++kloads;
                    rk.next();
                } else {
                    load_k();
                }
                next_step();
            }
        };
        if (KF8) start_loads();
        Walk w = w0;
        Ring<KS> ru;          // slot being read
        Ring<kSBufs> rs, rf;  // rf: the last segment's first step, kf
        for (int past = 0, seg = 0, k = 0, kf = 0; past < ntiles && ok; ++seg) {
            const Seg sc = segment<kConv>(w, ntiles - past);
            const int qb = seg & 1;
            ok = await(b_qfull, qb, seg >> 1);
            if (KF8) ok = ok && await(b_qsplit, qb, seg >> 1);
            for (int i = 0; i < sc.steps && ok; ++i, ++k) {
                ok = await(b_kfull, ru.slot, ru.parity);
                // the softmax has read the scores of step k - kSBufs
                if (k >= kSBufs) ok = ok && await(b_sfree, rs.slot, rs.parity ^ 1);
                // and the last segment's reference scores: implied unless its
                // first step is a later one (whose buffer then has no later
                // phase, so that the parity is exact)
                if (i == 0 && seg > 0 && k - kf < kSBufs)
                    ok = ok && await(b_sfree, rf.slot, rf.parity);
                if (!ok) break;
                fence_after();
                if (elect_one()) {
                    const uint32_t dS = tmem + (uint32_t)(rs.slot * N), dR = tmem + Lt::kRefCol;
                    const uint32_t slot = (uint32_t)(ru.slot * Lt::kKBytes) >> 4;
                    // the parts' K^T one after the other, 32 elements (32 bytes) per MMA
                    // (the queries are B of S^T, A of the reference scores); bf16: panel kk / 4, then 16 elements within the 128-byte row
                    const bool f8 = KF8 && 2 * i < sc.pairs;
                    auto key8 = [&](int kk) { return dk8 + (uint64_t)(slot + kk % (D / 32) * 2); };
                    auto qry8 = [&](int kk) {
                        return dq8 + (uint64_t)((kk / (D / 32) * Lt::kQ8Bytes + kk % (D / 32) * 32) >> 4);
                    };
                    auto key16 = [&](int kk) {
                        return dk + (uint64_t)(slot + (((kk >> 2) * (KF8 ? 8192 : 16384) +
                                                        (kk & 3) * 32) >> 4));
                    };
                    auto qry16 = [&](int kk) {
                        return dq + (uint64_t)((qb * Lt::kQBytes + (kk >> 2) * (N * 128) +
                                                (kk & 3) * 32) >> 4);
                    };
                    if (i == 0) {  // first: the softmax takes the references meanwhile
                        if (f8) {
#pragma unroll
                            for (int kk = 0; kk < Lt::kParts * (D / 32); ++kk)
                                mma_f8(dR, qry8(kk), key8(kk), id_r8, kk > 0);
                        } else {
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk)
                                mma(dR, qry16(kk), key16(kk), id_r, kk > 0);
                        }
                        mma_commit(b_rready);
                    }
                    if (f8) {
#pragma unroll
                        for (int kk = 0; kk < Lt::kParts * (D / 32); ++kk)
                            mma_f8(dS, key8(kk), qry8(kk), id_s8, kk > 0);
                    } else {
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            mma(dS, key16(kk), qry16(kk), id_s, kk > 0);
                    }
                    mma_commit(b_sready + 8 * rs.slot);
                    mma_commit(b_kempty + 8 * ru.slot);
                    if (i == sc.steps - 1) mma_commit(b_qempty + 8 * qb);
                }
                __syncwarp();
                // fill the slots not used yet, refill this one once these S are done
                if (!KF8 && k == 0) start_loads();
                if (done < ntiles) {  // refill the slot once these S are done
                    ok = await(b_kempty, ru.slot, ru.parity);
                    if (ok) {
                        if (si == 0) sg = segment<kConv>(wl, ntiles - done);
                        load_k();
                        next_step();
                    }
                }
                if (i == 0) {
                    rf = rs;
                    kf = k;
                }
                ru.next();
                rs.next();
            }
            past += sc.tiles;
            walk_segment(p, w, sc);
        }
    } else if (warp == kMmaWarp) {
        // ========================= O^T += V^T P^T, l += 1 P^T ====================
        // A is MN-major: V as it lies (dims contiguous).  D = 64: M = 128, the
        // second 64 rows of A are ones, so lanes 64.. accumulate the row sums
        // of P as rounded; D = 128: they take MMAs of their own, with the ones
        // in tensor memory (shared memory is the scarcer port).
        const uint64_t dp = sdesc(sbase + Lt::kPOff, 16, 16 * N, N == 64 ? kSw128 : N == 32 ? kSw64 : kSw32);
        const uint32_t vbase = sbase + (VF8 ? Lt::kWOff : Lt::kVOff);
        constexpr int kVStride = VF8 ? Lt::kTileBytes : Lt::kVBytes;
        const uint32_t b_v = VF8 ? b_wready : b_vfull, b_vdone = VF8 ? b_wfree : b_vempty;
        const uint32_t dO = tmem + Lt::kOCol;
        Walk w = w0;
        Ring<VF8 ? WS : VS> rv;
        bool ok = true;
        for (int done = 0, k = 0; done < ntiles && ok;) {
            const Seg sg = segment<kConv>(w, ntiles - done);
            // 16-key groups of the last tile that P V reads, and of a last step of it alone
            const int last_groups = (tile_keys(w, w.t + sg.tiles - 1) + 15) >> 4;
            for (int i = 0; i < sg.steps; ++i, ++k) {
                const int n = step_tiles(sg, i);
                const bool last = i == sg.steps - 1;
                // (a partly filled prefix tile before a block step of its own is all zeros past its keys)
                const int groups = !last ? 4 * n : n == 2 ? 4 + last_groups : max(last_groups, 1);
                const bool f16 = VF8 && 2 * i < sg.pairs;  // widened values: f16
                const uint32_t id_pv = f16 ? idesc_f16(128, N, 1, 1) : idesc(128, N, 1, 1);
                const uint32_t id_l = f16 ? idesc_f16(128, N, 0, 1) : idesc(128, N, 0, 1);
                const uint32_t ones = sbase + Lt::kOnesOff + (f16 ? 2048 : 0);
                const Ring<VF8 ? WS : VS> r0 = rv;
                ok = await(b_v, rv.slot, rv.parity);
                rv.next();
                const int slot1 = rv.slot;
                if (n == 2) {
                    ok = ok && await(b_v, rv.slot, rv.parity);
                    rv.next();
                }
                ok = ok && await(b_pready, k & 1, k >> 1);
                if (!ok) break;
                fence_after();
                if (elect_one()) {
                    const uint64_t b0 = dp + (uint64_t)(((k & 1) * Lt::kPBytes) >> 4);
                    const bool acc0 = i > 0;
                    const uint32_t va0 = vbase + r0.slot * kVStride, va1 = vbase + slot1 * kVStride;
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        if (g >= groups) break;
                        const uint32_t va = (g < 4 ? va0 : va1) + (g & 3) * 2048;
                        mma(dO, sdesc(va, D == 128 ? 8192 : ones - va, 1024, kSw128),
                            b0 + (uint64_t)((g * 32 * N) >> 4), id_pv, acc0 || g > 0);
                    }
                    if (D == 128) {
                        const uint32_t a = tmem + Lt::kOnesCol + (f16 ? 8 : 0);
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            if (g >= groups) break;
                            mma_ta(tmem + Lt::kLCol, a, b0 + (uint64_t)((g * 32 * N) >> 4), id_l,
                                   acc0 || g > 0);
                        }
                    }
                    mma_commit(b_pvdone + 8 * (k & 1));
                    mma_commit(b_vdone + 8 * r0.slot);
                    if (n == 2) mma_commit(b_vdone + 8 * slot1);
                }
                __syncwarp();
            }
            done += sg.tiles;
            walk_segment(p, w, sg);
        }
    } else if (kConv && warp >= kConvWarp0) {
        // ==================== query split, e4m3 -> f16 values ====================
        const int ct = threadIdx.x - kConvWarp0 * 32;
        float *qsc = reinterpret_cast<float *>(sm + Lt::kQscOff);
        Walk w = w0;
        int seg = -1, vt = 0;
        for (int j = 0; j < ntiles; ++j) {
            if (KF8 && (j == 0 || w.t == 0)) {
                // The parts are overwritten once the last segment's S are done
                // (a step or two before the softmax ends it), the scales of
                // buffer b once the segment before last's are read: qempty.
                ++seg;
                const int qb = seg & 1;
                if (seg >= 1 && !await(b_qempty, qb ^ 1, (seg - 1) >> 1)) break;
                if (!await(b_qfull, qb, seg >> 1)) break;
                split_q<D, N, Lt::kParts>(sbase + Lt::kQOff + qb * Lt::kQBytes,
                                          sbase + Lt::kQ8Off, qsc + qb * N, p.scale_log2, ct);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(b_qsplit + 8 * qb);
            }
            if (VF8) {
                const uint32_t wr = b_wready + 8 * (j % WS);
                const uint32_t dst = sbase + Lt::kWOff + (j % WS) * Lt::kTileBytes;
                if (j >= WS && !await(b_wfree, j % WS, j / WS - 1)) break;
                if (w.t == w.nt - 1) {
                    // the block's V is bf16: one lane loads it into the slot
                    // with a copy that completes on wready itself
                    if (warp == kConvWarp0) {
                        if (elect_one()) {
                            mbar_arrive_expect_tx(wr, Lt::kTileBytes);
#pragma unroll
                            for (int dp = 0; dp < Lt::kPanels; ++dp)
                                tma_4d(dst + dp * 8192, &tm_vb, wr, dp * 64, w.h, 0, w.b);
                        }
                        drain_copy = j;
                    } else if (lane == 0) {
                        mbar_arrive(wr);
                    }
                    __syncwarp();
                } else {
                    const int vs = vt % VS;
                    if (!await(b_vfull, vs, vt / VS)) break;
                    widen_f16<D>(sbase + Lt::kVOff + vs * Lt::kVBytes, dst, tile_keys(w, w.t), ct);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(wr);
                        mbar_arrive(b_vempty + 8 * vs);
                    }
                    ++vt;
                }
            }
            walk_next(p, w);
        }
    } else if (warp < kSoftWarps) {
        // ================================ softmax ================================
        // Thread j of a group holds key j of the step: its group's kCols scores
        // of that lane of S^T.  With N = 64 two groups take 32 columns each,
        // independent of one another up to P (two warps per scheduler, which
        // hide each other's latencies; one group of 64 columns needed 255
        // registers and was slower on every 64-column case).
        constexpr int NC = Lt::kCols;
        constexpr float kShift = VF8 ? kShiftF16 : 0.f, kTop = VF8 ? kTopF16 : kTopBf16;
        const int group = Lt::kGroups == 1 ? 0 : warp >> 2, key = threadIdx.x & 127;
        const int half = key >> 6, kidx = key & 63;  // tile of the step, key of the tile
        const int col0 = group * NC;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        // per query row, this group's: -reference, rescale factor, per-warp
        // partials [4][N], rounded row sum (shared memory); -reference and
        // score scale in every lane of tensor memory
        const uint32_t rows = sbase + Lt::kNmOff + col0 * 4;
        const uint32_t nm_sm = rows, al_sm = rows + (Lt::kAlphaOff - Lt::kNmOff),
                       red_sm = rows + (Lt::kRedOff - Lt::kNmOff),
                       lr_sm = rows + (Lt::kLrOff - Lt::kNmOff);
        const uint32_t pkey = sbase + Lt::kPOff + key * (2 * N);
        const int pswz = N == 64 ? key & 7 : N == 32 ? (key >> 1) & 3 : (key >> 2) & 1;
        const uint32_t nm_t = tmem + lane_base + (uint32_t)(Lt::kNmCol + col0),
                       sc_t = tmem + lane_base + (uint32_t)(Lt::kScCol + col0),
                       sum_t = tmem + lane_base + (uint32_t)(Lt::kSumCol + col0);
        Walk w = w0;
        Ring<VF8 ? WS : VS> rv;
        Ring<kSBufs> rs;
        for (int done = 0, seg = 0, k = 0; done < ntiles; ++seg) {
        const Seg sg = segment<kConv>(w, ntiles - done);
        const int rows_active = p.G * w.T - col0;
        const uint32_t sc_row = rows + (Lt::kQscOff - Lt::kNmOff) + (seg & 1) * N * 4;
        if (KF8) {
            await(b_qsplit, seg & 1, seg >> 1);
            row_values_to_tmem<NC>(sc_row, sc_t);
            // the scales are read: their buffer may take the segment after next's
            __syncwarp();
            if (lane == 0) mbar_arrive(b_qempty + 8 * (seg & 1));
        }
        for (int i = 0; i < sg.steps; ++i, ++k, rs.next()) {
            const bool first = i == 0;
            const bool last = i == sg.steps - 1;
            const bool full = i < sg.nfull;                  // every key visible to every row
            const bool f8s = KF8 && 2 * i < sg.pairs;        // the scores carry a scale per row
            const int n = step_tiles(sg, i);
            const int t0 = kConv && 2 * i >= sg.pairs ? w.nt - 1 : w.t + 2 * i;
            // this key is visible to the rows from r0 on: all for a valid
            // prefix key, rows i >= kidx (r / G >= kidx) for a block key
            int r0 = 0;
            if (!full) {
                const int t = t0 + half;
                const bool valid = half < n && kidx < tile_keys(w, t);
                r0 = !valid ? N : t == w.nt - 1 ? kidx * p.G - col0 : 0;
            }
            // ---- scores of the step ----
            const uint32_t s_addr = tmem + lane_base + (uint32_t)(rs.slot * N + col0);
            float v[NC];
            // v = score - reference (base 2), -inf where not visible
            auto to_exponents = [&]() {
                const float s0 = p.scale_log2;
                if constexpr (KF8) {  // (three loads of 32 would spill)
#pragma unroll
                    for (int c = 0; c < NC; c += 16) {
                        float m[16], s[16];
                        tmem_ld_scores(s_addr + c, nm_t + c, sc_t + c, v + c, m, s);
#pragma unroll
                        for (int j = 0; j < 16; j += 2)
                            fma2(v[c + j], v[c + j + 1], v[c + j], v[c + j + 1], f8s ? s[j] : s0,
                                 f8s ? s[j + 1] : s0, m[j], m[j + 1]);
                    }
                } else {
                    float m[NC];
                    tmem_ld_two<NC>(s_addr, nm_t, v, m);
#pragma unroll
                    for (int j = 0; j < NC; j += 2)
                        fma2(v[j], v[j + 1], v[j], v[j + 1], s0, s0, m[j], m[j + 1]);
                }
                if (!full)
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[c] = c >= r0 ? v[c] : -INFINITY;
            };
            if (first) {  // the first reference, while S is formed
                await(b_rready, 0, seg);
                fence_after();
                if ((warp & 3) * 16 >= col0 && (warp & 3) * 16 < col0 + NC) {
                    float x[kRefKeys];
                    tmem_ld<kRefKeys>(tmem + lane_base + (uint32_t)Lt::kRefCol, x);
                    const int r = (warp & 3) * 16 + lane - col0;  // lanes < 16
                    const int nv = min(kRefKeys, tile_keys(w, t0));
                    const int lim = t0 == w.nt - 1 ? min(nv, (r + col0) / p.G + 1) : nv;
                    float m = -INFINITY;
#pragma unroll
                    for (int c = 0; c < kRefKeys; ++c) m = fmaxf(m, c < lim ? x[c] : -INFINITY);
                    if (lane < 16) {
                        m *= f8s ? lds(sc_row + 4 * r) : p.scale_log2;
                        // a row with no finite score yet keeps a reference far below
                        // any; rows past the block weigh nothing and never move it
                        sts(nm_sm + 4 * r, r >= rows_active  ? -INFINITY
                                           : m == -INFINITY ? kNoRef
                                                            : kShift - m);
                    }
                }
                soft_sync(group);
                row_values_to_tmem<NC>(nm_sm, nm_t);
            }
            await(b_sready, rs.slot, rs.parity);
            fence_after();
            to_exponents();
            float m4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) m4[j] = fmaxf(v[j], v[j + 4]);
#pragma unroll
            for (int c = 8; c < NC; c += 8)
#pragma unroll
                for (int j = 0; j < 4; ++j) m4[j] = max3(m4[j], v[c + j], v[c + 4 + j]);
            // a score far beyond its row's reference: the references move
            const bool move =
                soft_any(group, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) > kTop);
            const uint32_t pbuf = (uint32_t)((k & 1) * Lt::kPBytes);
            if (move) {  // the same in all of the group's warps
                // the rows' maxima over the step, through the P buffer (free once
                // P V of step k - 2 is done)
                if (k >= kPBufs) await(b_pvdone, k & 1, (k >> 1) - 1);
#pragma unroll
                for (int c = 0; c < NC; c += 16) {
                    float m[16], s[16];
                    tmem_ld_scores(s_addr + c, nm_t + c, (KF8 ? sc_t : nm_t) + c, v + c, m, s);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        v[c + j] = c + j >= r0 ? v[c + j] * (f8s ? s[j] : p.scale_log2) : -INFINITY;
                }
                lane_reduce<true, NC, N>(v, sbase + Lt::kPOff + pbuf, red_sm + (warp & 3) * N * 4, group, key);
                soft_sync(group);
                if (key < NC) {
                    const int r = key;
                    const uint32_t red = red_sm + 4 * r;
                    const float m = fmaxf(fmaxf(lds(red), lds(red + 4 * N)),
                                          fmaxf(lds(red + 8 * N), lds(red + 12 * N)));
                    const float old = lds(nm_sm + 4 * r);
                    float nm = old, alpha = 1.f;
                    if (m + old > kShift && m != -INFINITY) {  // (old = -inf past the block)
                        nm = kShift - m;
                        alpha = ex2(nm - old);
                    }
                    sts(nm_sm + 4 * r, nm);
                    sts(al_sm + 4 * r, alpha);
                }
                soft_sync(group);
                row_values_to_tmem<NC>(nm_sm, nm_t);
                if (!first) {
                    // O is stable once P V of step k - 1 is done
                    await(b_pvdone, (k - 1) & 1, (k - 1) >> 1);
                    fence_after();
                    // the lane's sums, O and (D = 128) the rounded row sums
                    tmem_wait_st();
#pragma unroll 1
                    for (int c = 0; c < (D == 128 ? 3 : 2) * NC; c += 16) {
                        const int at = c < NC       ? Lt::kSumCol
                                       : c < 2 * NC ? Lt::kOCol - NC
                                                    : Lt::kLCol - 2 * NC;
                        const uint32_t ta = tmem + lane_base + (uint32_t)(at + col0 + c);
                        float o[16];
                        tmem_ld<16>(ta, o);
#pragma unroll
                        for (int r = 0; r < 16; r += 4) {
                            const float4 a = lds4(al_sm + 4 * ((c & (NC - 1)) + r));
                            mul2(o[r], o[r + 1], o[r], o[r + 1], a.x, a.y);
                            mul2(o[r + 2], o[r + 3], o[r + 2], o[r + 3], a.z, a.w);
                        }
                        tmem_st16(ta, o);
                    }
                    tmem_wait_st();
                }
                to_exponents();
            }
            // the scores are in registers: their buffer may take step k + kSBufs
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_sfree + 8 * rs.slot);
            // ---- P = 2^(s - m), as 16-bit floats into the P buffer ----
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = ex2(v[c]);
            uint32_t pk[NC / 2];
            if (VF8 && 2 * i < sg.pairs) {
#pragma unroll
                for (int c = 0; c < NC / 2; ++c) pk[c] = pack_f16(v[2 * c], v[2 * c + 1]);
            } else {
#pragma unroll
                for (int c = 0; c < NC / 2; ++c) pk[c] = pack_bf16(v[2 * c], v[2 * c + 1]);
            }
            // the P buffer is free once P V of step k - 2, its last reader, is done
            if (k >= kPBufs) await(b_pvdone, k & 1, (k >> 1) - 1);
            const uint32_t prow = pkey + pbuf;
#pragma unroll
            for (int c = 0; c < NC / 8; ++c)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                 prow + (((col0 / 8 + c) ^ pswz) << 4)),
                             "r"(pk[4 * c]), "r"(pk[4 * c + 1]), "r"(pk[4 * c + 2]),
                             "r"(pk[4 * c + 3])
                             : "memory");
            // keys past the end of a tile may hold anything: zero the V rows
            // that P V reads (widened tiles hold zeros there)
            for (int h = 0; h < n; ++h, rv.next()) {
                if (full || (VF8 && 2 * i < sg.pairs)) continue;
                const int nv = tile_keys(w, t0 + h);
                // a tile with another after it is read whole, the last up to its 16-key group
                const int end = !last || h + 1 < n ? kTileKeys : n == 1 && nv == 0 ? 16 : (nv + 15) & ~15;
                if (nv >= end) continue;
                await(VF8 ? b_wready : b_vfull, rv.slot, rv.parity);
                const uint32_t vt = sbase + (VF8 ? Lt::kWOff + rv.slot * Lt::kTileBytes
                                                 : Lt::kVOff + rv.slot * Lt::kVBytes);
                const int chunks = (end - nv) * 8;
                for (int c = threadIdx.x; c < chunks * Lt::kPanels; c += kSoftWarps * 32)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                                     vt + (c / chunks) * 8192 + nv * 128 + (c % chunks) * 16),
                                 "r"(0u)
                                 : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_pready + 8 * (k & 1));
            // The lane's part of the sum of each row's fp32 weights (for the
            // lse), after P has been handed on.  The sum of the weights as
            // rounded for the P V product, used for the normalisation so that
            // O / l is an exact convex combination of the values, is
            // accumulated by the tensor core.
            tmem_accumulate<NC>(sum_t, v, first);
        }
        // ---- end of segment: O / l and lse ----
        --k;  // the last step
        {
            const bool whole = w.t == 0 && sg.blk;
            const size_t slot = (size_t)(w.b * p.Hkv + w.h) + blockIdx.x;
            // while P V of the last step runs, the sums over the keys (through
            // the other P buffer)
            if (k >= 1) await(b_pvdone, (k - 1) & 1, (k - 1) >> 1);
            {
                float l[NC];
                tmem_wait_st();
                tmem_ld<NC>(sum_t, l);
                lane_reduce<false, NC, N>(l, sbase + Lt::kPOff + (uint32_t)((~k & 1) * Lt::kPBytes),
                                          red_sm + (warp & 3) * N * 4, group, key);
            }
            await(b_pvdone, k & 1, k >> 1);
            fence_after();
            if (D == 64) {  // lanes 64.. hold the rounded row sums: to all through shared memory
                if ((warp & 3) == 2) {
                    float lr[NC];
                    tmem_ld<NC>(tmem + lane_base + (uint32_t)(Lt::kOCol + col0), lr);
                    if (lane == 0)
#pragma unroll
                        for (int r = 0; r < NC; r += 4)
                            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(lr_sm + 4 * r),
                                         "f"(lr[r]), "f"(lr[r + 1]), "f"(lr[r + 2]), "f"(lr[r + 3])
                                         : "memory");
                }
                soft_sync(group);
            }
            // thread = dim (lane of O^T).  A whole pair's rows are staged as
            // bf16 in the group's slice of the P buffer (read by no MMA until
            // the group hands on its next P) and leave as 16-byte stores; a
            // partial's fp32 rows go straight out, 128 bytes a warp and row.
            constexpr int kUnit = 2 * NC;  // contiguous bytes of the slice
            const uint32_t pcur = sbase + Lt::kPOff + (uint32_t)((k & 1) * Lt::kPBytes);
            if (key < D) {
                float o[NC];
                const uint32_t o_t = tmem + lane_base + (uint32_t)(Lt::kOCol + col0);
                if constexpr (D == 64) tmem_ld<NC>(o_t, o);
#pragma unroll
                for (int c = 0; c < NC; c += 16) {
                    float lr[16];
                    if constexpr (D == 128) {
                        tmem_ld_two<16>(o_t + c, o_t + (Lt::kLCol - Lt::kOCol) + c, o + c, lr);
                    } else {
#pragma unroll
                        for (int r = 0; r < 16; r += 4) {
                            const float4 y = lds4(lr_sm + 4 * (c + r));
                            lr[r] = y.x;
                            lr[r + 1] = y.y;
                            lr[r + 2] = y.z;
                            lr[r + 3] = y.w;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 16; ++r) o[c + r] *= inverse(lr[r]);
                }
                if (whole) {
#pragma unroll
                    for (int r = 0; r < NC; ++r)
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(
                                         slice_at<N>(pcur, group, (r * D + key) * 2 / kUnit) +
                                         key * 2 % kUnit),
                                     "h"((uint16_t)pack_bf16(o[r], 0.f))
                                     : "memory");
                } else {
                    float *ob = p.part_o + (slot * p.rows_max + col0) * D + key;
#pragma unroll
                    for (int r = 0; r < NC; ++r)
                        if (r < rows_active) __stcg(ob + r * D, o[r]);
                }
            }
            soft_sync(group);  // the row sums of all warps
            if (key < NC && key < rows_active) {
                const int r = key, qr = col0 + r;
                const uint32_t red = red_sm + 4 * r;
                const float lsum = (lds(red) + lds(red + 4 * N)) + (lds(red + 8 * N) + lds(red + 12 * N));
                // m + log2(l), l's exponent apart: m and it may cancel
                const float e = (float)((int)(__float_as_uint(lsum) >> 23) - 127);
                const float f = __uint_as_float((__float_as_uint(lsum) & 0x7fffffu) | 0x3f800000u);
                const float lse = !(lsum <= 3.4e38f) ? lsum  // infinite or NaN
                                  : lsum > 0.f
                                      ? ((e - lds(nm_sm + 4 * r)) + __log2f(f)) * kLn2
                                      : -INFINITY;
                if (whole)
                    p.lse[((size_t)w.b * p.Hq + (size_t)w.h * p.G + qr % p.G) * p.max_block +
                          qr / p.G] = lse;
                else
                    p.part_lse[slot * p.rows_max + qr] = lse;
            }
            if (whole) {
                for (int c = key; c < min(rows_active, NC) * (D / 8); c += 128) {
                    const int r = c / (D / 8), x = c * 16;
                    uint4 y;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(y.x), "=r"(y.y), "=r"(y.z), "=r"(y.w)
                                 : "r"(slice_at<N>(pcur, group, x / kUnit) + x % kUnit)
                                 : "memory");
                    const int qr = col0 + r;
                    *reinterpret_cast<uint4 *>(
                        p.out + (((size_t)w.b * p.max_block + qr / p.G) * p.Hq + (size_t)w.h * p.G +
                                 qr % p.G) * D + (c % (D / 8)) * 8) = y;
                }
            }
            soft_sync(group);  // the rows' values and the slice may be written again
            if (whole) {  // rows past the block: 0 and lse -inf
                const int act = p.G * w.T;
                for (int idx = threadIdx.x; idx < (p.rows_max - act) * (D / 8);
                     idx += kSoftWarps * 32) {
                    const int r = act + idx / (D / 8), col = (idx % (D / 8)) * 8;
                    const int ii = r / p.G, gg = r % p.G;
                    *reinterpret_cast<uint4 *>(p.out + (((size_t)w.b * p.max_block + ii) *
                                                             p.Hq +
                                                         (size_t)w.h * p.G + gg) * D + col) =
                        make_uint4(0u, 0u, 0u, 0u);
                    if (col == 0)
                        p.lse[((size_t)w.b * p.Hq + (size_t)w.h * p.G + gg) * p.max_block +
                              ii] = -INFINITY;
                }
            }
            fence_before();
        }
        ++k;
        done += sg.tiles;
        walk_segment(p, w, sg);
        }
    }
    if (warp == kMmaWarp || warp == kSWarp) {
        // all MMAs this warp issued are complete before tensor memory is freed
        // (only a timed-out run can leave any in flight)
        const uint32_t drain = b_drain + (warp == kSWarp ? 8 : 0);
        if (elect_one()) mma_commit(drain);
        __syncwarp();
        const unsigned long long t0 = globaltimer();
        while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < kWaitNs) {
        }
    }
    // every MMA was waited on by its issuing warp and the softmax warps
    fence_before();
    __syncthreads();
    fence_after();
    if (lds(abort_flag) != 0.f) {  // a wait gave up: copies still in flight land before exit
        if (warp == kProducerWarp && elect_one()) {
            for (int s = loads - 1; s >= 0 && s >= loads - VS; --s)
                drain_wait(b_vfull + 8 * (s % VS), (uint32_t)((s / VS) & 1));
            for (int q = qseg; q >= 0 && q >= qseg - 1; --q)
                drain_wait(b_qfull + 8 * (q & 1), (uint32_t)((q >> 1) & 1));
        }
        if (warp == kSWarp && elect_one())
            for (int s = kloads - 1; s >= 0 && s >= kloads - KS; --s)
                drain_wait(b_kfull + 8 * (s % KS), (uint32_t)((s / KS) & 1));
        if (VF8 && warp == kConvWarp0 && lane == 0 && drain_copy >= 0)
            drain_wait(b_wready + 8 * (drain_copy % WS), (uint32_t)((drain_copy / WS) & 1));
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "n"(Lt::kTmemCols));
}

}  // namespace

// ---- split-K merge ------------------------------------------------------------
// One warp per RPW query rows of a split pair (rows w, w + 4, ... of the
// CTA's 4 RPW rows); lane l holds columns [VPL l, VPL (l+1)).  With partial s
// holding O_s / l_s and lse_s for the row:
//   out = sum_s e^(lse_s - M) O_s / l_s / sum_s e^(lse_s - M),
//   lse = M + ln sum_s e^(lse_s - M),  M = max_s lse_s,
// (NaN if any lse_s is) and rows past the block get 0 and lse -inf.  The pair's segments are found
// from the lengths before griddepcontrol.wait (the attention grid this one
// depends on started after every kernel that could write them had
// completed); the partials are read after it, SEGS segments of each of the
// RPW rows in flight at once.  SEGS x RPW trades round trips and CTAs for
// registers: at D = 128, 8 x 1 takes 116 registers a thread (4 CTAs per SM),
// 4 x 1 72 (7), 2 x 1 40 (12), 2 x 2 about the same as 4 x 1 with half the
// CTAs.
constexpr int kMergeWarps = 4;

template <int SEGS, int RPW>
constexpr int merge_min_blocks() {
    return SEGS * RPW >= 8 ? 4 : SEGS * RPW >= 4 ? 7 : 12;
}

template <int D, int SEGS, int RPW>
__global__ void __launch_bounds__(kMergeWarps * 32, merge_min_blocks<SEGS, RPW>())
    merge_kernel(const AttnParams p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int VPL = D / 32;
    constexpr int kRowsPerCta = kMergeWarps * RPW;
    const int rblocks = (p.rows_max + kRowsPerCta - 1) / kRowsPerCta;
    const int pair = blockIdx.x / rblocks;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = (blockIdx.x % rblocks) * kRowsPerCta + warp;  // rows row0 + r * kMergeWarps
    const int b = pair / p.Hkv, h = pair % p.Hkv;
    const int C = p.num_ctas;
    // one pass: all tiles, and the tiles of the sequences before b
    long long total = 0, before = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
        const int nt = seq_tiles(p, b0 + lane);
        total += (long long)__reduce_add_sync(kFull, (unsigned)nt) * p.Hkv;
        before += (long long)__reduce_add_sync(kFull, b0 + lane < b ? (unsigned)nt : 0u) * p.Hkv;
    }
    const Split sp = split_from_total(p, total);
    const int nt = tiles_of(clamp_prefix(p, b));
    const long long first = before + (long long)h * nt;  // the pair's first tile
    const long long first_w = first + (long long)sp.beta * pair;
    const int c0 = cta_of_w(first_w, sp, C);
    // every CTA holds a tile when beta > 0 or N >= C, so the pair's segments
    // are those of CTAs c0 .. c1; otherwise (beta = 0) each tile is a CTA of
    // its own
    const bool contiguous = sp.beta > 0 || sp.N >= C;
    const int nseg = contiguous ? cta_of_w(first_w + nt - 1, sp, C) - c0 + 1 : nt;
    const int rows_active = p.G * clamp_block(p, b);

    // partials come from the attention grid
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (nseg <= 1) return;  // a single segment wrote its output
    uint16_t *orow[RPW];
    float *lrow[RPW];
    bool act[RPW];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int row = row0 + r * kMergeWarps;
        const int i = row / p.G, g = row % p.G;
        orow[r] = p.out + (((size_t)b * p.max_block + i) * p.Hq + (size_t)h * p.G + g) * D +
                  VPL * lane;
        lrow[r] = p.lse + ((size_t)b * p.Hq + (size_t)h * p.G + g) * p.max_block + i;
        act[r] = row < rows_active;
        if (row < p.rows_max && !act[r]) {  // rows past the block: 0 and lse -inf
            if (VPL == 4)
                *reinterpret_cast<uint2 *>(orow[r]) = make_uint2(0u, 0u);
            else
                *reinterpret_cast<uint32_t *>(orow[r]) = 0u;
            if (lane == 0) *lrow[r] = -INFINITY;
        }
    }
    float M[RPW], L[RPW], acc[RPW][VPL];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        M[r] = -INFINITY;
        L[r] = 0.f;
#pragma unroll
        for (int v = 0; v < VPL; ++v) acc[r][v] = 0.f;
    }
#pragma unroll 1
    for (int s0 = 0; s0 < nseg; s0 += SEGS) {
        float ls[RPW][SEGS], os[RPW][SEGS][VPL];
#pragma unroll
        for (int r = 0; r < RPW; ++r)
#pragma unroll
            for (int u = 0; u < SEGS; ++u) {
                ls[r][u] = -INFINITY;
#pragma unroll
                for (int v = 0; v < VPL; ++v) os[r][u][v] = 0.f;
                if (act[r] && s0 + u < nseg) {
                    const int c = contiguous ? c0 + s0 + u : cta_of_w(first + s0 + u, sp, C);
                    const size_t rs = ((size_t)pair + c) * p.rows_max + row0 + r * kMergeWarps;
                    ls[r][u] = __ldcg(p.part_lse + rs);
                    const float *src = p.part_o + rs * D + VPL * lane;
                    if (VPL == 4) {
                        const float4 x = __ldcg(reinterpret_cast<const float4 *>(src));
                        os[r][u][0] = x.x;
                        os[r][u][1 % VPL] = x.y;
                        os[r][u][2 % VPL] = x.z;
                        os[r][u][VPL - 1] = x.w;
                    } else {
                        const float2 x = __ldcg(reinterpret_cast<const float2 *>(src));
                        os[r][u][0] = x.x;
                        os[r][u][VPL - 1] = x.y;
                    }
                }
            }
#pragma unroll
        for (int r = 0; r < RPW; ++r) {
            float mn = M[r];
#pragma unroll
            for (int u = 0; u < SEGS; ++u) mn = max_nan(mn, ls[r][u]);
            if (mn == -INFINITY) continue;
            const float a = __expf(M[r] - mn);  // 0 while M is -inf
            L[r] *= a;
#pragma unroll
            for (int v = 0; v < VPL; ++v) acc[r][v] *= a;
#pragma unroll
            for (int u = 0; u < SEGS; ++u) {
                const float wgt = __expf(ls[r][u] - mn);  // 0 for absent segments
                L[r] += wgt;
#pragma unroll
                for (int v = 0; v < VPL; ++v) acc[r][v] += wgt * os[r][u][v];
            }
            M[r] = mn;
        }
    }
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        if (!act[r]) continue;
        const float inv = L[r] > 0.f ? 1.f / L[r] : 0.f;
        if (VPL == 4)
            *reinterpret_cast<uint2 *>(orow[r]) =
                make_uint2(pack_bf16(acc[r][0] * inv, acc[r][1 % VPL] * inv),
                           pack_bf16(acc[r][2 % VPL] * inv, acc[r][VPL - 1] * inv));
        else
            *reinterpret_cast<uint32_t *>(orow[r]) =
                pack_bf16(acc[r][0] * inv, acc[r][VPL - 1] * inv);
        if (lane == 0) *lrow[r] = L[r] == 0.f ? -INFINITY : M[r] + __logf(L[r]);
    }
}

// The merge variants (segments in flight x rows per warp) and their resident
// CTAs per SM, looked up once per device.
constexpr int kMergeVariants = 4;
constexpr int kMergeSegs[kMergeVariants] = {8, 4, 2, 2};
constexpr int kMergeRpw[kMergeVariants] = {1, 1, 1, 2};

template <int D>
cudaError_t merge_occupancy(int dev, int occ[kMergeVariants]) {
    static std::atomic<int> cached[64][kMergeVariants];
    if (dev < 64 && cached[dev][kMergeVariants - 1].load(std::memory_order_acquire) > 0) {
        for (int v = 0; v < kMergeVariants; ++v)
            occ[v] = cached[dev][v].load(std::memory_order_relaxed);
        return cudaSuccess;
    }
    const void *fns[kMergeVariants] = {
        reinterpret_cast<const void *>(merge_kernel<D, 8, 1>),
        reinterpret_cast<const void *>(merge_kernel<D, 4, 1>),
        reinterpret_cast<const void *>(merge_kernel<D, 2, 1>),
        reinterpret_cast<const void *>(merge_kernel<D, 2, 2>)};
    for (int v = 0; v < kMergeVariants; ++v) {
        // few pairs: the shared-memory split of the attention kernel that the merge runs
        // beside; many rows to merge read faster with the default's larger L1
        cudaError_t e = cudaSuccess;
        if (kMergeSegs[v] > 2)
            e = cudaFuncSetAttribute(fns[v], cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[v], fns[v], kMergeWarps * 32, 0);
        if (e != cudaSuccess) return e;
        occ[v] = std::max(occ[v], 1);
    }
    if (dev < 64) {
        for (int v = 0; v < kMergeVariants - 1; ++v)
            cached[dev][v].store(occ[v], std::memory_order_relaxed);
        cached[dev][kMergeVariants - 1].store(occ[kMergeVariants - 1], std::memory_order_release);
    }
    return cudaSuccess;
}

template <int D, bool KF8, bool VF8, int N>
cudaError_t launch_n(const AttnParams &p, const CUtensorMap &tk, const CUtensorMap &tk2,
                     const CUtensorMap &tv,
                     const CUtensorMap &tkb, const CUtensorMap &tvb, const CUtensorMap &tq,
                     cudaStream_t stream) {
    using Lt = Layout<D, KF8, VF8, N>;
    constexpr int smem = Lt::kBytes;
    static std::atomic<bool> configured[64];  // the smem opt-in, once per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(attn_kernel<D, KF8, VF8, N>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(attn_kernel<D, KF8, VF8, N>,
                                 cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.num_ctas);
    cfg.blockDim = dim3(Lt::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, attn_kernel<D, KF8, VF8, N>, tk, tk2, tv, tkb, tvb, tq, p);
}

// The merge, a programmatic dependent of either attention kernel.
template <int D>
cudaError_t launch_merge(const AttnParams &p, cudaStream_t stream) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // The merge variant with the fewest estimated sequential steps: waves of
    // resident merge CTAs (at least one) times L2 round trips per row (at
    // least one), for a pair's average segment count 1 + C / (B Hkv).
    const double segs = 1.0 + (double)p.num_ctas / ((double)p.B * p.Hkv);
    int occ[kMergeVariants];
    e = merge_occupancy<D>(dev, occ);
    if (e != cudaSuccess) return e;
    int best = 0;
    double best_cost = 0.0;
    long long best_ctas = 0;
    for (int v = 0; v < kMergeVariants; ++v) {
        const int rows_per_cta = kMergeWarps * kMergeRpw[v];
        const long long ctas =
            (long long)p.B * p.Hkv * ((p.rows_max + rows_per_cta - 1) / rows_per_cta);
        const double waves = std::max(1.0, (double)ctas / ((double)occ[v] * p.num_ctas));
        const double cost = waves * std::max(1.0, segs / kMergeSegs[v]);
        if (v == 0 || cost < best_cost) {
            best = v;
            best_cost = cost;
            best_ctas = ctas;
        }
    }
    cfg.gridDim = dim3((unsigned)best_ctas);
    cfg.blockDim = dim3(kMergeWarps * 32);
    cfg.dynamicSmemBytes = 0;
    if (best == 0) return cudaLaunchKernelEx(&cfg, merge_kernel<D, 8, 1>, p);
    if (best == 1) return cudaLaunchKernelEx(&cfg, merge_kernel<D, 4, 1>, p);
    if (best == 2) return cudaLaunchKernelEx(&cfg, merge_kernel<D, 2, 1>, p);
    return cudaLaunchKernelEx(&cfg, merge_kernel<D, 2, 2>, p);
}

// The MMAs' query columns: the pair's G * max_block rows rounded up to 16, 32 or 64.
template <int D, bool KF8, bool VF8>
cudaError_t launch_d(const AttnParams &p, const CUtensorMap &tk, const CUtensorMap &tk2,
                     const CUtensorMap &tv,
                     const CUtensorMap &tkb, const CUtensorMap &tvb, const CUtensorMap &tq,
                     cudaStream_t stream) {
    if (p.rows_max <= 16) return launch_n<D, KF8, VF8, 16>(p, tk, tk2, tv, tkb, tvb, tq, stream);
    if (p.rows_max <= 32) return launch_n<D, KF8, VF8, 32>(p, tk, tk2, tv, tkb, tvb, tq, stream);
    return launch_n<D, KF8, VF8, 64>(p, tk, tk2, tv, tkb, tvb, tq, stream);
}

cudaError_t launch_attn(const AttnParams &p, int head_dim, bool keys_e4m3, bool values_e4m3,
                        const CUtensorMap &tk, const CUtensorMap &tk2, const CUtensorMap &tv,
                        const CUtensorMap &tkb, const CUtensorMap &tvb, const CUtensorMap &tq,
                        cudaStream_t stream) {
#define DAS_LAUNCH(D, K8, V8) launch_d<D, K8, V8>(p, tk, tk2, tv, tkb, tvb, tq, stream)
    if (head_dim == 128) {
        if (keys_e4m3)
            return values_e4m3 ? DAS_LAUNCH(128, true, true) : DAS_LAUNCH(128, true, false);
        if (values_e4m3) return DAS_LAUNCH(128, false, true);
    }
    if (head_dim == 64) {
        if (keys_e4m3) return values_e4m3 ? DAS_LAUNCH(64, true, true) : DAS_LAUNCH(64, true, false);
        return values_e4m3 ? DAS_LAUNCH(64, false, true) : DAS_LAUNCH(64, false, false);
    }
#undef DAS_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace tc

int attn_grid_size(int device) {
    static std::atomic<int> sms_of[64];  // the SM count, looked up once per device
    if (device >= 0 && device < 64) {
        const int known = sms_of[device].load(std::memory_order_relaxed);
        if (known > 0) return known;
    }
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return 0;
    if (device >= 0 && device < 64) sms_of[device].store(sms, std::memory_order_relaxed);
    return sms;
}

// Whether a call takes the kernel of das_rows.cu.  The transposed kernel costs less per
// tile and up to 3 us more per call (a segment's first scores wait for a whole step,
// its first references and its end take barriers), so it wins where the average
// segment, tiles / (pairs + CTAs), is long.  The prefix lengths are the device's, and
// a server's cache is longer than most of its prefixes; the capacity bounds them.  So
// the lines lie at twice the segments where the two kernels break even: no call over
// a cache at least half full is slower.  Below, at the least segments, the transposed
// kernel takes up to 1.15 (16 columns) and 1.4 (64) times as long.  (Both in one kernel,
// chosen by the lengths, cost each of them up to 10 to 25 %: their code is more than
// the instruction caches hold well.)  Measured, time of das_rows.cu's kernel over the
// transposed one's at that many tiles a segment (few: at most a pair a CTA / many):
//   bf16 keys and values, D = 64: 16 columns 2.0 0.94, 5.0 1.08, 11 1.11, 33 1.28; 32: 5.0 0.96,
//     11 1.02, 33 1.21; 64: 7.1 0.93, 19 1.01, 33 1.09
//   the same at D = 128: 16: 0.6 0.90, 5.0 1.05, 33 1.00; 32: 2.3 0.95, 33 1.01; 64: 5.5 0.89,
//     33 1.00, so never
//   e4m3 keys, D = 128: 16: 0.6 1.05, 2.3 0.96, 9.4 1.16, 33 1.09, so always; 32: 1.9 0.95, 3.2 1.01,
//     33 1.11; 64: 5.5 0.93, 19 1.01, 33 1.02 / 7.9 0.84, 23 1.02
//   e4m3 keys, D = 64: 16: 2.3 0.91, 5.5 1.04, 33 1.40 / 6.1 0.94, 7.9 1.14; 32: 5.5 0.95, 11 1.03,
//     33 1.26; 64: 19 0.97, 29 1.07 / 23 0.99
//   e4m3 keys and values, D = 128: 16: 0.6 0.95, 3.2 1.10, 33 1.40 / 6.1 0.97, 7.9 1.13; 32: 4.3 0.87,
//     5.5 1.01, 33 1.30 / 7.9 1.04; 64: 5.5 0.93, 11 1.00, 33 1.22 / 14 1.03
//   the same at D = 64: 16: 2.3 0.96, 5.5 1.08, 33 1.33 / 7.9 1.17; 32: 7.1 0.87, 12 0.98, 33 1.12 /
//     18 1.07; 64: 19 0.97, 33 1.04 / 23 1.00
// (e4m3 values alone take the lines of e4m3 keys and values.)
bool attn_short_ranges(int device, int batch, int kv_heads, int capacity, int head_dim,
                       int rows_max, bool keys_e4m3, bool values_e4m3) {
    const long long pairs = (long long)batch * kv_heads, C = attn_grid_size(device);
    const bool many = pairs > C;
    const int cols = rows_max <= 16 ? 0 : rows_max <= 32 ? 1 : 2;
    int need;
    if (!keys_e4m3 && !values_e4m3) {
        if (head_dim == 128) return true;
        need = cols == 0 ? 10 : cols == 1 ? 22 : 36;
    } else if (head_dim == 128 && !values_e4m3) {
        need = cols == 0 ? 0 : cols == 1 ? 6 : many ? 46 : 40;
    } else if (head_dim == 128) {
        need = cols == 0 ? (many ? 14 : 8) : cols == 1 ? (many ? 16 : 12) : (many ? 26 : 22);
    } else if (!values_e4m3) {
        need = cols == 0 ? (many ? 16 : 12) : cols == 1 ? 22 : many ? 48 : 40;
    } else {
        need = cols == 0 ? (many ? 16 : 12) : cols == 1 ? 30 : many ? 46 : 40;
    }
    const long long tiles = pairs * (((long long)capacity + kTileKeys - 1) / kTileKeys + 1);
    return tiles < need * (pairs + C);
}

namespace {
size_t round256(size_t n) { return (n + 255) & ~size_t(255); }
}  // namespace

// header | part_o [slots][rows_max][D] | part_lse [slots][rows_max], slots =
// B * Hkv + C (the slot of a segment is pair + CTA).
size_t attn_workspace_bytes(int device, int batch, int kv_heads, int rows_max, int head_dim) {
    const int C = attn_grid_size(device);
    if (C <= 0) return 0;
    const size_t slots = (size_t)batch * kv_heads + (size_t)C;
    return kWorkspaceHeader + round256(slots * rows_max * head_dim * sizeof(float)) +
           round256(slots * rows_max * sizeof(float));
}

void attn_workspace_layout(void *workspace, int batch, int kv_heads, int rows_max, int head_dim,
                           int num_ctas, AttnParams &p) {
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    const size_t slots = (size_t)batch * kv_heads + (size_t)num_ctas;
    p.status = reinterpret_cast<int32_t *>(ws);
    size_t off = kWorkspaceHeader;
    p.part_o = reinterpret_cast<float *>(ws + off);
    off += round256(slots * rows_max * head_dim * sizeof(float));
    p.part_lse = reinterpret_cast<float *>(ws + off);
}

cudaError_t attn_launch(AttnParams p, int head_dim, bool keys_e4m3, bool values_e4m3,
                        const CUtensorMap &tm_k, const CUtensorMap &tm_k2, const CUtensorMap &tm_v,
                        const CUtensorMap &tm_kb, const CUtensorMap &tm_vb,
                        const CUtensorMap &tm_q, cudaStream_t stream) {
    const int tile_bytes = kTileKeys * head_dim * ((keys_e4m3 ? 1 : 2) + (values_e4m3 ? 1 : 2));
    p.block_weight = p.short_ranges ? 3 : tc::kBlockBytes / tile_bytes;
    cudaError_t e;
    if (p.short_ranges)
        e = rows_launch(p, head_dim, keys_e4m3, values_e4m3, tm_k, tm_v, tm_kb, tm_vb, tm_q, stream);
    else
        e = tc::launch_attn(p, head_dim, keys_e4m3, values_e4m3, tm_k, tm_k2, tm_v, tm_kb, tm_vb, tm_q,
                            stream);
    if (e != cudaSuccess) return e;
    return head_dim == 128 ? tc::launch_merge<128>(p, stream) : tc::launch_merge<64>(p, stream);
}

}  // namespace das
