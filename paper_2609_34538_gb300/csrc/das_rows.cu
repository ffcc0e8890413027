// das_rows.cu -- the attention kernel for bf16 keys and values with 128-wide heads, and
// for short ranges of every form: query rows in the lanes of the accumulators
// (M = 64), one 64-key tile at a time.  das_attention.cu describes the work split,
// the segments and the merge, and has the kernel for longer ranges of the other
// forms; attn_short_ranges says where the line lies.  This one starts sooner (a
// row's maximum needs no MMA of its own, a segment ends without sums over the
// keys), which is what counts where a CTA has a few tiles, and costs more per tile.
//
// One CTA = four softmax warps + one TMA warp + two MMA warps (+ four conversion
// warps when prefix keys or values are stored as e4m3).
//   S = Q K^T    tcgen05.mma M=64 N=64 K=D   -> S buffer (k % 4) in TMEM
//                (e4m3 keys at D = 128: two e4m3 passes over the query rows
//                split exactly into hi + lo, see split_q)
//   O += P V     tcgen05.mma M=64 N=D K=64   -> O in TMEM
//   2 l += P 2   tcgen05.mma M=64 N=8 K=64   -> the rounded row sums, doubled
// e4m3 values are widened to f16 and meet f16 weights (a rounding of 2^-11 where bf16
// has 2^-8); all other operands are bf16 (e4m3 keys where they are not split: widened).
// An M=64 MMA puts row r in TMEM lane 32 (r / 16) + r % 16: softmax warp w owns
// rows 16w..16w+15 and two threads share a row.  A row's reference max moves only
// when a score exceeds it by more than 2^8.  Pairs of at most 16 (32) query rows
// (D = 128, bf16 values) load the rows four (two) times, and the softmax warps of a
// copy take a quarter (half) of every tile's keys; the copies are combined by
// log-sum-exp through shared memory at a segment's end.
#include <atomic>

#include "das_tc.h"

namespace das {
namespace tc {
namespace {

constexpr int kSoftWarps = 4;
constexpr int kProducerWarp = kSoftWarps;     // TMA loads
constexpr int kMmaWarp = kSoftWarps + 1;      // tcgen05 MMAs of P V
constexpr int kSWarp = kSoftWarps + 2;        // tcgen05 MMAs of S
constexpr int kConvWarp0 = kSoftWarps + 3;    // e4m3 -> bf16 widening, query split
constexpr int kRows = 64;            // M of every MMA (query rows per pair)
constexpr int kSBufs = 4;            // S buffers in tensor memory
constexpr int kTmemCols = 512;       // S buffers [0, 64 kSBufs), O [64 kSBufs, 64 kSBufs + D),
                                     // then 8 columns whose first is twice the rounded row sum
constexpr float kRescaleLog2 = 8.f;  // move the reference max only beyond 2^8
constexpr float kShiftF16 = 7.f;     // f16 weights are 2^7 larger: f16 holds 2^-25 to 2^16

// 32 columns of S for the calling thread (16 lanes x 2 halves): thread t < 16
// of a warp gets TMEM lane t, columns [c, c + 32), thread t + 16 the same lane,
// [c + 32, c + 64).  With M = 64 a warp's rows sit in its first 16 lanes, so
// two threads share each row.
__device__ __forceinline__ void tmem_ld_half32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32], "
        "32;\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}
// (Replicated rows) the calling thread's 8 scores: lane t < 16 of the warp
// reads TMEM lane t, columns [0, 8) from taddr, lane t + 16 the same lane,
// columns [8, 16).
__device__ __forceinline__ void tmem_ld_half8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], 8;\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}
// (Replicated rows, two copies) the calling thread's 16 scores: lane t < 16
// reads TMEM lane t, columns [0, 16) from taddr, lane t + 16 the same lane,
// columns [16, 32).
__device__ __forceinline__ void tmem_ld_half16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15}, [%16], 16;\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
// The O row of the calling thread's half: with M = 64, thread t < 16 of a warp
// gets TMEM lane t, columns [64 g, 64 g + 32) for g < D / 64, and thread t + 16
// the same lane, columns [64 g + 32, 64 g + 64).  All loads are issued before
// the single wait, so the epilogue pays one TMEM round trip.
template <int D>
__device__ __forceinline__ void tmem_ld_orow(uint32_t taddr, float (&v)[D / 2]);
template <>
__device__ __forceinline__ void tmem_ld_orow<128>(uint32_t taddr, float (&v)[64]) {
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%64], 32;\n"
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,"
        "%27,%28,%29,%30,%31}, [%65], 32;\n"
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,"
        "%43,%44,%45,%46,%47}, [%66], 32;\n"
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,"
        "%59,%60,%61,%62,%63}, [%67], 32;\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]),
          "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]),
          "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]),
          "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]),
          "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]),
          "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr), "r"(taddr + 16), "r"(taddr + 64), "r"(taddr + 80)
        : "memory");
#pragma unroll
    for (int j = 0; j < 64; ++j) v[j] = __uint_as_float(r[j]);
}
template <>
__device__ __forceinline__ void tmem_ld_orow<64>(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%32], 32;\n"
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,"
        "%27,%28,%29,%30,%31}, [%33], 32;\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr), "r"(taddr + 16)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(
            taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])),
        "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])), "r"(__float_as_uint(v[20])),
        "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
        "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])),
        "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])),
        "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Shared memory of one CTA.  Keys and values stored as e4m3 (the depths below
// R in a das_kv_cache_f8) land in the stage as 8-bit tiles [64 keys][D].
//   kQSplit (keys e4m3, values bf16, D = 128: Mature-V over a das_kv_cache_f8):
//     the key tile lands 128-byte swizzled and is read by the S MMAs as it is
//     (kind::f8f6f4).  The conversion warps split each segment's bf16 query
//     rows exactly into two e4m3 parts, 2^e q = hi + lo with one power of two
//     e per row (see split_q), and S = (hi + lo) K^T is two e4m3 products
//     accumulated in fp32, 2^e times the bf16 product.  The pair's block
//     tile (bf16 keys) has a bf16 key buffer of its own and bf16 MMAs.
//   otherwise: the conversion warps widen every e4m3 tile (keys to bf16, values to f16), in
//     the 128-byte-swizzled layout the MMAs read, held in a ring of kConvSlots
//     slots (tile j in slot j % kConvSlots) rather than one per stage: the
//     smaller stages then fit 6 (or 7) deep instead of 4, which is what keeps
//     more DRAM requests in flight per SM.  A pair's block tile is bf16: the
//     conversion warps load its e4m3-stored operands straight into the ring
//     slot, the producer the others into the stage.
template <int D, bool KF8, bool VF8, int NC = 1>
struct Layout {
    static constexpr bool REP = NC > 1;  // NC copies of the query rows (1, 2 or 4)
    static_assert(NC == 1 || NC == 2 || NC == 4, "copies: 1, 2 or 4");
    // bf16 keys, or e4m3 keys with the split-query scores; bf16 values; D = 128
    static_assert(!REP || (!VF8 && D == 128), "replicated rows: bf16 values, D = 128");
    static constexpr bool kQSplit = KF8 && !VF8 && D == 128;
    static constexpr bool kConv = KF8 || VF8;
    // (kQSplit: 4 stages of 24 KB measured faster than 5, e4m3 long 82.0 -> 81.5 us)
    static constexpr int kStages = kQSplit ? 4 : (KF8 && VF8) ? 7 : kConv ? 6 : 4;
    static constexpr int kConvSlots = 2;
    static constexpr int kThreads = (kSoftWarps + 3 + (kConv ? kConvWarps : 0)) * 32;
    static constexpr int kPanels = D / 64;
    static constexpr int kTileBytes = kTileKeys * D * 2;  // a bf16 K or V tile
    static constexpr int kTile8Bytes = kTileKeys * D;     // an e4m3 tile
    static constexpr int kKBytes = KF8 ? kTile8Bytes : kTileBytes;  // K part of a stage
    static constexpr int kVBytes = VF8 ? kTile8Bytes : kTileBytes;  // V part of a stage
    static constexpr int kStageBytes = kKBytes + kVBytes;
    static constexpr int kConvBytes =
        kQSplit ? 0 : (KF8 ? kTileBytes : 0) + (VF8 ? kTileBytes : 0);
    static constexpr int kQBytes = kPanels * kRows * 128;  // one query buffer
    static constexpr int kQ8Bytes = kRows * 128;           // one e4m3 query part (D = 128)
    static constexpr int kPBytes = kRows * kTileKeys * 2;  // one P buffer
    static constexpr int kStagesOff = 0;
    static constexpr int kConvOff = kStages * kStageBytes;  // the ring of widened tiles, or
    // (kQSplit) the block tile's bf16 keys, then hi / lo of both query buffers
    static constexpr int kBlkKOff = kConvOff;
    static constexpr int kQ8Off = kConvOff + kTileBytes;
    static constexpr int kExtraBytes =
        kQSplit ? kTileBytes + 4 * kQ8Bytes : kConvSlots * kConvBytes;
    static constexpr int kQOff = kConvOff + kExtraBytes;
    static constexpr int kPOff = kQOff + 2 * kQBytes;
    // the B operand of the row-sum MMA: [8][64], row 0 twos (0x4000 is 2 as bf16 and as
    // f16: the sums come doubled, which is exact), 128-byte swizzled
    static constexpr int kTwosOff = kPOff + 2 * kPBytes;
    static constexpr int kBarOff = kTwosOff + 1024;
    // barriers: full[kStages], empty[kStages], qfull[2], qempty[2],
    // sready[kSBufs], sfree[kSBufs], pready[2], pvdone[2], drain[2],
    // cready[kConvSlots], kfree[kConvSlots], vfree[kConvSlots], qsplit[2], bkfree
    static constexpr int kNumBars = 2 * kStages + 10 + 2 * kSBufs + 3 * kConvSlots + 3;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kLenOff = kMiscOff + 16;  // lengths read before the dependency wait
    static constexpr int kQeOff = kLenOff + 64 * 4;  // (kQSplit) e of each row, per query buffer
    // (REP) the segment end's exchange, then (m, l, rounded l) of every MMA
    // row [kRows][4]; rows are padded by 16 bytes so that consecutive rows
    // start in different bank groups.  Compacted (e4m3 keys, whose stages
    // leave too little shared memory for whole rows): a softmax thread holds
    // D / 2 values of its copy's O row, in NC groups of D / 2 / NC; each
    // group is combined by the thread of the copy with its index, so a thread
    // stores only the NC - 1 groups other copies combine: [2 halves][kRows]
    // [kXchStride] floats.
    // With bf16 keys there is room for the whole rows: every copy's O row
    // [kRows][kXchStride] (measured faster for bf16: decode 17.43 -> 17.12 us).
    static constexpr bool kCompactXch = KF8;
    static constexpr int kXchStride =
        !REP ? 0 : kCompactXch ? (NC - 1) * (D / 2 / NC) + 4 : D + 4;
    static constexpr int kXchOff = (kQeOff + (kQSplit ? 2 * kRows * 4 : 0) + 15) & ~15;
    static constexpr int kXchBytes =
        !REP ? 0
             : ((kCompactXch ? 2 * kRows * kXchStride : kRows * kXchStride) + kRows * 4) * 4;
    static constexpr int kBytes = kXchOff + kXchBytes + 1024;  // + alignment slack
    static_assert(kStageBytes % 1024 == 0 && kKBytes % 1024 == 0 && kConvBytes % 1024 == 0,
                  "swizzled tiles need 1024-byte alignment");
    static_assert(kBytes <= 232448, "shared memory per CTA");
};

// K-major 128B-swizzled address of bf16 element (row, col) of a [64][64] panel
__device__ __forceinline__ uint32_t p_chunk_addr(uint32_t base, int row, int chunk) {
    return base + row * 128 + ((chunk ^ (row & 7)) << 4);
}

// Two e4m3 codes (the low and high byte of a) -> bf16x2 (low, high half):
// the hardware conversion to f16x2 (exact: every e4m3 value, NaN included, is
// an f16 value), each half widened to f32 and the pair rounded to bf16x2
// (exact again: an e4m3 value has at most 4 significant bits).
__device__ __forceinline__ uint32_t e4m3x2_to_bf16x2(uint32_t a) {
    uint32_t h;
    asm("{\n .reg .b16 t;\n cvt.u16.u32 t, %1;\n cvt.rn.f16x2.e4m3x2 %0, t;\n}\n"
        : "=r"(h)
        : "r"(a));
    float f0, f1;
    asm("{\n .reg .b16 l, u;\n mov.b32 {l, u}, %2;\n cvt.f32.f16 %0, l;\n cvt.f32.f16 %1, u;\n}\n"
        : "=f"(f0), "=f"(f1)
        : "r"(h));
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(f1), "f"(f0));
    return r;
}

// Widen an e4m3 key tile [64 keys][D] (row-major, as the 8-bit TMA box lands)
// into the bf16 tile the MMAs read: D / 64 panels of [64 keys][128 bytes],
// 16-byte chunk j of key r at (j ^ (r % 8)) * 16 (128-byte swizzle).  The 128
// conversion threads (ct = 0..127) each take 16-element chunks.
template <int D>
__device__ __forceinline__ void widen_tile(uint32_t src, uint32_t dst, int ct) {
    constexpr int kChunks = kTileKeys * D / 16;
#pragma unroll
    for (int i = 0; i < kChunks / (kConvWarps * 32); ++i) {
        const int c = ct + i * kConvWarps * 32;
        // Chunk c: 16 elements jj of a 64-column panel of a key.  The 8 lanes
        // of a quarter warp (one shared-memory wavefront of 16-byte accesses)
        // take two keys of opposite parity, so their loads (rows of D bytes)
        // and their swizzled stores each touch 8 distinct 16-byte bank groups.
        const int jj = c & 3;
        const int pnl = D == 128 ? (c >> 2) & 1 : 0;
        const int key = D == 128 ? ((c >> 4) << 1) + (pnl ^ ((c >> 3) & 1)) : c >> 2;
        const int d0 = pnl * 64 + jj * 16;
        uint32_t w0, w1, w2, w3;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3)
                     : "r"(src + key * D + d0));
        const uint32_t row = dst + (d0 / 64) * 8192 + key * 128;
        const int j = (d0 % 64) / 8;  // the first of two 16-byte bf16 chunks
        // bytes 0,1 / 2,3 of each word into the 16-bit halves of a register
        auto lo = [](uint32_t w) { return w & 0xFFFFu; };
        auto hi = [](uint32_t w) { return w >> 16; };
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         row + ((j ^ (key & 7)) << 4)),
                     "r"(e4m3x2_to_bf16x2(lo(w0))), "r"(e4m3x2_to_bf16x2(hi(w0))),
                     "r"(e4m3x2_to_bf16x2(lo(w1))), "r"(e4m3x2_to_bf16x2(hi(w1)))
                     : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         row + (((j + 1) ^ (key & 7)) << 4)),
                     "r"(e4m3x2_to_bf16x2(lo(w2))), "r"(e4m3x2_to_bf16x2(hi(w2))),
                     "r"(e4m3x2_to_bf16x2(lo(w3))), "r"(e4m3x2_to_bf16x2(hi(w3)))
                     : "memory");
    }
}

// Exact split of the query rows for e4m3 keys (D = 128).  Row r of the bf16
// query buffer q (two 128-byte-swizzled panels of [64 rows][64 dims]) becomes
// two e4m3 rows hi, lo (128-byte swizzled [64 rows][128 dims]) with
//   2^e q = hi + lo,  e = 7 - floor(log2 max_d |q_d|)  (clamped to +-120),
// so that the row's largest element scales into [128, 256).  hi is 2^e q
// rounded to e4m3 (4 significant bits) and lo the rounded remainder: a bf16
// value has 8 significant bits, so the remainder fits e4m3 exactly unless it
// falls below e4m3's smallest subnormal (2^-9), i.e. for elements below about
// 2^-9 of the row's largest.  Thread ct of the 128 conversion threads takes
// row ct / 2, dims [64 (ct % 2), +64); e is written to qexp[row].  A row of
// zeros gives e = 0; a row with an infinity or NaN gives kNotFinite (its scores
// are then NaN; the parts of an infinity would be finite).
constexpr int kNotFinite = 1 << 20;
__device__ __forceinline__ void split_q(uint32_t q, uint32_t hi, uint32_t lo, int *qexp, int ct) {
    const int row = ct >> 1, half = ct & 1;
    uint32_t w[32];
#pragma unroll
    for (int c = 0; c < 8; ++c)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[4 * c]), "=r"(w[4 * c + 1]), "=r"(w[4 * c + 2]), "=r"(w[4 * c + 3])
                     : "r"(q + half * (kRows * 128) + row * 128 + ((c ^ (row & 7)) << 4)));
    uint32_t mb = 0;  // largest magnitude, as bits (a NaN's are the largest)
#pragma unroll
    for (int i = 0; i < 32; ++i)
        mb = max(mb, max((w[i] << 16) & 0x7fff0000u, w[i] & 0x7fff0000u));
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
    int e = 0;
    if (mb != 0u && mb < 0x7f800000u) {
        e = 7 - ((int)(mb >> 23) - 127);
        e = e < -120 ? -120 : (e > 120 ? 120 : e);
    }
    const float sc = __uint_as_float((uint32_t)(127 + e) << 23);
    // word i holds dims 2i (low half) and 2i + 1 of the thread's 64
    uint32_t h[16], l[16];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const float xa = __uint_as_float(w[i] << 16) * sc;
        const float xb = __uint_as_float(w[i] & 0xffff0000u) * sc;
        uint32_t h2, f2, l2;
        asm("{\n .reg .b16 t;\n cvt.rn.satfinite.e4m3x2.f32 t, %1, %2;\n cvt.u32.u16 %0, t;\n}"
            : "=r"(h2)
            : "f"(xb), "f"(xa));
        asm("{\n .reg .b16 t;\n cvt.u16.u32 t, %1;\n cvt.rn.f16x2.e4m3x2 %0, t;\n}"
            : "=r"(f2)
            : "r"(h2));
        float ha, hb;
        asm("{\n .reg .b16 a, b;\n mov.b32 {a, b}, %2;\n cvt.f32.f16 %0, a;\n cvt.f32.f16 %1, b;\n}"
            : "=f"(ha), "=f"(hb)
            : "r"(f2));
        asm("{\n .reg .b16 t;\n cvt.rn.satfinite.e4m3x2.f32 t, %1, %2;\n cvt.u32.u16 %0, t;\n}"
            : "=r"(l2)
            : "f"(xb - hb), "f"(xa - ha));
        if (i & 1) {
            h[i >> 1] |= h2 << 16;
            l[i >> 1] |= l2 << 16;
        } else {
            h[i >> 1] = h2;
            l[i >> 1] = l2;
        }
    }
    // 16-byte chunk c of the 128-byte e4m3 row holds dims 16 c .. 16 c + 15:
    // this thread's are chunks 4 half .. 4 half + 3
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t off = row * 128 + (((4 * half + m) ^ (row & 7)) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(hi + off), "r"(h[4 * m]),
                     "r"(h[4 * m + 1]), "r"(h[4 * m + 2]), "r"(h[4 * m + 3])
                     : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(lo + off), "r"(l[4 * m]),
                     "r"(l[4 * m + 1]), "r"(l[4 * m + 2]), "r"(l[4 * m + 3])
                     : "memory");
    }
    if (half == 0) qexp[row] = mb >= 0x7f800000u ? kNotFinite : e;
}

// Registers a thread of the query-split variant may use: 144 x 352 threads
// leave room for one merge CTA (128 threads x 116) beside the attention CTA,
// so the merge kernel is resident before the attention grid ends (measured:
// the e4m3 long call 89.9 -> 89.0 us against 165 registers, no spills).
template <int D, bool KF8, bool VF8>
constexpr int kRegCap = Layout<D, KF8, VF8>::kQSplit ? 144 : 255;

// KF8 / VF8: prefix keys / values are e4m3 (tm_k / tm_v are 8-bit maps).
// NC > 1 (D = 128, bf16 values, at most 64 / NC query rows per pair):
// replicated rows.  The pair's rows are loaded NC times, copy c at MMA rows [c 64 / NC,
// (c + 1) 64 / NC), so that the softmax warps of copy c take only keys
// [c 64 / NC, (c + 1) 64 / NC) of each tile (32 / NC a thread instead of 32).
// The other keys of their P rows stay zero (the P buffers are cleared once),
// so P V accumulates each copy's own keys, and each copy keeps its own
// reference max, sums and O rows; at a segment end the copies are combined
// by log-sum-exp through shared memory.
template <int D, bool KF8, bool VF8, int NC>
__global__ void __launch_bounds__(Layout<D, KF8, VF8, NC>::kThreads, 1)
    __maxnreg__((kRegCap<D, KF8, VF8>)) rows_kernel(const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_kb,
                   const __grid_constant__ CUtensorMap tm_vb,
                   const __grid_constant__ CUtensorMap tm_q, const AttnParams p) {
    using Lt = Layout<D, KF8, VF8, NC>;
    constexpr bool REP = Lt::REP;
    constexpr int kStages = Lt::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(sm);
    const uint32_t bars = sbase + Lt::kBarOff;
    const uint32_t b_full = bars, b_empty = bars + 8 * kStages, b_qfull = b_empty + 8 * kStages,
                   b_qempty = b_qfull + 16, b_sready = b_qempty + 16,
                   b_sfree = b_sready + 8 * kSBufs, b_pready = b_sfree + 8 * kSBufs,
                   b_pvdone = b_pready + 16, b_drain = b_pvdone + 16,
                   b_cready = b_drain + 16, b_kfree = b_cready + 8 * Lt::kConvSlots,
                   b_vfree = b_kfree + 8 * Lt::kConvSlots,
                   b_qsplit = b_vfree + 8 * Lt::kConvSlots, b_bkfree = b_qsplit + 16;
    constexpr int kSlots = Lt::kConvSlots;
    constexpr bool kQSplit = Lt::kQSplit;
    int *qexp = reinterpret_cast<int *>(sm + Lt::kQeOff);  // [2][kRows]
    // where the MMAs read tile j's bf16 K and V (stage s = j % kStages): the
    // TMA tile in the stage, or the ring slot j % kSlots the conversion warps
    // widened it into
    const uint32_t kconv0 = sbase + Lt::kConvOff, vconv0 = kconv0 + (KF8 ? Lt::kTileBytes : 0);
    auto k_src = [&](int st, long long j) {
        return KF8 ? kconv0 + (int)(j % kSlots) * Lt::kConvBytes : sbase + st * Lt::kStageBytes;
    };
    auto v_src = [&](int st, long long j) {
        return VF8 ? vconv0 + (int)(j % kSlots) * Lt::kConvBytes
                   : sbase + st * Lt::kStageBytes + Lt::kKBytes;
    };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sm + Lt::kMiscOff);
    const uint32_t abort_flag = sbase + Lt::kMiscOff + 4;
    // a ring slot is written for tile j once the MMAs of tile j - kSlots that
    // read it have completed (kfree after S, vfree after P V).  Only the
    // conversion warps wait on kfree / vfree, and they wait for every tile in
    // order: a parity wait is exact only when the barrier is at most one phase
    // behind, which a thread that skipped tiles (the producer, which runs
    // kStages tiles ahead of P V) could not ensure.
    auto slot_free = [&](uint32_t bar, long long j) {
        return j < kSlots || wait(bar + 8 * (int)(j % kSlots),
                                  (uint32_t)(((j - kSlots) / kSlots) & 1), abort_flag, p.status);
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;


    // set-up that touches no global memory: it may overlap the previous
    // kernel in the stream (programmatic dependent launch)
    auto init_bars = [&]() {  // one thread
        for (int s = 0; s < kStages; ++s) {
            mbar_init(b_full + 8 * s, 1);
            mbar_init(b_empty + 8 * s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(b_qfull + 8 * i, 1);
            // kQSplit: the last S of the segment and every softmax warp, once
            // it has read its row's e (the next split overwrites it)
            mbar_init(b_qempty + 8 * i, kQSplit ? 1 + kSoftWarps : 1);
            mbar_init(b_pready + 8 * i, kSoftWarps);
            mbar_init(b_qsplit + 8 * i, kConvWarps);
        }
        mbar_init(b_bkfree, 1);
        for (int i = 0; i < kSBufs; ++i) {
            mbar_init(b_sready + 8 * i, 1);
            mbar_init(b_sfree + 8 * i, kSoftWarps);
        }
        mbar_init(b_pvdone, 1);
        mbar_init(b_pvdone + 8, 1);
        mbar_init(b_drain, 1);
        mbar_init(b_drain + 8, 1);
        if (Lt::kConv)
            for (int c = 0; c < kSlots; ++c) {
                mbar_init(b_cready + 8 * c, kConvWarps);
                mbar_init(b_kfree + 8 * c, 1);
                mbar_init(b_vfree + 8 * c, 1);
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
            "n"(kTmemCols));
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
    if (threadIdx.x < 64) {  // the row-sum MMA's B operand: row 0 of [8][64] twos
        const uint32_t two2 = threadIdx.x < 8 ? 0x40004000u : 0u;
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                         sbase + Lt::kTwosOff + threadIdx.x * 16),
                     "r"(two2)
                     : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (REP) {  // both P buffers start (and, outside each copy's keys, stay) zero
        for (int i = threadIdx.x; i < 2 * Lt::kPBytes / 16; i += Lt::kThreads)
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                             sbase + Lt::kPOff + i * 16),
                         "r"(0u)
                         : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kProducerWarp && elect_one()) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_v)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_q)) : "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    // The plan from the lengths as they read before the dependency wait;
    // after the wait they are read again and the plan is kept only if every
    // length is unchanged.
    long long lo = 0, hi = 0, ntiles = 0;
    Walk w0 = {0, 0, 0, 1, 0, 0};
    int sP = 0, sT = 0;
    if (spec) {
        sP = len_sm[lane0];
        sT = len_sm[32 + lane0];
        ntiles = plan(p, sP, sT, lo, hi, w0) ? hi - lo : 0;
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
            for (long long j = 0; j < ntiles && j < prefetch && wp.t < wp.nt - 1; ++j) {
                const int tok = wp.t * kTileKeys;
#pragma unroll
                for (int dp = 0; dp < (KF8 ? 1 : Lt::kPanels); ++dp)
                    tma_prefetch_5d(&tm_k, dp * 64, wp.h, tok, wp.b, p.key_slab);
#pragma unroll
                for (int dp = 0; dp < (VF8 ? 1 : Lt::kPanels); ++dp)
                    tma_prefetch_5d(&tm_v, dp * 64, wp.h, tok, wp.b, p.value_slab);
                ++wp.t;  // stays inside the pair: its last (block) tile ends the loop
            }
        }
    }

    // Producer state and one step of its loop (tile j of the range): the
    // first steps may run before the lengths are checked (below).
    Walk wl = w0;
    int qseg = -1;
    long long nblk = 0;           // (kQSplit) block tiles whose keys were issued
    long long issued = 0, j = 0;  // tiles whose loads were issued; next tile
    bool ok = true;
    uint64_t policy = 0;
    if (warp == kProducerWarp)
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    auto produce = [&]() {
        if (j == 0 || wl.t == 0) {  // the segment's query rows
            ++qseg;
            const int qb = qseg & 1;
            if (qseg >= 2)
                ok = ok && wait(b_qempty + 8 * qb, (uint32_t)(((qseg - 2) >> 1) & 1),
                                abort_flag, p.status);
            if (ok && elect_one()) {
                const uint32_t full = b_qfull + 8 * qb;
                const uint32_t dst = sbase + Lt::kQOff + qb * Lt::kQBytes;
                // (NC > 1) copy c at rows c 64 / NC
                mbar_arrive_expect_tx(full, NC * Lt::kPanels * p.rows_max * 128);
#pragma unroll
                for (int dp = 0; dp < Lt::kPanels; ++dp)
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        tma_4d(dst + dp * (kRows * 128) + c * (kRows / NC * 128), &tm_q, full,
                               dp * 64, wl.h * p.G, 0, wl.b);
            }
        }
        const int s = (int)(j % kStages);
        if (j >= kStages)
            ok = ok && wait(b_empty + 8 * s, (uint32_t)(((j - kStages) / kStages) & 1),
                            abort_flag, p.status);
        const bool blk = wl.t == wl.nt - 1;
        // (kQSplit) the block-key buffer is free once the S of the last block tile is done
        if (kQSplit && blk && nblk >= 1)
            ok = ok && wait(b_bkfree, (uint32_t)((nblk - 1) & 1), abort_flag, p.status);
        if (ok && elect_one()) {
            const uint32_t full = b_full + 8 * s;
            const uint32_t kdst = sbase + Lt::kStagesOff + s * Lt::kStageBytes;
            const uint32_t vdst = kdst + Lt::kKBytes;
            if (wl.t < wl.nt - 1) {
                const int tok = wl.t * kTileKeys;
                mbar_arrive_expect_tx(full, Lt::kStageBytes);
                // an e4m3 tile is one {D, 1, 64} box, a bf16 tile D / 64 swizzled panels
                if (KF8) {
                    tma_5d(kdst, &tm_k, full, 0, wl.h, tok, wl.b, p.key_slab, policy);
                } else {
#pragma unroll
                    for (int dp = 0; dp < Lt::kPanels; ++dp)
                        tma_5d(kdst + dp * 8192, &tm_k, full, dp * 64, wl.h, tok, wl.b,
                               p.key_slab, policy);
                }
                if (VF8) {
                    tma_5d(vdst, &tm_v, full, 0, wl.h, tok, wl.b, p.value_slab, policy);
                } else {
#pragma unroll
                    for (int dp = 0; dp < Lt::kPanels; ++dp)
                        tma_5d(vdst + dp * 8192, &tm_v, full, dp * 64, wl.h, tok, wl.b,
                               p.value_slab, policy);
                }
            } else if (kQSplit) {  // the block's own K (bf16) into its buffer, V into the stage
                mbar_arrive_expect_tx(full, 2 * Lt::kTileBytes);
#pragma unroll
                for (int dp = 0; dp < Lt::kPanels; ++dp) {
                    tma_4d(sbase + Lt::kBlkKOff + dp * 8192, &tm_kb, full, dp * 64, wl.h, 0,
                           wl.b);
                    tma_4d(vdst + dp * 8192, &tm_vb, full, dp * 64, wl.h, 0, wl.b);
                }
            } else {  // the block's own K / V (bf16): the operands read from the
                      // stage; ring-slot operands are loaded by the conversion warps
                mbar_arrive_expect_tx(full, (KF8 ? 0 : Lt::kTileBytes) +
                                                (VF8 ? 0 : Lt::kTileBytes));
#pragma unroll
                for (int dp = 0; dp < Lt::kPanels; ++dp) {
                    if (!KF8) tma_4d(kdst + dp * 8192, &tm_kb, full, dp * 64, wl.h, 0, wl.b);
                    if (!VF8) tma_4d(vdst + dp * 8192, &tm_vb, full, dp * 64, wl.h, 0, wl.b);
                }
            }
        }
        __syncwarp();
        if (ok && kQSplit && blk) ++nblk;
        if (ok) issued = j + 1;
        walk_next(p, wl);
        ++j;
    };

    // every input (and the workspace) may be written by the previous kernel
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the first loads of the speculative plan go out while the lengths are
    // checked (no step here waits: fresh stages and query buffers only)
    if (spec && warp == kProducerWarp)
        while (j < ntiles && j < kStages && ok && !((j == 0 || wl.t == 0) && qseg + 1 >= 2) &&
               !(kQSplit && wl.t == wl.nt - 1 && nblk >= 1))
            produce();
    {
        const int P1 = lane0 < p.B ? len_cg(p.prefix_len, lane0, p.capacity) : 0;
        const int T1 = lane0 < p.B ? len_cg(p.block_len, lane0, p.max_block) : 0;
        if (!(spec && __all_sync(kFull, P1 == sP && T1 == sT))) {  // the same in every warp
            if (spec) {  // loads issued under the stale plan land, then the barriers restart
                if (warp == kProducerWarp) {
                    for (long long t = 0; t < issued; ++t)
                        wait(b_full + 8 * (int)t, 0u, abort_flag, p.status);
                    for (int q = 0; q <= qseg; ++q) wait(b_qfull + 8 * q, 0u, abort_flag, p.status);
                }
                __syncthreads();
                if (threadIdx.x == 0) init_bars();
                __syncthreads();
            }
            lo = hi = 0;
            w0 = {0, 0, 0, 1, 0, 0};
            ntiles = plan(p, P1, T1, lo, hi, w0) ? hi - lo : 0;
            wl = w0;
            qseg = -1;
            nblk = 0;
            issued = j = 0;
            ok = true;
        }
    }

    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (int b = 0; b < p.B; ++b)
            if (p.prefix_len[b] != clamp_prefix(p, b) || p.block_len[b] != clamp_block(p, b))
                atomicOr(p.status, kStatusClamped);
    // an empty range (only when N < C) runs no loop below

    // the last loads each issuing thread started, for the abort path's drain
    long long drain_tiles = 0, drain_copy = -1;
    int drain_qseg = -1;
    if (warp == kProducerWarp) {
        // ================================ producer ===============================
        // Warp-uniform loop; one elected lane issues.  Stage s is reused once
        // the P V that read it has completed (the P V warp commits empty[s]);
        // a query buffer once the last S of the segment before last completed.
        while (j < ntiles && ok) produce();
        drain_tiles = issued;
        drain_qseg = qseg;
    } else if (warp == kMmaWarp || warp == kSWarp) {
        // ================================== MMA ==================================
        // Two issuing warps, each blocking on its own in-order stream: P V of
        // tile k once its P is in shared memory (pready), and S of tile kn once
        // its K has landed (or been widened), its segment's queries are in and
        // TMEM buffer kn % kSBufs has been read by the softmax warps (sfree).
        const uint32_t id_s = idesc(kRows, kTileKeys, 0, 0);
        const uint32_t id_pv = idesc(kRows, D, 0, 1);
        // descriptors are affine in the address: build each base once and add
        // (byte offset >> 4) for buffers and k-steps
        const uint64_t dq0 = sdesc(sbase + Lt::kQOff, 16, 1024, kSw128);
        const uint64_t dk0 = sdesc(k_src(0, 0), 16, 1024, kSw128);
        // (kQSplit) e4m3 operands: query parts hi / lo of buffer b at
        // kQ8Off + (2 b + part) kQ8Bytes, prefix keys in the stage, block keys (bf16)
        const uint32_t id_s8 = idesc_e4m3(kRows, kTileKeys);
        const uint64_t dq8 = sdesc(sbase + Lt::kQ8Off, 16, 1024, kSw128);
        const uint64_t dk8 = sdesc(sbase + Lt::kStagesOff, 16, 1024, kSw128);
        const uint64_t dkb = sdesc(sbase + Lt::kBlkKOff, 16, 1024, kSw128);
        const uint64_t dv0 = sdesc(v_src(0, 0), 8192, 1024, kSw128);
        const uint64_t dp0 = sdesc(sbase + Lt::kPOff, 16, 1024, kSw128);
        // rounded row sums: D[64][8] += P[64][64] twos[8][64]^T, column 0 = twice the sum of P
        const uint64_t d1 = sdesc(sbase + Lt::kTwosOff, 16, 1024, kSw128);
        const uint32_t id_l = idesc(kRows, 8, 0, 0);
        const uint32_t id_pv16 = idesc_f16(kRows, D, 0, 1), id_l16 = idesc_f16(kRows, 8, 0, 0);
        bool ok = true;
        if (warp == kSWarp) {
            Walk wsn = w0;
            int qseg = -1, qcur = 0;
            for (long long kn = 0; kn < ntiles && ok; ++kn) {
                if (kn == 0 || wsn.t == 0) {
                    ++qseg;
                    qcur = qseg & 1;
                    ok = ok && wait(b_qfull + 8 * qcur, (uint32_t)((qseg >> 1) & 1), abort_flag,
                                    p.status);
                    // (kQSplit) and split into its e4m3 parts
                    if (kQSplit)
                        ok = ok && wait(b_qsplit + 8 * qcur, (uint32_t)((qseg >> 1) & 1),
                                        abort_flag, p.status);
                }
                const int s = (int)(kn % kStages);
                // the tile's K and V: landed, and widened if stored as e4m3 (kQSplit:
                // the e4m3 keys are read as they are)
                if (Lt::kConv && !kQSplit)
                    ok = ok && wait(b_cready + 8 * (int)(kn % kSlots),
                                    (uint32_t)((kn / kSlots) & 1), abort_flag, p.status);
                else
                    ok = ok && wait(b_full + 8 * s, (uint32_t)((kn / kStages) & 1), abort_flag,
                                    p.status);
                if (kn >= kSBufs)
                    ok = ok && wait(b_sfree + 8 * (int)(kn % kSBufs),
                                    (uint32_t)(((kn - kSBufs) / kSBufs) & 1), abort_flag,
                                    p.status);
                if (!ok) break;
                const bool blk_tile = wsn.t == wsn.nt - 1;
                const bool seg_end = blk_tile || (kn + 1 == ntiles);
                fence_after();
                if (elect_one()) {
                    const uint32_t dS = tmem + (uint32_t)((kn % kSBufs) * kTileKeys);
                    if (kQSplit && !blk_tile) {
                        // S = hi K^T + lo K^T: 2 x 4 MMAs of 32 e4m3 elements (32 bytes)
                        const uint64_t ah = dq8 + (uint64_t)((2 * qcur * Lt::kQ8Bytes) >> 4);
                        const uint64_t al = ah + (uint64_t)(Lt::kQ8Bytes >> 4);
                        const uint64_t b0 = dk8 + (uint64_t)((s * Lt::kStageBytes) >> 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_f8(dS, ah + (uint64_t)(kk * 2), b0 + (uint64_t)(kk * 2), id_s8,
                                     kk > 0);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_f8(dS, al + (uint64_t)(kk * 2), b0 + (uint64_t)(kk * 2), id_s8,
                                     1u);
                    } else {
                        const uint64_t a0 = dq0 + (uint64_t)((qcur * Lt::kQBytes) >> 4);
                        const uint64_t b0 =
                            kQSplit ? dkb
                                    : dk0 + (uint64_t)((k_src(s, kn) - k_src(0, 0)) >> 4);
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            // panel kk / 4, then 16 elements (32 bytes) within the 128-byte row
                            const uint32_t qoff =
                                ((kk >> 2) * (kRows * 128) + (kk & 3) * 32) >> 4;
                            const uint32_t koff = ((kk >> 2) * 8192 + (kk & 3) * 32) >> 4;
                            mma(dS, a0 + qoff, b0 + koff, id_s, kk > 0);
                        }
                    }
                    mma_commit(b_sready + 8 * (int)(kn % kSBufs));
                    if (KF8 && !kQSplit) mma_commit(b_kfree + 8 * (int)(kn % kSlots));
                    if (kQSplit && blk_tile) mma_commit(b_bkfree);
                    if (seg_end) mma_commit(b_qempty + 8 * qcur);
                }
                __syncwarp();
                walk_next(p, wsn);
            }
        } else {
            Walk wm = w0;
            for (long long k = 0; k < ntiles && ok; ++k) {
                const bool first = (k == 0) || (wm.t == 0);
                ok = wait(b_pready + 8 * (int)(k & 1), (uint32_t)((k >> 1) & 1), abort_flag,
                          p.status);
                if (!ok) break;
                fence_after();
                if (elect_one()) {
                    const int s = (int)(k % kStages);
                    const uint64_t a0 = dp0 + (uint64_t)(((k & 1) * Lt::kPBytes) >> 4);
                    const uint64_t b0 = dv0 + (uint64_t)((v_src(s, k) - v_src(0, 0)) >> 4);
                    const uint32_t dO = tmem + kSBufs * kTileKeys;
                    const bool f16 = VF8 && wm.t < wm.nt - 1;  // widened values
#pragma unroll
                    for (int kk = 0; kk < kTileKeys / 16; ++kk)
                        mma(dO, a0 + (uint64_t)((kk * 32) >> 4),
                            b0 + (uint64_t)((kk * 2048) >> 4), f16 ? id_pv16 : id_pv,
                            (!first || kk > 0) ? 1u : 0u);
#pragma unroll
                    for (int kk = 0; kk < kTileKeys / 16; ++kk)
                        mma(dO + D, a0 + (uint64_t)((kk * 32) >> 4), d1 + (uint64_t)((kk * 32) >> 4),
                            f16 ? id_l16 : id_l, (!first || kk > 0) ? 1u : 0u);
                    mma_commit(b_pvdone + 8 * (int)(k & 1));
                    mma_commit(b_empty + 8 * s);
                    if (VF8) mma_commit(b_vfree + 8 * (int)(k % kSlots));
                }
                __syncwarp();
                walk_next(p, wm);
            }
        }
        // all MMAs this warp issued are complete before tensor memory is freed
        // (only a timed-out run can leave any in flight)
        const uint32_t drain = b_drain + (warp == kSWarp ? 8 : 0);
        if (elect_one()) mma_commit(drain);
        __syncwarp();
        const unsigned long long t0 = globaltimer();
        while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < kWaitNs) {
        }
    } else if (kQSplit && warp >= kConvWarp0) {
        // ========================== query split (kQSplit) ========================
        // Once a segment's bf16 query rows have landed, split them into their
        // e4m3 parts for the S MMAs and record each row's e for the softmax
        // warps (qsplit).  Query buffer b is loaded again only after the S of
        // its segment and every softmax warp's read of e are done (qempty),
        // so neither the parts nor e are overwritten early.
        const int ct = threadIdx.x - kConvWarp0 * 32;
        Walk wc = w0;
        int qs = -1;
        for (long long j = 0; j < ntiles; ++j) {
            if (j == 0 || wc.t == 0) {
                ++qs;
                const int qb = qs & 1;
                if (!wait(b_qfull + 8 * qb, (uint32_t)((qs >> 1) & 1), abort_flag, p.status))
                    break;
                const uint32_t q8 = sbase + Lt::kQ8Off + 2 * qb * Lt::kQ8Bytes;
                split_q(sbase + Lt::kQOff + qb * Lt::kQBytes, q8, q8 + Lt::kQ8Bytes,
                        qexp + qb * kRows, ct);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(b_qsplit + 8 * qb);
            }
            walk_next(p, wc);
        }
    } else if (Lt::kConv && warp >= kConvWarp0) {
        // ======================== e4m3 -> bf16 keys, f16 values ==================
        // Widen every prefix tile's e4m3 K (and V) into its ring slot once it
        // has landed and the slot is free, then hand the tile to the S warp
        // (cready).  A block tile's K (V) is bf16 already: for a ring operand
        // one elected lane of the first conversion warp loads it into the slot
        // with a copy that completes on cready itself.
        const int ct = threadIdx.x - kConvWarp0 * 32;
        Walk wc = w0;
        bool ok = true;
        for (long long j = 0; j < ntiles && ok; ++j) {
            const int s = (int)(j % kStages);
            const uint32_t cready = b_cready + 8 * (int)(j % kSlots);
            ok = wait(b_full + 8 * s, (uint32_t)((j / kStages) & 1), abort_flag, p.status);
            if (!ok) break;
            if (wc.t == wc.nt - 1) {
                if (KF8) ok = slot_free(b_kfree, j);
                if (VF8) ok = ok && slot_free(b_vfree, j);
                if (!ok) break;
                if (warp == kConvWarp0) {
                    if (elect_one()) {
                        mbar_arrive_expect_tx(cready, ((KF8 ? 1 : 0) + (VF8 ? 1 : 0)) *
                                                          Lt::kTileBytes);
#pragma unroll
                        for (int dp = 0; dp < Lt::kPanels; ++dp) {
                            if (KF8)
                                tma_4d(k_src(s, j) + dp * 8192, &tm_kb, cready, dp * 64, wc.h, 0,
                                       wc.b);
                            if (VF8)
                                tma_4d(v_src(s, j) + dp * 8192, &tm_vb, cready, dp * 64, wc.h, 0,
                                       wc.b);
                        }
                    }
                    drain_copy = j;
                } else if (lane == 0) {
                    mbar_arrive(cready);
                }
                __syncwarp();
                walk_next(p, wc);
                continue;
            }
            if (KF8) {
                ok = slot_free(b_kfree, j);
                if (!ok) break;
                widen_tile<D>(sbase + s * Lt::kStageBytes, k_src(s, j), ct);
            }
            if (VF8) {
                ok = slot_free(b_vfree, j);
                if (!ok) break;
                widen_f16<D>(sbase + s * Lt::kStageBytes + Lt::kKBytes, v_src(s, j), kTileKeys, ct);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(cready);
            walk_next(p, wc);
        }
    } else {
        // ================================ softmax ================================
        // thread (warp, lane) handles row 16 warp + lane % 16, keys of its half
        // (lane / 16) of each tile; the epilogue's O rows are read by lanes < 16
        const int row = warp * 16 + (lane & 15);
        // (REP) MMA row c 64 / NC + r holds copy c of query row r: warp w
        // holds rows of copy cp = w / (4 / NC)
        constexpr int kRowsPerCopy = kRows / NC;
        const int cp = REP ? warp / (4 / NC) : 0;
        const int qrow = REP ? row - cp * kRowsPerCopy : row;
        const int half = lane >> 4;
        // scores a thread takes per tile, and the first of them
        constexpr int kVals = 32 / NC;
        const int key0 = cp * (kTileKeys / NC) + kVals * half;
        const bool owner = lane < 16;
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        Walk ws = w0;
        // l_sum: sum of the fp32 weights 2^(s - m), for the lse.  The sum of
        // the same weights as rounded to bf16 for the P V product, used for
        // the normalisation so that O / l is an exact convex combination of
        // the values (the rounding of P then moves the output by a fraction
        // of the values' spread around it, not of the values themselves), is
        // accumulated by the tensor core next to O (P times a ones column,
        // fp32), which takes its tree of adds off the softmax warps.
        float m_ref = -INFINITY, l_sum = 0.f;
        int rows_active = 0, irow = 0;
        long long seg_first = lo;
        // (kQSplit) scale of the prefix tiles' scores: S holds 2^e q.k for this row
        float row_scale = p.scale_log2;
        int qs = -1;
        for (long long k = 0; k < ntiles; ++k) {
            const bool first = (k == 0) || (ws.t == 0);
            const bool block_tile = ws.t == ws.nt - 1;
            const bool last = block_tile || (k + 1 == ntiles);
            if (first) {
                m_ref = -INFINITY;
                l_sum = 0.f;
                rows_active = p.G * ws.T;
                irow = qrow / p.G;
                seg_first = lo + k;
                if (kQSplit) {
                    ++qs;
                    const int qb = qs & 1;
                    wait(b_qsplit + 8 * qb, (uint32_t)((qs >> 1) & 1), abort_flag, p.status);
                    const int e = qexp[qb * kRows + row];
                    row_scale = e == kNotFinite
                                    ? __uint_as_float(0x7fc00000u)
                                    : p.scale_log2 * __uint_as_float((uint32_t)(127 - e) << 23);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(b_qempty + 8 * qb);
                }
            }
            const int nvalid = block_tile ? ws.T : min(kTileKeys, ws.P - ws.t * kTileKeys);
            const int s = (int)(k % kStages);
            // ---- scores of tile k ----
            const bool ok_s = wait(b_sready + 8 * (int)(k % kSBufs),
                                   (uint32_t)((k / kSBufs) & 1), abort_flag, p.status);
            fence_after();
            const uint32_t s_addr = tmem + lane_base + (uint32_t)((k % kSBufs) * kTileKeys) +
                                    (uint32_t)(cp * (kTileKeys / NC));
            const bool valid_row = qrow < rows_active && ok_s;
            // keys j < lim are visible to this row; a full prefix tile needs no
            // mask (rows of other lanes are computed but never stored)
            const int lim = !valid_row ? 0 : (block_tile ? min(nvalid, irow + 1) : nvalid);
            const bool full_tile = !block_tile && nvalid == kTileKeys;
            const float scale = kQSplit && !block_tile ? row_scale : p.scale_log2;
            // The thread's 32 scores in registers (masked keys -> -inf); the
            // row's tile max decides the reference first: the segment's first
            // tile sets it, a later tile moves it (rescaling O and l) only when
            // its max is beyond the reference by more than 2^8.
            float v[kVals];
            if constexpr (kVals == 8)
                tmem_ld_half8(s_addr, v);
            else if constexpr (kVals == 16)
                tmem_ld_half16(s_addr, v);
            else
                tmem_ld_half32(s_addr, v);
            // the scores are in registers: S buffer k % kSBufs may take tile k + kSBufs
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_sfree + 8 * (int)(k % kSBufs));
            if (!full_tile) {
#pragma unroll
                for (int j = 0; j < kVals; j += 2) {
                    float a, b;
                    mul2(a, b, v[j], v[j + 1], scale, scale);
                    v[j] = key0 + j < lim ? a : -INFINITY;
                    v[j + 1] = key0 + j + 1 < lim ? b : -INFINITY;
                }
            }
            float mt;
            if constexpr (kVals == 8) {
                const float m = max3(max3(v[0], v[1], v[2]), max3(v[3], v[4], v[5]), fmaxf(v[6], v[7]));
                mt = full_tile ? m * scale : m;
            } else if constexpr (kVals == 16) {  // 16 -> 6 -> 2 -> 1
                const float m = fmaxf(max3(max3(v[0], v[1], v[2]), max3(v[3], v[4], v[5]),
                                           max3(v[6], v[7], v[8])),
                                      max3(max3(v[9], v[10], v[11]), max3(v[12], v[13], v[14]), v[15]));
                mt = full_tile ? m * scale : m;
            } else {  // three-input maxima: 32 -> 11 -> 4 -> 1
                float m11[11];
#pragma unroll
                for (int j = 0; j < 10; ++j) m11[j] = max3(v[3 * j], v[3 * j + 1], v[3 * j + 2]);
                m11[10] = fmaxf(v[30], v[31]);
                const float m = fmaxf(max3(max3(m11[0], m11[1], m11[2]), max3(m11[3], m11[4], m11[5]),
                                           max3(m11[6], m11[7], m11[8])),
                                      fmaxf(m11[9], m11[10]));
                mt = full_tile ? m * scale : m;
            }
            // (f16 weights) 2^kShiftF16 times what they would be: the reference is that much lower
            mt = fmaxf(mt, __shfl_xor_sync(kFull, mt, 16)) - (VF8 ? kShiftF16 : 0.f);
            if (first) {
                m_ref = mt;
            } else {
                const bool jump = valid_row && mt > m_ref + kRescaleLog2;
                if (__any_sync(kFull, jump)) {
                    // O is stable once P V of tile k-1 is done
                    wait(b_pvdone + 8 * (int)((k - 1) & 1), (uint32_t)(((k - 1) >> 1) & 1),
                         abort_flag, p.status);
                    fence_after();
                    const float alpha = jump ? ex2(m_ref - mt) : 1.f;  // m_ref -inf gives 0
                    if (jump) {
                        m_ref = mt;
                        l_sum *= alpha;
                    }
                    // O and, in the next 32 columns, the rounded row sum
#pragma unroll 1
                    for (int c = 0; c < D + 32; c += 32) {
                        float o[32];
                        const uint32_t ta = tmem + lane_base + (uint32_t)(kSBufs * kTileKeys + c);
                        tmem_ld32(ta, o);
#pragma unroll
                        for (int j = 0; j < 32; ++j) o[j] *= alpha;
                        tmem_st32(ta, o);
                    }
                }
            }
            // P = 2^(s - m) as bf16 into the swizzled P buffer (32 keys = 4
            // chunks): all exponentials first, then the packs (measured faster
            // than one loop that does both per pair); their tree sum for l
            // comes after P has been handed on
            const float mu = m_ref == -INFINITY ? 0.f : m_ref;
            if (full_tile) {
#pragma unroll
                for (int j = 0; j < kVals; j += 2)
                    fma2(v[j], v[j + 1], v[j], v[j + 1], scale, scale, -mu, -mu);
            } else {
#pragma unroll
                for (int j = 0; j < kVals; j += 2) add2(v[j], v[j + 1], v[j], v[j + 1], -mu, -mu);
            }
#pragma unroll
            for (int j = 0; j < kVals; ++j) v[j] = ex2(v[j]);
            uint32_t w[kVals / 2];
#pragma unroll
            for (int e = 0; e < kVals / 2; ++e)
                w[e] = VF8 && !block_tile ? pack_f16(v[2 * e], v[2 * e + 1])
                                          : pack_bf16(v[2 * e], v[2 * e + 1]);
            // P buffer (k & 1) is free once P V of tile k-2, its last reader, is done
            // (pvdone[k & 1] completes once per P V of tiles with that parity)
            if (k >= 2) wait(b_pvdone + 8 * (int)(k & 1), (uint32_t)(((k - 2) >> 1) & 1), abort_flag,
                             p.status);
            fence_after();
            const uint32_t pbuf = sbase + Lt::kPOff + (uint32_t)((k & 1) * Lt::kPBytes);
#pragma unroll
            for (int q4 = 0; q4 < kVals / 8; ++q4)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                 p_chunk_addr(pbuf, row, key0 / 8 + q4)),
                             "r"(w[4 * q4]), "r"(w[4 * q4 + 1]), "r"(w[4 * q4 + 2]),
                             "r"(w[4 * q4 + 3])
                             : "memory");
            // keys past the end of the tile may hold anything: zero their V rows
            if (nvalid < kTileKeys) {
                const uint32_t vt = v_src(s, k);
                const int nzero = (kTileKeys - nvalid) * 8 * Lt::kPanels;  // 16-byte chunks
                for (int i = threadIdx.x; i < nzero; i += kSoftWarps * 32) {
                    const int panel = i / ((kTileKeys - nvalid) * 8);
                    const int rem = i % ((kTileKeys - nvalid) * 8);
                    const int key = nvalid + rem / 8, chunk = rem % 8;
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(
                                     vt + panel * 8192 + key * 128 + (chunk << 4)),
                                 "r"(0u)
                                 : "memory");
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_pready + 8 * (int)(k & 1));
            if constexpr (kVals == 8) {
                l_sum += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
            } else if constexpr (kVals == 16) {
                float a0, a1, b0, b1;
                add2(a0, a1, v[0], v[1], v[8], v[9]);
                add2(b0, b1, v[2], v[3], v[10], v[11]);
                float c0, c1, d0, d1;
                add2(c0, c1, v[4], v[5], v[12], v[13]);
                add2(d0, d1, v[6], v[7], v[14], v[15]);
                add2(a0, a1, a0, a1, c0, c1);
                add2(b0, b1, b0, b1, d0, d1);
                add2(a0, a1, a0, a1, b0, b1);
                l_sum += a0 + a1;
            } else {  // the row sum is needed only for l: after P has been handed on
                // (packed adds, in the order of the tree t[j] += t[j + w])
                float t[16];
#pragma unroll
                for (int j = 0; j < 16; j += 2)
                    add2(t[j], t[j + 1], v[j], v[j + 1], v[j + 16], v[j + 17]);
#pragma unroll
                for (int wd = 8; wd > 1; wd >>= 1)
#pragma unroll
                    for (int j = 0; j < wd; j += 2)
                        add2(t[j], t[j + 1], t[j], t[j + 1], t[j + wd], t[j + wd + 1]);
                l_sum += t[0] + t[1];
            }

            // ---- end of segment: O / l and lse ----
            if (last) {
                wait(b_pvdone + 8 * (int)(k & 1), (uint32_t)((k >> 1) & 1), abort_flag, p.status);
                fence_after();
                const long long pair_first = lo + k - ws.t;
                const bool whole = (seg_first == pair_first) && block_tile;
                const int pair = ws.b * p.Hkv + ws.h;
                const size_t slot = (size_t)pair + blockIdx.x;
                const bool write = qrow < rows_active;
                // the row's sums: this thread's half plus its partner's; the
                // rounded one from the tensor core (column 0 of the row-sum
                // accumulator in the low half, column 1, zero, in the high one)
                const float l_row = l_sum + __shfl_xor_sync(kFull, l_sum, 16);
                float l_rnd;
                {
                    uint32_t r;
                    asm volatile(
                        "tcgen05.ld.sync.aligned.16x32bx2.x1.b32 {%0}, [%1], 1;\n"
                        "tcgen05.wait::ld.sync.aligned;"
                        : "=r"(r)
                        : "r"(tmem + lane_base + (uint32_t)(kSBufs * kTileKeys + D))
                        : "memory");
                    l_rnd = 0.5f * __uint_as_float(r);
                }
                const float l_row_rnd = l_rnd + __shfl_xor_sync(kFull, l_rnd, 16);
                const int gq = qrow % p.G;
                // this thread's columns: [64 g + 32 half, +32) for each 64-column group g
                float v[D / 2];
                tmem_ld_orow<D>(tmem + lane_base + (uint32_t)(kSBufs * kTileKeys), v);
                if constexpr (REP && Lt::kCompactXch) {
                    // The NC copies of each row through shared memory: the
                    // groups of its O row (not normalised) that the other
                    // copies combine, and its (m, l, rounded l); then thread
                    // (copy cp, row r, half) combines group cp of half `half`
                    // of query row r by log-sum-exp over the copies.
                    constexpr int kG = D / 2 / NC;  // values per group
                    constexpr int kXS = Lt::kXchStride;
                    float *xo = reinterpret_cast<float *>(sm + Lt::kXchOff);
                    float *xm = xo + 2 * kRows * kXS;
                    float *dst = xo + (half * kRows + row) * kXS;
#pragma unroll
                    for (int g = 0; g < NC; ++g) {
                        if (g == cp) continue;
                        const int slot = g < cp ? g : g - 1;
#pragma unroll
                        for (int j = 0; j < kG; j += 4)
                            *reinterpret_cast<float4 *>(dst + slot * kG + j) =
                                make_float4(v[g * kG + j], v[g * kG + j + 1], v[g * kG + j + 2],
                                            v[g * kG + j + 3]);
                    }
                    if (half == 0)
                        *reinterpret_cast<float4 *>(xm + row * 4) =
                            make_float4(m_ref, l_row, l_row_rnd, 0.f);
                    // this thread's own group, selected without a dynamic register index
                    constexpr int kDims = kG;
                    float own[kG];
#pragma unroll
                    for (int j = 0; j < kG; ++j) own[j] = v[j];
#pragma unroll
                    for (int g = 1; g < NC; ++g)
                        if (cp == g)
#pragma unroll
                            for (int j = 0; j < kG; ++j) own[j] = v[g * kG + j];
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                    // group cp's dims: values [0, 32) of a half are dims 32 half + i,
                    // values [32, 64) dims 64 + 32 half + i - 32
                    const int i0 = cp * kG;
                    const int d0 = i0 < 32 ? 32 * half + i0 : 64 + 32 * half + (i0 - 32);
                    float4 ml[NC];
                    float M = -INFINITY;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ml[c] = *reinterpret_cast<const float4 *>(xm + (c * kRowsPerCopy + qrow) * 4);
                        M = fmaxf(M, ml[c].x);
                    }
                    float L = 0.f, Lr = 0.f, o[kDims];
#pragma unroll
                    for (int j = 0; j < kDims; ++j) o[j] = 0.f;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        // a copy that saw no visible key has m = -inf and weight 0
                        const float sc = ml[c].x == -INFINITY ? 0.f : ex2(ml[c].x - M);
                        L += sc * ml[c].y;
                        Lr += sc * ml[c].z;
                        if (c == cp) {
#pragma unroll
                            for (int j = 0; j < kDims; ++j) o[j] += sc * own[j];
                        } else {
                            const float *src = xo + (half * kRows + c * kRowsPerCopy + qrow) * kXS +
                                               (cp < c ? cp : cp - 1) * kG;
#pragma unroll
                            for (int j = 0; j < kDims; j += 4) {
                                const float4 x = *reinterpret_cast<const float4 *>(src + j);
                                o[j] += sc * x.x;
                                o[j + 1] += sc * x.y;
                                o[j + 2] += sc * x.z;
                                o[j + 3] += sc * x.w;
                            }
                        }
                    }
                    const float inv = Lr > 0.f ? 1.f / Lr : 0.f;
                    const float lse = L == 0.f ? -INFINITY : (M + __log2f(L)) * kLn2;
                    if (write) {
                        if (whole) {
                            uint16_t *orow = p.out + (((size_t)ws.b * p.max_block + irow) * p.Hq +
                                                      (size_t)ws.h * p.G + gq) * D + d0;
#pragma unroll
                            for (int j = 0; j < kDims; j += 8)
                                *reinterpret_cast<uint4 *>(orow + j) =
                                    make_uint4(pack_bf16(o[j] * inv, o[j + 1] * inv),
                                               pack_bf16(o[j + 2] * inv, o[j + 3] * inv),
                                               pack_bf16(o[j + 4] * inv, o[j + 5] * inv),
                                               pack_bf16(o[j + 6] * inv, o[j + 7] * inv));
                        } else {
                            float *prow = p.part_o + (slot * p.rows_max + qrow) * D + d0;
#pragma unroll
                            for (int j = 0; j < kDims; j += 4)
                                *reinterpret_cast<float4 *>(prow + j) =
                                    make_float4(o[j] * inv, o[j + 1] * inv, o[j + 2] * inv,
                                                o[j + 3] * inv);
                        }
                        if (cp == 0 && half == 0) {
                            if (whole)
                                p.lse[((size_t)ws.b * p.Hq + (size_t)ws.h * p.G + gq) *
                                          p.max_block +
                                      irow] = lse;
                            else
                                p.part_lse[slot * p.rows_max + qrow] = lse;
                        }
                    }
                    // the exchange area is free again once every thread has read it
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                } else if constexpr (REP) {
                    // The NC copies of each row through shared memory: every
                    // copy's O row (not normalised) and its (m, l, rounded l);
                    // then thread (copy cp, row r, half) combines kDims dims of
                    // query row r, from kDims (2 cp + half), by log-sum-exp
                    // over the copies.
                    constexpr int kDims = kRowsPerCopy * D / 128;
                    float *xo = reinterpret_cast<float *>(sm + Lt::kXchOff);
                    float *xm = xo + kRows * Lt::kXchStride;
                    float *dst = xo + row * Lt::kXchStride + 32 * half;
#pragma unroll
                    for (int g = 0; g < D / 64; ++g)
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            *reinterpret_cast<float4 *>(dst + 64 * g + j) =
                                make_float4(v[32 * g + j], v[32 * g + j + 1], v[32 * g + j + 2],
                                            v[32 * g + j + 3]);
                    if (half == 0)
                        *reinterpret_cast<float4 *>(xm + row * 4) =
                            make_float4(m_ref, l_row, l_row_rnd, 0.f);
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                    const int d0 = kDims * (2 * cp + half);
                    float4 ml[NC];
                    float M = -INFINITY;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ml[c] = *reinterpret_cast<const float4 *>(xm + (c * kRowsPerCopy + qrow) * 4);
                        M = fmaxf(M, ml[c].x);
                    }
                    float L = 0.f, Lr = 0.f, o[kDims];
#pragma unroll
                    for (int j = 0; j < kDims; ++j) o[j] = 0.f;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        // a copy that saw no visible key has m = -inf and weight 0
                        const float sc = ml[c].x == -INFINITY ? 0.f : ex2(ml[c].x - M);
                        L += sc * ml[c].y;
                        Lr += sc * ml[c].z;
                        const float *src = xo + (c * kRowsPerCopy + qrow) * Lt::kXchStride + d0;
#pragma unroll
                        for (int j = 0; j < kDims; j += 4) {
                            const float4 x = *reinterpret_cast<const float4 *>(src + j);
                            o[j] += sc * x.x;
                            o[j + 1] += sc * x.y;
                            o[j + 2] += sc * x.z;
                            o[j + 3] += sc * x.w;
                        }
                    }
                    const float inv = Lr > 0.f ? 1.f / Lr : 0.f;
                    const float lse = L == 0.f ? -INFINITY : (M + __log2f(L)) * kLn2;
                    if (write) {
                        if (whole) {
                            uint16_t *orow = p.out + (((size_t)ws.b * p.max_block + irow) * p.Hq +
                                                      (size_t)ws.h * p.G + gq) * D + d0;
#pragma unroll
                            for (int j = 0; j < kDims; j += 8)
                                *reinterpret_cast<uint4 *>(orow + j) =
                                    make_uint4(pack_bf16(o[j] * inv, o[j + 1] * inv),
                                               pack_bf16(o[j + 2] * inv, o[j + 3] * inv),
                                               pack_bf16(o[j + 4] * inv, o[j + 5] * inv),
                                               pack_bf16(o[j + 6] * inv, o[j + 7] * inv));
                        } else {
                            float *prow = p.part_o + (slot * p.rows_max + qrow) * D + d0;
#pragma unroll
                            for (int j = 0; j < kDims; j += 4)
                                *reinterpret_cast<float4 *>(prow + j) =
                                    make_float4(o[j] * inv, o[j + 1] * inv, o[j + 2] * inv,
                                                o[j + 3] * inv);
                        }
                        if (cp == 0 && half == 0) {
                            if (whole)
                                p.lse[((size_t)ws.b * p.Hq + (size_t)ws.h * p.G + gq) *
                                          p.max_block +
                                      irow] = lse;
                            else
                                p.part_lse[slot * p.rows_max + qrow] = lse;
                        }
                    }
                    // the exchange area is free again once every thread has read it
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                } else {
                const float inv = l_row_rnd > 0.f ? 1.f / l_row_rnd : 0.f;
                const float lse = l_row == 0.f ? -INFINITY : (m_ref + __log2f(l_row)) * kLn2;
                if (write) {
                    uint16_t *orow = p.out + (((size_t)ws.b * p.max_block + irow) * p.Hq +
                                              (size_t)ws.h * p.G + gq) * D + 32 * half;
                    float *prow = p.part_o + (slot * p.rows_max + row) * D + 32 * half;
#pragma unroll
                    for (int g = 0; g < D / 64; ++g) {
                        const float *x = v + 32 * g;
                        if (whole) {
#pragma unroll
                            for (int j = 0; j < 32; j += 8)
                                *reinterpret_cast<uint4 *>(orow + 64 * g + j) =
                                    make_uint4(pack_bf16(x[j] * inv, x[j + 1] * inv),
                                               pack_bf16(x[j + 2] * inv, x[j + 3] * inv),
                                               pack_bf16(x[j + 4] * inv, x[j + 5] * inv),
                                               pack_bf16(x[j + 6] * inv, x[j + 7] * inv));
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; j += 4)
                                *reinterpret_cast<float4 *>(prow + 64 * g + j) =
                                    make_float4(x[j] * inv, x[j + 1] * inv, x[j + 2] * inv,
                                                x[j + 3] * inv);
                        }
                    }
                }
                if (write && owner) {
                    if (whole)
                        p.lse[((size_t)ws.b * p.Hq + (size_t)ws.h * p.G + gq) * p.max_block +
                              irow] = lse;
                    else
                        p.part_lse[slot * p.rows_max + row] = lse;
                }
                }  // REP
                if (whole) {  // rows past the block: 0 and lse -inf
                    for (int idx = threadIdx.x; idx < (p.rows_max - rows_active) * (D / 8);
                         idx += kSoftWarps * 32) {
                        const int r = rows_active + idx / (D / 8), col = (idx % (D / 8)) * 8;
                        const int ii = r / p.G, gg = r % p.G;
                        *reinterpret_cast<uint4 *>(p.out + (((size_t)ws.b * p.max_block + ii) *
                                                                 p.Hq +
                                                             (size_t)ws.h * p.G + gg) * D + col) =
                            make_uint4(0u, 0u, 0u, 0u);
                        if (col == 0)
                            p.lse[((size_t)ws.b * p.Hq + (size_t)ws.h * p.G + gg) * p.max_block +
                                  ii] = -INFINITY;
                    }
                }
                fence_before();
            }
            walk_next(p, ws);
        }
    }
    // every MMA was waited on by the control lane and the softmax warps
    fence_before();
    __syncthreads();
    fence_after();
    if (lds(abort_flag) != 0.f) {  // a wait gave up: copies still in flight land before exit
        if (warp == kProducerWarp && elect_one()) {
            for (long long j = drain_tiles - 1; j >= 0 && j >= drain_tiles - kStages; --j)
                drain_wait(b_full + 8 * (int)(j % kStages), (uint32_t)((j / kStages) & 1));
            for (int q = drain_qseg; q >= 0 && q >= drain_qseg - 1; --q)
                drain_wait(b_qfull + 8 * (q & 1), (uint32_t)((q >> 1) & 1));
        }
        if (Lt::kConv && warp == kConvWarp0 && lane == 0 && drain_copy >= 0)
            drain_wait(b_cready + 8 * (int)(drain_copy % kSlots),
                       (uint32_t)((drain_copy / kSlots) & 1));
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "n"(kTmemCols));
}

template <int D, bool KF8, bool VF8, int NC = 1>
cudaError_t launch_rows(const AttnParams &p, const CUtensorMap &tk, const CUtensorMap &tv,
                        const CUtensorMap &tkb, const CUtensorMap &tvb, const CUtensorMap &tq,
                        cudaStream_t stream) {
    using Lt = Layout<D, KF8, VF8, NC>;
    constexpr int smem = Lt::kBytes;
    static std::atomic<bool> configured[64];  // the smem opt-in, once per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(rows_kernel<D, KF8, VF8, NC>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        // the split of the merge that runs beside it (an SM changes it only while idle:
        // 12.98 instead of 12.29 us for one call over 16 pairs of about 600 keys)
        e = cudaFuncSetAttribute(rows_kernel<D, KF8, VF8, NC>,
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
    return cudaLaunchKernelEx(&cfg, rows_kernel<D, KF8, VF8, NC>, tk, tv, tkb, tvb, tq, p);
}

}  // namespace
}  // namespace tc

cudaError_t rows_launch(const AttnParams &p, int head_dim, bool keys_e4m3, bool values_e4m3,
                        const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                        const CUtensorMap &tm_kb, const CUtensorMap &tm_vb,
                        const CUtensorMap &tm_q, cudaStream_t stream) {
#define DAS_ROWS(...) tc::launch_rows<__VA_ARGS__>(p, tm_k, tm_v, tm_kb, tm_vb, tm_q, stream)
    if (head_dim == 128) {
        if (values_e4m3)
            return keys_e4m3 ? DAS_ROWS(128, true, true) : DAS_ROWS(128, false, true);
        if (keys_e4m3)
            return p.rows_max <= 16   ? DAS_ROWS(128, true, false, 4)
                   : p.rows_max <= 32 ? DAS_ROWS(128, true, false, 2)
                                      : DAS_ROWS(128, true, false);
        return p.rows_max <= 16   ? DAS_ROWS(128, false, false, 4)
               : p.rows_max <= 32 ? DAS_ROWS(128, false, false, 2)
                                  : DAS_ROWS(128, false, false);
    }
    if (head_dim == 64) {
        if (keys_e4m3) return values_e4m3 ? DAS_ROWS(64, true, true) : DAS_ROWS(64, true, false);
        return values_e4m3 ? DAS_ROWS(64, false, true) : DAS_ROWS(64, false, false);
    }
#undef DAS_ROWS
    return cudaErrorInvalidValue;
}

}  // namespace das
