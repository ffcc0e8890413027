// das_tc.h -- what the attention kernels share: mbarrier, TMA and tcgen05
// wrappers, packed fp32 arithmetic, and the split of the tile list over the CTAs.
#pragma once

#include <cuda_bf16.h>

#include "das_internal.h"

namespace das {
namespace tc {
namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr unsigned long long kWaitNs = 2000000000ull;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kConvWarps = 4;        // query split, e4m3 -> f16 (e4m3 variants)
constexpr int kPrefetchTiles = 2;    // prefix tiles pulled into L2 before the dependency wait
constexpr int kLongRange = 80;       // ranges longer than this prefetch none (measured, us per
                                     // two calls, 2 tiles / 1 / none: verify, 108 tiles a range,
                                     // - / 169.3 / 169.4, long - / 166.0 / 165.8; decode, 14
                                     // tiles, 32.0 / - / 32.9)
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ float lds(uint32_t a) {
    float x;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
    return x;
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
    float4 x;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                 : "r"(a)
                 : "memory");
    return x;
}
__device__ __forceinline__ void sts(uint32_t a, float x) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}
// Bounded wait; false after 2 s or once another thread of the CTA gave up
// (abort: shared address of the CTA's flag, 0 until then).  Everything after the first
// try is out of line: the roles' code together is more than the nearest instruction
// cache holds, and eight tries in line at every wait made the warps fetch it again
// (us per step: two e4m3 calls of B8 ragged 87.1 -> 82.0, ragged B8 D64 58.2 -> 56.9;
// the short-range kernel: decode 65.6 -> 63.9, batched 235.5 -> 232.0, the draft, verify,
// accept and commit step of B2 90.1 -> 88.1).
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, uint32_t abort,
                                       int32_t *status) {
    unsigned long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it == 8 || (it & 63u) == 0) {
            if (lds(abort) != 0.f) return false;
            if (it == 8) t0 = globaltimer();
            if (globaltimer() - t0 > kWaitNs) {
                sts(abort, 1.f);
                atomicOr(status, kStatusWaitTimeout);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, uint32_t abort,
                                     int32_t *status) {
    if (mbar_try_wait(bar, parity)) return true;
    return wait_slow(bar, parity, abort, status);
}

// On the abort path only: wait (at most 20 ms, whatever the abort flag says)
// for a phase whose completion also means that the copies signalling it
// have landed, so that no bulk copy into shared memory outlives the CTA.
__device__ __noinline__ void drain_wait(uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(bar, parity) && globaltimer() - t0 < 20000000ull) {
    }
}

__device__ __forceinline__ void tma_5d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0,
                                       int c1, int c2, int c3, int c4, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        ".L2::cache_hint [%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(c4), "l"(policy)
        : "memory");
}
// L2 prefetch of one box (no shared memory, no barrier).
__device__ __forceinline__ void tma_prefetch_5d(const CUtensorMap *map, int c0, int c1, int c2,
                                                int c3, int c4) {
    asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global.tile [%0, {%1, %2, %3, %4, %5}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
                 : "memory");
}
__device__ __forceinline__ void tma_prefetch_4d(const CUtensorMap *map, int c0, int c1, int c2,
                                                int c3) {
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0,
                                       int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// ---- tcgen05 ----------------------------------------------------------------
// Shared-memory matrix descriptor: start, leading / stride byte offsets,
// descriptor version 1, swizzle of the rows.  K-major: stride = 8 rows.
// MN-major: leading = from one span of swizzled columns to the next, stride =
// 8 rows along K.
constexpr uint64_t kSw128 = 2, kSw64 = 4, kSw32 = 6;
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint64_t sw) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)((lbo >> 4) & 0x3FFF) << 16 |
           (uint64_t)((sbo >> 4) & 0x3FFF) << 32 | (uint64_t)1 << 46 | sw << 61;
}
// Instruction descriptors of kind::f16: f16 (or bf16) A and B, fp32 D, majors, N, M.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, int a_mn_major, int b_mn_major) {
    return (1u << 4) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__host__ __device__ constexpr uint32_t idesc(int M, int N, int a_mn_major, int b_mn_major) {
    return idesc_f16(M, N, a_mn_major, b_mn_major) | (1u << 7) | (1u << 10);
}
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id,
                                    uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate)
        : "memory");
}
// The same with A in tensor memory (K-major).
__device__ __forceinline__ void mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t id,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(id), "r"(accumulate)
        : "memory");
}
// kind::f8f6f4 with e4m3 A and B (format code 0 for both; bit 7 makes A, bit 10 B
// e5m2), fp32 D, both K-major.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_f8(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}
__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// true on exactly one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n .reg .pred P;\n .reg .b32 R;\n elect.sync R|P, 0xffffffff;\n"
        " selp.u32 %0, 1, 0, P;\n}\n"
        : "=r"(pred));
    return pred != 0;
}
// 32 lanes x 32 consecutive 32-bit columns; thread t gets lane (base + t).
// The load and its wait form one statement, so no use of the registers can
// be scheduled before the data is there.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
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
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 8 columns of the calling thread's lane, all set to x
__device__ __forceinline__ void tmem_fill8(uint32_t taddr, uint32_t x) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};\n"
        "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
        "r"(x)
        : "memory");
}

// 1 / x to within an ulp of the division for x of 1 to 2^120 (0 for x = 0): one step
// r + r (1 - x r) of Newton's iteration for 1 / r - x = 0 from the hardware's
// approximation.  (The weights' sums it is for are 1 or more.  Rounded divisions, 32 in
// a row at a segment's end, took two e4m3 calls of B8 ragged from 81.5 to 87.7 us.)
__device__ __forceinline__ float inverse(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return x > 0.f ? fmaf(r, fmaf(-x, r, 1.f), r) : 0.f;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Packed fp32 arithmetic (two independent IEEE operations per instruction,
// bit for bit the scalar results) and the three-input maximum.
__device__ __forceinline__ void fma2(float &d0, float &d1, float a0, float a1, float b0, float b1,
                                     float c0, float c1) {
    asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
        " mov.b64 c, {%6, %7};\n fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void add2(float &d0, float &d1, float a0, float a1, float b0, float b1) {
    asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
        " add.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void mul2(float &d0, float &d1, float a0, float a1, float b0, float b1) {
    asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
        " mul.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// The maximum, NaN if either is (fmaxf drops it).
__device__ __forceinline__ float max_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Widen an e4m3 value tile [64 keys][D] (row-major, as the 8-bit TMA box
// lands) into the f16 tile the P V MMAs read: D / 64 panels of [64 keys][128
// bytes], 16-byte chunk j of key r at (j ^ (r % 8)) * 16 (128-byte swizzle).
// Every e4m3 value is exactly an f16 value, so one conversion per pair does
// it (bf16 takes four).  Keys from nvalid on (anything, NaN included) become
// zeros.  The 128 conversion threads (ct = 0..127) each take 16-element chunks.
template <int D>
__device__ __forceinline__ void widen_f16(uint32_t src, uint32_t dst, int nvalid, int ct) {
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
        uint32_t w[4];
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                     : "r"(src + key * D + pnl * 64 + jj * 16));
        const uint32_t row = dst + pnl * 8192 + key * 128;
        const bool keep = key < nvalid;
        uint32_t h[8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n cvt.rn.f16x2.e4m3x2 %0, l;\n"
                " cvt.rn.f16x2.e4m3x2 %1, h;\n}\n"
                : "=r"(h[2 * u]), "=r"(h[2 * u + 1])
                : "r"(keep ? w[u] : 0u));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                             row + (((2 * jj + u) ^ (key & 7)) << 4)),
                         "r"(h[4 * u]), "r"(h[4 * u + 1]), "r"(h[4 * u + 2]), "r"(h[4 * u + 3])
                         : "memory");
    }
}

// ---- tile list ----------------------------------------------------------------
__device__ __forceinline__ int clamp_prefix(const AttnParams &p, int b) {
    int v = p.prefix_len[b];
    return v < 0 ? 0 : (v > p.capacity ? p.capacity : v);
}
__device__ __forceinline__ int clamp_block(const AttnParams &p, int b) {
    int v = p.block_len[b];
    return v < 0 ? 0 : (v > p.max_block ? p.max_block : v);
}
__device__ __forceinline__ int tiles_of(int P) { return (P + kTileKeys - 1) / kTileKeys + 1; }

struct Walk {
    int b, h, t, nt, P, T;
};
__device__ __forceinline__ void walk_load_seq(const AttnParams &p, Walk &w) {
    if (w.b < p.B) {
        w.P = clamp_prefix(p, w.b);
        w.T = clamp_block(p, w.b);
        w.nt = tiles_of(w.P);
    }
}
__device__ __forceinline__ void walk_next(const AttnParams &p, Walk &w) {
    if (++w.t == w.nt) {
        w.t = 0;
        if (++w.h == p.Hkv) {
            w.h = 0;
            ++w.b;
            walk_load_seq(p, w);
        }
    }
}

// Extra weight of a pair's block tile when the list is split (p.block_weight,
// in tiles).  Ending one segment and starting the next (the wait for the last
// P V, the sums, the output or partial, the next queries) costs a CTA a time
// that does not depend on the tile's size, so the weight is the number of
// tiles that many bytes take: kBlockBytes over a tile's K and V bytes, 3 for
// 32 KB (D = 128, bf16), 6 for 16 KB.  A range that holds a block tile takes
// that many tiles fewer while there is at least one CTA per pair; with more
// pairs than CTAs nearly every range holds one and the weight would only move
// work around.  Weights 3 / 5 / 7 in the transposed kernel, us per two calls: ragged
// B8 D64 bf16 55.6 / 53.8 / 52.7, ragged B8 D128 e4m3 keys and values 84.1 / 82.3 /
// 83.4.  (das_rows.cu's kernel: 3, whatever the tile.)
constexpr int kBlockBytes = 3 * 32768;
constexpr int kCtasPerPairForWeight = 1;

// The split of the tile list: tile x of pair q has weighted position
// x + beta q; CTA c takes the tiles whose weighted position lies in
// [c W / C, (c+1) W / C).  beta = p.block_weight if there are at least
// kCtasPerPairForWeight CTAs per pair and W >= (2 + beta) C (which leaves no
// CTA empty: weighted positions are at most 1 + beta apart), else 0.
struct Split {
    long long N;  // tiles
    long long W;  // N + beta * pairs
    int beta;
};

// The split, given the total tile count.
__device__ __forceinline__ Split split_from_total(const AttnParams &p, long long total) {
    const long long pairs = (long long)p.B * p.Hkv;
    Split sp;
    sp.N = total;
    sp.beta = pairs * kCtasPerPairForWeight <= p.num_ctas &&
                      total + p.block_weight * pairs >= (long long)(2 + p.block_weight) * p.num_ctas
                  ? p.block_weight
                  : 0;
    sp.W = total + sp.beta * pairs;
    return sp;
}

// Clamped length read from L2 (not kept in L1, so that a value read before
// the dependency wait can never be served stale to a later load).
__device__ __forceinline__ int len_cg(const int32_t *a, int b, int cap) {
    const int v = __ldcg(a + b);
    return v < 0 ? 0 : (v > cap ? cap : v);
}

// Tiles of one pair of sequence b (0 past the batch); at most 2^25, so sums
// over 32 sequences fit in 32 bits.
__device__ __forceinline__ int seq_tiles(const AttnParams &p, int b) {
    return b < p.B ? tiles_of(clamp_prefix(p, b)) : 0;
}

__device__ Split split_of(const AttnParams &p) {  // whole warp
    const int lane = threadIdx.x & 31;
    long long total = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32)
        total += (long long)__reduce_add_sync(kFull, (unsigned)seq_tiles(p, b0 + lane)) * p.Hkv;
    return split_from_total(p, total);
}

// a / b for 0 <= a, 0 < b: a 32-bit division when both fit (the usual case;
// a 64-bit division is a long dependent instruction sequence).
__device__ __forceinline__ long long udiv(long long a, long long b) {
    if ((((unsigned long long)a | (unsigned long long)b) >> 32) == 0)
        return (long long)((uint32_t)a / (uint32_t)b);
    return a / b;
}

// The CTA whose weighted range holds weighted position q.
__device__ __forceinline__ int cta_of_w(long long q, const Split &sp, int C) {
    return (int)udiv((q + 1) * C - 1, sp.W);
}

// Range [lo, hi) of this CTA and the walk state of its first tile (a whole
// warp executes this).  One pass over the sequences: a 32-bit inclusive scan
// of the per-pair tile counts gives, for sequence b of a chunk, both the
// tiles and the weighted positions before it; the tiles at the weighted
// positions c W / C and (c+1) W / C are located in the same pass.
// P0 / T0: the clamped lengths of sequence `lane` (0 past the batch), given
// by the caller; with B <= 32 they are all the plan reads.
__device__ bool plan(const AttnParams &p, int P0, int T0, long long &lo, long long &hi, Walk &w) {
    const int lane = threadIdx.x & 31;
    const int nt0 = lane < p.B ? tiles_of(P0) : 0;
    const Split sp =
        p.B <= 32 ? split_from_total(p, (long long)__reduce_add_sync(kFull, (unsigned)nt0) * p.Hkv)
                  : split_of(p);
    const long long lw = udiv((long long)blockIdx.x * sp.W, p.num_ctas);
    const long long hw = udiv(((long long)blockIdx.x + 1) * sp.W, p.num_ctas);
    lo = hi = sp.N;
    bool have_lo = false;
    long long run_w = 0, run_t = 0;  // weighted positions / tiles before the chunk
    for (int b0 = 0; b0 < p.B; b0 += 32) {
        const int nt = b0 == 0 ? nt0 : seq_tiles(p, b0 + lane);
        int inc = nt;  // inclusive scan over the chunk
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int u = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += u;
        }
        const int nseq = min(32, p.B - b0);
        // weighted position after this lane's sequence
        const long long after_w =
            run_w + ((long long)inc + (long long)sp.beta * min(lane + 1, nseq)) * p.Hkv;
        // tile x at weighted position q, q inside sequence f of this chunk
        auto locate = [&](long long q, int f, Walk *wk) {
            const int ntf = __shfl_sync(kFull, nt, f);
            const int excl = __shfl_sync(kFull, inc, f) - ntf;
            const long long seq_w = run_w + ((long long)excl + (long long)sp.beta * f) * p.Hkv;
            const long long seq_t = run_t + (long long)excl * p.Hkv;
            const long long off = q - seq_w;
            int h = (int)udiv(off, ntf + sp.beta);
            int t = (int)(off - (long long)h * (ntf + sp.beta));
            if (t >= ntf) {  // inside a block tile's extra weight: the next pair
                t = 0;
                ++h;
            }
            if (wk) {
                wk->b = b0 + f;
                wk->h = h;
                wk->t = t;
                if (b0 == 0) {  // lengths already in registers
                    wk->P = __shfl_sync(kFull, P0, f);
                    wk->T = __shfl_sync(kFull, T0, f);
                    wk->nt = tiles_of(wk->P);
                } else {
                    walk_load_seq(p, *wk);
                }
                if (wk->h == p.Hkv) {
                    wk->h = 0;
                    ++wk->b;
                    walk_load_seq(p, *wk);
                }
            }
            return seq_t + (long long)h * ntf + t;
        };
        if (!have_lo) {
            const unsigned m = __ballot_sync(kFull, after_w > lw);
            if (m) {
                lo = locate(lw, __ffs(m) - 1, &w);
                have_lo = true;
            }
        }
        if (have_lo) {
            const unsigned m = __ballot_sync(kFull, after_w > hw);
            if (m) {
                hi = locate(hw, __ffs(m) - 1, nullptr);
                break;
            }
        }
        run_w += ((long long)__shfl_sync(kFull, inc, 31) + (long long)sp.beta * nseq) * p.Hkv;
        run_t += (long long)__shfl_sync(kFull, inc, 31) * p.Hkv;
    }
    return lo < hi;
}

}  // namespace
}  // namespace tc
}  // namespace das
