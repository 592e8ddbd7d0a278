// QuaRTZ attention, one decode step (Appendix D, Table 6: attention with
// heads x 128 dimensions on LZS-coded operands, groups of 8 / 16 / 32), for
// sm_103a.
//
// One query per (batch x head) row attends over the first L tokens of that
// head's key / value cache.  Query, keys and values are QuaRTZ-encoded per
// token (Eq. 1 + Eq. 2, 64-wide groups along the head dimension):
//     score_t = scale * sum_g s_q[g] s_k[t,g] P_g[t],
//     P_g[t]  = sum_{k in g} v_q[k] v_k[t,k]            (exact integers)
//     o       = sum_t softmax(score)_t * s_v[t,g] v_v[t,.]
// The step is HBM-bound: per token and head it reads 2 x (64 code bytes +
// 128/G_s FLAG bytes + 4 scale bytes) and does about 2 operations per cached
// element, so the kernel streams the caches once, split over enough CTAs to
// keep every SM's memory pipe busy (split-L with a combine pass):
//
//   attn_decode_kernel<G_s>: CTA (split, bh), 128 threads, tokens in tiles
//     of 128.  Keys: one token per thread; the integer group sums are dp4a
//     products of the query's decoded values (int8, |v| <= 112, computed
//     once per CTA) with the key codes placed in the high nibble of each
//     byte (16 c), shifted per subgroup by the key's FLAG — the paper's
//     accumulator-shift schedule (Section 4.4) on the key side, exact.
//     Softmax: running maximum and sum per CTA in the log2 domain; each key
//     thread then writes p_t s_v 2^FLAG for its token's value subgroups
//     (the FLAG added to the scale's exponent field).  Values: 8 threads per
//     token row (one 8-byte piece of 16 codes each) x 16 token slots; each
//     code becomes a float exactly through the 2^23 magic number, and
//     o += p_t s_v 2^FLAG c with paired f32x2 subtract and fused
//     multiply-add (two instructions per two codes).  The code tiles of
//     both caches (8 KB each per 128 tokens) stream through a 2-stage
//     shared-memory ring filled by cp.async (chunks XOR-swizzled against
//     bank conflicts) one tile ahead (more stages measured slower: fewer
//     CTAs fit an SM); FLAGs and scales of the next tile are loaded into the
//     registers of this one's once these are used, before the value phase
//     (loaded a whole tile ahead, the copies and the registers they hold cost
//     more: G_s = 8 70.7 -> 69.2 us, 16 64.1 -> 63.1, 64 62.8 -> 59.8, 32 x 16
//     heads, 4096 tokens).  Output per CTA: unnormalised o, running
//     max, running sum.
//     What bounds it: instruction issue as much as memory.  A 128-token tile
//     took 842 instructions a warp (32 x 16 heads, 4096 tokens, G_s = 16:
//     issue slots 67% busy, the half-rate ALU 63%, DRAM 56%), of which the
//     unpack and the multiply-adds of the values need some 300.  So the rest
//     is kept small: addresses are a base per CTA plus 32-bit offsets, a full
//     tile is copied without row checks, the FLAG form (bytes or nibbles) is a
//     template argument, and a key's FLAG shifts the 16-fold dot product,
//     which is divided by 16 once per 64-wide group.  With what the comments
//     below add, 72.7 -> 62.0 us there, 80.7 -> 67.6 at G_s = 8, 68.4 -> 61.7
//     at G_s = 32, 131 -> 112 with 64 x 16 heads.  Measured and not used:
//     independent warps without CTA barriers (+-3%); the tiles of all heads
//     cut into equal runs, one wave of CTAs (0-8% slower); the even key codes
//     biased in their low nibbles instead of shifted (1-3% slower).
//   attn_combine_kernel: one CTA per bh merges the splits, where
//     attn_decode_kernel does not do it itself (one split, or one wave of
//     CTAs with at most 8 splits a head).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>

#include "lzs_e4m3.cuh"
#include "ptx.cuh"
#include "quartz_internal.h"

namespace quartz {
namespace {

constexpr int kD = 128;              // head dimension
constexpr int kWords = kD / 8;       // 32-bit code words per token row
constexpr int kTile = 128;           // tokens per tile = threads per CTA
constexpr int kAttnThreads = 128;
constexpr int kPfStride = kTile + 2;           // s_pf row stride: conflict-free reads and writes
constexpr int kPartStride = kD + 4;  // o[128], m, l (+ pad) per split
constexpr int kMaxSplits = 64;
constexpr int kMaxCluster = 8;       // splits merged within a cluster (the portable size)
constexpr float kLog2e = 1.4426950408889634f;

struct AttnArgs {
    const uint32_t *q_codes;
    const uint8_t *q_flags;
    const __half *q_scales;
    const uint32_t *k_codes;
    const uint8_t *k_flags;
    const __half *k_scales;
    const uint32_t *v_codes;
    const uint8_t *v_flags;
    const __half *v_scales;
    int q_packed, k_packed, v_packed;
    int64_t L_max;
    int L, n_split, chunk;
    float scale_log2;  // softmax scale * log2(e)
    float *part;       // [BH][n_split][kPartStride]; null: the splits of a head are one cluster
    void *out;         // with part == null: [BH][kD] of out_type
    int out_type;
};

// The FLAG bytes (or nibbles) of one token row: S = 128 / G_s subgroups,
// stored at subgroup index row * S + j (one byte each, or two per byte).
template <int GS, typename Row>
__device__ __forceinline__ void load_row_flags(const uint8_t *flags, Row row, bool packed, uint32_t (&f)[4])
{
    constexpr int S = kD / GS;
    f[0] = f[1] = f[2] = f[3] = 0u;
    const int bytes = packed ? S / 2 : S;
    const uint8_t *p = flags + row * bytes;
    if (bytes == 16) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
    } else if (bytes == 8) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        f[0] = v.x, f[1] = v.y;
    } else if (bytes == 4) {
        f[0] = *reinterpret_cast<const uint32_t *>(p);
    } else if (bytes == 2) {
        f[0] = *reinterpret_cast<const uint16_t *>(p);
    } else {
        f[0] = *p;
    }
}

__device__ __forceinline__ int row_flag(const uint32_t (&f)[4], int j, bool packed)
{
    return packed ? static_cast<int>((f[j >> 3] >> (4 * (j & 7))) & 0xFu)
                  : static_cast<int>((f[j >> 2] >> (8 * (j & 3))) & 0xFFu);
}

template <typename Row>
__device__ __forceinline__ float2 load_scales2(const __half *scales, Row row)
{
    const uint32_t w = *reinterpret_cast<const uint32_t *>(scales + 2 * row);
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
}

// The float 2^23 + x for the byte x selected by `sel` (byte b of
// `biased_bytes` into byte 0, 0x4B above it: 0x4B0000xx = 2^23 + xx).
__device__ __forceinline__ float magic_float(uint32_t biased_bytes, uint32_t sel)
{
    return __int_as_float(prmt_b32(biased_bytes, 0x4B000000u, sel));
}

__device__ __forceinline__ uint4 lds_u4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// s v 2^F for a float s that is 0 or normal: the exponent field grows by F
// (exact; for s = 0 the result is a tiny normal, only ever multiplied by 0).
__device__ __forceinline__ float scale_pow2(float s, int F)
{
    return __int_as_float(__float_as_int(s) + (F << 23));
}

// (acc0, acc1) += p * (c0, 16 c1), where f0 = 2^23 + 8 + c0 and f1 = 2^23 + 16
// (8 + c1): one paired subtraction and one paired fused multiply-add.  The
// odd codes stay in their high nibbles, which saves a shift per 8 codes; their
// sums are 16-fold until the end (a power of two: the roundings are the same).
// 32 x 16 heads, 4096 tokens: G_s = 8 69.2 -> 67.5 us, 16 63.1 -> 62.0.
__device__ __forceinline__ void fma_codes2(float &acc0, float &acc1, float p, float f0, float f1)
{
    asm("{\n\t.reg .b64 f, m, c, pp, acc;\n\t"
        "mov.b64 f, {%2, %3};\n\t"
        "mov.b64 m, {%5, %6};\n\t"
        "add.rn.f32x2 c, f, m;\n\t"
        "mov.b64 pp, {%4, %4};\n\t"
        "mov.b64 acc, {%0, %1};\n\t"
        "fma.rn.f32x2 acc, pp, c, acc;\n\t"
        "mov.b64 {%0, %1}, acc;\n\t}"
        : "+f"(acc0), "+f"(acc1)
        : "f"(f0), "f"(f1), "f"(p), "f"(-8388616.0f), "f"(-8388736.0f));
}

// Asynchronous 16-byte global -> shared copies (cp.async, completion tracked
// per thread in commit groups; the wait is the hardware's own).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Shared-memory offset of 16-byte chunk c (0..3) of token row r in a code
// tile: rows of 64 bytes, chunks XOR-swizzled by (r / 2) % 4 so that eight
// consecutive rows reading the same chunk hit eight different bank groups.
__device__ __forceinline__ uint32_t tile_off(int r, int c) { return r * 64 + ((c ^ ((r >> 1) & 3)) << 4); }

// Cluster barrier (all threads of all CTAs; the hardware's own wait) and
// reads of another CTA's shared memory.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void store_out(void *out, int type, int64_t i, float v)
{
    if (type == QUARTZ_OUT_F16) static_cast<__half *>(out)[i] = __float2half_rn(v);
    else if (type == QUARTZ_OUT_BF16) static_cast<__nv_bfloat16 *>(out)[i] = __float2bfloat16_rn(v);
    else static_cast<float *>(out)[i] = v;
}

// The FLAGs and scales of one token row of the key and value caches.
struct RowSide {
    uint32_t kf[4], vf[4];
    float2 sk, sv;
};

// The four arrays at a CTA's first token (uniform addresses), so that a
// thread's loads need a 32-bit token offset only.
struct SideBase {
    const uint8_t *kf, *vf;
    const __half *ks, *vs;
};

// PACK: 0 = one FLAG byte per subgroup in both caches, 1 = 4-bit FLAGs in
// both, -1 = as the arguments say (the caches differ).
template <int GS, int PACK>
__device__ __forceinline__ void load_side(const AttnArgs &a, const SideBase &b, uint32_t t, bool valid, RowSide &r)
{
    if (valid) {
        load_row_flags<GS>(b.kf, t, PACK < 0 ? a.k_packed != 0 : PACK, r.kf);
        load_row_flags<GS>(b.vf, t, PACK < 0 ? a.v_packed != 0 : PACK, r.vf);
        r.sk = load_scales2(b.ks, t);
        r.sv = load_scales2(b.vs, t);
    } else {
        r.kf[0] = r.kf[1] = r.kf[2] = r.kf[3] = 0u;
        r.vf[0] = r.vf[1] = r.vf[2] = r.vf[3] = 0u;
        r.sk = r.sv = make_float2(0.f, 0.f);
    }
}

constexpr int kStages = 2;                     // code tiles in flight per CTA
constexpr int kTileBytes = kTile * kD / 2;     // 8 KB of codes per tile and cache
constexpr int kAttnDynSmem = kStages * 2 * kTileBytes;
// Value phase layout: each thread takes kValDims = 16 dimensions (one 8-byte
// piece of a token row's codes, 16 accumulators) of kTile / kSlots tokens.
// With 32 dimensions (a 16-byte chunk) the registers of G_s = 32 spilled at
// 6 CTAs per SM: 65.0 us against 62.4 (32 x 16 heads, 4096 tokens).
constexpr int kValDims = 16;
static_assert(kAttnThreads * (kValDims + 1) * 4 <= kAttnDynSmem, "slot reduction fits the code ring");

// Resident CTAs per SM the register allocation is bounded for: more warps
// cover the memory latency.  The shared memory of 6 CTAs fits and the kernel
// compiles to at most 80 registers from G_s = 16 on (3-4% faster than 5, and
// 5 8-10% faster than an unbounded build; G_s = 64 64.8 -> 63.5 us with 6);
// at G_s = 8 shared memory allows only 5.
template <int GS>
constexpr int attn_min_ctas() { return GS >= 16 ? 6 : 5; }

template <int GS, int PACK>
__global__ void __launch_bounds__(kAttnThreads, attn_min_ctas<GS>()) attn_decode_kernel(const __grid_constant__ AttnArgs a)
{
    griddep_wait();
    constexpr int S = kD / GS;            // subgroups per row
    constexpr int kWordsPerSub = GS / 8;  // code words per subgroup
    extern __shared__ __align__(128) uint8_t s_ring[];  // [kStages][K, V][kTileBytes]
    __shared__ float s_pf[S][kPfStride];  // p_t s_v 2^FLAG per value subgroup and token
    __shared__ __align__(16) uint32_t s_q[2 * kWords];  // the query's decoded values (even, odd codes)
    __shared__ float s_wmax[kAttnThreads / 32];
    __shared__ float s_wsum[kAttnThreads / 32];

    const int tid = threadIdx.x;
    const int split = blockIdx.x;
    const int64_t bh = blockIdx.y;
    const int t_begin = split * a.chunk;
    const int t_end = min(t_begin + a.chunk, a.L);
    const int n_tiles = (t_end - t_begin + kTile - 1) / kTile;
    const uint32_t ring = static_cast<uint32_t>(__cvta_generic_to_shared(s_ring));
    const bool k_packed = PACK < 0 ? a.k_packed != 0 : PACK, v_packed = PACK < 0 ? a.v_packed != 0 : PACK;
    const int n_tok = t_end - t_begin;
    const int64_t row0 = bh * a.L_max + t_begin;  // the CTA's first token in the caches
    const SideBase side = {a.k_flags + row0 * (k_packed ? S / 2 : S), a.v_flags + row0 * (v_packed ? S / 2 : S),
                           a.k_scales + 2 * row0, a.v_scales + 2 * row0};
    // this thread's chunks of a code tile: rows tid / 4 + 32 k, whose swizzle is the same for every k
    const uint8_t *kbytes = reinterpret_cast<const uint8_t *>(a.k_codes) + row0 * (kD / 2);
    const uint8_t *vbytes = reinterpret_cast<const uint8_t *>(a.v_codes) + row0 * (kD / 2);
    const uint32_t ring_dst = ring + tile_off(tid >> 2, tid & 3);

    // Copies of tile `it` (both caches) into stage it % kStages; every thread
    // commits one group per call, empty past the last tile.
    auto issue = [&](int it) {
        const int left = n_tok - it * kTile;  // tokens from this tile on
        const uint32_t kdst = ring_dst + (it % kStages) * 2 * kTileBytes;
        const uint32_t src = static_cast<uint32_t>(it) * kTileBytes + tid * 16;
        if (left >= kTile) {
#pragma unroll
            for (int k = 0; k < kTileBytes / 16 / kAttnThreads; ++k) {
                cp_async16(kdst + k * kAttnThreads * 16, kbytes + src + k * kAttnThreads * 16);
                cp_async16(kdst + kTileBytes + k * kAttnThreads * 16, vbytes + src + k * kAttnThreads * 16);
            }
        } else if (left > 0) {
#pragma unroll
            for (int k = 0; k < kTileBytes / 16 / kAttnThreads; ++k) {
                if ((tid >> 2) + k * (kAttnThreads / 4) < left) {
                    cp_async16(kdst + k * kAttnThreads * 16, kbytes + src + k * kAttnThreads * 16);
                    cp_async16(kdst + kTileBytes + k * kAttnThreads * 16, vbytes + src + k * kAttnThreads * 16);
                }
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int it = 0; it < kStages - 1; ++it) issue(it);

    // ---- the query's decoded values, as int8 (even codes, odd codes) -------
    // decoded once per CTA by the first 16 threads (one code word each)
    if (tid < kWords) {
        uint32_t f[4];
        load_row_flags<GS>(a.q_flags, bh, a.q_packed != 0, f);
        const uint32_t word = a.q_codes[bh * kWords + tid];
        const int F = row_flag(f, tid / kWordsPerSub, a.q_packed != 0);
        uint32_t e = 0u, o = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int c0 = static_cast<int>(word << (28 - 8 * b)) >> 28;  // code 2b
            const int c1 = static_cast<int>(word << (24 - 8 * b)) >> 28;  // code 2b + 1
            e |= (static_cast<uint32_t>(c0 * (1 << F)) & 0xFFu) << (8 * b);
            o |= (static_cast<uint32_t>(c1 * (1 << F)) & 0xFFu) << (8 * b);
        }
        s_q[tid] = e;
        s_q[kWords + tid] = o;
    }
    const float2 sq = load_scales2(a.q_scales, bh);
    RowSide cur;
    load_side<GS, PACK>(a, side, tid, tid < n_tok, cur);
    __syncthreads();
    const uint32_t sq_addr = static_cast<uint32_t>(__cvta_generic_to_shared(s_q));

    constexpr int kPieces = kD / kValDims;             // code pieces per token row
    constexpr int kSlots = kAttnThreads / kPieces;     // token slots
    constexpr int kWordsPerPiece = kValDims / 8;       // 32-bit code words per piece
    const int vc = tid % kPieces;   // value phase: code piece (dims kValDims vc ..)
    const int slot = tid / kPieces; // value phase: token slot
    // offsets in a code tile: the thread's key row, and its value piece of token `slot`
    // (the swizzle is the same for tokens slot + i kSlots)
    static_assert(kSlots % 8 == 0, "the swizzle repeats every 8 rows");
    uint32_t key_off[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) key_off[c] = tile_off(tid, c);
    const uint32_t val_off = tile_off(slot, vc >> 1) + 8 * (vc & 1);
    float acc[kValDims];
#pragma unroll
    for (int k = 0; k < kValDims; ++k) acc[k] = 0.f;
    float m_run = -INFINITY;  // running maximum (log2 domain)
    float l_thr = 0.f;        // this thread's share of the running sum

    for (int it = 0; it < n_tiles; ++it) {
        issue(it + kStages - 1);     // into the stage tile it - 1 used
        cp_async_wait<kStages - 1>();  // this thread's copies of tile `it` have landed
        __syncthreads();     // ... and everyone else's
        const uint32_t kst = ring + (it % kStages) * 2 * kTileBytes;
        const uint32_t vst = kst + kTileBytes;

        // ---- keys: one token per thread -----------------------------------
        const bool valid = it * kTile + tid < n_tok;
        float s2 = -INFINITY;
        if (valid) {
            uint32_t kw[kWords], qe[kWords], qo[kWords];  // the query words: broadcast shared loads
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 v = lds_u4(kst + key_off[c]);
                kw[4 * c] = v.x, kw[4 * c + 1] = v.y, kw[4 * c + 2] = v.z, kw[4 * c + 3] = v.w;
                const uint4 e = lds_u4(sq_addr + 16 * c);
                qe[4 * c] = e.x, qe[4 * c + 1] = e.y, qe[4 * c + 2] = e.z, qe[4 * c + 3] = e.w;
                const uint4 o = lds_u4(sq_addr + 4 * kWords + 16 * c);
                qo[4 * c] = o.x, qo[4 * c + 1] = o.y, qo[4 * c + 2] = o.z, qo[4 * c + 3] = o.w;
            }
            int P[2] = {0, 0};
#pragma unroll
            for (int j = 0; j < S; ++j) {
                int dot = 0;  // 16 x the code dot product of subgroup j
#pragma unroll
                for (int w = j * kWordsPerSub; w < (j + 1) * kWordsPerSub; ++w) {
                    dot = __dp4a(static_cast<int>(qe[w]), static_cast<int>((kw[w] << 4) & 0xF0F0F0F0u), dot);
                    dot = __dp4a(static_cast<int>(qo[w]), static_cast<int>(kw[w] & 0xF0F0F0F0u), dot);
                }
                // 16 x the group sum, in 27 bits (the shift of a negative sum as unsigned)
                P[(j * GS) / 64] += static_cast<int>(static_cast<uint32_t>(dot) << row_flag(cur.kf, j, k_packed));
            }
            const float sc = __fmul_rn(__fmul_rn(sq.x, cur.sk.x), static_cast<float>(P[0] >> 4)) +
                             __fmul_rn(__fmul_rn(sq.y, cur.sk.y), static_cast<float>(P[1] >> 4));
            s2 = sc * a.scale_log2;
        }

        // ---- softmax: tile maximum, rescale, weights ----------------------
        float wm = s2;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
        if ((tid & 31) == 0) s_wmax[tid >> 5] = wm;
        __syncthreads();
        float tmax = s_wmax[0];
#pragma unroll
        for (int w = 1; w < kAttnThreads / 32; ++w) tmax = fmaxf(tmax, s_wmax[w]);
        const float m_new = fmaxf(m_run, tmax);
        const float alpha = exp2f(m_run - m_new);  // 0 on the first tile
        const float p = valid ? exp2f(s2 - m_new) : 0.f;
        l_thr = l_thr * alpha + p;
#pragma unroll
        for (int j = 0; j < S; ++j)  // p_t s_v 2^FLAG of every value subgroup (0 past the end)
            s_pf[j][tid] = p * scale_pow2((j * GS) / 64 ? cur.sv.y : cur.sv.x, row_flag(cur.vf, j, v_packed));
        // FLAGs and scales of the next tile, while the values are processed
        const int t_next = (it + 1) * kTile + tid;
        load_side<GS, PACK>(a, side, static_cast<uint32_t>(t_next), t_next < n_tok, cur);
        if (m_new != m_run) {  // CTA-uniform: rescale only when the maximum grew
#pragma unroll
            for (int k = 0; k < kValDims; ++k) acc[k] *= alpha;
        }
        m_run = m_new;
        __syncthreads();

        // ---- values: o += p_t s_v 2^FLAG c_t -------------------------------
#pragma unroll
        for (int i = 0; i < kTile / kSlots; ++i) {
            const int ti = slot + i * kSlots;
            uint32_t words[kWordsPerPiece];
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(words[0]), "=r"(words[1])
                         : "r"(vst + val_off + i * kSlots * 64));
#pragma unroll
            for (int w = 0; w < kWordsPerPiece; ++w) {
                // word kWordsPerPiece vc + w of the row; its subgroup's factor (0 past the end)
                const int sub = (kWordsPerPiece * vc + w) / kWordsPerSub;
                const float pf = s_pf[sub][ti];
                const uint32_t ev = (words[w] & 0x0F0F0F0Fu) ^ 0x08080808u;         // codes 0, 2, 4, 6 as c + 8
                const uint32_t od = (words[w] & 0xF0F0F0F0u) ^ 0x80808080u;  // codes 1, 3, 5, 7 as 16 (c + 8)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    fma_codes2(acc[8 * w + 2 * b], acc[8 * w + 2 * b + 1], pf, magic_float(ev, 0x7440u | b),
                               magic_float(od, 0x7440u | b));
            }
        }
        __syncthreads();  // s_pf and this stage are rewritten later
    }
    cp_async_wait<0>();

    // ---- reduce over token slots, write this split's partial result -------
    // (the code ring is free now: thread (slot, vc) stores its kValDims sums
    // at (kPieces slot + vc) * (kValDims + 1), which keeps both the stores and
    // the column reads below free of bank conflicts)
    __syncthreads();
    float *s_red = reinterpret_cast<float *>(s_ring);
#pragma unroll
    for (int k = 0; k < kValDims; ++k) s_red[(slot * kPieces + vc) * (kValDims + 1) + k] = k & 1 ? acc[k] * 0.0625f : acc[k];
    float ws = l_thr;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
    if ((tid & 31) == 0) s_wsum[tid >> 5] = ws;
    __syncthreads();
    float od = 0.f;
#pragma unroll 8
    for (int sl = 0; sl < kSlots; ++sl)
        od += s_red[(sl * kPieces + tid / kValDims) * (kValDims + 1) + (tid % kValDims)];
    float l = 0.f;
#pragma unroll
    for (int w = 0; w < kAttnThreads / 32; ++w) l += s_wsum[w];
    if (a.part) {
        float *part = a.part + (bh * a.n_split + split) * kPartStride;
        part[tid] = od;
        if (tid == 0) {
            part[kD] = m_run;
            part[kD + 1] = l;
        }
        return;
    }

    // ---- one cluster per head: its first CTA merges the splits -------------
    // from the others' shared memory, with the combine kernel's arithmetic
    if (a.n_split == 1) {
        store_out(a.out, a.out_type, bh * kD + tid, od / l);
        return;
    }
    constexpr int kMergeAt = 24 * 1024;  // in the code ring, past the slot sums
    static_assert(kAttnThreads * (kValDims + 1) * 4 <= kMergeAt && kMergeAt + kPartStride * 4 <= kAttnDynSmem, "");
    float *mine = reinterpret_cast<float *>(s_ring + kMergeAt);
    mine[tid] = od;
    if (tid == 0) {
        mine[kD] = m_run;
        mine[kD + 1] = l;
    }
    cluster_arrive();
    cluster_wait();
    if (split == 0) {
        const uint32_t base = ring + kMergeAt;
        float m[kMaxCluster], ls[kMaxCluster], os[kMaxCluster];
        float M = -INFINITY;
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r)
            if (r < a.n_split) {
                const uint32_t p = mapa(base, r);
                m[r] = ld_cluster_f32(p + 4 * kD);
                ls[r] = ld_cluster_f32(p + 4 * (kD + 1));
                os[r] = ld_cluster_f32(p + 4 * tid);
            }
        cluster_arrive();
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r)
            if (r < a.n_split) M = fmaxf(M, m[r]);
        float num = 0.f, den = 0.f;
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r)
            if (r < a.n_split) {
                const float w = exp2f(m[r] - M);  // 0 for an empty split
                num = fmaf(w, os[r], num);
                den = fmaf(w, ls[r], den);
            }
        store_out(a.out, a.out_type, bh * kD + tid, num / den);
    } else {
        cluster_arrive();
    }
    cluster_wait();  // this CTA's shared memory stays until the first has read it
}

template <int OUT>
__global__ void __launch_bounds__(kD) attn_combine_kernel(const float *__restrict__ part, int n_split, void *out)
{
    griddep_wait();
    const int64_t bh = blockIdx.x;
    const int d = threadIdx.x;
    const float *p = part + bh * n_split * kPartStride;
    // The kernel is all latency.  Up to 8 splits: their values are loaded
    // together, not maxima first: 32 x 4 heads with 8 splits 19.6 -> 18.6 us
    // for the whole step, 32 x 16 heads with 4 splits 64.6 -> 64.1; 4 or 16
    // instead of 8 measured within 0.3 us at 4 splits, and 4 costs 0.7 at 8.
    constexpr int kCombine = 8;
    float num = 0.f, den = 0.f;
    if (n_split <= kCombine) {
        float m[kCombine], l[kCombine], o[kCombine];
        float M = -INFINITY;
#pragma unroll
        for (int s = 0; s < kCombine; ++s) {
            const bool in = s < n_split;
            m[s] = in ? p[s * kPartStride + kD] : -INFINITY;
            l[s] = in ? p[s * kPartStride + kD + 1] : 0.f;
            o[s] = in ? p[s * kPartStride + d] : 0.f;
        }
#pragma unroll
        for (int s = 0; s < kCombine; ++s) M = fmaxf(M, m[s]);
#pragma unroll
        for (int s = 0; s < kCombine; ++s)
            if (s < n_split) {
                const float w = exp2f(m[s] - M);  // 0 for an empty split
                num = fmaf(w, o[s], num);
                den = fmaf(w, l[s], den);
            }
    } else {
        // More (few heads): thread s loads split s's maximum and sum and
        // computes its weight once, and the outputs come kBatch splits at a
        // time, the first of them before the weights are known.  Same
        // arithmetic in the same order.  A loop over the splits in every
        // thread, its loads one after the other, cost more than the step: 3
        // heads, 8097 tokens (64 splits), G_s = 8 14.6 -> 7.1 us; 15 heads,
        // 7534 tokens (59 splits), G_s = 64 13.8 -> 9.2.
        constexpr int kBatch = 16;
        static_assert(kMaxSplits == 64 && kD >= kMaxSplits, "two maxima per lane, a thread per split");
        __shared__ float s_m[kMaxSplits], s_w[kMaxSplits], s_l[kMaxSplits];
        float o[kBatch];
        auto load_o = [&](int s0) {
#pragma unroll
            for (int s = 0; s < kBatch; ++s) o[s] = s0 + s < n_split ? p[(s0 + s) * kPartStride + d] : 0.f;
        };
        load_o(0);
        float2 ml = make_float2(-INFINITY, 0.f);
        if (d < n_split) ml = *reinterpret_cast<const float2 *>(p + d * kPartStride + kD);
        if (d < kMaxSplits) s_m[d] = ml.x, s_l[d] = ml.y;
        __syncthreads();
        float M = fmaxf(s_m[d & 31], s_m[32 + (d & 31)]);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, k));
        if (d < n_split) s_w[d] = exp2f(ml.x - M);  // 0 for an empty split
        __syncthreads();
        for (int s0 = 0; s0 < n_split; s0 += kBatch) {
            if (s0 > 0) load_o(s0);
#pragma unroll
            for (int s = 0; s < kBatch; ++s)
                if (s0 + s < n_split) {
                    num = fmaf(s_w[s0 + s], o[s], num);
                    den = fmaf(s_w[s0 + s], s_l[s0 + s], den);
                }
        }
    }
    store_out(out, OUT, bh * kD + d, num / den);
}

// Splits of the L axis per head: chunks of about kSplitTiles tiles (1024
// tokens), and at least as many CTAs as fit the GPU at once.  Measured on the
// Table 6 settings against 1, 2, 3, 6, 8 and 16 splits and a wave-count
// model, this was the best or within 2% everywhere.
constexpr int64_t kSplitTiles = 8;
int attn_splits(int64_t BH, int64_t L, int64_t slots, int *chunk)
{
    const int64_t tiles = (L + kTile - 1) / kTile;
    int64_t n = (tiles + kSplitTiles - 1) / kSplitTiles;
    const int64_t fill = (slots + BH - 1) / BH;
    if (n < fill) n = fill;
    if (n > tiles) n = tiles;
    if (n > kMaxSplits) n = kMaxSplits;
    const int64_t per = (tiles + n - 1) / n;  // tiles per split
    *chunk = static_cast<int>(per * kTile);
    return static_cast<int>((tiles + per - 1) / per);
}

template <int GS, int PACK>
cudaError_t launch_decode(int64_t BH, AttnArgs &a, cudaStream_t s)
{
    // resident CTAs per SM of this instance, looked up on first use (any
    // host thread; they all store the same value)
    static std::atomic<int> occ_cache{0};
    cudaError_t e = cudaFuncSetAttribute(attn_decode_kernel<GS, PACK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kAttnDynSmem);
    if (e != cudaSuccess) return e;
    int occ = occ_cache.load(std::memory_order_relaxed);
    if (occ == 0) {
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, attn_decode_kernel<GS, PACK>, kAttnThreads, kAttnDynSmem);
        if (e != cudaSuccess) return e;
        occ = n > 0 ? n : 1;
        occ_cache.store(occ, std::memory_order_relaxed);
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
    const int64_t slots = static_cast<int64_t>(sms) * occ;
    a.n_split = attn_splits(BH, a.L, slots, &a.chunk);
    const dim3 grid(static_cast<unsigned>(a.n_split), static_cast<unsigned>(BH));
    // One split: it writes the output.  Up to 8 splits and all CTAs resident
    // at once: the splits of a head are a cluster and its first CTA merges
    // them, which saves the combine launch (40 heads, 777 tokens: 12.0 -> 9.5
    // us; 32 x 4 heads, 4096 tokens, 8 splits, more than one wave: even).
    // With several waves of CTAs a cluster waits until all its places are
    // free, which costs more than the launch (64 x 16 heads, 4096 tokens, 4
    // splits: 115.5 -> 119.7 us).
    if (a.n_split == 1) {
        a.part = nullptr;
        launch_pdl(attn_decode_kernel<GS, PACK>, dim3(grid), dim3(kAttnThreads), kAttnDynSmem, s, a);
    } else if (a.n_split <= kMaxCluster && BH * a.n_split <= slots) {
        a.part = nullptr;
        launch_pdl_cluster(attn_decode_kernel<GS, PACK>, a.n_split, dim3(grid), dim3(kAttnThreads), kAttnDynSmem, s, a);
    } else {
        launch_pdl(attn_decode_kernel<GS, PACK>, dim3(grid), dim3(kAttnThreads), kAttnDynSmem, s, a);
    }
    return cudaGetLastError();
}

// The FLAG form as a template argument: read at run time it cost about five
// instructions per FLAG and token (both forms extracted, one selected).
// Caches that differ in it take the instance that reads it from the arguments.
template <int GS>
cudaError_t launch_decode(int64_t BH, AttnArgs &a, cudaStream_t s)
{
    if (a.k_packed != a.v_packed) return launch_decode<GS, -1>(BH, a, s);
    return a.k_packed ? launch_decode<GS, 1>(BH, a, s) : launch_decode<GS, 0>(BH, a, s);
}

}  // namespace

size_t attention_workspace_bytes(int64_t BH, int64_t L)
{
    const int64_t tiles = (L + kTile - 1) / kTile;
    const int64_t splits = tiles < kMaxSplits ? tiles : kMaxSplits;
    return static_cast<size_t>(BH * splits * kPartStride) * sizeof(float);
}

cudaError_t launch_attention_decode(const quartz_encoded_t *q, const quartz_encoded_t *k, const quartz_encoded_t *v,
                                    int64_t L_max, int64_t L, float scale, void *o, int o_type, void *workspace,
                                    cudaStream_t s)
{
    const int64_t BH = q->rows;
    if (BH == 0) return cudaSuccess;
    AttnArgs a;
    a.q_codes = reinterpret_cast<const uint32_t *>(q->codes);
    a.q_flags = q->flags;
    a.q_scales = reinterpret_cast<const __half *>(q->scales);
    a.k_codes = reinterpret_cast<const uint32_t *>(k->codes);
    a.k_flags = k->flags;
    a.k_scales = reinterpret_cast<const __half *>(k->scales);
    a.v_codes = reinterpret_cast<const uint32_t *>(v->codes);
    a.v_flags = v->flags;
    a.v_scales = reinterpret_cast<const __half *>(v->scales);
    a.q_packed = q->p.flag_bits == 4;
    a.k_packed = k->p.flag_bits == 4;
    a.v_packed = v->p.flag_bits == 4;
    a.L_max = L_max;
    a.L = static_cast<int>(L);
    a.scale_log2 = scale * kLog2e;
    a.part = static_cast<float *>(workspace);
    a.out = o;
    a.out_type = o_type;
    cudaError_t e;
    switch (q->p.group_s) {
        case 8: e = launch_decode<8>(BH, a, s); break;
        case 16: e = launch_decode<16>(BH, a, s); break;
        case 32: e = launch_decode<32>(BH, a, s); break;
        default: e = launch_decode<64>(BH, a, s); break;
    }
    if (e != cudaSuccess || !a.part) return e;
    const unsigned cb = static_cast<unsigned>(BH);
    if (o_type == QUARTZ_OUT_F16) launch_pdl(attn_combine_kernel<QUARTZ_OUT_F16>, dim3(cb), dim3(kD), 0, s, a.part, a.n_split, o);
    else if (o_type == QUARTZ_OUT_BF16) launch_pdl(attn_combine_kernel<QUARTZ_OUT_BF16>, dim3(cb), dim3(kD), 0, s, a.part, a.n_split, o);
    else launch_pdl(attn_combine_kernel<QUARTZ_OUT_F32>, dim3(cb), dim3(kD), 0, s, a.part, a.n_split, o);
    return cudaGetLastError();
}

}  // namespace quartz
