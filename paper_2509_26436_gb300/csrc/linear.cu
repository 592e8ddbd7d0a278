// QuaRTZ W4A4 linear layer for sm_103a (Section 4.4; Appendix C scales).
//
// Pipeline of one quartz_linear call:
//   1. expand: the packed 4-bit codes and per-subgroup FLAGs of both operands
//      are decoded to v = sgn(c)(|c| << FLAG) and written as FP8 E4M3 (exact:
//      every decoded value is |c| <= 7 times a power of two up to 2^4, i.e.
//      at most 3 significant bits and |v| <= 112, inside E4M3's 4-bit
//      significand and 448 range), together with the group scales
//      transposed to [G][rows] fp32 (and the zero-point terms to records in
//      the same order, see ZeroRec) for contiguous per-group access.  This
//      pass is HBM-bound and touches each operand element once, instead of
//      once per output tile that reads it.
//   2. GEMM: a persistent warp-specialised tcgen05 kernel.  One TMA warp
//      streams 128x64 A and 256x64 W tiles (one 64-wide quantization group
//      per stage, 64-byte swizzle) into a 5-stage shared-memory ring, with
//      each group's scales on the same barrier; one lane issues
//      kind::f8f6f4 MMAs into a fresh fp32 TMEM accumulator for every group
//      (double-buffered, 2 x 256 columns), so each accumulator holds exactly
//      P_g = sum_{k in g} v_a v_w; sixteen epilogue warps read P_g with
//      tcgen05.ld and fold it into the register-resident output as
//      y += s_a * (s_w * P_g) with packed f32x2 arithmetic.
//
// Exactness of P_g: the products v_a * v_w are integers of magnitude at most
// 112^2 = 12544 and every partial sum over a group is an integer of
// magnitude at most 64 * 12544 < 2^20, all exactly representable in the fp32
// accumulator, so the tensor-core sum equals the integer sum.  (sm_103a has
// no integer tcgen05 MMA kind; this is why the integer GEMM runs on the
// floating-point pipe.)
//
// 16-bit stage-1 codes (Section 5 LLM variant): decoded values reach
// 7 * 2^12 and are expanded to E5M2 instead (exact, see lzs_e4m3.cuh).
// Each product is still exact, but a group sum can need more than fp32's 24
// significant bits (products from 2^0 to 49 * 2^24), so P_g is the fp32
// tensor-core sum of exact products rather than the exact integer; the
// accumulator-shift GEMM below is the exact path for those operands.
#include <cuda.h>
#include <cuda_fp16.h>
#include <atomic>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "lzs_e4m3.cuh"
#include "ptx.cuh"
#include "quartz_internal.h"

namespace quartz {
namespace {

constexpr int kGroupQ = 64;

// ---------------------------------------------------------------------------
// 1. expand
// ---------------------------------------------------------------------------
// Row order of the expanded weight operand: inside every block of 16 rows,
// W row 4a + b is stored at position 4b + a (a 4x4 transposition; the map is
// its own inverse).  The GEMM's TMEM column j then holds output column
// perm16(j), which makes the four TMEM columns a thread reads with the
// 16x128b shape four consecutive output columns.
__host__ __device__ __forceinline__ int64_t perm16(int64_t r)
{
    return (r & ~int64_t(15)) | ((r & 3) << 2) | ((r >> 2) & 3);
}

// Zero-point terms of one row and group.  With u = 64 z_a - A_g (A_g, W_g: the
// gsum side values) the integer correction is P + z_w u - z_a W_g, the dot
// product of an activation record (hi u, lo u, -z_a, -z_a) and a weight
// record (z_w, z_w, hi W, lo W), hi x the multiple of 16 toward zero and lo x
// the rest: |u| <= 64 * 128 + 64 * 112 < 2^14 and |W| <= 64 * 112, so every
// entry is exact in fp16 and the tensor core adds the correction to P_g in
// its fp32 accumulator, all integers below 2^23, as a K = 16 step of which 4
// are used.  Against two more fused multiply-adds per output and group in the
// epilogue (GEMM, CUDA events): 18432 x 3072 x 3072 461 -> 277 us, 4001 x 3456
// x 1152 53.9 -> 37.5; results are the same bits.  Activation records are
// stored in row order, weight records in operand order (perm16), the order of
// the GEMM's accumulator.
struct ZeroRec {
    __half v[4];
};
static_assert(sizeof(ZeroRec) == 8, "two 4-byte planes hold the records");

__device__ __forceinline__ ZeroRec zero_rec(int z, int gsum, bool is_a)
{
    const int x = is_a ? kGroupQ * z - gsum : gsum;
    const int lo = x % 16;
    const __half hx = __int2half_rn(x - lo), lx = __int2half_rn(lo), hz = __int2half_rn(is_a ? -z : z);
    ZeroRec r;
    r.v[0] = is_a ? hx : hz;
    r.v[1] = is_a ? lx : hz;
    r.v[2] = is_a ? hz : hx;
    r.v[3] = is_a ? hz : lx;
    return r;
}

// (z_a, u) of an activation record, (z_w, W) of a weight record.
__device__ __forceinline__ float2 zero_terms(const ZeroRec &r, bool is_a)
{
    const float a = __half2float(r.v[0]), b = __half2float(r.v[1]), c = __half2float(r.v[2]), d = __half2float(r.v[3]);
    return is_a ? make_float2(-c, a + b) : make_float2(a, c + d);
}

// The records that follow the scale plane [G][rows_pad].
__host__ __device__ __forceinline__ const ZeroRec *zero_recs(const float *side, int64_t G, int64_t rows_pad)
{
    return reinterpret_cast<const ZeroRec *>(side + G * rows_pad);
}

// One launch prepares both GEMM operands (jobs selected by block index):
//   expand A, expand W: 16 codes per thread (8 bytes in, 16 E4M3 bytes out);
//     the weight operand is row-permuted (perm16) and zero-padded to a
//     multiple of 16 rows;
//   side A, side W: side[0][g][.] = s[r, g], weight rows in natural order,
//     activation rows at perm32(r); asymmetric adds a ZeroRec per row and
//     group (see there) in the space of two more such planes.  Rows in
//     [rows, rows_pad) are 0.  One thread per row and 8 groups: its reads stay
//     in L1 lines, consecutive threads write consecutive rows.
struct ExpandJob {
    const uint2 *codes;          // [rows, K/16] units of 16 codes
    const uint8_t *flags;        // [rows, K/G_s]
    uint4 *out;                  // [rows_out, K/16] units of 16 E4M3 values
    int64_t units, units_pad, units_per_row;
    int permute;
    int packed_flags;            // FLAGs two per byte
};
struct SideJob {
    const __half *scales;
    const int8_t *zeros;
    const int32_t *gsum;
    float *side;
    int64_t rows, rows_pad;
    int is_a;
};
struct PrepArgs {
    ExpandJob ex_a, ex_w;
    SideJob sd_a, sd_w;
    int64_t block_end[4];        // cumulative block counts: expand A, expand W, side A, side W
    int G, nside;
};
constexpr int kPrepThreads = 256;
constexpr int kSideGroupsPerThread = 8;

// kExpandPairs pairs of units per thread, a block apart (every load and
// store instruction of a warp is contiguous), one 16-byte code load per
// pair; all loads are issued before any decode so that several are in
// flight per thread (measured against 1, 4 and 8 single units and 1 and 4
// pairs per thread, and a grid-stride loop: 1.2-1.25x faster than 4 single
// units, the next best).
constexpr int kExpandPairs = 2;

template <int GS>
__device__ __forceinline__ void load_unit_flags(const ExpandJob &j, int64_t u, int &f0, int &f1)
{
    if (GS == 8) {
        if (j.packed_flags) {
            const uint32_t ff = j.flags[u];
            f0 = static_cast<int>(ff & 0xFu);
            f1 = static_cast<int>(ff >> 4);
        } else {
            const uint32_t ff = reinterpret_cast<const uint16_t *>(j.flags)[u];
            f0 = static_cast<int>(ff & 0xFFu);
            f1 = static_cast<int>(ff >> 8);
        }
    } else {
        f0 = f1 = load_flag(j.flags, (u * 16) / GS, j.packed_flags != 0);
    }
}

template <int GS, bool WIDE>
__device__ __forceinline__ void decode_unit(uint2 c, int f0, int f1, uint4 &o)
{
    if (WIDE) {
        e5m2_from_codes8(c.x, f0, o.x, o.y);
        e5m2_from_codes8(c.y, f1, o.z, o.w);
    } else {
        e4m3_from_codes8(c.x, f0, o.x, o.y);
        e4m3_from_codes8(c.y, f1, o.z, o.w);
    }
}

// kExpandPairs pairs of units per thread (one 16-byte code load per pair),
// a block apart; units and units_pad are multiples of 4 (K % 64 == 0), so a
// pair never straddles a row or the end.
template <int GS, bool WIDE>
__device__ __forceinline__ void run_expand(const ExpandJob &j, int64_t p0)
{
    uint4 c[kExpandPairs];
    int f[kExpandPairs][4];
#pragma unroll
    for (int q = 0; q < kExpandPairs; ++q) {
        const int64_t u = 2 * (p0 + q * kPrepThreads);
        c[q] = make_uint4(0u, 0u, 0u, 0u);
        f[q][0] = f[q][1] = f[q][2] = f[q][3] = 0;
        if (u < j.units) {
            c[q] = __ldcs(reinterpret_cast<const uint4 *>(j.codes) + (u >> 1));
            load_unit_flags<GS>(j, u, f[q][0], f[q][1]);
            load_unit_flags<GS>(j, u + 1, f[q][2], f[q][3]);
        }
    }
#pragma unroll
    for (int q = 0; q < kExpandPairs; ++q) {
        const int64_t u = 2 * (p0 + q * kPrepThreads);
        if (u >= j.units_pad) continue;
        int64_t dst = u;
        if (j.permute) {
            int64_t r;  // the row (32-bit division wherever the units fit)
            if (j.units_pad <= 0xFFFFFFFFll)
                r = static_cast<uint32_t>(u) / static_cast<uint32_t>(j.units_per_row);
            else
                r = u / j.units_per_row;
            dst = perm16(r) * j.units_per_row + (u - r * j.units_per_row);
        }
        uint4 o0 = make_uint4(0u, 0u, 0u, 0u), o1 = o0;  // padding rows stay zero
        if (u < j.units) {
            decode_unit<GS, WIDE>(make_uint2(c[q].x, c[q].y), f[q][0], f[q][1], o0);
            decode_unit<GS, WIDE>(make_uint2(c[q].z, c[q].w), f[q][2], f[q][3], o1);
        }
        j.out[dst] = o0;
        j.out[dst + 1] = o1;
    }
}

__device__ __forceinline__ void run_side(const SideJob &j, int64_t t, int G, int nside)
{
    const int64_t r = t % j.rows_pad;
    const int g0 = static_cast<int>(t / j.rows_pad) * kSideGroupsPerThread;
    if (g0 >= G) return;
    const int g1 = min(g0 + kSideGroupsPerThread, G);
    ZeroRec *recs = const_cast<ZeroRec *>(zero_recs(j.side, G, j.rows_pad));
    const int64_t o = j.is_a ? perm32(r) : r, oz = j.is_a ? r : perm16(r);
    const bool in = r < j.rows;
    for (int g = g0; g < g1; ++g) {
        const int64_t i = static_cast<int64_t>(g) * j.rows_pad + o;
        j.side[i] = in ? __half2float(j.scales[r * G + g]) : 0.f;
        if (nside > 1) {
            recs[static_cast<int64_t>(g) * j.rows_pad + oz] =
                in ? zero_rec(j.zeros[r * G + g], j.gsum[r * G + g], j.is_a != 0) : zero_rec(0, 0, j.is_a != 0);
        }
    }
}

template <int GS, bool WIDE>
__global__ void __launch_bounds__(kPrepThreads) prep_kernel(const __grid_constant__ PrepArgs args)
{
    griddep_wait();
    const int64_t bid = blockIdx.x;
    if (bid < args.block_end[0]) {
        run_expand<GS, WIDE>(args.ex_a, bid * (kPrepThreads * kExpandPairs) + threadIdx.x);
    } else if (bid < args.block_end[1]) {
        run_expand<GS, WIDE>(args.ex_w, (bid - args.block_end[0]) * (kPrepThreads * kExpandPairs) + threadIdx.x);
    } else if (bid < args.block_end[2]) {
        run_side(args.sd_a, (bid - args.block_end[1]) * kPrepThreads + threadIdx.x, args.G, args.nside);
    } else {
        run_side(args.sd_w, (bid - args.block_end[2]) * kPrepThreads + threadIdx.x, args.G, args.nside);
    }
}

// ---------------------------------------------------------------------------
// 2. tcgen05 GEMM
// ---------------------------------------------------------------------------
constexpr int BM = 128;
constexpr int BN = 256;
constexpr int BK = kGroupQ;
constexpr int kABytes = BM * BK;      // E4M3 operands: one byte per element
constexpr int kBBytes = BN * BK;
// Warpgroups 0-3 dequantise (16 warps: four per 32-lane TMEM quarter, 64
// columns each); warpgroup 4 holds the TMA producer, the MMA issuer, the
// zero-point record warp and an idle one.  The dequant epilogue is the throughput-critical part (two fp32
// operations per output element per group), so it gets four warps per
// scheduler; the control roles sit on two different schedulers (warp w runs
// on scheduler w % 4) because each slows the epilogue warps that share its
// scheduler.
//
// What bounds the kernel is the time each epilogue warp spends per group
// outside its arithmetic: TMEM and shared loads and the hand-off.  So a group
// costs an epilogue warp one barrier wait and one arrival (its scales ride on
// the operands' barrier, see Smem), waits branch on a warp vote
// (mbar_wait_warp) and the control warps run their loops converged with one
// elected lane issuing, which took an operand stage's issue from about 460 to
// 60 cycles.  Together, against single-lane control loops, per-lane waits and
// a scale ring with barriers of its own (CUDA events, GEMM + combine):
// 18432 x 12288 x 3072 1178 -> 1053 us, 8192 x 4608 x 1152 96.9 -> 86.7,
// 2048 x 4096 x 11008 (E5M2) 166.6 -> 150.2; per-row scales 18432 x 3072 x
// 3072 251 -> 181, asymmetric 548 -> 478.
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 4) * 32;
constexpr int kProducerWarp = kEpiWarps;
constexpr int kMmaWarp = kEpiWarps + 1;
constexpr int kRecWarp = kEpiWarps + 2;  // zero-point records (asymmetric)
constexpr int kRecDepth = 3;             // groups of record copies in flight (below the stage count)
constexpr int kColsPerWarp = BN / 4;
// Register split (setmaxnreg): 640 threads launch with 96 registers each;
// warpgroup 4 drops to 32 so the epilogue warpgroups can hold 112
// (512*112 + 128*32 = 61440 = 640*96).
constexpr uint32_t kRegsLaunch = 96;
constexpr uint32_t kRegsEpilogue = 112;
constexpr uint32_t kRegsControl = 32;
static_assert(kEpiWarps * 32 * kRegsEpilogue + 128 * kRegsControl <= kThreads * kRegsLaunch,
              "register split exceeds the launch allocation");
constexpr uint32_t kTmemCols = 512;   // two fp32 accumulators of 256 columns
constexpr int kRasterM = 8;  // tiles are visited in bands of 8 M-tiles
constexpr int kRowRasterMaxN = 16;  // see tile_coords
// Per-row scales (group_q = K): the MMA accumulates kPerRowChunk stages (256
// of K) into one TMEM accumulator before the epilogue takes it; each such sum
// is an integer below 256 * 112^2 < 2^22, exact in fp32 and convertible with
// the 1.5 * 2^23 rounding addend, and the epilogue adds it to an int32.
constexpr int kPerRowChunk = 4;

struct GemmArgs {
    const float *a_side;  // scales [G][m_pad], then (asymmetric) the ZeroRecs [G][m_pad]
    const float *w_side;  // scales [G][n_pad], then (asymmetric) the ZeroRecs [G][n_pad]
    int64_t m_pad, n_pad;
    int M, N, G;
    int tiles_m, tiles_n, num_tiles;
    int raster_m;         // M-tiles per band of the visiting order: kRasterM or 1 (see tile_coords)
    const __half *bias;
    void *y;
    int y_type;
    int32_t *partials;
    int partials_group;
    int *dev_err;
    int per_row;          // scales per row (group_q = K) rather than per 64-group
    int wide;             // E5M2 operands (16-bit stage-1 codes) instead of E4M3
    // Split last wave: the first full_tiles tiles go round robin over the CTAs
    // (the same count each); each of the remaining tail_tiles is cut along K
    // into `split` group ranges taken by CTAs 0 .. tail_tiles * split - 1,
    // which leave partial tiles in tail_part (fp32 sums, or int32 sums with
    // scales per row); tail_combine_kernel adds them in part order and writes
    // the outputs.  Range forms (ls > 0): the
    // last tail_tiles tiles' tail_tiles * G group iterations (after at least
    // one wave of whole tiles, or every tile's when more than half but not
    // all of the SMs hold one) are cut into one contiguous range of ls per
    // CTA, one CTA per SM; a tile met by r ranges leaves parts 0 .. r - 1 in
    // group order (r <= 2 after whole tiles, where ls >= G; r <= 3 otherwise,
    // where ls >= G / 2), a tile inside one range is stored whole.
    int full_tiles, tail_tiles, split;
    int ls;
    float *tail_part;     // [tail_tiles][split][16][kEpiWarps * 32] of four 32-bit words (fp32, or int32 per row)
};

// Shared memory: the operand stages, the output blocks (one per epilogue warp,
// see TileOut), then a ring of scale slots (one group's BM activation and BN
// weight scales each), then the mbarriers.  5 stages (4 with zero points)
// cover the copy latency (a group takes 350 cycles or more; 4, 6 and 8
// measured no better).  A group's scales are copied with its operands and
// counted on the same barrier.  A slot needs no barrier of its own to be reused: the
// producer writes group i + kSideSlots once the MMA of group i + kSideSlots -
// kStages is done, which was issued after the epilogue had released group
// i + kSideSlots - kStages - 2, a group after i.
//
// With zero points (ZERO) a stage also holds its group's records as rows of 16
// bytes, the upper halves zero, 128 of activations and 256 of weights, and a
// zero block stands for the second 16 bytes of K of both.
constexpr int kOutBlockBytes = 32 * 128;  // 32 rows of 64 two-byte outputs
constexpr int kRecRow = 16;
constexpr int kRecBytes = (BM + BN) * kRecRow;
template <bool ZERO, bool STAGED>
struct Smem {
    static constexpr int kStages = ZERO ? 4 : 5;
    static constexpr int kSideSlots = ZERO ? 8 : 16;
    static constexpr int kStageBytes = kABytes + kBBytes + (ZERO ? kRecBytes : 0);
    static constexpr int kRecA = kABytes + kBBytes, kRecW = kRecA + BM * kRecRow;  // in a stage
    static_assert(kSideSlots >= kStages + 3, "a slot is rewritten only after its group's epilogue");
    static constexpr int kOperands = 0;
    static constexpr int kOut = kStages * kStageBytes;
    static constexpr int kSide = kOut + (STAGED ? kEpiWarps * kOutBlockBytes : 0);
    static constexpr int kSideABytes = BM * 4;
    static constexpr int kSideSlotBytes = (BM + BN) * 4;
    static constexpr int kZeros = kSide + kSideSlots * kSideSlotBytes;
    static constexpr int kZeroBytes = ZERO ? BN * kRecRow : 0;
    static constexpr int kBars = kZeros + kZeroBytes;
    // full, empty, acc_full x2, acc_empty x2, drain
    static constexpr int kNumBars = 2 * kStages + 4 + 1;
    static constexpr int kMisc = kBars + kNumBars * 8;
    static constexpr int kTotal = kMisc + 16;
    static constexpr int kAlloc = kTotal + 1024;  // slack to align the base to 1024 bytes
};

// Tile visiting order: bands of RM M-tiles, N-tiles inside a band (M
// fastest), so the CTAs resident at one time share few A row-blocks and W
// column-blocks and both stay in L2.  RM is kRasterM, or 1 (whole rows of
// tiles, one M-tile after the other) for layers at most kRowRasterMaxN
// tiles wide on the symmetric fast path: there a band of 8 M-tiles holds
// fewer tiles than one wave of CTAs, so the waves would cut bands and read
// an A row-block again in the next wave (measured 2.3x A reads for a
// 12-tile-wide, 192-group layer), while a row keeps each A row-block's
// consumers in one wave and the whole narrow W stays in L2.  RM is a
// template argument of the GEMM (a runtime band size measured 1.4% slower
// on the wide layers); a.raster_m holds it for the combine kernel.
template <int RM>
__device__ __forceinline__ void tile_coords(int tile, const GemmArgs &a, int &mt, int &nt)
{
    const int band = tile / (RM * a.tiles_n);
    const int m0 = band * RM;
    const int gm = min(RM, a.tiles_m - m0);
    const int r = tile - band * RM * a.tiles_n;
    mt = m0 + r % gm;
    nt = r / gm;
}

// This CTA's work: whole tiles, then (split last wave) one part of a tail tile.
struct WorkItem {
    int tile, g0, g1;  // tile index and group range [g0, g1)
    int part, tail;    // part of tail tile `tail` (part = -1: a whole tile)
};

__device__ __forceinline__ int work_items(const GemmArgs &a)
{
    const int c = blockIdx.x, P = gridDim.x;
    if (a.split <= 1) return (a.num_tiles - c + P - 1) / P;
    if (a.ls > 0) {  // (tail_tiles * G < 2^30: checked on the host)
        const int nf = a.full_tiles / P;
        const int U = a.tail_tiles * a.G, b = c * a.ls, e = min(b + a.ls, U);
        if (b >= e) return nf;
        return nf + (e - 1) / a.G - b / a.G + 1;
    }
    return a.full_tiles / P + (c < a.tail_tiles * a.split ? 1 : 0);
}

__device__ __forceinline__ WorkItem work_item(const GemmArgs &a, int k)
{
    WorkItem w;
    const int c = blockIdx.x, P = gridDim.x;
    if (a.ls > 0 && k >= a.full_tiles / P) {
        const int U = a.tail_tiles * a.G, b = c * a.ls, e = min(b + a.ls, U);
        const int t = b / a.G + (k - a.full_tiles / P);
        const int t0 = t * a.G;
        w.tile = a.full_tiles + t;
        w.g0 = max(b - t0, 0);
        w.g1 = min(e - t0, a.G);
        if (w.g0 == 0 && w.g1 == a.G) {
            w.part = -1;
            w.tail = 0;
        } else {
            w.part = c - t0 / a.ls;  // ranges before this one that meet the tile
            w.tail = t;
        }
        return w;
    }
    if (a.split <= 1 || k < a.full_tiles / P) {
        w.tile = c + k * P;
        w.g0 = 0;
        w.g1 = a.G;
        w.part = -1;
        w.tail = 0;
    } else {
        w.tail = c / a.split;
        w.part = c - w.tail * a.split;
        w.tile = a.full_tiles + w.tail;
        w.g0 = w.part * a.G / a.split;
        w.g1 = (w.part + 1) * a.G / a.split;
    }
    return w;
}

// Both halves of an fp32 pair += b.
__device__ __forceinline__ void add_to_pair(uint64_t &a, float b)
{
    const float lo = __fadd_rn(__uint_as_float(static_cast<uint32_t>(a)), b);
    const float hi = __fadd_rn(__uint_as_float(static_cast<uint32_t>(a >> 32)), b);
    a = (static_cast<uint64_t>(__float_as_uint(hi)) << 32) | __float_as_uint(lo);
}

// Two values rounded to a two-byte output type, the first in the low half.
template <int OUT>
__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    if (OUT == QUARTZ_OUT_BF16) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<const uint32_t *>(&a);
    }
    const __half2 a = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&a);
}

template <int OUT>
__device__ __forceinline__ void store_quad(void *y, int64_t off, float4 v)
{
    if (OUT == QUARTZ_OUT_F32)
        *reinterpret_cast<float4 *>(static_cast<float *>(y) + off) = v;
    else
        *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(y) + off) = make_uint2(pack2<OUT>(v.x, v.y), pack2<OUT>(v.z, v.w));
}

// v + bias[n .. n + 3] in fp32 (no bias: v).
__device__ __forceinline__ float4 add_bias4(const GemmArgs &args, int64_t n, float4 v)
{
    if (args.bias) {
        const uint2 braw = __ldg(reinterpret_cast<const uint2 *>(args.bias + n));
        const float2 b0 = __half22float2(*reinterpret_cast<const __half2 *>(&braw.x));
        const float2 b1 = __half22float2(*reinterpret_cast<const __half2 *>(&braw.y));
        v.x = __fadd_rn(v.x, b0.x);
        v.y = __fadd_rn(v.y, b0.y);
        v.z = __fadd_rn(v.z, b1.x);
        v.w = __fadd_rn(v.w, b1.y);
    }
    return v;
}

// Output of one epilogue warp's 32 x 64 slice of a tile.  Two-byte outputs go
// through the warp's block of shared memory (128-byte rows, 128-byte swizzle:
// the 8-byte writes of a warp then hit every bank twice at most) and leave it
// by one tensor store, which clips rows past M and columns past N, so that
// the warp is back at its next group while the tile is written: with direct
// 8-byte stores a tile held its warps for about 2 us.  fp32 outputs are
// stored directly (their blocks would not fit).
template <int OUT>
struct TileOut {
    static constexpr bool kStaged = OUT != QUARTZ_OUT_F32;
    const GemmArgs &args;
    const CUtensorMap *tmap;
    uint32_t block, at;  // this warp's block; this thread's 8 bytes of a row, before row and chunk
    uint32_t swz;
    int64_t m0, n0;      // first row and column of the slice
    int trow, tq, lane;

    // (m, n): first row and column of the slice.  Made at the end of a tile,
    // from a fresh read of the lane number, so that none of it takes
    // registers in the group loop.
    __device__ __forceinline__ TileOut(const GemmArgs &a, const CUtensorMap *t, uint32_t out_base, int warp, int64_t m,
                                       int64_t n)
        : args(a), tmap(t), m0(m), n0(n)
    {
        asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
        trow = lane >> 2;
        tq = 4 * (lane & 3);
        block = out_base + warp * kOutBlockBytes;
        at = block + trow * 128 + ((2 * tq) & 15);
        swz = static_cast<uint32_t>((trow ^ (tq >> 3)) << 4);
        if (kStaged) {
            bulk_wait_read();  // the previous tile has left the block (every lane asks, so none diverges)
            __syncwarp();
        }
    }

    // v: columns 16 chunk + tq .. + 3 of row r8 + trow (r8: 0, 8, 16, 24) of
    // the slice, rounded once to the output type.
    __device__ __forceinline__ void put_raw(int r8, int chunk, float4 v)
    {
        if (kStaged) {
            sts_b64(at + r8 * 128 + ((32u * chunk) ^ swz), pack2<OUT>(v.x, v.y), pack2<OUT>(v.z, v.w));
        } else {
            const int64_t m = m0 + r8 + trow, n = n0 + 16 * chunk + tq;
            if (m < args.M && n < args.N)
                *reinterpret_cast<float4 *>(static_cast<float *>(args.y) + m * args.N + n) = v;
        }
    }

    // The same after adding the bias in fp32.
    __device__ __forceinline__ void put(int r8, int chunk, float4 v)
    {
        const int64_t n = n0 + 16 * chunk + tq;
        if (n < args.N) v = add_bias4(args, n, v);
        put_raw(r8, chunk, v);
    }

    __device__ __forceinline__ void end()
    {
        if (!kStaged) return;
        fence_proxy_async();
        __syncwarp();
        if (lane == 0 && m0 < args.M && n0 < args.N) {
            tma_store_2d(tmap, block, static_cast<int32_t>(n0), static_cast<int32_t>(m0));
            bulk_commit();
        }
    }

    // Before the kernel ends: this warp's stores are complete.
    static __device__ __forceinline__ void drain(int lane)
    {
        if (kStaged && lane == 0) bulk_wait_all();
    }
};

// Half of one 16-column chunk: one 16x128b.x4 TMEM load (16 lanes), then
// acc[i] += s_a * (s_w[i] * P_i) for the four pairs P_i = (row, row + 8) of
// column i, on explicit 64-bit register pairs (q: the loaded pairs, s: the
// column scale duplicated into both halves, t: s_w * P).
__device__ __forceinline__ void epi_half_chunk_sym(uint32_t taddr, float4 sw, uint64_t sa, uint64_t *acc)
{
    asm volatile(
        "{\n\t"
        ".reg .b32 p<8>;\n\t"
        ".reg .b64 q<4>, t<4>, s<4>;\n\t"
        "tcgen05.ld.sync.aligned.16x128b.x4.b32 {p0, p1, p2, p3, p4, p5, p6, p7}, [%4];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t"
        "mov.b64 q0, {p0, p1};\n\t"
        "mov.b64 q1, {p2, p3};\n\t"
        "mov.b64 q2, {p4, p5};\n\t"
        "mov.b64 q3, {p6, p7};\n\t"
        "mov.b64 s0, {%5, %5};\n\t"
        "mov.b64 s1, {%6, %6};\n\t"
        "mov.b64 s2, {%7, %7};\n\t"
        "mov.b64 s3, {%8, %8};\n\t"
        "mul.rn.f32x2 t0, q0, s0;\n\t"
        "fma.rn.f32x2 %0, t0, %9, %0;\n\t"
        "mul.rn.f32x2 t1, q1, s1;\n\t"
        "fma.rn.f32x2 %1, t1, %9, %1;\n\t"
        "mul.rn.f32x2 t2, q2, s2;\n\t"
        "fma.rn.f32x2 %2, t2, %9, %2;\n\t"
        "mul.rn.f32x2 t3, q3, s3;\n\t"
        "fma.rn.f32x2 %3, t3, %9, %3;\n\t"
        "}"
        : "+l"(acc[0]), "+l"(acc[1]), "+l"(acc[2]), "+l"(acc[3])
        : "r"(taddr), "f"(sw.x), "f"(sw.y), "f"(sw.z), "f"(sw.w), "l"(sa)
        : "memory");
}

// Per-row-scale epilogue step for half of one 16-column chunk: one
// 16x128b.x4 TMEM load of an accumulator whose values are exact integers
// below 2^22, each turned into an int32 with the 1.5 * 2^23 rounding addend
// (the integer is the float's bit pattern minus 0x4B400000) and added to acc.
__device__ __forceinline__ void epi_half_chunk_int(uint32_t taddr, int32_t *acc)
{
    asm volatile(
        "{\n\t"
        ".reg .b32 p<8>;\n\t"
        ".reg .f32 f<8>;\n\t"
        "tcgen05.ld.sync.aligned.16x128b.x4.b32 {p0, p1, p2, p3, p4, p5, p6, p7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t"
        "add.rn.f32 f0, p0, 0f4B400000;\n\t"
        "add.rn.f32 f1, p1, 0f4B400000;\n\t"
        "add.rn.f32 f2, p2, 0f4B400000;\n\t"
        "add.rn.f32 f3, p3, 0f4B400000;\n\t"
        "add.rn.f32 f4, p4, 0f4B400000;\n\t"
        "add.rn.f32 f5, p5, 0f4B400000;\n\t"
        "add.rn.f32 f6, p6, 0f4B400000;\n\t"
        "add.rn.f32 f7, p7, 0f4B400000;\n\t"
        "mov.b32 p0, f0;\n\t"
        "mov.b32 p1, f1;\n\t"
        "mov.b32 p2, f2;\n\t"
        "mov.b32 p3, f3;\n\t"
        "mov.b32 p4, f4;\n\t"
        "mov.b32 p5, f5;\n\t"
        "mov.b32 p6, f6;\n\t"
        "mov.b32 p7, f7;\n\t"
        "sub.s32 p0, p0, 0x4B400000;\n\t"
        "sub.s32 p1, p1, 0x4B400000;\n\t"
        "sub.s32 p2, p2, 0x4B400000;\n\t"
        "sub.s32 p3, p3, 0x4B400000;\n\t"
        "sub.s32 p4, p4, 0x4B400000;\n\t"
        "sub.s32 p5, p5, 0x4B400000;\n\t"
        "sub.s32 p6, p6, 0x4B400000;\n\t"
        "sub.s32 p7, p7, 0x4B400000;\n\t"
        "add.s32 %0, %0, p0;\n\t"
        "add.s32 %1, %1, p1;\n\t"
        "add.s32 %2, %2, p2;\n\t"
        "add.s32 %3, %3, p3;\n\t"
        "add.s32 %4, %4, p4;\n\t"
        "add.s32 %5, %5, p5;\n\t"
        "add.s32 %6, %6, p6;\n\t"
        "add.s32 %7, %7, p7;\n\t"
        "}"
        : "+r"(acc[0]), "+r"(acc[1]), "+r"(acc[2]), "+r"(acc[3]), "+r"(acc[4]), "+r"(acc[5]),
          "+r"(acc[6]), "+r"(acc[7])
        : "r"(taddr)
        : "memory");
}

// Two 64-bit words from shared memory (one 16-byte load).
__device__ __forceinline__ void lds_b64x2(uint32_t addr, uint64_t &a, uint64_t &b)
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

// Partials dump: one epilogue warp's 32 x 64 slice (first row m0, first column
// n0) of group args.partials_group, read again from its accumulator at tbase.
// The exact integer P_g: with zero points (ZERO) the terms that the tensor core
// added are taken off again (all integers below 2^24, exact in fp32).  It runs
// for one group of a tile, beside the group loop that every call has.  Against a
// group loop of its own that fetched the zero points per group from global
// memory (GEMM 4001 x 3456 x 1152, fp16 / fp32 out): 203 -> 60 / 166 -> 64 us
// with zero points (37.5 / 44 without a dump), 85 -> 44 / 89 -> 52 without
// (33 / 40).
template <bool ZERO>
__device__ __forceinline__ void dump_partials(const GemmArgs &args, uint32_t tbase, int64_t m0, int64_t n0)
{
    int lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    m0 += lane >> 2;
    n0 += 4 * (lane & 3);
    const int64_t g = args.partials_group;
#pragma unroll 1
    for (int chunk = 0; chunk < 4; ++chunk, n0 += 16) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            uint32_t r[8];  // columns n0 + i of rows m0 + 16 h (r[2 i]) and 8 below (r[2 i + 1])
            __syncwarp();
            tmem_ld_16x128b_x4(tbase + (static_cast<uint32_t>(16 * h) << 16) + 16 * chunk, r);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t m = m0 + 16 * h + 8 * e;
                float2 ta = make_float2(0.f, 0.f);
                if (ZERO) ta = zero_terms(zero_recs(args.a_side, args.G, args.m_pad)[g * args.m_pad + m], true);
                int32_t P[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float p = __uint_as_float(r[2 * i + e]);
                    if (ZERO) {
                        const float2 tw = zero_terms(
                            zero_recs(args.w_side, args.G, args.n_pad)[g * args.n_pad + perm16(n0 + i)], false);
                        p = __fmaf_rn(ta.x, tw.y, __fmaf_rn(-tw.x, ta.y, p));
                    }
                    P[i] = __float2int_rn(p);
                }
                if (m < args.M && n0 < args.N)
                    *reinterpret_cast<int4 *>(args.partials + m * args.N + n0) = make_int4(P[0], P[1], P[2], P[3]);
            }
        }
    }
}

template <int MODE, int OUT, bool DUMP, bool PERROW, int RM = kRasterM>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_a,
                        const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_y,
                        const GemmArgs args)
{
    griddep_wait();
    constexpr bool ZERO = MODE == QUARTZ_ASYMMETRIC;  // zero-point terms by the tensor core
    using L = Smem<ZERO, OUT != QUARTZ_OUT_F32>;
    constexpr int kStages = L::kStages, kStageBytes = L::kStageBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bar_base = smem_base + L::kBars;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
    auto acc_full_bar = [&](int b) { return bar_base + 8u * (2 * kStages + b); };
    auto acc_empty_bar = [&](int b) { return bar_base + 8u * (2 * kStages + 2 + b); };
    const uint32_t drain_bar = bar_base + 8u * (2 * kStages + 4);
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + L::kMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kMisc + 4);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full_bar(s), ZERO ? 2 : 1);  // the copies, and the records
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full_bar(b), 2);  // the commit and the issuing lane
            mbar_init(acc_empty_bar(b), kEpiWarps);
        }
        mbar_init(drain_bar, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if constexpr (ZERO) {
        // the upper halves of the record rows and the zero block stay zero
        for (int i = threadIdx.x; i < L::kZeroBytes / 16; i += kThreads)
            *reinterpret_cast<uint4 *>(smem + L::kZeros + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
        for (int st = 0; st < kStages; ++st)
            for (int i = threadIdx.x; i < kRecBytes / 16; i += kThreads)
                *reinterpret_cast<uint4 *>(smem + st * kStageBytes + L::kRecA + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(tmem_holder), kTmemCols);
        tmem_relinquish();
    }
    if (warp == kProducerWarp && lane == 0) {
        tma_prefetch_desc(&tmap_a);
        tma_prefetch_desc(&tmap_w);
        if (OUT != QUARTZ_OUT_F32) tma_prefetch_desc(&tmap_y);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    const int G = args.G;

    if (warp >= kEpiWarps) {
      regs_decrease<kRegsControl>();
      if (warp == kProducerWarp) {
        // ------------------------------------------------------------------
        // TMA producer: one stage = one 64-wide group of A (128 rows) and W
        // (256 rows).  Rows past M or N are zero-filled by the tensor map.
        // The whole warp runs the loop and one elected lane issues (see
        // elect_one): a stage costs about 60 cycles this way, against 460
        // from a divergent lane.
        // ------------------------------------------------------------------
        const bool leader = elect_one();
        int it = 0, s = 0;   // groups whose operand copies were issued; the next stage
        uint32_t phase = 1;  // parity of that stage's last release (the first round waits for none)
        bool ok = true;
        const int n_items = work_items(args);
        for (int k = 0; k < n_items && ok; ++k) {
            const WorkItem wi = work_item(args, k);
            int mt, nt;
            tile_coords<RM>(wi.tile, args, mt, nt);
            const float *src_a = args.a_side + wi.g0 * args.m_pad + static_cast<int64_t>(mt) * BM;
            const float *src_w = args.w_side + wi.g0 * args.n_pad + static_cast<int64_t>(nt) * BN;
            for (int g = wi.g0; g < wi.g1; ++g, ++it) {
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, args.dev_err, kWaitLimitNs)) {
                    ok = false;
                    break;
                }
                if (leader) {
                    const uint32_t sa = smem_base + L::kOperands + s * kStageBytes;
                    mbar_arrive_expect_tx(full_bar(s), kABytes + kBBytes + (PERROW ? 0 : L::kSideSlotBytes));
                    tma_load_2d(sa, &tmap_a, g * BK, mt * BM, full_bar(s));
                    tma_load_2d(sa + kABytes, &tmap_w, g * BK, nt * BN, full_bar(s));
                    if (!PERROW) {
                        const uint32_t dst = smem_base + L::kSide + (it % L::kSideSlots) * L::kSideSlotBytes;
                        bulk_load(dst, src_a, BM * 4, full_bar(s));
                        bulk_load(dst + L::kSideABytes, src_w, BN * 4, full_bar(s));
                    }
                }
                __syncwarp();
                src_a += args.m_pad;
                src_w += args.n_pad;
                if (++s == kStages) {
                    s = 0;
                    phase ^= 1u;
                }
            }
        }
        // Never leave the CTA with copies in flight: wait for the last
        // load issued into every stage (bounded, even after an abort).
        if (leader) {
            int zero = 0;
            for (int i = 0; i < kStages && i < it; ++i) {
                const int last = it - 1 - ((it - 1 - i) % kStages);
                mbar_wait_bounded(full_bar(i), (last / kStages) & 1, &zero, args.dev_err, kWaitLimitNs);
            }
        }
        __syncwarp();
      } else if (ZERO && warp == kRecWarp) {
        // ------------------------------------------------------------------
        // Zero-point records: each group's 128 + 256 records go by 8-byte
        // asynchronous copies into the lower halves of the stage's rows,
        // kRecDepth groups in flight; a group is handed over once its copies
        // have landed and are visible to the async proxy.
        // ------------------------------------------------------------------
        int it = 0, s = 0, done = 0;  // groups issued, the next stage, the stage to hand over next
        uint32_t phase = 1;
        bool ok = true;
        const int n_items = work_items(args);
        for (int k = 0; k < n_items && ok; ++k) {
            const WorkItem wi = work_item(args, k);
            int mt, nt;
            tile_coords<RM>(wi.tile, args, mt, nt);
            const ZeroRec *src_a = zero_recs(args.a_side, G, args.m_pad) + wi.g0 * args.m_pad +
                                   static_cast<int64_t>(mt) * BM + lane;
            const ZeroRec *src_w = zero_recs(args.w_side, G, args.n_pad) + wi.g0 * args.n_pad +
                                   static_cast<int64_t>(nt) * BN + lane;
            for (int g = wi.g0; g < wi.g1; ++g, ++it) {
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, args.dev_err, kWaitLimitNs)) {
                    ok = false;
                    break;
                }
                const uint32_t dst = smem_base + s * kStageBytes + L::kRecA + lane * kRecRow;
#pragma unroll
                for (int i = 0; i < BM / 32; ++i) cp_async8(dst + 32 * i * kRecRow, src_a + 32 * i);
#pragma unroll
                for (int i = 0; i < BN / 32; ++i) cp_async8(dst + (BM + 32 * i) * kRecRow, src_w + 32 * i);
                cp_async_commit();
                src_a += args.m_pad;
                src_w += args.n_pad;
                if (it >= kRecDepth - 1) {
                    cp_async_wait<kRecDepth - 1>();  // group it - (kRecDepth - 1) has landed
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full_bar(done));
                    if (++done == kStages) done = 0;
                }
                if (++s == kStages) {
                    s = 0;
                    phase ^= 1u;
                }
            }
        }
        cp_async_wait<0>();
        fence_proxy_async();
        __syncwarp();
        if (lane == 0 && ok)
            for (int i = min(it, kRecDepth - 1); i > 0; --i) {
                mbar_arrive(full_bar(done));
                if (++done == kStages) done = 0;
            }
        __syncwarp();
      } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------
        // MMA issuer: 2 x (M=128, N=256, K=32) kind::f8f6f4 MMAs per group into
        // a fresh accumulator (first MMA overwrites), then two commits: one
        // frees the operand stage, one hands P_g to the epilogue.
        // ------------------------------------------------------------------
        {
            const uint32_t idesc = args.wide ? idesc_e5m2_f32(BM, BN) : idesc_e4m3_f32(BM, BN);
            const uint64_t desc_a0 = sdesc_k_major_sw64(smem_base + L::kOperands);
            const uint64_t desc_w0 = sdesc_k_major_sw64(smem_base + L::kOperands + kABytes);
            // records: 8-row blocks of 16-byte rows 128 bytes apart, the second
            // 16 bytes of K in the zero block
            const uint64_t desc_ra0 = sdesc_k_major_none(smem_base + L::kRecA, smem_base + L::kZeros);
            const uint64_t desc_rw0 = sdesc_k_major_none(smem_base + L::kRecW, smem_base + L::kZeros);
            const bool leader = elect_one();
            int s = 0;
            uint32_t phase = 0;
            bool ok = true;
            constexpr int CH = PERROW ? kPerRowChunk : 1;  // stages per TMEM accumulator
            int ic = 0;                                    // accumulators handed to the epilogue
            const int n_items = work_items(args);
            for (int k = 0; k < n_items && ok; ++k) {
                const WorkItem wi = work_item(args, k);
                for (int g = wi.g0; g < wi.g1; ++g) {
                    const int b = ic & 1;
                    const bool first = ((g - wi.g0) % CH) == 0;
                    const bool last = ((g - wi.g0) % CH) == CH - 1 || g == wi.g1 - 1;
                    if (!mbar_wait_warp(full_bar(s), phase, abort_flag, args.dev_err, kWaitLimitNs) ||
                        (first && ic >= 2 && !mbar_wait_warp(acc_empty_bar(b), ((ic >> 1) - 1) & 1, abort_flag,
                                                             args.dev_err, kWaitLimitNs))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t st = static_cast<uint64_t>(s * (kStageBytes / 16));  // (descriptor address units)
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < BK / 32; ++kk)
                            mma_f8_ss(tmem_base + static_cast<uint32_t>(b * BN), desc_a0 + st + 2 * kk,
                                      desc_w0 + st + 2 * kk, idesc, (kk > 0 || !first) ? 1u : 0u);
                        if (ZERO)  // (the distance to the zero block shrinks as the address grows)
                            mma_f16_ss(tmem_base + static_cast<uint32_t>(b * BN), desc_ra0 + st - (st << 16),
                                       desc_rw0 + st - (st << 16), idesc_f16_f32(BM, BN), 1u);
                        mma_commit(empty_bar(s));
                        if (last) {
                            mma_commit(acc_full_bar(b));
                            mbar_arrive(acc_full_bar(b));  // orders the side values, seen landed above, before their readers
                        }
                    }
                    __syncwarp();
                    if (last) ++ic;
                    if (++s == kStages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
            }
            // Make sure no MMA is still writing TMEM before it is freed.
            if (leader) {
                mma_commit(drain_bar);
                int zero = 0;
                mbar_wait_bounded(drain_bar, 0, &zero, args.dev_err, kWaitLimitNs);
            }
        }
        __syncwarp();
      }
    } else {
        regs_increase<kRegsEpilogue>();
        // ------------------------------------------------------------------
        // Epilogue.  Warp w reads TMEM lanes [32*(w%4), +32) (tile rows) and
        // TMEM columns [64*(w/4), +64) with the 16x128b shape: per 16-column
        // chunk, thread t holds TMEM columns t%4 + {0,4,8,12} of lanes t/4 and
        // t/4 + 8 (and t/4 + 16, t/4 + 24 from the second lane half).  With
        // the weight rows transposed inside each 16-row block, those four TMEM
        // columns are the four consecutive output columns 4*(t%4) + {0..3},
        // so one 16-byte shared load gives their scales (each used for four
        // rows) and the stores are 4-wide.  The thread's four row scales are
        // one 16-byte load as well (rows are permuted in the side values).
        // Per group, y += s_a * (s_w * P_g) on (row, row + 8) pairs with
        // f32x2 arithmetic (with zero points the tensor core has added their
        // exact integer terms to P_g).
        // ------------------------------------------------------------------
        const int quarter = warp & 3;
        const int slot = warp >> 2;
        const int trow = lane >> 2;          // row offset inside each 8-row band
        const int tq = 4 * (lane & 3);       // first of this thread's 4 output columns in a 16-column chunk

        // acc[h][j]: output column 16*(j/4) + tq + j%4 of this warp's slice,
        // rows trow + 16h (.x) and trow + 16h + 8 (.y)
        if constexpr (PERROW) {
            // Per-row scales (group_q = K, symmetric): each TMEM accumulator
            // holds the exact integer sum of kPerRowChunk stages; the epilogue
            // adds it into int32 accumulators and scales once per tile:
            // y = s_a * (s_w * P).  acci[c][4h + i] = rows trow + 16h (i < 4:
            // pairs 2i / 2i + 1 are rows +0 / +8) of column 16c + tq + i%4.
            int32_t acci[4][16];
            int ic = 0;
            bool ok = true;
            const int n_items = work_items(args);
            for (int k = 0; k < n_items && ok; ++k) {
                const WorkItem wi = work_item(args, k);
                const int nchunks = (wi.g1 - wi.g0 + kPerRowChunk - 1) / kPerRowChunk;
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int j = 0; j < 16; ++j) acci[c][j] = 0;
                for (int cc = 0; cc < nchunks; ++cc, ++ic) {
                    const int b = ic & 1;
                    if (!mbar_wait_warp(acc_full_bar(b), (ic >> 1) & 1, abort_flag, args.dev_err, kWaitLimitNs)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                                           static_cast<uint32_t>(b * BN + slot * kColsPerWarp);
#pragma unroll
                    for (int chunk = 0; chunk < 4; ++chunk) {
                        epi_half_chunk_int(tbase + 16 * chunk, acci[chunk]);
                        epi_half_chunk_int(tbase + (16u << 16) + 16 * chunk, acci[chunk] + 8);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_empty_bar(b));
                }
                if (!ok) break;
                if (!DUMP && wi.part >= 0) {  // a cut tile: this part's integer sums (planes as below)
                    uint4 *dst = reinterpret_cast<uint4 *>(args.tail_part) +
                                 ((wi.tail * args.split + wi.part) * 16 * (kEpiWarps * 32) + warp * 32 + lane);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            dst[(4 * c + j) * (kEpiWarps * 32)] =
                                make_uint4(static_cast<uint32_t>(acci[c][4 * j]), static_cast<uint32_t>(acci[c][4 * j + 1]),
                                           static_cast<uint32_t>(acci[c][4 * j + 2]), static_cast<uint32_t>(acci[c][4 * j + 3]));
                    continue;
                }
                int mt, nt;
                tile_coords<RM>(wi.tile, args, mt, nt);
                const int64_t n0 = static_cast<int64_t>(nt) * BN + slot * kColsPerWarp;
                TileOut<OUT> out(args, &tmap_y, smem_base + L::kOut, warp, static_cast<int64_t>(mt) * BM + quarter * 32,
                                 n0);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int r = 16 * h + 8 * e + trow;
                        const int64_t m = static_cast<int64_t>(mt) * BM + quarter * 32 + r;
                        const float s_a = args.a_side[perm32(m)];  // (side values are padded to whole tiles)
#pragma unroll
                        for (int chunk = 0; chunk < 4; ++chunk) {
                            const int64_t n = n0 + 16 * chunk + tq;
                            const float4 s_w = *reinterpret_cast<const float4 *>(args.w_side + n);
                            const float swv[4] = {s_w.x, s_w.y, s_w.z, s_w.w};
                            float vv[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int32_t P = acci[chunk][8 * h + 2 * i + e];
                                if (DUMP && m < args.M && n < args.N) args.partials[m * args.N + n + i] = P;
                                vv[i] = __fmul_rn(__fmul_rn(static_cast<float>(P), swv[i]), s_a);
                            }
                            out.put(16 * h + 8 * e, chunk, make_float4(vv[0], vv[1], vv[2], vv[3]));
                        }
                    }
                out.end();
            }
        } else {
            // Groups of 64 (with zero points the accumulator holds the corrected
            // sum): each half chunk (16 lanes x 16 columns: TMEM
            // load, wait and the scale arithmetic) is one PTX block on
            // explicit 64-bit pairs, which keeps the kernel free of spills.
            // The group loop carries only its accumulators, three offsets and
            // a count: with the work item and a group index carried too, ptxas
            // spilled and added moves (18432 x 12288 x 3072 1047 us, now 984;
            // 8192 x 4608 x 1152 84.6, now 79; both with TileOut).  A group takes
            // 850 cycles (18432 x 12288 x 3072, ends of tiles included) against
            // 512 of fp32 lanes: FMA pipe 64% busy, issue slots 65%.  Loads of
            // 32 columns or of both lane halves per wait, and scales loaded
            // ahead, measured 1-10% slower.
            // acc64[c][4h + i]: output column 16c + tq + i, rows trow + 16h (low) and + 8 (high)
            uint64_t acc64[4][8];
            uint32_t buf = 0, par = 0, side = 0;  // accumulator (column offset), its parity, scale slot offset
            const uint32_t tbase0 = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(slot * kColsPerWarp);
            const uint32_t side_a0 = smem_base + L::kSide + (quarter * 32 + 4 * trow) * 4;
            const uint32_t side_w0 = smem_base + L::kSide + L::kSideABytes + (slot * kColsPerWarp + tq) * 4;
            bool ok = true;
            const int n_items = work_items(args);
            for (int k = 0; k < n_items && ok; ++k) {
                int left;
                {
                    const WorkItem wi = work_item(args, k);
                    left = wi.g1 - wi.g0;
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc64[c][j] = 0ull;
                for (; left > 0; --left) {
                    const uint32_t full = acc_full_bar(0) + (buf >> 5);
                    if (!mbar_wait_warp(full, par, abort_flag, args.dev_err, kWaitLimitNs)) {
                        ok = false;
                        break;
                    }
                    uint64_t sa0, sa1;
                    lds_b64x2(side_a0 + side, sa0, sa1);
                    tc_fence_after();
                    const uint32_t tbase = tbase0 + buf;
#pragma unroll
                    for (int chunk = 0; chunk < 4; ++chunk) {
                        const float4 sw = lds_f4(side_w0 + side + 16 * chunk * 4);
                        epi_half_chunk_sym(tbase + 16 * chunk, sw, sa0, acc64[chunk]);
                        epi_half_chunk_sym(tbase + (16u << 16) + 16 * chunk, sw, sa1, acc64[chunk] + 4);
                    }
                    if (DUMP && left == G - args.partials_group) {  // (whole tiles: left counts down from G)
                        int mt, nt;
                        tile_coords<RM>(blockIdx.x + k * gridDim.x, args, mt, nt);
                        dump_partials<ZERO>(args, tbase, static_cast<int64_t>(mt) * BM + quarter * 32,
                                            static_cast<int64_t>(nt) * BN + slot * kColsPerWarp);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full + 16);
                    side += L::kSideSlotBytes;
                    if (side == L::kSideSlots * L::kSideSlotBytes) side = 0;
                    par ^= buf >> 8;
                    buf ^= BN;
                }
                if (!ok) break;
                asm volatile("" : "+r"(k));  // the item is looked up again rather than carried through the loop
                const WorkItem wi = work_item(args, k);
                if (!DUMP && wi.part >= 0) {
                    // split last wave: leave this part's fp32 partial tile for
                    // tail_combine_kernel: slot tail * split + part holds 16
                    // planes of one uint4 per epilogue thread (coalesced)
                    uint4 *dst = reinterpret_cast<uint4 *>(args.tail_part) +
                                 ((wi.tail * args.split + wi.part) * 16 * (kEpiWarps * 32) + warp * 32 + lane);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            dst[(4 * c + j) * (kEpiWarps * 32)] = make_uint4(static_cast<uint32_t>(acc64[c][2 * j]),
                                                        static_cast<uint32_t>(acc64[c][2 * j] >> 32),
                                                        static_cast<uint32_t>(acc64[c][2 * j + 1]),
                                                        static_cast<uint32_t>(acc64[c][2 * j + 1] >> 32));
                    continue;
                }
                int mt, nt;
                tile_coords<RM>(wi.tile, args, mt, nt);
                TileOut<OUT> out(args, &tmap_y, smem_base + L::kOut, warp, static_cast<int64_t>(mt) * BM + quarter * 32,
                                 static_cast<int64_t>(nt) * BN + slot * kColsPerWarp);
                // The bias goes into the accumulators, read once per column with all
                // four loads in flight, rather than through every put: prepare +
                // GEMM 18432 x 12288 x 3072 with a bias 1002 -> 983 us, without one
                // 999 -> 969; 8192 x 4608 x 1152 80.1 -> 79.4 and 79.7 -> 76.7.
                if (args.bias) {
                    uint2 braw[4];
#pragma unroll
                    for (int chunk = 0; chunk < 4; ++chunk) {
                        const int64_t n = out.n0 + 16 * chunk + tq;  // (columns past N take column 0's: they are not stored)
                        braw[chunk] = __ldg(reinterpret_cast<const uint2 *>(args.bias + (n < args.N ? n : 0)));
                    }
#pragma unroll
                    for (int chunk = 0; chunk < 4; ++chunk) {
                        const float2 b0 = __half22float2(*reinterpret_cast<const __half2 *>(&braw[chunk].x));
                        const float2 b1 = __half22float2(*reinterpret_cast<const __half2 *>(&braw[chunk].y));
                        const float bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            add_to_pair(acc64[chunk][i], bv[i & 3]);
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int chunk = 0; chunk < 4; ++chunk) {
                            float vv[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const uint64_t q = acc64[chunk][4 * h + i];
                                vv[i] = __uint_as_float(static_cast<uint32_t>(e ? (q >> 32) : q));
                            }
                            out.put_raw(16 * h + 8 * e, chunk, make_float4(vv[0], vv[1], vv[2], vv[3]));
                        }
                out.end();
            }
        }
        TileOut<OUT>::drain(lane);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Split last wave (see GemmArgs): adds each tail tile's partial tiles in part
// order (fp32, or int32 with scales per row, which are then applied), then
// stores the sum as the epilogue would have.  Grid: (tail tile, 16-column chunk c of every warp's slice); block:
// one thread per epilogue thread, which owns the chunk's 8 column pairs.
template <int OUT, bool PERROW>
__global__ void __launch_bounds__(kEpiWarps * 32) tail_combine_kernel(const __grid_constant__ GemmArgs args)
{
    griddep_wait();
    constexpr int T = kEpiWarps * 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tail = blockIdx.x >> 2, c = blockIdx.x & 3;
    // parts of this tile: every one of the split equal parts, or (range
    // forms) one per CTA range the tile's groups meet
    const int parts = args.ls > 0 ? ((tail + 1) * args.G - 1) / args.ls - (tail * args.G) / args.ls + 1
                                  : args.split;
    if (parts == 1) return;  // the tile lies in one CTA's range: stored whole by the GEMM
    const uint4 *src = reinterpret_cast<const uint4 *>(args.tail_part) +
                       static_cast<int64_t>(tail) * args.split * 16 * T + 4 * c * T + threadIdx.x;
    uint32_t acc[16];  // acc[4i' ..]: pairs (row, row + 8) of the chunk's columns, as the epilogue holds them
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint4 v = __ldcg(src + j * T);
        acc[4 * j] = v.x, acc[4 * j + 1] = v.y, acc[4 * j + 2] = v.z, acc[4 * j + 3] = v.w;
    }
    for (int p = 1; p < parts; ++p) {
        const uint4 *sp = src + static_cast<int64_t>(p) * 16 * T;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 v = __ldcg(sp + j * T);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
                acc[4 * j + i] = PERROW ? acc[4 * j + i] + w[i]
                                        : __float_as_uint(__fadd_rn(__uint_as_float(acc[4 * j + i]), __uint_as_float(w[i])));
        }
    }
    int mt, nt;
    if (args.raster_m == 1)
        tile_coords<1>(args.full_tiles + tail, args, mt, nt);
    else
        tile_coords<kRasterM>(args.full_tiles + tail, args, mt, nt);
    const int quarter = warp & 3, slot = warp >> 2, trow = lane >> 2, tq = 4 * (lane & 3);
    const int64_t n = static_cast<int64_t>(nt) * BN + slot * kColsPerWarp + 16 * c + tq;
    if (n >= args.N) return;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int64_t m = static_cast<int64_t>(mt) * BM + quarter * 32 + 16 * h + 8 * e + trow;
            if (m >= args.M) continue;
            float vv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t q = acc[8 * h + 2 * i + e];
                vv[i] = PERROW ? __fmul_rn(__fmul_rn(static_cast<float>(static_cast<int32_t>(q)), args.w_side[n + i]),
                                           args.a_side[perm32(m)])
                               : __uint_as_float(q);
            }
            store_quad<OUT>(args.y, m * args.N + n, add_bias4(args, n, make_float4(vv[0], vv[1], vv[2], vv[3])));
        }
}

// ---------------------------------------------------------------------------
// 3. SIMT GEMM: same decoded operands, same epilogue arithmetic, CUDA cores.
//    64x64 output tile per 256-thread block, 4x4 outputs per thread.
// ---------------------------------------------------------------------------
// Zero-point terms of group g for the tile's 64 rows from m0 (z[0]) and 64
// columns from n0 (z[1], column r at 16 (r % 4) + r / 4, so that a warp's reads
// of one of its 4 columns a thread are contiguous), converted once per tile and
// group by threads 0 .. 127 beside the operand loads (the side values are padded
// past the last tile).  With records read and converted for every output: SIMT
// 4001 x 3456 x 1152 2410 us, now 1676; SHIFT 2001 x 1600 x 1152 G_s = 8 310 ->
// 236, 16 267 -> 192, 32 242 -> 173, 64 242 -> 169.
__device__ __forceinline__ void stage_zero_terms(const GemmArgs &args, int g, int m0, int n0, float2 (&z)[2][64])
{
    const int r = threadIdx.x & 63;
    if (threadIdx.x < 64)
        z[0][r] = zero_terms(zero_recs(args.a_side, args.G, args.m_pad)[static_cast<int64_t>(g) * args.m_pad + m0 + r], true);
    else if (threadIdx.x < 128)
        z[1][(r & 3) * 16 + (r >> 2)] = zero_terms(
            zero_recs(args.w_side, args.G, args.n_pad)[static_cast<int64_t>(g) * args.n_pad + perm16(n0 + r)], false);
}

template <int MODE, int OUT>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const __nv_fp8_e4m3 *__restrict__ a_op,
                                                        const __nv_fp8_e4m3 *__restrict__ w_op,
                                                        const GemmArgs args, int K)
{
    griddep_wait();
    __shared__ int16_t sa[64][kGroupQ + 2];
    __shared__ int16_t sw[64][kGroupQ + 2];
    __shared__ float2 z[2][64];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    float y[4][4] = {};
    for (int g = 0; g < args.G; ++g) {
        for (int i = threadIdx.x; i < 64 * kGroupQ; i += 256) {
            const int r = i / kGroupQ, k = i % kGroupQ;
            const int64_t kk = static_cast<int64_t>(g) * kGroupQ + k;
            sa[r][k] = (m0 + r < args.M) ? static_cast<int16_t>(static_cast<float>(a_op[(int64_t)(m0 + r) * K + kk])) : 0;
            sw[r][k] = (n0 + r < args.N) ? static_cast<int16_t>(static_cast<float>(w_op[perm16(n0 + r) * K + kk])) : 0;
        }
        if constexpr (MODE == QUARTZ_ASYMMETRIC) stage_zero_terms(args, g, m0, n0, z);
        __syncthreads();
        int p[4][4] = {};
        for (int k = 0; k < kGroupQ; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) p[i][j] += sa[ty * 4 + i][k] * sw[tx * 4 + j][k];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = m0 + ty * 4 + i;
            const float s_a = args.a_side[static_cast<int64_t>(g) * args.m_pad + perm32(m)];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = n0 + tx * 4 + j;
                if (m >= args.M || n >= args.N) continue;
                float P = static_cast<float>(p[i][j]);
                if (args.partials && g == args.partials_group) args.partials[(int64_t)m * args.N + n] = p[i][j];
                if constexpr (MODE == QUARTZ_ASYMMETRIC) {
                    const float2 ta = z[0][ty * 4 + i], tw = z[1][16 * j + tx];
                    P = __fmaf_rn(tw.x, ta.y, P);
                    P = __fmaf_rn(-ta.x, tw.y, P);
                }
                const float t = __fmul_rn(P, args.w_side[static_cast<int64_t>(g) * args.n_pad + n]);
                y[i][j] = __fmaf_rn(t, s_a, y[i][j]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (m >= args.M || n >= args.N) continue;
            float v = y[i][j];
            if (args.bias) v = __fadd_rn(v, __half2float(args.bias[n]));
            const int64_t off = (int64_t)m * args.N + n;
            if (OUT == QUARTZ_OUT_F16) static_cast<__half *>(args.y)[off] = __float2half_rn(v);
            else if (OUT == QUARTZ_OUT_BF16) static_cast<__nv_bfloat16 *>(args.y)[off] = __float2bfloat16_rn(v);
            else static_cast<float *>(args.y)[off] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// 4. Accumulator-shift GEMM (the paper's own schedule, Section 4.4): works on
//    the packed 4-bit codes and FLAGs directly, with no decoded operand.  Per
//    subgroup j of G_s elements it forms the integer dot product of the codes
//    and shifts it by the two FLAGs: P_g = sum_j (sum_{k in j} c_a c_w)
//    << (F_a[j] + F_w[j]), which equals sum_k v_a v_w exactly.  The dot
//    products run on dp4a over the codes placed in the high nibble of each
//    byte (int8 value 16c, so a dot product is 256 x the code dot product).
//    The dequant arithmetic is the SIMT kernel's.  64x64 output tile per
//    256-thread block, 4x4 outputs per thread.  WIDE: operands with 16-bit
//    stage-1 codes (Section 5 LLM variant), FLAGs up to 12, so a shifted
//    subgroup product reaches 392 << 24 and the group sums are 64-bit.
// ---------------------------------------------------------------------------
template <int GS, int MODE, int OUT, bool WIDE>
__global__ void __launch_bounds__(256) gemm_shift_kernel(const uint32_t *__restrict__ a_codes,
                                                         const uint8_t *__restrict__ a_flags,
                                                         const uint32_t *__restrict__ w_codes,
                                                         const uint8_t *__restrict__ w_flags,
                                                         const GemmArgs args, int K, int a_packed, int w_packed)
{
    griddep_wait();
    constexpr int kSub = kGroupQ / GS;            // subgroups per group
    constexpr int kWordsPerSub = GS / 4;          // int8x4 words per subgroup
    __shared__ uint32_t sa[64][2 * kGroupQ / 8 + 1];
    __shared__ uint32_t sw[64][2 * kGroupQ / 8 + 1];
    __shared__ uint8_t fa[64][kSub];
    __shared__ uint8_t fw[64][kSub];
    __shared__ float2 z[2][64];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int64_t words_per_row = K / 8, flags_per_row = K / GS;
    float y[4][4] = {};
    for (int g = 0; g < args.G; ++g) {
        for (int i = threadIdx.x; i < 64 * (kGroupQ / 8); i += 256) {
            const int r = i / (kGroupQ / 8), wi = i % (kGroupQ / 8);
            const int64_t col = static_cast<int64_t>(g) * (kGroupQ / 8) + wi;
            const uint32_t ca = (m0 + r < args.M) ? a_codes[(m0 + r) * words_per_row + col] : 0u;
            const uint32_t cw = (n0 + r < args.N) ? w_codes[(n0 + r) * words_per_row + col] : 0u;
            sa[r][2 * wi] = (ca << 4) & 0xF0F0F0F0u;  // even codes, as 16c
            sa[r][2 * wi + 1] = ca & 0xF0F0F0F0u;     // odd codes, as 16c
            sw[r][2 * wi] = (cw << 4) & 0xF0F0F0F0u;
            sw[r][2 * wi + 1] = cw & 0xF0F0F0F0u;
        }
        for (int i = threadIdx.x; i < 64 * kSub; i += 256) {
            const int r = i / kSub, j = i % kSub;
            const int64_t col = static_cast<int64_t>(g) * kSub + j;
            fa[r][j] = (m0 + r < args.M) ? load_flag(a_flags, (m0 + r) * flags_per_row + col, a_packed != 0) : 0;
            fw[r][j] = (n0 + r < args.N) ? load_flag(w_flags, (n0 + r) * flags_per_row + col, w_packed != 0) : 0;
        }
        if constexpr (MODE == QUARTZ_ASYMMETRIC) stage_zero_terms(args, g, m0, n0, z);
        __syncthreads();
        using Acc = typename std::conditional<WIDE, long long, int>::type;
        Acc p[4][4] = {};
#pragma unroll
        for (int j = 0; j < kSub; ++j) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    int dot = 0;
#pragma unroll
                    for (int q = 0; q < kWordsPerSub; ++q)
                        dot = __dp4a(static_cast<int>(sa[ty * 4 + i][j * kWordsPerSub + q]),
                                     static_cast<int>(sw[tx * 4 + jj][j * kWordsPerSub + q]), dot);
                    p[i][jj] += static_cast<Acc>(dot >> 8) << (fa[ty * 4 + i][j] + fw[tx * 4 + jj][j]);
                }
        }
        float2 tws[4];
        if constexpr (MODE == QUARTZ_ASYMMETRIC) {
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) tws[jj] = z[1][16 * jj + tx];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = m0 + ty * 4 + i;
            if (m >= args.M) continue;
            const float s_a = args.a_side[static_cast<int64_t>(g) * args.m_pad + perm32(m)];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const int n = n0 + tx * 4 + jj;
                if (n >= args.N) continue;
                float P = static_cast<float>(p[i][jj]);
                if (!WIDE && args.partials && g == args.partials_group)
                    args.partials[(int64_t)m * args.N + n] = static_cast<int32_t>(p[i][jj]);
                if constexpr (MODE == QUARTZ_ASYMMETRIC) {
                    const float2 ta = z[0][ty * 4 + i], tw = tws[jj];
                    P = __fmaf_rn(tw.x, ta.y, P);
                    P = __fmaf_rn(-ta.x, tw.y, P);
                }
                const float t = __fmul_rn(P, args.w_side[static_cast<int64_t>(g) * args.n_pad + n]);
                y[i][jj] = __fmaf_rn(t, s_a, y[i][jj]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int n = n0 + tx * 4 + jj;
            if (m >= args.M || n >= args.N) continue;
            float v = y[i][jj];
            if (args.bias) v = __fadd_rn(v, __half2float(args.bias[n]));
            const int64_t off = (int64_t)m * args.N + n;
            if (OUT == QUARTZ_OUT_F16) static_cast<__half *>(args.y)[off] = __float2half_rn(v);
            else if (OUT == QUARTZ_OUT_BF16) static_cast<__nv_bfloat16 *>(args.y)[off] = __float2bfloat16_rn(v);
            else static_cast<float *>(args.y)[off] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }
size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn lookup_encode_tiled()
{
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
        return reinterpret_cast<EncodeTiledFn>(p);
    return nullptr;
}

// Looked up once (the initialisation of a function-local static is
// thread-safe, so concurrent first calls from several host threads are fine).
EncodeTiledFn encode_tiled_fn()
{
    static const EncodeTiledFn fn = lookup_encode_tiled();
    return fn;
}

// K-major E4M3 operand [rows, K] (one byte per element) read in boxes of
// [box_rows, 64] with the 64-byte swizzle; out-of-range rows read as zero.
bool make_operand_map(CUtensorMap *m, const void *base, int64_t rows, int64_t K, int box_rows)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(K)};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(BK), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Two-byte output [M, N], written in blocks of 32 rows x 64 columns (128-byte
// swizzle); parts of a block past M or N are not written.
bool make_output_map(CUtensorMap *m, void *y, int64_t M, int64_t N)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(M)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(N) * 2};
    const cuuint32_t box[2] = {kColsPerWarp, 32};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, y, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// SM count of the current device (0 if there is none), looked up once per device.
int device_sms_or_zero()
{
    constexpr int kMaxDevices = 64;
    static std::atomic<int> cached[kMaxDevices];  // 0: not looked up yet
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const bool slot = dev >= 0 && dev < kMaxDevices;
    if (slot && (n = cached[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 0;
    if (slot) cached[dev].store(n, std::memory_order_relaxed);
    return n;
}

int num_sms()
{
    const int n = device_sms_or_zero();
    return n > 0 ? n : 1;
}

template <int MODE, int OUT>
cudaError_t launch_tc(const CUtensorMap &ta, const CUtensorMap &tw, const CUtensorMap &ty, const GemmArgs &args,
                      cudaStream_t s)
{
    constexpr bool staged = OUT != QUARTZ_OUT_F32;
    constexpr int smem = Smem<MODE == QUARTZ_ASYMMETRIC, staged>::kAlloc;
    static_assert(smem <= 227 * 1024, "shared memory budget");
    auto kern = args.partials ? gemm_tcgen05_kernel<MODE, OUT, true, false>
                              : gemm_tcgen05_kernel<MODE, OUT, false, false>;
    if constexpr (MODE == QUARTZ_SYMMETRIC) {
        if (!args.partials && !args.per_row && args.raster_m == 1) kern = gemm_tcgen05_kernel<MODE, OUT, false, false, 1>;
    }
    if constexpr (MODE == QUARTZ_SYMMETRIC) {
        if (args.per_row)
            kern = args.partials ? gemm_tcgen05_kernel<MODE, OUT, true, true>
                                 : gemm_tcgen05_kernel<MODE, OUT, false, true>;
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int grid = args.num_tiles < num_sms() ? args.num_tiles : num_sms();
    if (args.split > 1 && args.ls == 0 && args.full_tiles == 0) grid = args.tail_tiles * args.split;
    if (args.ls > 0) grid = num_sms();  // one group range per SM
    launch_pdl(kern, dim3(grid), dim3(kThreads), smem, s, ta, tw, ty, args);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_tc_out(const CUtensorMap &ta, const CUtensorMap &tw, const CUtensorMap &ty, const GemmArgs &args,
                          int y_type, cudaStream_t s)
{
    switch (y_type) {
        case QUARTZ_OUT_F16: return launch_tc<MODE, QUARTZ_OUT_F16>(ta, tw, ty, args, s);
        case QUARTZ_OUT_BF16: return launch_tc<MODE, QUARTZ_OUT_BF16>(ta, tw, ty, args, s);
        default: return launch_tc<MODE, QUARTZ_OUT_F32>(ta, tw, ty, args, s);
    }
}

template <bool PERROW>
cudaError_t launch_tail_combine(const GemmArgs &args, int y_type, cudaStream_t s)
{
    const unsigned grid = static_cast<unsigned>(args.tail_tiles) * 4;
    switch (y_type) {
        case QUARTZ_OUT_F16: launch_pdl(tail_combine_kernel<QUARTZ_OUT_F16, PERROW>, dim3(grid), dim3(kEpiWarps * 32), 0, s, args); break;
        case QUARTZ_OUT_BF16: launch_pdl(tail_combine_kernel<QUARTZ_OUT_BF16, PERROW>, dim3(grid), dim3(kEpiWarps * 32), 0, s, args); break;
        default: launch_pdl(tail_combine_kernel<QUARTZ_OUT_F32, PERROW>, dim3(grid), dim3(kEpiWarps * 32), 0, s, args); break;
    }
    return cudaGetLastError();
}

template <int MODE, int OUT>
cudaError_t launch_simt(const LinearWorkspace &ws, const GemmArgs &args, int K, cudaStream_t s)
{
    dim3 grid(static_cast<unsigned>((args.N + 63) / 64), static_cast<unsigned>((args.M + 63) / 64));
    launch_pdl(gemm_simt_kernel<MODE, OUT>, dim3(grid), dim3(256), 0, s, static_cast<const __nv_fp8_e4m3 *>(ws.a_op),
                                                     static_cast<const __nv_fp8_e4m3 *>(ws.w_op), args, K);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_simt_out(const LinearWorkspace &ws, const GemmArgs &args, int K, int y_type,
                            cudaStream_t s)
{
    switch (y_type) {
        case QUARTZ_OUT_F16: return launch_simt<MODE, QUARTZ_OUT_F16>(ws, args, K, s);
        case QUARTZ_OUT_BF16: return launch_simt<MODE, QUARTZ_OUT_BF16>(ws, args, K, s);
        default: return launch_simt<MODE, QUARTZ_OUT_F32>(ws, args, K, s);
    }
}

GemmArgs make_args(const LinearWorkspace &ws, int64_t M, int64_t N, int64_t K, const void *bias,
                   void *y, int y_type, int32_t *partials, int partials_group, int *dev_err)
{
    GemmArgs a;
    a.per_row = 0;
    a.wide = 0;
    a.split = 1;
    a.ls = 0;
    a.tail_tiles = 0;
    a.tail_part = ws.tail_part;
    a.a_side = ws.a_side;
    a.w_side = ws.w_side;
    a.m_pad = ws.m_pad;
    a.n_pad = ws.n_pad;
    a.M = static_cast<int>(M);
    a.N = static_cast<int>(N);
    a.G = static_cast<int>(K / kGroupQ);
    a.tiles_n = static_cast<int>((N + BN - 1) / BN);
    a.tiles_m = static_cast<int>((M + BM - 1) / BM);
    a.num_tiles = a.tiles_m * a.tiles_n;
    a.raster_m = kRasterM;
    a.full_tiles = a.num_tiles;
    a.bias = static_cast<const __half *>(bias);
    a.y = y;
    a.y_type = y_type;
    a.partials = partials;
    a.partials_group = partials_group;
    a.dev_err = dev_err;
    return a;
}

}  // namespace

// Split of the GEMM's last wave on this device (symmetric mode; with scales per
// row row_split_pays decides whether it is taken): when the tiles left after whole waves fill at most half of one,
// each of them is cut along K into `split` group ranges (at most
// kMaxTailSplit, at least two groups each) for otherwise idle CTAs; with
// fewer tiles than SMs (a first wave that is also the last), every tile is
// cut that way and the grid has tiles x split CTAs.  When
// they fill more than half, the last two waves' group iterations are spread
// evenly over the CTAs (two-wave form), but only where that shortens the
// critical path by at least kMinStreamSaving group iterations: it costs
// about the time of 25 (partial tiles written and read back, the combine
// launch), measured on the LLaMA-2-7B o (saves 20: 3% slower) and down
// (saves 54: 9% faster) projections.
constexpr int kMaxTailSplit = 4;
constexpr int kMinStreamSaving = 32;

void tail_split(int64_t M, int64_t N, int64_t K, int mode, int *tail, int *split, int *ls = nullptr)
{
    *tail = 0;
    *split = 1;
    if (ls) *ls = 0;
    const int sms = device_sms_or_zero();
    if (mode != QUARTZ_SYMMETRIC || sms <= 0 || M <= 0) return;
    const int64_t T = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    const int64_t P = T < sms ? T : sms;
    const int64_t W = T / P, R = T % P, G = K / kGroupQ;
    if (W >= 1 && 2 * R > P) {
        const int64_t Ts = P + R, U = Ts * G;
        if (G * (P - R) < kMinStreamSaving * P || U >= (int64_t(1) << 30)) return;
        *tail = static_cast<int>(Ts);
        *split = 2;
        if (ls) *ls = static_cast<int>((U + P - 1) / P);
        return;
    }
    if (T < sms && 2 * T > sms) {
        // more than half the SMs hold a tile: the tiles' T * G group
        // iterations are cut into one contiguous range per SM (ls >= G / 2,
        // so a tile meets at most 3 ranges: 3 part slots per tile)
        const int64_t U = T * G;
        if (G * (sms - T) < kMinStreamSaving * sms || U >= (int64_t(1) << 30)) return;
        *tail = static_cast<int>(T);
        *split = 3;
        if (ls) *ls = static_cast<int>((U + sms - 1) / sms);
        return;
    }
    if (T < sms) {  // fewer tiles than SMs: every tile is cut along K for the idle SMs
        int64_t S = sms / T;
        if (S > kMaxTailSplit) S = kMaxTailSplit;
        if (S > G / 2) S = G / 2;
        if (S < 2) return;
        *tail = static_cast<int>(T);
        *split = static_cast<int>(S);
        return;
    }
    if (W < 1 || R == 0) return;
    int64_t S = P / R;
    if (S > kMaxTailSplit) S = kMaxTailSplit;
    if (S > G / 2) S = G / 2;
    if (S < 2) return;
    *tail = static_cast<int>(R);
    *split = static_cast<int>(S);
}

// With scales per row the same plan cuts the int32 sums (exact, so the cut
// changes no result).  A 64-wide stage takes about 0.27 us there, so it is
// taken only where the busiest CTA is spared kMinRowSaving of them, or
// kMinRowRangeSaving in the range forms, which leave more partial tiles.  GEMM
// + combine against whole tiles: 2048 x 1280 x 11520 (ranges, spares 85) 51.9
// -> 41.6 us, 2048 x 1280 x 5760 (42) 31.4 -> 31.4, 2560 x 3072 x 5120 (two
// waves, 34) 49.8 -> 53.9; 8192 x 640 x 5760 (3 parts, 60) 53.9 -> 45.7, 1790 x
// 3064 x 3072 (36) 35.5 -> 31.4, 1000 x 1304 x 2048 (21) 17.1 -> 17.0, 1000 x
// 1304 x 1152 (12) 15.0 -> 17.0.
constexpr int kMinRowSaving = 32;
constexpr int kMinRowRangeSaving = 48;

bool row_split_pays(int64_t M, int64_t N, int64_t K, int tail, int split, int ls)
{
    const int sms = num_sms();
    const int64_t T = ((M + BM - 1) / BM) * ((N + BN - 1) / BN), G = K / kGroupQ;
    const int64_t P = T < sms ? T : sms;
    const int64_t whole = (T + P - 1) / P * G;
    const int64_t cut = (T - tail) / P * G + (ls > 0 ? ls : (G + split - 1) / split);
    return whole - cut >= (ls > 0 ? kMinRowRangeSaving : kMinRowSaving);
}

int linear_tail_parts(int64_t M, int64_t N, int64_t K, int mode, bool per_row)
{
    int tail = 0, split = 1, ls = 0;
    tail_split(M, N, K, mode, &tail, &split, &ls);
    if (per_row && split > 1 && !row_split_pays(M, N, K, tail, split, ls)) return 1;
    return split;
}

size_t tail_part_bytes(int tail, int split) { return static_cast<size_t>(tail) * split * kEpiWarps * 32 * 64 * 4; }

size_t linear_workspace_bytes(int64_t M, int64_t N, int64_t K, int mode)
{
    const int nside = mode == QUARTZ_ASYMMETRIC ? 3 : 1;
    const int64_t G = K / kGroupQ;
    size_t b = align256(static_cast<size_t>(M) * K);
    b += align256(static_cast<size_t>(round_up(N, 16)) * K);
    b += align256(static_cast<size_t>(nside) * G * round_up(M > 0 ? M : 1, BM) * 4);
    b += align256(static_cast<size_t>(nside) * G * round_up(N, BN) * 4);
    int tail = 0, split = 1;
    tail_split(M, N, K, mode, &tail, &split);
    if (split > 1) b += align256(tail_part_bytes(tail, split));
    return b;
}

void linear_workspace_carve(void *base, int64_t M, int64_t N, int64_t K, int mode,
                            LinearWorkspace *ws)
{
    const int nside = mode == QUARTZ_ASYMMETRIC ? 3 : 1;
    const int64_t G = K / kGroupQ;
    uint8_t *p = static_cast<uint8_t *>(base);
    ws->nside = nside;
    ws->m_pad = round_up(M > 0 ? M : 1, BM);
    ws->n_pad = round_up(N, BN);
    ws->a_op = p;
    p += align256(static_cast<size_t>(M) * K);
    ws->w_op = p;
    p += align256(static_cast<size_t>(round_up(N, 16)) * K);
    ws->a_side = reinterpret_cast<float *>(p);
    p += align256(static_cast<size_t>(nside) * G * ws->m_pad * 4);
    ws->w_side = reinterpret_cast<float *>(p);
    p += align256(static_cast<size_t>(nside) * G * ws->n_pad * 4);
    tail_split(M, N, K, mode, &ws->tail_tiles, &ws->tail_split, &ws->tail_ls);
    ws->tail_part = ws->tail_split > 1 ? reinterpret_cast<float *>(p) : nullptr;
}

size_t prepared_weights_bytes(int64_t N, int64_t K, int mode)
{
    const int nside = mode == QUARTZ_ASYMMETRIC ? 3 : 1;
    const int64_t G = K / kGroupQ;
    return align256(static_cast<size_t>(round_up(N, 16)) * K) + align256(static_cast<size_t>(nside) * G * round_up(N, BN) * 4);
}

void prepared_weights_carve(const void *base, int64_t N, int64_t K, int mode, LinearWorkspace *ws)
{
    uint8_t *p = static_cast<uint8_t *>(const_cast<void *>(base));
    ws->w_op = p;
    ws->w_side = reinterpret_cast<float *>(p + align256(static_cast<size_t>(round_up(N, 16)) * K));
    ws->n_pad = round_up(N, BN);
    ws->nside = mode == QUARTZ_ASYMMETRIC ? 3 : 1;
}

cudaError_t launch_prepare(const quartz_encoded_t *a, const quartz_encoded_t *w, const LinearWorkspace &ws,
                           cudaStream_t s, bool expand, bool w_ready)
{
    const int64_t K = w->K;
    const int64_t upr = K / 16;
    PrepArgs p{};
    p.G = static_cast<int>(K / w->p.group_q);  // scale groups per row
    p.nside = ws.nside;
    if (a)
        p.ex_a = {reinterpret_cast<const uint2 *>(a->codes), a->flags, static_cast<uint4 *>(ws.a_op),
                  a->rows * upr, a->rows * upr, upr, 0, a->p.flag_bits == 4};
    // the weight operand is row-permuted and padded to a multiple of 16 rows
    p.ex_w = {reinterpret_cast<const uint2 *>(w->codes), w->flags, static_cast<uint4 *>(ws.w_op),
              w->rows * upr, round_up(w->rows, 16) * upr, upr, 1, w->p.flag_bits == 4};
    if (a)
        p.sd_a = {reinterpret_cast<const __half *>(a->scales), a->zeros, a->gsum, ws.a_side, a->rows, ws.m_pad, 1};
    p.sd_w = {reinterpret_cast<const __half *>(w->scales), w->zeros, w->gsum, ws.w_side, w->rows, ws.n_pad, 0};
    const int64_t side_chunks = (p.G + kSideGroupsPerThread - 1) / kSideGroupsPerThread;
    const int64_t items[4] = {expand ? p.ex_a.units_pad : 0, expand && !w_ready ? p.ex_w.units_pad : 0,
                              a ? ws.m_pad * side_chunks : 0, w_ready ? 0 : ws.n_pad * side_chunks};
    const int64_t per_block[4] = {2 * kPrepThreads * kExpandPairs, 2 * kPrepThreads * kExpandPairs, kPrepThreads,
                                  kPrepThreads};
    int64_t acc = 0;
    for (int i = 0; i < 4; ++i) {
        acc += (items[i] + per_block[i] - 1) / per_block[i];
        p.block_end[i] = acc;
    }
    if (acc == 0) return cudaSuccess;
    const unsigned blocks = static_cast<unsigned>(acc);
    if (w->p.code_bits == 16) {  // 16-bit stage-1 codes: E5M2 operands
        switch (w->p.group_s) {
            case 8: launch_pdl(prep_kernel<8, true>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
            case 16: launch_pdl(prep_kernel<16, true>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
            case 32: launch_pdl(prep_kernel<32, true>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
            default: launch_pdl(prep_kernel<64, true>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
        }
        return cudaGetLastError();
    }
    switch (w->p.group_s) {
        case 8: launch_pdl(prep_kernel<8, false>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
        case 16: launch_pdl(prep_kernel<16, false>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
        case 32: launch_pdl(prep_kernel<32, false>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
        default: launch_pdl(prep_kernel<64, false>, dim3(blocks), dim3(kPrepThreads), 0, s, p); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_gemm_tcgen05(const LinearWorkspace &ws, int64_t M, int64_t N, int64_t K,
                                int mode, const void *bias, void *y, int y_type,
                                int32_t *partials, int partials_group, int *dev_err,
                                cudaStream_t s, bool per_row, bool wide)
{
    if (M == 0) return cudaSuccess;
    CUtensorMap ta, tw, ty = {};
    if (y_type != QUARTZ_OUT_F32 && !make_output_map(&ty, y, M, N)) return cudaErrorInvalidValue;
    if (!make_operand_map(&ta, ws.a_op, M, K, BM) || !make_operand_map(&tw, ws.w_op, round_up(N, 16), K, BN))
        return cudaErrorInvalidValue;
    GemmArgs args = make_args(ws, M, N, K, bias, y, y_type, partials, partials_group, dev_err);
    args.per_row = per_row ? 1 : 0;
    args.wide = wide ? 1 : 0;
    if (mode == QUARTZ_SYMMETRIC && !partials && !per_row && args.tiles_n <= kRowRasterMaxN) args.raster_m = 1;
    int tail = 0, split = 1, ls = 0;  // the workspace's split must still match this device's grid
    if (mode == QUARTZ_SYMMETRIC && !partials && ws.tail_split > 1 && ws.tail_part)
        tail_split(M, N, K, mode, &tail, &split, &ls);
    if (per_row && split > 1 && !row_split_pays(M, N, K, tail, split, ls)) split = 1;
    if (split > 1 && split == ws.tail_split && tail == ws.tail_tiles && ls == ws.tail_ls) {
        args.split = ws.tail_split;
        args.ls = ls;
        args.tail_tiles = ws.tail_tiles;
        args.full_tiles = args.num_tiles - ws.tail_tiles;
        cudaError_t e = launch_tc_out<QUARTZ_SYMMETRIC>(ta, tw, ty, args, y_type, s);
        if (e != cudaSuccess) return e;
        return per_row ? launch_tail_combine<true>(args, y_type, s) : launch_tail_combine<false>(args, y_type, s);
    }
    if (per_row) return launch_tc_out<QUARTZ_SYMMETRIC>(ta, tw, ty, args, y_type, s);
    return mode == QUARTZ_ASYMMETRIC ? launch_tc_out<QUARTZ_ASYMMETRIC>(ta, tw, ty, args, y_type, s)
                                     : launch_tc_out<QUARTZ_SYMMETRIC>(ta, tw, ty, args, y_type, s);
}

cudaError_t launch_gemm_simt(const LinearWorkspace &ws, int64_t M, int64_t N, int64_t K, int mode,
                             const void *bias, void *y, int y_type, int32_t *partials,
                             int partials_group, cudaStream_t s)
{
    if (M == 0) return cudaSuccess;
    const GemmArgs args = make_args(ws, M, N, K, bias, y, y_type, partials, partials_group, nullptr);
    return mode == QUARTZ_ASYMMETRIC
               ? launch_simt_out<QUARTZ_ASYMMETRIC>(ws, args, static_cast<int>(K), y_type, s)
               : launch_simt_out<QUARTZ_SYMMETRIC>(ws, args, static_cast<int>(K), y_type, s);
}

namespace {
template <int GS, int MODE, int OUT, bool WIDE>
cudaError_t launch_shift(const quartz_encoded_t *a, const quartz_encoded_t *w, const GemmArgs &args,
                         cudaStream_t s)
{
    dim3 grid(static_cast<unsigned>((args.N + 63) / 64), static_cast<unsigned>((args.M + 63) / 64));
    launch_pdl(gemm_shift_kernel<GS, MODE, OUT, WIDE>, dim3(grid), dim3(256), 0, s, 
        reinterpret_cast<const uint32_t *>(a->codes), a->flags, reinterpret_cast<const uint32_t *>(w->codes),
        w->flags, args, static_cast<int>(a->K), a->p.flag_bits == 4, w->p.flag_bits == 4);
    return cudaGetLastError();
}

template <int GS, int MODE, bool WIDE>
cudaError_t launch_shift_out(const quartz_encoded_t *a, const quartz_encoded_t *w, const GemmArgs &args,
                             int y_type, cudaStream_t s)
{
    switch (y_type) {
        case QUARTZ_OUT_F16: return launch_shift<GS, MODE, QUARTZ_OUT_F16, WIDE>(a, w, args, s);
        case QUARTZ_OUT_BF16: return launch_shift<GS, MODE, QUARTZ_OUT_BF16, WIDE>(a, w, args, s);
        default: return launch_shift<GS, MODE, QUARTZ_OUT_F32, WIDE>(a, w, args, s);
    }
}

template <int GS>
cudaError_t launch_shift_mode(const quartz_encoded_t *a, const quartz_encoded_t *w, const GemmArgs &args,
                              int y_type, bool wide, cudaStream_t s)
{
    if (wide) return launch_shift_out<GS, QUARTZ_SYMMETRIC, true>(a, w, args, y_type, s);
    return a->p.mode == QUARTZ_ASYMMETRIC ? launch_shift_out<GS, QUARTZ_ASYMMETRIC, false>(a, w, args, y_type, s)
                                          : launch_shift_out<GS, QUARTZ_SYMMETRIC, false>(a, w, args, y_type, s);
}
}  // namespace

cudaError_t launch_gemm_shift(const LinearWorkspace &ws, const quartz_encoded_t *a, const quartz_encoded_t *w,
                              const void *bias, void *y, int y_type, int32_t *partials, int partials_group,
                              cudaStream_t s, bool wide)
{
    const int64_t M = a->rows, N = w->rows, K = a->K;
    if (M == 0) return cudaSuccess;
    const GemmArgs args = make_args(ws, M, N, K, bias, y, y_type, partials, partials_group, nullptr);
    switch (a->p.group_s) {
        case 8: return launch_shift_mode<8>(a, w, args, y_type, wide, s);
        case 16: return launch_shift_mode<16>(a, w, args, y_type, wide, s);
        case 32: return launch_shift_mode<32>(a, w, args, y_type, wide, s);
        default: return launch_shift_mode<64>(a, w, args, y_type, wide, s);
    }
}

// ---------------------------------------------------------------------------
// failure-detection self-test: a wait that nothing ever satisfies
// ---------------------------------------------------------------------------
namespace {
__global__ void selftest_timeout_kernel(uint64_t limit_ns, int *dev_err)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait_bounded(smem_u32(&bar), 0, &abort_flag, dev_err, limit_ns);
    __syncthreads();
}
}  // namespace

cudaError_t launch_selftest_timeout(int64_t limit_ns, int *dev_err, cudaStream_t s)
{
    selftest_timeout_kernel<<<1, 32, 0, s>>>(static_cast<uint64_t>(limit_ns), dev_err);
    return cudaGetLastError();
}

}  // namespace quartz
