// Tensor-core X stage on sm_103a: tcgen05 MMA with accumulators in tensor memory.
//
// For one channel the correlation matrix is the outer product of the sample vector with
// its conjugate, summed over time (Sec. 4, Fig. 2) -- a Hermitian rank-k update, i.e. a
// dense contraction over the time axis.  A 64-input block is held as 128 operand rows,
// interleaved: row 2m carries the real parts and row 2m+1 the imaginary parts of input m,
// one column per time sample.  With A = block I and B = block J in that form, one MMA per
// 16 samples accumulates D = A B^T (M = N = 128), whose 2 x 2 sub-blocks are
//     D[2i][2j] = sum xr_i xr_j    D[2i][2j+1] = sum xr_i xi_j
//     D[2i+1][2j] = sum xi_i xr_j  D[2i+1][2j+1] = sum xi_i xi_j
// so that Re V_ij = D[2i][2j] + D[2i+1][2j+1] and Im V_ij = D[2i+1][2j] - D[2i][2j+1]:
// x_i conj(x_j) summed over time (Sec. 2).  Rows 2i and 2i+1 sit in adjacent tensor-memory
// lanes, so the epilogue combines them with one lane-pair shuffle.  Only blocks with
// I <= J (the upper triangle of input pairs) are scheduled.
//
// Exactness for integer samples: 4/8-bit values are exact in fp16, their products
// (|p| <= 2^14) are exact, and each D element sums one product per sample, so a chunk of
// at most 1024 samples keeps every partial sum at or below 2^24 in magnitude, where fp32
// holds every integer.  Each D element is converted to int64 before the re/im sums, and
// chunks are flushed to int64; results are bit-exact.  4-bit samples (-8..7) are exact in
// fp8 e4m3 as well: their packed feed converts them to e4m3 operand bytes and issues
// kind::f8f6f4 MMAs (K = 32), with the same fp32 accumulation and chunking.
//
// Float samples (BF16x3): x = h + l with bf16 h, l; MMAs for h h^T, h l^T and l h^T with
// fp32 accumulation.
//
// Two ways to feed the operands:
//   planes  -- the unpack kernel has written fp16 (or bf16 hi/lo; e4m3 for 4-bit samples)
//              sample planes in the interleaved row order; TMA loads 128-row x 128-byte tiles
//              (64 fp16 or 128 e4m3 samples) with 128-byte swizzle straight into the operand
//              ring.
//   raw     -- (4/8-bit samples) TMA loads the packed [time][chan][input] bytes of a
//              64-input x 64-sample block (128 samples for 4-bit e4m3 operands) and eight
//              converter warps turn them into the swizzled operand tiles in shared memory: the
//              unpack/transpose step (Sec. 4) fused into the X kernel, so the samples cross
//              HBM once.  Float samples go the same way (8-byte complex floats in, bf16 hi and lo
//              tiles out) where that is faster than planes (tc_rawf32_pairs, tc_rawf32_odd).
//
// Arrays of several blocks mostly run in pairs of CTAs on 2 x 2 squares of tiles (PAIR below).
//
// CTA roles (one CTA per SM, persistent over work items = (dump, channel, I, J)):
//   warp 0       TMA producer
//   warp 1       tensor-memory allocator and single-thread MMA issuer
//   warps 2..9   epilogue, two warps per tensor-memory lane quarter: tensor memory ->
//                registers -> lane-pair combine -> int64 -> baseline order, staged in shared
//                memory and bulk-copied (single-block arrays: one run per quarter)
//   warps 10..17 (raw only) converters: packed bytes -> fp16 (floats -> bf16 hi/lo) K-major
//                swizzled tiles
// Shared memory is carved at launch: when the array has a single 64-input block every
// item is a diagonal tile (B = A), so stages hold one tile and the rings get deeper.
// Tensor memory holds two accumulators (128 columns each) so the epilogue of one item
// overlaps the MMAs of the next.  Every wait is bounded.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <mutex>
#include <new>

#include "corr_internal.h"
#include "launch.cuh"
#include "sample_convert.cuh"
#include "tc_ptx.cuh"

namespace corr {
namespace {

constexpr int kTileBytes = kBlockRows * kTimeBlock * 2;     // 16 KB: 128 rows x 64 fp16
constexpr uint64_t kWaitLimitNs = 2000000000ull;            // 2 s per wait
constexpr uint64_t kDrainLimitNs = 200000000ull;            // 0.2 s for in-flight work at exit
constexpr int kMaxOpStages = 16;
constexpr int kMaxRawStages = 32;
constexpr int kBarBytes = 8 * (3 * kMaxOpStages + 2 * kMaxRawStages + 13) + 16;
constexpr int kSmemBudget = 227 * 1024 - kBarBytes - 1024;  // ring space after barriers and alignment
// Staged epilogue: a warp's 16 rows of 64 baselines (16 bytes each), row pitch 65 x 16 B so
// that the 16-byte stores of a quarter-warp fall in 8 distinct bank groups.
constexpr int kStageRowBytes = 65 * 16;
constexpr int kStageBytes = 4 * 16 * kStageRowBytes;
// Dump mode stages 8-byte float pairs: rows of 66 slots (16-byte aligned pitch), element j of a
// row at slot (j - J0) + s, with s the parity of the row's first global element index, so a
// slot and its destination are 16-byte aligned together and the bulk copies stay aligned.
constexpr int kStageRowBytesF = 66 * 8;
constexpr int kStageWarpD = 16 * kStageRowBytesF + kBlockInputs * 8;   // dump mode: and the J block's phasors
// Single-block jobs: an item's tile holds whole channels, so the baselines of a warp's 16 rows are
// one contiguous run of the output.  The warp packs its rows there without gaps and issues one bulk
// copy (or one bulk add) for the run.  Quarter q's rows need at most sum of (64 - u), u = 16 q ..
// 16 q + 15, slots whatever the array's size and packing, so quarter q starts at slot kTriSlot(q)
// (float pairs: one more 16-byte unit per warp, for a run that starts at an odd element).
__host__ __device__ constexpr int tri_slot(int q) { return 64 * 16 * q - 8 * q * (16 * q - 1); }
constexpr int kTriBytes = tri_slot(4) * 16;                 // int64 pairs
constexpr int kTriPhasors = tri_slot(4) * 8 + 4 * 16;       // float pairs, then 64 phasors per warp
constexpr int kTriBytesF = kTriPhasors + 4 * kBlockInputs * 8;
static_assert(tri_slot(4) == 2080 && tri_slot(1) * 16 <= 16 * kStageRowBytes, "staging area");

enum Mode : int { kPlanesF16 = 0, kPlanesBF16x3 = 1, kRaw8 = 2, kRaw4 = 3, kRawF32 = 4, kRaw4F8 = 5, kPlanesF8 = 6 };

template <int MODE>
struct Cfg {
    // kRawF32: float32 complex samples loaded by TMA and split into bf16 hi + lo by the converter
    // warps (the BF16x3 products of the planes path, without the planes in memory)
    static constexpr bool kFloat = MODE == kRawF32;
    // kRaw4F8: 4-bit samples converted to e4m3 operand bytes (kind::f8f6f4): a 128-byte operand
    // row then holds 128 samples, so a stage covers 128 samples in four K = 32 MMAs.  kPlanesF8:
    // the same operands read from e4m3 planes.
    static constexpr bool kF8 = MODE == kRaw4F8 || MODE == kPlanesF8;
    static constexpr bool kRaw = (MODE == kRaw8 || MODE == kRaw4 || kFloat || MODE == kRaw4F8);
    static constexpr bool kBits8 = MODE == kRaw8;
    static constexpr bool kSplit = (MODE == kPlanesBF16x3 || kFloat);
    static constexpr int kEpiWarps = 8;     // two per tensor-memory lane quarter
    static constexpr int kConvWarps = 8;
    // groups of converter warps, each taking every other stage: the e4m3 and float conversions gain (4-bit
    // 64 inputs 126 -> 116 us, 128 inputs x 2048 samples 106 -> 86; BF16x3 109 -> 105), the 8-bit one,
    // whose loads and stores crowd the shared-memory port, does not on single blocks (129 -> 136; not
    // measured in pairs)
    static constexpr int kConvGroups = kF8 || kFloat ? 2 : 1;
    static constexpr int kGroupWarps = kConvWarps / kConvGroups;
    static constexpr int kThreads = 64 + 32 * kEpiWarps + (kRaw ? 32 * kConvWarps : 0);
    static constexpr int kBps = kFloat ? 8 : (kBits8 ? 2 : 1);            // packed bytes per sample
    static constexpr int kStageT = kF8 ? 2 * kTimeBlock : kTimeBlock;    // samples per stage
    static constexpr int kRawTileBytes = kRaw ? kStageT * kBlockInputs * kBps : 0;
    // x coordinate of a 64-input block in the raw tensor map: bytes, or 8-byte complex floats
    static constexpr int kMapX = kFloat ? kBlockInputs : kBlockInputs * kBps;
    static constexpr int kTilesPerOperand = kSplit ? 2 : 1;               // hi (+ lo)
};

constexpr int kMaxJobs = kMaxJobsPerLaunch;   // jobs one launch packs (kernel-parameter space holds their maps)

// One correlation job of a launch: its TMA map (packed bytes, or fp16/bf16 hi planes),
// sizes, output and the flat index of its first work item.
struct TcJob {
    CUtensorMap map;
    CUtensorMap map_wide;   // plane path, wide items: boxes of two blocks (256 rows)
    void* vis;
    int64_t item_begin;  // first flat item of this job
    int n_inputs;
    int n_chan;
    int nb;              // 64-input blocks
    int kp;              // samples per dump rounded up to 64
    int n_tiles;         // work items per channel group: nb (nb + 1) / 2 tiles, or S(nb) wide items
    int tw;              // 2: wide items (block I against blocks J0, J0 + 1, one N = 256 MMA); 1: tiles
    int cpi;             // tiles of adjacent channels per work item (2: single-block arrays)
    int n_groups;        // item groups per dump = ceil(ceil(n_chan / pack) / cpi)
    int pack;            // channels side by side in one 64-input tile (arrays of at most 32 inputs), else 1
    int x_step, y_step;  // TMA coordinates of channel tile k: x = I kMapX + k x_step, y = k y_step
    int pair_off;        // packed feed, cpi = 2: bytes from the first to the second tile in a sample row
    uint32_t idesc;      // instruction descriptor of a tile's MMA (N = the columns the tile uses)
    int chunk_kb;        // stages (64 samples; 128 with e4m3 operands) per exactly-flushed chunk
    // division by n_tiles and n_groups as q = (umulhi(n, m) + n) >> s (n < 2^31; Granlund and
    // Montgomery, division by invariant integers using multiplication)
    uint32_t tiles_m, groups_m;
    int tiles_s, groups_s;
    // 1: every D element of a chunk is at most 2^23 in magnitude, so rr + ii and ir - ri are
    // exact in fp32 and each needs one conversion (4-bit samples; 8-bit with <= 512 samples)
    int f32_combine;
    // 1: dump mode (Fig. 1, Sec. 2) -- the epilogue writes float32 V / n_accum rotated by
    // phasor_i conj(phasor_j) (phasor [n_chan][n_inputs] or nullptr: no rotation) instead of
    // the exact int64 sums; a dump must fit one exact chunk and is never accumulated
    int out_mode;
    const float2* phasor;
    float inv_n;
};

template <int MAXJ>
struct TcLaunch {
    CUtensorMap map_lo;  // BF16x3 lo planes (single-job launches only)
    int n_jobs;
    int64_t n_items;     // sum over jobs of n_dumps * n_groups * n_tiles
    int accumulate;
    int* status;
    uint32_t tmem_cols;  // 256 or 512 (two accumulator sets of up to 2 x 128 columns)
    // shared-memory carve-up (bytes; ring base is 1024-aligned)
    int op_stages;
    int op_stage_bytes;  // operand tiles of one stage: A (+ B, or a second channel) (x2 for hi/lo)
    int b_offset;        // offset of the B tile(s) inside an op stage (0: B = A)
    int raw_stages;
    int raw_stage_bytes;
    int raw_offset;      // start of the raw ring
    int bar_offset;      // start of the barriers
    uint64_t wait_limit_ns;  // bound of every mbarrier wait
    int64_t stall_item;  // self-test: the producer withholds the first stage of this item (-1: none)
    int staged;          // 1: the staging area holds tile rows (jobs of several blocks), 0: packed runs only
    int staging_offset;  // start of the staging area
    TcJob jobs[MAXJ];
};

// Work-item coordinates.  Items are visited in increasing order by every role, so the job
// index only moves forward.
struct ItemCtx {
    int j;
    int I, J;            // J: the first B block (wide items: J and J + 1 when nsub = 2)
    bool same;
    bool wide;
    int nsub;            // accumulators of the item: channels (cpi) or B blocks (wide)
    int64_t d;           // dump within the job
    int c0;              // first channel of the item
};

// Tiles are numbered row by row over I <= J: row I starts at off(I) = I nb - I (I - 1) / 2.
// The row is the larger root bound of off(I) <= tile, taken in float and corrected exactly.
__device__ __forceinline__ void tile_coords(int tile, int nb, int& I, int& J) {
    const int b = 2 * nb + 1;
    int i = (int)(((float)b - sqrtf((float)(b * b - 8 * tile))) * 0.5f);
    i = max(0, min(i, nb - 1));
    while (i > 0 && i * nb - i * (i - 1) / 2 > tile) --i;
    while (i + 1 < nb && (i + 1) * nb - (i + 1) * i / 2 <= tile) ++i;
    I = i;
    J = i + (tile - (i * nb - i * (i - 1) / 2));
}

// Wide items: row I holds the items J0 = I, I + 2, ... < nb, so the rows of lengths nb .. 1
// start at S(nb) - S(nb - I) with S(m) = floor((m + 1) / 2) floor((m + 2) / 2).  The row is
// the smallest m = nb - I with S(m) >= S(nb) - item, from S(m) ~ (m + 1.5)^2 / 4 in float and
// corrected exactly.
__device__ __forceinline__ int pairs_upto(int m) { return ((m + 1) >> 1) * ((m + 2) >> 1); }

__device__ __forceinline__ void wide_coords(int tile, int nb, int& I, int& J0) {
    const int R = pairs_upto(nb) - tile;
    int m = (int)(2.0f * sqrtf((float)R) - 1.5f);
    m = max(0, min(m, nb));
    while (m > 0 && pairs_upto(m - 1) >= R) --m;
    while (pairs_upto(m) < R) ++m;
    I = nb - m;
    J0 = I + 2 * (tile - (pairs_upto(nb) - pairs_upto(m)));
}

__device__ __forceinline__ uint32_t fast_div(uint32_t n, uint32_t m, int s) {
    return (uint32_t)(((uint64_t)__umulhi(n, m) + n) >> s);
}

// PAIR: tiles are the upper triangle of block pairs (a <= b); CTA `rank` takes block I = 2 a + rank
// against blocks J = 2 b and J + 1.
template <int MAXJ, bool PAIR>
__device__ __forceinline__ void decode_item(const TcLaunch<MAXJ>& L, int64_t item, int& j, ItemCtx& it, int rank) {
    // single-job launches: a constant index, so the job's fields are plain parameter operands
    if constexpr (MAXJ == 1) j = 0;
    else
        while (j + 1 < L.n_jobs && item >= L.jobs[j + 1].item_begin) ++j;
    const TcJob& jb = L.jobs[j];
    const uint32_t local = (uint32_t)(item - jb.item_begin);   // < 2^31 per job (host-checked)
    const uint32_t dg = fast_div(local, jb.tiles_m, jb.tiles_s);
    const int tile = (int)(local - dg * (uint32_t)jb.n_tiles);
    const uint32_t d = fast_div(dg, jb.groups_m, jb.groups_s);
    it.j = j;
    it.d = d;
    it.c0 = (int)(dg - d * (uint32_t)jb.n_groups) * jb.cpi;
    it.wide = PAIR || jb.tw == 2;
    if constexpr (PAIR) {
        int a, b;
        tile_coords(tile, (jb.nb + 1) >> 1, a, b);
        it.I = 2 * a + rank;
        it.J = 2 * b;
        it.nsub = 2;
        it.same = a == b;
        return;
    }
    if (it.wide) {
        wide_coords(tile, jb.nb, it.I, it.J);
        it.nsub = min(2, jb.nb - it.J);
    } else {
        tile_coords(tile, jb.nb, it.I, it.J);
        it.nsub = jb.cpi;
    }
    it.same = it.I == it.J;
}

__device__ __forceinline__ void record_error(int* status, volatile int* abort, int code, int detail) {
    *abort = 1;
    if (atomicCAS(status, 0, code) == 0) status[1] = detail;
}

using conv::lane_selector;
using conv::pair_to_half2;

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

__device__ __forceinline__ void st_shared_u64(uint32_t addr, uint64_t a) {
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(a) : "memory");
}

__device__ __forceinline__ void st_shared_f32(uint32_t addr, float a) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(a) : "memory");
}

__device__ __forceinline__ void st_shared_v2_f32(uint32_t addr, float a, float b) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}

__device__ __forceinline__ float2 ld_shared_v2_f32(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// Per-thread constants of the converters: for each of the 4 output rows a lane writes, the
// byte-lane selector, the row's swizzle-atom offset and (row & 7) << 4.  They depend only on
// the lane, so they are computed once per kernel.
struct ConvLane {
    uint32_t sel[4];
    uint32_t rowoff[4];
    uint32_t r7x16[4];
    // 4-bit: the lane writes its two rows of an input in the order (re, im) or (im, re): the
    // nibble shift of the first row's values and the byte offset of the second row from the first
    uint32_t first_shift;
    int32_t second_delta;
};

// 8-bit: lane l takes inputs 2l, 2l+1; byte lane k of a loaded word is re(2l), im(2l),
// re(2l+1), im(2l+1) = operand row 4l + k.  At step kk the lane writes k = (kk + l/2) & 3,
// so the rows of a quarter-warp (l = 8a .. 8a+7) fall in 8 distinct swizzle chunks: even l
// give (row & 7) in 0..3, odd l in 4..7, and the 16-byte stores never share a bank.
__device__ __forceinline__ ConvLane conv_lane8(int l) {
    ConvLane c;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const int k = (kk + (l >> 1)) & 3;
        const int row = 4 * l + k;
        c.sel[kk] = lane_selector(k);
        c.rowoff[kk] = (uint32_t)((row >> 3) * 1024 + (row & 7) * 128);
        c.r7x16[kk] = (uint32_t)((row & 7) << 4);
    }
    c.first_shift = 0;
    c.second_delta = 0;
    return c;
}

// 4-bit: lane l takes inputs 4m .. 4m+3 (m = l & 15); at step kk input 4m + k with
// k = (kk + m/2) & 3, and writes rows 2(4m + k) (re) and 2(4m + k) + 1 (im), the im row first
// when m is odd.  A quarter-warp's first rows then have (row & 7) = 2k + (m & 1), eight distinct
// values, and so do its second rows: each 16-byte store of the quarter-warp lands in its own
// swizzle chunk, free of bank conflicts.
__device__ __forceinline__ ConvLane conv_lane4(int l) {
    ConvLane c;
    const int m = l & 15;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const int k = (kk + (m >> 1)) & 3;
        const int row = 2 * (4 * m + k) + (m & 1);
        c.sel[kk] = lane_selector(k);
        c.rowoff[kk] = (uint32_t)((row >> 3) * 1024 + (row & 7) * 128);
        c.r7x16[kk] = (uint32_t)((row & 7) << 4);
    }
    c.first_shift = (m & 1) ? 0u : 4u;           // re is the high nibble, im the low one
    c.second_delta = (m & 1) ? -128 : 128;
    return c;
}

// One warp-sized slice of a packed 8-bit tile -> interleaved fp16 operand tile.  Lane l holds
// w[e] = bytes 4l .. 4l+3 (re, im of inputs 2l, 2l+1) of sample 8q + e; the slice is the 8
// samples of group q, written as four 16-byte swizzled row chunks.
__device__ __forceinline__ void convert_words8(const uint32_t (&w)[8], uint32_t dst, int q, const ConvLane& cl) {
    const __half2 bias = conv::bias8();
    const uint32_t flip = conv::kFlip8;   // exponent bytes 0x64, sign bit of each sample byte flipped
    const uint32_t q16 = (uint32_t)q << 4;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const uint32_t sel = cl.sel[kk];
        st_shared_v4(dst + cl.rowoff[kk] + (q16 ^ cl.r7x16[kk]), pair_to_half2(w[0], w[1], sel, flip, bias),
                     pair_to_half2(w[2], w[3], sel, flip, bias), pair_to_half2(w[4], w[5], sel, flip, bias),
                     pair_to_half2(w[6], w[7], sel, flip, bias));
    }
}

// Packed 4-bit words (high nibble re, low nibble im): lane l holds w[e] = inputs 4m .. 4m+3
// (m = l & 15) of the 8 samples of group q; writes the 16-byte chunk q of each of its 8 rows.
__device__ __forceinline__ void convert_words4(const uint32_t (&w)[8], uint32_t dst, int q, const ConvLane& cl) {
    const __half2 bias = conv::bias4();
    const uint32_t flip = conv::kFlip4;   // exponent bytes 0x64, sign bit of each 4-bit sample flipped
    uint32_t a[8], b[8];                  // nibbles of the first and the second row, one per byte
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        a[e] = (w[e] >> cl.first_shift) & 0x0F0F0F0Fu;
        b[e] = (w[e] >> (4u - cl.first_shift)) & 0x0F0F0F0Fu;
    }
    const uint32_t q16 = (uint32_t)q << 4;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const uint32_t sel = cl.sel[kk];
        const uint32_t at = dst + cl.rowoff[kk];
        st_shared_v4(at + (q16 ^ cl.r7x16[kk]), pair_to_half2(a[0], a[1], sel, flip, bias),
                     pair_to_half2(a[2], a[3], sel, flip, bias), pair_to_half2(a[4], a[5], sel, flip, bias),
                     pair_to_half2(a[6], a[7], sel, flip, bias));
        // the other row of the input: 128 bytes away, (row & 7) differing in its lowest bit
        st_shared_v4(at + (uint32_t)cl.second_delta + (q16 ^ (cl.r7x16[kk] ^ 16u)),
                     pair_to_half2(b[0], b[1], sel, flip, bias), pair_to_half2(b[2], b[3], sel, flip, bias),
                     pair_to_half2(b[4], b[5], sel, flip, bias), pair_to_half2(b[6], b[7], sel, flip, bias));
    }
}

// The e4m3 converter's lane constants: input 4m + k at step kk with k = (kk + m) & 3, its re row
// 2(4m + k) first and the im row after it.  Its stores are half as many as the fp16 ones and
// conflict in pairs; the conflict-free order of conv_lane4 and its loads (permuted row addresses,
// a lane-dependent order of the two rows) measured slower here (99 against 97 us on a 4-bit
// stream of 64 inputs x 768 channels x 4 dumps, 75 against 71 on 128 x 512 x 2048).
__device__ __forceinline__ ConvLane conv_lane4_f8(int l) {
    ConvLane c;
    const int m = l & 15;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const int k = (kk + m) & 3;
        const int row = 2 * (4 * m + k);
        c.sel[kk] = conv::gather_selector(k);
        c.rowoff[kk] = (uint32_t)((row >> 3) * 1024 + (row & 7) * 128);
        c.r7x16[kk] = (uint32_t)((row & 7) << 4);
    }
    c.first_shift = 4;
    c.second_delta = 128;
    return c;
}

// Packed 4-bit words -> e4m3 operand tile (128 samples per 128-byte row): lane l holds
// w[e] = inputs 4m .. 4m+3 (m = l & 15) of sample 16c + e, e = 0..15, and writes, for the re
// and im rows of each of its four inputs, the row's 16-byte chunk c (16 samples).
__device__ __forceinline__ void convert_words4_f8(const uint32_t (&w)[16], uint32_t dst, int c, const ConvLane& cl) {
    const uint32_t c16 = (uint32_t)c << 4;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const uint32_t sel = cl.sel[kk];
        const uint32_t at = dst + cl.rowoff[kk];
        uint32_t r[4], m[4];
#pragma unroll
        for (int o = 0; o < 4; ++o)
            conv::e4m3_of_nibbles(conv::gather4(w[4 * o], w[4 * o + 1], w[4 * o + 2], w[4 * o + 3], sel), r[o], m[o]);
        st_shared_v4(at + (c16 ^ cl.r7x16[kk]), r[0], r[1], r[2], r[3]);
        st_shared_v4(at + 128u + (c16 ^ (cl.r7x16[kk] + 16u)), m[0], m[1], m[2], m[3]);   // the im row
    }
}

// One warp-sized slice of a float32 tile -> bf16 hi and lo operand tiles (hi = bf16(x),
// lo = bf16(x - hi), both rounded to nearest, as the planes path splits).  A raw sample row
// holds 128 words, (re, im) of 64 inputs, so word w of a row is operand row w; lane l takes
// rows l + 32 kk (kk = 0..3) of samples 8q .. 8q + 7 and writes each row's 16-byte chunk q of
// the hi tile and of the lo tile (kTileBytes further).  A quarter-warp's rows differ in
// (row & 7), so its swizzled chunks fall in distinct banks.
__device__ __forceinline__ uint32_t bf16x2_bits(float a, float b) {   // a in the low half
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t bf16_pair(float a, float b, uint32_t& lo) {
    const uint32_t h = bf16x2_bits(a, b);   // one conversion for both, and again for what it dropped
    lo = bf16x2_bits(a - __uint_as_float(h << 16), b - __uint_as_float(h & 0xFFFF0000u));
    return h;
}

__device__ __forceinline__ void convert_slice_f32(uint32_t raw_tile, uint32_t dst_hi, int q, int lane) {
    constexpr uint32_t kRowBytes = kBlockInputs * 8;   // one sample row of the raw tile
    const uint32_t src = raw_tile + (uint32_t)q * 8u * kRowBytes + 4u * (uint32_t)lane;
    const uint32_t q16 = (uint32_t)q << 4;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const uint32_t row = (uint32_t)lane + 32u * kk;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(ld_shared_u32(src + (uint32_t)e * kRowBytes + 128u * kk));
        uint32_t h[4], l[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) h[p] = bf16_pair(v[2 * p], v[2 * p + 1], l[p]);
        const uint32_t at = dst_hi + (row >> 3) * 1024u + (row & 7u) * 128u + (q16 ^ ((row & 7u) << 4));
        st_shared_v4(at, h[0], h[1], h[2], h[3]);
        st_shared_v4(at + (uint32_t)kTileBytes, l[0], l[1], l[2], l[3]);
    }
}

__device__ __forceinline__ void bulk_store(void* gdst, uint32_t ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(ssrc), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_add_u64(void* gdst, uint32_t ssrc, uint32_t bytes) {
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.u64 [%0], [%1], %2;" ::"l"(gdst), "r"(ssrc),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void fence_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

// One K step of a stage: 16 fp16 samples (kind::f16) or 32 e4m3 samples (kind::f8f6f4); either
// way 32 bytes of each 128-byte operand row, so the descriptors advance alike.
template <bool F8>
__device__ __forceinline__ void mma_op(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                       uint32_t acc) {
    if constexpr (F8) ptx::mma_f8_lo(d, a_lo, b_lo, hi, idesc, acc);
    else ptx::mma_f16_lo(d, a_lo, b_lo, hi, idesc, acc);
}

// DUMP: the epilogue writes the dump-mode float pairs (out_mode = 1 jobs) instead of int64
// sums; a separate instantiation so the exact-output kernels keep their registers.
//
// PAIR (arrays of several blocks): two CTAs of a cluster work on a 2 x 2 square of tiles, blocks
// 2 a, 2 a + 1 against 2 b, 2 b + 1, with one M = 256, N = 256 MMA (cta_group::2) per K step: each
// CTA holds its own block's 128 rows of A and half of B, so it loads (or converts) two blocks for
// its two tiles -- one, on the diagonal -- where single tiles take two per tile, and its shared
// memory feeds 8 KB instead of 16 KB of operands per tile and K step.  The even CTA's MMA thread
// issues for both; converters and epilogue warps of the odd CTA arrive on its barriers, and its
// commits arrive in both.  On planes the odd CTA's MMA thread relays "stage loaded".  Float
// pairs have 64 KB of operands (two blocks, hi and lo) in a stage off the diagonal: two such stages
// and two raw slots of one 32 KB tile each fit, and the converter groups take a tile each.
template <int MODE, int MAXJ, bool DUMP, bool PAIR>
__global__ void __launch_bounds__(Cfg<MODE>::kThreads, 1) xeng_tc_kernel(const __grid_constant__ TcLaunch<MAXJ> prm) {
    using C = Cfg<MODE>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ring = smem;
    uint8_t* rawring = smem + prm.raw_offset;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + prm.bar_offset);
    const int OS = prm.op_stages, RS = prm.raw_stages;
    // barriers: op_full[OS], op_empty[OS], raw_full[RS], raw_empty[RS], acc_full[2], acc_empty[2], drain,
    // stage_free[4], stage_full[4] (the two epilogue warps of a lane quarter), peer_full[OS] (pairs)
    const uint32_t bar_op_full = ptx::smem_u32(bars);
    const uint32_t bar_op_empty = bar_op_full + 8 * OS;
    const uint32_t bar_raw_full = bar_op_empty + 8 * OS;
    const uint32_t bar_raw_empty = bar_raw_full + 8 * RS;
    const uint32_t bar_acc_full = bar_raw_empty + 8 * RS;
    const uint32_t bar_acc_empty = bar_acc_full + 16;
    const uint32_t bar_drain = bar_acc_empty + 16;
    const uint32_t bar_stage_free = bar_drain + 8;
    const uint32_t bar_stage_full = bar_stage_free + 32;
    const uint32_t bar_peer_full = bar_stage_full + 32;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3 * OS + 2 * RS + 13);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kCtas = PAIR ? 2 : 1;
    const int rank = PAIR ? (int)ptx::cluster_rank() : 0;
    const int64_t item0 = blockIdx.x / kCtas, item_step = gridDim.x / kCtas;   // the CTA's (pair's) items

    if (threadIdx.x == 0) {
        for (int s = 0; s < OS; ++s) {
            ptx::mbar_init(bar_op_full + 8 * s, C::kRaw ? C::kGroupWarps * kCtas * (C::kFloat && PAIR ? 2 : 1) : 1);
            ptx::mbar_init(bar_op_empty + 8 * s, 1);
            ptx::mbar_init(bar_peer_full + 8 * s, 1);
        }
        for (int s = 0; s < RS; ++s) {
            ptx::mbar_init(bar_raw_full + 8 * s, 1);
            ptx::mbar_init(bar_raw_empty + 8 * s, C::kGroupWarps);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(bar_acc_full + 8 * b, 1);
            ptx::mbar_init(bar_acc_empty + 8 * b, C::kEpiWarps * kCtas);
        }
        ptx::mbar_init(bar_drain, 1);
        for (int b = 0; b < 4; ++b) {
            ptx::mbar_init(bar_stage_free + 8 * b, 2);
            ptx::mbar_init(bar_stage_full + 8 * b, 2);
        }
        *abort_flag = 0;
        ptx::fence_mbar_init();
        for (int j = 0; j < prm.n_jobs; ++j) {
            ptx::prefetch_tensormap(&prm.jobs[j].map);
            if (!C::kRaw && prm.jobs[j].tw == 2) ptx::prefetch_tensormap(&prm.jobs[j].map_wide);
        }
        if (C::kSplit && !C::kRaw) ptx::prefetch_tensormap(&prm.map_lo);
    }
    if (warp == 1) {
        ptx::tmem_alloc<PAIR>(ptx::smem_u32(tmem_slot), prm.tmem_cols);
        ptx::tmem_relinquish<PAIR>();
    }
    ptx::tc_fence_before();
    if constexpr (PAIR) {
        __syncwarp();
        ptx::cluster_sync();   // the other CTA's barriers exist before anything arrives on them
    } else {
        __syncthreads();
    }
    ptx::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_wait();   // samples and outputs may be the preceding kernel's
    grid_release();


    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            const int S = C::kRaw ? RS : OS;
            const uint32_t bar_full = C::kRaw ? bar_raw_full : bar_op_full;
            const uint32_t bar_empty = C::kRaw ? bar_raw_empty : bar_op_empty;
            int s = 0;
            uint32_t ph = 0;
            int64_t n_slots = 0;       // ring slots used so far (issued or withheld)
            int64_t withheld = -1;     // the slot the self-test withheld
            bool ok = true;
            int jc = 0;
            for (int64_t item = item0; ok && item < prm.n_items; item += item_step) {
                ItemCtx it;
                decode_item<MAXJ, PAIR>(prm, item, jc, it, rank);
                const TcJob& jb = prm.jobs[MAXJ == 1 ? 0 : it.j];
                const int I = it.I, J = it.J;
                const bool same = it.same;
                const int nkb = jb.kp / C::kStageT;
                // float pairs: the two blocks of a square off the diagonal take a raw slot each
                const int units = C::kFloat && PAIR && !same ? 2 : 1;
                for (int ku = 0; ku < nkb * units; ++ku) {
                    const int kb = units == 2 ? ku >> 1 : ku;
                    if (!ptx::mbar_wait_bounded(bar_empty + 8 * s, ph ^ 1u, abort_flag, prm.wait_limit_ns)) {
                        record_error(prm.status, abort_flag, kDevTimeoutEmpty, kb);
                        ok = false;
                        break;
                    }
                    const uint32_t fb = bar_full + 8 * s;
                    if (item == prm.stall_item && ku == 0) {
                        // self-test of the bounded waits: nothing will complete this stage
                        withheld = n_slots++;
                        if (++s == S) {
                            s = 0;
                            ph ^= 1u;
                        }
                        continue;
                    }
                    if constexpr (C::kRaw) {
                        const uint32_t st = ptx::smem_u32(rawring + s * prm.raw_stage_bytes);
                        if constexpr (C::kFloat && PAIR) {
                            const int block = units == 2 && (ku & 1) ? J + rank : I;
                            ptx::mbar_expect_tx(fb, (uint32_t)C::kRawTileBytes);
                            tma_load_4d(st, &jb.map, block * C::kMapX, it.c0, kb * C::kStageT, (int)it.d, fb);
                        } else {
                        // one box covers cpi adjacent channels (cpi x 64 inputs per sample row)
                        ptx::mbar_expect_tx(fb, (same ? (uint32_t)jb.cpi : 2u) * (uint32_t)C::kRawTileBytes);
                        tma_load_4d(st, &jb.map, I * C::kMapX + it.c0 * jb.x_step, it.c0 * jb.y_step,
                                    kb * C::kStageT, (int)it.d, fb);
                        if (!same)
                            tma_load_4d(st + C::kRawTileBytes, &jb.map, (J + rank) * C::kMapX, it.c0, kb * C::kStageT,
                                        (int)it.d, fb);
                        }
                    } else {
                        const uint32_t st = ptx::smem_u32(ring + s * prm.op_stage_bytes);
                        const int64_t dc = it.d * jb.n_chan + it.c0;   // planes: one channel per item
                        const int rowA = (int)((dc * jb.nb + I) * kBlockRows);
                        const int rowB = (int)((dc * jb.nb + J + rank) * kBlockRows);
                        const uint32_t bo = (uint32_t)prm.b_offset;
                        if (!PAIR && it.wide) {
                            // B = blocks J (, J + 1) in one box at b_offset; A = block I, or on the
                            // diagonal the first half of the B box itself
                            const uint32_t nB = (uint32_t)it.nsub;
                            ptx::mbar_expect_tx(fb, (nB + (same ? 0u : 1u)) * (uint32_t)kTileBytes);
                            if (!same) ptx::tma_load_2d(st, &jb.map, kb * C::kStageT, rowA, fb);
                            ptx::tma_load_2d(st + bo, nB == 2 ? &jb.map_wide : &jb.map, kb * C::kStageT, rowB, fb);
                        } else {
                            ptx::mbar_expect_tx(fb, (same ? 1u : 2u) * (uint32_t)(C::kTilesPerOperand * kTileBytes));
                            ptx::tma_load_2d(st, &jb.map, kb * C::kStageT, rowA, fb);
                            if (!same) ptx::tma_load_2d(st + bo, &jb.map, kb * C::kStageT, rowB, fb);
                            if (C::kSplit) {
                                ptx::tma_load_2d(st + kTileBytes, &prm.map_lo, kb * C::kStageT, rowA, fb);
                                if (!same) ptx::tma_load_2d(st + bo + kTileBytes, &prm.map_lo, kb * C::kStageT, rowB, fb);
                            }
                        }
                    }
                    ++n_slots;
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            // no copy of ours may still be landing in shared memory when the CTA exits:
            // wait for the last phase issued on each stage (even after an abort)
            if (!ok || *abort_flag) {
                const int64_t n_last = n_slots < S ? n_slots : S;
                for (int64_t k = 0; k < n_last; ++k) {
                    const int64_t idx = n_slots - 1 - k;        // k-th most recent slot
                    if (idx == withheld) continue;              // nothing was issued there
                    const int st = (int)(idx % S);
                    const uint32_t par = (uint32_t)((idx / S) & 1);
                    ptx::mbar_wait_drain(bar_full + 8 * st, par, kDrainLimitNs);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (PAIR && rank != 0) {
            // planes: tell the issuing CTA which of this CTA's stages have landed
            if (!C::kRaw && lane == 0) {
                const uint32_t peer = ptx::map_shared(bar_peer_full, 0);
                int s = 0;
                uint32_t ph = 0;
                bool ok = true;
                int jc = 0;
                for (int64_t item = item0; ok && item < prm.n_items; item += item_step) {
                    ItemCtx it;
                    decode_item<MAXJ, PAIR>(prm, item, jc, it, rank);
                    const int nkb = prm.jobs[MAXJ == 1 ? 0 : it.j].kp / C::kStageT;
                    for (int kb = 0; kb < nkb; ++kb) {
                        if (!ptx::mbar_wait_bounded(bar_op_full + 8 * s, ph, abort_flag, prm.wait_limit_ns)) {
                            record_error(prm.status, abort_flag, kDevTimeoutFull, kb);
                            ok = false;
                            break;
                        }
                        ptx::mbar_arrive_cluster(peer + 8 * s);
                        if (++s == OS) {
                            s = 0;
                            ph ^= 1u;
                        }
                    }
                }
            }
        } else if (lane == 0) {
            constexpr uint32_t idesc_wide = ptx::idesc_f16(PAIR ? 256 : 128, 256, C::kSplit);
            auto wait = [&](uint32_t bar, uint32_t parity) {
                return ptx::mbar_wait_bounded(bar, parity, abort_flag, prm.wait_limit_ns);
            };
            auto commit = [&](uint32_t bar) {
                if constexpr (PAIR) ptx::mma_commit_pair(bar);
                else ptx::mma_commit(bar);
            };
            constexpr uint32_t desc_hi = ptx::sw128_desc_hi();
            const uint32_t desc_lo_ring = ptx::sw128_desc_lo(ptx::smem_u32(ring));
            const uint32_t stage16 = (uint32_t)prm.op_stage_bytes >> 4;
            const uint32_t boff16 = (uint32_t)prm.b_offset >> 4;
            int s = 0;
            uint32_t ph = 0;
            int abuf = 0;
            uint32_t aph = 0;
            bool ok = true;
            bool any = false;
            int jc = 0;
            for (int64_t item = item0; ok && item < prm.n_items; item += item_step) {
                ItemCtx it;
                decode_item<MAXJ, PAIR>(prm, item, jc, it, rank);
                const TcJob& jb = prm.jobs[MAXJ == 1 ? 0 : it.j];
                const uint32_t idesc = jb.idesc;
                const bool same = it.same;
                const int nkb = jb.kp / C::kStageT;
                for (int kb0 = 0; ok && kb0 < nkb; kb0 += jb.chunk_kb) {
                    const int kb1 = min(nkb, kb0 + jb.chunk_kb);
                    if (!wait(bar_acc_empty + 8 * abuf, aph ^ 1u)) {
                        record_error(prm.status, abort_flag, kDevTimeoutAccEmpty, kb0);
                        ok = false;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t dset = tmem_base + (uint32_t)(abuf * (int)(prm.tmem_cols / 2));
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!wait(bar_op_full + 8 * s, ph) ||
                            (PAIR && !C::kRaw && !wait(bar_peer_full + 8 * s, ph))) {
                            record_error(prm.status, abort_flag, kDevTimeoutFull, kb);
                            ok = false;
                            break;
                        }
                        ptx::tc_fence_after();
                        // descriptor low words, in 16-byte units: the stage, then +1024 per
                        // 16 KB tile, +2 per 16-sample step along the swizzled rows
                        const uint32_t a0 = desc_lo_ring + (uint32_t)s * stage16;
                        const uint32_t acc0 = kb > kb0 ? 1u : 0u;
                        if constexpr (PAIR) {
                            const uint32_t b0 = same ? a0 : a0 + boff16;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t ak = a0 + 2u * k, bk = b0 + 2u * k;
                                ptx::mma_pair_lo<C::kF8>(dset, ak, bk, desc_hi, idesc_wide, (k > 0) | acc0);
                                if constexpr (C::kSplit) {
                                    ptx::mma_pair_lo<false>(dset, ak, bk + 1024u, desc_hi, idesc_wide, 1u);   // h_i l_j
                                    ptx::mma_pair_lo<false>(dset, ak + 1024u, bk, desc_hi, idesc_wide, 1u);   // l_i h_j
                                }
                            }
                        } else if (!C::kRaw && !C::kSplit && it.wide) {
                            // one M = 128, N = 256 MMA covers tiles (I, J) and (I, J + 1); on the
                            // diagonal A is the first half of the B box
                            const uint32_t b0 = a0 + boff16;
                            const uint32_t aw = same ? b0 : a0;
                            const uint32_t id = it.nsub == 2 ? idesc_wide : idesc;
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                mma_op<C::kF8>(dset, aw + 2u * k, b0 + 2u * k, desc_hi, id, (k > 0) | acc0);
                        } else if constexpr (C::kSplit) {
                            const uint32_t b0 = same ? a0 : a0 + boff16;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t ak = a0 + 2u * k, bk = b0 + 2u * k;
                                ptx::mma_f16_lo(dset, ak, bk, desc_hi, idesc, (k > 0) | acc0);
                                ptx::mma_f16_lo(dset, ak, bk + 1024u, desc_hi, idesc, 1u);   // h_i l_j
                                ptx::mma_f16_lo(dset, ak + 1024u, bk, desc_hi, idesc, 1u);   // l_i h_j
                            }
                        } else if (jb.cpi == 2) {
                            // two channels, each its own diagonal tile (B = A), accumulators
                            // interleaved so consecutive MMAs are independent
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t acc = (k > 0) | acc0;
                                mma_op<C::kF8>(dset, a0 + 2u * k, a0 + 2u * k, desc_hi, idesc, acc);
                                mma_op<C::kF8>(dset + 128u, a0 + 1024u + 2u * k, a0 + 1024u + 2u * k, desc_hi, idesc,
                                               acc);
                            }
                        } else {
                            const uint32_t b0 = same ? a0 : a0 + boff16;
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                mma_op<C::kF8>(dset, a0 + 2u * k, b0 + 2u * k, desc_hi, idesc, (k > 0) | acc0);
                        }
                        any = true;
                        commit(bar_op_empty + 8 * s);
                        if (++s == OS) {
                            s = 0;
                            ph ^= 1u;
                        }
                    }
                    if (!ok) break;
                    commit(bar_acc_full + 8 * abuf);
                    if (++abuf == 2) {
                        abuf = 0;
                        aph ^= 1u;
                    }
                }
            }
            // every MMA of ours must be complete before tensor memory is released
            if (any) {
                commit(bar_drain);
                ptx::mbar_wait_drain(bar_drain, 0, kDrainLimitNs);
            } else if constexpr (PAIR) {
                ptx::mbar_arrive_cluster(ptx::map_shared(bar_drain, 1));   // nothing to come for the peer
            }
        }
        __syncwarp();
    } else if (warp < 2 + C::kEpiWarps) {
        // ---------------- epilogue (warps 2..9) ----------------
        // Lane L of quadrant q holds operand row 32q + L: input i_loc = 16q + L/2, real part
        // for even L, imaginary part for odd L.  Two warps share a quadrant: both stage into the
        // same 16 rows, warp `half` the column sixteenths m = half, half + 2, and each issues half
        // of the row copies.  (One warp per quadrant spent 4600 clocks on a 64 x 64 tile of a
        // 1024-input array, 1900 in the column loop and 1500 issuing copies, and bounded every
        // output-heavy shape.)
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int i_loc = 16 * q + (lane >> 1);
        const bool odd = lane & 1;
        constexpr bool kIntOut = !C::kSplit;
        const uint32_t staging = ptx::smem_u32(smem + prm.staging_offset);
        const uint32_t staging_q = staging + (uint32_t)(q * (kIntOut && !DUMP ? 16 * kStageRowBytes
                                                                              : DUMP ? kStageWarpD : 16 * kStageRowBytesF));
        int abuf = 0;
        uint32_t aph = 0, sph = 0;   // phases of the accumulator and of the quadrant's staging rows
        bool ok = true;
        int jc = 0;
        // Packed-triangle staging (single-block jobs): tile row u = sub n + i is input i of channel
        // cx + sub; its baselines j >= i sit in tile columns u .. t_end - 1 (t_end = sub n + n) and, in
        // the warp's part of the tile's run of elements, at slots t_slot + column.  The values depend
        // only on the job and on how many channels of the tile exist: kept from tile to tile.
        int t_rows = -1, t_job = -1, t_end = 0, t_slot = 0, t_len = 0, t_s0 = 0, t_mhi = 0;
        for (int64_t item = item0; ok && item < prm.n_items; item += item_step) {
            ItemCtx it;
            decode_item<MAXJ, PAIR>(prm, item, jc, it, rank);
            const TcJob& jb = prm.jobs[MAXJ == 1 ? 0 : it.j];
            const int n_in = jb.n_inputs;
            const int P = n_in * (n_in + 1) / 2;
            const int I = it.I, J = it.J;
            const int nkb = jb.kp / C::kStageT;
            const bool tri = jb.nb == 1;
            // baseline b(i, j) = row_off(i) + j within one channel's [P] block
            auto row_off = [&](int i) { return i * n_in - (i * (i - 1) >> 1) - i; };
            // float pairs: 1 when the output starts at an odd 8-byte unit (16-byte alignment of the copies)
            const int vis_odd = (int)((reinterpret_cast<uintptr_t>(jb.vis) >> 3) & 1);
            for (int kb0 = 0; kb0 < nkb; kb0 += jb.chunk_kb) {
                // An accumulator spans a whole chunk of stages, so this wait gets twice the bound: a
                // stage that never arrives is reported by the role waiting for that stage
                const bool got =
                    ptx::mbar_wait_bounded_warp(bar_acc_full + 8 * abuf, aph, abort_flag, 2 * prm.wait_limit_ns);
                if (!got) {   // the warp decides as one
                    if (lane == 0) record_error(prm.status, abort_flag, kDevTimeoutAccFull, kb0);
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const bool add = prm.accumulate || kb0 > 0;
                for (int ch = 0; ch < it.nsub; ++ch) {
                // a pair's square reaches below the diagonal and past the last block
                if (PAIR && (J + ch < I || J + ch >= jb.nb || I >= jb.nb)) continue;
                // sub-accumulator ch: channel tile c0 + ch of a single-block item, or tile
                // (I, J + ch) of a wide item
                const int Jx = it.wide ? J + ch : J;
                const int J0 = Jx * kBlockInputs;
                const int cx = (it.wide ? it.c0 : it.c0 + ch) * jb.pack;   // first channel of the tile
                const int64_t chan_base = (it.d * jb.n_chan + cx) * (int64_t)P;
                const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) +
                                       (uint32_t)(abuf * (int)(prm.tmem_cols / 2) + ch * 128);
                int m_lo = Jx == I ? q : 0, m_hi = 4;   // column sixteenths the quadrant needs
                if (tri) {
                    const int rows = max(0, min(jb.pack, jb.n_chan - cx)) * n_in;
                    if (rows != t_rows || it.j != t_job) {
                        t_rows = rows;
                        t_job = it.j;
                        const int r0 = 16 * q, r1 = min(r0 + 16, rows);
                        auto start = [&](int u) {   // element of row u's first baseline within the tile's run
                            const int sub = u / n_in, iu = u - sub * n_in;
                            return sub * P + row_off(iu) + iu;
                        };
                        t_mhi = t_len = t_end = 0;
                        if (r0 < r1) {
                            t_s0 = start(r0);
                            t_len = start(r1) - t_s0;
                            t_mhi = (((r1 - 1) / n_in + 1) * n_in + 15) >> 4;
                            t_end = i_loc < r1 ? (i_loc / n_in + 1) * n_in : 0;
                            t_slot = start(i_loc) - t_s0 - i_loc;
                        }
                    }
                    m_hi = t_mhi;
                }
                const int64_t tri_first = chan_base + t_s0;   // the quadrant's run of output elements
                const int tri_odd = (!kIntOut || DUMP) ? (int)((tri_first + vis_odd) & 1) : 0;
                // both warps' bulk copies of the previous tile must have read the staging rows; a later
                // chunk adds into elements that the copies of the one before it wrote
                if (lane < 16) {
                    if (kb0 > 0) bulk_wait_all();
                    else bulk_wait_read();
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar_stage_free + 8 * q);
                if (!ptx::mbar_wait_bounded_warp(bar_stage_free + 8 * q, sph, abort_flag, prm.wait_limit_ns)) {
                    if (lane == 0) record_error(prm.status, abort_flag, kDevTimeoutAccFull, kb0);
                    ok = false;
                    break;
                }
                // dump mode: this channel's phasors -- gi for the lane's row, and the J block's
                // 64 in shared memory after the warp's staging rows (staged launches)
                const float2* gch = nullptr;
                float2 gi = make_float2(1.f, 0.f);
                uint32_t phs = 0;
                if constexpr (DUMP) {
                    if (jb.phasor && cx < jb.n_chan) {   // warp-uniform: every lane stages
                        gch = jb.phasor + (size_t)cx * n_in;   // [channel][input]: tile column j of row cx
                        const int n_ph = tri ? t_rows : n_in;
                        if (I * kBlockInputs + i_loc < n_ph) gi = gch[I * kBlockInputs + i_loc];
                        phs = tri ? staging + (uint32_t)(kTriPhasors + q * kBlockInputs * 8)
                                  : staging_q + 16u * (uint32_t)kStageRowBytesF;
                        // each warp stages the 32 it uses: columns 16 m .. 16 m + 15, m = half, half + 2
                        const int u = (lane >> 4) * 32 + half * 16 + (lane & 15);
                        const float2 g = J0 + u < n_ph ? gch[J0 + u] : make_float2(1.f, 0.f);
                        st_shared_v2_f32(phs + 8u * (uint32_t)u, g.x, g.y);
                        __syncwarp();
                    }
                }
                // beside jobs of several blocks the run nests in the warp's own staging rows: another
                // warp may still be on such a job's tile
                const uint32_t tri_q = prm.staged ? staging_q
                                                  : staging + (kIntOut && !DUMP ? (uint32_t)(tri_slot(q) * 16)
                                                                                : (uint32_t)(tri_slot(q) * 8 + q * 16));
#pragma unroll 1
                for (int m = m_lo + ((m_lo ^ half) & 1); m < m_hi; m += 2) {
                    uint32_t v[32];
                    __syncwarp();
                    ptx::tmem_ld32(tbase + 32u * m, v);
                    ptx::tmem_wait_ld();
                    if constexpr (DUMP) {
                    // exchange: the even lane keeps j-slots 0..7 and receives the odd lane's
                    // (xi_i xr_j, xi_i xi_j) for them; the odd lane keeps 8..15 likewise
                    uint32_t own0[8], own1[8], oth0[8], oth1[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t s0 = odd ? v[2 * k] : v[2 * k + 16];
                        const uint32_t s1 = odd ? v[2 * k + 1] : v[2 * k + 17];
                        oth0[k] = __shfl_xor_sync(0xffffffffu, s0, 1);
                        oth1[k] = __shfl_xor_sync(0xffffffffu, s1, 1);
                        own0[k] = odd ? v[2 * k + 16] : v[2 * k];
                        own1[k] = odd ? v[2 * k + 17] : v[2 * k + 1];
                    }
                    const int j0 = 16 * m + (odd ? 8 : 0);   // first of the lane's 8 tile columns
                        // dump mode: rr + ii and ir - ri in fp32 (each term exact, the sum rounded
                        // once), scaled by 1 / n_accum and rotated by phasor_i conj(phasor_j)
                        float2 wv[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float rr = __uint_as_float(odd ? oth0[k] : own0[k]);
                            const float ri = __uint_as_float(odd ? oth1[k] : own1[k]);
                            const float ir = __uint_as_float(odd ? own0[k] : oth0[k]);
                            const float ii = __uint_as_float(odd ? own1[k] : oth1[k]);
                            float2 w = make_float2((rr + ii) * jb.inv_n, (ir - ri) * jb.inv_n);
                            if (gch) {   // columns past the array: phasor 1, never stored
                                const float2 gj = ld_shared_v2_f32(phs + 8u * (uint32_t)(j0 + k));
                                const float2 t = make_float2(w.x * gi.x - w.y * gi.y, w.x * gi.y + w.y * gi.x);
                                w = make_float2(t.x * gj.x + t.y * gj.y, t.y * gj.x - t.x * gj.y);
                            }
                            wv[k] = w;
                        }
                        if (tri) {
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                if (j0 + k >= i_loc && j0 + k < t_end)
                                    st_shared_v2_f32(tri_q + 8u * (uint32_t)(t_slot + tri_odd + j0 + k), wv[k].x, wv[k].y);
                        } else {   // dump mode of several blocks is always staged
                            // slot (j - J0) + s of row lane/2, s = parity of the row's element J0
                            const int s_r = (int)((chan_base + row_off(I * kBlockInputs + i_loc) + J0 + vis_odd) & 1);
                            const uint32_t rowp = staging_q + (uint32_t)(lane >> 1) * kStageRowBytesF +
                                                  (uint32_t)(j0 + s_r) * 8u;
#pragma unroll
                            for (int k = 0; k < 8; ++k) st_shared_v2_f32(rowp + 8u * (uint32_t)k, wv[k].x, wv[k].y);
                        }
                    } else {
                        // column k of the sixteenth: the real-part row (even lane) holds (rr, ri), the
                        // imaginary-part row (odd lane) (ir, ii); one exchange of the second values
                        // gives the even lane Re = rr + ii and the odd lane Im = ir - ri, with no
                        // selects, and each lane stores its half of the output pair
                        const float sgn = odd ? -1.f : 1.f;
                        const int col = 16 * m;
                        if constexpr (kIntOut) {
                            // every D element is an integer of magnitude <= 2^24: exact in int32
                            int w[16];
                            if (jb.f32_combine) {
#pragma unroll
                                for (int k = 0; k < 16; ++k) {
                                    const float x = __uint_as_float(__shfl_xor_sync(0xffffffffu, v[2 * k + 1], 1));
                                    w[k] = __float2int_rn(fmaf(sgn, x, __uint_as_float(v[2 * k])));
                                }
                            } else {
#pragma unroll
                                for (int k = 0; k < 16; ++k) {
                                    const float x = __uint_as_float(__shfl_xor_sync(0xffffffffu, v[2 * k + 1], 1));
                                    w[k] = __float2int_rn(__uint_as_float(v[2 * k])) + __float2int_rn(sgn * x);
                                }
                            }
                            if (tri) {
                                const uint32_t rowp = tri_q + (uint32_t)(t_slot + col) * 16u + (odd ? 8u : 0u);
#pragma unroll
                                for (int k = 0; k < 16; ++k)
                                    if (col + k >= i_loc && col + k < t_end)
                                        st_shared_u64(rowp + 16u * (uint32_t)k, (uint64_t)(long long)w[k]);
                            } else {
                                // row lane/2 of the warp's staging rows, slots j - J0: the pairs of a
                                // half-warp's 8 rows fall in distinct banks (row pitch 65 x 16 bytes)
                                const uint32_t rowp = staging_q + (uint32_t)(lane >> 1) * kStageRowBytes +
                                                      (uint32_t)col * 16u + (odd ? 8u : 0u);
#pragma unroll
                                for (int k = 0; k < 16; ++k)
                                    st_shared_u64(rowp + 16u * (uint32_t)k, (uint64_t)(long long)w[k]);
                            }
                        } else {
                            float w[16];
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                const float x = __uint_as_float(__shfl_xor_sync(0xffffffffu, v[2 * k + 1], 1));
                                w[k] = fmaf(sgn, x, __uint_as_float(v[2 * k]));
                            }
                            if (tri) {
                                const uint32_t rowp = tri_q + (uint32_t)(t_slot + tri_odd + col) * 8u + (odd ? 4u : 0u);
#pragma unroll
                                for (int k = 0; k < 16; ++k)
                                    if (col + k >= i_loc && col + k < t_end)
                                        st_shared_f32(rowp + 8u * (uint32_t)k, w[k]);
                            } else {
                                const int s_r = (int)((chan_base + row_off(I * kBlockInputs + i_loc) + J0 + vis_odd) & 1);
                                const uint32_t rowp = staging_q + (uint32_t)(lane >> 1) * kStageRowBytesF +
                                                      (uint32_t)(col + s_r) * 8u + (odd ? 4u : 0u);
#pragma unroll
                                for (int k = 0; k < 16; ++k) st_shared_f32(rowp + 8u * (uint32_t)k, w[k]);
                            }
                        }
                    }
                }
                // both warps have staged their columns: the staged rows are visible to the bulk-copy
                // engine and to the other warp
                fence_async_shared();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar_stage_full + 8 * q);
                if (!ptx::mbar_wait_bounded_warp(bar_stage_full + 8 * q, sph, abort_flag, prm.wait_limit_ns)) {
                    if (lane == 0) record_error(prm.status, abort_flag, kDevTimeoutAccFull, kb0);
                    ok = false;
                    break;
                }
                sph ^= 1u;
                // this warp's row of the tile in its lane (several blocks): lanes 0..7
                const int r_own = 8 * half + lane;
                const int i_own = I * kBlockInputs + 16 * q + r_own;
                const int j_lo = max(J0, i_own), j_hi = min(J0 + kBlockInputs, n_in);
                const bool own_ok = lane < 8 && i_own < n_in && j_lo < j_hi;   // one channel per tile: cx exists
                if (C::kSplit && add) {
                    // float sums in place: each warp adds half of the staged elements, lanes along the output
                    float2* const vis2 = reinterpret_cast<float2*>(jb.vis);
                    auto add_run = [&](int64_t first, uint32_t src, int len, int e0, int step) {
                        for (int e = e0 + lane; e < len; e += step) {
                            const float2 w = ld_shared_v2_f32(src + 8u * (uint32_t)e);
                            float2 o = vis2[first + e];
                            o.x += w.x;
                            o.y += w.y;
                            vis2[first + e] = o;
                        }
                    };
                    if (tri) {
                        add_run(tri_first, tri_q + 8u * (uint32_t)tri_odd, t_len, 32 * half, 64);
                    } else {
                        for (int r = 8 * half; r < 8 * half + 8; ++r) {
                            const int ir_ = I * kBlockInputs + 16 * q + r;
                            if (ir_ >= n_in) break;
                            const int lo = max(J0, ir_);
                            const int64_t rstart = chan_base + row_off(ir_);
                            const int s_r = (int)((rstart + J0 + vis_odd) & 1);
                            add_run(rstart + lo, staging_q + (uint32_t)r * kStageRowBytesF + (uint32_t)(lo - J0 + s_r) * 8u,
                                    j_hi - lo, 0, 32);
                        }
                    }
                } else if (tri) {
                    // one lane copies the quadrant's run: int64 pairs whole; float pairs the 16-byte-aligned
                    // body, with an unaligned first and an odd last element by plain stores
                    if (half == 0 && lane == 0 && t_len > 0) {
                        if constexpr (kIntOut && !DUMP) {
                            void* dst = reinterpret_cast<longlong2*>(jb.vis) + tri_first;
                            if (add) bulk_add_u64(dst, tri_q, (uint32_t)t_len * 16u);
                            else bulk_store(dst, tri_q, (uint32_t)t_len * 16u);
                        } else {
                            float2* dst = reinterpret_cast<float2*>(jb.vis) + tri_first;
                            if (tri_odd) dst[0] = ld_shared_v2_f32(tri_q + 8u);
                            const int body = (t_len - tri_odd) & ~1;
                            if (body > 0) bulk_store(dst + tri_odd, tri_q + 16u * (uint32_t)tri_odd, (uint32_t)body * 8u);
                            if (tri_odd + body < t_len)
                                dst[t_len - 1] = ld_shared_v2_f32(tri_q + 8u * (uint32_t)(t_len - 1 + tri_odd));
                        }
                    }
                    bulk_commit();
                } else if (DUMP || !kIntOut) {
                    // the row's float pairs [max(J0, i), min(J0 + 64, N)): an unaligned first element by
                    // a plain store, the 16-byte-aligned body by a bulk copy, an odd last element by a
                    // plain store
                    if (own_ok) {
                        const int64_t rstart = chan_base + row_off(i_own);
                        const int s_r = (int)((rstart + J0 + vis_odd) & 1);
                        const uint32_t row_src = staging_q + (uint32_t)r_own * kStageRowBytesF;
                        float2* vis2 = reinterpret_cast<float2*>(jb.vis);
                        int j = j_lo;
                        if ((rstart + j + vis_odd) & 1) {
                            vis2[rstart + j] = ld_shared_v2_f32(row_src + (uint32_t)(j - J0 + s_r) * 8u);
                            ++j;
                        }
                        const int body = (j_hi - j) & ~1;
                        if (body > 0)
                            bulk_store(vis2 + rstart + j, row_src + (uint32_t)(j - J0 + s_r) * 8u, (uint32_t)body * 8u);
                        j += body;
                        if (j < j_hi) vis2[rstart + j] = ld_shared_v2_f32(row_src + (uint32_t)(j - J0 + s_r) * 8u);
                    }
                    bulk_commit();
                } else {
                    // the row's run of baselines [max(J0, i), min(J0 + 64, N))
                    if (own_ok) {
                        const uint32_t src = staging_q + (uint32_t)r_own * kStageRowBytes + (uint32_t)(j_lo - J0) * 16u;
                        void* dst = reinterpret_cast<longlong2*>(jb.vis) + chan_base + (row_off(i_own) + j_lo);
                        const uint32_t bytes = (uint32_t)(j_hi - j_lo) * 16u;
                        if (add) bulk_add_u64(dst, src, bytes);
                        else bulk_store(dst, src, bytes);
                    }
                    bulk_commit();
                }
                }  // sub-accumulators of the item
                if (!ok) break;
                // accumulator drained (the loads completed at tcgen05.wait::ld): hand the
                // tensor-memory buffer back to the MMA warp
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) ptx::mbar_arrive_cluster(ptx::map_shared(bar_acc_empty + 8 * abuf, 0));
                    else ptx::mbar_arrive(bar_acc_empty + 8 * abuf);
                }
                if (++abuf == 2) {
                    abuf = 0;
                    aph ^= 1u;
                }
            }
        }
        // every bulk copy of ours must have completed before the CTA exits
        if (lane < 16) bulk_wait_all();
        // The issuing CTA's commits arrive in its peer as well, and the last must have before the peer exits.  The
        // limit runs from here, where the last accumulator has been seen, not from the start of a launch that may take
        // longer; it covers an issuer that gives up one wait later.  (Behind the closing barrier, outside
        // the roles, the same wait cost every pass of them: 224 inputs x 1218 channels x 77 samples x 4 640 -> 652 us.)
        if (PAIR && rank != 0 && warp == 2 && lane == 0)
            ptx::mbar_wait_drain(bar_drain, 0, prm.wait_limit_ns + kDrainLimitNs);
    } else if constexpr (C::kRaw) {
        // ---------------- converters (the last kConvWarps warps) ----------------
        // With two groups, one converts a whole stage while the other converts the next one: waits,
        // fence and arrivals (some 400 clocks of a stage with eight warps on it) are paid per warp and
        // visit, and a visit carries twice the work.  A barrier's phases are told apart by parity
        // only, so no group may wait for a phase two ahead of the barrier's: a group's previous stage
        // (two back) had its operand slot, so the MMAs are past the slot's use before last (rings have
        // two slots at least); and once this stage's operand slot is free, the raw slot's previous
        // stage is consumed -- where the raw ring is at least as deep as the operand ring, or its
        // slots stay with one group (an even depth; the host makes it so).
        const int cwarp = (warp - 2 - C::kEpiWarps) % C::kGroupWarps;
        const int group = (warp - 2 - C::kEpiWarps) / C::kGroupWarps;
        int turn = 0;
        const ConvLane cl = C::kBits8 ? conv_lane8(lane) : (C::kF8 ? conv_lane4_f8(lane) : conv_lane4(lane));
        constexpr uint32_t kRow = kBlockInputs * C::kBps;   // packed bytes of 64 inputs
        const uint32_t lane_byte = C::kBits8 ? 4u * lane : 4u * (lane & 15);
        int rs = 0, os = 0;
        uint32_t rph = 0, oph = 0;
        bool ok = true;
        int jc = 0;
        for (int64_t item = item0; ok && item < prm.n_items; item += item_step) {
            ItemCtx it;
            decode_item<MAXJ, PAIR>(prm, item, jc, it, rank);
            const int cpi = prm.jobs[MAXJ == 1 ? 0 : it.j].cpi;
            const uint32_t pair_off = (uint32_t)prm.jobs[MAXJ == 1 ? 0 : it.j].pair_off;
            const bool same = it.same;
            const int nkb = prm.jobs[MAXJ == 1 ? 0 : it.j].kp / C::kStageT;
            // The stage holds n_tl packed tiles: cpi channels side by side in each sample row
            // (diagonal items, row pitch cpi x kRow), or blocks I and J (off-diagonal items,
            // pitch kRow).  Each tile splits into warp-sized slices (8 for 8-bit, 4 for 4-bit);
            // the converter warps take slices round-robin.
            constexpr int kSlices = C::kBits8 ? 8 : 4;
            const int n_tl = same ? cpi : 2;
            const bool pair_pitch = same && cpi == 2;
            const int units = C::kFloat && PAIR && !same ? 2 : 1;
            for (int ku = 0; ku < nkb * units; ++ku) {
                const int kb = units == 2 ? ku >> 1 : ku;
                const bool mine = turn == group;
                if (++turn == C::kConvGroups) turn = 0;
                if (mine) {
                const bool got =
                    ptx::mbar_wait_bounded_warp2(bar_op_empty + 8 * os, oph ^ 1u, bar_raw_full + 8 * rs, rph,
                                                 abort_flag, prm.wait_limit_ns);
                if (!got) {   // the warp decides as one
                    if (lane == 0) record_error(prm.status, abort_flag, kDevTimeoutFull, kb);
                    ok = false;
                    break;
                }
                const uint32_t raw = ptx::smem_u32(rawring + rs * prm.raw_stage_bytes) + lane_byte;
                const uint32_t dst = ptx::smem_u32(ring + os * prm.op_stage_bytes);
                if constexpr (C::kFloat) {
                    // one tile a visit (B = A, or a square off the diagonal, whose two tiles go to the
                    // two groups): slice q of the tile per warp
                    const uint32_t raw_tile = ptx::smem_u32(rawring + rs * prm.raw_stage_bytes);
                    for (int sl = cwarp; sl < kTimeBlock / 8; sl += C::kGroupWarps)
                        convert_slice_f32(raw_tile, units == 2 && (ku & 1) ? dst + prm.b_offset : dst, sl, lane);
                } else if constexpr (C::kF8) {
                    // e4m3 operands, a slice per warp: 32 samples of one tile, lanes 0..15 chunk
                    // c = 2 part (samples 16c .. 16c + 15) and 16..31 chunk c + 1.  (The fp16
                    // converter's conflict-free orders below measured slower here: this converter
                    // is bound by its instruction count, not by shared-memory conflicts.)
                    const uint32_t pitch = pair_pitch ? 2 * kRow : kRow;
                    for (int sl = cwarp; sl < n_tl * kSlices; sl += C::kGroupWarps) {
                        const int tl = sl / kSlices;
                        const int c = 2 * (sl % kSlices) + (lane >> 4);
                        const uint32_t src = (same ? raw + tl * pair_off : raw + tl * C::kRawTileBytes) +
                                             (uint32_t)c * 16u * pitch;
                        uint32_t w[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) w[e] = ld_shared_u32(src + (uint32_t)e * pitch);
                        convert_words4_f8(w, dst + (same ? tl * kTileBytes : tl * prm.b_offset), c, cl);
                    }
                } else {
                const uint32_t pitch = pair_pitch ? 2 * kRow : kRow;
                // all loads of the warp's slices are issued before the first conversion, so their
                // shared-memory latencies overlap
                constexpr int kSlots = (2 * kSlices + C::kGroupWarps - 1) / C::kGroupWarps;
                uint32_t w[kSlots][8];
                // 4-bit slices (8 samples of 64 inputs per half-warp) split like the e4m3 ones:
                // by channel with channel pairs, else by sample group with the upper half-warp
                // reading rows in the order e ^ 1 (adjacent samples swapped alike in every odd
                // group of every operand row: a permutation of the sample axis shared by A and B)
                const bool split_ch = !C::kBits8 && pair_pitch;
                const int eflip = (!C::kBits8 && !pair_pitch) ? (lane >> 4) : 0;
#pragma unroll
                for (int v = 0; v < kSlots; ++v) {
                    const int sl = cwarp + C::kGroupWarps * v;
                    if (sl < n_tl * kSlices) {
                        const int tl = split_ch ? (lane >> 4) : sl / kSlices, part = sl % kSlices;
                        const int q = C::kBits8 ? part : (split_ch ? sl : 2 * part + (lane >> 4));
                        const uint32_t src = (same ? raw + tl * pair_off : raw + tl * C::kRawTileBytes) +
                                             (uint32_t)q * 8u * pitch;
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[v][e] = ld_shared_u32(src + (uint32_t)(e ^ eflip) * pitch);
                    }
                }
#pragma unroll
                for (int v = 0; v < kSlots; ++v) {
                    const int sl = cwarp + C::kGroupWarps * v;
                    if (sl < n_tl * kSlices) {
                        const int tl = split_ch ? (lane >> 4) : sl / kSlices, part = sl % kSlices;
                        const uint32_t out = dst + (same ? tl * kTileBytes : tl * prm.b_offset);
                        if constexpr (C::kBits8) convert_words8(w[v], out, part, cl);
                        else convert_words4(w[v], out, split_ch ? sl : 2 * part + (lane >> 4), cl);
                    }
                }
                }   // packed integers
                fence_async_shared();   // generic-proxy writes -> visible to the tensor core
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) {
                        const uint32_t full = ptx::map_shared(bar_op_full + 8 * os, 0);
                        ptx::mbar_arrive_cluster(full);
                        if (C::kFloat && units == 1) ptx::mbar_arrive_cluster(full);   // for the tile it has not
                    } else {
                        ptx::mbar_arrive(bar_op_full + 8 * os);
                    }
                    ptx::mbar_arrive(bar_raw_empty + 8 * rs);
                }
                }   // the group's stage
                if (++rs == RS) {
                    rs = 0;
                    rph ^= 1u;
                }
                if (units == 2 && !(ku & 1)) continue;   // the stage's second tile follows
                if (++os == OS) {
                    os = 0;
                    oph ^= 1u;
                }
            }
        }
    }

    ptx::tc_fence_before();
    if constexpr (PAIR) {
        __syncwarp();
        ptx::cluster_sync();   // neither CTA's memory goes while the other may still arrive there or read it
        // The issuing CTA has seen its last commit; the same commits must have arrived here before
        // this CTA exits.  The limit runs from here, not from the start of a launch that may take longer.
    } else {
        __syncthreads();
    }
    ptx::tc_fence_after();
    if (warp == 1) ptx::tmem_dealloc<PAIR>(tmem_base, prm.tmem_cols);
    if constexpr (PAIR) ptx::cluster_sync();
}

// ---- host side --------------------------------------------------------------------

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// 2-D map over plane rows: dim0 = Kp samples (fp16/bf16), dim1 = all 128-row blocks; boxes of
// one block (128 rows) or, for wide items, of two adjacent blocks (256 rows).
// Planes [rows][kp] of 2-byte elements (fp16/bf16: boxes of 64 samples) or of e4m3 bytes
// (UINT8: boxes of 128 samples); either way a box row is 128 bytes, loaded with 128-byte swizzle.
bool make_plane_map(CUtensorMap* map, const void* base, int kp, int64_t rows, CUtensorMapDataType dt,
                    int box_rows = kBlockRows) {
    auto enc = get_encode();
    if (!enc) return false;
    const int elem = dt == CU_TENSOR_MAP_DATA_TYPE_UINT8 ? 1 : 2;
    cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kp * elem};
    cuuint32_t box[2] = {(cuuint32_t)(128 / elem), (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// 4-D map over packed bytes [dump][time][chan][input*bps]; box = 64 inputs x box_chans channels
// x box_t samples (64, or 128 for e4m3 operands).
// Out-of-range inputs (ragged last block) and samples (ragged last block) read as zero.
// pack > 1 (arrays of at most 32 inputs): `pack` adjacent channels fill one 64-input tile, so the map
// runs over whole time samples (all channels' inputs as one row) and a box of one or two tiles
// starts at the first channel's input 0, a multiple of 16 bytes.
bool make_raw_map(CUtensorMap* map, const void* base, int n_inputs, int n_chan, int n_time, int n_dumps, int bps,
                  int box_chans, int box_t, int pack, int64_t pitch) {
    auto enc = get_encode();
    if (!enc) return false;
    const cuuint64_t row = pitch > 0 ? (cuuint64_t)pitch : (cuuint64_t)n_inputs * bps;
    cuuint64_t dims[4] = {(cuuint64_t)n_inputs * bps, (cuuint64_t)n_chan, (cuuint64_t)n_time, (cuuint64_t)n_dumps};
    cuuint64_t strides[3] = {row, row * n_chan, row * n_chan * n_time};
    cuuint32_t box[4] = {(cuuint32_t)(kBlockInputs * bps), (cuuint32_t)box_chans, (cuuint32_t)box_t, 1};
    if (pack > 1) {
        dims[0] = row * n_chan;
        dims[1] = 1;
        strides[0] = row * n_chan;
        box[0] = (cuuint32_t)(kBlockInputs * bps * box_chans);
        box[1] = 1;
    }
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// constants of fast_div for the divisor d (1 <= d <= 2^31)
void fast_div_make(uint32_t d, uint32_t& m, int& s) {
    int l = 0;
    while ((uint64_t{1} << l) < d) ++l;
    m = (uint32_t)(((uint64_t{1} << 32) * ((uint64_t{1} << l) - d)) / d + 1);
    s = l;
}

// S(m) = floor((m + 1) / 2) floor((m + 2) / 2): wide items of an array of m blocks
int wide_items(int m) { return ((m + 1) / 2) * ((m + 2) / 2); }

template <int MODE, int MAXJ>
cudaError_t launch_jobs(const TcJobSpec* specs, int n_jobs, const CUtensorMap* maps, const CUtensorMap* map_lo,
                        int accumulate, int* status, int n_sm, const TcTuning& tune, cudaStream_t s,
                        const CUtensorMap* maps_wide = nullptr) {
    using C = Cfg<MODE>;
    if (n_jobs < 1 || n_jobs > MAXJ) return cudaErrorInvalidValue;
    static_assert(sizeof(TcLaunch<MAXJ>) <= 32000, "kernel parameters exceed the launch limit");
    auto* prm = new (std::nothrow) TcLaunch<MAXJ>();
    if (!prm) return cudaErrorMemoryAllocation;
    prm->n_jobs = n_jobs;
    prm->accumulate = accumulate;
    prm->status = status;
    prm->wait_limit_ns = tune.wait_limit_ns ? tune.wait_limit_ns : kWaitLimitNs;
    prm->stall_item = tune.stall_item;
    if (map_lo) prm->map_lo = *map_lo;
    int64_t items = 0;
    int op_tiles = 1, raw_tiles = 1;
    bool any_pair = false, pair = tune.pair != 0 && MODE != kPlanesBF16x3 && MODE != kRaw4;
    for (int j = 0; j < n_jobs; ++j)
        pair = pair && specs[j].n_inputs > kBlockInputs;
    for (int j = 0; j < n_jobs; ++j) {
        const TcJobSpec& sp = specs[j];
        TcJob& jb = prm->jobs[j];
        jb.map = maps[j];
        // wide items only where the MMA feed reads fp16 planes (two blocks per TMA box)
        jb.tw = ((MODE == kPlanesF16 || MODE == kPlanesF8) && sp.tw == 2 && maps_wide && !pair) ? 2 : 1;
        if (jb.tw == 2) jb.map_wide = maps_wide[j];
        jb.vis = sp.vis;
        jb.n_inputs = sp.n_inputs;
        jb.n_chan = sp.n_chan;
        jb.nb = (sp.n_inputs + kBlockInputs - 1) / kBlockInputs;
        jb.kp = (sp.n_time + C::kStageT - 1) / C::kStageT * C::kStageT;   // whole stages (zeros past n_time)
        const int ng = (jb.nb + 1) / 2;
        jb.n_tiles = pair ? ng * (ng + 1) / 2 : jb.tw == 2 ? wide_items(jb.nb) : jb.nb * (jb.nb + 1) / 2;
        jb.cpi = sp.cpi;
        jb.pack = C::kRaw && jb.nb == 1 ? sp.pack : 1;
        jb.n_groups = ((sp.n_chan + jb.pack - 1) / jb.pack + jb.cpi - 1) / jb.cpi;
        // packed channels: the map's rows are whole time samples (all channels), see make_raw_map
        const int tile_x = jb.pack * sp.n_inputs * (C::kMapX / kBlockInputs);
        jb.x_step = jb.pack > 1 ? tile_x : 0;
        jb.y_step = jb.pack > 1 ? 0 : 1;
        jb.pair_off = jb.pack > 1 ? jb.pack * sp.n_inputs * C::kBps : kBlockInputs * C::kBps;
        // a single-block tile's MMA stops at the columns its inputs fill (N a multiple of 16)
        jb.idesc = ptx::idesc_f16(128, jb.nb == 1 ? (2 * jb.pack * sp.n_inputs + 15) / 16 * 16 : 128, C::kSplit);
        // samples per exact chunk: 8-bit 1024 (|sum| <= 1024 * 2^14 = 2^24), 4-bit 131072, float: all
        // (in stages: 64 samples each, 128 for e4m3 operands)
        jb.chunk_kb = C::kSplit ? (jb.kp / kTimeBlock)
                                : (sp.sample_bits == 4 ? 131072 / C::kStageT : 1024 / C::kStageT);
        // |D| <= chunk samples x max |x_a x_b|: 4-bit 2^17 x 2^6 = 2^23, 8-bit 512 x 2^14 = 2^23
        jb.f32_combine = !C::kSplit && (sp.sample_bits == 4 || jb.kp <= 512) ? 1 : 0;
        jb.out_mode = sp.out_mode;
        jb.phasor = static_cast<const float2*>(sp.phasor);
        jb.inv_n = sp.inv_n;
        if (jb.out_mode && (accumulate || jb.kp > jb.chunk_kb * C::kStageT)) {   // one exact chunk per dump
            delete prm;
            return cudaErrorInvalidValue;
        }
        jb.item_begin = items;
        const int64_t job_items = (int64_t)sp.n_dumps * jb.n_groups * jb.n_tiles;
        if (job_items >= (int64_t{1} << 31)) {   // decode_item divides 32-bit item indices
            delete prm;
            return cudaErrorInvalidValue;
        }
        fast_div_make((uint32_t)jb.n_tiles, jb.tiles_m, jb.tiles_s);
        fast_div_make((uint32_t)jb.n_groups, jb.groups_m, jb.groups_s);
        items += job_items;
        // operand tiles one stage needs: A + a two-block B box for wide items; float pairs of two
        // blocks have their diagonal square only, and float pairs' raw slots hold one tile
        const int tiles = jb.tw == 2 ? 3 : (jb.nb == 1 ? jb.cpi : C::kFloat && pair && jb.nb == 2 ? 1 : 2);
        op_tiles = tiles > op_tiles ? tiles : op_tiles;
        raw_tiles = C::kFloat && pair ? 1 : tiles > raw_tiles ? tiles : raw_tiles;
        any_pair = any_pair || jb.cpi == 2 || jb.tw == 2 || pair;   // two 256-column accumulator sets
    }
    prm->n_items = items;
    prm->tmem_cols = any_pair ? 512u : 256u;
    // shared-memory carve-up; arrays of several blocks stage tile rows, single-block ones packed runs
    bool any_multi = false, any_dump = false;
    for (int j = 0; j < n_jobs; ++j) {
        any_multi = any_multi || prm->jobs[j].nb > 1;
        any_dump = any_dump || prm->jobs[j].out_mode != 0;
    }
    prm->staged = any_multi ? 1 : 0;
    const int stage_space = any_dump ? (any_multi ? 4 * kStageWarpD : kTriBytesF)
                            : C::kSplit ? (any_multi ? 4 * 16 * kStageRowBytesF : kTriPhasors)
                                        : (any_multi ? kStageBytes : kTriBytes);
    const int operand_bytes = C::kTilesPerOperand * kTileBytes;
    prm->op_stage_bytes = op_tiles * operand_bytes;
    prm->b_offset = operand_bytes;
    if (C::kRaw) {
        prm->raw_stage_bytes = raw_tiles * C::kRawTileBytes;
        prm->op_stages = tune.op_stages > 0 ? tune.op_stages : (prm->staged ? 3 : 4);
        // a requested depth that leaves fewer than 3 raw stages is reduced to what fits
        while (prm->op_stages > 2 &&
               kSmemBudget - stage_space - prm->op_stages * prm->op_stage_bytes < 3 * prm->raw_stage_bytes)
            --prm->op_stages;
        int raw_space = kSmemBudget - stage_space - prm->op_stages * prm->op_stage_bytes;
        prm->raw_stages = raw_space / prm->raw_stage_bytes;
        if (prm->raw_stages > kMaxRawStages) prm->raw_stages = kMaxRawStages;
        // two converter groups on a shallower raw ring, or one whose slots are parts of stages, need an
        // even one (see the converters' waits)
        if (C::kConvGroups == 2 && (prm->raw_stages < prm->op_stages || (C::kFloat && pair && op_tiles == 2)))
            prm->raw_stages &= ~1;
        if (prm->raw_stages < 2) {
            delete prm;
            return cudaErrorInvalidValue;
        }
    } else {
        prm->raw_stage_bytes = 0;
        prm->raw_stages = 0;
        // as deep as fits (less any reserve for a kernel running beside it), or the requested
        // depth when that is smaller
        prm->op_stages = (kSmemBudget - stage_space - tune.smem_reserve) / prm->op_stage_bytes;
        if (prm->op_stages > kMaxOpStages) prm->op_stages = kMaxOpStages;
        if (tune.op_stages >= 2 && tune.op_stages < prm->op_stages) prm->op_stages = tune.op_stages;
    }
    if (prm->op_stages < 2 || prm->op_stages > kMaxOpStages) {
        delete prm;
        return cudaErrorInvalidValue;
    }
    prm->raw_offset = prm->op_stages * prm->op_stage_bytes;
    prm->staging_offset = prm->raw_offset + prm->raw_stages * prm->raw_stage_bytes;
    prm->bar_offset = prm->staging_offset + stage_space;
    const int smem_bytes = prm->bar_offset + kBarBytes + 1024;
    auto kern = xeng_tc_kernel<MODE, MAXJ, false, false>;
    if constexpr (MODE != kPlanesBF16x3 && MODE != kRaw4) {
        if (pair) kern = xeng_tc_kernel<MODE, MAXJ, false, true>;
    }
    if constexpr (C::kRaw && !C::kFloat && MAXJ == 1) {
        if (any_dump) kern = xeng_tc_kernel<MODE, MAXJ, true, false>;
        if constexpr (MODE != kRaw4) {
            if (any_dump && pair) kern = xeng_tc_kernel<MODE, MAXJ, true, true>;
        }
    } else if (any_dump) {   // dump mode is built for single-job packed-sample launches only
        delete prm;
        return cudaErrorInvalidValue;
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e == cudaSuccess && items > 0) {
        const int ctas = pair ? 2 : 1, slots = n_sm / ctas;
        e = launch_kernel(kern, dim3((unsigned)(items < slots ? items : slots) * ctas), C::kThreads, (size_t)smem_bytes,
                          s, ctas, C::kRaw, *prm);
    }
    delete prm;
    return e;
}

// Pairs on planes, except for short accumulating dumps of few squares, whose read-modify-write single tiles spread
// over more CTAs (256 inputs x 1 channel x 128 samples 16.5 -> 12.6 us, 512 x 16 x 64 24.5 -> 22.7).
bool plane_pairs(const Plan& p, int n_dumps, int accumulate) {
    const int ng = (p.nb + 1) / 2;
    if (accumulate && p.kp <= 512 && (int64_t)ng * (ng + 1) / 2 * n_dumps * p.n_chan <= p.n_sm) return false;
    return tc_use_pairs(p, false);
}

}  // namespace

cudaError_t launch_xeng_tc(const Plan& p, const void* d_planes, const void* d_planes_lo, int n_dumps, void* d_vis,
                           int accumulate, cudaStream_t s) {
    const int64_t rows = (int64_t)n_dumps * p.n_chan * p.nb * kBlockRows;
    if (rows >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // TMA row coordinates are int32
    CUtensorMap mh, ml;
    TcJobSpec sp{p.n_inputs, p.n_chan, p.n_time, n_dumps, p.sample_bits, d_planes, d_vis, 1};
    TcTuning tune{};
    tune.op_stages = p.tc_op_stages;
    if (d_planes_lo) {
        if (!make_plane_map(&mh, d_planes, p.kp, rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16) ||
            !make_plane_map(&ml, d_planes_lo, p.kp, rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16))
            return cudaErrorInvalidValue;
        return launch_jobs<kPlanesBF16x3, 1>(&sp, 1, &mh, &ml, accumulate, p.d_status, p.n_sm, tune, s);
    }
    if (!make_plane_map(&mh, d_planes, p.kp, rows, CU_TENSOR_MAP_DATA_TYPE_FLOAT16)) return cudaErrorInvalidValue;
    // wide items (one N = 256 MMA over blocks J, J + 1) unless the plan asks for single tiles; by
    // default also single tiles for accumulating dumps shorter than 1024 samples, whose
    // read-modify-write epilogue bounds them and which run faster on the deeper operand ring of
    // 32 KB stages (measured: 1024 inputs x 1228 channels x 472 samples, 4.05 against 4.41 ms)
    const bool wide = p.tc_items == 2 || (p.tc_items == 0 && !(accumulate && p.kp < 1024));
    tune.pair = plane_pairs(p, n_dumps, accumulate);
    CUtensorMap mw;
    if (!tune.pair && p.nb >= 2 && wide && make_plane_map(&mw, d_planes, p.kp, rows, CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                                            2 * kBlockRows)) {
        sp.tw = 2;
        return launch_jobs<kPlanesF16, 1>(&sp, 1, &mh, nullptr, accumulate, p.d_status, p.n_sm, tune, s, &mw);
    }
    return launch_jobs<kPlanesF16, 1>(&sp, 1, &mh, nullptr, accumulate, p.d_status, p.n_sm, tune, s);
}

// CTA pairs work on 2 x 2 squares of tiles, so an odd block count leaves a block row and column of
// squares half empty.  Measured (8-bit, 512 channels, us, single CTAs -> pairs): packed feed, 128
// inputs x 256 / 2048 samples 40 -> 36 / 205 -> 127 (but 32 -> 34 at 128 samples), 192 inputs 57 -> 68
// at 128 samples, 75 -> 72 / 417 -> 381 at 256 / 2048, 256 inputs x 2048 662 -> 396, 512 inputs x 2048
// (476 channels) 1712 -> 936; plane feed, 512 inputs x 2048 1104 -> 998, 1024 inputs x 2048 (158
// channels) 1107 -> 992, but 320 inputs x 2048 821 -> 856 and, 4-bit, 320 x 512 158 -> 179.
bool tc_use_pairs(const Plan& p, bool packed) {
    if (p.nb < 2 || p.tc_items != 0) return false;
    if (p.nb % 2 == 0) return p.nb > 2 || p.kp > 128;
    return packed && p.kp > 256;
}

// Arrays whose plan would take the plane feed but which pairs convert faster inside the kernel: each
// block is converted once per square instead of once per tile.  Measured (8-bit, us, planes with
// pairs -> packed with pairs; 128 / 512 / 2048 samples): 256 inputs 97 -> 85 / 168 -> 122 / 554 -> 396,
// 512 inputs 273 -> 255 / 427 -> 392 / 998 -> 936, 768 inputs 321 -> 313 / 432 -> 446 / 990 -> 1085, 1024
// inputs 310 -> 311 / 405 -> 451 / 992 -> 1185 (256 samples: 374 -> 344, 360 -> 343).  4-bit (e4m3
// planes): 256 inputs 89 -> 84 / 125 -> 109 / 303 -> 320, 512 inputs 342 -> 346 at 512 samples.
// Accumulating dumps gain more: the read-modify-write of the sums leaves the packed feed's port and
// the memory system less to share than planes do.  8-bit, 400 inputs x 512 / 1024 samples 424 -> 358 /
// 702 -> 642, 1024 x 512 / 768 / 1024 536 -> 446 / 579 -> 549 / 666 -> 695; 4-bit, 192 x 384 94 -> 77,
// 400 x 512 320 -> 308, 1024 x 512 / 768 527 -> 488 / 505 -> 457, 256 / 384 inputs x 1024 channels x 1000
// samples 450 -> 264 / 869 -> 572, but 400 x 768 356 -> 417.
// Few items of long dumps go the other way (int_planes_faster).
bool tc_packed_pairs(const Plan& p, int accumulate) {
    // one operand stage (set_tuning): the plane feed ignores it, the packed one could not run
    if (p.tc_operands != 0 || p.tc_items != 0 || p.nb < 2 || p.tc_op_stages == 1) return false;
    const bool even = p.nb % 2 == 0;
    if (accumulate)
        return p.sample_bits == 8 ? p.nb <= 8 || p.kp <= (p.nb <= 12 ? 1024 : 768) : p.kp <= (even ? 1024 : 512);
    if (!even || !tc_use_pairs(p, true)) return false;
    return p.sample_bits == 8 ? p.nb <= 8 || p.kp <= 256 : p.nb == 4 && p.kp <= 512;
}

// Planes are written by the whole chip and then read at the MMAs' own pace; the packed feeds convert in the few
// CTAs that have an item, at 1.3 to 1.6 times the time per 64 samples.  Where the launch does not fill the
// chip and the dump is long, that is what it takes, planes or no planes.  Both estimated in us, from the waves of
// items, the time of an item's stage and the bytes that the extra kernel and the planes move; measured, packed ->
// planes: 8-bit, 256 inputs x 1 channel x 20000 / 60000 samples 207 -> 140 / 600 -> 392, x 4 x 20000 209 -> 155; 129 x 1 x
// 20000 201 -> 134; 9 inputs x 1 channel x 20000 143 -> 113; 320 x 16 x 20000, accumulating, 392 -> 274; but 256 x 16 x 20000
// 300 there, 318 with planes.  Dumps of fewer than 1500 samples, and 4-bit ones, are no slower packed.
bool int_planes_faster(const Plan& p, int n_dumps, int accumulate) {
    const int stages = p.kp / kTimeBlock;
    const int64_t cd = (int64_t)n_dumps * p.n_chan;
    if (p.sample_bits != 8 || stages < 24 || cd * p.nb * kBlockRows >= (int64_t{1} << 31)) return false;
    const int ng = (p.nb + 1) / 2;
    const bool pairs = tc_use_pairs(p, true), ragged = !tc_raw_supported(p);
    const int pack = tc_channel_pack(p.n_inputs, 2, p.n_chan, n_dumps, p.n_sm);
    const int64_t tiles = p.nb * (p.nb + 1) / 2 * cd, squares = ng * (ng + 1) / 2 * cd;
    auto waves = [](int64_t items, int64_t slots) { return (double)((items + slots - 1) / slots); };
    const double w = pairs ? waves(squares, p.n_sm / 2) : waves(p.nb == 1 && pack > 1 ? tiles / pack : tiles, p.n_sm);
    if (w > (p.nb == 1 ? 1 : 2)) return false;   // full chips hide the conversion
    const double mb = 2e-6 * p.n_inputs * (double)p.n_time * cd;
    double packed = w * stages * (!pairs ? 0.44 : p.nb == 2 ? 0.48 : 0.66);
    if (ragged && pack < 2) packed += 5 + 0.31 * mb;   // the repacked copy
    const double w_pl = tc_use_pairs(p, false)                                            ? waves(squares, p.n_sm / 2)
                        : p.nb >= 2 && !(accumulate && p.kp < 1024) ? waves(wide_items(p.nb) * cd, p.n_sm)
                                                                    : waves(tiles, p.n_sm);
    const double planes = 5 + w_pl * stages * (p.nb == 1 ? 0.35 : 0.41) + 0.14 * (mb + 512e-6 * p.nb * (double)p.kp * cd);
    return planes < packed;
}

bool tc_planes_e4m3(const Plan& p) { return p.sample_bits == 4 && tc_raw_supported(p); }

int tc_kp_e4m3(const Plan& p) { return (p.n_time + 127) / 128 * 128; }

cudaError_t launch_xeng_tc_e4m3_planes(const Plan& p, const void* d_planes, int n_dumps, void* d_vis, int accumulate,
                                       cudaStream_t s) {
    const int64_t rows = (int64_t)n_dumps * p.n_chan * p.nb * kBlockRows;
    if (rows >= (int64_t)1 << 31 || p.sample_bits != 4) return cudaErrorInvalidValue;
    const int kp8 = tc_kp_e4m3(p);
    CUtensorMap mh, mw;
    TcJobSpec sp{p.n_inputs, p.n_chan, p.n_time, n_dumps, p.sample_bits, d_planes, d_vis, 1};
    TcTuning tune{};
    tune.op_stages = p.tc_op_stages;
    if (!make_plane_map(&mh, d_planes, kp8, rows, CU_TENSOR_MAP_DATA_TYPE_UINT8)) return cudaErrorInvalidValue;
    // item shape as for fp16 planes
    const bool wide = p.tc_items == 2 || (p.tc_items == 0 && !(accumulate && kp8 < 1024));
    tune.pair = plane_pairs(p, n_dumps, accumulate);
    if (!tune.pair && p.nb >= 2 && wide &&
        make_plane_map(&mw, d_planes, kp8, rows, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2 * kBlockRows)) {
        sp.tw = 2;
        return launch_jobs<kPlanesF8, 1>(&sp, 1, &mh, nullptr, accumulate, p.d_status, p.n_sm, tune, s, &mw);
    }
    return launch_jobs<kPlanesF8, 1>(&sp, 1, &mh, nullptr, accumulate, p.d_status, p.n_sm, tune, s);
}

bool tc_use_planes(const Plan& p) {
    if (!tc_raw_supported(p)) return true;
    if (p.tc_operands == 1 || p.tc_operands == 3) return false;
    if (p.tc_operands == 2) return true;
    return p.nb >= (tc_planes_e4m3(p) ? kPlaneMinBlocksE4m3 : kPlaneMinBlocks);
}

bool tc_raw_supported(int n_inputs, int sample_bits) {
    // TMA needs every global stride (the packed row of N samples) to be a multiple of 16 bytes
    if (sample_bits != 4 && sample_bits != 8) return false;
    const int64_t row = (int64_t)n_inputs * (sample_bits == 8 ? 2 : 1);
    return row % 16 == 0;
}

bool tc_raw_supported(const Plan& p) { return tc_raw_supported(p.n_inputs, p.sample_bits); }

bool tc_raw_by_packing(const Plan& p, int n_dumps, int accumulate) {
    return (p.sample_bits == 4 || p.sample_bits == 8) && !tc_raw_supported(p) && p.tc_operands == 0 &&
           p.tc_op_stages != 1 &&   // as in tc_packed_pairs
           tc_channel_pack(p.n_inputs, p.sample_bits == 8 ? 2 : 1, p.n_chan, 1, p.n_sm) > 1 &&
           !int_planes_faster(p, n_dumps, accumulate);
}

// Channel pairs (256-byte TMA rows, one item's epilogue under the next item's MMAs) for
// single-block arrays, unless there are too few channels to give every SM a pair: a small dump
// then spreads its channels over twice as many CTAs.
int tc_default_cpi(int n_inputs, int64_t channels, int n_sm) {
    if (n_inputs > kBlockInputs) return 1;
    return channels >= 2 * (int64_t)n_sm ? 2 : 1;
}

// Channels side by side in one 64-input tile for arrays of at most 32 inputs (1: one channel per
// tile; 0: the packed feed cannot address the samples).  A packed sample row holds the channels one
// after another, so `pack` adjacent channels of n inputs are pack n adjacent inputs of one tile, of
// whose products the epilogue keeps each channel's own: TMA boxes, conversions and MMAs then carry
// pack channels for the price of one padded one.  Tiles start at 16-byte multiples and time samples
// are 16-byte multiples (TMA), which also admits rows of fewer than 16 bytes or odd ones.  A tile's
// place in the time sample is a 32-bit coordinate (in bytes, or in complex floats), so longer time
// samples do not pack.  A small launch keeps one tile per SM rather than fewer fuller ones.
int tc_channel_pack(int n_inputs, int bps, int n_chan, int64_t n_dumps, int n_sm) {
    const int64_t row = (int64_t)n_inputs * bps;
    const int64_t extent = (bps == 8 ? n_inputs : row) * n_chan;
    const bool aligned = row % 16 == 0;
    if (n_inputs > kBlockInputs / 2 || row * n_chan % 16 != 0 || extent >= (int64_t{1} << 31)) return aligned ? 1 : 0;
    int step = 1;   // smallest pack whose tiles are 16-byte multiples
    while (row * step % 16) ++step;
    const int most = kBlockInputs / n_inputs;
    if (step > most) return 0;
    int64_t pk = n_sm > 0 ? n_dumps * n_chan / n_sm : most;
    pk = pk > most ? most : pk;
    pk = pk > n_chan ? n_chan : pk;
    pk = pk / step * step;
    return (int)(pk < step ? step : pk);
}

bool tc_make_raw_map(CUtensorMap* map, const TcJobSpec& sp, bool f8) {
    const int bps = sp.sample_bits == 8 ? 2 : 1;
    return make_raw_map(map, sp.data, sp.n_inputs, sp.n_chan, sp.n_time, sp.n_dumps, bps, sp.cpi,
                        f8 ? Cfg<kRaw4F8>::kStageT : kTimeBlock, sp.pack, sp.row_pitch);
}

cudaError_t launch_xeng_tc_raw_jobs(const TcJobSpec* specs, const CUtensorMap* maps, int n_jobs, int accumulate,
                                    int* status, int n_sm, const TcTuning& tune, cudaStream_t s) {
    if (n_jobs < 1) return cudaErrorInvalidValue;
    const int bits = specs[0].sample_bits;
    for (int j = 0; j < n_jobs; ++j)
        if (specs[j].sample_bits != bits || specs[j].pack < 1 ||
            (specs[j].pack > 1 ? specs[j].pack * specs[j].n_inputs > kBlockInputs
             : specs[j].row_pitch ? specs[j].row_pitch % 16 != 0
                                  : !tc_raw_supported(specs[j].n_inputs, bits)) ||
            (specs[j].cpi != 1 && specs[j].cpi != 2) || (specs[j].cpi == 2 && specs[j].n_inputs > kBlockInputs))
            return cudaErrorInvalidValue;
    if (tune.f8_operands) {   // e4m3 operands: 4-bit samples (maps with 128-sample boxes)
        if (bits != 4) return cudaErrorInvalidValue;
        if (n_jobs == 1) return launch_jobs<kRaw4F8, 1>(specs, 1, maps, nullptr, accumulate, status, n_sm, tune, s);
        if (n_jobs > kMaxJobs) return cudaErrorInvalidValue;
        return launch_jobs<kRaw4F8, kMaxJobs>(specs, n_jobs, maps, nullptr, accumulate, status, n_sm, tune, s);
    }
    if (n_jobs == 1) {
        if (bits == 8) return launch_jobs<kRaw8, 1>(specs, 1, maps, nullptr, accumulate, status, n_sm, tune, s);
        return launch_jobs<kRaw4, 1>(specs, 1, maps, nullptr, accumulate, status, n_sm, tune, s);
    }
    if (n_jobs > kMaxJobs) return cudaErrorInvalidValue;
    if (bits == 8) return launch_jobs<kRaw8, kMaxJobs>(specs, n_jobs, maps, nullptr, accumulate, status, n_sm, tune, s);
    return launch_jobs<kRaw4, kMaxJobs>(specs, n_jobs, maps, nullptr, accumulate, status, n_sm, tune, s);
}

bool tc_make_plane_map(CUtensorMap* map, const TcJobSpec& sp, bool f8) {
    const int nb = (sp.n_inputs + kBlockInputs - 1) / kBlockInputs;
    const int step = f8 ? Cfg<kPlanesF8>::kStageT : kTimeBlock;
    const int kp = (sp.n_time + step - 1) / step * step;
    const int64_t rows = (int64_t)sp.n_dumps * sp.n_chan * nb * kBlockRows;
    if (rows >= (int64_t{1} << 31)) return false;   // TMA row coordinates are int32
    return make_plane_map(map, sp.data, kp, rows, f8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
}

bool tc_make_plane_map_wide(CUtensorMap* map, const TcJobSpec& sp, bool f8) {
    const int nb = (sp.n_inputs + kBlockInputs - 1) / kBlockInputs;
    const int step = f8 ? Cfg<kPlanesF8>::kStageT : kTimeBlock;
    const int kp = (sp.n_time + step - 1) / step * step;
    const int64_t rows = (int64_t)sp.n_dumps * sp.n_chan * nb * kBlockRows;
    if (rows >= (int64_t{1} << 31) || rows < 2 * kBlockRows) return false;
    return make_plane_map(map, sp.data, kp, rows, f8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                          2 * kBlockRows);
}

cudaError_t launch_xeng_tc_plane_jobs(const TcJobSpec* specs, const CUtensorMap* maps, int n_jobs, int accumulate,
                                      int* status, int n_sm, const TcTuning& tune, cudaStream_t s,
                                      const CUtensorMap* maps_wide) {
    if (n_jobs < 1 || n_jobs > kMaxJobs) return cudaErrorInvalidValue;
    for (int j = 0; j < n_jobs; ++j)
        if ((specs[j].sample_bits != 4 && specs[j].sample_bits != 8) || specs[j].cpi != 1 ||
            (specs[j].tw == 2 && !maps_wide))
            return cudaErrorInvalidValue;
    if (tune.f8_operands) {   // e4m3 planes of 4-bit samples (maps of tc_make_plane_map(..., true))
        for (int j = 0; j < n_jobs; ++j)
            if (specs[j].sample_bits != 4) return cudaErrorInvalidValue;
        if (n_jobs == 1)
            return launch_jobs<kPlanesF8, 1>(specs, 1, maps, nullptr, accumulate, status, n_sm, tune, s, maps_wide);
        return launch_jobs<kPlanesF8, kMaxJobs>(specs, n_jobs, maps, nullptr, accumulate, status, n_sm, tune, s,
                                                maps_wide);
    }
    if (n_jobs == 1)
        return launch_jobs<kPlanesF16, 1>(specs, 1, maps, nullptr, accumulate, status, n_sm, tune, s, maps_wide);
    return launch_jobs<kPlanesF16, kMaxJobs>(specs, n_jobs, maps, nullptr, accumulate, status, n_sm, tune, s,
                                             maps_wide);
}

namespace {
cudaError_t launch_raw_impl(const Plan& p, const void* d_packed, int n_dumps, void* d_vis, int accumulate,
                            cudaStream_t s, const TcTuning* tune, int out_mode, const void* phasor, float inv_n,
                            int64_t pitch = 0) {
    const int bps = p.sample_bits == 8 ? 2 : 1;
    const int pack = pitch ? 1 : tc_channel_pack(p.n_inputs, bps, p.n_chan, n_dumps, p.n_sm);
    if ((p.sample_bits != 4 && p.sample_bits != 8) || pack < 1 || (reinterpret_cast<uintptr_t>(d_packed) & 15u))
        return cudaErrorInvalidValue;
    TcTuning plan_tune;
    plan_tune.op_stages = p.tc_op_stages;
    // 4-bit samples take e4m3 operands unless the plan asks for fp16 (CORR_OPERANDS_PACKED):
    // the same bits, half the operand bytes and MMAs per sample
    const bool f8 = p.sample_bits == 4 && (p.tc_operands == 0 || p.tc_operands == 3);
    TcTuning run_tune = tune ? *tune : plan_tune;
    run_tune.f8_operands = f8 ? 1 : 0;
    run_tune.pair = tc_use_pairs(p, true) && !(p.sample_bits == 4 && !f8);
    const int chan_tiles = (p.n_chan + pack - 1) / pack;
    const int cpi = tc_default_cpi(p.n_inputs, (int64_t)n_dumps * chan_tiles, p.n_sm);
    // one launch covers fewer than 2^31 work items (the kernel decodes 32-bit item indices)
    const int64_t items_per_dump = (int64_t)((chan_tiles + cpi - 1) / cpi) * (p.nb * (p.nb + 1) / 2);
    const int64_t max_dumps = ((int64_t{1} << 31) - 1) / items_per_dump;
    if (max_dumps < 1) return cudaErrorInvalidValue;
    const size_t packed_dump = (size_t)p.n_time * p.n_chan * (pitch ? (size_t)pitch : (size_t)p.n_inputs * bps);
    const size_t vis_dump = (size_t)p.n_chan * (size_t)p.n_baselines * (out_mode ? 8 : 16);
    for (int d0 = 0; d0 < n_dumps;) {
        const int nd = (int)((n_dumps - d0) < max_dumps ? (n_dumps - d0) : max_dumps);
        TcJobSpec sp{p.n_inputs, p.n_chan, p.n_time, nd, p.sample_bits,
                     static_cast<const uint8_t*>(d_packed) + (size_t)d0 * packed_dump,
                     static_cast<uint8_t*>(d_vis) + (size_t)d0 * vis_dump, cpi};
        sp.pack = pack;
        sp.row_pitch = pitch;
        sp.out_mode = out_mode;
        sp.phasor = phasor;
        sp.inv_n = inv_n;
        CUtensorMap m;
        if (!tc_make_raw_map(&m, sp, f8)) return cudaErrorInvalidValue;
        const cudaError_t e = launch_xeng_tc_raw_jobs(&sp, &m, 1, accumulate, p.d_status, p.n_sm, run_tune, s);
        if (e != cudaSuccess) return e;
        d0 += nd;
    }
    return cudaSuccess;
}
}  // namespace

bool tc_rawf32_supported(const Plan& p) {
    // the arrays that ask for no workspace: single-block ones (single CTAs), and a
    // row of N complex floats a multiple of 16 bytes (TMA strides)
    return p.sample_bits == 32 && p.n_inputs <= kBlockInputs && (p.n_inputs % 2) == 0;
}

// As int_planes_faster, for float samples that the kernel could split itself.  Measured, in the kernel -> planes:
// 128 inputs x 1 channel x 4000 / 20000 samples 57 -> 41 / 254 -> 171 us, 256 x 1 / 4 x 20000 347 -> 175 / 441 -> 232, 512 x 8 x
// 4000 161 -> 130, 65 x 1 x 1000 23 -> 19, 33 x 2 x 20000 202 -> 169; but 128 x 16 x 20000 257 in the kernel, 297 with planes, and
// from five waves on (nine of long dumps) always the kernel.  Accumulating dumps also pay for the tiles' read-modify-write,
// in pairs by few CTAs: short ones of two blocks (65 inputs x 256 channels x 64 samples 62 -> 45) are better spread.
bool float_planes_faster(const Plan& p, int n_dumps, int accumulate) {
    const int stages = p.kp / kTimeBlock, ng = (p.nb + 1) / 2;
    const int64_t cd = (int64_t)n_dumps * p.n_chan;
    if (cd * p.nb * kBlockRows >= (int64_t{1} << 31)) return false;
    const int pack = accumulate ? 1 : tc_channel_pack(p.n_inputs, 8, p.n_chan, n_dumps, p.n_sm);
    const bool repack = p.n_inputs % 2 && pack < 2;
    const int64_t tiles = p.nb * (p.nb + 1) / 2 * cd, squares = ng * (ng + 1) / 2 * cd;
    auto waves = [](int64_t items, int64_t slots) { return (double)((items + slots - 1) / slots); };
    const double mb = 8e-6 * p.n_inputs * (double)p.n_time * cd;
    double split;
    if (p.nb == 1) {
        const double w = waves((cd + (pack > 1 ? pack : 1) - 1) / (pack > 1 ? pack : 1), p.n_sm);
        if (w > 1) return false;
        split = w * stages * 0.66;
    } else {
        const double w = waves(squares, p.n_sm / 2);
        if (accumulate && p.nb == 2 && w > 1 && stages <= (repack ? 4 : 2)) return true;
        if (w > (stages >= 32 ? 8 : 4)) return false;
        const double item = accumulate ? (p.nb == 2 ? 13 : p.nb % 2 ? 6.5 : 9) : 1.5;
        split = w * (stages * (p.nb == 2 ? 0.82 : w == 1 || p.nb > 4 ? 1.45 : 1.15) + item);
    }
    if (repack) split += 4.5 + 0.31 * mb;
    const double planes = 5 + waves(tiles, p.n_sm) * (stages * 0.5 + (accumulate && p.nb > 1 ? 6.2 : 0.8)) +
                          0.14 * (mb + 1024e-6 * p.nb * (double)p.kp * cd);
    return split > 1.03 * planes;
}

// Arrays of several blocks: the CTAs of a pair split the blocks of a square themselves, where the plane
// feed writes hi and lo planes (half of its time) and reads them back.  Measured, planes -> pairs: 128
// inputs x 512 channels x 64 / 128 / 256 / 512 samples 50 -> 27 / 69 -> 31 / 99 -> 38 / 173 -> 63 us (45
// us for the bytes of 512), 1024 channels x 1024 634 -> 227, 80 inputs x 139 x 1222 112 -> 43, 20 x 100
// 16 -> 9; squares off the diagonal too: 256 x 512 x 128 / 512 162 -> 81 / 402 -> 201, 256 x 76 x 4096
// 433 -> 238, 192 x 202 x 506 116 -> 78, 130 x 139 x 1222 180 -> 136, 512 x 128 x 512 283 -> 178, 1024 x 64
// x 256 / 1024 281 -> 180 / 780 -> 602.  Odd block counts above one compute half-empty squares and gain
// nothing on long dumps (320 x 200 x 500 220 -> 167, but 320 x 30 x 2000 126 -> 127).
bool tc_rawf32_pairs(const Plan& p, int n_dumps, int accumulate) {
    return p.sample_bits == 32 && p.nb >= 2 && (p.nb % 2 == 0 || p.kp <= 1536) && (p.n_inputs % 2) == 0 &&
           !p.tc_float_planes &&
           p.tc_op_stages != 1 &&   // one operand stage: the plane feed ignores it, this one could not run
           !float_planes_faster(p, n_dumps, accumulate);
}

// Odd counts of inputs, whose rows TMA cannot address: several channels of at most 32 inputs packed into
// a tile start at 16-byte multiples again; other rows go into the workspace one sample longer.
// Measured, planes -> this: packed channels 9 / 31 inputs x 512 channels x 1000 samples 139 -> 25 / 147 -> 33
// us; repacked 9 / 31 x 513 x 1000 137 -> 56 / 150 -> 88, 41 x 762 x 318 x 3 dumps 211 -> 153, 75 x 139 x
// 1222 113 -> 73, 127 x 512 x 512 181 -> 145, x 20 x 100 15 -> 13, 255 x 202 x 506 177 -> 149, 1023 x 64 x
// 256 289 -> 227; odd block counts, whose squares are half empty, stay with the planes (141 x 179 x 833 172
// there, 182 here).
bool tc_rawf32_odd(const Plan& p, int n_dumps, int accumulate) {
    return p.sample_bits == 32 && p.n_inputs % 2 && (p.nb == 1 || p.nb % 2 == 0) && !p.tc_float_planes && p.tc_op_stages != 1 &&
           (int64_t)n_dumps * p.n_time * p.n_chan < (int64_t{1} << 31) && !float_planes_faster(p, n_dumps, accumulate);
}

cudaError_t launch_xeng_tc_rawf32_odd(const Plan& p, const void* d_samples, int n_dumps, void* d_ws, void* d_vis,
                                      int accumulate, cudaStream_t s) {
    if (!accumulate && tc_channel_pack(p.n_inputs, 8, p.n_chan, n_dumps, p.n_sm) > 1)
        return launch_xeng_tc_rawf32(p, d_samples, n_dumps, d_vis, accumulate, s);
    const cudaError_t e = launch_repack(p, d_samples, n_dumps, d_ws, s);
    if (e != cudaSuccess) return e;
    return launch_xeng_tc_rawf32(p, d_ws, n_dumps, d_vis, accumulate, s, repack_pitch(p));
}

cudaError_t launch_xeng_tc_rawf32(const Plan& p, const void* d_samples, int n_dumps, void* d_vis, int accumulate,
                                  cudaStream_t s, int64_t pitch) {
    const int pack = accumulate || pitch ? 1 : tc_channel_pack(p.n_inputs, 8, p.n_chan, n_dumps, p.n_sm);
    if (p.sample_bits != 32 || (p.n_inputs % 2 && !pitch && pack < 2) ||
        (reinterpret_cast<uintptr_t>(d_samples) & 15u))
        return cudaErrorInvalidValue;
    if ((int64_t)n_dumps * p.n_chan >= (int64_t{1} << 31)) return cudaErrorInvalidValue;   // 32-bit item indices
    auto enc = get_encode();
    if (!enc) return cudaErrorInvalidValue;
    // [dump][time][chan][input] of 8-byte complex floats; box = 64 inputs x 1 channel x 64 samples.
    // The register epilogue that adds float sums in place takes one channel per tile.
    CUtensorMap m;
    const cuuint64_t row = pitch ? (cuuint64_t)pitch : (cuuint64_t)p.n_inputs * 8;
    cuuint64_t dims[4] = {(cuuint64_t)p.n_inputs, (cuuint64_t)p.n_chan, (cuuint64_t)p.n_time, (cuuint64_t)n_dumps};
    cuuint64_t strides[3] = {row, row * p.n_chan, row * p.n_chan * p.n_time};
    if (pack > 1) {   // whole time samples as rows, as in make_raw_map
        dims[0] *= (cuuint64_t)p.n_chan;
        dims[1] = 1;
        strides[0] = row * p.n_chan;
    }
    // (an odd count of a padded row: what lies past it reads as zero)
    cuuint32_t box[4] = {(cuuint32_t)kBlockInputs, 1, (cuuint32_t)kTimeBlock, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    if (enc(&m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(d_samples), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    TcJobSpec sp{p.n_inputs, p.n_chan, p.n_time, n_dumps, 32, d_samples, d_vis, 1};
    sp.pack = pack;
    TcTuning tune;
    tune.op_stages = p.tc_op_stages;
    tune.pair = p.nb >= 2;
    return launch_jobs<kRawF32, 1>(&sp, 1, &m, nullptr, accumulate, p.d_status, p.n_sm, tune, s);
}

cudaError_t launch_xeng_tc_raw(const Plan& p, const void* d_packed, int n_dumps, void* d_vis, int accumulate,
                               cudaStream_t s, const TcTuning* tune) {
    return launch_raw_impl(p, d_packed, n_dumps, d_vis, accumulate, s, tune, 0, nullptr, 1.0f);
}

// Rows that TMA cannot address (and channels that do not pack into tiles it can) go into the
// workspace as rows of whole 16-byte pieces where the packed feed is the better one, and else
// straight into planes (e4m3 for 4-bit samples: the workspace holds fp16 ones, twice as large).
// Measured, 8-bit, 75 inputs x 333 channels x 777 samples x 2 dumps: 215 us with a general unpack into
// fp16 planes (147 us of it the unpack), 109 us repacked.
cudaError_t launch_tc_plane_path(const Plan& p, const void* d_packed, int n_dumps, void* d_ws, void* d_vis,
                                 int accumulate, cudaStream_t s) {
    const bool ragged = !tc_raw_supported(p), aligned = (reinterpret_cast<uintptr_t>(d_packed) & 15u) == 0;
    const bool packed = (tc_packed_pairs(p, accumulate) ||
                         (ragged && p.tc_operands == 0 && p.tc_op_stages != 1 &&
                          p.nb < (p.sample_bits == 4 ? kPlaneMinBlocksE4m3 : kPlaneMinBlocks))) &&
                        !int_planes_faster(p, n_dumps, accumulate);
    if (packed && aligned) {
        if (!ragged) return launch_xeng_tc_raw(p, d_packed, n_dumps, d_vis, accumulate, s);
        if ((int64_t)n_dumps * p.n_time * p.n_chan < (int64_t{1} << 31)) {
            const cudaError_t e = launch_repack(p, d_packed, n_dumps, d_ws, s);
            if (e != cudaSuccess) return e;
            return launch_raw_impl(p, d_ws, n_dumps, d_vis, accumulate, s, nullptr, 0, nullptr, 1.0f, repack_pitch(p));
        }
    }
    if (p.sample_bits == 4) {
        const cudaError_t e = launch_unpack_e4m3(p, d_packed, n_dumps, d_ws, s);
        return e == cudaSuccess ? launch_xeng_tc_e4m3_planes(p, d_ws, n_dumps, d_vis, accumulate, s) : e;
    }
    const cudaError_t e = launch_unpack_fp16(p, d_packed, n_dumps, d_ws, s);
    return e == cudaSuccess ? launch_xeng_tc(p, d_ws, nullptr, n_dumps, d_vis, accumulate, s) : e;
}

cudaError_t launch_xeng_tc_raw_dump(const Plan& p, const void* d_packed, int n_dumps, void* d_out, const void* phasor,
                                    float inv_n, cudaStream_t s) {
    return launch_raw_impl(p, d_packed, n_dumps, d_out, 0, s, nullptr, 1, phasor, inv_n);
}

}  // namespace corr
