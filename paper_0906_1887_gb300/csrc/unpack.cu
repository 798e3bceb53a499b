// Unpack/transpose kernels: packed time-ordered samples -> per-input sample planes.
//
// The paper's first GPU step (Sec. 4) takes a block of N_I x N_C samples ordered with
// the input index fastest, converts them to floating point and regroups them so each
// input's samples are contiguous -- a transpose of the block.  Here the transpose is
// staged through shared memory so both the reads (consecutive inputs) and the writes
// (consecutive time samples of one plane row) are coalesced.
//
// Output planes: [dump][chan][NB][128][Kp]; row 2r holds the real parts and row 2r + 1
// the imaginary parts of input r of the block's 64 inputs; Kp = n_time rounded up to 64;
// padded inputs and samples are zero.  Elements are fp16, or, for the e4m3 plane feed of 4-bit
// samples, e4m3 bytes with Kp = n_time rounded up to 128.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "corr_internal.h"
#include "launch.cuh"
#include "ragged_piece.h"
#include "sample_convert.cuh"

namespace corr {
namespace {

constexpr int kThreads = 256;
constexpr int kPad = 65;  // smem row stride (floats)

enum OutKind { kOutF32 = 0, kOutBF16Split = 1 };

template <int OUT>
__global__ void __launch_bounds__(kThreads) unpack_kernel(const float2* __restrict__ samples, int n_inputs,
                                                          int n_chan, int n_time, int nb_count, int kp,
                                                          int64_t n_tiles, void* __restrict__ out0,
                                                          void* __restrict__ out1) {
    __shared__ float s_re[kBlockInputs * kPad];
    __shared__ float s_im[kBlockInputs * kPad];
    const int tb_count = kp / kTimeBlock;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        // tile -> (dc, nb, tb); dc = dump * n_chan + chan
        const int tb = (int)(tile % tb_count);
        const int64_t rest = tile / tb_count;
        const int nb = (int)(rest % nb_count);
        const int64_t dc = rest / nb_count;
        const int64_t d = dc / n_chan;
        const int c = (int)(dc % n_chan);
        // load: warp w takes time rows w, w+8, ...; lanes take consecutive inputs
        for (int t = warp; t < kTimeBlock; t += kThreads / 32) {
            const int tg = tb * kTimeBlock + t;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = lane + 32 * h;
                const int ig = nb * kBlockInputs + i;
                float re = 0.f, im = 0.f;
                if (tg < n_time && ig < n_inputs) {
                    const int64_t idx = ((d * n_time + tg) * n_chan + c) * (int64_t)n_inputs + ig;
                    const float2 v = samples[idx];
                    re = v.x;
                    im = v.y;
                }
                s_re[i * kPad + t] = re;
                s_im[i * kPad + t] = im;
            }
        }
        __syncthreads();
        // store: 128 rows x 64 samples, 8 samples (one 16-byte fp16 chunk) per step
        const int64_t row0 = ((dc * nb_count) + nb) * (int64_t)kBlockRows;
        for (int q = threadIdx.x; q < kBlockRows * (kTimeBlock / 8); q += kThreads) {
            const int r = q >> 3, ch = q & 7;
            const float* src = ((r & 1) ? s_im : s_re) + (r >> 1) * kPad + ch * 8;
            const int64_t off = (row0 + r) * (int64_t)kp + tb * kTimeBlock + ch * 8;
            if constexpr (OUT == kOutF32) {
                float4* dst = reinterpret_cast<float4*>(static_cast<float*>(out0) + off);
                dst[0] = make_float4(src[0], src[1], src[2], src[3]);
                dst[1] = make_float4(src[4], src[5], src[6], src[7]);
            } else {
                __align__(16) __nv_bfloat16 hi[8];
                __align__(16) __nv_bfloat16 lo[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    hi[e] = __float2bfloat16_rn(src[e]);
                    lo[e] = __float2bfloat16_rn(src[e] - __bfloat162float(hi[e]));
                }
                *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out0) + off) = *reinterpret_cast<uint4*>(hi);
                *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out1) + off) = *reinterpret_cast<uint4*>(lo);
            }
        }
        __syncthreads();
    }
}

// Packed 4/8-bit rows -> fp16 planes, for arrays whose packed row of N samples is a multiple of
// 16 bytes (so every 64-input block's row starts 16-byte aligned and its valid part is whole
// 16-byte pieces).  A tile is 64 samples x 64 inputs of one channel, handled by one block of
// kTileThreads threads:
//   load:    16-byte pieces of the 64 packed rows (64 x 128 B for 8-bit, 64 x 64 B for 4-bit)
//            into a shared byte tile, with 16-byte chunk c of row t stored at chunk
//            c ^ ((t >> 3) & 7) (8-bit) -- the conversion's reads are then bank-conflict-free;
//            pieces past the array's last input or past the dump's last sample are zero;
//   convert: thread (p, q) takes one 32-bit word (8-bit: inputs 2p, 2p+1; 4-bit: inputs 4p ..
//            4p+3) of the 8 samples 8q .. 8q+7 and writes its 4 (8-bit) or 8 (4-bit) plane rows'
//            16-byte piece q, converted exactly to fp16; lanes with consecutive q write one
//            128-byte row piece together.
template <int BITS>
struct FastTile {
    static constexpr int kRowBytes = kBlockInputs * (BITS == 8 ? 2 : 1);   // 128 or 64
    static constexpr int kWords = kRowBytes / 4;                            // 32 or 16
    static constexpr int kThreads = kWords * 8;                             // 256 or 128
    static constexpr int kTileBytes = kTimeBlock * kRowBytes;
};

// kGroup: tiles whose loads a block issues together (1 for the full grid; 8 for a launch of one
// block per SM beside a tensor-core launch, 64 KB in flight per block).  F8 (4-bit only): the
// planes hold e4m3 bytes instead of fp16 (rows of kp bytes), for the e4m3 plane feed.
// RAGGED: rows that are no whole 16-byte pieces; a piece is put together from the aligned words
// around it (load_piece), and bytes past the row are zero.  Tiles are counted in 32 bits (2^31 tiles of planes are
// 17 TB); 64-bit divisions of the tile index took a tenth of the time.
template <int BITS, int kGroup, bool F8 = false, bool RAGGED = false>
__global__ void __launch_bounds__(FastTile<BITS>::kThreads) unpack_fast_kernel(
    const unsigned char* __restrict__ packed, int n_inputs, int n_chan, int n_time, int nb_count, int kp,
    uint32_t n_tiles, void* __restrict__ planes_out, int64_t n_bytes) {
    static_assert(!F8 || BITS == 4, "e4m3 planes hold 4-bit samples only");
    __half* __restrict__ planes = static_cast<__half*>(planes_out);
    using F = FastTile<BITS>;
    __shared__ __align__(16) uint32_t tile[F::kTileBytes / 4];
    const int tid = threadIdx.x;
    const int tb_count = kp / kTimeBlock;
    const int64_t row_bytes = (int64_t)n_inputs * (BITS == 8 ? 2 : 1);
    constexpr int kPieces = F::kRowBytes / 16;          // 16-byte pieces per packed row
    constexpr int kPer = kTimeBlock * kPieces / F::kThreads;   // pieces a thread moves per tile (2)
    static_assert(kPer * F::kThreads == kTimeBlock * kPieces, "whole pieces per thread");
    const uint32_t tail = RAGGED ? tail_word(packed, n_bytes) : 0u;
    // conversion task of this thread
    const int q = tid & 7, pw = tid >> 3;             // sample group, word within the row
    const uint32_t* src = tile + (size_t)(8 * q) * F::kWords;
    // A block takes kGroup tiles at a time (strided by the grid) and issues every load of the
    // group before converting any: kGroup x 8 KB in flight per block.
    for (uint32_t t_base = blockIdx.x; t_base < n_tiles; t_base += kGroup * gridDim.x) {
        uint4 v[kGroup][kPer];
#pragma unroll
        for (int gi = 0; gi < kGroup; ++gi) {
            const uint32_t t_idx = t_base + gi * gridDim.x;
            const bool tile_ok = t_idx < n_tiles;
            const uint32_t rest = tile_ok ? t_idx / (uint32_t)tb_count : 0;
            const int tb = tile_ok ? (int)(t_idx - rest * tb_count) : 0;
            const uint32_t dc = rest / (uint32_t)nb_count;   // dump * n_chan + chan
            const int nb = (int)(rest - dc * nb_count);
            const int64_t d = dc / (uint32_t)n_chan;
            const int c = (int)(dc - (uint32_t)d * n_chan);
            const int64_t valid = row_bytes - (int64_t)nb * F::kRowBytes;   // bytes of this block's row that exist
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int k = tid + u * F::kThreads;
                const int t = k / kPieces, piece = k % kPieces;
                const int tg = tb * kTimeBlock + t;
                v[gi][u] = make_uint4(0u, 0u, 0u, 0u);
                if (tile_ok && tg < n_time && (int64_t)piece * 16 < valid) {
                    const int64_t off =
                        ((d * n_time + tg) * n_chan + c) * row_bytes + (int64_t)nb * F::kRowBytes + piece * 16;
                    if constexpr (RAGGED) {
                        uint32_t x[4];
                        load_piece(packed, off, n_bytes, (int)(valid - piece * 16 < 16 ? valid - piece * 16 : 16), tail, x);
                        v[gi][u] = make_uint4(x[0], x[1], x[2], x[3]);
                    } else {
                        v[gi][u] = *reinterpret_cast<const uint4*>(packed + off);
                    }
                }
            }
        }
#pragma unroll
        for (int gi = 0; gi < kGroup; ++gi) {
            const uint32_t t_idx = t_base + gi * gridDim.x;
            if (t_idx >= n_tiles) break;   // uniform across the block
            const uint32_t rest = t_idx / (uint32_t)tb_count;
            const int tb = (int)(t_idx - rest * tb_count);
            const int64_t dc = rest / (uint32_t)nb_count;
            const int nb = (int)(rest - (uint32_t)dc * nb_count);
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int k = tid + u * F::kThreads;
                const int t = k / kPieces, piece = k % kPieces;
                const int chunk = BITS == 8 ? (piece ^ ((t >> 3) & 7)) : (piece ^ ((t >> 3) & 3));
                *reinterpret_cast<uint4*>(tile + t * F::kWords + chunk * 4) = v[gi][u];
            }
            __syncthreads();
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int t = 8 * q + e;
                const int word = BITS == 8 ? (pw ^ (((t >> 3) & 7) << 2)) : (pw ^ (((t >> 3) & 3) << 2));
                w[e] = src[e * F::kWords + word];
            }
            __syncthreads();   // the tile is free for the next store once every thread holds its words
            const int64_t row0 = (dc * nb_count + nb) * (int64_t)kBlockRows;
            __half* out = planes + row0 * kp + (int64_t)tb * kTimeBlock + 8 * q;
            if constexpr (BITS == 8) {
                // word pw = (re, im) of inputs 2pw, 2pw + 1 -> plane rows 4pw + k, k = byte lane
                const __half2 bias = conv::bias8();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t sel = conv::lane_selector(k);
                    uint4 o;
                    o.x = conv::pair_to_half2(w[0], w[1], sel, conv::kFlip8, bias);
                    o.y = conv::pair_to_half2(w[2], w[3], sel, conv::kFlip8, bias);
                    o.z = conv::pair_to_half2(w[4], w[5], sel, conv::kFlip8, bias);
                    o.w = conv::pair_to_half2(w[6], w[7], sel, conv::kFlip8, bias);
                    *reinterpret_cast<uint4*>(out + (int64_t)(4 * pw + k) * kp) = o;
                }
            } else if constexpr (F8) {
                // as below, each row's 8 samples written as 8 e4m3 bytes (rows of kp bytes)
                unsigned char* out8 = static_cast<unsigned char*>(planes_out) + row0 * kp +
                                      (int64_t)tb * kTimeBlock + 8 * q;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    constexpr uint32_t kSel[4] = {conv::gather_selector(0), conv::gather_selector(1),
                                                  conv::gather_selector(2), conv::gather_selector(3)};
                    uint2 re, im;
                    conv::e4m3_of_nibbles(conv::gather4(w[0], w[1], w[2], w[3], kSel[k]), re.x, im.x);
                    conv::e4m3_of_nibbles(conv::gather4(w[4], w[5], w[6], w[7], kSel[k]), re.y, im.y);
                    *reinterpret_cast<uint2*>(out8 + (int64_t)(8 * pw + 2 * k) * kp) = re;
                    *reinterpret_cast<uint2*>(out8 + (int64_t)(8 * pw + 2 * k + 1) * kp) = im;
                }
            } else {
                // word pw = inputs 4pw .. 4pw + 3, high nibble re, low nibble im -> rows 8pw + 2k (+1)
                const __half2 bias = conv::bias4();
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    hi[e] = (w[e] >> 4) & 0x0F0F0F0Fu;
                    lo[e] = w[e] & 0x0F0F0F0Fu;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t sel = conv::lane_selector(k);
                    uint4 o;
                    o.x = conv::pair_to_half2(hi[0], hi[1], sel, conv::kFlip4, bias);
                    o.y = conv::pair_to_half2(hi[2], hi[3], sel, conv::kFlip4, bias);
                    o.z = conv::pair_to_half2(hi[4], hi[5], sel, conv::kFlip4, bias);
                    o.w = conv::pair_to_half2(hi[6], hi[7], sel, conv::kFlip4, bias);
                    *reinterpret_cast<uint4*>(out + (int64_t)(8 * pw + 2 * k) * kp) = o;
                    o.x = conv::pair_to_half2(lo[0], lo[1], sel, conv::kFlip4, bias);
                    o.y = conv::pair_to_half2(lo[2], lo[3], sel, conv::kFlip4, bias);
                    o.z = conv::pair_to_half2(lo[4], lo[5], sel, conv::kFlip4, bias);
                    o.w = conv::pair_to_half2(lo[6], lo[7], sel, conv::kFlip4, bias);
                    *reinterpret_cast<uint4*>(out + (int64_t)(8 * pw + 2 * k + 1) * kp) = o;
                }
            }
        }
    }
}

// The whole GPU: many blocks, one tile each at a time; or, beside a tensor-core launch, few blocks
// with eight tiles of loads in flight each (blocks_per_sm > 0).  kp: samples of a plane row.
template <int BITS, bool F8>
cudaError_t launch_fast(const Plan& p, const void* d_packed, int n_dumps, void* planes, int kp, cudaStream_t s,
                        int blocks_per_sm) {
    using F = FastTile<BITS>;
    const int64_t n_tiles = (int64_t)n_dumps * p.n_chan * p.nb * (kp / kTimeBlock);
    if (n_tiles < 1) return cudaSuccess;
    if (n_tiles >= (int64_t{1} << 31)) return cudaErrorInvalidValue;
    const auto* src = static_cast<const unsigned char*>(d_packed);
    const int64_t bytes = (int64_t)n_dumps * p.n_time * p.n_chan * p.n_inputs * (BITS == 8 ? 2 : 1);
    const bool ragged = (int64_t)p.n_inputs * (BITS == 8 ? 2 : 1) % 16 != 0;
    const int64_t cap = (int64_t)p.n_sm * (blocks_per_sm > 0 ? blocks_per_sm : BITS == 8 ? 8 : 16);
    const dim3 grid((unsigned)(n_tiles < cap ? n_tiles : cap));
    auto kern = ragged ? unpack_fast_kernel<BITS, 1, F8, true>
                       : blocks_per_sm > 0 ? unpack_fast_kernel<BITS, 8, F8> : unpack_fast_kernel<BITS, 1, F8>;
    return launch_kernel(kern, grid, F::kThreads, 0, s, 1, false, src, p.n_inputs, p.n_chan, p.n_time, p.nb, kp,
                          (uint32_t)n_tiles, planes, bytes);
}

// Packed rows [row][row_bytes] -> [row][pitch], pitch a multiple of 16 bytes: rows that TMA can
// address (what lies between a row's end and the next row is never read).  A copy at the price of
// the packed samples twice over, where planes cost their two to four times as many bytes twice
// (75 inputs, 8-bit: 78 MB in, 83 out, against 284 MB of planes).
// FLOAT: rows of an odd number of 8-byte samples.
template <bool FLOAT>
__global__ void __launch_bounds__(256) repack_kernel(const unsigned char* __restrict__ packed,
                                                     unsigned char* __restrict__ out, uint32_t rows, int row_bytes,
                                                     int pieces, uint32_t rows_per_block, int64_t n_bytes) {
    grid_release();
    const uint32_t tail = FLOAT ? 0u : tail_word(packed, n_bytes);
    for (uint32_t r0 = blockIdx.x * rows_per_block; r0 < rows; r0 += gridDim.x * rows_per_block) {
        const uint32_t n = min(rows_per_block, rows - r0) * (uint32_t)pieces;
        uint4* dst = reinterpret_cast<uint4*>(out) + (int64_t)r0 * pieces;
        const int64_t base = (int64_t)r0 * row_bytes;
#pragma unroll 4
        for (uint32_t e = threadIdx.x; e < n; e += 256) {
            const uint32_t r = e / (uint32_t)pieces;
            const int64_t off = base + (int64_t)r * row_bytes + (e - r * pieces) * 16;
            if constexpr (FLOAT) {
                const uint2 a = *reinterpret_cast<const uint2*>(packed + off);
                const uint2 b = off + 16 <= n_bytes ? *reinterpret_cast<const uint2*>(packed + off + 8) : uint2{};
                dst[e] = make_uint4(a.x, a.y, b.x, b.y);
            } else {
                uint32_t x[4];
                load_piece(packed, off, n_bytes, 16, tail, x);
                dst[e] = make_uint4(x[0], x[1], x[2], x[3]);
            }
        }
    }
}

template <int OUT>
cudaError_t launch(const Plan& p, const void* d_packed, int n_dumps, void* o0, void* o1, cudaStream_t s) {
    const int64_t n_tiles = (int64_t)n_dumps * p.n_chan * p.nb * (p.kp / kTimeBlock);
    const int64_t cap = (int64_t)p.n_sm * 8;
    const int grid = (int)(n_tiles < cap ? n_tiles : cap);
    return launch_kernel(unpack_kernel<OUT>, dim3((unsigned)grid), kThreads, 0, s, 1, false,
                          static_cast<const float2*>(d_packed), p.n_inputs, p.n_chan, p.n_time, p.nb, p.kp,
                          n_tiles, o0, o1);
}

}  // namespace

cudaError_t launch_unpack_fp16(const Plan& p, const void* d_packed, int n_dumps, void* d_planes, cudaStream_t s,
                               int blocks_per_sm) {
    if (((reinterpret_cast<uintptr_t>(d_packed) | reinterpret_cast<uintptr_t>(d_planes)) & 15u) != 0)
        return cudaErrorInvalidValue;
    return p.sample_bits == 4 ? launch_fast<4, false>(p, d_packed, n_dumps, d_planes, p.kp, s, blocks_per_sm)
                              : launch_fast<8, false>(p, d_packed, n_dumps, d_planes, p.kp, s, blocks_per_sm);
}

cudaError_t launch_unpack_e4m3(const Plan& p, const void* d_packed, int n_dumps, void* d_planes, cudaStream_t s,
                               int blocks_per_sm) {
    if (p.sample_bits != 4 || (reinterpret_cast<uintptr_t>(d_packed) & 15u) || (reinterpret_cast<uintptr_t>(d_planes) & 15u))
        return cudaErrorInvalidValue;
    return launch_fast<4, true>(p, d_packed, n_dumps, d_planes, tc_kp_e4m3(p), s, blocks_per_sm);
}

int64_t repack_pitch(const Plan& p) {
    return ((int64_t)p.n_inputs * (p.sample_bits == 32 ? 8 : p.sample_bits == 8 ? 2 : 1) + 15) / 16 * 16;
}

cudaError_t launch_repack(const Plan& p, const void* d_packed, int n_dumps, void* d_out, cudaStream_t s) {
    const int64_t rows = (int64_t)n_dumps * p.n_time * p.n_chan;
    const int row_bytes = p.n_inputs * (p.sample_bits == 32 ? 8 : p.sample_bits == 8 ? 2 : 1);
    if (rows >= (int64_t{1} << 31) ||
        ((reinterpret_cast<uintptr_t>(d_packed) | reinterpret_cast<uintptr_t>(d_out)) & 15u) != 0)
        return cudaErrorInvalidValue;
    const int pieces = (int)(repack_pitch(p) / 16);
    const int per = 2048 / pieces > 0 ? 2048 / pieces : 1;
    const int64_t want = (rows + per - 1) / per, cap = (int64_t)p.n_sm * 8;
    return launch_kernel(p.sample_bits == 32 ? repack_kernel<true> : repack_kernel<false>, dim3((unsigned)(want < cap ? want : cap)), 256, 0, s, 1, false,
                          static_cast<const unsigned char*>(d_packed), static_cast<unsigned char*>(d_out), (uint32_t)rows,
                          row_bytes, pieces, (uint32_t)per, rows * row_bytes);
}

cudaError_t launch_unpack_f32(const Plan& p, const void* d_packed, int n_dumps, void* d_planes, cudaStream_t s) {
    return launch<kOutF32>(p, d_packed, n_dumps, d_planes, nullptr, s);
}

cudaError_t launch_unpack_bf16x2(const Plan& p, const void* d_packed, int n_dumps, void* d_hi, void* d_lo,
                                 cudaStream_t s) {
    return launch<kOutBF16Split>(p, d_packed, n_dumps, d_hi, d_lo, s);
}

}  // namespace corr
