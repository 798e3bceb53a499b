// F stage: transforms of 32 points and more, and the polyphase filterbank with its window in
// registers.  fengine.cu keeps the rest (fwide_takes below).
//
// Why not its layout.  fengine.cu gives a CTA 4096 points in two buffers: a 2048-point transform
// leaves two inputs per CTA, every load and store touches 2 to 16 bytes of a row and the L1
// wavefronts bound the kernel (128 inputs x 1024 real channels x 512 frames: 675 us, 82% of L1, 12%
// of DRAM, against 100 us for the bytes; 217 us here), and an array of 16 inputs leaves a short
// transform's CTA mostly empty.  Here the values of a Stockham stage stay in registers between its
// reads and its writes, so one buffer is enough, a CTA of T threads holds 16 T points (16 per
// thread), rows of up to 16 inputs go out as whole lines and a CTA takes several frames of a short
// transform.  What bounds it: the shared-memory port (60% busy with barriers between its phases).
//
// Real samples take half the points: z[n] = x[2n] + i x[2n + 1] is transformed at half length
// H = L / 2 and split, X[k] = E + W O and X[H - k] = conj(E - W O) with
// E = (Z[k] + conj Z[H - k]) / 2, O = -i (Z[k] - conj Z[H - k]) / 2, W = exp(-2 pi i k / L): both
// halves come from one input, so no input's rounding reaches another.  The last stage's task p
// yields channels p + q H / R and its mirror task H / R - p the partners, so a thread that does
// both tasks splits in registers.
//
// Columns.  A CTA transforms C = 16 T / H columns at a time, a column being one input of one
// frame: G inputs x FB frames.  Shared memory holds point i of column c at (pad(i) CP + c)
// float2, columns fastest, so every stage reads and writes runs of columns.
//
//   plain       packed samples of the next frames are copied to shared memory (cp.async) while
//               the present ones are transformed; the first stage unpacks them.
//   filterbank  (MT = 4 or 8 taps) y_f[s] = sum_m h[m L + s] x[(f + m) L + s].  A CTA walks a run
//               of consecutive frames and each thread keeps, for four points of every frame, the
//               MT - 1 partial sums that still wait for samples: a sample is loaded and unpacked
//               once and multiplied by MT taps, a_k <- a_{k+1} + h_{MT-2-k} x.  (fengine.cu reads
//               and unpacks every sample MT times through L2: 377 us for 64 inputs x 128 channels
//               x 10000 frames x 8 taps, 209 here, against 122 us for the bytes.)  Four frames of sums are
//               collected, then transformed together.
#include <cmath>
#include <type_traits>
#include <vector>

#include "corr_internal.h"
#include "fengine_wide.h"
#include "fft_reg.cuh"
#include "launch.cuh"

namespace corr {
namespace {

// ---- radices: 2 or 3 stages; the last one at most 8 where real spectra are split ----
__host__ __device__ constexpr int fw_stages(int lgh, bool real) { return lgh < 8 || (lgh == 8 && !real) ? 2 : 3; }
__host__ __device__ constexpr int fw_lgr(int lgh, bool real, int st) {
    if (lgh == 4) return 2;
    if (lgh == 5) return st == 0 ? 3 : 2;
    if (lgh == 6) return 3;
    if (lgh == 7) return st == 0 ? 4 : 3;
    if (lgh == 8) return real ? (st == 2 ? 2 : 3) : 4;
    if (lgh == 9) return 3;
    if (lgh == 10) return st == 0 ? 4 : 3;
    if (lgh == 11) return st == 2 ? 3 : 4;
    return 4;
}
__host__ __device__ constexpr int fw_lgns(int lgh, bool real, int st) {   // log2 of the product of earlier radices
    int o = 0;
    for (int u = 0; u < st; ++u) o += fw_lgr(lgh, real, u);
    return o;
}
// twiddle tables: stage st (>= 1) holds exp(-2 pi i k r / (Ns R)) at k (R - 1) + r - 1; after the
// stages, for real samples, w = exp(-2 pi i (p + q H / R) / L) at p R + q for p = 0 .. H / R / 2 of the
// last stage (one rounding each: a task's root times a 16th root cost 5 to 20% in the error), and in
// the same order what w's rounding dropped (FW::kExact)
__host__ __device__ constexpr int fw_tw_offset(int lgh, bool real, int st) {
    int o = 0;
    for (int u = 1; u < st; ++u) o += (1 << fw_lgns(lgh, real, u)) * ((1 << fw_lgr(lgh, real, u)) - 1);
    return o;
}
__host__ __device__ constexpr int fw_split_entries(int lgh, bool real) {
    const int lgr = fw_lgr(lgh, real, fw_stages(lgh, real) - 1);
    return real ? (1 << (lgh - 1)) + (1 << lgr) : 0;
}
__host__ __device__ constexpr int fw_tw_entries(int lgh, bool real) {
    return fw_tw_offset(lgh, real, fw_stages(lgh, real)) + fw_split_entries(lgh, real);
}

// ---- geometry of one kernel ----
// Threads: as few as leave rows of 16 inputs (whole 128-byte lines; several CTAs per SM hide each
// other's barriers): 2048 real samples with 4 / 8 / 16 inputs a row 235 / 147 / 114 us, 2048 complex
// ones with 4 / 8 354 / 216 us (2^26 samples).  The filterbank's partial sums take 128 registers a
// thread: 512 threads (256 with half the rows: 248 -> 218 us at L = 256, 8 taps).
__host__ __device__ constexpr int fw_threads(int lgh, int mt) {
    if (mt) return 512;
    return lgh <= 8 ? 256 : lgh == 9 ? 512 : 1024;
}

// ROW < 16: plain transforms in CTAs of 4096 points, with rows of at most ROW inputs (plain_row).  A column's
// arithmetic is the same in every geometry, and so are its bits.
template <int KIND, int LGL, int MT, int ROW = 16>
struct FW {
    static constexpr bool kReal = KIND == CORR_F_REAL8;
    static constexpr int BPS = f_bps<KIND>();
    static constexpr int L = 1 << LGL, LGH = LGL - (kReal ? 1 : 0), H = 1 << LGH;
    static constexpr int T = ROW < 16 ? 256 : fw_threads(LGH, MT);
    static constexpr int C = 16 * T / H;                       // columns
    static constexpr int G = MT ? C / 4 : (C < ROW ? C : ROW);   // inputs (16: whole 128-byte lines out)
    static constexpr int FB = C / G;                           // frames per batch
    static constexpr int NST = fw_stages(LGH, kReal);
    static constexpr int PS = fw_lgr(LGH, kReal, 0);           // one pad row after every first radix of rows
    // row pitch: the filterbank's 16-byte stores of a quarter-warp (2 x 4 rows, 1 x 8 rows for
    // few inputs) then fall in distinct banks
    static constexpr int CP = C + (MT && G == 8 ? 8 : MT && G == 4 ? 4 : MT && G == 2 ? 2 : 0);
    static constexpr int NOUT = kReal ? H + 1 : H;
    // How far a real spectrum's split keeps its roundings (fw_split): as far as the error must not exceed that
    // of the full-length transform, whose 0.97 to 1.08 a plain split has (least for plain transforms of
    // 512 points and more, most for filterbanks of 64).
    static constexpr int kExact = !kReal ? 0 : MT == 0 ? (LGL == 8 ? 1 : 0) : (LGL <= 8 || LGL == 11 ? 3 : 2);
    static constexpr int TWN = fw_tw_entries(LGH, kReal) + (kExact > 0 ? fw_split_entries(LGH, kReal) : 0);
    static constexpr int ROWB = G * BPS;                       // packed bytes of a sample row
    static constexpr int PIECE = ROWB < 16 ? ROWB : 16;        // bytes of one asynchronous copy, at most
    static constexpr int RAWB = MT ? 0 : FB * L * ROWB;        // packed bytes of a batch
    static constexpr int DATA = ((H - 1) + ((H - 1) >> PS) + 1) * CP;   // float2
    static constexpr int SMEM = (DATA + TWN) * 8 + RAWB + 16;
    static_assert(C >= 1 && (C & (C - 1)) == 0 && T % C == 0, "columns");
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static __host__ __device__ constexpr int pad(int i) { return i + (i >> PS); }
};

// read one stage's tasks into registers, apply its twiddles and DFTs
template <class F, int ST, int IT, int R>
__device__ __forceinline__ void fw_read(float2 (&v)[IT][R], const float2* buf, const float2* tws) {
    constexpr int LGNS = fw_lgns(F::LGH, F::kReal, ST), NS = 1 << LGNS, LR = F::H / R;
    const int c = threadIdx.x & (F::C - 1);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = (threadIdx.x + it * F::T) / F::C;
        const float2* src = buf + F::pad(j) * F::CP + c;
#pragma unroll
        for (int r = 0; r < R; ++r) v[it][r] = src[F::pad(r * LR) * F::CP];
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = (threadIdx.x + it * F::T) / F::C, k = j & (NS - 1);
        const float2* t = tws + fw_tw_offset(F::LGH, F::kReal, ST) + k * (R - 1) - 1;
#pragma unroll
        for (int r = 1; r < R; ++r) v[it][r] = cmul(v[it][r], t[r]);
        dft_reg<R>(v[it]);
    }
}

template <class F, int ST, int IT, int R>
__device__ __forceinline__ void fw_write(const float2 (&v)[IT][R], float2* buf) {
    constexpr int LGNS = fw_lgns(F::LGH, F::kReal, ST), NS = 1 << LGNS;
    const int c = threadIdx.x & (F::C - 1);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = (threadIdx.x + it * F::T) / F::C, k = j & (NS - 1);
        float2* dst = buf + F::pad((j - k) * R + k) * F::CP + c;
#pragma unroll
        for (int q = 0; q < R; ++q) dst[F::pad(q * NS) * F::CP] = v[it][q];
    }
}

// a + b = s + e exactly (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}

// a b = p + e exactly
__device__ __forceinline__ float two_prod(float a, float b, float& e) {
    const float p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
    return p;
}

// X[k] and X[H - k] from Z[k] and Z[H - k]; w = exp(-2 pi i k / L), wl what its rounding dropped.  The sums
// and differences 2 E and 2 O always keep their rounding errors.  EXACT = 1 adds wl and the errors
// of one product each of 2 W O, 2 those of both and of their sum, 3 that of the last sum as well, which
// leaves the rounding of the result.  Error relative to the full-length transform's, and time of 2^26
// samples of 128 inputs, 0 -> the one chosen (FW::kExact): filterbanks of 8 taps, L = 32 1.05 -> 0.97, 94
// -> 116 us; 64 1.06 -> 0.99, 97 -> 124; 128 1.05 -> 1.00, 116 -> 145; 256 1.03 -> 0.98, 127 -> 158; 512
// 1.02 -> 0.99, 170 -> 180; 1024 1.02 -> 0.99, 242 -> 269; 2048 1.03 -> 0.99, 436 -> 465; plain, L = 256
// 1.005 -> 0.97, 86 -> 89.
template <int EXACT>
__device__ __forceinline__ void fw_split(float2 z, float2 zp, float2 w, float2 wl, float2& xk, float2& xm) {
    float er, ei, fr, fi;
    const float sr = two_sum(z.x, zp.x, er), si = two_sum(z.y, -zp.y, ei);   // 2 E
    const float dr = two_sum(z.y, zp.y, fr), di = two_sum(zp.x, -z.x, fi);   // 2 O
    if constexpr (EXACT == 0) {
        const float pr = fmaf(fr, w.x, fmaf(-fi, w.y, fmaf(dr, w.x, -(di * w.y))));   // 2 W O
        const float pi = fmaf(fr, w.y, fmaf(fi, w.x, fmaf(dr, w.y, di * w.x)));
        xk = make_float2(0.5f * (sr + (pr + er)), 0.5f * (si + (pi + ei)));
        xm = make_float2(0.5f * (sr - (pr - er)), 0.5f * ((pi - ei) - si));
    } else {
        float b, d, pr, pi, cr, ci;   // 2 W O = pr + cr, pi + ci
        const float p1 = two_prod(di, w.y, b), q1 = two_prod(di, w.x, d);
        if constexpr (EXACT == 1) {
            pr = fmaf(dr, w.x, -p1);
            pi = fmaf(dr, w.y, q1);
            cr = -b;
            ci = d;
        } else {
            float a, c, e, f;
            const float p0 = two_prod(dr, w.x, a), q0 = two_prod(dr, w.y, c);
            pr = two_sum(p0, -p1, e);
            pi = two_sum(q0, q1, f);
            cr = e + (a - b);
            ci = f + (c + d);
        }
        cr = fmaf(dr, wl.x, fmaf(-di, wl.y, fmaf(fr, w.x, fmaf(-fi, w.y, cr))));
        ci = fmaf(dr, wl.y, fmaf(di, wl.x, fmaf(fr, w.y, fmaf(fi, w.x, ci))));
        if constexpr (EXACT < 3) {
            xk = make_float2(0.5f * (sr + (pr + (cr + er))), 0.5f * (si + (pi + (ci + ei))));
            xm = make_float2(0.5f * (sr - (pr + (cr - er))), 0.5f * ((pi + (ci - ei)) - si));
        } else {
            float g;
            const float kr = two_sum(sr, pr, g);
            xk.x = 0.5f * (kr + (g + (er + cr)));
            const float ki = two_sum(si, pi, g);
            xk.y = 0.5f * (ki + (g + (ei + ci)));
            const float mr = two_sum(sr, -pr, g);
            xm.x = 0.5f * (mr + (g + (er - cr)));
            const float mi = two_sum(pi, -si, g);
            xm.y = 0.5f * (mi + (g + (ci - ei)));
        }
    }
}

// the dropped part of the root at w, for FW::kExact
template <class F>
__device__ __forceinline__ float2 fw_low(const float2* w) {
    if constexpr (F::kExact > 0) return w[fw_split_entries(F::LGH, true)];
    else return float2{};
}

template <class F, int R, int Q>
__device__ __forceinline__ void fw_split_pairs(const float2 (&a)[R], const float2 (&b)[R], const float2* w, float2* o,
                                               int N, int p) {
    if constexpr (Q < R) {   // channel p + q H / R and its mirror, output R - 1 - q of the mirror task
        constexpr int NS = F::H / R;
        float2 xk, xm;
        fw_split<F::kExact>(a[Q], b[R - 1 - Q], w[Q], fw_low<F>(w + Q), xk, xm);
        const int k = p + Q * NS;
        o[k * N] = xk;
        o[(F::H - k) * N] = xm;
        fw_split_pairs<F, R, Q + 1>(a, b, w, o, N, p);
    }
}

template <class F, int R, int Q>
__device__ __forceinline__ void fw_split_self(const float2 (&a)[R], const float2* w, float2* o, int N) {
    if constexpr (Q < R / 2) {   // task 0: channels q H / R, mirrored at R - q of the same task
        constexpr int NS = F::H / R;
        float2 xk, xm;
        fw_split<F::kExact>(a[Q], a[R - Q], w[Q], fw_low<F>(w + Q), xk, xm);
        o[Q * NS * N] = xk;
        o[(F::H - Q * NS) * N] = xm;
        fw_split_self<F, R, Q + 1>(a, w, o, N);
    }
}

template <class F, int R, int Q>
__device__ __forceinline__ void fw_split_mid(const float2 (&b)[R], const float2* w, float2* o, int N) {
    if constexpr (Q < R / 2) {   // task H / R / 2: channels (q + 1/2) H / R, mirrored at R - 1 - q
        constexpr int NS = F::H / R;
        float2 xk, xm;
        fw_split<F::kExact>(b[Q], b[R - 1 - Q], w[Q], fw_low<F>(w + Q), xk, xm);
        o[(NS / 2 + Q * NS) * N] = xk;
        o[(F::H - NS / 2 - Q * NS) * N] = xm;
        fw_split_mid<F, R, Q + 1>(b, w, o, N);
    }
}

// stages 1 .. last of the columns in `buf`; the last stage stores the spectra.  `o`: channel 0 of
// the thread's column in the output (null: the column does not exist).  Ends with every read of
// buf done by this thread only: the caller's next barrier orders them before new writes.
template <class F>
__device__ __forceinline__ void fw_rest(float2* buf, const float2* tws, float2* o, int N) {
    if constexpr (F::NST == 3) {
        constexpr int R = 1 << fw_lgr(F::LGH, F::kReal, 1), IT = 16 / R;
        float2 v[IT][R];
        fw_read<F, 1, IT, R>(v, buf, tws);
        __syncthreads();
        fw_write<F, 1, IT, R>(v, buf);
        __syncthreads();
    }
    constexpr int ST = F::NST - 1;
    constexpr int R = 1 << fw_lgr(F::LGH, F::kReal, ST), NS = F::H / R;
    if constexpr (!F::kReal) {
        constexpr int IT = 16 / R;
        float2 v[IT][R];
        fw_read<F, ST, IT, R>(v, buf, tws);
        if (o) {
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                const int j = (threadIdx.x + it * F::T) / F::C;
#pragma unroll
                for (int q = 0; q < R; ++q) o[(j + q * NS) * N] = v[it][q];
            }
        }
    } else {
        constexpr int IT = 8 / R;   // task pairs per thread
        const int c = threadIdx.x & (F::C - 1);
        const float2* split = tws + fw_tw_offset(F::LGH, true, F::NST);
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int p = (threadIdx.x + it * F::T) / F::C;
            const int j2 = p ? NS - p : NS / 2;
            float2 a[R], b[R];
            const float2* sa = buf + F::pad(p) * F::CP + c;
            const float2* sb = buf + F::pad(j2) * F::CP + c;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                a[r] = sa[F::pad(r * NS) * F::CP];
                b[r] = sb[F::pad(r * NS) * F::CP];
            }
            const float2* ta = tws + fw_tw_offset(F::LGH, true, ST) + p * (R - 1) - 1;
            const float2* tb = tws + fw_tw_offset(F::LGH, true, ST) + j2 * (R - 1) - 1;
#pragma unroll
            for (int r = 1; r < R; ++r) {
                a[r] = cmul(a[r], ta[r]);
                b[r] = cmul(b[r], tb[r]);
            }
            dft_reg<R>(a);
            dft_reg<R>(b);
            if (o) {
                if (p) {
                    fw_split_pairs<F, R, 0>(a, b, split + p * R, o, N, p);
                } else {
                    // channel 0 and the Nyquist channel, the mirrored rest of task 0, channel H / 2
                    o[0] = make_float2(a[0].x + a[0].y, 0.f);
                    o[F::H * N] = make_float2(a[0].x - a[0].y, 0.f);
                    fw_split_self<F, R, 1>(a, split, o, N);
                    o[F::H / 2 * N] = make_float2(a[R / 2].x, -a[R / 2].y);
                    fw_split_mid<F, R, 0>(b, split + NS / 2 * R, o, N);
                }
            }
        }
    }
}

__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int bytes) {
    if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else if (bytes == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// packed samples of `rows` sample rows of the CTA's inputs -> shared memory [row][G], in pieces of P bytes
// where rows and their first byte are multiples of that (plain_piece), else sample by sample.  ODD: shorter
// pieces than F::PIECE, or none, in a kernel of their own: beside the whole ones they cost those 3% (c8 1024 points,
// 176 inputs x 1087 frames 506 -> 520 us)
template <class F, int P>
__device__ __forceinline__ void fw_fetch_pieces(uint8_t* raw, const uint8_t* src, int rows, int N, int g_n) {
    constexpr int PP = F::ROWB / P;
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(raw));
    for (int e = threadIdx.x; e < rows * PP; e += F::T) {
        const int row = e / PP, pc = e % PP;
        if (pc * (P / F::BPS) < g_n) cp_async(dst + (uint32_t)e * P, src + (size_t)row * N * F::BPS + pc * P, P);
    }
}

template <class F, bool ODD>
__device__ __forceinline__ void fw_fetch(uint8_t* raw, const uint8_t* src, int rows, int N, int g_n, int piece) {
    if constexpr (!ODD) return fw_fetch_pieces<F, F::PIECE>(raw, src, rows, N, g_n);
    if (F::PIECE > 8 && piece == 8) return fw_fetch_pieces<F, F::PIECE >= 8 ? 8 : F::ROWB>(raw, src, rows, N, g_n);
    if (F::PIECE > 4 && piece == 4) return fw_fetch_pieces<F, F::PIECE >= 4 ? 4 : F::ROWB>(raw, src, rows, N, g_n);
    // a thread's samples are rows apart: eight loads in flight
    using S = std::conditional_t<F::BPS == 2, unsigned short, uint8_t>;
    const int g = threadIdx.x % F::G;
    const S* in = reinterpret_cast<const S*>(src) + g;
    S* out = reinterpret_cast<S*>(raw) + g;
    constexpr int STEP = F::T / F::G;
    for (int row = threadIdx.x / F::G; row < rows; row += 8 * STEP) {
        S x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = g < g_n && row + u * STEP < rows ? in[(size_t)(row + u * STEP) * N] : S{};
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (row + u * STEP < rows) out[(row + u * STEP) * F::G] = x[u];
    }
}

// point i of a column from the packed rows at `raw` (the column's first sample)
template <class F, int KIND>
__device__ __forceinline__ float2 fw_point(const uint8_t* raw, int i) {
    if constexpr (KIND == CORR_F_COMPLEX8)
        return unpack1<KIND>(*reinterpret_cast<const unsigned short*>(raw + i * F::ROWB));
    else if constexpr (KIND == CORR_F_COMPLEX4) return unpack1<KIND>(raw[i * F::ROWB]);
    else return make_float2(unpack1<KIND>(raw[2 * i * F::ROWB]).x, unpack1<KIND>(raw[(2 * i + 1) * F::ROWB]).x);
}

template <int KIND, int LGL, int ROW, bool ODD>
__global__ void __launch_bounds__(FW<KIND, LGL, 0, ROW>::T, 1024 / FW<KIND, LGL, 0, ROW>::T)
    fengine_wide_kernel(const uint8_t* __restrict__ in, float2* __restrict__ out, const float2* __restrict__ tw, int N,
                        int n_frames, int piece) {
    using F = FW<KIND, LGL, 0, ROW>;
    extern __shared__ __align__(16) uint8_t fw_smem[];
    float2* const buf = reinterpret_cast<float2*>(fw_smem);
    float2* const tws = buf + F::DATA;
    uint8_t* const raw = reinterpret_cast<uint8_t*>(fw_smem) + ((F::DATA + F::TWN) * 8 + 15) / 16 * 16;
    const int n0 = blockIdx.x * F::G;
    const int g_n = min(F::G, N - n0);
    for (int k = threadIdx.x; k < F::TWN; k += F::T) tws[k] = tw[k];
    grid_release();
    const int n_batches = (n_frames + F::FB - 1) / F::FB;
    const size_t frame_bytes = (size_t)F::L * N * F::BPS;
    const uint8_t* const in0 = in + (size_t)n0 * F::BPS;
    const int c = threadIdx.x & (F::C - 1), cg = c % F::G, cf = c / F::G;   // the thread's column
    const uint8_t* const col = raw + cf * F::L * F::ROWB + cg * F::BPS;
    int b = blockIdx.y;
    if (b < n_batches)
        fw_fetch<F, ODD>(raw, in0 + (size_t)b * F::FB * frame_bytes, min(F::FB, n_frames - b * F::FB) * F::L, N, g_n, piece);
    for (; b < n_batches; b += gridDim.y) {
        cp_async_wait();
        __syncthreads();   // this batch's samples are here, and the last one's columns are read
        {
            constexpr int R = 1 << fw_lgr(F::LGH, F::kReal, 0), IT = 16 / R, LR = F::H / R;
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                const int j = (threadIdx.x + it * F::T) / F::C;
                float2 v[1][R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[0][r] = fw_point<F, KIND>(col, j + r * LR);
                dft_reg<R>(v[0]);
                float2* dst = buf + F::pad(j * R) * F::CP + c;
#pragma unroll
                for (int q = 0; q < R; ++q) dst[F::pad(q) * F::CP] = v[0][q];
            }
        }
        __syncthreads();
        // the samples are consumed: the next batch's arrive while the stages run
        const int bn = b + gridDim.y;
        if (bn < n_batches)
            fw_fetch<F, ODD>(raw, in0 + (size_t)bn * F::FB * frame_bytes, min(F::FB, n_frames - bn * F::FB) * F::L, N, g_n,
                        piece);
        const int f = b * F::FB + cf;
        float2* const o = (cg < g_n && f < n_frames) ? out + (size_t)f * F::NOUT * N + n0 + cg : nullptr;
        fw_rest<F>(buf, tws, o, N);
    }
}

// Filterbank of at most MT taps: CTA (x, y) takes inputs n0 .. n0 + G - 1 and the frames of run y.
// Thread: the four points i of inputs n0 + 4 gv .. + 3 (real samples: rows 2 i and 2 i + 1); where a CTA
// has room for two inputs only, points i and i + T of both.
template <int KIND, int LGL, int MT>
__global__ void __launch_bounds__(FW<KIND, LGL, MT>::T, 512 / FW<KIND, LGL, MT>::T)
    fengine_pfb_kernel(const uint8_t* __restrict__ in, float2* __restrict__ out, const float2* __restrict__ tw, int N,
                       int n_frames, int run, const float* __restrict__ taps, int M, int vec) {
    using F = FW<KIND, LGL, MT>;
    constexpr int SPP = F::kReal ? 2 : 1;                    // samples per point
    constexpr int QV = F::G < 4 ? F::G : 4, NI = 4 / QV;                   // inputs and points of each of a thread
    constexpr int NR = NI * SPP;                             // its sample rows
    constexpr int VB = QV * F::BPS;                          // bytes of QV inputs of a sample
    extern __shared__ __align__(16) uint8_t fw_smem[];
    float2* const buf = reinterpret_cast<float2*>(fw_smem);
    float2* const tws = buf + F::DATA;
    for (int k = threadIdx.x; k < F::TWN; k += F::T) tws[k] = tw[k];
    const int n0 = blockIdx.x * F::G;
    const int g_n = min(F::G, N - n0);
    const int f0 = blockIdx.y * run, f1 = min(n_frames, f0 + run);
    const int n_in = n_frames + M - 1;                       // input frames
    const int gv = threadIdx.x % (F::G / QV), i = threadIdx.x / (F::G / QV);
    const size_t frame_bytes = (size_t)F::L * N * F::BPS;
    const uint8_t* const src = in + ((size_t)SPP * i * N + n0 + QV * gv) * F::BPS;
    const int g_left = g_n - QV * gv;                        // inputs of the thread's that exist
    using Raw = std::conditional_t<VB == 8, uint2, uint32_t>;
    using Load = std::conditional_t<VB == 2, unsigned short, Raw>;
    auto row = [](int s) { return s / SPP * F::T * SPP + s % SPP; };   // sample row s of the thread, from its first
    auto load = [&](int t, Raw (&w)[NR]) {                   // input frame t: its packed samples, or zeros
#pragma unroll
        for (int s = 0; s < NR; ++s) {
            w[s] = Raw{};
            if (t >= n_in || g_left <= 0) continue;
            const uint8_t* p = src + (size_t)t * frame_bytes + (size_t)row(s) * N * F::BPS;
            if (vec) {
                w[s] = *reinterpret_cast<const Load*>(p);
            } else {
                uint32_t u[2] = {0u, 0u};
#pragma unroll
                for (int k = 0; k < QV; ++k)
                    if (k < g_left) {
                        const uint32_t x = F::BPS == 2 ? (uint32_t)*reinterpret_cast<const unsigned short*>(p + 2 * k)
                                                       : (uint32_t)p[k];
                        u[(k * F::BPS) >> 2] |= x << (((k * F::BPS) & 3) * 8);
                    }
                if constexpr (VB == 8) w[s] = make_uint2(u[0], u[1]);
                else w[s] = u[0];
            }
        }
    };
    auto point = [&](const Raw (&w)[NR], int q) -> float2 {   // point q: input q % QV, row q / QV
        const int k = q % QV, s = q / QV * SPP;
        if constexpr (KIND == CORR_F_COMPLEX8) {
            uint32_t u;
            if constexpr (VB == 8) u = (k < 2 ? w[s].x : w[s].y) ^ 0x80808080u;
            else u = w[s] ^ 0x80808080u;
            const uint32_t b0 = 2u * (k & 1);
            return make_float2(f_byte(u, 0x7540u | b0, kBias8), f_byte(u, 0x7541u + b0, kBias8));
        } else if constexpr (KIND == CORR_F_COMPLEX4) {
            const uint32_t u = w[s] ^ 0x88888888u;
            return make_float2(f_byte((u >> 4) & 0x0F0F0F0Fu, 0x7540u | (uint32_t)k, kBias4),
                               f_byte(u & 0x0F0F0F0Fu, 0x7540u | (uint32_t)k, kBias4));
        } else {
            return make_float2(f_byte(w[s] ^ 0x80808080u, 0x7540u | (uint32_t)k, kBias8),
                               f_byte(w[s + 1] ^ 0x80808080u, 0x7540u | (uint32_t)k, kBias8));
        }
    };
    float h[MT][NR];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int s = 0; s < NR; ++s) h[m][s] = m < M ? taps[m * F::L + SPP * i + row(s)] : 0.f;
    float2 a[MT - 1][4];   // a[k]: partial sum of the output frame that k + 1 more samples complete
#pragma unroll
    for (int k = 0; k < MT - 1; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[k][q] = make_float2(0.f, 0.f);
    // taps past M are zero, so frame f completes with input frame f + MT - 1 (zeros past the last)
    auto step = [&](const Raw (&w)[NR], float2 (&y)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 x = point(w, q);
            const int s0 = q / QV * SPP, s1 = s0 + SPP - 1;
            y[q] = make_float2(fmaf(h[MT - 1][s0], x.x, a[0][q].x), fmaf(h[MT - 1][s1], x.y, a[0][q].y));
#pragma unroll
            for (int k = 0; k < MT - 2; ++k)
                a[k][q] = make_float2(fmaf(h[MT - 2 - k][s0], x.x, a[k + 1][q].x),
                                      fmaf(h[MT - 2 - k][s1], x.y, a[k + 1][q].y));
            a[MT - 2][q] = make_float2(h[0][s0] * x.x, h[0][s1] * x.y);
        }
    };
    Raw w[4][NR];
    grid_release();
    if (f0 < f1) {
        for (int t = f0; t < f0 + MT - 1; ++t) {   // the run's first sums
            float2 y[4];
            load(t, w[0]);
            step(w[0], y);
        }
    }
    const int c = threadIdx.x & (F::C - 1), cg = c % F::G, cf = c / F::G;
    const bool second = (threadIdx.x >> 2) & 1;   // which half of the four goes first (distinct banks)
    float2* const wr = buf + F::pad(i) * F::CP + QV * gv;
#pragma unroll
    for (int fb = 0; fb < 4; ++fb) load(f0 + MT - 1 + fb, w[fb]);
    for (int f = f0; f < f1; f += 4) {
        __syncthreads();   // the previous frames' columns are read
#pragma unroll
        for (int fb = 0; fb < 4; ++fb) {
            float2 y[4];
            step(w[fb], y);
            const float4 lo = make_float4(y[0].x, y[0].y, y[1].x, y[1].y);
            const float4 hi = make_float4(y[2].x, y[2].y, y[3].x, y[3].y);
            float4* const d = reinterpret_cast<float4*>(wr + fb * F::G);
            if constexpr (QV == 4) {
                d[second ? 1 : 0] = second ? hi : lo;
                d[second ? 0 : 1] = second ? lo : hi;
            } else {
                d[0] = lo;
                d[F::pad(F::T) * F::CP / 2] = hi;   // point i + T (pad(i + T) = pad(i) + pad(T))
            }
        }
#pragma unroll
        for (int fb = 0; fb < 4; ++fb) load(f + 4 + MT - 1 + fb, w[fb]);
        __syncthreads();
        {
            constexpr int R = 1 << fw_lgr(F::LGH, F::kReal, 0), IT = 16 / R, LR = F::H / R;
            float2 v[IT][R];
#pragma unroll
            for (int it = 0; it < IT; ++it) {
                const int j = (threadIdx.x + it * F::T) / F::C;
                const float2* s = buf + F::pad(j) * F::CP + c;
#pragma unroll
                for (int r = 0; r < R; ++r) v[it][r] = s[F::pad(r * LR) * F::CP];
                dft_reg<R>(v[it]);
            }
            __syncthreads();
            fw_write<F, 0, IT, R>(v, buf);
            __syncthreads();
        }
        float2* const o = (cg < g_n && f + cf < f1) ? out + (size_t)(f + cf) * F::NOUT * N + n0 + cg : nullptr;
        fw_rest<F>(buf, tws, o, N);
    }
}

// rows of CTAs along the frames, each with the same number of batches: the number of waves whose
// waves x (batches of a CTA + 1) is least, the 1 being what a CTA spends before its first batch.  One
// wave alone leaves up to half the chip idle when the groups are more than half of it.
// *walk: the batches that a slot then takes one after another.
int fw_rows(int groups, int n_batches, int slots, long long* walk = nullptr) {
    const int w0 = (groups + slots - 1) / slots;
    long long best_cost = 0;
    int best = 1;
    for (int w = w0; w < w0 + 8; ++w) {
        long long rows = (long long)w * slots / groups;
        if (rows > n_batches) rows = n_batches;
        const long long per = (n_batches + rows - 1) / rows, cost = w * (per + 1);
        if (w == w0 || cost < best_cost) {
            best_cost = cost;
            best = (int)((n_batches + per - 1) / per);
            if (walk) *walk = w * per;
        }
    }
    return best > 65535 ? 65535 : best;
}

template <class F>
constexpr int plain_per_sm() {
    return 1024 / F::T < 227 * 1024 / (F::SMEM + 1024) ? 1024 / F::T : 227 * 1024 / (F::SMEM + 1024);
}

// bytes of the pieces a sample row can be fetched in (0: single samples)
template <class F>
int plain_piece(const FWideArgs& p) {
    for (int piece = 16; piece >= 4; piece /= 2)
        if (piece <= F::PIECE && (size_t)p.n_inputs * F::BPS % piece == 0 && reinterpret_cast<uintptr_t>(p.d_in) % piece == 0)
            return piece;
    return 0;
}

template <int KIND, int LGL, int ROW>
cudaError_t launch_plain(const FWideArgs& p, cudaStream_t s) {
    using F = FW<KIND, LGL, 0, ROW>;
    const int piece = plain_piece<F>(p);
    auto kern = fengine_wide_kernel<KIND, LGL, ROW, true>;
    if constexpr (F::PIECE >= 4)
        if (piece == F::PIECE) kern = fengine_wide_kernel<KIND, LGL, ROW, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F::SMEM);
    if (e != cudaSuccess) return e;
    const int groups = (p.n_inputs + F::G - 1) / F::G;
    const int rows = fw_rows(groups, (p.n_frames + F::FB - 1) / F::FB, p.n_sm * plain_per_sm<F>());
    return launch_kernel(kern, dim3(groups, rows), F::T, F::SMEM, s, 1, false, static_cast<const uint8_t*>(p.d_in),
                          static_cast<float2*>(p.d_out), static_cast<const float2*>(p.d_tw), p.n_inputs, p.n_frames,
                          piece);
}

// Inputs of a row of a plain transform's CTAs.  Rows of 16 leave columns empty where the inputs are few or no
// multiple of 16 (one input of 2048 real points: 1/16 of the CTA) and give a call of few frames a few CTAs
// of 1024 threads.  CTAs of 4096 points with rows of 4 (of one, for one or two inputs of long
// transforms) cost 1.2 to 2.2 times as much for as many points where both are full, so the choice is by the
// batches that a slot walks, weighted.  us, rows of 16 -> chosen: c8 512 points, 1 / 8 inputs x 4096 frames
// 142 -> 50 / 126 -> 51; r8 2048 points, 2 inputs x 4096 frames 305 -> 61, 20 x 256 47 -> 23, 16 x 1 10.6 -> 6.4;
// c8 1024 points, 100 x 64 31 -> 27.  128 inputs and more keep rows of 16.
template <int KIND, int LGL>
int plain_row(const FWideArgs& p) {
    using W = FW<KIND, LGL, 0, 16>;
    using N = FW<KIND, LGL, 0, 4>;
    if (p.n_inputs <= 12 - W::LGH && W::LGH >= 10) return 1;   // up to 2 / 1 inputs of 1024 / 2048 points
    const int gn = (p.n_inputs + N::G - 1) / N::G, bn = (p.n_frames + N::FB - 1) / N::FB;
    if (W::LGH >= 9 && (long long)gn * bn <= p.n_sm) return 4;   // a CTA each at most
    long long walk_w = 0, walk_n = 0;
    fw_rows((p.n_inputs + W::G - 1) / W::G, (p.n_frames + W::FB - 1) / W::FB, p.n_sm * plain_per_sm<W>(), &walk_w);
    fw_rows(gn, bn, p.n_sm * plain_per_sm<N>(), &walk_n);
    // rows of one or two inputs (LGH 12, 11) write parts of sectors where there are more
    const double cost = W::LGH <= 8 ? 1.45 : W::LGH <= 10 ? 1.2 : W::LGH == 11 ? (p.n_inputs <= 6 ? 1.0 : 1.5)
                                                                               : (p.n_inputs <= 2 ? 0.9 : 2.2);
    return walk_n * cost <= walk_w ? 4 : 16;
}

template <int KIND, int LGL, int MT>
cudaError_t launch_pfb(const FWideArgs& p, cudaStream_t s) {
    using F = FW<KIND, LGL, MT>;
    auto kern = fengine_pfb_kernel<KIND, LGL, MT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F::SMEM);
    if (e != cudaSuccess) return e;
    const int groups = (p.n_inputs + F::G - 1) / F::G;
    const int batches = (p.n_frames + 3) / 4;
    const int rows = fw_rows(groups, batches, p.n_sm * (512 / F::T));
    const int run = (batches + rows - 1) / rows * 4;
    constexpr int kVec = F::G < 4 ? F::G : 4;
    const int vec = (size_t)p.n_inputs % kVec == 0 && reinterpret_cast<uintptr_t>(p.d_in) % (kVec * F::BPS) == 0;
    return launch_kernel(kern, dim3(groups, rows), F::T, F::SMEM, s, 1, false, static_cast<const uint8_t*>(p.d_in),
                          static_cast<float2*>(p.d_out), static_cast<const float2*>(p.d_tw), p.n_inputs, p.n_frames, run,
                          p.d_taps, p.n_taps, vec);
}

template <int KIND, int LGL>
cudaError_t launch_len(const FWideArgs& p, cudaStream_t s) {
    if constexpr (LGL <= (KIND == CORR_F_REAL8 ? 11 : 10)) {
        if (p.d_taps) return p.n_taps <= 4 ? launch_pfb<KIND, LGL, 4>(p, s) : launch_pfb<KIND, LGL, 8>(p, s);
    }
    if constexpr (KIND != CORR_F_REAL8 || LGL >= 8) {
        if (!p.d_taps) {
            const int row = plain_row<KIND, LGL>(p);
            constexpr int lgh = FW<KIND, LGL, 0>::LGH;
            if constexpr (lgh == 10 || lgh == 11)
                if (row == 1) return launch_plain<KIND, LGL, 1>(p, s);
            return row == 4 ? launch_plain<KIND, LGL, 4>(p, s) : launch_plain<KIND, LGL, 16>(p, s);
        }
    }
    return cudaErrorInvalidValue;
}

template <int KIND>
cudaError_t launch_kind(const FWideArgs& p, cudaStream_t s) {
    switch (p.log2L) {
        case 5: return launch_len<KIND, 5>(p, s);
        case 6: return launch_len<KIND, 6>(p, s);
        case 7: return launch_len<KIND, 7>(p, s);
        case 8: return launch_len<KIND, 8>(p, s);
        case 9: return launch_len<KIND, 9>(p, s);
        case 10: return launch_len<KIND, 10>(p, s);
        case 11: return launch_len<KIND, 11>(p, s);
        case 12: return launch_len<KIND, 12>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Which plans take these kernels (us on 2^26 samples, fengine.cu -> here).
// Plain complex transforms of 32 points and more: c8 of 128 inputs, L = 32 .. 4096: 138 -> 115,
// (110 -> 116), 126 -> 119, 153 -> 123, 238 -> 163, 274 -> 179, 465 -> 216, 1067 -> 402; 16 inputs,
// L = 64: 270 -> 115.  L = 64 of whole groups of 64 inputs stays with fengine.cu.
// Plain real transforms of 256 points and more: 112 -> 89, 194 -> 94, 226 -> 108, 339 -> 119,
// 755 -> 166.  Shorter ones keep fengine.cu.
// Filterbanks of up to 8 taps where four frames of at least two inputs fit: 8 taps, c8, L = 32 ..
// 512: 403 -> 158, 302 -> 163, 313 -> 178, 421 -> 212, 515 -> 331; r8, L = 32 .. 1024: 308 -> 116,
// 244 -> 124, 252 -> 145, 342 -> 158, 440 -> 180, 942 -> 269.  With two inputs, 8 taps, 128 / 336 inputs:
// c8, L = 1024: 1025 -> 577 / 1411 -> 582; r8, L = 2048: 1604 -> 465 / 1418 -> 480, 4 taps 915 -> 404 /
// 882 -> 394.  Real spectra of either kind have no more error than the full-length transform (fw_split).
// The few taps of a long complex transform stay with fengine.cu, which pays for each tap: c8 of 128
// inputs, L = 512, 2 / 3 / 4 taps: 267 / 304 / 335 there, 313 here; c4, L = 256, 2 / 4 taps: 193 / 258
// there, 205 / 200 here; L = 1024, 4 / 6 taps: 476 / 823 there, 544 / 577 here.
// A CTA of the filterbank spends 3 or 7 frames of samples before its first batch of four, so calls that give
// a slot one batch, and fengine.cu no more than one either, stay there (8 taps, 1 input x 64 frames, r8
// L = 1024: 8.9 us there, 14.5 here; 256 inputs x 8 frames 41 there, 19 here), except the cheap ones (complex, up
// to 128 points, up to 4 taps: 7.5 there, 6.3 here); and so do the few taps of short transforms where groups
// are part empty or more than one (L = 32, 1 tap, 16 inputs, c8 / r8: 1.2 / 1.6 times faster there; 64 points, 1 / 2
// taps, 40 to 256 inputs 1.2 / 1.05; r8 2048 points, 1 tap 1.1).
bool fwide_takes(int kind, int log2L, int n_inputs, int n_taps, int n_frames, int n_sm) {
    const bool real = kind == CORR_F_REAL8;
    if (log2L < 5) return false;
    if (n_taps == 0) {
        // rows of no whole words, of 64 and 128 points: read sample by sample, better there (c4, 50 inputs, 31 / 60
        // us there, 42 / 84 here)
        if (!real && (log2L == 6 || log2L == 7) && n_inputs > 32 && n_inputs * (kind == CORR_F_COMPLEX8 ? 2 : 1) % 4) return false;
        return real ? log2L >= 8 : log2L != 6 || n_inputs % 64 != 0;
    }
    if (n_taps > 8 || log2L > (real ? 11 : 10)) return false;
    const int group = 2048 >> (log2L - (real ? 1 : 0));   // inputs of a CTA
    if (real) {
        if (log2L == 5 && n_inputs <= 64) return false;
        if (n_taps == 1 && (log2L <= 8 || log2L == 11) && log2L != 5) return false;
        if (n_taps == 2 && log2L <= 7 && n_inputs < 8) return false;
    } else {
        if (log2L >= 8 && n_taps < log2L - 5) return false;
        if (log2L == 5 && (n_taps == 1 || (n_taps == 2 && n_inputs % 4))) return false;
        if ((log2L == 6 || log2L == 7) && n_taps <= 2 && n_inputs > group) return false;
        if (log2L < 8 && n_taps <= 4) return true;
    }
    long long walk = 0;
    fw_rows((n_inputs + group - 1) / group, (n_frames + 3) / 4, n_sm, &walk);
    const long long there = log2L >= 6 ? 4096 >> log2L : 64;   // fengine.cu's inputs per CTA, two CTAs per SM
    return walk >= 2 || (n_inputs + there - 1) / there * n_frames > 2LL * n_sm;
}

std::vector<float2> fwide_tables(int kind, int log2L) {
    const bool real = kind == CORR_F_REAL8;
    const int lgh = log2L - (real ? 1 : 0);
    std::vector<float2> tw;
    auto root = [](int num, int den) {   // exp(-2 pi i num / den), rounded from double
        const double ang = -2.0 * M_PI * (double)num / (double)den;
        return make_float2((float)cos(ang), (float)sin(ang));
    };
    for (int st = 1; st < fw_stages(lgh, real); ++st) {
        const int ns = 1 << fw_lgns(lgh, real, st), r_ = 1 << fw_lgr(lgh, real, st);
        for (int k = 0; k < ns; ++k)
            for (int r = 1; r < r_; ++r) tw.push_back(root(k * r, ns * r_));
    }
    if (real) {
        const int r_ = 1 << fw_lgr(lgh, real, fw_stages(lgh, real) - 1), ns = (1 << lgh) / r_;
        for (int low = 0; low < 2; ++low)
            for (int p = 0; p <= ns / 2; ++p)
                for (int q = 0; q < r_; ++q) {
                    const float2 w = root(p + q * ns, 1 << log2L);
                    const double ang = -2.0 * M_PI * (double)(p + q * ns) / (double)(1 << log2L);
                    tw.push_back(low ? make_float2((float)(cos(ang) - (double)w.x), (float)(sin(ang) - (double)w.y)) : w);
                }
    }
    return tw;
}

cudaError_t launch_fwide(const FWideArgs& p, cudaStream_t s) {
    if (p.kind == CORR_F_COMPLEX8) return launch_kind<CORR_F_COMPLEX8>(p, s);
    if (p.kind == CORR_F_COMPLEX4) return launch_kind<CORR_F_COMPLEX4>(p, s);
    return launch_kind<CORR_F_REAL8>(p, s);
}

}  // namespace corr
