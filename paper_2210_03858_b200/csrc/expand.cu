// Forward (Eq. 2) and input gradient (Eq. 3) kernels of the BCQ linear layer.
//
//   forward   D[j, t] = sum_k  W_hat[j, k] * X[t, k]
//   dX        D[k, t] = sum_j  W_hat[j, k] * dY[t, j]
//
// W_hat = sum_i alpha_i b_i (Eq. 1) never exists in global memory: worker warps rebuild it tile by
// tile from the packed planes, straight into the 128-byte-swizzled shared-memory operand layout of
// tcgen05.mma (K-major for the forward, where j is the M index; MN-major for dX, where k is the M
// index and one 128-byte line holds 64 consecutive k of one row j).  Accumulators live in tensor
// memory (128 lanes x TN fp32 columns).
//
// Number format.  A scaled weight rounded to bf16 (8 significant bits) alone already costs about
// 1.7e-3 relative error on the outputs, so both operands are fp16 (11 bits):
//   * the scaled weight takes one of 2^q values per (row, group).  For q <= 4 the workers build
//     a byte-wise lookup table of the fp16 levels in four registers and index it with PRMT; the
//     selector nibbles are stored instead of the planes (lut.cuh).  For q = 4 the table holds the
//     eight levels with b_4 = +1; b_4 = -1 mirrors the index and flips the sign.  q > 4 falls back
//     to fp32 sums of +-alpha_i.
//   * activations are bf16 at the interface.  A short pre-pass writes them to the workspace as
//     fp16, each token row multiplied by a power of two that brings its largest magnitude to
//     2^14..2^15 (exact; undone in the epilogue), so neither large activations nor small
//     gradients leave the fp16 range.  The same pre-pass finds max|alpha|, from which a power of
//     two for the weights is derived.
//   * q > 4: the sums come out in the order 0,4,1,5,2,6,3,7 of a byte of a plane word, so the pre-pass,
//     which regroups the plane words anyway, stores the bits of every byte as 0,2,4,6,1,3,5,7.
#include <algorithm>

#include "expand_rules.h"
#include "gemm_common.cuh"
#include "lut.cuh"

namespace {

using namespace bcq;

__device__ int g_timeout_flag = 0;

enum { MODE_FWD = 0, MODE_BWDX = 1 };
enum { QM_LUT3 = 0, QM_LUT4 = 1, QM_GENERIC = 2 };

// 16 weights of one row (bits 0..15 of the plane words w) as fp32 sums of +-alpha_i, any q <= 8, stored as two
// 16-byte chunks (slots chunk0, chunk0 + 1) of the 128-byte line at `line` (swizzle key lx); a[i] = scales.
__device__ __forceinline__ void expand16_sum(const uint32_t (&w)[BCQ_MAX_Q], const float (&a)[BCQ_MAX_Q],
                                             int q, uint32_t line, uint32_t lx, uint32_t chunk0) {
    float v[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) v[p] = 0.0f;
#pragma unroll
    for (int i = 0; i < BCQ_MAX_Q; ++i) {
        if (i < q) {
            const uint32_t ai = __float_as_uint(a[i]);
            const uint32_t nw = ~w[i];
#pragma unroll
            for (int p = 0; p < 16; ++p) v[p] += __uint_as_float(ai ^ ((nw << (31 - p)) & 0x80000000u));
        }
    }
#pragma unroll
    for (int cc = 0; cc < 2; ++cc)
        ptx::st_shared_v4(line + (((chunk0 + cc) ^ lx) << 4), pack_half2(v[8 * cc + 0], v[8 * cc + 4]),
                          pack_half2(v[8 * cc + 1], v[8 * cc + 5]), pack_half2(v[8 * cc + 2], v[8 * cc + 6]),
                          pack_half2(v[8 * cc + 3], v[8 * cc + 7]));
}

template <int QM>
struct NumWords {
    static constexpr int value = (QM == QM_GENERIC) ? BCQ_MAX_Q : 4;
};

// Stored words per 32 weights when the planes are kept as selector codes (q <= 4): the q = 4
// packing for four planes, the q = 3 packing for one to three (missing planes read as index bits 0).
template <int QM>
struct CodeWords {
    static constexpr int value = (QM == QM_LUT4) ? 4 : 3;
};

// ------------------------------------------------------------------------------------------
// pre-pass: activations -> fp16 with a per-token power-of-two scale; max |alpha|
// ------------------------------------------------------------------------------------------

constexpr int kMaxAlphaBlocks = 128;

// Head of the forward / dX workspace: max |alpha| of each pre-pass block that scanned alpha (bit patterns), zeros
// for blocks that there are not: a lane of the consumer takes four with one load, and nothing has to be read first.
struct WsHeader {
    uint32_t block_max[kMaxAlphaBlocks];
};

// Power of two for the weights: q * max|alpha| lands in [2^13, 2^14).  Called by whole warps.
__device__ __forceinline__ int weight_shift(const WsHeader* hdr, int q) {
    const uint4 v = ld(reinterpret_cast<const uint4*>(hdr->block_max) + (threadIdx.x & 31));
    uint32_t m = max(max(v.x, v.y), max(v.z, v.w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    return shift_for(exponent_of_bits(__float_as_uint(__uint_as_float(m) * (float)q)), 13);
}

struct PrepParams {
    int n, K, act_blocks;
    long long ld_in, ld_out;
    const __nv_bfloat16* in;
    __half* out;
    float* tok_inv_scale;  // [n]
    const float* alpha;
    long long alpha_count;
    WsHeader* hdr;
    // Weights regrouped into the chunks one pipeline stage consumes, each chunk contiguous so that
    // a single bulk copy brings it into shared memory (rows past d_out are written as zeros):
    //   forward  bits_t  [m_tile][kb][q][128 rows][2 words]   the 64 k of stage kb
    //            alpha_t [m_tile][G][q][128 rows]
    //   dX       bits_t  [u][jb][q][64 rows][4 words]         u = 128-wide k tile, jb = 64-row block
    //            alpha_t [jb][G][q][64 rows]
    int mode, d_out, q, G, pitch, num_kb, amax_blocks, bits_blocks;
    int row_tiles;   // ceil(d_out / 128)
    int alpha_w;     // groups to a block of the scales' regrouping: a power of two, at most 32
    int bits_cblk;   // ceil(pitch / 32): 32-word column blocks of the plane words
    const uint32_t* bits;
    float* alpha_t;
    uint32_t* bits_t;
    uint32_t* counters;  // zeroed for the GEMM kernel (arrivals at tiles that several pairs share)
    int num_counters;
};

// WPT warps per token row.  A lane keeps up to HELD 16-byte vectors of the row in registers between finding the row's
// largest magnitude and writing the scaled fp16 row.  Rows of up to 1024 WPT elements take HELD = 4 (40 registers), longer
// ones 8 (62, up to 16384 elements) or 12 (76, up to 24576): all of these are read once.  Rows past that go to <8, 4>
// and are read again from L2.
// The token blocks are bound by memory (n x K x 4 bytes; with a warp per token and two reads, 4096 x 6400 took 21 us and
// 4096 x 1600 8.5 us) and need warps in flight, so registers that no vector comes to cost time.  Whole forward, g = d_in,
// q = 3, 2048 tokens, with two reads / 12 vectors / the fewest that hold the row, us:
//   8200 -> 512 43.7 / 50.2 / 42.9    10240 -> 1024 59.9 / 63.8 / 57.9    16384 -> 512 62.8 / 64.7 / 60.3    20480 -> 512 74.0 / 69.1 / 69.1
// (12 vectors with two blocks of 90 registers an SM instead of three: 20480 -> 512 72.4).
// Blocks past the activation blocks scan alpha instead.
constexpr int kPrepWarps = 8;

__device__ __forceinline__ uint32_t max_mag_bf16x8(const uint4& x, int k0, int K) {
    if (k0 + 8 <= K) {
        // whole vector inside the row: magnitudes are 15-bit integers, compared two per word
        const uint32_t a = __vmaxu2(x.x & 0x7FFF7FFFu, x.y & 0x7FFF7FFFu);
        const uint32_t b = __vmaxu2(x.z & 0x7FFF7FFFu, x.w & 0x7FFF7FFFu);
        const uint32_t c = __vmaxu2(a, b);
        return max(c & 0xFFFFu, c >> 16);
    }
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
    uint32_t m = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (k0 + e < K) m = max(m, (xs[e >> 1] >> ((e & 1) * 16)) & 0x7FFFu);
    return m;
}

__device__ __forceinline__ uint4 scale_to_fp16x8(const uint4& x, int k0, int K, float scale) {
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
    if (k0 + 8 <= K) {
        // bf16 -> fp32 is a shift (low half) or a mask (high half); the product with a power of two
        // is exact and one conversion packs two of them
        uint4 o;
        uint32_t* ow = &o.x;
#pragma unroll
        for (int w = 0; w < 4; ++w)
            ow[w] = pack_half2(__uint_as_float(xs[w] << 16) * scale, __uint_as_float(xs[w] & 0xFFFF0000u) * scale);
        return o;
    }
    float f[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const uint32_t b = (xs[e >> 1] >> ((e & 1) * 16)) & 0xFFFFu;
        f[e] = (k0 + e < K) ? __uint_as_float(b << 16) * scale : 0.0f;
    }
    uint4 o;
    o.x = pack_half2(f[0], f[1]);
    o.y = pack_half2(f[2], f[3]);
    o.z = pack_half2(f[4], f[5]);
    o.w = pack_half2(f[6], f[7]);
    return o;
}

template <int WPT, int HELD = 4>
__global__ void __launch_bounds__(256, HELD == 12 ? 3 : 0) prepare_kernel(const PrepParams p) {
    constexpr bool AGAIN = WPT == kPrepWarps && HELD == 4;  // there may be more vectors than are held
    __shared__ uint32_t red[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_trigger();
    pdl_wait();
    // roles by block id: tokens, then max|alpha|, then the regrouping blocks.  The hardware starts
    // blocks in index order, and the short, latency-bound regrouping blocks should not queue
    // behind the register-heavy token blocks, so the ids run backwards.
    const int bid = (int)gridDim.x - 1 - (int)blockIdx.x;
    if (bid >= p.act_blocks + p.amax_blocks) {
        __shared__ uint32_t tile[128][33];
        int b = bid - p.act_blocks - p.amax_blocks;
        if (b >= p.bits_blocks) {
            b -= p.bits_blocks;
            // ---- scales of one plane, 128 rows x alpha_w groups: coalesced reads along the groups (alpha[i][j][c] is
            // contiguous over (j, c)), coalesced writes along the rows (rows past d_out become zeros).  All loads
            // of a thread are in flight at once: a block for all groups of 128 rows, one load at a time, took
            // 0.8 us for every second group (d_in = 20480, g = 128, 2048 tokens: 70 us for the pre-pass, now 37)
            const int w = p.alpha_w, shift = __ffs(w) - 1;
            const int cblk = (p.G + w - 1) >> shift;
            const int c0 = (b % cblk) << shift;
            const int rt = (b / cblk) % p.row_tiles;
            const int i = b / (cblk * p.row_tiles);
            const float* src = p.alpha + ((long long)i * p.d_out + (long long)rt * 128) * p.G + c0;
            const int rows_left = p.d_out - rt * 128;
            float held[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int e = threadIdx.x + 256 * k, r = e >> shift, c = e & (w - 1);
                held[k] = r < 128 && r < rows_left && c0 + c < p.G ? ld(src + (long long)r * p.G + c) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int e = threadIdx.x + 256 * k, r = e >> shift, c = e & (w - 1);
                if (r < 128) tile[r][c] = __float_as_uint(held[k]);
            }
            __syncthreads();
            for (int e = threadIdx.x; e < 128 * w; e += 256) {
                const int r = e & 127, c = e >> 7;
                if (c0 + c >= p.G) break;
                long long o;
                if (p.mode == MODE_FWD) {
                    o = (((long long)rt * p.G + c0 + c) * p.q + i) * 128 + r;
                } else {
                    const int jb = rt * 2 + (r >> 6), rr = r & 63;
                    if (jb >= p.num_kb) continue;
                    o = (((long long)jb * p.G + c0 + c) * p.q + i) * 64 + rr;
                }
                p.alpha_t[o] = __uint_as_float(tile[r][c]);
            }
            return;
        }
        // ---- plane words (q > 4), 128 rows x 32 words of one plane: coalesced reads into shared memory,
        // then coalesced writes of the stage chunks
        const int cb = b % p.bits_cblk;
        const int rt = (b / p.bits_cblk) % p.row_tiles;
        const int i = b / (p.bits_cblk * p.row_tiles);
        const uint32_t* src = p.bits + (long long)i * p.d_out * p.pitch;
        // all sixteen loads of a thread in flight at once: the block's time is one memory latency
        uint32_t held[16];
        const int col_l = cb * 32 + lane;
#pragma unroll
        for (int pass = 0; pass < 16; ++pass) {
            const int j = rt * 128 + pass * 8 + warp;
            held[pass] = (j < p.d_out && col_l < p.pitch) ? ld(src + (long long)j * p.pitch + col_l) : 0u;
        }
#pragma unroll
        for (int pass = 0; pass < 16; ++pass) {
            // even bits of every byte to its low nibble, odd bits to the high nibble: one PRMT
            // pair of the expansion emits weights 0,4,1,5,2,6,3,7 of a byte, so with the bits
            // stored as 0,2,4,6,1,3,5,7 the expanded tile comes out in natural k order
            uint32_t v = held[pass];
            uint32_t t = (v ^ (v >> 1)) & 0x22222222u;
            v ^= t ^ (t << 1);
            t = (v ^ (v >> 2)) & 0x0C0C0C0Cu;
            v ^= t ^ (t << 2);
            tile[pass * 8 + warp][lane] = v;
        }
        __syncthreads();
        const int t = threadIdx.x;
#pragma unroll 4
        for (int pass = 0; pass < 16; ++pass) {
            int r, cl;
            if (p.mode == MODE_FWD) { r = t >> 1; cl = pass * 2 + (t & 1); }
            else { r = (pass & 1) * 64 + (t >> 2); cl = (pass >> 1) * 4 + (t & 3); }
            const int col = cb * 32 + cl;
            if (col >= p.pitch) continue;
            long long o;
            if (p.mode == MODE_FWD) {
                const int kb = col >> 1;
                if (kb >= p.num_kb) continue;
                o = ((((long long)rt * p.num_kb + kb) * p.q + i) * 128 + r) * 2 + (col & 1);
            } else {
                const int jb = rt * 2 + (r >> 6), rr = r & 63;
                if (jb >= p.num_kb) continue;
                o = ((((long long)(col >> 2) * p.num_kb + jb) * p.q + i) * 64 + rr) * 4 + (col & 3);
            }
            p.bits_t[o] = tile[r][cl];
        }
        return;
    }
    if (bid >= p.act_blocks) {
        // ---- max |alpha| of this block's share of the scales
        if (bid == p.act_blocks) {
            for (int i = threadIdx.x; i < p.num_counters; i += 256) p.counters[i] = 0u;
            for (int i = p.amax_blocks + threadIdx.x; i < kMaxAlphaBlocks; i += 256) p.hdr->block_max[i] = 0u;
        }
        // (eight loads in flight; 16 bytes each where the scales are aligned)
        const long long step = (long long)p.amax_blocks * 256, at = ((long long)bid - p.act_blocks) * 256 + threadIdx.x;
        uint32_t m = 0u;
        long long done = 0;
        if ((reinterpret_cast<uintptr_t>(p.alpha) & 15u) == 0) {
            const long long nv = p.alpha_count >> 2;
            const uint4* v4 = reinterpret_cast<const uint4*>(p.alpha);
            for (long long o = at; o < nv; o += 8 * step) {
                uint4 v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = o + k * step < nv ? ld(v4 + o + k * step) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    m = max(m, max(max(v[k].x & 0x7FFFFFFFu, v[k].y & 0x7FFFFFFFu), max(v[k].z & 0x7FFFFFFFu, v[k].w & 0x7FFFFFFFu)));
            }
            done = nv << 2;
        }
        for (long long o = done + at; o < p.alpha_count; o += 8 * step) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = o + k * step < p.alpha_count ? __float_as_uint(ld(p.alpha + o + k * step)) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) m = max(m, v[k] & 0x7FFFFFFFu);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) red[warp] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int w = 0; w < 8; ++w) m = max(m, red[w]);
            p.hdr->block_max[bid - p.act_blocks] = m;
        }
        return;
    }
    const int slot = warp / WPT;                        // of the block's kPrepWarps / WPT tokens
    const int t = bid * (kPrepWarps / WPT) + slot;
    const int tl = (warp % WPT) * 32 + lane;            // thread of the token
    constexpr int kThreadsPerToken = WPT * 32;
    const bool live = t < p.n;
    const uint4* src = reinterpret_cast<const uint4*>(p.in + (long long)(live ? t : 0) * p.ld_in);
    uint4* dst = reinterpret_cast<uint4*>(p.out + (long long)t * p.ld_out);
    const int nvec = live ? (p.K + 7) / 8 : 0;
    uint32_t m = 0u;
    uint4 held[HELD];
    int v0 = tl;
    do {
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const int v = v0 + kThreadsPerToken * i;
            held[i] = (v < nvec) ? ld(src + v) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const int v = v0 + kThreadsPerToken * i;
            // (HELD = 8 for rows of 1025 to 2048 vectors, so up to three of a lane's eight are not there)
            if (HELD != 8 || v < nvec) m = max(m, max_mag_bf16x8(held[i], v * 8, p.K));
        }
        v0 += HELD * kThreadsPerToken;
    } while (AGAIN && v0 - tl < nvec);
    m = __reduce_max_sync(0xffffffffu, m);
    if (WPT > 1) {
        if (lane == 0) red[warp] = m;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WPT; ++w) m = max(m, red[slot * WPT + w]);
    }
    const int sh = shift_for(exponent_of_bits(m << 16), 14);
    const float scale = pow2f(sh);
    if (live && tl == 0) p.tok_inv_scale[t] = pow2f(-sh);
    if (!AGAIN || nvec <= HELD * kThreadsPerToken) {
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            const int v = tl + kThreadsPerToken * i;
            if (v < nvec) dst[v] = scale_to_fp16x8(held[i], v * 8, p.K, scale);
        }
    } else {
        for (v0 = tl; v0 < nvec; v0 += HELD * kThreadsPerToken) {
#pragma unroll
            for (int i = 0; i < HELD; ++i) {
                const int v = v0 + kThreadsPerToken * i;
                held[i] = (v < nvec) ? ld(src + v) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int i = 0; i < HELD; ++i) {
                const int v = v0 + kThreadsPerToken * i;
                if (v < nvec) dst[v] = scale_to_fp16x8(held[i], v * 8, p.K, scale);
            }
        }
    }
}

// Selector codes of the planes (q <= 4) in the chunk order of the GEMM kernel; one thread per (row,
// 32-weight block).  The planes are frozen, so this runs once per layer (bcq_prepare_planes); a call
// that is not given prepared planes runs it into its workspace.
//   forward  codes [m_tile][kb][128 rows][2 halves][NW words]    NW = CodeWords
//   dX       codes [u][jb][64 rows][4 quarters][NW words]
// Rows past d_out and blocks past the row pitch are written as zeros (their levels are zero or
// meet zero activations).
template <int NW>
__global__ void __launch_bounds__(256) code_planes_kernel(int mode, int d_out, int pitch, int q, int rows_padded,
                                                           int words_padded, int num_kb, int early, const uint32_t* bits,
                                                           uint32_t* codes) {
    if (early) pdl_trigger();
    pdl_wait();
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)rows_padded * words_padded) return;
    const int wd = (int)(idx % words_padded);
    const int j = (int)(idx / words_padded);
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    const bool valid = (j < d_out) && (wd < pitch);
    for (int i = 0; i < q; ++i)
        if (valid) w[i] = ld(bits + ((long long)i * d_out + j) * pitch + wd);
    uint32_t S[4];
    selectors_from_planes(w, q, S);
    if (!valid)
        for (int r = 0; r < 4; ++r) S[r] = 0u;
    long long o;
    if (mode == MODE_FWD)
        o = ((((long long)(j >> 7) * num_kb + (wd >> 1)) * 128 + (j & 127)) * 2 + (wd & 1)) * NW;
    else
        o = ((((long long)(wd >> 2) * num_kb + (j >> 6)) * 64 + (j & 63)) * 4 + (wd & 3)) * NW;
    pack_selectors<NW>(S, codes + o);
}

// ------------------------------------------------------------------------------------------
// forward / dX for n > 16: A expanded from the bit-planes, B (fp16 activations) by TMA
// ------------------------------------------------------------------------------------------

struct ExpandParams {
    int q, g, G, n;
    int Mdim;          // d_out (fwd) or d_in (dX)
    int num_kb;        // K blocks of 64 over d_in (fwd) or d_out (dX)
    // The first full_tiles output tiles go whole to the pairs in turn; the res_tiles tiles after them
    // are cut into `pieces` pieces of piece_len stages, one for each of the first res_tiles * pieces pairs
    int full_tiles, res_tiles, pieces, piece_len;
    int m_tiles;           // row tiles of 128 of the regrouped planes
    int m_pairs;           // output tiles of a token tile: pairs of row tiles
    int tn;                // token tile width
    uint32_t acc_cols;     // tensor-memory columns per accumulator
    // pipeline geometry (chosen on the host)
    int a_slots;           // ring of expanded weight tiles (16 KiB each), >= the number of worker groups
    int b_slots;           // ring of activation tiles (TN / 2 x 128 B each), filled by TMA
    uint32_t chunk_words;  // words of one stage's chunk of the regrouped planes
    const uint32_t* bits_t;      // regrouped plane words (see PrepParams)
    const float* alpha_t;        // regrouped scales
    const float* bias;           // fwd only, may be null
    const WsHeader* hdr;         // max |alpha| per pre-pass block
    const float* tok_inv_scale;  // [n]
    void* out;                   // [n][ldo]
    long long ldo;
    int out_bf16;
    int fast_epi;                // bf16 output written by TMA stores (aligned base and pitch, no K split)
    int helpers;                 // the worker warps share the epilogue of a CTA's last tile (see run_expand)
    float* partial;              // [pair][rank][TN columns][128 rows]
    uint32_t* counters;          // [shared tile][rank][quarter][box class]
};

// Prefill kernel.  Persistent: every pair of CTAs walks over output tiles of 256 rows x TN tokens (rows
// fastest, so that pairs running at the same time share activation tiles in L2).  A pair, because
// shared memory bounds a CTA alone: per 64-wide stage of a 128 x 256 tile (512 tensor-core cycles) the
// workers write 16 KiB, TMA writes 32 KiB and the tensor core reads 48 KiB, 768 cycles at 128 bytes a
// cycle (measured: 755 - 820 cycles a stage).  In a pair each CTA expands its own 128 rows but holds
// only half of the tokens: 512 cycles (measured: 600 - 700, now set by the workers).
// Each CTA has 22 warps:
//   warps 0..15   workers in four groups of four; group g takes the pipeline stages whose running
//                 index is g mod 4 (the workers set the pace by latency, not by issue rate: 6400 -> 1600
//                 with 4096 tokens takes 106 us with three groups, 97 with four, 100 with five).  A
//                 thread expands 64 weights of one row per stage (one 128-byte line of the operand
//                 tile), so a group rebuilds one 128 x 64 weight tile.  The thread reads its selector
//                 codes (or plane words) and scales straight from the regrouped arrays in global
//                 memory, one task ahead of the one it expands, so the loads are hidden behind a
//                 whole turn of the group
//   warps 16..19  epilogue: drain one accumulator while the main loop fills the other (warp w
//                 reaches the tensor-memory lanes 32 * (w % 4) .. + 31)
//   warp 20       owner of the tensor-memory allocation (two accumulators); in the leader of the
//                 pair, UMMA issuer for both CTAs
//   warp 21       producer of this CTA's half of the activation tiles (TMA)
// Shared memory: a ring of weight tiles (16 KiB each; the workers refill one as soon as the tensor core
// is done with it), a ring of activation tiles (TN / 2 x 128 B each; a TMA load takes about a
// microsecond to land), the epilogue's staging, barriers and output scales.  The barriers "operand
// in place" and "accumulator drained" are the leader's and count both CTAs; the others exist in both
// CTAs and are signalled by one commit to both.
//
// Where a ragged last wave of tiles (or a problem with few tiles) would leave at least half of the pairs
// idle, its tiles are cut along K into as many pieces as there are pairs for; a pair does its piece
// first.  It writes its fp32 sums to the workspace, and for each box of the output the warp that arrives
// last (a counter) adds the pieces in order and writes the result, so no warp waits for another and the
// result does not depend on which one is last.
constexpr int kPfGroupWarps = 4;
constexpr int kPfWorkerWarps = kPfGroups * kPfGroupWarps;  // 16
constexpr int kPfEpiWarp0 = kPfWorkerWarps;
constexpr int kPfEpiWarps = 4;
constexpr int kPfMmaWarp = kPfEpiWarp0 + kPfEpiWarps;
constexpr int kPfProdWarp = kPfMmaWarp + 1;
constexpr int kPfThreads = (kPfProdWarp + 1) * 32;         // 704
static_assert(kPfEpiWarp0 % 4 == 0, "epilogue warp e must sit on tensor-memory lane quarter e");
__device__ __forceinline__ int pf_worker_index(int warp) { return warp < kPfWorkerWarps ? warp : -1; }
__device__ __forceinline__ int pf_epilogue_index(int warp) {
    return warp >= kPfEpiWarp0 && warp < kPfEpiWarp0 + kPfEpiWarps ? warp - kPfEpiWarp0 : -1;
}
constexpr int kPfMaxSlots = 8;                                // per ring
constexpr uint32_t kPfGroupBar0 = 4;                           // named barriers 4..7: one per worker group
constexpr uint32_t kPfCtlBytes = 384;                          // barriers, TMEM handle, abort flag
constexpr uint32_t kPfScaleBytes = 256 * 4;                    // [TN] output scales of the tile being drained
// per epilogue warp one 1 KiB buffer of 32 rows x 16 bf16 (8 fp32) tokens; two such sets
constexpr uint32_t kPfStagingBuf = kPfEpiWarps * 1024;

template <int MODE, int QM>
__global__ void __launch_bounds__(kPfThreads, 1)
expand_gemm_kernel(const __grid_constant__ CUtensorMap tmap_b, const __grid_constant__ CUtensorMap tmap_out,
                   const ExpandParams p) {
    const int TN = p.tn;                                   // token tile: a multiple of 16, <= 256
    const uint32_t kBBytes = (uint32_t)(TN / 2) * kBlockK * 2;  // this CTA's half of the tokens
    const uint32_t kAccCols = p.acc_cols;                  // tensor-memory columns of one accumulator
    const uint32_t kTmemCols = 2 * kAccCols;               // a power of two >= 32
    constexpr int kRows = (MODE == MODE_FWD) ? 128 : 64;  // weight rows of one stage
    constexpr int kUnit = (MODE == MODE_FWD) ? 2 : 4;     // 32-weight blocks per row and stage
    constexpr int NW = NumWords<QM>::value;
    // fp16 x fp16 -> fp32; A is MN-major for dX
    const uint32_t kIdesc = (ptx::make_idesc_bf16(2 * kBlockM, TN, MODE == MODE_BWDX ? 1 : 0, 0)) &
                            ~((1u << 7) | (1u << 10));

    extern __shared__ uint8_t smem_raw[];
    const int NA = p.a_slots, NB = p.b_slots;
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t b_base = smem_base + NA * kABytes;
    const uint32_t staging_base = b_base + NB * kBBytes;  // 1 KiB aligned: the output boxes are swizzled
    constexpr uint32_t staging_bytes = 2 * kPfStagingBuf;
    const uint32_t ctl_base = staging_base + staging_bytes;
    uint8_t* ctl_gen = smem_gen + NA * kABytes + NB * kBBytes + staging_bytes;

    Ctl ctl;
    ctl.aready = ctl_base;                      // + 8*s : the workers have written weight slot s
    ctl.empty = ctl_base + 8 * kPfMaxSlots;     // + 8*s : the UMMAs that read weight slot s are done
    ctl.full = ctl_base + 16 * kPfMaxSlots;     // + 8*s : the activation tile of slot s has landed
    const uint32_t b_empty = ctl_base + 24 * kPfMaxSlots;  // + 8*s : the UMMAs that read activation slot s are done
    ctl.accum = ctl_base + 32 * kPfMaxSlots;    // accumulator full [2]
    const uint32_t acc_empty = ctl.accum + 16;  // accumulator drained [2]
    ctl.spare = acc_empty + 16;
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(ctl_gen + 32 * kPfMaxSlots + 40);
    ctl.abort_flag = reinterpret_cast<volatile int*>(ctl_gen + 32 * kPfMaxSlots + 44);
    ctl.device_flag = &g_timeout_flag;
    float* scale = reinterpret_cast<float*>(ctl_gen + kPfCtlBytes);  // [TN]: 1 / (weight scale * token scale)
    const uint32_t scale_addr = ctl_base + kPfCtlBytes;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_rank();
    const int pair0 = (int)blockIdx.x >> 1, num_pairs = (int)gridDim.x >> 1;

    if (warp == 0) {
        // the barriers are initialised by the lanes of one warp side by side (one after the other
        // they cost a few tenths of a microsecond before any copy can start)
        if (lane < NA) {
            ptx::mbar_init(ctl.aready + 8 * lane, 2 * kPfGroupWarps);
            ptx::mbar_init(ctl.empty + 8 * lane, 1);
        } else if (lane >= 8 && lane < 8 + NB) {
            ptx::mbar_init(ctl.full + 8 * (lane - 8), 1);
            ptx::mbar_init(b_empty + 8 * (lane - 8), 1);
        } else if (lane >= 16 && lane < 18) {
            ptx::mbar_init(ctl.accum + 8 * (lane - 16), 1);
            ptx::mbar_init(acc_empty + 8 * (lane - 16), 2 * kPfEpiWarps);
        } else if (lane == 18) {
            ptx::mbar_init(ctl.spare, 1);
            *ctl.abort_flag = 0;
        } else if (lane == 19) {
            ptx::prefetch_tmap(&tmap_b);
            if (p.fast_epi) ptx::prefetch_tmap(&tmap_out);
        }
        ptx::fence_mbar_init();
        __syncwarp();
    }
    if (warp == kPfMmaWarp) {
        ptx::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t*>(tmem_holder)), kTmemCols);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();  // the peer's barriers exist
    ptx::tc_fence_after_sync();
    pdl_wait();
    const uint32_t tmem_base = *tmem_holder;

    // every role walks the same sequence of segments (a tile, or this pair's part of one) and pipeline
    // stages
    const int nres = pair0 < p.res_tiles * p.pieces ? 1 : 0;
    const int nseg = nres + (pair0 < p.full_tiles ? (p.full_tiles - 1 - pair0) / num_pairs + 1 : 0);
    // res: index of the shared tile of which the segment is a part, or -1 for a whole tile
    auto tile_coords = [&](int seg, int& m0, int& t0, int& res, int& kb_begin, int& iters) {
        int tile;
        res = -1;
        if (seg < nres) {
            res = pair0 / p.pieces;
            kb_begin = (pair0 - res * p.pieces) * p.piece_len;
            iters = min(p.piece_len, p.num_kb - kb_begin);
            tile = p.full_tiles + res;
        } else {
            kb_begin = 0;
            iters = p.num_kb;
            tile = pair0 + (seg - nres) * num_pairs;
        }
        m0 = (2 * (tile % p.m_pairs) + rank) * kBlockM;
        t0 = (tile / p.m_pairs) * TN;
    };

    // bf16 output through TMA stores, 16 tokens x 32 rows at a time: the accumulator is read as MMA
    // fragments (thread t: rows g = t/4 and g + 8 of each half of the warp's 32 lanes, token pairs
    // 2(t%4)), scaled, packed to bf16 pairs and transposed by stmatrix into a 64-byte-swizzled
    // [16 tokens][32 rows] box at `buf`, which one lane then hands to the TMA.  s0*, s1* are the
    // output scales of the thread's tokens in the first and second group of eight.
    auto store_box = [&](uint32_t t_row, int col, uint32_t buf, float s0x, float s0y, float s1x, float s1y,
                         const float (&b4)[4], int x, int y) {
        const int tok = ((lane >> 4) << 3) + (lane & 7);  // token row this lane addresses
        const uint32_t st_off = (uint32_t)tok * 64u;
        const uint32_t st_sw = (uint32_t)((tok >> 1) & 3);
        const uint32_t jb = (uint32_t)((lane >> 3) & 1);
        uint32_t va[8], vb[8];
        ptx::tmem_ld_16x256b_x2(t_row + (uint32_t)col, va);
        ptx::tmem_ld_16x256b_x2(t_row + (16u << 16) + (uint32_t)col, vb);
        ptx::tmem_ld_wait();
        auto pk = [](uint32_t u, uint32_t v, float sx, float sy, float b) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(u) * sx + b, __uint_as_float(v) * sy + b);
            return *reinterpret_cast<const uint32_t*>(&h);
        };
        const uint32_t a0 = pk(va[0], va[1], s0x, s0y, b4[0]), a1 = pk(va[2], va[3], s0x, s0y, b4[1]);
        const uint32_t a2 = pk(va[4], va[5], s1x, s1y, b4[0]), a3 = pk(va[6], va[7], s1x, s1y, b4[1]);
        const uint32_t c0 = pk(vb[0], vb[1], s0x, s0y, b4[2]), c1 = pk(vb[2], vb[3], s0x, s0y, b4[3]);
        const uint32_t c2 = pk(vb[4], vb[5], s1x, s1y, b4[2]), c3 = pk(vb[6], vb[7], s1x, s1y, b4[3]);
        ptx::stmatrix_x4_trans(buf + st_off + ((jb ^ st_sw) << 4), a0, a1, a2, a3);
        ptx::stmatrix_x4_trans(buf + st_off + (((jb + 2u) ^ st_sw) << 4), c0, c1, c2, c3);
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            ptx::tma_store_2d(&tmap_out, x, y, buf);
            ptx::bulk_commit_group();
        }
    };
    // Any other output, 16 tokens x 32 rows at a time: transposed through the staging buffer `stg`
    // ([token][row]), then 16-byte pieces of one token's 32 rows as coalesced stores.  sc: the output
    // scales of the 16 tokens.
    auto store_box_any = [&](uint32_t t_row, int col, uint32_t stg, const float (&sc)[16], float bias, int m0w, int t0) {
        const int esz = p.out_bf16 ? 2 : 4;
        uint8_t* out_base = reinterpret_cast<uint8_t*>(p.out);
        // 16-byte stores need an aligned base and pitch
        const bool full_rows = ((reinterpret_cast<uintptr_t>(out_base) & 15u) == 0) && ((p.ldo * esz) % 16 == 0) &&
                               (m0w + 32 <= p.Mdim);
        const int pieces = 2 * esz;          // 16-byte vectors of one token's 32 rows
        const int toks = 1024 / (32 * esz);  // tokens per staging round: 16 (bf16) or 8 (fp32)
        uint32_t v[16];
        ptx::tmem_ld_x16(t_row + (uint32_t)col, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (esz == 2) {
                if (half == 1) break;
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const __nv_bfloat16 h = __float2bfloat16_rn(__uint_as_float(v[c]) * sc[c] + bias);
                    asm volatile("st.shared.b16 [%0], %1;" ::"r"(stg + c * 64 + lane * 2),
                                 "h"(*reinterpret_cast<const unsigned short*>(&h)) : "memory");
                }
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float f = __uint_as_float(v[8 * half + c]) * sc[8 * half + c] + bias;
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(stg + c * 128 + lane * 4), "f"(f) : "memory");
                }
            }
            __syncwarp();
            const int tbase = t0 + col + ((esz == 4) ? 8 * half : 0);
            for (int pc = lane; pc < toks * pieces; pc += 32) {
                const int c = pc / pieces, piece = pc - c * pieces;
                const int t = tbase + c;
                if (t >= p.n) continue;
                uint32_t x0, x1, x2, x3;
                asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(x0), "=r"(x1), "=r"(x2), "=r"(x3)
                             : "r"(stg + pc * 16) : "memory");
                uint8_t* dst = out_base + ((long long)t * p.ldo + m0w) * esz + piece * 16;
                if (full_rows) {
                    *reinterpret_cast<uint4*>(dst) = make_uint4(x0, x1, x2, x3);
                } else {
                    const uint32_t rr[4] = {x0, x1, x2, x3};
                    const int per = 16 / esz;  // elements in this piece
#pragma unroll
                    for (int e2 = 0; e2 < 8; ++e2) {
                        if (e2 < per && m0w + piece * per + e2 < p.Mdim) {
                            if (esz == 2)
                                reinterpret_cast<unsigned short*>(dst)[e2] =
                                    (unsigned short)(rr[e2 >> 1] >> ((e2 & 1) * 16));
                            else
                                reinterpret_cast<uint32_t*>(dst)[e2] = rr[e2 & 3];
                        }
                    }
                }
            }
            __syncwarp();
        }
    };
    // Output of a segment: emit(col) for the boxes first, first + step, ... of this warp's 32 rows.  For
    // a part of a shared tile the sums go to the workspace, and emit() follows for those classes of
    // boxes (box mod kPfHelpers) of which this warp's part is the last to arrive.
    constexpr int kPfHelpers = 1 + kPfWorkerWarps / 4;  // 5
    auto drain = [&](int res, int m0w, int t0, uint32_t t_row, int quarter, int first, int step, auto&& emit) {
        if (m0w >= p.Mdim) return;
        const int nbox = min(TN >> 4, (p.n - t0 + 15) >> 4);
        if (res < 0) {
#pragma unroll 1
            for (int b = first; b < nbox; b += step) emit(16 * b);
            return;
        }
        const size_t part = (size_t)TN * 256;  // floats of one contribution, both CTAs
        const int e0 = rank * TN * 128 + quarter * 32 + lane;
        float* mine = p.partial + (size_t)pair0 * part + e0;
#pragma unroll 1
        for (int b = first; b < nbox; b += step) {
            uint32_t v[16];
            ptx::tmem_ld_x16(t_row + 16u * b, v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 16; ++c) __stcg(mine + (16 * b + c) * 128, __uint_as_float(v[c]));
        }
        __threadfence();
        __syncwarp();
        const int p_first = res * p.pieces, p_last = p_first + p.pieces - 1;
        uint32_t* cnt = p.counters + ((res * 2 + rank) * 4 + quarter) * kPfHelpers;
        const int cl_end = min(nbox, step == 1 ? kPfHelpers : first + 1);
#pragma unroll 1
        for (int cl = first; cl < cl_end; ++cl) {
            uint32_t before = 0u;
            if (lane == 0) before = atomicAdd(cnt + cl, 1u);
            before = __shfl_sync(0xffffffffu, before, 0);
            if (before != (uint32_t)(p_last - p_first)) continue;
            __threadfence();
#pragma unroll 1
            for (int b = cl; b < nbox; b += kPfHelpers) {
                float sum[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) sum[c] = 0.0f;
#pragma unroll 2
                for (int q = p_first; q <= p_last; ++q) {
                    const float* src = p.partial + (size_t)q * part + e0 + (size_t)(16 * b) * 128;
                    float x[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) x[c] = __ldcg(src + c * 128);
#pragma unroll
                    for (int c = 0; c < 16; ++c) sum[c] += x[c];
                }
                ptx::tmem_st_x16(t_row + 16u * b, sum);
                ptx::tmem_st_wait();
                emit(16 * b);
            }
        }
    };
    // On the last segment of a CTA the worker warps have nothing left to expand, so they share its
    // epilogue: of the five warps on a tensor-memory lane quarter (one epilogue warp, four workers)
    // warp h takes the boxes h, h + 5, ...

    if (warp == kPfProdWarp) {
        // ---------------- producer: the activation tile of every stage (TMA), into a ring of its
        // own that runs as far ahead of the tensor core as shared memory allows
        if (lane == 0) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int seg = 0; seg < nseg && ok; ++seg) {
                int m0, t0, res, kb_begin, iters;
                tile_coords(seg, m0, t0, res, kb_begin, iters);
                for (int it = 0; it < iters; ++it) {
                    ok = wait_bar(b_empty + 8 * s, ph ^ 1u, ctl, 1, 256u);
                    if (!ok) break;
                    if (rank == 0) ptx::mbar_arrive_expect_tx(ctl.full + 8 * s, 2u * kBBytes);
                    ptx::tma_load_2d_pair(b_base + s * kBBytes, &tmap_b, (kb_begin + it) * kBlockK, t0 + rank * (TN / 2),
                                          ptx::leader_addr(ctl.full + 8 * s));
                    if (++s == NB) { s = 0; ph ^= 1u; }
                }
            }
            // (no pdl_trigger here: blocks of the next call's pre-pass that start under this kernel crowd
            // onto the few SMs it leaves free, and the pre-pass then lacks the others' bandwidth; measured
            // on a training step of a layer of width 1600: 872 us without, 914 with)
            // giving up: the copies in flight are counted on the leader's barriers, which may never
            // complete; they land within microseconds, so wait a thousand times as long
            if (!ok) for (int i = 0; i < 1000; ++i) __nanosleep(2000);
        }
        __syncwarp();
    } else if (warp == kPfMmaWarp) {
        // ---------------- UMMA issuer.  One elected thread runs the whole loop: per stage it has
        // to get through two barrier checks, a fence, four UMMAs and two commits in less time
        // than the tensor core needs for the stage (512 cycles at the full width), so nothing
        // warp-wide (election, reconvergence) is left inside the loop and the two barrier checks
        // are issued together.
        if (rank == 0 && ptx::elect_one()) {
            bool ok = true;
            int sa = 0, sb = 0, lt = 0;
            uint32_t pha = 0, phb = 0;
            // shared-memory descriptor halves (128-byte swizzle, version 1): low = start address >> 4 and
            // leading offset >> 4 at bit 16, high = stride offset >> 4, version at bit 14, swizzle at bit 29
            constexpr uint32_t kHiCommon = (1024u >> 4) | (1u << 14) | (2u << 29);
            constexpr uint32_t kAHi = kHiCommon, kBHi = kHiCommon;
            constexpr uint32_t kALoExtra = ((MODE == MODE_FWD) ? (16u >> 4) : (8192u >> 4)) << 16;  // leading offset of A
            constexpr uint32_t kBLoExtra = (16u >> 4) << 16;
            constexpr uint32_t kAStep = (MODE == MODE_FWD) ? (32u >> 4) : (2048u >> 4);
            const uint32_t a_lo0 = ((smem_base >> 4) & 0x3FFFu) | kALoExtra;
            const uint32_t b_lo0 = ((b_base >> 4) & 0x3FFFu) | kBLoExtra;
            for (; lt < nseg && ok; ++lt) {
                int m0, t0, res, kb_begin, iters;
                tile_coords(lt, m0, t0, res, kb_begin, iters);
                const int acc = lt & 1;
                const uint32_t acc_ph = (lt >> 1) & 1;
                ok = wait_bar(acc_empty + 8 * acc, acc_ph ^ 1u, ctl, 8);  // the epilogue has drained it
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)acc * kAccCols;
                for (int it = 0; it < iters; ++it) {
                    // both operands of the stage in place?  (the common case: yes, both at once)
                    const bool fb = ptx::mbar_try_wait(ctl.full + 8 * sb, phb);
                    const bool fa = ptx::mbar_try_wait(ctl.aready + 8 * sa, pha);
                    if (!fb) ok = wait_bar(ctl.full + 8 * sb, phb, ctl, 4, 32u);
                    if (!fa && ok) ok = wait_bar(ctl.aready + 8 * sa, pha, ctl, 3, 32u);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    // descriptors: only the start-address field changes, by 32 bytes (K-major) or
                    // 2048 bytes (MN-major A) per UMMA
                    const uint32_t a_lo = a_lo0 + (uint32_t)sa * (kABytes >> 4);
                    const uint32_t b_lo = b_lo0 + (uint32_t)sb * (kBBytes >> 4);
#pragma unroll
                    for (int kk = 0; kk < kBlockK / 16; ++kk)
                        ptx::umma_f16_pair(d_tmem, a_lo + kk * kAStep, kAHi, b_lo + kk * 2, kBHi, kIdesc,
                                           (it > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit_pair(ctl.empty + 8 * sa);
                    ptx::umma_commit_pair(b_empty + 8 * sb);
                    if (++sa == NA) { sa = 0; pha ^= 1u; }
                    if (++sb == NB) { sb = 0; phb ^= 1u; }
                }
                if (ok) ptx::umma_commit_pair(ctl.accum + 8 * acc);
            }
            if (!ok) {
                ptx::umma_commit_pair(ctl.spare);
                wait_bar(ctl.spare, 0, ctl, 5);
            }
        }
        __syncwarp();
    } else if (pf_worker_index(warp) >= 0) {
        // ---------------- workers
        const int wid = pf_worker_index(warp);  // 0..15
        const int group = wid / kPfGroupWarps;  // takes the stages whose running index is `group` mod kPfGroups
        const int wl = wid % kPfGroupWarps;
        float wscale = 0.0f;  // known once the first loads are on their way

        // A task is one 128-byte line of the weight tile: 64 weights of one row.
        // fwd : (weight row m0 + row, the stage's 64 k); a warp takes 32 consecutive rows
        // dX  : (K index j = 64*kb + row, 64-wide half of the tile's 128 k); the two halves of a row
        //       sit in adjacent lanes
        // Either way the 32 lanes of a warp write their 16-byte chunks to all banks evenly.
        const int row = (MODE == MODE_FWD) ? wl * 32 + lane : wl * 16 + (lane >> 1);
        const int half = (MODE == MODE_FWD) ? 0 : (lane & 1);
        const uint32_t line_off = (uint32_t)half * 8192u + (uint32_t)row * 128u;
        const uint32_t lx = row & 7;
        constexpr int NWC = CodeWords<QM>::value;
        constexpr int NL = (QM == QM_GENERIC) ? NW : NWC;   // words a 32-weight block loads
        constexpr int NSC = (QM == QM_GENERIC) ? NW : 4;    // scales a task loads
        // the task's words within a chunk [m_tile][kb] (fwd) or [u][jb] (dX) of the regrouped planes:
        // q <= 4 selector codes [row][block][NWC], q > 4 plane words [plane][row][block]; its two
        // 32-weight blocks are neighbours
        const uint32_t block0 = (uint32_t)(row * kUnit + half * 2);
        const uint32_t word_off = (QM == QM_GENERIC) ? block0 : block0 * NWC;
        const uint32_t chunk_words = p.chunk_words;
        const uint32_t alpha_block = (uint32_t)p.q * kRows;  // floats per (row block, group): [plane][row]

        // The task stream of this thread: the stages whose running index over all tiles of the CTA
        // is `group` mod kPfGroups.  A cursor names one of them.
        struct Cur {
            int seg, it, iters, kb_begin, mt;
            int c, kpos, next_edge;  // group index of the task's first 32 k (forward: advances with the stage)
            uint32_t code_idx;       // this thread's first word of the task in the regrouped planes
            uint32_t alpha_idx;      // its first scale (plane 0, group c) in the regrouped scales
            bool split;              // the second 32 k belong to the next group (g not a multiple of 64)
            bool fresh;              // the scales differ from the previous task's: load them, rebuild the table
            bool valid;
        };
        auto enter_tile = [&](Cur& x) {
            int m0, t0, res;
            tile_coords(x.seg, m0, t0, res, x.kb_begin, x.iters);
            x.mt = min(m0 >> 7, p.m_tiles - 1);  // a pair whose second row tile does not exist expands the first again
        };
        const uint32_t code_step = kPfGroups * chunk_words;
        const uint32_t alpha_step = kPfGroups * (uint32_t)p.G * alpha_block;  // dX: the next task's rows
        auto locate = [&](Cur& x) {  // group index and array positions at (seg, it), from scratch
            x.kpos = (MODE == MODE_FWD) ? (x.kb_begin + x.it) * kBlockK : x.mt * kBlockM + half * 64;
            x.c = min(x.kpos / p.g, p.G - 1);
            x.next_edge = (x.c + 1) * p.g;
            x.split = (x.kpos + 32 >= x.next_edge) && (x.c < p.G - 1);
            x.code_idx = (uint32_t)(x.mt * p.num_kb + x.kb_begin + x.it) * chunk_words + word_off;
            const int blk = (MODE == MODE_FWD) ? x.mt : x.kb_begin + x.it;
            x.alpha_idx = (uint32_t)(blk * p.G + x.c) * alpha_block + (uint32_t)row;
        };
        // to the next task: kPfGroups stages on
        auto advance = [&](Cur& x) {
            x.it += kPfGroups;
            bool moved = false;
            while (x.it >= x.iters) {
                x.it -= x.iters;
                if (++x.seg >= nseg) { x.valid = false; return; }
                enter_tile(x);
                moved = true;
            }
            if (moved) {
                locate(x);
                x.fresh = true;
            } else if (MODE == MODE_FWD) {
                const int c0 = x.c;
                x.kpos += kPfGroups * kBlockK;
                while (x.kpos >= x.next_edge && x.c < p.G - 1) { ++x.c; x.next_edge += p.g; }
                x.split = (x.kpos + 32 >= x.next_edge) && (x.c < p.G - 1);
                x.fresh = (QM == QM_GENERIC) || (x.c != c0) || x.split;
                x.code_idx += code_step;
                x.alpha_idx += (uint32_t)(x.c - c0) * alpha_block;
            } else {
                x.fresh = true;  // dX: every stage brings other rows
                x.code_idx += code_step;
                x.alpha_idx += alpha_step;
            }
        };
        // global loads of a task: its plane words or codes and, when they change, its scales
        auto issue = [&](const Cur& x, uint32_t (&cv)[2][NL], float (&av)[NSC]) {
            const uint32_t* src = p.bits_t + x.code_idx;
            if (QM == QM_GENERIC) {
#pragma unroll
                for (int i = 0; i < NL; ++i) {
                    if (i < p.q) {
                        const uint2 v = ld_stream(reinterpret_cast<const uint2*>(src + i * (kRows * kUnit)));
                        cv[0][i] = v.x; cv[1][i] = v.y;
                    } else {
                        cv[0][i] = 0u; cv[1][i] = 0u;
                    }
                }
            } else if (NWC == 4) {
                const uint4 v0 = ld_stream(reinterpret_cast<const uint4*>(src)), v1 = ld_stream(reinterpret_cast<const uint4*>(src + 4));
                cv[0][0] = v0.x; cv[0][1] = v0.y; cv[0][2] = v0.z; cv[0][NL - 1] = v0.w;
                cv[1][0] = v1.x; cv[1][1] = v1.y; cv[1][2] = v1.z; cv[1][NL - 1] = v1.w;
            } else {
                // six words, 8-byte aligned
                const uint2 v0 = ld_stream(reinterpret_cast<const uint2*>(src)), v1 = ld_stream(reinterpret_cast<const uint2*>(src + 2)), v2 = ld_stream(reinterpret_cast<const uint2*>(src + 4));
                cv[0][0] = v0.x; cv[0][1] = v0.y; cv[0][2] = v1.x;
                cv[1][0] = v1.y; cv[1][1] = v2.x; cv[1][2] = v2.y;
            }
            if (x.fresh) {
                const float* ap = p.alpha_t + x.alpha_idx;
#pragma unroll
                for (int i = 0; i < NSC; ++i)
                    av[i] = (i < p.q) ? ld_stream(ap + i * kRows) : 0.0f;
            }
        };

        Lut lut = {0u, 0u, 0u, 0u};
        bool ok = true;
        int s = group;  // weight slot of the current task (a_slots >= kPfGroups)
        uint32_t ph = 0;
        // One task: wait until the UMMAs that read the slot's previous contents are done (the first
        // warp of the group polls the barrier, the others park on a hardware barrier: a polling
        // warp takes issue slots from the warps that expand), expand, publish.
        auto process = [&](const Cur& x, const uint32_t (&cv)[2][NL], const float (&av)[NSC]) -> bool {
            if (wl == 0) wait_bar(ctl.empty + 8 * s, ph ^ 1u, ctl, 9, 256u);  // a timeout shows in the abort flag
            ptx::named_bar_sync(kPfGroupBar0 + group, kPfGroupWarps * 32);
            if (*ctl.abort_flag) return false;
            const uint32_t line = smem_base + (uint32_t)s * kABytes + line_off;
            float a2[NSC];  // scales of the second 32 weights when they belong to the next group
            if (x.split) {
                const float* ap = p.alpha_t + x.alpha_idx + alpha_block;  // group c + 1
#pragma unroll
                for (int i = 0; i < NSC; ++i)
                    a2[i] = (i < p.q) ? ld_stream(ap + i * kRows) : 0.0f;
            }
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const bool second = (b == 1) && x.split;
                if (QM == QM_GENERIC) {
                    float a8[BCQ_MAX_Q];
                    uint32_t w8[BCQ_MAX_Q];
#pragma unroll
                    for (int i = 0; i < BCQ_MAX_Q; ++i) {
                        a8[i] = (second ? a2[i % NSC] : av[i % NSC]) * wscale;
                        w8[i] = cv[b][i % NL];
                    }
                    expand16_sum(w8, a8, p.q, line, lx, 4 * b);
#pragma unroll
                    for (int i = 0; i < BCQ_MAX_Q; ++i) w8[i] >>= 16;
                    expand16_sum(w8, a8, p.q, line, lx, 4 * b + 2);
                } else {
                    if ((b == 0 && x.fresh) || second) {
                        float a[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) a[i] = (second ? a2[i % NSC] : av[i % NSC]) * wscale;
                        lut = (QM == QM_LUT4) ? build_lut(a[0], a[1], a[2], a[3]) : build_lut(a[0], a[1], a[2], 0.0f);
                    }
                    uint32_t cw[NWC], S[4];
#pragma unroll
                    for (int i = 0; i < NWC; ++i) cw[i] = cv[b][i % NL];
                    selectors<NWC>(cw, S);
                    expand32_codes<NWC>(S, lut, line, lx, 4 * b);
                }
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::leader_addr(ctl.aready + 8 * s));
            s += kPfGroups;
            if (s >= NA) { s -= NA; ph ^= 1u; }
            return true;
        };

        Cur cur;
        cur.seg = 0;
        cur.valid = nseg > 0;
        cur.fresh = true;
        cur.split = false;
        cur.it = group;
        cur.iters = 0; cur.kb_begin = 0; cur.mt = 0; cur.c = 0; cur.kpos = 0; cur.next_edge = 0;
        cur.code_idx = 0; cur.alpha_idx = 0;
        if (cur.valid) {
            enter_tile(cur);
            while (cur.it >= cur.iters) {
                cur.it -= cur.iters;
                if (++cur.seg >= nseg) { cur.valid = false; break; }
                enter_tile(cur);
            }
            if (cur.valid) locate(cur);
        }
        uint32_t cvA[2][NL], cvB[2][NL];
        float avA[NSC], avB[NSC];
        if (QM == QM_GENERIC) {
            // q > 4: one set of registers, loaded at the head of the task (under the wait for the slot)
            wscale = pow2f(weight_shift(p.hdr, p.q));
            while (cur.valid && ok) {
                issue(cur, cvA, avA);
                ok = process(cur, cvA, avA);
                advance(cur);
            }
        } else {
            // q <= 4: the loads of the next task are in flight while this one is expanded (two
            // register sets, so that nothing has to wait for a load in order to be moved)
            if (cur.valid) issue(cur, cvA, avA);
            wscale = pow2f(weight_shift(p.hdr, p.q));
            while (cur.valid && ok) {
                Cur nxt = cur;
                advance(nxt);
                if (nxt.valid) issue(nxt, cvB, avB);
                ok = process(cur, cvA, avA);
                cur = nxt;
                if (!cur.valid || !ok) break;
                advance(nxt);
                if (nxt.valid) issue(nxt, cvA, avA);
                ok = process(cur, cvB, avB);
                cur = nxt;
            }
        }
        if (p.helpers && ok && nseg > 0) {
            // share the output of this CTA's last segment.  Its operand slots are free once the
            // accumulator is complete, so each warp stages its boxes in 1 KiB of the first slots.
            const int lt = nseg - 1;
            int m0, t0, res, kb_begin, iters;
            tile_coords(lt, m0, t0, res, kb_begin, iters);
            const int acc = lt & 1;
            ok = wait_bar(ctl.accum + 8 * acc, (uint32_t)(lt >> 1) & 1u, ctl, 10);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                ptx::tc_fence_after_sync();
                const int quarter = warp & 3, helper = 1 + (warp >> 2);  // 1..4
                const int m0w = m0 + quarter * 32;
                const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * kAccCols;
                const uint32_t buf = smem_base + (uint32_t)warp * 1024u;
                const float winv = 1.0f / wscale;  // a power of two
                auto scale_of = [&](int t) { return (t < p.n) ? winv * ld(p.tok_inv_scale + t) : 0.0f; };
                auto bias_of = [&](int m) { return (MODE == MODE_FWD && p.bias != nullptr && m < p.Mdim) ? ld(p.bias + m) : 0.0f; };
                if (p.fast_epi) {
                    const int g = lane >> 2, tq = lane & 3;
                    float b4[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) b4[i] = bias_of(m0w + g + 8 * i);
                    bool stored = false;
                    drain(res, m0w, t0, t_row, quarter, helper, kPfHelpers, [&](int col) {
                        if (stored && lane == 0) ptx::bulk_wait_group_read<0>();
                        __syncwarp();
                        const int ta = t0 + col + 2 * tq, tb = ta + 8;
                        store_box(t_row, col, buf, scale_of(ta), scale_of(ta + 1), scale_of(tb), scale_of(tb + 1), b4, m0w, t0 + col);
                        stored = true;
                    });
                    if (lane == 0) ptx::bulk_wait_group<0>();
                } else {
                    const float bias = bias_of(m0w + lane);
                    drain(res, m0w, t0, t_row, quarter, helper, kPfHelpers, [&](int col) {
                        float sc[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) sc[c] = scale_of(t0 + col + c);
                        store_box_any(t_row, col, buf, sc, bias, m0w, t0);
                    });
                }
            }
        }
    } else if (pf_epilogue_index(warp) >= 0) {
        // ---------------- epilogue warps: D[row, col] -> out[t0 + col][m0 + row]
        const int ew = pf_epilogue_index(warp);  // 0..3
        const int quarter = warp & 3;       // TMEM lanes 32 * quarter .. + 31
        const int et = ew * 32 + lane;      // 0..127
        const float winv = pow2f(-weight_shift(p.hdr, p.q));
        // this warp's staging: [tokens][32 rows], 1 KiB (a second one kPfStagingBuf further)
        const uint32_t stg = staging_base + ew * 1024;
        bool ok = true;
        int lt = 0;
        uint32_t chunks = 0;  // output boxes stored so far (fast path): selects the staging buffer
        for (; lt < nseg && ok; ++lt) {
            int m0, t0, res, kb_begin, iters;
            tile_coords(lt, m0, t0, res, kb_begin, iters);
            const int acc = lt & 1;
            const uint32_t acc_ph = (lt >> 1) & 1;
            for (int i = et; i < TN; i += kPfEpiWarps * 32)
                scale[i] = (t0 + i < p.n) ? winv * ld(p.tok_inv_scale + t0 + i) : 0.0f;
            // one warp polls the accumulator's barrier (a whole tile away), the others park on the
            // hardware barrier that also publishes the scale row; a timeout shows in the abort flag
            if (ew == 0) wait_bar(ctl.accum + 8 * acc, acc_ph, ctl, 7, 1000u);
            asm volatile("bar.sync 2, %0;" ::"n"(kPfEpiWarps * 32) : "memory");
            if (*ctl.abort_flag) { ok = false; break; }
            ptx::tc_fence_after_sync();
            const int m0w = m0 + quarter * 32;
            const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * kAccCols;
            auto bias_of = [&](int m) { return (MODE == MODE_FWD && p.bias != nullptr && m < p.Mdim) ? ld(p.bias + m) : 0.0f; };
            const int step = (p.helpers && lt == nseg - 1) ? kPfHelpers : 1;  // the workers take the other boxes
            if (p.fast_epi) {
                const int g = lane >> 2, tq = lane & 3;
                float b4[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) b4[i] = bias_of(m0w + g + 8 * i);
                drain(res, m0w, t0, t_row, quarter, 0, step, [&](int col) {
                    // the store that last read this buffer has to be done with it
                    if (chunks >= 2 && lane == 0) ptx::bulk_wait_group_read<1>();
                    __syncwarp();
                    const uint32_t buf = stg + (chunks & 1u) * kPfStagingBuf;
                    float s0x, s0y, s1x, s1y;
                    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(s0x), "=f"(s0y) : "r"(scale_addr + (col + 2 * tq) * 4) : "memory");
                    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(s1x), "=f"(s1y) : "r"(scale_addr + (col + 8 + 2 * tq) * 4) : "memory");
                    store_box(t_row, col, buf, s0x, s0y, s1x, s1y, b4, m0w, t0 + col);
                    ++chunks;
                });
            } else {
                const float bias = bias_of(m0w + lane);
                drain(res, m0w, t0, t_row, quarter, 0, step, [&](int col) {
                    float sc[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) sc[c] = scale[col + c];
                    store_box_any(t_row, col, stg, sc, bias, m0w, t0);
                });
            }
            // the accumulator (and this tile's scale row) may be reused
            ptx::tc_fence_before_sync();
            asm volatile("bar.sync 2, %0;" ::"n"(kPfEpiWarps * 32) : "memory");
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::leader_addr(acc_empty + 8 * acc));
        }
        if (p.fast_epi && lane == 0) ptx::bulk_wait_group<0>();  // all output boxes written before the CTA ends
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();  // neither CTA's memory goes away under the other
    if (warp == kPfMmaWarp) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------

struct ExpandPlan {
    int TN, num_kb, m_tiles, m_pairs, n_tiles;
    int full_tiles, res_tiles, pieces, piece_len, pairs;                 // see ExpandParams
    int a_slots, b_slots;
    uint32_t bits_bytes, alpha_bytes;                                    // one stage's chunk of the planes; the scales of one (row block, group)
    size_t planes_bytes;                                                 // the regrouped planes (codes for q <= 4)
    size_t smem;                                                         // dynamic shared memory of the GEMM kernel
    size_t off_tok, off_act, off_alpha, off_bits, off_counters, off_partial, total;  // workspace layout (bytes)
    int ld_act;                                                          // pitch of the fp16 activations (elements)
};

constexpr int kPfMinPiece = 4;
constexpr int kPfBoxClasses = 1 + kPfWorkerWarps / 4;                  // counters per shared tile, CTA and lane quarter
constexpr size_t kPfFixedBytes = 1024 + kPfCtlBytes + kPfScaleBytes;   // alignment slack, barriers, output scales

// Tile width over tokens, the K split and the pipeline geometry.  Wide token tiles amortise the
// expansion of a weight tile over more tokens; the K split fills the SMs when the output has few
// tiles.
ExpandPlan plan_expand(int mode, int d_out, int d_in, int q, int g, int n) {
    ExpandPlan pl;
    const int pairs = std::max(1, sm_count() / 2);
    const int Mdim = (mode == MODE_FWD) ? d_out : d_in;
    const int Kdim = (mode == MODE_FWD) ? d_in : d_out;
    const int G = (int)bcq_num_groups(d_in, g);
    pl.m_tiles = ceil_div(Mdim, kBlockM);
    pl.m_pairs = ceil_div(pl.m_tiles, 2);
    pl.num_kb = ceil_div(Kdim, kBlockK);
    // Token tiles and K pieces, by the time a call is expected to take.  All in stages of a pair at q <= 4 (about
    // 0.3 us, set by the expansion of the weight tiles and hence nearly the same at every width; 140
    // tiles of 208 tokens take 2 % longer than 112 of 256, two waves both; q > 4 adds +-alpha_i weight by
    // weight, four times as long):
    //   * whole waves of tiles, then the ragged last wave (or all of a problem with fewer tiles than
    //     pairs), whole or cut into d pieces;
    //   * pieces that end the call are added by all 20 output warps of a CTA: 2.4 us for the way through
    //     memory, 0.33 us per piece for each of a warp's boxes of 16 tokens, and their bytes written and read
    //     at 11 TB/s.  Measured, 4096 -> 256, q = 3, 64 tokens, 1 / 2 / 4 / 8 / 16 pieces: 33.0 / 27.0 / 23.2 /
    //     22.2 / 23.2 us, 16 tokens 33.3 / 26.3 / 22.2 / 20.8 / 22.2; 64 tokens, q = 8: 86.7 / 52.2 / 34.1 / 26.6 /
    //     23.6; 4096 -> 1024 at 2048 tokens, one piece (32 tiles of 256) or two (36 of 240) 31.7 / 30.0;
    //   * pieces before whole tiles are added by four warps under the main loop of those, so they
    //     cost nothing if that is much longer (measured: 5120 -> 20480 dX with 2048 tokens, 12 of 160
    //     tiles in pieces, 429 -> 359 us; 1600 -> 6400, whose tiles are 25 stages, 79 -> 92 us);
    //   * the last output, TN / 64 stages.
    // That is the time of a call with the chip to itself.  A layer stack that runs on several streams pays for the
    // pairs that a plan holds and for how long, so a whole chip's time counts for a quarter on top of it.
    // (The rule before counted stages, not the time that pieces take to be added, and cut 4096 -> 1024 in two
    // on 72 pairs where 32 take 6 % longer: GPT-2-medium stack, 24 layers at 2048 tokens, forward, dalpha and
    // dX on nine streams 732 TFLOP/s, 792 now.)
    const int nt0 = ceil_div(n, 256), nt1 = std::min(ceil_div(n, 32), 8 * nt0);
    double best = -1.0;
    for (int nt = nt0; nt <= nt1; ++nt) {
        const int tn = std::max(32, ceil_div(ceil_div(n, nt), 16) * 16);
        if (ceil_div(n, tn) != nt) continue;
        const int tiles = pl.m_pairs * nt;
        const int waves = tiles / pairs, ragged = tiles % pairs;
        const double stage = (q <= 4 ? 1.0 : 4.0) * (1.1 - 0.1 * tn / 256.0), out = 1.0 + tn / 64.0;
        const int dmax = ragged > 0 ? std::min(pairs / ragged, pl.num_kb / kPfMinPiece) : 1;
        for (int d = 1; d <= std::max(1, dmax); ++d) {
            const int len = ceil_div(pl.num_kb, d), pieces = ceil_div(pl.num_kb, len);
            double add = 0.0;
            if (d > 1 && waves == 0)
                add = 8.0 + 1.1 * ceil_div(tn, 80) * pieces + 0.62e-6 * tiles * pieces * (double)(tn * 256 * 4);
            if (d > 1 && waves > 0 && waves * pl.num_kb < 3 * 40 * d) break;  // would not stay hidden
            const double cost = (waves * pl.num_kb + (ragged > 0 ? len : 0)) * stage + add + out;
            const int used = waves == 0 ? tiles * pieces : pieces > 1 ? pairs : ceil_div(tiles, waves + (ragged > 0 ? 1 : 0));
            const double score = cost + 0.25 * used * cost / pairs;
            if (best >= 0.0 && score >= best) continue;
            best = score;
            pl.TN = tn;
            pl.n_tiles = nt;
            pl.pieces = pieces;
            pl.piece_len = len;
            pl.res_tiles = pieces > 1 ? ragged : 0;
            pl.full_tiles = tiles - pl.res_tiles;
            pl.pairs = used;
        }
    }
    const int tn = pl.TN;

    const int rows = (mode == MODE_FWD) ? 128 : 64;
    pl.bits_bytes = (q <= 3 ? 3u : (uint32_t)q) * 1024u;  // q <= 4: selector codes (3 or 4 words per 32 weights)
    pl.alpha_bytes = (uint32_t)(q * rows * 4);
    // Shared memory.  A worker group takes about a microsecond from "the tensor core is done with my
    // slot" to "the slot holds the next tile", and a TMA load as long to land; both rings must be deep
    // enough to cover that at one stage per ~0.3 us.  These fit at every token-tile width.
    pl.a_slots = kPfWeightSlots;
    pl.b_slots = 6;
    pl.smem = pl.a_slots * (size_t)kABytes + pl.b_slots * (size_t)(tn / 2) * kBlockK * 2 +
              2 * (size_t)kPfStagingBuf + kPfFixedBytes;

    const size_t chunks_bits = (size_t)pl.m_tiles * pl.num_kb;                       // [m_tile][kb] or [u][jb]
    const size_t blocks_alpha = (size_t)((mode == MODE_FWD) ? pl.m_tiles : pl.num_kb) * G;  // [m_tile][G] or [jb][G]
    pl.ld_act = (int)align_up((size_t)Kdim, 8);
    pl.off_tok = align_up(sizeof(WsHeader), 128);
    pl.off_act = align_up(pl.off_tok + (size_t)n * sizeof(float), 128);
    pl.off_alpha = align_up(pl.off_act + (size_t)n * pl.ld_act * 2, 128);
    pl.off_bits = align_up(pl.off_alpha + blocks_alpha * pl.alpha_bytes, 128);
    pl.planes_bytes = chunks_bits * pl.bits_bytes;
    pl.off_counters = align_up(pl.off_bits + pl.planes_bytes, 128);
    pl.off_partial = align_up(pl.off_counters + (size_t)pl.res_tiles * 8 * kPfBoxClasses * sizeof(uint32_t), 128);
    pl.total = pl.off_partial + (size_t)(pl.res_tiles * pl.pieces) * tn * 256 * sizeof(float);
    return pl;
}

template <int MODE>
bcq_status ensure_expand_smem(int q, size_t smem) {
    if (q <= 3) return ensure_dynamic_smem(expand_gemm_kernel<MODE, QM_LUT3>, smem);
    if (q == 4) return ensure_dynamic_smem(expand_gemm_kernel<MODE, QM_LUT4>, smem);
    return ensure_dynamic_smem(expand_gemm_kernel<MODE, QM_GENERIC>, smem);
}

template <int MODE, int QM>
bcq_status launch_expand(const CUtensorMap& tm, const CUtensorMap& tmo, const ExpandParams& p, const ExpandPlan& pl,
                         cudaStream_t stream) {
    auto kern = expand_gemm_kernel<MODE, QM>;
    bcq_status st0 = ensure_dynamic_smem(kern, pl.smem);
    if (st0 != BCQ_OK) return st0;
    BCQ_CUDA_TRY(launch_pdl(kern, dim3(2u * (unsigned)pl.pairs), kPfThreads, pl.smem, stream, 2, tm, tmo, p));
    return BCQ_OK;
}

template <int MODE>
bcq_status launch_expand_q(const CUtensorMap& tm, const CUtensorMap& tmo, const ExpandParams& p, const ExpandPlan& pl,
                           cudaStream_t stream) {
    if (p.q <= 3) return launch_expand<MODE, QM_LUT3>(tm, tmo, p, pl, stream);
    if (p.q == 4) return launch_expand<MODE, QM_LUT4>(tm, tmo, p, pl, stream);
    return launch_expand<MODE, QM_GENERIC>(tm, tmo, p, pl, stream);
}

// Writes the selector codes of the planes (q <= 4) in the chunk order of mode `mode`.
bcq_status launch_code_planes(int mode, int d_out, int d_in, int q, const ExpandPlan& pl, const uint32_t* bits,
                              uint32_t* codes, cudaStream_t s) {
    const int pitch = (int)bcq_pitch_words(d_in);
    const int rows_padded = (mode == MODE_FWD) ? pl.m_tiles * 128 : pl.num_kb * 64;
    const int words_padded = (mode == MODE_FWD) ? pl.num_kb * 2 : pl.m_tiles * 4;
    const long long total = (long long)rows_padded * words_padded;
    const unsigned grid = (unsigned)((total + 255) / 256);
    // the pre-pass may come in early where this kernel's blocks leave room on every SM (see launch_pdl):
    // 1024 x 1024 at 64 tokens, q = 1, 128 blocks, 14.2 us a call with it and 15.4 without
    const int early = grid <= (unsigned)sm_count() ? 1 : 0;
    BCQ_CUDA_TRY(launch_pdl(q == 4 ? code_planes_kernel<4> : code_planes_kernel<3>, dim3(grid), 256, 0, s, 1, mode, d_out, pitch, q,
                            rows_padded, words_padded, pl.num_kb, early, bits, codes));
    return BCQ_OK;
}

// act: bf16 [n][ldact] with Kdim valid columns (X for the forward, dY for dX).  `prepared`: the
// planes as written by bcq_prepare_planes for this mode, or null (then `bits` is regrouped into
// the workspace by this call).
template <int MODE>
bcq_status run_expand(int d_out, int d_in, int q, int g, int n, const void* act, size_t ldact,
                      const uint32_t* bits, const void* prepared, const float* alpha, const float* bias, void* out,
                      size_t ldo, int out_dtype, void* ws, size_t ws_bytes, void* stream) {
    const int Mdim = (MODE == MODE_FWD) ? d_out : d_in;
    const int Kdim = (MODE == MODE_FWD) ? d_in : d_out;
    const ExpandPlan pl = plan_expand(MODE, d_out, d_in, q, g, n);
    // the kernel indexes the regrouped planes and scales with 32-bit word offsets
    if ((pl.planes_bytes >> 2) >= (1ull << 32) || (pl.off_bits - pl.off_alpha) / 4 >= (1ull << 32)) return BCQ_ERR_UNSUPPORTED;
    if (ws == nullptr) return BCQ_ERR_NULL;
    if (ws_bytes < pl.total) return BCQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return BCQ_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* wsb = reinterpret_cast<uint8_t*>(ws);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(wsb);
    float* tok = reinterpret_cast<float*>(wsb + pl.off_tok);
    __half* act16 = reinterpret_cast<__half*>(wsb + pl.off_act);
    const int pitch = (int)bcq_pitch_words(d_in);

    CUtensorMap tm;
    bcq_status st = make_tmap_16bit(&tm, act16, 1, pl.ld_act, n, (size_t)pl.ld_act, pl.TN / 2);
    if (st != BCQ_OK) return st;

    // everything that can fail is done before the first launch: the output tensor map and the
    // shared-memory limits of the kernels this call may run
    const bool fast_epi = (out_dtype == BCQ_BF16 && aligned16(out) && (ldo * 2) % 16 == 0 &&
                           ldo >= (size_t)Mdim);
    CUtensorMap tmo = tm;
    if (fast_epi) {
        st = make_tmap_out_bf16(&tmo, out, Mdim, n, ldo);
        if (st != BCQ_OK) return st;
    }
    if ((st = ensure_expand_smem<MODE>(q, pl.smem)) != BCQ_OK) return st;

    PrepParams pp;
    pp.n = n; pp.K = Kdim; pp.act_blocks = n;
    pp.ld_in = (long long)ldact; pp.ld_out = pl.ld_act;
    pp.in = reinterpret_cast<const __nv_bfloat16*>(act); pp.out = act16; pp.tok_inv_scale = tok;
    pp.alpha = alpha; pp.alpha_count = (long long)bcq_alpha_count(d_out, d_in, q, g); pp.hdr = hdr;
    long long ablocks = (pp.alpha_count + 256 * 16 - 1) / (256 * 16);
    if (ablocks > kMaxAlphaBlocks) ablocks = kMaxAlphaBlocks;
    if (ablocks < 1) ablocks = 1;
    pp.mode = MODE; pp.d_out = d_out; pp.q = q; pp.G = (int)bcq_num_groups(d_in, g); pp.pitch = pitch;
    pp.num_kb = pl.num_kb;
    pp.amax_blocks = (int)ablocks;
    pp.row_tiles = ceil_div(d_out, 128);
    pp.bits_cblk = ceil_div(pitch, 32);
    const bool coded = q <= 4;  // selector codes (written once, or by the launch below); q > 4: plane words
    pp.bits_blocks = coded ? 0 : q * pp.row_tiles * pp.bits_cblk;
    pp.alpha_w = 1;
    while (pp.alpha_w < 32 && pp.alpha_w < pp.G) pp.alpha_w *= 2;
    const int alpha_tr_blocks = q * pp.row_tiles * ceil_div(pp.G, pp.alpha_w);
    pp.bits = bits;
    pp.alpha_t = reinterpret_cast<float*>(wsb + pl.off_alpha);
    pp.bits_t = reinterpret_cast<uint32_t*>(wsb + pl.off_bits);
    pp.counters = reinterpret_cast<uint32_t*>(wsb + pl.off_counters);
    pp.num_counters = pl.res_tiles * 8 * kPfBoxClasses;
    if (coded && prepared == nullptr) {
        if ((st = launch_code_planes(MODE, d_out, d_in, q, pl, bits, pp.bits_t, s)) != BCQ_OK) return st;
    }
    const int nvec = (Kdim + 7) / 8;
    int wpt = 1;  // warps per token (see prepare_kernel)
    while (wpt < kPrepWarps && nvec > wpt * 128) wpt *= 2;
    const int tok_blocks = ceil_div(n, kPrepWarps / wpt);
    pp.act_blocks = tok_blocks;
    const unsigned pgrid = (unsigned)(tok_blocks + ablocks + pp.bits_blocks + alpha_tr_blocks);
    auto prep = wpt == 1 ? prepare_kernel<1> : wpt == 2 ? prepare_kernel<2> : wpt == 4 ? prepare_kernel<4>
                : nvec <= 1024 || nvec > 3072 ? prepare_kernel<8> : nvec <= 2048 ? prepare_kernel<8, 8> : prepare_kernel<8, 12>;
    BCQ_CUDA_TRY(launch_pdl(prep, dim3(pgrid), 256, 0, s, 1, pp));

    ExpandParams p;
    p.q = q; p.g = g;
    p.G = (int)bcq_num_groups(d_in, g);
    p.n = n; p.Mdim = Mdim; p.num_kb = pl.num_kb;
    p.full_tiles = pl.full_tiles; p.res_tiles = pl.res_tiles; p.pieces = pl.pieces; p.piece_len = pl.piece_len;
    p.m_tiles = pl.m_tiles; p.m_pairs = pl.m_pairs;
    p.tn = pl.TN;
    p.acc_cols = 32;
    while ((int)p.acc_cols < pl.TN) p.acc_cols *= 2;
    p.a_slots = pl.a_slots; p.b_slots = pl.b_slots; p.chunk_words = pl.bits_bytes / 4;
    p.bits_t = (coded && prepared != nullptr) ? reinterpret_cast<const uint32_t*>(prepared) : pp.bits_t;
    p.alpha_t = pp.alpha_t; p.bias = bias; p.hdr = hdr; p.tok_inv_scale = tok;
    p.out = out; p.ldo = (long long)ldo; p.out_bf16 = (out_dtype == BCQ_BF16);
    p.partial = reinterpret_cast<float*>(wsb + pl.off_partial);
    p.counters = pp.counters;
    // bf16 output with an aligned base and pitch goes out through TMA stores
    p.fast_epi = fast_epi ? 1 : 0;
    p.helpers = helpers_may_share(pl.full_tiles, pl.res_tiles > 0, pl.pairs, pl.num_kb) ? 1 : 0;
    return launch_expand_q<MODE>(tm, tmo, p, pl, s);
}

bcq_status run_decode(int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx,
                      const uint32_t* bits, const float* alpha, const float* bias, void* Y, size_t ldy,
                      int y_dtype, void* ws, size_t ws_bytes, void* stream) {
    const size_t need = decode_workspace_bytes(d_out, d_in, q, g, n);
    if (need > 0) {
        if (ws == nullptr) return BCQ_ERR_NULL;
        if (ws_bytes < need) return BCQ_ERR_WORKSPACE;
        if (!aligned16(ws)) return BCQ_ERR_ALIGN;
    }
    return run_decode_planes(d_out, d_in, q, g, n, X, ldx, bits, alpha, bias, Y, ldy, y_dtype, (cudaStream_t)stream);
}

// Argument checks of the forward and decode entry points (host arithmetic and pointer tests only).
bcq_status check_fwd_args(int decode, int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx,
                          const uint32_t* bits, const float* alpha, const void* Y, size_t ldy, int y_dtype) {
    bcq_status st = check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1 || (decode && n > 16)) return BCQ_ERR_SHAPE;
    if (!bits || !alpha || !Y) return BCQ_ERR_NULL;
    if ((st = check_act(X, ldx, d_in)) != BCQ_OK) return st;
    if (ldy < (size_t)d_out) return BCQ_ERR_SHAPE;
    if (y_dtype != BCQ_F32 && y_dtype != BCQ_BF16) return BCQ_ERR_SHAPE;
    if (!aligned16(bits)) return BCQ_ERR_ALIGN;
    return BCQ_OK;
}

bcq_status fwd_common(int decode, int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx,
                      const uint32_t* bits, const float* alpha, const float* bias, void* Y, size_t ldy,
                      int y_dtype, void* ws, size_t ws_bytes, void* stream) {
    const bcq_status st = check_fwd_args(decode, d_out, d_in, q, g, n, X, ldx, bits, alpha, Y, ldy, y_dtype);
    if (st != BCQ_OK) return st;
    if (decode)
        return run_decode(d_out, d_in, q, g, n, X, ldx, bits, alpha, bias, Y, ldy, y_dtype, ws, ws_bytes, stream);
    return run_expand<MODE_FWD>(d_out, d_in, q, g, n, X, ldx, bits, nullptr, alpha, bias, Y, ldy, y_dtype, ws,
                                ws_bytes, stream);
}

}  // namespace

namespace bcq {
bcq_status expand_timeout_flag(int* flag_out, int reset) {
    int v = 0;
    BCQ_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_timeout_flag, sizeof(int)));
    *flag_out = v;
    if (reset && v != 0) {
        const int zero = 0;
        BCQ_CUDA_TRY(cudaMemcpyToSymbol(g_timeout_flag, &zero, sizeof(int)));
    }
    return BCQ_OK;
}

size_t fwd_workspace_bytes(int d_out, int d_in, int q, int g, int n) {
    return plan_expand(MODE_FWD, d_out, d_in, q, g, n).total;
}
// The scratch that callers of bcq_linear_decode provide: partial sums of a split over d_in that gives every
// SM two row tiles of 128.  The kernel (decode.cu) keeps its sums on chip; the size and the checks on it
// stay as callers know them.
size_t decode_workspace_bytes(int d_out, int d_in, int, int, int n) {
    const int num_kb = ceil_div(d_in, kBlockK);
    const int splits = std::min({std::max(1, 2 * sm_count() / ceil_div(d_out, kBlockM)), (num_kb + 7) / 8, 64});
    const int used = ceil_div(num_kb, ceil_div(num_kb, splits));
    return used > 1 ? (size_t)used * n * d_out * sizeof(float) : 0;
}
size_t bwd_x_workspace_bytes(int d_out, int d_in, int q, int g, int n) {
    return plan_expand(MODE_BWDX, d_out, d_in, q, g, n).total;
}
}  // namespace bcq

extern "C" bcq_status bcq_linear_fwd(int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx,
                                     const uint32_t* bits, const float* alpha, const float* bias, void* Y,
                                     size_t ldy, int y_dtype, void* ws, size_t ws_bytes, void* stream) {
    return fwd_common(0, d_out, d_in, q, g, n, X, ldx, bits, alpha, bias, Y, ldy, y_dtype, ws, ws_bytes,
                      stream);
}

extern "C" bcq_status bcq_linear_decode(int d_out, int d_in, int q, int g, int n, const void* X,
                                        size_t ldx, const uint32_t* bits, const float* alpha,
                                        const float* bias, void* Y, size_t ldy, int y_dtype, void* ws,
                                        size_t ws_bytes, void* stream) {
    return fwd_common(1, d_out, d_in, q, g, n, X, ldx, bits, alpha, bias, Y, ldy, y_dtype, ws, ws_bytes,
                      stream);
}

// ------------------------------------------------------------------------------------------
// decode without a caller-provided workspace
// ------------------------------------------------------------------------------------------

extern "C" bcq_status bcq_linear_decode_noalloc(int d_out, int d_in, int q, int g, int n, const void* X,
                                                size_t ldx, const uint32_t* bits, const float* alpha,
                                                const float* bias, void* Y, size_t ldy, int y_dtype,
                                                void* stream) {
    bcq_status st = check_fwd_args(1, d_out, d_in, q, g, n, X, ldx, bits, alpha, Y, ldy, y_dtype);
    if (st != BCQ_OK) return st;
    if (bcq::decode_workspace_bytes(d_out, d_in, q, g, n) > (size_t)BCQ_NOALLOC_SCRATCH_BYTES)
        return BCQ_ERR_WORKSPACE;
    return bcq::run_decode_planes(d_out, d_in, q, g, n, X, ldx, bits, alpha, bias, Y, ldy, y_dtype, (cudaStream_t)stream);
}

extern "C" bcq_status bcq_linear_bwd_x(int d_out, int d_in, int q, int g, int n, const void* dY,
                                       size_t lddy, const uint32_t* bits, const float* alpha, void* dX,
                                       size_t lddx, int dx_dtype, void* ws, size_t ws_bytes,
                                       void* stream) {
    bcq_status st = check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1) return BCQ_ERR_SHAPE;
    if (!bits || !alpha || !dX) return BCQ_ERR_NULL;
    if ((st = check_act(dY, lddy, d_out)) != BCQ_OK) return st;
    if (lddx < (size_t)d_in) return BCQ_ERR_SHAPE;
    if (dx_dtype != BCQ_F32 && dx_dtype != BCQ_BF16) return BCQ_ERR_SHAPE;
    if (!aligned16(bits)) return BCQ_ERR_ALIGN;
    return run_expand<MODE_BWDX>(d_out, d_in, q, g, n, dY, lddy, bits, nullptr, alpha, nullptr, dX, lddx, dx_dtype,
                                 ws, ws_bytes, stream);
}

// ------------------------------------------------------------------------------------------
// planes prepared once (B is frozen)
// ------------------------------------------------------------------------------------------

namespace {
bcq_status check_prepared(int op, int d_out, int d_in, int q, int g) {
    bcq_status st = check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (op != BCQ_OP_FWD && op != BCQ_OP_BWD_X) return BCQ_ERR_SHAPE;
    if (q > 4) return BCQ_ERR_UNSUPPORTED;
    return BCQ_OK;
}
}  // namespace

extern "C" size_t bcq_prepared_bytes(int op, int d_out, int d_in, int q, int g) {
    if (check_prepared(op, d_out, d_in, q, g) != BCQ_OK) return 0;
    return plan_expand(op == BCQ_OP_FWD ? MODE_FWD : MODE_BWDX, d_out, d_in, q, g, 256).planes_bytes;
}

extern "C" bcq_status bcq_prepare_planes(int op, int d_out, int d_in, int q, int g, const uint32_t* bits,
                                         void* prepared, size_t prepared_bytes, void* stream) {
    bcq_status st = check_prepared(op, d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (!bits || !prepared) return BCQ_ERR_NULL;
    if (!aligned16(bits) || !aligned16(prepared)) return BCQ_ERR_ALIGN;
    const int mode = (op == BCQ_OP_FWD) ? MODE_FWD : MODE_BWDX;
    const ExpandPlan pl = plan_expand(mode, d_out, d_in, q, g, 256);
    if (prepared_bytes < pl.planes_bytes) return BCQ_ERR_WORKSPACE;
    return launch_code_planes(mode, d_out, d_in, q, pl, bits, reinterpret_cast<uint32_t*>(prepared),
                              (cudaStream_t)stream);
}

extern "C" bcq_status bcq_linear_fwd_prepared(int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx,
                                              const void* prepared, const float* alpha, const float* bias,
                                              void* Y, size_t ldy, int y_dtype, void* ws, size_t ws_bytes,
                                              void* stream) {
    bcq_status st = check_prepared(BCQ_OP_FWD, d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1) return BCQ_ERR_SHAPE;
    if (!prepared || !alpha || !Y) return BCQ_ERR_NULL;
    if ((st = check_act(X, ldx, d_in)) != BCQ_OK) return st;
    if (ldy < (size_t)d_out) return BCQ_ERR_SHAPE;
    if (y_dtype != BCQ_F32 && y_dtype != BCQ_BF16) return BCQ_ERR_SHAPE;
    if (!aligned16(prepared)) return BCQ_ERR_ALIGN;
    return run_expand<MODE_FWD>(d_out, d_in, q, g, n, X, ldx, nullptr, prepared, alpha, bias, Y, ldy, y_dtype, ws,
                                ws_bytes, stream);
}

extern "C" bcq_status bcq_linear_bwd_x_prepared(int d_out, int d_in, int q, int g, int n, const void* dY,
                                                size_t lddy, const void* prepared, const float* alpha, void* dX,
                                                size_t lddx, int dx_dtype, void* ws, size_t ws_bytes, void* stream) {
    bcq_status st = check_prepared(BCQ_OP_BWD_X, d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1) return BCQ_ERR_SHAPE;
    if (!prepared || !alpha || !dX) return BCQ_ERR_NULL;
    if ((st = check_act(dY, lddy, d_out)) != BCQ_OK) return st;
    if (lddx < (size_t)d_in) return BCQ_ERR_SHAPE;
    if (dx_dtype != BCQ_F32 && dx_dtype != BCQ_BF16) return BCQ_ERR_SHAPE;
    if (!aligned16(prepared)) return BCQ_ERR_ALIGN;
    return run_expand<MODE_BWDX>(d_out, d_in, q, g, n, dY, lddy, nullptr, prepared, alpha, nullptr, dX, lddx,
                                 dx_dtype, ws, ws_bytes, stream);
}
