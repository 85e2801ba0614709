// Decode (1..16 tokens): from a packed copy of the frozen weights (bcq_decode_pack and
// bcq_linear_decode_packed), and from the canonical planes and scales (the kernel of bcq_linear_decode).
//
// Decode streams every weight once and uses it for at most 16 tokens, so the time is set by the
// bytes of the pack and by how cheaply a weight gets from its bits into a tensor-core operand
// (Section "Inference Speed": the cost of a small-batch layer is moving its weights).  B and, at
// inference, alpha are frozen, so everything that does not depend on the activations is done once,
// when the pack is written:
//
//   codes   for every weight the index of its level among the 2^q sums +-alpha_1 .. +-alpha_q of
//           its (row, group), as a 4-bit selector nibble for PRMT (lut.cuh), q bits per weight;
//   tables  for every (row, group) the eight fp16 levels as a byte-wise lookup table of four
//           registers, pre-multiplied by a power of two per row that brings q * max|alpha| of the
//           row to [2^13, 2^14).
//
// A warp expands codes straight into the A fragments of mma.m16n8k16 (fp16): no operand tile in shared
// memory, no barrier between expansion and product, no accumulator to fetch from tensor memory.  What is
// left per weight is 1.6 (q = 4) or 1.2 (q = 3) instructions of the logic pipe (64 lanes per clock and SM),
// 39 - 53 weights per clock and SM where HBM delivers 37 - 46.
//
// Work split: a unit is 16 rows x 128 k.  The 16-row tiles are dealt to the CTAs (one per SM).  The
// units of a CTA, numbered step by step with all tiles of a step together, are dealt to its warps, so a
// step's activations are converted once (bf16 -> fp16 times a power of two per token and step) and stay in
// registers as B fragments.  Its sums wait in a private slot of shared memory per tile; the slots of a
// tile are added at the end, in order.  Where there are too few tiles for the SMs, the CTAs of a cluster
// share the steps of a tile (deal_tiles); otherwise no CTA needs another.
//
// One CTA of 16 warps an SM: with two of 8 warps, each CTA had half as many tiles to use a step's activations
// for (OPT-6.7B layer, q = 4, one token: 68 us against 53); 20 or 24 warps with fewer registers each
// were no faster (54 us) and slower for 16 tokens (73 and 92 us against 66).
//
// Weights go from global memory to registers a unit ahead of their use, and the code of a unit is there once: two register
// sets in turn, two units ahead, doubled it, and a loop that fits the instruction caches gains more than the distance
// (4096 -> 16384, q = 4, one token 15.2 us and 13.9; the same pack from L2 takes no less time than from memory, so what
// bounds a unit is not its way here but the logic pipe).  The kernel may start
// while the previous kernel of the stream is finishing (programmatic dependent launch).  That may be the
// kernel that writes the pack, and only the grid dependency wait makes its writes visible, so nothing
// is read before it; the first two units are merely brought into L2.
#include <algorithm>

#include "gemm_common.cuh"
#include "lut.cuh"

namespace {

using namespace bcq;

constexpr int kDpWarps = 16;
constexpr int kDpThreads = kDpWarps * 32;
constexpr int kDpStepK = 128;      // weights of a row per unit: eight K = 16 MMAs
constexpr int kDpRows = 16;        // rows of a unit: the M of the MMA
constexpr uint32_t kDpTableBytes = kDpRows * 16;  // tables of one (tile, group)
constexpr size_t kDpMaxSmem = 232448;  // of a CTA
constexpr int kDpMaxRound = 24;    // tiles a CTA takes between two additions of its warps' sums

// ------------------------------------------------------------------------------------------
// pack layout (host and device)
//   rinv    float  [tile][16 rows]      inverse of the row's power of two
//   tables  uint4  [tile][G][16 rows]
//   codes   uint32 [tile][step][2 q words per lane], words ordered for the widest loads
// Lane (g = lane / 4, t = lane % 4) of a unit has the q words of rows g and g + 8; nibble e of its
// selector word r is the weight k = 32 r + 8 t + e of the step.
// ------------------------------------------------------------------------------------------

struct PackLayout {
    int tiles, steps, parts, G;
    size_t off_tables, off_codes, total;
};

// Pieces of a step that may belong to different groups.
__host__ __device__ inline int dp_parts(int g, int G) {
    if (G == 1 || g % 128 == 0) return 1;
    if (g % 64 == 0) return 2;
    return 4;
}

PackLayout pack_layout(int d_out, int d_in, int q, int g) {
    PackLayout L;
    L.tiles = ceil_div(d_out, kDpRows);
    L.steps = ceil_div(d_in, kDpStepK);
    L.G = (int)bcq_num_groups(d_in, g);
    L.parts = dp_parts(g, L.G);
    L.off_tables = align_up((size_t)L.tiles * kDpRows * 4, 128);
    L.off_codes = align_up(L.off_tables + (size_t)L.tiles * L.G * kDpTableBytes, 128);
    L.total = L.off_codes + (size_t)L.tiles * L.steps * q * 256u;
    return L;
}

// Position (in words) of word `w` (row half w / Q, word w % Q) of a lane inside a unit's codes: as many
// 16-byte vectors per lane as there are, then one 8-byte vector (odd q).
template <int Q>
__device__ __forceinline__ uint32_t code_pos(int w, int lane) {
    if (w >= (Q / 2) * 4) return (uint32_t)(Q / 2) * 128u + lane * 2 + (w & 1);
    return (uint32_t)(w >> 2) * 128u + lane * 4 + (w & 3);
}

// ------------------------------------------------------------------------------------------
// writing the pack
// ------------------------------------------------------------------------------------------

// One thread per weight row: the power of two of the row and its inverse.
__global__ void pack_rowscale_kernel(int d_out, int q, int G, int rows_padded, const float* alpha,
                                     float* rinv) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= rows_padded) return;
    float inv = 1.0f;
    if (j < d_out) {
        uint32_t am = 0u;
        for (int i = 0; i < q; ++i)
            for (int c = 0; c < G; ++c)
                am = max(am, __float_as_uint(ld(alpha + ((long long)i * d_out + j) * G + c)) & 0x7FFFFFFFu);
        inv = pow2f(-shift_for(exponent_of_bits(__float_as_uint(__uint_as_float(am) * (float)q)), 13));
    }
    rinv[j] = inv;
}

// One thread per (tile, group, row): the lookup table of the row's levels in that group.
__global__ void pack_tables_kernel(int d_out, int q, int G, long long total, const float* alpha,
                                   const float* rinv, uint4* tables) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int c = (int)((idx >> 4) % G);
    const int j = (int)((idx >> 4) / G) * kDpRows + (int)(idx & 15);
    uint4 out = make_uint4(0u, 0u, 0u, 0u);  // rows past d_out expand to zeros
    if (j < d_out) {
        const float wscale = 1.0f / ld(rinv + j);  // a power of two
        float a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            a[i] = (i < q) ? ld(alpha + ((long long)i * d_out + j) * G + c) * wscale : 0.0f;
        const Lut t = build_lut(a[0], a[1], a[2], a[3]);  // q <= 3: a[3] = 0 is the base
        out = make_uint4(t.tl0, t.tl1, t.th0, t.th1);
    }
    tables[idx] = out;
}

// One warp per unit.
template <int Q>
__global__ void __launch_bounds__(256) pack_codes_kernel(int d_out, int pitch, int tiles, int steps,
                                                         const uint32_t* bits, uint32_t* codes) {
    const long long unit = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (unit >= (long long)tiles * steps) return;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int st = (int)(unit % steps);
    const int tile = (int)(unit / steps);
    uint32_t* dst = codes + unit * (Q * 64);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int j = tile * kDpRows + g + 8 * half;
        uint32_t out[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) out[i] = 0u;
        if (j < d_out) {
            // byte r of w[i]: the plane's bits of this lane's eight weights in the step's r-th word
            uint32_t w[4] = {0u, 0u, 0u, 0u}, S[4];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const uint4 src = ld(reinterpret_cast<const uint4*>(bits + ((long long)i * d_out + j) * pitch) + st);
                w[i] = ((src.x >> (8 * t)) & 0xFFu) | (((src.y >> (8 * t)) & 0xFFu) << 8) |
                       (((src.z >> (8 * t)) & 0xFFu) << 16) | (((src.w >> (8 * t)) & 0xFFu) << 24);
            }
            selectors_from_planes(w, Q, S);
            pack_selectors<Q>(S, out);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) dst[code_pos<Q>(half * Q + i, lane)] = out[i];
    }
}

// ------------------------------------------------------------------------------------------
// the decode kernel
// ------------------------------------------------------------------------------------------

// Where the sums of a decode kernel go.
struct DecOut {
    int d_out, n;
    const float* bias;
    void* out;
    long long ldo;
    int out_bf16;
};

// The sums of `ntiles` 16-row tiles from tile0 on: added over the warps of the CTA, in order, and written.
//   sums [warp][max_tiles][NT][32 lanes]: lane (g, t) has rows g (x, y) and g + 8 (z, w), tokens 2 t, 2 t + 1
// SPLIT: the `split` CTAs of a cluster hold parts of the same sums; the first one adds them, in order of rank.
template <int NT, bool SPLIT>
__device__ __forceinline__ void add_and_store(const DecOut& o, float4* sums, int max_tiles, int ntiles, int tile0,
                                              const float* rinv, int split) {
    const int items = ntiles * NT * 32;
    auto over_warps = [&](int e) {
        const float4* src = sums + e;
        float4 s = src[0];
        for (int w = 1; w < kDpWarps; ++w) {
            const float4 x = src[(size_t)w * max_tiles * (NT * 32)];
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        return s;
    };
    const int rank = SPLIT ? (int)ptx::cluster_rank() : 0;
    if (SPLIT) {
        if (rank > 0)
            for (int e = threadIdx.x; e < items; e += kDpThreads) sums[e] = over_warps(e);
        __syncthreads();
        ptx::cluster_sync();
    }
    for (int e = threadIdx.x; rank == 0 && e < items; e += kDpThreads) {
        const int ti = e / (NT * 32), ln = e & 31, nt = (e >> 5) % NT;
        float4 s = over_warps(e);
        for (int r = 1; SPLIT && r < split; ++r) {
            const float4 x = ptx::ld_cluster_v4(ptx::cluster_addr(ptx::smem_u32(sums + e), (uint32_t)r));
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        const int tok = nt * 8 + 2 * (ln & 3);
        if (tok >= o.n) continue;
        const int j0 = (tile0 + ti) * kDpRows + (ln >> 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + 8 * h;
            if (j >= o.d_out) continue;
            const float scale = rinv != nullptr ? ld(rinv + j) : 1.0f, bias = o.bias != nullptr ? ld(o.bias + j) : 0.0f;
            const float v[2] = {(h ? s.z : s.x) * scale + bias, (h ? s.w : s.y) * scale + bias};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (tok + c >= o.n) continue;
                const long long at = (long long)(tok + c) * o.ldo + j;
                if (o.out_bf16) reinterpret_cast<__nv_bfloat16*>(o.out)[at] = __float2bfloat16_rn(v[c]);
                else reinterpret_cast<float*>(o.out)[at] = v[c];
            }
        }
    }
    if (SPLIT) {  // the sums have been read
        __syncthreads();
        ptx::cluster_sync();
    }
}

// 32 activations of one token as fp16 times a power of two per (token, 128-k step): the four lanes of a
// quad hold the step, v[r] the eight elements from k0 + r * stride on.  Returns the inverse scale.
__device__ __forceinline__ float scale_fragment(uint4 (&v)[4], int k0, int stride, int d_in, bool ragged) {
    if (ragged) {  // columns past d_in count as zeros
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            uint32_t* w = &v[r].x;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (k0 + r * stride + e >= d_in) w[e >> 1] &= (e & 1) ? 0x0000FFFFu : 0xFFFF0000u;
        }
    }
    uint32_t mm = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r)
        mm = __vmaxu2(mm, __vmaxu2(__vmaxu2(v[r].x & 0x7FFF7FFFu, v[r].y & 0x7FFF7FFFu),
                                   __vmaxu2(v[r].z & 0x7FFF7FFFu, v[r].w & 0x7FFF7FFFu)));
    uint32_t mag = max(mm & 0xFFFFu, mm >> 16);
    mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, 1));
    mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, 2));
    const int sh = shift_for(exponent_of_bits(mag << 16), 14);
    const float sc = pow2f(sh);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        uint32_t* w = &v[r].x;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[e] = pack_half2(__uint_as_float(w[e] << 16) * sc, __uint_as_float(w[e] & 0xFFFF0000u) * sc);
    }
    return pow2f(-sh);
}

struct DecPackedParams {
    int d_out, d_in, g, G, n;
    int steps;
    int per, rem;            // row tiles per CTA and remainder
    int round;               // tiles between two additions
    int split;               // CTAs of a cluster that share the steps of their tiles
    uint32_t x_stride;       // XS: bytes of a token's fragments in shared memory
    uint32_t g_magic;        // ceil(2^32 / g) where k / g = hi32(k g_magic) for every k < d_in, else 0
    const __nv_bfloat16* X;
    long long ldx;
    const uint8_t* codes;
    const uint8_t* tables;
    const float* rinv;
    DecOut o;
};

// D += A B, 16 x 8 x 16, fp16 operands.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Eight weights of one row: their selector word through the row's table to four fp16 pairs.
template <int Q>
__device__ __forceinline__ void expand8(uint32_t S, const uint4& t, uint32_t (&out)[4]) {
    // (shifts written as multiplications run on the multiply-add pipe; the logic pipe, which does the
    // PRMTs, is the one that paces this loop)
    const uint32_t s = (Q == 4) ? (S & 0x77777777u) : S;
    const uint32_t sh = __umulhi(s, 1u << 16);
    const uint32_t lbl = prmt(t.x, t.y, s), lbh = prmt(t.x, t.y, sh);
    uint32_t hbl = prmt(t.z, t.w, s), hbh = prmt(t.z, t.w, sh);
    if (Q == 4) {
        // bit 3 of nibble e = "negate": replicated over byte e by PRMT's sign mode
        const uint32_t fa = S * 16u;
        hbl ^= prmt(fa, S, 0xD9C8u) & 0x80808080u;
        hbh ^= prmt(fa, S, 0xFBEAu) & 0x80808080u;
    }
    out[0] = prmt(lbl, hbl, 0x5140u);
    out[1] = prmt(lbl, hbl, 0x7362u);
    out[2] = prmt(lbh, hbh, 0x5140u);
    out[3] = prmt(lbh, hbh, 0x7362u);
}

// The words of a unit that one lane needs, on their way from global memory.
template <int Q, int PARTS>
struct UnitWords {
    uint32_t c[2 * Q];
    uint4 ta[PARTS], tb[PARTS];  // tables of rows g and g + 8
};

// XS (few tokens, see launch_decode_packed): the CTA's activations are converted once, by all threads, into shared memory.  A
// warp that converts a step for itself works for eight tokens whatever their number, and again for every step.
template <int Q, int NT, int PARTS, bool SPLIT, bool XS>
__global__ void __launch_bounds__(kDpThreads, 1)
decode_packed_kernel(const DecPackedParams p) {
    extern __shared__ float4 sums[];  // [warp][slot][NT][32 lanes]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gr = lane >> 2, tq = lane & 3;
    const int cta = SPLIT ? (int)blockIdx.x / p.split : (int)blockIdx.x;
    const int tile0 = cta * p.per + min(cta, p.rem);
    const int ntiles = p.per + (cta < p.rem ? 1 : 0);
    // the CTA's steps: all of them, or its rank's share
    const int part = SPLIT ? (int)blockIdx.x - cta * p.split : 0;
    const int step0 = SPLIT ? (int)((long long)p.steps * part / p.split) : 0;
    const int nsteps = SPLIT ? (int)((long long)p.steps * (part + 1) / p.split) - step0 : p.steps;
    float4* mine = sums + (size_t)warp * p.round * (NT * 32) + lane;

    // XS: fragments [token][step][r][t] of 16 bytes, then the inverse scales [token][step]
    uint8_t* xfrag = reinterpret_cast<uint8_t*>(sums + (size_t)kDpWarps * p.round * (NT * 32));
    float* xinv = reinterpret_cast<float*>(xfrag + (size_t)p.n * p.x_stride);

    pdl_trigger();
    for (int first = 0; first < ntiles; first += p.round) {
        const int round_n = min(p.round, ntiles - first);
        // the warp's units: an equal, contiguous share of the round's, numbered step by step
        const int all = round_n * nsteps;
        const int u0 = all * warp / kDpWarps, u1 = all * (warp + 1) / kDpWarps;
        const int st0 = step0 + u0 / round_n, i0 = u0 - (st0 - step0) * round_n;

        // ---- loading: unit (step, tile) pairs in the order of use
        const uint8_t* lp_codes = p.codes;
        const uint8_t* lp_tables[PARTS];
        int l_st = st0, l_i = i0, l_left = u1 - u0;
        auto seek = [&]() {  // to tile l_i of step l_st
            const size_t tile = (size_t)(tile0 + first + l_i);
            lp_codes = p.codes + (tile * p.steps + l_st) * (Q * 256) + lane * 16;
#pragma unroll
            for (int a = 0; a < PARTS; ++a) {
                const int k = l_st * kDpStepK + a * (kDpStepK / PARTS);
                const int c = min(p.g_magic != 0u ? (int)__umulhi((uint32_t)k, p.g_magic) : k / p.g, p.G - 1);
                lp_tables[a] = p.tables + (tile * p.G + c) * kDpTableBytes + gr * 16;
            }
        };
        const size_t codes_stride = (size_t)p.steps * (Q * 256), tables_stride = (size_t)p.G * kDpTableBytes;
        auto touch = [&]() {  // into L2: the first unit and the next one of the step
            for (int u = 0; u < min(2, l_left); ++u) {
                if (u > 0 && l_i + u >= round_n) break;
#pragma unroll
                for (int v = 0; v < (Q + 1) / 2; ++v) ptx::prefetch_l2(lp_codes + u * codes_stride + v * 512 - (2 * v + 1 == Q ? lane * 8 : 0));
#pragma unroll
                for (int a = 0; a < PARTS; ++a) {
                    ptx::prefetch_l2(lp_tables[a] + u * tables_stride);
                    ptx::prefetch_l2(lp_tables[a] + u * tables_stride + 128);
                }
            }
        };
        auto load = [&](UnitWords<Q, PARTS>& u) {
            if (l_left == 0) return;
            --l_left;
#pragma unroll
            for (int v = 0; v < Q / 2; ++v) {
                const uint4 x = ld_stream(reinterpret_cast<const uint4*>(lp_codes + v * 512));
                u.c[4 * v] = x.x; u.c[4 * v + 1] = x.y; u.c[4 * v + 2] = x.z; u.c[4 * v + 3] = x.w;
            }
            if (Q & 1) {
                const uint2 x = ld_stream(reinterpret_cast<const uint2*>(lp_codes + (Q / 2) * 512 - lane * 8));
                u.c[2 * Q - 2] = x.x; u.c[2 * Q - 1] = x.y;
            }
#pragma unroll
            for (int a = 0; a < PARTS; ++a) {
                u.ta[a] = ld_stream(reinterpret_cast<const uint4*>(lp_tables[a]));
                u.tb[a] = ld_stream(reinterpret_cast<const uint4*>(lp_tables[a] + 128));
            }
            if (++l_i == round_n) {
                l_i = 0;
                ++l_st;
                seek();
            } else {
                lp_codes += codes_stride;
#pragma unroll
                for (int a = 0; a < PARTS; ++a) lp_tables[a] += tables_stride;
            }
        };
        UnitWords<Q, PARTS> next;
        seek();
        if (first == 0) touch();
        for (int i = 0; i < round_n * NT; ++i) mine[i * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (first == 0) pdl_wait();
        load(next);
        if (XS && first == 0) {
            const int items = p.n * nsteps * 4;  // four lanes hold a step of a token
            for (int e = threadIdx.x; e < ((items + 31) & ~31); e += kDpThreads) {
                const int ts = e >> 2, tok = ts / nsteps, st = ts - tok * nsteps;
                const int kb = (step0 + st) * kDpStepK + tq * 8;
                const __nv_bfloat16* src = p.X + (long long)tok * p.ldx + kb;
                uint4 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    v[r] = make_uint4(0u, 0u, 0u, 0u);
                    if (e < items && kb + r * 32 < p.d_in) v[r] = ld(reinterpret_cast<const uint4*>(src + r * 32));
                }
                const float inv = scale_fragment(v, kb, 32, p.d_in, (step0 + st) * kDpStepK + kDpStepK > p.d_in);
                if (e < items) {
                    uint4* dst = reinterpret_cast<uint4*>(xfrag + (size_t)tok * p.x_stride + st * 256) + tq;
#pragma unroll
                    for (int r = 0; r < 4; ++r) dst[4 * r] = v[r];
                    if (tq == 0) xinv[tok * nsteps + st] = inv;
                }
            }
            __syncthreads();
        }
        if (!XS && first == 0) {
            // the activations of the warp's later steps: into L1 while the first step is at work
            // (32 lanes: 16 tokens x two 128-byte lines of a step)
            for (int s = st0 + 1; (s - step0) * round_n < u1; ++s) {
                const int k = s * kDpStepK + (lane & 1) * 64;
                if ((lane >> 1) < p.n && k < p.d_in)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(p.X + (long long)(lane >> 1) * p.ldx + k));
            }
        }

        // ---- a step's activations as B fragments: lane (g, t) holds token g of each tile of eight, the
        // eight k 32 r + 8 t .. + 7 for both MMAs of selector word r
        uint4 xb[NT][4];
        float f0[NT], f1[NT];  // inverse scales of the tokens of this lane's sums: 2 t, 2 t + 1
        auto load_x = [&](int st) {
            if constexpr (XS) {
                const int at = st - step0;
                const uint4* src = reinterpret_cast<const uint4*>(xfrag + (size_t)gr * p.x_stride + at * 256) + tq;
#pragma unroll
                for (int r = 0; r < 4; ++r) xb[0][r] = gr < p.n ? src[4 * r] : make_uint4(0u, 0u, 0u, 0u);
                f0[0] = 2 * tq < p.n ? xinv[2 * tq * nsteps + at] : 0.f;
                f1[0] = 2 * tq + 1 < p.n ? xinv[(2 * tq + 1) * nsteps + at] : 0.f;
                return;
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const int tok = nt * 8 + gr;
                const int kb = st * kDpStepK + tq * 8;
                const __nv_bfloat16* src = p.X + (long long)tok * p.ldx + kb;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    xb[nt][r] = make_uint4(0u, 0u, 0u, 0u);
                    if (tok < p.n && kb + r * 32 < p.d_in) xb[nt][r] = ld(reinterpret_cast<const uint4*>(src + r * 32));
                }
                const float inv = scale_fragment(xb[nt], kb, 32, p.d_in, st * kDpStepK + kDpStepK > p.d_in);
                f0[nt] = __shfl_sync(0xffffffffu, inv, 8 * tq);
                f1[nt] = __shfl_sync(0xffffffffu, inv, 8 * tq + 4);
            }
        };

        int u_st = st0, u_i = i0;
        bool fresh = true;
        auto unit = [&](const UnitWords<Q, PARTS>& u) {
            float d[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
            uint32_t wa[Q], wb[Q], Sa[4], Sb[4];
#pragma unroll
            for (int e = 0; e < Q; ++e) { wa[e] = u.c[e]; wb[e] = u.c[Q + e]; }
            selectors<Q>(wa, Sa);
            selectors<Q>(wb, Sb);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                uint32_t ra[4], rb[4];
                expand8<Q>(Sa[r], u.ta[r * PARTS / 4], ra);
                expand8<Q>(Sb[r], u.tb[r * PARTS / 4], rb);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    mma_f16(d[nt], ra[0], rb[0], ra[1], rb[1], xb[nt][r].x, xb[nt][r].y);
                    mma_f16(d[nt], ra[2], rb[2], ra[3], rb[3], xb[nt][r].z, xb[nt][r].w);
                }
            }
            float4* slot = mine + u_i * (NT * 32);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float4 s = slot[nt * 32];
                s.x = fmaf(f0[nt], d[nt][0], s.x);
                s.y = fmaf(f1[nt], d[nt][1], s.y);
                s.z = fmaf(f0[nt], d[nt][2], s.z);
                s.w = fmaf(f1[nt], d[nt][3], s.w);
                slot[nt * 32] = s;
            }
            fresh = (++u_i == round_n);
            if (fresh) { u_i = 0; ++u_st; }
        };
#pragma unroll 1
        for (int u = u0; u < u1; ++u) {
            if (fresh) load_x(u_st);
            const UnitWords<Q, PARTS> now = next;
            load(next);
            unit(now);
        }

        __syncthreads();
        add_and_store<NT, SPLIT>(p.o, sums, p.round, round_n, tile0 + first, p.rinv, p.split);
        if (first + p.round < ntiles) __syncthreads();  // the slots are written again
    }
}

// ------------------------------------------------------------------------------------------
// decode from the canonical planes (bcq_linear_decode: the scales may change between calls, any q <= 8)
// ------------------------------------------------------------------------------------------
//
// The same kernel with another way from memory to a fragment.  Lane (g, t) takes the plane words of rows g
// and g + 8 that hold the k 32 t .. + 31 of the step, and the scales of their group.  q <= 4: the level
// table of a (row, group) is built in registers and the selector nibbles of four weights are gathered
// from the plane bits with shifts and masks (2.75 instructions per weight where the pack needs 1.6); q > 4:
// fp32 sums of +-alpha_i.  Levels carry a power of two per (row, step) that brings the largest sum of
// |alpha_i| to [2^13, 2^14), taken out of the sums again in fp32.
// This replaced a tcgen05 kernel with a split over K and a second kernel that added the parts.
//
// Weights are on their way one unit ahead, as in the kernel above, or (DEEP, see launch_decode_planes) two units ahead in
// two register sets that take turns.

struct DecPlanesParams {
    int d_out, d_in, q, g, G, n;
    int steps, pitch;
    int per, rem, round, split;  // see DecPackedParams
    uint32_t g_magic;
    const __nv_bfloat16* X;
    long long ldx;
    const uint32_t* bits;
    const float* alpha;
    DecOut o;
};

// Planes and scales of one (16-row tile, step) as one lane needs them: rows g and g + 8.
template <int NQ>
struct PlaneWords {
    uint32_t wa[NQ], wb[NQ];
    float aa[NQ], ab[NQ];
};

// Pairs of one row's 32 weights for the MMA (r, h): weights 16 h + r and + 4, + 8 and + 12.  NQ = 3: levels of
// three planes; 4: table for b_4 = +1, mirrored and negated where b_4 = -1; 8: fp32 sums.
template <int NQ>
struct RowExpand {
    Lut t;
    uint32_t x[NQ == 8 ? 8 : 4];  // plane words (NQ = 4: mirrored; x[3] bit set where b_4 = -1)
    float a[NQ == 8 ? 8 : 1];

    __device__ __forceinline__ void begin(const uint32_t (&w)[NQ], const float (&al)[NQ], float scale) {
        if constexpr (NQ == 8) {
#pragma unroll
            for (int i = 0; i < 8; ++i) { x[i] = ~w[i]; a[i] = al[i] * scale; }
        } else if constexpr (NQ == 4) {
            t = build_lut(al[0] * scale, al[1] * scale, al[2] * scale, al[3] * scale);
#pragma unroll
            for (int i = 0; i < 3; ++i) x[i] = ~(w[i] ^ w[3]);
            x[3] = ~w[3];
        } else {
            t = build_lut(al[0] * scale, al[1] * scale, al[2] * scale, 0.0f);
#pragma unroll
            for (int i = 0; i < 3; ++i) x[i] = w[i];
        }
    }
    // selector word of residue r: nibble m = level index of weight 4 m + r
    __device__ __forceinline__ uint32_t select(int r) const {
        constexpr uint32_t M = 0x11111111u;
        const uint32_t b = r >= 1 ? x[1] >> (r >= 1 ? r - 1 : 0) : x[1] << 1;
        const uint32_t c = r >= 2 ? x[2] >> (r >= 2 ? r - 2 : 0) : x[2] << (r >= 2 ? 0 : 2 - r);
        return ((x[0] >> r) & M) | (b & (M << 1)) | (c & (M << 2));
    }
    __device__ __forceinline__ void pairs(uint32_t S, int r, int h, uint32_t& lo, uint32_t& hi) const {
        if constexpr (NQ == 8) {
            float v[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                v[m] = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i)  // planes past q have zero scales
                    v[m] += __uint_as_float(__float_as_uint(a[i]) ^ ((x[i] << (31 - (16 * h + r + 4 * m))) & 0x80000000u));
            }
            lo = pack_half2(v[0], v[1]);
            hi = pack_half2(v[2], v[3]);
        } else {
            const uint32_t sel = h ? (S >> 16) : S;
            uint32_t hb = prmt(t.th0, t.th1, sel);
            const uint32_t lb = prmt(t.tl0, t.tl1, sel);
            if (NQ == 4) {
                // bytes of the flag word = 0xFF where the weight's b_4 is -1 (weights m = 0..3 sit 4 bits apart)
                const int p0 = 16 * h + r;
                const uint32_t s02 = (p0 <= 7) ? (x[3] << (p0 <= 7 ? 7 - p0 : 0)) : (x[3] >> (p0 > 7 ? p0 - 7 : 0));
                const uint32_t s13 = (p0 <= 3) ? (x[3] << (p0 <= 3 ? 3 - p0 : 0)) : (x[3] >> (p0 > 3 ? p0 - 3 : 0));
                hb ^= prmt(s02, s13, 0xD9C8u) & 0x80808080u;
            }
            lo = prmt(lb, hb, 0x5140u);
            hi = prmt(lb, hb, 0x7362u);
        }
    }
};

template <int NQ, int NT, bool SPLIT, bool DEEP>
__global__ void __launch_bounds__(kDpThreads, 1)
decode_planes_kernel(const DecPlanesParams p) {
    extern __shared__ float4 sums[];  // [warp][tile][NT][32 lanes]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gr = lane >> 2, tq = lane & 3;
    const int cta = SPLIT ? (int)blockIdx.x / p.split : (int)blockIdx.x;
    const int tile0 = cta * p.per + min(cta, p.rem);
    const int ntiles = p.per + (cta < p.rem ? 1 : 0);
    // the CTA's steps: all of them, or its rank's share
    const int part = SPLIT ? (int)blockIdx.x - cta * p.split : 0;
    const int step0 = SPLIT ? (int)((long long)p.steps * part / p.split) : 0;
    const int nsteps = SPLIT ? (int)((long long)p.steps * (part + 1) / p.split) - step0 : p.steps;
    float4* mine = sums + (size_t)warp * p.round * (NT * 32) + lane;
    const size_t plane_bits = (size_t)p.d_out * p.pitch, plane_alpha = (size_t)p.d_out * p.G;

    pdl_trigger();
    pdl_wait();  // the scales may come from the kernel before this one
    for (int first = 0; first < ntiles; first += p.round) {
        const int round_n = min(p.round, ntiles - first);
        const int all = round_n * nsteps;
        const int u0 = all * warp / kDpWarps, u1 = all * (warp + 1) / kDpWarps;
        const int st0 = step0 + u0 / round_n, i0 = u0 - (st0 - step0) * round_n;

        int l_st = st0, l_i = i0, l_c = 0, l_left = u1 - u0;
        auto group_of = [&](int st) {  // group of this lane's 32 weights
            const int k = st * kDpStepK + 32 * tq;
            return min(p.g_magic != 0u ? (int)__umulhi((uint32_t)k, p.g_magic) : k / p.g, p.G - 1);
        };
        l_c = group_of(l_st);
        auto load = [&](PlaneWords<NQ>& u) {
            if (l_left == 0) return;
            --l_left;
            const int ja = (tile0 + first + l_i) * kDpRows + gr, jb = ja + 8;
            const uint32_t* pb = p.bits + (size_t)ja * p.pitch + l_st * 4 + tq;
            const float* pa = p.alpha + (size_t)ja * p.G + l_c;
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const bool va = i < p.q && ja < p.d_out, vb = i < p.q && jb < p.d_out;
                u.wa[i] = va ? ld(pb + i * plane_bits) : 0u;
                u.wb[i] = vb ? ld(pb + i * plane_bits + 8 * (size_t)p.pitch) : 0u;
                u.aa[i] = va ? ld(pa + i * plane_alpha) : 0.0f;
                u.ab[i] = vb ? ld(pa + i * plane_alpha + 8 * (size_t)p.G) : 0.0f;
            }
            if (++l_i == round_n) {
                l_i = 0;
                l_c = group_of(++l_st);
            }
        };
        PlaneWords<NQ> next, after;
        load(next);
        if (DEEP) load(after);
        for (int i = 0; i < round_n * NT; ++i) mine[i * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (first == 0) {
            for (int s = st0 + 1; (s - step0) * round_n < u1; ++s) {
                const int k = s * kDpStepK + (lane & 1) * 64;
                if ((lane >> 1) < p.n && k < p.d_in)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(p.X + (long long)(lane >> 1) * p.ldx + k));
            }
        }

        // a step's activations: lane (g, t) holds token g of each tile of eight, k 32 t .. + 31, paired as the
        // expansion pairs the weights: xb[nt][r][h] = (16 h + r, + 4), (+ 8, + 12)
        uint2 xb[NT][4][2];
        float f0[NT], f1[NT];
        auto load_x = [&](int st) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const int tok = nt * 8 + gr;
                const int kb = st * kDpStepK + tq * 32;
                const __nv_bfloat16* src = p.X + (long long)tok * p.ldx + kb;
                uint4 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    v[r] = make_uint4(0u, 0u, 0u, 0u);
                    if (tok < p.n && kb + r * 8 < p.d_in) v[r] = ld(reinterpret_cast<const uint4*>(src + r * 8));
                }
                const float inv = scale_fragment(v, kb, 8, p.d_in, st * kDpStepK + kDpStepK > p.d_in);
                const uint32_t P[16] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w,
                                        v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = 8 * h + (r >> 1);
                        const uint32_t sel = (r & 1) ? 0x7632u : 0x5410u;
                        xb[nt][r][h] = make_uint2(prmt(P[e], P[e + 2], sel), prmt(P[e + 4], P[e + 6], sel));
                    }
                f0[nt] = __shfl_sync(0xffffffffu, inv, 8 * tq);
                f1[nt] = __shfl_sync(0xffffffffu, inv, 8 * tq + 4);
            }
        };

        int u_st = st0, u_i = i0;
        bool fresh = true;
        auto row_shift = [&](const float (&a)[NQ]) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < NQ; ++i) s += fabsf(a[i]);
            uint32_t m = __float_as_uint(s);
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
            return shift_for(exponent_of_bits(m), 13);
        };
        auto unit = [&](const PlaneWords<NQ>& u) {
            const int sa = row_shift(u.aa), sb = row_shift(u.ab);
            RowExpand<NQ> ea, eb;
            ea.begin(u.wa, u.aa, pow2f(sa));
            eb.begin(u.wb, u.ab, pow2f(sb));
            float d[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                uint32_t Sa = 0u, Sb = 0u;
                if (NQ < 8) { Sa = ea.select(r); Sb = eb.select(r); }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t a0, a1, a2, a3;
                    ea.pairs(Sa, r, h, a0, a2);
                    eb.pairs(Sb, r, h, a1, a3);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) mma_f16(d[nt], a0, a1, a2, a3, xb[nt][r][h].x, xb[nt][r][h].y);
                }
            }
            const float ia = pow2f(-sa), ib = pow2f(-sb);
            float4* slot = mine + u_i * (NT * 32);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float4 s = slot[nt * 32];
                s.x = fmaf(f0[nt] * ia, d[nt][0], s.x);
                s.y = fmaf(f1[nt] * ia, d[nt][1], s.y);
                s.z = fmaf(f0[nt] * ib, d[nt][2], s.z);
                s.w = fmaf(f1[nt] * ib, d[nt][3], s.w);
                slot[nt * 32] = s;
            }
            fresh = (++u_i == round_n);
            if (fresh) { u_i = 0; ++u_st; }
        };
#pragma unroll 1
        for (int u = u0; u < u1; ++u) {
            if (fresh) load_x(u_st);
            if (DEEP) {
                unit(next);
                load(next);
                if (++u == u1) break;
                if (fresh) load_x(u_st);
                unit(after);
                load(after);
            } else if (NQ == 8) {  // one unit's registers are all there is room for
                unit(next);
                load(next);
            } else {
                const PlaneWords<NQ> now = next;
                load(next);
                unit(now);
            }
        }
        __syncthreads();
        add_and_store<NT, SPLIT>(p.o, sums, p.round, round_n, tile0 + first, nullptr, p.split);
        if (first + p.round < ntiles) __syncthreads();  // the slots are written again
    }
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------

// ceil(2^32 / g): k / g = hi32(k magic) while k g < 2^32, since k magic - k 2^32 / g < k; else 0
uint32_t group_magic(int d_in, int g) {
    return (long long)d_in * g < (1ll << 32) && g > 1 ? (uint32_t)(((1ull << 32) + g - 1) / g) : 0u;
}

// Row tiles dealt to one CTA per SM; bytes of the warps' sums (at most 192 KiB).  A matrix with few row tiles
// gives each to a cluster of 2, 4 or 8 CTAs that share its steps, as long as a CTA keeps a step for every
// warp (fewer: 2048 -> 256, q = 4, one token 4.6 us without a cluster, 5.5 in pairs) and the clusters find
// their places at once (on 148 SMs at most 65, 32 and 16 of them).  Measured, one CTA a tile, now, and the
// kernels with the columns dealt over all SMs that these replaced, 16 tokens:
//   planes, q = 4   16384 -> 512 32.4 / 12.0 / 18.8 us   16384 -> 128 32.0 / 8.0 / 18.3   4096 -> 512 10.4 / 7.7 / 17.2
//   planes, q = 6   16384 -> 512 61.6 / 19.1 / 32.3      32768 -> 32 113 / 18.3 / 27.7
//   packed, q = 4   16384 -> 512 20.1 / 9.2 / 26.3       65536 -> 16 70.5 / 12.6 / 63.7
template <int NT, typename Params>
size_t deal_tiles(Params& p, int tiles, int* ctas) {
    const int sms = sm_count();
    p.split = 1;
    while (p.split < 8 && p.steps >= 2 * kDpWarps * p.split && 2 * p.split * tiles <= sms - sms / 8) p.split *= 2;
    const int clusters = std::min(tiles, sms);
    *ctas = clusters * p.split;
    p.per = tiles / clusters;
    p.rem = tiles % clusters;
    p.round = std::min(p.per + (p.rem > 0 ? 1 : 0), kDpMaxRound / NT);
    return (size_t)kDpWarps * p.round * NT * 512;
}

template <int Q, int NT, int PARTS>
bcq_status launch_decode_packed(DecPackedParams p, int tiles, cudaStream_t s) {
    int ctas;
    size_t smem = deal_tiles<NT>(p, tiles, &ctas);
    const int steps = ceil_div(p.steps, p.split);  // of a CTA, at most
    p.x_stride = (uint32_t)steps * 256u + 64u;     // (64 bytes more: tokens next to each other in other banks)
    const size_t x_bytes = (size_t)p.n * (p.x_stride + steps * sizeof(float));
    // Activations by way of shared memory: for up to four tokens, where they fit.  With two tokens the CTA's conversion is an eighth
    // to a quarter of what its warps do otherwise; with four the CTA needs more than one step a warp for it to be less, with eight it
    // is as much, behind a barrier; four tables a step (PARTS = 4) leave no registers for it.  q = 4, without and with, us:
    //   4096 -> 4096   one token 6.12 / 5.84, two 6.18 / 5.99, four 6.22 / 6.17, eight 6.30 / 7.01
    //   16384 -> 4096, one token 19.0 / 15.6; 4096 -> 16384, one token 13.9 / 13.3; 2048 -> 2048, four tokens 3.27 / 3.38
    //   2048 -> 2048, g = 32, one token 3.60 / 4.11; 4096 -> 512, in clusters of two with 16 steps each, four tokens 4.34 / 4.45
    constexpr bool CAN = NT == 1 && PARTS <= 2;
    const bool xs = CAN && p.n <= (steps > kDpWarps ? 4 : 2) && smem + x_bytes <= kDpMaxSmem;
    if (xs) smem += x_bytes;
    void (*kern)(DecPackedParams) = p.split > 1 ? decode_packed_kernel<Q, NT, PARTS, true, false> : decode_packed_kernel<Q, NT, PARTS, false, false>;
    if constexpr (CAN)
        if (xs) kern = p.split > 1 ? decode_packed_kernel<Q, NT, PARTS, true, true> : decode_packed_kernel<Q, NT, PARTS, false, true>;
    const bcq_status st = ensure_dynamic_smem(kern, smem);
    if (st != BCQ_OK) return st;
    BCQ_CUDA_TRY(launch_pdl(kern, dim3((unsigned)ctas), kDpThreads, smem, s, (unsigned)p.split, p));
    return BCQ_OK;
}

template <int Q, int NT>
bcq_status launch_decode_parts(const DecPackedParams& p, const PackLayout& L, cudaStream_t s) {
    if (L.parts == 1) return launch_decode_packed<Q, NT, 1>(p, L.tiles, s);
    if (L.parts == 2) return launch_decode_packed<Q, NT, 2>(p, L.tiles, s);
    return launch_decode_packed<Q, NT, 4>(p, L.tiles, s);
}

template <int Q>
bcq_status launch_decode_tokens(const DecPackedParams& p, const PackLayout& L, cudaStream_t s) {
    return p.n <= 8 ? launch_decode_parts<Q, 1>(p, L, s) : launch_decode_parts<Q, 2>(p, L, s);
}

template <int NQ, int NT>
bcq_status launch_decode_planes(DecPlanesParams p, cudaStream_t s) {
    int ctas;
    const size_t smem = deal_tiles<NT>(p, ceil_div(p.d_out, kDpRows), &ctas);
    void (*kern)(DecPlanesParams) = p.split > 1 ? decode_planes_kernel<NQ, NT, true, false> : decode_planes_kernel<NQ, NT, false, false>;
    // Two units ahead (DEEP) where a warp has few units and the start of its loads counts for more than a loop that is there
    // once.  us, one ahead / two ahead, one token; in front: units of a CTA, to be dealt to its 16 warps:
    //   q = 3   6   768 -> 768 2.78 / 2.67      16   2048 -> 2048 3.80 / 3.62   20  1280 -> 5120 5.46 / 5.04   39  1600 -> 4800 6.07 / 5.70
    //           50  6400 -> 1600 8.88 / 8.54    64   4096 -> 4096 8.74 / 8.73   256 16384 -> 4096 27.8 / 28.6
    // With nine tokens and more one ahead is the faster (1024 -> 1024, 16 tokens 4.38 / 4.72).  q = 4 is left alone: two ahead
    // gains where the units do not divide evenly among the warps (33  1408 -> 6400 6.92 / 6.63) and loses where they do (32  2048 -> 4096
    // 6.50 / 6.97), and a layer whose linears then take turns in two kernels fetches the code of both (the four linears of width
    // 1600, four tokens 30.4 us, with a rule of that kind 30.7).
    if constexpr (NQ == 3 && NT == 1)
        if (p.round * ceil_div(p.steps, p.split) < 4 * kDpWarps)
            kern = p.split > 1 ? decode_planes_kernel<NQ, NT, true, true> : decode_planes_kernel<NQ, NT, false, true>;
    const bcq_status st = ensure_dynamic_smem(kern, smem);
    if (st != BCQ_OK) return st;
    BCQ_CUDA_TRY(launch_pdl(kern, dim3((unsigned)ctas), kDpThreads, smem, s, (unsigned)p.split, p));
    return BCQ_OK;
}

template <int NQ>
bcq_status launch_decode_planes_tokens(const DecPlanesParams& p, cudaStream_t s) {
    return p.n <= 8 ? launch_decode_planes<NQ, 1>(p, s) : launch_decode_planes<NQ, 2>(p, s);
}

bcq_status check_pack_shape(int d_out, int d_in, int q, int g) {
    bcq_status st = check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (q > 4) return BCQ_ERR_UNSUPPORTED;
    return BCQ_OK;
}

template <int Q>
void launch_pack_codes(int d_out, int pitch, const PackLayout& L, const uint32_t* bits, uint32_t* codes, cudaStream_t s) {
    const long long threads = (long long)L.tiles * L.steps * 32;
    pack_codes_kernel<Q><<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(d_out, pitch, L.tiles, L.steps, bits, codes);
}

}  // namespace

namespace bcq {
bcq_status run_decode_planes(int d_out, int d_in, int q, int g, int n, const void* X, size_t ldx, const uint32_t* bits,
                             const float* alpha, const float* bias, void* Y, size_t ldy, int y_dtype, cudaStream_t s) {
    DecPlanesParams p = {};
    p.d_out = d_out; p.d_in = d_in; p.q = q; p.g = g; p.G = (int)bcq_num_groups(d_in, g); p.n = n;
    p.steps = ceil_div(d_in, kDpStepK); p.pitch = (int)bcq_pitch_words(d_in);
    p.g_magic = group_magic(d_in, g);
    p.X = reinterpret_cast<const __nv_bfloat16*>(X); p.ldx = (long long)ldx;
    p.bits = bits; p.alpha = alpha;
    p.o = {d_out, n, bias, Y, (long long)ldy, y_dtype == BCQ_BF16};
    if (q <= 3) return launch_decode_planes_tokens<3>(p, s);
    if (q == 4) return launch_decode_planes_tokens<4>(p, s);
    return launch_decode_planes_tokens<8>(p, s);
}
}  // namespace bcq

extern "C" size_t bcq_decode_pack_bytes(int d_out, int d_in, int q, int g) {
    if (check_pack_shape(d_out, d_in, q, g) != BCQ_OK) return 0;
    return pack_layout(d_out, d_in, q, g).total;
}

extern "C" bcq_status bcq_decode_pack(int d_out, int d_in, int q, int g, const uint32_t* bits,
                                      const float* alpha, void* pack, size_t pack_bytes, void* stream) {
    bcq_status st = check_pack_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (!bits || !alpha || !pack) return BCQ_ERR_NULL;
    if (!aligned16(bits) || (reinterpret_cast<uintptr_t>(pack) & 127u) != 0) return BCQ_ERR_ALIGN;
    const PackLayout L = pack_layout(d_out, d_in, q, g);
    if (pack_bytes < L.total) return BCQ_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* pk = reinterpret_cast<uint8_t*>(pack);
    float* rinv = reinterpret_cast<float*>(pk);
    const int rows_padded = L.tiles * kDpRows;
    pack_rowscale_kernel<<<ceil_div(rows_padded, 128), 128, 0, s>>>(d_out, q, L.G, rows_padded, alpha, rinv);
    bcq::count_launch();
    BCQ_CUDA_TRY(cudaGetLastError());
    const long long nt = (long long)L.tiles * L.G * kDpRows;
    pack_tables_kernel<<<(unsigned)((nt + 255) / 256), 256, 0, s>>>(d_out, q, L.G, nt, alpha, rinv,
                                                                   reinterpret_cast<uint4*>(pk + L.off_tables));
    bcq::count_launch();
    BCQ_CUDA_TRY(cudaGetLastError());
    const int pitch = (int)bcq_pitch_words(d_in);
    uint32_t* codes = reinterpret_cast<uint32_t*>(pk + L.off_codes);
    switch (q) {
        case 1: launch_pack_codes<1>(d_out, pitch, L, bits, codes, s); break;
        case 2: launch_pack_codes<2>(d_out, pitch, L, bits, codes, s); break;
        case 3: launch_pack_codes<3>(d_out, pitch, L, bits, codes, s); break;
        default: launch_pack_codes<4>(d_out, pitch, L, bits, codes, s); break;
    }
    bcq::count_launch();
    BCQ_CUDA_TRY(cudaGetLastError());
    return BCQ_OK;
}

extern "C" bcq_status bcq_linear_decode_packed(int d_out, int d_in, int q, int g, int n, const void* X,
                                               size_t ldx, void* pack, const float* bias, void* Y, size_t ldy,
                                               int y_dtype, void* /*ws*/, size_t /*ws_bytes*/, void* stream) {
    bcq_status st = check_pack_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1 || n > 16) return BCQ_ERR_SHAPE;
    if (!pack || !Y) return BCQ_ERR_NULL;
    if ((st = check_act(X, ldx, d_in)) != BCQ_OK) return st;
    if (ldy < (size_t)d_out) return BCQ_ERR_SHAPE;
    if (y_dtype != BCQ_F32 && y_dtype != BCQ_BF16) return BCQ_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(pack) & 127u) != 0) return BCQ_ERR_ALIGN;
    const PackLayout L = pack_layout(d_out, d_in, q, g);
    const uint8_t* pk = reinterpret_cast<const uint8_t*>(pack);
    DecPackedParams p = {};
    p.d_out = d_out; p.d_in = d_in; p.g = g; p.G = L.G; p.n = n;
    p.steps = L.steps;
    p.g_magic = group_magic(d_in, g);
    p.X = reinterpret_cast<const __nv_bfloat16*>(X); p.ldx = (long long)ldx;
    p.codes = pk + L.off_codes; p.tables = pk + L.off_tables;
    p.rinv = reinterpret_cast<const float*>(pk);
    p.o = {d_out, n, bias, Y, (long long)ldy, y_dtype == BCQ_BF16};
    cudaStream_t s = (cudaStream_t)stream;
    switch (q) {
        case 1: return launch_decode_tokens<1>(p, L, s);
        case 2: return launch_decode_tokens<2>(p, L, s);
        case 3: return launch_decode_tokens<3>(p, L, s);
        default: return launch_decode_tokens<4>(p, L, s);
    }
}
