// BCQ post-training quantizer (greedy and alternating) and the dequantize helper.
//
// One "team" of threads owns one (row, group) problem and keeps its weights in registers.
//
// team_quantize_kernel (greedy for every q, alternating for q <= 4): a thread holds up to 32 weights, so
// a group of 128 is four lanes and a warp works on eight groups (greedy; alternating takes 8 or 16
// lanes, see launch_team_size); a team is up to a warp for g <= 1024 (two warps for short alternating
// problems) and a whole CTA above that.  Four lanes share 128 consecutive weights, lane l taking the 16-byte
// pieces l, l + 4, ...: full 32-byte sectors from memory, and the four lanes' sign bits make four
// container words with one 4 x 4 byte transpose.  With a warp per group (four weights a lane), as
// this kernel worked before, a plane of 128 weights cost five rounds of 64-bit shuffles and a
// ballot per 32 weights; now two rounds, and per weight and plane two fp64 additions and one shift
// that collects the sign.  Measured, before and after: greedy q = 4, g = 128, the four linears of a
// layer of width 1600 (30.7 M weights) 162 -> 59 us (2.5 TB/s; the logic pipe is 55 % busy, the fp64
// pipe 21 %); five alternating rounds, q = 3, g = 128, 5120 x 5120: 1119 -> 360 us (instruction fetch of
// the unrolled rounds and fp64 latency at five warps per scheduler bound it).
//
// Sums are fp64 and are reduced in a fixed order, so a result never depends on scheduling.
//
// quantize_kernel (alternating, q > 4): one warp per group up to 1024 weights, a CTA above.
//
// Appendix "Details on BCQ Format": Eq. ap:1-ap:3 (greedy), Eq. ap:4 and the following
// paragraph (alternating).
#include "common.h"

namespace {

struct QuantParams {
    int d_out, d_in, q, g, G, alt_iters;
    long long ldw;
    int pitch;
    const float* W;
    uint32_t* bits;
    float* alpha;
    double* sq_err;
    long long items;  // d_out * G
    int vec;          // rows and groups start on 16-byte boundaries
    double inv_g;     // 1 / g where that is exact (a power of two), else 0
    uint32_t g_magic; // where not 0: row of an item = hi32(item * g_magic) >> g_shift
    uint32_t g_shift;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the team.  TW == 1: the warp.  TW > 1: the CTA (all threads must call).
template <int TW>
__device__ __forceinline__ double team_sum(double v, double* scratch) {
    v = warp_sum(v);
    if (TW == 1) return v;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll 1
    for (int w = 0; w < TW; ++w) t += scratch[w];
    return t;
}

// Sum of small non-negative counts over the team, as a double.  A warp adds them with one
// integer reduction (exact, like the fp64 tree: the values are integers far below 2^53).
template <int TW>
__device__ __forceinline__ double team_count(int v, double* scratch) {
    if (TW == 1) return (double)__reduce_add_sync(0xffffffffu, v);
    return team_sum<TW>((double)v, scratch);
}

template <int TW>
__device__ __forceinline__ void team_sync() {
    if (TW == 1)
        __syncwarp();
    else
        __syncthreads();
}

// Least-squares scales for fixed signs (Eq. ap:4): solve (B^T B) x = B^T w by Gaussian
// elimination with partial pivoting.  Every thread of the team runs the same arithmetic on the
// same numbers.  Products and differences are rounded separately (no fused multiply-add).
// Returns false (alpha untouched) when a pivot is below 1e-12 * m.
__device__ bool solve_ls(int q, double m, double (*A)[BCQ_MAX_Q + 1], float* alpha) {
    const double tiny = 1e-12 * m;
    for (int col = 0; col < q; ++col) {
        int piv = col;
        for (int r = col + 1; r < q; ++r)
            if (fabs(A[r][col]) > fabs(A[piv][col])) piv = r;
        if (fabs(A[piv][col]) < tiny) return false;
        if (piv != col)
            for (int l = 0; l <= q; ++l) {
                double tmp = A[col][l];
                A[col][l] = A[piv][l];
                A[piv][l] = tmp;
            }
        for (int r = col + 1; r < q; ++r) {
            const double f = __ddiv_rn(A[r][col], A[col][col]);
            for (int l = col; l <= q; ++l) A[r][l] = __dsub_rn(A[r][l], __dmul_rn(f, A[col][l]));
        }
    }
    double x[BCQ_MAX_Q];
    for (int r = q - 1; r >= 0; --r) {
        double s = A[r][q];
        for (int l = r + 1; l < q; ++l) s = __dsub_rn(s, __dmul_rn(A[r][l], x[l]));
        x[r] = __ddiv_rn(s, A[r][r]);
    }
    for (int i = 0; i < q; ++i) alpha[i] = (float)x[i];
    return true;
}

// The same elimination for a plane count known at compile time: every index is static, so the
// matrix stays in registers (the pivot row is found by value and swapped in by predicated moves).
// Same operations in the same order as solve_ls, hence the same result.
template <int Q>
__device__ __forceinline__ bool solve_ls_static(double m, double (&A)[Q][Q + 1], float (&alpha)[Q]) {
    const double tiny = 1e-12 * m;
#pragma unroll
    for (int col = 0; col < Q; ++col) {
        int piv = col;
        double best = fabs(A[col][col]);
#pragma unroll
        for (int r = col + 1; r < Q; ++r) {
            const double v = fabs(A[r][col]);
            if (v > best) { best = v; piv = r; }
        }
        if (best < tiny) return false;
#pragma unroll
        for (int r = col + 1; r < Q; ++r) {
            if (r == piv) {
#pragma unroll
                for (int l = 0; l <= Q; ++l) {
                    const double tmp = A[col][l];
                    A[col][l] = A[r][l];
                    A[r][l] = tmp;
                }
            }
        }
#pragma unroll
        for (int r = col + 1; r < Q; ++r) {
            const double f = __ddiv_rn(A[r][col], A[col][col]);
#pragma unroll
            for (int l = col; l <= Q; ++l) A[r][l] = __dsub_rn(A[r][l], __dmul_rn(f, A[col][l]));
        }
    }
    double x[Q];
#pragma unroll
    for (int r = Q - 1; r >= 0; --r) {
        double s = A[r][Q];
#pragma unroll
        for (int l = r + 1; l < Q; ++l) s = __dsub_rn(s, __dmul_rn(A[r][l], x[l]));
        x[r] = __ddiv_rn(s, A[r][r]);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) alpha[i] = (float)x[i];
    return true;
}

// Alternating method for any number of planes.
template <int EPT, int TW>
__global__ void __launch_bounds__(TW == 1 ? 128 : TW * 32)
quantize_kernel(const QuantParams p) {
    const int q = p.q;
    constexpr int NT = TW * 32;
    constexpr int TEAMS = (TW == 1) ? 4 : 1;
    __shared__ double red_scratch[32];
    bcq::pdl_wait();  // (and no pdl_trigger, see launch_pdl)
    __shared__ double level_smem[TEAMS][1 << BCQ_MAX_Q];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int team = (TW == 1) ? warp : 0;
    const int tid = (TW == 1) ? lane : (int)threadIdx.x;  // index inside the team
    const int twarp = (TW == 1) ? 0 : warp;               // warp index inside the team
    double* levels = level_smem[team];

    const long long first = (long long)blockIdx.x * TEAMS + team;
    const long long stride = (long long)gridDim.x * TEAMS;
    // TW > 1 uses __syncthreads(): every team of the CTA is the CTA, so the trip count is uniform.
    for (long long item = first; item < p.items; item += stride) {
        const int j = (int)(item / p.G);
        const int c = (int)(item - (long long)j * p.G);
        const int k0 = c * p.g;
        const int m = min(p.g, p.d_in - k0);
        const double md = (double)m;
        const bool m_pow2 = (m & (m - 1)) == 0;
        const double inv_m = 1.0 / md;

        double r[EPT];
        float w[EPT];
        uint32_t code[EPT];
        const float* wrow = p.W + (long long)j * p.ldw + k0;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int kl = e * NT + tid;
            const float v = (kl < m) ? bcq::ld(wrow + kl) : 0.0f;
            r[e] = (double)v;
            w[e] = v;
            code[e] = 0u;
        }

        float a[BCQ_MAX_Q];
        // ---- greedy planes
        for (int i = 0; i < q; ++i) {
            double local = 0.0;
#pragma unroll
            for (int e = 0; e < EPT; ++e)
                if (e * NT + tid < m) local += fabs(r[e]);
            const double S = team_sum<TW>(local, red_scratch);
            // a power-of-two group size divides exactly by multiplying with its reciprocal
            a[i] = (float)(m_pow2 ? __dmul_rn(S, inv_m) : __ddiv_rn(S, md));
            const double ad = (double)a[i];
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                const bool pos = r[e] >= 0.0;
                if (e * NT + tid < m) r[e] = pos ? r[e] - ad : r[e] + ad;
                if (pos) code[e] |= (1u << i);
            }
        }

        {
            const int ncodes = 1 << q;
            for (int it = 0; it <= p.alt_iters; ++it) {
                // ---- least-squares alpha for the current signs
                double A[BCQ_MAX_Q][BCQ_MAX_Q + 1];
                for (int i = 0; i < q; ++i) {
                    double local = 0.0;
#pragma unroll
                    for (int e = 0; e < EPT; ++e)
                        if (e * NT + tid < m) local += ((code[e] >> i) & 1u) ? (double)w[e] : -(double)w[e];
                    A[i][q] = team_sum<TW>(local, red_scratch);
                    A[i][i] = md;
                    for (int l = i + 1; l < q; ++l) {
                        int cnt = 0;
#pragma unroll
                        for (int e = 0; e < EPT; ++e)
                            if (e * NT + tid < m) cnt += (int)(((code[e] >> i) ^ (code[e] >> l)) & 1u);
                        const double mism = team_count<TW>(cnt, red_scratch);
                        A[i][l] = md - 2.0 * mism;
                        A[l][i] = A[i][l];
                    }
                }
                solve_ls(q, md, A, a);
                if (it == p.alt_iters) break;  // the last pass is the final refit only
                // ---- every weight moves to the nearest level; largest code wins ties
                team_sync<TW>();
                for (int s = tid; s < ncodes; s += NT) {
                    double L = 0.0;
                    for (int i = 0; i < q; ++i) L = ((s >> i) & 1) ? L + (double)a[i] : L - (double)a[i];
                    levels[s] = L;
                }
                team_sync<TW>();
#pragma unroll
                for (int e = 0; e < EPT; ++e) {
                    const double wv = (double)w[e];
                    int best = ncodes - 1;
                    double dbest = fabs(wv - levels[best]);
#pragma unroll 1
                    for (int s = ncodes - 2; s >= 0; --s) {
                        const double d = fabs(wv - levels[s]);
                        if (d < dbest) {
                            dbest = d;
                            best = s;
                        }
                    }
                    code[e] = (uint32_t)best;
                }
            }
            // ---- write the planes
            for (int i = 0; i < q; ++i) {
                uint32_t* brow = p.bits + ((long long)i * p.d_out + j) * p.pitch + (k0 >> 5);
#pragma unroll
                for (int e = 0; e < EPT; ++e) {
                    const bool valid = (e * NT + tid) < m;
                    const uint32_t word = __ballot_sync(0xffffffffu, valid && ((code[e] >> i) & 1u));
                    if (lane == 0 && (e * NT + twarp * 32) < m) brow[e * TW + twarp] = word;
                }
            }
        }

        // ---- scales, zero padding words of the row, optional squared error
        if (tid < q) p.alpha[((long long)tid * p.d_out + j) * p.G + c] = a[tid];
        if (c == p.G - 1) {
            const int first_pad = (p.d_in + 31) >> 5;
            const int npad = p.pitch - first_pad;  // 0..3
            for (int t = tid; t < npad * q; t += NT) {
                const int i = t / npad, wdx = t - i * npad;
                p.bits[((long long)i * p.d_out + j) * p.pitch + first_pad + wdx] = 0u;
            }
        }
        if (p.sq_err != nullptr) {
            double local = 0.0;
#pragma unroll
            for (int e = 0; e < EPT; ++e)
                if (e * NT + tid < m) {
                    double wh = 0.0;
                    for (int i = 0; i < q; ++i)
                        wh = ((code[e] >> i) & 1u) ? wh + (double)a[i] : wh - (double)a[i];
                    const double d = (double)w[e] - wh;
                    local += d * d;
                }
            const double E = team_sum<TW>(local, red_scratch);
            if (tid == 0) p.sq_err[(long long)j * p.G + c] = E;
        }
    }
}

// ------------------------------------------------------------------------------------------
// the team kernel
// ------------------------------------------------------------------------------------------

// A sum over a group is a tree whose shape depends on the group size alone, so a row gets the same scales whichever
// team takes it, and hence whatever else is in the call.  Where a group may be taken by teams of different
// size (alternating, up to 2048 weights) its leaves are two neighbouring 16-byte pieces of one lane of a
// quad, 8 weights.  Over them, neighbours first: the leaves of a lane (tree_of_leaves), the quads of a
// warp, the warps; the four lanes of a quad come last.
template <int N>
__device__ __forceinline__ double tree_of_leaves(const double (&p)[N]) {
    static_assert(N == 1 || N == 2 || N == 4, "leaves of a thread");
    if constexpr (N == 1) return p[0];
    else if constexpr (N == 2) return p[0] + p[1];
    else return (p[0] + p[1]) + (p[2] + p[3]);
}

// A value of each warp, uniform in the warp: added over the CTA, in order.
template <int TW>
__device__ __forceinline__ double warps_sum(double v, double* scratch) {
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll 1
    for (int w = 0; w < TW; ++w) t += scratch[w];
    return t;
}

// Sum over a team of L lanes (TW = 1) or TW warps of the lanes' leaves.
template <int L, int TW>
__device__ __forceinline__ double lanes_sum(double v, double* scratch) {
#pragma unroll
    for (int o = 4; o < L; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if constexpr (TW == 2 || TW == 4) {
        __syncthreads();
        if ((threadIdx.x & 31) < 4) scratch[(threadIdx.x >> 5) * 4 + (threadIdx.x & 3)] = v;
        __syncthreads();
        double t[4];
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            t[l] = scratch[l] + scratch[4 + l];
            if (TW == 4) t[l] += scratch[8 + l] + scratch[12 + l];
        }
        return (t[0] + t[1]) + (t[2] + t[3]);
    } else {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if constexpr (TW == 1) return v;
        else return warps_sum<TW>(v, scratch);
    }
}

// Four lanes hold the bits of 128 consecutive weights: bit 4 i + e of a lane's word is weight
// 16 i + 4 l + e.  Returns container word l (weights 32 l .. 32 l + 31) to lane l.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t v) {
    const uint32_t l = threadIdx.x & 3u;
    uint32_t o = __shfl_xor_sync(0xffffffffu, v, 1);
    v = (l & 1u) ? __byte_perm(v, o, 0x3715u) : __byte_perm(v, o, 0x6240u);
    o = __shfl_xor_sync(0xffffffffu, v, 2);
    v = (l & 2u) ? __byte_perm(v, o, 0x3276u) : __byte_perm(v, o, 0x5410u);
    // byte l' = (low nibble: weights 4 l' .. + 3, high nibble: weights 16 + 4 l' .. + 3)
    uint32_t lo = v & 0x0F0F0F0Fu, hi = (v >> 4) & 0x0F0F0F0Fu;
    lo |= lo >> 4;
    hi |= hi >> 4;
    return __byte_perm(lo, hi, 0x6420u);
}

// (value, code) pairs into ascending order of the values.
template <int N>
__device__ __forceinline__ void sort_levels(double (&L)[N], uint32_t (&c)[N]) {
    auto ce = [&](int x, int y) {
        if (L[y] < L[x]) {
            const double t = L[x]; L[x] = L[y]; L[y] = t;
            const uint32_t u = c[x]; c[x] = c[y]; c[y] = u;
        }
    };
    if constexpr (N == 2) ce(0, 1);
    if constexpr (N == 4) { ce(0, 1); ce(2, 3); ce(0, 2); ce(1, 3); ce(1, 2); }
    if constexpr (N == 8) {
        ce(0, 1); ce(2, 3); ce(4, 5); ce(6, 7);
        ce(0, 2); ce(1, 3); ce(4, 6); ce(5, 7);
        ce(1, 2); ce(5, 6); ce(0, 4); ce(3, 7);
        ce(1, 5); ce(2, 6);
        ce(1, 4); ce(3, 6);
        ce(2, 4); ce(3, 5);
        ce(3, 4);
    }
}

// Nearest of the 2^Q levels, the largest code among equidistant ones: the definition.
template <int Q>
__device__ __noinline__ uint32_t nearest_code(double w, const float (&a)[Q]) {
    uint32_t best = 0u;
    double dbest = 0.0;
#pragma unroll 1
    for (int s = (1 << Q) - 1; s >= 0; --s) {
        double L = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) L = ((s >> i) & 1) ? L + (double)a[i] : L - (double)a[i];
        const double d = fabs(w - L);
        if (s == (1 << Q) - 1 || d < dbest) {
            dbest = d;
            best = (uint32_t)s;
        }
    }
    return best;
}

// What a round of the alternating method needs to know about the levels of a group.  They come in
// pairs +-L, so only the positive ones are kept: sorted, as fp32 midpoints, with the code of each
// (bit i set where plane i is -1) in a nibble of `codes`.  A magnitude finds its level in Q - 1
// comparisons instead of 2^Q fp64 distances.
template <int Q>
struct LevelSearch {
    static constexpr int N = 1 << (Q - 1);
    float mid[N];     // mid[k], k >= 1: between level k - 1 and level k
    uint32_t codes;
    float delta;      // a weight closer than this to a midpoint (or to 0) is decided by nearest_code

    // amax: at least the group's largest magnitude
    __device__ __forceinline__ void build(const float (&a)[Q], float amax) {
        double L[N];
        uint32_t c[N];
#pragma unroll
        for (int s = 0; s < N; ++s) {
            double v = 0.0;
#pragma unroll
            for (int i = 0; i < Q; ++i) v = (i == Q - 1 || ((s >> i) & 1)) ? v + (double)a[i] : v - (double)a[i];
            const uint32_t neg = ~((uint32_t)s | (1u << (Q - 1))) & ((1u << Q) - 1u);
            const bool flip = v < 0.0;
            L[s] = flip ? -v : v;
            c[s] = flip ? neg ^ ((1u << Q) - 1u) : neg;
        }
        sort_levels<N>(L, c);
        codes = 0u;
        double gap = 2.0 * L[0];
        mid[0] = 0.f;
#pragma unroll
        for (int s = 0; s < N; ++s) {
            codes |= c[s] << (4 * s);
            if (s > 0) {
                gap = fmin(gap, L[s] - L[s - 1]);
                mid[s] = (float)(0.5 * (L[s] + L[s - 1]));
            }
        }
        // fp32 decides exactly as the fp64 distances do when the weight is 2^-21 of the largest level
        // away from every midpoint: the midpoint is rounded by 2^-24 of itself, the distances by
        // 2^-53 of the weight.  Levels (almost) on top of each other, or far below the weights, are
        // left to the definition: delta then covers everything.
        const float top = (float)L[N - 1];
        delta = (gap > 9.6e-7 * fmax((double)top, (double)amax * 2.5e-4)) ? top * 4.8e-7f : __int_as_float(0x7F800000);
        if (!(top < 3.0e38f)) delta = __int_as_float(0x7F800000);
    }
    // the code (as in `codes`) of magnitude x in the low Q bits of the result; near = min(near, distances)
    __device__ __forceinline__ uint32_t find(float x, float& near) const {
        if constexpr (Q == 1) return codes;
        float d = x - mid[N / 2];
        near = fminf(near, fabsf(d));
        bool p0 = d >= 0.f;
        if constexpr (Q == 2) return p0 ? codes >> 4 : codes;
        if constexpr (Q == 3) {
            d = x - (p0 ? mid[3] : mid[1]);
            near = fminf(near, fabsf(d));
            const uint32_t h = p0 ? codes >> 8 : codes;
            return d >= 0.f ? h >> 4 : h;
        }
        if constexpr (Q == 4) {
            const float lo = p0 ? mid[5] : mid[1], hi = p0 ? mid[7] : mid[3];
            d = x - (p0 ? mid[6] : mid[2]);
            near = fminf(near, fabsf(d));
            const bool p1 = d >= 0.f;
            d = x - (p1 ? hi : lo);
            near = fminf(near, fabsf(d));
            uint32_t h = p0 ? codes >> 16 : codes;
            h = p1 ? h >> 8 : h;
            return d >= 0.f ? h >> 4 : h;
        }
    }
};

// Groups with an infinite or NaN weight.  The team kernel keeps residuals as magnitudes and signs, and the sign of a
// NaN says nothing: r >= 0 is false for it.  The first scale a1 of such a group is infinite or NaN, so the
// residuals of the second plane are w -+ a1 and everything after it is NaN.
__device__ __forceinline__ bool greedy_sign_not_finite(float w, float a1, int plane) {
    if (plane == 0) return w >= 0.f;
    return plane == 1 && (w >= 0.f ? (double)w - (double)a1 : (double)w + (double)a1) >= 0.0;
}

// First scale of a group: the mean of |w|.
__device__ __noinline__ float first_scale(const float* w, int m) {
    double S = 0.0;
#pragma unroll 1
    for (int k = 0; k < m; ++k) S += fabs((double)bcq::ld(w + k));
    return (float)__ddiv_rn(S, (double)m);
}

// Container word `wi` of such a group in the greedy planes.
__device__ __noinline__ void greedy_word_not_finite(const QuantParams p, long long item, int wi) {
    const int j = (int)(item / p.G), k0 = (int)(item % p.G) * p.g + 32 * wi, m = min(min(p.g - 32 * wi, p.d_in - k0), 32);
    if (m <= 0) return;
    const float* w = p.W + (long long)j * p.ldw + k0;
    const float a1 = first_scale(w - 32 * wi, min(p.g, p.d_in - k0 + 32 * wi));
#pragma unroll 1
    for (int i = 0; i < p.q; ++i) {
        uint32_t word = 0u;
#pragma unroll 1
        for (int e = 0; e < m; ++e)
            if (greedy_sign_not_finite(bcq::ld(w + e), a1, i)) word |= 1u << e;
        p.bits[((long long)i * p.d_out + j) * p.pitch + (k0 >> 5)] = word;
    }
}

// The scales (and the squared error) of such a group after alternating rounds, by the definition.  The right-hand
// sides of a fit are not finite, so no level is nearer than another: after the first round every weight
// has the largest code, and for q > 1 the fit is singular from then on.
__device__ __noinline__ void fit_not_finite(const QuantParams p, long long item) {
    const int j = (int)(item / p.G), k0 = (int)(item % p.G) * p.g, m = min(p.g, p.d_in - k0), q = p.q;
    const float* w = p.W + (long long)j * p.ldw + k0;
    const float a1 = first_scale(w, m);
    if (fabsf(a1) <= 3.402823466e38f) return;  // finite weights, a scale that a fit took out of range
    double A[BCQ_MAX_Q][BCQ_MAX_Q + 1], plain = 0.0;
    float a[BCQ_MAX_Q];
    a[0] = a1;
#pragma unroll 1
    for (int i = 1; i < q; ++i) a[i] = __int_as_float(0x7FFFFFFF);
#pragma unroll 1
    for (int i = 0; i < q; ++i) {
        A[i][q] = 0.0;
#pragma unroll 1
        for (int l = 0; l < q; ++l) A[i][l] = (double)m;
    }
#pragma unroll 1
    for (int k = 0; k < m; ++k) {
        const float x = bcq::ld(w + k);
        plain += (double)x;
#pragma unroll 1
        for (int i = 0; i < q; ++i) {
            const bool pos = greedy_sign_not_finite(x, a1, i);
            A[i][q] += pos ? (double)x : -(double)x;
#pragma unroll 1
            for (int l = 0; l < q; ++l) A[i][l] -= pos != greedy_sign_not_finite(x, a1, l) ? 2.0 : 0.0;
        }
    }
    solve_ls(q, (double)m, A, a);
    if (q == 1) a[0] = (float)__ddiv_rn(plain, (double)m);
#pragma unroll 1
    for (int i = 0; i < q; ++i) p.alpha[i * p.items + item] = a[i];
    if (p.sq_err != nullptr) {
        double E = 0.0, wh = 0.0;
#pragma unroll 1
        for (int i = 0; i < q; ++i) wh += (double)a[i];
#pragma unroll 1
        for (int k = 0; k < m; ++k) {
            const double d = (double)bcq::ld(w + k) - wh;
            E += d * d;
        }
        p.sq_err[item] = E;
    }
}

// Q = 0: greedy, p.q planes; Q > 0: alternating with Q planes.  A thread holds 4 NI weights, a team is L
// lanes (TW = 1) or TW warps.
template <int NI, int L, int TW, int Q>
__global__ void __launch_bounds__(TW == 1 ? 128 : TW * 32,
                                  TW == 1   ? (NI == 2 || (Q == 0 && NI == 4) ? 6 : Q == 0 || NI == 4 ? 5 : 3)
                                  : TW <= 4 ? (NI == 4 ? 20 : 12) / TW
                                            : 1)
team_quantize_kernel(const QuantParams p) {
    constexpr bool ALT = Q > 0;
    constexpr int EPT = 4 * NI;
    constexpr int NT = L * TW;                       // threads of a team
    constexpr int LEAVES = !ALT || (NI == 8 && TW >= 4) ? 1 : NI / 2;  // see lanes_sum
    constexpr int LEAF = EPT / LEAVES;
    constexpr int TEAMS = TW == 1 ? 128 / L : 1;     // per CTA
    __shared__ double scratch[TW == 1 ? 1 : 32];
    bcq::pdl_trigger();
    bcq::pdl_wait();
    const int tl = TW == 1 ? (int)(threadIdx.x & (L - 1)) : (int)threadIdx.x;
    const long long item0 = (long long)blockIdx.x * TEAMS + (TW == 1 ? threadIdx.x / L : 0);
    // teams past the last item repeat it (the shuffles need every lane) and store nothing
    const bool live = item0 < p.items;
    const long long item = live ? item0 : p.items - 1;
    int j, c;
    if (p.g_magic != 0u) {
        j = (int)(__umulhi((uint32_t)item, p.g_magic) >> p.g_shift);
        c = (int)((uint32_t)item - (uint32_t)j * (uint32_t)p.G);
    } else {
        j = (int)(item / p.G);
        c = (int)(item - (long long)j * p.G);
    }
    const int k0 = c * p.g;
    const int m = min(p.g, p.d_in - k0);
    const double md = (double)m;
    const int kt = (tl >> 2) * (16 * NI) + (tl & 3) * 4;  // first weight of the thread; piece i is 16 i further

    // ---- load; bit t of `valid`: the thread's t-th weight exists
    const float* src = p.W + (long long)j * p.ldw + k0 + kt;
    float w[EPT];
    constexpr uint32_t kAll = EPT == 32 ? 0xFFFFFFFFu : (1u << (EPT & 31)) - 1u;
    uint32_t valid = kAll;
    int pieces = NI;       // 16-byte pieces that hold weights
    bool partial = false;  // the last of them is not full
    double inv_m = p.inv_g;
    if (m == EPT * NT && p.vec) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float4 v = bcq::ld(reinterpret_cast<const float4*>(src + 16 * i));
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
        }
    } else {
        valid = 0u;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int left = m - (kt + 16 * i);
            if (p.vec && left >= 4) {
                const float4 v = bcq::ld(reinterpret_cast<const float4*>(src + 16 * i));
                w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) w[4 * i + e] = (e < left) ? bcq::ld(src + 16 * i + e) : 0.0f;
            }
            valid |= (left >= 4 ? 0xFu : left > 0 ? (1u << left) - 1u : 0u) << (4 * i);
        }
        pieces = min(NI, max(0, (m - kt + 15) >> 4));
        partial = pieces > 0 && m - (kt + 16 * (pieces - 1)) < 4;
        inv_m = (m & (m - 1)) == 0 ? 1.0 / md : 0.0;
    }

    // ---- greedy planes.  A residual is kept as a magnitude |t| and a sign bit in `negs`: taking a off in
    // the direction of its sign leaves |t| - a with the sign kept, or a - |t| with the sign turned.
    // t = a - |t| is one addition, and the collected sign bits of all t turn `negs` at once.
    // Weights that do not exist are zeros throughout.  (-0.0 as an input counts as positive.)
    double t[EPT];
    uint32_t negs = 0u;
#pragma unroll
    for (int e = EPT - 1; e >= 0; --e) {
        w[e] += 0.0f;
        negs = __funnelshift_l(__float_as_uint(w[e]), negs, 1);
        t[e] = (double)w[e];
    }
    const int q = ALT ? Q : p.q;
    constexpr int QN = ALT ? Q : 1;
    float a[QN];
    uint32_t neg[QN];  // bit t: plane i of the thread's t-th weight is -1
    const int wi = (tl >> 2) * (NI / 2) + (tl & 3);           // container word of the group this thread writes
    const bool writes = live && (tl & 3) < NI / 2 && 32 * wi < m;
    const uint32_t word_mask = m - 32 * wi >= 32 ? 0xFFFFFFFFu : (1u << ((m - 32 * wi) & 31)) - 1u;
    uint32_t* dst = p.bits + (long long)j * p.pitch + (k0 >> 5) + wi;
    const long long plane_words = (long long)p.d_out * p.pitch, plane_alpha = (long long)p.d_out * p.G;
    float* adst = p.alpha + (long long)j * p.G + c;
    // scale of the next plane; `negs` are its signs
    auto scale_of = [&]() {
        double leaf[LEAVES];
#pragma unroll
        for (int k = 0; k < LEAVES; ++k) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll
            for (int e = k * LEAF; e < (k + 1) * LEAF; e += 4) {
                s0 += fabs(t[e]);
                s1 += fabs(t[e + 1]);
                s2 += fabs(t[e + 2]);
                s3 += fabs(t[e + 3]);
            }
            leaf[k] = (s0 + s1) + (s2 + s3);
        }
        const double S = lanes_sum<L, TW>(tree_of_leaves(leaf), scratch);
        // a power-of-two group size divides exactly by multiplying with its reciprocal
        return (float)(inv_m != 0.0 ? __dmul_rn(S, inv_m) : __ddiv_rn(S, md));
    };
    // the residual after a plane with scale ai
    auto next_residual = [&](float ai) {
        const double ad = (double)ai;
        uint32_t kept = 0u, least = 0xFFFFFFFFu;
        if (__all_sync(0xffffffffu, valid == kAll)) {
#pragma unroll
            for (int e = EPT - 1; e >= 0; --e) {
                t[e] = ad - fabs(t[e]);
                kept = __funnelshift_l((uint32_t)__double2hiint(t[e]), kept, 1);
                least = min(least, (uint32_t)__double2hiint(t[e]));
            }
        } else {
#pragma unroll
            for (int i4 = NI - 1; i4 >= 0; --i4) {  // a piece without weights: -0.0 - 0.0 is -0.0
                const double ap = i4 < pieces ? ad : -0.0;
#pragma unroll
                for (int e = 4 * i4 + 3; e >= 4 * i4; --e) {
                    t[e] = ap - fabs(t[e]);
                    kept = __funnelshift_l((uint32_t)__double2hiint(t[e]), kept, 1);
                    least = min(least, (uint32_t)__double2hiint(t[e]));
                }
            }
            if (partial) {
#pragma unroll
                for (int e = 0; e < EPT; ++e)
                    if (!((valid >> e) & 1u)) t[e] = -0.0;
            }
        }
        negs ^= ~kept;
        if (least == 0u) {  // a residual of exactly zero counts as positive
#pragma unroll
            for (int e = 0; e < EPT; ++e)
                if (t[e] == 0.0 && ((valid >> e) & 1u)) negs &= ~(1u << e);
        }
    };
    float last = 0.f;  // a scale that is not finite if a weight of the group is not
    if constexpr (!ALT) {
        for (int i = 0; i < q; ++i) {
            const float ai = last = scale_of();
            const uint32_t word = transpose_bits(~negs);
            if (writes) dst[i * plane_words] = word & word_mask;
            if (live && tl == 0) adst[i * plane_alpha] = ai;
            if (i + 1 < q || p.sq_err != nullptr) next_residual(ai);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            a[i] = scale_of();
            neg[i] = negs;
            if (i + 1 < Q) next_residual(a[i]);
        }

        // ---- alternating rounds.  From here on only magnitudes count: b_i w = (b_i sign(w)) |w|, so the
        // sums run over |w| with the signs `neg` relative to sign(w), and so do the mismatch counts.
        uint32_t sgn = 0u, zero = 0u;
        float tiny = __int_as_float(0x7F800000), amax = 0.f;
#pragma unroll
        for (int e = EPT - 1; e >= 0; --e) {
            sgn = __funnelshift_l(__float_as_uint(w[e]), sgn, 1);
            w[e] = fabsf(w[e]);
            zero = (zero << 1) | (w[e] == 0.f ? 1u : 0u);
            if (w[e] != 0.f) tiny = fminf(tiny, w[e]);
            amax = fmaxf(amax, w[e]);
        }
        zero &= valid;
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        if constexpr (TW > 1) amax = (float)warps_sum<TW>((double)amax, scratch);  // a bound: the sum over the warps
#pragma unroll
        for (int i = 0; i < Q; ++i) neg[i] ^= sgn;

        double S[Q];  // this thread's part of B^T w; a leaf is added from its last weight to its first
        double leaf[Q], odd[Q], upper[Q];
        auto end_leaf = [&](int k) {  // leaves come from the last to the first
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (LEAVES == 1) S[i] = leaf[i];
                else if (k & 1) odd[i] = leaf[i];
                else if (LEAVES == 4 && k == 2) upper[i] = leaf[i] + odd[i];
                else S[i] = LEAVES == 4 ? (leaf[i] + odd[i]) + upper[i] : leaf[i] + odd[i];
            }
        };
        auto sums_from_signs = [&]() {
#pragma unroll
            for (int k = LEAVES - 1; k >= 0; --k) {
#pragma unroll
                for (int i = 0; i < Q; ++i) leaf[i] = 0.0;
#pragma unroll
                for (int e = (k + 1) * LEAF - 1; e >= k * LEAF; --e) {
                    const double x = (double)w[e];
                    const int hi = __double2hiint(x), lo = __double2loint(x);
#pragma unroll
                    for (int i = 0; i < Q; ++i)
                        leaf[i] += __hiloint2double(hi ^ (int)((neg[i] << (31 - e)) & 0x80000000u), lo);
                }
                end_leaf(k);
            }
        };
        sums_from_signs();
        uint32_t flip0 = 0u;  // the code of an exact zero is the complement of the smallest level's
        for (int it = 0;; ++it) {
            // ---- least-squares alpha for the current signs
            double A[Q][Q + 1];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                A[i][Q] = lanes_sum<L, TW>(S[i], scratch);
                A[i][i] = md;
            }
            // mismatch counts, two to a word (at most 1024 weights to a warp)
            constexpr int PAIRS = Q * (Q - 1) / 2;
            uint32_t cnt[PAIRS > 0 ? (PAIRS + 1) / 2 : 1] = {};
            {
                int n = 0;
#pragma unroll
                for (int i = 0; i < Q; ++i)
#pragma unroll
                    for (int l = i + 1; l < Q; ++l, ++n)
                        cnt[n / 2] += (uint32_t)__popc((neg[i] ^ neg[l]) & valid) << (16 * (n & 1));
            }
            if (PAIRS > 0) {
#pragma unroll
                for (int v = 0; v < (PAIRS + 1) / 2; ++v) {
#pragma unroll
                    for (int o = L / 2; o > 0; o >>= 1) cnt[v] += __shfl_xor_sync(0xffffffffu, cnt[v], o);
                }
                int n = 0;
#pragma unroll
                for (int i = 0; i < Q; ++i)
#pragma unroll
                    for (int l = i + 1; l < Q; ++l, ++n) {
                        double mism = (double)((cnt[n / 2] >> (16 * (n & 1))) & 0xFFFFu);
                        if constexpr (TW > 1) mism = warps_sum<TW>(mism, scratch);
                        A[i][l] = md - 2.0 * mism;
                        A[l][i] = A[i][l];
                    }
            }
            solve_ls_static<Q>(md, A, a);
            if (it == p.alt_iters) break;  // the last pass is the final refit only
            // ---- every weight moves to the nearest level
            // (opaque to the compiler, which would keep all fp64 copies across the rounds and spill)
#pragma unroll
            for (int e = 0; e < EPT; ++e) asm volatile("" : "+f"(w[e]));
            LevelSearch<Q> ls;
            ls.build(a, amax);
            flip0 = (ls.codes >> (Q - 1)) & 1u;
            float near = tiny;
#pragma unroll
            for (int i = 0; i < Q; ++i) neg[i] = 0u;
#pragma unroll
            for (int k = LEAVES - 1; k >= 0; --k) {
#pragma unroll
                for (int i = 0; i < Q; ++i) leaf[i] = 0.0;
#pragma unroll
                for (int e = (k + 1) * LEAF - 1; e >= k * LEAF; --e) {
                    const uint32_t y = ls.find(w[e], near);
                    const double x = (double)w[e];
                    const int hi = __double2hiint(x), lo = __double2loint(x);
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const uint32_t b = y << (31 - i);
                        neg[i] = __funnelshift_l(b, neg[i], 1);
                        leaf[i] += __hiloint2double(hi ^ (int)(b & 0x80000000u), lo);
                    }
                }
                end_leaf(k);
            }
            if (!(near > ls.delta)) {
                // some weight of this thread is too close to call in fp32
                flip0 = 0u;
#pragma unroll
                for (int i = 0; i < Q; ++i) neg[i] = 0u;
#pragma unroll
                for (int e = EPT - 1; e >= 0; --e) {
                    const uint32_t code = nearest_code<Q>(((sgn >> e) & 1u) ? -(double)w[e] : (double)w[e], a);
#pragma unroll
                    for (int i = 0; i < Q; ++i) neg[i] |= (~(code >> i) & 1u) << e;
                }
#pragma unroll
                for (int i = 0; i < Q; ++i) neg[i] ^= sgn;
                sums_from_signs();
            }
        }
        last = a[0];
        // ---- write the planes
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            // flip0: a zero is equidistant from +L and -L, the larger code (plane Q - 1 at +1) wins
            neg[i] ^= sgn ^ (flip0 ? zero : 0u);
            const uint32_t word = transpose_bits(~neg[i]);
            if (writes) dst[i * plane_words] = word & word_mask;
            if (live && tl == 0) adst[i * plane_alpha] = a[i];
        }
        if (p.sq_err != nullptr) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                double wh = 0.0;
#pragma unroll
                for (int i = 0; i < Q; ++i) wh = ((neg[i] >> e) & 1u) ? wh - (double)a[i] : wh + (double)a[i];
                t[e] = ((valid >> e) & 1u) ? (((sgn >> e) & 1u) ? -(double)w[e] : (double)w[e]) - wh : 0.0;
            }
        }
    }

    // ---- zero padding words of the row, optional squared error
    if (c == p.G - 1 && live) {
        const int first_pad = (p.d_in + 31) >> 5;
        const int npad = p.pitch - first_pad;  // 0..3
        for (int e = tl; e < npad * q; e += NT) {
            const int i = e / npad;
            p.bits[i * plane_words + (long long)j * p.pitch + first_pad + (e - i * npad)] = 0u;
        }
    }
    if (p.sq_err != nullptr) {
        double leaf[LEAVES];
#pragma unroll
        for (int k = 0; k < LEAVES; ++k) {
            leaf[k] = 0.0;
#pragma unroll
            for (int e = k * LEAF; e < (k + 1) * LEAF; ++e) leaf[k] += t[e] * t[e];
        }
        const double E = lanes_sum<L, TW>(tree_of_leaves(leaf), scratch);
        if (live && tl == 0) p.sq_err[(long long)j * p.G + c] = E;
    }
    if (!(fabsf(last) <= 3.402823466e38f)) {
        // rare: everything is formed again, so that nothing of it is kept for the sake of these calls
        uint32_t block;
        asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(block));
        const long long again = (long long)block * TEAMS + (TW == 1 ? threadIdx.x / L : 0);
        const int t = TW == 1 ? (int)(threadIdx.x & (L - 1)) : (int)threadIdx.x;
        if (!ALT && again < p.items && (t & 3) < NI / 2) greedy_word_not_finite(p, again, (t >> 2) * (NI / 2) + (t & 3));
        if (ALT && again < p.items && t == 0) fit_not_finite(p, again);
    }
}

template <int NI, int L, int TW, int Q>
cudaError_t launch_team(const QuantParams& p, cudaStream_t stream) {
    constexpr int TEAMS = TW == 1 ? 128 / L : 1;
    const int threads = TW == 1 ? 128 : TW * 32;
    const unsigned blocks = (unsigned)((p.items + TEAMS - 1) / TEAMS);
    return bcq::launch_pdl(team_quantize_kernel<NI, L, TW, Q>, dim3(blocks), threads, 0, stream, 1, p);
}

// Greedy: the smallest team that holds a group at 32 weights a thread (8 or 16 for groups of 32 or 64).
// Alternating: a thread goes through its weights one after the other in every round, so a problem that
// is over in a few waves takes as long as one thread does, and fewer weights a thread are better;
// more lanes mean more shuffles and more copies of the solve, which a long one pays for.  Measured, five
// rounds, at 32 / 16 / 8 weights a thread:
//   g = 128, q = 4   512 x 512 56 / 37 / 28 us   2048 x 1536 209 / 138 / 118   3000 x 4096 401 / 333 / 401
//                    5120 x 5120 711 / 653 / 851
//   g = 128, q = 3   512 x 512 31 / 20 / 21 us   1406 x 1582 93 / 55 / 58   5120 x 5120 357 / 345 / 468
//   g = 128, 1600 x 1600, 16 / 8 a thread: q = 1 18.6 / 15.5 us, q = 2 37.9 / 33.4, q = 3 72.7 / 63.8;
//                    64 x 512, q = 3 13.0 / 10.1 (so for every q, though two problems of q = 3 above lose 5 %)
//   g = 256, q = 3   1406 x 1582 106 / 57 us     5120 x 5120 355 / 346
//   a row, q = 3     1024 x 1024 80 / 53 us      2048 x 1536 128 / 98       3000 x 4096 231 / 288
// The line between "few waves" and "long" is 30720 weights per SM (4.5 M on 148, three waves of the
// 16-weight teams).
template <int Q>
cudaError_t launch_team_size(const QuantParams& p, cudaStream_t s) {
    const int g = p.g;
    const bool few = Q > 0 && p.items * g <= 30720ll * bcq::sm_count();
    if (g <= 32) return launch_team<2, 4, 1, Q>(p, s);
    if (g <= 64) return launch_team<4, 4, 1, Q>(p, s);
    if constexpr (Q > 0) {
        if (g <= 128) return few ? launch_team<2, 16, 1, Q>(p, s) : launch_team<4, 8, 1, Q>(p, s);
        if (g <= 256) return launch_team<4, 16, 1, Q>(p, s);
        if (g <= 512) return launch_team<4, 32, 1, Q>(p, s);
        if (g <= 1024 && few) return launch_team<4, 32, 2, Q>(p, s);
        if (g <= 2048 && few) return launch_team<4, 32, 4, Q>(p, s);
    } else {
        if (g <= 128) return launch_team<8, 4, 1, Q>(p, s);
        if (g <= 256) return launch_team<8, 8, 1, Q>(p, s);
        if (g <= 512) return launch_team<8, 16, 1, Q>(p, s);
    }
    if (g <= 1024) return launch_team<8, 32, 1, Q>(p, s);
    if (g <= 2048) return launch_team<8, 32, 2, Q>(p, s);
    if (g <= 4096) return launch_team<8, 32, 4, Q>(p, s);
    if (g <= 8192) return launch_team<8, 32, 8, Q>(p, s);
    if (g <= 16384) return launch_team<8, 32, 16, Q>(p, s);
    return launch_team<8, 32, 32, Q>(p, s);
}

template <int EPT, int TW>
cudaError_t launch_quantize(const QuantParams& p, cudaStream_t stream) {
    constexpr int TEAMS = (TW == 1) ? 4 : 1;
    const int threads = (TW == 1) ? 128 : TW * 32;
    long long blocks = (p.items + TEAMS - 1) / TEAMS;
    const long long cap = (long long)bcq::sm_count() * 64;  // grid-stride beyond this
    if (blocks > cap) blocks = cap;
    return bcq::launch_pdl(quantize_kernel<EPT, TW>, dim3((unsigned)blocks), threads, 0, stream, 1, p);
}

__global__ void dequantize_kernel(int d_out, int d_in, int q, int g, int G, int pitch,
                                  const uint32_t* bits,
                                  const float* alpha, float* W_hat,
                                  long long ldw) {
    const int j = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d_in) return;
    const int c = k / g;
    float s = 0.0f;
    for (int i = 0; i < q; ++i) {
        const uint32_t word = bcq::ld(bits + ((long long)i * d_out + j) * pitch + (k >> 5));
        const float a = bcq::ld(alpha + ((long long)i * d_out + j) * G + c);
        s += ((word >> (k & 31)) & 1u) ? a : -a;
    }
    W_hat[(long long)j * ldw + k] = s;
}

}  // namespace

extern "C" bcq_status bcq_quantize(int d_out, int d_in, int q, int g, const float* W, size_t ldw,
                                   int alt_iters, uint32_t* bits, float* alpha, double* sq_err,
                                   void* stream) {
    bcq_status st = bcq::check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (!W || !bits || !alpha) return BCQ_ERR_NULL;
    if (ldw < (size_t)d_in || alt_iters < 0) return BCQ_ERR_SHAPE;
    if (g > BCQ_MAX_QUANT_G) return BCQ_ERR_UNSUPPORTED;
    if (!bcq::aligned16(bits)) return BCQ_ERR_ALIGN;
    QuantParams p;
    p.d_out = d_out; p.d_in = d_in; p.q = q; p.g = g;
    p.G = (int)bcq_num_groups(d_in, g);
    p.alt_iters = alt_iters;
    p.ldw = (long long)ldw;
    p.pitch = (int)bcq_pitch_words(d_in);
    p.W = W; p.bits = bits; p.alpha = alpha; p.sq_err = sq_err;
    p.items = (long long)d_out * p.G;
    p.vec = bcq::aligned16(W) && ldw % 4 == 0;
    p.inv_g = (g & (g - 1)) == 0 ? 1.0 / g : 0.0;
    p.g_magic = 0; p.g_shift = 0;
    if (p.G > 1 && p.items < (1ll << 31)) {
        // ceil(2^(32 + s) / G) with 2^s < G <= 2^(s+1): exact for every item below 2^31
        int sh = 0;
        while ((2ll << sh) < p.G) ++sh;
        p.g_shift = (uint32_t)sh;
        p.g_magic = (uint32_t)(((1ull << (32 + sh)) + p.G - 1) / p.G);
    }
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    if (alt_iters == 0) e = launch_team_size<0>(p, s);
    else if (q == 1) e = launch_team_size<1>(p, s);
    else if (q == 2) e = launch_team_size<2>(p, s);
    else if (q == 3) e = launch_team_size<3>(p, s);
    else if (q == 4) e = launch_team_size<4>(p, s);
    else if (g <= 128) e = launch_quantize<4, 1>(p, s);
    else if (g <= 256) e = launch_quantize<8, 1>(p, s);
    else if (g <= 512) e = launch_quantize<16, 1>(p, s);
    else if (g <= 1024) e = launch_quantize<32, 1>(p, s);
    else if (g <= 2048) e = launch_quantize<8, 8>(p, s);
    else if (g <= 4096) e = launch_quantize<16, 8>(p, s);
    else if (g <= 8192) e = launch_quantize<32, 8>(p, s);
    else e = launch_quantize<32, 32>(p, s);
    if (e != cudaSuccess) return bcq::cuda_fail(e);
    return BCQ_OK;
}

extern "C" bcq_status bcq_dequantize(int d_out, int d_in, int q, int g, const uint32_t* bits,
                                     const float* alpha, float* W_hat, size_t ldw, void* stream) {
    bcq_status st = bcq::check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (!bits || !alpha || !W_hat) return BCQ_ERR_NULL;
    if (ldw < (size_t)d_in) return BCQ_ERR_SHAPE;
    if (d_out > 65535 * 1) {
        // grid.y limit: fold rows is not needed for the layer sizes this library targets
        if (d_out > 65535) return BCQ_ERR_UNSUPPORTED;
    }
    dim3 grid((unsigned)bcq::ceil_div(d_in, 256), (unsigned)d_out);
    dequantize_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(
        d_out, d_in, q, g, (int)bcq_num_groups(d_in, g), (int)bcq_pitch_words(d_in), bits, alpha,
        W_hat, (long long)ldw);
    bcq::count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return bcq::cuda_fail(e);
    return BCQ_OK;
}
