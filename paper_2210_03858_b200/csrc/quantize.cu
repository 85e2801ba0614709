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
// layer of width 1600 (30.7 M weights) 162 -> 56 us (2.6 TB/s; the logic pipe is 55 % busy, the fp64
// pipe 21 %); two alternating rounds, q = 3, g = 128, 5120 x 5120: 190 us (instruction fetch of the
// unrolled rounds and fp64 latency at five warps per scheduler bound it).
//
// Sums are fp64 and are reduced in a fixed order, so a result never depends on scheduling.
//
// sorted_quantize_kernel (alternating, q = 2 .. 4, groups of up to 256, three rounds or more): see there.
//
// quantize_kernel (alternating, q > 4): one warp per group up to 1024 weights, a CTA above.
//
// Appendix "Details on BCQ Format": Eq. ap:1-ap:3 (greedy), Eq. ap:4 and the following
// paragraph (alternating).
#include <algorithm>

#include "gemm_common.cuh"

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
    int row_items;    // items that the order of the items counts to a row: G, or see team_quantize_kernel
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

// Nearest of the 2^Q levels, the largest code among equidistant ones: the definition.  (Unrolled, so that the chains
// of the levels run side by side; scales by value, which keeps the callers' out of local memory.)
template <int Q>
__device__ __noinline__ uint32_t nearest_code_of(double w, float a0, float a1, float a2, float a3) {
    const float a[4] = {a0, a1, a2, a3};
    uint32_t best = 0u;
    double dbest = 0.0;
#pragma unroll
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
template <int Q>
__device__ __forceinline__ uint32_t nearest_code(double w, const float (&a)[Q]) {
    return nearest_code_of<Q>(w, a[0], a[Q > 1 ? 1 : 0], a[Q > 2 ? 2 : 0], a[Q > 3 ? 3 : 0]);
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
// TAILS: the items are the full groups, row by row, and after them the short last group of every row.  A warp that
// holds a short group goes another way for all its groups; row by row that were 61 % of the warps at 1600 columns and
// g = 128 (6400 rows, q = 4: 20.1 us row by row and 18.2 with the short groups last; 2222 x 3331, q = 3: 18.9 and 15.6).  An
// instance of its own, because the order costs matrices without short groups 3 to 6 %.
// Blocks to an SM: with four planes and 8 weights a lane four, since the 80 registers of six are too few (512 x 512, g = 32, two
// rounds: 17.1 us with six and 13.5 with four; 5120 x 5120 539 and 522; with three, 170 registers, 12.9 and 592).
template <int NI, int L, int TW, int Q, bool TAILS>
__global__ void __launch_bounds__(TW == 1 ? 128 : TW * 32,
                                  TW == 1   ? ((NI == 2 && Q < 4) || (Q == 0 && NI == 4) ? 6 : NI == 2 ? 4 : Q == 0 || NI == 4 ? 5 : 3)
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
        c = (int)((uint32_t)item - (uint32_t)j * (uint32_t)p.row_items);
    } else {
        j = (int)(item / p.row_items);
        c = (int)(item - (long long)j * p.row_items);
    }
    if (TAILS && item >= (long long)p.d_out * p.row_items) {
        j = (int)(item - (long long)p.d_out * p.row_items);
        c = p.row_items;
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
        long long again = (long long)block * TEAMS + (TW == 1 ? threadIdx.x / L : 0);
        if (TAILS && again < p.items) {
            const long long full_items = (long long)p.d_out * p.row_items;
            again = again < full_items ? again / p.row_items * p.G + again % p.row_items : (again - full_items) * p.G + p.row_items;
        }
        const int t = TW == 1 ? (int)(threadIdx.x & (L - 1)) : (int)threadIdx.x;
        if (!ALT && again < p.items && (t & 3) < NI / 2) greedy_word_not_finite(p, again, (t >> 2) * (NI / 2) + (t & 3));
        if (ALT && again < p.items && t == 0) fit_not_finite(p, again);
    }
}

// ------------------------------------------------------------------------------------------
// alternating, groups of up to 256 weights: rounds on sorted magnitudes
// ------------------------------------------------------------------------------------------
//
// In a round a weight's code depends on its magnitude alone, and does not decrease with it: the levels cut the
// sorted magnitudes of a group into 2^(Q-1) runs.  So a group is sorted once, with the running sums of its
// magnitudes beside it, and a round is Q = 3: three searches and as many differences of running sums,
// whatever the group's size.  The greedy start is a tree of such cuts too.
//
// A warp takes up to 32 groups.  (1) In teams of L lanes it loads 32 / L groups at a time, sorts them in registers
// (a network in each lane, then merges across the lanes) and puts keys and running sums into shared memory.
// (2) Lane k does all rounds of group k (or four lanes do, see SHARE), so a least-squares solve is done once per group
// and not by every lane of a team.  (3) In teams again, the weights are read once more (from L2), find their levels and are
// written as planes.  Warps are blocks of their own, so that some sort while others wait for the chains of fp64
// divisions of (2); eight or nine fit an SM (25 KiB each).
//
// The team kernel keeps a group in registers and goes through its weights in every round, and all lanes of a team solve.
// Measured, that and this: 5120 x 5120, g = 128, five rounds: q = 3 331 and 167 us, q = 4 599 and 278 (launch_team_size has
// more).  What bounds it now: min and max of the sort run at half rate (the logic pipe), and the code, 15 to 30 KiB for
// a pass, comes slowly to eight warps an SM (stall no_instruction; 4.2 an issue with everything unrolled, 250 us).
//
// Key of a weight: its magnitude's bits shifted left by one, below them 1 where it is not negative: integers in the
// order of the magnitudes, of equal ones the negative first.  That is the order in which sign(0) = +1 decides
// a residual of exactly zero (a negative weight with |w| = a gets b = +1, that is, against its own sign, like
// the smaller magnitudes; a positive one like the larger).
constexpr uint32_t kNoKey = 0xFFFFFFFFu;  // behind every weight
constexpr int kRun = 4;                   // keys between two running sums

template <int N>
__device__ __forceinline__ void sort_keys(uint32_t (&v)[N]) {  // Batcher's odd-even merge sort
#pragma unroll
    for (int p = 1; p < N; p *= 2)
#pragma unroll
        for (int k = p; k >= 1; k /= 2)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int at = i - k % p;  // pairs (i, i + k) inside blocks of 2 k from k mod p on
                if (at >= 0 && at % (2 * k) < k && i + k < N && i / (2 * p) == (i + k) / (2 * p)) {
                    const uint32_t a = v[i], b = v[i + k];
                    v[i] = min(a, b);
                    v[i + k] = max(a, b);
                }
            }
}

// N keys a lane, ascending in each lane, to ascending over the L lanes of a team (lane l: N l .. N l + N - 1).
template <int N, int L>
__device__ __forceinline__ void merge_lanes(uint32_t (&v)[N], int tl) {
    // (loops: unrolled, the code of the kernel would not fit the instruction caches)
#pragma unroll 1
    for (int w = 2; w <= L; w *= 2) {
        // the smaller half of two neighbouring sequences to the lower lanes ...
        const bool upper = (tl & (w / 2)) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const uint32_t a = __shfl_xor_sync(0xffffffffu, v[N - 1 - i], w - 1), b = __shfl_xor_sync(0xffffffffu, v[i], w - 1);
            v[i] = upper ? max(v[i], a) : min(v[i], a);
            v[N - 1 - i] = upper ? max(v[N - 1 - i], b) : min(v[N - 1 - i], b);
        }
        // ... and each half, which rises and falls once, into order
#pragma unroll 1
        for (int d = w / 4; d >= 1; d /= 2) {
            const bool up = (tl & d) != 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t a = __shfl_xor_sync(0xffffffffu, v[i], d);
                v[i] = up ? max(v[i], a) : min(v[i], a);
            }
        }
#pragma unroll
        for (int d = N / 2; d >= 1; d /= 2)
#pragma unroll
            for (int i = 0; i < N; ++i)
                if ((i & d) == 0) {
                    const uint32_t a = v[i], b = v[i + d];
                    v[i] = min(a, b);
                    v[i + d] = max(a, b);
                }
    }
}

// Keys of weights below the cut t of a greedy plane: magnitudes under t, and of those equal to t the negative ones.
__device__ __forceinline__ uint32_t key_below(double t) {
    if (!(t > 0.0)) return 0u;  // a zero counts as positive
    const float f = __double2float_rd(t);
    return (__float_as_uint(f) << 1) + ((double)f == t ? 1u : 2u);
}

__device__ __forceinline__ float key_magnitude(uint32_t key) { return __uint_as_float(key >> 1); }

template <int NI, int L>
struct SortedShape {
    static_assert(L >= 4, "four lanes share 128 weights");
    static constexpr int EPT = 4 * NI, C = EPT * L, TEAMS = 32 / L, RUNS = C / kRun;
    static constexpr int GROUPS = C > 128 ? 16 : 32;  // of a warp: what leaves room for eight warps on an SM
    static constexpr size_t bytes = (size_t)C * GROUPS * 4 + (size_t)(RUNS + 1) * GROUPS * 8;
};

constexpr int kSortWarps = 4;         // of a block, at most
constexpr long long kSortPlaces = 9;  // warps that an SM holds

// PIECES: the full groups leave some of the lanes' 16-byte pieces empty.  An instance of its own, because asking for each piece
// costs full lanes 1 % (5120 x 5120, g = 128, q = 3, five rounds 166.7 us and 168.4), and taking such groups one weight at a
// time, as short last groups of an odd size are taken, costs more (g = 224, q = 3, three rounds, 3200 x 5376: 146.4 and 138.4).
// SHARE: four lanes to a group in (2), for calls that give a warp at most eight, whose other lanes would be idle: each looks for
// every fourth cut, and all do the rest alike.  One lane goes through the cuts one instruction at a time, which a chip
// full of warps hides and a small call does not: 512 x 512, g = 256, q = 4, five rounds 27.4 us and 22.5, q = 3 15.9 and 15.1.
template <int NI, int L, int Q, bool PIECES, bool SHARE>
__global__ void __launch_bounds__(32 * kSortWarps, 2)
sorted_quantize_kernel(const QuantParams p, int batch) {
    using Sh = SortedShape<NI, L>;
    constexpr int EPT = Sh::EPT, C = Sh::C, TEAMS = Sh::TEAMS, RUNS = Sh::RUNS, GROUPS = Sh::GROUPS;
    constexpr int N = 1 << (Q - 1);
    constexpr int LEAF = 8, LEAVES = EPT / LEAF;  // see lanes_sum
    constexpr uint32_t kMask = (1u << Q) - 1u;
    extern __shared__ double sorted_smem[];
    const int warp = threadIdx.x >> 5;
    double* sums = sorted_smem + warp * (Sh::bytes / 8);                       // [RUNS + 1][GROUPS], the last row: of all
    uint32_t* keys = reinterpret_cast<uint32_t*>(sums + (RUNS + 1) * GROUPS);  // [C][GROUPS]
    const int lane = threadIdx.x & 31;
    const int tl = lane & (L - 1);
    // the column of a group is turned by the lane that holds the position, so that the lanes of a team store to
    // different banks
    auto key_at = [&](int pos, int grp) { return pos * GROUPS + (grp ^ ((pos / EPT) * TEAMS & (GROUPS - 1))); };
    auto sum_at = [&](int run, int grp) { return run * GROUPS + (grp ^ ((run * kRun / EPT) * TEAMS & (GROUPS - 1))); };

    bcq::pdl_wait();  // (and no pdl_trigger: a long kernel, see launch_pdl)
    // (warps past the last group do it again)
    const long long first = min(((long long)blockIdx.x * (blockDim.x >> 5) + warp) * batch, p.items - 1);
    const int count = (int)min((long long)batch, p.items - first);  // groups of this warp

    struct Place { int j, c, m; };
    auto place = [&](long long item) {
        Place x;
        if (p.g_magic != 0u) {
            x.j = (int)(__umulhi((uint32_t)item, p.g_magic) >> p.g_shift);
            x.c = (int)((uint32_t)item - (uint32_t)x.j * (uint32_t)p.G);
        } else {
            x.j = (int)(item / p.G);
            x.c = (int)(item - (long long)x.j * p.G);
        }
        x.m = min(p.g, p.d_in - x.c * p.g);
        return x;
    };
    // Weight 4 i + e of a lane: 16 i + e after its first.
    const int kt = (tl >> 2) * (16 * NI) + (tl & 3) * 4;
    // pieces from .. of a lane
    auto load = [&](const Place& x, int from, auto& w) {
        constexpr int COUNT = sizeof(w) / sizeof(float);
        const float* src = p.W + (long long)x.j * p.ldw + x.c * p.g + kt + 16 * from;
        const int left = x.m - kt - 16 * from;
        if (p.vec && (PIECES ? (x.m & 3) == 0 : x.m == C)) {
#pragma unroll
            for (int i = 0; i < COUNT / 4; ++i) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!PIECES || 16 * i < left) v = bcq::ld(reinterpret_cast<const float4*>(src + 16 * i));
                w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int e = 0; e < COUNT; ++e) w[e] = 16 * (e / 4) + e % 4 < left ? bcq::ld(src + 16 * (e / 4) + e % 4) : 0.0f;
        }
    };
    // teams past the last group repeat it (the shuffles need every lane) and store nothing
    auto group_of = [&](int pass) { return min(pass * TEAMS + lane / L, count - 1); };
    const int passes = (batch + TEAMS - 1) / TEAMS;

    // ---- (1) sort
    {
        Place at = place(first + group_of(0)), next = at;
        float w[EPT];
        load(at, 0, w);
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
            __syncthreads();
            uint32_t v[EPT];
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                const uint32_t b = __float_as_uint(__fmul_rn(w[e], -1.0f));
                v[e] = __funnelshift_l(b, b, 1);
            }
            if (at.m < C) {
#pragma unroll
                for (int e = 0; e < EPT; ++e)
                    v[e] = kt + 16 * (e / 4) + e % 4 >= at.m ? kNoKey : min(v[e], kNoKey - 1u);  // (a NaN has these bits)
            }
            if (pass + 1 < passes) {
                next = place(first + group_of(pass + 1));
                load(next, 0, w);
            }
            sort_keys<EPT>(v);
            merge_lanes<EPT, L>(v, tl);
            // running sums: in blocks of 16 keys from the left, the blocks in a scan over their numbers: an order that the
            // lanes' share of a group does not show in
            constexpr int BLOCK = EPT < 16 ? EPT : 16, BLOCKS = EPT / BLOCK;
            double before[EPT / kRun], upto[BLOCKS];
            auto add_blocks = [&](bool all) {
#pragma unroll
                for (int b = 0; b < BLOCKS; ++b) {
                    double s = 0.0;
#pragma unroll
                    for (int e = b * BLOCK; e < (b + 1) * BLOCK; ++e) {
                        if (e % kRun == 0) before[e / kRun] = s;
                        if (all || v[e] != kNoKey) s += (double)key_magnitude(v[e]);
                    }
                    upto[b] = s;
                }
            };
            if (at.m == C) add_blocks(true);
            else add_blocks(false);
#pragma unroll
            for (int o = 1; o < C / BLOCK; o <<= 1) {
                double from[BLOCKS];
#pragma unroll
                for (int b = 0; b < BLOCKS; ++b)  // block o before this one
                    from[b] = o < BLOCKS && b >= o ? upto[b - o]
                                                   : __shfl_up_sync(0xffffffffu, upto[(b - o) & (BLOCKS - 1)], o < BLOCKS ? 1 : o / BLOCKS, L);
#pragma unroll
                for (int b = 0; b < BLOCKS; ++b)
                    if (tl * BLOCKS + b >= o) upto[b] = from[b] + upto[b];
            }
            double base[BLOCKS];
            base[0] = __shfl_up_sync(0xffffffffu, upto[BLOCKS - 1], 1, L);
            if (tl == 0) base[0] = 0.0;
#pragma unroll
            for (int b = 1; b < BLOCKS; ++b) base[b] = upto[b - 1];
            const int grp = pass * TEAMS + lane / L;
            if (grp < count) {
#pragma unroll
                for (int e = 0; e < EPT; ++e) keys[key_at(tl * EPT + e, grp)] = v[e];
#pragma unroll
                for (int r = 0; r < EPT / kRun; ++r) sums[sum_at(tl * (EPT / kRun) + r, grp)] = base[r * kRun / BLOCK] + before[r];
                if (tl == L - 1) sums[RUNS * GROUPS + grp] = upto[BLOCKS - 1];
            }
            at = next;
        }
    }
    __syncwarp();

    // ---- (2) rounds: a group per lane, or per four
    constexpr int SHARES = SHARE ? 4 : 1, OWN = (N - 1 + SHARES - 1) / SHARES;  // cuts that a lane looks for: s = share + 1, + SHARES, ...
    const int slot = SHARE ? lane & 7 : lane, share = SHARE ? lane >> 3 : 0;
    const int grp = min(slot, count - 1);
    auto own = [&](const auto& of_cut, int o) {  // (of the last cut again, where there are fewer)
        auto v = of_cut[min(SHARES * o + 1, N - 1)];
#pragma unroll
        for (int k = 1; k < SHARES; ++k) v = share == k ? of_cut[min(SHARES * o + 1 + k, N - 1)] : v;
        return v;
    };
    const long long item = first + grp;
    float a[Q], a_cut[Q];  // scales; the scales that the last cuts were made for
    LevelSearch<Q> ls;
    {
        const int m = place(item).m;
        const double md = (double)m;
        const double inv_m = m == p.g ? p.inv_g : (m & (m - 1)) == 0 ? 1.0 / md : 0.0;
        const double total = sums[RUNS * GROUPS + grp];
        auto mean = [&](double S) { return (float)(inv_m != 0.0 ? __dmul_rn(S, inv_m) : __ddiv_rn(S, md)); };
        auto key = [&](int pos) { return keys[key_at(pos, grp)]; };
        // number of keys below k, and the sum of their magnitudes
        auto cut = [&](uint32_t k, double& sum) {
            int r = 0;
#pragma unroll
            for (int s = RUNS / 2; s >= 1; s /= 2)
                if (key((r + s) * kRun) < k) r += s;
            double t = sums[sum_at(r, grp)];
            int n = r * kRun;
#pragma unroll
            for (int e = 0; e < kRun; ++e) {
                const uint32_t x = key(r * kRun + e);
                if (x < k) {
                    t += (double)key_magnitude(x);
                    ++n;
                }
            }
            sum = t;
            return n;
        };
        // the runs: run s is cuts[s] .. cuts[s + 1] - 1; below[s] = sum of the magnitudes before it
        int cuts[N + 1];
        double below[N + 1];
        cuts[0] = 0; below[0] = 0.0;
        cuts[N] = m; below[N] = total;

        const float amax = key_magnitude(key(m - 1));
        float tiny = __int_as_float(0x7F800000);  // smallest magnitude that is not zero
        {
            int zeros = 0;
#pragma unroll 1
            while (zeros < m && key(zeros) < 2u) ++zeros;
            if (zeros < m) tiny = key_magnitude(key(zeros));
        }
        // Greedy: plane i cuts every run of the planes before it at its centre, a sum of +-a_1 .. +-a_(i-1).  Cut s of
        // the final ones, 1 .. N - 1, comes with plane turn(s).
        auto turn = [](int s) {
            int i = Q - 1;
            for (; (s & 1) == 0; s >>= 1) --i;
            return i;
        };
        double centre[N];
        uint32_t at[N];  // keys below at[s] are below cut s
#pragma unroll
        for (int s = 0; s < N; ++s) { centre[s] = 0.0; at[s] = 0u; }
        a[0] = mean(total);
        centre[N / 2] = (double)a[0];
        // codes of the runs, a nibble each: bit i set where plane i is against the sign of the weight
        ls.codes = 0u;
#pragma unroll
        for (int s = 0; s < N; ++s)
#pragma unroll
            for (int i = 1; i < Q; ++i) ls.codes |= (uint32_t)(~(s >> (Q - 1 - i)) & 1) << (4 * s + i);
        ls.delta = 0.f;
#pragma unroll
        for (int s = 0; s < N; ++s) ls.mid[s] = 0.f;
#pragma unroll
        for (int i = 0; i < Q; ++i) a_cut[i] = 0.f;
        bool close = false;    // some weight is too close to a cut to call in fp32
        bool settled = false;  // further rounds change nothing
        // Rounds 1 - Q .. -1 are the greedy planes, one body for all: unrolled, it would not fit the instruction caches
#pragma unroll 1
        for (int it = 1 - Q;; ++it) {
            __syncthreads();
            if (it < 0) {
                const int plane = it + Q;
#pragma unroll
                for (int s = 1; s < N; ++s)
                    if (plane == turn(s)) at[s] = key_below(centre[s]);
            } else {
            // ---- B^T w and B^T B from the runs
            double A[Q][Q + 1], S[Q];
            int agree[Q][Q];  // weights on which planes i and l agree, less the others
            double part[N];
            int num[N];
#pragma unroll
            for (int s = 0; s < N; ++s) {
                part[s] = below[s + 1] - below[s];
                num[s] = cuts[s + 1] - cuts[s];
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                S[i] = 0.0;
#pragma unroll
                for (int s = 0; s < N; ++s) {
                    const uint32_t b = (ls.codes << (31 - 4 * s - i)) & 0x80000000u;
                    S[i] += __hiloint2double(__double2hiint(part[s]) ^ (int)b, __double2loint(part[s]));
                }
#pragma unroll
                for (int l = i + 1; l < Q; ++l) {
                    agree[i][l] = 0;
#pragma unroll
                    for (int s = 0; s < N; ++s) {
                        const uint32_t x = (ls.codes >> (4 * s + i)) ^ (ls.codes >> (4 * s + l));
                        agree[i][l] += (x & 1u) ? -num[s] : num[s];
                    }
                }
            }
            // those weights get the code that the definition gives: the whole warp looks through the group
            for (uint32_t todo = __ballot_sync(0xffffffffu, close); todo != 0u; todo &= todo - 1u) {
                const int f = __ffs(todo) - 1;
                auto of = [&](auto v) { return __shfl_sync(0xffffffffu, v, f); };
                const int fm = of(m);
                const uint32_t fcodes = of(ls.codes);
                const float fdelta = of(0.5f * ls.delta);
                float fmid[N], fa[Q];
                int fcut[N];
#pragma unroll
                for (int s = 1; s < N; ++s) { fmid[s] = of(ls.mid[s]); fcut[s] = of(cuts[s]); }
#pragma unroll
                for (int i = 0; i < Q; ++i) fa[i] = of(a_cut[i]);
                bool changed = false;
                double dS[Q];
                int dagree[Q][Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    dS[i] = 0.0;
#pragma unroll
                    for (int l = i + 1; l < Q; ++l) dagree[i][l] = 0;
                }
#pragma unroll 1
                for (int e = lane; e < fm; e += 32) {
                    const uint32_t k = keys[key_at(e, f)];
                    const float x = key_magnitude(k);
                    float near = x == 0.f ? __int_as_float(0x7F800000) : x;
                    int run = 0;
#pragma unroll
                    for (int s = 1; s < N; ++s) {
                        near = fminf(near, fabsf(x - fmid[s]));
                        run += e >= fcut[s] ? 4 : 0;
                    }
                    if (near > fdelta) continue;
                    const bool negative = (k & 1u) == 0u;
                    const uint32_t was = (fcodes >> run) & kMask;
                    const uint32_t now = (~nearest_code<Q>(negative ? -(double)x : (double)x, fa) & kMask) ^ (negative ? kMask : 0u);
                    changed |= now != was;
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        if (((was ^ now) >> i) & 1u) dS[i] += ((now >> i) & 1u) ? -2.0 * (double)x : 2.0 * (double)x;
#pragma unroll
                        for (int l = i + 1; l < Q; ++l)
                            dagree[i][l] += 2 * ((int)(((was >> i) ^ (was >> l)) & 1u) - (int)(((now >> i) ^ (now >> l)) & 1u));
                    }
                }
                if (!__any_sync(0xffffffffu, changed)) continue;
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const double d = warp_sum(dS[i]);
                    if (slot == f) S[i] += d;
#pragma unroll
                    for (int l = i + 1; l < Q; ++l) {
                        const int n = __reduce_add_sync(0xffffffffu, dagree[i][l]);
                        if (slot == f) agree[i][l] += n;
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                A[i][Q] = S[i];
                A[i][i] = md;
#pragma unroll
                for (int l = i + 1; l < Q; ++l) A[i][l] = A[l][i] = (double)agree[i][l];
            }
            // ---- least-squares alpha for the current signs
            float fit[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) fit[i] = a[i];
            solve_ls_static<Q>(md, A, fit);
            // scales that come out as they went in stay so, and with them the codes (where all magnitudes are alike every
            // weight is too close to a cut, and this spares all rounds but one of looking at each)
            bool same = it > 0;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (!settled) a[i] = fit[i];
                same = same && a[i] == a_cut[i];
            }
            settled = settled || same;
            if (it == p.alt_iters) break;  // the last pass is the final refit only
            // ---- every weight moves to the nearest level
#pragma unroll
            for (int i = 0; i < Q; ++i) a_cut[i] = a[i];
            ls.build(a, amax);
#pragma unroll
            for (int s = 1; s < N; ++s) at[s] = __float_as_uint(ls.mid[s]) << 1;
            }
            int own_cut[OWN];
            double own_below[OWN];
#pragma unroll
            for (int o = 0; o < OWN; ++o) own_cut[o] = cut(own(at, o), own_below[o]);
#pragma unroll
            for (int s = 1; s < N; ++s) {
                const int o = (s - 1) / SHARES, from = slot + 8 * ((s - 1) % SHARES);
                cuts[s] = SHARE ? __shfl_sync(0xffffffffu, own_cut[o], from) : own_cut[o];
                below[s] = SHARE ? __shfl_sync(0xffffffffu, own_below[o], from) : own_below[o];
            }
            if (it < 0) {
                const int plane = it + Q;
                double S = 0.0;
#pragma unroll
                for (int t = 1; t < Q; ++t)
#pragma unroll
                    for (int s = 1; s < N; ++s)
                        if (t == turn(s) && plane >= t) {
                            const int half = N >> t, lo = s - half, hi = s + half;
                            if (cuts[s] <= cuts[lo]) { cuts[s] = cuts[lo]; below[s] = below[lo]; }
                            if (cuts[s] >= cuts[hi]) { cuts[s] = cuts[hi]; below[s] = below[hi]; }
                            if (plane == t)
                                S += ((below[hi] - below[s]) - (double)(cuts[hi] - cuts[s]) * centre[s]) +
                                     ((double)(cuts[s] - cuts[lo]) * centre[s] - (below[s] - below[lo]));
                        }
                const float ai = mean(S);
#pragma unroll
                for (int i = 1; i < Q; ++i)
                    if (plane == i) a[i] = ai;
#pragma unroll
                for (int s = 1; s < N; ++s)
                    if (plane == turn(s)) {
                        const int half = (N >> turn(s)) / 2;
                        if (half > 0) {
                            centre[s - half] = centre[s] - (double)ai;
                            centre[s + half] = centre[s] + (double)ai;
                        }
                    }
            } else {
                float near = tiny;
#pragma unroll
                for (int o = 0; o < OWN; ++o) {
                    const float mid = own(ls.mid, o);
                    if (own_cut[o] > 0) near = fminf(near, mid - key_magnitude(key(own_cut[o] - 1)));
                    if (own_cut[o] < m) near = fminf(near, key_magnitude(key(own_cut[o])) - mid);
                }
                if (SHARE) {
                    near = fminf(near, __shfl_xor_sync(0xffffffffu, near, 8));
                    near = fminf(near, __shfl_xor_sync(0xffffffffu, near, 16));
                }
                // fp32 decides where a weight is 2^-22 of the largest level away from the midpoint, which is rounded by
                // 2^-24 of itself; half of ls.delta keeps the neighbourhoods of two midpoints apart
                close = lane < count && !settled && !(near > 0.5f * ls.delta);
            }
        }
    }
    __syncwarp();
    // what (3) needs of a group, in place of its keys
    float* hand = reinterpret_cast<float*>(keys);  // [row][GROUPS]
    constexpr int ROW_CODES = 0, ROW_DELTA = 1, ROW_CUT = 2, ROW_MID = ROW_CUT + Q, ROW_A = ROW_MID + N;
    constexpr int ROWS = ROW_A + Q;
    static_assert(ROWS * GROUPS + (EPT < 16 ? EPT : 16) * 32 <= C * GROUPS, "space of the keys");
    if (lane < count) {
        keys[ROW_CODES * GROUPS + lane] = ls.codes;
        hand[ROW_DELTA * GROUPS + lane] = ls.delta;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            hand[(ROW_CUT + i) * GROUPS + lane] = a_cut[i];
            hand[(ROW_A + i) * GROUPS + lane] = a[i];
            p.alpha[i * p.items + item] = a[i];
        }
#pragma unroll
        for (int s = 1; s < N; ++s) hand[(ROW_MID + s) * GROUPS + lane] = ls.mid[s];
    }
    __syncwarp();

    // ---- (3) planes, 16 weights of a lane at a time
    {
        constexpr int PART = EPT < 16 ? EPT : 16, PARTS = EPT / PART;
        const long long plane_words = (long long)p.d_out * p.pitch;
        Place at = place(first + group_of(0)), next = at;
        float wn[PART];
        uint32_t neg[Q];
        double leaf[LEAVES];
        load(at, (PARTS - 1) * (PART / 4), wn);
#pragma unroll 1
        for (int turn = 0; turn < passes * PARTS; ++turn) {
            __syncthreads();
            const int pass = turn / PARTS, part = PARTS - 1 - turn % PARTS;  // the last weights first
            const int g3 = group_of(pass);
            float w[PART];
#pragma unroll
            for (int e = 0; e < PART; ++e) w[e] = wn[e] + 0.0f;
            if (turn + 1 < passes * PARTS) {
                if (part == 0) next = place(first + group_of(pass + 1));
                load(next, (part == 0 ? PARTS - 1 : part - 1) * (PART / 4), wn);
            }
            const uint32_t codes = keys[ROW_CODES * GROUPS + g3];
            // bit e of past[s]: weight e is below cut s; every midpoint is subtracted from every weight, which leaves the
            // choice of the code to a few operations on whole words
            uint32_t sgn = 0u, zero = 0u, now[Q], past[N];
            float mid[N];
#pragma unroll
            for (int s = 1; s < N; ++s) {
                mid[s] = hand[(ROW_MID + s) * GROUPS + g3];
                past[s] = 0u;
            }
            float near = __int_as_float(0x7F800000), least = near;
#pragma unroll
            for (int e = PART - 1; e >= 0; --e) {
                sgn = __funnelshift_l(__float_as_uint(w[e]), sgn, 1);
                const float x = fabsf(w[e]);
                least = fminf(least, x);
#pragma unroll
                for (int s = 1; s < N; ++s) {
                    const float d = x - mid[s];
                    near = fminf(near, fabsf(d));
                    past[s] = __funnelshift_l(__float_as_uint(d), past[s], 1);
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                now[i] = 0u - ((codes >> (4 * (N - 1) + i)) & 1u);
#pragma unroll
                for (int s = 1; s < N; ++s) {
                    const uint32_t turns = ((codes >> (4 * s + i)) ^ (codes >> (4 * s - 4 + i))) & 1u;
                    now[i] ^= past[s] & (0u - turns);
                }
            }
            if (least == 0.f) {
                least = __int_as_float(0x7F800000);
#pragma unroll
                for (int e = 0; e < PART; ++e) {
                    if (w[e] == 0.f) zero |= 1u << e;
                    else least = fminf(least, fabsf(w[e]));
                }
                // a zero is equidistant from +L and -L, the larger code (plane Q - 1 at +1) wins
                if (((codes >> (Q - 1)) & 1u) == 0u) zero = 0u;
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) now[i] = (now[i] ^ sgn ^ zero) & ((1u << PART) - 1u);
            const float delta = hand[ROW_DELTA * GROUPS + g3];
            if (!(fminf(near, least) > delta)) {
                // some weights of this lane are too close to a cut to call in fp32
                uint32_t hits = 0u;
#pragma unroll
                for (int e = 0; e < PART; ++e) {
                    float d = fabsf(w[e]);
                    if (d == 0.f && delta < 3.0e38f) d = __int_as_float(0x7F800000);
#pragma unroll
                    for (int s = 1; s < N; ++s) d = fminf(d, fabsf(fabsf(w[e]) - mid[s]));
                    if (!(d > delta)) hits |= 1u << e;
                }
                float ac[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) ac[i] = hand[(ROW_CUT + i) * GROUPS + g3];
                float* copy = hand + ROWS * GROUPS + lane;  // (by way of shared memory: registers have no index)
#pragma unroll
                for (int e = 0; e < PART; ++e) copy[e * 32] = w[e];
#pragma unroll 1
                for (; hits != 0u; hits &= hits - 1u) {
                    const int e = __ffs(hits) - 1;
                    const uint32_t code = nearest_code<Q>((double)copy[e * 32], ac);
#pragma unroll
                    for (int i = 0; i < Q; ++i) now[i] = (now[i] & ~(1u << e)) | ((~(code >> i) & 1u) << e);
                }
            }
            const bool live = pass * TEAMS + lane / L < count;
            if (p.sq_err != nullptr) {
#pragma unroll
                for (int k = 0; k < PART / LEAF; ++k) {
                    double sum = 0.0;
#pragma unroll
                    for (int e = k * LEAF; e < (k + 1) * LEAF; ++e) {
                        double wh = 0.0;
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            const double ai = (double)hand[(ROW_A + i) * GROUPS + g3];
                            wh = ((now[i] >> e) & 1u) ? wh - ai : wh + ai;
                        }
                        const double d = kt + 4 * PART * part + 16 * (e / 4) + e % 4 < at.m ? (double)w[e] - wh : 0.0;
                        sum += d * d;
                    }
#pragma unroll
                    for (int h = 0; h < PARTS; ++h)
                        if (h == part) leaf[h * (PART / LEAF) + k] = sum;
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) neg[i] = part == PARTS - 1 ? now[i] : (neg[i] << (PART & 31)) | now[i];
            if (part > 0) continue;
            const int wi = (tl >> 2) * (NI / 2) + (tl & 3);  // container word of the group this lane writes
            const bool writes = live && (tl & 3) < NI / 2 && 32 * wi < at.m;
            const uint32_t word_mask = at.m - 32 * wi >= 32 ? 0xFFFFFFFFu : (1u << ((at.m - 32 * wi) & 31)) - 1u;
            uint32_t* row = p.bits + (long long)at.j * p.pitch;
            uint32_t* dst = row + ((at.c * p.g) >> 5) + wi;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const uint32_t word = transpose_bits(~neg[i]);
                if (writes) dst[i * plane_words] = word & word_mask;
            }
            // zero padding words of the row, optional squared error
            if (at.c == p.G - 1 && live) {
                const int first_pad = (p.d_in + 31) >> 5;
                const int npad = p.pitch - first_pad;  // 0..3
#pragma unroll 1
                for (int e = tl; e < npad * Q; e += L) {
                    const int i = e / npad;
                    row[i * plane_words + first_pad + (e - i * npad)] = 0u;
                }
            }
            if (p.sq_err != nullptr) {
                double unused[1];
                const double E = lanes_sum<L, 1>(tree_of_leaves(leaf), unused);
                if (live && tl == 0) p.sq_err[(long long)at.j * p.G + at.c] = E;
            }
            at = next;
        }
    }
    __syncwarp();
    if (lane < count && !(fabsf(a[0]) <= 3.402823466e38f)) fit_not_finite(p, item);
}

// Groups to a warp: as few as fill the chip once (a warp goes through (1) and (3) 32 / L groups at a time, so a
// small problem is over sooner with fewer), at most the 32 that (2) has lanes for (1600 x 1600, q = 2, g = 128: 26 us with 650
// warps of 32 groups, 20 with 1300 of 16).  Four warps to a block in lockstep where there are three waves of them: they
// share what they fetch of the code (5120 x 5120, g = 128, with warps on their own: q = 3 186 us and 183, q = 4 415 and 381).
template <int NI, int L, int Q>
cudaError_t launch_sorted(const QuantParams& p, cudaStream_t stream) {
    using Sh = SortedShape<NI, L>;
    const long long places = kSortPlaces * bcq::sm_count();
    int batch = std::max(Sh::TEAMS, 4);
    while (batch < Sh::GROUPS && (p.items + batch - 1) / batch > places) batch *= 2;
    void (*kern)(const QuantParams, int) = sorted_quantize_kernel<NI, L, Q, false, false>;
    if constexpr (NI == 8 && Q < 4)  // (q = 4: no difference, the rounds are most of the time)
        if (p.g < Sh::C && p.vec) kern = sorted_quantize_kernel<NI, L, Q, true, false>;
    if constexpr (Q > 2)  // (q = 2 has one cut)
        if (batch <= 8) kern = sorted_quantize_kernel<NI, L, Q, false, true>;
    const bcq_status st = bcq::ensure_dynamic_smem(kern, kSortWarps * Sh::bytes);
    if (st != BCQ_OK) return cudaErrorUnknown;
    const long long warps = (p.items + batch - 1) / batch;
    const int per_block = warps >= 24ll * bcq::sm_count() ? kSortWarps : 1;
    return bcq::launch_pdl(kern, dim3((unsigned)((warps + per_block - 1) / per_block)), 32 * per_block, per_block * Sh::bytes, stream, 1, p, batch);
}

void set_row_items(QuantParams& p, int n) {
    p.row_items = n;
    p.g_magic = 0; p.g_shift = 0;
    if (n > 1 && p.items < (1ll << 31)) {
        // ceil(2^(32 + s) / n) with 2^s < n <= 2^(s+1): exact for every item below 2^31
        int sh = 0;
        while ((2ll << sh) < n) ++sh;
        p.g_shift = (uint32_t)sh;
        p.g_magic = (uint32_t)(((1ull << (32 + sh)) + n - 1) / n);
    }
}

template <int NI, int L, int TW, int Q>
cudaError_t launch_team(QuantParams p, cudaStream_t stream) {
    constexpr int TEAMS = TW == 1 ? 128 / L : 1;
    const int threads = TW == 1 ? 128 : TW * 32;
    const dim3 blocks((unsigned)((p.items + TEAMS - 1) / TEAMS));
    if constexpr (Q == 0 && TW == 1)
        if (p.d_in % p.g != 0) {
            set_row_items(p, p.d_in / p.g);
            return bcq::launch_pdl(team_quantize_kernel<NI, L, TW, Q, true>, blocks, threads, 0, stream, 1, p);
        }
    return bcq::launch_pdl(team_quantize_kernel<NI, L, TW, Q, false>, blocks, threads, 0, stream, 1, p);
}

// Greedy: the smallest team that holds a group at 32 weights a thread (8 or 16 for groups of 32 or 64).
// Alternating: a thread goes through its weights one after the other in every round, so a problem that
// is over in a few waves takes as long as one thread does, and fewer weights a thread are better;
// more lanes mean more shuffles and more copies of the solve, which a long one pays for.  Measured, us a call:
//   g = 128, two rounds, 8 / 16 weights a thread (groups of q > 1 come here with one or two rounds, see below)
//     q = 1   64 x 512 2.3 / 2.4   512 x 512 3.2 / 2.8    1600 x 1600 10.4 / 9.2    5120 x 5120 77.6 / 57.3
//     q = 2   64 x 512 3.6 / 4.3   1024 x 1024 8.7 / 9.2    1600 x 1600 17.7 / 15.6   5120 x 5120 143 / 106
//     q = 3   512 x 512 9.2 / 9.8   1024 x 1024 14.5 / 15.7   1600 x 1600 29.8 / 24.9   5120 x 5120 249 / 190
//     q = 4   512 x 512 12.1 / 15.9   1024 x 1024 22.5 / 24.6   1600 x 1600 52.4 / 43.1   5120 x 5120 458 / 318
//   g = 256, two rounds, 16 / 32 weights a thread (g = 512 is alike)
//     q = 2   1600 x 1600 16.3 / 17.9   2560 x 2560 30.7 / 29.7   3200 x 3072 43.7 / 40.6   5120 x 5120 108 / 94.4
//     q = 3   512 x 512 10.4 / 15.1   2048 x 2048 35.0 / 35.4   2560 x 2560 52.6 / 50.6   3200 x 3072 73.9 / 67.2   5120 x 5120 187 / 160
//     q = 4   2048 x 2048 58.8 / 57.8   3200 x 3072 125 / 113   5120 x 5120 315 / 282
//     q = 1, five rounds   3200 x 3072 36.1 / 36.8   4096 x 4096 60.4 / 60.9   5120 x 5120 87.7 / 82.5
//   a row, five rounds, 16 / 32 weights a thread
//     q = 3   1024 x 1024 30.8 / 35.7   2000 x 1024 44.0 / 48.9   3000 x 1024 59.0 / 57.2   1500 x 2048 63.2 / 60.0   4000 x 2048 142 / 116
//     q = 4   2000 x 1024 72.2 / 79.8   3000 x 1024 102 / 101   1024 x 2048 79.3 / 91.1   1500 x 2048 105 / 97.5
// The line between "few waves" and "long" is thus 18432 weights per SM for rows (2.7 M on 148), 49152 for groups of 129 to 512
// (7.3 M; with one plane 98304) and 8192 for groups of 65 to 128 (1.2 M; with one plane, whose rounds are short, 1024).
// From three rounds on groups of up to 256 go to the sorted kernel, with two planes groups of more than 128 from four on
// (g = 256, three rounds: 64 x 512 4.9 us here and 8.0 there, 1600 x 1600 20.2 / 28.3, 3200 x 3072 50.2 / 58.2, 5120 x 5120 119 / 125).  5120 x 5120, g = 128, q = 2 / 3 / 4: one round 82 / 139 / 218 us
// here and 100 / 129 / 189 there, two 107 / 192 / 320 and 105 / 140 / 210, three 132 / 239 / 413 and 109 / 146 / 231, five 178 / 331 / 599 and
// 118 / 167 / 278.  Small problems are chains of latencies in both, and there sorting costs: 1600 x 1600, three rounds
// 19 / 32 / 58 and 24 / 33 / 52; 512 x 512, five rounds 9.3 / 16.2 / 22.0 and 8.6 / 12.4 / 20.6; 64 x 512, three rounds 4.3 / 6.7 / 10.5 and
// 6.4 / 9.5 / 15.4.  They go there all the same: the choice may not depend on the number of rows, because the two kernels add in
// different orders and a row gets the same scales whatever else is in the call.
template <int Q>
cudaError_t launch_team_size(const QuantParams& p, cudaStream_t s) {
    const int g = p.g;
    const long long line = g > 512 ? 18432 : g > 128 ? (Q == 1 ? 98304 : 49152) : Q == 1 ? 1024 : 8192;  // weights per SM
    const bool few = Q > 0 && p.items * g <= line * bcq::sm_count();
    // (whatever the number of rows, see above)
    if constexpr (Q > 1)
        if (p.alt_iters >= (Q == 2 && g > 128 ? 4 : 3)) {
            if (g <= 32) return launch_sorted<2, 4, Q>(p, s);
            if (g <= 64) return launch_sorted<4, 4, Q>(p, s);
            // Groups of 65 to 128 in eight lanes, as long as warps of four groups find their places at once: half the weights to
            // sort in a lane (512 x 512, g = 128, three rounds, q = 2 / 3 / 4: 8.2 / 11.6 / 18.5 us in four lanes, 6.8 / 9.7 / 16.2 in eight;
            // 1024 x 1024 9.7 / 13.7 / 22.4 and 10.3 / 14.3 / 22.9; groups of 256 in sixteen 8.8 / 12.0 / 18.2 and 9.1 / 12.7 / 19.0)
            if (g <= 128) return p.items <= 4 * kSortPlaces * bcq::sm_count() ? launch_sorted<4, 8, Q>(p, s) : launch_sorted<8, 4, Q>(p, s);
            if (g <= 256) return launch_sorted<8, 8, Q>(p, s);
        }
    if (g <= 32) return launch_team<2, 4, 1, Q>(p, s);
    if (g <= 64) return launch_team<4, 4, 1, Q>(p, s);
    if constexpr (Q > 0) {
        if (g <= 128) return few ? launch_team<2, 16, 1, Q>(p, s) : launch_team<4, 8, 1, Q>(p, s);
        if (g <= 256) return few ? launch_team<4, 16, 1, Q>(p, s) : launch_team<8, 8, 1, Q>(p, s);
        if (g <= 512) return few ? launch_team<4, 32, 1, Q>(p, s) : launch_team<8, 16, 1, Q>(p, s);
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
    set_row_items(p, p.G);
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
