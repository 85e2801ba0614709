// Scale gradient of the BCQ linear layer (Eq. 4):
//     dalpha_i[j, c] = scale * sum_{k in group c} b_i[j,k] * (dY^T X)[j,k].
//
// D[j, k] = sum_t dY[t, j] X[t, k] is a 256 x 256 x 64 UMMA tile product of a CTA pair with both
// operands MN-major (tokens are the K index; dY and X rows are contiguous in j and k), loaded by TMA
// in 64 x 64 boxes.  A pair, because operand traffic bounds this kernel: per 512 tensor-core cycles a
// 128 x 256 tile of a CTA alone takes 48 KiB into shared memory and reads 48 KiB back, 192 bytes a
// cycle against the 128 of shared memory; in a pair each CTA holds half of the columns, 128 bytes a
// cycle.  Measured, CTA alone and pair: 1600 -> 6400 with 4096 tokens 75.5 and 68.5 us, 5120 -> 20480
// with 2048 tokens 326 and 276 us (1558 TFLOP/s).  The epilogue never writes D: thread = (row j, half of
// the tile's columns) reads its accumulator row from tensor memory 32 columns at a time, applies the signs of every
// requested plane from one 32-bit word of the packed planes, and sums per group.  Partial sums
// (one per split over tokens, column sub-tile and group piece) go to the workspace and a second
// kernel adds them in a fixed order, so the result does not depend on scheduling.  When every
// output has exactly one partial (no token split and a group per column sub-tile, e.g. g = 128)
// the epilogue writes dalpha itself and the second kernel is not launched.
#include <algorithm>

#include "gemm_common.cuh"

namespace {

using namespace bcq;

__device__ int g_timeout_flag = 0;

struct DalphaParams {
    int d_out, d_in, q, g, G, pitch, n;
    int num_kb;          // K blocks of 64 tokens
    int kb_per_split;
    int splits;
    int m_tiles, n_tiles;
    int n_subtiles;      // column sub-tiles of width kHN over d_in
    int slots;           // partial slots per sub-tile
    uint32_t planes;     // nibble k: the k-th plane of the mask
    int num_planes;
    const uint32_t* bits;
    float* partial;      // [splits][n_subtiles][q][slots][d_out]
    // direct != 0: every output has exactly one partial (no token split, one group per column
    // sub-tile), so the epilogue writes dalpha itself and no second kernel runs
    int direct, accumulate;
    float scale;
    float* dalpha;       // [q][d_out][G]
};


// ------------------------------------------------------------------------------------------
// dalpha: D[j, k] = sum_t dY[t, j] X[t, k], sign-weighted group sums in the epilogue
// ------------------------------------------------------------------------------------------

constexpr int kTN = 256;       // columns of a tile
constexpr int kHN = kTN / 2;   // of an epilogue sub-tile, and of the half of B that one CTA holds
constexpr int kTM = 2 * kBlockM;
constexpr int kStages = 6;
constexpr uint32_t kStageBytes = kABytes + kHN * kBlockK * 2;  // 32 KiB
// sign words of the epilogue's threads, [plane of the mask][thread][column chunk of 32]
constexpr uint32_t kSignBytes = (kHN / 32) * BCQ_MAX_Q * kWorkerWarps * 32 * 4;  // 32 KiB
static_assert(kHN == 128, "a sub-tile's sign words of a row are one 16-byte load");
constexpr size_t kDalphaSmem = (size_t)kStages * kStageBytes + 1024 + 256 + kSignBytes;
static_assert(kDalphaSmem <= 232448, "shared memory of a CTA");

// Persistent: every pair of CTAs walks over (row tile, column tile, token split) tiles; two
// accumulators in tensor memory, so the sign-and-sum epilogue of one tile runs under the main loop of
// the next.  In each CTA:
//   warp 0      TMA producer (its dY and X boxes of every K block of 64 tokens)
//   warp 1      owner of the tensor-memory allocation; in the leader, UMMA issuer for both
//   warps 2..9  epilogue: thread = (row j of this CTA's 128, half of the tile's columns)
// `full` and `acc_empty` are the leader's barriers; `empty` and `accum` exist in both CTAs and are
// signalled by one commit to both.
__global__ void __launch_bounds__(kThreads, 1)
dalpha_kernel(const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_x,
              const DalphaParams p) {
    constexpr int HN = kHN;
    constexpr int NCH = HN / 32;
    constexpr uint32_t kAccCols = kTN;
    constexpr uint32_t kTmemCols = 2 * kAccCols;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t ctl_base = smem_base + kStages * kStageBytes;
    uint8_t* ctl_gen = smem_gen + kStages * kStageBytes;

    Ctl ctl;
    ctl.full = ctl_base;
    ctl.aready = 0;
    ctl.empty = ctl_base + 8 * kStages;
    ctl.accum = ctl_base + 16 * kStages;        // + 8c : accumulator c complete
    const uint32_t acc_empty = ctl.accum + 16;  // + 8c : accumulator c drained by both CTAs
    ctl.spare = ctl.accum + 32;
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(ctl_gen + 16 * kStages + 40);
    ctl.abort_flag = reinterpret_cast<volatile int*>(ctl_gen + 16 * kStages + 44);
    ctl.device_flag = &g_timeout_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_rank();
    const int num_tiles = p.m_tiles * p.n_tiles * p.splits;
    const int pair0 = (int)blockIdx.x >> 1, num_pairs = (int)gridDim.x >> 1;
    // row tile fastest: pairs running together share the X boxes of a column tile in L2
    auto tile_coords = [&](int tile, int& j0, int& k0, int& z, int& kb_begin, int& iters) {
        const int mt = tile % p.m_tiles;
        const int rest = tile / p.m_tiles;
        j0 = mt * kTM + rank * kBlockM;
        k0 = (rest % p.n_tiles) * kTN;
        z = rest / p.n_tiles;
        kb_begin = z * p.kb_per_split;
        iters = min(p.num_kb, kb_begin + p.kb_per_split) - kb_begin;
    };
    // a column tile that reaches past d_in multiplies only the 64-column blocks that hold columns of
    // the matrix; half of them are in each CTA
    auto tile_width = [&](int k0) { return min(kTN, (p.d_in - k0 + 63) / 64 * 64); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(ctl.full + 8 * s, 1);
            ptx::mbar_init(ctl.empty + 8 * s, 1);
        }
        for (int c = 0; c < 2; ++c) {
            ptx::mbar_init(ctl.accum + 8 * c, 1);
            ptx::mbar_init(acc_empty + 8 * c, 2 * kWorkerWarps);
        }
        ptx::mbar_init(ctl.spare, 1);
        *ctl.abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&tmap_dy);
        ptx::prefetch_tmap(&tmap_x);
    }
    __syncwarp();
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t*>(tmem_holder)), kTmemCols);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();  // the peer's barriers exist
    ptx::tc_fence_after_sync();
    pdl_wait();
    const uint32_t tmem_base = *tmem_holder;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int tile = pair0; tile < num_tiles && ok; tile += num_pairs) {
                int j0, k0, z, kb_begin, iters;
                tile_coords(tile, j0, k0, z, kb_begin, iters);
                const int half = tile_width(k0) / 2;  // columns this CTA brings
                const int boxes = (half + 63) / 64;
                const int kx = k0 + rank * half;
                for (int it = 0; it < iters; ++it) {
                    ok = wait_bar(ctl.empty + 8 * s, ph ^ 1u, ctl, 11);
                    if (!ok) break;
                    const uint32_t sa = smem_base + s * kStageBytes;
                    const uint32_t bar = ptx::leader_addr(ctl.full + 8 * s);
                    const int tok = (kb_begin + it) * kBlockK;
                    if (rank == 0) ptx::mbar_arrive_expect_tx(ctl.full + 8 * s, 2u * (kABytes + (uint32_t)boxes * 8192u));
                    // A: two blocks of 64 rows j (inner) x 64 tokens; B: blocks of 64 k x 64 tokens
                    ptx::tma_load_2d_pair(sa, &tmap_dy, j0, tok, bar);
                    ptx::tma_load_2d_pair(sa + 8192, &tmap_dy, j0 + 64, tok, bar);
                    ptx::tma_load_2d_pair(sa + kABytes, &tmap_x, kx, tok, bar);
                    if (boxes > 1) ptx::tma_load_2d_pair(sa + kABytes + 8192, &tmap_x, kx + 64, tok, bar);
                    if (++s == kStages) { s = 0; ph ^= 1u; }
                }
            }
            // (no pdl_trigger here: the reduction's blocks would crowd onto the SMs that this kernel leaves
            // free, see launch_pdl; 1528 x 1000 at 777 tokens, four planes, 16.4 us with it and 13.7 without)
            // giving up: the copies in flight are counted on the leader's barriers, which may never
            // complete; they land within microseconds, so wait a thousand times as long
            if (!ok) for (int i = 0; i < 1000; ++i) __nanosleep(2000);
        }
        __syncwarp();
    } else if (warp == 1) {
        // One elected thread runs the whole loop: between two stages it has a barrier check, a
        // fence, four UMMAs and a commit to get through in less time than the tensor core needs
        // for a stage, so nothing warp-wide (election, reconvergence) is left inside the loop.
        if (rank == 0 && ptx::elect_one()) {
            bool ok = true;
            int s = 0, lt = 0;
            uint32_t ph = 0;
            // descriptor halves (128-byte swizzle, MN-major: leading offset 8192 B between blocks of 64
            // rows, stride 1024 B between groups of eight token lines); a UMMA steps the start by 2048 B
            constexpr uint32_t kHi = (1024u >> 4) | (1u << 14) | (2u << 29);
            constexpr uint32_t kLoExtra = (8192u >> 4) << 16;
            for (int tile = pair0; tile < num_tiles && ok; tile += num_pairs, ++lt) {
                int j0, k0, z, kb_begin, iters;
                tile_coords(tile, j0, k0, z, kb_begin, iters);
                const int acc = lt & 1;
                ok = wait_bar(acc_empty + 8 * acc, (uint32_t)((lt >> 1) & 1) ^ 1u, ctl, 17);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + (uint32_t)acc * kAccCols;
                const uint32_t idesc = ptx::make_idesc_bf16(kTM, tile_width(k0), 1, 1);
                for (int it = 0; it < iters; ++it) {
                    ok = wait_bar(ctl.full + 8 * s, ph, ctl, 13, 32u);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    const uint32_t a_lo = (((smem_base + (uint32_t)s * kStageBytes) >> 4) & 0x3FFFu) | kLoExtra;
                    const uint32_t b_lo = a_lo + (kABytes >> 4);
#pragma unroll
                    for (int kk = 0; kk < kBlockK / 16; ++kk)
                        ptx::umma_f16_pair(d_tmem, a_lo + kk * (2048u >> 4), kHi, b_lo + kk * (2048u >> 4), kHi, idesc,
                                           (it > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit_pair(ctl.empty + 8 * s);
                    if (++s == kStages) { s = 0; ph ^= 1u; }
                }
                if (ok) ptx::umma_commit_pair(ctl.accum + 8 * acc);
            }
            if (!ok) {
                ptx::umma_commit_pair(ctl.spare);
                wait_bar(ctl.spare, 0, ctl, 15);
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: thread = (row j, HN columns of the tile).  Loops over chunks and planes, not
        // unrolled: a CTA has one to three tiles, so the code runs from cold instruction caches, and the time is what
        // fetching it takes (written out for all planes and chunks, 50 KiB: the last epilogue of a call took 5.1 us with
        // one plane; 1024 x 1024, one plane, 64 tokens 8.3 us a call and 6.1 now, 2048 tokens 11.9 and 9.8)
        const int quarter = warp & 3;
        const int half = (warp - kWorkerWarp0) >> 2;
        const int et = (int)threadIdx.x - kWorkerWarp0 * 32;
        constexpr int ET = kWorkerWarps * 32;
        uint32_t* mine = reinterpret_cast<uint32_t*>(ctl_gen + 256) + 4 * et;  // this thread's; [plane][thread][chunk]
        const uint32_t words = ptx::smem_u32(mine);
        const long long plane_words = (long long)p.d_out * p.pitch;
        const int np = p.num_planes;
        bool ok = true;
        int lt = 0;
        for (int tile = pair0; tile < num_tiles && ok; tile += num_pairs, ++lt) {
            int j0, k0, z, kb_begin, iters;
            tile_coords(tile, j0, k0, z, kb_begin, iters);
            const int acc = lt & 1;
            const int j = j0 + quarter * 32 + lane;
            const bool j_ok = j < p.d_out;
            const int kbase = k0 + half * HN;
            const int subtile = (k0 / kTN) * 2 + half;

            // The sign words do not depend on the accumulator: they are on their way into shared memory while the main
            // loop runs, all planes' at once (a row's words of a sub-tile are 16 bytes, aligned).  Loaded plane after
            // plane through registers they were a chain of as many memory latencies, longer than a short main loop:
            // 1024 x 1024, 64 tokens, four planes 9.2 us and 8.0 so; 6400 -> 1600, eight planes 30.7 and 27.6.
            if (j_ok && kbase < p.d_in) {
#pragma unroll 1
                for (int i = 0; i < np; ++i)
                    ptx::cp_async_16(words + (uint32_t)i * (ET * 16), p.bits + (long long)((p.planes >> (4 * i)) & 15u) * plane_words +
                                                                          (long long)j * p.pitch + (kbase >> 5));
            }

            ok = wait_bar(ctl.accum + 8 * acc, (uint32_t)(lt >> 1) & 1u, ctl, 16, 512u);
            ptx::cp_async_wait_all();
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (kbase < p.d_in) {
                const int c_first = min(kbase / p.g, p.G - 1);
                int c = c_first, next_edge = c < p.G - 1 ? (c + 1) * p.g : p.d_in;  // first column of the next group
                bool fresh = true;
#pragma unroll 1
                for (int ch = 0; ch < NCH; ++ch) {
                    const int kg = kbase + ch * 32;
                    if (kg >= p.d_in) break;  // uniform in the warp
                    uint32_t v[32];
                    ptx::tmem_ld_x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * kAccCols +
                                         (uint32_t)(half * HN + ch * 32), v);
                    ptx::tmem_ld_wait();
                    const bool last = ch == NCH - 1 || kg + 32 >= next_edge;  // of this group in this sub-tile
#pragma unroll 1
                    for (int i = 0; i < np; ++i) {
                        uint32_t* so_far = mine + i * (4 * ET);
                        const uint32_t w = ~so_far[ch];
                        float sum = 0.0f;
#pragma unroll
                        for (int b = 0; b < 32; ++b)
                            sum += __uint_as_float(v[b] ^ ((w << (31 - b)) & 0x80000000u));
                        // the group's sum so far waits in place of the plane's first sign word, which is used up
                        if (!fresh) sum = __uint_as_float(*so_far) + sum;
                        if (!last) {
                            *so_far = __float_as_uint(sum);
                        } else if (j_ok) {
                            const int plane = (int)(p.planes >> (4 * i)) & 15;
                            if (p.direct) {
                                float* dst = p.dalpha + ((long long)plane * p.d_out + j) * p.G + c;
                                *dst = p.accumulate ? (*dst + p.scale * sum) : (p.scale * sum);
                            } else {
                                p.partial[((((long long)z * p.n_subtiles + subtile) * p.q + plane) * p.slots + (c - c_first)) * p.d_out + j] = sum;
                            }
                        }
                    }
                    fresh = last;
                    if (kg + 32 >= next_edge) {
                        ++c;
                        next_edge = c < p.G - 1 ? next_edge + p.g : p.d_in;
                    }
                }
            }
            // the accumulator may be overwritten by the tile after next
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::leader_addr(acc_empty + 8 * acc));
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();  // neither CTA's memory goes away under the other
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// dalpha[i][j][c] (+)= scale * sum over splits and over the sub-tiles that meet group c.
// Block = 32 consecutive rows j x 8 parts: part y adds every 8th partial of its output (so that
// eight loads per output are in flight at once), then the eight sums are added in order 0..7.  Nibble k of
// `planes` is the k-th plane of the mask.
__global__ void __launch_bounds__(256)
dalpha_reduce_kernel(int d_out, int d_in, int q, int g, int G, int HN, int splits, int n_subtiles, int slots,
                     uint32_t planes, float scale, int accumulate, const float* partial,
                     float* dalpha) {
    __shared__ float sums[8][32];
    pdl_trigger();
    pdl_wait();
    const int jx = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int jblocks = (d_out + 31) / 32;
    const int jb = blockIdx.x % jblocks;
    const int r = blockIdx.x / jblocks;  // (plane of the mask, group)
    const int c = r % G;
    const int i = (int)(planes >> (4 * (r / G))) & 15;
    const int j = jb * 32 + jx;
    const int k_lo = c * g;
    const int k_hi = min(k_lo + g, d_in) - 1;
    const int st_lo = k_lo / HN, st_n = k_hi / HN - st_lo + 1;
    const int total = splits * st_n;
    float s = 0.0f;
    if (j < d_out) {
        for (int e = part; e < total; e += 8) {
            const int z = e / st_n, st = st_lo + (e - z * st_n);
            const int slot = c - min((st * HN) / g, G - 1);
            s += ld(partial + ((((long long)z * n_subtiles + st) * q + i) * slots + slot) * d_out + j);
        }
    }
    sums[part][jx] = s;
    __syncthreads();
    if (part == 0 && j < d_out) {
        float t = 0.0f;
#pragma unroll
        for (int y = 0; y < 8; ++y) t += sums[y][jx];
        float* dst = dalpha + ((long long)i * d_out + j) * G + c;
        *dst = accumulate ? (*dst + scale * t) : (scale * t);
    }
}

struct DalphaPlan {
    int splits, kb_per_split, num_kb, m_tiles, n_tiles, n_subtiles, slots;
};

DalphaPlan plan_dalpha(int d_out, int d_in, int g, int n) {
    DalphaPlan pl;
    const int pairs = std::max(1, sm_count() / 2);
    pl.m_tiles = ceil_div(d_out, kTM);
    pl.num_kb = ceil_div(n, kBlockK);
    pl.n_tiles = ceil_div(d_in, kTN);
    pl.n_subtiles = pl.n_tiles * 2;
    if (g % kHN == 0) pl.slots = 1;
    else if (kHN % g == 0) pl.slots = kHN / g;
    else pl.slots = kHN / g + 2;
    const int tiles = pl.m_tiles * pl.n_tiles;
    int splits = pairs / tiles;
    if (splits < 1) splits = 1;
    const int max_splits = (pl.num_kb + 3) / 4;
    if (splits > max_splits) splits = max_splits;
    if (splits > 32) splits = 32;
    pl.kb_per_split = ceil_div(pl.num_kb, splits);
    pl.splits = ceil_div(pl.num_kb, pl.kb_per_split);
    return pl;
}


size_t dalpha_ws_bytes(const DalphaPlan& pl, int d_out, int q) {
    return (size_t)pl.splits * pl.n_subtiles * q * pl.slots * d_out * sizeof(float);
}

}  // namespace

namespace bcq {
bcq_status dalpha_timeout_flag(int* flag_out, int reset) {
    int v = 0;
    BCQ_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_timeout_flag, sizeof(int)));
    *flag_out = v;
    if (reset && v != 0) {
        const int zero = 0;
        BCQ_CUDA_TRY(cudaMemcpyToSymbol(g_timeout_flag, &zero, sizeof(int)));
    }
    return BCQ_OK;
}

size_t bwd_alpha_workspace_bytes(int d_out, int d_in, int q, int g, int n) {
    return dalpha_ws_bytes(plan_dalpha(d_out, d_in, g, n), d_out, q);
}
}  // namespace bcq

extern "C" bcq_status bcq_linear_bwd_alpha(int d_out, int d_in, int q, int g, int n, const void* dY,
                                           size_t lddy, const void* X, size_t ldx, const uint32_t* bits,
                                           uint32_t plane_mask, float scale, int accumulate,
                                           float* dalpha, void* ws, size_t ws_bytes, void* stream) {
    bcq_status st = check_shape(d_out, d_in, q, g);
    if (st != BCQ_OK) return st;
    if (n < 1) return BCQ_ERR_SHAPE;
    if (!bits || !dalpha) return BCQ_ERR_NULL;
    if ((st = check_act(dY, lddy, d_out)) != BCQ_OK) return st;
    if ((st = check_act(X, ldx, d_in)) != BCQ_OK) return st;
    if (!aligned16(bits)) return BCQ_ERR_ALIGN;
    plane_mask &= (1u << q) - 1u;
    if (plane_mask == 0) return BCQ_OK;
    const DalphaPlan pl = plan_dalpha(d_out, d_in, g, n);
    const size_t need = dalpha_ws_bytes(pl, d_out, q);
    if (ws == nullptr) return BCQ_ERR_NULL;
    if (ws_bytes < need) return BCQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return BCQ_ERR_ALIGN;

    CUtensorMap tm_dy, tm_x;
    if ((st = make_tmap_16bit(&tm_dy, dY, 0, d_out, n, lddy, 64)) != BCQ_OK) return st;
    if ((st = make_tmap_16bit(&tm_x, X, 0, d_in, n, ldx, 64)) != BCQ_OK) return st;
    DalphaParams p;
    p.d_out = d_out; p.d_in = d_in; p.q = q; p.g = g;
    p.G = (int)bcq_num_groups(d_in, g);
    p.pitch = (int)bcq_pitch_words(d_in);
    p.n = n; p.num_kb = pl.num_kb; p.kb_per_split = pl.kb_per_split; p.splits = pl.splits;
    p.m_tiles = pl.m_tiles; p.n_tiles = pl.n_tiles;
    p.n_subtiles = pl.n_subtiles; p.slots = pl.slots;
    p.planes = 0; p.num_planes = 0;
    for (int i = 0; i < q; ++i)
        if ((plane_mask >> i) & 1u) p.planes |= (uint32_t)i << (4 * p.num_planes++);
    p.bits = bits; p.partial = reinterpret_cast<float*>(ws);
    p.direct = (pl.splits == 1 && g == kHN) ? 1 : 0;
    p.accumulate = accumulate; p.scale = scale; p.dalpha = dalpha;
    cudaStream_t s = (cudaStream_t)stream;
    // persistent, one CTA per SM; every pair gets the same number of tiles (as many as the busiest
    // would get anyway), which leaves whole SMs to other kernels instead of a ragged last wave
    const int tiles = pl.m_tiles * pl.n_tiles * pl.splits;
    const int per_pair = ceil_div(tiles, std::max(1, sm_count() / 2));
    if ((st = ensure_dynamic_smem(dalpha_kernel, kDalphaSmem)) != BCQ_OK) return st;
    BCQ_CUDA_TRY(launch_pdl(dalpha_kernel, dim3(2u * (unsigned)ceil_div(tiles, per_pair)), kThreads, kDalphaSmem, s, 2, tm_dy, tm_x, p));
    if (p.direct) return BCQ_OK;
    // (only blocks of planes in the mask: the others would wait for this kernel and leave.  q = 8, one plane,
    // 5120 x 5120, g = 64, 64 tokens: 143 us with them, 52 without)
    const long long rblocks = (long long)p.num_planes * p.G * ((d_out + 31) / 32);
    BCQ_CUDA_TRY(launch_pdl(dalpha_reduce_kernel, dim3((unsigned)rblocks), 256, 0, s, 1, d_out, d_in, q, g, p.G, kHN, pl.splits,
                            pl.n_subtiles, pl.slots, p.planes, scale, accumulate, (const float*)p.partial, dalpha));
    return BCQ_OK;
}
