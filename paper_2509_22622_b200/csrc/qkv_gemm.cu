// QKV projection with the path's front end in its epilogue (sm_100a):
//
//   y = x W^T + b          x [n_tokens, d_model] bf16, W [3*H*D, d_model] bf16, fp32 accumulation
//   q | k | v = y          (the rows of W are the q features, then k, then v)
//   q, k: optional RMS norm over the token's whole row of H*D elements with a learned gain,
//         then the 3-D rotation;  rotated q -> q_out, rotated k and raw v -> the cache rows.
//
// The GEMM is a persistent tcgen05 kernel on pairs of CTAs (cta_group::2): a pair works on 256
// tokens x TN output features, each CTA holding 128 tokens' rows of x and half of the W tile's rows in
// its shared memory and the accumulators of its own 128 tokens in its tensor memory, so an operand
// byte fetched from L2 is used for 256 rows (or TN columns) instead of 128.  K blocks of 64 go
// through a TMA ring in each CTA that reports to the leader's barriers; accumulators are
// double-buffered (2 x TN columns) so that the epilogue of a tile runs under the main loop of
// the next.  Warp 0 (one lane): TMA producer.  Warp 1 of the leader (one elected lane): MMA issuer for the
// pair.  Warps 4-19: epilogue, a warp = 16 token rows of half the features, 32 at a time in the 16x256b
// TMEM shape: a register pair is one rotation pair, four threads share a row, so the (cos, sin) pairs
// of a load lie in 8 sectors instead of 32 (one row per thread), and 16-bit rows go out through
// shared memory in 64-byte pieces.
//   What bounds it (4680 tokens, 1536 -> 3 x 1536, norm): the MMAs alone take 46 us of the 57 us at
// the clock this load gets (1.7 GHz; 342 tiles on 74 pairs are 5 rounds where 4.6 would do), the operands
// from L2 add 1 us, the epilogue's stores and the last round's epilogue the rest.  With one
// 128 x 192 tile per CTA and one row per epilogue thread it was 72 us: 107 B/clk and SM of operands, and
// scattered epilogue accesses that kept the L1 63 % busy.  Eight instead of sixteen epilogue
// warps: 64 us; features instead of tokens running fastest over the tiles: 61 us.
//   TN is 256, 192 or 128, whichever leaves the pairs less idle in the last round of tiles.
//
// The norm needs the sum of squares of a token's whole q (or k) row, which is spread over
// H*D/TN tiles that run on different SMs at different times.  The factor is one scalar per
// token and everything after it is linear, so a tile stores rotate(gain * y) without it and
// leaves its part of the sum of squares in a table (one slot per token and warp: no atomics,
// the sum is taken in a fixed order).  For q the scalar then travels with q_out to the
// attention call as a per-row softmax scale; for k a small second kernel applies it: the
// epilogue parks the un-normalised rotated k rows in fp32 in the caller's workspace and the
// second kernel scales, rounds once to bf16 and writes the cache rows.
#include <cuda_bf16.h>

#include "bounded_wait.cuh"
#include "ll_internal.h"
#include "ptx.cuh"

namespace ll {

namespace {

using namespace ptx;

constexpr int kTileM = 256, kBlockK = 64;              // tokens of a pair's tile
constexpr int kABytes = 128 * kBlockK * 2;             // a CTA's half of the tokens: 16 KB

template <int TN>
struct GemmCfg {
    static_assert(TN == 256 || TN == 192 || TN == 128, "tile widths built");
    // epilogue warps: 16 rows of half the features each, or of all 128 (the table of the sums of squares has
    // room for one slot per 96 features)
    static constexpr int kEpiWarps = TN == 128 ? 8 : 16;
    static constexpr int kEpiCols = TN == 128 ? 128 : TN / 2;
    static constexpr int kThreads = 128 + 32 * kEpiWarps;  // TMA, MMA, two idle warps, epilogue
    static constexpr int kStages = TN == 128 ? 7 : 6;
    static constexpr int kBBytes = TN / 2 * kBlockK * 2;   // a CTA's half of the features
    static constexpr int kStageBytes = kABytes + kBBytes;  // per CTA
    static constexpr int kStaging = kStages * kStageBytes; // 16 rows x 64 bytes per epilogue warp
    static constexpr int kBarOff = kStaging + kEpiWarps * 1024;
    static constexpr int kSmem = kBarOff + 1024 /*barriers*/ + 1024 /*alignment*/;
    // barrier indices: full and acc-empty are the leader's, empty and acc-full each CTA's own, start the other CTA's
    static constexpr int kFull = 0, kEmpty = kStages, kAccFull = 2 * kStages, kAccEmpty = 2 * kStages + 2, kStart = 2 * kStages + 4,
                         kBars = 2 * kStages + 5;
};

// ---- pairs of CTAs ----
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// 3-D tiled load into this CTA's shared memory, bytes counted on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *m, uint32_t cluster_bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(cluster_bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// D[both CTAs' tmem] (+)= A B over the pair; issued by one thread of the leader.
__device__ __forceinline__ void mma_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The barrier at this offset in both CTAs arrives once the pair's tcgen05 operations issued so far are done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}

// What an epilogue thread knows about one of its two token rows.
struct EpiRow {
    bool live;
    int token;
    size_t cache_row;
    const float2 *t_row, *h_row, *w_row;
    __device__ EpiRow(const QkvParams &p, int tok, int n_t, int n_h) : live(tok < p.n_tokens), token(live ? tok : 0)
    {
        const int frame = token / p.P, cell = token - frame * p.P, y = cell / p.grid_w;
        cache_row = (size_t)p.slot[frame] * p.P + cell;
        t_row = p.t_tab + (size_t)frame * n_t;
        h_row = p.h_tab + (size_t)y * n_h;
        w_row = p.w_tab + (size_t)(cell - y * p.grid_w) * n_h;
    }
    // (cos, sin) of rotation pair j of a head row
    template <int kNt, int kNh>
    __device__ float2 turn(int j) const { return *(j < kNt ? t_row + j : j < kNt + kNh ? h_row + (j - kNt) : w_row + (j - kNt - kNh)); }
};

// A warp's 16 rows x COLS features of the accumulator tile, 32 features at a time: bias, sum of squares,
// gain, rotation, stores.  A thread holds rows lane / 4 and lane / 4 + 8, of every 8 features the pair
// 2 (lane % 4).  Returns its two rows' sums of squares (complete in all four threads of a row).
template <int D, int COLS>
__device__ __forceinline__ float2 epilogue_rows(const QkvParams &p, uint32_t taddr, int token0, int n0, int lane, uint32_t staging)
{
    constexpr int kNh = D / 6, kNt = D / 2 - 2 * kNh;  // pairs of the h (= w) and t bands
    const int HD = p.heads * D, which = n0 / HD, c0 = n0 - which * HD;      // 0 q, 1 k, 2 v: a tile never straddles them
    const EpiRow ra(p, token0 + (lane >> 2), kNt, kNh), rb(p, token0 + (lane >> 2) + 8, kNt, kNh);
    const bool park = which == 1 && p.with_norm;       // k under the norm: fp32, finished by the second kernel
    const float *gain = which == 0 ? p.gain_q : p.gain_k;
    const int cq = 2 * (lane & 3);
    // staging: row r at 64 r, its 16-byte chunk k at position k ^ (r / 2 % 4); lane 8 m + r stores row r of chunk m
    const uint32_t st_at = staging + (uint32_t)(lane & 7) * 64 + ((uint32_t)((lane >> 3) ^ ((lane & 7) >> 1)) << 4);
    const int out_r = lane >> 2, out_k = lane & 3;
    const uint32_t ld_at = staging + (uint32_t)out_r * 64 + ((uint32_t)(out_k ^ ((out_r >> 1) & 3)) << 4);
    // the rows this thread writes 16 bytes of: out_r and out_r + 8, i.e. its own two rows
    float ssq_a = 0.f, ssq_b = 0.f;
#pragma unroll 1
    for (int ch = 0; ch < COLS / 32; ++ch) {
        const int cw = c0 + 32 * ch, head = cw / D, d0 = cw - head * D;     // first feature inside q, k or v; inside its head
        uint32_t r[16];
        tmem_ld_16x256b_x4(taddr + 32 * ch, r);
        float2 ca[4], cb[4];
        if (which < 2) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = d0 / 2 + 4 * k + (lane & 3);
                ca[k] = ra.turn<kNt, kNh>(j);
                cb[k] = rb.turn<kNt, kNh>(j);
            }
        }
        float2 bias[4], gg[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            bias[k] = p.bias ? *reinterpret_cast<const float2 *>(p.bias + n0 + 32 * ch + 8 * k + cq) : make_float2(0.f, 0.f);
            gg[k] = which < 2 && p.with_norm ? *reinterpret_cast<const float2 *>(gain + cw + 8 * k + cq) : make_float2(1.f, 1.f);
        }
        tmem_wait_ld();
        float2 va[4], vb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            va[k] = make_float2(__uint_as_float(r[4 * k]) + bias[k].x, __uint_as_float(r[4 * k + 1]) + bias[k].y);
            vb[k] = make_float2(__uint_as_float(r[4 * k + 2]) + bias[k].x, __uint_as_float(r[4 * k + 3]) + bias[k].y);
        }
        if (which < 2) {
            auto turn = [](float2 v, float2 g, float2 cs) {
                const float a = v.x * g.x, b = v.y * g.y;
                return make_float2(fmaf(a, cs.x, -(b * cs.y)), fmaf(a, cs.y, b * cs.x));
            };
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ssq_a = fmaf(va[k].y, va[k].y, fmaf(va[k].x, va[k].x, ssq_a));
                ssq_b = fmaf(vb[k].y, vb[k].y, fmaf(vb[k].x, vb[k].x, ssq_b));
                va[k] = turn(va[k], gg[k], ca[k]);
                vb[k] = turn(vb[k], gg[k], cb[k]);
            }
        }
        if (park) {
            float2 *da = reinterpret_cast<float2 *>(p.k_park + (size_t)ra.token * HD + cw + cq);
            float2 *db = reinterpret_cast<float2 *>(p.k_park + (size_t)rb.token * HD + cw + cq);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (ra.live) da[4 * k] = va[k];
                if (rb.live) db[4 * k] = vb[k];
            }
            continue;
        }
        stmatrix_x4(st_at, cvt_bf16x2(va[0].x, va[0].y), cvt_bf16x2(va[1].x, va[1].y), cvt_bf16x2(va[2].x, va[2].y), cvt_bf16x2(va[3].x, va[3].y));
        stmatrix_x4(st_at + 512, cvt_bf16x2(vb[0].x, vb[0].y), cvt_bf16x2(vb[1].x, vb[1].y), cvt_bf16x2(vb[2].x, vb[2].y), cvt_bf16x2(vb[3].x, vb[3].y));
        __syncwarp();
        const uint4 xa = ld_shared_v4(ld_at), xb = ld_shared_v4(ld_at + 512);
        auto row_of = [&](const EpiRow &e) -> ll_bf16 * {
            if (which == 0) return p.q_out + ((size_t)e.token * p.heads + head) * D + d0;
            return (which == 1 ? p.kcache : p.vcache) + ((size_t)head * p.rows_per_head + e.cache_row) * D + d0;
        };
        if (ra.live) *reinterpret_cast<uint4 *>(row_of(ra) + 8 * out_k) = xa;
        if (rb.live) *reinterpret_cast<uint4 *>(row_of(rb) + 8 * out_k) = xb;
        __syncwarp();                                  // the staging rows are read before the next 32 features
    }
#pragma unroll
    for (int m = 1; m < 4; m <<= 1) {
        ssq_a += __shfl_xor_sync(0xffffffffu, ssq_a, m);
        ssq_b += __shfl_xor_sync(0xffffffffu, ssq_b, m);
    }
    return make_float2(ssq_a, ssq_b);
}

template <int D, int TN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GemmCfg<TN>::kThreads, 1)
qkv_gemm_kernel(const __grid_constant__ QkvParams p, const __grid_constant__ CUtensorMap xmap,
                const __grid_constant__ CUtensorMap wmap)
{
    using G = GemmCfg<TN>;
    constexpr int kStages = G::kStages, kStageBytes = G::kStageBytes;
    constexpr int kFull = G::kFull, kEmpty = G::kEmpty, kAccFull = G::kAccFull, kAccEmpty = G::kAccEmpty, kStart = G::kStart;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t bars = smem_base + G::kBarOff;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + G::kBarOff + G::kBars * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile uint32_t *verdict = tmem_slot + 2;        // the leader's look at the status word: 1 the pair starts, 2 it does not
    auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();              // 0: the leader, whose barriers and issuer serve the pair
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

    grid_dep_launch();
    if (threadIdx.x == 0) {
        for (int i = 0; i < G::kBars; ++i) mbar_init(bar(i), (i >= kAccEmpty && i < kStart) ? 2u * G::kEpiWarps : 1u);   // both CTAs' epilogue warps free a buffer
        *abort_flag = 0;
        *verdict = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {                      // (the maps are launch parameters)
        prefetch_tensormap(&xmap);
        prefetch_tensormap(&wmap);
    }
    tc_fence_before_sync();
    __syncwarp();
    cluster_sync();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    WaitCtx ctx{abort_flag, p.status, warp};
    grid_dep_wait();
    // An earlier kernel gave up on a wait: the pair does not start (flag value 2).  The leader's look at the status word decides for both
    // CTAs.  The load warps do not wait to hear of it: their first tiles are under way meanwhile, and they find the flag when they run out
    // of stages.  (In front of the first load stood the read of the status word, the pair's barrier and a look at the leader's flag:
    // 270 tokens, 256 -> 3 x 1536 with norm 13.3 -> 12.7 us; 312 tokens, 1024 -> 3 x 192 15.2 -> 14.6; 200 tokens, 2048 -> 3 x 5120
    // 33.3 -> 32.6.)
    if (warp == 2) {                                   // (which has nothing else to do)
        if (rank == 1) {
            wait_bar<true>(bar(kStart), 0, ctx, kStart, 0);
        } else if (lane == 0) {
            *verdict = *reinterpret_cast<volatile uint32_t *>(p.status) != kStatusOk ? 2u : 1u;
            st_shared_remote(smem_u32(tmem_slot + 2), 1, *verdict);
            mbar_arrive_remote(bar(kStart), 1);
        }
        if (lane == 0 && *verdict != 1u && *abort_flag == 0) *abort_flag = 2;
        __syncwarp();
    }
    if (warp != 0) named_sync(1, G::kThreads - 32);
    const bool skip = warp != 0 && *verdict != 1u;
    auto wait = [&](int bar_id, uint32_t parity, int iter) -> bool {
        return wait_bar(bar(bar_id), parity & 1u, ctx, bar_id, iter);
    };
    const int n_kb = (p.d_model + kBlockK - 1) / kBlockK;
    const int n_tiles = p.m_tiles * p.n_tiles;

    if (skip) {
        // an earlier kernel gave up on a wait: nothing to do
    } else if (warp == 0 && lane == 0) {
        // ---- TMA producer (each CTA its own halves): tiles in the order all roles walk them; tokens
        // run fastest, so that the last round, whose epilogue nothing hides, is of v: no norm, no rotation ----
        uint32_t n = 0;
        for (int tile = pair; tile < n_tiles; tile += n_pairs) {
            const int m0 = (tile % p.m_tiles) * kTileM + 128 * (int)rank, n0 = (tile / p.m_tiles) * TN + TN / 2 * (int)rank;
            for (int kb = 0; kb < n_kb; ++kb, ++n) {
                const int stage = n % kStages;
                if (!wait(kEmpty + stage, (n / kStages) ^ 1u, (int)n)) goto done;
                if (rank == 0) mbar_arrive_expect_tx(bar(kFull + stage), 2 * kStageBytes);
                const uint32_t a = smem_base + stage * kStageBytes, full = map_to_rank(bar(kFull + stage), 0);
                tma_load_3d_pair(a, &xmap, full, kb * kBlockK, m0, 0);
                tma_load_3d_pair(a + kABytes, &wmap, full, kb * kBlockK, n0, 0);
            }
        }
    } else if (warp == 1 && rank == 0) {
        // ---- MMA issuer of the pair ----
        const bool elected = elect_one();
        constexpr uint32_t idesc = idesc_bf16_f32(kTileM, TN, 0, 0);
        constexpr uint32_t hi = smem_desc_hi_sw128(1024);
        uint32_t n = 0, t = 0;
        for (int tile = pair; tile < n_tiles; tile += n_pairs, ++t) {
            const uint32_t buf = t & 1u;
            // both epilogues have read this accumulator buffer out (two tiles ago)
            if (t >= 2 && !wait(kAccEmpty + buf, (t >> 1) - 1, (int)t)) goto done;
            tc_fence_after_sync();
            for (int kb = 0; kb < n_kb; ++kb, ++n) {
                const int stage = n % kStages;
                if (!wait(kFull + stage, n / kStages, (int)n)) goto done;
                tc_fence_after_sync();
                if (elected) {
                    const uint32_t a_lo = smem_desc_lo(smem_base + stage * kStageBytes, 16);
                    const uint32_t b_lo = smem_desc_lo(smem_base + stage * kStageBytes + kABytes, 16);
#pragma unroll
                    for (int kk = 0; kk < kBlockK / 16; ++kk)
                        mma_ss_pair(tmem + buf * TN, smem_desc_join(a_lo + ((kk * 32) >> 4), hi),
                                    smem_desc_join(b_lo + ((kk * 32) >> 4), hi), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                    tc_commit_pair(bar(kEmpty + stage));
                    if (kb == n_kb - 1) tc_commit_pair(bar(kAccFull + buf));
                }
                __syncwarp();
            }
        }
    } else if (warp >= 4) {
        // ---- epilogue: warp = 16 token rows x kEpiCols features ----
        constexpr int kCols = G::kEpiCols;
        const int e = warp - 4, row0 = 32 * (warp & 3) + 16 * ((e >> 2) & 1), col0 = kCols * (e >> 3);
        const uint32_t staging = smem_base + G::kStaging + (uint32_t)e * 1024;
        const uint32_t acc_empty = map_to_rank(bar(kAccEmpty), 0);
        uint32_t t = 0;
        for (int tile = pair; tile < n_tiles; tile += n_pairs, ++t) {
            const uint32_t buf = t & 1u;
            const int m0 = (tile % p.m_tiles) * kTileM + 128 * (int)rank, n0 = (tile / p.m_tiles) * TN + col0;
            if (!__all_sync(0xffffffffu, wait(kAccFull + buf, t >> 1, (int)t))) goto done;
            tc_fence_after_sync();
            const float2 ssq = epilogue_rows<D, kCols>(p, tmem + buf * TN + col0 + ((uint32_t)row0 << 16), m0 + row0, n0, lane, staging);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty + 8u * buf);
            // the warp's part of the rows' sums of squares: one slot per token and kCols features
            const int HD = p.heads * D, which = n0 / HD, token = m0 + row0 + (lane >> 2);
            if (p.with_norm && which < 2 && (lane & 3) == 0) {
                float *dst = p.ssq + ((size_t)which * p.n_tokens + token) * p.ssq_slots + (n0 - which * HD) / kCols;
                if (token < p.n_tokens) dst[0] = ssq.x;
                if (token + 8 < p.n_tokens) dst[(size_t)8 * p.ssq_slots] = ssq.y;
            }
        }
    }
done:
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag != 0) {
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    // neither CTA leaves while the other may still reach its barriers, its operands or its tensor memory
    __syncthreads();
    __syncwarp();
    cluster_sync();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// The norm's second step, one warp per token: the row factors from the sums of squares per tile
// (added in feature order), q's to q_row_scale, k's applied to the parked fp32 row, which is rounded
// once to bf16 into the cache row.  A lane takes kHeld 8-feature vectors at a time, all their loads in
// flight together and before the factor is known.
__global__ void __launch_bounds__(256)
qkv_finish_kernel(const __grid_constant__ QkvParams p)
{
    // (3, 4 and 6 are the same within what runs differ, 1 to 3 %: the projection with norm of 4680 tokens, widths 1536 / 2048 / 3072 / 5120,
    // 72.4 / 146.3 / 297.8 / 772.8 us with 3, 75.1 / 146.8 / 298.2 / 774.9 with 6)
    constexpr int kHeld = 3;
    const int token = (int)((blockIdx.x * 256u + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    grid_dep_launch();
    grid_dep_wait();
    if (token >= p.n_tokens) return;
    const int HD = p.heads * p.head_dim, vecs = HD / 8, per_head = p.head_dim / 8;
    const int frame = token / p.P, cell = token - frame * p.P;
    const float4 *src = reinterpret_cast<const float4 *>(p.k_park + (size_t)token * HD);
    ll_bf16 *dst = p.kcache + ((size_t)p.slot[frame] * p.P + cell) * p.head_dim;
    float rk = 0.f;
    for (int v0 = 0; v0 < vecs; v0 += 32 * kHeld) {
        float4 x[kHeld][2];
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int v = v0 + 32 * i + lane;
            if (v < vecs) {
                x[i][0] = __ldcg(src + 2 * v);
                x[i][1] = __ldcg(src + 2 * v + 1);
            }
        }
        if (v0 == 0) {
            float factor = 0.f;
            if (lane < 2) {
                const float *ssq = p.ssq + ((size_t)lane * p.n_tokens + token) * p.ssq_slots;
                float sum = 0.f;
                for (int t = 0; t < p.ssq_slots; ++t) sum += __ldcg(ssq + t);
                factor = 1.f / sqrtf(fmaf(sum, 1.f / (float)HD, p.eps));
            }
            if (lane == 0) p.q_row_scale[token] = factor;
            rk = __shfl_sync(0xffffffffu, factor, 1);
        }
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int v = v0 + 32 * i + lane;
            if (v < vecs) {
                const float4 a = x[i][0], b = x[i][1];
                const int head = v / per_head;
                *reinterpret_cast<uint4 *>(dst + (size_t)head * p.rows_per_head * p.head_dim + (v - head * per_head) * 8) =
                    make_uint4(cvt_bf16x2(a.x * rk, a.y * rk), cvt_bf16x2(a.z * rk, a.w * rk), cvt_bf16x2(b.x * rk, b.y * rk),
                               cvt_bf16x2(b.z * rk, b.w * rk));
            }
        }
    }
}

}  // namespace

cudaError_t launch_qkv_gemm(const QkvParams &p, const CUtensorMap &xmap, const CUtensorMap &wmap, int sm_count,
                            cudaStream_t stream)
{
    const int n_tiles = p.m_tiles * p.n_tiles;
    if (n_tiles <= 0) return cudaSuccess;
    const int pairs = sm_count / 2 > 0 ? sm_count / 2 : 1, grid = 2 * (n_tiles < pairs ? n_tiles : pairs);
    cudaError_t e = cudaErrorInvalidValue;
#define LL_GEMM_CASE(DD, TT)                                                                                                  \
    if (p.head_dim == DD && p.tile_n == TT) {                                                                                  \
        e = cudaFuncSetAttribute(qkv_gemm_kernel<DD, TT>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<TT>::kSmem);   \
        if (e != cudaSuccess) return e;                                                                                        \
        e = launch_dependent(true, qkv_gemm_kernel<DD, TT>, grid, GemmCfg<TT>::kThreads, GemmCfg<TT>::kSmem, stream, p, xmap, wmap); \
    }
    LL_GEMM_CASE(128, 256)
    LL_GEMM_CASE(128, 192)
    LL_GEMM_CASE(128, 128)
    LL_GEMM_CASE(64, 256)
    LL_GEMM_CASE(64, 192)
    LL_GEMM_CASE(64, 128)
#undef LL_GEMM_CASE
    count_launch();
    if (e != cudaSuccess || !p.with_norm) return e;
    e = launch_spread<&qkv_finish_kernel>((unsigned)((p.n_tokens + 7) / 8), 256, stream, p);
    count_launch();
    return e;
}

}  // namespace ll
