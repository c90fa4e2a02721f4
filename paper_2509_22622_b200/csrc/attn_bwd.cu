// Backward of the clip step on tcgen05 tensor cores (sm_100a): gradients of a loss with respect to
// the clip's q, k, v given the gradient of the attention output.
//
// With s_ij = q_i.k_j / sqrt(D) over the keys visible to row i, p_ij = exp(s_ij - lse_i):
//   delta_i = d_out_i . out_i                                  (delta kernel)
//   dP_ij = d_out_i . v_j,   dS_ij = p_ij (dP_ij - delta_i)
//   dq_i = sum_j dS_ij k_j / sqrt(D)                            (dq blocks, one CTA per query tile)
//   dk_j = sum_i dS_ij q_i / sqrt(D),  dv_j = sum_i p_ij d_out_i   (dk/dv blocks, one CTA per key tile)
// q, k are the rotated tensors; dq and dk are turned back through the rotation before they are
// stored.  Only the clip's own keys get dk, dv (the sink and the context are detached).
//
// Two passes over the products instead of one with atomics: every gradient element is accumulated by one CTA in one
// order, so the result is run-to-run deterministic, at the price of forming S and dP twice.  Both kinds of
// block have one warp that issues the MMAs (all its lanes walk the loop so that descriptors are warp-uniform;
// one elected lane issues) and eight compute warps (one thread per tile row and 64-column half, the 32x32b TMEM
// shape).  The dq blocks' issuer also loads (TMA); their compute warps take S into registers and release its tensor
// memory at once, so the next step's S is formed while they are in the exponentials.  The dk/dv blocks have a
// load warp of their own, and form the next S once P has been read.  dP is read only for the last multiply.
//   Neither kind needs what the other writes, so one launch holds both, the dq blocks in front: the dk/dv blocks fill the SMs that a
// short dq part leaves idle, or the end of a long one, and every block waits for delta as the kernels of a stream do.
// Against two kernels one behind the other, in us: 650 rows, 2 heads of 128: 33.1 -> 20.6; 2394 rows, 3 of 128: 71.6 -> 42.7; 3240 rows, 2 of 64:
// 82.0 -> 49.8; 11628 rows, 1 of 128: 381 -> 261; 768 rows, 16 of 64: 19.1 -> 18.3; the 21-frame clip 8919 and 8908.
//   What they compute goes back to tensor memory as the A operand of the products that follow: dS over dP, and in
// the dk/dv blocks P over S (at head_dim 64 beside them, where columns are left).  Through shared memory those tiles
// cost a store and a read of 32 KB each beside operands of 64 KB per 512 clk of products.
//   Products run in the order of their issue only if they share accumulator and shape.  One that overwrites columns
// which an earlier one reads as its A operand is therefore issued behind that one's commit; stores from registers are
// behind a later product's commit anyway, which covers all products before it.
//   21-frame clip of the benchmark layer (32760 rows, 12 heads of 128): 9.25 -> 8.80 ms in a loop at the power limit (8.65 without
// the waits between products).  Serving the two 64-key halves of the dq blocks' steps as chains of their own, half a step
// apart, was slower (64-wide products: 4.66 ms for them where they took 4.07 without those waits).
#include <cuda_bf16.h>

#include "bounded_wait.cuh"
#include "exp2_poly.cuh"
#include "ll_internal.h"
#include "ptx.cuh"

namespace ll {

namespace {

using namespace ptx;

constexpr int kComputeWarps = 8;
constexpr int kIssueWarp = 8;                          // issues the MMAs; in the dq blocks the loads too
constexpr int kLoadWarp = 9;                           // of the dk/dv blocks
constexpr int kBwdThreads = 320;
constexpr int kTile = 128;
constexpr int kStatBytes = 2 * kTile * 4;              // a query tile's row statistics in the dk/dv blocks
constexpr int kBwdBars = 17;

__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const uint32_t *r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
                 : "memory");
}

__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}

// delta[h][i] = sum_d d_out[i][h][d] * out[i][h][d].  D / 8 threads share a row of a head, 16 bytes each, and take
// kRows consecutive rows, all loads in flight together; bound by the read of the two tensors.  (With a
// warp per row and head and 4-byte loads 74 us, now 34 us, for 32760 rows of 12 heads of 128: 201 MB, 31 us
// at the copy rate.)
template <int D>
__global__ void __launch_bounds__(256) bwd_delta_kernel(const __grid_constant__ BwdParams p)
{
    constexpr int kLanes = D / 8, kRows = 4;
    grid_dep_launch();
    const int lane = threadIdx.x & (kLanes - 1);
    const long long group = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
    const int head = (int)(group % p.heads);
    const long long row0 = group / p.heads * kRows;
    grid_dep_wait();
    uint4 a[kRows], b[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const bool live = row0 + r < p.nq_total;
        const size_t off = ((size_t)(row0 + r) * p.heads + head) * D + 8 * lane;
        a[r] = live ? *reinterpret_cast<const uint4 *>(p.out + off) : make_uint4(0u, 0u, 0u, 0u);
        b[r] = live ? *reinterpret_cast<const uint4 *>(p.d_out + off) : make_uint4(0u, 0u, 0u, 0u);
    }
    float mine = 0.f;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const uint32_t x[4] = {a[r].x, a[r].y, a[r].z, a[r].w}, y[4] = {b[r].x, b[r].y, b[r].z, b[r].w};
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            s = fmaf(as_f(x[i] << 16), as_f(y[i] << 16), s);
            s = fmaf(as_f(x[i] & 0xffff0000u), as_f(y[i] & 0xffff0000u), s);
        }
#pragma unroll
        for (int m = kLanes / 2; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        if (lane == r) mine = s;
    }
    if (lane < kRows && row0 + lane < p.nq_total) p.delta[(size_t)head * p.nq_total + row0 + lane] = mine;
}

// Half `half` of the D columns of 128 rows x D fp32 in TMEM (row = thread), times `mul`,
// optionally turned back through the rotation of the row's grid position, rounded to bf16 and
// stored at dst (one head row of D).
template <int D, bool kRotateBack>
__device__ __forceinline__ void store_grad_row(uint32_t taddr, float mul, ll_bf16 *dst, const BwdParams &p, int frame,
                                               int y, int x, bool live, int half)
{
    constexpr int kNh = D / 6, kNt = D / 2 - 2 * kNh;
    const float2 *t_row = p.t_tab + (size_t)frame * kNt, *h_row = p.h_tab + (size_t)y * kNh, *w_row = p.w_tab + (size_t)x * kNh;
#pragma unroll
    for (int c = 0; c < D / 64; ++c) {
        const int ch = half * (D / 64) + c;
        uint32_t r[32];
        tmem_ld_32x32b_x32(taddr + 32 * ch, r);
        tmem_wait_ld();
        uint32_t o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float a = as_f(r[2 * i]) * mul, b = as_f(r[2 * i + 1]) * mul;
            if (kRotateBack) {
                const int j = 16 * ch + i;
                const float2 cs = j < kNt ? t_row[j] : j < kNt + kNh ? h_row[j - kNt] : w_row[j - kNt - kNh];
                const float a2 = fmaf(a, cs.x, b * cs.y), b2 = fmaf(b, cs.x, -(a * cs.y));
                a = a2;
                b = b2;
            }
            o[i] = cvt_bf16x2(a, b);
        }
        if (live) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                reinterpret_cast<uint4 *>(dst + 32 * ch)[i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
        }
    }
}

// Walks the 128-row key tiles of a group's visible runs.
struct RunTiles {
    const AttnGroup *g;
    int r, off;
    __device__ RunTiles(const AttnGroup *grp) : g(grp), r(0), off(0) {}
    __device__ int row() const { return g->k_start[r] + off; }
    __device__ int valid() const { return min(kTile, g->k_len[r] - off); }
    __device__ void next()
    {
        off += kTile;
        if (off >= g->k_len[r]) { ++r; off = 0; }
    }
};


template <int D>
struct BwdCfg {
    static constexpr int kAtomBytes = 128 * 128;
    static constexpr int kTileBytes = (D / 64) * kAtomBytes;     // 128 rows x D bf16
    static constexpr int kBarOff = 6 * kTileBytes + 2 * kStatBytes;      // behind the tiles and the dk/dv blocks' statistics
    static constexpr int kSmemBytes = kBarOff + 2048;            // barriers, tensor memory address, flag; alignment of the tiles
};

// What a block has once its barriers and its tensor memory are set up and the kernels in front of this one have completed.
struct BwdSetup {
    uint32_t base, bars, tmem;                         // shared addresses of the tiles and the barriers; tensor memory
    uint8_t *gen;                                      // the tiles again
    volatile int *abort_flag;
    bool skip;                                         // an earlier kernel gave up on a wait: nothing to do
    int warp, head;
};

// MMA helpers: all tiles are 128-byte-swizzled, 128 rows, tile base 1024-byte aligned.  The low
// descriptor word of a tile is formed once; a slice of the contraction adds a constant to it.
//   K-major operand [rows][64-element atoms]: slice kk = 16 elements of the contraction.
//   MN-major operand: the tile's rows are the contraction index, its columns the M (or N) index;
//   slice kk = rows 16 kk .. 16 kk + 15.
__device__ __forceinline__ uint32_t lo_kmajor(uint32_t tile) { return smem_desc_lo(tile, 16); }
__device__ __forceinline__ uint32_t lo_mnmajor(uint32_t tile) { return smem_desc_lo(tile, 128 * 128); }
__host__ __device__ constexpr uint32_t slice_kmajor(int kk) { return (uint32_t)(((kk / 4) * (128 * 128) + (kk % 4) * 32) >> 4); }
__host__ __device__ constexpr uint32_t slice_mnmajor(int kk) { return (uint32_t)((kk * 2048) >> 4); }

// D = A B over kSlices slices, both operands K-major in shared memory.
template <int kSlices>
__device__ __forceinline__ void mma_kmajor(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc)
{
    constexpr uint32_t hi = smem_desc_hi_sw128(1024);
#pragma unroll
    for (int kk = 0; kk < kSlices; ++kk)
        mma_ss(d, smem_desc_join(a_lo + slice_kmajor(kk), hi), smem_desc_join(b_lo + slice_kmajor(kk), hi), idesc, kk > 0);
}

__device__ __forceinline__ void key_mask(int nvalid, uint32_t (&valid)[4])
{
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        valid[ch] = nvalid >= 32 * (ch + 1) ? 0xffffffffu : nvalid > 32 * ch ? ((1u << (nvalid - 32 * ch)) - 1u) : 0u;
}

// This thread's 64 columns of a score row (fp32 words in s) to the weights p = 2^(s c - lse2),
// in place; columns whose bit in vlo (first 32) / vhi is clear give zero.  (Moving a quarter or
// a half of the exponentials to the FMA-pipe polynomial of the forward kernel made the pass
// slower, 8.46 and 8.59 ms against 8.35 ms at the 21-frame clip, so all of them stay on the
// special-function unit.)
__device__ __forceinline__ void scores_to_weights(uint32_t (&s)[64], float c, float lse2, uint32_t vlo, uint32_t vhi)
{
    const uint64_t c2 = pack2(c, c), nl2 = pack2(-lse2, -lse2);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        float e0, e1;
        unpack2(exp2_sfu2(fma2(pack2(as_f(s[2 * i]), as_f(s[2 * i + 1])), c2, nl2)), e0, e1);
        s[2 * i] = __float_as_uint(e0);
        s[2 * i + 1] = __float_as_uint(e1);
    }
    if ((vlo & vhi) != 0xffffffffu) {
#pragma unroll
        for (int i = 0; i < 64; ++i)
            if (!(((i < 32 ? vlo : vhi) >> (i & 31)) & 1u)) s[i] = 0u;
    }
}

// ---- dq: one CTA per (128-row query tile, head) ---------------------------------------------
// The tile's Q and dO rows are the stationary A operands of S = Q K^T and dP = dO V^T: they are
// written once into tensor memory (bf16, two elements per column), so those products read only
// K and V from shared memory.  Eight compute warps share a step (thread = tile row x 64-key
// half).  Per 128-key step j the tensor pipe runs S(j+1) | dQ(j) | dP(j+1) ...: the compute warps
// take S(j) into registers and release it at once, so S(j+1) is formed while they are in the
// exponentials; dP(j) is only needed for the last multiply, dS = P (dP - delta), which goes back
// over it as bf16, so that dP(j+1) waits for dQ(j), or at head_dim 64 into columns of its own.  K and V tiles sit in
// three stages; K is needed until the step's dQ product, V only until its dP.
//   tensor memory columns: S 0..127, dP 128..255, dQ 256..256+D-1, Q 384.., dO 448..; dS of key half h at 128 + 64 h.. or 416 + 64 h..
template <int D>
struct DqBlock {
    using C = BwdCfg<D>;
    enum { kKFull = 0, kVFull = 3, kKEmpty = 6, kVEmpty = 9, kSFull = 12, kSFree = 13, kDpFull = 14, kDsFull = 15, kDone = 16, kBars = 17 };
    static __device__ uint32_t arrivals(int bar_id) { return bar_id == kSFree || bar_id == kDsFull ? kComputeWarps : 1; }

    int g, tile;                                       // query group, and which tile of it
    __device__ DqBlock(const BwdParams &p, int t) : g(0), tile(t)
    {
        while (tile >= (p.g[g].q_rows + kTile - 1) / kTile) { tile -= (p.g[g].q_rows + kTile - 1) / kTile; ++g; }
    }
    __device__ __forceinline__ void run(const BwdParams &p, const BwdMaps &maps, const BwdSetup &b) const;
};

template <int D>
__device__ __forceinline__ void DqBlock<D>::run(const BwdParams &p, const BwdMaps &maps, const BwdSetup &b) const
{
    constexpr int kStages = 3;
    const uint32_t k_s = b.base, v_s = k_s + kStages * C::kTileBytes;
    const int warp = b.warp, lane = threadIdx.x & 31, head = b.head;
    auto bar = [&](int i) -> uint32_t { return b.bars + 8u * (uint32_t)i; };
    const AttnGroup &G = p.g[g];
    const int q0 = G.q_begin + tile * kTile, rows = min(kTile, G.q_rows - tile * kTile);
    const int n_kt = G.n_kt;
    const uint32_t tmem = b.tmem;
    const WaitCtx ctx{b.abort_flag, p.status, warp};
    auto wait = [&](int bar_id, uint32_t parity, int iter) -> bool { return wait_bar(bar(bar_id), parity & 1u, ctx, bar_id, iter); };
    const bool skip = b.skip;
    constexpr bool kOverDp = D == 128;                           // dS takes the place of dP
    const uint32_t t_s = tmem, t_dp = tmem + 128, t_dq = tmem + 256, t_q = tmem + 384, t_do = tmem + 448,
                   t_ds = kOverDp ? t_dp : tmem + 416;

    // the tile's Q rows (warps 0-3) and dO rows (warps 4-7) into tensor memory; rows past the
    // group's end become zeros
    if (!skip && warp < kIssueWarp) {
        const int row = threadIdx.x & 127, half = threadIdx.x >> 7;
        const bool live = row < rows;
        const uint4 *src = reinterpret_cast<const uint4 *>((half ? p.d_out : p.q) + ((size_t)(q0 + (live ? row : 0)) * p.heads + head) * D);
        const uint32_t dst = (half ? t_do : t_q) + ((uint32_t)(32 * (warp & 3)) << 16);
#pragma unroll
        for (int c = 0; c < D / 64; ++c) {
            uint32_t w[32];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 u = live ? src[8 * c + i] : make_uint4(0u, 0u, 0u, 0u);
                w[4 * i] = u.x; w[4 * i + 1] = u.y; w[4 * i + 2] = u.z; w[4 * i + 3] = u.w;
            }
            tmem_st_32x32b_x32(dst + 32 * c, w);
        }
        tmem_wait_st();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();

    if (skip) {
    } else if (warp == kIssueWarp) {
        // All 32 lanes walk the loop and the waits, so that addresses and descriptors are
        // warp-uniform values; one elected lane issues the copies, the MMAs and the commits.
        [&]() {
            const bool elected = elect_one();
            constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0), idesc_dq = idesc_bf16_f32(128, D, 0, 1);
            constexpr uint32_t hi = smem_desc_hi_sw128(1024);
            RunTiles kt(&G);                                     // walks ahead of the products: tile of the next load
            int loaded = 0;
            auto load_kv = [&]() {                               // K and V tiles of step `loaded`
                const int st = loaded % kStages, row = kt.row();
                if (elected) {
                    mbar_arrive_expect_tx(bar(kKFull + st), C::kTileBytes);
                    for (int a = 0; a < D / 64; ++a)
                        tma_load_3d(k_s + st * C::kTileBytes + a * C::kAtomBytes, &maps.k, bar(kKFull + st), a * 64, row, head);
                    mbar_arrive_expect_tx(bar(kVFull + st), C::kTileBytes);
                    for (int a = 0; a < D / 64; ++a)
                        tma_load_3d(v_s + st * C::kTileBytes + a * C::kAtomBytes, &maps.v, bar(kVFull + st), a * 64, row, head);
                }
                __syncwarp();
                ++loaded;
                kt.next();
            };
            auto commit = [&](int bar_id) { if (elected) tc_commit(bar(bar_id)); };
            const uint32_t k_lo = lo_kmajor(k_s), v_lo = lo_kmajor(v_s);
            auto issue_s = [&](int j) -> bool {                  // S(j) = Q K(j)^T
                const int st = j % kStages;
                if (!wait(kKFull + st, j / kStages, j)) return false;
                tc_fence_after_sync();
                const uint32_t b_lo = k_lo + ((uint32_t)(st * C::kTileBytes) >> 4);
                if (elected) {
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        mma_ts(t_s, t_q + 8 * kk, smem_desc_join(b_lo + slice_kmajor(kk), hi), idesc_s, kk > 0);
                }
                __syncwarp();
                commit(kSFull);
                return true;
            };
            auto issue_dp = [&](int j) -> bool {                 // dP(j) = dO V(j)^T
                const int st = j % kStages;
                if (!wait(kVFull + st, j / kStages, j)) return false;
                const uint32_t b_lo = v_lo + ((uint32_t)(st * C::kTileBytes) >> 4);
                if (kOverDp && j > 0 && !wait(kKEmpty + (j - 1) % kStages, (j - 1) / kStages, j)) return false;      // dQ(j-1) has read dS(j-1)
                tc_fence_after_sync();
                if (elected) {
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        mma_ts(t_dp, t_do + 8 * kk, smem_desc_join(b_lo + slice_kmajor(kk), hi), idesc_s, kk > 0);
                }
                __syncwarp();
                commit(kDpFull);
                commit(kVEmpty + st);
                return true;
            };
            for (int i = 0; i < kStages && i < n_kt; ++i) load_kv();
            if (!issue_s(0) || !issue_dp(0)) return;
            for (int j = 0; j < n_kt; ++j) {
                const int st = j % kStages;
                if (j >= 1 && j + 2 < n_kt) {                    // the stage step j - 1 used takes step j + 2
                    const int free_st = (j - 1) % kStages;
                    if (!wait(kVEmpty + free_st, (j - 1) / kStages, j) || !wait(kKEmpty + free_st, (j - 1) / kStages, j)) return;
                    load_kv();
                }
                if (j + 1 < n_kt) {
                    if (!wait(kSFree, j, j)) return;             // S(j) is in the compute warps' registers
                    if (!issue_s(j + 1)) return;
                }
                if (!wait(kDsFull, j, j)) return;                // dS(j) is in tensor memory, dP(j) has been read
                tc_fence_after_sync();
                const uint32_t k_mn = lo_mnmajor(k_s + st * C::kTileBytes);
                if (elected) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        mma_ts(t_dq, t_ds + (kk >= 4 ? 64 : 0) + 8 * (kk & 3), smem_desc_join(k_mn + slice_mnmajor(kk), hi), idesc_dq,
                               (j > 0 || kk > 0) ? 1u : 0u);
                }
                __syncwarp();
                commit(kKEmpty + st);
                if (j + 1 < n_kt && !issue_dp(j + 1)) return;
            }
            commit(kDone);
        }();
    } else if (warp < kIssueWarp) {
        bool alive = true;
        auto wait_c = [&](int bar_id, uint32_t parity, int iter) {
            if (alive && !__all_sync(0xffffffffu, wait(bar_id, parity, iter))) alive = false;
        };
        const int row = threadIdx.x & 127, half = threadIdx.x >> 7;      // tile row = TMEM lane; 64-key half
        const bool live = row < rows;
        const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
        const size_t stat = (size_t)head * p.nq_total + q0 + (live ? row : 0);
        const float lse2 = p.lse[stat] * 1.4426950408889634f, delta = p.delta[stat];
        RunTiles kt(&G);
        for (int j = 0; j < n_kt; ++j, kt.next()) {
            uint32_t valid[4];
            key_mask(kt.valid(), valid);
            wait_c(kSFull, j, j);
            tc_fence_after_sync();
            uint32_t w[64];
            tmem_ld_32x32b_x32(t_s + lane_off + 64 * half, w);
            tmem_ld_32x32b_x32(t_s + lane_off + 64 * half + 32, w + 32);
            tmem_wait_ld();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kSFree));
            scores_to_weights(w, p.scale_log2, lse2, live ? (half ? valid[2] : valid[0]) : 0u, live ? (half ? valid[3] : valid[1]) : 0u);
            wait_c(kDpFull, j, j);
            tc_fence_after_sync();
            const uint64_t nd2 = pack2(-delta, -delta);
#pragma unroll
            for (int h = 0; h < 2; ++h) {                        // dS = p (dP - delta), bf16
                uint32_t dp[32], dw[16];
                tmem_ld_32x32b_x32(t_dp + lane_off + 64 * half + 32 * h, dp);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    float d0, d1;
                    unpack2(mul2(pack2(as_f(w[32 * h + 2 * i]), as_f(w[32 * h + 2 * i + 1])),
                                 add2(pack2(as_f(dp[2 * i]), as_f(dp[2 * i + 1])), nd2)), d0, d1);
                    dw[i] = cvt_bf16x2(d0, d1);
                }
                tmem_st_32x32b_x16(t_ds + lane_off + 64 * half + 16 * h, dw);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kDsFull));
        }
        wait_c(kDone, 0, n_kt);
        tc_fence_after_sync();
        const int token = q0 + (live ? row : 0);
        const int frame = token / p.P, cell = token % p.P;
        if (alive)
            store_grad_row<D, true>(t_dq + lane_off, p.scale, p.dq + ((size_t)token * p.heads + head) * D, p, frame,
                                    cell / p.grid_w, cell % p.grid_w, live, half);
    }
}

// Which of the 128 cache rows starting at r0 a group can see (bit c of word c / 32 = row r0 + c).
__device__ __forceinline__ bool group_mask(const AttnGroup &G, int r0, uint32_t (&valid)[4])
{
    valid[0] = valid[1] = valid[2] = valid[3] = 0u;
    bool any = false;
    for (int r = 0; r < G.n_ranges; ++r) {
        const int lo = max(G.k_start[r], r0) - r0, hi = min(G.k_start[r] + G.k_len[r], r0 + kTile) - r0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int a = min(max(lo - 32 * w, 0), 32), b = min(max(hi - 32 * w, 0), 32);
            if (b > a) valid[w] |= (b == 32 ? 0xffffffffu : (1u << b) - 1u) & ~((1u << a) - 1u);
        }
        any |= hi > lo;
    }
    return any;
}

// Whether any of the 128 cache rows starting at r0 is visible to the group.
__device__ __forceinline__ bool group_sees(const AttnGroup &G, int r0)
{
    bool any = false;
    for (int r = 0; r < G.n_ranges; ++r)
        any |= min(G.k_start[r] + G.k_len[r], r0 + kTile) > max(G.k_start[r], r0);
    return any;
}

// The (group, 128-row query tile) pairs a key tile takes part in, in order.  The group's first row
// and tile count are kept, so a step inside a group costs an increment.
struct QTiles {
    const BwdParams &p;
    int r0, g, i, tiles, q_begin;
    __device__ QTiles(const BwdParams &params, int first_row) : p(params), r0(first_row), g(-1), i(0), tiles(0), q_begin(0) { next(); }
    __device__ bool done() const { return g >= p.n_groups; }
    __device__ int q_row() const { return q_begin + i * kTile; }
    __device__ int live() const { return p.g[g].q_rows - i * kTile; }      // rows of the group from this tile on
    __device__ void next()
    {
        if (++i < tiles) return;
        i = 0;
        for (++g; g < p.n_groups; ++g) {
            const AttnGroup &G = p.g[g];
            if (G.q_rows > 0 && group_sees(G, r0)) {
                tiles = (G.q_rows + kTile - 1) / kTile;
                q_begin = G.q_begin;
                return;
            }
        }
    }
};

// ---- dk, dv: one CTA per (128-row tile of the clip's cache rows, head) -----------------------
// K and V of the tile stay in shared memory; per step j one query tile's Q and dO stream in (two slots each, loaded
// by a warp of their own).  Scores are formed with the keys as rows, S^T = K Q^T and dP^T = V dO^T, so that
// P^T and dS^T are the A operands of dV += P^T dO and dK += dS^T Q in the rows they are computed in: they go back to
// tensor memory as bf16 and never through shared memory.  At head_dim 128 all 512 columns are taken and they go over S and
// dP, so that S(j+1) waits for dV(j), and dP(j+1) for dK(j); at 64 they have columns of their own.
//   The tensor pipe runs, per step,  dV(j) | S(j+1) | dK(j) | dP(j+1).  P(j) is handed over in two pieces, so that half of
// dV(j) runs under the second piece's exponentials, and dS(j) is formed under the rest of dV(j) and S(j+1).
// The row statistics are per column here: the load warp lays them out in shared memory (negated, in pairs for
// the packed arithmetic).
//   tensor memory columns: S 0..127, dP 128..255, dK and dV 256..256+2D-1; P (16-query slices 0-3 at 0.., 4-7 at 64.. of it) at 0
// or 384, dS (likewise) at 128 or 416.
template <int D>
struct DkdvBlock {
    using C = BwdCfg<D>;
    enum { kKvFull = 0, kQFull = 1, kDoFull = 3, kQEmpty = 5, kDoEmpty = 7, kStatFull = 9, kSFull = 11, kPHalf = 12, kPFull = 13,
           kDpFull = 14, kDsFull = 15, kDone = 16, kBars = 17 };
    static __device__ uint32_t arrivals(int bar_id) { return bar_id == kPHalf || bar_id == kPFull || bar_id == kDsFull ? kComputeWarps : 1; }

    int r0, run_end;                                   // the tile's first cache row and the end of the run it belongs to
    __device__ DkdvBlock(const BwdParams &p, int t)
    {
        int run = 0;
        while (t >= (p.krun_len[run] + kTile - 1) / kTile) { t -= (p.krun_len[run] + kTile - 1) / kTile; ++run; }
        r0 = p.krun_start[run] + t * kTile;
        run_end = p.krun_start[run] + p.krun_len[run];
    }
    __device__ __forceinline__ void run(const BwdParams &p, const BwdMaps &maps, const BwdSetup &b) const;
};

template <int D>
__device__ __forceinline__ void DkdvBlock<D>::run(const BwdParams &p, const BwdMaps &maps, const BwdSetup &b) const
{
    const uint32_t k_s = b.base, v_s = k_s + C::kTileBytes, q_s = v_s + C::kTileBytes, do_s = q_s + 2 * C::kTileBytes;
    uint8_t *const stats = b.gen + 6 * C::kTileBytes;            // two slots of kStatBytes
    const int warp = b.warp, lane = threadIdx.x & 31, head = b.head;
    auto bar = [&](int i) -> uint32_t { return b.bars + 8u * (uint32_t)i; };
    const uint32_t tmem = b.tmem;
    const WaitCtx ctx{b.abort_flag, p.status, warp};
    auto wait = [&](int bar_id, uint32_t parity, int iter) -> bool { return wait_bar(bar(bar_id), parity & 1u, ctx, bar_id, iter); };
    const bool skip = b.skip;
    constexpr bool kOver = D == 128;                             // P and dS take the places of S and dP
    const uint32_t t_s = tmem, t_dp = tmem + 128, t_dk = tmem + 256, t_dv = tmem + 256 + D,
                   t_p = kOver ? t_s : tmem + 384, t_ds = kOver ? t_dp : tmem + 416;

    if (skip) {
    } else if (warp == kLoadWarp) {
        // ---- loads: all lanes walk the loop, one elected lane issues the copies ----
        [&]() {
            const bool elected = elect_one();
            auto load_tile = [&](uint32_t dst, const CUtensorMap *map, int bar_id, int q_row) {
                if (elected) {
                    mbar_arrive_expect_tx(bar(bar_id), C::kTileBytes);
                    for (int a = 0; a < D / 64; ++a) tma_load_3d(dst + a * C::kAtomBytes, map, bar(bar_id), a * 64, head, q_row);
                }
                __syncwarp();
            };
            int j = 0;
            for (QTiles qt(p, r0); !qt.done(); qt.next(), ++j) {
                const int sl = j & 1, row = qt.q_row(), live = qt.live();
                float nl[4], nd[4];                              // rows lane + 32 i of the tile
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool in = lane + 32 * i < live;
                    const size_t stat = (size_t)head * p.nq_total + row + (in ? lane + 32 * i : 0);
                    nl[i] = in ? -1.4426950408889634f * p.lse[stat] : 0.f;
                    nd[i] = in ? -p.delta[stat] : 0.f;
                }
                if (j == 0) {
                    if (elected) {
                        mbar_arrive_expect_tx(bar(kKvFull), 2 * C::kTileBytes);
                        for (int a = 0; a < D / 64; ++a) {
                            tma_load_3d(k_s + a * C::kAtomBytes, &maps.k, bar(kKvFull), a * 64, r0, head);
                            tma_load_3d(v_s + a * C::kAtomBytes, &maps.v, bar(kKvFull), a * 64, r0, head);
                        }
                    }
                    __syncwarp();
                }
                if (j >= 2 && !wait(kQEmpty + sl, (j >> 1) - 1, j)) return;      // dK(j-2) has read Q(j-2), and step j-2 its statistics
                load_tile(q_s + sl * C::kTileBytes, &maps.q, kQFull + sl, row);
                if (j >= 2 && !wait(kDoEmpty + sl, (j >> 1) - 1, j)) return;     // dV(j-2) has read dO(j-2)
                load_tile(do_s + sl * C::kTileBytes, &maps.d_out, kDoFull + sl, row);
                float *st = reinterpret_cast<float *>(stats + sl * kStatBytes);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    st[lane + 32 * i] = nl[i];
                    st[kTile + lane + 32 * i] = nd[i];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kStatFull + sl));
            }
        }();
    } else if (warp == kIssueWarp) {
        // ---- MMA issue: all lanes walk the loop and the waits, one elected lane issues ----
        [&]() {
            const bool elected = elect_one();
            constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0), idesc_g = idesc_bf16_f32(128, D, 0, 1);
            constexpr uint32_t hi = smem_desc_hi_sw128(1024);
            auto commit = [&](int bar_id) { if (elected) tc_commit(bar(bar_id)); };
            int n_steps = 0;
            for (QTiles qt(p, r0); !qt.done(); qt.next()) ++n_steps;
            if (n_steps == 0) return;
            const uint32_t k_k = lo_kmajor(k_s), v_k = lo_kmajor(v_s);
            auto issue_s = [&](int j) -> bool {                  // S^T(j) = K Q(j)^T
                const int sl = j & 1;
                if (!wait(kQFull + sl, j >> 1, j)) return false;
                if (kOver && j > 0 && !wait(kDoEmpty + (sl ^ 1), (j - 1) >> 1, j)) return false;     // dV(j-1) has read P(j-1)
                tc_fence_after_sync();
                if (elected) mma_kmajor<D / 16>(t_s, k_k, lo_kmajor(q_s + sl * C::kTileBytes), idesc_s);
                __syncwarp();
                commit(kSFull);
                return true;
            };
            auto issue_dp = [&](int j) -> bool {                 // dP^T(j) = V dO(j)^T
                const int sl = j & 1;
                if (!wait(kDoFull + sl, j >> 1, j)) return false;
                if (kOver && j > 0 && !wait(kQEmpty + (sl ^ 1), (j - 1) >> 1, j)) return false;      // dK(j-1) has read dS(j-1)
                tc_fence_after_sync();
                if (elected) mma_kmajor<D / 16>(t_dp, v_k, lo_kmajor(do_s + sl * C::kTileBytes), idesc_s);
                __syncwarp();
                commit(kDpFull);
                return true;
            };
            // 16-query slice kk of grad += A^T(tensor memory) B(shared memory, rows = queries)
            auto slice = [&](uint32_t t_grad, uint32_t t_a, uint32_t b_mn, int kk, uint32_t acc) {
                mma_ts(t_grad, t_a + (kk >= 4 ? 64 : 0) + 8 * (kk & 3), smem_desc_join(b_mn + slice_mnmajor(kk), hi), idesc_g, acc);
            };
            if (!wait(kKvFull, 0, 0)) return;
            if (!issue_s(0) || !issue_dp(0)) return;
            for (int j = 0; j < n_steps; ++j) {
                const int sl = j & 1;
                const bool more = j + 1 < n_steps;
                const uint32_t do_mn = lo_mnmajor(do_s + sl * C::kTileBytes), q_mn = lo_mnmajor(q_s + sl * C::kTileBytes);
#pragma unroll
                for (int h = 0; h < 2; ++h) {                    // dV += P^T dO, a piece's slices at a time
                    if (!wait(h ? kPFull : kPHalf, j, j)) return;
                    tc_fence_after_sync();
                    if (elected) {
                        slice(t_dv, t_p, do_mn, 2 * h, (j > 0 || h > 0) ? 1u : 0u);
                        slice(t_dv, t_p, do_mn, 2 * h + 1, 1u);
                        slice(t_dv, t_p, do_mn, 2 * h + 4, 1u);
                        slice(t_dv, t_p, do_mn, 2 * h + 5, 1u);
                    }
                    __syncwarp();
                }
                commit(kDoEmpty + sl);
                if (more && !issue_s(j + 1)) return;
                if (!wait(kDsFull, j, j)) return;
                tc_fence_after_sync();
                if (elected) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) slice(t_dk, t_ds, q_mn, kk, (j > 0 || kk > 0) ? 1u : 0u);
                }
                __syncwarp();
                commit(kQEmpty + sl);
                if (more && !issue_dp(j + 1)) return;
            }
            commit(kDone);
        }();
    } else {
        bool alive = true;
        auto wait_c = [&](int bar_id, uint32_t parity, int iter) {
            if (alive && !__all_sync(0xffffffffu, wait(bar_id, parity, iter))) alive = false;
        };
        const int row = threadIdx.x & 127, half = threadIdx.x >> 7;      // key row of the tile = TMEM lane; 64-query half
        const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
        const uint32_t t_sh = t_s + lane_off + 64 * half, t_dph = t_dp + lane_off + 64 * half,
                       t_ph = t_p + lane_off + 64 * half, t_dsh = t_ds + lane_off + 64 * half;
        const uint64_t c2 = pack2(p.scale_log2, p.scale_log2);
        uint32_t step = 0;
        for (int g = 0; g < p.n_groups; ++g) {
            const AttnGroup &G = p.g[g];
            uint32_t valid[4];
            if (!group_mask(G, r0, valid)) continue;
            const uint32_t word = row < 32 ? valid[0] : row < 64 ? valid[1] : row < 96 ? valid[2] : valid[3];
            const bool seen = (word >> (row & 31)) & 1u;         // whether the group sees this key
            for (int i = 0; i * kTile < G.q_rows; ++i, ++step) {
                const float4 *nl = reinterpret_cast<const float4 *>(stats + (step & 1) * kStatBytes) + 16 * half;
                const float4 *nd = nl + kTile / 4;
                const int n_live = seen ? G.q_rows - i * kTile - 64 * half : 0;      // live columns of this thread's 64 (or more)
                wait_c(kStatFull + (step & 1), step >> 1, (int)step);
                wait_c(kSFull, step, (int)step);
                tc_fence_after_sync();
                uint32_t w[64];
                tmem_ld_32x32b_x32(t_sh, w);
                tmem_ld_32x32b_x32(t_sh + 32, w + 32);
                tmem_wait_ld();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pw[16];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 n = nl[8 * h + k];
                        uint32_t *v = w + 32 * h + 4 * k;
                        float e0, e1, e2, e3;
                        unpack2(exp2_sfu2(fma2(pack2(as_f(v[0]), as_f(v[1])), c2, pack2(n.x, n.y))), e0, e1);
                        unpack2(exp2_sfu2(fma2(pack2(as_f(v[2]), as_f(v[3])), c2, pack2(n.z, n.w))), e2, e3);
                        v[0] = as_u(e0); v[1] = as_u(e1); v[2] = as_u(e2); v[3] = as_u(e3);
                    }
                    if (n_live < 64) {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (32 * h + k >= n_live) w[32 * h + k] = 0u;
                    }
#pragma unroll
                    for (int k = 0; k < 16; ++k) pw[k] = cvt_bf16x2(as_f(w[32 * h + 2 * k]), as_f(w[32 * h + 2 * k + 1]));
                    tmem_st_32x32b_x16(t_ph + 16 * h, pw);
                    tmem_wait_st();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(h ? kPFull : kPHalf));
                }
                wait_c(kDpFull, step, (int)step);
                tc_fence_after_sync();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t dp[32], dw[16];
                    tmem_ld_32x32b_x32(t_dph + 32 * h, dp);
                    tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 n = nd[8 * h + k];
                        const uint32_t *v = w + 32 * h + 4 * k, *x = dp + 4 * k;
                        float d0, d1;
                        unpack2(mul2(pack2(as_f(v[0]), as_f(v[1])), add2(pack2(as_f(x[0]), as_f(x[1])), pack2(n.x, n.y))), d0, d1);
                        dw[2 * k] = cvt_bf16x2(d0, d1);
                        unpack2(mul2(pack2(as_f(v[2]), as_f(v[3])), add2(pack2(as_f(x[2]), as_f(x[3])), pack2(n.z, n.w))), d0, d1);
                        dw[2 * k + 1] = cvt_bf16x2(d0, d1);
                    }
                    tmem_st_32x32b_x16(t_dsh + 16 * h, dw);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kDsFull));
            }
        }
        // this thread's key row: stored only if it is one of the clip's rows inside this run
        const int r = r0 + row;
        const int slot = r / p.P, cell = r % p.P;
        const int cf = (r < run_end && slot < LL_MAX_SLOTS) ? p.slot_clip_frame[slot] : -1;
        const bool live = cf >= 0;
        const size_t token = live ? (size_t)cf * p.P + cell : 0;
        if (step > 0) wait_c(kDone, 0, (int)step);
        tc_fence_after_sync();
        if (alive && step > 0) {
            store_grad_row<D, true>(t_dk + lane_off, p.scale, p.dk + (token * p.heads + head) * D, p, live ? cf : 0,
                                    cell / p.grid_w, cell % p.grid_w, live, half);
            store_grad_row<D, false>(t_dv + lane_off, 1.f, p.dv + (token * p.heads + head) * D, p, 0, 0, 0, live, half);
        }
    }
}

// The dq blocks of the call, tile after tile and head after head, then its dk/dv blocks.
template <int D>
__global__ void __launch_bounds__(kBwdThreads, 1)
bwd_kernel(const __grid_constant__ BwdParams p, const __grid_constant__ BwdMaps maps)
{
    using C = BwdCfg<D>;
    static_assert(DqBlock<D>::kBars <= kBwdBars && DkdvBlock<D>::kBars <= kBwdBars, "more barriers than there is room for");
    extern __shared__ uint8_t smem_raw[];
    BwdSetup b;
    b.base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    b.gen = smem_raw + (b.base - smem_u32(smem_raw));
    b.bars = b.base + C::kBarOff;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(b.gen + C::kBarOff + kBwdBars * 8);
    b.abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    b.warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int n_dq = p.n_qtiles * p.heads;
    const bool is_dq = (int)blockIdx.x < n_dq;
    const int index = is_dq ? (int)blockIdx.x : (int)blockIdx.x - n_dq, tiles = is_dq ? p.n_qtiles : p.n_ktiles;
    b.head = index / tiles;
    const int tile = index - b.head * tiles;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kBwdBars; ++i) mbar_init(b.bars + 8u * (uint32_t)i, is_dq ? DqBlock<D>::arrivals(i) : DkdvBlock<D>::arrivals(i));
        fence_mbar_init();
    }
    if (b.warp == kIssueWarp) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); }
    grid_dep_launch();
    grid_dep_wait();
    if (threadIdx.x == 0) *b.abort_flag = (*reinterpret_cast<volatile uint32_t *>(p.status) != kStatusOk) ? 2 : 0;
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    b.tmem = *tmem_slot;
    b.skip = *b.abort_flag != 0;
    if (is_dq) DqBlock<D>(p, tile).run(p, maps, b);
    else DkdvBlock<D>(p, tile).run(p, maps, b);
    tc_fence_before_sync();
    __syncthreads();
    if (*b.abort_flag == 1) {
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (b.warp == kIssueWarp) { __syncwarp(); tc_fence_after_sync(); tmem_dealloc(b.tmem, 512); }
}

}  // namespace

cudaError_t launch_attn_backward(const BwdParams &p, const BwdMaps &maps, int sm_count, cudaStream_t stream)
{
    const int D = p.head_dim;
    const int smem = D == 128 ? BwdCfg<128>::kSmemBytes : BwdCfg<64>::kSmemBytes;
    cudaError_t e = D == 128 ? cudaFuncSetAttribute(bwd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                             : cudaFuncSetAttribute(bwd_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    // D / 8 threads per four rows of a head
    const long long threads = (long long)((p.nq_total + 3) / 4) * p.heads * (D / 8);
    const unsigned dblocks = (unsigned)((threads + 255) / 256);
    e = D == 128 ? launch_spread<&bwd_delta_kernel<128>>(dblocks, 256, stream, p) : launch_spread<&bwd_delta_kernel<64>>(dblocks, 256, stream, p);
    count_launch();
    if (e != cudaSuccess) return e;
    long long steps = 0;
    for (int g = 0; g < p.n_groups; ++g) steps += (long long)p.heads * ((p.g[g].q_rows + kTile - 1) / kTile) * p.g[g].n_kt;
    const bool early = steps <= kEarlySteps * sm_count;
    const dim3 grid((unsigned)(p.n_qtiles + p.n_ktiles) * (unsigned)p.heads);
    e = D == 128 ? launch_dependent(early, bwd_kernel<128>, grid, kBwdThreads, smem, stream, p, maps)
                 : launch_dependent(early, bwd_kernel<64>, grid, kBwdThreads, smem, stream, p, maps);
    count_launch();
    return e;
}

}  // namespace ll
