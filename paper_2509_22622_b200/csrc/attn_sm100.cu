// Sink+window attention on tcgen05 tensor cores (sm_100a).
//
// Work decomposition.  A *column* is up to 256 query rows of one head (two
// 128-row MMA tiles, "lanes" 0 and 1) and a *step* is one 128-key tile of that
// column's visible cache rows.  One persistent CTA runs per SM.  The columns of
// all query groups of a launch (one per chunk of queries, of one or several
// streams) are numbered through.  As long as there is a column for every CTA,
// columns are handed out whole: the CTAs of a head then walk the keys in step and
// each K/V tile is fetched from HBM once and shared through L2.  The steps of the
// columns left over are laid end to end and cut into one share per CTA, sized on
// the host so that every SM ends up with the same number of steps whatever the
// number and length of the columns (very short columns go out whole instead).  Equally long
// columns may also go out by their 128-row tiles, every CTA as many as any other or one more, two of one head at a
// time as a column and what is left over alone (AttnParams::tile_ctas); then nothing is split.
// A column whose steps fall into several CTAs is finished by whichever of them
// arrives last:
// every part leaves its unnormalised O rows, reference maxima and sums in a
// scratch slot, bumps the column's arrival counter, and the last one merges the
// parts and writes the output.  Nothing waits on another CTA.  Columns in up to eight equal parts are held by the
// CTAs of a cluster (AttnParams::cluster_parts), which run at the same time, wait for one another and merge a share of the
// head's columns each (merge_in_cluster).
//
// Inside a CTA (640 threads):
//   warp 16 (one lane)  TMA producer: the column's Q tiles, then K_j V_j K_j+1 ...
//                       into a ring of 128-byte-swizzled shared-memory stages
//   warps 17, 18        MMA issuers of lane 0 and lane 1 (one elected thread each):
//                       S_w = Q_w K_j^T and O_w += P_w V_j, operands in shared memory
//                       (P in TMEM at head_dim 64), accumulators in TMEM
//   warps 0-15          softmax: warp (w, q, h) owns the 16 rows 32q + 16h .. of
//                       lane w; its threads read S with the 16x256b TMEM shape, so
//                       a row lives in the four threads of a quad.  P (bf16) goes to
//                       a swizzled shared-memory tile (head_dim 128) or to TMEM columns of
//                       its own (64), 64 keys at a time and as soon as a 64-key piece is
//                       computed (its registers are then free for the next piece).  The rows' reference maxima move, and O is
//                       rescaled in TMEM, only when a weight computed against the old
//                       reference would have been large.
//   P does not go back over S: a lane's S buffer is free as soon as its softmax
//   warps hold the tile in registers, so the MMA warp issues QK of step j+1 while
//   the softmax of step j is still running, and the softmax warps find the next S
//   waiting.  The tensor pipe then sees, per lane and step, QK of the next step and
//   PV of this one, whenever their inputs arrive.  A share of the exponentials can be
//   evaluated with a cubic on the FMA pipe instead of the special-function unit
//   (kPolyMask: none at head_dim 128, a quarter at head_dim 64, as measured).
//
// TMEM columns: S_0 | S_1 | O_0 | O_1 (fp32), at head_dim 64 | P_0 | P_1 (bf16).  There a P that went through
// shared memory made that carry 128 KB per tile and step; from TMEM
// it is 64 KB, and one store instruction replaces four (24 heads of 64 on the benchmark grid: 714 -> 700 us in a
// loop at the power limit, 660 -> 644 us in bursts).  At head_dim 128 all columns are taken.  The visible keys are a short list of
// contiguous cache-row runs (sink, ring, wrapped ring); softmax does not care about
// key order, so the only masking is the ragged last tile of each run.
//
// Every mbarrier wait is bounded: a role that waits longer than kWaitLimitNs
// records a status word, raises the CTA's abort flag, and all roles drain to the
// common exit where TMEM is released.
#include <cuda_bf16.h>

#include <atomic>

#include "bounded_wait.cuh"
#include "exp2_poly.cuh"
#include "ll_internal.h"
#include "ptx.cuh"

namespace ll {

namespace {

using namespace ptx;

constexpr int kThreads = 640;
constexpr int kSoftmaxWarps = 16;
constexpr int kTmaWarp = 16;
constexpr int kMmaWarp = 17;
// A piece's 16 weights per thread and row were safe to compute if they sum to less than this:
// no weight can exceed the sum, and a score too far above the row's reference shows up as a
// weight of at least 2^127 on the special-function unit and of just under 256 (the top of its
// clamped range) on the polynomial path.  (A limit of 2^32 moves the references less often and makes
// eight streams with outliers 6 % faster, but the largest weight of a row is then hardly ever exactly
// 1, and its rounding shows: relative error 1.8e-3 instead of 1.6e-3.)
constexpr float kSafeSum = 128.f;
// Register reallocation draws on what the CTA was launched with: 640 threads x 96
// registers = (16 softmax warps x kSoftmaxRegs + 4 producer-group warps x kProducerRegs) x 32.  A
// request beyond that total would block forever.  The softmax warps take what the producers can spare: at head_dim 64
// they hold a whole score tile, at 128 a row's O when the references move (64 registers either way).
constexpr int kLaunchRegs = 96, kSoftmaxRegs = 112, kProducerRegs = 32;
static_assert(kSoftmaxWarps * kSoftmaxRegs + (kThreads / 32 - kSoftmaxWarps) * kProducerRegs <= (kThreads / 32) * kLaunchRegs,
              "setmaxnreg targets exceed the CTA's register allocation");
// 8-key groups (bit k of 16 per 128-key tile) whose exponentials use the cubic instead of the
// special-function unit.  head_dim 128: none - the special-function unit is not what a step
// waits for, and the cubic's ten instructions per pair cost time and power (0.4027 ms against
// 0.4047 ms with one group in four, 0.4218 ms with two; 0.4664 / 0.4715 / 0.4915 ms in a long
// loop at the power cap).  head_dim 64 has twice the exponentials per flop and is bound by
// them: one group in four (24 heads on the same grid, 605 us in bursts and 672 in a loop; the other 14 of 15 masks of none
// to half of the groups take 606 to 718 and 671 to 782).
template <int D> constexpr uint32_t kPolyMask = D == 64 ? 0x8888u : 0x0000u;

template <int D>
struct Cfg {
    static constexpr int kAtoms = D / 64;                   // 128-byte swizzle atoms per row
    static constexpr int kAtomBytes = 128 * 128;            // 128 rows x 128 bytes
    static constexpr int kTileBytes = kAtoms * kAtomBytes;  // one 128-row tile of Q, K or V
    static constexpr bool kPInTmem = D == 64;               // P (bf16) in tensor memory, or in shared memory
    static constexpr int kPBytes = (kPInTmem ? kAtoms : 2) * kAtomBytes;   // one lane's P: 128 rows x 128 keys; or its output rows
    static constexpr int kStages = (D == 128) ? 3 : 8;
    static constexpr int kSmemTiles = 2 * kTileBytes + 2 * kPBytes + kStages * kTileBytes;
    static constexpr int kSmemBytes = kSmemTiles + 1024 /*barriers*/ + 1024 /*alignment slack*/;
    static constexpr int kTmemCols = 512;
    static constexpr int kColS = 0;                         // S_w at kColS + 128 w
    static constexpr int kColO = 256;                       // O_w at kColO + D w
    static constexpr int kColP = 384;                       // P_w at kColP + 64 w (kPInTmem; two keys per column)
    // A move of the references rescales the O rows behind the piece's P instead of in front of it: then the piece's registers
    // are free and all loads of a row go out together (eight streams with outliers, which move in every fourth piece:
    // 3750 -> 3512 us; the benchmark layer's decode, which hardly moves, 473 us, the same within what runs differ).  In chunks of 64
    // columns with 104 registers the decode took 507 us; at head_dim 64, whose loop has no registers to spare, 742 instead of 702 us.
    static constexpr bool kRescaleLate = D == 128;
    static constexpr int kOChunks = D / 64;                 // 64-column pieces of an O row
};

// barrier indices inside the shared barrier array (+ lane or + stage)
enum Bar {
    kQFull = 0, kQEmpty = 2, kSFull = 4, kSEmpty = 6, kPFull = 8, kPEmpty = 10, kOFull = 12, kOEmpty = 14,
    kKvFull = 16, kKvEmpty = 24, kNumBars = 32,
    kPartFull = 32, kNumBarsParts = kPartFull + kSlabs      // kFormParts: the other parts' rows of a slab are in their slots
};

// Which launches an instance of the kernel serves.  At head_dim 128 one serves columns and tiles; at 64, whose loop has no registers
// to spare, the code for tiles costs the others 0.7 % (698 -> 703 us, 24 heads of 64 on the benchmark grid).
enum Form { kFormColumns, kFormTiles /* columns too */, kFormParts /* AttnParams::cluster_parts */ };

// Walks the visible key tiles of a group: runs in order, 128 rows at a time.
struct KeyIter {
    const AttnGroup *g;
    int r, off;
    __device__ KeyIter(const AttnGroup *grp, int run, int offset) : g(grp), r(run), off(offset) {}
    __device__ KeyIter(const AttnGroup *grp, int first_tile) : g(grp), r(0), off(0)
    {
        while (first_tile > 0) {
            const int nt = (g->k_len[r] + kKeyTile - 1) / kKeyTile;
            if (first_tile >= nt) { first_tile -= nt; ++r; }
            else { off = first_tile * kKeyTile; first_tile = 0; }
        }
    }
    __device__ int row() const { return g->k_start[r] + off; }
    __device__ void next()
    {
        off += kKeyTile;
        if (off >= g->k_len[r]) { ++r; off = 0; }
    }
};

// One CTA's piece of one column.
struct Segment {
    int g, head, tile;      // the column
    int kt0, kt1;           // its steps [kt0, kt1) run here
    int q0;                 // first query row of the column
    int rows_valid;         // live rows of the 256
    int n_sub;              // live 128-row tiles
    int col_begin;          // shared-step index of the column's first step (split columns only)
};

// A CTA's work in order: its whole columns, wave by wave, then its share of the steps
// that are left.  Every role of the CTA walks the same sequence.
template <int kForm>
struct WorkIter {
    static constexpr bool kTiles = kForm == kFormTiles;
    const AttnParams &p;
    int cta, g, wave, share;
    int u, end;
    __device__ WorkIter(const AttnParams &prm, int cta_)
        : p(prm), cta(cta_), g(0), wave(0), share(kForm == kFormParts ? cta_ : prm.share_of_cta[cta_]), u(0), end(0)
    {
        if (kForm == kFormParts) {
        } else if (kTiles && p.tile_ctas > 0) {
            u = cta * p.tiles_each + min(cta, p.tiles_extra);
            end = u + p.tiles_each + (cta < p.tiles_extra ? 1 : 0);
        } else if (share >= 0) {
            u = p.share_begin[share];
            end = p.share_begin[share + 1];
        }
    }
    // Goes on behind the piece of work that was looked up first (First).
    __device__ WorkIter(const AttnParams &prm, int cta_, const int (&state)[4])
        : p(prm), cta(cta_), g(state[0]), wave(state[1]), share(0), u(state[2]), end(state[3]) {}
    __device__ void fill(Segment &s, int grp, int col, int kt0, int kt1) const
    {
        const AttnGroup &G = p.g[grp];
        s.g = grp;
        s.head = col / G.tiles;
        s.tile = col - s.head * G.tiles;
        s.kt0 = kt0;
        s.kt1 = kt1;
        s.q0 = G.q_begin + s.tile * kQTileRows;
        s.rows_valid = min(kQTileRows, G.q_rows - s.tile * kQTileRows);
        s.n_sub = s.rows_valid > 128 ? 2 : 1;
    }
    __device__ bool next(Segment &s)
    {
        if (kForm == kFormParts) {                       // share `cta`, from its definition: the n-th part of a column
            if (wave++ > 0) return false;
            const int n = p.cluster_parts, col = cta / n, i = cta - col * n;
            while (col >= p.g[g].col_begin + p.heads * p.g[g].tiles) ++g;
            const AttnGroup &G = p.g[g];
            fill(s, g, col - G.col_begin, i * G.n_kt / n, (i + 1) * G.n_kt / n);
            s.col_begin = 0;
            return true;
        }
        if (kTiles && p.tile_ctas > 0) {
            if (u >= end) return false;
            while (u >= p.g[g].tile_begin + p.heads * p.g[g].row_tiles) ++g;
            const AttnGroup &G = p.g[g];
            const int off = u - G.tile_begin, head = off / G.row_tiles, t = off - head * G.row_tiles;
            s.g = g;
            s.head = head;
            s.tile = 0;
            s.kt0 = s.col_begin = 0;
            s.kt1 = G.n_kt;
            s.n_sub = min(min(2, end - u), G.row_tiles - t);
            s.q0 = G.q_begin + 128 * t;
            s.rows_valid = min(128 * s.n_sub, G.q_rows - 128 * t);
            u += s.n_sub;
            return true;
        }
        if (wave < p.n_waves) {
            const int col = wave * p.n_ctas + cta;                  // launch-wide column number
            ++wave;
            if (col < p.all_cols) {
                while (col >= p.g[g].col_begin + p.heads * p.g[g].tiles) ++g;
                fill(s, g, col - p.g[g].col_begin, 0, p.g[g].n_kt);
                s.col_begin = 0;
                return true;
            }
        }
        if (u >= end) return false;
        int gg = 0;
        while (gg + 1 < p.n_groups && u >= p.g[gg + 1].step_begin) ++gg;
        const AttnGroup &G = p.g[gg];
        const int off = u - (int)G.step_begin;
        const int col = off / G.n_kt;
        const int kt0 = off - col * G.n_kt;
        const int kt1 = min(G.n_kt, kt0 + (end - u));
        fill(s, gg, G.wave_cols + col, kt0, kt1);
        s.col_begin = u - kt0;
        u += kt1 - kt0;
        return true;
    }
};

// A CTA's first piece of work, where its keys begin, and what its WorkIter goes on from, in shared memory.
struct First {
    Segment s;
    int any, run, off, state[4];
};

// -inf into the registers of one 64-column piece (first column col0) whose key is not valid.
__device__ __forceinline__ void mask_piece(uint32_t *v, int col0, int cq, int nvalid)
{
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (col0 + 8 * k + cq >= nvalid) v[4 * k] = v[4 * k + 2] = 0xff800000u;
        if (col0 + 8 * k + cq + 1 >= nvalid) v[4 * k + 1] = v[4 * k + 3] = 0xff800000u;
    }
}

// The warp's 16 O rows times their rows' factors, WIDTH columns (half as many registers) at a time.
template <int WIDTH, int D>
__device__ __forceinline__ void rescale_o(uint32_t t_o, float al_a, float al_b)
{
    constexpr int kRegs = WIDTH / 2;
    tc_fence_after_sync();
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += WIDTH) {
        uint32_t o[kRegs];
        if constexpr (WIDTH == 32) {
            tmem_ld_16x256b_x4(t_o + c0, o);
        } else {
#pragma unroll
            for (int c = 0; c < WIDTH; c += 64) tmem_ld_16x256b_x8(t_o + c0 + c, o + c / 2);
        }
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < kRegs; k += 4) {
            o[k] = as_u(as_f(o[k]) * al_a);
            o[k + 1] = as_u(as_f(o[k + 1]) * al_a);
            o[k + 2] = as_u(as_f(o[k + 2]) * al_b);
            o[k + 3] = as_u(as_f(o[k + 3]) * al_b);
        }
        if constexpr (WIDTH == 32) {
            tmem_st_16x256b_x4(t_o + c0, o);
        } else {
#pragma unroll
            for (int c = 0; c < WIDTH; c += 64) tmem_st_16x256b_x8(t_o + c0 + c, o + c / 2);
        }
    }
    tmem_wait_st();
    tc_fence_before_sync();
}

// Where a softmax warp's 16 rows sit: q = TMEM lane quarter, w = lane (query tile) of the column, h = half
// of the quarter.
struct WarpRows {
    int lane, q, w, h;
    __device__ WarpRows(int warp, int lane_) : lane(lane_), q(warp & 3), w(warp >> 3), h((warp >> 2) & 1) {}
    __device__ int first() const { return 32 * q + 16 * h; }              // inside the lane's 128-row tile
    __device__ int row_a() const { return first() + (lane >> 2); }        // row of registers 4k+{0,1}; 4k+{2,3} are row_a + 8
    __device__ int slab() const { return w * 8 + q * 2 + h; }
};

// 64 columns (chunk ch) of the warp's rows, packed as pp of a softmax piece, to the output.  They go through
// the lane's P tile (its last PV has completed; every warp uses its own 16 rows), so that eight
// threads store 128 contiguous bytes of a row instead of four storing 16: 30.0 -> 26.7 us for a launch of
// two columns of four steps per CTA (4680 queries, 512 keys, 12 heads of 128).
template <int D>
__device__ __forceinline__ void store_rows(const AttnParams &p, const AttnItem &item, const Segment &s, const WarpRows &wr, uint32_t p_smem,
                                           uint32_t p_at, int ch, const uint32_t (&pk)[16])
{
    using C = Cfg<D>;
    const uint32_t at = p_at + ch * C::kAtomBytes;
    stmatrix_x4(at, pk[0], pk[2], pk[4], pk[6]);                       // rows a, chunks 0..3
    stmatrix_x4(at ^ 64u, pk[8], pk[10], pk[12], pk[14]);               // rows a, chunks 4..7
    stmatrix_x4(at + 8 * 128, pk[1], pk[3], pk[5], pk[7]);              // rows a + 8
    stmatrix_x4((at ^ 64u) + 8 * 128, pk[9], pk[11], pk[13], pk[15]);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {                                      // rows 4 i + lane / 8 of the warp's 16, 16-byte chunk lane % 8
        const int r = 4 * i + (wr.lane >> 3), row = 128 * wr.w + wr.first() + r;
        const uint4 x = ld_shared_v4(p_smem + wr.w * C::kPBytes + ch * C::kAtomBytes + (uint32_t)(wr.first() + r) * 128 +
                                     ((uint32_t)((wr.lane ^ r) & 7) << 4));
        if (row < s.rows_valid)
            *reinterpret_cast<uint4 *>(item.out + ((size_t)(s.q0 + row) * p.heads + s.head) * D + 64 * ch + 8 * (wr.lane & 7)) = x;
    }
}

// The log of the rows' sums (reference maxima m, sums l of rows a and a + 8), when the caller wants it.
__device__ __forceinline__ void store_lse(const AttnItem &item, const Segment &s, const WarpRows &wr, float m_a, float m_b, float l_a, float l_b)
{
    if (!item.lse || (wr.lane & 3)) return;
    const int row = 128 * wr.w + wr.row_a();
    float *lse = item.lse + (size_t)s.head * item.nq_total + s.q0 + row;
    if (row < s.rows_valid) lse[0] = (m_a + log2f(l_a)) * 0.6931471805599453f;
    if (row + 8 < s.rows_valid) lse[8] = (m_b + log2f(l_b)) * 0.6931471805599453f;
}

// The shares that hold parts of a split column: the first one, and how many (they are consecutive).
__device__ __forceinline__ void parts_of(const AttnParams &p, const Segment &s, int own, int &i0, int &n_parts)
{
    int i1 = own;
    i0 = own;
    while (p.share_begin[i0] > s.col_begin) --i0;
    while (p.share_begin[i1 + 1] < s.col_begin + p.g[s.g].n_kt) ++i1;
    n_parts = i1 - i0 + 1;
}

// Merges the parts of a split column for the warp's rows: reference maxima and sums first, then the O rows,
// always from the slots and in the order of the parts, so the result does not depend on
// which part happened to arrive last.  Up to kBatch parts it is bound by the latency of its loads, which
// therefore go out together (columns of three parts: 6.5 -> 3 us).  More parts are bound by their bytes, up to 128 KB
// each that one SM reads back: they go one by one, nothing read twice (in batches of four, the last one again
// behind the last: 8 heads of 128, 352 queries of two streams, six parts, 47.1 us a step, now 42.9).
template <int D>
__device__ __forceinline__ void merge_column(const AttnParams &p, const Segment &s, int own, const WarpRows &wr, uint32_t p_smem, uint32_t p_at)
{
    constexpr int kBatch = D == 64 ? 2 : 4;
    constexpr size_t kSlotFloats = (size_t)kQTileRows * (D + 2);
    int i0, n_parts;
    parts_of(p, s, own, i0, n_parts);
    const AttnItem &item = p.item[p.g[s.g].item];
    const int last = i0 + n_parts - 1, slab = wr.slab(), lane = wr.lane;
    auto part_slot = [&](int i) -> const float * { return p.partial + (size_t)(2 * i + (i == i0 ? 1 : 0)) * kSlotFloats; };
    auto part_ml = [&](int i) { return reinterpret_cast<const float2 *>(part_slot(i) + (size_t)kQTileRows * D) + slab * 16 + (lane >> 2); };
    float2 pa[kBatch], pb[kBatch];                     // (reference, sum) of a batch of parts, rows a and a + 8
    auto load_ml = [&](int first) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float2 *ml = part_ml(min(first + u, last));
            pa[u] = __ldcg(ml);
            pb[u] = __ldcg(ml + 8);
        }
    };
    float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
    for (int i = i0; i <= last; i += kBatch) {
        load_ml(i);                                    // (the last part again behind the last: no new maximum)
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            m_a = fmaxf(m_a, pa[u].x);
            m_b = fmaxf(m_b, pb[u].x);
        }
    }
    for (int i = i0; i <= last; i += kBatch) {
        if (n_parts > kBatch) load_ml(i);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (i + u > last) break;
            l_a = fmaf(pa[u].y, ex2(pa[u].x - m_a), l_a);
            l_b = fmaf(pb[u].y, ex2(pb[u].x - m_b), l_b);
        }
    }
    const float v_scale = item.v_scale ? item.v_scale[s.head] : 1.f;   // 8-bit caches: value codes x scale
    const float inv_a = v_scale / l_a, inv_b = v_scale / l_b;
#pragma unroll 1
    for (int ch = 0; ch < D / 64; ++ch) {
        uint32_t pk[16];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float o[16];                               // 32 columns: of each 16, this thread's four of row a, then of row a + 8
#pragma unroll
            for (int k = 0; k < 16; ++k) o[k] = 0.f;
            auto load_part = [&](float4 (&x)[4], int i) {
                const float4 *src = reinterpret_cast<const float4 *>(part_slot(i)) +
                                    (size_t)(slab * (D / 16) + 4 * ch + 2 * half) * 64 + lane;
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = __ldcg(src + 32 * k);
            };
            auto add_part = [&](const float4 (&x)[4], float ref_a, float ref_b) {
                const float wa = ex2(ref_a - m_a) * inv_a, wb = ex2(ref_b - m_b) * inv_b;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float wk = (k & 1) ? wb : wa;
                    o[4 * k] = fmaf(x[k].x, wk, o[4 * k]);
                    o[4 * k + 1] = fmaf(x[k].y, wk, o[4 * k + 1]);
                    o[4 * k + 2] = fmaf(x[k].z, wk, o[4 * k + 2]);
                    o[4 * k + 3] = fmaf(x[k].w, wk, o[4 * k + 3]);
                }
            };
            if (n_parts <= kBatch) {
                float4 x[kBatch][4];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) load_part(x[u], min(i0 + u, last));
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    if (i0 + u > last) break;
                    add_part(x[u], pa[u].x, pb[u].x);
                }
            } else {
                for (int i = i0; i <= last; ++i) {
                    const float2 *ml = part_ml(i);
                    const float ref_a = __ldcg(ml).x, ref_b = __ldcg(ml + 8).x;
                    float4 x[4];
                    load_part(x, i);
                    add_part(x, ref_a, ref_b);
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int g = 0; g < 2; ++g) {          // 8-column group 4 half + 2 k + g
                    pk[2 * (4 * half + 2 * k + g)] = cvt_bf16x2(o[8 * k + 2 * g], o[8 * k + 2 * g + 1]);
                    pk[2 * (4 * half + 2 * k + g) + 1] = cvt_bf16x2(o[8 * k + 4 + 2 * g], o[8 * k + 5 + 2 * g]);
                }
        }
        store_rows<D>(p, item, s, wr, p_smem, p_at, ch, pk);
    }
    store_lse(item, s, wr, m_a, m_b, l_a, l_b);
    __syncwarp();                                      // the P rows are read before another column's are staged
}

// The parts of a column that the CTAs of a cluster hold, merged for the warp's 16 rows.  Every CTA leaves what the others merge of
// its unnormalised rows in its scratch slot, tells the same warp of each of them, and merges an n-th of the columns itself: those
// of the 8-column groups k with k n / (D / 8) == its rank.  All SMs of the cluster then read and write (n - 1) / n of a part, where the one
// that arrives last reads back all parts: from the last product to the end 5 us for two parts of 256 rows where that takes 8
// (12 heads of 128, 1479 queries over 5916 keys; 450 over 2250, 8 heads: 24.6 us a call in four parts, 17.5 in six).  Through the cluster's shared memory the same exchange is slower (64 KB
// each way 4100 clk to send for two CTAs, 7800 for four; to L2 2900 and 3500), so only the barriers are there.
//   kPeers and kUnroll: other parts that x has room for, and groups at a time, so that about eight to fourteen loads are in flight.
template <int D, int kPeers, int kUnroll>
__device__ __forceinline__ void merge_groups(const AttnParams &p, const WarpRows &wr, int cta, int rank, int n, int g0, int g1, uint32_t t_o,
                                             float v_scale, uint32_t stage, float &m_a, float &m_b, float &l_a, float &l_b)
{
    constexpr int kGroups = D / 8;
    constexpr size_t kSlotFloats = (size_t)kQTileRows * (D + 2);
    const int lane = wr.lane, slab = wr.slab();
    // of the j-th peer (part j below this CTA's rank, part j + 1 from there on)
    auto slot = [&](int j) { return p.partial + (size_t)2 * (cta - rank + j + (j >= rank ? 1 : 0)) * kSlotFloats; };
    float4 x[kPeers][kUnroll];                         // of each group this thread's two columns of row a, then of row a + 8
    auto load_groups = [&](int k0) {
#pragma unroll
        for (int j = 0; j < kPeers; ++j) {
            const float4 *src = reinterpret_cast<const float4 *>(slot(j)) + (size_t)(slab * kGroups + k0) * 32 + lane;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                x[j][u] = (j < n - 1 && k0 + u < g1) ? __ldcg(src + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float2 ra[kPeers], rb[kPeers];                     // (reference, sum), rows a and a + 8
#pragma unroll
    for (int j = 0; j < kPeers; ++j) {
        const float2 *ml = reinterpret_cast<const float2 *>(slot(j) + (size_t)kQTileRows * D) + slab * 16 + (lane >> 2);
        ra[j] = j < n - 1 ? __ldcg(ml) : make_float2(-INFINITY, 0.f);
        rb[j] = j < n - 1 ? __ldcg(ml + 8) : make_float2(-INFINITY, 0.f);
    }
    constexpr bool kAhead = kPeers <= 3;               // the first groups are in flight with them (with more the registers do not suffice)
    if (kAhead) load_groups(g0);
    const float own_a = m_a, own_b = m_b;
#pragma unroll
    for (int j = 0; j < kPeers; ++j) {
        m_a = fmaxf(m_a, ra[j].x);
        m_b = fmaxf(m_b, rb[j].x);
    }
    float w_a = ex2(own_a - m_a), w_b = ex2(own_b - m_b);
    l_a *= w_a;
    l_b *= w_b;
#pragma unroll
    for (int j = 0; j < kPeers; ++j) {                 // from here on .x is the part's weight (0 behind the last)
        ra[j].x = ex2(ra[j].x - m_a);
        rb[j].x = ex2(rb[j].x - m_b);
        l_a = fmaf(ra[j].y, ra[j].x, l_a);
        l_b = fmaf(rb[j].y, rb[j].x, l_b);
    }
    const float inv_a = v_scale / l_a, inv_b = v_scale / l_b;
    w_a *= inv_a;
    w_b *= inv_b;
#pragma unroll
    for (int j = 0; j < kPeers; ++j) {
        ra[j].x *= inv_a;
        rb[j].x *= inv_b;
    }
#pragma unroll 1
    for (int k0 = g0; k0 < g1; k0 += kUnroll) {
        if (!kAhead || k0 > g0) load_groups(k0);
        uint32_t own[4 * kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            tmem_ld_16x256b_x1(t_o + 8 * min(k0 + u, kGroups - 1), own[4 * u], own[4 * u + 1], own[4 * u + 2], own[4 * u + 3]);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            float4 o = make_float4(as_f(own[4 * u]) * w_a, as_f(own[4 * u + 1]) * w_a, as_f(own[4 * u + 2]) * w_b, as_f(own[4 * u + 3]) * w_b);
#pragma unroll
            for (int j = 0; j < kPeers; ++j) {
                o.x = fmaf(x[j][u].x, ra[j].x, o.x);
                o.y = fmaf(x[j][u].y, ra[j].x, o.y);
                o.z = fmaf(x[j][u].z, rb[j].x, o.z);
                o.w = fmaf(x[j][u].w, rb[j].x, o.w);
            }
            const int k = k0 + u;
            if (k < g1)
                stmatrix_x2(stage + (k >> 3) * Cfg<D>::kAtomBytes + (((uint32_t)k ^ lane) & 7u) * 16, cvt_bf16x2(o.x, o.y), cvt_bf16x2(o.z, o.w));
        }
    }
}

template <int D, class Wait>
__device__ __forceinline__ bool merge_in_cluster(const AttnParams &p, const Segment &s, const WarpRows &wr, int cta, uint32_t t_o, float m_own_a,
                                                 float m_own_b, float l_own_a, float l_own_b, uint32_t p_smem, uint32_t part_bar, bool &told, Wait wait)
{
    using C = Cfg<D>;
    constexpr int kGroups = D / 8;
    const int n = p.cluster_parts, rank = (int)cluster_rank(), lane = wr.lane, slab = wr.slab();
    const int g0 = (rank * kGroups + n - 1) / n, g1 = ((rank + 1) * kGroups + n - 1) / n;
    float *slot = p.partial + (size_t)2 * cta * kQTileRows * (D + 2);
#pragma unroll 1
    for (int ch = 0; ch < C::kOChunks; ++ch) {
        uint32_t o[32];
        tmem_ld_16x256b_x8(t_o + 64 * ch, o);
        tmem_wait_ld();
        uint4 *dst = reinterpret_cast<uint4 *>(slot) + (size_t)(slab * kGroups + 8 * ch) * 32 + lane;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (8 * ch + k < g0 || 8 * ch + k >= g1) dst[32 * k] = make_uint4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
    }
    if ((lane & 3) == 0) {
        float2 *ml = reinterpret_cast<float2 *>(slot + (size_t)kQTileRows * D) + slab * 16 + (lane >> 2);
        ml[0] = make_float2(m_own_a, l_own_a);
        ml[8] = make_float2(m_own_b, l_own_b);
    }
    fence_cluster();
    __syncwarp();
    if (lane < n && lane != rank) mbar_arrive_remote(part_bar, (uint32_t)lane);
    told = true;
    if (!__all_sync(0xffffffffu, wait())) return false;
    const AttnItem &item = p.item[p.g[s.g].item];
    const float v_scale = item.v_scale ? item.v_scale[s.head] : 1.f;   // 8-bit caches: value codes x scale
    // the merged rows wait in the lane's P tile (its last PV has completed; every warp uses its own 16 rows) for 16-byte stores
    const uint32_t tile = p_smem + wr.w * C::kPBytes, stage = tile + (uint32_t)(wr.first() + (lane & 15)) * 128;
    float m_a = m_own_a, m_b = m_own_b, l_a = l_own_a, l_b = l_own_b;
    if (n == 2) merge_groups<D, 1, 8>(p, wr, cta, rank, n, g0, g1, t_o, v_scale, stage, m_a, m_b, l_a, l_b);
    else if (n <= 4) merge_groups<D, 3, 4>(p, wr, cta, rank, n, g0, g1, t_o, v_scale, stage, m_a, m_b, l_a, l_b);
    else merge_groups<D, 7, 2>(p, wr, cta, rank, n, g0, g1, t_o, v_scale, stage, m_a, m_b, l_a, l_b);
    __syncwarp();
    const int groups = g1 - g0, inv = (65536 + groups - 1) / groups;           // i / groups = i inv / 65536 for i below 128
    for (int i = lane; i < 16 * groups; i += 32) {
        const int r = (i * inv) >> 16, k = g0 + i - r * groups, row = 128 * wr.w + wr.first() + r;
        const uint4 v = ld_shared_v4(tile + (k >> 3) * C::kAtomBytes + (uint32_t)(wr.first() + r) * 128 + ((uint32_t)((k ^ r) & 7) << 4));
        if (row < s.rows_valid) *reinterpret_cast<uint4 *>(item.out + ((size_t)(s.q0 + row) * p.heads + s.head) * D + 8 * k) = v;
    }
    if (rank == 0) store_lse(item, s, wr, m_a, m_b, l_a, l_b);
    return true;
}

template <int D, int kForm>
__global__ void __launch_bounds__(kThreads, 1)
attn_sm100_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ AttnMaps maps)
{
    using C = Cfg<D>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t q_smem = smem_base;                                  // 2 tiles
    const uint32_t p_smem = smem_base + 2 * C::kTileBytes;              // one 64-key P tile per lane
    const uint32_t kv_smem = p_smem + 2 * C::kPBytes;                   // kStages tiles
    const uint32_t bars = smem_base + C::kSmemTiles;                    // kNumBars x 8 bytes
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_gen + C::kSmemTiles + kNumBarsParts * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    First *first = reinterpret_cast<First *>(tmem_slot + 2);
    static_assert(kNumBarsParts * 8 + 8 + sizeof(First) <= 1024, "barriers and first piece of work exceed their kilobyte");
    auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };

    // (the shuffle tells the compiler that the warp index is the same in all lanes, which
    // keeps the role code of the MMA warps on the uniform datapath)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int cta = blockIdx.x;

    // ---- setup ------------------------------------------------------------------
    grid_dep_launch();
    constexpr bool kParts = kForm == kFormParts;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < kNumBars; ++i) {
            uint32_t count = 1;
            if ((i >= kSEmpty && i < kSEmpty + 2) || (i >= kPFull && i < kPFull + 2) || (i >= kOEmpty && i < kOEmpty + 2))
                count = kSoftmaxWarps / 2;                                     // one arrival per softmax warp of the lane
            if (i == kQEmpty || i >= kKvEmpty) count = 2;                      // both MMA warps release Q and every K/V stage
            mbar_init(bar(i), count);
        }
        if (kParts)
            for (int i = 0; i < kSlabs; ++i) mbar_init(bar(kPartFull + i), p.cluster_parts - 1);     // the same warp of every other CTA of the cluster
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (kParts) cluster_arrive();
    if (warp == kTmaWarp) {
        tmem_alloc(smem_u32(tmem_slot), C::kTmemCols);
        tmem_relinquish();
        if (lane == 0)                                 // (the maps are launch parameters)
            for (int i = 0; i < p.n_items; ++i) {
                prefetch_tensormap(&maps.q[i]);
                prefetch_tensormap(&maps.k[i]);
                prefetch_tensormap(&maps.v[i]);
            }
    }
    // What a CTA's first piece of work is comes from the launch parameters: divisions, and loads from a constant cache that is cold, 1000
    // to 2500 clk which the first tiles would stand behind.  It is looked up for the load warp while the barriers and the tensor
    // memory are being set up; the other roles do so themselves while the tiles are on their way.  (With the maps fetched up here, too,
    // and the load warp not waiting for the status word: 12 heads of 128, 44 queries over 220 keys, 7.85 -> 7.24 us a call;
    // 4680 over 512 keys 22.1 -> 21.4 us.)
    if (threadIdx.x == 32) {
        WorkIter<kForm> it(p, cta);
        first->any = it.next(first->s);
        if (first->any) {
            const KeyIter k(&p.g[first->s.g], first->s.kt0);
            first->run = k.r;
            first->off = k.off;
        }
        first->state[0] = it.g;
        first->state[1] = it.wave;
        first->state[2] = it.u;
        first->state[3] = it.end;
    }
    if (kParts) cluster_wait();                        // every CTA of the cluster has its barriers
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_dep_wait();
    // An earlier CTA already gave up on a wait: this one does not start (flag value 2).  The load warp does not wait to hear of that: its
    // first tiles are under way meanwhile, and it finds the flag when it runs out of stages.
    if (warp == kTmaWarp) {
        named_arrive(1, kThreads);
    } else {
        if (threadIdx.x == 0 && *reinterpret_cast<volatile uint32_t *>(p.status) != kStatusOk) *abort_flag = 2;
        named_sync(1, kThreads);
    }

    WaitCtx ctx{abort_flag, p.status, warp};
    // (in a cluster another CTA may set the flag at any time: the lanes of a warp agree on what they saw)
    const bool skip = warp != kTmaWarp && (kParts ? __any_sync(0xffffffffu, *abort_flag != 0) : *abort_flag != 0);
    bool told = false;                                 // kParts: this warp has arrived at its peers' barriers
    auto wait = [&](int bar_id, uint32_t parity, int iter) -> bool {
        return wait_bar(bar(bar_id), parity & 1u, ctx, bar_id, iter);
    };

    if (warp >= kSoftmaxWarps) {
        // Register reallocation: the softmax warps hold 32 or 64 scores per thread,
        // the producer warpgroup (TMA, MMA and two idle warps) needs little.
        setmaxnreg_dec<kProducerRegs>();
        if (skip) {
            // an earlier CTA gave up: nothing to do
        } else if (warp == kTmaWarp && lane == 0) {
            // =========================== TMA producer ===========================
            [&]() {
                uint32_t n = 0;                 // K/V tiles issued so far
                uint32_t seg = 0;
                WorkIter<kForm> it(p, cta, first->state);
                Segment s = first->s;
                int run = first->run, off = first->off;
                for (bool more = first->any; more; more = it.next(s), ++seg) {
                    // Tile order K_0, K_1, V_0, K_2, V_1, ... : the QK of a step is issued a whole
                    // softmax ahead of the step's PV, so K runs one step ahead of V and three stages
                    // (the V in use, the K in use, one in flight) keep both fed.
                    if (seg > 0) {
                        const KeyIter k(&p.g[s.g], s.kt0);
                        run = k.r;
                        off = k.off;
                    }
                    KeyIter kit(&p.g[s.g], run, off);
                    int row = kit.row();
                    const int item = p.g[s.g].item;
                    const CUtensorMap *qmap = &maps.q[item], *kmap = &maps.k[item], *vmap = &maps.v[item];
                    auto load_kv = [&](const CUtensorMap *m, int row) -> bool {
                        const int stage = n % C::kStages;
                        if (!wait(kKvEmpty + stage, (n / C::kStages) ^ 1u, (int)n)) return false;
                        mbar_arrive_expect_tx(bar(kKvFull + stage), C::kTileBytes);
                        for (int a = 0; a < C::kAtoms; ++a)
                            tma_load_3d(kv_smem + stage * C::kTileBytes + a * C::kAtomBytes, m,
                                        bar(kKvFull + stage), a * 64, p.kv_token_major ? s.head : row,
                                        p.kv_token_major ? row : s.head);
                        ++n;
                        return true;
                    };
                    // the first key tile goes out before Q: it needs no Q buffer and is in
                    // flight while the previous column's last products drain
                    if (!load_kv(kmap, row)) return;
                    if (seg > 0 && !wait(kQEmpty, seg - 1, (int)seg)) return;
                    for (int w = 0; w < s.n_sub; ++w) {
                        mbar_arrive_expect_tx(bar(kQFull + w), C::kTileBytes);
                        for (int a = 0; a < C::kAtoms; ++a)
                            tma_load_3d(q_smem + w * C::kTileBytes + a * C::kAtomBytes, qmap, bar(kQFull + w),
                                        a * 64, s.head, s.q0 + 128 * w);
                    }
                    for (int j = s.kt0; j < s.kt1; ++j) {
                        const int v_row = row;
                        if (j + 1 < s.kt1) {
                            kit.next();
                            row = kit.row();
                            if (!load_kv(kmap, row)) return;
                        }
                        if (!load_kv(vmap, v_row)) return;
                    }
                }
            }();
        } else if (warp == kMmaWarp || warp == kMmaWarp + 1) {
            // ====================== MMA issuer of lane w = warp - kMmaWarp ======================
            // One issuing warp per lane.  Both walk the same K/V ring and both release every
            // stage (a lane that sits a column out releases it unused).  All 32 lanes walk the
            // loops and the waits, so that addresses and descriptors are warp-uniform values;
            // one elected lane issues the MMAs, commits and arrivals.
            [&]() {
                const int w = warp - kMmaWarp;
                const bool elected = elect_one();
                constexpr uint32_t idesc_qk = idesc_bf16_f32(128, 128, 0, 0);
                constexpr uint32_t idesc_pv = idesc_bf16_f32(128, D, 0, 1);
                constexpr uint32_t hi = smem_desc_hi_sw128(1024);
                const uint32_t t_sw = tmem + C::kColS + 128 * w, t_ow = tmem + C::kColO + D * w, t_pw = tmem + C::kColP + 64 * w;
                // S_w = Q_w K^T: both operands K-major, 64-element atoms, 16 elements (32 bytes) per MMA
                const uint32_t q_lo = smem_desc_lo(q_smem + w * C::kTileBytes, 16);
                const uint32_t k_lo0 = smem_desc_lo(kv_smem, 16);
                // O_w += P_w V: P K-major (one 64-key atom, 16 keys = 32 bytes per MMA); V is MN-major:
                // 8-key groups 1024 bytes apart, 64-wide d atoms kAtomBytes apart
                const uint32_t p_lo = smem_desc_lo(p_smem + w * C::kPBytes, 16);
                const uint32_t v_lo0 = smem_desc_lo(kv_smem, C::kAtomBytes);
                auto issue_qk = [&](uint32_t stage) {
                    const uint32_t k_lo = k_lo0 + stage * (C::kTileBytes >> 4);
                    if (elected) {
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint32_t off = ((kk / 4) * C::kAtomBytes + (kk % 4) * 32) >> 4;
                            mma_ss(t_sw, smem_desc_join(q_lo + off, hi), smem_desc_join(k_lo + off, hi), idesc_qk, kk > 0);
                        }
                    }
                    __syncwarp();
                };
                auto issue_pv = [&](uint32_t stage, bool first) {
                    const uint32_t v_lo = v_lo0 + stage * (C::kTileBytes >> 4);
                    if (elected) {
#pragma unroll
                        for (int kk = 0; kk < kKeyTile / 16; ++kk)
                            if (C::kPInTmem)
                                mma_ts(t_ow, t_pw + 8 * kk, smem_desc_join(v_lo + ((kk * 2048) >> 4), hi), idesc_pv, (!first || kk > 0) ? 1u : 0u);
                            else
                                mma_ss(t_ow, smem_desc_join(p_lo + (((kk / 4) * C::kAtomBytes + (kk % 4) * 32) >> 4), hi),
                                       smem_desc_join(v_lo + ((kk * 2048) >> 4), hi), idesc_pv, (!first || kk > 0) ? 1u : 0u);
                    }
                    __syncwarp();
                };
                auto commit = [&](int bar_id) { if (elected) tc_commit(bar(bar_id)); };
                auto arrive = [&](int bar_id) { if (elected) mbar_arrive(bar(bar_id)); };
                // tile n of the producer's sequence K_0, K_1, V_0, K_2, V_1, ... sits in stage n % kStages
                auto kv_wait = [&](uint32_t n) -> bool { return wait(kKvFull + n % C::kStages, n / C::kStages, (int)n); };
                uint32_t n0 = 0;                // producer index of the column's first tile
                uint32_t sc = 0;                // steps this lane has been through
                uint32_t oc = 0;                // columns this lane took part in so far
                uint32_t seg = 0;
                Segment s;
                for (WorkIter<kForm> it(p, cta); it.next(s); ++seg) {
                    const int n_steps = s.kt1 - s.kt0;
                    if (w >= s.n_sub) {
                        // not this lane's column: pass every stage on once its tile has landed, and
                        // the Q buffers once the previous column's release is complete
                        for (int t = 0; t < 2 * n_steps; ++t) {
                            if (!kv_wait(n0 + t)) return;
                            arrive(kKvEmpty + (n0 + t) % C::kStages);
                        }
                        n0 += 2 * n_steps;
                        if (seg > 0 && !wait(kQEmpty, seg - 1, (int)seg)) return;
                        arrive(kQEmpty);
                        continue;
                    }
                    if (!wait(kQFull + w, oc, 0)) return;
                    // QK of the column's first step: its S buffer was read out by the last softmax
                    if (!kv_wait(n0)) return;
                    if (sc > 0 && !wait(kSEmpty + w, sc - 1, (int)sc)) return;
                    tc_fence_after_sync();
                    issue_qk(n0 % C::kStages);
                    commit(kSFull + w);
                    commit(kKvEmpty + n0 % C::kStages);
                    if (n_steps == 1) commit(kQEmpty);
                    for (int j = 0; j < n_steps; ++j, ++sc) {
                        const bool more = j + 1 < n_steps;
                        const uint32_t nk = n0 + 2 * j + 1;                     // K_j+1 (if any)
                        const uint32_t nv = more ? nk + 1 : nk;                 // V_j
                        // QK of the next step as soon as the softmax warps hold S_j in registers
                        if (more) {
                            if (!kv_wait(nk)) return;
                            if (!wait(kSEmpty + w, sc, (int)sc)) return;
                            tc_fence_after_sync();
                            issue_qk(nk % C::kStages);
                            commit(kSFull + w);
                            commit(kKvEmpty + nk % C::kStages);
                            if (j + 2 == n_steps) commit(kQEmpty);               // the column's last QK is in the pipe
                        }
                        if (!kv_wait(nv)) return;
                        // the previous column's O rows must have been read out
                        if (j == 0 && oc > 0 && !wait(kOEmpty + w, oc - 1, (int)oc)) return;
                        if (!wait(kPFull + w, sc, (int)sc)) return;
                        tc_fence_after_sync();
                        issue_pv(nv % C::kStages, j == 0);
                        commit(kPEmpty + w);
                        commit(kKvEmpty + nv % C::kStages);
                        if (!more) commit(kOFull + w);
                    }
                    n0 += 2 * n_steps;
                    ++oc;
                }
            }();
        }
    } else {
        // ============================= softmax warps =============================
        setmaxnreg_inc<kSoftmaxRegs>();
        if (!skip) [&]() {
            const WarpRows wr(warp, lane);
            const int w = wr.w;
            const uint32_t lane_off = (uint32_t)wr.first() << 16;   // the TMEM lanes this warp reads
            const uint32_t t_s = tmem + lane_off + C::kColS + 128 * w;
            const uint32_t t_o = tmem + lane_off + C::kColO + D * w;
            const uint32_t t_p = tmem + lane_off + C::kColP + 64 * w;
            const int cq = 2 * (lane & 3);                     // first of this thread's two columns in each group of 8
            // P at head_dim 128, and output rows, go to shared memory with stmatrix: of the warp's 16 rows x 64 keys, one call
            // stores four 8-row x 8-key blocks (a block row = one 16-byte chunk); lane 8m + r gives the
            // address of row r of the block holding chunk m, which sits at chunk position m ^ r.
            // Chunks 4..7 are at the same address ^ 64, the second eight rows 1024 bytes on.
            const uint32_t p_at = p_smem + w * C::kPBytes + (uint32_t)(wr.first() + (lane & 7)) * 128 +
                                  ((uint32_t)((lane >> 3) ^ (lane & 7)) << 4);
            uint32_t sc = 0, oc = 0;
            constexpr bool kMergeLate = D == 64;
            uint32_t to_merge = 0;                             // which of the CTA's two parts complete a column here
            Segment s;
            for (WorkIter<kForm> it(p, cta); it.next(s);) {
                if (w >= s.n_sub) continue;
                const AttnGroup &G = p.g[s.g];
                // keys left in the current run of the visible set (its last tile may be ragged)
                int run, left;
                {
                    const KeyIter first(&G, s.kt0);
                    run = first.r;
                    left = G.k_len[run] - first.off;
                }
                // log2(e)/sqrt(D), times the head's key scale when the cache holds 8-bit codes
                const float *k_scale = p.item[G.item].k_scale;
                const float c = k_scale ? p.scale_log2 * k_scale[s.head] : p.scale_log2;
                // ... and times the query row's own factor when the caller brings one (a q/k norm whose
                // per-token factor was left out of the stored q)
                float c_a = c, c_b = c;
                if (const float *q_scale = p.item[G.item].q_scale) {
                    const int r = 128 * w + wr.row_a();
                    if (r < s.rows_valid) c_a *= q_scale[s.q0 + r];
                    if (r + 8 < s.rows_valid) c_b *= q_scale[s.q0 + r + 8];
                }
                float m_a = -INFINITY, m_b = -INFINITY;
                uint64_t acc_a = 0ull, acc_b = 0ull;       // two partial sums per row
                for (int j = s.kt0; j < s.kt1; ++j, ++sc) {
                    if (!__all_sync(0xffffffffu, wait(kSFull + w, sc, j))) return;
                    tc_fence_after_sync();
                    const int nvalid = min(left, kKeyTile);
                    left -= kKeyTile;
                    if (left <= 0 && j + 1 < s.kt1) left = G.k_len[++run];
                    // head_dim 64: the whole tile goes to registers at once and the S buffer back to the
                    // MMA warp, so that the next QK and its hand-overs run under all of this step's
                    // weights (2480 -> 2350 clk per step; 24 heads of 64: 0.744 -> 0.707 ms at the power
                    // limit).  At head_dim 128 it is taken 64 columns at a time: there the early release
                    // costs cycles and energy (0.478 ms against 0.514 ms; 455 mJ against 488 mJ per call).
                    constexpr bool kWholeTile = D == 64;
                    uint32_t s_tile[kWholeTile ? 64 : 32];
                    auto release_s = [&]() {
                        tmem_wait_ld();
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kSEmpty + w));
                    };
                    if (kWholeTile) {
                        tmem_ld_16x256b_x8(t_s, s_tile);
                        tmem_ld_16x256b_x8(t_s + 64, s_tile + (kWholeTile ? 32 : 0));
                        release_s();
                    }
                    // The tile is worked through in two 64-key pieces.  A piece's exponentials are computed
                    // against the rows' current reference maxima straight away; its sums then tell
                    // whether that was safe (no weight can exceed the sum).  Only when some sum in
                    // the warp is too large or not finite - and on a column's first piece, which has
                    // no references yet - are the exact row maxima taken, the references moved,
                    // what has been accumulated rescaled, and the piece computed against them.
#pragma unroll
                    for (int piece = 0; piece < 2; ++piece) {
                        uint32_t *v = s_tile + (kWholeTile ? 32 * piece : 0);
                        uint32_t pp[16];                           // the piece's P: 16 rows x 64 keys per warp
                        if (!kWholeTile) {
                            tmem_ld_16x256b_x8(t_s + 64 * piece, v);
                            if (piece == 0) tmem_wait_ld(); else release_s();
                        }
                        if (nvalid < kKeyTile) mask_piece(v, 64 * piece, cq, nvalid);
                        uint64_t ts_a = 0ull, ts_b = 0ull;         // the piece's sums, two partials per row
                        const bool fresh = piece == 0 && j == s.kt0;   // nothing accumulated yet, no references
                        if (!fresh) {
                            const uint64_t na2 = pack2(-m_a, -m_a), nb2 = pack2(-m_b, -m_b);
                            const uint64_t c2a = pack2(c_a, c_a), c2b = pack2(c_b, c_b);
                            const PolyRow ra{c_a * (1.f / 128.f), ((float)kPolyLow - m_a) * (1.f / 128.f)};
                            const PolyRow rb{c_b * (1.f / 128.f), ((float)kPolyLow - m_b) * (1.f / 128.f)};
                            // Four 8-key groups at a time, stage by stage, so that the exponentials of a
                            // batch are all in flight before the first result is needed.
#pragma unroll
                            for (int g = 0; g < 2; ++g) {
                                uint64_t xa[4], xb[4];
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk) {
                                    const int k = 4 * g + kk;
                                    if (!((kPolyMask<D> >> (8 * piece + k)) & 1u)) {
                                        xa[kk] = fma2(pack2(as_f(v[4 * k]), as_f(v[4 * k + 1])), c2a, na2);
                                        xb[kk] = fma2(pack2(as_f(v[4 * k + 2]), as_f(v[4 * k + 3])), c2b, nb2);
                                    }
                                }
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk) {
                                    const int k = 4 * g + kk;
                                    if ((kPolyMask<D> >> (8 * piece + k)) & 1u) {
                                        xa[kk] = exp2_poly2(as_f(v[4 * k]), as_f(v[4 * k + 1]), ra);
                                        xb[kk] = exp2_poly2(as_f(v[4 * k + 2]), as_f(v[4 * k + 3]), rb);
                                    } else {
                                        xa[kk] = exp2_sfu2(xa[kk]);
                                        xb[kk] = exp2_sfu2(xb[kk]);
                                    }
                                }
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk) {
                                    const int k = 4 * g + kk;
                                    ts_a = add2(ts_a, xa[kk]);
                                    ts_b = add2(ts_b, xb[kk]);
                                    float a0, a1, b0, b1;
                                    unpack2(xa[kk], a0, a1);
                                    unpack2(xb[kk], b0, b1);
                                    pp[2 * k] = cvt_bf16x2(a0, a1);        // key 8k + cq in the low half
                                    pp[2 * k + 1] = cvt_bf16x2(b0, b1);
                                }
                            }
                        }
                        bool move = fresh;
                        float al_a = 0.f, al_b = 0.f;              // what a move multiplies everything before it by
                        if (!fresh) {
                            float x0, x1, y0, y1;
                            unpack2(ts_a, x0, x1);
                            unpack2(ts_b, y0, y1);
                            move = __any_sync(0xffffffffu, !(x0 + x1 < kSafeSum) || !(y0 + y1 < kSafeSum));
                        }
                        if (move) {
                            // exact maxima of the piece's rows: 16 columns per thread, then across the quad
                            float ta = fmaxf(as_f(v[0]), as_f(v[1])), tb = fmaxf(as_f(v[2]), as_f(v[3]));
#pragma unroll
                            for (int k = 1; k < 8; ++k) {
                                ta = max3(ta, as_f(v[4 * k]), as_f(v[4 * k + 1]));
                                tb = max3(tb, as_f(v[4 * k + 2]), as_f(v[4 * k + 3]));
                            }
                            ta = fmaxf(ta, __shfl_xor_sync(0xffffffffu, ta, 1));
                            tb = fmaxf(tb, __shfl_xor_sync(0xffffffffu, tb, 1));
                            ta = fmaxf(ta, __shfl_xor_sync(0xffffffffu, ta, 2)) * c_a;
                            tb = fmaxf(tb, __shfl_xor_sync(0xffffffffu, tb, 2)) * c_b;
                            const float new_a = fresh ? ta : fmaxf(m_a, ta), new_b = fresh ? tb : fmaxf(m_b, tb);
                            if (!fresh) {
                                al_a = ex2(m_a - new_a);
                                al_b = ex2(m_b - new_b);
                            }
                            m_a = new_a;
                            m_b = new_b;
                            acc_a = fma2(acc_a, pack2(al_a, al_a), 0ull);
                            acc_b = fma2(acc_b, pack2(al_b, al_b), 0ull);
                            if (piece == 1) {
                                // the first piece's P is stored already, against the old
                                // references: take it back, rescale, store again (nobody else reads it
                                // before this step's hand-over)
                                auto scale = [](uint32_t x, float al) {
                                    return cvt_bf16x2(as_f(x << 16) * al, as_f(x & 0xffff0000u) * al);
                                };
                                if constexpr (C::kPInTmem) {
                                    uint32_t r[16];
                                    tmem_wait_st();
                                    tmem_ld_16x128b_x8(t_p, r);
                                    tmem_wait_ld();
#pragma unroll
                                    for (int k = 0; k < 8; ++k) {
                                        r[2 * k] = scale(r[2 * k], al_a);
                                        r[2 * k + 1] = scale(r[2 * k + 1], al_b);
                                    }
                                    tmem_st_16x128b_x8(t_p, r);
                                } else {
                                    __syncwarp();
#pragma unroll
                                    for (int half = 0; half < 2; ++half) {
                                        const uint32_t at = half ? (p_at ^ 64u) : p_at;
                                        uint32_t ra0, ra1, ra2, ra3, rb0, rb1, rb2, rb3;
                                        ldmatrix_x4(at, ra0, ra1, ra2, ra3);
                                        ldmatrix_x4(at + 8 * 128, rb0, rb1, rb2, rb3);
                                        __syncwarp();
                                        stmatrix_x4(at, scale(ra0, al_a), scale(ra1, al_a), scale(ra2, al_a), scale(ra3, al_a));
                                        stmatrix_x4(at + 8 * 128, scale(rb0, al_b), scale(rb1, al_b), scale(rb2, al_b), scale(rb3, al_b));
                                    }
                                }
                            }
                            if (!C::kRescaleLate && j != s.kt0) {
                                // The O rows hold every earlier tile of the column: once the last PV issued
                                // (the previous step's) has completed they can be rescaled; this step's PV
                                // waits for this step's P.
                                if (!__all_sync(0xffffffffu, wait(kPEmpty + w, sc - 1, (int)sc))) return;
                                rescale_o<32, D>(t_o, al_a, al_b);
                            }
                            // the piece against the new references
                            const uint64_t na2 = pack2(-m_a, -m_a), nb2 = pack2(-m_b, -m_b);
                            const uint64_t c2a = pack2(c_a, c_a), c2b = pack2(c_b, c_b);
                            ts_a = ts_b = 0ull;
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const uint64_t pa = exp2_sfu2(fma2(pack2(as_f(v[4 * k]), as_f(v[4 * k + 1])), c2a, na2));
                                const uint64_t pb = exp2_sfu2(fma2(pack2(as_f(v[4 * k + 2]), as_f(v[4 * k + 3])), c2b, nb2));
                                ts_a = add2(ts_a, pa);
                                ts_b = add2(ts_b, pb);
                                float a0, a1, b0, b1;
                                unpack2(pa, a0, a1);
                                unpack2(pb, b0, b1);
                                pp[2 * k] = cvt_bf16x2(a0, a1);
                                pp[2 * k + 1] = cvt_bf16x2(b0, b1);
                            }
                        }
                        acc_a = add2(acc_a, ts_a);
                        acc_b = add2(acc_b, ts_b);
                        // The piece's P (bf16) goes into the lane's P tile straight away (the first piece's once the PV
                        // that read the previous step's P has completed), so its registers are free while the
                        // second piece is computed.  In shared memory the tile is the K-major, 128-byte-swizzled A
                        // operand of PV: one 64-key atom per piece, row r at r * 128 bytes, its 16-byte chunk k
                        // (8 keys) at chunk position k ^ (r % 8).  In tensor memory a row is a lane, two keys a column.
                        if (piece == 0 && sc > 0 && !__all_sync(0xffffffffu, wait(kPEmpty + w, sc - 1, (int)sc))) return;
                        if (C::kPInTmem) {
                            if (piece == 0) tc_fence_after_sync();
                            tmem_st_16x128b_x8(t_p + 32 * piece, pp);
                        } else {
                            const uint32_t at = p_at + piece * C::kAtomBytes;
                            stmatrix_x4(at, pp[0], pp[2], pp[4], pp[6]);                       // rows a, chunks 0..3
                            stmatrix_x4(at ^ 64u, pp[8], pp[10], pp[12], pp[14]);               // rows a, chunks 4..7
                            stmatrix_x4(at + 8 * 128, pp[1], pp[3], pp[5], pp[7]);              // rows a + 8
                            stmatrix_x4((at ^ 64u) + 8 * 128, pp[9], pp[11], pp[13], pp[15]);
                        }
                        // (the last PV that was issued has completed, see the wait above; this step's waits for this
                        // step's P)
                        if (C::kRescaleLate && move && j != s.kt0) rescale_o<D, D>(t_o, al_a, al_b);
                    }
                    if (C::kPInTmem) {
                        tmem_wait_st();
                        tc_fence_before_sync();
                    } else {
                        fence_proxy_async_smem();                  // the stores above are read by the tensor pipe
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kPFull + w));
                }

                // ---- the column's (or this part's) O rows are complete ----
                if (!__all_sync(0xffffffffu, wait(kOFull + w, oc, s.kt1))) return;
                tc_fence_after_sync();
                float l_a, l_b;
                {
                    float x0, x1;
                    unpack2(acc_a, x0, x1);
                    l_a = x0 + x1;
                    unpack2(acc_b, x0, x1);
                    l_b = x0 + x1;
                    l_a += __shfl_xor_sync(0xffffffffu, l_a, 1);
                    l_b += __shfl_xor_sync(0xffffffffu, l_b, 1);
                    l_a += __shfl_xor_sync(0xffffffffu, l_a, 2);
                    l_b += __shfl_xor_sync(0xffffffffu, l_b, 2);
                }
                const AttnItem &item = p.item[G.item];
                if constexpr (kParts) {
                    const int part_bar = kPartFull + wr.slab();
                    if (!merge_in_cluster<D>(p, s, wr, cta, t_o, m_a, m_b, l_a, l_b, p_smem, bar(part_bar), told,
                                             [&]() { return wait_bar<true>(bar(part_bar), 0, ctx, part_bar, s.kt1) && *abort_flag == 0; }))
                        return;
                } else if (s.kt0 == 0 && s.kt1 == G.n_kt) {
                    // a whole column: normalise and store
                    const float v_scale = item.v_scale ? item.v_scale[s.head] : 1.f;   // 8-bit caches: value codes x scale
                    const float inv_a = v_scale / l_a, inv_b = v_scale / l_b;
#pragma unroll 1
                    for (int ch = 0; ch < C::kOChunks; ++ch) {
                        uint32_t o[32], pk[16];
                        tmem_ld_16x256b_x8(t_o + 64 * ch, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            pk[2 * k] = cvt_bf16x2(as_f(o[4 * k]) * inv_a, as_f(o[4 * k + 1]) * inv_a);
                            pk[2 * k + 1] = cvt_bf16x2(as_f(o[4 * k + 2]) * inv_b, as_f(o[4 * k + 3]) * inv_b);
                        }
                        store_rows<D>(p, item, s, wr, p_smem, p_at, ch, pk);
                    }
                    store_lse(item, s, wr, m_a, m_b, l_a, l_b);
                } else {
                    // a part of a column: into its slot, and count the arrival; the warp that arrives last
                    // merges the parts.  At head_dim 64 it does so when the CTA's steps are done (a CTA has at
                    // most two parts: the end of its share's first column and the beginning of the last
                    // one): with the merge inside the column loop the softmax of a whole tile does not fit the
                    // registers (0.710 -> 0.815 ms, 24 heads of 64); at 128 it fits, and the loop
                    // is faster with it (0.484 against 0.490 ms).
                    const int own = p.share_of_cta[cta], which = s.kt0 == 0 ? 1 : 0;
                    int i0, n_parts;
                    parts_of(p, s, own, i0, n_parts);
                    float *slot = p.partial + (size_t)(2 * own + which) * kQTileRows * (D + 2);
#pragma unroll 1
                    for (int ch = 0; ch < C::kOChunks; ++ch) {
                        uint32_t o[32];
                        tmem_ld_16x256b_x8(t_o + 64 * ch, o);
                        tmem_wait_ld();
                        uint4 *dst = reinterpret_cast<uint4 *>(slot) + (size_t)(wr.slab() * (D / 16) + 4 * ch) * 64 + lane;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {              // 16 columns: this thread's four of row a, then of row a + 8
                            dst[64 * k] = make_uint4(o[8 * k], o[8 * k + 1], o[8 * k + 4], o[8 * k + 5]);
                            dst[64 * k + 32] = make_uint4(o[8 * k + 2], o[8 * k + 3], o[8 * k + 6], o[8 * k + 7]);
                        }
                    }
                    if ((lane & 3) == 0) {
                        float2 *ml = reinterpret_cast<float2 *>(slot + (size_t)kQTileRows * D) + wr.slab() * 16 + (lane >> 2);
                        ml[0] = make_float2(m_a, l_a);
                        ml[8] = make_float2(m_b, l_b);
                    }
                    __threadfence();
                    __syncwarp();
                    uint32_t arrived = 0;
                    if (lane == 0) arrived = atomicAdd(p.counters + i0 * kSlabs + wr.slab(), 1u);
                    arrived = __shfl_sync(0xffffffffu, arrived, 0);
                    if (arrived == (uint32_t)(n_parts - 1)) {
                        if (lane == 0) p.counters[i0 * kSlabs + wr.slab()] = 0;    // ready for the next launch
                        if (kMergeLate) {
                            to_merge |= 1u << which;
                        } else {
                            __threadfence();
                            merge_column<D>(p, s, own, wr, p_smem, p_at);
                        }
                    }
                }
                // the O columns may be overwritten by the next column's first PV
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kOEmpty + w));
                ++oc;
            }
            if (!kParts && kMergeLate && to_merge) {
                __threadfence();                                   // the other parts' slots, seen complete above
                const int own = p.share_of_cta[cta];
                for (WorkIter<kForm> it(p, cta); it.next(s);) {
                    if (w >= s.n_sub || (s.kt0 == 0 && s.kt1 == p.g[s.g].n_kt)) continue;
                    if ((to_merge >> (s.kt0 == 0 ? 1 : 0)) & 1u) merge_column<D>(p, s, own, wr, p_smem, p_at);
                }
            }
        }();
    }

    // ---- common exit -------------------------------------------------------------
    // In a cluster every warp that merges arrives at its peers exactly once, whatever becomes of its CTA, and leaves only when
    // all of them have arrived: a CTA that did not start, or gave up, sets the others' flags in front of its arrivals (value 3), so that
    // they neither merge rows that are not there nor wait for them.  A CTA that ends with its flag clear has heard of
    // every peer, and no peer sets it any more.
    auto merges = [&]() { return kParts && warp < 8 * first->s.n_sub; };
    if (kParts && !told && merges() && lane < p.cluster_parts && lane != (int)cluster_rank()) {
        st_shared_remote(smem_u32(tmem_slot + 1), (uint32_t)lane, 3u);
        mbar_arrive_remote(bar(kPartFull + WarpRows(warp, lane).slab()), (uint32_t)lane);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag != 0) {
        // give copies and MMAs that may still be in flight time to land before the
        // shared and tensor memory go back to the SM
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (kParts && *abort_flag != 0) {
        // (the limit is longer than a peer can take to give up)
        const uint64_t t0 = globaltimer_ns();
        if (merges() && lane == 0)
            while (!mbar_try_wait_cluster(bar(kPartFull + warp), 0) && globaltimer_ns() - t0 < 2 * kWaitLimitNs) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == kTmaWarp) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem, C::kTmemCols);
    }
}

// The bounded-wait machinery on its own: one warp waits on a barrier that nobody will ever
// complete, gives up after limit_ns, leaves the record and returns normally.
__global__ void wait_probe_kernel(uint32_t *status, unsigned long long limit_ns)
{
    __shared__ uint64_t never;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&never), 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    WaitCtx ctx{&abort_flag, status, (int)(threadIdx.x >> 5)};
    wait_bar(smem_u32(&never), 0, ctx, kProbeBarrierId, kProbeIteration, limit_ns);
}

}  // namespace

cudaError_t launch_wait_probe(uint32_t *status, uint64_t limit_ns, cudaStream_t stream)
{
    wait_probe_kernel<<<1, 32, 0, stream>>>(status, (unsigned long long)limit_ns);
    count_launch();
    return cudaGetLastError();
}

namespace {

template <int D, int kForm>
cudaError_t launch_instance(const AttnParams &p, const AttnMaps &maps, dim3 grid, bool early, cudaStream_t stream)
{
    // Once per device: the in-kernel register reallocation assumes the launch
    // allocation it was sized for, and the kernel needs its dynamic shared memory opted in.
    constexpr int kMaxDevices = 64;
    static std::atomic<unsigned char> prepared[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices || !prepared[dev].load(std::memory_order_acquire)) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, attn_sm100_kernel<D, kForm>);
        if (e != cudaSuccess) return e;
        if (fa.numRegs != kLaunchRegs) return cudaErrorLaunchOutOfResources;
        e = cudaFuncSetAttribute(attn_sm100_kernel<D, kForm>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDevices) prepared[dev].store(1, std::memory_order_release);
    }
    return launch_dependent(early, -1, kForm == kFormParts ? p.cluster_parts : 1, attn_sm100_kernel<D, kForm>, grid, kThreads, Cfg<D>::kSmemBytes,
                            stream, p, maps);
}

}  // namespace

namespace {

// Asked once per device and size.
template <int D>
int clusters_held(int n)
{
    constexpr int kMaxDevices = 64;
    static std::atomic<int> known[kMaxDevices][kMaxClusterParts + 1];      // 0: not asked, else one more than are held
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev < kMaxDevices)
        if (const int k = known[dev][n].load(std::memory_order_acquire)) return k - 1;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof attr);
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)n;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)n);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<D>::kSmemBytes;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int held = 0;
    cudaError_t e = cudaFuncSetAttribute(attn_sm100_kernel<D, kFormParts>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&held, attn_sm100_kernel<D, kFormParts>, &cfg);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        held = 0;
    }
    if (dev < kMaxDevices) known[dev][n].store(held + 1, std::memory_order_release);
    return held;
}

}  // namespace

int attn_clusters(int head_dim, int n) { return n < 1 || n > kMaxClusterParts ? 0 : head_dim == 128 ? clusters_held<128>(n) : clusters_held<64>(n); }

cudaError_t launch_attn_sm100(const AttnParams &p, int head_dim, const AttnMaps &maps, cudaStream_t stream)
{
    if (p.n_ctas <= 0) return cudaSuccess;
    dim3 grid((unsigned)(p.tile_ctas > 0 ? p.tile_ctas : p.n_ctas));
    cudaError_t e;
    long long steps = 0;
    for (int g = 0; g < p.n_groups; ++g) steps += (long long)p.heads * p.g[g].tiles * p.g[g].n_kt;
    const bool early = steps <= kEarlySteps * p.n_ctas;
    if (p.cluster_parts > 0)
        e = head_dim == 128 ? launch_instance<128, kFormParts>(p, maps, grid, early, stream) : launch_instance<64, kFormParts>(p, maps, grid, early, stream);
    else if (head_dim == 128) e = launch_instance<128, kFormTiles>(p, maps, grid, early, stream);
    else if (p.tile_ctas > 0) e = launch_instance<64, kFormTiles>(p, maps, grid, early, stream);
    else e = launch_instance<64, kFormColumns>(p, maps, grid, early, stream);
    count_launch();
    return e;
}

}  // namespace ll
