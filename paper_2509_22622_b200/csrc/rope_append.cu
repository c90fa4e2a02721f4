// Fused 3-D RoPE + K/V append (HBM-bound).
//
// One thread owns one 16-byte vector (8 bf16 = 4 rotation pairs) of one token
// for a group of kHeadsPerThread heads: it fetches the four (cos, sin) pairs
// once (they depend on the token's (t, y, x) only, not on the head and not on
// Q vs K), then streams Q, K, V of its heads through registers.  All global
// accesses are 16-byte vectors; 16 consecutive threads cover one 256-byte head
// row, so reads of the token-major inputs and writes of the head-major cache
// rows are fully coalesced.
#include <cuda_bf16.h>

#include <algorithm>

#include "bounded_wait.cuh"
#include "ll_internal.h"
#include "ptx.cuh"
#include "rope_math.cuh"

namespace ll {

namespace {

constexpr int kHeadsPerThread = 4;
constexpr int kThreads = 256;
constexpr int kNormThreads = 128;                      // of the kernel with the norm: one token per warp
constexpr int kStreamThreads = 384;                    // ... at most, when it streams its rows through shared memory
constexpr int kStreamSmem = 227 * 1024;                // and the shared memory it has for that
constexpr int kStreamed = -1;

// fp64-accurate sine/cosine tables, rounded once to fp32.
//   t_tab[(f - t_base) * n_t + i] = (cos, sin)(f * theta^(-i/n_t))
//   h_tab[y * n_hw + i], w_tab[x * n_hw + i] likewise with n_hw pairs per axis
__global__ void rope_table_kernel(float2 *t_tab, long long t_base, int n_t_frames, int n_t,
                                  float2 *h_tab, int grid_h, float2 *w_tab, int grid_w, int n_hw,
                                  double theta, int do_t, int do_hw)
{
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int n_tt = do_t ? n_t_frames * n_t : 0;
    const int n_hh = do_hw ? grid_h * n_hw : 0;
    const int n_ww = do_hw ? grid_w * n_hw : 0;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n_tt + n_hh + n_ww;
         idx += gridDim.x * blockDim.x) {
        double pos; int i, n_a; float2 *dst;
        if (idx < n_tt) {
            pos = (double)(t_base + idx / n_t); i = idx % n_t; n_a = n_t; dst = t_tab + idx;
        } else if (idx < n_tt + n_hh) {
            int j = idx - n_tt;
            pos = (double)(j / n_hw); i = j % n_hw; n_a = n_hw; dst = h_tab + j;
        } else {
            int j = idx - n_tt - n_hh;
            pos = (double)(j / n_hw); i = j % n_hw; n_a = n_hw; dst = w_tab + j;
        }
        double ang = pos * pow(theta, -(double)i / (double)n_a);
        double s, c;
        sincos(ang, &s, &c);
        *dst = make_float2((float)c, (float)s);
    }
}

__device__ __forceinline__ uint4 ld16(const ll_bf16 *p) { return *reinterpret_cast<const uint4 *>(p); }
__device__ __forceinline__ void st16(ll_bf16 *p, uint4 v) { *reinterpret_cast<uint4 *>(p) = v; }

__device__ __forceinline__ uint4 rotate_vec(uint4 x, const float2 (&cs)[4])
{
    return make_uint4(rotate_pair(x.x, cs[0]), rotate_pair(x.y, cs[1]),
                      rotate_pair(x.z, cs[2]), rotate_pair(x.w, cs[3]));
}

template <int D>
__global__ void __launch_bounds__(kThreads)
rope_append_kernel(const __grid_constant__ RopeAppendParams p)
{
    constexpr int kVecs = D / 8;                       // 16-byte vectors per head row
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int head_groups = (p.heads + kHeadsPerThread - 1) / kHeadsPerThread;
    const long long gid = (long long)blockIdx.x * kThreads + threadIdx.x;
    const int vec = (int)(gid % kVecs);
    const long long rest = gid / kVecs;
    const int hg = (int)(rest % head_groups);
    const long long token = rest / head_groups;
    if (token >= p.n_tokens) return;

    const int frame = (int)(token / p.P);
    const int cell = (int)(token % p.P);
    const int y = cell / p.grid_w, x = cell % p.grid_w;
    if ((unsigned)p.slot[frame] >= (unsigned)p.n_slots) {         // never with the host's slot rule: refuse, report
        record_status(p.status, kStatusBadRow, (uint32_t)p.slot[frame], (uint32_t)frame);
        return;
    }

    float2 cs[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = vec * 4 + u;                     // rotation pair inside the head row
        const float2 *src;
        if (j < p.n_t)             src = p.t_tab + (size_t)frame * p.n_t + j;
        else if (j < p.n_t + p.n_h) src = p.h_tab + (size_t)y * p.n_h + (j - p.n_t);
        else                        src = p.w_tab + (size_t)x * p.n_h + (j - p.n_t - p.n_h);
        cs[u] = *src;
    }

    const int h0 = hg * kHeadsPerThread;
    const size_t in_base = ((size_t)token * p.heads + h0) * D + (size_t)vec * 8;
    const size_t cache_row = (size_t)p.slot[frame] * p.P + cell;

    uint4 kq[kHeadsPerThread], kk[kHeadsPerThread], kv[kHeadsPerThread];
#pragma unroll
    for (int u = 0; u < kHeadsPerThread; ++u) {
        if (h0 + u < p.heads) {
            kk[u] = ld16(p.k + in_base + (size_t)u * D);
            kv[u] = ld16(p.v + in_base + (size_t)u * D);
            if (p.q_out) kq[u] = ld16(p.q + in_base + (size_t)u * D);
        }
    }
#pragma unroll
    for (int u = 0; u < kHeadsPerThread; ++u) {
        if (h0 + u < p.heads) {
            const size_t dst = (((size_t)(h0 + u)) * p.rows_per_head + cache_row) * D + (size_t)vec * 8;
            st16(static_cast<ll_bf16 *>(p.kcache) + dst, rotate_vec(kk[u], cs));
            st16(static_cast<ll_bf16 *>(p.vcache) + dst, kv[u]);
            if (p.q_out) st16(p.q_out + in_base + (size_t)u * D, rotate_vec(kq[u], cs));
        }
    }
}

// ---- the same into an 8-bit cache ---------------------------------------------------------
//
// K (rotated, fp32) and V are divided by their head's scale (the correctly rounded quotient) and rounded to
// E4M3, round to nearest even, saturating; a thread's eight elements make one 8-byte store, 16
// consecutive threads cover a 128-byte cache row.  Q is rotated to bf16 as in the bf16 kernel.
//   The quotient comes from the correctly rounded reciprocal r of the scale by Markstein's correction
// (P. Markstein, IBM J. Res. Dev. 34, 1990): q = x r, then q + (x - q s) r with fused operations is x / s
// correctly rounded, as long as nothing leaves the exponent range.  Scales in [2^-60, 2^60] keep it
// inside for every quotient that is not rounded to zero or saturated anyway; other scales divide.  With the
// division for every element and each head's loads behind the stores of the one before: 20.9 us, now 16.9 us for 4680
// tokens of 12 heads of 128 (72 MB, 11 us at the copy rate).
__device__ __forceinline__ uint2 quantise_vec(const float (&x)[8], float scale, float recip)
{
    uint32_t c[4];
    if (scale >= 0x1p-60f && scale <= 0x1p60f) {
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float q0 = x[u] * recip, q1 = fmaf(fmaf(-q0, scale, x[u]), recip, q0);
            q[u] = fabsf(q0) < 1024.f && q0 != 0.f ? q1 : q0;   // else saturated, infinite, NaN, or a zero with its sign
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = cvt_e4m3x2(q[2 * u], q[2 * u + 1]);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = cvt_e4m3x2(__fdiv_rn(x[2 * u], scale), __fdiv_rn(x[2 * u + 1], scale));
    }
    return make_uint2(c[0] | (c[1] << 16), c[2] | (c[3] << 16));
}

template <int D>
__global__ void __launch_bounds__(kThreads)
rope_append_e4m3_kernel(const __grid_constant__ RopeAppendParams p)
{
    constexpr int kVecs = D / 8;
    ptx::grid_dep_launch();
    const int head_groups = (p.heads + kHeadsPerThread - 1) / kHeadsPerThread;
    const long long gid = (long long)blockIdx.x * kThreads + threadIdx.x;
    const int vec = (int)(gid % kVecs);
    const long long rest = gid / kVecs;
    const int hg = (int)(rest % head_groups);
    const long long token = rest / head_groups;
    if (token >= p.n_tokens) return;

    const int frame = (int)(token / p.P);
    const int cell = (int)(token % p.P);
    const int y = cell / p.grid_w, x = cell % p.grid_w;
    const int h0 = hg * kHeadsPerThread;
    const size_t in_base = ((size_t)token * p.heads + h0) * D + (size_t)vec * 8;
    ptx::grid_dep_wait();
    if ((unsigned)p.slot[frame] >= (unsigned)p.n_slots) {         // never with the host's slot rule: refuse, report
        record_status(p.status, kStatusBadRow, (uint32_t)p.slot[frame], (uint32_t)frame);
        return;
    }
    // everything a thread reads goes out at once
    uint4 kq[kHeadsPerThread], kk[kHeadsPerThread], kv[kHeadsPerThread];
    float ks[kHeadsPerThread], vs[kHeadsPerThread];
#pragma unroll
    for (int u = 0; u < kHeadsPerThread; ++u) {
        if (h0 + u < p.heads) {
            kk[u] = ld16(p.k + in_base + (size_t)u * D);
            kv[u] = ld16(p.v + in_base + (size_t)u * D);
            if (p.q_out) kq[u] = ld16(p.q + in_base + (size_t)u * D);
            ks[u] = p.k_scale[h0 + u];
            vs[u] = p.v_scale[h0 + u];
        }
    }
    float2 cs[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = vec * 4 + u;
        const float2 *src;
        if (j < p.n_t)             src = p.t_tab + (size_t)frame * p.n_t + j;
        else if (j < p.n_t + p.n_h) src = p.h_tab + (size_t)y * p.n_h + (j - p.n_t);
        else                        src = p.w_tab + (size_t)x * p.n_h + (j - p.n_t - p.n_h);
        cs[u] = *src;
    }
    const size_t cache_row = (size_t)p.slot[frame] * p.P + cell;
    uint8_t *kc = static_cast<uint8_t *>(p.kcache), *vc = static_cast<uint8_t *>(p.vcache);
#pragma unroll
    for (int u = 0; u < kHeadsPerThread; ++u) {
        if (h0 + u >= p.heads) break;
        const uint32_t kw[4] = {kk[u].x, kk[u].y, kk[u].z, kk[u].w}, vw[4] = {kv[u].x, kv[u].y, kv[u].z, kv[u].w};
        float kr[8], vr[8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            rotate_pair_f32(kw[t], cs[t], kr[2 * t], kr[2 * t + 1]);
            vr[2 * t] = __uint_as_float(vw[t] << 16);
            vr[2 * t + 1] = __uint_as_float(vw[t] & 0xffff0000u);
        }
        const size_t dst = (((size_t)(h0 + u)) * p.rows_per_head + cache_row) * D + (size_t)vec * 8;
        *reinterpret_cast<uint2 *>(kc + dst) = quantise_vec(kr, ks[u], __frcp_rn(ks[u]));
        *reinterpret_cast<uint2 *>(vc + dst) = quantise_vec(vr, vs[u], __frcp_rn(vs[u]));
        if (p.q_out) st16(p.q_out + in_base + (size_t)u * D, rotate_vec(kq[u], cs));
    }
}

// Codes of the listed cache-row runs, all heads, K and V: to bf16 at the same rows of the
// staging pair.  One thread converts 16 codes (one 16-byte load, two 16-byte stores).
template <int D>
__global__ void __launch_bounds__(kThreads)
stage_e4m3_kernel(const __grid_constant__ StageParams p)
{
    constexpr int kVecs = D / 16;                      // 16-code vectors per row
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    long long gid = (long long)blockIdx.x * kThreads + threadIdx.x;
    const int vec = (int)(gid % kVecs);
    gid /= kVecs;
    int run = 0;
    long long rows_before = 0;
    // threads are numbered run by run, within a run head-major over its rows
    while (run < p.n_runs && gid >= rows_before + (long long)p.len[run] * p.heads) {
        rows_before += (long long)p.len[run] * p.heads;
        ++run;
    }
    if (run >= p.n_runs) return;
    const long long r = gid - rows_before;
    const int head = (int)(r / p.len[run]);
    const long long row = p.start[run] + r % p.len[run];
    const size_t off = ((size_t)head * p.rows_per_head + row) * D + (size_t)vec * 16;
    auto expand = [&](const uint8_t *src, ll_bf16 *dst) {
        const uint4 c = *reinterpret_cast<const uint4 *>(src + off);
        const uint32_t w[4] = {c.x, c.y, c.z, c.w};
        uint32_t o[8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            o[2 * t] = e4m3x2_to_bf16x2(w[t] & 0xffffu);
            o[2 * t + 1] = e4m3x2_to_bf16x2(w[t] >> 16);
        }
        st16(dst + off, make_uint4(o[0], o[1], o[2], o[3]));
        st16(dst + off + 8, make_uint4(o[4], o[5], o[6], o[7]));
    };
    expand(p.k8, p.k16);
    expand(p.v8, p.v16);
}

// ---- the same with the RMS norm of q and k in front -----------------------------------
//
// One warp owns one token at a time: a first pass over q and k sums the squares (fp32, then a butterfly over the
// warp), a second pass scales by the row's factor and the gain, rotates and stores; v leaves in between.  The row stride in
// vectors (32) is a multiple of the vectors per head (8 or 16), so a lane meets the same four rotation pairs in
// every vector it owns; their (cos, sin) are fetched with the row.  Both forms add in the same order: same bits.
//   Bound by memory, if enough of it is in flight.  With the row in registers between the passes (up to 192 vectors: 1536
// elements at head_dim 128) an SM holds 16 warps of 104 registers and meets their two dependent phases in turn: 21.7 us a
// pass for 4680 tokens of 1536 (86 MB, 13.2 us at the copy rate).  With the rows, which are contiguous in q, k and v, copied in
// bulk into shared memory, the next token's while one is worked on, 100 KB per SM are in flight at any time whatever the
// registers: 18.0 us.  Rows that fit neither are read again (from L1/L2) by the second pass.
__device__ __forceinline__ uint64_t widen(uint32_t packed)
{
    return ptx::pack2(__uint_as_float(packed << 16), __uint_as_float(packed & 0xffff0000u));
}

__device__ __forceinline__ uint64_t add_squares(uint4 x, uint64_t acc)
{
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint64_t v = widen(w[u]);
        acc = ptx::fma2(v, v, acc);
    }
    return acc;
}

// One packed pair times the row's factor (both halves of r), then its gains, turned by cs, in fp32, one rounding.  In
// this order: the factor brings the elements to the order of 1, element times gain alone may leave the range.
__device__ __forceinline__ uint32_t norm_rotate_pair(uint32_t packed, uint64_t r, float gx, float gy, float2 cs)
{
    float a, b;
    ptx::unpack2(ptx::mul2(ptx::mul2(widen(packed), r), ptx::pack2(gx, gy)), a, b);
    return ptx::cvt_bf16x2(fmaf(a, cs.x, -(b * cs.y)), fmaf(a, cs.y, b * cs.x));
}

__device__ __forceinline__ uint4 norm_rotate_vec(uint4 x, uint64_t r, const float *gain, const float2 (&cs)[4])
{
    const float4 g0 = *reinterpret_cast<const float4 *>(gain), g1 = *reinterpret_cast<const float4 *>(gain + 4);
    return make_uint4(norm_rotate_pair(x.x, r, g0.x, g0.y, cs[0]), norm_rotate_pair(x.y, r, g0.z, g0.w, cs[1]),
                      norm_rotate_pair(x.z, r, g1.x, g1.y, cs[2]), norm_rotate_pair(x.w, r, g1.z, g1.w, cs[3]));
}

// Shared memory of a block that streams its rows: the gains, then two buffers (q, k and v row) and their barriers per warp.
__host__ __device__ inline int norm_buffer_bytes(int heads, int head_dim) { return 3 * heads * head_dim * 2; }
__host__ __device__ inline int norm_gain_bytes(int heads, int head_dim) { return 2 * heads * head_dim * 4; }
__host__ __device__ inline int norm_smem_bytes(int heads, int head_dim, int warps)
{
    return norm_gain_bytes(heads, head_dim) + warps * (2 * norm_buffer_bytes(heads, head_dim) + 16) + 16;
}

// What a warp has of that.
template <int D>
struct NormStream {
    float *gains;                                      // q, then k
    uint8_t *own;                                      // its two buffers
    volatile int *abort_flag;
    uint32_t bars;                                     // and their barriers
    __device__ NormStream(int heads, uint8_t *smem)
    {
        const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5, buffers = 2 * norm_buffer_bytes(heads, D);
        gains = reinterpret_cast<float *>(smem);
        own = smem + norm_gain_bytes(heads, D) + (size_t)warp * buffers;
        bars = ptx::smem_u32(smem + norm_gain_bytes(heads, D) + (size_t)warps * buffers) + 16u * warp;
        abort_flag = reinterpret_cast<volatile int *>(smem + norm_smem_bytes(heads, D, warps) - 16);
    }
    // no memory but shared: before the wait for the kernel in front
    __device__ void init_barriers() const
    {
        if ((threadIdx.x & 31) < 2) ptx::mbar_init(bars + 8u * (threadIdx.x & 31), 1);
        if (threadIdx.x == 0) *abort_flag = 0;
        ptx::fence_mbar_init();
    }
};

// The rows through shared memory: one persistent block per SM, two buffers per warp.
template <int D>
__device__ __forceinline__ void norm_rows_streamed(const RopeAppendParams &p, const float *gain_q, const float *gain_k, float eps,
                                                   const NormStream<D> &stream)
{
    constexpr int kVecs = D / 8, kBatch = 6;           // 16-byte vectors per head row; vectors per lane whose loads go out together
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int row_vecs = p.heads * kVecs, row_bytes = row_vecs * 16;
    const bool with_q = p.q_out != nullptr;
    const int vec = lane % kVecs;                      // the lane's vector inside every head row it meets
    float *gains = stream.gains;
    uint8_t *own = stream.own;
    const uint32_t bars = stream.bars;
    WaitCtx ctx{stream.abort_flag, p.status, warp};
    // tokens go round the blocks first, so that every SM gets its share of the last round
    const int first = blockIdx.x + gridDim.x * warp, stride = gridDim.x * warps;
    auto fetch = [&](int token, int buf) {             // lane 0: q, k and v row of a token
        const uint32_t dst = ptx::smem_u32(own + buf * 3 * row_bytes), bar = bars + 8u * buf;
        const size_t off = (size_t)token * row_vecs * 8;
        ptx::mbar_arrive_expect_tx(bar, (with_q ? 3 : 2) * row_bytes);
        if (with_q) ptx::bulk_load(dst, p.q + off, row_bytes, bar);
        ptx::bulk_load(dst + row_bytes, p.k + off, row_bytes, bar);
        ptx::bulk_load(dst + 2 * row_bytes, p.v + off, row_bytes, bar);
    };
    if (lane == 0 && first < p.n_tokens) fetch(first, 0);
    for (int i = threadIdx.x; i < p.heads * D / 4; i += blockDim.x) {
        if (with_q) reinterpret_cast<float4 *>(gains)[i] = reinterpret_cast<const float4 *>(gain_q)[i];
        reinterpret_cast<float4 *>(gains)[p.heads * D / 4 + i] = reinterpret_cast<const float4 *>(gain_k)[i];
    }
    __syncthreads();
    int n = 0;                                         // tokens this warp has been through
    for (int token = first; token < p.n_tokens; token += stride, ++n) {
        const int frame = token / p.P, cell = token - frame * p.P;
        const int y = cell / p.grid_w, x = cell - y * p.grid_w;
        const bool bad = (unsigned)p.slot[frame] >= (unsigned)p.n_slots;    // never with the host's slot rule: refuse, report
        const size_t in_base = (size_t)token * row_vecs * 8;
        if (lane == 0 && token + stride < p.n_tokens) fetch(token + stride, (n + 1) & 1);
        float2 cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = vec * 4 + u;
            const float2 *src;
            if (j < p.n_t)             src = p.t_tab + (size_t)frame * p.n_t + j;
            else if (j < p.n_t + p.n_h) src = p.h_tab + (size_t)y * p.n_h + (j - p.n_t);
            else                        src = p.w_tab + (size_t)x * p.n_h + (j - p.n_t - p.n_h);
            cs[u] = *src;
        }
        const size_t cache_row = (size_t)p.slot[frame] * p.P + cell;
        auto cache_at = [&](int v) -> size_t { return ((size_t)(v / kVecs) * p.rows_per_head + cache_row) * D + (size_t)vec * 8; };
        if (!__all_sync(0xffffffffu, wait_bar(bars + 8u * (n & 1), (n >> 1) & 1, ctx, n & 1, n))) {
            const uint64_t t0 = ptx::globaltimer_ns();           // the copies in flight get time to land before the block goes
            while (ptx::globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            break;
        }
        const ll_bf16 *src_q = reinterpret_cast<const ll_bf16 *>(own + (n & 1) * 3 * row_bytes);
        const ll_bf16 *src_k = src_q + row_vecs * 8, *src_v = src_k + row_vecs * 8;
        const float *g_q = gains, *g_k = gains + p.heads * D;
        if (bad) {
            record_status(p.status, kStatusBadRow, (uint32_t)p.slot[frame], (uint32_t)frame);
            continue;
        }
        uint64_t sq2 = 0ull, sk2 = 0ull;
        for (int v0 = lane; v0 < row_vecs; v0 += 32 * kBatch) {
            uint4 xk[kBatch], xq[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (v0 + 32 * i < row_vecs) {
                    xk[i] = ld16(src_k + (size_t)(v0 + 32 * i) * 8);
                    if (with_q) xq[i] = ld16(src_q + (size_t)(v0 + 32 * i) * 8);
                }
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (v0 + 32 * i < row_vecs) {
                    sk2 = add_squares(xk[i], sk2);
                    if (with_q) sq2 = add_squares(xq[i], sq2);
                }
        }
        // v needs no factor
        for (int v0 = lane; v0 < row_vecs; v0 += 32 * kBatch)
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (v0 + 32 * i < row_vecs)
                    st16(static_cast<ll_bf16 *>(p.vcache) + cache_at(v0 + 32 * i), ld16(src_v + (size_t)(v0 + 32 * i) * 8));
        float sq, sk;
        {
            float a, b;
            ptx::unpack2(sq2, a, b);
            sq = a + b;
            ptx::unpack2(sk2, a, b);
            sk = a + b;
        }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            sq += __shfl_xor_sync(0xffffffffu, sq, m);
            sk += __shfl_xor_sync(0xffffffffu, sk, m);
        }
        const float inv_n = 1.f / (float)(row_vecs * 8);
        const float rq = 1.f / sqrtf(fmaf(sq, inv_n, eps)), rk = 1.f / sqrtf(fmaf(sk, inv_n, eps));
        const uint64_t rq2 = ptx::pack2(rq, rq), rk2 = ptx::pack2(rk, rk);
        for (int v0 = lane; v0 < row_vecs; v0 += 32 * kBatch) {
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const int v = v0 + 32 * i;
                if (v < row_vecs) {
                    st16(static_cast<ll_bf16 *>(p.kcache) + cache_at(v), norm_rotate_vec(ld16(src_k + (size_t)v * 8), rk2, g_k + (size_t)v * 8, cs));
                    if (with_q)
                        st16(p.q_out + in_base + (size_t)v * 8, norm_rotate_vec(ld16(src_q + (size_t)v * 8), rq2, g_q + (size_t)v * 8, cs));
                }
            }
        }
        __syncwarp();                                  // the buffer has been read
    }
}

// kIters > 0: the row's vectors fit kIters per lane and stay in registers between the two
// passes (one read of q, k, v from memory); 0: any row length, second pass re-reads; kStreamed: norm_rows_streamed.
template <int D, int kIters>
__global__ void __launch_bounds__(kIters == kStreamed ? kStreamThreads : kNormThreads)
norm_rope_append_kernel(const __grid_constant__ RopeAppendParams p, const float *gain_q,
                        const float *gain_k, float eps)
{
    constexpr int kVecs = D / 8;                       // 16-byte vectors per head row
    static_assert(32 % kVecs == 0, "a lane must meet the same rotation pairs in all its vectors");
    constexpr int kHeld = kIters > 0 ? kIters : 1;
    ptx::grid_dep_launch();
    extern __shared__ __align__(128) uint8_t smem[];
    const NormStream<D> stream(p.heads, smem);
    if constexpr (kIters == kStreamed) stream.init_barriers();
    // The index arithmetic stays behind the wait.  In front of it, append and attention of 1 head of 64, 1188 tokens, take 19.97 us
    // instead of 19.80 in a stream, 23.46 instead of 23.60 in a replayed graph; 6 heads, 240 tokens, 10.33 / 10.28 and 13.28 / 13.38.
    ptx::grid_dep_wait();
    if constexpr (kIters == kStreamed) {
        norm_rows_streamed<D>(p, gain_q, gain_k, eps, stream);
        return;
    }
    const int lane = threadIdx.x & 31;
    const long long token = (long long)blockIdx.x * (kNormThreads / 32) + (threadIdx.x >> 5);
    if (token >= p.n_tokens) return;
    const int row_vecs = p.heads * kVecs;
    const int frame = (int)(token / p.P);
    const int cell = (int)(token % p.P);
    const int y = cell / p.grid_w, x = cell % p.grid_w;
    const size_t in_base = (size_t)token * row_vecs * 8;
    const bool with_q = p.q_out != nullptr;
    if ((unsigned)p.slot[frame] >= (unsigned)p.n_slots) {         // never with the host's slot rule: refuse, report
        record_status(p.status, kStatusBadRow, (uint32_t)p.slot[frame], (uint32_t)frame);
        return;
    }

    uint4 hq[kHeld], hk[kHeld], hv[kHeld];
    uint64_t sq2 = 0ull, sk2 = 0ull;
    if (kIters > 0) {
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int v = lane + 32 * i;
            if (v < row_vecs) {
                hk[i] = ld16(p.k + in_base + (size_t)v * 8);
                if (with_q) hq[i] = ld16(p.q + in_base + (size_t)v * 8);
                hv[i] = ld16(p.v + in_base + (size_t)v * 8);
            }
        }
    }
    const int vec = lane % kVecs;                      // the lane's vector inside every head row it meets
    float2 cs[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = vec * 4 + u;
        const float2 *src;
        if (j < p.n_t)             src = p.t_tab + (size_t)frame * p.n_t + j;
        else if (j < p.n_t + p.n_h) src = p.h_tab + (size_t)y * p.n_h + (j - p.n_t);
        else                        src = p.w_tab + (size_t)x * p.n_h + (j - p.n_t - p.n_h);
        cs[u] = *src;
    }
    const size_t cache_row = (size_t)p.slot[frame] * p.P + cell;
    auto cache_at = [&](int v) -> size_t { return ((size_t)(v / kVecs) * p.rows_per_head + cache_row) * D + (size_t)vec * 8; };
    if (kIters > 0) {
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            if (lane + 32 * i < row_vecs) {
                sk2 = add_squares(hk[i], sk2);
                if (with_q) sq2 = add_squares(hq[i], sq2);
            }
        }
        // v needs no factor: it leaves while the sums are on their way round the warp
#pragma unroll
        for (int i = 0; i < kHeld; ++i)
            if (lane + 32 * i < row_vecs) st16(static_cast<ll_bf16 *>(p.vcache) + cache_at(lane + 32 * i), hv[i]);
    } else {
        for (int v = lane; v < row_vecs; v += 32) {
            sk2 = add_squares(ld16(p.k + in_base + (size_t)v * 8), sk2);
            if (with_q) sq2 = add_squares(ld16(p.q + in_base + (size_t)v * 8), sq2);
            st16(static_cast<ll_bf16 *>(p.vcache) + cache_at(v), ld16(p.v + in_base + (size_t)v * 8));
        }
    }
    float sq, sk;
    {
        float a, b;
        ptx::unpack2(sq2, a, b);
        sq = a + b;
        ptx::unpack2(sk2, a, b);
        sk = a + b;
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, m);
        sk += __shfl_xor_sync(0xffffffffu, sk, m);
    }
    const float inv_n = 1.f / (float)(row_vecs * 8);
    const float rq = 1.f / sqrtf(fmaf(sq, inv_n, eps)), rk = 1.f / sqrtf(fmaf(sk, inv_n, eps));
    const uint64_t rq2 = ptx::pack2(rq, rq), rk2 = ptx::pack2(rk, rk);
    auto emit = [&](int v, uint4 xq, uint4 xk) {
        st16(static_cast<ll_bf16 *>(p.kcache) + cache_at(v), norm_rotate_vec(xk, rk2, gain_k + (size_t)v * 8, cs));
        if (with_q) st16(p.q_out + in_base + (size_t)v * 8, norm_rotate_vec(xq, rq2, gain_q + (size_t)v * 8, cs));
    };
    if (kIters > 0) {
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int v = lane + 32 * i;
            if (v < row_vecs) emit(v, hq[i], hk[i]);
        }
    } else {
        for (int v = lane; v < row_vecs; v += 32) {
            const size_t src = in_base + (size_t)v * 8;
            emit(v, with_q ? ld16(p.q + src) : make_uint4(0, 0, 0, 0), ld16(p.k + src));
        }
    }
}

// Warps of a streaming block: as many as their buffers fit, at least four up to 32 heads of 128.
int norm_stream_warps(int heads, int head_dim)
{
    int warps = kStreamThreads / 32;
    while (norm_smem_bytes(heads, head_dim, warps) > kStreamSmem) --warps;
    return warps;
}

template <int D>
cudaError_t launch_norm_variant(const RopeAppendParams &p, const float *gain_q, const float *gain_k, float eps, int sm_count, cudaStream_t stream)
{
    const int iters = (p.heads * (D / 8) + 31) / 32, sms = sm_count > 0 ? sm_count : 148;
    if (norm_append_streams(p.heads, D, p.n_tokens, p.q_out != nullptr, sm_count)) {
        const int warps = norm_stream_warps(p.heads, D);
        // never less than half of an SM's shared memory: blocks of an early kernel go to the SMs that come free first, and two
        // on one would leave another idle
        const int need = norm_smem_bytes(p.heads, D, warps), smem = need > kStreamSmem / 2 ? need : kStreamSmem / 2 + 2048;
        const cudaError_t e = cudaFuncSetAttribute(norm_rope_append_kernel<D, kStreamed>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
        if (e != cudaSuccess) return e;
        return launch_dependent(true, norm_rope_append_kernel<D, kStreamed>, dim3((unsigned)(p.n_tokens < sms ? p.n_tokens : sms)), 32 * warps, smem, stream,
                                p, gain_q, gain_k, eps);
    }
    const unsigned blocks = (unsigned)((p.n_tokens + kNormThreads / 32 - 1) / (kNormThreads / 32));
    if (iters <= 2) return launch_spread<&norm_rope_append_kernel<D, 2>>(blocks, kNormThreads, stream, p, gain_q, gain_k, eps);
    if (iters <= 4) return launch_spread<&norm_rope_append_kernel<D, 4>>(blocks, kNormThreads, stream, p, gain_q, gain_k, eps);
    if (iters <= 6) return launch_spread<&norm_rope_append_kernel<D, 6>>(blocks, kNormThreads, stream, p, gain_q, gain_k, eps);
    return launch_spread<&norm_rope_append_kernel<D, 0>>(blocks, kNormThreads, stream, p, gain_q, gain_k, eps);
}

}  // namespace

// Whether the append with the norm streams its rows through shared memory.  Both kernels go through the tokens in rounds: a
// streaming SM one per warp at a time (12 up to 11 heads of 128, 8 at 16 heads, 4 at 32), the other kernel, with its rows in
// registers, 24 tokens an SM at a time up to 8 heads of 128 and 16 up to 12.  Streamed rows gain where the other kernel
// begins a round and lose where they begin one of their own while it is still in its first; the longer the row, the more
// a round of theirs gains.  us, streamed against not, buffers not in L2, 148 SMs, q too unless noted:
//   5 heads of 128:   888 tokens 5.9 / 6.1, 2000 9.2 / 7.2, 4680 12.6 / 12.0, 7104 16.4 / 15.9
//   8 heads:         1184 tokens 7.1 / 7.3, 1776 8.5 / 8.2, 2000 10.5 / 8.9, 2516 11.0 / 10.6, 2960 11.2 / 12.3, 4680 14.7 / 16.1, 7104 19.9 / 21.8
//   12 heads:        1479 tokens 9.4 / 9.9, 2368 13.2 / 11.8, 2516 13.3 / 16.1, 4680 18.8 / 21.0, 7104 27.5 / 28.5, 14400 52.0 / 48.9
//   14 heads:         444 tokens 7.4 / 11.2, 2960 17.0 / 17.4, 4736 25.0 / 23.4
//   16 heads:        1184 tokens 10.1 / 13.9, 4680 24.8 / 26.8, 14400 64.1 / 70.9; k and v alone 2960 14.5 / 15.1, 4736 18.9 / 18.7
//   24 heads:        1184 tokens 15.2 / 18.9, 2368 27.1 / 25.4, 4736 42.8 / 41.7; k and v alone 1924 16.3 / 17.3, 2368 20.2 / 18.4
//   32 heads:        1184 tokens 18.6 / 24.1, 2368 31.3 / 35.4; k and v alone 1776 19.0 / 20.7, 2368 24.2 / 23.7
//   k and v alone up to 8 heads: nothing to gain (8 heads, 888 tokens 5.7 / 5.6, 2368 8.8 / 7.3, 4736 11.8 / 11.9).
// Heads of 64 go by the length of their rows as well (24 of 64 as 12 of 128, within 2 %).  Rows of up to 4 heads are too short (2 heads,
// 14400 tokens: 20.6 / 9.0), from 33 heads on too few warps' buffers fit (40 heads, 4680 tokens: 81.9 / 64.9).
bool norm_append_streams(int heads, int head_dim, int n_tokens, bool with_q, int sm_count)
{
    const int iters = (heads * (head_dim / 8) + 31) / 32;         // 16-byte vectors of a row per lane of a warp
    const int sms = sm_count > 0 ? sm_count : 148, each = (int)(((long long)n_tokens + sms - 1) / sms);
    if (iters <= 2 || iters > 16) return false;
    if (iters <= 4) return with_q && (each <= (iters == 3 ? 6 : 10) || (iters == 4 && each > 18 && each <= 48));
    if (iters <= 6) return each <= norm_stream_warps(heads, head_dim) || (each > 16 && each <= 48);
    if (iters <= 8) return each <= 24 || (iters == 8 && with_q);
    return each <= (with_q ? 16 : std::min(16, 3 * norm_stream_warps(heads, head_dim)));
}

cudaError_t launch_norm_rope_append(const RopeAppendParams &p, int head_dim, const float *gain_q, const float *gain_k,
                                    float eps, int sm_count, cudaStream_t stream)
{
    if (p.n_tokens <= 0) return cudaSuccess;
    const cudaError_t e = head_dim == 128 ? launch_norm_variant<128>(p, gain_q, gain_k, eps, sm_count, stream)
                                          : launch_norm_variant<64>(p, gain_q, gain_k, eps, sm_count, stream);
    count_launch();
    return e;
}

cudaError_t launch_rope_tables(float2 *t_tab, int64_t t_base, int n_t_frames, int n_t, float2 *h_tab,
                               int grid_h, float2 *w_tab, int grid_w, int n_hw, float theta, bool do_t,
                               bool do_hw, cudaStream_t stream)
{
    int total = (do_t ? n_t_frames * n_t : 0) + (do_hw ? (grid_h + grid_w) * n_hw : 0);
    if (total == 0) return cudaSuccess;
    int blocks = (total + 127) / 128;
    const cudaError_t e = launch_dependent(true, rope_table_kernel, blocks, 128, 0, stream, t_tab, (long long)t_base, n_t_frames, n_t, h_tab,
                                           grid_h, w_tab, grid_w, n_hw, (double)theta, (int)do_t, (int)do_hw);
    count_launch();
    return e;
}

cudaError_t launch_rope_append_e4m3(const RopeAppendParams &p, int head_dim, cudaStream_t stream)
{
    const int head_groups = (p.heads + kHeadsPerThread - 1) / kHeadsPerThread;
    const long long threads = (long long)p.n_tokens * head_groups * (head_dim / 8);
    const unsigned blocks = (unsigned)((threads + kThreads - 1) / kThreads);
    if (blocks == 0) return cudaSuccess;
    const cudaError_t e = head_dim == 128 ? launch_spread<&rope_append_e4m3_kernel<128>>(blocks, kThreads, stream, p)
                                          : launch_spread<&rope_append_e4m3_kernel<64>>(blocks, kThreads, stream, p);
    count_launch();
    return e;
}

cudaError_t launch_stage_e4m3(const StageParams &p, int head_dim, cudaStream_t stream)
{
    long long rows = 0;
    for (int i = 0; i < p.n_runs; ++i) rows += (long long)p.len[i] * p.heads;
    const long long threads = rows * (head_dim / 16);
    const unsigned blocks = (unsigned)((threads + kThreads - 1) / kThreads);
    if (blocks == 0) return cudaSuccess;
    const cudaError_t e = head_dim == 128 ? launch_spread<&stage_e4m3_kernel<128>>(blocks, kThreads, stream, p)
                                          : launch_spread<&stage_e4m3_kernel<64>>(blocks, kThreads, stream, p);
    count_launch();
    return e;
}

cudaError_t launch_rope_append(const RopeAppendParams &p, int head_dim, cudaStream_t stream)
{
    const int head_groups = (p.heads + kHeadsPerThread - 1) / kHeadsPerThread;
    const long long threads = (long long)p.n_tokens * head_groups * (head_dim / 8);
    const unsigned blocks = (unsigned)((threads + kThreads - 1) / kThreads);
    if (blocks == 0) return cudaSuccess;
    const cudaError_t e = head_dim == 128 ? launch_spread<&rope_append_kernel<128>>(blocks, kThreads, stream, p)
                                          : launch_spread<&rope_append_kernel<64>>(blocks, kThreads, stream, p);
    count_launch();
    return e;
}

}  // namespace ll
