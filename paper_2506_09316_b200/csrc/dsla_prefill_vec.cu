// Prefill with gates per key channel (the gated-linear-attention form of Sec. 2) on the tensor cores: bf16 inputs, d = 128, dual
// state.  With one gate per state row there is no decay per token pair to mask a score matrix with; inside a chunk of
// C = 32 tokens the decays go into the operands, as plain products of gates (all <= 1: nothing overflows, and a zero
// gate is exact), with p_j[c] = prod_{t <= j} g_t[c] and s_j[c] = prod_{t > j} g_t[c] over the chunk:
//     O^T   = sum_i S_i^T (W_i p_i (.) Q)^T + V^T P~^T             A_i[c] = prod of the chunk's gates
//     S_i^T <- S_i^T diag(A_i) + V^T (s_i (.) K)                   P~ = sum_i W_i A_i[j][s],  s <= j
//     A_i[j][s] = sum_c q_j[c] k_s[c] prod_{s < t <= j} g_t[c]     (the scores; here A_i[j][s] is per token pair)
//
// Precision.  The token-by-token kernel this replaces works in fp32, and so does this one: q, k and v are exact in bf16, a
// scaled operand is an fp32 value cut into bf16 terms.  K enters the states with three terms (24 bits); for the outputs, which are
// rounded to bf16, Q, the states and P~ have two (products down to 2^-16 of the leading one are kept).  The scores inside a
// 16-token block are fp32 on CUDA cores, those between the chunk's two blocks are products of two-term operands scaled
// to the block boundary.
//
// CTA = (sequence, head, segment), 16 warps, no fixed roles: the chunk loop alternates between the two states.
//   phase A: pass over S_1 (two bf16 terms of it for the readout, then S_1 diag(A_1)) | MMAs of state 1 | operands of state 2
//   phase B: pass over S_2, P~                                                        | MMAs of state 2 | operands of state 1, next chunk
// so the operands of one state are built while the tensor core works on the other and nothing is double-buffered but
// the raw Q, K and V.  Bound by instruction issue: about 85 slots per token and SM sub-partition for the operands and scores and
// 40 for the passes over the states.
//
// A sequence is split into segments when there are few (sequence, head) pairs and the caller's workspace has room: a first
// grid accumulates each segment's state from zero, walking the chunks backwards with the product of all later gates (no pass
// over the states), an elementwise kernel turns these summaries into initial states, the main grid starts from them.
// T = 4096, 32 heads: 540 us (413 of them this file's main grid); 2490 us with the token-by-token kernel.
#include "dsla_prefill_tc.cuh"

namespace dsla {

namespace {

constexpr int VC = 32, VB = 16;                      // tokens per chunk, per block
constexpr int V_NTHREADS = 512;
constexpr int V_TILE = VC * D * 2, V_HALF = V_TILE / 2;          // bf16 tile of 32 tokens: two halves [32][64], 128-byte swizzle
constexpr int V_BTILE = VB * D * 2, V_BHALF = V_BTILE / 2;       // the same for one block
// shared memory
constexpr int OFF_V = 0;                             // V, two buffers
constexpr int OFF_QT = OFF_V + 2 * V_TILE;           // Q~: [state][term 2]
constexpr int OFF_KT = OFF_QT + 4 * V_TILE;          // K~: [state][term 3]  (summaries: [parity][state][term])
constexpr int OFF_PT = OFF_KT + 6 * V_TILE;          // P~: [term 2], rows of 128 bytes of which 64 are used
constexpr int OFF_QB = OFF_PT + 2 * VC * 128;        // Q of block 1 scaled from its start, two terms
constexpr int OFF_KB = OFF_QB + 2 * V_BTILE;         // K of block 0 scaled to its end, two terms
constexpr int OFF_RAW = OFF_KB + 2 * V_BTILE;        // raw Q, K: [buffer][32][128] bf16
constexpr int OFF_RAWK = OFF_RAW + 2 * V_TILE;
constexpr int OFF_G = OFF_RAWK + 2 * V_TILE;         // gates: [state][32][128] fp32
constexpr int OFF_SC = OFF_G + 2 * VC * D * 4;       // scores: [state][32][32] fp32
constexpr int OFF_A = OFF_SC + 2 * VC * VC * 4;      // chunk decays: [state][128] fp32
constexpr int V_SMEM = OFF_A + 2 * D * 4 + 1024;
// summaries reuse the front: V buffers, then K~ [parity][state][term]
constexpr int OFF_SKT = 2 * V_TILE;
constexpr int OFF_SG = OFF_SKT + 12 * V_TILE;        // gates [parity][state][32][128] fp32
constexpr int OFF_SK = OFF_SG + 4 * VC * D * 4;      // raw K [parity]
constexpr int V_SMEM_SUM = OFF_SK + 2 * V_TILE + 1024;
// TMEM columns
constexpr uint32_t VCOL_S = 0, VCOL_SB = 256, VCOL_O = 384;      // fp32 states 2 x 128, bf16 terms of one state 2 x 64, O^T 32
constexpr size_t VEC_STRIDE = (2 * D * D + 2 * D) * sizeof(float);      // one summary: U[2][d][d], A[2][d]

struct VecParams {
    PrefillParams p;
    float* ws;           // summaries / initial states [(n*H + h)*nseg + g], or nullptr (nseg = 1)
    int nseg, cps;       // segments per sequence, chunks per segment
};

struct alignas(16) VecShared {
    uint64_t raw_full[2], g2_full, done[2];
    uint32_t tmem_base;
    int abort_flag;
    short pair[2][72];   // score pair numbers -> row * 32 + column inside a block
};

// bf16 terms of a pair of fp32 values; x is left with what the term does not hold
__device__ __forceinline__ uint32_t take_term(float2& x) {
    const uint32_t t = pack_bf16(x.x, x.y);
    const float2 f = unpack_bf16(t);
    x = __fadd2_rn(x, make_float2(-f.x, -f.y));
    return t;
}
__device__ __forceinline__ float2 clamp0(float2 g) { return make_float2(fmaxf(g.x, 0.f), fmaxf(g.y, 0.f)); }

// Sum over the lanes of 32 values per lane: lane l is left with the total of v[l] (31 exchanges).
__device__ __forceinline__ float transpose_sum(float (&v)[32], int lane) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float send = up ? v[i] : v[i + off], keep = up ? v[i + off] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

struct VecUnit {
    int n, h, g, len, slot, t_begin, nchunks, c_begin, c_end;
};
__device__ __forceinline__ VecUnit vec_unit(const VecParams& vp, int block, int nseg_grid) {
    const PrefillParams& p = vp.p;
    VecUnit u;
    u.g = block % nseg_grid;
    u.h = (block / nseg_grid) % p.H;
    u.n = block / (nseg_grid * p.H);
    u.t_begin = p.cu_seqlens ? p.cu_seqlens[u.n] : u.n * p.T;
    u.len = (p.cu_seqlens ? p.cu_seqlens[u.n + 1] : (u.n + 1) * p.T) - u.t_begin;
    u.slot = p.slots ? p.slots[u.n] : u.n;
    u.nchunks = (u.len + VC - 1) / VC;
    u.c_begin = u.g * vp.cps;
    u.c_end = u.g == vp.nseg - 1 ? u.nchunks : min(u.nchunks, u.c_begin + vp.cps);     // the last segment takes whatever is left
    return u;
}

// One score block of 16 tokens: pairs (j, s < j) with s in [S0, S1), this lane's four channels, all pairs of a batch of 32 reduced
// together.  q, k: raw rows of the block; g: gates.
template <int S0, int S1>
__device__ __forceinline__ void block_scores(const uint8_t* q, const uint8_t* k, const float* g, int valid, int lane, const short* pair, float* out) {
    float2 kd[S1 - S0][2];
#pragma unroll
    for (int s = S0; s < S1; ++s) {
        const uint2 x = *reinterpret_cast<const uint2*>(k + s * 256 + lane * 8);
        kd[s - S0][0] = s < valid ? unpack_bf16(x.x) : make_float2(0.f, 0.f);
        kd[s - S0][1] = s < valid ? unpack_bf16(x.y) : make_float2(0.f, 0.f);
    }
    float v[32];
    int at = 0;      // (compile-time: every loop below is unrolled)
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = 0.f;
#pragma unroll
    for (int j = S0 + 1; j < VB; ++j) {
        const uint2 x = *reinterpret_cast<const uint2*>(q + j * 256 + lane * 8);
        const float4 gg = *reinterpret_cast<const float4*>(g + j * D + lane * 4);
        const float2 q0 = unpack_bf16(x.x), q1 = unpack_bf16(x.y);
        const float2 g0 = clamp0(make_float2(gg.x, gg.y)), g1 = clamp0(make_float2(gg.z, gg.w));
#pragma unroll
        for (int s = S0; s < S1; ++s) {
            if (s >= j) continue;
            float2(&w)[2] = kd[s - S0];
            w[0] = __fmul2_rn(w[0], g0);
            w[1] = __fmul2_rn(w[1], g1);
            const float2 y = __ffma2_rn(q1, w[1], __fmul2_rn(q0, w[0]));
            v[at % 32] = y.x + y.y;
            if (++at % 32 == 0) {
                const float total = transpose_sum(v, lane);
                out[pair[at - 32 + lane]] = total;
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = 0.f;
            }
        }
    }
    if (at % 32) {
        const float total = transpose_sum(v, lane);
        if (lane < at % 32) out[pair[at - at % 32 + lane]] = total;
    }
}
constexpr int SPLIT_S = 5;      // keys 0..4 of a block: 65 pairs, keys 5..14: 55

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t saddr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(bytes),
                 "r"(smem_u32(bar))
                 : "memory");
}

// Byte offset of this lane's channel pair (channels 64 hh + 2 lane, + 1) of a row in a swizzled tile whose halves are `half` bytes.
__device__ __forceinline__ uint32_t pair_at(int row, int hh, int lane, int half) {
    return (uint32_t)(hh * half + row * 128 + ((((lane >> 2) ^ (row & 7)) << 4) | ((lane & 3) << 2)));
}

// Q~ of one state: rows 16 b .. 16 b + 15, channels 64 hh ..; block 1 also leaves its copy scaled from the block's start.
__device__ __forceinline__ void build_q(uint8_t* tiles, const uint8_t* qraw, const uint8_t* graw, int i, int hh, int b, int valid, float W, int lane) {
    const uint8_t* q = qraw + hh * 128 + lane * 4;
    const uint8_t* g = graw + hh * 256 + lane * 8;
    uint8_t* qt = tiles + OFF_QT + 2 * i * V_TILE;
    float2 first = make_float2(W, W);          // weight times the decay before this block
    if (b == 1) {
#pragma unroll 4
        for (int t = 0; t < VB; ++t) first = __fmul2_rn(first, clamp0(*reinterpret_cast<const float2*>(g + t * 512)));      // (valid > 16, or the rows do not matter)
    }
    float2 pr = make_float2(1.f, 1.f);
#pragma unroll 4
    for (int t = VB * b; t < VB * b + VB; ++t) {
        const float2 gg = clamp0(*reinterpret_cast<const float2*>(g + t * 512));
        if (t < valid) pr = __fmul2_rn(pr, gg);
        float2 x = __fmul2_rn(unpack_bf16(*reinterpret_cast<const uint32_t*>(q + t * 256)), pr);
        float2 y = __fmul2_rn(x, first);
        const uint32_t at = pair_at(t, hh, lane, V_HALF);
        *reinterpret_cast<uint32_t*>(qt + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(qt + V_TILE + at) = pack_bf16(y.x, y.y);
        if (b == 1) {
            const uint32_t bt = pair_at(t - VB, hh, lane, V_BHALF);
            *reinterpret_cast<uint32_t*>(tiles + OFF_QB + bt) = take_term(x);
            *reinterpret_cast<uint32_t*>(tiles + OFF_QB + V_BTILE + bt) = pack_bf16(x.x, x.y);
        }
    }
}

// K~ of one state in three terms (kt), rows 16 b .. 16 b + 15, weighted to the end of the chunk times `carry`; block 0 also leaves its
// copy scaled to the block's end (kb, unless null).  Returns the product of the chunk's gates.
__device__ __forceinline__ float2 build_k(uint8_t* kt, uint8_t* kb, const uint8_t* kraw, const uint8_t* graw, int hh, int b, int valid, float2 carry, int lane) {
    const uint8_t* k = kraw + hh * 128 + lane * 4;
    const uint8_t* g = graw + hh * 256 + lane * 8;
    float2 other = make_float2(1.f, 1.f);      // product of the other block's gates
#pragma unroll 4
    for (int t = VB * (1 - b); t < VB * (1 - b) + VB; ++t) {
        const float2 gg = clamp0(*reinterpret_cast<const float2*>(g + t * 512));
        if (t < valid) other = __fmul2_rn(other, gg);
    }
    const float2 behind = b == 0 ? __fmul2_rn(other, carry) : carry;      // decay behind this block
    float2 sf = make_float2(1.f, 1.f);
#pragma unroll 4
    for (int t = VB * b + VB - 1; t >= VB * b; --t) {
        const float2 kk = t < valid ? unpack_bf16(*reinterpret_cast<const uint32_t*>(k + t * 256)) : make_float2(0.f, 0.f);
        float2 x = __fmul2_rn(kk, sf);
        float2 y = __fmul2_rn(x, behind);
        const uint32_t at = pair_at(t, hh, lane, V_HALF);
        *reinterpret_cast<uint32_t*>(kt + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(kt + V_TILE + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(kt + 2 * V_TILE + at) = pack_bf16(y.x, y.y);
        if (b == 0 && kb) {
            const uint32_t bt = pair_at(t, hh, lane, V_BHALF);
            *reinterpret_cast<uint32_t*>(kb + bt) = take_term(x);
            *reinterpret_cast<uint32_t*>(kb + V_BTILE + bt) = pack_bf16(x.x, x.y);
        }
        const float2 gg = clamp0(*reinterpret_cast<const float2*>(g + t * 512));
        if (t < valid) sf = __fmul2_rn(sf, gg);
    }
    return __fmul2_rn(sf, other);
}

// Scores between the blocks, rows 16..31 x columns 8 nt .. 8 nt + 7: two-term operands, the product of the two low terms left out.
__device__ __forceinline__ void cross_scores(const uint8_t* tiles, int nt, int lane, float* out) {
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t qb = smem_u32(tiles + OFF_QB), kb = smem_u32(tiles + OFF_KB);
    const int arow = lane & 15, brow = 8 * nt + (lane & 7);
#pragma unroll 2
    for (int k2 = 0; k2 < 4; ++k2) {           // 32 channels per round
        const int half = (k2 >> 1) * V_BHALF;
        uint32_t b[2][4];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int piece = 4 * (k2 & 1) + (lane >> 3);
            ldmatrix_x4(kb + (uint32_t)(t * V_BTILE + half + brow * 128 + ((piece ^ (brow & 7)) << 4)), b[t]);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            uint32_t a[2][4];
            const int piece = 4 * (k2 & 1) + 2 * s + (lane >> 4);
#pragma unroll
            for (int t = 0; t < 2; ++t) ldmatrix_x4(qb + (uint32_t)(t * V_BTILE + half + arow * 128 + ((piece ^ (arow & 7)) << 4)), a[t]);
            mma16816(c, a[1], b[0][2 * s], b[0][2 * s + 1]);
            mma16816(c, a[0], b[1][2 * s], b[1][2 * s + 1]);
            mma16816(c, a[0], b[0][2 * s], b[0][2 * s + 1]);
        }
    }
    float* o = out + (VB + (lane >> 2)) * VC + 8 * nt + 2 * (lane & 3);
    *reinterpret_cast<float2*>(o) = make_float2(c[0], c[1]);
    *reinterpret_cast<float2*>(o + 8 * VC) = make_float2(c[2], c[3]);
}

// Everything state i needs of a chunk from its raw Q, K and gates.
__device__ __forceinline__ void build_operands(uint8_t* tiles, const VecShared& sh, int i, int buf, int valid, float W, int warp, int lane) {
    const uint8_t* qraw = tiles + OFF_RAW + buf * V_TILE;
    const uint8_t* kraw = tiles + OFF_RAWK + buf * V_TILE;
    const uint8_t* graw = tiles + OFF_G + i * VC * D * 4;
    float* sc = reinterpret_cast<float*>(tiles + OFF_SC) + i * VC * VC;
    if (warp < 4) {
        build_q(tiles, qraw, graw, i, warp & 1, warp >> 1, valid, W, lane);
        if (warp >= 2) asm volatile("bar.arrive 1, 192;" ::: "memory");
    } else if (warp < 8) {
        const int hh = warp & 1, b = (warp - 4) >> 1;
        const float2 a = build_k(tiles + OFF_KT + 3 * i * V_TILE, tiles + OFF_KB, kraw, graw, hh, b, valid, make_float2(1.f, 1.f), lane);
        if (b == 0) {
            asm volatile("bar.arrive 1, 192;" ::: "memory");
            reinterpret_cast<float2*>(tiles + OFF_A)[i * (D / 2) + 32 * hh + lane] = a;
        }
    } else if (warp < 12) {
        const int b = (warp - 8) >> 1;
        const uint8_t *q = qraw + b * VB * 256, *k = kraw + b * VB * 256;
        const float* g = reinterpret_cast<const float*>(graw) + b * VB * D;
        float* out = sc + b * (VB * VC + VB);
        if (warp & 1) block_scores<SPLIT_S, VB - 1>(q, k, g, valid - b * VB, lane, sh.pair[1], out);
        else block_scores<0, SPLIT_S>(q, k, g, valid - b * VB, lane, sh.pair[0], out);
    } else if (warp < 14) {
        asm volatile("bar.sync 1, 192;" ::: "memory");
        cross_scores(tiles, warp - 12, lane, sc);
    } else if (warp == 14 && i == 0) {
        // the current token is undecayed: its score is the same for both states
        float v[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) {
            const uint2 x = *reinterpret_cast<const uint2*>(qraw + t * 256 + lane * 8), y = *reinterpret_cast<const uint2*>(kraw + t * 256 + lane * 8);
            const float2 z = __ffma2_rn(unpack_bf16(x.y), unpack_bf16(y.y), __fmul2_rn(unpack_bf16(x.x), unpack_bf16(y.x)));
            v[t] = t < valid ? z.x + z.y : 0.f;
        }
        const float total = transpose_sum(v, lane);
        sc[lane * (VC + 1)] = total;
        sc[VC * VC + lane * (VC + 1)] = total;
    } else if (warp == 15 && i == 0) {
        // V rows past the end belong to the next sequence: they meet only zero weights, but 0 * inf is not 0
        for (int t = VC - 1; t >= valid; --t)
            if (lane < 16) *reinterpret_cast<uint4*>(tiles + OFF_V + buf * V_TILE + (lane >> 3) * V_HALF + t * 128 + (lane & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
}

__device__ __forceinline__ void vec_setup(VecShared& sh, int tid, int warp, int mma_warp) {
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.raw_full[i], 1); mbar_init(&sh.done[i], 1); }
        mbar_init(&sh.g2_full, 1);
        sh.abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == mma_warp) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
}

// ============================================================================================
// Main kernel
// ============================================================================================
__global__ void __launch_bounds__(V_NTHREADS, 1) prefill_vec_kernel(const __grid_constant__ CUtensorMap map_v, const VecParams vp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ VecShared sh;
    const PrefillParams& p = vp.p;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const VecUnit u = vec_unit(vp, blockIdx.x, vp.nseg);
    if (u.slot < 0 || u.slot >= p.num_slots) return;
    float* slot1 = p.state + ((size_t)u.slot * 2 * p.H + u.h) * (size_t)(D * D);
    const size_t state_stride = (size_t)p.H * D * D;
    if (u.len <= 0) {  // empty sequence: a fresh start leaves zero states, a resume leaves the slot alone
        if (u.g == 0 && !p.use_initial_state)
            for (int i = tid; i < 2 * D * D; i += V_NTHREADS) slot1[(size_t)(i / (D * D)) * state_stride + i % (D * D)] = 0.f;
        return;
    }
    if (u.c_begin >= u.c_end) return;
    const int nc = u.c_end - u.c_begin, tok0 = u.c_begin * VC, t0 = u.t_begin + tok0;
    const bool last = u.c_end == u.nchunks;
    vec_setup(sh, tid, warp, 0);
    if (tid >= 64 && tid < 96) {      // (row, column) of every score pair, in the order block_scores produces them; a row per lane
        const int j = lane + 1;
        for (int part = 0; part < 2; ++part) {
            const int s0 = part ? SPLIT_S : 0, s1 = part ? VB - 1 : SPLIT_S;
            int at = 0;
            for (int r = s0 + 1; r < j; ++r) at += min(r, s1) - s0;
            if (j < VB)
                for (int s = s0; s < min(j, s1); ++s, ++at) sh.pair[part][at] = (short)(j * VC + s);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    volatile int* abortp = &sh.abort_flag;
    const int q = warp & 3, cg = warp >> 2;          // TMEM lane quadrant and column group of this warp's share of a pass
    const uint32_t lane_addr = (uint32_t)(32 * q) << 16;      // (all of TMEM is allocated: column 0 is its base)
    const int v = 32 * q + lane;
    const float W1 = p.gamma[u.h] * p.scale, W2 = (1.f - p.gamma[u.h]) * p.scale;
    const __nv_bfloat16* qg = reinterpret_cast<const __nv_bfloat16*>(p.q);
    const __nv_bfloat16* kg = reinterpret_cast<const __nv_bfloat16*>(p.k);
    __nv_bfloat16* og = reinterpret_cast<__nv_bfloat16*>(p.o);
#define WAIT(bar, ph) mbar_wait(bar, (uint32_t)(ph), abortp, p.status)

    // one warp, a row per lane
    auto load_raw = [&](int c) {
        const int valid = min(VC, u.len - tok0 - c * VC), b = c & 1;
        if (lane == 0) mbar_arrive_expect_tx(&sh.raw_full[b], (uint32_t)(valid * (256 + 256 + 512) + V_TILE));
        __syncwarp();
        if (lane < valid) {
            const size_t off = ((size_t)(t0 + c * VC + lane) * p.H + u.h) * D;
            bulk_load(tiles + OFF_RAW + b * V_TILE + lane * 256, qg + off, 256, &sh.raw_full[b]);
            bulk_load(tiles + OFF_RAWK + b * V_TILE + lane * 256, kg + off, 256, &sh.raw_full[b]);
            bulk_load(tiles + OFF_G + lane * 512, p.g_hist + off, 512, &sh.raw_full[b]);
        }
        if (lane == 0) tma_load_4d(tiles + OFF_V + b * V_TILE, &map_v, &sh.raw_full[b], 0, t0 + c * VC, 0, u.h);
    };
    auto load_g2 = [&](int c) {
        const int valid = min(VC, u.len - tok0 - c * VC);
        if (lane == 0) mbar_arrive_expect_tx(&sh.g2_full, (uint32_t)(valid * 512));
        __syncwarp();
        if (lane < valid) bulk_load(tiles + OFF_G + VC * D * 4 + lane * 512, p.g_rec + ((size_t)(t0 + c * VC + lane) * p.H + u.h) * D, 512, &sh.g2_full);
    };
    // S_i -> two bf16 terms for the readout, then S_i diag(A_i); 32 columns (key channels) of one lane quadrant per warp
    auto pass = [&](int i) {
        uint32_t r[32], hi[16], lo[16];
        tmem_ld32(lane_addr + VCOL_S + 128 * i + 32 * cg, r);
        const float4* A = reinterpret_cast<const float4*>(tiles + OFF_A) + i * (D / 4) + 8 * cg;
        tc_wait_ld();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 a = A[k];
            float2 x = make_float2(__uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1])), y = make_float2(__uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3]));
            const float2 xs = __fmul2_rn(x, make_float2(a.x, a.y)), ys = __fmul2_rn(y, make_float2(a.z, a.w));
            hi[2 * k] = take_term(x); lo[2 * k] = pack_bf16(x.x, x.y);
            hi[2 * k + 1] = take_term(y); lo[2 * k + 1] = pack_bf16(y.x, y.y);
            r[4 * k] = __float_as_uint(xs.x); r[4 * k + 1] = __float_as_uint(xs.y); r[4 * k + 2] = __float_as_uint(ys.x); r[4 * k + 3] = __float_as_uint(ys.y);
        }
        tmem_st16(lane_addr + VCOL_SB + 16 * cg, hi);
        tmem_st16(lane_addr + VCOL_SB + 64 + 16 * cg, lo);
        tmem_st32(lane_addr + VCOL_S + 128 * i + 32 * cg, r);
        tc_wait_st();
    };
    auto outputs = [&](int c) {      // tokens 8 cg .. 8 cg + 7, one d_v lane per thread
        uint32_t r[8];
        tmem_ld8(lane_addr + VCOL_O + 8 * cg, r);
        const int valid = u.len - tok0 - c * VC - 8 * cg;
        __nv_bfloat16* dst = og + ((size_t)(t0 + c * VC + 8 * cg) * p.H + u.h) * D + v;
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < valid) dst[(size_t)j * p.H * D] = __float2bfloat16_rn(__uint_as_float(r[j]));
    };
    const uint32_t sa = (smem_u32(smem_raw) + 1023u) & ~1023u;
    auto issue = [&](int i, int buf) {      // by one thread
        constexpr uint32_t ID_RO = idesc_bf16(128, VC, 0, 0), ID_PV = idesc_bf16(128, VC, 1, 0), ID_U = idesc_bf16(128, 128, 1, 1);
        const uint32_t vd = smem_desc_lo(sa + OFF_V + buf * V_TILE, V_HALF), qd = smem_desc_lo(sa + OFF_QT + 2 * i * V_TILE, 16);
        const uint32_t kd = smem_desc_lo(sa + OFF_KT + 3 * i * V_TILE, V_HALF), pd = smem_desc_lo(sa + OFF_PT, 16);
#pragma unroll 1
        for (int m = 0; m < 3; ++m) {       // low x high, high x low, high x high terms
            const uint32_t a = VCOL_SB + (m == 0 ? 64 : 0), b = qd + (m == 1 ? V_TILE >> 4 : 0);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) mma_ts_lo(VCOL_O, a + 8 * kk, b + (uint32_t)((kk >> 2) * (V_HALF >> 4) + 2 * (kk & 3)), ID_RO, (i | m | kk) ? 1u : 0u);
        }
        if (i == 1) {
#pragma unroll
            for (int m = 0; m < 4; ++m) mma_ss_lo(VCOL_O, vd + (m & 1) * 128, pd + (uint32_t)((m >> 1) * (VC * 128 >> 4) + 2 * (m & 1)), ID_PV, 1u);
        }
#pragma unroll
        for (int m = 0; m < 6; ++m) mma_ss_lo(VCOL_S + 128 * i, vd + (m & 1) * 128, kd + (uint32_t)((m >> 1) * (V_TILE >> 4) + (m & 1) * 128), ID_U, 1u);
        tc_commit(&sh.done[i]);
    };

    if (warp == 15) { load_raw(0); load_g2(0); }
    {   // initial states: the slot, what the summaries were folded into, or zero
        const int i = warp >> 3, half = (warp >> 2) & 1;
        const bool load = u.g > 0 || p.use_initial_state;
        const float* base = vp.ws ? vp.ws + ((size_t)(u.n * p.H + u.h) * vp.nseg + u.g) * (VEC_STRIDE / 4) + (size_t)i * D * D : slot1 + (size_t)i * state_stride;
#pragma unroll 1
        for (int bt = 2 * half; bt < 2 * half + 2; ++bt) {
            uint32_t r[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) r[k] = load ? __float_as_uint(base[(size_t)(32 * bt + k) * D + v]) : 0u;
            tmem_st32(lane_addr + VCOL_S + 128 * i + 32 * bt, r);
        }
        tc_wait_st();
        tc_fence_before();
    }
    WAIT(&sh.raw_full[0], 0);
    build_operands(tiles, sh, 0, 0, min(VC, u.len - tok0), W1, warp, lane);
    fence_proxy_async_smem();
    __syncthreads();
    tc_fence_after();
#pragma unroll 1
    for (int c = 0; c < nc; ++c) {
        const int b = c & 1, valid = min(VC, u.len - tok0 - c * VC);
        // ---- phase A
        if (c > 0) {
            WAIT(&sh.done[1], (c - 1) & 1);
            tc_fence_after();
        }
        if (warp == 15 && c + 1 < nc) load_raw(c + 1);
        if (c > 0) outputs(c - 1);
        pass(0);
        tc_fence_before();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            issue(0, b);
        }
        __syncwarp();
        WAIT(&sh.g2_full, c & 1);
        build_operands(tiles, sh, 1, b, valid, W2, warp, lane);
        fence_proxy_async_smem();
        __syncthreads();
        // ---- phase B
        if (warp == 15 && c + 1 < nc) load_g2(c + 1);
        WAIT(&sh.done[0], c & 1);
        tc_fence_after();
        pass(1);
        {   // P~: two columns of one row per thread
            const int j = tid >> 4, s = (tid & 15) * 2;
            const float2 x = *reinterpret_cast<const float2*>(tiles + OFF_SC + (j * VC + s) * 4), y = *reinterpret_cast<const float2*>(tiles + OFF_SC + (VC * VC + j * VC + s) * 4);
            float2 z = make_float2(s <= j ? fmaf(W2, y.x, W1 * x.x) : 0.f, s + 1 <= j ? fmaf(W2, y.y, W1 * x.y) : 0.f);
            uint8_t* at = tiles + OFF_PT + j * 128 + (((s >> 3) ^ (j & 7)) << 4) + (s & 7) * 2;
            *reinterpret_cast<uint32_t*>(at) = take_term(z);
            *reinterpret_cast<uint32_t*>(at + VC * 128) = pack_bf16(z.x, z.y);
        }
        tc_fence_before();
        fence_proxy_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            issue(1, b);
        }
        __syncwarp();
        if (c + 1 < nc) {
            WAIT(&sh.raw_full[b ^ 1], ((c + 1) >> 1) & 1);
            build_operands(tiles, sh, 0, b ^ 1, min(VC, u.len - tok0 - (c + 1) * VC), W1, warp, lane);
        }
        fence_proxy_async_smem();
        __syncthreads();
    }
    WAIT(&sh.done[1], (nc - 1) & 1);
    tc_fence_after();
    outputs(nc - 1);
    if (last) store_state(slot1 + (size_t)(warp >> 3) * state_stride, v, lane_addr + VCOL_S + 128 * (warp >> 3), 2 * ((warp >> 2) & 1), 2 * ((warp >> 2) & 1) + 2);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(0, 512);
}

// ============================================================================================
// Segments: summaries and initial states
// ============================================================================================
// U_g (both states, accumulated from zero) and A_g (products of the segment's gates) of a segment that has a successor.  Warps 0..7
// build K~ (state, channel half, block), warp 8 loads and issues.
constexpr int VS_NTHREADS = 288;
__global__ void __launch_bounds__(VS_NTHREADS, 1) prefill_vec_summary_kernel(const __grid_constant__ CUtensorMap map_v, const VecParams vp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ VecShared sh;
    const PrefillParams& p = vp.p;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const VecUnit u = vec_unit(vp, blockIdx.x, vp.nseg - 1);
    if (u.slot < 0 || u.slot >= p.num_slots || u.len <= 0 || u.c_end >= u.nchunks) return;      // (c_end < nchunks: whole chunks only)
    const int nc = u.c_end - u.c_begin, t0 = u.t_begin + u.c_begin * VC;
    float* out = vp.ws + ((size_t)(u.n * p.H + u.h) * vp.nseg + u.g) * (VEC_STRIDE / 4);
    vec_setup(sh, tid, warp, 8);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    volatile int* abortp = &sh.abort_flag;
    const __nv_bfloat16* kg = reinterpret_cast<const __nv_bfloat16*>(p.k);
    const uint32_t sa = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int i = warp >> 2, hh = warp & 1, b = (warp >> 1) & 1;
    float2 carry = make_float2(1.f, 1.f);
    // step it = chunk nc - 1 - it; buffers by the parity of it
    auto load = [&](int it) {
        const int par = it & 1, t = t0 + (nc - 1 - it) * VC;
        const size_t off = ((size_t)(t + lane) * p.H + u.h) * D;
        if (lane == 0) mbar_arrive_expect_tx(&sh.raw_full[par], VC * (256 + 1024) + V_TILE);
        __syncwarp();
        bulk_load(tiles + OFF_SK + par * V_TILE + lane * 256, kg + off, 256, &sh.raw_full[par]);
        bulk_load(tiles + OFF_SG + par * 2 * VC * D * 4 + lane * 512, p.g_hist + off, 512, &sh.raw_full[par]);
        bulk_load(tiles + OFF_SG + (par * 2 + 1) * VC * D * 4 + lane * 512, p.g_rec + off, 512, &sh.raw_full[par]);
        if (lane == 0) tma_load_4d(tiles + OFF_V + par * V_TILE, &map_v, &sh.raw_full[par], 0, t, 0, u.h);
    };
    if (warp == 8) load(0);
#pragma unroll 1
    for (int it = 0; it < nc; ++it) {
        const int par = it & 1;
        if (warp == 8) {
            if (it + 1 < nc) {
                if (it >= 1) WAIT(&sh.done[par ^ 1], ((it - 1) >> 1) & 1);      // the MMAs of step it - 1 have read V
                load(it + 1);
            }
        } else {
            WAIT(&sh.raw_full[par], (it >> 1) & 1);
            if (it >= 2) WAIT(&sh.done[par], ((it >> 1) - 1) & 1);              // ... and those of step it - 2 this K~
            const float2 a = build_k(tiles + OFF_SKT + (par * 6 + 3 * i) * V_TILE, nullptr, tiles + OFF_SK + par * V_TILE,
                                     tiles + OFF_SG + (par * 2 + i) * VC * D * 4, hh, b, VC, carry, lane);
            carry = __fmul2_rn(carry, a);
            fence_proxy_async_smem();
        }
        __syncthreads();
        if (warp == 8 && elect_one()) {
            constexpr uint32_t ID_U = idesc_bf16(128, 128, 1, 1);
            WAIT(&sh.raw_full[par], (it >> 1) & 1);
            tc_fence_after();
            const uint32_t vd = smem_desc_lo(sa + OFF_V + par * V_TILE, V_HALF), kd = smem_desc_lo(sa + OFF_SKT + par * 6 * V_TILE, V_HALF);
#pragma unroll 1
            for (int m = 0; m < 6; ++m) {       // (state, term)
                const uint32_t d = VCOL_S + (m >= 3 ? 128 : 0), k = kd + (uint32_t)(m * (V_TILE >> 4)), fresh = (it == 0 && (m == 0 || m == 3)) ? 0u : 1u;
                mma_ss_lo(d, vd, k, ID_U, fresh);
                mma_ss_lo(d, vd + 128, k + 128, ID_U, 1u);
            }
            tc_commit(&sh.done[par]);
        }
        __syncwarp();
    }
    WAIT(&sh.done[(nc - 1) & 1], ((nc - 1) >> 1) & 1);
    tc_fence_after();
    if (warp < 8) {
        store_state(out + (size_t)i * D * D, 32 * (warp & 3) + lane, ((uint32_t)(32 * (warp & 3)) << 16) + VCOL_S + 128 * i, 0, 4);
        if (b == 0) reinterpret_cast<float2*>(out + 2 * D * D)[i * (D / 2) + 32 * hh + lane] = carry;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(0, 512);
}
#undef WAIT

// Summaries -> initial states, in place: S_g = fold over earlier segments of (S <- diag(A_j) S + U_j), from the slot or zero.  Four
// elements of one state row per thread.
__global__ void __launch_bounds__(256) prefill_vec_fold_kernel(const VecParams vp) {
    const PrefillParams& p = vp.p;
    const int part = blockIdx.x % (2 * 16), unit = blockIdx.x / (2 * 16), i = part >> 4;
    const int e = ((part & 15) * 256 + threadIdx.x) * 4, row = e / D;
    const int n = unit / p.H, h = unit % p.H;
    const int slot = p.slots ? p.slots[n] : n;
    if (slot < 0 || slot >= p.num_slots) return;
    const int len = p.cu_seqlens ? p.cu_seqlens[n + 1] - p.cu_seqlens[n] : p.T;
    if (len <= 0) return;
    const int last = min(vp.nseg - 1, ((len + VC - 1) / VC - 1) / vp.cps);
    float* at = vp.ws + (size_t)unit * vp.nseg * (VEC_STRIDE / 4) + (size_t)i * D * D + e;
    const float* A = vp.ws + (size_t)unit * vp.nseg * (VEC_STRIDE / 4) + 2 * D * D + i * D + row;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.use_initial_state) s = *reinterpret_cast<const float4*>(p.state + (((size_t)slot * 2 + i) * p.H + h) * (size_t)(D * D) + e);
#pragma unroll 4
    for (int g = 0; g <= last; ++g, at += VEC_STRIDE / 4, A += VEC_STRIDE / 4) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        float a = 0.f;
        if (g < last) { x = *reinterpret_cast<const float4*>(at); a = *A; }
        *reinterpret_cast<float4*>(at) = s;
        s.x = fmaf(a, s.x, x.x); s.y = fmaf(a, s.y, x.y); s.z = fmaf(a, s.z, x.z); s.w = fmaf(a, s.w, x.w);
    }
}

}  // namespace

// bf16, d = 128, both gate tensors on 16-byte boundaries (their rows are copied in bulk)
bool prefill_vec_applies(const dsla_prefill_args* a) {
    return a->dtype == DSLA_BF16 && a->d_k == D && a->T_total > 0 && reinterpret_cast<uintptr_t>(a->g_hist) % 16 == 0 &&
           reinterpret_cast<uintptr_t>(a->g_rec) % 16 == 0;
}

dsla_status launch_prefill_vec(const PrefillParams& p, const dsla_prefill_args* a, cudaStream_t s) {
    VecParams vp;
    vp.p = p;
    const long long units = (long long)p.N * p.H;
    const int max_chunks = (a->max_seqlen + VC - 1) / VC;
    // Segments: as many as keep every SM at one CTA, at least eight chunks each (below that the two extra launches cost more than the
    // shorter chains save), and no more than the workspace holds (these calls need none: without one a sequence is one segment).
    int ns = (int)(148 / units);
    if (ns > 16) ns = 16;
    while (ns > 1 && ((max_chunks + ns - 1) / ns < 8 || (size_t)units * ns * VEC_STRIDE > a->workspace_bytes)) --ns;
    if (ns < 1 || !a->workspace || reinterpret_cast<uintptr_t>(a->workspace) % 16 != 0) ns = 1;
    vp.nseg = ns;
    vp.cps = ns > 1 ? (max_chunks + ns - 1) / ns : max_chunks;
    vp.ws = ns > 1 ? static_cast<float*>(a->workspace) : nullptr;
    if (units * ns > 0x7fffffffLL / 32) return DSLA_ERR_UNSUPPORTED;
    CUtensorMap mv;
    if (!make_tile_map(&mv, p.v, a->T_total, p.H, VC)) return DSLA_ERR_CUDA;
    if (ns > 1) {
        if (cudaFuncSetAttribute(prefill_vec_summary_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, V_SMEM_SUM) != cudaSuccess) return DSLA_ERR_CUDA;
        prefill_vec_summary_kernel<<<dim3((unsigned)(units * (ns - 1))), dim3(VS_NTHREADS), V_SMEM_SUM, s>>>(mv, vp);
        prefill_vec_fold_kernel<<<dim3((unsigned)(units * 2 * 16)), dim3(256), 0, s>>>(vp);
        count_launch(2);
    }
    if (cudaFuncSetAttribute(prefill_vec_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, V_SMEM) != cudaSuccess) return DSLA_ERR_CUDA;
    prefill_vec_kernel<<<dim3((unsigned)(units * ns)), dim3(V_NTHREADS), V_SMEM, s>>>(mv, vp);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DSLA_OK : DSLA_ERR_CUDA;
}

}  // namespace dsla
