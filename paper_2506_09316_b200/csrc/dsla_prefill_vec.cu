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
// The tensor core cuts its fp32 sums off instead of rounding them: every MMA onto a state would move it by up to an ulp, always
// towards zero (six per chunk: states off by 1.5e-6 after 4096 tokens, 3.4e-7 token by token).  So what a chunk adds to a
// state, V^T (s_i (.) K), is a sum of its own from zero, smallest terms first, and is added on CUDA cores.
// An infinity or NaN in V would reach the tokens before it through the zeros of P~: the outputs of such a chunk are finished on CUDA cores.
//
// CTA = (sequence, head, segment), 16 warps in step: each step takes one state through its pass (two bf16 terms of it for the
// readout, then S_i diag(A_i)) and its MMAs, and meanwhile builds the operands of the other state for its next turn, so
// nothing but the raw inputs is double-buffered.  16.7 k cycles per chunk, of which 7600 issue a warp instruction on each SM
// sub-partition (57 %; half of the instructions for the operands, a quarter for the scores): the warps have unequal shares and wait for
// the longest one at the barriers of every step.
//
// A sequence is split into segments when there are few (sequence, head) pairs and the caller's workspace has room: a first
// grid accumulates each segment's state from zero, walking the chunks backwards with the product of all later gates (no pass
// over the states), and the main grid folds the summaries of the earlier segments into its initial states.
// T = 4096, 32 heads: 300 us (of them 64 for the summaries; 280 with the MMAs onto the states); 2490 us with the token-by-token kernel.
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
constexpr int V_GBYTES = 2 * VC * D * 4;
constexpr int OFF_G = OFF_RAWK + 2 * V_TILE;         // gates: [buffer][state][32][128] fp32
constexpr int OFF_SC = OFF_G + 2 * V_GBYTES;         // blended scores [buffer][32][32] fp32
constexpr int OFF_A = OFF_SC + 2 * VC * VC * 4;          // chunk decays: [state][128] fp32
constexpr int V_SMEM = OFF_A + 2 * D * 4 + 1024;
// summaries reuse the front: V buffers, then K~ [parity][state][term]
constexpr int OFF_SKT = 2 * V_TILE;
constexpr int OFF_SG = OFF_SKT + 12 * V_TILE;        // gates [parity][state][32][128] fp32
constexpr int OFF_SK = OFF_SG + 2 * V_GBYTES;        // raw K [parity]
constexpr int V_SMEM_SUM = OFF_SK + 2 * V_TILE + 1024;
// TMEM columns: fp32 states 2 x 128; the bf16 terms of one state, per 32 key channels 16 columns of high ones, then 16 of low ones, and when the
// readout has read them what the chunk adds to that state, fp32 (so that each warp overwrites only columns it has read); O^T 32
constexpr uint32_t VCOL_S = 0, VCOL_SB = 256, VCOL_O = 384;
constexpr size_t VEC_STRIDE = (2 * D * D + 2 * D) * sizeof(float);      // one summary: U[2][d][d], A[2][d]

struct VecParams {
    PrefillParams p;
    float* ws;           // summaries / initial states [(n*H + h)*nseg + g], or nullptr (nseg = 1)
    int nseg, cps;       // segments per sequence, chunks per segment
};

struct alignas(16) VecShared {
    uint64_t raw_full[2], done[2], ro;
    uint32_t tmem_base;
    int abort_flag;
    int inf_in_v[4];     // [chunk % 4]: chunk + 1 if V of the chunk holds an infinity or NaN
};

// bf16 terms of a pair of fp32 values; x is left with what the term does not hold
__device__ __forceinline__ uint32_t take_term(float2& x) {
    const uint32_t t = pack_bf16(x.x, x.y);
    const float2 f = unpack_bf16(t);
    x = __ffma2_rn(f, make_float2(-1.f, -1.f), x);      // exact
    return t;
}

// Sums over the lanes of N values per lane (a power of two): lane l is left with the total of v[l % N].
template <int N>
__device__ __forceinline__ float transpose_sum(float* v, int lane) {
#pragma unroll
    for (int off = N / 2; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float send = up ? v[i] : v[i + off], keep = up ? v[i + off] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (int off = N; off < 32; off <<= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
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

// Blended scores of a block of 16 tokens: keys s0 .. s0 + 3 with tokens j_begin .. j_end - 1 (the current token, undecayed, included), four
// channels per lane, four tokens per round.  Both states share the product with q and the sums over the lanes: their
// decayed copies of k are added first.
// (A loop over the tokens, not unrolled code: every role of this kernel passes through its code once per phase, and when that
// does not fit the instruction cache all of them wait for it.  Unrolled to all pairs: twice the time per phase.)
__device__ __forceinline__ void block_scores(const uint8_t* q, const uint8_t* k, const uint8_t* g, int s0, int j_begin, int j_end, float W1, float W2, int lane, float* out) {
    float2 k1[4][2], k2[4][2];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint2 x = *reinterpret_cast<const uint2*>(k + (s0 + e) * 256 + lane * 8);
        const float2 a = unpack_bf16(x.x), b = unpack_bf16(x.y);
        k1[e][0] = __fmul2_rn(a, make_float2(W1, W1)); k1[e][1] = __fmul2_rn(b, make_float2(W1, W1));
        k2[e][0] = __fmul2_rn(a, make_float2(W2, W2)); k2[e][1] = __fmul2_rn(b, make_float2(W2, W2));
    }
#pragma unroll 1
    for (int j = s0 + 1; j < j_begin; ++j) {      // decays up to the first token of this warp's part
        const float4 g1 = *reinterpret_cast<const float4*>(g + j * 512 + lane * 16), g2 = *reinterpret_cast<const float4*>(g + V_GBYTES / 2 + j * 512 + lane * 16);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (s0 + e < j) {
                k1[e][0] = __fmul2_rn(k1[e][0], make_float2(g1.x, g1.y)); k1[e][1] = __fmul2_rn(k1[e][1], make_float2(g1.z, g1.w));
                k2[e][0] = __fmul2_rn(k2[e][0], make_float2(g2.x, g2.y)); k2[e][1] = __fmul2_rn(k2[e][1], make_float2(g2.z, g2.w));
            }
    }
#pragma unroll 1
    for (int j0 = j_begin; j0 < j_end; j0 += 4) {
        float v[16];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int j = j0 + r;
            const uint2 x = *reinterpret_cast<const uint2*>(q + j * 256 + lane * 8);
            const float4 g1 = *reinterpret_cast<const float4*>(g + j * 512 + lane * 16), g2 = *reinterpret_cast<const float4*>(g + V_GBYTES / 2 + j * 512 + lane * 16);
            const float2 q0 = unpack_bf16(x.x), q1 = unpack_bf16(x.y);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (e < r || j0 > s0) {      // key s0 + e is earlier than token j
                    k1[e][0] = __fmul2_rn(k1[e][0], make_float2(g1.x, g1.y)); k1[e][1] = __fmul2_rn(k1[e][1], make_float2(g1.z, g1.w));
                    k2[e][0] = __fmul2_rn(k2[e][0], make_float2(g2.x, g2.y)); k2[e][1] = __fmul2_rn(k2[e][1], make_float2(g2.z, g2.w));
                }
                const float2 y = __ffma2_rn(q1, __fadd2_rn(k1[e][1], k2[e][1]), __fmul2_rn(q0, __fadd2_rn(k1[e][0], k2[e][0])));
                v[4 * r + e] = y.x + y.y;
            }
        }
        const float total = transpose_sum<16>(v, lane);
        if (lane < 16) out[(j0 + (lane >> 2)) * VC + s0 + (lane & 3)] = total;      // (above the diagonal: never read)
    }
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t saddr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}

// Byte offset of this lane's channel pair (channels 64 hh + 2 lane, + 1) of a row in a swizzled tile whose halves are `half` bytes.
__device__ __forceinline__ uint32_t pair_at(int row, int hh, int lane, int half) {
    return (uint32_t)(hh * half + row * 128 + ((((lane >> 2) ^ (row & 7)) << 4) | ((lane & 3) << 2)));
}
__device__ __forceinline__ float2 gate_pair(const uint8_t* g, int t) { return *reinterpret_cast<const float2*>(g + t * 512); }

// The four builders below take the raw rows and gates of one channel half (a channel pair per lane).
// Q~ of one state, two terms: rows 16 b .. 16 b + 15 of Q scaled from the chunk's start.
__device__ __forceinline__ void build_q(uint8_t* qt, const uint8_t* q, const uint8_t* g, int hh, int b, float W, int lane) {
    float2 pr = make_float2(W, W);
    if (b == 1) {
#pragma unroll 8
        for (int t = 0; t < VB; ++t) pr = __fmul2_rn(pr, gate_pair(g, t));
    }
    q += b * VB * 256; g += b * VB * 512; qt += b * VB * 128;
#pragma unroll 4
    for (int t = 0; t < VB; ++t) {
        pr = __fmul2_rn(pr, gate_pair(g, t));
        float2 y = __fmul2_rn(unpack_bf16(*reinterpret_cast<const uint32_t*>(q + t * 256)), pr);
        const uint32_t at = pair_at(t, hh, lane, V_HALF);
        *reinterpret_cast<uint32_t*>(qt + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(qt + V_TILE + at) = pack_bf16(y.x, y.y);
    }
}
// Rows 16..31 of Q scaled from their block's start, two terms.
__device__ __forceinline__ void build_qb(uint8_t* qb, const uint8_t* q, const uint8_t* g, int hh, float W, int lane) {
    float2 pr = make_float2(W, W);
    q += VB * 256; g += VB * 512;
#pragma unroll 4
    for (int t = 0; t < VB; ++t) {
        pr = __fmul2_rn(pr, gate_pair(g, t));
        float2 y = __fmul2_rn(unpack_bf16(*reinterpret_cast<const uint32_t*>(q + t * 256)), pr);
        const uint32_t at = pair_at(t, hh, lane, V_BHALF);
        *reinterpret_cast<uint32_t*>(qb + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(qb + V_BTILE + at) = pack_bf16(y.x, y.y);
    }
}
// Rows 0..15 of K scaled to their block's end, two terms.
__device__ __forceinline__ void build_kb(uint8_t* kb, const uint8_t* k, const uint8_t* g, int hh, int lane) {
    float2 sf = make_float2(1.f, 1.f);
#pragma unroll 4
    for (int t = VB - 1; t >= 0; --t) {
        float2 y = __fmul2_rn(unpack_bf16(*reinterpret_cast<const uint32_t*>(k + t * 256)), sf);
        const uint32_t at = pair_at(t, hh, lane, V_BHALF);
        *reinterpret_cast<uint32_t*>(kb + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(kb + V_BTILE + at) = pack_bf16(y.x, y.y);
        sf = __fmul2_rn(sf, gate_pair(g, t));
    }
}
// K~ of one state, three terms: rows t_begin .. t_begin + ROWS - 1 of K scaled to the chunk's end times `carry`.  Returns the
// product of the gates from row t_begin on, times carry.
template <int ROWS, bool CLAMP>
__device__ __forceinline__ float2 build_k(uint8_t* kt, const uint8_t* k, const uint8_t* g, int hh, int t_begin, float2 carry, int lane) {
    auto gate = [&](int t) {
        const float2 x = gate_pair(g, t);
        return CLAMP ? make_float2(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f)) : x;
    };
    float2 sf = carry;
#pragma unroll 8
    for (int t = VC - 1; t >= t_begin + ROWS; --t) sf = __fmul2_rn(sf, gate(t));
    k += t_begin * 256; g += t_begin * 512; kt += t_begin * 128;
#pragma unroll 4
    for (int t = ROWS - 1; t >= 0; --t) {
        float2 y = __fmul2_rn(unpack_bf16(*reinterpret_cast<const uint32_t*>(k + t * 256)), sf);
        const uint32_t at = pair_at(t, hh, lane, V_HALF);      // (t_begin is a multiple of 8)
        *reinterpret_cast<uint32_t*>(kt + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(kt + V_TILE + at) = take_term(y);
        *reinterpret_cast<uint32_t*>(kt + 2 * V_TILE + at) = pack_bf16(y.x, y.y);
        sf = __fmul2_rn(sf, gate(t));
    }
    return sf;
}

// Scores between the blocks, rows 16..31 x columns 8 nt .. 8 nt + 7: two-term operands, the product of the two low terms left out.
__device__ __forceinline__ void cross_scores(const uint8_t* tiles, int nt, int lane, bool add, float* out) {
    float* o = out + (VB + (lane >> 2)) * VC + 8 * nt + 2 * (lane & 3);
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    if (add) { c[0] = o[0]; c[1] = o[1]; c[2] = o[8 * VC]; c[3] = o[8 * VC + 1]; }
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
    *reinterpret_cast<float2*>(o) = make_float2(c[0], c[1]);
    *reinterpret_cast<float2*>(o + 8 * VC) = make_float2(c[2], c[3]);
}

// The operands of state i of a chunk, and half of its scores: block i of 16 tokens and this state's share between the blocks.
__device__ __forceinline__ void build_operands(uint8_t* tiles, int i, int buf, float W1, float W2, int warp, int lane) {
    const uint8_t* qraw = tiles + OFF_RAW + buf * V_TILE;
    const uint8_t* kraw = tiles + OFF_RAWK + buf * V_TILE;
    const uint8_t* graw = tiles + OFF_G + buf * V_GBYTES;
    float* sc = reinterpret_cast<float*>(tiles + OFF_SC) + buf * VC * VC;
    const int hh = warp & 1;
    const float W = i == 0 ? W1 : W2;
    const uint8_t *qh = qraw + hh * 128 + lane * 4, *kh = kraw + hh * 128 + lane * 4, *gh = graw + i * (V_GBYTES / 2) + hh * 256 + lane * 8;
    if (warp < 4) {
        build_q(tiles + OFF_QT + 2 * i * V_TILE, qh, gh, hh, warp >> 1, W, lane);
    } else if (warp < 8) {
        const int b = (warp - 4) >> 1;
        const float2 a = build_k<VB, false>(tiles + OFF_KT + 3 * i * V_TILE, kh, gh, hh, b * VB, make_float2(1.f, 1.f), lane);
        if (b == 0) reinterpret_cast<float2*>(tiles + OFF_A)[i * (D / 2) + 32 * hh + lane] = a;
    } else if (warp < 12) {
        // ten rounds of 4 x 4 tokens and keys: 2 + 1, 3, 2 and 2 (behind eight tokens' decays)
        const uint8_t *q = qraw + i * VB * 256, *k = kraw + i * VB * 256, *g = graw + i * VB * 512;
#pragma unroll 1
        for (int part = 0; part < (warp == 8 ? 2 : 1); ++part) {
            const int s0 = warp == 8 ? 12 * part : warp == 11 ? 0 : 4 * (warp - 8);
            block_scores(q, k, g, s0, warp == 11 ? 8 : s0, warp == 8 && part == 0 ? 8 : VB, W1, W2, lane, sc + i * (VB * VC + VB));
        }
    } else if (warp < 14) {
        build_qb(tiles + OFF_QB, qh, gh, hh, W, lane);
        asm volatile("bar.arrive 1, 128;" ::: "memory");
    } else {
        build_kb(tiles + OFF_KB, kh, gh, hh, lane);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        cross_scores(tiles, hh, lane, i == 1, sc);
    }
}

// Outputs of a chunk whose V holds an infinity or NaN (cold path, out of line).  A product with P~ would carry that to the tokens before
// it, whose weight for it is 0: O^T from the states alone, and V of the tokens up to each one added here.
__device__ __noinline__ void outputs_by_hand(const uint8_t* tiles, int buf, __nv_bfloat16* o, int H, int valid, int warp, int lane) {
    const int v = 32 * (warp & 3) + lane, j0 = 8 * (warp >> 2);
    const float* sc = reinterpret_cast<const float*>(tiles + OFF_SC) + buf * VC * VC;
    const uint8_t* vt = tiles + OFF_V + buf * V_TILE + (v >> 6) * V_HALF + (v & 7) * 2;
    uint32_t r[8];
    tmem_ld8(((uint32_t)(32 * (warp & 3)) << 16) + VCOL_O + j0, r);
    tc_wait_ld();
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int j = j0 + e;
        float x = __uint_as_float(r[e]);
#pragma unroll 1
        for (int s = 0; s <= j; ++s)
            x = fmaf(sc[j * VC + s], __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(vt + s * 128 + ((((v & 63) >> 3) ^ (s & 7)) << 4))), x);
        if (j < valid) o[(size_t)j * H * D + v] = __float2bfloat16_rn(x);
    }
}

__device__ __forceinline__ void vec_setup(VecShared& sh, int tid, int warp, int mma_warp) {
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.raw_full[i], 1); mbar_init(&sh.done[i], 1); }
        mbar_init(&sh.ro, 1);
        for (int i = 0; i < 4; ++i) sh.inf_in_v[i] = 0;
        sh.abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == mma_warp) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
}

// ============================================================================================
// Main kernel
// ============================================================================================
__global__ void __launch_bounds__(V_NTHREADS, 1) prefill_vec_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                                                                   const __grid_constant__ CUtensorMap map_g1, const __grid_constant__ CUtensorMap map_g2, const VecParams vp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ VecShared sh;
    const PrefillParams& p = vp.p;
    uint8_t* tiles = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);      // (an offset, not a rounded address: the compiler still knows that it is shared memory)
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
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    volatile int* abortp = &sh.abort_flag;
    const int q = warp & 3, cg = warp >> 2;          // TMEM lane quadrant and column group of this warp's share of a pass
    const uint32_t lane_addr = (uint32_t)(32 * q) << 16;      // (all of TMEM is allocated: column 0 is its base)
    const int v = 32 * q + lane;
    const float W1 = p.gamma[u.h] * p.scale, W2 = (1.f - p.gamma[u.h]) * p.scale;
    __nv_bfloat16* og = reinterpret_cast<__nv_bfloat16*>(p.o);
#define WAIT(bar, ph) mbar_wait(bar, (uint32_t)(ph), abortp, p.status)

    auto load_raw = [&](int c) {      // by one thread
        const int b = c & 1, t = t0 + c * VC;
        mbar_arrive_expect_tx(&sh.raw_full[b], 3 * V_TILE + V_GBYTES);
        tma_load_3d(tiles + OFF_G + b * V_GBYTES, &map_g1, &sh.raw_full[b], 0, u.h, t);
        tma_load_3d(tiles + OFF_G + b * V_GBYTES + V_GBYTES / 2, &map_g2, &sh.raw_full[b], 0, u.h, t);
        tma_load_3d(tiles + OFF_RAW + b * V_TILE, &map_q, &sh.raw_full[b], 0, u.h, t);
        tma_load_3d(tiles + OFF_RAWK + b * V_TILE, &map_k, &sh.raw_full[b], 0, u.h, t);
        tma_load_4d(tiles + OFF_V + b * V_TILE, &map_v, &sh.raw_full[b], 0, t, 0, u.h);
    };
    // Gates below 0 count as 0; past the end of the sequence gates are 1 and the other rows 0 (what landed there belongs to the next
    // sequence: it would meet only zero weights, but 0 * inf is not 0).
    auto clean = [&](int c) {
        const int b = c & 1, valid = u.len - tok0 - c * VC;
        float4* g = reinterpret_cast<float4*>(tiles + OFF_G + b * V_GBYTES);
#pragma unroll
        for (int m = 0; m < V_GBYTES / 16 / V_NTHREADS; ++m) {
            const int idx = tid + m * V_NTHREADS;
            const float4 x = g[idx];
            g[idx] = ((idx >> 5) & (VC - 1)) < valid ? make_float4(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f), fmaxf(x.z, 0.f), fmaxf(x.w, 0.f)) : make_float4(1.f, 1.f, 1.f, 1.f);
        }
        if (valid < VC) {
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            if ((tid >> 4) >= valid) {
                reinterpret_cast<uint4*>(tiles + OFF_RAW + b * V_TILE)[tid] = zero;
                reinterpret_cast<uint4*>(tiles + OFF_RAWK + b * V_TILE)[tid] = zero;
            }
            if (((tid >> 3) & (VC - 1)) >= valid) reinterpret_cast<uint4*>(tiles + OFF_V + b * V_TILE)[tid] = zero;
        }
        const uint4 y = reinterpret_cast<const uint4*>(tiles + OFF_V + b * V_TILE)[tid];      // (this thread's own piece in both cases)
        if (hfma2_u32(y.x, 0u, hfma2_u32(y.y, 0u, hfma2_u32(y.z, 0u, hmul2_u32(y.w, 0u)))) & 0x7fff7fffu) sh.inf_in_v[c & 3] = c + 1;
    };
    // S_i += d, which its last chunk added; 32 columns (key channels) of one lane quadrant per warp
    auto merge = [&](int i, const uint32_t (&d)[32]) {
        uint32_t r[32];
        tmem_ld32(lane_addr + VCOL_S + 128 * i + 32 * cg, r);
        tc_wait_ld();
#pragma unroll
        for (int k = 0; k < 32; k += 2) {
            const float2 x = __fadd2_rn(make_float2(__uint_as_float(r[k]), __uint_as_float(r[k + 1])), make_float2(__uint_as_float(d[k]), __uint_as_float(d[k + 1])));
            r[k] = __float_as_uint(x.x); r[k + 1] = __float_as_uint(x.y);
        }
        tmem_st32(lane_addr + VCOL_S + 128 * i + 32 * cg, r);
        tc_wait_st();
        tc_fence_before();
    };
    // S_i -> two bf16 terms for the readout, over the other state's sum (which moves into d), then S_i diag(A_i)
    auto pass = [&](int i, bool sum, uint32_t (&d)[32]) {
        uint32_t r[32], hl[32];
        if (sum) tmem_ld32(lane_addr + VCOL_SB + 32 * cg, d);
        tmem_ld32(lane_addr + VCOL_S + 128 * i + 32 * cg, r);
        const float4* A = reinterpret_cast<const float4*>(tiles + OFF_A) + i * (D / 4) + 8 * cg;
        tc_wait_ld();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 a = A[k];
            float2 x = make_float2(__uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1])), y = make_float2(__uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3]));
            const float2 xs = __fmul2_rn(x, make_float2(a.x, a.y)), ys = __fmul2_rn(y, make_float2(a.z, a.w));
            hl[2 * k] = take_term(x); hl[16 + 2 * k] = pack_bf16(x.x, x.y);
            hl[2 * k + 1] = take_term(y); hl[17 + 2 * k] = pack_bf16(y.x, y.y);
            r[4 * k] = __float_as_uint(xs.x); r[4 * k + 1] = __float_as_uint(xs.y); r[4 * k + 2] = __float_as_uint(ys.x); r[4 * k + 3] = __float_as_uint(ys.y);
        }
        tmem_st32(lane_addr + VCOL_SB + 32 * cg, hl);
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
    auto inf_in_v = [&](int c) { return sh.inf_in_v[c & 3] == c + 1; };
    auto readout = [&](int i, int buf, bool with_v) {      // by one thread
        constexpr uint32_t ID_RO = idesc_bf16(128, VC, 0, 0), ID_PV = idesc_bf16(128, VC, 1, 0);
        const uint32_t vd = smem_desc_lo(sa + OFF_V + buf * V_TILE, V_HALF), qd = smem_desc_lo(sa + OFF_QT + 2 * i * V_TILE, 16), pd = smem_desc_lo(sa + OFF_PT, 16);
#pragma unroll 1
        for (int m = 0; m < 3; ++m) {       // low x high, high x low, high x high terms
            const uint32_t a = VCOL_SB + (m == 0 ? 16 : 0), b = qd + (m == 1 ? V_TILE >> 4 : 0);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_ts_lo(VCOL_O, a + 32 * (kk >> 1) + 8 * (kk & 1), b + (uint32_t)((kk >> 2) * (V_HALF >> 4) + 2 * (kk & 3)), ID_RO, (i | m | kk) ? 1u : 0u);
        }
        if (i == 1 && with_v) {
#pragma unroll
            for (int m = 0; m < 4; ++m) mma_ss_lo(VCOL_O, vd + (m & 1) * 128, pd + (uint32_t)((m >> 1) * (VC * 128 >> 4) + 2 * (m & 1)), ID_PV, 1u);
        }
        tc_commit(&sh.ro);
    };
    auto update = [&](int i, int buf) {       // by one thread, behind the readout: over the terms that it has read
        constexpr uint32_t ID_U = idesc_bf16(128, 128, 1, 1);
        const uint32_t vd = smem_desc_lo(sa + OFF_V + buf * V_TILE, V_HALF), kd = smem_desc_lo(sa + OFF_KT + 3 * i * V_TILE, V_HALF);
#pragma unroll
        for (int m = 0; m < 6; ++m) mma_ss_lo(VCOL_SB, vd + (m & 1) * 128, kd + (uint32_t)((2 - (m >> 1)) * (V_TILE >> 4) + (m & 1) * 128), ID_U, m ? 1u : 0u);
        tc_commit(&sh.done[i]);
    };

    if (warp == 15 && lane == 0) load_raw(0);
    // Initial states: the slot (or zero) pushed through the summaries of the earlier segments, S <- diag(A_j) S + U_j.  The summary
    // of the first one holds the slot's share already, and the entry of the last segment, which has no summary, a copy of the
    // slot for the first (the CTA of the last segment overwrites the slot itself).
    if (vp.ws) asm volatile("griddepcontrol.wait;" ::: "memory");
    {
        const int i = warp >> 3, half = (warp >> 2) & 1;
        const float* unit = vp.ws ? vp.ws + (size_t)(u.n * p.H + u.h) * vp.nseg * (VEC_STRIDE / 4) : nullptr;
        const float* first = (u.g == 0 && last) ? slot1 + (size_t)i * state_stride : u.g == 0 ? unit + (size_t)(vp.nseg - 1) * (VEC_STRIDE / 4) + (size_t)i * D * D : unit + (size_t)i * D * D;
        const bool load = u.g > 0 || p.use_initial_state;
#pragma unroll 1
        for (int bt = 2 * half; bt < 2 * half + 2; ++bt) {
            float acc[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) acc[k] = load ? first[(size_t)(32 * bt + k) * D + v] : 0.f;
#pragma unroll 1
            for (int jg = 1; jg < u.g; ++jg) {
                const float* U = unit + (size_t)jg * (VEC_STRIDE / 4);
                const float4* A = reinterpret_cast<const float4*>(U + 2 * D * D + i * D + 32 * bt);
                float x[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) x[k] = U[(size_t)i * D * D + (size_t)(32 * bt + k) * D + v];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 a = A[k];
                    acc[4 * k] = fmaf(a.x, acc[4 * k], x[4 * k]); acc[4 * k + 1] = fmaf(a.y, acc[4 * k + 1], x[4 * k + 1]);
                    acc[4 * k + 2] = fmaf(a.z, acc[4 * k + 2], x[4 * k + 2]); acc[4 * k + 3] = fmaf(a.w, acc[4 * k + 3], x[4 * k + 3]);
                }
            }
            uint32_t r[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) r[k] = __float_as_uint(acc[k]);
            tmem_st32(lane_addr + VCOL_S + 128 * i + 32 * bt, r);
        }
        tc_wait_st();
        tc_fence_before();
    }
    WAIT(&sh.raw_full[0], 0);
    clean(0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Step hs = 2 c + i: pass over state i, its MMAs for chunk c, the operands of the other state.  One body for both phases (and for the
    // first operands, hs = -1): the code has to stay in the instruction cache.
#pragma unroll 1
    for (int hs = -1; hs < 2 * nc; ++hs) {
        const int i = hs & 1, c = hs >> 1, b = c & 1;
        if (hs >= 0) {
            if (hs > 0) {
                WAIT(&sh.done[i ^ 1], ((hs - 1) >> 1) & 1);
                tc_fence_after();
            }
            if (i == 0) {
                const bool by_hand = c > 0 && inf_in_v(c - 1);
                if (by_hand) {      // before the next V takes the place of that one
                    outputs_by_hand(tiles, b ^ 1, og + ((size_t)(t0 + (c - 1) * VC) * p.H + u.h) * D, p.H, VC, warp, lane);
                    __syncthreads();
                }
                if (warp == 15 && lane == 0 && c + 1 < nc && !*abortp) load_raw(c + 1);
                __syncwarp();
                if (c > 0 && !by_hand) outputs(c - 1);
            } else {      // P~: two columns of one row per thread
                const int j = tid >> 4, s = (tid & 15) * 2;
                const float2 x = *reinterpret_cast<const float2*>(tiles + OFF_SC + (b * VC * VC + j * VC + s) * 4);
                float2 z = make_float2(s <= j ? x.x : 0.f, s + 1 <= j ? x.y : 0.f);
                uint8_t* at = tiles + OFF_PT + j * 128 + (((s >> 3) ^ (j & 7)) << 4) + (s & 7) * 2;
                *reinterpret_cast<uint32_t*>(at) = take_term(z);
                *reinterpret_cast<uint32_t*>(at + VC * 128) = pack_bf16(z.x, z.y);
                fence_proxy_async_smem();
            }
            uint32_t d[32];
            pass(i, hs > 0, d);
            tc_fence_before();
            if (warp == 1) {      // only the issuing warp waits for the others
                asm volatile("bar.sync 2, 512;" ::: "memory");
                if (elect_one()) {
                    tc_fence_after();
                    readout(i, b, !inf_in_v(c));
                }
                __syncwarp();
            } else {
                asm volatile("bar.arrive 2, 512;" ::: "memory");
            }
            if (hs > 0) merge(i ^ 1, d);
        }
        if (hs >= 0 && warp == 12) {      // (one of the warps with the least to build; behind its build: 1 % of the kernel's time more)
            WAIT(&sh.ro, hs & 1);
            if (elect_one()) {
                tc_fence_after();
                update(i, b);
            }
            __syncwarp();
        }
        if (hs + 1 < 2 * nc) build_operands(tiles, i ^ 1, i == 0 ? b : b ^ 1, W1, W2, warp, lane);
        if (i == 0 && c + 1 < nc) {
            WAIT(&sh.raw_full[b ^ 1], ((c + 1) >> 1) & 1);
            clean(c + 1);
        }
        fence_proxy_async_smem();
        __syncthreads();
    }
    WAIT(&sh.done[1], (nc - 1) & 1);
    tc_fence_after();
    if (inf_in_v(nc - 1)) outputs_by_hand(tiles, (nc - 1) & 1, og + ((size_t)(t0 + (nc - 1) * VC) * p.H + u.h) * D, p.H, u.len - tok0 - (nc - 1) * VC, warp, lane);
    else outputs(nc - 1);
    {
        uint32_t d[32];
        tmem_ld32(lane_addr + VCOL_SB + 32 * cg, d);
        merge(1, d);
    }
    __syncthreads();
    tc_fence_after();
    if (last) store_state(slot1 + (size_t)(warp >> 3) * state_stride, v, lane_addr + VCOL_S + 128 * (warp >> 3), 2 * ((warp >> 2) & 1), 2 * ((warp >> 2) & 1) + 2);
    settle_after_timeout(abortp);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(0, 512);
}

// ============================================================================================
// Segment summaries
// ============================================================================================
// U_g (both states, accumulated from zero) and A_g (products of the segment's gates) of a segment that has a successor.  Warps 0..15
// build K~ (state, channel half, eight rows each) and add up U in registers, warp 16 loads and issues.  The first segment of a sequence that continues
// from its slot also pushes that through its summary, and leaves a copy of it in the entry of the last segment.
constexpr int VS_NTHREADS = 17 * 32;
__global__ void __launch_bounds__(VS_NTHREADS, 1)
prefill_vec_summary_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g1,
                           const __grid_constant__ CUtensorMap map_g2, const VecParams vp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ VecShared sh;
    __shared__ float2 carries[2][2][D / 2];      // [parity][state]: product of the gates of all later chunks
    const PrefillParams& p = vp.p;
    uint8_t* tiles = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);      // (an offset, not a rounded address: the compiler still knows that it is shared memory)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const VecUnit u = vec_unit(vp, blockIdx.x, vp.nseg - 1);
    if (u.slot < 0 || u.slot >= p.num_slots || u.len <= 0 || u.c_end >= u.nchunks) return;      // (c_end < nchunks: whole chunks only)
    const int nc = u.c_end - u.c_begin, t0 = u.t_begin + u.c_begin * VC;
    float* unit = vp.ws + (size_t)(u.n * p.H + u.h) * vp.nseg * (VEC_STRIDE / 4);
    float* out = unit + (size_t)u.g * (VEC_STRIDE / 4);
    vec_setup(sh, tid, warp, 16);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    volatile int* abortp = &sh.abort_flag;
    const uint32_t sa = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int i = warp >> 3, hh = warp & 1, rows = 8 * ((warp >> 1) & 3);
    float2 after = make_float2(1.f, 1.f);
    // U of state warp / 8, key channels 64 ((warp / 4) % 2) .. + 63, one d_v lane per thread.  What a chunk adds to both states is a sum of
    // its own in the TMEM columns of its parity.
    const int q = warp & 3, ch0 = 64 * ((warp >> 2) & 1);
    float2 U[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) U[k] = make_float2(0.f, 0.f);
    auto merge = [&](int par) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            uint32_t r[16];
            tmem_ld16(((uint32_t)(32 * q) << 16) + 256 * par + 128 * i + ch0 + 16 * b, r);
            tc_wait_ld();
#pragma unroll
            for (int k = 0; k < 8; ++k) U[8 * b + k] = __fadd2_rn(U[8 * b + k], make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1])));
        }
        tc_fence_before();
    };
    // step it = chunk nc - 1 - it; buffers by the parity of it
    auto load = [&](int it) {      // by one thread
        const int par = it & 1, t = t0 + (nc - 1 - it) * VC;
        mbar_arrive_expect_tx(&sh.raw_full[par], 2 * V_TILE + V_GBYTES);
        tma_load_3d(tiles + OFF_SG + par * V_GBYTES, &map_g1, &sh.raw_full[par], 0, u.h, t);
        tma_load_3d(tiles + OFF_SG + par * V_GBYTES + V_GBYTES / 2, &map_g2, &sh.raw_full[par], 0, u.h, t);
        tma_load_3d(tiles + OFF_SK + par * V_TILE, &map_k, &sh.raw_full[par], 0, u.h, t);
        tma_load_4d(tiles + OFF_V + par * V_TILE, &map_v, &sh.raw_full[par], 0, t, 0, u.h);
    };
    if (warp == 16 && lane == 0) load(0);
#pragma unroll 1
    for (int it = 0; it < nc; ++it) {
        const int par = it & 1;
        if (warp == 16) {
            if (it + 1 < nc) {
                if (it >= 1) WAIT(&sh.done[par ^ 1], ((it - 1) >> 1) & 1);      // the MMAs of step it - 1 have read V
                if (lane == 0 && !*abortp) load(it + 1);
            }
        } else {
            if (it > 0) after = carries[par][i][32 * hh + lane];
            WAIT(&sh.raw_full[par], (it >> 1) & 1);
            if (it >= 2) {                                                      // ... and those of step it - 2 this K~
                WAIT(&sh.done[par], ((it >> 1) - 1) & 1);
                tc_fence_after();
                merge(par);
            }
            const float2 a = build_k<8, true>(tiles + OFF_SKT + (par * 6 + 3 * i) * V_TILE, tiles + OFF_SK + par * V_TILE + hh * 128 + lane * 4,
                                              tiles + OFF_SG + par * V_GBYTES + i * (V_GBYTES / 2) + hh * 256 + lane * 8, hh, rows, after, lane);
            if (rows == 0) carries[par ^ 1][i][32 * hh + lane] = a;
            fence_proxy_async_smem();
        }
        __syncthreads();
        if (warp == 16 && elect_one()) {
            constexpr uint32_t ID_U = idesc_bf16(128, 128, 1, 1);
            tc_fence_after();
            const uint32_t vd = smem_desc_lo(sa + OFF_V + par * V_TILE, V_HALF), kd = smem_desc_lo(sa + OFF_SKT + par * 6 * V_TILE, V_HALF);
            WAIT(&sh.raw_full[par], (it >> 1) & 1);
#pragma unroll
            for (int m = 5; m >= 0; --m) {      // (state, term), smallest terms first
                const uint32_t d = 256 * par + (m >= 3 ? 128 : 0), k = kd + (uint32_t)(m * (V_TILE >> 4));
                mma_ss_lo(d, vd, k, ID_U, m % 3 == 2 ? 0u : 1u);
                mma_ss_lo(d, vd + 128, k + 128, ID_U, 1u);
            }
            tc_commit(&sh.done[par]);
        }
        __syncwarp();
    }
    if (nc > 1) WAIT(&sh.done[nc & 1], ((nc - 2) >> 1) & 1);
    WAIT(&sh.done[(nc - 1) & 1], ((nc - 1) >> 1) & 1);
    tc_fence_after();
    if (warp < 16) {
        if (nc > 1) merge(nc & 1);
        merge((nc - 1) & 1);
        const float* A = reinterpret_cast<const float*>(carries[nc & 1][i]);
        const int v = 32 * q + lane;
        const bool from_slot = u.g == 0 && p.use_initial_state;
        const float* slot = p.state + (((size_t)u.slot * 2 + i) * p.H + u.h) * (size_t)(D * D) + v;
        float* copy = unit + (size_t)(vp.nseg - 1) * (VEC_STRIDE / 4) + (size_t)i * D * D + v;
        float* dst = out + (size_t)i * D * D + v;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int k0 = ch0 + 8 * b;
            float x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = from_slot ? slot[(size_t)(k0 + k) * D] : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (from_slot) copy[(size_t)(k0 + k) * D] = x[k];
                dst[(size_t)(k0 + k) * D] = fmaf(A[k0 + k], x[k], (k & 1) ? U[4 * b + (k >> 1)].y : U[4 * b + (k >> 1)].x);
            }
        }
        if (tid < 64) reinterpret_cast<float4*>(out + 2 * D * D)[tid] = reinterpret_cast<const float4*>(&carries[nc & 1][0][0])[tid];
    }
    settle_after_timeout(abortp);
    tc_fence_before();
    __syncthreads();
    if (warp == 16) tmem_dealloc(0, 512);
}
#undef WAIT

// [T_total, H, 128] of 2- or 4-byte elements, a chunk of one head per copy, rows as they are
bool make_row_map(CUtensorMap* m, const void* base, bool f32, int T_total, int H) {
    const cuuint64_t es = f32 ? 4 : 2;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)T_total};
    cuuint64_t strides[2] = {D * es, (cuuint64_t)H * D * es};
    cuuint32_t box[3] = {D, 1, VC};
    return encode_tile_map(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

}  // namespace

// bf16, d = 128, both gate tensors on 16-byte boundaries (their rows are copied in bulk)
bool prefill_vec_applies(const dsla_prefill_args* a) {
    return a->dtype == DSLA_BF16 && a->d_k == D && a->T_total > 0 && reinterpret_cast<uintptr_t>(a->g_hist) % 16 == 0 &&
           reinterpret_cast<uintptr_t>(a->g_rec) % 16 == 0;
}

// Segments per sequence: as many as keep every SM at one CTA, at least eight chunks each (below that the extra launch costs more than the
// shorter chains save), and no more than there is room for (these calls need none: without any a sequence is one segment).
static int plan_segments(const dsla_prefill_args* a, size_t room) {
    const long long units = (long long)a->N * a->H;
    const int max_chunks = (a->max_seqlen + VC - 1) / VC;
    int ns = units > 0 ? (int)(sm_count() / units) : 1;
    if (ns > 16) ns = 16;
    while (ns > 1 && ((max_chunks + ns - 1) / ns < 8 || (size_t)units * ns * VEC_STRIDE > room)) --ns;
    return ns < 1 ? 1 : ns;
}

size_t prefill_vec_workspace_bytes(const dsla_prefill_args* a) {
    const int ns = prefill_vec_applies(a) ? plan_segments(a, SIZE_MAX) : 1;
    return ns > 1 ? (size_t)a->N * a->H * ns * VEC_STRIDE : 0;
}

dsla_status launch_prefill_vec(const PrefillParams& p, const dsla_prefill_args* a, cudaStream_t s) {
    VecParams vp;
    vp.p = p;
    const long long units = (long long)p.N * p.H;
    const int max_chunks = (a->max_seqlen + VC - 1) / VC;
    const int ns = a->workspace && reinterpret_cast<uintptr_t>(a->workspace) % 16 == 0 ? plan_segments(a, a->workspace_bytes) : 1;
    vp.nseg = ns;
    vp.cps = ns > 1 ? (max_chunks + ns - 1) / ns : max_chunks;
    vp.ws = ns > 1 ? static_cast<float*>(a->workspace) : nullptr;
    if (units * ns > 0x7fffffffLL / 32) return DSLA_ERR_UNSUPPORTED;
    CUtensorMap mq, mk, mv, m1, m2;
    if (!make_row_map(&mq, p.q, false, a->T_total, p.H) || !make_row_map(&mk, p.k, false, a->T_total, p.H) || !make_tile_map(&mv, p.v, a->T_total, p.H, VC) ||
        !make_row_map(&m1, p.g_hist, true, a->T_total, p.H) || !make_row_map(&m2, p.g_rec, true, a->T_total, p.H))
        return DSLA_ERR_CUDA;
    if (ns > 1) {
        if (cudaFuncSetAttribute(prefill_vec_summary_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, V_SMEM_SUM) != cudaSuccess) return DSLA_ERR_CUDA;
        prefill_vec_summary_kernel<<<dim3((unsigned)(units * (ns - 1))), dim3(VS_NTHREADS), V_SMEM_SUM, s>>>(mk, mv, m1, m2, vp);
        count_launch();
    }
    if (cudaFuncSetAttribute(prefill_vec_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, V_SMEM) != cudaSuccess) return DSLA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * ns));
    cfg.blockDim = dim3(V_NTHREADS);
    cfg.dynamicSmemBytes = V_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ns > 1 ? 1 : 0;      // its prologue under the summaries' tail
    if (cudaLaunchKernelEx(&cfg, prefill_vec_kernel, mq, mk, mv, m1, m2, vp) != cudaSuccess) return DSLA_ERR_CUDA;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DSLA_OK : DSLA_ERR_CUDA;
}

}  // namespace dsla
