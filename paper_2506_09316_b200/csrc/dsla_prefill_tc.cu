// Tensor-core prefill of the dual-state linear attention layer for sm_100a (DSLA_IMPL_TENSOR): bf16 inputs,
// d = 128, fp32 states, both states of a (sequence, head) pair in one CTA.  Chunkwise form of the Sec. 4.1
// recurrence (chunks of 128 tokens, cumulative log-gates b^i_j inside the chunk, a^i = e^{b^i_last},
// w^i_s = e^{b^i_last - b^i_s}, r^i_j = weight_i e^{b^i_j}, weight = (gamma, 1 - gamma) * scale):
//     P      = Q K^T                                        tcgen05, fp32 in TMEM
//     P~     = P (.) [s<=j] (w1 e^{b1_j-b1_s} + w2 e^{b2_j-b2_s})     CUDA cores -> bf16 in smem
//     O^T    = S1^T (r1 (.) Q)^T + S2^T (r2 (.) Q)^T + V^T P~^T       tcgen05, states read from TMEM
//     S^i^T <- a^i S^i^T + (w^i (.) V)^T K                            rescale on CUDA cores, MMA accumulates
// States and outputs are computed transposed (d_v on the 128 TMEM lanes), so every MMA has M = 128.  The two fp32
// states live in TMEM for the whole segment; their bf16 copies in TMEM are the A operand of the readout, and once that
// has read them the weighted V^T, A operand of the update, takes their columns.  The scores and the outputs share the last
// 128 columns.  TMA lands Q, K and V ahead of their use in five 32 KB slots (128-byte swizzle).
//
// What bounds it: per chunk a loop  state pass (TMEM -> registers -> bf16 copy and rescaled state) -> readout -> update ->
// next pass,  and the 128 B/clk of shared memory that an M = N = 128 MMA with both operands there uses up alone.  Hence
// chunks of 128 tokens (half the passes of 64-token chunks), the update's A operand in TMEM, raw K and V as
// operands, and Q the only tile that is copied.
//
// A sequence may be split into segments along T so that few (sequence, head) pairs still fill the
// GPU (dsla_prefill_summary.cu computes the segment summaries); the main kernel, launched as the
// summary grid's programmatic dependent, folds the summaries of earlier segments into its initial
// state.  Packed batches are visited longest sequence first.  This file also holds the host side
// of both tensor-core variants (segment plan, workspace layout, launches).
#include "dsla_prefill_tc.cuh"

namespace dsla {

namespace {

// Warp roles of the main kernel: 0 = TMA producer, 1 = MMA issuer, 2..9 = tile warps (masked scores, scaled copies of Q),
// 10..17 = state warps (state rescale + bf16 copy, weighted V^T, outputs, initial/final state), 18, 19 = gate warps.
// A warp may touch only the 32 TMEM lanes of its quadrant (warp index mod 4).
constexpr int WARP_TMA = 0, WARP_MMA = 1, TILE_W0 = 2, STATE_W0 = 10, GATE_W0 = 18;
constexpr int NTHREADS = 20 * 32;
constexpr int CM = 128;                      // tokens per chunk of this kernel
// Shared memory, tiles of 128 tokens x 128 elements (32 KB, two halves of 64 elements, 128-byte swizzle).  Q of chunk c lands in
// slot c % 3 of a ring and V of chunk c in slot (c + 2) % 3: V of chunk c + 1 takes the place of Q of chunk c (read out by
// then), Q of chunk c + 3 that of V.  K alternates between two slots.  Q is scaled in place for state 1.
constexpr int TILE_BYTES = 32768, HALF_BYTES = 16384;
constexpr int OFF_K = 3 * TILE_BYTES;
constexpr int OFF_Q2 = OFF_K + 2 * TILE_BYTES;       // Q scaled for state 2
constexpr int OFF_PT = OFF_Q2 + TILE_BYTES;          // P~: columns 0..63 of 128 rows (16 KB), columns 64..127 of rows 64..127 (8 KB)
constexpr int SMEM_TILES = OFF_PT + HALF_BYTES + HALF_BYTES / 2;
constexpr int SMEM_DYN = SMEM_TILES + 1024;          // + alignment slack
// TMEM columns
constexpr uint32_t COL_S = 0;      // fp32 S1^T [0,128), S2^T [128,256)
constexpr uint32_t COL_SB = 256;   // per state 64 columns: the bf16 copy of S^T (readout), then the weighted V~^T (update)
constexpr uint32_t COL_R = 384;    // P (scores, tokens x tokens), then O^T (d_v x tokens): 128 columns

// Per-token terms of one chunk; the first index is the state.
struct alignas(16) GateSmem {
    float L[2][CM];                  // cumulative log2-gate from the chunk start, inclusive
    uint32_t rowf[2][CM];            // weight_i * (decay from the chunk start through the token), bf16 in both halves
    __nv_bfloat16 E[2][CM];          // decay from the token to the end of its block of 32 tokens
    __nv_bfloat16 w[2][CM];          // decay from the token to the end of the chunk; 0 past the end of the sequence
    float a[2];                      // product of the chunk's gates
};

struct alignas(16) Shared {
    uint64_t kq_full[2], v_full[2], p_full, prep_ready, sb_ready[2], ro_done, vt_ready[2], o_full, o_free, o_staged, u_full[2], g_ready[2], g_free[2], init_done;
    uint32_t tmem_base;
    int abort_flag;
    GateSmem gs[2];
};

// Four MMAs whose operands advance by a constant.
template <uint32_t ASTEP, uint32_t BSTEP>
__device__ __forceinline__ void issue4_ss(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) mma_ss_lo(d, a + k * ASTEP, b + k * BSTEP, idesc, k ? 1u : acc);
}
template <uint32_t BSTEP>
__device__ __forceinline__ void issue4_ts(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) mma_ts_lo(d, a + 8 * k, b + k * BSTEP, idesc, k ? 1u : acc);
}

// ============================================================================================
// Main kernel
// ============================================================================================
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, const TcParams tp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const PrefillParams& p = tp.p;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Blocks are handed out in index order: the last segments first.  When this grid starts as a programmatic dependent
    // of the summary grid, the blocks that fit next to it are then the ones with the longest fold of summaries ahead of
    // them, and their prologue (TMEM, first tiles, first scores) is hidden behind the summary grid's tail.
    const int units = p.N * p.H;
    const int g = tp.nseg - 1 - (int)(blockIdx.x / units);
    const int h = (blockIdx.x % units) % p.H;
    const int rank = (blockIdx.x % units) / p.H;
    const int n = tp.order ? tp.order[rank] : rank;
    const SeqInfo sq = seq_info(p, n, g, tp);
    if (sq.slot < 0 || sq.slot >= p.num_slots) return;
    if (tid == 0 && g == 0 && sq.nchunks > seg_begin(tp.nseg, tp.nseg, tp.cps, tp.skew8)) atomicExch(p.status, (int)DSLA_ERR_INVALID_ARG);
    float* slot1 = p.state + (((size_t)sq.slot * p.n_total + p.state_first) * p.H + h) * (size_t)(D * D);
    const size_t state_stride = (size_t)p.H * D * D;
    // where the initial state is read: the slot, or the snapshot taken before this grid (split sequences)
    const float* init1 = tp.init ? tp.init + (size_t)(n * p.H + h) * 2 * (size_t)(D * D) : slot1;
    const size_t init_stride = tp.init ? (size_t)(D * D) : state_stride;
    if (sq.len <= 0) {  // empty sequence: a fresh start leaves zero states, a resume leaves the slot alone
        if (g == 0 && !p.use_initial_state)
            for (int i = tid; i < (p.single ? 1 : 2) * D * D; i += NTHREADS) slot1[(size_t)(i / (D * D)) * state_stride + i % (D * D)] = 0.f;
        return;
    }
    if (sq.c_begin >= sq.c_end) return;
    const int nc = sq.c_end - sq.c_begin;
    const int t0 = sq.t_begin + sq.c_begin * CM;  // first token of this segment
    const int tok0 = sq.c_begin * CM;             // its index inside the sequence
    const bool last = g == sq.last_seg;           // the final state is kept; other segments skip the last chunk's update
    const bool init_shared = (g > 0 && tp.ws) || p.use_initial_state;   // the initial state is loaded, not just zero
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // a dependent launch behind this grid (the decode step) may be scheduled early

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.kq_full[i], 1); mbar_init(&sh.v_full[i], 1);
            mbar_init(&sh.sb_ready[i], 4); mbar_init(&sh.vt_ready[i], 4); mbar_init(&sh.u_full[i], 1);
            mbar_init(&sh.g_ready[i], 2); mbar_init(&sh.g_free[i], 16);
        }
        mbar_init(&sh.p_full, 1); mbar_init(&sh.prep_ready, 8); mbar_init(&sh.ro_done, 1);
        mbar_init(&sh.o_full, 1); mbar_init(&sh.o_free, 8); mbar_init(&sh.o_staged, 8);
        mbar_init(&sh.init_done, 8);     // the tile warps' share of the initial state
        sh.abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == WARP_MMA) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = 0;      // all 512 columns are allocated: the base is column 0
    volatile int* abortp = &sh.abort_flag;
#define WAIT(bar, ph) mbar_wait(bar, (uint32_t)(ph), abortp, p.status)

    if (warp == WARP_TMA) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            prefetch_tensormap(&map_q); prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
            auto load_kq = [&](int c, int q3) {
                mbar_arrive_expect_tx(&sh.kq_full[c & 1], 2 * TILE_BYTES);
                tma_load_4d(tiles + q3 * TILE_BYTES, &map_q, &sh.kq_full[c & 1], 0, t0 + c * CM, 0, h);
                tma_load_4d(tiles + OFF_K + (c & 1) * TILE_BYTES, &map_k, &sh.kq_full[c & 1], 0, t0 + c * CM, 0, h);
            };
            auto load_v = [&](int c, int v3) {
                mbar_arrive_expect_tx(&sh.v_full[c & 1], TILE_BYTES);
                tma_load_4d(tiles + v3 * TILE_BYTES, &map_v, &sh.v_full[c & 1], 0, t0 + c * CM, 0, h);
            };
            load_kq(0, 0);
            load_v(0, 2);
            if (nc > 1) load_kq(1, 1);
            const int nfull = (sq.len - tok0) / CM;         // whole chunks leave through shared memory and a tile store
            int c3 = 0;
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                const int v3 = c3 == 0 ? 2 : c3 - 1;
                if (c + 1 < nc) {
                    WAIT(&sh.ro_done, c & 1);              // Q of chunk c has been read: its slot takes V of chunk c + 1
                    load_v(c + 1, c3);
                    // pull what the next loads will need into L2 (a tile's slot frees only about one load latency before it is used)
                    if (c + 2 < nc) tma_prefetch_4d(&map_v, 0, t0 + (c + 2) * CM, 0, h);
                }
                if (c < nfull) {
                    WAIT(&sh.o_staged, c & 1);             // the outputs of chunk c are in the slot of its V
                    tma_store_4d(&map_o, tiles + v3 * TILE_BYTES, 0, t0 + c * CM, 0, h);
                    bulk_commit();
                    bulk_wait_read();
                }
                if (c + 2 < nc) {
                    WAIT(&sh.u_full[1], c & 1);            // K of chunk c has been read
                    load_kq(c + 2, v3);
                    if (c + 3 < nc) {
                        tma_prefetch_4d(&map_q, 0, t0 + (c + 3) * CM, 0, h);
                        tma_prefetch_4d(&map_k, 0, t0 + (c + 3) * CM, 0, h);
                    }
                }
                c3 = c3 == 2 ? 0 : c3 + 1;
            }
            bulk_wait_all();
        }
    } else if (warp == WARP_MMA) {
        // ------------------------------------------------------------------ MMA issuer
        // Per chunk:  O^T = S1^T Q~1^T + S2^T Q~2^T,  O^T += V^T P~^T,  S1^T += V~1^T K,  P of the next chunk,  S2^T += V~2^T K.
        // The readout of a state starts as soon as its bf16 copy is there; V~ is stored under the P~ part, O^T is read out under
        // the first update, the next scores are masked under the second.
        if (elect_one()) {
            const uint32_t sa = (smem_u32(smem_raw) + 1023u) & ~1023u;
            constexpr uint32_t ID_KK = idesc_bf16(128, 128, 0, 0);     // both operands K-major (scores; readout with A in TMEM)
            constexpr uint32_t ID_V128 = idesc_bf16(128, 128, 1, 0), ID_V64 = idesc_bf16(128, 64, 1, 0);
            constexpr uint32_t ID_U = idesc_bf16(128, 128, 0, 1);      // A in TMEM, B = raw K, MN-major
            constexpr uint32_t T_STEP = TILE_BYTES >> 4, H_STEP = HALF_BYTES >> 4;
            const uint32_t dq0 = smem_desc_lo(sa, 16), dq2 = smem_desc_lo(sa + OFF_Q2, 16), dkk = smem_desc_lo(sa + OFF_K, 16);
            const uint32_t dkn = smem_desc_lo(sa + OFF_K, HALF_BYTES), dv0 = smem_desc_lo(sa, HALF_BYTES), dp0 = smem_desc_lo(sa + OFF_PT, 16);
            auto scores = [&](int c, int q3) {
                WAIT(&sh.kq_full[c & 1], (c >> 1) & 1);
                tc_fence_after();
                const uint32_t a = dq0 + (uint32_t)q3 * T_STEP, b = dkk + (uint32_t)(c & 1) * T_STEP;
                issue4_ss<2, 2>(COL_R, a, b, ID_KK, 0u);
                issue4_ss<2, 2>(COL_R, a + H_STEP, b + H_STEP, ID_KK, 1u);
                tc_commit(&sh.p_full);
            };
            scores(0, 0);
            int c3 = 0;
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                const int v3 = c3 == 0 ? 2 : c3 - 1, n3 = c3 == 2 ? 0 : c3 + 1;
                WAIT(&sh.v_full[c & 1], (c >> 1) & 1);
                WAIT(&sh.prep_ready, c & 1);               // P read out of TMEM, P~, Q~1, Q~2 in place
#pragma unroll 1
                for (int i = 0; i < 2; ++i) {
                    WAIT(&sh.sb_ready[i], c & 1);
                    tc_fence_after();
                    const uint32_t a = COL_SB + 64 * i, b = i == 0 ? dq0 + (uint32_t)c3 * T_STEP : dq2;
                    issue4_ts<2>(COL_R, a, b, ID_KK, i ? 1u : 0u);
                    issue4_ts<2>(COL_R, a + 32, b + H_STEP, ID_KK, 1u);
                }
                tc_commit(&sh.ro_done);
                const uint32_t v = dv0 + (uint32_t)v3 * T_STEP;
                issue4_ss<128, 2>(COL_R, v, dp0, ID_V128, 1u);
                issue4_ss<128, 2>(COL_R + 64, v + 512, dp0 + H_STEP, ID_V64, 1u);     // keys 64..127 reach only the outputs of tokens 64..127
                tc_commit(&sh.o_full);
                const bool update = last || c + 1 < nc;
                const uint32_t bk = dkn + (uint32_t)(c & 1) * T_STEP;
#pragma unroll 1
                for (int i = 0; i < 2; ++i) {
                    if (update) {
                        WAIT(&sh.vt_ready[i], c & 1);
                        tc_fence_after();
                        issue4_ts<128>(COL_S + 128 * i, COL_SB + 64 * i, bk, ID_U, 1u);
                        issue4_ts<128>(COL_S + 128 * i, COL_SB + 64 * i + 32, bk + 512, ID_U, 1u);
                        tc_commit(&sh.u_full[i]);
                    }
                    if (i == 0 && c + 1 < nc) {
                        WAIT(&sh.o_free, c & 1);           // O^T is in registers: its columns take the next scores
                        scores(c + 1, n3);
                    }
                }
                c3 = n3;
            }
        }
    } else if (warp < STATE_W0) {
        // ------------------------------------------------------------------ tile warps 2..9
        const int tt = tid - TILE_W0 * 32;                // 0..255
        const int q = warp & 3;                           // TMEM lane quadrant: rows (tokens) 32 q .. 32 q + 31
        const int half = (warp - TILE_W0) >> 2;           // column half: keys 64 half .. 64 half + 63
        const uint32_t lane_addr = tb + ((uint32_t)(32 * q) << 16);
        const int j = 32 * q + lane;
        const float W1 = (p.weights ? p.weights[(size_t)h * p.n_total + p.state_first] : p.gamma[h]) * p.scale;
        const float W2 = p.single ? 0.f : (p.weights ? p.weights[(size_t)h * p.n_total + p.state_first + 1] : 1.f - p.gamma[h]) * p.scale;

        if (init_shared) {
            // d_k rows 64..127 of the initial state of state `half` for this lane quadrant, while the first tiles are in flight
            WAIT(&sh.g_ready[0], 0);
            if (g > 0 && tp.ws) asm volatile("griddepcontrol.wait;" ::: "memory");
            init_state_pass(init1 + (size_t)half * init_stride, p.use_initial_state && !(p.single && half == 1),
                            tp.ws ? tp.ws + ((size_t)(n * p.H + h) * tp.nseg) * (SUMMARY_STRIDE / 4) : nullptr, g, half, j, sh.gs[0].a[half],
                            lane_addr + COL_S + 128 * half, lane_addr + COL_SB + 64 * half, 2, 4);
            tc_wait_st();
            tc_fence_before();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.init_done);
        // The ten 32 x 32 blocks of the lower triangle: a quadrant's q + 1 blocks are split between its two warps (the second one
        // has the diagonal block).  The two blocks above the diagonal that the MMAs read are zeroed once.
        const int blk0 = half == 0 ? 0 : (q == 1 ? 1 : 2), nblk = q == 0 ? 1 - half : (q == 3 || (q == 2 && half == 0)) ? 2 : 1;
        if (half == 0 && (q == 0 || q == 2))
            for (int m4 = 0; m4 < 4; ++m4)
                *reinterpret_cast<uint4*>(tiles + OFF_PT + (q == 2 ? HALF_BYTES - 64 * 128 : 0) + sw128_offset(j, 32 + 8 * m4)) = make_uint4(0u, 0u, 0u, 0u);
        int c3 = 0;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            const GateSmem& gs = sh.gs[s];
            uint8_t* qs = tiles + c3 * TILE_BYTES;
            WAIT(&sh.g_ready[s], (c >> 1) & 1);
            WAIT(&sh.kq_full[s], (c >> 1) & 1);           // the TMA writes of Q are visible to this thread
            // ---- scaled copies of Q, eight 16-byte pieces per thread.  The copy for state 2 is written as soon as the readout of the
            // previous chunk is done with its buffer, the one for state 1 waits in registers until the scores have read the raw Q.
            if (c > 0) WAIT(&sh.ro_done, (c - 1) & 1);
            uint4 q1[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) q1[m] = reinterpret_cast<const uint4*>(qs)[tt + 256 * m];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int idx = tt + 256 * m, row = (idx >> 3) & 127;
                reinterpret_cast<uint4*>(tiles + OFF_Q2)[idx] = scale8(q1[m], gs.rowf[1][row]);
                q1[m] = scale8(q1[m], gs.rowf[0][row]);
            }
            mbar_wait_inline(&sh.p_full, c & 1, abortp, p.status);
            tc_fence_after();
#pragma unroll
            for (int m = 0; m < 8; ++m) reinterpret_cast<uint4*>(qs)[tt + 256 * m] = q1[m];
            // ---- P~ = P (.) M; the decays of a block left of the diagonal factor through the block's last token
            const float L1 = gs.L[0][j], L2 = gs.L[1][j];
#pragma unroll 1
            for (int blk = blk0; blk < blk0 + nblk; ++blk) {
                uint8_t* at = tiles + OFF_PT + (blk >= 2 ? HALF_BYTES - 64 * 128 : 0);
                uint32_t r[32], pk[16];
                tmem_ld32(lane_addr + COL_R + 32 * blk, r);
                if (blk < q) {
                    const float R1 = W1 * ex2(L1 - gs.L[0][32 * blk + 31]), R2 = W2 * ex2(L2 - gs.L[1][32 * blk + 31]);
                    const float2 RR1 = make_float2(R1, R1), RR2 = make_float2(R2, R2);
                    uint4 E1[4], E2[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        E1[e] = *reinterpret_cast<const uint4*>(&gs.E[0][32 * blk + 8 * e]);
                        E2[e] = *reinterpret_cast<const uint4*>(&gs.E[1][32 * blk + 8 * e]);
                    }
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float2 m = __ffma2_rn(RR2, unpack_bf16(word_of(E2[e >> 2], e & 3)), __fmul2_rn(RR1, unpack_bf16(word_of(E1[e >> 2], e & 3))));
                        const float2 y = __fmul2_rn(m, make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])));
                        pk[e] = pack_bf16(y.x, y.y);
                    }
                } else {
                    tc_wait_ld();
#pragma unroll
                    for (int e4 = 0; e4 < 8; ++e4) {
                        const float4 K1 = *reinterpret_cast<const float4*>(&gs.L[0][32 * blk + 4 * e4]), K2 = *reinterpret_cast<const float4*>(&gs.L[1][32 * blk + 4 * e4]);
                        const float m0 = fmaf(W2, ex2(L2 - K2.x), W1 * ex2(L1 - K1.x)), m1 = fmaf(W2, ex2(L2 - K2.y), W1 * ex2(L1 - K1.y));
                        const float m2 = fmaf(W2, ex2(L2 - K2.z), W1 * ex2(L1 - K1.z)), m3 = fmaf(W2, ex2(L2 - K2.w), W1 * ex2(L1 - K1.w));
                        const int e = 4 * e4;      // keys later than the row's token carry nothing
                        pk[2 * e4] = pack_bf16(e <= lane ? __uint_as_float(r[e]) * m0 : 0.f, e + 1 <= lane ? __uint_as_float(r[e + 1]) * m1 : 0.f);
                        pk[2 * e4 + 1] = pack_bf16(e + 2 <= lane ? __uint_as_float(r[e + 2]) * m2 : 0.f, e + 3 <= lane ? __uint_as_float(r[e + 3]) * m3 : 0.f);
                    }
                }
#pragma unroll
                for (int m4 = 0; m4 < 4; ++m4)
                    *reinterpret_cast<uint4*>(at + sw128_offset(j, 32 * (blk & 1) + 8 * m4)) = make_uint4(pk[4 * m4], pk[4 * m4 + 1], pk[4 * m4 + 2], pk[4 * m4 + 3]);
            }
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) { mbar_arrive(&sh.prep_ready); mbar_arrive(&sh.g_free[s]); }
            c3 = c3 == 2 ? 0 : c3 + 1;
        }
    } else if (warp >= GATE_W0) {
        // ------------------------------------------------------------------ gate warps: 18 = state 1, 19 = state 2
        // Everything the chunk needs from the gates comes from the cumulative log-gates
        //     L_j = sum_{t <= j} log2 g_t        (inclusive, from the chunk start; a zero gate counts as -130, so any product
        //                                         that contains one flushes to an exact zero)
        // through independent exponentials.  Lane l holds tokens 4 l .. 4 l + 3.  The chunk decay that carries the state
        // is the plain product of the gates.
        const int i = warp - GATE_W0;
        const float* gsrc = i == 0 ? p.g_hist : p.g_rec;
        const float Wi = (p.weights ? (i == 1 && p.single ? 0.f : p.weights[(size_t)h * p.n_total + p.state_first + i])
                                    : (i == 0 ? p.gamma[h] : 1.f - p.gamma[h])) * p.scale;
        float nx[4];
        auto fetch = [&](int c) {      // raw values: nothing may consume them here, or the warp would sit out the load latency in every chunk
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = c * CM + 4 * lane + e;
                nx[e] = load_gate(gsrc, t0 + j, p.H, h, c < nc && tok0 + j < sq.len);
            }
        };
        fetch(0);
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            GateSmem& gs = sh.gs[s];
            float L[4], pr = 1.f, run = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float x = fmaxf(nx[e], 0.f);
                pr *= x;
                run += lg2_gate(x);
                L[e] = run;
            }
            fetch(c + 1);
            const float incl = warp_prefix_sum(run, lane);
            float excl = __shfl_up_sync(0xffffffffu, incl, 1);
            if (lane == 0) excl = 0.f;
            const float block_end = __shfl_sync(0xffffffffu, incl, lane | 7), end = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) pr *= __shfl_xor_sync(0xffffffffu, pr, off);
            const int valid = min(CM, sq.len - tok0 - c * CM);
            if (c >= 2) WAIT(&sh.g_free[s], ((c >> 1) - 1) & 1);
            float f[4], E[4], w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                L[e] = e == 3 ? incl : excl + L[e];      // (block_end is some lane's incl: keep the two consistent)
                f[e] = Wi * ex2(L[e]);
                E[e] = ex2(block_end - L[e]);
                w[e] = 4 * lane + e < valid ? ex2(end - L[e]) : 0.f;
            }
            *reinterpret_cast<float4*>(&gs.L[i][4 * lane]) = make_float4(L[0], L[1], L[2], L[3]);
            *reinterpret_cast<uint4*>(&gs.rowf[i][4 * lane]) = make_uint4(dup_bf16(f[0]), dup_bf16(f[1]), dup_bf16(f[2]), dup_bf16(f[3]));
            *reinterpret_cast<uint2*>(&gs.E[i][4 * lane]) = make_uint2(pack_bf16(E[0], E[1]), pack_bf16(E[2], E[3]));
            *reinterpret_cast<uint2*>(&gs.w[i][4 * lane]) = make_uint2(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]));
            if (lane == 0) gs.a[i] = pr;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.g_ready[s]);
        }
    } else {
        // ------------------------------------------------------------------ state warps 10..17
        const int q = warp & 3, hi = (warp - STATE_W0) >> 2;   // TMEM lane quadrant, state index
        const uint32_t lane_addr = tb + ((uint32_t)(32 * q) << 16);
        const uint32_t s_addr = lane_addr + COL_S + 128 * hi;
        const uint32_t sb_addr = lane_addr + COL_SB + 64 * hi;
        const int v = 32 * q + lane;
        __nv_bfloat16* og = reinterpret_cast<__nv_bfloat16*>(p.o);
        // ldmatrix: this thread addresses row mr of matrix mk; matrices (tokens 0..7 | 8..15) x (d_v 0..7 | 8..15)
        const int mk = lane >> 3, mr = lane & 7;
        int v3 = 2;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            const GateSmem& gs = sh.gs[s];
            WAIT(&sh.g_ready[s], (c >> 1) & 1);
            const float a = gs.a[hi];
            if (c == 0) {
                // With programmatic dependent launch this grid may start while the summary grid is still running;
                // everything up to here (and all of chunk 0's operand work in the other warps) is independent of it.
                if (g > 0 && tp.ws) asm volatile("griddepcontrol.wait;" ::: "memory");
                init_state_pass(init1 + (size_t)hi * init_stride, p.use_initial_state && !(p.single && hi == 1),
                                tp.ws ? tp.ws + ((size_t)(n * p.H + h) * tp.nseg) * (SUMMARY_STRIDE / 4) : nullptr, g, hi, v, a, s_addr, sb_addr,
                                0, init_shared ? 2 : 4);
                WAIT(&sh.init_done, 0);     // the other half (or nothing) from the tile warps
            } else {
                WAIT(&sh.u_full[hi], (c - 1) & 1);
                tc_fence_after();
                // ---- one pass over the state (TMEM -> registers once): the bf16 copy of S_{c-1} that the readout of chunk c
                // multiplies, and a_c S_{c-1} in place, onto which the update MMA of chunk c accumulates
                const float2 a2 = make_float2(a, a);
#pragma unroll 1
                for (int b = 0; b < 4; ++b) {
                    uint32_t r[32], pk[16];
                    tmem_ld32(s_addr + 32 * b, r);
                    tc_wait_ld();
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        pk[k] = pack_bf16(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
                        const float2 y = __fmul2_rn(make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1])), a2);
                        r[2 * k] = __float_as_uint(y.x); r[2 * k + 1] = __float_as_uint(y.y);
                    }
                    tmem_st16(sb_addr + 16 * b, pk);
                    tmem_st32(s_addr + 32 * b, r);
                }
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.sb_ready[hi]);
            // ---- V~^T[v][s] = w_s V[s][v] of this state and quadrant: built in registers under the readout, stored over the bf16 copy as
            // soon as that has been read; the P~ part of the outputs, which follows, leaves shared memory no room for other reads (ldmatrix.trans hands out the element pairs a 16x128b TMEM store takes)
            WAIT(&sh.v_full[s], (c >> 1) & 1);
            WAIT(&sh.prep_ready, c & 1);      // (under the readout: before it the tile warps need the issue slots and shared memory)
            {
                const uint32_t vrow = smem_u32(tiles + v3 * TILE_BYTES) + (uint32_t)((8 * (mk >> 1) + mr) * 128);
                const uint32_t wp = smem_u32(&gs.w[hi][2 * (lane & 3)]);
                uint32_t vt[2][32];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {       // the two 16-lane halves of this warp's TMEM quadrant
                    const int d = 32 * q + 16 * hh + 8 * (mk & 1);            // first d_v column of the matrix this thread addresses
                    const uint32_t row0 = vrow + (uint32_t)(d >> 6) * HALF_BYTES + (((uint32_t)((d & 63) >> 3) ^ (uint32_t)mr) << 4);
#pragma unroll
                    for (int t16 = 0; t16 < 8; ++t16)
                        ldmatrix_x4_trans(row0 + (uint32_t)(t16 * 16 * 128), vt[hh][4 * t16], vt[hh][4 * t16 + 1], vt[hh][4 * t16 + 2], vt[hh][4 * t16 + 3]);
                }
#pragma unroll
                for (int t16 = 0; t16 < 8; ++t16) {
                    const uint32_t w0 = ld_shared_u32(wp + 32 * t16), w1 = ld_shared_u32(wp + 32 * t16 + 16);
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        uint32_t* r = vt[hh] + 4 * t16;
                        r[0] = hmul2_u32(r[0], w0); r[1] = hmul2_u32(r[1], w0);
                        r[2] = hmul2_u32(r[2], w1); r[3] = hmul2_u32(r[3], w1);
                    }
                }
                mbar_wait_inline(&sh.ro_done, c & 1, abortp, p.status);
                tc_fence_after();
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    tmem_st_16x128b_x8(sb_addr + ((uint32_t)(16 * hh) << 16), vt[hh]);
                    tmem_st_16x128b_x8(sb_addr + ((uint32_t)(16 * hh) << 16) + 32, vt[hh] + 16);
                }
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { mbar_arrive(&sh.vt_ready[hi]); mbar_arrive(&sh.g_free[s]); }
            // ---- outputs, tokens 64 hi .. 64 hi + 63 of this warp's lane quadrant.  Whole chunks: token-major bf16 tile in the slot of
            // this chunk's V (stmatrix transposes the fragments of a 16x256b load), which the producer warp stores with one TMA
            // copy; 64 stores of one token's 64 bytes each held the warps up for 2400 cycles.
            WAIT(&sh.o_full, c & 1);
            const int valid = min(CM, sq.len - tok0 - c * CM);
            tc_fence_after();
            if (valid == CM) {
                uint32_t o4[4][16];
#pragma unroll
                for (int b = 0; b < 4; ++b) tmem_ld_16x256b_x4(lane_addr + ((uint32_t)(16 * (b & 1)) << 16) + COL_R + 64 * hi + 32 * (b >> 1), o4[b]);
                tc_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.o_free);
                mbar_wait_inline(&sh.vt_ready[0], c & 1, abortp, p.status);    // every state warp is done with V
                mbar_wait_inline(&sh.vt_ready[1], c & 1, abortp, p.status);
                const uint32_t tok = (uint32_t)(64 * hi + (lane & 7)), piece = (uint32_t)(4 * (q & 1) + (lane >> 3));
                const uint32_t at = smem_u32(tiles + v3 * TILE_BYTES + (q >> 1) * HALF_BYTES) + tok * 128u + ((piece ^ (tok & 7)) << 4);
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const uint32_t *x = o4[2 * (b >> 2)] + 4 * (b & 3), *y = o4[2 * (b >> 2) + 1] + 4 * (b & 3);
                    stmatrix_x4_trans(at + (uint32_t)(8 * b * 128), pack_bf16(__uint_as_float(x[0]), __uint_as_float(x[1])), pack_bf16(__uint_as_float(x[2]), __uint_as_float(x[3])),
                                      pack_bf16(__uint_as_float(y[0]), __uint_as_float(y[1])), pack_bf16(__uint_as_float(y[2]), __uint_as_float(y[3])));
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.o_staged);
            } else {      // the sequence's ragged last chunk: each thread owns one d_v lane of O^T
                __nv_bfloat16* dst = og + ((size_t)(t0 + c * CM + 64 * hi) * p.H + h) * D + v;
                const size_t row = (size_t)p.H * D;
#pragma unroll 1
                for (int b = 64 * hi; b < 64 * hi + 64; b += 16) {
                    uint32_t r[16];
                    tmem_ld16(lane_addr + COL_R + b, r);
                    tc_wait_ld();
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        if (b + jj < valid) *dst = __float2bfloat16_rn(__uint_as_float(r[jj]));
                        dst += row;
                    }
                }
            }
            v3 = v3 == 2 ? 0 : v3 + 1;
        }
        if (last) {
            WAIT(&sh.u_full[hi], (nc - 1) & 1);
            tc_fence_after();
            if (!(p.single && hi == 1)) store_state(slot1 + (size_t)hi * state_stride, v, s_addr, 0, 4);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) tmem_dealloc(tb, 512);
#undef WAIT
}

}  // namespace

namespace {

bool wants_order(const dsla_prefill_args* a) { return a->cu_seqlens != nullptr && a->N > 1 && a->N <= ORDER_MAX_N; }

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
        (void)cudaGetLastError();
        return 148;      // a B200, when there is no device to ask (sizing a workspace on a build machine)
    }
    return sms;
}

// Segments per sequence: enough work items (CTAs, or clusters of the pair variant) to cover the SMs when there
// are few (sequence, head) pairs, never shorter than 256 tokens per segment.
void plan(const dsla_prefill_args* a, bool pair, int* nseg, int* cps, int* skew8) {
    const int chunk = pair ? C : CM, min_cps = pair ? 4 : 2;
    const int max_chunks = (a->max_seqlen + chunk - 1) / chunk;
    const long long units = (long long)a->N * a->H;
    const int room = pair ? pair_resident_clusters() : sm_count();     // work items resident at once
    int ns = 1;
    if (units > 0 && units < room) ns = (int)(room / units);
    if (ns > 16) ns = 16;
    while (ns > 1 && (max_chunks + ns - 1) / ns < min_cps) --ns;
    if (max_chunks <= 0) ns = 1;
    *nseg = ns;
    *cps = max_chunks > 0 ? (max_chunks + ns - 1) / ns : 1;
    // later segments fold more summaries into their initial state before they start (about 50 tokens' time each):
    // make consecutive segments about that much shorter, as far as the shortest keeps at least 192 tokens
    int sk = ns > 1 ? (8 * (*cps - (pair ? 3 : 2))) / (ns - 1) : 0;
    const int most = pair ? 3 : 2;
    *skew8 = sk < 0 ? 0 : (sk > most ? most : sk);
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
size_t summaries_bytes(const dsla_prefill_args* a, int nseg) { return nseg > 1 ? (size_t)a->N * a->H * nseg * SUMMARY_STRIDE : 0; }
size_t order_bytes(const dsla_prefill_args* a) { return wants_order(a) ? up256((size_t)a->N * sizeof(int)) : 0; }
// room for the snapshot of the initial states of split sequences (used when use_initial_state is set)
size_t snapshot_bytes(const dsla_prefill_args* a, int nseg) { return nseg > 1 ? (size_t)a->N * a->H * 2 * D * D * sizeof(float) : 0; }

dsla_status launch_main(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mo, const TcParams& tp,
                        bool dependent, cudaStream_t s) {
    if (cudaFuncSetAttribute(prefill_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_DYN) != cudaSuccess) return DSLA_ERR_CUDA;
    const long long units = (long long)tp.p.N * tp.p.H;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * tp.nseg));
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = SMEM_DYN;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, prefill_tc_kernel, mq, mk, mv, mo, tp) != cudaSuccess) return DSLA_ERR_CUDA;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DSLA_OK : DSLA_ERR_CUDA;
}

}  // namespace

bool prefill_tc_available() { return true; }

size_t prefill_tc_workspace_bytes(const dsla_prefill_args* a, bool pair) {
    int nseg, cps, skew8;
    plan(a, pair, &nseg, &cps, &skew8);
    return summaries_bytes(a, nseg) + order_bytes(a) + snapshot_bytes(a, nseg);     // each a multiple of 256
}

dsla_status launch_prefill_tc(const PrefillParams& p, const dsla_prefill_args* a, bool pair, cudaStream_t s) {
    if (p.N == 0 || a->T_total == 0) {
        // only empty sequences: the CUDA-core kernel handles the slot bookkeeping
        return launch_prefill_simt(p, D, C, DSLA_BF16, s);
    }
    TcParams tp;
    tp.p = p;
    tp.chunk = pair ? C : CM;
    plan(a, pair, &tp.nseg, &tp.cps, &tp.skew8);
    char* wsp = static_cast<char*>(a->workspace);
    tp.ws = tp.nseg > 1 ? reinterpret_cast<float*>(wsp) : nullptr;
    tp.order = nullptr;
    tp.init = nullptr;
    if (wants_order(a)) {
        int* order = reinterpret_cast<int*>(wsp + summaries_bytes(a, tp.nseg));
        launch_seq_order(p.cu_seqlens, p.N, order, s);
        tp.order = order;
    }
    if (tp.nseg > 1 && p.use_initial_state) {
        // The CTA of a sequence's last segment overwrites the slot with the final state; CTAs of earlier segments read the
        // slot as their initial state and nothing orders the two inside the grid: they read a copy taken beforehand.
        float* snap = reinterpret_cast<float*>(wsp + summaries_bytes(a, tp.nseg) + order_bytes(a));
        launch_state_snapshot(p, snap, s);
        tp.init = snap;
    }
    CUtensorMap mq, mk, mv, mo;
    if (!make_tile_map(&mq, p.q, a->T_total, p.H, tp.chunk) || !make_tile_map(&mk, p.k, a->T_total, p.H, tp.chunk) ||
        !make_tile_map(&mv, p.v, a->T_total, p.H, tp.chunk) || !make_tile_map(&mo, p.o, a->T_total, p.H, tp.chunk))
        return DSLA_ERR_CUDA;
    const long long units = (long long)p.N * p.H;
    if (2 * units * tp.nseg > 0x7fffffffLL) return DSLA_ERR_UNSUPPORTED;
    if (tp.nseg > 1) {
        CUtensorMap sk, sv;
        if (!make_tile_map(&sk, p.k, a->T_total, p.H, C) || !make_tile_map(&sv, p.v, a->T_total, p.H, C)) return DSLA_ERR_CUDA;
        const dsla_status rc = launch_summary(sk, sv, tp, s);
        if (rc != DSLA_OK) return rc;
    }
    return pair ? launch_main_pair(mq, mk, mv, tp, tp.nseg > 1, s) : launch_main(mq, mk, mv, mo, tp, tp.nseg > 1, s);
}

}  // namespace dsla
