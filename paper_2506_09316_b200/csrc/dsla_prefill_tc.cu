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
// A sequence may be split into segments along T so that few (sequence, head) pairs still fill the GPU.  The segments of a
// sequence are the CTAs of a thread-block cluster: each first accumulates the state its own tokens leave behind, from zero (its
// summary U, with the product A of its gates), then the initial states travel down the cluster, S <- A S + U, in
// pieces, and each segment runs its chunks.  (As a kernel of its own the summaries took 21 of 68 us at T = 4096, 32 heads: launch,
// fill and drain of a second pipeline.  Stores into another CTA's shared memory ran at 26 bytes a cycle, loads from it at 12:
// hence a chain that only stores.  Its last of four CTAs has its initial state 13 to 15 k cycles after the first began to send, of which the
// first hop takes 9 to 11 k and a further one 2 k; a fold in which every CTA loads its share of all summaries and stores it back took 16 k.)
// Packed batches are visited longest sequence first.  This file also holds the host side of both tensor-core variants (segment
// plan, workspace layout, launches).
#include <atomic>
#include <cstddef>

#include "dsla_prefill_tc.cuh"

namespace dsla {

namespace {

// Warp roles of the main kernel: 0 = TMA producer, 1 = MMA issuer, 2, 3 = gate warps, 4..11 = tile warps (masked scores, scaled copies
// of Q), 12..19 = state warps (state rescale + bf16 copy, weighted V^T, outputs, initial/final state).
// A warp may touch only the 32 TMEM lanes of its quadrant (warp index mod 4).
constexpr int WARP_TMA = 0, WARP_MMA = 1, GATE_W0 = 2, TILE_W0 = 4, STATE_W0 = 12;
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

// Where the initial states of a segment arrive: per state a ring of two pieces of 32 d_k (16 KB each, [d_k / 4][d_v] of four d_k), in slots that
// nothing of the first chunk uses, so that its tiles are loaded and its scores masked meanwhile (with room for whole states, over V and
// Q~2 of that chunk, its outputs came 3 k cycles later).
__device__ constexpr int initial_off(int i) { return i == 0 ? TILE_BYTES : OFF_K + TILE_BYTES; }
constexpr int SUM_STAGES = 3;        // K and V tiles of the summaries: two slots each, in order

// Per-token terms of one chunk; the first index is the state.
struct alignas(16) GateSmem {
    float L[2][CM];                  // cumulative log2-gate from the chunk start, inclusive
    float E[2][CM];                  // decay from the token to the end of its block of 32 tokens
    __nv_bfloat16 w[2][CM];          // decay from the token to the end of the chunk, and what its rounding left; 0 past the end of the sequence
    __nv_bfloat16 w_rest[2][CM];
    float a[2];                      // product of the chunk's gates
};

struct alignas(16) Shared {
    uint64_t kq_full[2], v_full[2], p_full, prep_ready, sb_ready[2], ro_done, vt_ready[2], o_full, o_free, o_staged, u_full[2], g_ready[2], g_free[2], init_done;
    uint64_t s_full[SUM_STAGES], s_empty[SUM_STAGES], sw_ready[2], sw_free[2], svt_ready[2], svt_free[2], s_done;      // summaries
    uint64_t s_in[8][4], s_taken[8][2], next_ready;      // initial state: a piece has arrived, the next segment has taken its one, has room for it
    uint32_t tmem_base;
    int abort_flag;
    float* slot;                          // the first state of this (sequence, head) in its slot: read where it is needed, not kept in registers
    GateSmem gs[2];
    float a_seg[2];                       // products of the segment's gates
    uint64_t o_tail;                      // the pair of states before this one has written a ragged last chunk's outputs
    uint32_t o_turn;                      // and the first o_turn whole chunks'
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

// Rows valid .. CM - 1 of a K and a V tile, by 256 threads.
__device__ __forceinline__ void zero_rows(uint8_t* kt, uint8_t* vt, int valid, int t) {
#pragma unroll 1
    for (int i = 16 * valid + t; i < 16 * CM; i += 256) {
        const int at = (i & 8 ? HALF_BYTES : 0) + (i >> 4) * 128 + (i & 7) * 16;
        *reinterpret_cast<uint4*>(kt + at) = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(vt + at) = make_uint4(0u, 0u, 0u, 0u);
    }
}
// (the same as a call: in the variants with more code it spills less)
__device__ __noinline__ void zero_rows_call(uint8_t* kt, uint8_t* vt, int valid, int t) { zero_rows(kt, vt, valid, t); }

// ============================================================================================
// Main kernel
// ============================================================================================
// The rank-th longest of up to 64 sequences, ties by index (the order of seq_order_kernel); one warp, every lane gets the result.
// The slots are read along with the lengths.
struct SeqPlace {
    int n, t_begin, t_end, slot;
};
__device__ __forceinline__ SeqPlace longest_first(const PrefillParams& p, int rank, int lane) {
    int begin[2], end[2], slot[2], before[2] = {0, 0};
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int i = lane + 32 * x;
        begin[x] = i < p.N ? p.cu_seqlens[i] : 0;
        end[x] = i < p.N ? p.cu_seqlens[i + 1] : -1;
        slot[x] = i < p.N && p.slots ? p.slots[i] : i;
    }
    const int len0 = end[0] - begin[0], len1 = end[1] - begin[1];
#pragma unroll 1
    for (int j = 0; j < p.N; ++j) {
        const int lj = __shfl_sync(0xffffffffu, j < 32 ? len0 : len1, j & 31);
        before[0] += (lj > len0 || (lj == len0 && j < lane)) ? 1 : 0;
        before[1] += (lj > len1 || (lj == len1 && j < lane + 32)) ? 1 : 0;
    }
    const unsigned lo = __ballot_sync(0xffffffffu, lane < p.N && before[0] == rank), hi = __ballot_sync(0xffffffffu, lane + 32 < p.N && before[1] == rank);
    const int from = lo ? __ffs(lo) - 1 : __ffs(hi) - 1;
    SeqPlace r;
    r.n = lo ? from : from + 32;
    r.t_begin = __shfl_sync(0xffffffffu, lo ? begin[0] : begin[1], from);
    r.t_end = __shfl_sync(0xffffffffu, lo ? end[0] : end[1], from);
    r.slot = __shfl_sync(0xffffffffu, lo ? slot[0] : slot[1], from);
    return r;
}

// SPLIT: the sequences are cut into segments (a variant of its own: with that code in it the chunk loop of whole sequences
// ran 2 % longer).  PAIRS: the pairs of states of the n-state form side by side in the cluster (a variant for the same reason).
template <bool SPLIT, bool PAIRS>
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, const TcParams tp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const PrefillParams& p = tp.p;
    uint8_t* tiles = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);      // (an offset, not a rounded address: the compiler still knows that it is shared memory)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // The launch may overlap the tail of what precedes it in the stream: nothing is read from or written to global memory before
    // griddepcontrol.wait, which a dense batch reaches after its index arithmetic.
    if (p.cu_seqlens || p.slots) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int nseg = SPLIT ? tp.nseg : 1;
    const int pairs = PAIRS ? tp.pairs : 1;
    const int cta = blockIdx.x % (nseg * pairs);      // rank in the cluster
    const int pr = PAIRS ? cta / nseg : 0, g = cta - pr * nseg;
    const int unit = blockIdx.x / (nseg * pairs), h = unit % p.H, rank = unit / p.H;
    // (read where they are needed, not kept in registers)
    auto first = [&] { return p.state_first + 2 * pr; };
    auto accumulate = [&] { return PAIRS && pr > 0 ? true : p.accumulate != 0; };
    SeqInfo sq;
    if (tp.order_here) {
        const SeqPlace at = longest_first(p, rank, lane);
        sq = seq_info_at(at.t_begin, at.t_end, at.slot, g, tp);
    } else {
        sq = seq_info(p, tp.order ? tp.order[rank] : rank, g, tp);
    }
    if (sq.slot < 0 || sq.slot >= p.num_slots) return;
    if (tid == 0 && g == 0 && sq.nchunks > seg_begin(tp.nseg, tp.nseg, tp.cps, tp.skew8)) atomicExch(p.status, (int)DSLA_ERR_INVALID_ARG);
    float* slot1 = p.state + (((size_t)sq.slot * p.n_total + first()) * p.H + h) * (size_t)(D * D);
    const size_t state_stride = (size_t)p.H * D * D;
    if (sq.len <= 0) {  // empty sequence: a fresh start leaves zero states, a resume leaves the slot alone
        if (g == 0 && !p.use_initial_state)
            for (int i = tid; i < (p.single ? 1 : 2) * D * D; i += NTHREADS) slot1[(size_t)(i / (D * D)) * state_stride + i % (D * D)] = 0.f;
        return;
    }
    const int nc = max(0, sq.c_end - sq.c_begin);  // 0: a segment behind the end of its sequence
    const int t0 = sq.t_begin + sq.c_begin * CM;  // first token of this segment
    const int tok0 = sq.c_begin * CM;             // its index inside the sequence
    const bool last = g == sq.last_seg;           // the final state is kept; other segments skip the last chunk's update
    const bool summarize = SPLIT && g < sq.last_seg;
    const bool zero_start = !p.use_initial_state && g == 0;      // no readout of chunk 0, its update starts from zero

    // Set-up: the barriers are initialised by several warps, the TMA warp starts the first loads on its own ones, the gate warps request
    // their first gates.  (One thread for all barriers, and everything else behind it: 2200 cycles before the first load.)
    if (lane == 0) {
        if (warp == WARP_TMA) {
            for (int i = 0; i < 2; ++i) { mbar_init(&sh.kq_full[i], 1); mbar_init(&sh.v_full[i], 1); }
            for (int i = 0; i < SUM_STAGES; ++i) mbar_init(&sh.s_full[i], 1);
            fence_barrier_init();
        } else if (warp == TILE_W0) {
            mbar_init(&sh.p_full, 1); mbar_init(&sh.prep_ready, 8); mbar_init(&sh.ro_done, 1);
            mbar_init(&sh.o_full, 1); mbar_init(&sh.o_free, 8); mbar_init(&sh.o_staged, 8); mbar_init(&sh.init_done, SPLIT ? 8 : 16); mbar_init(&sh.s_done, 1);
            mbar_init(&sh.next_ready, 8);
            if (PAIRS) {
                mbar_init(&sh.o_tail, 8);
                sh.o_turn = 0;
                __threadfence();      // before the cluster barrier, behind which another CTA writes it
            }
            sh.abort_flag = 0;
            sh.slot = slot1;
            fence_barrier_init();
        } else if (warp == TILE_W0 + 1 || warp == TILE_W0 + 2) {
            const int i = warp - TILE_W0 - 1;
            mbar_init(&sh.sb_ready[i], 4); mbar_init(&sh.vt_ready[i], 8); mbar_init(&sh.u_full[i], 1); mbar_init(&sh.g_ready[i], 2); mbar_init(&sh.g_free[i], 16);
            fence_barrier_init();
        } else if (SPLIT && (warp == TILE_W0 + 3 || warp == TILE_W0 + 4)) {
            const int i = warp - TILE_W0 - 3;
            mbar_init(&sh.sw_ready[i], 2); mbar_init(&sh.sw_free[i], 8); mbar_init(&sh.svt_ready[i], 8); mbar_init(&sh.svt_free[i], 1);
            fence_barrier_init();
        } else if (SPLIT && warp == TILE_W0 + 5) {
            for (int i = 0; i < SUM_STAGES; ++i) mbar_init(&sh.s_empty[i], 9);      // eight V~ warps + the MMAs on K
            fence_barrier_init();
        } else if (SPLIT && warp >= STATE_W0) {
            for (int i = 0; i < 4; ++i) mbar_init(&sh.s_in[warp - STATE_W0][i], 1);
            for (int i = 0; i < 2; ++i) mbar_init(&sh.s_taken[warp - STATE_W0][i], 1);
            fence_barrier_init();
            if (g > 0 && nc > 0)
                for (int i = 0; i < 4; ++i) mbar_arrive_expect_tx(&sh.s_in[warp - STATE_W0][i], 32 * 128);      // 32 d_k x 32 d_v
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto load_kq = [&](int c, int q3) {
        mbar_arrive_expect_tx(&sh.kq_full[c & 1], 2 * TILE_BYTES);
        tma_load_4d(tiles + q3 * TILE_BYTES, &map_q, &sh.kq_full[c & 1], 0, t0 + c * CM, 0, h);
        tma_load_4d(tiles + OFF_K + (c & 1) * TILE_BYTES, &map_k, &sh.kq_full[c & 1], 0, t0 + c * CM, 0, h);
    };
    auto load_v = [&](int c, int v3) {
        mbar_arrive_expect_tx(&sh.v_full[c & 1], TILE_BYTES);
        tma_load_4d(tiles + v3 * TILE_BYTES, &map_v, &sh.v_full[c & 1], 0, t0 + c * CM, 0, h);
    };
    auto load_summary = [&](int it) {      // step it = chunk nc - 1 - it
        const int st = it % SUM_STAGES, t = t0 + (nc - 1 - it) * CM;
        mbar_arrive_expect_tx(&sh.s_full[st], 2 * TILE_BYTES);
        tma_load_4d(tiles + (2 * st + 1) * TILE_BYTES, &map_v, &sh.s_full[st], 0, t, 0, h);
        tma_load_4d(tiles + 2 * st * TILE_BYTES, &map_k, &sh.s_full[st], 0, t, 0, h);
    };
    if (warp == WARP_TMA && lane == 0) {
        if (summarize) {
            for (int it = 0; it < min(nc, SUM_STAGES); ++it) load_summary(it);
        } else if (nc > 0) {
            load_kq(0, 0);
            if (!SPLIT) {
                load_v(0, 2);
                if (nc > 1 && zero_start) load_kq(1, 1);
            }
        }
    }
    if (p.use_initial_state && warp >= TILE_W0)      // 128-byte lines of both states into L2
        for (int i = tid - TILE_W0 * 32; i < (p.single ? 512 : 1024); i += 512)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(slot1 + (size_t)(i >> 9) * state_stride + (size_t)(i & 511) * 32));
    float nx[4];      // gate warps: the next chunk's gates, four tokens a lane
    auto fetch = [&](int c) {      // raw values: nothing may consume them here, or the warp would sit out the load latency in every chunk
        const float* gsrc = (warp == GATE_W0 ? p.g_hist : p.g_rec) + (PAIRS ? (size_t)pr * p.pair_stride : 0);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = c * CM + 4 * lane + e;
            nx[e] = load_gate(gsrc, t0 + j, p.H, h, c >= 0 && c < nc && tok0 + j < sq.len);
        }
    };
    if (warp >= GATE_W0 && warp < TILE_W0) fetch(summarize ? nc - 1 : 0);
    if (warp == WARP_MMA) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncwarp();
    // Cluster barrier, phase 1: every CTA's barriers are initialised (waited for before the first use of another CTA's).  Phase 2: this
    // warp writes nothing more into other CTAs.  No CTA leaves before it is complete: a wait that gave up would otherwise let a CTA go that
    // its neighbours still write into.  Each warp arrives as early as it can, so that nobody waits for it at the end.
    if (SPLIT) cluster_arrive_relaxed();
    auto started_alone = [&] {      // a warp that keeps to its own CTA: both at once
        __syncwarp();
        cluster_wait();
        cluster_arrive_relaxed();
    };
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = 0;      // all 512 columns are allocated: the base is column 0
    volatile int* abortp = &sh.abort_flag;
#define WAIT(bar, ph) mbar_wait(bar, (uint32_t)(ph), abortp, p.status)

    // Whole sequences: d_k rows 64 part .. 64 part + 63 of state i from the slot, one d_v lane per thread, while the first gates are on
    // their way.
    auto start_state = [&](int i, int part, uint32_t lane_addr, int v) {
        uint32_t x[2][32];
        const float* src = sh.slot + (size_t)i * state_stride + (size_t)(64 * part) * D + v;
#pragma unroll
        for (int k = 0; k < 64; ++k) x[k >> 5][k & 31] = p.single && i == 1 ? 0u : __float_as_uint(src[(size_t)k * D]);
        tmem_st32(lane_addr + COL_S + 128 * i + 64 * part, x[0]);
        tmem_st32(lane_addr + COL_S + 128 * i + 64 * part + 32, x[1]);
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&sh.init_done);
    };

    if (warp == WARP_TMA) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0 && summarize) {
            for (int it = SUM_STAGES; it < nc; ++it) {
                WAIT(&sh.s_empty[it % SUM_STAGES], (it / SUM_STAGES - 1) & 1);
                if (*abortp) break;
                load_summary(it);
            }
            WAIT(&sh.s_done, 0);
            if (!*abortp) load_kq(0, 0);
        }
        if (PAIRS) {
            __syncwarp();
            cluster_wait();
        } else if (SPLIT) {
            started_alone();
        }
        if (lane == 0 && nc > 0) {
            const uint32_t next_turn = PAIRS && pr + 1 < pairs ? map_to_cta(smem_u32(&sh.o_turn), (uint32_t)(cta + nseg)) : 0u;
            if (SPLIT) {
                if (!*abortp) load_v(0, 2);
                if (g > 0) WAIT(&sh.init_done, 0);      // the initial state is in TMEM, its place free
                if (nc > 1 && !*abortp) load_kq(1, 1);      // (not onto pieces that may still arrive, where a wait for them gave up)
            }
            if (!SPLIT && !zero_start && nc > 1) {
                WAIT(&sh.init_done, 0);      // behind the initial state, which is needed first
                if (!*abortp) load_kq(1, 1);
            }
            const int nfull = (sq.len - tok0) / CM;         // whole chunks leave through shared memory and a tile store
            int c3 = 0;
#pragma unroll 1
            for (int c = 0; c < nc && !*abortp; ++c) {
                const int v3 = c3 == 0 ? 2 : c3 - 1;
                if (c + 1 < nc) {
                    WAIT(&sh.ro_done, c & 1);              // Q of chunk c has been read: its slot takes V of chunk c + 1
                    load_v(c + 1, c3);
                    // pull what the next loads will need into L2 (a tile's slot frees only about one load latency before it is used)
                    if (c + 2 < nc) tma_prefetch_4d(&map_v, 0, t0 + (c + 2) * CM, 0, h);
                }
                if (c < nfull) {
                    WAIT(&sh.o_staged, c & 1);             // the outputs of chunk c are in the slot of its V
                    if (PAIRS && pr > 0) {                 // behind the pair of states before this one: sums in a fixed order
                        wait_count_cluster(&sh.o_turn, (uint32_t)(c + 1), abortp, p.status);
                        fence_proxy_async_global();
                    }
                    if (accumulate()) tma_add_4d(&map_o, tiles + v3 * TILE_BYTES, 0, t0 + c * CM, 0, h);      // bf16 sums, one rounding each
                    else tma_store_4d(&map_o, tiles + v3 * TILE_BYTES, 0, t0 + c * CM, 0, h);
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
                if (PAIRS && pr + 1 < pairs && c < nfull) {
                    bulk_wait_all();
                    st_release_cluster(next_turn, (uint32_t)(c + 1));
                }
                c3 = c3 == 2 ? 0 : c3 + 1;
            }
            bulk_wait_all();
        }
        if (PAIRS) {
            __syncwarp();
            cluster_arrive_relaxed();
        }
    } else if (warp == WARP_MMA) {
        // ------------------------------------------------------------------ MMA issuer
        // Per chunk:  O^T = S1^T Q~1^T + S2^T Q~2^T,  O^T += V^T P~^T,  S1^T += V~1^T K,  P of the next chunk,  S2^T += V~2^T K.
        // The readout of a state starts as soon as its bf16 copy is there; V~ is stored under the P~ part, O^T is read out under
        // the first update, the next scores are masked under the second.
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
        if (elect_one()) {
            if (summarize) {
#pragma unroll 1
                for (int it = 0; it < nc; ++it) {
                    const int st = it % SUM_STAGES, b = it & 1;
                    WAIT(&sh.s_full[st], (it / SUM_STAGES) & 1);
                    WAIT(&sh.svt_ready[b], (it >> 1) & 1);
                    tc_fence_after();
                    const uint32_t bk = dv0 + (uint32_t)(2 * st) * T_STEP;      // K in slot 2 st, MN-major like V
#pragma unroll 1
                    for (int i = 0; i < 2; ++i) {
                        const uint32_t a = (b ? COL_R : COL_SB) + 64 * i;
                        issue4_ts<128>(COL_S + 128 * i, a, bk, ID_U, it ? 1u : 0u);
                        issue4_ts<128>(COL_S + 128 * i, a + 32, bk + 512, ID_U, 1u);
                    }
                    tc_commit(&sh.s_empty[st]);
                    tc_commit(&sh.svt_free[b]);
                }
                tc_commit(&sh.s_done);
            }
            if (nc > 0) scores(0, 0);
        }
        __syncwarp();
        if (SPLIT) started_alone();
        if (elect_one()) {
            int c3 = 0;
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                const int v3 = c3 == 0 ? 2 : c3 - 1, n3 = c3 == 2 ? 0 : c3 + 1;
                WAIT(&sh.v_full[c & 1], (c >> 1) & 1);
                WAIT(&sh.prep_ready, c & 1);               // P read out of TMEM, P~, Q~1, Q~2 in place
                const bool first = zero_start && c == 0;   // nothing to read out, nothing to add to
                if (first) tc_fence_after();
#pragma unroll 1
                for (int i = first ? 2 : 0; i < 2; ++i) {
                    WAIT(&sh.sb_ready[i], c & 1);
                    tc_fence_after();
                    const uint32_t a = COL_SB + 64 * i, b = i == 0 ? dq0 + (uint32_t)c3 * T_STEP : dq2;
                    issue4_ts<2>(COL_R, a, b, ID_KK, i ? 1u : 0u);
                    issue4_ts<2>(COL_R, a + 32, b + H_STEP, ID_KK, 1u);
                }
                tc_commit(&sh.ro_done);
                const uint32_t v = dv0 + (uint32_t)v3 * T_STEP;
                issue4_ss<128, 2>(COL_R, v, dp0, ID_V128, first ? 0u : 1u);
                issue4_ss<128, 2>(COL_R + 64, v + 512, dp0 + H_STEP, ID_V64, 1u);     // keys 64..127 reach only the outputs of tokens 64..127
                tc_commit(&sh.o_full);
                const bool update = last || c + 1 < nc;
                const uint32_t bk = dkn + (uint32_t)(c & 1) * T_STEP;
#pragma unroll 1
                for (int i = 0; i < 2; ++i) {
                    if (update) {
                        WAIT(&sh.vt_ready[i], c & 1);
                        tc_fence_after();
                        issue4_ts<128>(COL_S + 128 * i, COL_SB + 64 * i, bk, ID_U, first ? 0u : 1u);
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
    } else if (warp >= TILE_W0 && warp < STATE_W0) {
        // ------------------------------------------------------------------ tile warps 4..11
        const int tt = tid - TILE_W0 * 32;                // 0..255
        const int q = warp & 3;                           // TMEM lane quadrant: rows (tokens) 32 q .. 32 q + 31
        const int half = (warp - TILE_W0) >> 2;           // column half: keys 64 half .. 64 half + 63
        const uint32_t lane_addr = tb + ((uint32_t)(32 * q) << 16);
        const int j = 32 * q + lane;
        const uint32_t row_at = (uint32_t)(j * 128 + ((j & 7) << 4));      // row j of a swizzled half tile: piece m is at row_at ^ (m << 4)
        const float W1 = (p.weights ? p.weights[(size_t)h * p.n_total + first()] : p.gamma[h]) * p.scale;
        const float W2 = p.single ? 0.f : (p.weights ? p.weights[(size_t)h * p.n_total + first() + 1] : 1.f - p.gamma[h]) * p.scale;

        if (!SPLIT && !zero_start) start_state(half, 1, lane_addr, j);
        // The ten 32 x 32 blocks of the lower triangle: a quadrant's q + 1 blocks are split between its two warps, the second one
        // takes the diagonal block first.  The decays of a warp's first block are computed ahead of the scores.  The two blocks above the
        // diagonal that the MMAs read are zeroed once.
        const int blk0 = half == 0 ? 0 : q, blk1 = half == 0 ? (q >= 2 ? 1 : -1) : (q == 3 ? 2 : -1);
        if (half == 0 && (q == 0 || q == 2))
            for (int m4 = 0; m4 < 4; ++m4)
                *reinterpret_cast<uint4*>(tiles + OFF_PT + (q == 2 ? HALF_BYTES - 64 * 128 : 0) + sw128_offset(j, 32 + 8 * m4)) = make_uint4(0u, 0u, 0u, 0u);
        // a block left of the diagonal: its decays factor through its last token
        auto block_decays = [&](const GateSmem& gs, int blk, float L1, float L2, float2 (&mk)[16]) {
            const float R1 = W1 * ex2(L1 - gs.L[0][32 * blk + 31]), R2 = W2 * ex2(L2 - gs.L[1][32 * blk + 31]);
            const float2 RR1 = make_float2(R1, R1), RR2 = make_float2(R2, R2);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 E1 = *reinterpret_cast<const float4*>(&gs.E[0][32 * blk + 4 * e]), E2 = *reinterpret_cast<const float4*>(&gs.E[1][32 * blk + 4 * e]);
                mk[2 * e] = __ffma2_rn(RR2, make_float2(E2.x, E2.y), __fmul2_rn(RR1, make_float2(E1.x, E1.y)));
                mk[2 * e + 1] = __ffma2_rn(RR2, make_float2(E2.z, E2.w), __fmul2_rn(RR1, make_float2(E1.z, E1.w)));
            }
        };
        if (SPLIT) started_alone();
        // The decays of a block (32 registers) and the scaled Q (32) are alive across the waits of this loop, where a call costs spills.  Whole
        // sequences: the wait for Q and K comes before the decays, rows are cleared without a call (16 prompts of 335K tokens 2791 to
        // 2756 us, 8 x 512 tokens 50.0 to 48.7, pieces of one chunk 14.9 to 14.7, 232 tokens 13.0 to 12.8).  Segments: decays first, since the tiles come late, and waits without
        // a call (777 tokens 20.9 to 20.6; with the other order 21.8).  Pairs of states keep the calls (eight states 156 us, without them 170).
        auto tile_wait = [&](uint64_t* bar, int ph) {
            if (SPLIT && !PAIRS) mbar_wait_inline(bar, (uint32_t)ph, abortp, p.status);
            else WAIT(bar, ph);
        };
        int c3 = 0;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            const GateSmem& gs = sh.gs[s];
            uint8_t* qs = tiles + c3 * TILE_BYTES;
            tile_wait(&sh.g_ready[s], (c >> 1) & 1);
            if (!SPLIT) tile_wait(&sh.kq_full[s], (c >> 1) & 1);      // the TMA writes of Q are visible to this thread
            // ---- decays of this warp's first block, ahead of the scores that they multiply
            const float L1 = gs.L[0][j], L2 = gs.L[1][j];
            float2 mk[16];
            if (half == 0) {
                if (q > 0) block_decays(gs, 0, L1, L2, mk);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 K1 = *reinterpret_cast<const float4*>(&gs.L[0][32 * q + 4 * e]), K2 = *reinterpret_cast<const float4*>(&gs.L[1][32 * q + 4 * e]);
                    mk[2 * e].x = fmaf(W2, ex2(L2 - K2.x), W1 * ex2(L1 - K1.x)); mk[2 * e].y = fmaf(W2, ex2(L2 - K2.y), W1 * ex2(L1 - K1.y));
                    mk[2 * e + 1].x = fmaf(W2, ex2(L2 - K2.z), W1 * ex2(L1 - K1.z)); mk[2 * e + 1].y = fmaf(W2, ex2(L2 - K2.w), W1 * ex2(L1 - K1.w));
                }
            }
            if (SPLIT) tile_wait(&sh.kq_full[s], (c >> 1) & 1);
            // Rows of K and V past the end of the sequence belong to the next one.  They would meet only zero weights, but 0 * inf is not 0.  (The
            // scores, which may be reading K, meet them only in columns that no row of this sequence uses; V~ and the other MMAs wait for
            // prep_ready.  Here, under the scores; ahead of prep_ready it took 1 % of a packed batch's time, ahead of the decays 2 % of a call of
            // 129 tokens.)
            const int valid = sq.len - tok0 - c * CM;
            if (valid < CM) {
                tile_wait(&sh.v_full[s], (c >> 1) & 1);
                uint8_t *kt = tiles + OFF_K + s * TILE_BYTES, *vt = tiles + (c3 == 0 ? 2 : c3 - 1) * TILE_BYTES;
                if (SPLIT) zero_rows_call(kt, vt, valid, tt);
                else zero_rows(kt, vt, valid, tt);
            }
            // ---- scaled copies of Q, eight 16-byte pieces (half a row) per thread: one factor per state for all of them.  (Consecutive pieces per
            // thread needed the factors of eight rows from shared memory, which the loop is bound by.)  The copy for state 2 is written as soon as the readout
            // of the previous chunk is done with its buffer, the one for state 1 waits in registers until the scores have read the raw Q.
            if (c > 0) tile_wait(&sh.ro_done, (c - 1) & 1);
            uint8_t* qh = qs + half * HALF_BYTES;
            const uint32_t f1 = dup_bf16(W1 * ex2(L1)), f2 = dup_bf16(W2 * ex2(L2));      // weight * decay from the chunk start through the token
            uint4 q1[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) q1[m] = *reinterpret_cast<const uint4*>(qh + (row_at ^ (m << 4)));
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                *reinterpret_cast<uint4*>(tiles + OFF_Q2 + half * HALF_BYTES + (row_at ^ (m << 4))) = scale8(q1[m], f2);
                q1[m] = scale8(q1[m], f1);
            }
            mbar_wait_inline(&sh.p_full, c & 1, abortp, p.status);
            tc_fence_after();
#pragma unroll
            for (int m = 0; m < 8; ++m) *reinterpret_cast<uint4*>(qh + (row_at ^ (m << 4))) = q1[m];
            // ---- P~ = P (.) M
            auto store_masked = [&](int blk, const float2 (&m)[16], int upto) {      // keys later than `upto` carry nothing
                uint8_t* at = tiles + OFF_PT + (blk >= 2 ? HALF_BYTES - 64 * 128 : 0);
                uint32_t r[32], pk[16];
                tmem_ld32(lane_addr + COL_R + 32 * blk, r);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float2 y = __fmul2_rn(m[e], make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])));
                    pk[e] = pack_bf16(2 * e <= upto ? y.x : 0.f, 2 * e + 1 <= upto ? y.y : 0.f);
                }
#pragma unroll
                for (int m4 = 0; m4 < 4; ++m4)
                    *reinterpret_cast<uint4*>(at + (row_at ^ ((4 * (blk & 1) + m4) << 4))) = make_uint4(pk[4 * m4], pk[4 * m4 + 1], pk[4 * m4 + 2], pk[4 * m4 + 3]);
            };
            if (half == 1 || q > 0) store_masked(blk0, mk, half == 0 ? 31 : lane);
            if (blk1 >= 0) {
                block_decays(gs, blk1, L1, L2, mk);
                store_masked(blk1, mk, 31);
            }
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) { mbar_arrive(&sh.prep_ready); mbar_arrive(&sh.g_free[s]); }
            c3 = c3 == 2 ? 0 : c3 + 1;
        }
    } else if (warp < TILE_W0) {
        // ------------------------------------------------------------------ gate warps: 2 = state 1, 3 = state 2
        // Everything the chunk needs from the gates comes from the cumulative log-gates
        //     L_j = sum_{t <= j} log2 g_t        (inclusive, from the chunk start; a zero gate counts as -130, so any product
        //                                         that contains one flushes to an exact zero)
        // through independent exponentials.  Lane l holds tokens 4 l .. 4 l + 3.  The chunk decay that carries the state
        // is the plain product of the gates.
        const int i = warp - GATE_W0;
        auto decays = [&](const float (&x)[4], float (&L)[4], float& pr, float& incl) {      // L: inclusive from the chunk start; incl: of the lane's last token
            float run = 0.f;
            pr = 1.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float y = fmaxf(x[e], 0.f);
                pr *= y;
                run += lg2_gate(y);
                L[e] = run;
            }
            incl = warp_prefix_sum(run, lane);
            float excl = __shfl_up_sync(0xffffffffu, incl, 1);
            if (lane == 0) excl = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) L[e] = e == 3 ? incl : excl + L[e];      // (`incl` is what other lanes see: keep the two consistent)
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) pr *= __shfl_xor_sync(0xffffffffu, pr, off);
        };
        auto store_weights = [&](GateSmem& gs, const float (&w)[4]) {
            const uint2 x = make_uint2(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]));
            const float2 lo = unpack_bf16(x.x), hi = unpack_bf16(x.y);
            *reinterpret_cast<uint2*>(&gs.w[i][4 * lane]) = x;
            *reinterpret_cast<uint2*>(&gs.w_rest[i][4 * lane]) = make_uint2(pack_bf16(w[0] - lo.x, w[1] - lo.y), pack_bf16(w[2] - hi.x, w[3] - hi.y));
        };
        if (summarize) {      // weights to the end of the segment, chunks from the last to the first
            float after = 0.f, A = 1.f;      // log2 and product of the gates of all later chunks
            for (int it = 0; it < nc; ++it) {
                const int b = it & 1;
                const float x[4] = {nx[0], nx[1], nx[2], nx[3]};
                fetch(nc - 2 - it);
                float L[4], pr, incl;
                decays(x, L, pr, incl);
                const float end = __shfl_sync(0xffffffffu, incl, 31);
                if (it >= 2) WAIT(&sh.sw_free[b], ((it >> 1) - 1) & 1);
                const float w[4] = {ex2(end - L[0] + after), ex2(end - L[1] + after), ex2(end - L[2] + after), ex2(end - L[3] + after)};
                store_weights(sh.gs[b], w);
                after += end;
                A *= pr;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.sw_ready[b]);
            }
            if (lane == 0) sh.a_seg[i] = A;
            for (int it = max(0, nc - 2); it < nc; ++it) WAIT(&sh.sw_free[it & 1], (it >> 1) & 1);      // the ring is reused for the chunks below
            fetch(0);
        }
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            GateSmem& gs = sh.gs[s];
            const float x[4] = {nx[0], nx[1], nx[2], nx[3]};
            fetch(c + 1);
            float L[4], pr, incl;
            decays(x, L, pr, incl);
            const float block_end = __shfl_sync(0xffffffffu, incl, lane | 7), end = __shfl_sync(0xffffffffu, incl, 31);
            const int valid = min(CM, sq.len - tok0 - c * CM);
            if (c >= 2) WAIT(&sh.g_free[s], ((c >> 1) - 1) & 1);
            float E[4], w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                E[e] = ex2(block_end - L[e]);
                w[e] = 4 * lane + e < valid ? ex2(end - L[e]) : 0.f;
            }
            *reinterpret_cast<float4*>(&gs.L[i][4 * lane]) = make_float4(L[0], L[1], L[2], L[3]);
            *reinterpret_cast<float4*>(&gs.E[i][4 * lane]) = make_float4(E[0], E[1], E[2], E[3]);
            store_weights(gs, w);
            if (lane == 0) gs.a[i] = pr;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.g_ready[s]);
            if (SPLIT && c == 0) started_alone();
        }
        if (SPLIT && nc == 0) started_alone();
    } else {
        // ------------------------------------------------------------------ state warps 12..19
        const int q = warp & 3, hi = (warp - STATE_W0) >> 2;   // TMEM lane quadrant, state index
        const uint32_t lane_addr = tb + ((uint32_t)(32 * q) << 16);
        const uint32_t s_addr = lane_addr + COL_S + 128 * hi;
        const uint32_t sb_addr = lane_addr + COL_SB + 64 * hi;
        const int v = 32 * q + lane;
        __nv_bfloat16* og = reinterpret_cast<__nv_bfloat16*>(p.o);
        // ldmatrix: this thread addresses row mr of matrix mk; matrices (tokens 0..7 | 8..15) x (d_v 0..7 | 8..15)
        const int mk = lane >> 3, mr = lane & 7;
        // V~_i^T[v][s] = w^i_s V[s][v] of both states, for the 32 d_v lanes of this quadrant and tokens 64 hi .. 64 hi + 63 (16 lanes and all tokens
        // took twice the loads of weights): ldmatrix.trans hands out the element pairs a 16x128b TMEM store takes.  `wait` runs between the
        // arithmetic and the stores.  The weights have two bf16 terms, so that the product is rounded once: with one term, over chunks of 128 tokens,
        // states were 2.11e-3 from the exact ones, now 1.65e-3 (T = 4096, 59.3 to 59.7 us; other sizes lose up to 2 %).
        auto weighted_v = [&](const uint8_t* vtile, const GateSmem& gs, uint32_t col, auto wait) {
            const int d = 32 * q + 8 * (mk & 1);                      // first d_v column of the matrix this thread addresses, lanes 0..15 of the quadrant
            const uint32_t row0 = smem_u32(vtile) + (uint32_t)((64 * hi + 8 * (mk >> 1) + mr) * 128) + (uint32_t)(d >> 6) * HALF_BYTES +
                                  (((uint32_t)((d & 63) >> 3) ^ (uint32_t)mr) << 4);
            uint32_t r[32], y[32];      // [lanes 0..15 | 16..31][16 tokens][4]
#pragma unroll
            for (int t16 = 0; t16 < 8; ++t16) {
                const uint32_t at = (t16 < 4 ? row0 : row0 ^ 32u) + (uint32_t)((t16 & 3) * 16 * 128);
                ldmatrix_x4_trans(at, r[4 * t16], r[4 * t16 + 1], r[4 * t16 + 2], r[4 * t16 + 3]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                constexpr uint32_t REST = (uint32_t)(offsetof(GateSmem, w_rest) - offsetof(GateSmem, w));
                const uint32_t wp = smem_u32(&gs.w[i][64 * hi + 2 * (lane & 3)]);
                uint32_t* o = i == 0 ? y : r;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const uint32_t w0 = ld_shared_u32(wp + 32 * t), w1 = ld_shared_u32(wp + 32 * t + 16);
                    const uint32_t l0 = ld_shared_u32(wp + REST + 32 * t), l1 = ld_shared_u32(wp + REST + 32 * t + 16);
#pragma unroll
                    for (int x = 4 * t; x < 32; x += 16) {
                        o[x] = hfma2_u32(r[x], w0, hmul2_u32(r[x], l0)); o[x + 1] = hfma2_u32(r[x + 1], w0, hmul2_u32(r[x + 1], l0));
                        o[x + 2] = hfma2_u32(r[x + 2], w1, hmul2_u32(r[x + 2], l1)); o[x + 3] = hfma2_u32(r[x + 3], w1, hmul2_u32(r[x + 3], l1));
                    }
                }
            }
            wait();
            const uint32_t at = lane_addr + col + 32 * hi, at16 = at + (16u << 16);
            tmem_st_16x128b_x8(at, y); tmem_st_16x128b_x8(at16, y + 16);
            tmem_st_16x128b_x8(at + 64, r); tmem_st_16x128b_x8(at16 + 64, r + 16);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
        };
        if (summarize) {
#pragma unroll 1
            for (int it = 0; it < nc; ++it) {
                const int st = it % SUM_STAGES, b = it & 1;
                WAIT(&sh.sw_ready[b], (it >> 1) & 1);
                WAIT(&sh.s_full[st], (it / SUM_STAGES) & 1);
                weighted_v(tiles + (2 * st + 1) * TILE_BYTES, sh.gs[b], b ? COL_R : COL_SB, [&] {
                    if (it >= 2) WAIT(&sh.svt_free[b], ((it >> 1) - 1) & 1);
                    tc_fence_after();
                });
                if (lane == 0) { mbar_arrive(&sh.svt_ready[b]); mbar_arrive(&sh.s_empty[st]); mbar_arrive(&sh.sw_free[b]); }
            }
            WAIT(&sh.s_done, 0);
            tc_fence_after();
        }
        // Initial state of this warp's state and d_v lanes, in pieces of 32 d_k: from the slot (or zero) in the first segment, else from the
        // same warp of the segment before; what the next segment starts from goes to the same warp there.
        auto chain = [&](float a) {
            const float A = sh.a_seg[hi];
            const uint32_t mine = (uint32_t)(initial_off(hi) + v * 16), w = warp - STATE_W0;
            const uint32_t next = map_to_cta(smem_u32(tiles + mine), (uint32_t)(g + 1 < nseg ? cta + 1 : cta));
            const uint32_t next_bar = map_to_cta(smem_u32(&sh.s_in[w][0]), (uint32_t)(g + 1 < nseg ? cta + 1 : cta));
            if (summarize) mbar_wait_cluster(&sh.next_ready, 0, abortp, p.status);
#pragma unroll 1
            for (int b = 0; b < 8; ++b) {      // 16 d_k at a time, handed over in pairs
                uint32_t u[16];
                float x[16];
                if (summarize) tmem_ld16(s_addr + 16 * b, u);
                if (g > 0) {
                    if ((b & 1) == 0) mbar_wait_cluster(&sh.s_in[w][b >> 1], 0, abortp, p.status);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 y = *reinterpret_cast<const float4*>(tiles + mine + (4 * (b & 3) + k) * (D * 16));
                        x[4 * k] = y.x; x[4 * k + 1] = y.y; x[4 * k + 2] = y.z; x[4 * k + 3] = y.w;
                    }
                } else {
                    const float* src = sh.slot + (size_t)hi * state_stride + (size_t)(16 * b) * D + v;
                    const bool load = p.use_initial_state && !(p.single && hi == 1);
#pragma unroll
                    for (int k = 0; k < 16; ++k) x[k] = load ? src[(size_t)k * D] : 0.f;
                }
                if (summarize) {
                    tc_wait_ld();
                    if (b == 4 || b == 6) mbar_wait_cluster(&sh.s_taken[w][(b >> 1) - 2], 0, abortp, p.status);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        st_async_f32x4(next + (uint32_t)((4 * (b & 3) + k) * (D * 16)), fmaf(A, x[4 * k], __uint_as_float(u[4 * k])), fmaf(A, x[4 * k + 1], __uint_as_float(u[4 * k + 1])),
                                       fmaf(A, x[4 * k + 2], __uint_as_float(u[4 * k + 2])), fmaf(A, x[4 * k + 3], __uint_as_float(u[4 * k + 3])), next_bar + 8u * (b >> 1));
                }
                if (!zero_start) {
                    uint32_t pk[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) pk[k] = pack_bf16(x[2 * k], x[2 * k + 1]);
#pragma unroll
                    for (int k = 0; k < 16; ++k) u[k] = __float_as_uint(x[k] * a);
                    tmem_st8(sb_addr + 8 * b, pk);
                    tmem_st16(s_addr + 16 * b, u);
                }
                if (g > 0 && (b == 1 || b == 3)) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&sh.s_taken[w][b >> 1]), (uint32_t)(cta - 1)));
                }
            }
            tc_wait_st();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.init_done);
        };
        if (SPLIT) {
            __syncwarp();
            cluster_wait();
            if (g > 0 && nc > 0 && lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&sh.next_ready), (uint32_t)(cta - 1)));      // room for this segment's initial state
        }
        if (!SPLIT && !zero_start) {
            start_state(hi, 0, lane_addr, v);
            WAIT(&sh.init_done, 0);     // the tile warps' half
        }
        int v3 = 2;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            const int s = c & 1;
            const GateSmem& gs = sh.gs[s];
            WAIT(&sh.g_ready[s], (c >> 1) & 1);
            const float a = gs.a[hi];
            if (SPLIT && c == 0) {
                chain(a);
                __syncwarp();
                if (!PAIRS) cluster_arrive_relaxed();
            } else if (c > 0 || !zero_start) {
                if (c > 0) WAIT(&sh.u_full[hi], (c - 1) & 1);
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
            // ---- V~ of both states: built in registers under the readout, stored over the bf16 copies as soon as those have been read; the
            // P~ part of the outputs, which follows, leaves shared memory no room for other reads
            WAIT(&sh.v_full[s], (c >> 1) & 1);
            WAIT(&sh.prep_ready, c & 1);      // (under the readout: before it the tile warps need the issue slots and shared memory)
            weighted_v(tiles + v3 * TILE_BYTES, gs, COL_SB, [&] {
                mbar_wait_inline(&sh.ro_done, c & 1, abortp, p.status);
                tc_fence_after();
            });
            if (lane == 0) { mbar_arrive(&sh.vt_ready[0]); mbar_arrive(&sh.vt_ready[1]); mbar_arrive(&sh.g_free[s]); }
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
                if (PAIRS && pr > 0) mbar_wait_cluster(&sh.o_tail, 0, abortp, p.status);
#pragma unroll 1
                for (int b = 64 * hi; b < 64 * hi + 64; b += 16) {
                    uint32_t r[16];
                    tmem_ld16(lane_addr + COL_R + b, r);
                    tc_wait_ld();
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        if (b + jj < valid) {
                            const __nv_bfloat16 y = __float2bfloat16_rn(__uint_as_float(r[jj]));
                            *dst = accumulate() ? __hadd(*dst, y) : y;
                        }
                        dst += row;
                    }
                }
                if (PAIRS && pr + 1 < pairs) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&sh.o_tail), (uint32_t)(cta + nseg)));
                }
            }
            v3 = v3 == 2 ? 0 : v3 + 1;
        }
        if (SPLIT && (PAIRS || nc == 0)) {
            __syncwarp();
            cluster_arrive_relaxed();
        }
        if (last && nc > 0) {
            WAIT(&sh.u_full[hi], (nc - 1) & 1);
            tc_fence_after();
            if (!(p.single && hi == 1)) store_state(sh.slot + (size_t)hi * state_stride, v, s_addr, 0, 4);
        }
    }
    __syncwarp();
    if (SPLIT) cluster_wait();      // phase 2
    settle_after_timeout(abortp);
    tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) tmem_dealloc(tb, 512);
#undef WAIT
}

}  // namespace

namespace {

// Packed batches are visited longest first; up to ORDER_HERE_MAX_N sequences the main kernel of the single-CTA variant finds its place
// in the order by itself (a kernel for it takes 3 us of a call).
bool wants_order(const dsla_prefill_args* a) { return a->cu_seqlens != nullptr && a->N > 1 && a->N <= ORDER_MAX_N; }
bool orders_here(const dsla_prefill_args* a) { return a->N <= ORDER_HERE_MAX_N; }

// The most clusters of each size (one CTA per SM) that fit on the device at once; sizes over 8 are opt-in.
constexpr int MAX_SEG = 16;
int resident_clusters(int size) {
    static std::atomic<int> cached[64][MAX_SEG + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return sm_count() / size; }
    int n = cached[dev][size].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(size * sm_count()));
        cfg.blockDim = dim3(NTHREADS);
        cfg.dynamicSmemBytes = SMEM_DYN;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaFuncSetAttribute(prefill_tc_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_DYN) != cudaSuccess ||
            (size > 8 && cudaFuncSetAttribute(prefill_tc_kernel<true, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
            cudaOccupancyMaxActiveClusters(&n, prefill_tc_kernel<true, false>, &cfg) != cudaSuccess || n <= 0)
            n = -1;
        (void)cudaGetLastError();
        cached[dev][size].store(n, std::memory_order_relaxed);
    }
    return n > 0 ? n : 0;
}

// Segments per sequence: the most that keep all work items resident at once (CTAs of a cluster, or clusters of the pair variant).
// The single-CTA kernel's segments hold at least one chunk of 128 tokens, and a sequence of two chunks stays whole (summary and
// chain cost more than the chunk they would save: 256 tokens, 8 heads 11.6 us whole, 13.8 in two segments; 74 heads 12.7 and 16.9); the pair
// variant's at least four of 64.
// Several pairs of states of the n-state form in one launch: the CTAs of all of them and of all segments form one cluster; *nseg = 0 if
// they cannot all be resident.
void plan(const dsla_prefill_args* a, bool pair, int pairs, int* nseg, int* cps, int* skew8) {
    const int chunk = pair ? C : CM;
    const int max_chunks = (a->max_seqlen + chunk - 1) / chunk;
    const long long units = (long long)a->N * a->H;
    int ns = 1;
    *skew8 = 0;
    if (pair) {
        const int room = pair_resident_clusters();
        if (units > 0 && units < room) ns = (int)(room / units);
        if (ns > MAX_SEG) ns = MAX_SEG;
        while (ns > 1 && (max_chunks + ns - 1) / ns < 4) --ns;
    } else if (pairs > 1) {
        ns = units > 0 ? (int)(sm_count() / (units * pairs)) : 1;
        if (ns > MAX_SEG / pairs) ns = MAX_SEG / pairs;
        if (ns > 1 && (ns > max_chunks || max_chunks <= 2)) ns = max_chunks <= 2 ? 1 : max_chunks;
        while (ns > 0 && resident_clusters(ns * pairs) < units) --ns;
        if (ns > 1) ns = (max_chunks + (max_chunks + ns - 1) / ns - 1) / ((max_chunks + ns - 1) / ns);
    } else if (units > 0 && units < sm_count() && max_chunks > 2) {
        ns = (int)(sm_count() / units);
        if (ns > MAX_SEG) ns = MAX_SEG;
        if (ns > max_chunks) ns = max_chunks;
        while (ns > 1 && resident_clusters(ns) < units) --ns;
        ns = (max_chunks + (max_chunks + ns - 1) / ns - 1) / ((max_chunks + ns - 1) / ns);      // no segment without a chunk in the longest sequence
    }
    if (max_chunks <= 0) ns = 1;
    *nseg = ns;
    *cps = max_chunks > 0 && ns > 0 ? (max_chunks + ns - 1) / ns : 1;
    // The pair variant's later segments fold more summaries into their initial state before they start (about 50 tokens' time
    // each): make consecutive segments about that much shorter, as far as the shortest keeps at least 192 tokens.
    if (pair && ns > 1) {
        const int sk = (8 * (*cps - 3)) / (ns - 1);
        *skew8 = sk < 0 ? 0 : (sk > 3 ? 3 : sk);
    }
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
size_t order_bytes(const dsla_prefill_args* a, bool pair) { return wants_order(a) && (pair || !orders_here(a)) ? up256((size_t)a->N * sizeof(int)) : 0; }
// The pair variant's summaries (the single-CTA kernel's stay on chip)
size_t summaries_bytes(const dsla_prefill_args* a, int nseg) { return nseg > 1 ? (size_t)a->N * a->H * nseg * SUMMARY_STRIDE : 0; }
// room for the snapshot of the initial states of split sequences (used when use_initial_state is set)
size_t snapshot_bytes(const dsla_prefill_args* a, int nseg) { return nseg > 1 ? (size_t)a->N * a->H * 2 * D * D * sizeof(float) : 0; }

dsla_status launch_main(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mo, const TcParams& tp, cudaStream_t s) {
    const int size = tp.nseg * tp.pairs;      // CTAs of a cluster
    const auto kernel = tp.pairs > 1 ? prefill_tc_kernel<true, true> : size > 1 ? prefill_tc_kernel<true, false> : prefill_tc_kernel<false, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_DYN) != cudaSuccess) return DSLA_ERR_CUDA;
    if (size > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return DSLA_ERR_CUDA;
    const long long units = (long long)tp.p.N * tp.p.H;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * size));
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = SMEM_DYN;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)size; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = size > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kernel, mq, mk, mv, mo, tp) != cudaSuccess) return DSLA_ERR_CUDA;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DSLA_OK : DSLA_ERR_CUDA;
}

}  // namespace

bool prefill_tc_available() { return true; }

// Pairs of states side by side need fewer segments per sequence, so shorter chains of initial states, and read Q, K and V from L2
// the second time (four states, T = 4096, 32 heads: 112 us as two launches, 89 as one; eight: 221 and 152); but SMs may be left over,
// or the sequences be cut less than a launch for each pair would.  Weights: a chunk 8, set-up and drain 5, a summary 2 per chunk, a hop of the
// initial states 3.  (Stamped now, a chunk is 6.6 to 7.1 k cycles, a summary 1.9 to 2.5 k, the first hop 9 k and further ones 2 k.  With these
// weights the choice is within 3 % of the best of 1, 2 and 4 on 272 of 278 shapes of four and eight states; the worst are eight states of
// 3000 tokens, 16 heads, 141 us where all pairs in one launch take 128, and of 2048 tokens, 40 heads, 168 and 159.)
int prefill_tc_pairs(const dsla_prefill_args* a, int npairs) {
    int best = 1;
    long long least = 0;
    for (int k = 1; k <= npairs; k *= 2) {
        int nseg, cps, skew8;
        plan(a, false, k, &nseg, &cps, &skew8);
        if (nseg < 1) break;
        const long long cost = (npairs / k) * (8ll * cps + 5 + (nseg > 1 ? 2ll * cps + 3 * (nseg - 1) : 0));
        if (k == 1 || cost < least) { best = k; least = cost; }
    }
    return best;
}

// What a call is refused without: of the single-CTA kernel only the visiting order of large packed batches.
size_t prefill_tc_required_bytes(const dsla_prefill_args* a, bool pair) { return pair ? prefill_tc_workspace_bytes(a, true) : order_bytes(a, false); }

// What a caller is told to hand over.  (The single-CTA kernel's summaries stay on chip; where it cuts sequences the answer is one block more
// than it needs, so that it says, as it always has, which calls are cut.)
size_t prefill_tc_workspace_bytes(const dsla_prefill_args* a, bool pair) {
    int nseg, cps, skew8;
    plan(a, pair, 1, &nseg, &cps, &skew8);
    if (!pair) return order_bytes(a, false) + (nseg > 1 ? 256 : 0);
    return summaries_bytes(a, nseg) + order_bytes(a, true) + snapshot_bytes(a, nseg);     // each a multiple of 256
}

dsla_status launch_prefill_tc(const PrefillParams& p, const dsla_prefill_args* a, bool pair, cudaStream_t s) {
    if (p.N == 0 || a->T_total == 0) {
        // only empty sequences: the CUDA-core kernel handles the slot bookkeeping
        return launch_prefill_simt(p, D, C, DSLA_BF16, s);
    }
    TcParams tp;
    tp.p = p;
    tp.chunk = pair ? C : CM;
    tp.pairs = p.pairs > 1 ? p.pairs : 1;
    plan(a, pair, tp.pairs, &tp.nseg, &tp.cps, &tp.skew8);
    char* wsp = static_cast<char*>(a->workspace);
    tp.ws = pair && tp.nseg > 1 ? reinterpret_cast<float*>(wsp) : nullptr;
    tp.order = nullptr;
    tp.order_here = !pair && wants_order(a) && orders_here(a);
    tp.init = nullptr;
    if (wants_order(a) && !tp.order_here) {
        int* order = reinterpret_cast<int*>(wsp + (pair ? summaries_bytes(a, tp.nseg) : 0));
        launch_seq_order(p.cu_seqlens, p.N, order, s);
        tp.order = order;
    }
    if (pair && tp.nseg > 1 && p.use_initial_state) {
        // The CTA of a sequence's last segment overwrites the slot with the final state; CTAs of earlier segments read the
        // slot as their initial state and nothing orders the two inside the grid: they read a copy taken beforehand.
        float* snap = reinterpret_cast<float*>(wsp + summaries_bytes(a, tp.nseg) + order_bytes(a, true));
        launch_state_snapshot(p, snap, s);
        tp.init = snap;
    }
    CUtensorMap mq, mk, mv, mo;
    if (!make_tile_map(&mq, p.q, a->T_total, p.H, tp.chunk) || !make_tile_map(&mk, p.k, a->T_total, p.H, tp.chunk) ||
        !make_tile_map(&mv, p.v, a->T_total, p.H, tp.chunk) || (!pair && !make_tile_map(&mo, p.o, a->T_total, p.H, tp.chunk)))
        return DSLA_ERR_CUDA;
    const long long units = (long long)p.N * p.H;
    if (2 * units * tp.nseg > 0x7fffffffLL) return DSLA_ERR_UNSUPPORTED;
    if (pair && tp.nseg > 1) {
        const dsla_status rc = launch_summary(mk, mv, tp, s);
        if (rc != DSLA_OK) return rc;
    }
    return pair ? launch_main_pair(mq, mk, mv, tp, tp.nseg > 1, s) : launch_main(mq, mk, mv, mo, tp, s);
}

}  // namespace dsla
