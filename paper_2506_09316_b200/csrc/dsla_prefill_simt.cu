// Chunkwise prefill of the dual-state linear attention layer on CUDA cores, fp32 arithmetic.
// Serves the fp32 configuration (1e-4 tolerance rules out bf16/tf32 tensor-core products) and any
// shape the tensor-core kernel does not cover.  Mathematics (derived from the recurrence of
// Sec. 4.1 and its unrolled score form): inside a chunk with inclusive cumulative log-gates b^i_j,
//     o_j = sum_{s<=j} (q_j.k_s) [gamma e^{b1_j-b1_s} + (1-gamma) e^{b2_j-b2_s}] v_s
//           + gamma e^{b1_j} q_j S^1 + (1-gamma) e^{b2_j} q_j S^2
//     S^i <- e^{b^i_last} S^i + sum_s e^{b^i_last - b^i_s} k_s^T v_s
// Exponents are always differences b_j - b_s <= 0, so nothing overflows.  A gate that is exactly 0
// is not pushed through log(): zero gates are counted (zc) and a factor is 0 whenever a zero gate
// lies between the two tokens, which keeps tokens after the zero exact.
//
// CTA = (sequence, head, 32-column slab of d_v, segment of the sequence).  The chunks of a sequence are a serial chain,
// and a layer of few heads has few slabs: one CTA per slab leaves most of the chip idle (4 heads of 64: 8 CTAs).  The
// segments of a sequence therefore run on the 2, 4 or 8 CTAs of a thread-block cluster.  Every segment but the last
// first accumulates its own state from zero (K and V only) and leaves it, with the product of its gates, in its
// shared memory; after a cluster barrier the initial states are folded out of the summaries through distributed
// shared memory and every CTA runs its chunks.  No scratch in global memory, no second launch.
// 4 heads of 64, T = 512, fp32: 16 us, 106 us with one CTA per slab.  Bound by shared-memory reads, FMA issue and the barriers between
// the steps of a chunk: the 4 x 4 tiles of the update, the scores and the outputs do 8 packed FMAs (two products each) per two
// 16-byte reads.  Scalar FMAs, and output tiles of 4 x 2, took 18; scores behind the fold instead of under its barriers 21.
#include "dsla_internal.cuh"
#include "tc_utils.cuh"

namespace dsla {

namespace {

template <typename T> struct Vec4;
template <> struct Vec4<float> {
    using Raw = float4;
    static __device__ __forceinline__ Raw zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
    static __device__ __forceinline__ Raw load(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ float4 widen(Raw x) { return x; }
};
template <> struct Vec4<__nv_bfloat16> {
    using Raw = uint2;
    static __device__ __forceinline__ Raw zero() { return make_uint2(0u, 0u); }
    static __device__ __forceinline__ Raw load(const __nv_bfloat16* p) { return *reinterpret_cast<const uint2*>(p); }
    static __device__ __forceinline__ float4 widen(Raw u) {
        const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&u.x);
        const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
        return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
    }
};

__device__ __forceinline__ void store_row(float* p, const float2 (&y)[1]) { *reinterpret_cast<float2*>(p) = y[0]; }
__device__ __forceinline__ void store_row(float* p, const float2 (&y)[2]) { *reinterpret_cast<float4*>(p) = make_float4(y[0].x, y[0].y, y[1].x, y[1].y); }
__device__ __forceinline__ void store_row(__nv_bfloat16* p, const float2 (&y)[1]) { *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(y[0].x, y[0].y); }
__device__ __forceinline__ void store_row(__nv_bfloat16* p, const float2 (&y)[2]) {
    const __nv_bfloat162 z[2] = {__floats2bfloat162_rn(y[0].x, y[0].y), __floats2bfloat162_rn(y[1].x, y[1].y)};
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&z[0]), *reinterpret_cast<const uint32_t*>(&z[1]));
}
// Operands of __ffma2_rn: one instruction for two fp32 FMAs, each rounded as fmaf rounds it.
__device__ __forceinline__ float2 lo(const float4& x) { return make_float2(x.x, x.y); }
__device__ __forceinline__ float2 hi(const float4& x) { return make_float2(x.z, x.w); }
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

constexpr int DVS = 32;      // d_v columns per CTA

// Shared memory, in floats: Q, K [C][D], V [C][36], masked scores [C][C+4], states [2][D][36], per-token terms.  The 16-byte
// pieces of a Q or K row are XORed with the row's group of four: in the score loop neighbouring lanes read rows four
// apart, which a padded pitch would put on two banks.
template <int D, int C> struct Layout {
    static constexpr int VP = DVS + 4, CP = C + 4;
    static constexpr int Q = 0, K = Q + C * D, V = K + C * D, P = V + C * VP, S = P + C * CP;
    static constexpr int BB = S + 2 * D * VP;      // [2][C] cumulative log-gate (zeros skipped)
    static constexpr int ROWF = BB + 2 * C;        // [2][C] weight_i * e^{b_j} (0 behind a zero gate)
    static constexpr int WW = ROWF + 2 * C;        // [2][C] e^{b_last - b_s}
    static constexpr int ZC = WW + 2 * C;          // [2][C] zero-gate count, inclusive (int)
    static constexpr int END = ZC + 2 * C;
    static __device__ __forceinline__ int qk(int row, int col) { return row * D + (col ^ (((row >> 2) & 7) << 2)); }      // col: a multiple of 4
};

}  // namespace

// acc[a][columns] += sum_e x[a][e] y[e][columns], tiles of 4 rows and 2 NB columns
template <int NB> __device__ __forceinline__ void tile_fma(float2 (&acc)[4][NB], const float4 (&x)[4], const float2 (&y)[4][NB]) {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const float xe[4] = {x[a].x, x[a].y, x[a].z, x[a].w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[a][b] = __ffma2_rn(both(xe[e]), y[e][b], acc[a][b]);
    }
}
__device__ __forceinline__ void load_row(const float* p, float2 (&y)[1]) { y[0] = *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void load_row(const float* p, float2 (&y)[2]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    y[0] = lo(x); y[1] = hi(x);
}

// 4 D threads.  In the state update a thread owns a 4 x 4 tile of one state (in registers across the chunk loop, with a
// copy in shared memory for the readout); in the readout two neighbouring lanes share a tile of the output, one
// per state.  Q K^T is recomputed per slab (D / 32 times).  D = 64: two CTAs per SM (16 heads, T = 512: 45 us with one).
template <int D, int C, typename T>
__global__ void __launch_bounds__(4 * D, D == 64 ? 2 : 1) prefill_simt_kernel(const PrefillParams p, const int segs) {
    using L = Layout<D, C>;
    using V4 = Vec4<T>;
    constexpr int SLABS = D / DVS, VP = L::VP, CP = L::CP, NT = 4 * D;
    constexpr int SPLIT = D / 64;            // lanes that share a score tile
    constexpr int NB = 2 / SPLIT, MW = 2 * NB;      // columns of an output tile, in pairs and in all
    extern __shared__ __align__(16) float smem[];
    float *Qs = smem + L::Q, *Ks = smem + L::K, *Vs = smem + L::V, *Ps = smem + L::P, *Ss = smem + L::S;
    float *bb = smem + L::BB, *rowf = smem + L::ROWF, *ww = smem + L::WW;
    int* zc = reinterpret_cast<int*>(smem + L::ZC);
    __shared__ float a_dec[2], a_seg[2];

    // The launch may overlap the tail of what precedes it in the stream; nothing is read or written before this wait.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x;
    const int seg = blockIdx.x % segs;       // rank in the cluster
    const int slab = (blockIdx.x / segs) % SLABS;
    const int h = (blockIdx.x / (segs * SLABS)) % p.H;
    const int n = blockIdx.x / (segs * SLABS * p.H);
    const int t_begin = p.cu_seqlens ? p.cu_seqlens[n] : n * p.T;
    const int t_end = p.cu_seqlens ? p.cu_seqlens[n + 1] : (n + 1) * p.T;
    const int len = t_end - t_begin;
    const int slot = p.slots ? p.slots[n] : n;
    if (slot < 0 || slot >= p.num_slots) return;
    if (len <= 0 && p.use_initial_state) return;  // nothing to do, slot untouched
    const int col0 = slab * DVS;
    const int nchunks = (len + C - 1) / C, per = (nchunks + segs - 1) / segs;
    const int c_begin = min(seg * per, nchunks), c_end = min(c_begin + per, nchunks);

    // state tile of this thread
    const int si = tid / (2 * D);
    const int k0 = ((tid % (2 * D)) >> 3) * 4, n0 = (tid & 7) * 4;
    float* G = p.state + (((size_t)slot * 2 + si) * p.H + h) * (size_t)(D * D) + (size_t)k0 * D + col0 + n0;
    float* Sme = Ss + (si * D + k0) * VP + n0;
    float s[4][4];

    const float gam = p.gamma[h];
    const float W1 = gam * p.scale, W2 = (1.f - gam) * p.scale;
    const T* qg = reinterpret_cast<const T*>(p.q);
    const T* kg = reinterpret_cast<const T*>(p.k);
    const T* vg = reinterpret_cast<const T*>(p.v);
    T* og = reinterpret_cast<T*>(p.o);

    // One chunk ahead in registers: the loads of the next chunk are in flight while this one is computed.
    constexpr int NQ = (C * (D / 4) + NT - 1) / NT, NV = (C * (DVS / 4) + NT - 1) / NT;
    typename V4::Raw rq[NQ], rk[NQ], rv[NV];
    float rg[C > 32 ? 2 : 1];
    auto fetch = [&](int c, bool with_q) {
        const int c0 = c * C, valid = min(C, len - c0);
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int idx = tid + i * NT, row = idx / (D / 4);
            rq[i] = V4::zero(); rk[i] = V4::zero();
            if (row < valid) {
                const size_t off = ((size_t)(t_begin + c0 + row) * p.H + h) * D + (idx % (D / 4)) * 4;
                if (with_q) rq[i] = V4::load(qg + off);
                rk[i] = V4::load(kg + off);
            }
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int idx = tid + i * NT, row = idx / (DVS / 4);
            rv[i] = V4::zero();
            if (row < valid) rv[i] = V4::load(vg + ((size_t)(t_begin + c0 + row) * p.H + h) * D + col0 + (idx % (DVS / 4)) * 4);
        }
        if (tid < 64) {
            constexpr int PER = C >= 32 ? C / 32 : 1;
            const float* gp = (tid >> 5) == 0 ? p.g_hist : p.g_rec;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                const int j = (tid & 31) * PER + e;
                rg[e] = j < valid ? gp[(size_t)(t_begin + c0 + j) * p.H + h] : 1.f;
            }
        }
    };
    // Registers -> shared memory (rows past the end of the sequence are zeros), then the per-token decay terms.
    auto stage = [&](bool with_q) {
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int idx = tid + i * NT, row = idx / (D / 4), c = (idx % (D / 4)) * 4;
            if (row < C) {
                if (with_q) *reinterpret_cast<float4*>(Qs + L::qk(row, c)) = V4::widen(rq[i]);
                *reinterpret_cast<float4*>(Ks + L::qk(row, c)) = V4::widen(rk[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int idx = tid + i * NT, row = idx / (DVS / 4);
            if (row < C) *reinterpret_cast<float4*>(Vs + row * VP + (idx % (DVS / 4)) * 4) = V4::widen(rv[i]);
        }
        // ---- inclusive scan of log-gates (fp64 accumulation) and of the zero-gate count
        if (tid < 64) {
            constexpr int PER = C >= 32 ? C / 32 : 1;
            const int i = tid >> 5, lane = tid & 31;
            double lg[PER];
            int zz[PER];
            double run = 0.0;
            int zrun = 0;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                const float g = rg[e];
                const bool zero = !(g > 0.f);
                run += zero ? 0.0 : (double)logf(g);
                zrun += zero ? 1 : 0;
                lg[e] = run;
                zz[e] = zrun;
            }
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const double up = __shfl_up_sync(0xffffffffu, run, off);
                const int zup = __shfl_up_sync(0xffffffffu, zrun, off);
                if (lane >= off) { run += up; zrun += zup; }
            }
            const double excl = run - lg[PER - 1], last = __shfl_sync(0xffffffffu, run, 31);
            const int zexcl = zrun - zz[PER - 1], zl = __shfl_sync(0xffffffffu, zrun, 31);
            const float bl = (float)last, Wi = i == 0 ? W1 : W2;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                const int j = lane * PER + e;
                if (j < C) {
                    const float b = (float)(excl + lg[e]);
                    const int z = zexcl + zz[e];
                    bb[i * C + j] = b;
                    zc[i * C + j] = z;
                    rowf[i * C + j] = z == 0 ? Wi * expf(b) : 0.f;
                    ww[i * C + j] = z == zl ? expf(bl - b) : 0.f;
                }
            }
            if (lane == 0) a_dec[i] = zl == 0 ? expf(bl) : 0.f;
        }
    };
    // S <- a S + (K (.) w)^T V on this thread's tile
    auto update = [&]() {
        float2 u[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a) u[a][0] = u[a][1] = both(0.f);
        const float* w = ww + si * C;
#pragma unroll 4
        for (int t0 = 0; t0 < C; t0 += 4) {
            const float4 w4 = *reinterpret_cast<const float4*>(w + t0);
            const float we[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 kv = *reinterpret_cast<const float4*>(Ks + L::qk(t0 + e, k0));
                const float4 vv = *reinterpret_cast<const float4*>(Vs + (t0 + e) * VP + n0);
                const float ka[4] = {kv.x * we[e], kv.y * we[e], kv.z * we[e], kv.w * we[e]};
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    u[a][0] = __ffma2_rn(both(ka[a]), lo(vv), u[a][0]);
                    u[a][1] = __ffma2_rn(both(ka[a]), hi(vv), u[a][1]);
                }
            }
        }
        const float ad = a_dec[si];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) s[a][b] = fmaf(ad, s[a][b], (b & 1) ? u[a][b >> 1].y : u[a][b >> 1].x);
    };
    auto publish = [&]() {      // the tile -> its place in shared memory
#pragma unroll
        for (int a = 0; a < 4; ++a) *reinterpret_cast<float4*>(Sme + a * VP) = make_float4(s[a][0], s[a][1], s[a][2], s[a][3]);
    };

#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) s[a][b] = 0.f;
    // ---- masked scores: 4 x 4 tiles of the lower triangle, tile t of row group r is number r (r + 1) / 2 + t
    auto scores = [&]() {
        constexpr int TILES = (C / 4) * (C / 4 + 1) / 2;
        for (int it = tid; it < ((TILES * SPLIT + 31) & ~31); it += NT) {
            const int tile = min(it / SPLIT, TILES - 1), part = it % SPLIT;
            int r = (int)((sqrtf(8.f * (float)tile + 1.f) - 1.f) * 0.5f);
            if (r * (r + 1) / 2 > tile) --r;
            if ((r + 1) * (r + 2) / 2 <= tile) ++r;
            const int j0 = 4 * r, s0 = 4 * (tile - r * (r + 1) / 2);
            float2 acc2[4][4];      // sums over even and odd columns
            float acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc2[a][b] = both(0.f);
#pragma unroll 2
            for (int kk = 4 * part; kk < D; kk += 4 * SPLIT) {
                float4 qv[4], kv[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) qv[a] = *reinterpret_cast<const float4*>(Qs + L::qk(j0 + a, kk));
#pragma unroll
                for (int b = 0; b < 4; ++b) kv[b] = *reinterpret_cast<const float4*>(Ks + L::qk(s0 + b, kk));
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        acc2[a][b] = __ffma2_rn(lo(qv[a]), lo(kv[b]), acc2[a][b]);
                        acc2[a][b] = __ffma2_rn(hi(qv[a]), hi(kv[b]), acc2[a][b]);
                    }
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = acc2[a][b].x + acc2[a][b].y;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (SPLIT > 1) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) acc[a][b] += __shfl_xor_sync(0xffffffffu, acc[a][b], 1);
                }
                if (part == 0) *reinterpret_cast<float4*>(Ps + (j0 + a) * CP + s0) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
            }
        }
    };
    // ---- decay mask: a thread keeps to one column, four rows at a time, so that the loads and exponentials of four elements overlap
    // (one element after the other: 6800 cycles)
    auto mask = [&]() {
        constexpr int JS = NT / C;      // rows apart
        const int t = tid % C;
        const float b1 = bb[t], b2 = bb[C + t];
        const int z1 = zc[t], z2 = zc[C + t];
#pragma unroll 1
        for (int j0 = tid / C; j0 < C; j0 += 4 * JS) {
            if (t > ((j0 + 3 * JS) | 3)) continue;
            float x[4], m[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = min(j0 + e * JS, C - 1);
                x[e] = Ps[j * CP + t];
                const float d1 = zc[j] == z1 ? expf(bb[j] - b1) : 0.f;
                const float d2 = zc[C + j] == z2 ? expf(bb[C + j] - b2) : 0.f;
                m[e] = t <= j ? W1 * d1 + W2 * d2 : 0.f;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = j0 + e * JS;
                if (j < C && t <= (j | 3)) Ps[j * CP + t] = x[e] * m[e];
            }
        }
    };
    bool ahead = false;       // the segment's first chunk is in shared memory, its masked scores too
    if (segs > 1) {
        // ---- summary of this segment, left in Ss and a_seg for the later segments.  The first chunk's scores need no state: they and
        // their mask are computed while the cluster barriers on both sides of the fold complete.
        ahead = c_begin < c_end;
        const bool only = c_end - c_begin == 1;      // the summary's last chunk is the first of the second pass
        if (c_end < nchunks) {
            float as = 1.f;
            fetch(c_begin, only);
            for (int c = c_begin; c < c_end; ++c) {
                stage(only);
                __syncthreads();
                if (c + 1 < c_end) fetch(c + 1, false);
                else if (!only) fetch(c_begin, true);
                update();
                as *= a_dec[si];
                __syncthreads();
            }
            publish();
            if (tid % (2 * D) == 0) a_seg[si] = as;
        } else if (ahead) {
            fetch(c_begin, true);
        }
        tc::cluster_arrive();
        if (ahead) {
            if (!only || c_end == nchunks) { stage(true); __syncthreads(); }
            if (!only) fetch(c_begin + 1, true);
            scores();
            __syncthreads();
        }
        tc::cluster_wait();
        // ---- initial states: the slot (or zero) pushed through the earlier segments.  Each CTA does this for its share of the
        // elements and for every segment: it reads the share out of all summaries and writes the initial states over them, so
        // every CTA reads and writes 1 / segs of what a fold per segment would pull from the first CTAs of the cluster.
        for (int f = seg * (2 * D * 8 / segs) + tid; f < (seg + 1) * (2 * D * 8 / segs); f += NT) {
            const int fi = f / (D * 8), k = (f / 8) % D, c = (f & 7) * 4;
            const float* slot_at = p.state + (((size_t)slot * 2 + fi) * p.H + h) * (size_t)(D * D) + (size_t)k * D + col0 + c;
            float4 x = p.use_initial_state ? *reinterpret_cast<const float4*>(slot_at) : make_float4(0.f, 0.f, 0.f, 0.f);
            const uint32_t at = tc::smem_u32(Ss + (fi * D + k) * VP + c), a_at = tc::smem_u32(&a_seg[fi]);
            float4 u[7];
            float as[7];
#pragma unroll
            for (int e = 0; e < 7; ++e)
                if (e < segs - 1) {
                    u[e] = tc::ld_cluster_f32x4(tc::map_to_cta(at, (uint32_t)e));
                    as[e] = tc::ld_cluster_f32(tc::map_to_cta(a_at, (uint32_t)e));
                }
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (e < segs) {
                    tc::st_cluster_f32x4(tc::map_to_cta(at, (uint32_t)e), x.x, x.y, x.z, x.w);
                    // (segments behind the sequence's last chunk have no summary, and nobody uses what they would start from)
                    if (e < 7) { x.x = fmaf(as[e], x.x, u[e].x); x.y = fmaf(as[e], x.y, u[e].y); x.z = fmaf(as[e], x.z, u[e].z); x.w = fmaf(as[e], x.w, u[e].w); }
                }
        }
        tc::cluster_arrive();
        if (ahead) mask();
        tc::cluster_wait();      // the initial states are in place; every read of the slot is done
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float4 x = *reinterpret_cast<const float4*>(Sme + a * VP);
            s[a][0] = x.x; s[a][1] = x.y; s[a][2] = x.z; s[a][3] = x.w;
        }
        if (c_begin >= c_end && !(seg == 0 && nchunks == 0)) return;
    } else if (p.use_initial_state) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float4 x = *reinterpret_cast<const float4*>(G + (size_t)a * D);
            s[a][0] = x.x; s[a][1] = x.y; s[a][2] = x.z; s[a][3] = x.w;
        }
    }
    if (!ahead && c_begin < c_end) fetch(c_begin, true);
    for (int c = c_begin; c < c_end; ++c) {
        const int c0 = c * C, valid = min(C, len - c0);
        if (!ahead) {
            publish();
            stage(true);
            __syncthreads();
            if (c + 1 < c_end) fetch(c + 1, true);
            scores();
            __syncthreads();
            mask();
        }
        ahead = false;
        __syncthreads();
        // ---- outputs: tiles of 4 rows x 4 columns (x 2 when D = 128), shared by two lanes, one per state, which also take turns in the
        // columns of P
        for (int it = tid; it < (C / 4) * (DVS / MW) * 2; it += NT) {
            const int st = it & 1, tile = it >> 1;
            const int j0 = (tile / (DVS / MW)) * 4, m0 = (tile % (DVS / MW)) * MW;
            float2 acc[4][NB];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) acc[a][b] = both(0.f);
            const float* S = Ss + st * D * VP + m0;
#pragma unroll 2
            for (int kk = 0; kk < D; kk += 4) {
                float4 qv[4];
                float2 x[4][NB];
#pragma unroll
                for (int a = 0; a < 4; ++a) qv[a] = *reinterpret_cast<const float4*>(Qs + L::qk(j0 + a, kk));
#pragma unroll
                for (int e = 0; e < 4; ++e) load_row(S + (kk + e) * VP, x[e]);
                tile_fma(acc, qv, x);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) acc[a][b] = __fmul2_rn(both(rowf[st * C + j0 + a]), acc[a][b]);
            for (int t = 4 * st; t < j0 + 4; t += 8) {  // masked scores are 0 beyond the diagonal tile
                float4 pv[4];
                float2 x[4][NB];
#pragma unroll
                for (int a = 0; a < 4; ++a) pv[a] = *reinterpret_cast<const float4*>(Ps + (j0 + a) * CP + t);
#pragma unroll
                for (int e = 0; e < 4; ++e) load_row(Vs + (t + e) * VP + m0, x[e]);
                tile_fma(acc, pv, x);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    acc[a][b].x += __shfl_xor_sync(0xffffffffu, acc[a][b].x, 1);
                    acc[a][b].y += __shfl_xor_sync(0xffffffffu, acc[a][b].y, 1);
                }
                const int j = j0 + a;
                if (a / 2 == st && j < valid) store_row(og + ((size_t)(t_begin + c0 + j) * p.H + h) * D + col0 + m0, acc[a]);
            }
        }
        if (c_end < nchunks && c + 1 == c_end) break;      // not the last segment: its final state is nobody's
        update();
        __syncthreads();  // every read of this chunk's tiles and of the old state copy is done
    }
    if (c_end == nchunks) {
#pragma unroll
        for (int a = 0; a < 4; ++a) *reinterpret_cast<float4*>(G + (size_t)a * D) = make_float4(s[a][0], s[a][1], s[a][2], s[a][3]);
    }
}

// Segments per sequence: while a doubling still fits on the device at once (two CTAs per SM with D = 64, one with 128) (the extra pass over K and V for the summaries costs
// less than idle SMs) and some segment has more than one chunk of the longest sequence (three chunks take four segments,
// one of them empty: T = 130, 2 heads of 64: 34 us with two).
static int plan_segments(long long units, int max_chunks, int per_sm) {
    const int room = per_sm * sm_count();
    int segs = 1;
    while (segs < 8 && units * segs * 2 <= room && segs < max_chunks) segs *= 2;
    return segs;
}

template <int D, int C, typename T>
static dsla_status launch_one(const PrefillParams& p, cudaStream_t s) {
    constexpr size_t smem = sizeof(float) * Layout<D, C>::END;
    if (cudaFuncSetAttribute(prefill_simt_kernel<D, C, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return DSLA_ERR_CUDA;
    const long long units = (long long)p.N * p.H * (D / DVS);
    const int segs = plan_segments(units, p.max_chunks, D == 64 ? 2 : 1);
    if (units * segs > 0x7fffffffLL) return DSLA_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * segs));
    cfg.blockDim = dim3(4 * D);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)segs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = segs > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, prefill_simt_kernel<D, C, T>, p, segs) != cudaSuccess) return DSLA_ERR_CUDA;
    count_launch();
    return cudaGetLastError() == cudaSuccess ? DSLA_OK : DSLA_ERR_CUDA;
}

template <int D, typename T>
static dsla_status launch_chunk(const PrefillParams& p, int chunk, cudaStream_t s) {
    switch (chunk) {
        case 16: return launch_one<D, 16, T>(p, s);
        case 32: return launch_one<D, 32, T>(p, s);
        case 64: return launch_one<D, 64, T>(p, s);
        default: return DSLA_ERR_UNSUPPORTED;
    }
}

dsla_status launch_prefill_simt(const PrefillParams& p, int d, int chunk, dsla_dtype dt, cudaStream_t s) {
    if (p.N == 0) return DSLA_OK;
    if (d == 128 && dt == DSLA_BF16) return launch_chunk<128, __nv_bfloat16>(p, chunk, s);
    if (d == 128 && dt == DSLA_F32) return launch_chunk<128, float>(p, chunk, s);
    if (d == 64 && dt == DSLA_BF16) return launch_chunk<64, __nv_bfloat16>(p, chunk, s);
    if (d == 64 && dt == DSLA_F32) return launch_chunk<64, float>(p, chunk, s);
    return DSLA_ERR_UNSUPPORTED;
}

}  // namespace dsla
