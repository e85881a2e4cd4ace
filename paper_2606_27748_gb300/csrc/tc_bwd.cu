// Backward of RFF linear attention on the tensor cores (tcgen05).
//
// Gradient of L = sum(dout * out) for Eq. (linear att).  With unscaled features phi'
// (the M^{-1/2} cancels), den' = M den, g_i = dout_i / den'_i, c_i = -(dout_i . out_i)/den'_i:
//   dA_ij    = g_i . v_j + c_i                      (j <= i when causal)
//   dphi(q_i) = sum_j dA_ij phi(k_j)   = [intra-chunk] + S_i g_i + c_i z_i
//   dphi(k_j) = sum_i dA_ij phi(q_i)   = [intra-chunk] + R_j v_j + r_j
//   dv_j      = sum_i A_ij g_i         = [intra-chunk] + R_j^T phi(k_j)
// with S = sum phi(k) v^T, z = sum phi(k) (forward running sums) and R = sum phi(q) g^T,
// r = sum c phi(q) (reverse running sums), then through the feature map (Eq. phi_n /
// phi_non) by the chain rule: dx = da W, dW += da^T x.
//
// Every term splits over feature groups (64 frequencies = 128 features), and A enters dv
// linearly, so one CTA handles one (sequence, group) pair and the group results are summed.
// With two groups (M = 128) the two CTAs of a (pass, sequence) form a cluster: each chunk,
// CTA r finishes rows 64r..64r+63 of dq (pass F) or dk and dv (pass R): it sends its
// fp32 partial rows of the other half to the partner (staged in its own shared memory, one
// bulk copy into a region the partner has declared free), adds the partner's partial to its
// own rows and stores bf16.  dW goes through per-(pass, sequence, group) partials reduced
// over the batch in a fixed order.  Pass F runs the chunks forward (dq and the q part of
// dW, state S, z), pass R runs them backward (dk, dv and the k part of dW, state R, r); the
// two are independent and run as the two halves of one grid, pass R (the longer) first.
//
// Norm prefactor (Sec. 3.2, optional): with key weights w_j = exp(|k_j|^2 exp(-tau)) (kw,
// one pass over k before this kernel), phi(k) is stored weighted, so S, z, A and dv come
// out weighted and T_D holds the gradient with respect to the weighted features.  In pass
// R the chain rule then needs dphi(k) = w dphi~(k) (the stationary feature tile already
// carries w; the nonstationary recomputation multiplies by it), s_j = phi~(k_j).dphi~(k_j)
// adds 2 exp(-tau) s_j k_j to dk_j (folded into the same row adds) and -ln(w_j) s_j to
// dtau (per-CTA slots, reduced with dW in a fixed order).
//
// Roles: warp 16 (one elected lane per operation) loads the tiles by TMA and issues every MMA;
// warp 17 tells the partner CTA when its copies have landed; 16 compute warps (four per
// tensor-memory lane quadrant, each a quarter of the columns) do the CUDA-core work and never meet at a CTA barrier: each hand-off is one
// arrival per warp on an mbarrier the issuer waits for, and the MMAs' completion, which
// follows every warp's arrival, releases the compute warps again.  Work that does not depend
// on a running MMA group (masks, row stores, the next chunk's g tile, the state snapshot)
// is placed while it runs, and groups are ordered so that what the compute warps need first
// is committed first.  The phases of a chunk, [MMA group] / compute:
//   causal F   g / [q and k projections, dA] / phi(k), mask dA / [dphi(q)] [S, z] / chain
//              rule / [dq, dW] / snapshot, dq rows
//   causal R   g / [q and k projections, dA] / phi(q), phi(k) / [A] / mask dA, mask A /
//              [dphi(k), dv] [R, r] / chain rule / [dk, dW] / dv rows, snapshot, dk rows
//   kState     [projection of the next chunk] / features, g / [state]
//   kGrad F    [q projection, dphi(q)] / chain rule, next chunk's g / [dq, dW] / dq rows
//   kGrad R    [k projection, dphi(k)] / phi(k), chain rule / [dv, dk, dW] / dv, dk rows
// The phases of a chunk depend on one another (an SM holds one CTA's tensor memory), so the
// length of this chain bounds the kernel, not DRAM (14%) or the tensor pipe (18%): a chunk of s M128
// takes about 15 us in F and R together, from 19.4 with all threads meeting at CTA barriers
// and thread 0 issuing; measured forward and backward: s B8 H12 N8192 M128 2.16 -> 1.57 ms,
// n non-causal B32 H8 N4000 M64 1.30 -> 0.89 ms.
// Every wait is bounded.  Tiles of the following chunks are loaded as soon as the region
// each one occupies is free (two buffers where the pass leaves room).
//
// Exchange regions (staging -> the partner's receive region; each free when it is used):
//   causal   pass F  dq: PQ -> DA2 (s), PK (n)   pass R  dv: PQ -> DA2, dk: PK -> XR (s), PQ+16K -> PK (n)
//   kGrad    pass F  dq: K  -> PK        pass R  dv: Q  -> DO,  dk: DA2 -> O
//
// Tensor memory (512 columns): [0,128) T_P: projection of q (causal F and R, kGrad F) or k,
// then (causal) dx (0-63) and dW (64-127); [128,256) T_A: dA, then dv (causal R); kGrad: dx
// (0-63), dv (64-127); [256,384) T_D: projection of k and A (causal), dphi; [384,464) S|z or
// R|r (kGrad n: dW).  kState: T_P and T_A are two projection buffers.
#include <algorithm>
#include <type_traits>

#include "flex_internal.h"
#include "tc_common.cuh"
#include "tc_util.cuh"

namespace flex {
namespace {
using namespace tc;

constexpr int kC = 128;
constexpr int kComputeWarps = 16;  // four per lane quadrant, each a quarter of the columns
constexpr int kThreadsB = 32 * kComputeWarps + 64;  // and the issuer's and the relay's warps
constexpr uint32_t kXBytes = 64 * 64 * 4;  // one exchanged half: 64 rows x 64 fp32
enum { kPassF = 0, kPassR = 1 };
// kCausal: the chunked scans of the causal gradient.  Non-causal (every key for every query):
// kState sums partial states over a range of chunks (pass F: [S | z] = sum phi(k) [v | 1],
// pass R: [R | r] = sum phi(q) [g | c]); kGrad starts from their totals and needs no scan:
// pass F dphi(q) = S g + c z, pass R dphi(k) = R v + r and dv = R^T phi(k).
enum { kCausal = 0, kState = 1, kGrad = 2 };

template <bool NS>
struct BwCfg {
    static constexpr int P = NS ? 128 : 64;  // projection rows (and dW rows) per group
    // shared memory (bytes).  Pass R keeps bf16(dA) in [Q | DA2] and bf16(A) in [DO | O].
    static constexpr uint32_t Q = 0, DA2 = 16384, K = 32768, V = 49152, DO = 65536, O = 81920;
    static constexpr uint32_t GT = 98304;     // g tile [token][dcol], bf16
    static constexpr uint32_t C16 = 114688;   // K-major [16][128 tokens]: ones (F) / c (R)
    static constexpr uint32_t W = 118784;     // this group's projection rows
    static constexpr uint32_t PQ = W + P * 128, PK = PQ + 32768;  // features (then da in place)
    static constexpr uint32_t SN = PK + 32768;     // state snapshot [feature][64 dcol], bf16
    static constexpr uint32_t ZR = SN + 16384;     // z or r [2 chunk parities][128] fp32
    static constexpr uint32_t CROW = ZR + 1024;    // c_t [2 chunk parities][128] fp32
    // s_t partials [4 column quarters][128] fp32; kGrad has a second set behind them, by chunk
    // parity
    static constexpr uint32_t SPART = CROW + 1024;
    // s: a receive block for dk (its W rows take half the space; causal only, so the second
    // set of partials shares its place); n has no room for one
    static constexpr uint32_t XR = NS ? PK : SPART + 2048;
    static constexpr uint32_t BYTES = SPART + 2048 + (NS ? 2048 : 16384);
    static constexpr uint32_t T_P = 0, T_A = 128, T_D = 256, T_S = 384;
    static_assert(BYTES + 1024 <= 232448, "shared memory budget");
};


__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d)
{
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(a), "f"(b),
                 "f"(c), "f"(d)
                 : "memory");
}

// KW: key weights of the norm prefactor given (compile-time; the plain kernel is unchanged);
// CS: CTAs per cluster = frequency groups (1 or 2; 1 for kState, which exchanges nothing);
// MODE: kCausal, kState or kGrad
template <bool NS, bool KW, int CS, int MODE, int PASS>
__device__ __forceinline__ void tc_bwd_body(const CUtensorMap& tmap_q, const CUtensorMap& tmap_k,
    const CUtensorMap& tmap_v, const CUtensorMap& tmap_do, const CUtensorMap& tmap_o, int H,
    int N, int M, int G, const __nv_bfloat16* __restrict__ q,
    const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
    const float* __restrict__ W1, const float* __restrict__ W2,
    const __nv_bfloat16* __restrict__ outp, const float* __restrict__ den,
    const __nv_bfloat16* __restrict__ dout, __nv_bfloat16* __restrict__ dq,
    __nv_bfloat16* __restrict__ dk, __nv_bfloat16* __restrict__ dv, float* dw_part,
    const float* kw, const float* __restrict__ tau, float* dtau_part,
    int units, int nsplit, float* state_part, const float* state_total,
    int* status)
{
    using L = BwCfg<NS>;
    // blocks [0, half): pass R, [half, 2 half): pass F, half = units * nsplit; within a pass
    // idx = (sequence * nsplit + split) * G + group (the groups of a cluster adjacent); the
    // chunks are split into nsplit ranges (causal scans: 1 unless a small batch is cut).
    // Partial slots are indexed by slot = pass * half + idx.
    const int half_grid = units * nsplit;
    const int idx = (int)blockIdx.x % half_grid;
    const int split = (idx / G) % nsplit;
    const int unit = (idx / G / nsplit) * G + idx % G;
    const int slot = PASS * half_grid + idx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sb = smem_u32(sm);
    __shared__ uint32_t tmem_base_sh;
    // tiles landed: tx[buffer] (q, k, v as the mode reads them), tg (dout and out), tv[buffer]
    // (v in kState); compute -> issuer, one arrival
    // per warp: rdy (operands written, tensor memory read), rdyg (the g tile), rdys[buffer]
    // (kState, where a warp may be a chunk ahead of another), srdy (the dk
    // rows taken); fin: every warp's rdy has been seen (kLate); MMA groups complete: m0, m1, mt[buffer]
    __shared__ __align__(8) uint64_t tx[2], tg, tv[3], rdy, rdyg, rdys[2], srdy, fin, m0, m1, mt[2];
    // cluster exchange i (0: dq (F) or dv (R), 1: dk (R)): xready: the partner's receive region
    // is free; xfull: the partner's partial landed (transaction count); xdone: this CTA's
    // partial landed there, so its staging region may be rewritten
    __shared__ __align__(8) uint64_t xready[2], xdone[2], xfull[2];
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wg = warp >> 2, quad = warp & 3, t = 32 * quad + lane;
    const int bh = unit / G, g = unit % G, h = bh % H;
    const size_t base = (size_t)bh * N * 64;
    float* zr = reinterpret_cast<float*>(sm + L::ZR);
    float* crow = reinterpret_cast<float*>(sm + L::CROW);
    float* spart = reinterpret_cast<float*>(sm + L::SPART);
    const float itau = KW ? expf(-tau[h]) : 0.f;
    float dtau_acc = 0.f;

    // ---- set-up: this group's projection rows, zero state, C16 ----
    grid_dep_launch();
    for (int idx = tid; idx < L::P * 8; idx += kThreadsB) {
        const int r = idx >> 3, c = idx & 7, f = 64 * g + (r & 63);
        const float* w1 = W1 + ((size_t)h * M + f) * 64 + c * 8;
        float x[8];
        if (!NS) {
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = w1[e];
        } else {
            const float* w2 = W2 + ((size_t)h * M + f) * 64 + c * 8;
            const float sgn = r < 64 ? 1.f : -1.f;  // U = (W1+W2)/2, V = (W1-W2)/2
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = 0.5f * (w1[e] + sgn * w2[e]);
        }
        st_shared_v4(sb + L::W + swz128(r, c * 8), pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]),
                     pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
    }
    for (int idx = tid; idx < 16384 / 16; idx += kThreadsB) st_shared_v4(sb + L::SN + idx * 16, 0, 0, 0, 0);
    for (int idx = tid; idx < 4096 / 16; idx += kThreadsB) {
        const uint32_t fill = PASS == kPassF ? 0x3F803F80u : 0u;  // ones (z) or zeros (c rows)
        st_shared_v4(sb + L::C16 + idx * 16, fill, fill, fill, fill);
    }
    for (int idx = tid; idx < 256; idx += kThreadsB) zr[idx] = 0.f;
    const int rank = CS > 1 ? (int)cluster_rank() : 0;  // = g
    if (tid == 0) {
        for (uint64_t* b : {&tx[0], &tx[1], &tg, &tv[0], &tv[1], &tv[2], &m0, &m1, &mt[0], &mt[1]})
            mbar_init(b, 1);
        for (uint64_t* b : {&rdy, &rdyg, &rdys[0], &rdys[1], &srdy}) mbar_init(b, kComputeWarps);
        mbar_init(&fin, 1);
        mbar_init(&xready[0], 1);
        mbar_init(&xready[1], 1);
        mbar_init(&xdone[0], 1);
        mbar_init(&xdone[1], 1);
        mbar_init(&xfull[0], 1);
        mbar_init(&xfull[1], 1);
        abort_flag = 0;
        fence_mbar_init();
        if (CS > 1) {  // the first chunk's exchanges
            mbar_arrive_expect_tx(&xfull[0], kXBytes);
            if (PASS == kPassR) mbar_arrive_expect_tx(&xfull[1], kXBytes);
        }
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, 512);
        tmem_relinquish();
    }
    grid_dep_wait();  // the key weights, partial states or totals (set-up needs none of them)
    fence_proxy_async();
    fence_before_sync();
    if (CS > 1)
        cluster_sync();  // the partner's barriers exist before anything arrives on them
    else
        __syncthreads();
    fence_after_sync();
    const uint32_t tm = tmem_base_sh;
    const uint32_t tm_row = tm + ((uint32_t)(32 * quad) << 16);
    // dtau = -sum_j ln(w_j) s_j with s_j = phi~(k_j) . dphi~(k_j) = dL / d ln(w_j).  Scaling
    // every key weight of a sequence by one factor leaves every output row unchanged, so the
    // s_j of a sequence sum to zero and any per-sequence constant may be subtracted from
    // ln(w_j); the log weight of the sequence's first key removes the common part, whose
    // terms would otherwise cancel only to the rounding of the s_j.
    const float lw0 = KW ? logf(kw[(size_t)bh * N]) : 0.f;
    uint32_t ph_xfull[2] = {0, 0};
    const uint32_t partner = (uint32_t)rank ^ 1u;

    // A phase of `bar`, and the tensor-memory accesses ordered after it; `ph` is the caller's
    // parity.  Called by a whole warp (one verdict).
    auto wwait = [&](uint64_t* bar, uint32_t& ph) -> bool {
        const bool ok = bar_wait_w(bar, ph, &abort_flag, status);
        ph ^= 1;
        fence_after_sync();
        return ok;
    };
    // This warp's shared-memory writes are visible to the tensor core and the copies, its
    // tensor-memory accesses done: one arrival.
    auto arrive = [&](uint64_t* bar) {
        fence_proxy_async();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    auto adv = [](uint64_t d, uint32_t bytes) { return d + (bytes >> 4); };
    const uint64_t dQ = sdesc(sb + L::Q, 16, 1024), dK = sdesc(sb + L::K, 16, 1024);
    const uint64_t dV = sdesc(sb + L::V, 16, 1024), dG = sdesc(sb + L::GT, 16, 1024);
    const uint64_t dW = sdesc(sb + L::W, 16, 1024), dWmn = sdesc(sb + L::W, 16384, 1024);
    const uint64_t dPQ = sdesc(sb + L::PQ, 16, 1024), dPK = sdesc(sb + L::PK, 16, 1024);
    const uint64_t dPQmn = sdesc(sb + L::PQ, 16384, 1024), dPKmn = sdesc(sb + L::PK, 16384, 1024);
    const uint64_t dVmn = sdesc(sb + L::V, 16384, 1024), dGmn = sdesc(sb + L::GT, 16384, 1024);
    const uint64_t dQmn = sdesc(sb + L::Q, 16384, 1024), dKmn = sdesc(sb + L::K, 16384, 1024);
    const uint64_t dSN = sdesc(sb + L::SN, 16, 1024), dSNmn = sdesc(sb + L::SN, 16384, 1024);
    const uint64_t dC16 = sdesc(sb + L::C16, 16, 1024);
    const uint64_t dDAmn = sdesc(sb + L::Q, L::DA2 - L::Q, 1024);  // bf16(dA) as [query][key]
    const uint64_t dAmn = sdesc(sb + L::DO, L::O - L::DO, 1024);   // bf16(A)  as [query][key]
    constexpr uint32_t I_PROJ = idesc_bf16(128, L::P, 0, 0);
    constexpr uint32_t I_KK128 = idesc_bf16(128, 128, 0, 0);   // K-major A, K-major B, N=128
    constexpr uint32_t I_KM128 = idesc_bf16(128, 128, 0, 1);   // K-major A, MN-major B, N=128
    constexpr uint32_t I_MM128 = idesc_bf16(128, 128, 1, 1);   // MN-major A and B, N=128
    constexpr uint32_t I_KM64 = idesc_bf16(128, 64, 0, 1);
    constexpr uint32_t I_MM64 = idesc_bf16(128, 64, 1, 1);
    constexpr uint32_t I_M16 = idesc_bf16(128, 16, 1, 0);      // MN-major A, K-major B, N=16

    // projection of a tile into tensor-memory column col
    auto issue_projection = [&](uint64_t dx, uint32_t col) {
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
            wmma_bf16(tm + col, adv(dx, ks * 32), adv(dW, ks * 32), I_PROJ, ks > 0);
    };
    // features of this group into dst (K-major rows) from the projection at column tcol; this
    // thread: row t, frequencies 16 wg .. 16 wg + 15
    auto features = [&](uint32_t dst, uint32_t tcol, bool valid, float wsc) {
        float a[16], w[16], m0, m1 = 0.f;  // m: max |x| per load
        tmem_ld16_maxabs(tm_row + tcol + 16 * wg, a, m0);
        if (NS) tmem_ld16_maxabs(tm_row + tcol + 64 + 16 * wg, w, m1);
        tmem_wait_ld();
        const float mabs = fmaxf(m0, m1);
        if (NS)
            cos_w_args(a, w, mabs);  // w <- cos(w)
        else
            reduce_2pi_if_needed(a, mabs);
        uint32_t pc[8], ps[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float s0, c0, s1, c1;
            __sincosf(a[2 * i], &s0, &c0);
            __sincosf(a[2 * i + 1], &s1, &c1);
            if (NS) {
                mul2x2(c0, c1, s0, s1, w[2 * i], w[2 * i + 1]);
            }
            if (KW) { c0 *= wsc; s0 *= wsc; c1 *= wsc; s1 *= wsc; }
            pc[i] = pack_bf16(c0, c1);
            ps[i] = pack_bf16(s0, s1);
        }
        // Rows past N are zeroed for the totals only.  Elsewhere TMA's zeros make x, v and g (and
        // c) zero in them, so they add nothing to dW or the state R; dA and A are masked; S after
        // the ragged last chunk is not used; their own result rows are not stored.
        if (MODE == kState && __any_sync(0xffffffffu, !valid) && !valid) {
#pragma unroll
            for (int i = 0; i < 8; ++i) pc[i] = ps[i] = 0u;
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t off = swz128(t, (2 * wg + j) * 8);
            st_shared_v4(dst + off, pc[4 * j], pc[4 * j + 1], pc[4 * j + 2], pc[4 * j + 3]);
            st_shared_v4(dst + 16384 + off, ps[4 * j], ps[4 * j + 1], ps[4 * j + 2], ps[4 * j + 3]);
        }
    };
    // Chain rule through the features of this thread's 16 frequencies: dphi from T_D plus
    // the per-feature term zrow * scale; da to the blocks at da0, da1 (s: da and, for the dW
    // MMA, its low part da - bf16(da); n: du | dw).  The cos and sin come from the projection
    // in T_P (TILE false; with phi != 0 the key features are written there as well), or, s
    // in the causal pass R, whose projection is gone by then, from the feature tile at da0,
    // which da replaces (TILE; its features carry the key weight).  wkey: the key weight
    // (pass R with the prefactor, else 1); returns this thread's part of
    // s_t = phi~(k_t) . dphi~(k_t) (pass R with the prefactor, else 0).
    auto feature_backward = [&](auto tile_tag, const float* zrow, uint32_t phi, uint32_t da0, uint32_t da1, float scale,
                                bool valid, float wkey) -> float {
        constexpr bool TILE = decltype(tile_tag)::value;
        static_assert(!(NS && TILE), "n takes cos and sin from the projection");
        float dc[16], ds[16];
        tmem_ld16(tm_row + L::T_D + 16 * wg, dc);
        tmem_ld16(tm_row + L::T_D + 64 + 16 * wg, ds);
        float a[16], w[16], ma = 0.f, mw = 0.f;  // m: max |x| per load
        if (!TILE) tmem_ld16_maxabs(tm_row + L::T_P + 16 * wg, a, ma);
        if (NS) tmem_ld16_maxabs(tm_row + L::T_P + 64 + 16 * wg, w, mw);
        tmem_wait_ld();
        if (NS)
            reduce_2pi_if_needed(a, w, fmaxf(ma, mw));
        else if (!TILE)
            reduce_2pi_if_needed(a, ma);
        const bool wt = KW && PASS == kPassR;
        float sdot = 0.f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {  // eight frequencies: one 16-byte store per block
            const uint32_t off = swz128(t, (2 * wg + j) * 8);
            uint32_t cp[4], sp[4];  // cos and sin pairs of the tile
            if (TILE) {
                const uint4 c4 = *reinterpret_cast<const uint4*>(sm + (da0 - sb) + off);
                const uint4 s4 = *reinterpret_cast<const uint4*>(sm + (da1 - sb) + off);
                cp[0] = c4.x; cp[1] = c4.y; cp[2] = c4.z; cp[3] = c4.w;
                sp[0] = s4.x; sp[1] = s4.y; sp[2] = s4.z; sp[3] = s4.w;
            }
            uint32_t o1[4], o2[4], pc[4], ps[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float r1[2], r2[2], fc[2], fs[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int fi = 8 * j + 2 * i + e, zi = 16 * wg + fi;
                    const float dphic = fmaf(scale, zrow[zi], dc[fi]);
                    const float dphis = fmaf(scale, zrow[64 + zi], ds[fi]);
                    float su, cu, sw = 0.f, cw = 1.f;
                    if (TILE) {
                        cu = __uint_as_float(e ? cp[i] & 0xFFFF0000u : cp[i] << 16);
                        su = __uint_as_float(e ? sp[i] & 0xFFFF0000u : sp[i] << 16);
                    } else {
                        __sincosf(a[fi], &su, &cu);
                        if (NS) __sincosf(w[fi], &sw, &cw);
                        if (wt && !NS) {
                            su *= wkey;
                            cu *= wkey;
                        }
                    }
                    fc[e] = NS ? cu * cw : cu;
                    fs[e] = NS ? su * cw : su;
                    r1[e] = fc[e] * dphis - fs[e] * dphic;
                    r2[e] = NS ? -sw * (cu * dphic + su * dphis) : 0.f;
                    if (wt) {
                        sdot = fmaf(fc[e], dphic, fmaf(fs[e], dphis, sdot));
                        if (NS) {
                            r1[e] *= wkey;
                            r2[e] *= wkey;
                            fc[e] *= wkey;
                            fs[e] *= wkey;
                        }
                    }
                    // (not needed, but ptxas spills 28 bytes instead of 8 without it: 921 -> 910
                    // us for the training step of B32 H8 N4000 M64)
                    if (NS && MODE == kGrad && !valid) r1[e] = r2[e] = fc[e] = fs[e] = 0.f;
                }
                o1[i] = pack_bf16(r1[0], r1[1]);
                if (!NS) {
                    // s: the sin half of the tile (unused by dx = da W) carries da - bf16(da),
                    // so the dW MMA (all 128 rows) gets da to ~2^-17: rows 64-127 of dW are
                    // added to rows 0-63 in the reduction
                    r2[0] = r1[0] - __uint_as_float(o1[i] << 16);
                    r2[1] = r1[1] - __uint_as_float(o1[i] & 0xFFFF0000u);
                }
                o2[i] = pack_bf16(r2[0], r2[1]);
                pc[i] = pack_bf16(fc[0], fc[1]);
                ps[i] = pack_bf16(fs[0], fs[1]);
            }
            st_shared_v4(da0 + off, o1[0], o1[1], o1[2], o1[3]);
            st_shared_v4(da1 + off, o2[0], o2[1], o2[2], o2[3]);
            if (!TILE && phi) {
                st_shared_v4(phi + off, pc[0], pc[1], pc[2], pc[3]);
                st_shared_v4(phi + 16384 + off, ps[0], ps[1], ps[2], ps[3]);
            }
        }
        if (!valid) sdot = 0.f;
        return NS ? sdot * wkey : sdot;  // n: phi~ = w cos u cos w, w sin u cos w
    };
    // dx = da W into column T_X, dW = da^T x into T_DW: n in the causal modes: this chunk's;
    // s: summed over the chunks beside the projection (T_P[64,128)); n in kGrad: summed in
    // T_S, which holds no state without a scan.  da's blocks lie at a0, a1; x is MN-major.
    constexpr bool kDwPerChunk = NS && MODE != kGrad;
    // kLate (causal s with a partner): dx and dv lie where the next chunk's first MMAs do not
    // write, so its rows can be finished late: dx beside the key projection, and in pass R dv
    // in place of the running dW, which is then summed per chunk like n's (dw_per_chunk).
    constexpr bool kLate = !NS && MODE == kCausal && CS == 2;
    const bool dw_per_chunk = kDwPerChunk || (kLate && PASS == kPassR);
    constexpr uint32_t T_X = MODE == kGrad ? L::T_A : kLate ? L::T_D + 64 : L::T_P;
    const uint32_t T_DW = NS && MODE == kGrad        ? L::T_S
                          : kLate && PASS == kPassR ? L::T_A + 64
                                                    : L::T_P + 64;
    constexpr uint32_t T_DV = MODE == kGrad ? L::T_A + 64 : kLate ? L::T_P + 64 : L::T_A;
    auto issue_back = [&](uint32_t a0, uint32_t a1, uint64_t d_x_mn, bool first) {
        const uint64_t dA0 = sdesc(a0, 16, 1024), dA1 = sdesc(a1, 16, 1024);
        const uint64_t dAm = sdesc(a0, a1 - a0, 1024);
#pragma unroll
        for (int ks = 0; ks < (NS ? 8 : 4); ++ks)  // K = P rows of W (s: the da block only)
            wmma_bf16(tm + T_X, adv(ks < 4 ? dA0 : dA1, (ks & 3) * 32), adv(dWmn, ks * 2048), I_KM64,
                     ks > 0);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            wmma_bf16(tm + T_DW, adv(dAm, ks * 2048), adv(d_x_mn, ks * 2048), I_MM64,
                     (dw_per_chunk ? ks > 0 : (!first || ks > 0)) ? 1u : 0u);
    };
    // dW rows of this chunk (lane = row of this group's projection) into the partial slot
    // (all 128 rows; s: rows 64-127 hold the low part's contribution), 16 columns a thread.
    // A slot is stored as [16 column quads][128 rows][4], so a warp's accesses are contiguous.
    // After the first chunk by reductions: each address is this thread's alone, so they apply
    // in its program order (repeatable), and no thread waits for the old values (a load, add
    // and store of rows took 6-7 of the 20-27 thousand cycles of a chunk).
    auto dw_accumulate = [&](bool first) {
        float v_[16];
        tmem_ld16(tm_row + T_DW + 16 * wg, v_);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float* dst = dw_part + ((size_t)slot * 16 + 4 * wg + j) * 512 + 4 * t;
            if (first)
                *reinterpret_cast<float4*>(dst) =
                    make_float4(v_[4 * j], v_[4 * j + 1], v_[4 * j + 2], v_[4 * j + 3]);
            else
                red_add_v4(dst, v_[4 * j], v_[4 * j + 1], v_[4 * j + 2], v_[4 * j + 3]);
        }
    };
    // state snapshot [feature][64] bf16 + column 64 (z or r) fp32, from T_S (lane = feature)
    auto snapshot = [&](float* zrow) {
        float s_[16], zz[16];
        tmem_ld16(tm_row + L::T_S + 16 * wg, s_);
        if (wg == 0) tmem_ld16(tm_row + L::T_S + 64, zz);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 2; ++j)
            st_shared_v4(sb + L::SN + swz128(t, (2 * wg + j) * 8),
                         pack_bf16(s_[8 * j], s_[8 * j + 1]), pack_bf16(s_[8 * j + 2], s_[8 * j + 3]),
                         pack_bf16(s_[8 * j + 4], s_[8 * j + 5]), pack_bf16(s_[8 * j + 6], s_[8 * j + 7]));
        if (wg == 0) zrow[t] = zz[0];
    };
    // ---- cluster exchange of the dq / dk / dv partials (CS = 2) ----
    // This CTA's receive region of exchange xi is free for the partner's next copies (issuer).
    auto signal_ready = [&](int xi) {
        if (CS > 1 && elect_one()) mbar_arrive_cluster(mapa(smem_u32(&xready[xi]), partner));
    };
    // An exchange block holds 64 rows x 64 fp32 as eight pieces of 2 KB, one per warp (two row
    // halves x four column quarters): byte offset of 16-byte chunk j (0-3) of this lane's row
    // in its warp's piece (64-byte rows, chunks swizzled by row).
    const uint32_t piece = 2048u * (uint32_t)(4 * (quad & 1) + wg);
    auto xoff = [&](int j) {
        return piece + 64u * lane + (((uint32_t)j ^ ((uint32_t)(lane >> 1) & 3u)) << 4);
    };
    auto store_quarter = [&](__nv_bfloat16* out, int t0, const float (&v_)[16]) {
        store_32b(out + base + (size_t)(t0 + t) * 64 + 16 * wg,
                  make_uint4(pack_bf16(v_[0], v_[1]), pack_bf16(v_[2], v_[3]), pack_bf16(v_[4], v_[5]),
                             pack_bf16(v_[6], v_[7])),
                  make_uint4(pack_bf16(v_[8], v_[9]), pack_bf16(v_[10], v_[11]),
                             pack_bf16(v_[12], v_[13]), pack_bf16(v_[14], v_[15])));
    };
    // Rows of the [128 x 64] block at tensor-memory column `col` -> bf16 rows of `out` for the
    // chunk at t0.  kcoef != 0 adds kcoef * k_t (the prefactor's dk term; k from the tile at
    // ktile).  Without a partner every row is stored.  With one, a warp whose rows the partner
    // finishes stages its piece and copies it to the partner's `recv`, once the partner has
    // signalled that the region is free; this CTA's own rows (64 rank .. + 63) stay in tensor memory (written back when the dk term was
    // added) for finalize_rows.  (Eight copies of 2 KB from the warps overlap; one copy of
    // 16 KB by the issuer, after every warp had staged, took 3 thousand cycles to land.)
    uint32_t ph_xready[2] = {0, 0};
    auto take_rows = [&](__nv_bfloat16* out, uint32_t col, int t0, bool valid, float kcoef,
                         uint32_t ktile, int xi, uint32_t stage, uint32_t recv) -> bool {
        float v_[16];
        tmem_ld16(tm_row + col + 16 * wg, v_);
        tmem_wait_ld();
        if (KW && kcoef != 0.f) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint4 k4 = *reinterpret_cast<const uint4*>(sm + ktile + swz128(t, 16 * wg + 8 * j));
                const uint32_t kw4[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v_[8 * j + 2 * e] = fmaf(kcoef, __uint_as_float(kw4[e] << 16), v_[8 * j + 2 * e]);
                    v_[8 * j + 2 * e + 1] =
                        fmaf(kcoef, __uint_as_float(kw4[e] & 0xFFFF0000u), v_[8 * j + 2 * e + 1]);
                }
            }
        }
        if (CS == 1) {
            if (valid) store_quarter(out, t0, v_);
        } else if ((t >> 6) != rank) {  // uniform over a warp
#pragma unroll
            for (int j = 0; j < 4; ++j)
                st_shared_v4(stage + xoff(j), __float_as_uint(v_[4 * j]),
                             __float_as_uint(v_[4 * j + 1]), __float_as_uint(v_[4 * j + 2]),
                             __float_as_uint(v_[4 * j + 3]));
            fence_proxy_async();
            const bool ok = __all_sync(
                0xffffffffu, bar_wait_cluster(&xready[xi], ph_xready[xi], &abort_flag, status));
            ph_xready[xi] ^= 1;
            if (!ok) return false;
            if (lane == 0)
                bulk_copy_cluster(mapa(recv + piece, partner), stage + piece, 2048,
                                  mapa(smem_u32(&xfull[xi]), partner));
        } else if (KW && PASS == kPassR) {
            uint32_t w_[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w_[i] = __float_as_uint(v_[i]);
            tmem_st16(tm_row + col + 16 * wg, w_);
            tmem_wait_st();
        }
        return true;
    };
    // With a partner: once its partial of this CTA's own rows has landed at `recv`, adds it
    // to the rows still at `col` and stores bf16 rows of the chunk at t0 (CL valid rows);
    // re-arms exchange xi for the next chunk and tells the partner that the data is read.
    auto finalize_rows = [&](__nv_bfloat16* out, uint32_t col, int t0, int CL, int xi,
                             uint32_t recv) -> bool {
        if (CS == 1) return true;
        if ((t >> 6) != rank) return true;  // uniform over a warp
        float v_[16];
        tmem_ld16(tm_row + col + 16 * wg, v_);
        const bool ok = bar_wait_w(&xfull[xi], ph_xfull[xi], &abort_flag, status);
        ph_xfull[xi] ^= 1;
        tmem_wait_ld();
        if (!ok) return false;
        if (wg == 0 && quad == 2 * rank && lane == 0) mbar_arrive_expect_tx(&xfull[xi], kXBytes);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 p4 = *reinterpret_cast<const float4*>(sm + (recv - sb) + xoff(j));
            v_[4 * j] += p4.x;
            v_[4 * j + 1] += p4.y;
            v_[4 * j + 2] += p4.z;
            v_[4 * j + 3] += p4.w;
        }
        if (t < CL) store_quarter(out, t0, v_);
        return true;
    };
    const float dscale = 1.0f / (float)M;  // den' = M den
    // g = dout / den' (bf16, the tile at gt) and c_t = -(g . out) (crow; with c_row also row 0
    // of the c operand at c16, and with c_lo row 1 = c - bf16(c)) from the dout and out tiles
    // of the chunk at t0; four lanes per row, eight rows per warp.
    // den_r: load_den's value for this chunk, loaded well before.
    auto load_den = [&](int t0) {
        const int r = t0 + 8 * warp + (lane >> 2);
        return r >= 0 && r < N ? den[(size_t)bh * N + r] : 1.f;
    };
    auto build_g = [&](uint32_t gt, float* crow_, uint32_t c16, float den_r, int CL, bool c_row,
                       bool c_lo) {
        const int r = 8 * warp + (lane >> 2), part = lane & 3;
        const bool valid_ = r < CL;
        const float gsc = valid_ ? dscale / den_r : 0.f;
        float dot = 0.f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t off = swz128(r, (2 * part + j) * 8);
            const uint4 a4 = *reinterpret_cast<const uint4*>(sm + L::DO + off);
            const uint4 o4 = *reinterpret_cast<const uint4*>(sm + L::O + off);
            const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, ow[4] = {o4.x, o4.y, o4.z, o4.w};
            uint32_t gp[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float a0 = __uint_as_float(aw[e] << 16), a1 = __uint_as_float(aw[e] & 0xFFFF0000u);
                const float b0 = __uint_as_float(ow[e] << 16), b1 = __uint_as_float(ow[e] & 0xFFFF0000u);
                // c uses the same bf16-rounded g as the MMAs, so g.v_j + c_i cancels
                // exactly where out_i = v_j (e.g. the first causal position)
                const uint32_t gw = pack_bf16(a0 * gsc, a1 * gsc);
                gp[e] = gw;
                dot = fmaf(__uint_as_float(gw << 16), b0,
                           fmaf(__uint_as_float(gw & 0xFFFF0000u), b1, dot));
            }
            st_shared_v4(gt + off, gp[0], gp[1], gp[2], gp[3]);
        }
        dot += __shfl_xor_sync(0xffffffffu, dot, 1);
        dot += __shfl_xor_sync(0xffffffffu, dot, 2);
        if (part == 0) {
            const float cval = valid_ ? -dot : 0.f;
            crow_[r] = cval;
            if (c_row) {  // row 0 of the K-major [16][tokens] c operand
                uint8_t* c16p = sm + (c16 - sb) + (r >> 6) * 2048;
                const __nv_bfloat16 chi = __float2bfloat16_rn(cval);
                *reinterpret_cast<__nv_bfloat16*>(c16p + swz128(0, r & 63)) = chi;
                if (c_lo)
                    *reinterpret_cast<__nv_bfloat16*>(c16p + swz128(1, r & 63)) =
                        __float2bfloat16_rn(cval - __bfloat162float(chi));
            }
        }
    };
    // row t's s_t partials in `sp`, in order
    auto row_sum = [&](const float* sp) { return (sp[t] + sp[128 + t]) + (sp[256 + t] + sp[384 + t]); };
    // TMA of one tile of chunk cn into shared memory, and of a chunk's rows into L2
    auto load_tile = [&](uint32_t dst, const CUtensorMap* map, int cn, uint64_t* bar) {
        wtma_load_3d(sb + dst, map, 0, cn * kC, bh, bar);
    };
    auto to_l2 = [&](const __nv_bfloat16* p, int cn) {
        if (elect_one()) prefetch_l2(p + base + (size_t)cn * kC * 64, (uint32_t)min(kC, N - cn * kC) * 128);
    };
    // [D] (+)= A B over 128 rows of K (both MN-major), the state sums' form, N = 64, and the
    // c / ones column block (N = 16)
    auto issue_state = [&](uint64_t dphi, uint64_t dval, uint64_t dcol, bool first) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const uint32_t acc = (!first || ks > 0) ? 1u : 0u;
            wmma_bf16(tm + L::T_S, adv(dphi, ks * 2048), adv(dval, ks * 2048), I_MM64, acc);
            wmma_bf16(tm + L::T_S + 64, adv(dphi, ks * 2048),
                     adv(dcol, (ks >> 2) * 2048 + (ks & 3) * 32), I_M16, acc);
        }
    };
    const int nch = (N + kC - 1) / kC;
    const bool issuer = warp == kComputeWarps, relay = warp == kComputeWarps + 1;
    // the chunks [cbeg, cend) of this split
    const int cps = (nch + nsplit - 1) / nsplit;
    const int cbeg = split * cps, cend = min(nch, cbeg + cps), n = cend - cbeg;
    // The relay's thread tells the partner when its partial of a chunk has landed here.
    auto relay_landings = [&](int n) {
        if (CS == 1 || lane != 0) return;
        uint32_t ph = 0;
        for (int i = 0; i < n; ++i, ph ^= 1)
            for (int xi = 0; xi < (PASS == kPassR ? 2 : 1); ++xi) {
                if (!bar_wait(&xfull[xi], ph, &abort_flag, status)) return;
                mbar_arrive_cluster(mapa(smem_u32(&xdone[xi]), partner));
            }
    };
    // A compute warp, before it rewrites the staging region of exchange xi.  Every warp that waits
    // has to gate the next exchange, or that one may complete first and the parity wait miss its
    // phase: in kGrad, where the staging regions hold nothing else, only the warps that send wait
    // (the partner's next landing takes their rows); in the causal passes all wait, before the
    // arrival that gates the MMAs whose rows are sent.
    uint32_t ph_xdone[2] = {0, 0};
    auto staging_free = [&](int xi) -> bool {
        if (CS == 1 || (MODE == kGrad && (t >> 6) == rank)) return true;  // uniform over a warp
        const bool ok = __all_sync(0xffffffffu,
                                   bar_wait_cluster(&xdone[xi], ph_xdone[xi], &abort_flag, status));
        ph_xdone[xi] ^= 1;
        return ok;
    };
    if constexpr (MODE == kCausal) {
        const bool seeded = nsplit > 1;  // ranges: each starts from the sums before (after) it
        if (relay) {
            relay_landings(n);
            __syncwarp();
        } else if (issuer) {
            [&]() {
                uint32_t p_tx = 0, p_rdy = 0, p_m0 = 0, p_m1 = 0, p_s = 0;
                // q, k, v of a chunk complete on tx[0], dout and out on tg; each tile is loaded
                // once its region is free
                const int c0 = PASS == kPassF ? cbeg : cend - 1;
                wmbar_arrive_expect_tx(&tg, 2 * kTileBytes);
                load_tile(L::DO, &tmap_do, c0, &tg);
                load_tile(L::O, &tmap_o, c0, &tg);
                wmbar_arrive_expect_tx(&tx[0], 3 * kTileBytes);
                load_tile(L::Q, &tmap_q, c0, &tx[0]);
                load_tile(L::K, &tmap_k, c0, &tx[0]);
                load_tile(L::V, &tmap_v, c0, &tx[0]);
                for (int it = 0; it < n; ++it) {
                    const int c = PASS == kPassF ? cbeg + it : cend - 1 - it;
                    const int cn = PASS == kPassF ? c + 1 : c - 1;  // the next chunk, if any
                    const bool has_next = it + 1 < n;
                    if (!wwait(&tx[0], p_tx) || !wwait(&rdy, p_rdy)) return;  // g; the previous rows are out of T_P, T_A
                    issue_projection(dQ, L::T_P);
                    issue_projection(dK, L::T_D);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)  // dA = g v^T
                        wmma_bf16(tm + L::T_A, adv(dG, ks * 32), adv(dV, ks * 32), I_KK128, ks > 0);
                    wmma_commit(&m0);
                    p_m0 ^= 1;
                    if (PASS == kPassF && has_next) {
                        wmbar_arrive_expect_tx(&tg, 2 * kTileBytes);
                        load_tile(L::DO, &tmap_do, cn, &tg);
                        load_tile(L::O, &tmap_o, cn, &tg);
                        wmbar_arrive_expect_tx(&tx[0], 3 * kTileBytes);
                    }
                    if (it + 2 < n) {  // the chunk after next into L2
                        const int c2 = PASS == kPassF ? c + 2 : c - 2;
                        to_l2(q, c2); to_l2(k, c2); to_l2(v, c2); to_l2(dout, c2); to_l2(outp, c2);
                    }
                    if (!wwait(&rdy, p_rdy)) return;  // features (F: and the masked dA)
                    if (PASS == kPassF) {
                        // dphi(q) = dA phi(K) + g S^T; S += phi(K)^T v; z += phi(K)^T 1
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            wmma_bf16_tmem_a(tm + L::T_D, tm + L::T_A + 32 * (ks >> 1) + 8 * (ks & 1),
                                            adv(dPKmn, ks * 2048), I_KM128, ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dG, ks * 32), adv(dSN, ks * 32), I_KK128, 1u);
                        wmma_commit(&m0);
                        p_m0 ^= 1;
                        issue_state(dPKmn, dVmn, dC16, it == 0 && !seeded);
                        wmma_commit(&m1);
                        if (kLate) signal_ready(0);  // DA2: the previous dq is finished
                        if (has_next) load_tile(L::K, &tmap_k, cn, &tx[0]);
                        if (!wwait(&m1, p_m1)) return;
                        if (!kLate) signal_ready(0);  // PK is free for the partner's dq partial
                        if (has_next) load_tile(L::V, &tmap_v, cn, &tx[0]);
                        if (!wwait(&rdy, p_rdy)) return;  // da
                        issue_back(sb + L::PQ, sb + L::PQ + 16384, dQmn, it == 0);
                        wmma_commit(&m0);
                        if (!wwait(&m0, p_m0)) return;
                        if (has_next) load_tile(L::Q, &tmap_q, cn, &tx[0]);
                    } else {
                        if (kLate && elect_one()) mbar_arrive(&fin);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {  // A = phi(Q) phi(K)^T
                            const uint32_t kofs = (ks >> 2) * 16384 + (ks & 3) * 32;
                            wmma_bf16(tm + L::T_D, adv(dPQ, kofs), adv(dPK, kofs), I_KK128, ks > 0);
                        }
                        wmma_commit(&m0);
                        p_m0 ^= 1;
                        if (!wwait(&rdy, p_rdy)) return;  // the masked dA and A
                        // n: u, w of k again for the chain rule; dphi(k) = dA^T phi(Q) + v R^T;
                        // dv = A^T g + phi(K) R; then R += phi(Q)^T g; r += phi(Q)^T c
                        if (NS) issue_projection(dK, L::T_P);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dDAmn, ks * 2048), adv(dPQmn, ks * 2048), I_MM128,
                                     ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dV, ks * 32), adv(dSN, ks * 32), I_KK128, 1u);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            wmma_bf16(tm + T_DV, adv(dAmn, ks * 2048), adv(dGmn, ks * 2048), I_MM64,
                                     ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            wmma_bf16(tm + T_DV, adv(dPK, (ks >> 2) * 16384 + (ks & 3) * 32),
                                     adv(dSNmn, ks * 2048), I_KM64, 1u);
                        wmma_commit(&m0);
                        p_m0 ^= 1;
                        issue_state(dPQmn, dGmn, dC16, it == 0 && !seeded);
                        wmma_commit(&m1);
                        if (kLate) signal_ready(1);  // XR: the previous dk is finished
                        if (!wwait(&m1, p_m1)) return;
                        signal_ready(0);  // DA2 is free for the partner's dv partial
                        if (!wwait(&rdy, p_rdy)) return;  // da
                        issue_back(sb + L::PK, sb + L::PK + 16384, dKmn, it == 0);
                        wmma_commit(&m0);
                        if (has_next) {  // Q, V, DO, O are free
                            wmbar_arrive_expect_tx(&tg, 2 * kTileBytes);
                            load_tile(L::DO, &tmap_do, cn, &tg);
                            load_tile(L::O, &tmap_o, cn, &tg);
                            wmbar_arrive_expect_tx(&tx[0], 3 * kTileBytes);
                            load_tile(L::Q, &tmap_q, cn, &tx[0]);
                            load_tile(L::V, &tmap_v, cn, &tx[0]);
                        }
                        if (!wwait(&m0, p_m0)) return;
                        if (!kLate) signal_ready(1);  // PK is free for the partner's dk partial
                        if (KW && !wwait(&srdy, p_s)) return;  // dk rows have read the k tile
                        if (has_next) load_tile(L::K, &tmap_k, cn, &tx[0]);
                    }
                }
            }();
            __syncwarp();
        } else {
            uint32_t p_tg = 0, p_m0 = 0, p_m1 = 0, p_fin = 0;
            int prev_t0 = 0, prev_CL = 0;  // the chunk whose rows await the partner
            // A copy takes about 3.5 us to land (8 KB/us a CTA when all exchange), so with kLate
            // the previous chunk's rows are finished after this chunk's features; n, whose
            // projections need that tensor memory, finishes them before its projections.
            constexpr uint32_t kRecvQ = kLate ? L::DA2 : L::PK;  // DA2 is unused in pass F
            auto finalize = [&](bool late) {
                if (CS == 1 || late != kLate) return true;
                if (PASS == kPassF) return finalize_rows(dq, T_X, prev_t0, prev_CL, 0, sb + kRecvQ);
                return finalize_rows(dv, T_DV, prev_t0, prev_CL, 0, sb + L::DA2) &&
                       finalize_rows(dk, T_X, prev_t0, prev_CL, 1, sb + L::XR);
            };
            // bf16 of the block at `col` masked to j <= i (+ add), this warp's 32 keys
            auto mask32 = [&](uint32_t col, float add, int CL, bool valid, uint32_t (&pk2)[16]) {
                // whole chunks: blocks above the diagonal block of this warp's rows are zeros
                // (nothing loaded), those below it need no mask
                const bool full = CL == kC && wg != quad;
                if (full && wg > quad) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) pk2[i] = 0u;
                    return;
                }
                float a[32];
                tmem_ld16(tm_row + col + 32 * wg, *reinterpret_cast<float(*)[16]>(&a[0]));
                tmem_ld16(tm_row + col + 32 * wg + 16, *reinterpret_cast<float(*)[16]>(&a[16]));
                tmem_wait_ld();
                if (full) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) pk2[i] = pack_bf16(a[2 * i] + add, a[2 * i + 1] + add);
                    return;
                }
                const int keys = (valid ? min(t + 1, CL) : 0) - 32 * wg;  // of this block
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    pk2[i] = pack_bf16(2 * i < keys ? a[2 * i] + add : 0.f,
                                       2 * i + 1 < keys ? a[2 * i + 1] + add : 0.f);
            };
            auto mask_to_smem = [&](uint32_t col, float add, int CL, bool valid, uint32_t dst) {
                uint32_t pk2[16];
                mask32(col, add, CL, valid, pk2);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    st_shared_v4(dst + (wg >> 1) * 16384 + swz128(t, (4 * (wg & 1) + j) * 8), pk2[4 * j],
                                 pk2[4 * j + 1], pk2[4 * j + 2], pk2[4 * j + 3]);
            };
            if (seeded) {
                // what the range starts from (zeros for the first), into the running state, its
                // snapshot and zr
                const float* st = state_part + ((size_t)slot * 128 + t) * 80;
                float x[16];
                uint32_t w_[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 f4 = reinterpret_cast<const float4*>(st + 16 * wg)[j];
                    x[4 * j] = f4.x; x[4 * j + 1] = f4.y; x[4 * j + 2] = f4.z; x[4 * j + 3] = f4.w;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) w_[i] = __float_as_uint(x[i]);
                tmem_st16(tm_row + L::T_S + 16 * wg, w_);
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    st_shared_v4(sb + L::SN + swz128(t, (2 * wg + j) * 8),
                                 pack_bf16(x[8 * j], x[8 * j + 1]), pack_bf16(x[8 * j + 2], x[8 * j + 3]),
                                 pack_bf16(x[8 * j + 4], x[8 * j + 5]),
                                 pack_bf16(x[8 * j + 6], x[8 * j + 7]));
                if (wg == 0) {
                    zr[t] = st[64];
#pragma unroll
                    for (int i = 0; i < 16; ++i) w_[i] = i == 0 ? __float_as_uint(st[64]) : 0u;
                    tmem_st16(tm_row + L::T_S + 64, w_);
                }
                tmem_wait_st();
            }
            float den_r = load_den(PASS == kPassF ? cbeg * kC : (cend - 1) * kC);
            for (int it = 0; it < n; ++it) {
                const int c = PASS == kPassF ? cbeg + it : cend - 1 - it;
                const int t0 = c * kC, CL = min(kC, N - t0);
                const bool valid = t < CL;
                const float wk = (KW && valid) ? kw[(size_t)bh * N + t0 + t] : 1.f;
                if (it > 0 && !finalize(false)) goto done;
                if (!wwait(&tg, p_tg)) goto done;
                build_g(sb + L::GT, crow, sb + L::C16, den_r, CL, PASS == kPassR, false);
                den_r = load_den(PASS == kPassF ? t0 + kC : t0 - kC);
                arrive(&rdy);
                if (!wwait(&m0, p_m0)) goto done;
                if (PASS == kPassF) {
                    features(sb + L::PK, L::T_D, valid, wk);
                    if (it > 0 && !finalize(true)) goto done;
                    {  // dA + c, masked, as the A operand: over the first 16 columns this warp read
                        uint32_t pk2[16];
                        mask32(L::T_A, crow[t], CL, valid, pk2);
                        tmem_st16(tm_row + L::T_A + 32 * wg, pk2);
                        tmem_wait_st();
                    }
                    arrive(&rdy);
                    if (!wwait(&m0, p_m0)) goto done;  // dphi(q)
                    if (it > 0 && !staging_free(0)) goto done;
                    feature_backward(std::false_type{}, zr + 128 * (it & 1), 0, sb + L::PQ,
                                     sb + L::PQ + 16384, crow[t], valid, 1.f);
                    arrive(&rdy);
                    if (!wwait(&m1, p_m1)) goto done;  // the state with this chunk
                    snapshot(zr + 128 * ((it + 1) & 1));
                    if (!wwait(&m0, p_m0)) goto done;  // dq, dW
                    if (!take_rows(dq, T_X, t0, valid, 0.f, 0, 0, sb + L::PQ, sb + kRecvQ)) goto done;
                    if (NS) dw_accumulate(it == 0);
                } else {
                    if (it > 0 && (!staging_free(0) || (!kLate && !staging_free(1)))) goto done;
                    features(sb + L::PQ, L::T_P, valid, 1.f);
                    if (kLate && it > 0 && !staging_free(1)) goto done;
                    features(sb + L::PK, L::T_D, valid, wk);
                    if (it > 0 && !finalize(true)) goto done;
                    arrive(&rdy);
                    // every warp has read the partner's dv in DA2, which the masked dA overwrites
                    if (kLate && !wwait(&fin, p_fin)) goto done;
                    // dA + c, masked, as [query][key] in [Q | DA2], while A is computed
                    mask_to_smem(L::T_A, crow[t], CL, valid, sb + L::Q);
                    if (!wwait(&m0, p_m0)) goto done;
                    mask_to_smem(L::T_D, 0.f, CL, valid, sb + L::DO);  // A in [DO | O]
                    arrive(&rdy);
                    if (!wwait(&m0, p_m0)) goto done;  // dphi(k), dv
                    const float sp = feature_backward(std::integral_constant<bool, !NS>{}, zr + 128 * (it & 1), 0,
                                                      sb + L::PK, sb + L::PK + 16384, 1.0f, valid, wk);
                    if (KW) {
                        spart[128 * wg + t] = sp;
                        // ln w = |k|^2 exp(-tau), centred on the sequence's first key (the s_j of
                        // a sequence sum to zero): the cancelling part drops out exactly
                        dtau_acc = fmaf(lw0 - logf(wk), sp, dtau_acc);
                    }
                    arrive(&rdy);
                    if (!wwait(&m1, p_m1)) goto done;  // the state; PQ is free for staging
                    if (!take_rows(dv, T_DV, t0, valid, 0.f, 0, 0, sb + L::PQ, sb + L::DA2)) goto done;
                    snapshot(zr + 128 * ((it + 1) & 1));
                    if (!wwait(&m0, p_m0)) goto done;  // dk, dW
                    if (!take_rows(dk, T_X, t0, valid, KW ? 2.f * itau * row_sum(spart) : 0.f, L::K, 1,
                                   sb + (kLate ? L::PK : L::PQ + 16384), sb + L::XR))
                        goto done;
                    if (KW) arrive(&srdy);
                    if (dw_per_chunk) dw_accumulate(it == 0);
                }
                prev_t0 = t0;
                prev_CL = CL;
            }
            // the last chunk's rows
            if (!finalize(kLate)) goto done;
        }
    } else if constexpr (MODE == kState) {
        // this CTA reads q, dout, out (pass R) or k, v (pass F); two tile, feature, g and c
        // buffers (three of v)
        const bool fq = PASS == kPassR;
        const uint32_t xb[2] = {fq ? L::Q : L::K, fq ? L::K : L::Q};
        const uint32_t vb[3] = {L::V, L::DO, L::O};
        const uint32_t gb[2] = {L::GT, L::V}, cb[2] = {L::C16, fq ? L::SN : L::C16};
        const uint32_t pb[2] = {L::PQ, L::PK}, tb[2] = {L::T_P, L::T_A};
        if (relay) {
        } else if (issuer) {
            [&]() {
                uint32_t p_tx[2] = {0, 0}, p_tv[3] = {0, 0, 0}, p_rdys[2] = {0, 0}, p_m1 = 0;
                auto load_x = [&](int i) {
                    wmbar_arrive_expect_tx(&tx[i & 1], kTileBytes);
                    load_tile(xb[i & 1], fq ? &tmap_q : &tmap_k, cbeg + i, &tx[i & 1]);
                };
                auto load_v = [&](int i) {
                    wmbar_arrive_expect_tx(&tv[i % 3], kTileBytes);
                    load_tile(vb[i % 3], &tmap_v, cbeg + i, &tv[i % 3]);
                };
                auto load_g = [&](int i) {
                    wmbar_arrive_expect_tx(&tg, 2 * kTileBytes);
                    load_tile(L::DO, &tmap_do, cbeg + i, &tg);
                    load_tile(L::O, &tmap_o, cbeg + i, &tg);
                };
                auto project = [&](int i) {
                    if (!wwait(&tx[i & 1], p_tx[i & 1])) return false;
                    issue_projection(sdesc(sb + xb[i & 1], 16, 1024), tb[i & 1]);
                    wmma_commit(&mt[i & 1]);
                    return true;
                };
                for (int i = 0; i < min(2, n); ++i) load_x(i);
                if (fq && n > 0) load_g(0);
                if (!fq)
                    for (int i = 0; i < min(2, n); ++i) load_v(i);
                if (n > 0 && !project(0)) return;
                for (int i = 0; i < n; ++i) {
                    if (i + 3 < n) {  // a later chunk into L2
                        const int c3 = cbeg + i + 3;
                        if (fq) {
                            to_l2(q, c3); to_l2(dout, c3); to_l2(outp, c3);
                        } else {
                            to_l2(k, c3); to_l2(v, c3);
                        }
                    }
                    if (i + 1 < n && !project(i + 1)) return;
                    if (!wwait(&rdys[i & 1], p_rdys[i & 1])) return;  // features (and g) of chunk i
                    if (i + 2 < n) load_x(i + 2);
                    if (fq && i + 1 < n) load_g(i + 1);
                    if (!fq && !wwait(&tv[i % 3], p_tv[i % 3])) return;
                    // the sums of chunk i - 1 (waited for before the next commit on m1, so
                    // that no phase of it is missed): its v buffer is free
                    if (i > 0 && !wwait(&m1, p_m1)) return;
                    if (!fq && i + 2 < n) load_v(i + 2);
                    // [S | z] += phi(K)^T [V | 1]  or  [R | r] += phi(Q)^T [G | c]
                    issue_state(sdesc(sb + pb[i & 1], 16384, 1024),
                                sdesc(sb + (fq ? gb[i & 1] : vb[i % 3]), 16384, 1024),
                                sdesc(sb + cb[i & 1], 16, 1024), i == 0);
                    wmma_commit(&m1);
                }
                if (n > 0) wwait(&m1, p_m1);
            }();
            __syncwarp();
        } else {
            uint32_t p_mt[2] = {0, 0}, p_tg = 0;
            float den_r = fq ? load_den(cbeg * kC) : 1.f;
            for (int i = 0; i < n; ++i) {
                const int t0 = (cbeg + i) * kC, CL = min(kC, N - t0);
                const bool valid = t < CL;
                const float wk = (KW && !fq && valid) ? kw[(size_t)bh * N + t0 + t] : 1.f;
                // projected; and the sums of chunk i - 2, issued before it, have read this
                // parity's feature, g and c buffers
                if (!wwait(&mt[i & 1], p_mt[i & 1])) break;
                features(sb + pb[i & 1], tb[i & 1], valid, fq ? 1.f : wk);
                if (fq) {
                    // c as high and low bf16 parts, so r carries c to ~2^-17 like the
                    // exact-cancelling term g . v
                    if (!wwait(&tg, p_tg)) break;
                    build_g(sb + gb[i & 1], crow, sb + cb[i & 1], den_r, CL, true, true);
                    den_r = load_den(t0 + kC);
                }
                arrive(&rdys[i & 1]);
            }
        }
        __syncthreads();  // reached after an abort as well: the last sums are complete
        fence_after_sync();
        if (abort_flag) goto done;
        if (!issuer && !relay) {
            // this CTA's partial state [128 features][80] fp32: S (or R) in columns 0-63,
            // z (or r) in column 64
            float s_[16], zz[16];
            tmem_ld16(tm_row + L::T_S + 16 * wg, s_);
            if (wg == 0) tmem_ld16(tm_row + L::T_S + 64, zz);
            tmem_wait_ld();
            float* dst = state_part + ((size_t)slot * 128 + t) * 80;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                reinterpret_cast<float4*>(dst + 16 * wg)[j] =
                    make_float4(s_[4 * j], s_[4 * j + 1], s_[4 * j + 2], s_[4 * j + 3]);
            // r = column 64 (c high) + column 65 (c low); z: column 64 (every C16 row is 1)
            if (wg == 0) dst[64] = PASS == kPassR ? zz[0] + zz[1] : zz[0];
        }
    } else {
        // the low part of the state snapshot, in a region the pass does not use
        const uint32_t sl = sb + (PASS == kPassF ? L::V : L::PQ);
        if (!issuer && !relay) {
            // the totals ([S | z] for pass F, [R | r] for pass R) as the state snapshot, split
            // into bf16 high (SN) and low (SL) parts [feature][64] so that the two MMAs carry
            // the fp32 totals to ~2^-17: the terms S g and c z (R v and r) cancel exactly
            // where the result is 0 (e.g. dq at N = 1); column 64 in zr (fp32)
            const float* st = state_total + ((size_t)PASS * units + unit) * 128 * 80 + (size_t)t * 80;
            float s_[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 f4 = reinterpret_cast<const float4*>(st + 16 * wg)[j];
                s_[4 * j] = f4.x; s_[4 * j + 1] = f4.y; s_[4 * j + 2] = f4.z; s_[4 * j + 3] = f4.w;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint32_t hi[4], lo[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x0 = s_[8 * j + 2 * e], x1 = s_[8 * j + 2 * e + 1];
                    hi[e] = pack_bf16(x0, x1);
                    lo[e] = pack_bf16(x0 - __uint_as_float(hi[e] << 16),
                                      x1 - __uint_as_float(hi[e] & 0xFFFF0000u));
                }
                const uint32_t off = swz128(t, (2 * wg + j) * 8);
                st_shared_v4(sb + L::SN + off, hi[0], hi[1], hi[2], hi[3]);
                st_shared_v4(sl + off, lo[0], lo[1], lo[2], lo[3]);
            }
            if (wg == 0) zr[t] = st[64];
        }
        fence_proxy_async();
        __syncthreads();
        const uint64_t dSL = sdesc(sl, 16, 1024), dSLmn = sdesc(sl, 16384, 1024);
        const uint32_t da1 = sb + L::PQ + 16384;
        if (PASS == kPassF) {
            const uint32_t qb[2] = {L::Q, L::DA2}, gb[2] = {L::GT, L::PK + 16384};
            if (relay) {
                relay_landings(n);
                __syncwarp();
            } else if (issuer) {
                [&]() {
                    uint32_t p_tx[2] = {0, 0}, p_rdy = 0, p_rdyg = 0, p_m1 = 0;
                    auto load_x = [&](int i) {
                        wmbar_arrive_expect_tx(&tx[i & 1], kTileBytes);
                        load_tile(qb[i & 1], &tmap_q, cbeg + i, &tx[i & 1]);
                    };
                    auto load_g = [&](int i) {
                        wmbar_arrive_expect_tx(&tg, 2 * kTileBytes);
                        load_tile(L::DO, &tmap_do, cbeg + i, &tg);
                        load_tile(L::O, &tmap_o, cbeg + i, &tg);
                    };
                    if (n > 0) load_g(0);
                    for (int i = 0; i < min(2, n); ++i) load_x(i);
                    signal_ready(0);  // PK is free for the first exchange
                    for (int i = 0; i < n; ++i) {
                        if (i + 2 < n) {
                            const int c2 = cbeg + i + 2;
                            to_l2(q, c2); to_l2(dout, c2); to_l2(outp, c2);
                        }
                        if (!wwait(&rdyg, p_rdyg)) return;  // g of chunk i; its dout, out are read
                        if (i + 1 < n) load_g(i + 1);
                        if (!wwait(&tx[i & 1], p_tx[i & 1])) return;
                        // the projection, and dphi(q) = g S^T (+ c z in the chain rule)
                        issue_projection(sdesc(sb + qb[i & 1], 16, 1024), L::T_P);
                        const uint64_t dGi = sdesc(sb + gb[i & 1], 16, 1024);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dGi, ks * 32), adv(dSN, ks * 32), I_KK128, ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dGi, ks * 32), adv(dSL, ks * 32), I_KK128, 1u);
                        wmma_commit(&m0);
                        if (i > 0) {
                            if (!wwait(&m1, p_m1)) return;
                            if (i + 1 < n) load_x(i + 1);
                        }
                        if (!wwait(&rdy, p_rdy)) return;  // da; chunk i - 1's rows are finished
                        if (CS > 1 && i > 0) {
                            signal_ready(0);
                        }
                        issue_back(sb + L::PQ, da1, sdesc(sb + qb[i & 1], 16384, 1024), i == 0);
                        wmma_commit(&m1);
                    }
                }();
                __syncwarp();
            } else {
                uint32_t p_tg = 0, p_m0 = 0, p_m1 = 0;
                float den_r = load_den(cbeg * kC);
                auto next_g = [&](int i) {
                    if (!wwait(&tg, p_tg)) return false;
                    const int t0 = (cbeg + i) * kC;
                    build_g(sb + gb[i & 1], crow + 128 * (i & 1), 0, den_r, min(kC, N - t0), false, false);
                    den_r = load_den(t0 + kC);
                    arrive(&rdyg);
                    return true;
                };
                if (n > 0 && !next_g(0)) goto done;
                for (int i = 0; i < n; ++i) {
                    const int t0 = (cbeg + i) * kC, CL = min(kC, N - t0);
                    const bool valid = t < CL;
                    if (!wwait(&m0, p_m0)) goto done;
                    feature_backward(std::false_type{}, zr, 0, sb + L::PQ, da1, crow[128 * (i & 1) + t],
                                     valid, 1.f);
                    if (i > 0 && !finalize_rows(dq, T_X, t0 - kC, kC, 0, sb + L::PK)) goto done;
                    arrive(&rdy);
                    if (i + 1 < n && !next_g(i + 1)) goto done;
                    if (!wwait(&m1, p_m1)) goto done;
                    if (i > 0 && !staging_free(0)) goto done;
                    if (!take_rows(dq, T_X, t0, valid, 0.f, 0, 0, sb + L::K, sb + L::PK)) goto done;
                }
                if (n > 0 && !finalize_rows(dq, T_X, (cend - 1) * kC, N - (cend - 1) * kC, 0, sb + L::PK))
                    goto done;
            }
        } else {
            // two buffers of k and v where no exchange needs the space
            constexpr int NB = CS == 1 ? 2 : 1;
            const uint32_t kb[2] = {L::K, L::Q}, vb[2] = {L::V, L::DO};
            if (relay) {
                relay_landings(n);
                __syncwarp();
            } else if (issuer) {
                [&]() {
                    uint32_t p_tx[2] = {0, 0}, p_rdy = 0, p_m1 = 0, p_s = 0;
                    auto load_x = [&](int i) {
                        const int b = i % NB;
                        wmbar_arrive_expect_tx(&tx[b], 2 * kTileBytes);
                        load_tile(kb[b], &tmap_k, cbeg + i, &tx[b]);
                        load_tile(vb[b], &tmap_v, cbeg + i, &tx[b]);
                    };
                    for (int i = 0; i < min(NB, n); ++i) load_x(i);
                    signal_ready(0);  // DO, O are free for the first exchange
                    signal_ready(1);
                    for (int i = 0; i < n; ++i) {
                        const int b = i % NB;
                        if (i + 2 < n) {
                            to_l2(k, cbeg + i + 2);
                            to_l2(v, cbeg + i + 2);
                        }
                        if (!wwait(&tx[b], p_tx[b])) return;
                        // the projection, and dphi(k) = v R^T (+ r in the chain rule)
                        issue_projection(sdesc(sb + kb[b], 16, 1024), L::T_P);
                        const uint64_t dVi = sdesc(sb + vb[b], 16, 1024);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dVi, ks * 32), adv(dSN, ks * 32), I_KK128, ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            wmma_bf16(tm + L::T_D, adv(dVi, ks * 32), adv(dSL, ks * 32), I_KK128, 1u);
                        wmma_commit(&m0);
                        if (NB == 2 && i > 0) {  // chunk i - 1's buffers: its MMAs and rows done
                            if (!wwait(&m1, p_m1)) return;
                            if (!wwait(&srdy, p_s)) return;
                            if (i + 1 < n) load_x(i + 1);
                        }
                        if (!wwait(&rdy, p_rdy)) return;  // phi(k), da; chunk i - 1's rows finished
                        if (CS > 1 && i > 0) {
                            signal_ready(0);
                            signal_ready(1);
                        }
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)  // dv = phi(K) R
                            wmma_bf16(tm + T_DV, adv(dPK, (ks >> 2) * 16384 + (ks & 3) * 32),
                                     adv(dSNmn, ks * 2048), I_KM64, ks > 0);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            wmma_bf16(tm + T_DV, adv(dPK, (ks >> 2) * 16384 + (ks & 3) * 32),
                                     adv(dSLmn, ks * 2048), I_KM64, 1u);
                        issue_back(sb + L::GT, da1, sdesc(sb + kb[b], 16384, 1024), i == 0);
                        wmma_commit(&m1);
                        if (NB == 1) {
                            if (!wwait(&m1, p_m1)) return;
                            if (!wwait(&srdy, p_s)) return;
                            if (i + 1 < n) load_x(i + 1);
                        }
                    }
                }();
                __syncwarp();
            } else {
                uint32_t p_m0 = 0, p_m1 = 0;
                auto finalize = [&](int t0, int CL) {
                    return finalize_rows(dv, T_DV, t0, CL, 0, sb + L::DO) &&
                           finalize_rows(dk, T_X, t0, CL, 1, sb + L::O);
                };
                for (int i = 0; i < n; ++i) {
                    const int t0 = (cbeg + i) * kC, CL = min(kC, N - t0);
                    const bool valid = t < CL;
                    const float wk = (KW && valid) ? kw[(size_t)bh * N + t0 + t] : 1.f;
                    if (!wwait(&m0, p_m0)) goto done;
                    const float sp = feature_backward(std::false_type{}, zr, sb + L::PK, sb + L::GT, da1, 1.0f,
                                                      valid, wk);
                    // Two sets of partials: with two tile buffers a warp may be here while another
                    // still reads the row sums of chunk i - 1 below.  None may be a chunk further
                    // ahead: m0 of chunk i + 1 follows every warp's srdy of chunk i - 1.
                    float* sp_ = spart + 512 * (i & 1);
                    if (KW) {
                        sp_[128 * wg + t] = sp;
                        dtau_acc = fmaf(lw0 - logf(wk), sp, dtau_acc);  // centred, as above
                    }
                    if (i > 0 && !finalize(t0 - kC, kC)) goto done;
                    arrive(&rdy);
                    if (!wwait(&m1, p_m1)) goto done;
                    if (i > 0 && (!staging_free(0) || !staging_free(1))) goto done;
                    if (!take_rows(dv, T_DV, t0, valid, 0.f, 0, 0, sb + L::Q, sb + L::DO) ||
                        !take_rows(dk, T_X, t0, valid, KW ? 2.f * itau * row_sum(sp_) : 0.f, kb[i % NB],
                                   1, sb + L::DA2, sb + L::O))
                        goto done;
                    arrive(&srdy);
                }
                if (n > 0 && !finalize((cend - 1) * kC, N - (cend - 1) * kC)) goto done;
            }
        }
    }
    // s (and n in kGrad): the sum over the chunks, held in tensor memory
    if (!issuer && !relay && MODE != kState && !dw_per_chunk) dw_accumulate(true);
done:
    __syncthreads();
    if (KW && MODE != kState && !abort_flag) {
        // this CTA's dtau (pass R; 0 in pass F): warps, then in order
        for (int o = 16; o > 0; o >>= 1) dtau_acc += __shfl_xor_sync(0xffffffffu, dtau_acc, o);
        if (lane == 0) spart[warp] = dtau_acc;
        __syncthreads();
        if (tid == 0) {
            float sum = 0.f;
            for (int w8 = 0; w8 < kComputeWarps; ++w8) sum += spart[w8];
            dtau_part[slot] = sum;
        }
    }
    if (tid == 0) drain_after_abort(abort_flag != 0);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 0) tmem_dealloc(tm, 512);
    if (CS > 1) cluster_sync();  // no CTA leaves while its partner may still copy into it
}

// One instantiation of the body per pass: each compiles with its own constants and registers.
template <bool NS, bool KW, int CS, int MODE>
__global__ void __launch_bounds__(kThreadsB, 1)
    tc_bwd_kernel(const __grid_constant__ CUtensorMap tmap_q,
                  const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_v,
                  const __grid_constant__ CUtensorMap tmap_do,
                  const __grid_constant__ CUtensorMap tmap_o, int H, int N, int M, int G,
                  const __nv_bfloat16* __restrict__ q,
                  const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                  const float* __restrict__ W1, const float* __restrict__ W2,
                  const __nv_bfloat16* __restrict__ outp, const float* __restrict__ den,
                  const __nv_bfloat16* __restrict__ dout, __nv_bfloat16* __restrict__ dq,
                  __nv_bfloat16* __restrict__ dk, __nv_bfloat16* __restrict__ dv,
                  float* dw_part,
                  const float* kw, const float* __restrict__ tau,
                  float* dtau_part, int units, int nsplit,
                  float* state_part, const float* state_total,
                  int* status)
{
    if ((int)blockIdx.x < units * nsplit)
        tc_bwd_body<NS, KW, CS, MODE, kPassR>(
            tmap_q, tmap_k, tmap_v, tmap_do, tmap_o, H, N, M, G, q, k, v, W1, W2,
            outp, den, dout, dq, dk, dv, dw_part, kw, tau, dtau_part, units, nsplit,
            state_part, state_total, status);
    else
        tc_bwd_body<NS, KW, CS, MODE, kPassF>(
            tmap_q, tmap_k, tmap_v, tmap_do, tmap_o, H, N, M, G, q, k, v, W1, W2,
            outp, den, dout, dq, dk, dv, dw_part, kw, tau, dtau_part, units, nsplit,
            state_part, state_total, status);
}

// dW over the batch (and the chunk splits) in a fixed order.  Partial slots
// [pass][((b * H + h) * nsplit + s) * G + g][16 column quads][128 rows][4]; s: rows < 64 are
// frequencies 64g + row (from the high bf16 part of da), rows >= 64 the same frequencies
// (from its low part); n: rows < 64 are dU, rows >= 64 are dV of frequency 64g + row%64.
// One block per (head, group, column quad): thread (row, lane) sums every fourth slot with
// LD loads in flight, the four lanes are then added in order.  It is bound by reading the slots
// (32 KB each) at memory latency and by the index arithmetic: B32 H8 in two ranges 29.5 us with one
// thread per output, 13.3 with eight loads in flight, 9.1 with 16 and no division per slot.
constexpr int kReduceThreads = 512;
template <int LD>  // loads in flight per thread (wide_reduce)
__global__ void __launch_bounds__(kReduceThreads)
    tc_dw_reduce_kernel(int B, int H, int M, int G, int nsplit, int nonstat,
                        const float* part, float* __restrict__ dW1,
                        float* __restrict__ dW2, const float* dtau_part,
                        float* __restrict__ dtau)
{
    __shared__ float4 sums[3][128];
    grid_dep_wait();
    const int quad = blockIdx.x % 16, g = blockIdx.x / 16 % G, h = blockIdx.x / (16 * G);
    const int row = threadIdx.x % 128, ln = threadIdx.x / 128;
    // slot i = bb nsplit + sp, bb = pass B + b < 2 B: pass F's slots, then R's; from one slot
    // to the fourth after it without a division
    const int dbb = 4 / nsplit, dsp = 4 % nsplit;
    int bb = ln / nsplit, sp = ln % nsplit;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    while (bb < 2 * B) {
        float4 x[LD];
#pragma unroll
        for (int u = 0; u < LD; ++u) {
            const size_t slot = ((size_t)(bb * H + h) * nsplit + sp) * G + g;
            x[u] = bb < 2 * B ? reinterpret_cast<const float4*>(part)[(slot * 16 + quad) * 128 + row]
                              : make_float4(0.f, 0.f, 0.f, 0.f);
            bb += dbb;
            sp += dsp;
            if (sp >= nsplit) {
                sp -= nsplit;
                ++bb;
            }
        }
#pragma unroll
        for (int u = 0; u < LD; ++u)
            a = make_float4(a.x + x[u].x, a.y + x[u].y, a.z + x[u].z, a.w + x[u].w);
    }
    if (ln > 0) sums[ln - 1][row] = a;
    __syncthreads();
    if (ln == 0) {
        for (int l = 0; l < 3; ++l) {
            const float4 x = sums[l][row];
            a = make_float4(a.x + x.x, a.y + x.y, a.z + x.z, a.w + x.w);
        }
        if (row >= 64) sums[0][row] = a;
    }
    __syncthreads();
    if (ln == 0 && row < 64) {
        const float4 b = sums[0][64 + row];  // n: dV rows; s: the dW rows of the low part of da
        const size_t o = (((size_t)h * M + 64 * g + row) * 64 + 4 * quad) / 4;
        if (!nonstat) {
            reinterpret_cast<float4*>(dW1)[o] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        } else {
            reinterpret_cast<float4*>(dW1)[o] = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y),
                                                            0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
            reinterpret_cast<float4*>(dW2)[o] = make_float4(0.5f * (a.x - b.x), 0.5f * (a.y - b.y),
                                                            0.5f * (a.z - b.z), 0.5f * (a.w - b.w));
        }
    }
    if (dtau && quad == 0 && g == 0 && threadIdx.x < 32) {  // dtau[h]: head h's pass R slots
        float t = 0.f;
        const size_t half = (size_t)B * H * nsplit * G;  // slots per pass
        for (int i = threadIdx.x; i < B * nsplit * G; i += 32)
            t += dtau_part[half + ((size_t)(i / (nsplit * G) * H + h) * nsplit + i / G % nsplit) * G + i % G];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) dtau[h] = t;
    }
}

// Partial states are [pass][(bh * nsplit + s) * G + g][128 rows][80], columns 0-64 in use: one
// block of kStateThreads covers an eighth (blockIdx.y) of the 128 x 17 float4 of a (pass, unit),
// blockIdx.x = pass * units + unit (unit = bh * G + g); the splits' loads are independent.
constexpr int kStateThreads = 272;
__device__ __forceinline__ float4* state_at(float* part, size_t slot)
{
    const int i = blockIdx.y * kStateThreads + threadIdx.x;
    return reinterpret_cast<float4*>(part) + (slot * 128 + i / 17) * 20 + i % 17;
}
__device__ __forceinline__ void add4(float4& a, const float4& x)
{
    a = make_float4(a.x + x.x, a.y + x.y, a.z + x.z, a.w + x.w);
}

// Non-causal totals: total[pass][unit][row][0..64] = sum over the splits, in order.
__global__ void __launch_bounds__(kStateThreads)
    nc_state_reduce_kernel(int units, int G, int nsplit, float* part,
                           float* total)
{
    const int u = blockIdx.x % units, pass = blockIdx.x / units, bh = u / G, g = u % G;
    grid_dep_launch();
    grid_dep_wait();
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int sp = 0; sp < nsplit; ++sp)
        add4(a, *state_at(part, (size_t)pass * units * nsplit + ((size_t)bh * nsplit + sp) * G + g));
    *state_at(total, (size_t)pass * units + u) = a;
}

// Causal ranges: each range's partial state becomes, in place, what the range starts from:
// pass F the sum over the earlier ranges, pass R over the later ones, in order.
__global__ void __launch_bounds__(kStateThreads)
    causal_state_scan_kernel(int units, int G, int nsplit, float* part)
{
    const int u = blockIdx.x % units, pass = blockIdx.x / units, bh = u / G, g = u % G;
    grid_dep_launch();
    grid_dep_wait();
    auto at = [&](int o) {
        const int sp = pass == kPassF ? o : nsplit - 1 - o;
        return state_at(part, (size_t)pass * units * nsplit + ((size_t)bh * nsplit + sp) * G + g);
    };
    float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int o0 = 0; o0 < nsplit; o0 += 8) {
        float4 x[8];
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (o0 + o < nsplit) x[o] = *at(o0 + o);
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (o0 + o < nsplit) {
                *at(o0 + o) = run;
                add4(run, x[o]);
            }
    }
}

// Ranges per sequence for the causal mode.  One range per CTA runs the chunks in order, so a
// small batch leaves SMs idle (2 B H G CTAs); cut into ranges, each (pass, sequence, group)
// first sums its ranges' states (kState, about 0.16 of a causal chunk each) and scans them.
// The count minimises rounds of CTAs on 152 SMs x (set-up + chunks), in causal chunk times
// (about 8 us; the two extra launches cost about one); short sequences (under 8 chunks) gain
// nothing.  Forward and backward of n with tau, B2 H8 N2000 M64 (32 CTAs uncut, 128 in four
// ranges): 248 -> 160 us (109 with the later steps).
int causal_splits(const Problem& p)
{
    const long long units = (long long)p.B * p.H * (p.M / 64);
    const int nch = (p.N + kC - 1) / kC;
    if (nch < 8) return 1;
    int best_ns = 1;
    double best = 0.;
    for (int want = 1; want <= nch / 2; ++want) {
        const int per = (nch + want - 1) / want, ns = (nch + per - 1) / per;
        const double rounds = (double)((2 * units * ns + 151) / 152);
        const double cost = rounds * (0.4 + per) + (ns > 1 ? rounds * (0.4 + 0.16 * per) + 1. : 0.);
        if (want == 1 || cost < 0.95 * best) {
            best = cost;
            best_ns = ns;
        }
    }
    return best_ns;
}

// Chunk splits per (pass, sequence, group) for the non-causal modes: enough CTAs for a few
// waves of ~152 SMs, every split non-empty (depends on the shape only, so the workspace size
// is known before the call).
int nc_splits(const Problem& p)
{
    const int units = p.B * p.H * (p.M / 64), nch = (p.N + kC - 1) / kC;
    const int target = std::max(1, std::min(nch, (4 * 152 + 2 * units - 1) / (2 * units)));
    const int cps = (nch + target - 1) / target;
    return (nch + cps - 1) / cps;
}

int bwd_splits(const Problem& p) { return p.causal ? causal_splits(p) : nc_splits(p); }

// Scratch layout (every region 256-byte aligned): dW partials [2 half][128][64], key
// weights [B*H*N] (prefactor), dtau partials [2 half]; non-causal and causal in ranges also
// partial states [2 half][128][80], non-causal totals [2 units][128][80] (half =
// B*H*G*nsplit, units = B*H*G).
struct BwdWs {
    size_t part, kw, dtau, state_part, state_total, total;
};
BwdWs bwd_ws(const Problem& p, int nsplit)
{
    const size_t units = (size_t)p.B * p.H * (p.M / 64);
    const size_t half = units * nsplit;
    auto a64 = [](size_t n) { return align_up(n, 64); };  // floats
    BwdWs w;
    w.part = 0;
    w.kw = a64(w.part + 2 * half * 128 * 64);
    w.dtau = a64(w.kw + (size_t)p.B * p.H * p.N);
    w.state_part = a64(w.dtau + 2 * half);
    w.state_total = a64(w.state_part + (p.causal && nsplit == 1 ? 0 : 2 * half * 128 * 80));
    w.total = a64(w.state_total + (p.causal ? 0 : 2 * units * 128 * 80));
    return w;  // in floats
}

struct BwdArgs {
    CUtensorMap mq, mk, mv, mdo, mo;
};

// One launch of tc_bwd_kernel<NS, KW, CS, MODE>: 2 * units * nsplit CTAs, clusters of CS.
template <bool NS, bool KW, int CS, int MODE>
cudaError_t launch_mode(const Problem& p, const BwdArgs& m, const void* q, const void* k,
                        const void* v, const float* W1, const float* W2, const float* tau,
                        const void* out, const float* den, const void* dout, void* dq, void* dk,
                        void* dv, float* f, const BwdWs& w, int nsplit, int* status,
                        cudaStream_t s)
{
    const int smem = (int)BwCfg<NS>::BYTES + 1024;
    auto kb = tc_bwd_kernel<NS, KW, CS, MODE>;
    cudaError_t e = cudaFuncSetAttribute(kb, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    typedef const __nv_bfloat16* CB;
    typedef __nv_bfloat16* B16;
    const int units = p.B * p.H * (p.M / 64);
    // (the first kernel of a call, without key weights, starts in stream order)
    const bool after = KW || MODE == kGrad || (MODE == kCausal && nsplit > 1);
    return launch_after(kb, dim3((unsigned)(2 * units * nsplit)), kThreadsB, smem, CS, after, s, m.mq, m.mk,
                        m.mv, m.mdo, m.mo, p.H, p.N, p.M, p.M / 64, (CB)q, (CB)k, (CB)v, W1,
                        W2, (CB)out, den, (CB)dout, (B16)dq, (B16)dk, (B16)dv, f + w.part,
                        KW ? (const float*)(f + w.kw) : (const float*)nullptr, tau, f + w.dtau, units,
                        nsplit, f + w.state_part, (const float*)(f + w.state_total), status);
}

template <bool NS, bool KW>
cudaError_t launch_bwd(const Problem& p, const void* q, const void* k, const void* v,
                       const float* W1, const float* W2, const float* tau, const void* out,
                       const float* den, const void* dout, void* dq, void* dk, void* dv,
                       float* dW1, float* dW2, float* dtau, void* scratch, int nsplit, int* status,
                       cudaStream_t s)
{
    const int BH = p.B * p.H, G = p.M / 64;
    float* f = static_cast<float*>(scratch);
    const BwdWs w = bwd_ws(p, nsplit);
    cudaError_t e = cudaSuccess;
    if (KW && (e = launch_key_weights(p, k, tau, f + w.kw, s)) != cudaSuccess) return e;
    BwdArgs m;
    if (!make_act_map(&m.mq, q, BH, p.N) || !make_act_map(&m.mk, k, BH, p.N) ||
        !make_act_map(&m.mv, v, BH, p.N) || !make_act_map(&m.mdo, dout, BH, p.N) ||
        !make_act_map(&m.mo, out, BH, p.N))
        return cudaErrorInvalidValue;
    const int units = BH * G;
    if (!p.causal || nsplit > 1) {
        e = launch_mode<NS, KW, 1, kState>(p, m, q, k, v, W1, W2, tau, out, den, dout, dq, dk, dv,
                                           f, w, nsplit, status, s);
        if (e != cudaSuccess) return e;
        const dim3 sgrid(2 * units, 128 * 17 / kStateThreads);
        e = p.causal ? launch_after(causal_state_scan_kernel, sgrid, kStateThreads, 0, 0, true, s, units,
                                    G, nsplit, f + w.state_part)
                     : launch_after(nc_state_reduce_kernel, sgrid, kStateThreads, 0, 0, true, s, units, G,
                                    nsplit, f + w.state_part, f + w.state_total);
        if (e != cudaSuccess) return e;
    }
    if (p.causal)
        e = G == 2 ? launch_mode<NS, KW, 2, kCausal>(p, m, q, k, v, W1, W2, tau, out, den, dout, dq,
                                                     dk, dv, f, w, nsplit, status, s)
                   : launch_mode<NS, KW, 1, kCausal>(p, m, q, k, v, W1, W2, tau, out, den, dout, dq,
                                                     dk, dv, f, w, nsplit, status, s);
    else
        e = G == 2 ? launch_mode<NS, KW, 2, kGrad>(p, m, q, k, v, W1, W2, tau, out, den, dout, dq,
                                                   dk, dv, f, w, nsplit, status, s)
                   : launch_mode<NS, KW, 1, kGrad>(p, m, q, k, v, W1, W2, tau, out, den, dout, dq,
                                                   dk, dv, f, w, nsplit, status, s);
    if (e != cudaSuccess) return e;
    auto reduce = wide_reduce(16LL * p.H * G) ? tc_dw_reduce_kernel<16> : tc_dw_reduce_kernel<8>;
    return launch_after(reduce, dim3((unsigned)(p.H * G * 16)), kReduceThreads, 0, 0, true, s,
                        p.B, p.H, p.M, G, nsplit, p.nonstat, (const float*)(f + w.part), dW1, dW2,
                        (const float*)(f + w.dtau), KW ? dtau : (float*)nullptr);
}

}  // namespace

// bf16, d = 64, M in {64, 128}: causal (two scans) and non-causal (totals, then every
// chunk independently).
bool tc_bwd_supported(const Problem& p)
{
    return p.bf16 && p.d == 64 && (p.M == 64 || p.M == 128);
}

// Ranges used with a workspace of `bytes`: one (the minimum a workspace has to hold in the
// causal mode) when the ranges' scratch does not fit.
static int tc_bwd_splits(const Problem& p, size_t bytes)
{
    const int ns = bwd_splits(p);
    return p.causal && bwd_ws(p, ns).total * sizeof(float) > bytes ? 1 : ns;
}

int tc_bwd_launches(const Problem& p, bool tau, size_t bytes)
{
    return (p.causal && tc_bwd_splits(p, bytes) == 1 ? 2 : 4) + (tau ? 1 : 0);
}

size_t tc_bwd_ws_bytes(const Problem& p, bool least)
{
    return bwd_ws(p, least && p.causal ? 1 : bwd_splits(p)).total * sizeof(float);
}

cudaError_t launch_tc_bwd(const Problem& p, const void* q, const void* k, const void* v,
                          const float* W1, const float* W2, const float* tau, const void* out,
                          const float* den, const void* dout, void* dq, void* dk, void* dv,
                          float* dW1, float* dW2, float* dtau, void* scratch, size_t bytes,
                          int* status, cudaStream_t s)
{
    const int ns = tc_bwd_splits(p, bytes);
#define FLEX_BWD_ARGS p, q, k, v, W1, W2, tau, out, den, dout, dq, dk, dv, dW1, dW2, dtau, scratch, ns, status, s
    if (p.nonstat)
        return tau ? launch_bwd<true, true>(FLEX_BWD_ARGS) : launch_bwd<true, false>(FLEX_BWD_ARGS);
    return tau ? launch_bwd<false, true>(FLEX_BWD_ARGS) : launch_bwd<false, false>(FLEX_BWD_ARGS);
#undef FLEX_BWD_ARGS
}

}  // namespace flex
