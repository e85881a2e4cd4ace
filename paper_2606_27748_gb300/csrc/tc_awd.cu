// Attention-weight distillation loss on the tensor cores.
//
// The loss of the softmax-recovery experiments (the appendix's distillation setting): per
// query i the teacher distribution P_ij = softmax_j(q_i . k_j / sqrt(d)) and the kernel's
// normalised weights R_ij = A~_ij / D_i, A~_ij = phi~(q_i) . phi~(k_j), D_i = sum_l A~_il;
//   L = -(1/N) sum_i sum_j P_ij log R_ij     (j over all keys, or j <= i when causal).
// The query's prefactor and the feature scale cancel in R, so A~ uses phi(q) and the
// weighted key features w_j phi(k_j) (both written by a feature pass before this kernel).
// Entries with a non-positive R_ij count log(1e-6) (RFF estimates and row sums can be
// negative; the logarithm is undefined there).
//
// One CTA per (sequence, block of 128 queries), 256 threads: TMA loads the query tile and
// its features once, then per block of 128 keys the key tile and its features (the next
// block's load is issued once the MMAs have read the current one, so it overlaps the
// epilogue); thread 0 issues S = Q K^T (K = d = 64) into T_S and A = phi(Q) phi~(K)^T
// (K = 2M) into T_A; every thread then takes half of one query row's 128 columns and keeps
// online statistics in base 2: the running maximum m of the scores, Z = sum 2^(s-m), and
// for positive and negative A separately Z+- = sum 2^(s-m) and T+- = sum 2^(s-m) log2|A|,
// and D = sum A.  At the end the two halves merge and, by the sign of D,
//   L_i = -(ln2 T_sign - Z_sign ln|D| + (Z - Z_sign) ln 1e-6) / Z,
// which is the definition with the reading above applied.  Block sums of L_i go to
// partial slots, summed per sequence in a fixed order.  Every wait is bounded.  For the
// gradient the same kernel also writes each row's statistics (below).
#include <algorithm>
#include <type_traits>

#include "flex_internal.h"
#include "tc_common.cuh"
#include "tc_util.cuh"

namespace flex {
namespace {
using namespace tc;

constexpr int kC = 128;
constexpr int kThreadsA = 256;
constexpr int kOnePerSm = 116 * 1024;  // more than half of an SM's 228 KB

template <int G2>  // 64-feature blocks of phi: 2M / 64
struct AwdCfg {
    static constexpr uint32_t Q = 0, K = 16384, PQ = 32768, PK = PQ + G2 * 16384;
    static constexpr uint32_t BYTES = PK + G2 * 16384;
    static constexpr uint32_t T_S = 0, T_A = 128;
    static_assert(BYTES + 1024 <= 232448, "shared memory budget");
};

__device__ __forceinline__ float ex2f(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2f(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcpf(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct Stats {
    float m, z, zp, zn, tp, tn, den;
};

template <int G2>
__global__ void __launch_bounds__(kThreadsA, 1)
    tc_awd_kernel(const __grid_constant__ CUtensorMap tmap_q,
                  const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_pq,
                  const __grid_constant__ CUtensorMap tmap_pk, int N, int causal,
                  float score_scale, int nqb, float* part,
                  float4* rowstat, int* status)
{
    using L = AwdCfg<G2>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sb = smem_u32(sm);
    __shared__ uint32_t tmem_base_sh;
    __shared__ __align__(8) uint64_t mbar, tma_bar;
    __shared__ volatile int abort_flag;
    __shared__ float merge[7][kC];
    __shared__ float wsum[kThreadsA / 32];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wg = warp >> 2, quad = warp & 3, t = 32 * quad + lane;
    const int bh = blockIdx.x / nqb, qb = blockIdx.x % nqb;
    const int row = qb * kC + t;

    if (tid == 0) {
        mbar_init(&mbar, 1);
        mbar_init(&tma_bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, 256);
        tmem_relinquish();
    }
    grid_dep_launch();
    grid_dep_wait();  // the feature maps
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tm = tmem_base_sh;
    const uint32_t tm_row = tm + ((uint32_t)(32 * quad) << 16);
    uint32_t phase = 0, tma_phase = 0;
    auto adv = [](uint64_t dsc, uint32_t bytes) { return dsc + (bytes >> 4); };
    const uint64_t dQ = sdesc(sb + L::Q, 16, 1024), dK = sdesc(sb + L::K, 16, 1024);
    const uint64_t dPQ = sdesc(sb + L::PQ, 16, 1024), dPK = sdesc(sb + L::PK, 16, 1024);
    constexpr uint32_t I_KK128 = idesc_bf16(128, 128, 0, 0);

    Stats st = {-INFINITY, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int nkb = causal ? qb + 1 : (N + kC - 1) / kC;
    bool ok = true;

    // key tiles of block kb (one arrival per phase; the first also brings the query side)
    auto load_keys = [&](int kb) {
        mbar_arrive_expect_tx(&tma_bar, (1 + G2) * kTileBytes * (kb == 0 ? 2 : 1));
        if (kb == 0) {
            tma_load_3d(sb + L::Q, &tmap_q, 0, qb * kC, bh, &tma_bar);
            for (int g = 0; g < G2; ++g)
                tma_load_3d(sb + L::PQ + g * 16384, &tmap_pq, 64 * g, qb * kC, bh, &tma_bar);
        }
        tma_load_3d(sb + L::K, &tmap_k, 0, kb * kC, bh, &tma_bar);
        for (int g = 0; g < G2; ++g)
            tma_load_3d(sb + L::PK + g * 16384, &tmap_pk, 64 * g, kb * kC, bh, &tma_bar);
    };
    if (tid == 0) load_keys(0);
    for (int kb = 0; kb < nkb && ok; ++kb) {
        ok = bar_wait(&tma_bar, tma_phase, &abort_flag, status);
        tma_phase ^= 1;
        ok = !__syncthreads_or(!ok);
        if (!ok) break;
        fence_after_sync();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_bf16(tm + L::T_S, adv(dQ, ks * 32), adv(dK, ks * 32), I_KK128, ks > 0);
#pragma unroll
            for (int ks = 0; ks < 4 * G2; ++ks) {
                const uint32_t kofs = (ks >> 2) * 16384 + (ks & 3) * 32;
                mma_bf16(tm + L::T_A, adv(dPQ, kofs), adv(dPK, kofs), I_KK128, ks > 0);
            }
            mma_commit(&mbar);
        }
        ok = bar_wait(&mbar, phase, &abort_flag, status);
        phase ^= 1;
        ok = !__syncthreads_or(!ok);
        if (!ok) break;
        fence_after_sync();
        // the MMAs have read the key tiles: the next block's load overlaps this epilogue
        if (tid == 0 && kb + 1 < nkb) load_keys(kb + 1);
        // statistics over this thread's 64 columns, two rounds of 32; a block with no
        // masked key (not the ragged last one, not on the causal diagonal) takes the
        // unmasked path (rows past N are computed and discarded at the end)
        const bool full = (kb + 1) * kC <= N && (!causal || kb < qb);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint32_t col = 64 * wg + 32 * b;
            float s[32], a[32];
            tmem_ld16(tm_row + L::T_S + col, *reinterpret_cast<float(*)[16]>(&s[0]));
            tmem_ld16(tm_row + L::T_S + col + 16, *reinterpret_cast<float(*)[16]>(&s[16]));
            tmem_ld16(tm_row + L::T_A + col, *reinterpret_cast<float(*)[16]>(&a[0]));
            tmem_ld16(tm_row + L::T_A + col + 16, *reinterpret_cast<float(*)[16]>(&a[16]));
            tmem_wait_ld();
            if (full) {  // no mask: every key of the block is valid for every row
                float bmax = s[0];
#pragma unroll
                for (int e = 1; e < 32; ++e) bmax = fmaxf(bmax, s[e]);
                bmax *= score_scale;  // > 0, so the maximum commutes with the scale
                if (bmax > st.m) {
                    const float f = ex2f(st.m - bmax);
                    st.z *= f; st.zp *= f; st.zn *= f; st.tp *= f; st.tn *= f;
                    st.m = bmax;
                }
                const float nm = -st.m;
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float p = ex2f(fmaf(s[e], score_scale, nm));
                    const float pl = p * lg2f(fabsf(a[e]));
                    st.z += p;
                    st.den += a[e];
                    if (a[e] > 0.f) { st.zp += p; st.tp += pl; }
                    if (a[e] < 0.f) { st.zn += p; st.tn += pl; }
                }
                continue;
            }
            const int j0 = kb * kC + (int)col;
            float bmax = -INFINITY;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const int j = j0 + e;
                const bool v = row < N && j < N && (!causal || j <= row);
                s[e] = v ? s[e] * score_scale : -INFINITY;
                bmax = fmaxf(bmax, s[e]);
            }
            if (bmax == -INFINITY) continue;  // no key of this round for this row
            if (bmax > st.m) {
                const float f = ex2f(st.m - bmax);  // 0 on the first valid round
                st.z *= f; st.zp *= f; st.zn *= f; st.tp *= f; st.tn *= f;
                st.m = bmax;
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                if (s[e] == -INFINITY) continue;
                const float p = ex2f(s[e] - st.m);
                st.z += p;
                st.den += a[e];
                if (a[e] > 0.f) {
                    st.zp += p;
                    st.tp = fmaf(p, lg2f(a[e]), st.tp);
                } else if (a[e] < 0.f) {
                    st.zn += p;
                    st.tn = fmaf(p, lg2f(-a[e]), st.tn);
                }
            }
        }
        // tensor memory and the key tiles are free once every thread is here
        fence_before_sync();
        __syncthreads();
    }

    // merge the two halves of each row (wg 1 hands its statistics to wg 0)
    float lsum = 0.f;
    if (ok) {
        if (wg == 1) {
            merge[0][t] = st.m; merge[1][t] = st.z; merge[2][t] = st.zp; merge[3][t] = st.zn;
            merge[4][t] = st.tp; merge[5][t] = st.tn; merge[6][t] = st.den;
        }
        __syncthreads();
        if (wg == 0 && row < N) {
            const float m2 = merge[0][t], m = fmaxf(st.m, m2);
            const float f1 = st.m == -INFINITY ? 0.f : ex2f(st.m - m);
            const float f2 = m2 == -INFINITY ? 0.f : ex2f(m2 - m);
            const float z = st.z * f1 + merge[1][t] * f2;
            const float zp = st.zp * f1 + merge[2][t] * f2, zn = st.zn * f1 + merge[3][t] * f2;
            const float tp = st.tp * f1 + merge[4][t] * f2, tn = st.tn * f1 + merge[5][t] * f2;
            const float den = st.den + merge[6][t];
            constexpr float kLn2 = 0.69314718055994531f, kLnEps = -13.815510557964274f;  // ln 1e-6
            float li;
            if (den > 0.f)
                li = -(kLn2 * tp - zp * logf(den) + (z - zp) * kLnEps) / z;
            else if (den < 0.f)
                li = -(kLn2 * tn - zn * logf(-den) + (z - zn) * kLnEps) / z;
            else
                li = -kLnEps;
            lsum = li;
            if (rowstat) {  // what the gradient needs of this row (see the gradient kernel)
                const float sg = den > 0.f ? 1.f : (den < 0.f ? -1.f : 0.f);
                const float zs = den > 0.f ? zp : zn;
                const float e = sg != 0.f ? (zs / z) / den : 0.f;
                rowstat[(size_t)bh * N + row] = make_float4(m + log2f(z), sg, e, 0.f);
            }
        }
    }
    // block sum in a fixed order
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) wsum[warp] = lsum;
    __syncthreads();
    if (tid == 0) {
        float tot = 0.f;
        for (int w8 = 0; w8 < kThreadsA / 32; ++w8) tot += wsum[w8];
        part[blockIdx.x] = tot;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 0) {
        drain_after_abort(!ok);
        tmem_dealloc(tm, 256);
    }
}

__global__ void awd_reduce_kernel(int BH, int nqb, int N, const float* part,
                                  float* __restrict__ loss)
{
    grid_dep_launch();
    grid_dep_wait();
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < BH; u += gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int b = 0; b < nqb; ++b) s += part[(size_t)u * nqb + b];  // fixed order
        loss[u] = s / (float)N;
    }
}

// ---- gradient with respect to the kernel's parameters ------------------------------------
//
// The distillation trains only the feature map, so the gradient is taken with respect to
// W1, W2 and tau.  With the row statistics of the loss kernel (l_i = log2 of the softmax
// normaliser in the scaled base-2 scores, the sign of D_i, e_i = c_i / D_i where c_i is the
// teacher mass on the entries with R_ij > 0) and sigma = -dloss / N:
//   dL/dA~_ij = sigma G_ij,   G_ij = [A~_ij sign(D_i) > 0] P_ij / A~_ij - e_i   (j in row i)
//   dphi(q_i) = sigma sum_j G_ij phi~(k_j),   dphi~(k_j) = sigma sum_i G_ij phi(q_i).
// A sequence's query side holds blocks of 128 queries and streams the key blocks; its key
// side holds blocks of 128 keys and streams the query blocks; each side's held blocks are
// split over `hsplit` CTAs.  The other side's rows are streamed 64 at a time: S = X_own
// X_other^T and A = Phi_own Phi_other^T into one of two tensor-memory buffers, the buffer's
// group of 8 compute warps turns them into G (ex2 and a reciprocal an entry), writes it as
// bf16 in place over A, and G Phi_other (A operand in tensor memory, features MN-major)
// accumulates into T_D.  A loader warp and an issuing warp run ahead of the compute warps,
// which only meet them at mbarriers.  M = 64: the held block's x and features are tensor-memory
// operands and the next held block is loaded meanwhile.  Then, per group of 64 frequencies, the
// chain rule through the feature map runs on the tensor cores: the projection X_own W'^T is
// recomputed, the epilogue forms da (du | dw for Flexformer_n) from T_D, and dW' += da^T X_own.
// What bounds it: per step of 128 x 64 entries the 16 small MMAs (about 0.4 us) and the two
// groups' arithmetic (0.7 us each, overlapping); per CTA about a third of the time is set-up
// and the chain rule.  Measured, one distillation step n B32 H8 N512 M64: 361 us with all
// warps in step and thread 0 issuing, 307 us now (mask and side as compile-time cases 357 ->
// 333, the held block as a tensor-memory operand -> 324, loads by their own warp -> 307); 281 with
// overlapped launches, the feature pass's 32-byte stores and the wider sum of the slots (12.7 ->
// 9 us), 196 of them here.  The rows of dW' are added into this CTA's slot; a reduction sums the
// slots over the sides, the batch and the splits in a fixed order, so the result does not depend on scheduling.  On the
// key side, with the prefactor, the chain rule takes dphi(k_j) = w_j dphi~(k_j) and dtau
// gains -(phi~(k_j) . dphi~(k_j)) |k_j|^2 exp(-tau).  Every wait is bounded.
constexpr int kComputeG = 16;                    // compute warps, four per lane quadrant
constexpr int kThreadsG = 32 * kComputeG + 64;   // and the issuer's and the loader's warps
constexpr int kHalf = 64;                        // streamed rows per step
template <int G2>
struct AwdBwCfg {
    // M = 64 has tensor memory left for the held block's x and features (bf16) as operands, so
    // every step's S and A read only the streamed rows from shared memory; it also has two
    // buffers for held blocks, the features' place taking da once they are copied.
    static constexpr bool OWN_T = G2 == 2;
    static constexpr int STAGES = OWN_T ? 4 : 2, OWN = OWN_T ? 2 : 1;  // steps, blocks in flight
    static constexpr uint32_t OWN_BYTES = (1 + G2) * 16384;     // x tile, then features
    static constexpr uint32_t ST0 = OWN * OWN_BYTES;
    static constexpr uint32_t STAGE_BYTES = (1 + G2) * 8192;    // x rows, then features
    static constexpr uint32_t WG = ST0 + STAGES * STAGE_BYTES;  // W' rows of every group
    static constexpr uint32_t BYTES = WG + (G2 / 2) * 16384;    // (at most 16 KB a group)
    __host__ __device__ static constexpr uint32_t XO(int ob) { return OWN_T ? (uint32_t)(ob & 1) * OWN_BYTES : 0u; }
    __host__ __device__ static constexpr uint32_t PO(int ob) { return XO(ob) + 16384; }
    // da [du | dw], after the streamed steps
    __host__ __device__ static constexpr uint32_t DA(int ob) { return OWN_T ? PO(ob) : ST0; }
    // tensor memory: two buffers of S (64 columns) and A (64), the projection and dW' of the
    // chain rule over them, dphi
    static constexpr uint32_t T_SA = 0, T_C = 0, T_W = 128, T_D = 256;
    static constexpr uint32_t T_XO = 384, T_PO = 416;
    static_assert(G2 >= 2 && BYTES + 1024 <= 232448, "shared memory budget");
    static_assert(OWN_T || STAGES * STAGE_BYTES >= 32768, "da fits the stages");
};

template <int G2, bool NS, bool KW>
__global__ void __launch_bounds__(kThreadsG, 1)
    tc_awd_bwd_kernel(const __grid_constant__ CUtensorMap tmap_q,
                      const __grid_constant__ CUtensorMap tmap_k,
                      const __grid_constant__ CUtensorMap tmap_pq,
                      const __grid_constant__ CUtensorMap tmap_pk, int BH, int H, int N, int M,
                      int causal, int hsplit, float score_scale,
                      const float4* rowstat, const float* __restrict__ dloss,
                      const float* __restrict__ W1, const float* __restrict__ W2,
                      const float* kw, const float* __restrict__ tau,
                      float* slots, float* dtau_part, int* status)
{
    using L = AwdBwCfg<G2>;
    constexpr int P = NS ? 128 : 64;  // projection rows per group of 64 frequencies
    constexpr int G = G2 / 2;
    constexpr int ST = L::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sb = smem_u32(sm);
    __shared__ uint32_t tmem_base_sh;
    // tiles landed: town[buffer] (held block), tx[stage]; their last use done: ofree, sfree; one arrival per compute warp: rdy[buffer] (G of
    // a step, from the group of warps that takes that buffer's steps), rdyc (start of a held block, chain rule); MMA groups complete: msa[buffer]
    // (S and A of a step), md (dphi of a step), mc (chain rule)
    __shared__ __align__(8) uint64_t town[L::OWN], ofree[L::OWN], tx[ST], sfree[ST], rdy[2],
        rdyc, msa[2], md, mc;
    __shared__ volatile int abort_flag;
    __shared__ float4 ostat[4][kHalf];  // key side: statistics of the streamed query rows
    __shared__ float wsum[kThreadsG / 32];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int qd = warp >> 2, quad = warp & 3, t = 32 * quad + lane;  // qd: column quarter
    const int seq = (int)blockIdx.x / hsplit, split = (int)blockIdx.x % hsplit;
    const bool kside = seq >= BH;
    const int bh = seq % BH, h = bh % H;
    const CUtensorMap* x_own = kside ? &tmap_k : &tmap_q;
    const CUtensorMap* x_oth = kside ? &tmap_q : &tmap_k;
    const CUtensorMap* f_own = kside ? &tmap_pk : &tmap_pq;
    const CUtensorMap* f_oth = kside ? &tmap_pq : &tmap_pk;
    const int nblk = (N + kC - 1) / kC, nhalf = (N + kHalf - 1) / kHalf;
    const int hb0 = split * nblk / hsplit, hb1 = (split + 1) * nblk / hsplit;
    const float sigma = -dloss[bh] / (float)N;
    const float itau = KW ? expf(-tau[h]) : 0.f;
    const float cM = rsqrtf((float)M);
    float dtau_acc = 0.f;

    if (tid == 0) {
        for (int s = 0; s < L::OWN; ++s) {
            mbar_init(&town[s], 1);
            mbar_init(&ofree[s], 1);
        }
        for (int s = 0; s < ST; ++s) {
            mbar_init(&tx[s], 1);
            mbar_init(&sfree[s], 1);
        }
        mbar_init(&rdy[0], kComputeG / 2);
        mbar_init(&rdy[1], kComputeG / 2);
        mbar_init(&rdyc, kComputeG);
        for (uint64_t* b : {&msa[0], &msa[1], &md, &mc}) mbar_init(b, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_sh, 512);
        tmem_relinquish();
    }
    // this head's W' rows, all groups, once
    if (warp < kComputeG) stage_freq_rows<NS, G, 32 * kComputeG>(sb + L::WG, W1, W2, h, M, tid);
    grid_dep_launch();
    grid_dep_wait();  // the feature maps, the rows' statistics
    fence_proxy_async();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tm = tmem_base_sh;
    const uint32_t tm_row = tm + ((uint32_t)(32 * quad) << 16);
    auto wwait = [&](uint64_t* bar, uint32_t& ph) -> bool {  // a whole warp, one verdict
        const bool ok = bar_wait_w(bar, ph, &abort_flag, status);
        ph ^= 1;
        fence_after_sync();
        return ok;
    };
    auto arrive = [&](uint64_t* bar) {  // this warp's shared- and tensor-memory accesses are done
        fence_proxy_async();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    // streamed steps (64 rows) of held block ob: causal queries see keys j <= i
    auto first_step = [&](int ob) { return (kside && causal) ? 2 * ob : 0; };
    auto last_step = [&](int ob) { return (!kside && causal) ? min(nhalf, 2 * ob + 2) : nhalf; };

    if (warp == kComputeG + 1) {
        // ================= loader (a tile load takes the issuing warp about 0.2 us) ==========
        [&]() {
            int gs = 0;  // steps loaded so far: stage gs % ST
            for (int ob = hb0; ob < hb1; ++ob) {
                const int io = ob - hb0, b = io % L::OWN;
                if (io >= L::OWN && !bar_wait_w(&ofree[b], (io / L::OWN - 1) & 1, &abort_flag, status))
                    return;
                const uint32_t xo = sb + L::XO(io);
                wmbar_arrive_expect_tx(&town[b], L::OWN_BYTES);
                for (int r = 0; r < 2; ++r) {  // (64-row boxes)
                    wtma_load_3d(xo + r * 8192, x_own, 0, ob * kC + r * 64, bh, &town[b]);
                    for (int g = 0; g < G2; ++g)
                        wtma_load_3d(xo + 16384 + g * 16384 + r * 8192, f_own, 64 * g, ob * kC + r * 64, bh,
                                     &town[b]);
                }
                const int n = last_step(ob) - first_step(ob);
                for (int j = 0; j < n; ++j, ++gs) {
                    const int st = gs % ST;
                    if (gs >= ST && !bar_wait_w(&sfree[st], (gs / ST - 1) & 1, &abort_flag, status)) return;
                    const uint32_t dst = sb + L::ST0 + (uint32_t)st * L::STAGE_BYTES;
                    const int r0 = (first_step(ob) + j) * kHalf;
                    wmbar_arrive_expect_tx(&tx[st], L::STAGE_BYTES);
                    wtma_load_3d(dst, x_oth, 0, r0, bh, &tx[st]);
                    for (int g = 0; g < G2; ++g)
                        wtma_load_3d(dst + 8192 + g * 8192, f_oth, 64 * g, r0, bh, &tx[st]);
                }
            }
        }();
        __syncwarp();
    } else if (warp == kComputeG) {
        // ================= issuer (a whole warp, one elected lane per operation) =============
        constexpr uint32_t I_S = idesc_bf16(128, kHalf, 0, 0);
        constexpr uint32_t I_DPHI = idesc_bf16(128, 64 * G2, 0, 1);  // N = 2M features
        constexpr uint32_t I_PROJ = idesc_bf16(128, P, 0, 0);
        constexpr uint32_t I_DW = idesc_bf16(128, 64, 1, 1);
        [&]() {
            auto adv = [](uint64_t dsc, uint32_t bytes) { return dsc + (bytes >> 4); };
            uint32_t p_rdy[2] = {0, 0}, p_rdyc = 0, p_md = 0, p_mc = 0;
            int gs0 = 0;  // steps of the earlier held blocks
            for (int ob = hb0; ob < hb1; ++ob) {
                const int io = ob - hb0, n = last_step(ob) - first_step(ob);
                const uint32_t xo = sb + L::XO(io), po = sb + L::PO(io);
                const uint64_t dXO = sdesc(xo, 16, 1024), dPO = sdesc(po, 16, 1024);
                const uint64_t dXOmn = sdesc(xo, 16384, 1024);
                const uint64_t dDAmn = sdesc(sb + L::DA(io), 16384, 1024);
                // dphi += G Phi of step j (G bf16 over its A columns, 16 keys in 8 columns)
                auto issue_dphi = [&](int j) {
                    const uint64_t dPT = sdesc(
                        sb + L::ST0 + (uint32_t)((gs0 + j) % ST) * L::STAGE_BYTES + 8192, 8192, 1024);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        wmma_bf16_tmem_a(tm + L::T_D, tm + L::T_SA + 128 * (j & 1) + 64 + 16 * ks,
                                         adv(dPT, ks * 2048), I_DPHI, (j > 0 || ks > 0) ? 1u : 0u);
                    wmma_commit(&md);
                    wmma_commit(&sfree[(gs0 + j) % ST]);
                };
                // the compute warps are done with the previous held block (M = 64: and this one
                // is in tensor memory)
                if (!wwait(&rdyc, p_rdyc)) return;
                if (!bar_wait_w(&town[io % L::OWN], (io / L::OWN) & 1, &abort_flag, status)) return;
                fence_after_sync();
                for (int j = 0; j <= n; ++j) {
                    // (waited for before the next commit on md)
                    if (j >= 2 && !wwait(&md, p_md)) return;
                    if (j < n) {
                        const int gs = gs0 + j, st = gs % ST;
                        if (!bar_wait_w(&tx[st], (gs / ST) & 1, &abort_flag, status)) return;
                        fence_after_sync();
                        // (step j - 2's dphi, which reads this buffer, is complete)
                        const uint32_t sa = tm + L::T_SA + 128 * (j & 1);
                        const uint32_t xs = sb + L::ST0 + (uint32_t)st * L::STAGE_BYTES;
                        const uint64_t dXT = sdesc(xs, 16, 1024), dPT = sdesc(xs + 8192, 16, 1024);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            if (L::OWN_T)
                                wmma_bf16_tmem_a(sa, tm + L::T_XO + 8 * ks, adv(dXT, ks * 32), I_S, ks > 0);
                            else
                                wmma_bf16(sa, adv(dXO, ks * 32), adv(dXT, ks * 32), I_S, ks > 0);
                        }
#pragma unroll
                        for (int ks = 0; ks < 4 * G2; ++ks) {
                            const uint64_t pt = adv(dPT, (ks >> 2) * 8192 + (ks & 3) * 32);
                            if (L::OWN_T)
                                wmma_bf16_tmem_a(sa + 64, tm + L::T_PO + 8 * ks, pt, I_S, ks > 0);
                            else
                                wmma_bf16(sa + 64, adv(dPO, (ks >> 2) * 16384 + (ks & 3) * 32), pt, I_S,
                                          ks > 0);
                        }
                        wmma_commit(&msa[j & 1]);
                    }
                    if (j > 0) {
                        if (!wwait(&rdy[(j - 1) & 1], p_rdy[(j - 1) & 1])) return;  // G of step j - 1
                        issue_dphi(j - 1);
                    }
                }
                // chain rule through the feature map, one group of 64 frequencies at a time; it
                // writes over the buffer the last step's dphi reads
                if (!wwait(&md, p_md)) return;
                for (int g = 0; g < G; ++g) {
                    if (g > 0 && !wwait(&rdyc, p_rdyc)) return;  // the previous group's dW' is read
                    const uint64_t dWg = sdesc(sb + L::WG + (uint32_t)g * P * 128, 16, 1024);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        wmma_bf16(tm + L::T_C, adv(dXO, ks * 32), adv(dWg, ks * 32), I_PROJ, ks > 0);
                    wmma_commit(&mc);
                    p_mc ^= 1;
                    if (!wwait(&rdyc, p_rdyc)) return;  // da
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        wmma_bf16(tm + L::T_W, adv(dDAmn, ks * 2048), adv(dXOmn, ks * 2048), I_DW, ks > 0);
                    wmma_commit(&mc);
                    if (g + 1 == G) wmma_commit(&ofree[io % L::OWN]);
                    if (!wwait(&mc, p_mc)) return;
                }
                gs0 += n;
            }
        }();
        __syncwarp();
    } else {
        // ================= compute =================
        // Steps: warps 0-7 take the even ones, 8-15 the odd ones (their tensor-memory latency
        // then falls into the other group's arithmetic), a warp 32 of the 64 columns.
        const int grp = warp / (kComputeG / 2);
        uint32_t p_own[2] = {0, 0}, p_msa = 0, p_mc = 0;
        for (int ob = hb0; ob < hb1; ++ob) {
            const int own_row = ob * kC + t;
            const bool own_valid = own_row < N;
            const int o0 = first_step(ob), n = last_step(ob) - o0;
            float4 qs = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!kside && own_valid) qs = rowstat[(size_t)bh * N + own_row];
            // Key side: the streamed queries' statistics of step j, written by the group that
            // takes it while that group's previous step runs (its other warps are past step
            // j - 4, which had the slot).
            auto stage_stat = [&](int j) {
                const int c = tid & (32 * kComputeG / 2 - 1);
                if (kside && c < kHalf && j < n) {
                    const int r = (o0 + j) * kHalf + c;
                    ostat[j & 3][c] =
                        r < N ? rowstat[(size_t)bh * N + r] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            };
            stage_stat(grp);
            if (!L::OWN_T) arrive(&rdyc);
            const int ow = L::OWN_T ? (ob - hb0) & 1 : 0;
            const uint32_t xo = L::XO(ob - hb0), po = L::PO(ob - hb0), da = sb + L::DA(ob - hb0);
            if (!wwait(&town[ow], p_own[ow])) goto done;
            if (L::OWN_T) {  // row t: x columns 16 qd .. + 15, features 32 qd .. + 31
                auto to_tmem = [&](uint32_t src, uint32_t col, int chunk) {  // 16 values
                    uint32_t r[8];
                    *reinterpret_cast<uint4*>(&r[0]) =
                        *reinterpret_cast<const uint4*>(sm + src + swz128(t, 8 * chunk));
                    *reinterpret_cast<uint4*>(&r[4]) =
                        *reinterpret_cast<const uint4*>(sm + src + swz128(t, 8 * chunk + 8));
                    tmem_st8(tm_row + col, r);
                };
                to_tmem(xo, L::T_XO + 8 * qd, 2 * qd);
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    to_tmem(po + (qd >> 1) * 16384, L::T_PO + 16 * qd + 8 * b, 4 * (qd & 1) + 2 * b);
                tmem_wait_st();
                arrive(&rdyc);
            }
            float kk = 0.f;  // key side: |k_j|^2 from the held tile
            if (KW && kside) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint4 k4 = *reinterpret_cast<const uint4*>(sm + xo + swz128(t, 8 * j));
                    const uint32_t kw4[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float k0 = __uint_as_float(kw4[e] << 16);
                        const float k1 = __uint_as_float(kw4[e] & 0xFFFF0000u);
                        kk = fmaf(k0, k0, fmaf(k1, k1, kk));
                    }
                }
            }
            for (int j = grp; j < n; j += 2) {
                if (!wwait(&msa[grp], p_msa)) goto done;
                stage_stat(j + 2);
                // G over this warp's 32 columns, sixteen at a time, bf16 over the first 8 of the
                // sixteen in A; a step with no masked entry skips the mask tests.  The step's
                // two conditions are compile-time: tested per entry they cost as much as G.
                const int r0 = (o0 + j) * kHalf;
                const bool full = r0 + kHalf <= N && (ob + 1) * kC <= N &&
                                  (!causal || (kside ? r0 >= ob * kC + kC - 1 : r0 + kHalf - 1 <= ob * kC));
                auto form_g = [&](auto full_tag, auto kside_tag) {
                    constexpr bool FULL = decltype(full_tag)::value, KS = decltype(kside_tag)::value;
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const int c0 = 32 * (qd & 1) + 16 * b;
                        const uint32_t sa = tm_row + L::T_SA + 128 * grp + c0;
                        float sv[16], av[16];
                        tmem_ld16(sa, sv);
                        tmem_ld16(sa + 64, av);
                        tmem_wait_ld();
                        uint32_t pk[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float gv[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const int c = c0 + 2 * i + e;
                                const float4 sts = KS ? ostat[j & 3][c] : qs;
                                const float a = av[2 * i + e];
                                const float p = ex2f(fmaf(sv[2 * i + e], score_scale, -sts.x));
                                // (branch-free: what p / a gives at a <= 0 is not used)
                                gv[e] = (a * sts.y > 0.f ? p * rcpf(a) : 0.f) - sts.z;
                                if (!FULL) {
                                    const int orow = r0 + c;
                                    const int qi = KS ? orow : own_row, kj = KS ? own_row : orow;
                                    if (!(own_valid && orow < N && (!causal || kj <= qi))) gv[e] = 0.f;
                                }
                            }
                            pk[i] = pack_bf16(gv[0], gv[1]);
                        }
                        tmem_st8(sa + 64, pk);
                    }
                };
                if (kside)
                    full ? form_g(std::true_type{}, std::true_type{})
                         : form_g(std::false_type{}, std::true_type{});
                else
                    full ? form_g(std::true_type{}, std::false_type{})
                         : form_g(std::false_type{}, std::false_type{});
                tmem_wait_st();
                arrive(&rdy[grp]);
            }
            const float wk = (KW && kside && own_valid) ? kw[(size_t)bh * N + own_row] : 1.f;
            const float scl = sigma * wk;  // dphi(x) = scl T_D (key side: dphi = w dphi~)
            float sdot = 0.f;              // key side: phi(k) . T_D over this thread's features
            for (int g = 0; g < G; ++g) {
                if (!wwait(&mc, p_mc)) goto done;  // dphi complete, the projection of group g
                // this thread's 16 frequencies of the group: 64 g + 16 qd + [0, 16)
                float dc[16], ds[16], u[16], w[16];
                tmem_ld16(tm_row + L::T_D + 64 * g + 16 * qd, dc);
                tmem_ld16(tm_row + L::T_D + M + 64 * g + 16 * qd, ds);
                float mu, mw = 0.f;  // max |x| per load
                tmem_ld16_maxabs(tm_row + L::T_C + 16 * qd, u, mu);
                if (NS) tmem_ld16_maxabs(tm_row + L::T_C + 64 + 16 * qd, w, mw);
                tmem_wait_ld();
                if (NS)
                    reduce_2pi_if_needed(u, w, fmaxf(mu, mw));
                else
                    reduce_2pi_if_needed(u, mu);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint32_t o1[4], o2[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float r1[2], r2[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int f = 8 * j + 2 * i + e;
                            float su, cu;
                            __sincosf(u[f], &su, &cu);
                            float cw = 1.f, sw = 0.f;
                            if (NS) __sincosf(w[f], &sw, &cw);
                            const float dpc = scl * dc[f], dps = scl * ds[f];
                            r1[e] = cM * cw * (-su * dpc + cu * dps);
                            r2[e] = NS ? -cM * sw * (cu * dpc + su * dps) : 0.f;
                            if (KW) sdot = fmaf(cu * cw, dc[f], fmaf(su * cw, ds[f], sdot));
                            if (!own_valid) r1[e] = r2[e] = 0.f;
                        }
                        o1[i] = pack_bf16(r1[0], r1[1]);
                        o2[i] = pack_bf16(r2[0], r2[1]);
                    }
                    const uint32_t off = swz128(t, (2 * qd + j) * 8);
                    st_shared_v4(da + off, o1[0], o1[1], o1[2], o1[3]);
                    st_shared_v4(da + 16384 + off, o2[0], o2[1], o2[2], o2[3]);
                }
                arrive(&rdyc);
                if (!wwait(&mc, p_mc)) goto done;
                // rows of dW' (lane = projection row), this thread's 16 columns, into the slot
                // ([16 column quads][128 rows][4]: a warp's accesses are contiguous)
                float v[16];
                tmem_ld16(tm_row + L::T_W + 16 * qd, v);
                tmem_wait_ld();
                float4* dst = reinterpret_cast<float4*>(slots) +
                              (((size_t)blockIdx.x * G + g) * 16 + 4 * qd) * 128 + t;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 old = ob == hb0 ? make_float4(0.f, 0.f, 0.f, 0.f) : dst[128 * j];
                    dst[128 * j] = make_float4(old.x + v[4 * j], old.y + v[4 * j + 1],
                                               old.z + v[4 * j + 2], old.w + v[4 * j + 3]);
                }
                if (g + 1 < G) arrive(&rdyc);  // (after the last group: the next block's arrival)
            }
            if (KW && kside && own_valid)  // s_j = phi~(k_j) . dphi~(k_j) = w cM sigma sdot
                dtau_acc -= wk * cM * sigma * sdot * kk * itau;
        }
    }

done:
    __syncthreads();
    if (tid == 0) drain_after_abort(abort_flag != 0);
    // dtau partial of this CTA, summed in a fixed order
    float dsum = dtau_acc;
    for (int o = 16; o > 0; o >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
    if (lane == 0) wsum[warp] = dsum;
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (tid == 0) {
        float tot = 0.f;
        for (int w8 = 0; w8 < kComputeG; ++w8) tot += wsum[w8];
        dtau_part[blockIdx.x] = tot;
    }
    if (warp == 0) tmem_dealloc(tm, 512);
}

// dW1, dW2 [H][M][64] and dtau [H] from the slots [2 sides][B*H][hsplit][G][16 column
// quads][128 rows][4].  One block per (head, group, column quad): thread (row, lane) sums
// every fourth slot (slots in (side, batch entry, split) order) with LD loads in flight;
// the four lanes are then added in order.  For Flexformer_n rows 0-63 of a group are dU, rows
// 64-127 dV (U = (W1+W2)/2, V = (W1-W2)/2), so dW1 = (dU+dV)/2, dW2 = (dU-dV)/2.
constexpr int kReduceThreads = 512;
template <int LD>  // loads in flight per thread (wide_reduce)
__global__ void __launch_bounds__(kReduceThreads)
    awd_dw_reduce_kernel(int B, int H, int M, int nonstat, int hsplit,
                         const float* slots, const float* dtau_part,
                         float* __restrict__ dW1, float* __restrict__ dW2,
                         float* __restrict__ dtau)
{
    grid_dep_wait();
    __shared__ float4 sums[3][128];
    const int BH = B * H, G = M / 64, per_side = B * hsplit;
    const int quad = blockIdx.x % 16, g = blockIdx.x / 16 % G, h = blockIdx.x / (16 * G);
    const int row = threadIdx.x % 128, ln = threadIdx.x / 128;
    auto add = [](float4& a, const float4& x) {
        a = make_float4(a.x + x.x, a.y + x.y, a.z + x.z, a.w + x.w);
    };
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    // slot i = bb hsplit + sp, bb = side B + b < 2 B; from one slot to the fourth after it
    // without a division
    const int dbb = 4 / hsplit, dsp = 4 % hsplit;
    int bb = ln / hsplit, sp = ln % hsplit;
    while (bb < 2 * B) {
        float4 x[LD];
#pragma unroll
        for (int e = 0; e < LD; ++e) {
            const size_t cta = (size_t)(bb * H + h) * hsplit + sp;
            x[e] = bb < 2 * B ? reinterpret_cast<const float4*>(slots)[((cta * G + g) * 16 + quad) * 128 + row]
                              : make_float4(0.f, 0.f, 0.f, 0.f);
            bb += dbb;
            sp += dsp;
            if (sp >= hsplit) {
                sp -= hsplit;
                ++bb;
            }
        }
#pragma unroll
        for (int e = 0; e < LD; ++e) add(a, x[e]);
    }
    if (ln > 0) sums[ln - 1][row] = a;
    __syncthreads();
    if (ln == 0) {
        for (int l = 0; l < 3; ++l) add(a, sums[l][row]);
        if (row >= 64) sums[0][row] = a;
    }
    __syncthreads();
    if (ln == 0 && row < 64) {
        const size_t o = (((size_t)h * M + 64 * g + row) * 64 + 4 * quad) / 4;
        if (nonstat) {
            const float4 b = sums[0][64 + row];
            reinterpret_cast<float4*>(dW1)[o] = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y),
                                                            0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
            reinterpret_cast<float4*>(dW2)[o] = make_float4(0.5f * (a.x - b.x), 0.5f * (a.y - b.y),
                                                            0.5f * (a.z - b.z), 0.5f * (a.w - b.w));
        } else {
            reinterpret_cast<float4*>(dW1)[o] = a;
        }
    }
    if (dtau && quad == 0 && g == 0 && threadIdx.x < 32) {  // the key side's partials of head h
        float t = 0.f;
        for (int i = threadIdx.x; i < per_side; i += 32)
            t += dtau_part[(size_t)(BH + i / hsplit * H + h) * hsplit + i % hsplit];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) dtau[h] = t;
    }
}

template <int G2>
cudaError_t launch_typed(const Problem& p, const void* q, const void* k, const void* pq,
                         const void* pk, float* part, float* loss, float4* rowstat, int* status,
                         cudaStream_t s)
{
    const int BH = p.B * p.H, nqb = (p.N + kC - 1) / kC;
    CUtensorMap mq, mk, mpq, mpk;
    if (!make_act_map(&mq, q, BH, p.N) || !make_act_map(&mk, k, BH, p.N) ||
        !make_feat_map(&mpq, pq, BH, p.N, 2 * p.M) || !make_feat_map(&mpk, pk, BH, p.N, 2 * p.M))
        return cudaErrorInvalidValue;
    // A grid of at most one block an SM asks for so much shared memory that an SM takes one
    // (M = 64 would fit two): it starts while the feature map's blocks still leave, on whatever
    // SMs are free by then, and pairs on some of them leave others idle.  Loss of one sequence, n,
    // N 16384 M 64 (128 blocks): 375 us, 248 with one block an SM.
    int smem = (int)AwdCfg<G2>::BYTES + 1024;
    if ((long long)BH * nqb <= sm_count()) smem = std::max(smem, kOnePerSm);
    auto kern = tc_awd_kernel<G2>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const float score_scale = 1.4426950408889634f / sqrtf((float)p.d);  // log2(e) / sqrt(d)
    e = launch_after(kern, dim3((unsigned)(BH * nqb)), kThreadsA, smem, 0, true, s, mq, mk, mpq, mpk, p.N,
                     p.causal, score_scale, nqb, part, rowstat, status);
    if (e != cudaSuccess || !loss) return e;
    return launch_after(awd_reduce_kernel, dim3((BH + 255) / 256), 256, 0, 0, true, s, BH, nqb, p.N,
                        (const float*)part, loss);
}

// CTAs per (side, sequence) of the gradient kernel: held blocks are split until the grid
// covers the GPU about four times over (whole blocks per CTA).
int awd_hsplit(const Problem& p)
{
    const int nblk = (p.N + kC - 1) / kC;
    int hs = 1;
    while (hs * 2 <= nblk && 2LL * p.B * p.H * hs < 4LL * 152) hs *= 2;
    return hs;
}

template <int G2, bool NS, bool KW>
cudaError_t launch_bwd_typed(const Problem& p, const void* q, const void* k, const void* pq,
                             const void* pk, const float* W1, const float* W2, const float* kw,
                             const float* tau, const float* dloss, const float4* rowstat,
                             float* slots, float* dtau_part, float* dW1, float* dW2, float* dtau,
                             int* status, cudaStream_t s)
{
    const int BH = p.B * p.H;
    CUtensorMap mq, mk, mpq, mpk;
    if (!make_feat_map(&mq, q, BH, p.N, 64, kHalf) || !make_feat_map(&mk, k, BH, p.N, 64, kHalf) ||
        !make_feat_map(&mpq, pq, BH, p.N, 2 * p.M, kHalf) ||
        !make_feat_map(&mpk, pk, BH, p.N, 2 * p.M, kHalf))
        return cudaErrorInvalidValue;
    const int smem = (int)AwdBwCfg<G2>::BYTES + 1024;
    auto kern = tc_awd_bwd_kernel<G2, NS, KW>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const float score_scale = 1.4426950408889634f / sqrtf((float)p.d);
    const int hs = awd_hsplit(p);
    e = launch_after(kern, dim3((unsigned)(2 * BH * hs)), kThreadsG, smem, 0, true, s, mq, mk, mpq, mpk, BH,
                     p.H, p.N, p.M, p.causal, hs, score_scale, rowstat, dloss, W1, W2, kw, tau, slots,
                     dtau_part, status);
    if (e != cudaSuccess) return e;
    const long long blocks = 16LL * p.H * (p.M / 64);
    auto reduce = wide_reduce(blocks) ? awd_dw_reduce_kernel<16> : awd_dw_reduce_kernel<8>;
    return launch_after(reduce, dim3((unsigned)blocks), kReduceThreads, 0, 0, true, s, p.B, p.H, p.M,
                        p.nonstat, hs, (const float*)slots, (const float*)dtau_part, dW1, dW2,
                        tau ? dtau : (float*)nullptr);
}

template <int G2>
cudaError_t launch_bwd_g2(const Problem& p, const void* q, const void* k, const void* pq,
                          const void* pk, const float* W1, const float* W2, const float* kw,
                          const float* tau, const float* dloss, const float4* rowstat,
                          float* slots, float* dtau_part, float* dW1, float* dW2, float* dtau,
                          int* status, cudaStream_t s)
{
    if (p.nonstat)
        return tau ? launch_bwd_typed<G2, true, true>(p, q, k, pq, pk, W1, W2, kw, tau, dloss,
                                                      rowstat, slots, dtau_part, dW1, dW2, dtau,
                                                      status, s)
                   : launch_bwd_typed<G2, true, false>(p, q, k, pq, pk, W1, W2, kw, tau, dloss,
                                                       rowstat, slots, dtau_part, dW1, dW2, dtau,
                                                       status, s);
    return tau ? launch_bwd_typed<G2, false, true>(p, q, k, pq, pk, W1, W2, kw, tau, dloss,
                                                   rowstat, slots, dtau_part, dW1, dW2, dtau,
                                                   status, s)
               : launch_bwd_typed<G2, false, false>(p, q, k, pq, pk, W1, W2, kw, tau, dloss,
                                                    rowstat, slots, dtau_part, dW1, dW2, dtau,
                                                    status, s);
}

}  // namespace

bool tc_awd_supported(const Problem& p)
{
    return p.bf16 && p.d == 64 && (p.M == 64 || p.M == 128);
}

size_t tc_awd_part_floats(const Problem& p)
{
    return (size_t)p.B * p.H * ((p.N + kC - 1) / kC);
}

size_t tc_awd_slot_floats(const Problem& p)
{
    return (size_t)2 * p.B * p.H * awd_hsplit(p) * (p.M / 64) * 128 * 64;
}

cudaError_t launch_tc_awd(const Problem& p, const void* q, const void* k, const void* pq,
                          const void* pk, float* part, float* loss, int* status, cudaStream_t s)
{
    return p.M == 64 ? launch_typed<2>(p, q, k, pq, pk, part, loss, nullptr, status, s)
                     : launch_typed<4>(p, q, k, pq, pk, part, loss, nullptr, status, s);
}

cudaError_t launch_tc_awd_bwd(const Problem& p, const void* q, const void* k, const void* pq,
                              const void* pk, const float* W1, const float* W2, const float* kw,
                              const float* tau, const float* dloss, float* part, float* loss,
                              float4* rowstat, float* slots, float* dtau_part, float* dW1,
                              float* dW2, float* dtau, int* status, cudaStream_t s)
{
    cudaError_t e = p.M == 64 ? launch_typed<2>(p, q, k, pq, pk, part, loss, rowstat, status, s)
                              : launch_typed<4>(p, q, k, pq, pk, part, loss, rowstat, status, s);
    if (e != cudaSuccess) return e;
    return p.M == 64 ? launch_bwd_g2<2>(p, q, k, pq, pk, W1, W2, kw, tau, dloss, rowstat, slots,
                                        dtau_part, dW1, dW2, dtau, status, s)
                     : launch_bwd_g2<4>(p, q, k, pq, pk, W1, W2, kw, tau, dloss, rowstat, slots,
                                        dtau_part, dW1, dW2, dtau, status, s);
}

}  // namespace flex
