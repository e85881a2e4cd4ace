// SIMT kernels: fp32 arithmetic on the CUDA cores.
//
// These kernels serve the fp32 storage type, whose tolerance (relative L2 <= 1e-4)
// excludes bf16/tf32 tensor-core operands, bf16 shapes off the tensor-core path, the
// feature-map entry point and the workspace-free backward.  They run the chunked form of
// Eq. (linear att): inside a chunk of T tokens the masked T x T kernel matrix
// phi(Q) phi(K)^T is applied directly, across chunks the running state
// S = sum phi(k) v^T, z = sum phi(k) carries the prefix.
//
// Inside the attention kernels the features are unscaled, phi' = [cos, sin] (times cos w
// for the nonstationary map): the global factor M^{-1/2} of Eq. phi_n / phi_non cancels in
// out and in every gradient, and only the stored denominator is rescaled, den = den'/M.
//
// Norm prefactor (Sec. 3.2, optional, tau per head): phi~(x) = exp(|x|^2 / exp(tau)) phi(x).
// The query's factor cancels row by row; the key's is a weight w_j, carried by turning the
// key rows [v_j | 1] into [w_j v_j | w_j].  The backward then multiplies dv_j by w_j and,
// with s_j = phi(k_j) . dphi(k_j), adds 2 exp(-tau) s_j k_j to dk_j and
// -exp(-tau) |k_j|^2 s_j to dtau.
#include "flex_internal.h"

#include <math.h>

#include <algorithm>

#include "tc_common.cuh"
#include "tc_util.cuh"

namespace flex {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxCluster = 8;   // CTAs that share one sequence
constexpr int kMaxT = 128;       // tokens per chunk (over 64: the non-causal forward only)
constexpr int kMaxMG = 32;       // frequencies per group (64 features) of chunks over 32 tokens

__device__ __forceinline__ float load_act(const float* p, size_t i) { return p[i]; }
__device__ __forceinline__ float load_act(const __nv_bfloat16* p, size_t i)
{
    return __bfloat162float(p[i]);
}
__device__ __forceinline__ void store_act(float* p, size_t i, float x) { p[i] = x; }
__device__ __forceinline__ void store_act(__nv_bfloat16* p, size_t i, float x)
{
    p[i] = __float2bfloat16_rn(x);
}
// Four consecutive elements (d % 4 == 0 and 16-byte aligned tensors: aligned accesses).
__device__ __forceinline__ float4 load_act4(const float* p, size_t i)
{
    return *reinterpret_cast<const float4*>(p + i);
}
__device__ __forceinline__ float4 load_act4(const __nv_bfloat16* p, size_t i)
{
    const uint2 u = *reinterpret_cast<const uint2*>(p + i);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void store_act4(float* p, size_t i, float4 x)
{
    *reinterpret_cast<float4*>(p + i) = x;
}
__device__ __forceinline__ void store_act4(__nv_bfloat16* p, size_t i, float4 x)
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
    *reinterpret_cast<uint2*>(p + i) = make_uint2(*reinterpret_cast<const uint32_t*>(&a),
                                                  *reinterpret_cast<const uint32_t*>(&b));
}

// ------------------------------------------------------------------------------------
// Feature map entry point (writes phi, scaled by M^{-1/2}).
// ------------------------------------------------------------------------------------
template <typename T>
__global__ void featmap_kernel(Problem p, const T* x, const float* W1, const float* W2, T* phi,
                               float scale, const float* rowscale)
{
    const int d = p.d, M = p.M;
    const size_t rows = (size_t)p.B * p.H * p.N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < rows * M;
         idx += (size_t)gridDim.x * blockDim.x) {
        size_t row = idx / M;
        int m = (int)(idx % M);
        int h = (int)((row / p.N) % p.H);
        const float* w1 = W1 + ((size_t)h * M + m) * d;
        float a = 0.f, w = 0.f;
        if (!p.nonstat) {
            for (int i = 0; i < d; ++i) a = fmaf(load_act(x, row * d + i), w1[i], a);
        } else {
            const float* w2 = W2 + ((size_t)h * M + m) * d;
            for (int i = 0; i < d; ++i) {
                float xi = load_act(x, row * d + i);
                a = fmaf(xi, 0.5f * (w1[i] + w2[i]), a);
                w = fmaf(xi, 0.5f * (w1[i] - w2[i]), w);
            }
        }
        float sa, ca;
        sincosf(a, &sa, &ca);
        float cw = (p.nonstat ? cosf(w) : 1.f) * scale * (rowscale ? rowscale[row] : 1.f);
        store_act(phi, row * 2 * M + m, ca * cw);
        store_act(phi, row * 2 * M + M + m, sa * cw);
    }
}

// ------------------------------------------------------------------------------------
// Attention: plan, tile products, features.
// ------------------------------------------------------------------------------------
// One cluster of CL CTAs per (b, h) sequence; CTA r owns a contiguous range of chunks of
// T tokens.  When the sequence is split (or not causal) each CTA first sums its own range's
// state; the cluster then turns those into what each range starts from (the total, or the
// exclusive prefix or suffix) through distributed shared memory, so no workspace and no
// second launch is needed.  Frequencies are taken MG at a time: a group has F = 2 MG
// features, feature columns 4x..4x+3 being cos, sin of frequency 2x and cos, sin of 2x + 1,
// so the thread that projects two frequencies writes (and later differentiates) its own
// four features.  All products run as 4 x 4 register tiles over shared-memory operands: per
// four k 8 float4 loads feed 64 fmas, so the fma pipe and not the shared-memory port is the
// limit (one output per thread took two loads per fma), and a short sequence spreads over
// up to 8 SMs instead of one.  Measured on GB300 against one CTA per sequence with
// one output per thread: forward f32 s B1 H1 N256 d32 M32 132 -> 16 us, bf16 n B32 H4
// N1024 d32 M16 477 -> 73 us; forward and backward f32 n tau B4 H4 N1000 d64 M64
// 8.58 -> 0.33 ms (10 of the 78 TFLOP/s fp32 peak: 96 of 152 SMs, and there per chunk the
// products run between barriers, one backward CTA per SM: issue slots 43% and the fma pipe
// 32% busy over all SMs, the rest shared-memory latency, barriers and instruction fetch).
struct Plan {
    int T;              // tokens per chunk (a multiple of 8, at most kMaxT)
    int lpr;            // lanes per row in row-wise sums: 4, or 2 with 128 tokens
    int ng, MG;         // frequency groups; frequencies per group (a multiple of 4)
    int CT;             // feature column tiles of a group, MG / 2
    int F;              // features of a group, 2 MG
    int KP;             // projection rows of a group: MG (s), 2 MG (n: u and w)
    int pd, pp, pa;     // pitches (floats) of rows of d, of features, of T x T blocks
    int wres;           // every group's projection rows stay in shared memory
    int CL;             // CTAs per sequence
    int S, W, dW, Xq, Xk, V, G, Pq, Pk, A, red, total;  // offsets (floats)
    int nt;             // threads per CTA
    int any;            // a plan of the kernels with NT = 0
};

// NT: threads of the CTA, kThreads or (0) Plan::nt.  Kernels with NT = 0 take the plans of short
// sequences and of many small ones: any thread count, groups of any size, no products with a
// state that is still zero and none that nothing reads.  (One kernel for every plan was 1-3%
// slower on long sequences; so is the count by a function instead of this expression.)
#define FLEX_THREADS (NT ? NT : (int)blockDim.x)

// Row of column tile x, column c in arrays whose rows are read four at a time by
// neighbouring x (projection rows, state rows): c CT + x, so that 16 lanes with
// consecutive x read consecutive rows (pitch 4 mod 32: no bank conflicts).
__device__ __forceinline__ int prow(const Plan& L, int feature)
{
    return (feature & 3) * L.CT + (feature >> 2);
}

// acc[r][c] += sum_k a[r pa + k] b[c pb + k], K a multiple of 4.
template <int NC>
__device__ __forceinline__ void mm_nt(const float* a, int pa, const float* b, int pb, int K,
                                      float (&acc)[4][NC])
{
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 x[4], y[NC];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(a + r * pa + k);
#pragma unroll
        for (int c = 0; c < NC; ++c) y[c] = *reinterpret_cast<const float4*>(b + c * pb + k);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                acc[r][c] = fmaf(x[r].x, y[c].x, acc[r][c]);
                acc[r][c] = fmaf(x[r].y, y[c].y, acc[r][c]);
                acc[r][c] = fmaf(x[r].z, y[c].z, acc[r][c]);
                acc[r][c] = fmaf(x[r].w, y[c].w, acc[r][c]);
            }
    }
}

// acc[r][c] += sum_k a[r pa + k] b[row(k)][c]; the rows of k..k+3 lie at o0..o3 from b,
// which advances by `step` every four (plain rows or the permuted rows of prow).
__device__ __forceinline__ void mm_nn(const float* a, int pa, const float* b, int o1, int o2,
                                      int o3, int step, int K, float (&acc)[4][4])
{
#pragma unroll 1
    for (int k = 0; k < K; k += 4, b += step) {
        float4 x[4], y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(a + r * pa + k);
        y[0] = *reinterpret_cast<const float4*>(b);
        y[1] = *reinterpret_cast<const float4*>(b + o1);
        y[2] = *reinterpret_cast<const float4*>(b + o2);
        y[3] = *reinterpret_cast<const float4*>(b + o3);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float xr[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                acc[r][0] = fmaf(xr[kk], y[kk].x, acc[r][0]);
                acc[r][1] = fmaf(xr[kk], y[kk].y, acc[r][1]);
                acc[r][2] = fmaf(xr[kk], y[kk].z, acc[r][2]);
                acc[r][3] = fmaf(xr[kk], y[kk].w, acc[r][3]);
            }
        }
    }
}

// acc[r][c] += sum_k a[k pa + r] b[k pb + c], K a multiple of 4.
__device__ __forceinline__ void mm_tn(const float* a, int pa, const float* b, int pb, int K,
                                      float (&acc)[4][4])
{
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 x = *reinterpret_cast<const float4*>(a + k * pa);
        const float4 y = *reinterpret_cast<const float4*>(b + k * pb);
        const float xr[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            acc[r][0] = fmaf(xr[r], y.x, acc[r][0]);
            acc[r][1] = fmaf(xr[r], y.y, acc[r][1]);
            acc[r][2] = fmaf(xr[r], y.z, acc[r][2]);
            acc[r][3] = fmaf(xr[r], y.w, acc[r][3]);
        }
    }
}

// Products with a masked T x T block M (M[i][j] = 0 for j > i) end at the diagonal: half the
// work, and a masked key or query is left out, not multiplied by zero, so an infinite or NaN
// value (or a key weight that overflows) reaches no row that does not see it.
// Rows 4y..4y+3 of M B: acc[r][c] += sum_{j <= 4y + r} M[4y + r][j] b[j pb + c].
__device__ __forceinline__ void mm_masked(const float* M, int pm, int y, const float* b, int pb,
                                          float (&acc)[4][4])
{
    mm_nn(M + 4 * y * pm, pm, b, pb, 2 * pb, 3 * pb, 4 * pb, 4 * y, acc);
    float4 x[4];  // the diagonal block
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(M + (4 * y + r) * pm + 4 * y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 v = *reinterpret_cast<const float4*>(b + (4 * y + k) * pb);
#pragma unroll
        for (int r = k; r < 4; ++r) {
            const float m = k == 0 ? x[r].x : k == 1 ? x[r].y : k == 2 ? x[r].z : x[r].w;
            acc[r][0] = fmaf(m, v.x, acc[r][0]);
            acc[r][1] = fmaf(m, v.y, acc[r][1]);
            acc[r][2] = fmaf(m, v.z, acc[r][2]);
            acc[r][3] = fmaf(m, v.w, acc[r][3]);
        }
    }
}
// Rows 4y..4y+3 of M^T B over T rows: acc[r][c] += sum_{i >= 4y + r} M[i][4y + r] b[i pb + c].
__device__ __forceinline__ void mm_masked_t(const float* M, int pm, int y, const float* b, int pb,
                                            int T, float (&acc)[4][4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // the diagonal block
        const float4 x = *reinterpret_cast<const float4*>(M + (4 * y + k) * pm + 4 * y);
        const float4 v = *reinterpret_cast<const float4*>(b + (4 * y + k) * pb);
        const float xr[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int r = 0; r <= k; ++r) {
            acc[r][0] = fmaf(xr[r], v.x, acc[r][0]);
            acc[r][1] = fmaf(xr[r], v.y, acc[r][1]);
            acc[r][2] = fmaf(xr[r], v.z, acc[r][2]);
            acc[r][3] = fmaf(xr[r], v.w, acc[r][3]);
        }
    }
    const int i = 4 * y + 4;
    mm_tn(M + i * pm + 4 * y, pm, b + i * pb, pb, T - i, acc);
}

template <int R, int C>
__device__ __forceinline__ void zero(float (&acc)[R][C])
{
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[r][c] = 0.f;
}

// Projection rows of group g of one head.  s: column c (0, 1) of tile x is frequency
// 2x + c; n: columns 0..3 are u, w of frequency 2x, then u, w of 2x + 1, with
// U = (W1+W2)/2, V = (W1-W2)/2.  Rows past M are zero.
template <bool NS, int NT>
__device__ void stage_projection(const Problem& p, const Plan& L, const float* W1,
                                 const float* W2, int h, int g, float* W)
{
    const int d = p.d, dq = d / 4, total = L.KP * dq;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * FLEX_THREADS) {  // four loads in flight
        float4 w[4], w2[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * FLEX_THREADS, row = idx / dq, c = row / L.CT, x = row % L.CT;
            const int f = g * L.MG + 2 * x + (NS ? c >> 1 : c);
            w[u] = w2[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (idx < total && f < p.M) {
                const size_t o = ((size_t)h * p.M + f) * d + 4 * (idx % dq);
                w[u] = *reinterpret_cast<const float4*>(W1 + o);
                if (NS) w2[u] = *reinterpret_cast<const float4*>(W2 + o);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * FLEX_THREADS, row = idx / dq;
            if (idx >= total) break;
            if (NS) {
                const float sg = (row / L.CT & 1) ? -1.f : 1.f;
                w[u] = make_float4(0.5f * (w[u].x + sg * w2[u].x), 0.5f * (w[u].y + sg * w2[u].y),
                                   0.5f * (w[u].z + sg * w2[u].z), 0.5f * (w[u].w + sg * w2[u].w));
            }
            *reinterpret_cast<float4*>(W + row * L.pd + 4 * (idx % dq)) = w[u];
        }
    }
}

// Rows of a chunk from one tensor, or from two (src2 non-null), zero from row `rows` on; the
// loads of a thread (up to eight) are issued before its stores.
template <int NT, typename T>
__device__ void load_rows(const T* src, const T* src2, size_t base, int rows, int d, float* dst,
                          float* dst2, int pitch, int nrows)
{
    const int dq = d / 4, total = nrows * dq;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * FLEX_THREADS) {
        float4 x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * FLEX_THREADS, t = idx / dq, e = 4 * (idx % dq);
            x[u] = y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < rows) {
                x[u] = load_act4(src, base + (size_t)t * d + e);
                if (src2) y[u] = load_act4(src2, base + (size_t)t * d + e);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * FLEX_THREADS, t = idx / dq, e = 4 * (idx % dq);
            if (idx >= total) break;
            *reinterpret_cast<float4*>(dst + t * pitch + e) = x[u];
            if (src2) *reinterpret_cast<float4*>(dst2 + t * pitch + e) = y[u];
        }
    }
}

// Column d of the value rows: 1 for the chunk's keys, 0 past its end.
__device__ __forceinline__ void unit_weights(const Plan& L, int d, int rows, float* V)
{
    if (threadIdx.x < L.T) V[threadIdx.x * L.pd + d] = threadIdx.x < rows ? 1.f : 0.f;
}

// Prefactor: [v_j | 1] -> [w_j v_j | w_j], w_j = exp(|k_j|^2 itau); |k_j|^2 to kn2.  lpr
// lanes per row.
__device__ __forceinline__ void weight_keys(const Plan& L, const float* Xk, int rows, int d,
                                            float itau, float* V, float* kn2)
{
    if (threadIdx.x >= L.lpr * L.T) return;
    const int j = threadIdx.x / L.lpr, part = threadIdx.x % L.lpr, step = 4 * L.lpr;
    float n2 = 0.f;
    for (int e = 4 * part; e < d; e += step) {
        const float4 x = *reinterpret_cast<const float4*>(Xk + j * L.pd + e);
        n2 = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, n2))));
    }
    n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
    if (L.lpr == 4) n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
    const float w = j < rows ? expf(n2 * itau) : 0.f;
    for (int e = 4 * part; e < d; e += step) {
        float4* v = reinterpret_cast<float4*>(V + j * L.pd + e);
        if (j < rows) *v = make_float4(w * v->x, w * v->y, w * v->z, w * v->w);
    }
    if (part == 0) {
        V[j * L.pd + d] = w;
        kn2[j] = n2;
    }
}

// This thread's place in the feature tile of a chunk: rows 4y..4y+3, column tile x.
struct Place {
    int y, x;
    bool on;
};

// sin and cos of two arguments in fp32, on packed pairs: reduction by pi/2 in three constants
// (Cody and Waite: the fp32 values of pi/2 and of the two remainders, each step one fma), then
// polynomials on [-pi/4, pi/4], sin r = r + r y (s0 + s1 y + s2 y^2) and
// cos r = 1 + y (-1/2 + y (c0 + c1 y + c2 y^2)) with y = r^2, fitted here by least squares on
// 4000 Chebyshev nodes refined by Lawson's iteration (approximation error of these, in fp32,
// 2.3e-9 and 5.1e-10).
// Max error against fp64 over |x| <= 10^4: 7.1e-8 (rms 1.7e-8; rounding the exact value:
// 1.5e-8), as the CUDA library's sincosf, which larger arguments take.  About 15 instructions
// an argument instead of 45; inlined library calls also overflowed the instruction cache.
__device__ __noinline__ float2 sincos_large(float x)
{
    float s, c;
    sincosf(x, &s, &c);
    return make_float2(s, c);
}
__device__ __forceinline__ void sincos2(float x0, float x1, float (&s)[2], float (&c)[2])
{
    if (!(fmaxf(fabsf(x0), fabsf(x1)) <= 1.0e4f)) {  // large or infinite (a lone NaN stays NaN below)
        const float2 a = sincos_large(x0), b = sincos_large(x1);
        s[0] = a.x; c[0] = a.y; s[1] = b.x; c[1] = b.y;
        return;
    }
    auto k2 = [](float k) { return tc::f2_pack(k, k); };
    constexpr float kRound = 12582912.f;  // 1.5 * 2^23: the sum's low bits hold rint(x 2/pi)
    const uint64_t x = tc::f2_pack(x0, x1);
    const uint64_t t = tc::f2_fma(x, k2(0.63661977236758134f), k2(kRound));
    const uint64_t n = tc::f2_fma(t, k2(1.f), k2(-kRound));
    uint64_t r = tc::f2_fma(n, k2(-1.57079637050628662f), x);
    r = tc::f2_fma(n, k2(4.371138828673793e-8f), r);
    r = tc::f2_fma(n, k2(1.7151244994428828e-15f), r);
    const uint64_t y = tc::f2_mul(r, r);
    uint64_t p = tc::f2_fma(k2(-1.9495636e-4f), y, k2(8.331979e-3f));
    p = tc::f2_fma(p, y, k2(-1.6666651e-1f));
    const uint64_t sn = tc::f2_fma(tc::f2_mul(p, y), r, r);
    uint64_t q = tc::f2_fma(k2(2.4438452e-5f), y, k2(-1.3887368e-3f));
    q = tc::f2_fma(q, y, k2(4.1666646e-2f));
    q = tc::f2_fma(q, y, k2(-0.5f));
    const uint64_t cs = tc::f2_fma(q, y, k2(1.f));
    float tn[2], sr[2], cr[2];
    tc::f2_unpack(t, tn[0], tn[1]);
    tc::f2_unpack(sn, sr[0], sr[1]);
    tc::f2_unpack(cs, cr[0], cr[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t quad = __float_as_uint(tn[i]);
        const float a = (quad & 1u) ? cr[i] : sr[i], b = (quad & 1u) ? sr[i] : cr[i];
        s[i] = __uint_as_float(__float_as_uint(a) ^ ((quad & 2u) << 30));
        c[i] = __uint_as_float(__float_as_uint(b) ^ (((quad + 1u) & 2u) << 30));
    }
}

// Unscaled features of this thread's 4 rows x 2 frequencies: pf = (cos, sin) of each (times
// cos w), zero for rows from `rows` on and frequencies past M.  With CHAIN also
// qf = (cos u sin w, sin u sin w) (n), for the derivative with respect to w.
template <bool NS, bool CHAIN>
__device__ __forceinline__ void features(const Problem& p, const Plan& L, const Place& f,
                                         const float* X, int rows, const float* W, int g,
                                         float (&pf)[4][4], float (&qf)[4][4])
{
    constexpr int NC = NS ? 4 : 2;
    float a[4][NC];
    zero(a);
    mm_nt<NC>(X + 4 * f.y * L.pd, L.pd, W + f.x * L.pd, L.CT * L.pd, p.d, a);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float su[2], cu[2], sw[2], cw[2];
        sincos2(a[r][0], a[r][NC / 2], su, cu);
        if (NS) sincos2(a[r][1], a[r][NC - 1], sw, cw);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const bool ok = 4 * f.y + r < rows && g * L.MG + 2 * f.x + i < p.M;
            pf[r][2 * i] = ok ? (NS ? cu[i] * cw[i] : cu[i]) : 0.f;
            pf[r][2 * i + 1] = ok ? (NS ? su[i] * cw[i] : su[i]) : 0.f;
            if (NS && CHAIN) {
                qf[r][2 * i] = ok ? cu[i] * sw[i] : 0.f;
                qf[r][2 * i + 1] = ok ? su[i] * sw[i] : 0.f;
            }
        }
    }
}
__device__ __forceinline__ void store_tile(float* P, int pitch, const Place& f, const float (&v)[4][4])
{
#pragma unroll
    for (int r = 0; r < 4; ++r)
        *reinterpret_cast<float4*>(P + (4 * f.y + r) * pitch + 4 * f.x) =
            make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
}

// acc = sum_k a[k pa + r] b[k pb + c] over K rows: ks (1, 2 or 4) neighbouring lanes share a
// 4 x 4 tile, each sums every ks-th row, and every lane of the group returns the sum.
__device__ __forceinline__ void mm_tn_split(const float* a, int pa, const float* b, int pb, int K,
                                            int ks, float (&acc)[4][4])
{
    const int part = threadIdx.x & (ks - 1);
    mm_tn(a + part * pa, ks * pa, b + part * pb, ks * pb, K / ks, acc);
    for (int o = 1; o < ks; o *= 2)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] += __shfl_xor_sync(0xffffffffu, acc[r][c], o);
}

// State of one group: S[prow(f)][e] += sum_j P[j][f] Y[j][e] and, in column d, the sum
// weighted by Y[j][d] (z, or r from G = [g | c]).
template <int NT>
__device__ __forceinline__ void state_update(const Plan& L, int d, const float* P, const float* Y,
                                             float* S)
{
    const int dq = d / 4, tiles = L.CT * dq;
    // over long chunks, lanes without a tile of their own share one
    const int ks = L.T <= 64 ? 1 : 4 * tiles <= FLEX_THREADS ? 4 : 2 * tiles <= FLEX_THREADS ? 2 : 1;
    for (int i0 = threadIdx.x & ~31; i0 < tiles * ks; i0 += FLEX_THREADS) {
        // (whole warps take part in the exchange: lanes past the end repeat the last tile)
        const int at = i0 + (threadIdx.x & 31), id = min(at / ks, tiles - 1);
        const int x = id / dq, e = 4 * (id % dq);
        float acc[4][4];
        zero(acc);
        mm_tn_split(P + 4 * x, L.pp, Y + e, L.pd, L.T, ks, acc);
        if (at >= tiles * ks || (at & (ks - 1))) continue;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float4* s = reinterpret_cast<float4*>(S + (r * L.CT + x) * L.pd + e);
            *s = make_float4(s->x + acc[r][0], s->y + acc[r][1], s->z + acc[r][2],
                             s->w + acc[r][3]);
        }
    }
    // column d: four lanes per feature (4 F is a multiple of 32)
    if constexpr (NT == kThreads) {
        if (threadIdx.x < 4 * L.F) {
            const int f = threadIdx.x >> 2;
            float z = 0.f;
            for (int j = threadIdx.x & 3; j < L.T; j += 4) z = fmaf(P[j * L.pp + f], Y[j * L.pd + d], z);
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            z += __shfl_xor_sync(0xffffffffu, z, 2);
            if ((threadIdx.x & 3) == 0) S[prow(L, f) * L.pd + d] += z;
        }
    } else {
        for (int i = threadIdx.x; i < 4 * L.F; i += FLEX_THREADS) {
            const int f = i >> 2;
            float z = 0.f;
            for (int j = i & 3; j < L.T; j += 4) z = fmaf(P[j * L.pp + f], Y[j * L.pd + d], z);
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            z += __shfl_xor_sync(0xffffffffu, z, 2);
            if ((i & 3) == 0) S[prow(L, f) * L.pd + d] += z;
        }
    }
}

// The ranges' states, summed over the cluster in rank order: every CTA's S becomes the
// total, or the sum over the lower (prefix) or higher (suffix) ranks.  Each CTA owns a slice
// of the state: it alone reads and rewrites that slice in all CTAs, so it works in place.
enum { kTotal, kPrefix, kSuffix };
template <int NT>
__device__ void exchange_state(float* S, int n, int CL, int mode)
{
    tc::cluster_sync();
    const uint32_t base = tc::smem_u32(S);
    const int rank = (int)tc::cluster_rank();
    for (int i = rank * FLEX_THREADS + threadIdx.x; i < n / 4; i += CL * FLEX_THREADS) {
        float4 v[kMaxCluster];
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r)
            if (r < CL) v[r] = tc::ld_cluster_v4(tc::mapa(base + 16 * i, r));
        float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
        auto add = [&](const float4& x) {
            run = make_float4(run.x + x.x, run.y + x.y, run.z + x.z, run.w + x.w);
        };
        if (mode == kTotal)
#pragma unroll
            for (int r = 0; r < kMaxCluster; ++r)
                if (r < CL) add(v[r]);
#pragma unroll
        for (int o = 0; o < kMaxCluster; ++o) {
            const int r = mode == kSuffix ? kMaxCluster - 1 - o : o;
            if (r < CL) {
                tc::st_cluster_v4(tc::mapa(base + 16 * i, r), run.x, run.y, run.z, run.w);
                if (mode != kTotal) {
                    float4 x = v[0];
#pragma unroll
                    for (int s = 1; s < kMaxCluster; ++s)
                        if (s == r) x = v[s];
                    add(x);
                }
            }
        }
    }
    tc::cluster_sync();
}

// Chunks [cb, ce) of this CTA.
__device__ __forceinline__ void chunk_range(const Plan& L, int N, int rank, int* cb, int* ce)
{
    const int nch = (N + L.T - 1) / L.T, per = (nch + L.CL - 1) / L.CL;
    *cb = min(nch, rank * per);
    *ce = min(nch, *cb + per);
}

// ------------------------------------------------------------------------------------
// Forward.
// ------------------------------------------------------------------------------------
template <typename T, bool NS, int ND, int NT>
__global__ void __launch_bounds__(kThreads, 2)
    simt_fwd_kernel(Problem p, Plan L, const T* q, const T* k, const T* v, const float* W1,
                    const float* W2, const float* tau, T* out, float* den)
{
    extern __shared__ float4 sm4[];
    float* sm = reinterpret_cast<float*>(sm4);
    const int tid = threadIdx.x, d = p.d, N = p.N, dq = d / 4;
    const int rank = L.CL > 1 ? (int)tc::cluster_rank() : 0;
    const int bh = blockIdx.x / L.CL, h = bh % p.H;
    const size_t base = (size_t)bh * N * d;
    float *S = sm + L.S, *Xq = sm + L.Xq, *Xk = sm + L.Xk, *V = sm + L.V;
    float *Pq = sm + L.Pq, *Pk = sm + L.Pk, *A = sm + L.A, *red = sm + L.red;
    const float inv_m = 1.0f / (float)p.M, itau = tau ? expf(-tau[h]) : 0.f;
    const int gS = L.F * L.pd, gW = L.wres ? L.KP * L.pd : 0;  // strides of a group
    const Place f = {tid / L.CT, tid % L.CT, tid / L.CT < L.T / 4};
    const int TT = L.T / 4, ay = tid / TT, ax = tid % TT;  // T x T tile: rows 4 ay + r, cols ax + TT c
    const bool a_on = ay < TT;
    const int lpr = L.lpr, row = tid / lpr, part = tid % lpr;  // row-wise sums
    int cb, ce;
    chunk_range(L, N, rank, &cb, &ce);

    if (L.wres)
        for (int g = 0; g < L.ng; ++g)
            stage_projection<NS, NT>(p, L, W1, W2, h, g, sm + L.W + g * gW);
    for (int i = tid; i < L.ng * gS; i += FLEX_THREADS) S[i] = 0.f;

    if (!p.causal || L.CL > 1) {  // this range's sums
        for (int c = cb; c < ce; ++c) {
            const int t0 = c * L.T, rows = min(L.T, N - t0);
            load_rows<NT>(k, v, base + (size_t)t0 * d, rows, d, Xk, V, L.pd, L.T);
            unit_weights(L, d, rows, V);
            __syncthreads();
            if (tau) weight_keys(L, Xk, rows, d, itau, V, red);
            for (int g = 0; g < L.ng; ++g) {
                float* W = sm + L.W + g * gW;
                if (!L.wres) {
                    stage_projection<NS, NT>(p, L, W1, W2, h, g, W);
                    __syncthreads();
                }
                if (f.on) {
                    float pf[4][4], qf[4][4];
                    features<NS, false>(p, L, f, Xk, rows, W, g, pf, qf);
                    store_tile(Pk, L.pp, f, pf);
                }
                __syncthreads();
                state_update<NT>(L, d, Pk, V, S + g * gS);
                __syncthreads();
            }
        }
        if (L.CL > 1) exchange_state<NT>(S, L.ng * gS, L.CL, p.causal ? kPrefix : kTotal);
    }
    __syncthreads();

    for (int c = cb; c < ce; ++c) {
        const int t0 = c * L.T, rows = min(L.T, N - t0);
        const bool seen = NT || !p.causal || L.CL > 1 || c > cb;  // (else the state is still zero)
        load_rows<NT>(q, (const T*)nullptr, base + (size_t)t0 * d, rows, d, Xq, (float*)nullptr, L.pd, L.T);
        if (p.causal) {
            load_rows<NT>(k, v, base + (size_t)t0 * d, rows, d, Xk, V, L.pd, L.T);
            unit_weights(L, d, rows, V);
        }
        __syncthreads();
        if (tau && p.causal) weight_keys(L, Xk, rows, d, itau, V, red);
        float aa[4][4], num[ND][4][4], dsum = 0.f;
        zero(aa);
#pragma unroll
        for (int n = 0; n < ND; ++n) zero(num[n]);
        for (int g = 0; g < L.ng; ++g) {
            float* W = sm + L.W + g * gW;
            float* Sg = S + g * gS;
            if (!L.wres) {
                stage_projection<NS, NT>(p, L, W1, W2, h, g, W);
                __syncthreads();
            }
            if (f.on) {
                float pf[4][4], qf[4][4];
                features<NS, false>(p, L, f, Xq, rows, W, g, pf, qf);
                store_tile(Pq, L.pp, f, pf);
                if (p.causal) {
                    features<NS, false>(p, L, f, Xk, rows, W, g, pf, qf);
                    store_tile(Pk, L.pp, f, pf);
                }
            }
            __syncthreads();
            if (p.causal && a_on)
                mm_nt<4>(Pq + 4 * ay * L.pp, L.pp, Pk + ax * L.pp, TT * L.pp, L.F, aa);
#pragma unroll
            for (int n = 0; n < ND; ++n) {
                const int id = tid + n * FLEX_THREADS, y = id / dq, e = 4 * (id % dq);
                if (seen && y < TT)
                    mm_nn(Pq + 4 * y * L.pp, L.pp, Sg + e, L.CT * L.pd, 2 * L.CT * L.pd,
                          3 * L.CT * L.pd, L.pd, L.F, num[n]);
            }
            if (seen && tid < lpr * L.T)  // denominator
                for (int i = part; i < L.CT; i += lpr) {
                    const float4 x = *reinterpret_cast<const float4*>(Pq + row * L.pp + 4 * i);
                    const float* z = Sg + i * L.pd + d;
                    dsum = fmaf(x.x, z[0], dsum);
                    dsum = fmaf(x.y, z[L.CT * L.pd], dsum);
                    dsum = fmaf(x.z, z[2 * L.CT * L.pd], dsum);
                    dsum = fmaf(x.w, z[3 * L.CT * L.pd], dsum);
                }
            __syncthreads();
            if (p.causal) {
                if (NT || c + 1 < ce) state_update<NT>(L, d, Pk, V, Sg);  // (else nothing reads it)
                if (g + 1 < L.ng) __syncthreads();
            }
        }
        if (p.causal) {
            if (a_on)
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        const int i = 4 * ay + r, j = ax + TT * cc;
                        A[i * L.pa + j] = j <= i ? aa[r][cc] : 0.f;
                    }
            __syncthreads();
#pragma unroll
            for (int n = 0; n < ND; ++n) {
                const int id = tid + n * FLEX_THREADS, y = id / dq, e = 4 * (id % dq);
                if (y < TT) mm_masked(A, L.pa, y, V + e, L.pd, num[n]);
            }
            if (tid < lpr * L.T)
                for (int j = part; j <= row; j += lpr)
                    dsum = fmaf(A[row * L.pa + j], V[j * L.pd + d], dsum);
        }
        if (tid < lpr * L.T) {
            dsum += __shfl_xor_sync(0xffffffffu, dsum, 1);
            if (lpr == 4) dsum += __shfl_xor_sync(0xffffffffu, dsum, 2);
            if (part == 0) {
                red[kMaxT + row] = dsum;
                if (den && row < rows) den[(size_t)bh * N + t0 + row] = dsum * inv_m;
            }
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < ND; ++n) {
            const int id = tid + n * FLEX_THREADS, y = id / dq, e = 4 * (id % dq);
            if (y < TT)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = 4 * y + r;
                    if (i >= rows) break;
                    const float dn = red[kMaxT + i];
                    store_act4(out, base + (size_t)(t0 + i) * d + e,
                               make_float4(num[n][r][0] / dn, num[n][r][1] / dn,
                                           num[n][r][2] / dn, num[n][r][3] / dn));
                }
        }
    }
    if (L.CL > 1) tc::cluster_sync();  // no CTA leaves while another may read its state
}

// ------------------------------------------------------------------------------------
// Backward.
// ------------------------------------------------------------------------------------
// G[t] = [dout_t / den'_t | -(dout_t . out_t) / den'_t] with den' = M den; zero past `rows`.
// Four lanes per row.
template <typename T>
__device__ __forceinline__ void load_upstream(const Problem& p, const Plan& L, const T* dout,
                                              const T* out, const float* den, size_t base,
                                              size_t den_base, int rows, float* G)
{
    if (threadIdx.x >= 4 * L.T) return;
    const int d = p.d, t = threadIdx.x >> 2, part = threadIdx.x & 3;
    const bool ok = t < rows;
    const float dn = ok ? den[den_base + t] * (float)p.M : 1.f;
    float s = 0.f;
    for (int e = 4 * part; e < d; e += 16) {
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok) {
            g = load_act4(dout, base + (size_t)t * d + e);
            const float4 o = load_act4(out, base + (size_t)t * d + e);
            s = fmaf(g.x, o.x, fmaf(g.y, o.y, fmaf(g.z, o.z, fmaf(g.w, o.w, s))));
            g = make_float4(g.x / dn, g.y / dn, g.z / dn, g.w / dn);
        }
        *reinterpret_cast<float4*>(G + t * L.pd + e) = g;
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (part == 0) G[t * L.pd + d] = -s / dn;
}

// Chain rule through the features: dP = (dL/dcos, dL/dsin) of two frequencies a row ->
// dL/da (s), or dL/du, dL/dw of each (n), stored as projection columns.
template <bool NS>
__device__ __forceinline__ void store_chain(const Plan& L, const Place& f, const float (&dp)[4][4],
                                            const float (&pf)[4][4], const float (&qf)[4][4],
                                            float* D)
{
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float a0 = fmaf(-pf[r][1], dp[r][0], pf[r][0] * dp[r][1]);
        const float a1 = fmaf(-pf[r][3], dp[r][2], pf[r][2] * dp[r][3]);
        float* row = D + (4 * f.y + r) * L.pp;
        if (NS) {
            const float b0 = -fmaf(qf[r][0], dp[r][0], qf[r][1] * dp[r][1]);
            const float b1 = -fmaf(qf[r][2], dp[r][2], qf[r][3] * dp[r][3]);
            *reinterpret_cast<float4*>(row + 4 * f.x) = make_float4(a0, b0, a1, b1);
        } else {
            *reinterpret_cast<float2*>(row + 2 * f.x) = make_float2(a0, a1);
        }
    }
}

// dx tiles += da W and dW += da^T X of one group.
template <bool NS, int ND, int NT>
__device__ __forceinline__ void project_back(const Plan& L, int d, const float* D, const float* W,
                                             const float* X, float* dW, float (&dx)[ND][4][4])
{
    const int dq = d / 4, TT = L.T / 4, o = L.CT * L.pd;
#pragma unroll
    for (int n = 0; n < ND; ++n) {
        const int id = threadIdx.x + n * FLEX_THREADS, y = id / dq, e = 4 * (id % dq);
        if (y < TT) {
            if (NS)
                mm_nn(D + 4 * y * L.pp, L.pp, W + e, o, 2 * o, 3 * o, L.pd, L.KP, dx[n]);
            else
                mm_nn(D + 4 * y * L.pp, L.pp, W + e, o, L.pd, o + L.pd, 2 * L.pd, L.KP, dx[n]);
        }
    }
    for (int id = threadIdx.x; id < L.KP / 4 * dq; id += FLEX_THREADS) {
        const int x = id / dq, e = 4 * (id % dq);
        float acc[4][4];
        zero(acc);
        mm_tn(D + 4 * x, L.pp, X + e, L.pd, L.T, acc);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float4* w = reinterpret_cast<float4*>(dW + (4 * x + r) * d + e);
            *w = make_float4(w->x + acc[r][0], w->y + acc[r][1], w->z + acc[r][2],
                             w->w + acc[r][3]);
        }
    }
}

template <typename T, int ND, int NT>
__device__ __forceinline__ void store_rows(const Plan& L, int d, const float (&x)[ND][4][4],
                                           T* dst, size_t base, int rows)
{
    const int dq = d / 4;
#pragma unroll
    for (int n = 0; n < ND; ++n) {
        const int id = threadIdx.x + n * FLEX_THREADS, y = id / dq, e = 4 * (id % dq);
        if (y < L.T / 4)
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (4 * y + r < rows)
                    store_act4(dst, base + (size_t)(4 * y + r) * d + e,
                               make_float4(x[n][r][0], x[n][r][1], x[n][r][2], x[n][r][3]));
    }
}

template <typename T, bool NS, int ND, int NT>
__global__ void __launch_bounds__(kThreads, 1)
    simt_bwd_kernel(Problem p, Plan L, const T* q, const T* k, const T* v, const float* W1,
                    const float* W2, const float* tau, const T* out, const float* den,
                    const T* dout, T* dq, T* dk, T* dv, float* dw_part, float* dtau_part)
{
    extern __shared__ float4 sm4[];
    float* sm = reinterpret_cast<float*>(sm4);
    const int tid = threadIdx.x, d = p.d, N = p.N, d4 = d / 4;
    const int rank = L.CL > 1 ? (int)tc::cluster_rank() : 0;
    const int bh = blockIdx.x / L.CL, h = bh % p.H;
    const size_t base = (size_t)bh * N * d, den_base = (size_t)bh * N;
    float *S = sm + L.S, *Xq = sm + L.Xq, *Xk = sm + L.Xk, *V = sm + L.V, *G = sm + L.G;
    float *Pq = sm + L.Pq, *Pk = sm + L.Pk, *dA = sm + L.A, *dW = sm + L.dW, *red = sm + L.red;
    float* A = Pq;  // masked phi(Q) phi(K)^T, once the features are no longer needed
    const float itau = tau ? expf(-tau[h]) : 0.f;
    const int gS = L.F * L.pd, gW = L.wres ? L.KP * L.pd : 0, gD = L.KP * d;
    const Place f = {tid / L.CT, tid % L.CT, tid / L.CT < L.T / 4};
    const int TT = L.T / 4, ay = tid / TT, ax = tid % TT;
    const bool a_on = ay < TT;
    float dtau_acc = 0.f;
    // |k_0|^2 of the sequence: dtau = -exp(-tau) sum_j (|k_j|^2 - |k_0|^2) s_j (the s_j of a
    // sequence sum to zero, as every output row is invariant to a common key-weight scale)
    float n20 = 0.f;
    if (tau)
        for (int e = 0; e < d; ++e) {
            const float x = load_act(k, base + e);
            n20 = fmaf(x, x, n20);
        }
    int cb, ce;
    chunk_range(L, N, rank, &cb, &ce);

    if (L.wres)
        for (int g = 0; g < L.ng; ++g)
            stage_projection<NS, NT>(p, L, W1, W2, h, g, sm + L.W + g * gW);
    for (int i = tid; i < L.ng * gS; i += FLEX_THREADS) S[i] = 0.f;
    for (int i = tid; i < L.ng * gD; i += FLEX_THREADS) dW[i] = 0.f;

    auto load_kv = [&](int t0, int rows) {
        load_rows<NT>(k, v, base + (size_t)t0 * d, rows, d, Xk, V, L.pd, L.T);
        unit_weights(L, d, rows, V);
    };
    auto load_qg = [&](int t0, int rows) {
        load_rows<NT>(q, (const T*)nullptr, base + (size_t)t0 * d, rows, d, Xq, (float*)nullptr, L.pd, L.T);
        load_upstream(p, L, dout, out, den, base + (size_t)t0 * d, den_base + t0, rows, G);
    };
    auto group_W = [&](int g) {  // the group's projection rows, staged now unless resident
        float* W = sm + L.W + g * gW;
        if (!L.wres) {
            stage_projection<NS, NT>(p, L, W1, W2, h, g, W);
            __syncthreads();
        }
        return W;
    };
    // dA_ij = g_i . v_j + c_i (weighted keys), j <= i
    auto build_dA = [&]() {
        if (!a_on) return;
        float acc[4][4];
        zero(acc);
        mm_nt<4>(G + 4 * ay * L.pd, L.pd, V + ax * L.pd, TT * L.pd, d, acc);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = 4 * ay + r;
            const float ci = G[i * L.pd + d];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int j = ax + TT * c;
                dA[i * L.pa + j] = j <= i ? fmaf(ci, V[j * L.pd + d], acc[r][c]) : 0.f;
            }
        }
    };
    // this range's sums of phi(x) [y | y_d], over its chunks, into S (zeroed)
    auto range_state = [&](bool keys) {
        for (int c = cb; c < ce; ++c) {
            const int t0 = c * L.T, rows = min(L.T, N - t0);
            if (keys)
                load_kv(t0, rows);
            else
                load_qg(t0, rows);
            __syncthreads();
            if (keys && tau) weight_keys(L, Xk, rows, d, itau, V, red);
            for (int g = 0; g < L.ng; ++g) {
                float* W = group_W(g);
                if (f.on) {
                    float pf[4][4], qf[4][4];
                    features<NS, false>(p, L, f, keys ? Xk : Xq, rows, W, g, pf, qf);
                    store_tile(keys ? Pk : Pq, L.pp, f, pf);
                }
                __syncthreads();
                state_update<NT>(L, d, keys ? Pk : Pq, keys ? V : G, S + g * gS);
                __syncthreads();
            }
        }
    };

    // ---- dq: forward direction with S_i, z_i ----
    if (!p.causal || L.CL > 1) {
        __syncthreads();
        range_state(true);
        if (L.CL > 1) exchange_state<NT>(S, L.ng * gS, L.CL, p.causal ? kPrefix : kTotal);
    }
    __syncthreads();
    for (int c = cb; c < ce; ++c) {
        const int t0 = c * L.T, rows = min(L.T, N - t0);
        const bool seen = NT || !p.causal || L.CL > 1 || c > cb;  // (else the state is still zero)
        load_qg(t0, rows);
        if (p.causal) load_kv(t0, rows);
        __syncthreads();
        if (p.causal) {
            if (tau) {
                weight_keys(L, Xk, rows, d, itau, V, red);
                __syncthreads();
            }
            build_dA();
        }
        float dx[ND][4][4];
#pragma unroll
        for (int n = 0; n < ND; ++n) zero(dx[n]);
        for (int g = 0; g < L.ng; ++g) {
            float* W = group_W(g);
            float* Sg = S + g * gS;
            float pf[4][4], qf[4][4], dp[4][4];
            if (f.on) {
                if (p.causal) {
                    features<NS, false>(p, L, f, Xk, rows, W, g, pf, qf);
                    store_tile(Pk, L.pp, f, pf);
                }
                features<NS, true>(p, L, f, Xq, rows, W, g, pf, qf);
            }
            __syncthreads();
            if (f.on) {
                zero(dp);
                if (p.causal) mm_masked(dA, L.pa, f.y, Pk + 4 * f.x, L.pp, dp);
                if (seen) mm_nt<4>(G + 4 * f.y * L.pd, L.pd, Sg + f.x * L.pd, L.CT * L.pd, d, dp);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float ci = G[(4 * f.y + r) * L.pd + d];
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        dp[r][cc] = fmaf(ci, Sg[(cc * L.CT + f.x) * L.pd + d], dp[r][cc]);
                }
            }
            __syncthreads();
            if (f.on) store_chain<NS>(L, f, dp, pf, qf, Pq);
            if (p.causal && (NT || c + 1 < ce)) state_update<NT>(L, d, Pk, V, Sg);
            __syncthreads();
            project_back<NS, ND, NT>(L, d, Pq, W, Xq, dW + g * gD, dx);
            __syncthreads();
        }
        store_rows<T, ND, NT>(L, d, dx, dq, base + (size_t)t0 * d, rows);
    }

    // ---- dk, dv: reverse direction with R_j, r_j (S's buffer is reused for R) ----
    for (int i = tid; i < L.ng * gS; i += FLEX_THREADS) S[i] = 0.f;
    __syncthreads();
    if (!p.causal || L.CL > 1) {
        range_state(false);
        if (L.CL > 1) exchange_state<NT>(S, L.ng * gS, L.CL, p.causal ? kSuffix : kTotal);
        __syncthreads();
    }
    for (int c = ce - 1; c >= cb; --c) {
        const int t0 = c * L.T, rows = min(L.T, N - t0);
        const bool seen = NT || !p.causal || L.CL > 1 || c < ce - 1;  // (else the state is still zero)
        load_kv(t0, rows);
        if (p.causal) load_qg(t0, rows);
        __syncthreads();
        if (tau) {
            weight_keys(L, Xk, rows, d, itau, V, red);
            __syncthreads();
        }
        if (p.causal) build_dA();
        float dx[ND][4][4], dvt[ND][4][4], aa[4][4], sdot[4] = {0.f, 0.f, 0.f, 0.f};
        zero(aa);
#pragma unroll
        for (int n = 0; n < ND; ++n) {
            zero(dx[n]);
            zero(dvt[n]);
        }
        for (int g = 0; g < L.ng; ++g) {
            float* W = group_W(g);
            float* Rg = S + g * gS;
            float pf[4][4], qf[4][4], dp[4][4];
            if (f.on) {
                if (p.causal) {
                    features<NS, false>(p, L, f, Xq, rows, W, g, pf, qf);
                    store_tile(Pq, L.pp, f, pf);
                }
                features<NS, true>(p, L, f, Xk, rows, W, g, pf, qf);
                store_tile(Pk, L.pp, f, pf);
            }
            __syncthreads();
            if (p.causal && a_on)
                mm_nt<4>(Pq + 4 * ay * L.pp, L.pp, Pk + ax * L.pp, TT * L.pp, L.F, aa);
#pragma unroll
            for (int n = 0; n < ND; ++n) {
                const int id = tid + n * FLEX_THREADS, y = id / d4, e = 4 * (id % d4);
                if (seen && y < TT)
                    mm_nn(Pk + 4 * y * L.pp, L.pp, Rg + e, L.CT * L.pd, 2 * L.CT * L.pd,
                          3 * L.CT * L.pd, L.pd, L.F, dvt[n]);
            }
            if (f.on) {
                zero(dp);
                if (p.causal) mm_masked_t(dA, L.pa, f.y, Pq + 4 * f.x, L.pp, L.T, dp);
                if (seen) mm_nt<4>(V + 4 * f.y * L.pd, L.pd, Rg + f.x * L.pd, L.CT * L.pd, d, dp);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float wj = V[(4 * f.y + r) * L.pd + d];
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        dp[r][cc] = fmaf(wj, Rg[(cc * L.CT + f.x) * L.pd + d], dp[r][cc]);
                        sdot[r] = fmaf(pf[r][cc], dp[r][cc], sdot[r]);
                    }
                }
            }
            __syncthreads();
            if (f.on) store_chain<NS>(L, f, dp, pf, qf, Pk);
            if (p.causal && (NT || c > cb)) state_update<NT>(L, d, Pq, G, Rg);
            __syncthreads();
            project_back<NS, ND, NT>(L, d, Pk, W, Xk, dW + g * gD, dx);
            __syncthreads();
        }
        if (p.causal && a_on)
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const int i = 4 * ay + r, j = ax + TT * cc;
                    A[i * L.pa + j] = j <= i ? aa[r][cc] : 0.f;
                }
        if (tau && f.on)  // s_j = phi(k_j) . dphi(k_j), one partial per column tile
#pragma unroll
            for (int r = 0; r < 4; ++r) dA[(4 * f.y + r) * L.pa + f.x] = sdot[r];
        __syncthreads();
        if (tau) {  // dk_j += 2 itau s_j k_j, dtau -= itau |k_j|^2 s_j
            if (tid < L.T) {
                float sj = 0.f;
                for (int x = 0; x < L.CT; ++x) sj += dA[tid * L.pa + x];
                red[kMaxT + tid] = 2.f * itau * sj;
                if (tid < rows) dtau_acc = fmaf(-itau * (red[tid] - n20), sj, dtau_acc);
            }
            __syncthreads();
        }
#pragma unroll
        for (int n = 0; n < ND; ++n) {
            const int id = tid + n * FLEX_THREADS, y = id / d4, e = 4 * (id % d4);
            if (y < TT) {
                if (p.causal) mm_masked_t(A, L.pa, y, G + e, L.pd, L.T, dvt[n]);
                if (tau)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int j = 4 * y + r;
                        const float wj = V[j * L.pd + d], kc = red[kMaxT + j];
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            dvt[n][r][cc] *= wj;  // dv_j = w_j R_j^T phi(k_j)
                            dx[n][r][cc] = fmaf(kc, Xk[j * L.pd + e + cc], dx[n][r][cc]);
                        }
                    }
            }
        }
        store_rows<T, ND, NT>(L, d, dvt, dv, base + (size_t)t0 * d, rows);
        store_rows<T, ND, NT>(L, d, dx, dk, base + (size_t)t0 * d, rows);
        __syncthreads();
    }

    // ---- the sequence's dW and dtau: the cluster's partials in rank order ----
    if (tau) {
        for (int o = 16; o > 0; o >>= 1) dtau_acc += __shfl_xor_sync(0xffffffffu, dtau_acc, o);
        if ((tid & 31) == 0) red[tid >> 5] = dtau_acc;
        __syncthreads();
        if (tid == 0) {
            float t = 0.f;
            for (int w = 0; w < FLEX_THREADS / 32; ++w) t += red[w];
            red[kMaxT] = t;
        }
    }
    if (L.CL > 1)
        tc::cluster_sync();
    else
        __syncthreads();
    const int Mc = NS ? 2 * p.M : p.M;
    float* part = dw_part + (size_t)bh * Mc * d;
    const uint32_t dw_addr = tc::smem_u32(dW);
    for (int i = rank * FLEX_THREADS + tid; i < L.ng * gD / 4; i += L.CL * FLEX_THREADS) {
        const int row = 4 * i / d, e = 4 * i % d, g = row / L.KP, kk = row % L.KP;
        const int fr = g * L.MG + (NS ? 2 * (kk >> 2) + ((kk >> 1) & 1) : kk);
        if (fr >= p.M) continue;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (L.CL == 1) {
            a = *reinterpret_cast<const float4*>(dW + 4 * i);
        } else {
            for (int r = 0; r < L.CL; ++r) {
                const float4 x = tc::ld_cluster_v4(tc::mapa(dw_addr + 16 * i, r));
                a = make_float4(a.x + x.x, a.y + x.y, a.z + x.z, a.w + x.w);
            }
        }
        // n: rows < M of the partial hold dU, rows >= M dV
        *reinterpret_cast<float4*>(part + (size_t)(NS && (kk & 1) ? p.M + fr : fr) * d + e) = a;
    }
    if (tau && rank == 0 && tid == 0) {
        float t = red[kMaxT];
        for (int r = 1; r < L.CL; ++r) t += tc::ld_cluster_f32(tc::mapa(tc::smem_u32(red + kMaxT), r));
        dtau_part[bh] = t;
    }
    if (L.CL > 1) tc::cluster_sync();  // no CTA leaves while another may read its partials
}

// Key weights of the norm prefactor for the tensor-core forwards: kw[row] =
// exp(|k_row|^2 exp(-tau_h)) for every row of k [B*H*N][d]; one thread per row, vector
// loads of 4 elements (d % 4 == 0).
template <typename T>
__global__ void __launch_bounds__(kThreads) key_weights_kernel(Problem p, const T* k,
                                                               const float* tau, float* kw)
{
    const size_t rows = (size_t)p.B * p.H * p.N;
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
         r += (size_t)gridDim.x * blockDim.x) {
        const T* x = k + r * p.d;
        float n2 = 0.f;
        for (int e = 0; e < p.d; e += 4) {
            float v[4];
            if constexpr (sizeof(T) == 4) {
                const float4 f = *reinterpret_cast<const float4*>(x + e);
                v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
            } else {
                const uint2 u = *reinterpret_cast<const uint2*>(x + e);
                v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
                v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) n2 = fmaf(v[i], v[i], n2);
        }
        const int h = (int)((r / p.N) % p.H);
        kw[r] = expf(n2 * expf(-tau[h]));
    }
}

// The same for bf16 rows of d = 64 (the tensor-core shapes): 8 lanes per row, one 16-byte
// load each (fully coalesced), 4 rows in flight per lane, the 8 partial sums combined by
// xor shuffles.
__global__ void __launch_bounds__(kThreads) key_weights_bf16_d64_kernel(Problem p,
                                                                         const __nv_bfloat16* k,
                                                                         const float* tau,
                                                                         float* kw)
{
    tc::grid_dep_launch();
    constexpr int kUnroll = 4;
    const size_t rows = (size_t)p.B * p.H * p.N;
    const int lane = threadIdx.x & 31, sub = lane & 7;
    const size_t warps = (size_t)gridDim.x * (blockDim.x / 32);
    const size_t gw = (size_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    for (size_t r0 = gw * 4 * kUnroll; r0 < rows; r0 += warps * 4 * kUnroll) {
        uint4 x[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const size_t r = r0 + 4 * u + (lane >> 3);
            x[u] = r < rows ? *reinterpret_cast<const uint4*>(k + r * 64 + 8 * sub)
                            : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const uint32_t wv[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
            float n2 = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float a = __uint_as_float(wv[e] << 16), b = __uint_as_float(wv[e] & 0xffff0000u);
                n2 = fmaf(a, a, fmaf(b, b, n2));
            }
            n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
            n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
            n2 += __shfl_xor_sync(0xffffffffu, n2, 4);
            const size_t r = r0 + 4 * u + (lane >> 3);
            if (sub == 0 && r < rows) kw[r] = expf(n2 * expf(-tau[(r / p.N) % p.H]));
        }
    }
}

// dW over the batch, in a fixed order (deterministic).  Nonstationary: the partials hold
// dU (rows < M) and dV (rows >= M); dW1 = (dU + dV)/2, dW2 = (dU - dV)/2.
__global__ void dw_reduce_kernel(Problem p, const float* part, float* dW1, float* dW2,
                                 const float* dtau_part, float* dtau)
{
    tc::grid_dep_wait();
    const int d = p.d, M = p.M, Mc = p.nonstat ? 2 * M : M;
    const size_t per = (size_t)M * d;
    if (dtau && blockIdx.x == 0)  // dtau[h] = sum over the batch, in order
        for (int h = threadIdx.x; h < p.H; h += blockDim.x) {
            float t = 0.f;
            for (int bb = 0; bb < p.B; ++bb) t += dtau_part[(size_t)bb * p.H + h];
            dtau[h] = t;
        }
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < (size_t)p.H * per;
         idx += (size_t)gridDim.x * blockDim.x) {
        int h = (int)(idx / per);
        size_t e = idx % per;
        float a = 0.f, b = 0.f;
        for (int bb = 0; bb < p.B; ++bb) {
            const float* pp = part + ((size_t)bb * p.H + h) * Mc * d;
            a += pp[e];
            if (p.nonstat) b += pp[per + e];
        }
        if (!p.nonstat) {
            dW1[idx] = a;
        } else {
            dW1[idx] = 0.5f * (a + b);
            dW2[idx] = 0.5f * (a - b);
        }
    }
}


// ---- sizes taken by the entry points ----------------------------------------------------
// A sequence's frequencies and state (and eight tokens of every operand) have to fit one
// CTA's shared memory: 227 KB of fp32.
constexpr size_t kSmemFloats = 227 * 1024 / 4;
constexpr size_t kMaxDw = 16384;  // Mc * d, the backward's frequency gradient

bool fits_fwd(const Problem& p)
{
    const size_t d = p.d, D = 2 * (size_t)p.M, Mc = p.nonstat ? D : D / 2;
    return Mc * (d + 1) + D * (d + 1) + 8 * (2 * d + 2 * (d + 1) + 2 * (D + 1) + 8) <= kSmemFloats;
}
bool fits_bwd(const Problem& p)
{
    const size_t d = p.d, D = 2 * (size_t)p.M, Mc = p.nonstat ? D : D / 2;
    return Mc * d <= kMaxDw && Mc * (d + 1) + D * (d + 1) +
                                       8 * (2 * d + 2 * (d + 1) + 3 * (D + 1) + 16 + Mc + 1 + 1) <=
                                   kSmemFloats;
}

// The plan for groups of at most mg frequencies and T tokens per chunk, with or without
// resident projection rows.
Plan layout(const Problem& p, bool bwd, int mg, int T, bool wres, int nt = kThreads)
{
    Plan L = {};
    L.T = T;
    L.lpr = T > 64 ? 2 : 4;
    L.nt = nt;
    L.wres = wres;
    L.CL = 1;
    L.ng = (p.M + mg - 1) / mg;
    L.MG = ((p.M + L.ng - 1) / L.ng + 3) / 4 * 4;
    L.CT = L.MG / 2;
    L.F = 2 * L.MG;
    L.KP = p.nonstat ? 2 * L.MG : L.MG;
    L.pd = p.d + 4;
    L.pp = L.F + 4;
    L.pa = (std::max(T, L.CT) + 3) / 4 * 4 + 4;  // (also the backward's s_j partials, CT a row)
    int o = 0;
    auto take = [&](int n) {
        const int at = o;
        o += n;
        return at;
    };
    const int rows = T * L.pd, feats = T * std::max(L.pp, L.pa);
    L.S = take(L.ng * L.F * L.pd);
    L.W = take((wres ? L.ng : 1) * L.KP * L.pd);
    L.dW = bwd ? take(L.ng * L.KP * p.d) : 0;
    // without the mask one pass holds only queries or only keys: their regions are one
    L.Xk = take(rows);
    L.Xq = p.causal ? take(rows) : L.Xk;
    L.V = take(rows);
    L.G = !bwd ? 0 : p.causal ? take(rows) : L.V;
    L.Pk = take(feats);
    L.Pq = p.causal ? take(feats) : L.Pk;
    // forward: phi(Q) phi(K)^T replaces phi(Q); backward: dA has its own block (causal), and
    // without the mask only the prefactor's s_j go there, after the features' last use
    L.A = bwd && p.causal ? take(T * L.pa) : L.Pq;
    L.red = take(2 * kMaxT);
    L.total = o;
    return L;
}

// The largest chunk that fits, with the projection rows resident when they fit beside it
// (M <= 32 has one group, staged once either way); then the CTAs per sequence: the count
// that minimises the rounds of CTAs on the SMs times the work of one, counted in chunks
// (a range's own sums, needed when the sequence is split or not causal, cost about 0.4 of
// a forward chunk, a backward chunk about 3; set-up about one).
bool make_plan(const Problem& p, bool bwd, Plan* plan)
{
    if (!(bwd ? fits_bwd(p) : fits_fwd(p))) return false;
    bool found = false;
    // 128 tokens where 64 would give no more than half of the threads a tile of features and of
    // the output (non-causal forward, long enough sequences): bf16 n B32 H4 N1024 d32 M16
    // 90 -> 73 us.
    const Plan small = layout(p, bwd, kMaxMG, 64, true);
    const int tiles = 16 * std::max(small.CT, p.d / 4);
    if (!bwd && !p.causal && 2 * tiles <= kThreads && p.N >= 512) {
        *plan = layout(p, bwd, kMaxMG, 128, true);
        found = 2 * ((size_t)plan->total * 4 + 1024) <= 228 * 1024;
    }
    // Short sequences: a chunk no longer than needed and groups as large as its threads take (the
    // groups run one after the other); more sequences than run at once (two CTAs an SM) take no
    // more threads than have a tile.  The kernels before these (one output a thread), chunks of
    // 64, this: forward n non-causal N16 d64 M64, 64 sequences 41, 31, 19 us, 2048 sequences 519,
    // 391, 154; d16 M256, 64 sequences 47, 60, 29.  At N 1 still up to 1.5 times the kernels before
    // (d16 M256: 19, 60, 28; d32 M32, 2048 sequences: 33, 107, 41), backwards at most even.
    const bool many = p.d <= 64 && (long long)p.B * p.H > 2 * 152;
    if (!found && p.N <= 32) {
        const int T = p.N <= 16 ? 16 : 32, mg = 8 * kThreads / T;
        const int ct = layout(p, bwd, mg, T, true).CT;
        int nt = 4 * T;
        while (nt < kThreads && (!many || nt < T / 4 * std::max(ct, p.d / 4))) nt *= 2;
        *plan = layout(p, bwd, mg, T, true, nt);
        found = (size_t)plan->total <= kSmemFloats;
    }
    // Many sequences of small heads: half the threads of a 64-token chunk would have no tile.
    // Forward n, N65 d16 M16, 1024 sequences, the same three: causal 76, 97, 58 us, not 58, 72, 54.
    // (d4 M4, N200, 2048 sequences, not causal: 91, 193, 179.)
    if (!found && many && tiles <= kThreads / 2) {
        *plan = layout(p, bwd, kMaxMG, 32, true, 128);
        found = true;  // (a 64-token chunk fits)
    }
    plan->any = found && plan->T < 64;
    for (int mg = kMaxMG; mg >= 4 && !found; mg /= 2)  // smaller groups: the largest shapes only
        for (int T = 64; T >= 8 && !found; T /= 2)
            for (int wres = 1; wres >= 0 && !found; --wres) {
                *plan = layout(p, bwd, mg, T, wres != 0);
                found = (size_t)plan->total <= kSmemFloats;
            }
    if (!found) return false;
    // (16 sequences: 8 CTAs each take two rounds, 0.51 ms on the training shape above; 6 take one,
    // 0.36 ms.)
    // Clusters of 1..8 CTAs that run at once with one CTA per SM (cudaOccupancyMaxActiveClusters
    // on GB300: 152 SMs in eight groups, of which a cluster takes its SMs from one).
    static const int kClusters[kMaxCluster] = {152, 76, 46, 36, 28, 23, 15, 15};
    const int occ = !bwd && 2 * ((size_t)plan->total * 4 + 1024) <= 228 * 1024 ? 2 : 1;
    const long long bh = (long long)p.B * p.H, nch = (p.N + plan->T - 1) / plan->T;
    double best = 0.;
    for (int cl = 1; cl <= kMaxCluster && (cl == 1 || cl <= nch); ++cl) {
        const double per = (double)((nch + cl - 1) / cl);
        const double pre = !p.causal || cl > 1 ? (bwd ? 0.8 : 0.4) : 0.;
        const long long cap = (long long)kClusters[cl - 1] * occ;
        double rounds = (double)((bh + cap - 1) / cap);
        if (occ == 2 && bh > kClusters[cl - 1]) rounds *= 1.6;  // two CTAs share an SM
        const double cost = rounds * (per * ((bwd ? 3. : 1.) + pre) + 1. + (cl > 1 ? 0.5 : 0.));
        if (cl == 1 || cost < best) {
            best = cost;
            plan->CL = cl;
        }
    }
    return true;
}

// Launches `kern` with CL CTAs per sequence as one cluster.
template <typename... KArgs, typename... Args>
cudaError_t launch_plan(void (*kern)(KArgs...), const Problem& p, const Plan& L, cudaStream_t s,
                        Args... args)
{
    const size_t smem = (size_t)L.total * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)p.B * p.H * L.CL));
    cfg.blockDim = dim3((unsigned)L.nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)L.CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, L, args...);
}

template <typename T, bool NS>
cudaError_t launch_fwd_t(const Problem& p, const Plan& L, const void* q, const void* k,
                         const void* v, const float* W1, const float* W2, const float* tau,
                         void* out, float* den, cudaStream_t s)
{
    auto kern = L.any ? simt_fwd_kernel<T, NS, 2, 0>
                : p.d > 64 ? simt_fwd_kernel<T, NS, 2, kThreads>
                           : simt_fwd_kernel<T, NS, 1, kThreads>;
    return launch_plan(kern, p, L, s, (const T*)q, (const T*)k, (const T*)v, W1, W2, tau, (T*)out,
                       den);
}

template <typename T, bool NS>
cudaError_t launch_bwd_t(const Problem& p, const Plan& L, const void* q, const void* k,
                         const void* v, const float* W1, const float* W2, const float* tau,
                         const void* out, const float* den, const void* dout, void* dq, void* dk,
                         void* dv, float* part, float* tpart, cudaStream_t s)
{
    auto kern = L.any ? simt_bwd_kernel<T, NS, 2, 0>
                : p.d > 64 ? simt_bwd_kernel<T, NS, 2, kThreads>
                           : simt_bwd_kernel<T, NS, 1, kThreads>;
    return launch_plan(kern, p, L, s, (const T*)q, (const T*)k, (const T*)v, W1, W2, tau,
                       (const T*)out, den, (const T*)dout, (T*)dq, (T*)dk, (T*)dv, part, tpart);
}

}  // namespace

bool simt_fwd_supported(const Problem& p)
{
    Plan L;
    return make_plan(p, false, &L);
}

bool simt_bwd_supported(const Problem& p)
{
    Plan L;
    return make_plan(p, true, &L);
}

// dW partials [B*H][Mc][d], then dtau partials [B*H].
size_t simt_bwd_ws_bytes(const Problem& p)
{
    const int Mc = p.nonstat ? 2 * p.M : p.M;
    return (size_t)p.B * p.H * (Mc * p.d + 1) * sizeof(float);
}

cudaError_t launch_key_weights(const Problem& p, const void* k, const float* tau, float* kw,
                               cudaStream_t s)
{
    const size_t rows = (size_t)p.B * p.H * p.N;
    if (p.bf16 && p.d == 64) {  // 16 rows per warp and iteration, 8 warps per block
        const int blocks = (int)std::min<size_t>((rows + 127) / 128, 152 * 16);
        key_weights_bf16_d64_kernel<<<blocks, kThreads, 0, s>>>(p, (const __nv_bfloat16*)k, tau,
                                                                 kw);
        return cudaGetLastError();
    }
    const int blocks = (int)std::min<size_t>((rows + kThreads - 1) / kThreads, 152 * 16);
    if (p.bf16)
        key_weights_kernel<<<blocks, kThreads, 0, s>>>(p, (const __nv_bfloat16*)k, tau, kw);
    else
        key_weights_kernel<<<blocks, kThreads, 0, s>>>(p, (const float*)k, tau, kw);
    return cudaGetLastError();
}

cudaError_t launch_featmap(const Problem& p, const void* x, const float* W1, const float* W2,
                           void* phi, cudaStream_t s)
{
    return launch_featmap_scaled(p, x, W1, W2, nullptr, phi, s);
}

cudaError_t launch_featmap_scaled(const Problem& p, const void* x, const float* W1,
                                  const float* W2, const float* rowscale, void* phi,
                                  cudaStream_t s)
{
    const size_t work = (size_t)p.B * p.H * p.N * p.M;
    const int blocks = (int)std::min<size_t>((work + kThreads - 1) / kThreads, 152 * 16);
    const float scale = 1.0f / sqrtf((float)p.M);
    if (p.bf16)
        featmap_kernel<<<blocks, kThreads, 0, s>>>(p, (const __nv_bfloat16*)x, W1, W2,
                                                   (__nv_bfloat16*)phi, scale, rowscale);
    else
        featmap_kernel<<<blocks, kThreads, 0, s>>>(p, (const float*)x, W1, W2, (float*)phi,
                                                   scale, rowscale);
    return cudaGetLastError();
}

cudaError_t launch_simt_fwd(const Problem& p, const void* q, const void* k, const void* v,
                            const float* W1, const float* W2, const float* tau, void* out,
                            float* den, cudaStream_t s)
{
    Plan L;
    if (!make_plan(p, false, &L)) return cudaErrorInvalidValue;
    typedef __nv_bfloat16 B16;
    auto run = p.bf16 ? (p.nonstat ? launch_fwd_t<B16, true> : launch_fwd_t<B16, false>)
                      : (p.nonstat ? launch_fwd_t<float, true> : launch_fwd_t<float, false>);
    return run(p, L, q, k, v, W1, W2, tau, out, den, s);
}

cudaError_t launch_simt_bwd(const Problem& p, const void* q, const void* k, const void* v,
                            const float* W1, const float* W2, const float* tau,
                            const void* out, const float* den, const void* dout, void* dq,
                            void* dk, void* dv, float* dW1, float* dW2, float* dtau,
                            void* scratch, cudaStream_t s)
{
    Plan L;
    if (!make_plan(p, true, &L)) return cudaErrorInvalidValue;
    const int Mc = p.nonstat ? 2 * p.M : p.M;
    float* part = (float*)scratch;
    float* tpart = part + (size_t)p.B * p.H * Mc * p.d;
    typedef __nv_bfloat16 B16;
    auto run = p.bf16 ? (p.nonstat ? launch_bwd_t<B16, true> : launch_bwd_t<B16, false>)
                      : (p.nonstat ? launch_bwd_t<float, true> : launch_bwd_t<float, false>);
    cudaError_t e = run(p, L, q, k, v, W1, W2, tau, out, den, dout, dq, dk, dv, part, tpart, s);
    if (e != cudaSuccess) return e;
    const size_t work = (size_t)p.H * p.M * p.d;
    const int blocks = (int)std::min<size_t>((work + kThreads - 1) / kThreads, 152 * 8);
    return tc::launch_after(dw_reduce_kernel, dim3((unsigned)blocks), kThreads, 0, 0, true, s, p, (const float*)part,
                            dW1, dW2, (const float*)tpart, tau ? dtau : (float*)nullptr);
}

}  // namespace flex
