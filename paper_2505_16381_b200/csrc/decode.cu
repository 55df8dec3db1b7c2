// Decoding step with an in-place key cache (paper Sec. 3.4).
//
// The cache holds kc_j = H_{t-1} ... H_{j+1} k_j for every past position, in float32: when token t arrives every
// cached key gets kc_j <- H_t kc_j = kc_j - beta_t w_t (w_t . kc_j), then (k_t, v_t) are appended untouched, and the
// step's output is plain softmax attention of q_t over the cache.  The update and the attention are one pass over the
// cache (each key row is read once, updated, written back and used for its logit while still in registers), so the
// step is bound by memory bandwidth: 2 * 4 d bytes per cached key plus 2 d for its value.  The cache is float32
// because it is rewritten at every step: a bf16 cache would be rounded t times.
//
// One half-warp handles U cached keys at a time, the head dimension spread over its 16 lanes; a CTA covers a contiguous
// range of positions of one (batch, head) slice and leaves a partial softmax state (max, sum, weighted values), which
// a small second kernel merges over the CTAs of the slice.  The length of the ranges is set by `splits`: a fixed 256
// positions per CTA left 129 states per head to merge at 32768 cached tokens (23 of 237 us).  GPU time of a step, before (256
// positions per CTA, one position per half-warp at a time) and after: 32 heads x 32768, d = 128: 237 -> 220 us (6.1 TB/s);
// the same with d = 64: 173 -> 119; 128 heads x 700, d = 64: 24.2 -> 15.2; 16 heads x 2000, d = 128: 20.6 -> 14.2.
#include "common.cuh"

namespace path {

namespace {

constexpr int kWarps = 8, kSlots = 3 * 148, kMinKeys = 64, kMaxSplits = 96;

// The number of SMs is a constant here because the workspace query, which needs no device, has to come to the same answer.
// The merge counts on every range but the last having a position (an empty state would be a NaN in it): for one of n ranges over t
// positions to stay empty, (n - 2) ceil(t / n) >= t, n would have to exceed 2 ceil(t / n), and ceil(t / n) is at least kMinKeys - 1.
static_assert(kMaxSplits <= 2 * kMinKeys - 2, "a range could be empty");

// CTAs per slice for n positions: one wave of the GPU (three CTAs per SM), ranges of at least 64 positions and no more states
// than the merge reads quickly (2 heads x 20000 tokens, d = 128: 29 us with 222 states, 24 with 79).  Long ranges are cut in
// four: with 2500 positions per CTA the wave's end is ragged (32 heads x 32768 x 128: 230 us, 220 with 600 per CTA), with
// 1200 the larger merge costs more than that (8 heads x 65000: 121 against 137).
__host__ __device__ inline int splits(int S, int n) {
    int most = kSlots / S > 1 ? kSlots / S : 1;
    if (n / most > 1536) most *= 4;
    const int fit = (n + kMinKeys - 1) / kMinKeys;
    most = most < kMaxSplits ? most : kMaxSplits;
    return fit < most ? fit : most;
}

// part: [S][nsplit][HD + 2] = (max, sum, weighted values) of each CTA's positions
//
// A half-warp (16 lanes) owns one cached position: lane j of the half holds the elements [4j, 4j+4) of every 64-element
// panel of the row (16-byte loads, a half-warp covers 256 contiguous bytes per instruction).  It works on U positions at
// once, so a warp has 2 U key rows and 2 U value rows in flight; U = 2 (d = 128) or 4 (d = 64) makes that 3 KB per warp.
template <int HD>
__global__ void __launch_bounds__(32 * kWarps, 3) decode_update_kernel(
    const __nv_bfloat16* __restrict__ q_t, const __nv_bfloat16* __restrict__ k_t, const __nv_bfloat16* __restrict__ v_t,
    const __nv_bfloat16* __restrict__ w_t, const float* __restrict__ beta_t, const float* __restrict__ log_f_t, float* kc,
    __nv_bfloat16* vc, float* gc, int t, int cap, int per_cta, float scale, float* __restrict__ part) {
    grid_wait();
    grid_launch();
    constexpr int NP = HD / 64;          // 64-element panels per row
    constexpr int NH = 2 * kWarps;       // half-warps per CTA
    constexpr int U = 4 / NP;            // positions per half-warp and step
    __shared__ float sm_m[NH], sm_l[NH], sm_acc[NH][HD];
    const int lane = threadIdx.x & 31, hl = lane & 15, hw = threadIdx.x >> 4;   // lane in the half-warp, half-warp in the CTA
    const int s = blockIdx.y, nsplit = gridDim.x;
    const int lo = blockIdx.x * per_cta, hi = min(lo + per_cta, t);             // cached positions; the new token is apart
    auto unpack = [](const uint2& u, float (&x)[4]) {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
        const float2 b2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
        x[0] = a.x; x[1] = a.y; x[2] = b2.x; x[3] = b2.y;
    };
    auto ld_bf16 = [&](const __nv_bfloat16* row, float (&x)[NP][4]) {
#pragma unroll
        for (int pn = 0; pn < NP; ++pn) unpack(*reinterpret_cast<const uint2*>(row + pn * 64 + hl * 4), x[pn]);
    };
    float q[NP][4], w[NP][4];
    ld_bf16(q_t + (size_t)s * HD, q);
    ld_bf16(w_t + (size_t)s * HD, w);
    const float b = beta_t[s];
    float qw = 0.f;
#pragma unroll
    for (int pn = 0; pn < NP; ++pn)
#pragma unroll
        for (int e = 0; e < 4; ++e) qw = fmaf(q[pn][e], w[pn][e], qw);
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) qw += __shfl_xor_sync(0xffffffffu, qw, off);
    const float Gt = gc ? ((t > 0 ? gc[(size_t)s * cap + t - 1] : 0.f) + log_f_t[s]) : 0.f;
    float* kcs = kc + (size_t)s * cap * HD;
    __nv_bfloat16* vcs = vc + (size_t)s * cap * HD;
    float m = -INFINITY, l = 0.f, acc[NP][4];
#pragma unroll
    for (int pn = 0; pn < NP; ++pn)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[pn][e] = 0.f;

    // both halves of a warp run the same number of iterations (the shuffles below name all 32 lanes)
    for (int i0 = lo + hw; i0 - hw < hi; i0 += NH * U) {
        float4 kk[U][NP];
        uint2 vv[U][NP];
        float Gi[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * NH;
            Gi[u] = 0.f;
#pragma unroll
            for (int pn = 0; pn < NP; ++pn) { kk[u][pn] = make_float4(0.f, 0.f, 0.f, 0.f); vv[u][pn] = make_uint2(0u, 0u); }
            if (i < hi) {
#pragma unroll
                for (int pn = 0; pn < NP; ++pn) {
                    kk[u][pn] = *reinterpret_cast<const float4*>(kcs + (size_t)i * HD + pn * 64 + hl * 4);
                    vv[u][pn] = *reinterpret_cast<const uint2*>(vcs + (size_t)i * HD + pn * 64 + hl * 4);
                }
                if (gc) Gi[u] = gc[(size_t)s * cap + i];
            }
        }
        float a[U], c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = c[u] = 0.f;
#pragma unroll
            for (int pn = 0; pn < NP; ++pn) {
                const float4 f = kk[u][pn];
                a[u] = fmaf(q[pn][0], f.x, a[u]); a[u] = fmaf(q[pn][1], f.y, a[u]);
                a[u] = fmaf(q[pn][2], f.z, a[u]); a[u] = fmaf(q[pn][3], f.w, a[u]);
                c[u] = fmaf(w[pn][0], f.x, c[u]); c[u] = fmaf(w[pn][1], f.y, c[u]);
                c[u] = fmaf(w[pn][2], f.z, c[u]); c[u] = fmaf(w[pn][3], f.w, c[u]);
            }
        }
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1)   // within the half-warp
#pragma unroll
            for (int u = 0; u < U; ++u) {
                a[u] += __shfl_xor_sync(0xffffffffu, a[u], off);
                c[u] += __shfl_xor_sync(0xffffffffu, c[u], off);
            }
        float sc[U], mn = m;
#pragma unroll
        for (int u = 0; u < U; ++u) {   // kc_i <- H_t kc_i; its logit follows from the two dot products already known
            const int i = i0 + u * NH;
            const float coef = b * c[u];
            sc[u] = -INFINITY;
            if (i < hi) {
#pragma unroll
                for (int pn = 0; pn < NP; ++pn) {
                    float4 f = kk[u][pn];
                    f.x = fmaf(-coef, w[pn][0], f.x); f.y = fmaf(-coef, w[pn][1], f.y);
                    f.z = fmaf(-coef, w[pn][2], f.z); f.w = fmaf(-coef, w[pn][3], f.w);
                    *reinterpret_cast<float4*>(kcs + (size_t)i * HD + pn * 64 + hl * 4) = f;
                }
                sc[u] = fmaf(scale, a[u] - coef * qw, Gt - Gi[u]);
            }
            mn = fmaxf(mn, sc[u]);
        }
        if (mn > m) {   // uniform over the half-warp
            const float r = expf(m - mn);
            l *= r;
#pragma unroll
            for (int pn = 0; pn < NP; ++pn)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[pn][e] *= r;
            m = mn;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * NH >= hi) continue;
            const float pj = expf(sc[u] - m);
            l += pj;
#pragma unroll
            for (int pn = 0; pn < NP; ++pn) {
                float x[4];
                unpack(vv[u][pn], x);
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[pn][e] = fmaf(pj, x[e], acc[pn][e]);
            }
        }
    }
    // the new token, appended as it is by the first half-warp of the slice's last CTA
    if (blockIdx.x == nsplit - 1 && threadIdx.x < 32) {
        float kk[NP][4], vv[NP][4], a = 0.f;
        ld_bf16(k_t + (size_t)s * HD, kk);
        ld_bf16(v_t + (size_t)s * HD, vv);
#pragma unroll
        for (int pn = 0; pn < NP; ++pn)
#pragma unroll
            for (int e = 0; e < 4; ++e) a = fmaf(q[pn][e], kk[pn][e], a);
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (hw == 0) {
            const float sc = scale * a, mn = fmaxf(m, sc), r = expf(m - mn), pj = expf(sc - mn);
            m = mn;
            l = fmaf(l, r, pj);
#pragma unroll
            for (int pn = 0; pn < NP; ++pn) {
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[pn][e] = fmaf(acc[pn][e], r, pj * vv[pn][e]);
                *reinterpret_cast<float4*>(kcs + (size_t)t * HD + pn * 64 + hl * 4) = make_float4(kk[pn][0], kk[pn][1], kk[pn][2], kk[pn][3]);
                *reinterpret_cast<uint2*>(vcs + (size_t)t * HD + pn * 64 + hl * 4) =
                    *reinterpret_cast<const uint2*>(v_t + (size_t)s * HD + pn * 64 + hl * 4);
            }
            if (gc && hl == 0) gc[(size_t)s * cap + t] = Gt;
        }
    }
    // merge the half-warps of the CTA
    if (hl == 0) { sm_m[hw] = m; sm_l[hw] = l; }
#pragma unroll
    for (int pn = 0; pn < NP; ++pn)
#pragma unroll
        for (int e = 0; e < 4; ++e) sm_acc[hw][pn * 64 + hl * 4 + e] = acc[pn][e];
    __syncthreads();
    float M = -INFINITY;
#pragma unroll
    for (int x = 0; x < NH; ++x) M = fmaxf(M, sm_m[x]);
    float* out = part + ((size_t)s * nsplit + blockIdx.x) * (HD + 2);
    if (threadIdx.x < HD) {
        float a = 0.f;
#pragma unroll
        for (int x = 0; x < NH; ++x) a += sm_acc[x][threadIdx.x] * expf(sm_m[x] - M);   // an idle half-warp has max = -inf: factor 0
        out[2 + threadIdx.x] = a;
    }
    if (threadIdx.x == 0) {
        float a = 0.f;
#pragma unroll
        for (int x = 0; x < NH; ++x) a += sm_l[x] * expf(sm_m[x] - M);
        out[0] = M; out[1] = a;
    }
}

// One CTA per slice; the partial states are read HD at a time, all loads of a pass in flight together.
template <int HD>
__global__ void __launch_bounds__(HD) decode_merge_kernel(const float* __restrict__ part, int nsplit, __nv_bfloat16* __restrict__ o_t,
                                                         float* __restrict__ lse_t) {
    grid_wait();
    grid_launch();
    constexpr int kAhead = 8;
    __shared__ float sf[kMaxSplits];
    __shared__ float sm_x[HD / 32], sl_x[HD / 32];
    const int s = blockIdx.x, tid = threadIdx.x;
    const float* p = part + (size_t)s * nsplit * (HD + 2);
    float M = -INFINITY;
    for (int c = tid; c < nsplit; c += HD) M = fmaxf(M, p[(size_t)c * (HD + 2)]);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    if ((tid & 31) == 0) sm_x[tid >> 5] = M;
    __syncthreads();
#pragma unroll
    for (int x = 0; x < HD / 32; ++x) M = fmaxf(M, sm_x[x]);
    float l = 0.f;
    for (int c = tid; c < nsplit; c += HD) {
        const float f = expf(p[(size_t)c * (HD + 2)] - M);
        sf[c] = f;
        l = fmaf(p[(size_t)c * (HD + 2) + 1], f, l);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if ((tid & 31) == 0) sl_x[tid >> 5] = l;
    __syncthreads();
    l = 0.f;
#pragma unroll
    for (int x = 0; x < HD / 32; ++x) l += sl_x[x];
    float a = 0.f;
    for (int c0 = 0; c0 < nsplit; c0 += kAhead) {
        float x[kAhead];
#pragma unroll
        for (int y = 0; y < kAhead; ++y) x[y] = c0 + y < nsplit ? p[(size_t)(c0 + y) * (HD + 2) + 2 + tid] : 0.f;
#pragma unroll
        for (int y = 0; y < kAhead; ++y)
            if (c0 + y < nsplit) a = fmaf(x[y], sf[c0 + y], a);
    }
    o_t[(size_t)s * HD + tid] = __float2bfloat16_rn(a / l);
    if (tid == 0) lse_t[s] = M + logf(l);
}

}  // namespace

size_t decode_partials_bytes(int S, int cap, int hd) {
    return (size_t)S * splits(S, cap) * (hd + 2) * sizeof(float);
}

cudaError_t launch_decode_step(const void* q_t, const void* k_t, const void* v_t, const void* w_t, const float* beta_t,
                               const float* log_f_t, float* kc, void* vc, float* gc, int t, int cap, void* o_t, float* lse_t,
                               int S, int hd, float scale, float* part, cudaStream_t st) {
    typedef __nv_bfloat16 bf;
    const int n = splits(S, t + 1), per_cta = (t + n - 1) / n;
    for (int s0 = 0; s0 < S; s0 += 65535) {   // (a grid's second dimension ends there)
        const dim3 grid(n, S - s0 < 65535 ? S - s0 : 65535);
        const size_t x = (size_t)s0 * hd, y = (size_t)s0 * cap;
        const bf *q = (const bf*)q_t + x, *k = (const bf*)k_t + x, *v = (const bf*)v_t + x, *w = (const bf*)w_t + x;
        const float *b = beta_t + s0, *f = log_f_t ? log_f_t + s0 : nullptr;
        float *kcs = kc + y * hd, *gcs = gc ? gc + y : nullptr, *ps = part + (size_t)s0 * n * (hd + 2);
        bf* vcs = (bf*)vc + y * hd;
        const cudaError_t e =
            hd == 64 ? launch<decode_update_kernel<64>>(grid, 32 * kWarps, 0, st, q, k, v, w, b, f, kcs, vcs, gcs, t, cap, per_cta, scale, ps)
                     : launch<decode_update_kernel<128>>(grid, 32 * kWarps, 0, st, q, k, v, w, b, f, kcs, vcs, gcs, t, cap, per_cta, scale, ps);
        if (e != cudaSuccess) return e;
    }
    return hd == 64 ? launch<decode_merge_kernel<64>>(S, 64, 0, st, (const float*)part, n, (bf*)o_t, lse_t)
                    : launch<decode_merge_kernel<128>>(S, 128, 0, st, (const float*)part, n, (bf*)o_t, lse_t);
}

}  // namespace path
