// Forward pass for float32 tensors (PATH_FP32), in float32 on the CUDA cores: the accuracy path.
//
// The definition walks the keys j = i, i-1, ..., 0 of a query i carrying u_{i,j} = H_{j+1} ... H_i q_i (paper Sec. 2.2: logit
// s_ij = scale * k_j . u_{i,j} + G_i - G_j, then u <- u - beta_j w_j (w_j . u)): one dependent dot product per key.  Here the
// walk goes 32 keys at a time (the UT form of Sec. 3.1 on small blocks).  With u0 = u at a block's last key and
// t = W u0 (32 dot products at once),
//     T = (I + C)^-1,  C_jm = beta_m w_j . w_m  (m > j),      Y = strictUpper(K W^T) D T
//     logits of the block:  K u0 - Y t = (K - Y W) u0 = Kr u0,      u after the block:  u0 - ((D T)^T W)^T t = u0 - Wt^T t
// Kr, Wt and Y belong to the keys alone: fp32_block_kernel makes them once per block.  A query's own block uses K, Y and t with
// the entries after the query set to zero.
//
// Blocks with a NaN or an infinity, in k, v, w, beta or in what is made of them, are walked key by key: products with zeros
// would carry it into rows before its position, and sums in another order turn an infinite logit, which the definition handles
// (minus infinity has no weight), into a NaN.  fp32_block_kernel marks them.
//
// fp32_fwd_kernel: a warp owns RW queries of one block, lane j the block's key j: two dot products per lane with rows from
// shared memory (u0 broadcast), then the lanes turn to the head dimension for the update of u and for P V.  What bounds it
// at the sizes it is for (a few slices, a few hundred tokens) is the chain of dependent phases of one block, L / 32 times.
// B=1, H=2, L=256, d=64: 69.7 -> 20.8 us per call (one key per step: 520 cycles each).
#include "common.cuh"

namespace path {

namespace {

constexpr int kBlk = 32;           // keys per block
constexpr int kWarps = 4;          // warps per CTA

template <int HD>
__device__ __host__ constexpr int ld() { return HD + 4; }   // row stride in floats: 16-byte rows, lanes on different banks

__device__ __forceinline__ float dot4(const float4& a, const float4& b) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}

// ---------------------------------------------------------------------------------------------- per block of keys
// grid = (blocks, S), 256 threads.  kr, wt: [S][nblk * 32][HD], ym: [S][nblk * 32][32], odd: [S][nblk].
template <int HD>
__global__ void __launch_bounds__(256) fp32_block_kernel(const float* __restrict__ k, const float* __restrict__ w,
                                                         const float* __restrict__ beta, const float* __restrict__ v,
                                                         float* __restrict__ kr, float* __restrict__ wt, float* __restrict__ ym,
                                                         int* __restrict__ odd, uint32_t* clear, int L) {
    grid_wait();
    grid_launch();
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 64) clear[threadIdx.x] = 0u;   // the workspace's status block
    constexpr int LD = ld<HD>(), LC = kBlk + 4;
    __shared__ __align__(16) float sw[kBlk][LD], sk[kBlk][LD], sc[kBlk][LC], skw[kBlk][LC];
    __shared__ float sb[kBlk];
    const int tid = threadIdx.x, blk = blockIdx.x, s = blockIdx.y, nblk = gridDim.x;
    const int row = tid >> 3, part = tid & 7;
    const bool live = blk * kBlk + row < L;
    const size_t src = ((size_t)s * L + blk * kBlk + row) * HD, dst = ((size_t)s * nblk + blk) * kBlk + row;
    float zero = 0.f;   // 0, or NaN if anything in this block is not finite
    auto look = [&](const float4& x) { zero = fmaf(x.x, 0.f, fmaf(x.y, 0.f, fmaf(x.z, 0.f, fmaf(x.w, 0.f, zero)))); };
#pragma unroll
    for (int c = 0; c < HD / 32; ++c) {
        const int e = c * 32 + part * 4;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        look(live ? *reinterpret_cast<const float4*>(v + src + e) : z);
        *reinterpret_cast<float4*>(&sw[row][e]) = live ? *reinterpret_cast<const float4*>(w + src + e) : z;
        *reinterpret_cast<float4*>(&sk[row][e]) = live ? *reinterpret_cast<const float4*>(k + src + e) : z;
    }
    if (tid < kBlk) sb[tid] = blk * kBlk + tid < L ? beta[(size_t)s * L + blk * kBlk + tid] : 0.f;
    __syncthreads();
    {   // C and K W^T above the diagonal: row `row`, columns part, part + 8, ...
        float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int e = 0; e < HD; e += 4) {
            const float4 wr = *reinterpret_cast<const float4*>(&sw[row][e]), kk = *reinterpret_cast<const float4*>(&sk[row][e]);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float4 wm = *reinterpret_cast<const float4*>(&sw[part + 8 * x][e]);
                a[x] += dot4(wr, wm);
                b[x] += dot4(kk, wm);
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int m = part + 8 * x;
            sc[m][row] = m > row ? sb[m] * a[x] : 0.f;   // (C transposed: the substitution goes column by column)
            skw[row][m] = m > row ? b[x] : 0.f;
        }
    }
    __syncthreads();
    if (tid < kBlk) {   // column tid of T by back substitution, in registers; D T replaces C
        float x[kBlk];
#pragma unroll
        for (int j = 0; j < kBlk; ++j) x[j] = j == tid ? 1.f : 0.f;
#pragma unroll
        for (int j = kBlk - 1; j > 0; --j)
#pragma unroll
            for (int i = 0; i < j; ++i) x[i] = fmaf(-sc[j][i], x[j], x[i]);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kBlk; ++j) sc[j][tid] = sb[j] * x[j];
    }
    __syncthreads();
    float y[4] = {0.f, 0.f, 0.f, 0.f};   // Y[row][4 part ..]
#pragma unroll 8
    for (int p = 0; p < kBlk; ++p) {
        const float c = skw[row][p];
        const float4 d4 = *reinterpret_cast<const float4*>(&sc[p][4 * part]);
        y[0] = fmaf(c, d4.x, y[0]); y[1] = fmaf(c, d4.y, y[1]); y[2] = fmaf(c, d4.z, y[2]); y[3] = fmaf(c, d4.w, y[3]);
    }
    *reinterpret_cast<float4*>(ym + dst * kBlk + 4 * part) = make_float4(y[0], y[1], y[2], y[3]);
    look(make_float4(y[0], y[1], y[2], y[3]));
    __syncthreads();
    *reinterpret_cast<float4*>(&skw[row][4 * part]) = make_float4(y[0], y[1], y[2], y[3]);
    __syncthreads();
    float ok[HD / 8], ow[HD / 8];
#pragma unroll
    for (int c = 0; c < HD / 8; ++c) { ok[c] = sk[row][(c >> 2) * 32 + part * 4 + (c & 3)]; ow[c] = 0.f; }
#pragma unroll 4
    for (int m = 0; m < kBlk; ++m) {
        const float cy = skw[row][m], ct = sc[m][row];
#pragma unroll
        for (int c = 0; c < HD / 32; ++c) {
            const float4 wm = *reinterpret_cast<const float4*>(&sw[m][c * 32 + part * 4]);
            const float t[4] = {wm.x, wm.y, wm.z, wm.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                ok[4 * c + x] = fmaf(-cy, t[x], ok[4 * c + x]);
                ow[4 * c + x] = fmaf(ct, t[x], ow[4 * c + x]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < HD / 32; ++c) {
        const float4 a = make_float4(ok[4 * c], ok[4 * c + 1], ok[4 * c + 2], ok[4 * c + 3]);
        const float4 b = make_float4(ow[4 * c], ow[4 * c + 1], ow[4 * c + 2], ow[4 * c + 3]);
        *reinterpret_cast<float4*>(kr + dst * HD + c * 32 + part * 4) = a;
        *reinterpret_cast<float4*>(wt + dst * HD + c * 32 + part * 4) = b;
        look(a);
        look(b);
    }
    const int any = __syncthreads_or(!(zero == 0.f));
    if (tid == 0) odd[(size_t)s * nblk + blk] = any;
}

// ---------------------------------------------------------------------------------------------- queries
__device__ __forceinline__ void cp16(float* dst, const float* src, bool live) {   // 16 bytes, zeros where not live
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(live ? 16 : 0) : "memory");
}

template <int HD, int RW>
__global__ void __launch_bounds__(32 * kWarps) fp32_fwd_kernel(const float* __restrict__ q, const float* __restrict__ k,
                                                               const float* __restrict__ v, const float* __restrict__ w,
                                                               const float* __restrict__ beta, const float* __restrict__ kr,
                                                               const float* __restrict__ wt, const float* __restrict__ ym,
                                                               const int* __restrict__ odd, const float* __restrict__ G,
                                                               float* __restrict__ o, float* __restrict__ lse, int S, int L,
                                                               int ldG, float scale) {
    grid_wait();
    grid_launch();
    constexpr int LD = ld<HD>(), E = HD / 32, TILE = kBlk * LD, GROUPS = kBlk / (kWarps * RW);
    extern __shared__ __align__(16) float sm[];      // [2 stages][W, Kr, Wt, V][32][LD], then per warp u [RW][HD], t and p [RW][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nblk = (L + kBlk - 1) / kBlk;
    // long rows first, the slices of one row group side by side
    const int s = blockIdx.x % S, grp = nblk * GROUPS - 1 - blockIdx.x / S;
    const int nb = grp / GROUPS, r0 = (grp % GROUPS) * kWarps * RW + warp * RW;   // own block, first row of the warp in it
    float* su = sm + 8 * TILE + warp * RW * (HD + 2 * kBlk);
    float* st = su + RW * HD;
    float* sp = st + RW * kBlk;
    auto request = [&](int n, int stage) {   // the four tiles of key block n; the own block takes K itself
        float* d = sm + stage * 4 * TILE;
        const size_t in = ((size_t)s * L + n * kBlk) * HD, pre = ((size_t)s * nblk + n) * kBlk * HD;
        const float* ksrc = n == nb ? k + in : kr + pre;
        for (int c = threadIdx.x; c < kBlk * HD / 4; c += 32 * kWarps) {
            const int row = c / (HD / 4), e = (c % (HD / 4)) * 4;
            const bool live = n * kBlk + row < L;
            const size_t at = (size_t)row * HD + e, in_at = live ? at : 0;
            float* t = d + row * LD + e;
            cp16(t, w + in + in_at, live);
            cp16(t + TILE, ksrc + (n == nb ? in_at : at), n == nb ? live : true);
            cp16(t + 2 * TILE, wt + pre + at, true);
            cp16(t + 3 * TILE, v + in + in_at, live);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    request(nb, 0);
    const int* odds = odd + (size_t)s * nblk;
    float acc[RW][E], m[RW], l[RW], Gi[RW];
    int i[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        i[r] = nb * kBlk + r0 + r;
        m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            acc[r][e] = 0.f;
            su[r * HD + e * 32 + lane] = i[r] < L ? q[((size_t)s * L + i[r]) * HD + e * 32 + lane] : 0.f;
        }
        Gi[r] = G && i[r] < L ? G[(size_t)s * ldG + i[r]] : 0.f;
    }
    __syncwarp();
    // Query r over block n, one key after the other, as fp32_walk_kernel does it (the lanes over the head dimension).
    auto walk = [&](const int r_, const int n) {
        const int last = min(n == nb ? nb * kBlk + r0 + r_ : n * kBlk + kBlk - 1, L - 1);
        float* u = su + r_ * HD;
#pragma unroll 1
        for (int j = last; j >= n * kBlk; --j) {
            const size_t at = ((size_t)s * L + j) * HD + lane;
            float a = 0.f, t = 0.f, ww[E], vv[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                ww[e] = w[at + e * 32];
                vv[e] = v[at + e * 32];
                a = fmaf(u[e * 32 + lane], k[at + e * 32], a);
                t = fmaf(u[e * 32 + lane], ww[e], t);
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, off);
                t += __shfl_xor_sync(0xffffffffu, t, off);
            }
            const float bt = beta[(size_t)s * L + j] * t, Gj = G ? G[(size_t)s * ldG + j] : 0.f;
#pragma unroll
            for (int r = 0; r < RW; ++r)
                if (r == r_) {   // (registers: the index has to be a constant)
                    const float sc = fmaf(scale, a, Gi[r] - Gj);
                    if (sc > m[r]) {
                        const float c = expf(m[r] - sc);
                        l[r] *= c;
#pragma unroll
                        for (int e = 0; e < E; ++e) acc[r][e] *= c;
                        m[r] = sc;
                    }
                    const float pj = expf(sc - m[r]);
                    if (lane == 0) l[r] += pj;
#pragma unroll
                    for (int e = 0; e < E; ++e) acc[r][e] = fmaf(pj, vv[e], acc[r][e]);
                }
#pragma unroll
            for (int e = 0; e < E; ++e) u[e * 32 + lane] = fmaf(-bt, ww[e], u[e * 32 + lane]);
        }
        __syncwarp();
    };
#pragma unroll 1
    for (int n = nb; n >= 0; --n) {
        const int stage = (nb - n) & 1;
        const bool own = n == nb;
        if (n > 0) {
            request(n - 1, stage ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        const int key = n * kBlk + lane;
        const float Gj = G && key < L ? G[(size_t)s * ldG + key] : 0.f;
        const int walked = odds[n];
        __syncthreads();
        if (walked) {   // (the whole CTA)
#pragma unroll 1
            for (int r = 0; r < RW; ++r) walk(r, n);
            __syncthreads();
            continue;
        }
        const float* tw = sm + stage * 4 * TILE + lane * LD;
        float t[RW][4], a[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int x = 0; x < 4; ++x) t[r][x] = a[r][x] = 0.f;
#pragma unroll 8
        for (int e = 0; e < HD; e += 4) {
            const float4 w4 = *reinterpret_cast<const float4*>(tw + e), k4 = *reinterpret_cast<const float4*>(tw + TILE + e);
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const float4 u4 = *reinterpret_cast<const float4*>(su + r * HD + e);
                t[r][0] = fmaf(w4.x, u4.x, t[r][0]); t[r][1] = fmaf(w4.y, u4.y, t[r][1]);
                t[r][2] = fmaf(w4.z, u4.z, t[r][2]); t[r][3] = fmaf(w4.w, u4.w, t[r][3]);
                a[r][0] = fmaf(k4.x, u4.x, a[r][0]); a[r][1] = fmaf(k4.y, u4.y, a[r][1]);
                a[r][2] = fmaf(k4.z, u4.z, a[r][2]); a[r][3] = fmaf(k4.w, u4.w, a[r][3]);
            }
        }
        float lg[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const float tt = (t[r][0] + t[r][1]) + (t[r][2] + t[r][3]);
            st[r * kBlk + lane] = own && lane > r0 + r ? 0.f : tt;
            lg[r] = (a[r][0] + a[r][1]) + (a[r][2] + a[r][3]);
        }
        __syncwarp();
        if (own) {   // logits of the own block: K q - Y t
            const float4* yr = reinterpret_cast<const float4*>(ym + (((size_t)s * nblk + n) * kBlk + lane) * kBlk);
#pragma unroll
            for (int c = 0; c < kBlk / 4; ++c) {
                const float4 y4 = yr[c];
#pragma unroll
                for (int r = 0; r < RW; ++r) lg[r] -= dot4(y4, *reinterpret_cast<const float4*>(st + r * kBlk + 4 * c));
            }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            float sc = fmaf(scale, lg[r], Gi[r] - Gj);
            if (own && lane > r0 + r) sc = -INFINITY;
            float mx = sc;
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float mn = fmaxf(m[r], mx), c = expf(m[r] - mn), pj = expf(sc - mn);
            m[r] = mn;
            l[r] = fmaf(l[r], c, pj);            // this lane's keys only: added up at the end
            sp[r * kBlk + lane] = pj;
#pragma unroll
            for (int e = 0; e < E; ++e) acc[r][e] *= c;
        }
        __syncwarp();
        // the lanes turn to the head dimension: u -= Wt^T t, acc += V^T p
        float du[RW][E];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int e = 0; e < E; ++e) du[r][e] = 0.f;
        const float* cw = sm + stage * 4 * TILE + 2 * TILE + lane;
#pragma unroll 4
        for (int j = 0; j < kBlk; j += 4) {
            float4 t4[RW], p4[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                t4[r] = *reinterpret_cast<const float4*>(st + r * kBlk + j);
                p4[r] = *reinterpret_cast<const float4*>(sp + r * kBlk + j);
            }
#pragma unroll
            for (int y = 0; y < 4; ++y)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const float ww = cw[(j + y) * LD + e * 32], vv = cw[TILE + (j + y) * LD + e * 32];
#pragma unroll
                    for (int r = 0; r < RW; ++r) {
                        const float tj = y == 0 ? t4[r].x : y == 1 ? t4[r].y : y == 2 ? t4[r].z : t4[r].w;
                        const float pj = y == 0 ? p4[r].x : y == 1 ? p4[r].y : y == 2 ? p4[r].z : p4[r].w;
                        du[r][e] = fmaf(tj, ww, du[r][e]);
                        acc[r][e] = fmaf(pj, vv, acc[r][e]);
                    }
                }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int e = 0; e < E; ++e) su[r * HD + e * 32 + lane] -= du[r][e];
        __syncthreads();   // everyone is done with this stage's tiles
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], off);
        if (i[r] >= L) continue;
        const float inv = 1.f / l[r];
#pragma unroll
        for (int e = 0; e < E; ++e) o[((size_t)s * L + i[r]) * HD + e * 32 + lane] = acc[r][e] * inv;
        if (lane == 0) lse[(size_t)s * L + i[r]] = m[r] + logf(l[r]);
    }
}

// ---------------------------------------------------------------------------------------------- without the per-block tiles
// The definition as it stands, one key at a time, for callers whose scratch does not hold the tiles (path_attn_fwd_static with
// more than 16 MiB of them): a warp per query, the head dimension spread over the lanes, the two dot products of a step
// reduced together by one butterfly.  About 520 cycles per key.
constexpr int kRowsPerCta = 8;

template <int HD>
__global__ void __launch_bounds__(32 * kRowsPerCta) fp32_walk_kernel(const float* __restrict__ q, const float* __restrict__ k,
                                                                   const float* __restrict__ v, const float* __restrict__ w,
                                                                   const float* __restrict__ beta, const float* __restrict__ G,
                                                                   float* __restrict__ o, float* __restrict__ lse, int S, int L,
                                                                   int ldG, float scale) {
    grid_wait();
    grid_launch();
    constexpr int E = HD / 32;   // elements per lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nblk = (L + kRowsPerCta - 1) / kRowsPerCta;
    // long rows first, the slices of one row block side by side
    const int slice = blockIdx.x % S, blk = nblk - 1 - blockIdx.x / S;
    const int i = blk * kRowsPerCta + warp;
    if (i >= L) return;
    const size_t base = (size_t)slice * L;
    auto load = [&](const float* p, int pos, float (&x)[E]) {
        const float* r = p + (base + pos) * HD + lane * E;
        if (E == 2) {
            const float2 t = *reinterpret_cast<const float2*>(r);
            x[0] = t.x; x[1] = t.y;
        } else {
            const float4 t = *reinterpret_cast<const float4*>(r);
            x[0] = t.x; x[1] = t.y; x[E - 2] = t.z; x[E - 1] = t.w;
        }
    };
    float u[E], acc[E], kj[E], wj[E], vj[E];
    load(q, i, u);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    const float Gi = G ? G[(size_t)slice * ldG + i] : 0.f;
    float m = -INFINITY, l = 0.f;
    load(k, i, kj); load(w, i, wj); load(v, i, vj);
    float bj = beta[base + i], Gj = Gi;
    for (int j = i; j >= 0; --j) {
        // the next key's row is requested before this step's reductions
        float kn[E], wn[E], vn[E], bn = 0.f, Gn = 0.f;
        if (j > 0) {
            load(k, j - 1, kn); load(w, j - 1, wn); load(v, j - 1, vn);
            bn = beta[base + j - 1];
            Gn = G ? G[(size_t)slice * ldG + j - 1] : 0.f;
        }
        float a = 0.f, t = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            a = fmaf(u[e], kj[e], a);
            t = fmaf(u[e], wj[e], t);
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, off);
            t += __shfl_xor_sync(0xffffffffu, t, off);
        }
        const float s = fmaf(scale, a, Gi - Gj);
        if (s > m) {   // warp-uniform: every lane holds the same s
            const float c = expf(m - s);
            l *= c;
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] *= c;
            m = s;
        }
        const float pj = expf(s - m);
        l += pj;
        const float bt = bj * t;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            acc[e] = fmaf(pj, vj[e], acc[e]);
            u[e] = fmaf(-bt, wj[e], u[e]);
        }
        if (j > 0) {
#pragma unroll
            for (int e = 0; e < E; ++e) { kj[e] = kn[e]; wj[e] = wn[e]; vj[e] = vn[e]; }
            bj = bn; Gj = Gn;
        }
    }
    const float inv = 1.f / l;
    float* orow = o + (base + i) * HD + lane * E;
    if (E == 2) {
        *reinterpret_cast<float2*>(orow) = make_float2(acc[0] * inv, acc[1] * inv);
    } else {
        *reinterpret_cast<float4*>(orow) = make_float4(acc[0] * inv, acc[1] * inv, acc[E - 2] * inv, acc[E - 1] * inv);
    }
    if (lane == 0) lse[base + i] = m + logf(l);
}

template <int HD, int RW>
cudaError_t launch_rows(const float* q, const float* k, const float* v, const float* w, const float* beta, const float* kr, const float* wt,
                        const float* ym, const int* odd, const float* G, float* o, float* lse, int S, int L, int ldG, float scale,
                        cudaStream_t st) {
    const int smem = (8 * kBlk * ld<HD>() + kWarps * RW * (HD + 2 * kBlk)) * 4;
    const int nblk = (L + kBlk - 1) / kBlk;
    return launch<fp32_fwd_kernel<HD, RW>>((unsigned)((size_t)S * nblk * (kBlk / (kWarps * RW))), 32 * kWarps, smem, st, q, k, v, w, beta,
                                           kr, wt, ym, odd, G, o, lse, S, L, ldG, scale);
}

template <int HD>
cudaError_t launch_hd(const float* q, const float* k, const float* v, const float* w, const float* beta, const float* G, float* o,
                      float* lse, int S, int L, int ldG, float scale, float* scratch, uint32_t* clear, cudaStream_t st) {
    const size_t nblk = (L + kBlk - 1) / kBlk, rows = (size_t)S * nblk * kBlk;
    float* kr = scratch;
    float* wt = kr + rows * HD;
    float* ym = wt + rows * HD;
    int* odd = reinterpret_cast<int*>(ym + rows * kBlk);
    for (int s0 = 0; s0 < S; s0 += 65535) {   // (a grid's second dimension ends there)
        const int ns = S - s0 < 65535 ? S - s0 : 65535;
        const size_t in = (size_t)s0 * L, out = (size_t)s0 * nblk * kBlk;
        const cudaError_t e = launch<fp32_block_kernel<HD>>(dim3((unsigned)nblk, ns), 256, 0, st, k + in * HD, w + in * HD, beta + in, v + in * HD,
                                                            kr + out * HD, wt + out * HD, ym + out * kBlk, odd + (size_t)s0 * nblk, s0 == 0 ? clear : nullptr, L);
        if (e != cudaSuccess) return e;
    }
    // One query per warp for few rows, four that share a warp's tile reads otherwise.  us with one / with four (slices x positions x
    // d): 2 x 256 x 64 20 / 25, 4 x 448 x 64 49 / 42, 4 x 592 x 64 62 / 63, 8 x 512 x 64 78 / 62; 2 x 256 x 128 32 / 53,
    // 4 x 448 x 128 88 / 89, 4 x 592 x 128 134 / 121, 8 x 512 x 128 184 / 106.  The line lies at four rows per warp of every SM.
    if (rows <= 148 * 4 * 4) return launch_rows<HD, 1>(q, k, v, w, beta, kr, wt, ym, odd, G, o, lse, S, L, ldG, scale, st);
    return launch_rows<HD, 4>(q, k, v, w, beta, kr, wt, ym, odd, G, o, lse, S, L, ldG, scale, st);
}

}  // namespace

size_t fp32_scratch_bytes(int S, int L, int hd) {
    const size_t rows = (size_t)S * ((L + kBlk - 1) / kBlk) * kBlk;
    return (rows * (2 * hd + kBlk) + rows / kBlk) * sizeof(float);
}

cudaError_t launch_fp32_fwd(const float* q, const float* k, const float* v, const float* w, const float* beta, const float* G,
                            float* o, float* lse, int S, int L, int ldG, int hd, float scale, float* scratch, uint32_t* clear, cudaStream_t st) {
    if (!scratch) {
        const dim3 grid((unsigned)((size_t)S * ((L + kRowsPerCta - 1) / kRowsPerCta)));
        const cudaError_t e = cudaMemsetAsync(clear, 0, 256, st);
        if (e != cudaSuccess) return e;
        return hd == 64 ? launch<fp32_walk_kernel<64>>(grid, 32 * kRowsPerCta, 0, st, q, k, v, w, beta, G, o, lse, S, L, ldG, scale)
                        : launch<fp32_walk_kernel<128>>(grid, 32 * kRowsPerCta, 0, st, q, k, v, w, beta, G, o, lse, S, L, ldG, scale);
    }
    return hd == 64 ? launch_hd<64>(q, k, v, w, beta, G, o, lse, S, L, ldG, scale, scratch, clear, st)
                    : launch_hd<128>(q, k, v, w, beta, G, o, lse, S, L, ldG, scale, scratch, clear, st);
}

}  // namespace path
