// Memory-bound helpers: prefix sum of the log gate (PaTH-FoX, paper Sec. 2.2) and suffix sum of its gradient, block skipping,
// decoding cache and segment buffers (copies, gate terms, padding), the forward-state record, clearing.
#include "linear.cuh"
#include "tc5.cuh"

namespace path {

namespace {

// Slices in a grid's second dimension, which ends at 65535: the kernels below walk on from there.
constexpr int kMaxGridY = 65535;

__global__ void pad_rows_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, int S, int L, int Lp, int rowbytes16) {
    grid_wait();
    grid_launch();
    // one 16-byte vector per thread and slice; grid.x covers Lp * rowbytes16
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long total = (long)Lp * rowbytes16;
    if (i >= total) return;
    const long row = i / rowbytes16, col = i % rowbytes16;
    for (int s = blockIdx.y; s < S; s += gridDim.y)
        dst[((long)s * Lp + row) * rowbytes16 + col] = row < L ? src[((long)s * L + row) * rowbytes16 + col] : make_uint4(0, 0, 0, 0);
}

// Sum of `x` over the threads before this one in a CTA of 1024; `total` = the sum over all of them.  Nothing is added and taken
// off again: the sums in front of a huge or infinite value (a gate that resets) must not feel it.
__device__ __forceinline__ float block_scan(float x, float* part, float& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    float w = part[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += y;
    }
    total = __shfl_sync(0xffffffffu, w, 31);
    const float warps = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0), lanes = __shfl_up_sync(0xffffffffu, x, 1);
    __syncthreads();   // (`part` is written again by the next call)
    return (warp > 0 ? warps : 0.f) + (lane > 0 ? lanes : 0.f);
}

// One CTA (1024 threads) per slice, 4096 positions at a time, four neighbouring ones per thread.  Latency-bound (32 KB per
// slice).  One contiguous segment per thread with a shared-memory scan of 20 barriers took 32 us at 32 slices x 8192 positions;
// the warp scans of this file together take 47 us off the training step of that shape and 27 us off one of 16 x 3001 x 64.
__global__ void __launch_bounds__(1024) gate_prefix_kernel(const float* __restrict__ g, float* __restrict__ G, int L,
                                                           int Lp, uint32_t* clear) {
    grid_wait();
    grid_launch();
    if (clear && blockIdx.x == 0 && threadIdx.x < 64) clear[threadIdx.x] = 0u;   // the workspace's status block (256 bytes)
    __shared__ float part[32];
    const float* gs = g + (size_t)blockIdx.x * L;
    float* Gs = G + (size_t)blockIdx.x * Lp;
    float carry = 0.f;
    for (int base = 0; base < Lp; base += 4096) {
        const int i0 = base + threadIdx.x * 4;
        float v[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) v[x] = i0 + x < L ? gs[i0 + x] : 0.f;
        v[1] += v[0]; v[2] += v[1]; v[3] += v[2];
        float total;
        const float before = carry + block_scan(v[3], part, total);
        if (i0 < Lp) *reinterpret_cast<float4*>(Gs + i0) = make_float4(before + v[0], before + v[1], before + v[2], before + v[3]);
        carry += total;
    }
}

// out[s][i] = sum over positions t >= i of dG + dGrow + the four partial row sums of the diagonal chunks' dS ([chunk][4][128]).
// One CTA per slice, from the end, 4096 positions at a time (see gate_prefix_kernel).
__global__ void __launch_bounds__(1024) gate_suffix_kernel(const float* __restrict__ dGa, const float* __restrict__ dGb,
                                                           const float* __restrict__ diag, float* __restrict__ out, int L, int Lp) {
    grid_wait();
    grid_launch();
    __shared__ float part[32];
    const size_t so = (size_t)blockIdx.x * Lp;
    float* os = out + (size_t)blockIdx.x * L;
    float carry = 0.f;
    for (int top = Lp; top > 0; top -= 4096) {
        const int i0 = top - 4 - (int)threadIdx.x * 4;   // this thread: positions i0 + 3, i0 + 2, i0 + 1, i0
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (i0 >= 0) {
            const float4 a = *reinterpret_cast<const float4*>(dGa + so + i0), b = *reinterpret_cast<const float4*>(dGb + so + i0);
            v[0] = a.w + b.w; v[1] = a.z + b.z; v[2] = a.y + b.y; v[3] = a.x + b.x;
            const float* d = diag + (so + (i0 & ~(CHUNK - 1))) * 4 + (i0 & (CHUNK - 1));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 c = *reinterpret_cast<const float4*>(d + q * CHUNK);
                v[0] += c.w; v[1] += c.z; v[2] += c.y; v[3] += c.x;
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (i0 + 3 - x >= L) v[x] = 0.f;   // the padded tail
        }
        v[1] += v[0]; v[2] += v[1]; v[3] += v[2];
        float total;
        const float before = carry + block_scan(v[3], part, total);
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (i0 >= 0 && i0 + 3 - x < L) os[i0 + 3 - x] = before + v[x];
        carry += total;
    }
}

// ---- block skipping for gated problems (the paper notes that PaTH-FoX keeps FoX's pruning of negligible blocks)
//
// |k_j^T (H_{j+1} ... H_i) q_i| <= |k_j| |q_i| prod_s max(1, |1 - beta_s |w_s|^2|)   (each factor bounds the 2-norm of H_s;
// it is 1 whenever 0 <= beta_s |w_s|^2 <= 2), and every row's largest logit is at least its own diagonal one,
// s_ii = scale q_i . k_i.  So if for a pair of chunks (I, J)
//     |scale| max_I|q| max_J|k| exp(sum of the log factors over chunks J..I) + max_I G - min_J G  <  min_I s_ii - kSkipMargin
// every probability of the pair is below exp(-kSkipMargin) of its row's normaliser and the pair can be left out.  A
// query chunk keeps the key chunks up to the farthest one that fails this test.
constexpr float kSkipMargin = 30.f;   // exp(-30) ~ 1e-13 per logit, far below bf16 resolution even summed over a long row

// stats[tile] = {max|q|, max|k|, max G, min G, min s_ii over real rows, sum of log factors, 0, 0}; tile_ranges_kernel leaves the
// distance of the slice's farthest kept pair, in chunks, in entry 6 of its first tile
// A row takes hd/8 lanes (16-byte loads), so a warp works on 2 (hd = 128) or 4 (hd = 64) rows at a time.
// Bound by its bytes, q, k and w once.  LPR lanes share a row, eight channels each.  The row's four sums are reduced together: at the
// first two steps a lane gives away half of what it holds, so that it ends up with one of them (role 0: |q|^2, 1: |k|^2, 2: q k,
// 3: |w|^2) in 5 shuffles instead of 16, and keeps that one's running maximum or sum.  2 x 16 x 8192 x 128: 49 -> 40 us.
template <int HD>
__global__ void __launch_bounds__(256) tile_stats_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                                                        const __nv_bfloat16* __restrict__ w, const float* __restrict__ beta,
                                                        const float* __restrict__ G, float* __restrict__ stats, int L, int Lp,
                                                        float scale) {
    grid_wait();
    grid_launch();
    __shared__ float red[8][6];
    constexpr int LPR = HD / 8, ROWS = 32 / LPR;   // lanes per row, rows per warp and instruction
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / LPR, li = lane % LPR;
    const bool up1 = li & (LPR / 2), up2 = li & (LPR / 4);
    const int role = 2 * (int)up1 + (int)up2;
    const int N = Lp / CHUNK, sl = blockIdx.x / N, c = blockIdx.x % N;
    // roles 0 - 2: maximum of factor * sum (the least q k as the greatest of its negative); role 3: the sum of the growth
    const float factor = role == 2 ? -scale : 1.f;
    float top = role == 2 ? -INFINITY : 0.f, gmax = -INFINITY, gmin = INFINITY, gam = 0.f;
    auto dot8 = [](const uint4& a, const uint4& b) {
        const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc = fmaf(__uint_as_float(x[i] << 16), __uint_as_float(y[i] << 16), acc);
            acc = fmaf(__uint_as_float(x[i] & 0xffff0000u), __uint_as_float(y[i] & 0xffff0000u), acc);
        }
        return acc;
    };
    constexpr int U = 4;   // rows per lane group in flight (CHUNK / (8 * ROWS) is 4 or 8)
    for (int r0 = warp * ROWS + grp; r0 < CHUNK; r0 += 8 * ROWS * U) {
        uint4 a[U], b[U], x[U];
        float g[U], bt[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = c * CHUNK + r0 + u * 8 * ROWS;
            const size_t row = (size_t)sl * L + t;
            a[u] = b[u] = x[u] = make_uint4(0u, 0u, 0u, 0u);
            bt[u] = 0.f;
            if (t < L) {
                a[u] = *reinterpret_cast<const uint4*>(q + row * HD + li * 8);
                b[u] = *reinterpret_cast<const uint4*>(k + row * HD + li * 8);
                x[u] = *reinterpret_cast<const uint4*>(w + row * HD + li * 8);
                bt[u] = beta[row];
            }
            g[u] = G[(size_t)sl * Lp + t];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float qq = dot8(a[u], a[u]), kk = dot8(b[u], b[u]), qk = dot8(a[u], b[u]), ww = dot8(x[u], x[u]);
            float s0 = up1 ? qk : qq, s1 = up1 ? ww : kk;
            s0 += __shfl_xor_sync(0xffffffffu, up1 ? qq : qk, LPR / 2);
            s1 += __shfl_xor_sync(0xffffffffu, up1 ? kk : ww, LPR / 2);
            float s = up2 ? s1 : s0;
            s += __shfl_xor_sync(0xffffffffu, up2 ? s0 : s1, LPR / 4);
#pragma unroll
            for (int off = LPR / 8; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (role != 2 || c * CHUNK + r0 + u * 8 * ROWS < L) top = fmaxf(top, factor * s);
            gam += logf(fmaxf(1.f, fabsf(1.f - bt[u] * s)));   // (counts for role 3)
            gmax = fmaxf(gmax, g[u]); gmin = fminf(gmin, g[u]);
        }
    }
    // combine the groups of the warp
    for (int off = LPR; off < 32; off <<= 1) {
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
        gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, off)); gmin = fminf(gmin, __shfl_xor_sync(0xffffffffu, gmin, off));
        gam += __shfl_xor_sync(0xffffffffu, gam, off);
    }
    if (lane < LPR && li % (LPR / 4) == 0) {
        if (role == 0) {
            red[warp][0] = sqrtf(top); red[warp][2] = gmax; red[warp][3] = gmin;
        } else if (role == 1) {
            red[warp][1] = sqrtf(top);
        } else if (role == 2) {
            red[warp][4] = -top;
        } else {
            red[warp][5] = gam;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float qn = red[0][0], kn = red[0][1], mlo = red[0][4];
        gmax = red[0][2]; gmin = red[0][3]; gam = red[0][5];
        for (int x = 1; x < 8; ++x) {
            qn = fmaxf(qn, red[x][0]); kn = fmaxf(kn, red[x][1]); gmax = fmaxf(gmax, red[x][2]); gmin = fminf(gmin, red[x][3]);
            mlo = fminf(mlo, red[x][4]); gam += red[x][5];
        }
        float* o = stats + (size_t)blockIdx.x * 8;
        // the norms and the growth go up, the row maximum goes down by a rounding margin: the test must err towards keeping
        o[0] = qn * 1.001f; o[1] = kn * 1.001f; o[2] = gmax; o[3] = gmin;
        o[4] = mlo - 1e-3f * fabsf(mlo); o[5] = gam * 1.001f + 1e-6f;
        o[6] = o[7] = 0.f;
    }
}

// One CTA per slice.  First, a warp per query chunk I finds the farthest key chunk that fails the test (lanes over the key
// chunks, the growth summed up by a warp scan).  Then the kept ranges are made a staircase: the first kept key chunk of a query
// chunk never lies after that of a later query chunk (ranges only grow, which is always safe).  Then "key chunk J is kept by
// query chunk I" holds for exactly the I in J .. far(J), so the key-major sweep of the backward (nvisit[J] = far(J) - J + 1 query
// chunks) computes the same pairs as the query-major sweeps, and every version a sweep asks for lies within the levels its
// chunk reaches.  Also counts the kept pairs.  (Two kernels with one serial thread per query chunk and per slice took
// 30 us at 32 slices x 64 chunks.)
__global__ void __launch_bounds__(1024) tile_ranges_kernel(float* stats, int* __restrict__ nkeep,
                                                           int* __restrict__ nvisit, unsigned long long* counters, int N,
                                                           float ascale) {
    grid_wait();
    grid_launch();
    // the ranges sit in shared memory when they fit (N <= kMax chunks, i.e. sequences up to a million tokens)
    constexpr int kMax = 8192;
    __shared__ int snk[kMax];
    const int sl = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* st = stats + (size_t)sl * N * 8;
    int* gk = nkeep + (size_t)sl * N;
    int* gv = nvisit + (size_t)sl * N;
    int* nk = N <= kMax ? snk : gk;
    for (int I = warp; I < N; I += 32) {
        const float* me = st + (size_t)I * 8;
        const float qn = me[0], gmax = me[2], need = me[4] - kSkipMargin;
        float grown = 0.f;
        int keep = 1;
        for (int n0 = 0; n0 <= I; n0 += 32) {
            const int n = n0 + lane;
            const bool in = n <= I;
            const float* o = st + (size_t)(in ? I - n : 0) * 8;
            float acc = in ? o[5] : 0.f;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, acc, off);
                if (lane >= off) acc += y;
            }
            const float bound = ascale * qn * o[1] * expf(grown + acc) + gmax - o[3];
            const unsigned kept = __ballot_sync(0xffffffffu, in && !(bound < need));   // a NaN or an infinity keeps as well
            if (kept) keep = n0 + 32 - __clz((int)kept);
            grown += __shfl_sync(0xffffffffu, acc, 31);
        }
        if (lane == 0) nk[I] = keep;
    }
    __syncthreads();
    if (warp == 0) {   // from the last chunk down: start(I) = min over I' >= I of the first kept chunk
        unsigned long long kept = 0;
        int start = N, far = 0;
        for (int top = N; top > 0; top -= 32) {
            const int I = top - 1 - lane;
            int first = I >= 0 ? I - nk[I] + 1 : N;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, first, off);
                if (lane >= off) first = min(first, y);
            }
            first = min(first, start);
            if (I >= 0) {
                nk[I] = I - first + 1;
                far = max(far, I - first);
                kept += (unsigned long long)nk[I];
            }
            start = __shfl_sync(0xffffffffu, first, 31);
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            kept += __shfl_xor_sync(0xffffffffu, kept, off);
            far = max(far, __shfl_xor_sync(0xffffffffu, far, off));
        }
        if (lane == 0) {
            stats[(size_t)sl * N * 8 + 6] = (float)far;
            atomicAdd(&counters[0], kept);
            atomicAdd(&counters[1], (unsigned long long)N * (N + 1) / 2);
        }
    }
    __syncthreads();
    // far(J) = the last I whose first kept key chunk I - nk[I] + 1 is <= J; those first chunks do not decrease with I, so a
    // binary search per J finds it
    for (int J = threadIdx.x; J < N; J += blockDim.x) {
        int lo = J, hi = N - 1;   // invariant: chunk lo keeps J (a chunk always keeps itself)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (mid - nk[mid] + 1 <= J) lo = mid; else hi = mid - 1;
        }
        gv[J] = lo - J + 1;
        if (nk != gk) gk[J] = nk[J];
    }
}

// Values and gate prefix of a prompt into the decoding cache: vc[S][cap][d] <- v[S][L][d], gc[S][cap] <- G[S][Lp] (L rows of every
// slice).  grid = (blocks of 1024 16-byte vectors, slices), four vectors per thread in flight: 99 us for 32 x 32768 x 128 (5.4 TB/s),
// where cudaMemcpy2DAsync took 273.
__global__ void __launch_bounds__(256) cache_rows_kernel(const uint4* __restrict__ v, uint4* __restrict__ vc, const float* __restrict__ G,
                                                         float* __restrict__ gc, long n16, long cap16, int L, int Lp, int cap, int S) {
    grid_wait();
    grid_launch();
    for (int s = blockIdx.y; s < S; s += gridDim.y) {
        const long i0 = (long)blockIdx.x * 1024 + threadIdx.x;
        uint4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * 256 < n16) x[u] = __ldcs(v + (size_t)s * n16 + i0 + u * 256);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * 256 < n16) __stcs(vc + (size_t)s * cap16 + i0 + u * 256, x[u]);
        if (gc)
            for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < L; i += (long)gridDim.x * 256) gc[(size_t)s * cap + i] = G[(size_t)s * Lp + i];
    }
}

// ---- context-parallel path: gate terms of a segment, final result
__global__ void cp_gate_kernel(const float* __restrict__ G, float* __restrict__ gq, float* __restrict__ gk,
                               float* __restrict__ gtot, int S, int L, int Lp) {
    grid_wait();
    grid_launch();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    for (int s = blockIdx.y; s < S; s += gridDim.y) {
        const float tot = G ? G[(size_t)s * Lp + L - 1] : 0.f;
        if (i == 0) gtot[s] = tot;
        if (i >= Lp) continue;
        const float g = G ? G[(size_t)s * Lp + i] : 0.f;
        gq[(size_t)s * Lp + i] = i < L ? g : 0.f;
        gk[(size_t)s * Lp + i] = i < L ? g - tot : 1e30f;
    }
}
// one thread per 4 outputs of a row
__global__ void cp_finish_kernel(const float* __restrict__ o_acc, const float* __restrict__ lse_acc, __nv_bfloat16* __restrict__ o,
                                 float* __restrict__ lse, size_t rows, int hd4) {
    grid_wait();
    grid_launch();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * hd4) return;
    const float4 a = reinterpret_cast<const float4*>(o_acc)[i];
    __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
    reinterpret_cast<uint2*>(o)[i] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
    if (i % hd4 == 0) lse[i / hd4] = lse_acc[i / hd4];
}

// ---- forward-state record and the wait self-test
__global__ void state_write_kernel(StateRecord* dst, const StateRecord rec) {
    grid_wait();
    grid_launch();
    if (threadIdx.x == 0) *dst = rec;
}
__global__ void state_check_kernel(const StateRecord* have, const StateRecord want, uint32_t* status) {
    grid_wait();
    grid_launch();
    if (threadIdx.x < 8) status[threadIdx.x] = 0u;   // the status word and the sweeps' item counters; the rest is the forward's
    __syncwarp();
    if (threadIdx.x != 0) return;
    const StateRecord h = *have;
    const bool same = h.magic == want.magic && h.q == want.q && h.k == want.k && h.v == want.v && h.w == want.w &&
                      h.beta == want.beta && h.log_f == want.log_f && h.B == want.B && h.H == want.H && h.L == want.L &&
                      h.d == want.d && h.gate == want.gate && (!want.gate || h.scale == want.scale);
    if (!same) atomicCAS(status, 0u, (uint32_t)ST_STATE);
}
// The same bounded wait every kernel of the library uses, on a barrier that never completes: after `ticks` cycles it
// gives up, raises the CTA's abort flag with its code, and the kernel forwards the flag to the status word and returns.
__global__ void selftest_wait_kernel(uint32_t* status, long long ticks) {
    __shared__ uint64_t bar;
    __shared__ uint32_t abort_word;
    volatile uint32_t* abort_flag = &abort_word;
    if (threadIdx.x == 0) {
        tc5::mbar_init(&bar, 1);
        *abort_flag = 0;
        tc5::mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok = tc5::mbar_try_wait(&bar, 0);
        if (!ok) ok = tc5::mbar_wait_slow(&bar, 0, abort_flag, ST_SELFTEST, ticks);
        if (!ok) tc5::report_abort(abort_flag, status);
    }
}

// Buffers that the next kernels add to, and the status block.  A kernel instead of one memset per buffer: it starts under the
// end of the kernel before and the next one under its own, where a memset waits for everything and takes 2 - 3 us of its own
// (the low-rank layer's backward had three: 44.8 -> 37.7 us for 8192 rows, 512 -> 64 -> 768; 59.0 -> 48.9 us for 1000 rows,
// 768 -> 128 -> 512).
__global__ void __launch_bounds__(256) clear_kernel(uint32_t* a, size_t na, uint32_t* b, size_t nb, uint32_t* c, size_t nc) {
    grid_wait();
    grid_launch();
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < na + nb + nc; i += (size_t)gridDim.x * 256) {
        if (i < na) a[i] = 0u;
        else if (i < na + nb) b[i - na] = 0u;
        else c[i - na - nb] = 0u;
    }
}

}  // namespace

cudaError_t launch_gate_suffix(const float* dGa, const float* dGb, const float* diag, float* out, int S, int L, int Lp,
                               cudaStream_t st) {
    return launch<gate_suffix_kernel>(S, 1024, 0, st, dGa, dGb, diag, out, L, Lp);
}

cudaError_t launch_clear(void* a, size_t na, void* b, size_t nb, void* c, size_t nc, cudaStream_t st) {
    const size_t blocks = (na + nb + nc + 1023) / 1024;   // (at most about eight per SM: the rest is the loop's)
    return launch<clear_kernel>((unsigned)(blocks < 1184 ? blocks : 1184), 256, 0, st, (uint32_t*)a, na, (uint32_t*)b, nb, (uint32_t*)c, nc);
}

cudaError_t launch_pad_rows(const void* src, void* dst, int S, int L, int Lp, int d, cudaStream_t st) {
    const int rowbytes16 = d * 2 / 16;
    const long total = (long)Lp * rowbytes16;
    const dim3 grid((unsigned)((total + 255) / 256), S < kMaxGridY ? S : kMaxGridY);
    return launch<pad_rows_kernel>(grid, 256, 0, st, (const uint4*)src, (uint4*)dst, S, L, Lp, rowbytes16);
}

cudaError_t launch_gate_prefix(const float* g, float* G, int S, int L, int Lp, uint32_t* clear, cudaStream_t st) {
    return launch<gate_prefix_kernel>(S, 1024, 0, st, g, G, L, Lp, clear);
}

cudaError_t launch_gate_skip(const void* q, const void* k, const void* w, const float* beta, const float* G, float* stats,
                             int* nkeep, int* nvisit, unsigned long long* counters, int S, int L, int Lp, int hd, float scale,
                             cudaStream_t st) {
    typedef __nv_bfloat16 bf;
    const int N = Lp / CHUNK;
    const cudaError_t e = hd == 64 ? launch<tile_stats_kernel<64>>(S * N, 256, 0, st, (const bf*)q, (const bf*)k, (const bf*)w, beta, G, stats, L, Lp, scale)
                                   : launch<tile_stats_kernel<128>>(S * N, 256, 0, st, (const bf*)q, (const bf*)k, (const bf*)w, beta, G, stats, L, Lp, scale);
    if (e != cudaSuccess) return e;
    return launch<tile_ranges_kernel>(S, 1024, 0, st, stats, nkeep, nvisit, counters, N, fabsf(scale));
}

cudaError_t launch_cache_rows(const void* v, void* vc, const float* G, float* gc, int S, int L, int Lp, int cap, int hd, cudaStream_t st) {
    const long n16 = (long)L * hd / 8, cap16 = (long)cap * hd / 8;
    const dim3 grid((unsigned)((n16 + 1023) / 1024), S < kMaxGridY ? S : kMaxGridY);
    return launch<cache_rows_kernel>(grid, 256, 0, st, (const uint4*)v, (uint4*)vc, G, gc, n16, cap16, L, Lp, cap, S);
}

cudaError_t launch_cp_gate(const float* G, float* gq, float* gk, float* gtot, int S, int L, int Lp, cudaStream_t st) {
    return launch<cp_gate_kernel>(dim3((Lp + 255) / 256, S < kMaxGridY ? S : kMaxGridY), 256, 0, st, G, gq, gk, gtot, S, L, Lp);
}
cudaError_t launch_cp_finish(const float* o_acc, const float* lse_acc, void* o, float* lse, size_t rows, int hd,
                             cudaStream_t st) {
    const size_t n = rows * (hd / 4);
    return launch<cp_finish_kernel>((unsigned)((n + 255) / 256), 256, 0, st, o_acc, lse_acc, (__nv_bfloat16*)o, lse, rows, hd / 4);
}

cudaError_t launch_state_write(void* record, const StateRecord& rec, cudaStream_t st) {
    return launch<state_write_kernel>(1, 32, 0, st, (StateRecord*)record, rec);
}
cudaError_t launch_state_check(const void* record, const StateRecord& want, uint32_t* status, cudaStream_t st) {
    return launch<state_check_kernel>(1, 32, 0, st, (const StateRecord*)record, want, status);
}
cudaError_t launch_selftest_wait(uint32_t* status, long long ticks, cudaStream_t st) {
    return (selftest_wait_kernel<<<1, 32, 0, st>>>(status, ticks), cudaGetLastError());
}

}  // namespace path
