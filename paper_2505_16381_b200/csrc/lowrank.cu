// The low-rank linear layer in front of the short convolution (paper Sec. 2.2, footnote to the definition of H_t: w_t
// comes from "a low-rank linear layer followed by a short convolution and L2 normalisation"):
//     t = x W1^T   [M, r],      z = t W2^T   [M, C]        (x [M, D];  W1 [r, D],  W2 [C, r]:  nn.Linear layouts)
// and its backward
//     dt = dz W2,   dW2 = dz^T t,   dx = dt W1,   dW1 = dt^T x.
// Two tcgen05 kernels.  z and dx (contraction over r, M x N output): wide_kernel below.  The other four, with their long
// contraction: gemm_kernel, C[M', N'] (+)= op(A) op(B) on 128 x 128 output tiles, operands fetched by TMA into a
// three-stage ring of 128-byte-swizzled tiles, one thread issuing the products into a tensor-memory accumulator, four
// warps writing the tile out.  Whether an operand enters as stored or transposed is a matter of its descriptor's
// major-ness, as everywhere in this library: a K-major operand is a [rows][K] matrix (box 128 rows x 64 k), an MN-major
// one a [K][rows] matrix (box 64 k x 64 rows, two per stage).  The weight gradients contract over the M tokens: their
// K range is split over CTAs and the partial tiles are added with float32 atomics (reproducible to rounding).
// These products have a short contraction or a narrow output: they are bound by the bytes of x, z and their
// gradients, not by the tensor pipe.
#include "tileops.cuh"

namespace path {
using namespace tc5;

namespace {

constexpr int kStages = 3;   // 3 x 32 KB: two CTAs per SM, so one writes its tile out while the other multiplies
constexpr uint32_t kStageBytes = 32768;   // A tile [128 x 64] + B tile [128 x 64], bf16
constexpr uint32_t kGemmSmem = kStages * kStageBytes + 256 + 1024;

// Descriptor low words of the k-th 16-wide step inside a 64-deep stage tile.
__device__ __forceinline__ uint32_t step_lo(uint32_t tile, int mn_major, int kk) {
    // K-major: [128 rows][64 k], 32 bytes per step.  MN-major: two panels [64 k][64 rows], 8192 bytes apart, 2048 bytes per step.
    return mn_major ? umma_desc_lo(tile + kk * 2048u, 8192u) : umma_desc_lo(tile + kk * 32u, 16u);
}

__global__ void __launch_bounds__(192, 2) gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                                                      const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint64_t* full = (uint64_t*)(smem + kStages * kStageBytes);
    uint64_t* empty = full + kStages;
    uint64_t* done = empty + kStages;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(done, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, 128);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * 128;
    // this CTA's share of the contraction, in stages of 64
    const int stages_total = (p.K + 63) / 64, per = (stages_total + (int)gridDim.z - 1) / (int)gridDim.z;
    const int s_lo = blockIdx.z * per, s_hi = min(stages_total, s_lo + per), ns = s_hi - s_lo;
    if (warp == 0 && lane == 0) {
        // ---------------------------------------------------------------- producer
        bool ok = true;
        for (int i = 0; i < ns && ok; ++i) {
            const int st = i % kStages, k0 = (s_lo + i) * 64;
            if (i >= kStages && !mbar_wait(&empty[st], ((i / kStages) - 1) & 1, abort_flag, ST_GEMM)) { ok = false; break; }
            uint8_t* a = smem + st * kStageBytes;
            uint8_t* b = a + 16384;
            mbar_expect_tx(&full[st], kStageBytes);
            if (p.a_mn) { tma_load_2d(a, &map_a, &full[st], m0, k0); tma_load_2d(a + 8192, &map_a, &full[st], m0 + 64, k0); }
            else tma_load_2d(a, &map_a, &full[st], k0, m0);
            if (p.b_mn) { tma_load_2d(b, &map_b, &full[st], n0, k0); tma_load_2d(b + 8192, &map_b, &full[st], n0 + 64, k0); }
            else tma_load_2d(b, &map_b, &full[st], k0, n0);
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------------------------------------------------------- product issue
        const uint32_t idesc = umma_idesc(128, 128, p.a_mn, p.b_mn);
        bool ok = true;
        for (int i = 0; i < ns && ok; ++i) {
            const int st = i % kStages;
            if (!mbar_wait(&full[st], (i / kStages) & 1, abort_flag, ST_GEMM)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t a = smem_u32(smem + st * kStageBytes), b = a + 16384;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                umma_ss(tmem, umma_desc_join(step_lo(a, p.a_mn, kk)), umma_desc_join(step_lo(b, p.b_mn, kk)), idesc,
                        (i > 0 || kk > 0) ? 1u : 0u);
            umma_commit(&empty[st]);
        }
        if (ok) umma_commit(done);
    } else if (warp >= 2) {
        // ---------------------------------------------------------------- write-out: one row per thread
        const int q4 = warp & 3, row = q4 * 32 + lane, m = m0 + row;
        const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
        bool ok = ns > 0 ? mbar_wait(done, 0, abort_flag, ST_GEMM) : true;
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after_sync();
        if (ok) {
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                const int n = n0 + c * 32;
                if (n >= p.N) break;
                float v[32];
                if (ns > 0) tile::tmem_row32(tl + c * 32, v);
                else {
#pragma unroll
                    for (int x = 0; x < 32; ++x) v[x] = 0.f;
                }
                if (p.c_atomic) {
                    if (m < p.M && ns > 0) {
                        float* dst = (float*)p.c + (size_t)m * p.ldc + n;
#pragma unroll
                        for (int x = 0; x < 32; x += 4)   // (N is a multiple of 64)
                            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + x), "f"(v[x]), "f"(v[x + 1]),
                                         "f"(v[x + 2]), "f"(v[x + 3]) : "memory");
                    }
                } else {   // bf16, N a multiple of 32 (checked on the host)
                    tile::gstore_bf16x32<true>((__nv_bfloat16*)p.c + (size_t)(m < p.M ? m : 0) * p.ldc + n, v, m < p.M);
                }
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, p.status);
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 128);
    }
}

// ---------------------------------------------------------------------------------------------- wide outputs
// C[M, N] = A B with a contraction of R = 64 or 128 only:  z = t W2^T (B K-major, [N][R])  and  dx = dt W1 (B MN-major, [R][N]).
// Bound by the bytes of C.  A persistent CTA takes units of one 128-row tile of A and `per_unit` column tiles: the A tile is
// fetched once per unit, B tiles go through a ring of two, accumulators alternate between two in tensor memory, and a tile
// leaves as two TMA stores of 64 columns from a staging panel each, so that loads, products and stores of different tiles
// overlap.  As 16384 CTAs of gemm_kernel with one 64-deep stage each, the output of 131072 x 2048 took 188 us
// (2.9 TB/s); it takes 120 us here (4.6 TB/s).
template <int R, bool BMN>
struct WideSmem {
    static constexpr uint32_t tile = R * 256;                 // [128 x R] bf16
    static constexpr uint32_t offA = 0, offB = 2 * tile, offC = offB + 2 * tile, offBar = offC + 32768;
    static constexpr uint32_t alloc = offBar + 256 + 1024;
};
template <int R, bool BMN>
__global__ void __launch_bounds__(192, R == 64 ? 2 : 1) wide_kernel(const __grid_constant__ CUtensorMap map_a,
                                                                    const __grid_constant__ CUtensorMap map_b,
                                                                    const __grid_constant__ CUtensorMap map_c, const int mtiles,
                                                                    const int ntiles, const int per_unit, const int N, uint32_t* status) {
    typedef WideSmem<R, BMN> Sm;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint64_t* bars = (uint64_t*)(smem + Sm::offBar);
    enum { AFULL = 0, AEMPTY = 2, BFULL = 4, BEMPTY = 6, CFULL = 8, CEMPTY = 10, COUNT = 12 };
    uint32_t* tmem_slot = (uint32_t*)(bars + COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < COUNT; ++i) mbar_init(&bars[i], i >= CEMPTY ? 4u : 1u);   // accumulators are handed back by four warps
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, 256);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    const int groups = (ntiles + per_unit - 1) / per_unit, units = mtiles * groups;
    auto wait = [&](int b, uint32_t parity) { return mbar_wait(&bars[b], parity & 1u, abort_flag, ST_GEMM); };
    if (warp == 0 && elect_one()) {
        // ---------------------------------------------------------------- producer
        uint32_t na = 0, nb = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++na) {
            const int m0 = u / groups * 128, t0 = u % groups * per_unit, t1 = min(t0 + per_unit, ntiles);
            if (!(ok = wait(AEMPTY + (na & 1), (na >> 1) ^ 1))) break;
            uint8_t* a = smem + Sm::offA + (na & 1) * Sm::tile;
            mbar_expect_tx(&bars[AFULL + (na & 1)], Sm::tile);
            for (int h = 0; h < R / 64; ++h) tma_load_2d(a + h * 16384, &map_a, &bars[AFULL + (na & 1)], h * 64, m0);
            for (int t = t0; t < t1; ++t, ++nb) {
                if (!(ok = wait(BEMPTY + (nb & 1), (nb >> 1) ^ 1))) break;
                uint8_t* b = smem + Sm::offB + (nb & 1) * Sm::tile;
                mbar_expect_tx(&bars[BFULL + (nb & 1)], Sm::tile);
                if (BMN) {   // panels of [R][64 columns], boxes of 64 x 64
                    for (int h = 0; h < 2; ++h)
                        for (int k = 0; k < R / 64; ++k)
                            tma_load_2d(b + h * (R * 128) + k * 8192, &map_b, &bars[BFULL + (nb & 1)], t * 128 + h * 64, k * 64);
                } else {     // panels of [128 rows][64 k]
                    for (int h = 0; h < R / 64; ++h) tma_load_2d(b + h * 16384, &map_b, &bars[BFULL + (nb & 1)], h * 64, t * 128);
                }
            }
        }
    } else if (warp == 1 && elect_one()) {
        // ---------------------------------------------------------------- product issue
        constexpr uint32_t idesc = umma_idesc(128, 128, 0, BMN ? 1 : 0);
        uint32_t na = 0, nb = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++na) {
            const int t0 = u % groups * per_unit, t1 = min(t0 + per_unit, ntiles);
            if (!(ok = wait(AFULL + (na & 1), na >> 1))) break;
            const uint32_t a_lo = umma_desc_lo(smem_u32(smem + Sm::offA + (na & 1) * Sm::tile), 16);
            for (int t = t0; t < t1; ++t, ++nb) {
                if (!(ok = wait(BFULL + (nb & 1), nb >> 1) && wait(CEMPTY + (nb & 1), (nb >> 1) ^ 1))) break;
                tc_fence_after_sync();
                const uint32_t b_lo = umma_desc_lo(smem_u32(smem + Sm::offB + (nb & 1) * Sm::tile), BMN ? R * 128 : 16);
#pragma unroll
                for (int kk = 0; kk < R / 16; ++kk) {
                    const uint32_t ko = (uint32_t)(kk >> 2) * 1024u + (uint32_t)(kk & 3) * 2u;
                    umma_ss(tmem + (nb & 1) * 128, umma_desc_join(a_lo + ko), umma_desc_join(b_lo + (BMN ? kk * 128u : ko)), idesc, kk > 0);
                }
                umma_commit(&bars[BEMPTY + (nb & 1)]);
                umma_commit(&bars[CFULL + (nb & 1)]);
            }
            if (ok) umma_commit(&bars[AEMPTY + (na & 1)]);
        }
    } else if (warp >= 2) {
        // ---------------------------------------------------------------- write-out: one row per thread, 64 columns at a time
        const int q4 = warp & 3, row = q4 * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
        uint32_t nb = 0;
        bool ok = true;
        auto sync = [&]() { __syncwarp(); asm volatile("bar.sync 1, 128;" ::: "memory"); };
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
            const int m0 = u / groups * 128, t0 = u % groups * per_unit, t1 = min(t0 + per_unit, ntiles);
            for (int t = t0; t < t1; ++t, ++nb) {
                ok = __all_sync(0xffffffffu, wait(CFULL + (nb & 1), nb >> 1));
                tc_fence_after_sync();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint8_t* panel = smem + Sm::offC + h * 16384;
                    uint32_t r0[32], r1[32];
                    if (ok) {
                        tmem_ld32(tl + (nb & 1) * 128 + h * 64, r0);
                        tmem_ld32(tl + (nb & 1) * 128 + h * 64 + 32, r1);
                        tmem_ld_wait();
                    }
                    if (h == 1) {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars[CEMPTY + (nb & 1)]);
                    }
                    // the panel's previous store (two stores ago) has read it
                    if (tid == 64) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    if (h == 0) ok = barrier_and<1, 128>(ok);   // the four warps go on, or leave after this tile, together
                    else sync();
                    if (ok) {
                        float v[32];
#pragma unroll
                        for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r0[x]);
                        tile::tile_store32(panel, row, 0, v);
#pragma unroll
                        for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r1[x]);
                        tile::tile_store32(panel, row, 32, v);
                    }
                    fence_proxy_async_smem();
                    sync();
                    if (tid == 64) {
                        if (ok && t * 128 + h * 64 < N) tma_store_2d(&map_c, panel, t * 128 + h * 64, m0);   // (rows past M are clipped)
                        tma_store_commit();
                    }
                }
                if (!ok) break;
            }
        }
        if (tid == 64) tma_store_wait_all();
    }
    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, status);
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 256);
    }
}

}  // namespace

cudaError_t launch_gemm(const CUtensorMap& map_a, const CUtensorMap& map_b, const GemmParams& p, int split_k, cudaStream_t st) {
    const dim3 grid((p.M + 127) / 128, (p.N + 127) / 128, split_k);
    return launch<gemm_kernel>(grid, 192, kGemmSmem, st, map_a, map_b, p);
}

cudaError_t launch_wide(const CUtensorMap& map_a, const CUtensorMap& map_b, const CUtensorMap& map_c, int M, int N, int R, int b_mn,
                        uint32_t* status, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const int mtiles = (M + 127) / 128, ntiles = (N + 127) / 128, slots = (R == 64 ? 2 : 1) * sms;
    // column tiles per unit: up to four share an A tile, as long as every CTA still gets a few units
    int per_unit = (int)((long)mtiles * ntiles / (4L * slots));
    per_unit = per_unit < 1 ? 1 : (per_unit > 4 ? 4 : per_unit);
    const long units = (long)mtiles * ((ntiles + per_unit - 1) / per_unit);
    const int grid = units < slots ? (int)units : slots;
    if (R == 64)
        return b_mn ? launch<wide_kernel<64, true>>(grid, 192, WideSmem<64, true>::alloc, st, map_a, map_b, map_c, mtiles, ntiles, per_unit, N, status)
                    : launch<wide_kernel<64, false>>(grid, 192, WideSmem<64, false>::alloc, st, map_a, map_b, map_c, mtiles, ntiles, per_unit, N, status);
    return b_mn ? launch<wide_kernel<128, true>>(grid, 192, WideSmem<128, true>::alloc, st, map_a, map_b, map_c, mtiles, ntiles, per_unit, N, status)
                : launch<wide_kernel<128, false>>(grid, 192, WideSmem<128, false>::alloc, st, map_a, map_b, map_c, mtiles, ntiles, per_unit, N, status);
}

}  // namespace path
