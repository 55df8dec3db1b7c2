// Per-chunk chain rule of the backward pass (the paper gives no backward): from the gradients of the
// boundary-adjusted tiles (dQl, dKr), of the diagonal-chunk logits (dSd) and of the chunk product (dP) back through
// the UT transform to dq, dk, dw, dbeta.  With Xq = lower(Q W^T), Xk = strictLower(W K^T), Y = T~ Xk, U = T~ W,
// T~ = Ainv D, Ainv = (I + strictLower(D W W^T))^-1 and s = scale:
//   dXq = lower(-dQl U^T - s dSd Y^T)            dY  = -W dKr^T - s Xq^T dSd           dU = -Xq^T dQl - W dP
//   dT  = lower(dY Xk^T + dU W^T)                dXk = strictLower(T~^T dY)
//   M   = Ainv^T dT,   dbeta_c  = M_cc,          dA  = strictLower(-M T~^T)       (Ainv^T = D^-1 T~^T: beta is never exactly 0 here)
//   dbeta_r += sum_c dA_rc (W W^T)_rc,           dGm = D dA
//   dq = dQl + s dSd K + dXq W                   dk = dKr + s dSd^T Q + dXk^T W
//   dw = -Y dKr - U dP^T + T~^T dU + dXq^T Q + dXk K + (dGm + dGm^T) W
// A persistent CTA (one per SM) walks over chunks and runs these ~31 products per chunk as tcgen05 MMAs on swizzled
// shared-memory tiles.  Sixteen worker warps turn accumulators (tensor memory, 32 columns of one row per thread) into the next
// operand tiles; one lane of another warp requests every tile (TMA) and issues every product.  The two sides meet only
// through mbarriers: the workers hand tiles over and go on (they wait for products, never for the issuer), the issuer
// sends out first whatever does not depend on the read-out in progress, starts the next chunk's first products while
// the current chunk's results are still leaving, and requests tiles the moment their slots are free.  dQl and dKr
// arrive as bf16 tiles.  T~ enters as a bf16 hi + lo pair, and so do the in-kernel intermediates dT, M and dGm;
// everything else is rounded to bf16 once.  dw accumulates in tensor memory across all phases.
#include "tileops.cuh"

namespace path {
using namespace tile;

namespace {

constexpr int kSlots = 7;
constexpr int kChainWorkers = 512, kChainThreads = kChainWorkers + 32;   // sixteen worker warps + the one that loads tiles and issues products
constexpr uint32_t kBarOff = kSlots * kTileB;
constexpr uint32_t kChainSmem = kBarOff + 64 + 3 * kT * 4 + 1024;

template <int HD>
__global__ void __launch_bounds__(kChainThreads, 1) chunk_chain_kernel(const __grid_constant__ ChainTensorMaps tm,
                                                             const ChainParams p, const int nchunks) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint64_t* bars = (uint64_t*)(smem + kBarOff);  // two for loads, two for product groups, two for the workers' hand-overs
    uint32_t* tmem_slot = (uint32_t*)(bars + 6);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    float* t1 = (float*)(smem + kBarOff + 64);
    float* parts = t1 + kT;   // [2][128]

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane, cg = (warp >> 2) & 3;   // a worker's row and which 32 of an accumulator's columns it has

    if (tid == 0) {
        for (int i = 0; i < 6; ++i) mbar_init(&bars[i], i < 4 ? 1u : (uint32_t)kChainWorkers);   // B_R0, B_R1: every worker arrives
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    auto slot = [&](int i) { return smem + i * kTileB; };
    auto sa = [&](int i) { return smem_u32(smem + i * kTileB); };
    constexpr int KD = HD / 16, K8 = 8;
    constexpr uint32_t cDW = 0, cA = 128, cB = 256, cG = 384;   // tensor-memory columns: dw, two work accumulators, W W^T
    enum { B_LOAD = 0, B_LOAD2, B_MMA, B_MMA2, B_R0, B_R1, B_COUNT };
    const int grid = (int)gridDim.x;

    if (warp == kChainWorkers / 32) {
    if (elect_one()) {
    // ------------------------------------------------------------------ leader: TMA loads and every product
    bool ok = true;
    uint32_t ph[7] = {0, 0, 0, 0, 0, 0, 0};
    auto wait = [&](int b) {   // false (and nothing more is issued) once a wait has run out
        if (ok && !mbar_wait(&bars[b], ph[b], abort_flag, ST_CHAIN)) ok = false;
        ph[b] ^= 1;
        tc_fence_after_sync();
        return ok;
    };
    // slots: 0 U->dXq   1 dQl->T~ hi->K   2 Y->Xq->Xk->dT hi->M hi->dGm hi   3 dSd->T~ lo->dSd
    //        4 W   5 dKr->dY->dXk->dGm lo   6 dP->dU->dT lo->M lo->Q
    // First tiles of a chunk, in two parts: five of the seven slots are free as soon as the products that finish dq and dk
    // have retired, and these five tiles are all that the chunk's first two products read; the other two slots feed the
    // previous chunk's very last products.
    auto first_loads_a = [&](int ch) {
        mbar_expect_tx(&bars[B_LOAD], 2 * kT * HD * 2 + HD * HD * 2 + 2 * kTileB);
        tma_tile(slot(1), &tm.dql, &bars[B_LOAD], HD, ch * kT);
        tma_tile(slot(0), &tm.u, &bars[B_LOAD], HD, ch * kT);
        tma_tile(slot(3), &tm.dsdt, &bars[B_LOAD], kT, ch * kT);   // (s dSd)^T: every use takes the transposed view
        tma_tile(slot(2), &tm.y, &bars[B_LOAD], kT, ch * kT);
        tma_tile(slot(6), &tm.dp, &bars[B_LOAD], HD, ch * HD);
    };
    auto first_loads_b = [&](int ch) {
        mbar_expect_tx(&bars[B_LOAD2], 2 * kT * HD * 2);
        tma_tile(slot(5), &tm.dkr, &bars[B_LOAD2], HD, ch * kT);
        tma_rows(slot(4), &tm.w, &bars[B_LOAD2], HD, (ch % p.N) * kT, ch / p.N);
    };
    // Tiles on their way into L2 before their slots are free: a load that has to come from memory holds the chain up for 2 to 3 thousand
    // cycles.  Only where the copy engine has nothing to load meanwhile: it works requests off in order.  (As prefetch.global of
    // worker threads or of a warp of their own they held up the next hand-over or the stores to shared memory.)  At d = 128, where
    // the bytes themselves take as long as the chain, it changes nothing.  8 x 16 x 2048 x 64: 231 -> 216 us.
    constexpr bool kPrefetch = HD == 64;
    auto fetch = [&](const CUtensorMap* m, int ncols, int row0) {
        for (int h = 0; h < ncols / 64; ++h) tma_prefetch_2d(m, h * 64, row0);
    };
    auto fetch_rows = [&](const CUtensorMap* m, int ch) {
        for (int h = 0; h < HD / 64; ++h) tma_prefetch_3d(m, h * 64, (ch % p.N) * kT, ch / p.N);
    };
    if ((int)blockIdx.x < nchunks) {
        first_loads_a(blockIdx.x);
        first_loads_b(blockIdx.x);
    }
#pragma unroll 1
    for (int chunk = blockIdx.x; chunk < nchunks && ok; chunk += grid) {
        const int r0 = chunk * kT;
        // ---- phase 0: dXq = lower(-(dQl U^T + s dSd Y^T)) -> cA, while the previous chunk's results are still leaving
        // the other columns; then dw = -Y dKr - U dP^T
        if (!wait(B_LOAD)) break;
        mma<OP_K, OP_K, KD, 128, true>(tmem + cA, sa(1), sa(0), false);
        mma<OP_MN, OP_K, K8, 128, true>(tmem + cA, sa(3), sa(2), true);
        if (chunk != (int)blockIdx.x && !wait(B_R1)) break;                      // the previous chunk's dw has left cDW
        if (!wait(B_LOAD2)) break;
        mma<OP_K, OP_MN, K8, HD, true>(tmem + cDW, sa(2), sa(5), false);
        mma<OP_K, OP_K, KD, HD, true>(tmem + cDW, sa(0), sa(6), true);
        umma_commit(&bars[B_MMA]);
        // ---- phase 1: dY = -(W dKr^T + Xq^T s dSd) -> cA,  dU = -(Xq^T dQl + W dP) -> cB.  dU's products read no tile
        // that the workers are writing and go to their own columns: they run underneath the read-out of dXq.
        if (!wait(B_MMA)) break;
        mbar_expect_tx(&bars[B_LOAD], kTileB);
        tma_tile(slot(2), &tm.xq, &bars[B_LOAD], kT, r0);
        mma<OP_K, OP_MN, KD, HD, true>(tmem + cB, sa(4), sa(6), false);     // W dP needs no new tile
        if (!wait(B_LOAD)) break;
        mma<OP_MN, OP_MN, K8, HD, true>(tmem + cB, sa(2), sa(1), true);
        if (!wait(B_R0)) break;                                                  // dXq has left cA
        mma<OP_K, OP_K, KD, 128, true>(tmem + cA, sa(4), sa(5), false);
        mma<OP_MN, OP_K, K8, 128, true>(tmem + cA, sa(2), sa(3), true);
        umma_commit(&bars[B_MMA]);
        // ---- phase 2: dT = lower(dY Xk^T + dU W^T) -> cA, and phase 3 right behind it (the same dY and dU tiles and T~):
        // dXk = strictLower(T~^T dY) -> cB,  dw += T~^T dU.  (s dSd)^T is not needed again before phase 5, where it is
        // loaded once more: until then its slot (3) holds T~ lo.
        if (!wait(B_MMA)) break;
        mbar_expect_tx(&bars[B_LOAD], 3 * kTileB);
        tma_tile(slot(2), &tm.xk, &bars[B_LOAD], kT, r0);
        tma_tile(slot(1), &tm.th, &bars[B_LOAD], kT, r0);
        tma_tile(slot(3), &tm.tl, &bars[B_LOAD], kT, r0);
        // (from here to phase 5 nothing is loaded: what phase 5 and the next chunk's first phases need)
        if (kPrefetch) {
            fetch_rows(&tm.q, chunk);
            fetch_rows(&tm.k, chunk);
        }
        if (kPrefetch && chunk + grid < nchunks) {
            const int ch = chunk + grid;
            fetch(&tm.dql, HD, ch * kT);
            fetch(&tm.u, HD, ch * kT);
            fetch(&tm.dsdt, kT, ch * kT);
            fetch(&tm.y, kT, ch * kT);
            fetch(&tm.dp, HD, ch * HD);
            fetch(&tm.dkr, HD, ch * kT);
            fetch_rows(&tm.w, ch);
            fetch(&tm.xq, kT, ch * kT);
        }
        if (!wait(B_R1)) break;                                                  // dY, dU tiles
        mma<OP_K, OP_K, KD, 128>(tmem + cA, sa(6), sa(4), false);           // dU W^T needs no new tile
        if (!wait(B_LOAD)) break;
        mma<OP_K, OP_K, K8, 128>(tmem + cA, sa(5), sa(2), true);
        umma_commit(&bars[B_MMA]);
        mma<OP_MN, OP_MN, K8, 128>(tmem + cB, sa(1), sa(5), false);
        mma<OP_MN, OP_MN, K8, 128>(tmem + cB, sa(3), sa(5), true);
        mma<OP_MN, OP_MN, K8, HD>(tmem + cDW, sa(1), sa(6), true);
        mma<OP_MN, OP_MN, K8, HD>(tmem + cDW, sa(3), sa(6), true);
        umma_commit(&bars[B_MMA2]);
        // ---- phase 4: D M = T~^T dT -> cG;  dA = strictLower(-M T~^T) -> cA;  W W^T -> cB (for dbeta).  T~ is still there.
        if (!wait(B_MMA) || !wait(B_MMA2)) break;
        if (!wait(B_R0)) break;                                                  // dT hi, lo tiles
        mma<OP_MN, OP_MN, K8, 128>(tmem + cG, sa(1), sa(2), false);
        mma<OP_MN, OP_MN, K8, 128>(tmem + cG, sa(3), sa(2), true);
        mma<OP_MN, OP_MN, K8, 128>(tmem + cG, sa(1), sa(6), true);
        umma_commit(&bars[B_MMA]);
        if (!wait(B_R1)) break;                                                  // dXk has left cB
        mma<OP_K, OP_K, KD, 128>(tmem + cB, sa(4), sa(4), false);          // retires with the next group
        if (!wait(B_MMA)) break;
        if (!wait(B_R0)) break;                                                  // M hi, lo tiles
        mma<OP_K, OP_K, K8, 128, true>(tmem + cA, sa(2), sa(1), false);
        mma<OP_K, OP_K, K8, 128, true>(tmem + cA, sa(2), sa(3), true);
        mma<OP_K, OP_K, K8, 128, true>(tmem + cA, sa(6), sa(1), true);
        umma_commit(&bars[B_MMA]);
        // ---- phase 5: dq -> cB, dk -> cG and the rest of dw, in three groups.  K, (s dSd)^T and Q replace T~ and M
        // lo.  First the products that need neither dGm nor the columns that dbeta still reads; when they have
        // retired, dXk's slot is free for dGm lo.  The second group finishes dq and dk, the third (dGm lo) only dw.
        if (!wait(B_MMA)) break;
        mbar_expect_tx(&bars[B_LOAD], 2 * kT * HD * 2 + kTileB);
        tma_tile(slot(3), &tm.dsdt, &bars[B_LOAD], kT, r0);
        tma_rows(slot(6), &tm.q, &bars[B_LOAD], HD, (chunk % p.N) * kT, chunk / p.N);
        tma_rows(slot(1), &tm.k, &bars[B_LOAD], HD, (chunk % p.N) * kT, chunk / p.N);
        mma<OP_MN, OP_MN, K8, HD>(tmem + cG, sa(5), sa(4), false);          // dXk^T W needs no new tile
        if (!wait(B_LOAD)) break;
        mma<OP_K, OP_MN, K8, HD>(tmem + cG, sa(3), sa(6), true);            // s dSd^T Q
        mma<OP_MN, OP_MN, K8, HD>(tmem + cDW, sa(0), sa(6), true);          // dXq^T Q
        mma<OP_K, OP_MN, K8, HD>(tmem + cDW, sa(5), sa(1), true);           // dXk K
        umma_commit(&bars[B_MMA2]);
        if (!wait(B_R1)) break;                                                  // dGm hi tile; W W^T has left cB
        mma<OP_MN, OP_MN, K8, HD>(tmem + cB, sa(3), sa(1), false);          // s dSd K
        mma<OP_K, OP_MN, K8, HD>(tmem + cB, sa(0), sa(4), true);            // dXq W
        mma<OP_K, OP_MN, K8, HD>(tmem + cDW, sa(2), sa(4), true);           // dGm W
        mma<OP_MN, OP_MN, K8, HD>(tmem + cDW, sa(2), sa(4), true);          // dGm^T W
        umma_commit(&bars[B_MMA]);
        if (!wait(B_MMA2)) break;
        // (the last two products cannot start before the second group has left the pipe anyway: the next chunk's tiles are
        // requested first, the moment their slots are free)
        const int next = chunk + grid;
        if (!wait(B_MMA)) break;
        if (next < nchunks) first_loads_a(next);                                 // slots 0 - 3 and 6 are free
        if (!wait(B_R0)) break;                                                  // dGm lo tile (over dXk)
        mma<OP_K, OP_MN, K8, HD>(tmem + cDW, sa(5), sa(4), true);
        mma<OP_MN, OP_MN, K8, HD>(tmem + cDW, sa(5), sa(4), true);
        umma_commit(&bars[B_MMA2]);
        if (!wait(B_MMA2)) break;
        if (next < nchunks) {
            first_loads_b(next);                                                 // and the other two
            if (kPrefetch) {
                fetch(&tm.xk, kT, next * kT);
                fetch(&tm.th, kT, next * kT);
                fetch(&tm.tl, kT, next * kT);
            }
        }
    }
    }
    __syncwarp();
    } else {
    // ------------------------------------------------------------------ workers: accumulators -> next operand tiles
    bool ok = true;
    uint32_t ph_mma = 0, ph_mma2 = 0;
    float v[32];
    uint32_t hi[16], lo[16];
    auto wsync = [&]() {
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(kChainWorkers) : "memory");
    };
    // lane 0 of every warp waits for the product group; the vote that follows releases the other lanes
    auto mma_wait = [&](int b = B_MMA) {
        uint32_t& ph = b == B_MMA ? ph_mma : ph_mma2;
        bool good = true;
        if (lane == 0) good = mbar_wait(&bars[b], ph, abort_flag, ST_CHAIN);
        ph ^= 1;
        ok = barrier_and<1, kChainWorkers>(good);
        tc_fence_after_sync();
    };
    // tiles written by this thread become visible to the MMA unit, its accumulator reads are ordered, the leader learns
    auto publish = [&](int b) {
        fence_proxy_async_smem();
        tc_fence_before_sync();
        mbar_arrive(&bars[b]);
    };
    // This thread's 32 columns of an accumulator's lower triangle.  `above` = columns minus rows of the warp's 32 x 32 block: > 0 nothing
    // of it counts, < 0 everything, 0 it lies on the diagonal, which counts itself or not.
    const int above = cg * 32 - (warp & 3) * 32;
    auto read_lower = [&](uint32_t col, int diagonal) {
        if (above > 0) {
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] = 0.f;
            return;
        }
        tmem_row32(tl + col + cg * 32, v);
        if (above == 0) {
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] = x < lane + diagonal ? v[x] : 0.f;
        }
    };
    // A tile of the head dimension: its 32 columns from head_c0 on belong to this thread if `mine`.  At d = 64 two of the four column
    // groups would have none; the second of two such tiles then goes to them.
    auto has = [&](int which) { return HD == 128 || (cg >> 1) == which; };
    const int head_c0 = (HD == 128 ? cg : cg & 1) * 32;

#pragma unroll 1
    for (int chunk = blockIdx.x; chunk < nchunks; chunk += grid) {
        const int s_idx = chunk / p.N, pos = (chunk % p.N) * kT + row;   // slice and position of this thread's row
        const bool row_valid = pos < p.L;
        const size_t urow = (size_t)s_idx * p.L + pos;                   // row in the caller's [S][L][.] tensors
        const float beta = beta_floor(row_valid ? p.beta[urow] : 0.f), inv_b = 1.f / beta;
        mma_wait();                                                 // phase 0
        if (!ok) break;
        read_lower(cA, 1);
        tile_store32(slot(0), row, cg * 32, v);                     // dXq (over U)
        publish(B_R0);
        mma_wait();                                                 // phase 1
        if (!ok) break;
        tmem_row32(tl + cA + cg * 32, v);
        tile_store32(slot(5), row, cg * 32, v);                     // dY (over dKr)
        if (has(0)) {
            tmem_row32(tl + cB + head_c0, v);
            tile_store32(slot(6), row, head_c0, v);                 // dU (over dP)
        }
        publish(B_R1);
        mma_wait();                                                 // phase 2
        if (!ok) break;
        // dT: its bf16 hi part goes over Xk now, the lo part follows once dU has been read
        read_lower(cA, 1);
        split32(v, hi, lo);
        tile_store_w16(slot(2), row, cg * 32, hi);
        mma_wait(B_MMA2);                                           // phase 3
        if (!ok) break;
        tile_store_w16(slot(6), row, cg * 32, lo);                  // dT lo (over dU)
        publish(B_R0);
        // dXk leaves its columns while M is being computed; W W^T takes them over as soon as it has
        read_lower(cB, 0);
        tile_store32(slot(5), row, cg * 32, v);                     // dXk (over dY)
        publish(B_R1);
        mma_wait();                                                 // D M
        if (!ok) break;
        {   // M, hi (over dT hi) and lo (over dT lo); its diagonal is dbeta's column part
            tmem_row32(tl + cG + cg * 32, v);
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] *= inv_b;
            if (above == 0) {
                float m = 0.f;
#pragma unroll
                for (int x = 0; x < 32; ++x) m = x == lane ? v[x] : m;
                t1[row] = m;
            }
            split32(v, hi, lo);
            tile_store_w16(slot(2), row, cg * 32, hi);
            tile_store_w16(slot(6), row, cg * 32, lo);
        }
        publish(B_R0);
        mma_wait();                                                 // dA and W W^T
        if (!ok) break;
        float part = 0.f;
        {   // dA = strictLower(cA);  dbeta_r = t1_r + sum_c dA_rc (W W^T)_rc;  dGm = D dA, hi now, lo once dXk's slot is free
            read_lower(cA, 0);
            if (above <= 0) {
                float gm[32];
                tmem_row32(tl + cB + cg * 32, gm);
#pragma unroll
                for (int x = 0; x < 32; ++x)
                    if (above < 0 || x < lane) part += v[x] * gm[x];
            }
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] *= beta;
            split32(v, hi, lo);
            tile_store_w16(slot(2), row, cg * 32, hi);
        }
        publish(B_R1);
        // (global stores and loads come after a hand-over, never just before it: the hand-over waits for them)
        // The dQl / dKr rows of the final sums are fetched while the products run.  (d = 64: a thread finishes either dq or dk and
        // keeps one row segment.  With an array for each the kernel spilled 72 bytes per thread, in a loop that has no L1 to speak of:
        // 211 / 199 us at 8 x 16 x 2048 x 64.)
        uint32_t fetched[HD / 64][2][8];
        auto is_k = [&](int i) { return HD == 128 ? i == 1 : has(1); };
#pragma unroll
        for (int i = 0; i < HD / 64; ++i)
            gload_bf16_issue((is_k(i) ? p.dkr : p.dql) + ((size_t)chunk * kT + row) * HD + head_c0, fetched[i]);
        // the four threads of a row add their parts through shared memory
        if (cg >= 2) parts[(cg - 2) * kT + row] = part;
        wsync();
        if (cg < 2) part += parts[cg * kT + row];
        if (cg == 1) parts[kT + row] = part;
        wsync();
        if (cg == 0 && row_valid) p.dbeta[urow] = t1[row] + (part + parts[kT + row]);
        mma_wait(B_MMA2);                                           // phase 5, first group: dXk's slot is free
        if (!ok) break;
        tile_store_w16(slot(5), row, cg * 32, lo);                  // dGm lo (over dXk)
        publish(B_R0);
        mma_wait();                                                 // phase 5, second group
        if (!ok) break;
        // dq and dk are complete: they leave while the last two products run
#pragma unroll
        for (int i = 0; i < HD / 64; ++i) {
            uint32_t w[16];
            gload_bf16_finish(fetched[i], w);
            tmem_row32(tl + (is_k(i) ? cG : cB) + head_c0, v);
#pragma unroll
            for (int x = 0; x < 16; ++x) {
                v[2 * x] += __uint_as_float(w[x] << 16);
                v[2 * x + 1] += __uint_as_float(w[x] & 0xffff0000u);
            }
            gstore_bf16x32<true>((is_k(i) ? p.dk : p.dq) + urow * HD + head_c0, v, row_valid);
        }
        mma_wait(B_MMA2);                                           // the last of dw
        if (!ok) break;
        if (has(0)) {
            tmem_row32(tl + cDW + head_c0, v);
            gstore_bf16x32<true>(p.dw + urow * HD + head_c0, v, row_valid);
        }
        publish(B_R1);   // the next chunk's first products overwrite the accumulators read above
    }
    }

    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, p.status);
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace

cudaError_t launch_chunk_chain(const ChainTensorMaps& tm, const ChainParams& p, int hd, int nchunks, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const int grid = nchunks < sms ? nchunks : sms;
    return hd == 64 ? launch<chunk_chain_kernel<64>>(grid, kChainThreads, kChainSmem, st, tm, p, nchunks)
                    : launch<chunk_chain_kernel<128>>(grid, kChainThreads, kChainSmem, st, tm, p, nchunks);
}

}  // namespace path
