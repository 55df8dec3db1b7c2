// Backward of the attention sweep (the paper gives no backward; this is the FlashAttention-2 style
// recomputation applied to the dyadic query / key versions of fa_fwd.cu).
//
//   P = exp(S - LSE),  dP = dO V^T,  dS = P o (dP - delta),  delta_i = dO_i . O_i
//   dV_J  = sum_I P^T dO_I                       dKv[l][J] = scale sum_{I at level l} dS^T Qv[l][I]
//   dQv[l][I] = scale sum_{J at level l} dS Kv[l][J]
//   gate prefix:  dG_m = sum_j dS_mj - sum_i dS_im  (row sums are written by dq_kernel, column sums by dkv_kernel;
//                 the row sums vanish in exact arithmetic but cancel the rounding of delta in the suffix sums)
//   diagonal chunk: (scale lower(dS))^T is stored for the per-chunk chain rule; its row sums in float32 if gated.
//
// Two kernels so that every accumulator stays in tensor memory and nothing is added atomically:
//   dkv_kernel, dkv64_kernel: one CTA per key chunk J, sweeps the query chunks I = J..N-1 with transposed tiles
//               (TMEM lanes = keys): S^T = K Q^T, dP^T = V dO^T, dV += P^T dO, dK += dS^T Q.
//   dq_kernel : one CTA per query chunk I, sweeps J = I-1..0: S = Q K^T, dP = dO V^T, dQ += dS K.
// The accumulator of a version is flushed to global memory when the sweep crosses into the next level.
// P^T / dS^T (dkv) and dS (dq) never touch shared memory: they overwrite the first half of the columns their thread
// read, as packed bf16, and enter the second products as tensor-memory A operands.
//
// The elementwise work of a step is split in two so that it overlaps the tensor pipe: part A turns S into P (the
// exponentials) as soon as S is there, while the dP product still runs; part B forms dS once dP has arrived.  dkv_kernel
// issues its products in the order  dV(t), S(t+1), dK(t), dP(t+1),  so the pipe always has the next step's logits in flight.
// Where tensor memory has room for two S tiles (dq_kernel; dkv64_kernel for d = 64 without a gate) the two parts of
// neighbouring steps share one pass.
// Warps of dkv_kernel: 0 = TMA producer, 1 = tcgen05 MMA issuer, 2-3 idle (their registers go to the others), 4-11 = elementwise
// math (two warps per TMEM lane quadrant, each taking 64 of the 128 columns of a row).
#include <type_traits>
#include "common.cuh"
#include "tc5.cuh"
#include "tileops.cuh"

namespace path {
using namespace tc5;

namespace {

constexpr int kTile = 128;
constexpr uint32_t kSlotBytes = 32768;
constexpr uint32_t kPanelBytes = 16384;
constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t kSmemAlloc = 232448;   // everything an SM offers one CTA

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// A warp writes its 32 accumulator rows as bf16: lane L holds CW consecutive columns of row L, scaled by `mul`; `dst`
// is the first of them in the lane's own row.  One 32-column piece at a time (this runs inside the sweeps' hot loops).
template <int CW>
__device__ __forceinline__ void store_acc_bf16(__nv_bfloat16* dst, uint32_t tcol, float mul) {
#pragma unroll 1
    for (int c = 0; c < CW / 32; ++c) {
        uint32_t r[32], w[16];
        tmem_ld32(tcol + c * 32, r);
        tmem_ld_wait();
#pragma unroll
        for (int x = 0; x < 16; ++x) w[x] = pack_bf16(__uint_as_float(r[2 * x]) * mul, __uint_as_float(r[2 * x + 1]) * mul);
        tile::gstore_bf16_w16(dst + c * 32, w);
    }
}

// D[tmem] (+)= A B^T with both operands K-major [rows][kdim] tiles (two 64-column panels per 128 of kdim).  Descriptors
// advance by their low word only (32 bytes per step, the next panel after four steps).
__device__ __forceinline__ void mma_kk(uint32_t d_tmem, uint32_t a0, uint32_t b0, int kdim, uint32_t idesc, bool acc) {
    uint32_t a_lo = umma_desc_lo(a0, 16), b_lo = umma_desc_lo(b0, 16);
#pragma unroll
    for (int kk = 0; kk < kdim / 16; ++kk) {
        umma_ss(d_tmem, umma_desc_join(a_lo), umma_desc_join(b_lo), idesc, (acc || kk > 0) ? 1u : 0u);
        const uint32_t step = (kk & 3) == 3 ? (kPanelBytes - 96u) >> 4 : 2u;
        a_lo += step;
        b_lo += step;
    }
}
// D[tmem] (+)= A B with A in tensor memory (packed bf16: the 64 contraction indices [64h, 64h+64) of a row sit in the
// 32 columns starting at a_col + 64h) and B MN-major [128 (k)][HD] in shared memory (2048 bytes per step).
__device__ __forceinline__ void mma_tn(uint32_t d_tmem, uint32_t a_col, uint32_t b0, uint32_t idesc, bool acc) {
    uint32_t b_lo = umma_desc_lo(b0, kPanelBytes);
#pragma unroll
    for (int kk = 0; kk < kTile / 16; ++kk) {
        umma_ts(d_tmem, a_col + (kk >> 2) * 64 + (kk & 3) * 8, umma_desc_join(b_lo), idesc, (acc || kk > 0) ? 1u : 0u);
        b_lo += 128u;
    }
}

using tile::tma_rows;
using tile::tma_tile;

// ------------------------------------------------------------------------------------------------ dK, dV
// Persistent: the work items (one key chunk of one slice each) are listed slice after slice as pairs (longest,
// shortest), (second longest, second shortest), ...; CTA c takes the pairs c, c + gridDim.x, ...  Every ring and phase
// counter runs on across items, so the loads and the first products of the next item overlap the write-out of the
// current one.
enum { K_KFULL = 0, K_KEMPTY, K_VFULL, K_VEMPTY, K_QFULL, K_QEMPTY = K_QFULL + 3, K_DOFULL = K_QEMPTY + 3,
       K_DOEMPTY = K_DOFULL + 2, K_SFULL = K_DOEMPTY + 2, K_DPFULL, K_PFULL, K_DSFULL, K_ACCFULL, K_ACCFREE,
       K_STFULL, K_STEMPTY = K_STFULL + 2, K_COUNT = K_STEMPTY + 2 };
constexpr uint32_t kDkvStat = 7 * kSlotBytes + 256;           // [2][2][128] floats: -lse2 (plus gate), -delta
constexpr uint32_t kDkvTotal = kDkvStat + 2 * 2 * kTile * 4 + kTile * 4;   // + [128] exchange of the gate column sums

template <int HD, bool GATE>
__global__ void __launch_bounds__(384, 1) dkv_kernel(const __grid_constant__ BwdTensorMaps tm, const BwdParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    if ((uint32_t)(smem - smem_raw) + kDkvTotal > kSmemAlloc) {   // uniform over the CTA
        grid_wait();   // (the status word belongs to the kernels before)
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)ST_DKV_PRODUCER);
        return;
    }
    uint8_t* sK = smem;
    uint8_t* sV = sK + kSlotBytes;
    uint8_t* sQ = sV + kSlotBytes;          // ring of 3; per item: rawQ, Xq, then Q of step t >= 1 (entry t + 1)
    uint8_t* sDO = sQ + 3 * kSlotBytes;     // ring of 2; per item: Y, then dO of step t (entry t + 1)
    uint64_t* bars = (uint64_t*)(smem + 7 * kSlotBytes);
    uint32_t* tmem_slot = (uint32_t*)(bars + K_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    float* rowstat = (float*)(smem + kDkvStat);
    float* dsum_x = rowstat + 2 * 2 * kTile;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = p.N * p.S;

    if (threadIdx.x == 0) {
        for (int i = 0; i < K_COUNT; ++i)
            mbar_init(&bars[i], (i == K_PFULL || i == K_DSFULL || i == K_ACCFREE || i == K_STEMPTY || i == K_STEMPTY + 1)
                                    ? 256u : 1u);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 2 && lane < 8) tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&tm) + lane);
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    constexpr uint32_t colS = 0, colDP = 128, colDV = 256, colDK = 384;
    // k-th work item of this CTA
    auto item_of = [&](int k, int& J, int& s) {
        const int w = 2 * ((int)blockIdx.x + (k >> 1) * (int)gridDim.x) + (k & 1);
        if (w >= items) return false;
        s = w / p.N;
        const int j = w % p.N;
        J = (j & 1) ? p.N - 1 - (j >> 1) : (j >> 1);
        return true;
    };
    int J = 0, s = 0;   // current item of this thread's role
    auto qrow = [&](int lvl, int chunk) { return qver_row(p.vl, s, lvl, chunk); };   // first row of a version tile
    auto krow = [&](int lvl, int chunk) { return kver_row(p.vl, s, lvl, chunk); };
    auto row0 = [&](int chunk) { return (long)s * p.Lp + (long)chunk * kTile; };      // plane 0
    auto level = [&](int t) { return t == 0 ? -1 : msb32((unsigned)((J + t) ^ J)); };
    // query chunks this key chunk meets (I = J .. J + T - 1): all later ones, or fewer when the gate has made the far
    // pairs negligible (every warp role reads the same precomputed number)
    auto steps_of = [&](int J, int s) { return p.nvisit ? min(p.N - J, p.nvisit[s * p.N + J]) : p.N - J; };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp == 0 && elect_one()) {
            bool ok = true;
            int nk = 0, nv = 0, qn = 0, dn = 0, sn = 0;   // fills so far: K, V, Q ring, dO ring, statistics ring
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_DKV_PRODUCER)) ok = false;
            };
            auto load_q = [&](const CUtensorMap* m, int kdim, int row0, int slice = -1) {   // slice >= 0: a caller's tensor
                const int slot = qn % 3;
                wait_empty(K_QEMPTY + slot, qn / 3);
                if (!ok) return;
                mbar_expect_tx(&bars[K_QFULL + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tma_rows(sQ + slot * kSlotBytes, m, &bars[K_QFULL + slot], kdim, row0, slice);
                else tma_tile(sQ + slot * kSlotBytes, m, &bars[K_QFULL + slot], kdim, row0);
                ++qn;
            };
            auto load_do = [&](const CUtensorMap* m, int kdim, int row0, int slice = -1) {
                const int slot = dn & 1;
                wait_empty(K_DOEMPTY + slot, dn >> 1);
                if (!ok) return;
                mbar_expect_tx(&bars[K_DOFULL + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tma_rows(sDO + slot * kSlotBytes, m, &bars[K_DOFULL + slot], kdim, row0, slice);
                else tma_tile(sDO + slot * kSlotBytes, m, &bars[K_DOFULL + slot], kdim, row0);
                ++dn;
            };
#pragma unroll 1
            for (int it = 0; ok && item_of(it, J, s); ++it) {
                const int T = steps_of(J, s), rowJ = s * p.Lp + J * kTile;
#pragma unroll 1
                for (int t = 0; t < T && ok; ++t) {
                    const int I = J + t, l = level(t);
                    if (t == 0 || l != level(t - 1)) {
                        wait_empty(K_KEMPTY, nk);
                        if (!ok) break;
                        mbar_expect_tx(&bars[K_KFULL], kTile * HD * 2);
                        if (t == 0) tma_rows(sK, &tm.k_raw, &bars[K_KFULL], HD, J * kTile, s);
                        else tma_tile(sK, &tm.kv, &bars[K_KFULL], HD, (int)krow(l, J));
                        ++nk;
                    }
                    if (t == 0) {
                        load_q(&tm.q_raw, HD, J * kTile, s);
                        load_q(&tm.xq, kTile, rowJ);
                        load_do(&tm.y, kTile, rowJ);
                        wait_empty(K_VEMPTY, nv);
                        if (!ok) break;
                        mbar_expect_tx(&bars[K_VFULL], kTile * HD * 2);
                        tma_rows(sV, &tm.v, &bars[K_VFULL], HD, J * kTile, s);
                        ++nv;
                        load_do(&tm.d_o, HD, J * kTile, s);
                    } else {
                        load_q(&tm.qv, HD, (int)qrow(l, I));
                        load_do(&tm.d_o, HD, I * kTile, s);
                    }
                    // per-query statistics of the step
                    wait_empty(K_STEMPTY + (sn & 1), sn >> 1);
                    if (!ok) break;
                    mbar_expect_tx(&bars[K_STFULL + (sn & 1)], 2 * kTile * 4);
                    const size_t gi = (size_t)s * p.Lp + I * kTile;
                    bulk_load(rowstat + (sn & 1) * 2 * kTile, p.lse2 + gi, kTile * 4, &bars[K_STFULL + (sn & 1)]);
                    bulk_load(rowstat + (sn & 1) * 2 * kTile + kTile, p.delta + gi, kTile * 4, &bars[K_STFULL + (sn & 1)]);
                    ++sn;
                }
            }
        } else if (warp == 1 && elect_one()) {
            constexpr uint32_t idescT = umma_idesc(128, 128, 0, 0);
            constexpr uint32_t idescD = umma_idesc(128, HD, 0, 1);
            bool ok = true;
            int nk = 0, nv = 0, qb = 0, db = 0, g = 0;   // K / V fills consumed; ring entries and steps before this item
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_DKV_MMA)) ok = false;
            };
            auto q_wait = [&](int e) { wait(K_QFULL + e % 3, e / 3); };
            auto do_wait = [&](int e) { wait(K_DOFULL + (e & 1), e >> 1); };
            auto q_addr = [&](int e) { return smem_u32(sQ + (e % 3) * kSlotBytes); };
            auto do_addr = [&](int e) { return smem_u32(sDO + (e & 1) * kSlotBytes); };
#pragma unroll 1
            for (int it = 0; ok && item_of(it, J, s); ++it) {
                const int T = steps_of(J, s);
                // step 0: S^T of the diagonal chunk (two contractions) and its dP^T
                wait(K_KFULL, nk); ++nk;
                q_wait(qb);
                q_wait(qb + 1);
                do_wait(db);
                tc_fence_after_sync();
                if (!ok) break;
                mma_kk(tmem + colS, smem_u32(sK), q_addr(qb), HD, idescT, false);
                {   // S^T -= Y^T Xq^T: Y as stored ([contraction][keys], MN-major), Xq K-major
                    const uint32_t a_lo = umma_desc_lo(do_addr(db), kPanelBytes), b_lo = umma_desc_lo(q_addr(qb + 1), 16);
#pragma unroll
                    for (int kk = 0; kk < kTile / 16; ++kk)
                        umma_ss(tmem + colS, umma_desc_join(a_lo + kk * 128u),
                                umma_desc_join(b_lo + (uint32_t)(kk >> 2) * (kPanelBytes >> 4) + (uint32_t)(kk & 3) * 2u),
                                umma_idesc(128, 128, 1, 0) | (1u << 13), 1u);
                }
                umma_commit(&bars[K_SFULL]);
                umma_commit(&bars[K_QEMPTY + qb % 3]);         // raw q and the two correction operands are only needed here
                umma_commit(&bars[K_QEMPTY + (qb + 1) % 3]);
                umma_commit(&bars[K_DOEMPTY + (db & 1)]);
                umma_commit(&bars[K_KEMPTY]);                  // raw k as well: step 1 uses a key version
                wait(K_VFULL, nv); ++nv;
                do_wait(db + 1);
                tc_fence_after_sync();
                if (!ok) break;
                mma_kk(tmem + colDP, smem_u32(sV), do_addr(db + 1), HD, idescT, false);
                umma_commit(&bars[K_DPFULL]);
                if (T == 1) umma_commit(&bars[K_VEMPTY]);
#pragma unroll 1
                for (int t = 0; t < T && ok; ++t) {
                    const int l = level(t);
                    const int qe = qb + (t == 0 ? 0 : t + 1), de = db + 1 + t;
                    // dV += P^T dO; the first product of an item overwrites the accumulators the previous item's
                    // write-out must have read
                    wait(K_PFULL, g + t);
                    if (t == 0 && it > 0) wait(K_ACCFREE, it - 1);
                    tc_fence_after_sync();
                    if (!ok) break;
                    mma_tn(tmem + colDV, tmem + colS, do_addr(de), idescD, t > 0);
                    umma_commit(&bars[K_DOEMPTY + (de & 1)]);
                    // S^T of the next step overwrites P^T: in-order execution puts it after the product above
                    if (t + 1 < T) {
                        const int l1 = level(t + 1);
                        if (l1 != l) { wait(K_KFULL, nk); ++nk; }
                        q_wait(qb + t + 2);
                        tc_fence_after_sync();
                        if (!ok) break;
                        mma_kk(tmem + colS, smem_u32(sK), q_addr(qb + t + 2), HD, idescT, false);
                        umma_commit(&bars[K_SFULL]);
                        if (t + 2 >= T || level(t + 2) != l1) umma_commit(&bars[K_KEMPTY]);
                    }
                    // dK += dS^T Q
                    wait(K_DSFULL, g + t);
                    tc_fence_after_sync();
                    if (!ok) break;
                    if (t > 0) {
                        mma_tn(tmem + colDK, tmem + colDP, q_addr(qe), idescD, !(t == 1 || l != level(t - 1)));
                        umma_commit(&bars[K_QEMPTY + qe % 3]);
                    }
                    if (t + 1 < T) {
                        do_wait(de + 1);
                        tc_fence_after_sync();
                        if (!ok) break;
                        mma_kk(tmem + colDP, smem_u32(sV), do_addr(de + 1), HD, idescT, false);
                        umma_commit(&bars[K_DPFULL]);
                        if (t + 2 == T) umma_commit(&bars[K_VEMPTY]);   // that was the item's last use of V
                    } else {
                        umma_commit(&bars[K_ACCFULL]);
                    }
                }
                g += T; qb += T + 1; db += T + 1;
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
        const int q4 = warp & 3, h = (warp - 4) >> 2, row = q4 * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)(q4 * 32) << 16);
        const float sl2 = p.scale * kLog2e;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        uint64_t ngj2 = 0;
        float dsum = 0.f;
        bool ok = true;
        int g = 0;                               // steps before the current item
        constexpr int CW = HD / 2;               // accumulator columns per thread when flushing
        auto flush_dk = [&](int lvl) {   // the version's gradient leaves as bf16, the form the version chain rule multiplies
            store_acc_bf16<CW>(p.dkv + ((size_t)krow(lvl, J) + row) * HD + h * CW, tlane + colDK + h * CW, p.scale);
        };
        auto step = [&](auto first_tag, const int t) {
            constexpr bool FIRST = decltype(first_tag)::value;   // the diagonal chunk: causal mask, dS^T written out
            const int gs = g + t;                                // running step number: ring slot and phase
            const float* st_ = rowstat + (gs & 1) * 2 * kTile;   // [0,128): -lse2 (+gate), [128,256): -delta of the queries
            const int c0 = h * 64;               // query columns of this thread
            uint32_t pr[2][32];                  // S^T, then P^T (float bits)
            // ---- part A: P^T = exp2(S^T * scale - lse)
            if (ok && !mbar_wait(&bars[K_STFULL + (gs & 1)], (gs >> 1) & 1, abort_flag, ST_DKV_COMPUTE)) ok = false;
            if (ok && !mbar_wait(&bars[K_SFULL], gs & 1, abort_flag, ST_DKV_COMPUTE)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            if (ok) {
                tmem_ld32(tlane + colS + c0, pr[0]);
                tmem_ld32(tlane + colS + c0 + 32, pr[1]);
                tmem_ld_wait();
                uint32_t pk[32];
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int x = 0; x < 32; x += 4) {
                        const float4 ls = *reinterpret_cast<const float4*>(st_ + c0 + c * 32 + x);
                        uint64_t v01 = fma2(pack2(__uint_as_float(pr[c][x]), __uint_as_float(pr[c][x + 1])), sl2x2, pack2(ls.x, ls.y));
                        uint64_t v23 = fma2(pack2(__uint_as_float(pr[c][x + 2]), __uint_as_float(pr[c][x + 3])), sl2x2, pack2(ls.z, ls.w));
                        if (GATE) { v01 = add2(v01, ngj2); v23 = add2(v23, ngj2); }
                        float e[4];
                        unpack2(v01, e[0], e[1]);
                        unpack2(v23, e[2], e[3]);
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            e[y] = ex2(e[y]);
                            if (FIRST && c0 + c * 32 + x + y < row) e[y] = 0.f;
                            pr[c][x + y] = __float_as_uint(e[y]);
                        }
                        pk[c * 16 + (x >> 1)] = pack_bf16(e[0], e[1]);
                        pk[c * 16 + (x >> 1) + 1] = pack_bf16(e[2], e[3]);
                    }
                tmem_st32(tlane + colS + c0, pk);
                tmem_st_wait();
            }
            tc_fence_before_sync();
            mbar_arrive(&bars[K_PFULL]);
            // ---- part B: dS^T = P^T o (dP^T - delta)
            if (ok && !mbar_wait(&bars[K_DPFULL], gs & 1, abort_flag, ST_DKV_COMPUTE)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            // dP^T ready means every product issued before it has retired: dK of a finished level can be flushed
            if (!FIRST && ok && t >= 2 && level(t) != level(t - 1)) flush_dk(level(t - 1));
            uint32_t dsw[FIRST ? 32 : 1];   // this thread's 64 entries of the transposed diagonal tile
            if (ok) {
                const float* dl_ = st_ + kTile;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t dp[32], pk[16];
                    tmem_ld32(tlane + colDP + c0 + c * 32, dp);
                    tmem_ld_wait();
#pragma unroll
                    for (int x = 0; x < 32; x += 4) {
                        const float4 dl = *reinterpret_cast<const float4*>(dl_ + c0 + c * 32 + x);
                        const uint64_t d01 = mul2(pack2(__uint_as_float(pr[c][x]), __uint_as_float(pr[c][x + 1])),
                                                  add2(pack2(__uint_as_float(dp[x]), __uint_as_float(dp[x + 1])), pack2(dl.x, dl.y)));
                        const uint64_t d23 = mul2(pack2(__uint_as_float(pr[c][x + 2]), __uint_as_float(pr[c][x + 3])),
                                                  add2(pack2(__uint_as_float(dp[x + 2]), __uint_as_float(dp[x + 3])), pack2(dl.z, dl.w)));
                        float d[4];
                        unpack2(d01, d[0], d[1]);
                        unpack2(d23, d[2], d[3]);
                        if (GATE) dsum += (d[0] + d[1]) + (d[2] + d[3]);
                        pk[x >> 1] = pack_bf16(d[0], d[1]);
                        pk[(x >> 1) + 1] = pack_bf16(d[2], d[3]);
                        if (FIRST) {   // (scale * dS)^T of the diagonal chunk for the chain rule; and float32 row sums if gated
                            dsw[c * 16 + (x >> 1)] = pack_bf16(d[0] * p.scale, d[1] * p.scale);
                            dsw[c * 16 + (x >> 1) + 1] = pack_bf16(d[2] * p.scale, d[3] * p.scale);
                            if (GATE) {
#pragma unroll
                                for (int y = 0; y < 4; ++y) dp[x + y] = __float_as_uint(d[y]);
                            }
                        }
                    }
                    tmem_st16(tlane + colDP + c0 + c * 16, pk);
                    if (FIRST && GATE) {   // row sums of dS over this warp's 32 keys: lane q of the warp ends up with query column q
#pragma unroll
                        for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
                            for (int x = 0; x < off; ++x) {
                                const bool up = lane & off;
                                const float keep = __uint_as_float(up ? dp[x + off] : dp[x]), give = __uint_as_float(up ? dp[x] : dp[x + off]);
                                dp[x] = __float_as_uint(keep + __shfl_xor_sync(0xffffffffu, give, off));
                            }
                        p.dsd[((size_t)(s * p.N + J) * 4 + q4) * kTile + c0 + c * 32 + lane] = __uint_as_float(dp[0]);
                    }
                }
                tmem_st_wait();
            }
            tc_fence_before_sync();
            mbar_arrive(&bars[K_DSFULL]);
            mbar_arrive(&bars[K_STEMPTY + (gs & 1)]);
            if constexpr (FIRST) {   // rows = keys (this warp's 32 lanes), 64 query columns = 128 bytes per row
                if (ok)
                    warp_store_rows128<false>(p.dsdt + ((size_t)(s * p.N + J) * kTile + q4 * 32) * kTile + h * 64, (size_t)kTile * 2,
                                       dsw);
            }
        };
#pragma unroll 1
        for (int it = 0; item_of(it, J, s); ++it) {
            const int T = steps_of(J, s);
            const int kj = J * kTile + row;          // key position of this thread's row
            if (GATE) {
                const float gj2 = p.G[(size_t)s * p.Lp + kj] * kLog2e;
                ngj2 = pack2(-gj2, -gj2);
                dsum = 0.f;
            }
            step(std::true_type{}, 0);
#pragma unroll 1
            for (int t = 1; t < T; ++t) step(std::false_type{}, t);
            g += T;
            if (ok && !mbar_wait(&bars[K_ACCFULL], it & 1, abort_flag, ST_DKV_COMPUTE)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            if (GATE) {   // the two threads of a key row add their halves of the column sum
                if (h == 1) dsum_x[row] = dsum;
                ok = barrier_and<1, 256>(ok);   // (all warps leave below, or none)
                if (h == 0 && ok) p.dG[(size_t)s * p.Lp + kj] = -(dsum + dsum_x[row]);
                { __syncwarp(); asm volatile("bar.sync 1, 256;" ::: "memory"); }
            }
            if (!ok) {
                mbar_arrive(&bars[K_ACCFREE]);
                break;
            }
            auto zero_dk = [&]() {
                uint4* dst = reinterpret_cast<uint4*>(p.dkv + ((size_t)row0(J) + row) * HD + h * CW);
                for (int x = 0; x < CW / 8; ++x) dst[x] = make_uint4(0u, 0u, 0u, 0u);
            };
            if (T > 1) flush_dk(level(T - 1));
            else zero_dk();   // no later query chunk met: the boundary-adjusted keys get a zero gradient from the sweep
            // (levels that a sweep shortened by block skipping did not reach stay unwritten: the version chain rule starts
            // at the highest level reached)
            if (CW == 64) {   // 64 bf16 = one 128-byte line per row: coalesced exchange
                uint32_t r0[32], r1[32], w[32];
                tmem_ld32(tlane + colDV + h * CW, r0);
                tmem_ld32(tlane + colDV + h * CW + 32, r1);
                tmem_ld_wait();
                tc_fence_before_sync();
                mbar_arrive(&bars[K_ACCFREE]);   // both accumulators have been read
#pragma unroll
                for (int x = 0; x < 16; ++x) {
                    w[x] = pack_bf16(__uint_as_float(r0[2 * x]), __uint_as_float(r0[2 * x + 1]));
                    w[16 + x] = pack_bf16(__uint_as_float(r1[2 * x]), __uint_as_float(r1[2 * x + 1]));
                }
                const int row0 = J * kTile + q4 * 32;
                warp_store_rows128<true>((__nv_bfloat16*)p.dv + ((size_t)s * p.L + row0) * HD + h * CW, (size_t)HD * 2, w,
                                   p.L - row0);
            } else {
                uint32_t r[32];
                tmem_ld32(tlane + colDV + h * CW, r);
                tmem_ld_wait();
                tc_fence_before_sync();
                mbar_arrive(&bars[K_ACCFREE]);
                if (kj < p.L) {
                    uint4* dst = reinterpret_cast<uint4*>((__nv_bfloat16*)p.dv + ((size_t)s * p.L + kj) * HD + h * CW);
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        dst[x] = make_uint4(pack_bf16(__uint_as_float(r[8 * x]), __uint_as_float(r[8 * x + 1])),
                                            pack_bf16(__uint_as_float(r[8 * x + 2]), __uint_as_float(r[8 * x + 3])),
                                            pack_bf16(__uint_as_float(r[8 * x + 4]), __uint_as_float(r[8 * x + 5])),
                                            pack_bf16(__uint_as_float(r[8 * x + 6]), __uint_as_float(r[8 * x + 7])));
                }
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, p.status);
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------------------------ dQ
// Persistent like the dK/dV sweep: items are the query chunks of a slice, paired (longest, shortest).  The steps of all
// items of a CTA form one sequence.  Round i of the elementwise warps does part A of step i and part B of step i - 1 in one
// pass over 16 columns at a time, so that exponentials, products and tensor-memory traffic of two steps share the issue
// slots: one after the other they took 1600 + 1200 cycles of which the exponentials alone are 1024.  What a round needs is
// produced while the previous one runs: S(i) alternates between two tiles, dP(i - 1) is released as soon as every thread
// has it in registers, and dS(i - 1) goes into the columns of S(i) that its thread has just read.  Everything else is kept
// out of these warps: the K producer describes each step in shared memory, four more warps write finished levels out.
// 8 x 16 x 2048 x 64: 150 -> 123 us (a round takes 2050 cycles, 1290 of them the pass itself); 4 x 16 x 4096 x 128: 342 ->
// 314 us, where the products alone are 1560 of 2500 cycles a round and the power limit is reached.
// Warps: 0 = producer of Q, K, gate prefix and step descriptions, 1 = tcgen05 issue of S and dQ, 2 = producer of dO and V,
// 3 = tcgen05 issue of dP, 4-11 = elementwise math, 12-15 = write-out.
enum { Q_QFULL = 0, Q_QEMPTY = 2, Q_DOFULL = 4, Q_DOEMPTY = 6, Q_KFULL = 8, Q_KEMPTY = Q_KFULL + 6, Q_VFULL = Q_KEMPTY + 6,
       Q_VEMPTY = Q_VFULL + 4, Q_GKEMPTY = Q_VEMPTY + 4, Q_READY = Q_GKEMPTY + 2, Q_DPFREE = Q_READY + 2, Q_ROUND, Q_ACCFULL = Q_ROUND + 2,
       Q_ACCFREE, Q_SUM, Q_COUNT = Q_SUM + 3 };
constexpr uint32_t kDqDesc = 7 * kSlotBytes + 336;            // [8] step descriptions
constexpr uint32_t kDqGk = kDqDesc + 8 * 16;                  // [2][128] gate prefix of the key chunk, [3][128] row sums of an item
constexpr uint32_t kDqTotal = kDqGk + 5 * kTile * 4;
static_assert(Q_COUNT * 8 + 8 <= 336 && kDqTotal <= kSmemAlloc, "shared memory of the dQ sweep");

// A CTA's steps one after the other: items come from `item_of(k, chunk, slice)`, their step counts from
// `steps_of(chunk, slice)`, fetched one item ahead; `skipped(chunk, slice)` sees the items without a step.
template <class ItemOf, class StepsOf, class Skipped>
struct Flow {
    ItemOf item_of;
    StepsOf steps_of;
    Skipped skipped;
    int c = 0, s = 0, t = -1, T = 0;              // current step: chunk, slice, step t of T
    int nc = 0, ns = 0, nT = 0, k = 0;            // the next item with steps, if there is one
    bool more;
    __device__ Flow(ItemOf io, StepsOf so, Skipped sk) : item_of(io), steps_of(so), skipped(sk) { fetch(); }
    __device__ void fetch() {
        while ((more = item_of(k++, nc, ns))) {
            nT = steps_of(nc, ns);
            if (nT > 0) break;
            skipped(nc, ns);
        }
    }
    __device__ bool next() {
        if (++t < T) return true;
        if (!more) return false;
        c = nc; s = ns; T = nT; t = 0;
        fetch();
        return true;
    }
};
template <class ItemOf, class StepsOf, class Skipped>
__device__ __forceinline__ Flow<ItemOf, StepsOf, Skipped> make_flow(ItemOf io, StepsOf so, Skipped sk) {
    return Flow<ItemOf, StepsOf, Skipped>(io, so, sk);
}
template <class ItemOf, class StepsOf>
__device__ __forceinline__ auto make_flow(ItemOf io, StepsOf so) { return make_flow(io, so, [](int, int) {}); }
enum { FL_VALID = 1, FL_FIRST = 2, FL_LAST = 4, FL_LVL0 = 8, FL_LVL1 = 16 };   // a step: first / last of its item / of a level

template <int N>
__device__ __forceinline__ void set_fewer_regs() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void set_more_regs() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
// Waits for this thread's tensor-memory loads; nothing that uses r may be moved in front of it.
__device__ __forceinline__ void tmem_ld_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// D[tmem] (+)= A B with A in tensor memory: the 16 contraction indices of step kk in the 8 columns at a_col + 16 kk.
__device__ __forceinline__ void mma_t16(uint32_t d_tmem, uint32_t a_col, uint32_t b0, uint32_t idesc, bool acc) {
    uint32_t b_lo = umma_desc_lo(b0, kPanelBytes);
#pragma unroll 2
    for (int kk = 0; kk < kTile / 16; ++kk) {
        umma_ts(d_tmem, a_col + kk * 16, umma_desc_join(b_lo), idesc, (acc || kk > 0) ? 1u : 0u);
        b_lo += 128u;
    }
}

template <int HD, bool GATE>
__global__ void __launch_bounds__(512, 1) dq_kernel(const __grid_constant__ BwdTensorMaps tm, const BwdParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    if ((uint32_t)(smem - smem_raw) + kDqTotal > kSmemAlloc) {   // uniform over the CTA
        grid_wait();   // (the status word belongs to the kernels before)
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)ST_DQ_PRODUCER);
        return;
    }
    // Tiles in flight.  K is needed from S(i + 2) to dQ(i - 1), four steps; V only for dP.
    constexpr int NQ = HD == 64 ? 2 : 1, NDO = NQ, NK = HD == 64 ? 6 : 4, NV = HD == 64 ? 4 : 1;
    constexpr uint32_t kBytes = kTile * HD * 2;
    // Registers.  Without a gate a math thread fetches its 64 columns of dP at once, so that the next dP can start early, and a
    // level is written out 32 columns at a time.  With one (more live values, and with block skipping a level may be one step
    // long) dP comes 16 columns at a time and a level is read whole, so that the next one can start.  dQ sweep, us, early / late:
    // d = 128, 4 x 16 x 4096 ungated 316 / 361; 2 x 16 x 8192 gated 154 / 144;  d = 64, 8 x 16 x 2048 ungated 121 / 146.
    constexpr bool EARLY = !GATE;
    constexpr int kRegsMath = EARLY ? 200 : 168, kRegsOut = EARLY ? 56 : 112, kRegsIssue = EARLY ? 56 : 64;
    static_assert(256 * kRegsMath + 128 * (kRegsOut + kRegsIssue) <= 65536, "no more than the block was launched with");
    static_assert((NQ + NDO + NK + NV) * kBytes == 7 * kSlotBytes, "tiles fill the 7 slots");
    uint8_t* sQ = smem;
    uint8_t* sDO = sQ + NQ * kBytes;
    uint8_t* sK = sDO + NDO * kBytes;
    uint8_t* sV = sK + NK * kBytes;
    uint64_t* bars = (uint64_t*)(smem + 7 * kSlotBytes);
    uint32_t* tmem_slot = (uint32_t*)(bars + Q_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    int4* desc = (int4*)(smem + kDqDesc);   // flags, first row of the query chunk, -, the same of the next item (-1: none)
    float* gk = (float*)(smem + kDqGk);
    float* dsum_x = gk + 2 * kTile;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = p.N * p.S;

    if (threadIdx.x == 0) {
        for (int i = 0; i < Q_COUNT; ++i)
            mbar_init(&bars[i], i == Q_READY || i == Q_READY + 1 ? 3u
                              : i == Q_DPFREE || i == Q_ROUND || i == Q_ROUND + 1 || i == Q_GKEMPTY || i == Q_GKEMPTY + 1 ? 256u
                              : i >= Q_SUM ? 256u : i == Q_ACCFREE ? 128u : 1u);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (GATE && threadIdx.x < 3 * kTile) dsum_x[threadIdx.x] = 0.f;
    if (warp == 3 && lane < 8) tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&tm) + lane);
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    constexpr uint32_t colS = 0, colDP = 256, colDQ = 384;   // two S tiles at 0 and 128
    // k-th work item of this CTA; query chunk I has I steps (t = 0..I-1, key chunk J = I-1-t)
    auto item_of = [&](int k, int& I, int& s) {
        const int w = 2 * ((int)blockIdx.x + (k >> 1) * (int)gridDim.x) + (k & 1);
        if (w >= items) return false;
        s = w / p.N;
        const int j = w % p.N;
        I = (j & 1) ? (j >> 1) : p.N - 1 - (j >> 1);
        return true;
    };
    // earlier key chunks this query chunk visits (J = I-1 .. I-T): all of them, or fewer when the gate has made the far
    // ones negligible (every warp role reads the same precomputed number; the diagonal chunk is not part of this sweep)
    auto steps_of = [&](int I, int s) { return p.nkeep ? min(I, p.nkeep[s * p.N + I] - 1) : I; };
    auto level = [](int I, int t) { return msb32((unsigned)(I ^ (I - 1 - t))); };
    auto flags_of = [](int I, int t, int T, int l) {   // level l covers the key chunks whose low l bits run from all ones down to zero
        const int J = I - 1 - t, m = (1 << l) - 1, last = t + 1 == T;
        return FL_VALID | (t == 0 ? FL_FIRST : 0) | (last ? FL_LAST : 0) | ((J & m) == m ? FL_LVL0 : 0) |
               (last || (J & m) == 0 ? FL_LVL1 : 0);
    };

    if (warp < 4) {
        set_fewer_regs<kRegsIssue>();
        if (warp == 0 && elect_one()) {
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            int nq = 0, n = 0;   // Q tiles, steps so far
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_DQ_PRODUCER)) ok = false;
                return ok;
            };
#pragma unroll 1
            for (; ok; ++n) {
                const bool more = flow.next();
                // K(n - NK) is released after round n - NK + 1, past the last look at description n - 8
                if (!wait_empty(Q_KEMPTY + n % NK, n / NK)) break;
                if (!more) {
                    desc[n & 7] = make_int4(0, 0, 0, -1);
                    mbar_arrive(&bars[Q_KFULL + n % NK]);
                    break;
                }
                const int I = flow.c, s = flow.s, J = I - 1 - flow.t, l = level(I, flow.t), f = flags_of(I, flow.t, flow.T, l);
                desc[n & 7] = make_int4(f, s * p.Lp + I * kTile, 0, flow.more ? flow.ns * p.Lp + flow.nc * kTile : -1);
                mbar_expect_tx(&bars[Q_KFULL + n % NK], kBytes + (GATE ? kTile * 4 : 0));
                tma_tile(sK + (n % NK) * kBytes, &tm.kv, &bars[Q_KFULL + n % NK], HD, (int)kver_row(p.vl, s, l, J));
                if (f & FL_LVL0) {
                    const int b = nq % NQ;
                    if (!wait_empty(Q_QEMPTY + b, nq / NQ)) break;
                    mbar_expect_tx(&bars[Q_QFULL + b], kBytes);
                    tma_tile(sQ + b * kBytes, &tm.qv, &bars[Q_QFULL + b], HD, (int)qver_row(p.vl, s, l, I));
                    ++nq;
                }
                if (GATE) {   // gate prefix of the key chunk (counted with K)
                    if (!wait_empty(Q_GKEMPTY + (n & 1), n >> 1)) break;
                    bulk_load(gk + (n & 1) * kTile, p.G + (size_t)s * p.Lp + J * kTile, kTile * 4, &bars[Q_KFULL + n % NK]);
                }
            }
        } else if (warp == 2 && elect_one()) {
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            int nd = 0;
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_DQ_PRODUCER)) ok = false;
                return ok;
            };
#pragma unroll 1
            for (int n = 0; flow.next(); ++n) {
                if (flow.t == 0) {
                    const int b = nd % NDO;
                    if (!wait_empty(Q_DOEMPTY + b, nd / NDO)) break;
                    mbar_expect_tx(&bars[Q_DOFULL + b], kBytes);
                    tma_rows(sDO + b * kBytes, &tm.d_o, &bars[Q_DOFULL + b], HD, flow.c * kTile, flow.s);
                    ++nd;
                }
                if (!wait_empty(Q_VEMPTY + n % NV, n / NV)) break;
                mbar_expect_tx(&bars[Q_VFULL + n % NV], kBytes);
                tma_rows(sV + (n % NV) * kBytes, &tm.v, &bars[Q_VFULL + n % NV], HD, (flow.c - 1 - flow.t) * kTile, flow.s);
            }
        } else if (warp == 1 && elect_one()) {
            constexpr uint32_t idescS = umma_idesc(128, 128, 0, 0);
            constexpr uint32_t idescD = umma_idesc(128, HD, 0, 1);
            bool ok = true;
            int nq = 0, na = 0;   // Q tiles so far, levels finished so far
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_DQ_MMA)) ok = false;
                return ok;
            };
            // S of step g; returns the step's flags, 0 after the last one.  A round begins on three arrivals: S, dP, and one
            // that hands the description on.
            auto issue_s = [&](int g) {
                if (!wait(Q_KFULL + g % NK, g / NK)) return 0;
                const int f = desc[g & 7].x;
                if (f) {
                    if (f & FL_LVL0) { wait(Q_QFULL + nq % NQ, nq / NQ); ++nq; }
                    const int b = (nq - 1) % NQ;
                    tc_fence_after_sync();
                    if (!ok) return 0;
                    mma_kk(tmem + colS + (g & 1) * 128, smem_u32(sQ + b * kBytes), smem_u32(sK + (g % NK) * kBytes), HD, idescS, false);
                    umma_commit(&bars[Q_READY + (g & 1)]);
                    if (f & FL_LVL1) umma_commit(&bars[Q_QEMPTY + b]);
                } else {   // the last round has no S: its tile is free once dQ(g - 3) has retired
                    umma_commit(&bars[Q_READY + (g & 1)]);
                }
                mbar_arrive(&bars[Q_READY + (g & 1)]);
                return f;
            };
            int fm = 0, f0 = issue_s(0), f1 = f0 ? issue_s(1) : 0;   // steps i - 1, i, i + 1
            if (ok) mbar_arrive(&bars[Q_READY]);                     // (no dP before round 0)
#pragma unroll 1
            for (int i = 0; ok && (f0 | fm); ++i) {
                if (!wait(Q_ROUND + (i & 1), i >> 1)) break;
                if (fm) {                    // dQ (+)= dS(i - 1) K
                    if ((fm & FL_LVL0) && na > 0 && !wait(Q_ACCFREE, na - 1)) break;   // the previous level has been read
                    tc_fence_after_sync();
                    mma_t16(tmem + colDQ, tmem + colS + (i & 1) * 128, smem_u32(sK + ((i - 1) % NK) * kBytes), idescD, !(fm & FL_LVL0));
                    umma_commit(&bars[Q_KEMPTY + (i - 1) % NK]);
                    if (fm & FL_LVL1) { umma_commit(&bars[Q_ACCFULL]); ++na; }
                }
                // in-order execution keeps S(i + 2) behind the product that reads dS(i - 1) from the same tile
                const int f2 = f1 ? issue_s(i + 2) : 0;
                fm = f0; f0 = f1; f1 = f2;
            }
        } else if (warp == 3 && elect_one()) {
            // dP has an issuing thread of its own: its waits and those for S and dQ are not paid one after the other
            constexpr uint32_t idescS = umma_idesc(128, 128, 0, 0);
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_DQ_MMA)) ok = false;
                return ok;
            };
#pragma unroll 1
            for (int i = 0, nd = 0; flow.next(); ++i) {
                if (flow.t == 0) { wait(Q_DOFULL + nd % NDO, nd / NDO); ++nd; }
                const int b = (nd - 1) % NDO;
                wait(Q_VFULL + i % NV, i / NV);
                if (i > 0) wait(Q_DPFREE, i - 1);   // every thread holds dP(i - 1)
                tc_fence_after_sync();
                if (!ok) break;
                mma_kk(tmem + colDP, smem_u32(sDO + b * kBytes), smem_u32(sV + (i % NV) * kBytes), HD, idescS, false);
                umma_commit(&bars[Q_READY + ((i + 1) & 1)]);
                umma_commit(&bars[Q_VEMPTY + i % NV]);
                if (flow.t + 1 == flow.T) umma_commit(&bars[Q_DOEMPTY + b]);
            }
        }
    } else if (warp >= 12) {
        // ---------------------------------------------------------------- write-out of finished levels, one row per thread
        set_fewer_regs<kRegsOut>();
        const int row = (warp & 3) * 32 + lane;
        const uint32_t tacc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + colDQ;
        // no key chunk visited (chunk 0, or block skipping left only the diagonal): the boundary-adjusted queries get a
        // zero gradient from the sweep.  Levels that a shortened sweep does not reach stay unwritten: the version
        // chain rule starts at the highest level reached.
        auto zero_item = [&](int I, int s) {
            uint4* dst = reinterpret_cast<uint4*>(p.dqv + ((size_t)s * p.Lp + (size_t)I * kTile) * HD);
            for (int x = threadIdx.x - 384; x < kTile * HD / 8; x += 128) dst[x] = make_uint4(0u, 0u, 0u, 0u);
            if (GATE) p.dGrow[(size_t)s * p.Lp + I * kTile + row] = 0.f;
        };
        auto flow = make_flow(item_of, steps_of, zero_item);
#pragma unroll 1
        for (int na = 0, nsum = 0; flow.next();) {
            const int l = level(flow.c, flow.t), f = flags_of(flow.c, flow.t, flow.T, l);
            if (!(f & FL_LVL1)) continue;
            bool ok = mbar_wait(&bars[Q_ACCFULL], na & 1, abort_flag, ST_DQ_COMPUTE);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after_sync();
            __nv_bfloat16* dst = p.dqv + ((size_t)qver_row(p.vl, flow.s, l, flow.c) + row) * HD;
            constexpr int PIECES = EARLY ? 1 : HD / 32;   // of 32 columns, held at a time
#pragma unroll 1
            for (int c0 = 0; c0 < HD / 32; c0 += PIECES) {
                uint32_t w[PIECES][16];
#pragma unroll
                for (int c = 0; c < PIECES; ++c) {
                    float v[32];
                    tile::tmem_row32(tacc + (c0 + c) * 32, v);
#pragma unroll
                    for (int x = 0; x < 16; ++x) w[c][x] = pack_bf16(v[2 * x] * p.scale, v[2 * x + 1] * p.scale);
                }
                if (c0 + PIECES == HD / 32) {
                    if (GATE && (f & FL_LAST)) {   // before the accumulators are handed back: three items on, the buffer is in use again
                        const int buf = nsum % 3;
                        ok = mbar_wait(&bars[Q_SUM + buf], (nsum / 3) & 1, abort_flag, ST_DQ_COMPUTE);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        p.dGrow[(size_t)flow.s * p.Lp + flow.c * kTile + row] = dsum_x[buf * kTile + row];
                        dsum_x[buf * kTile + row] = 0.f;
                        ++nsum;
                    }
                    tc_fence_before_sync();
                    mbar_arrive(&bars[Q_ACCFREE]);
                }
#pragma unroll
                for (int c = 0; c < PIECES; ++c) tile::gstore_bf16_w16(dst + (c0 + c) * 32, w[c]);
            }
            ++na;
        }
    } else {
        set_more_regs<kRegsMath>();
        const int q4 = warp & 3, h = (warp - 4) >> 2, row = q4 * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)(q4 * 32) << 16) + h * 64;   // this thread's 64 key columns
        const float sl2 = p.scale * kLog2e;
        const uint64_t sl2x2 = pack2(sl2, sl2), nlog2 = pack2(-kLog2e, -kLog2e);
        float nl_n = 0.f, nd_n = 0.f, nd_a = 0.f;   // minus lse2 (plus gate prefix) and minus delta: next item; delta of A's row
        uint64_t nl2 = 0, nd2 = 0;               // of A's row, of B's row
        float dsum = 0.f;
        float pr[64];                            // P of step i - 1, then of step i
        int nsum = 0;
        // One round: part A of step i from its S tile, part B of step i - 1 into it.
        auto round = [&](auto a_tag, auto b_tag, const int i) {
            constexpr bool A = decltype(a_tag)::value, B = decltype(b_tag)::value;
            const uint32_t ts = tlane + colS + (i & 1) * 128;
            constexpr int DC = EARLY ? 4 : 2;          // 16-column pieces of dP held at a time
            uint32_t dp[DC][16], sv[2][16];
            if (B) {
#pragma unroll
                for (int c = 0; c < DC - (EARLY ? 0 : 1); ++c) tmem_ld16(tlane + colDP + c * 16, dp[c]);
            }
            if (A) tmem_ld16(ts, sv[0]);
            auto release_dp = [&]() {
                tc_fence_before_sync();
                mbar_arrive(&bars[Q_DPFREE]);
            };
            const float* g_ = gk + (i & 1) * kTile + h * 64;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (B && (c == 0 || !EARLY)) tmem_ld_wait16(dp[c % DC]);
                if (A) tmem_ld_wait16(sv[c & 1]);
                if (B && EARLY && c == 0) {
#pragma unroll
                    for (int x = 1; x < DC; ++x) tmem_ld_wait16(dp[x]);
                    release_dp();
                }
                if (B && !EARLY && c < 3) tmem_ld16(tlane + colDP + (c + 1) * 16, dp[(c + 1) % DC]);
                if (A && c < 3) tmem_ld16(ts + (c + 1) * 16, sv[(c + 1) & 1]);
                if (B && !EARLY && c == 3) release_dp();
                if (B) {   // dS = P o (dP - delta)
                    uint32_t pk[8];
#pragma unroll
                    for (int x = 0; x < 16; x += 2) {
                        const uint32_t* d_ = &dp[c % DC][x];
                        const uint64_t d01 = mul2(pack2(pr[c * 16 + x], pr[c * 16 + x + 1]),
                                                  add2(pack2(__uint_as_float(d_[0]), __uint_as_float(d_[1])), nd2));
                        float d0, d1;
                        unpack2(d01, d0, d1);
                        if (GATE) dsum += d0 + d1;
                        pk[x >> 1] = pack_bf16(d0, d1);
                    }
                    tmem_st8(ts + c * 16, pk);
                }
                if (A) {   // P = exp2(S * scale - lse)
#pragma unroll
                    for (int x = 0; x < 16; x += 4) {
                        const uint32_t* s_ = &sv[c & 1][x];
                        uint64_t v01 = fma2(pack2(__uint_as_float(s_[0]), __uint_as_float(s_[1])), sl2x2, nl2);
                        uint64_t v23 = fma2(pack2(__uint_as_float(s_[2]), __uint_as_float(s_[3])), sl2x2, nl2);
                        if (GATE) {
                            const float4 g4 = *reinterpret_cast<const float4*>(g_ + c * 16 + x);
                            v01 = fma2(pack2(g4.x, g4.y), nlog2, v01);
                            v23 = fma2(pack2(g4.z, g4.w), nlog2, v23);
                        }
                        float e[4];
                        unpack2(v01, e[0], e[1]);
                        unpack2(v23, e[2], e[3]);
#pragma unroll
                        for (int y = 0; y < 4; ++y) pr[c * 16 + x + y] = ex2(e[y]);
                    }
                }
            }
            if (B) tmem_st_wait();
            tc_fence_before_sync();
            // (two barriers: round i + 1 does not wait for the slowest warp of round i, round i + 2 does)
            mbar_arrive(&bars[Q_ROUND + (i & 1)]);
            if (GATE && A) mbar_arrive(&bars[Q_GKEMPTY + (i & 1)]);
        };
        int fb = 0;   // flags of step i - 1
#pragma unroll 1
        for (int i = 0;; ++i) {
            bool ok = mbar_wait(&bars[Q_READY + (i & 1)], (i >> 1) & 1, abort_flag, ST_DQ_COMPUTE);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after_sync();
            const int4 de = desc[i & 7];
            const int fa = de.x;
            if (fb & FL_FIRST) nd2 = pack2(nd_a, nd_a);
            if (fa & FL_FIRST) {   // this item's row constants were requested when the previous item began
                if (i == 0) { nl_n = p.lse2[de.y + row]; nd_n = p.delta[de.y + row]; }
                nl2 = pack2(nl_n, nl_n);
                nd_a = nd_n;
                if (de.w >= 0) { nl_n = p.lse2[de.w + row]; nd_n = p.delta[de.w + row]; }
            }
            if (fa) {
                if (fb) round(std::true_type{}, std::true_type{}, i);
                else round(std::true_type{}, std::false_type{}, i);
            } else {
                if (fb) round(std::false_type{}, std::true_type{}, i);
            }
            if (GATE && (fb & FL_LAST)) {   // the two threads of a row add their halves (two addends: in any order)
                const int buf = nsum++ % 3;
                atomicAdd(dsum_x + buf * kTile + row, dsum);
                mbar_arrive(&bars[Q_SUM + buf]);
                dsum = 0.f;
            }
            if (!fa) break;
            fb = fa;
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, p.status);
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------------------------ dK, dV for d = 64, no gate
// dkv_kernel's sweep in the rounds of dq_kernel: at d = 64 the accumulators leave room for two S^T tiles, and the products
// (1050 cycles a step) are not what bounds it.  Round i of the math warps turns S^T(i) into P^T(i) and forms dS^T(i - 1); of the 16
// columns of a group of S^T(i) P^T(i) takes the first 8 and dS^T(i - 1) the last 8.  A round takes 1900 cycles (4400 one half after
// the other), 2000 to 3000 more on the diagonal step, whose passes are fetched anew each time.  Then dK (+)= dS^T(i - 1) Q, dV (+)= P^T(i) dO
// and S^T(i + 2) into the same tile follow in order.
// Warps: 0 = producer of Q (ring of 4), K (2), Xq, row constants (4) and step descriptions, 1 = tcgen05 issue of S, dK and dV,
// 2 = producer of dO (ring of 4) and V, 3 = tcgen05 issue of dP, 4-11 = elementwise math, 12-15 = write-out.
// Y of a diagonal step takes two entries of the dO ring, in halves of 64 columns.  Ring sizes: S(i + 2) is issued before
// Q(i) is released, and dO(i + 1) is still held when Y of a step i + 2 has to be there.
enum { D_QFULL = 0, D_QEMPTY = 4, D_DOFULL = 8, D_DOEMPTY = 12, D_KFULL = 16, D_KEMPTY = 18, D_VFULL = 20, D_VEMPTY, D_XFULL, D_XEMPTY, D_STEMPTY,
       D_READY = D_STEMPTY + 4, D_DPFREE = D_READY + 2, D_ROUND, D_DKFULL = D_ROUND + 2, D_DKFREE, D_DVFULL, D_DVFREE, D_COUNT };
constexpr uint32_t kD64Tile = kTile * 64 * 2;
constexpr uint32_t kD64Bars = 13 * kD64Tile, kD64Desc = kD64Bars + 384, kD64Stat = kD64Desc + 8 * 8;
constexpr uint32_t kD64Total = kD64Stat + 4 * 2 * kTile * 4;
static_assert(D_COUNT * 8 + 8 <= 384 && kD64Total + 1024 <= kSmemAlloc, "shared memory of the d = 64 dK/dV sweep");

// Causal mask of a diagonal chunk: zeros in the first `n` of this thread's 64 entries of P^T (columns ts + 16 g .. + 7, two entries
// each), whatever their exponents were.  (Minus infinity in the logits beforehand is not enough: a row whose log-normaliser is
// NaN made dV of all later keys of its chunk NaN.)  A function of its own, so that the rounds' code does not grow: the sweep
// of 8 x 16 x 2048 x 64 takes 243 us like this, 250 with the pass unrolled in the round, 238 with the mask in the logits.
__device__ __noinline__ void mask_pt(uint32_t ts, int n) {
#pragma unroll 1
    for (int c = 0; c < 64; c += 16) {
        uint32_t m[16];
        tmem_ld16(ts + c, m);
        tmem_ld_wait16(m);
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            if (c + 2 * x < n) m[x] &= 0xffff0000u;
            if (c + 2 * x + 1 < n) m[x] &= 0x0000ffffu;
        }
        tmem_st16(ts + c, m);
    }
    tmem_st_wait();
}

__global__ void __launch_bounds__(512, 1) dkv64_kernel(const __grid_constant__ BwdTensorMaps tm, const BwdParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    constexpr int HD = 64, NQ = 4, ND = 4;
    uint8_t* sQ = smem;
    uint8_t* sDO = sQ + NQ * kD64Tile;
    uint8_t* sK = sDO + ND * kD64Tile;
    uint8_t* sV = sK + 2 * kD64Tile;
    uint8_t* sX = sV + kD64Tile;                  // two panels
    uint64_t* bars = (uint64_t*)(smem + kD64Bars);
    uint32_t* tmem_slot = (uint32_t*)(bars + D_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    int2* desc = (int2*)(smem + kD64Desc);        // flags, first row of the key chunk
    float* stat = (float*)(smem + kD64Stat);      // [4][2][128]: -lse2, -delta of the queries of a step

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = p.N * p.S;
    if (threadIdx.x == 0) {
        for (int i = 0; i < D_COUNT; ++i)
            mbar_init(&bars[i], i == D_READY || i == D_READY + 1 ? 3u
                              : i >= D_DOEMPTY && i < D_DOEMPTY + ND ? 2u        // dO serves dP and dV
                              : i == D_DPFREE || i == D_ROUND || i == D_ROUND + 1 || (i >= D_STEMPTY && i < D_READY) ? 256u
                              : i == D_DKFREE || i == D_DVFREE ? 128u : 1u);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 3 && lane < 8) tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&tm) + lane);
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    constexpr uint32_t colS = 0, colDP = 256, colDV = 384, colDK = 448;   // two S tiles at 0 and 128
    static_assert(256 * 200 + 256 * 56 <= 65536, "registers: no more than the block was launched with");
    // items and steps as in dkv_kernel
    auto item_of = [&](int k, int& J, int& s) {
        const int w = 2 * ((int)blockIdx.x + (k >> 1) * (int)gridDim.x) + (k & 1);
        if (w >= items) return false;
        s = w / p.N;
        const int j = w % p.N;
        J = (j & 1) ? p.N - 1 - (j >> 1) : (j >> 1);
        return true;
    };
    auto steps_of = [&](int J, int s) { return p.N - J; };
    auto level = [](int J, int t) { return msb32((unsigned)((J + t) ^ J)); };   // t >= 1
    auto flags_of = [](int J, int t, int T, int l) {   // level l covers the query chunks whose low l bits run from zero up to all ones
        const int I = J + t, m = (1 << l) - 1, last = t + 1 == T;
        if (t == 0) return FL_VALID | FL_FIRST | FL_LVL0 | FL_LVL1 | (last ? FL_LAST : 0);   // raw q and k: a level of its own
        return FL_VALID | (last ? FL_LAST : 0) | ((I & m) == 0 ? FL_LVL0 : 0) | (last || (I & m) == m ? FL_LVL1 : 0);
    };

    if (warp < 4) {
        set_fewer_regs<56>();
        if (warp == 0 && elect_one()) {
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            int nk = 0, nx = 0, n = 0;   // K tiles, items, steps (Q ring entries) so far
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_DKV_PRODUCER)) ok = false;
                return ok;
            };
#pragma unroll 1
            for (; ok; ++n) {
                const bool more = flow.next();
                if (!wait_empty(D_QEMPTY + n % NQ, n / NQ)) break;
                if (!more) {
                    desc[n & 7] = make_int2(0, 0);
                    mbar_arrive(&bars[D_QFULL + n % NQ]);
                    break;
                }
                const int J = flow.c, s = flow.s, I = J + flow.t, l = flow.t ? level(J, flow.t) : 0, f = flags_of(J, flow.t, flow.T, l);
                desc[n & 7] = make_int2(f, s * p.Lp + J * kTile);
                // the row constants of the step travel with Q
                const int sb = n & 3, q0 = n % NQ;
                mbar_expect_tx(&bars[D_QFULL + q0], kD64Tile + 2 * kTile * 4);
                if (f & FL_FIRST) tma_rows(sQ + q0 * kD64Tile, &tm.q_raw, &bars[D_QFULL + q0], HD, J * kTile, s);
                else tma_tile(sQ + q0 * kD64Tile, &tm.qv, &bars[D_QFULL + q0], HD, (int)qver_row(p.vl, s, l, I));
                if (!wait_empty(D_STEMPTY + sb, n >> 2)) break;
                const size_t gi = (size_t)s * p.Lp + I * kTile;
                bulk_load(stat + sb * 2 * kTile, p.lse2 + gi, kTile * 4, &bars[D_QFULL + q0]);
                bulk_load(stat + sb * 2 * kTile + kTile, p.delta + gi, kTile * 4, &bars[D_QFULL + q0]);
                if (f & FL_LVL0) {
                    const int b = nk & 1;
                    if (!wait_empty(D_KEMPTY + b, nk >> 1)) break;
                    mbar_expect_tx(&bars[D_KFULL + b], kD64Tile);
                    if (f & FL_FIRST) tma_rows(sK + b * kD64Tile, &tm.k_raw, &bars[D_KFULL + b], HD, J * kTile, s);
                    else tma_tile(sK + b * kD64Tile, &tm.kv, &bars[D_KFULL + b], HD, (int)kver_row(p.vl, s, l, J));
                    ++nk;
                }
                if (f & FL_FIRST) {
                    if (!wait_empty(D_XEMPTY, nx)) break;
                    mbar_expect_tx(&bars[D_XFULL], 2 * kD64Tile);
                    tma_tile(sX, &tm.xq, &bars[D_XFULL], kTile, s * p.Lp + J * kTile);
                    ++nx;
                }
            }
        } else if (warp == 2 && elect_one()) {
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            int dn = 0, nv = 0;
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_DKV_PRODUCER)) ok = false;
                return ok;
            };
            auto entry = [&]() { return wait_empty(D_DOEMPTY + dn % ND, dn / ND); };
#pragma unroll 1
            while (ok && flow.next()) {
                const int J = flow.c, s = flow.s;
                if (flow.t == 0) {
                    if (dn & 1) {   // the halves of Y lie one after the other: an entry is left out
                        if (!entry()) break;
                        mbar_arrive(&bars[D_DOFULL + dn % ND]);
                        ++dn;
                    }
                    for (int h = 0; h < 2; ++h, ++dn) {
                        if (!entry()) break;
                        mbar_expect_tx(&bars[D_DOFULL + dn % ND], kD64Tile);
                        tma_load_2d(sDO + (dn % ND) * kD64Tile, &tm.y, &bars[D_DOFULL + dn % ND], h * 64, s * p.Lp + J * kTile);
                    }
                    if (!wait_empty(D_VEMPTY, nv)) break;
                    mbar_expect_tx(&bars[D_VFULL], kD64Tile);
                    tma_rows(sV, &tm.v, &bars[D_VFULL], HD, J * kTile, s);
                    ++nv;
                }
                if (!entry()) break;
                mbar_expect_tx(&bars[D_DOFULL + dn % ND], kD64Tile);
                tma_rows(sDO + (dn % ND) * kD64Tile, &tm.d_o, &bars[D_DOFULL + dn % ND], HD, (J + flow.t) * kTile, s);
                ++dn;
            }
        } else if (warp == 1 && elect_one()) {
            constexpr uint32_t idescT = umma_idesc(128, 128, 0, 0);
            constexpr uint32_t idescD = umma_idesc(128, HD, 0, 1);
            bool ok = true;
            int dn = 0, nk = 0, nx = 0, ndk = 0, ndv = 0;   // entries of the dO ring, K tiles, items, levels and items finished so far
            int d2 = 0;                                     // ring entry of dO of the step that issue_s looked at last
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_DKV_MMA)) ok = false;
                return ok;
            };
            // S^T of step g; returns its flags, 0 after the last step (see dq_kernel)
            auto issue_s = [&](int g) {
                if (!wait(D_QFULL + g % NQ, g / NQ)) return 0;
                const int f = desc[g & 7].x;
                if (f) {
                    if (f & FL_LVL0) { wait(D_KFULL + (nk & 1), nk >> 1); ++nk; }
                    const int kb = (nk - 1) & 1;
                    if (f & FL_FIRST) {
                        if (dn & 1) {
                            wait(D_DOFULL + dn % ND, dn / ND);
                            mbar_arrive(&bars[D_DOEMPTY + dn % ND]);
                            mbar_arrive(&bars[D_DOEMPTY + dn % ND]);
                            ++dn;
                        }
                        for (int h = 0; h < 2; ++h) wait(D_DOFULL + (dn + h) % ND, (dn + h) / ND);
                        wait(D_XFULL, nx);
                        ++nx;
                    }
                    tc_fence_after_sync();
                    if (!ok) return 0;
                    mma_kk(tmem + colS + (g & 1) * 128, smem_u32(sK + kb * kD64Tile), smem_u32(sQ + (g % NQ) * kD64Tile), HD, idescT, false);
                    if (f & FL_FIRST) {   // S^T -= Y^T Xq^T: Y as stored ([contraction][keys], MN-major), Xq K-major
                        const uint32_t a_lo = umma_desc_lo(smem_u32(sDO + (dn % ND) * kD64Tile), kPanelBytes), b_lo = umma_desc_lo(smem_u32(sX), 16);
#pragma unroll
                        for (int kk = 0; kk < kTile / 16; ++kk)
                            umma_ss(tmem + colS + (g & 1) * 128, umma_desc_join(a_lo + kk * 128u),
                                    umma_desc_join(b_lo + (uint32_t)(kk >> 2) * (kPanelBytes >> 4) + (uint32_t)(kk & 3) * 2u),
                                    umma_idesc(128, 128, 1, 0) | (1u << 13), 1u);
                        umma_commit(&bars[D_QEMPTY + g % NQ]);   // (raw q serves no other product)
                        umma_commit(&bars[D_XEMPTY]);
                        for (int h = 0; h < 4; ++h) umma_commit(&bars[D_DOEMPTY + (dn + (h & 1)) % ND]);
                        dn += 2;
                    }
                    d2 = dn++;
                    umma_commit(&bars[D_READY + (g & 1)]);
                    if (f & FL_LVL1) umma_commit(&bars[D_KEMPTY + kb]);
                } else {   // the last round has no S: its tile is free once the products that read it have retired
                    umma_commit(&bars[D_READY + (g & 1)]);
                }
                mbar_arrive(&bars[D_READY + (g & 1)]);
                return f;
            };
            int fm = 0;                                  // flags of step i - 1
            int f0 = issue_s(0), d0 = d2;                // step i
            int f1 = f0 ? issue_s(1) : 0, d1 = d2;
            if (ok) mbar_arrive(&bars[D_READY]);         // (no dP before round 0)
#pragma unroll 1
            for (int i = 0; ok && (f0 | fm); ++i) {
                if (!wait(D_ROUND + (i & 1), i >> 1)) break;
                const uint32_t tile = tmem + colS + (i & 1) * 128;
                if (fm && !(fm & FL_FIRST)) {            // dK (+)= dS^T(i - 1) Q
                    if ((fm & FL_LVL0) && ndk > 0 && !wait(D_DKFREE, ndk - 1)) break;
                    tc_fence_after_sync();
                    mma_t16(tmem + colDK, tile + 8, smem_u32(sQ + ((i - 1) % NQ) * kD64Tile), idescD, !(fm & FL_LVL0));
                    umma_commit(&bars[D_QEMPTY + (i - 1) % NQ]);
                    if (fm & FL_LVL1) { umma_commit(&bars[D_DKFULL]); ++ndk; }
                }
                if (f0) {                                // dV (+)= P^T(i) dO
                    if ((f0 & FL_FIRST) && ndv > 0 && !wait(D_DVFREE, ndv - 1)) break;
                    if (!wait(D_DOFULL + d0 % ND, d0 / ND)) break;
                    tc_fence_after_sync();
                    mma_t16(tmem + colDV, tile, smem_u32(sDO + (d0 % ND) * kD64Tile), idescD, !(f0 & FL_FIRST));
                    umma_commit(&bars[D_DOEMPTY + d0 % ND]);
                    if (f0 & FL_LAST) { umma_commit(&bars[D_DVFULL]); ++ndv; }
                }
                const int f2 = f1 ? issue_s(i + 2) : 0;
                fm = f0;
                f0 = f1; d0 = d1;
                f1 = f2; d1 = d2;
            }
        } else if (warp == 3 && elect_one()) {
            constexpr uint32_t idescT = umma_idesc(128, 128, 0, 0);
            auto flow = make_flow(item_of, steps_of);
            bool ok = true;
            int dn = 0, nv = 0;
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_DKV_MMA)) ok = false;
                return ok;
            };
#pragma unroll 1
            for (int i = 0; flow.next(); ++i) {
                if (flow.t == 0) {
                    dn = ((dn + 1) & ~1) + 2;
                    wait(D_VFULL, nv);
                    ++nv;
                }
                // Every thread holds dP(i - 1).  This comes first: it says that S(i) is there, hence Y and all entries before it, which
                // this thread does not wait for; a slot's phase below is then the current one.
                if (i > 0) wait(D_DPFREE, i - 1);
                wait(D_DOFULL + dn % ND, dn / ND);
                tc_fence_after_sync();
                if (!ok) break;
                mma_kk(tmem + colDP, smem_u32(sV), smem_u32(sDO + (dn % ND) * kD64Tile), HD, idescT, false);
                umma_commit(&bars[D_READY + ((i + 1) & 1)]);
                umma_commit(&bars[D_DOEMPTY + dn % ND]);
                if (flow.t + 1 == flow.T) umma_commit(&bars[D_VEMPTY]);
                ++dn;
            }
        }
    } else if (warp >= 12) {
        // ---------------------------------------------------------------- write-out of finished levels and items, one row per thread
        set_fewer_regs<56>();
        const int row = (warp & 3) * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        auto flow = make_flow(item_of, steps_of);
        int ndk = 0, ndv = 0;
        bool ok = true;
        auto ready = [&](int bar, int n) {
            ok = mbar_wait(&bars[bar], n & 1, abort_flag, ST_DKV_COMPUTE);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            return ok;
        };
        auto write = [&](auto caller, uint32_t col, float mul, int free_bar, __nv_bfloat16* dst, bool valid) {
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                float v[32];
                uint32_t w[16];
                tile::tmem_row32(tl + col + c * 32, v);
                if (c == 1) {
                    tc_fence_before_sync();
                    mbar_arrive(&bars[free_bar]);
                }
#pragma unroll
                for (int x = 0; x < 16; ++x) w[x] = pack_bf16(v[2 * x] * mul, v[2 * x + 1] * mul);
                tile::gstore_bf16_w16<decltype(caller)::value>(dst + c * 32, w, valid);
            }
        };
#pragma unroll 1
        while (flow.next()) {
            const int J = flow.c, s = flow.s, kj = J * kTile + row;
            const bool last = flow.t + 1 == flow.T;
            if (last) {   // dV first: the next item's first product waits for it
                if (!ready(D_DVFULL, ndv)) break;
                write(std::true_type{}, colDV, 1.f, D_DVFREE, (__nv_bfloat16*)p.dv + ((size_t)s * p.L + (kj < p.L ? kj : 0)) * HD, kj < p.L);
                ++ndv;
            }
            if (flow.t == 0) {
                if (last) {   // no later query chunk met: the boundary-adjusted keys get a zero gradient from the sweep
                    uint4* dst = reinterpret_cast<uint4*>(p.dkv + ((size_t)s * p.Lp + kj) * HD);
                    for (int x = 0; x < HD / 8; ++x) dst[x] = make_uint4(0u, 0u, 0u, 0u);
                }
                continue;
            }
            const int l = level(J, flow.t);
            if (!(flags_of(J, flow.t, flow.T, l) & FL_LVL1)) continue;
            if (!ready(D_DKFULL, ndk)) break;
            write(std::false_type{}, colDK, p.scale, D_DKFREE, p.dkv + ((size_t)kver_row(p.vl, s, l, J) + row) * HD, true);
            ++ndk;
        }
    } else {
        set_more_regs<200>();
        const int q4 = warp & 3, h = (warp - 4) >> 2, row = q4 * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)(q4 * 32) << 16) + h * 64;   // this thread's 64 query columns
        const float sl2 = p.scale * kLog2e;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        float pr[64];                              // P^T of step i - 1, then of step i
#pragma unroll
        for (int x = 0; x < 64; ++x) pr[x] = 0.f;
        // One round: part A of step i from its S^T tile, part B of step i - 1 into it.  The first and the last round use this code too
        // (the half without a step works on what it finds and nothing reads its results), and so do the diagonal steps: instruction
        // fetch is what a round waits for most, and a copy of this code that runs once per item cost 3000 cycles each time.
        auto round = [&](const int i, const int fa, const int fb) {
            const uint32_t ts = tlane + colS + (i & 1) * 128;
            uint32_t dp[4][16], sv[2][16];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld16(tlane + colDP + c * 16, dp[c]);
            tmem_ld16(ts, sv[0]);
            const float* ls_ = stat + (i & 3) * 2 * kTile + h * 64;                    // -lse2 of step i
            const float* dl_ = stat + ((i - 1) & 3) * 2 * kTile + kTile + h * 64;      // -delta of step i - 1
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tmem_ld_wait16(sv[c & 1]);
                if (c == 0) {   // dP too has arrived
#pragma unroll
                    for (int x = 0; x < 4; ++x) tmem_ld_wait16(dp[x]);
                    tc_fence_before_sync();
                    if (fb) mbar_arrive(&bars[D_DPFREE]);
                }
                if (c < 3) tmem_ld16(ts + (c + 1) * 16, sv[(c + 1) & 1]);
                uint32_t pk[16];   // P^T(i), dS^T(i - 1)
#pragma unroll
                for (int x = 0; x < 16; x += 4) {   // dS^T = P^T o (dP^T - delta)
                    const uint32_t* d_ = &dp[c][x];
                    const float4 dl = *reinterpret_cast<const float4*>(dl_ + c * 16 + x);
                    float d[4];
                    unpack2(mul2(pack2(pr[c * 16 + x], pr[c * 16 + x + 1]),
                                 add2(pack2(__uint_as_float(d_[0]), __uint_as_float(d_[1])), pack2(dl.x, dl.y))), d[0], d[1]);
                    unpack2(mul2(pack2(pr[c * 16 + x + 2], pr[c * 16 + x + 3]),
                                 add2(pack2(__uint_as_float(d_[2]), __uint_as_float(d_[3])), pack2(dl.z, dl.w))), d[2], d[3]);
                    pk[8 + (x >> 1)] = pack_bf16(d[0], d[1]);
                    pk[9 + (x >> 1)] = pack_bf16(d[2], d[3]);
                }
#pragma unroll
                for (int x = 0; x < 16; x += 4) {   // P^T = exp2(S^T * scale - lse)
                    const uint32_t* s_ = &sv[c & 1][x];
                    const float4 ls = *reinterpret_cast<const float4*>(ls_ + c * 16 + x);
                    uint64_t v01 = fma2(pack2(__uint_as_float(s_[0]), __uint_as_float(s_[1])), sl2x2, pack2(ls.x, ls.y));
                    uint64_t v23 = fma2(pack2(__uint_as_float(s_[2]), __uint_as_float(s_[3])), sl2x2, pack2(ls.z, ls.w));
                    float e[4];
                    unpack2(v01, e[0], e[1]);
                    unpack2(v23, e[2], e[3]);
#pragma unroll
                    for (int y = 0; y < 4; ++y) pr[c * 16 + x + y] = ex2(e[y]);
                    pk[x >> 1] = pack_bf16(pr[c * 16 + x], pr[c * 16 + x + 1]);
                    pk[(x >> 1) + 1] = pack_bf16(pr[c * 16 + x + 2], pr[c * 16 + x + 3]);
                }
                tmem_st16(ts + c * 16, pk);
            }
            tmem_st_wait();
            if (fa & FL_FIRST) mask_pt(ts, row - h * 64);   // causal mask of the diagonal chunk
            tc_fence_before_sync();
            mbar_arrive(&bars[D_ROUND + (i & 1)]);
            if (fb) mbar_arrive(&bars[D_STEMPTY + ((i - 1) & 3)]);
        };
        // The diagonal chunk's (scale * dS)^T in bf16 for the chain rule; `base` = the chunk's first row.
        auto diagonal = [&](const int i, const int base) {
            const float* dl_ = stat + (i & 3) * 2 * kTile + kTile + h * 64;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t dp[16], w[8];
                float d[16];
                tmem_ld16(tlane + colDP + c * 16, dp);
                tmem_ld_wait16(dp);
#pragma unroll
                for (int x = 0; x < 16; x += 4) {
                    const float4 dl = *reinterpret_cast<const float4*>(dl_ + c * 16 + x);
                    d[x] = pr[c * 16 + x] * (__uint_as_float(dp[x]) + dl.x);
                    d[x + 1] = pr[c * 16 + x + 1] * (__uint_as_float(dp[x + 1]) + dl.y);
                    d[x + 2] = pr[c * 16 + x + 2] * (__uint_as_float(dp[x + 2]) + dl.z);
                    d[x + 3] = pr[c * 16 + x + 3] * (__uint_as_float(dp[x + 3]) + dl.w);
                }
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    if (h * 64 + c * 16 + x < row) d[x] = 0.f;   // (mask_pt has masked what the product takes, not pr)
#pragma unroll
                for (int x = 0; x < 8; ++x) w[x] = pack_bf16(d[2 * x] * p.scale, d[2 * x + 1] * p.scale);
                st_global_32<false>(p.dsdt + ((size_t)base + row) * kTile + h * 64 + c * 16, w);
            }
        };
        int fb = 0, base = 0;   // step i - 1: flags, first row of the key chunk
#pragma unroll 1
        for (int i = 0;; ++i) {
            bool ok = mbar_wait(&bars[D_READY + (i & 1)], (i >> 1) & 1, abort_flag, ST_DKV_COMPUTE);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after_sync();
            const int2 de = desc[i & 7];
            const int fa = de.x;
            if (!(fa | fb)) break;
            if (fb & FL_FIRST) diagonal(i - 1, base);
            round(i, fa, fb);
            if (!fa) break;
            fb = fa;
            base = de.y;
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    report_abort(abort_flag, p.status);
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

// Per-row constants of the backward sweeps, stored negated so that they enter as addends:
//   delta[i] = -(dO_i . O_i),   lse2[i] = (G_i - lse_i) * log2(e)   (G: gate prefix, absent = 0),
// padded to Lp (tail rows: delta 0, lse2 -1e30 so that their probabilities vanish).  One warp per row.
template <int HD>
__global__ void rowstats_kernel(const __nv_bfloat16* __restrict__ o, const __nv_bfloat16* __restrict__ d_o,
                                const float* __restrict__ lse, const float* __restrict__ G, float* __restrict__ delta,
                                float* __restrict__ lse2, int S, int L, int Lp) {
    grid_wait();
    grid_launch();
    constexpr int TPR = HD / 8;                 // threads per row: 16 bytes (8 values) of o and of dO each
    const int i = blockIdx.x * (256 / TPR) + threadIdx.x / TPR;
    const int sub = threadIdx.x % TPR;
    for (int s = blockIdx.y; s < S; s += gridDim.y) {   // (a grid's second dimension ends at 65535)
        float acc = 0.f;
        if (i < L) {
            const size_t base = ((size_t)s * L + i) * HD + sub * 8;
            const uint4 a = *reinterpret_cast<const uint4*>(o + base), b = *reinterpret_cast<const uint4*>(d_o + base);
            const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[x]));
                const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[x]));
                acc += fa.x * fb.x + fa.y * fb.y;
            }
        }
#pragma unroll
        for (int off = TPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (sub == 0 && i < Lp) {
            delta[(size_t)s * Lp + i] = -acc;
            // rows of the zero-padded tail get a huge negative value: their probabilities must come out as exact zeros.  (A
            // plain 0 would do without a gate; with one, exp2(0 - G_j log2 e) of a strongly decayed key overflows and the
            // product with the row's zero dP - delta is a NaN.)
            float v = -1e30f;
            if (i < L) v = ((G ? G[(size_t)s * Lp + i] : 0.f) - lse[(size_t)s * L + i]) * kLog2e;
            lse2[(size_t)s * Lp + i] = v;
        }
    }
}

template <int HD, bool GATE>
cudaError_t launch_one(const BwdTensorMaps& tm, const BwdParams& p, int which, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const int pairs = (p.N * p.S + 1) / 2, grid = pairs < sms ? pairs : sms;
    // dK/dV sweep, us, dkv64_kernel / dkv_kernel: 8 x 16 x 2048 x 64 226 / 275, 4 x 32 x 4096 x 64 742 / 950 (taken with the mask in
    // the logits, see mask_pt: 3 % more now); gated, its further live values and passes cost more than the rounds give (2 x 8 x
    // 3001 x 64: 75 / 68)
    if constexpr (HD == 64 && !GATE) {
        if (which == 0) return launch<dkv64_kernel>(grid, 512, kD64Total + 1024, st, tm, p);
    } else {
        if (which == 0) return launch<dkv_kernel<HD, GATE>>(grid, 384, kSmemAlloc, st, tm, p);
    }
    return launch<dq_kernel<HD, GATE>>(grid, 512, kSmemAlloc, st, tm, p);
}

}  // namespace

// which = 0: dK/dV sweep, which = 1: dQ sweep.
cudaError_t launch_fa_bwd(const BwdTensorMaps& tm, const BwdParams& p, int hd, int which, cudaStream_t st) {
    if (hd == 64) return p.G ? launch_one<64, true>(tm, p, which, st) : launch_one<64, false>(tm, p, which, st);
    return p.G ? launch_one<128, true>(tm, p, which, st) : launch_one<128, false>(tm, p, which, st);
}

cudaError_t launch_rowstats(const void* o, const void* d_o, const float* lse, const float* G, float* delta, float* lse2,
                            int S, int L, int Lp, int hd, cudaStream_t st) {
    const int rows_per_cta = 256 / (hd / 8);
    const dim3 grid((Lp + rows_per_cta - 1) / rows_per_cta, S < 65535 ? S : 65535);
    typedef __nv_bfloat16 bf;
    return hd == 64 ? launch<rowstats_kernel<64>>(grid, 256, 0, st, (const bf*)o, (const bf*)d_o, lse, G, delta, lse2, S, L, Lp)
                    : launch<rowstats_kernel<128>>(grid, 256, 0, st, (const bf*)o, (const bf*)d_o, lse, G, delta, lse2, S, L, Lp);
}

}  // namespace path
