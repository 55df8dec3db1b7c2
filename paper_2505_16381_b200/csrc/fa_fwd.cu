// Fused forward sweep of PaTH attention (paper Sec. 3.3, the FlashAttention-style loop).
//
// Query chunk I of one (batch, head) slice walks the key chunks J = I, I-1, ..., 0.  The diagonal chunk uses the raw q, k
// plus the in-chunk Householder correction as a second contraction (Sec. 3.3, case i = j):
//     S = Q K^T - lower(Q W^T) (T~ strictLower(W K^T))                [operands q_raw, k_raw, xq, y]
// Every earlier chunk J < I is an ordinary tile product of a query version and a key version that meet at the dyadic
// boundary of (I, J):  S = Qv[l][I] Kv[l][J]^T, l = msb(I xor J).  The versions are prepared beforehand, so this loop
// contains no query update.
//
// Two kernels.  fa_fwd_kernel: a work item is a PAIR of neighbouring query chunks (2k, 2k+1), one stream each: both meet
// every key chunk J < 2k at the same level (the indices differ in bit 0 only), so one load of a key and a value tile
// serves both.  fa_split_kernel: a work item is one query chunk whose key chunks are dealt alternately to the two streams
// and whose two partial results are merged at the end; half the latency per chunk, twice the tile traffic: for problems
// whose pairs do not fill the GPU.  The rule is at launch_fa_fwd.
//
// A stream has its own softmax warpgroup (one query row per thread, the whole 128-wide logit row held in registers), its
// own S tile and O accumulator in tensor memory and its own running (max, sum).  While one warpgroup does its
// exponentials the tensor pipe works for the other stream.  P never touches shared memory: it is written to tensor memory
// as packed bf16 and enters O += P V as the tensor-memory A operand.  It is handed over in two parts, so that
// the P V of the first three quarters runs underneath the last quarter's exponentials.
//
// Warps of both kernels: 0 = TMA producer, 1 = tcgen05 MMA issuer, 2-3 idle (they give their registers to the softmax
// warps), 4-7 = softmax of stream 0, 8-11 = softmax of stream 1.
#include <type_traits>
#include "common.cuh"
#include "tc5.cuh"
#include "tileops.cuh"

namespace path {
using namespace tc5;

constexpr int kTile = 128;
constexpr uint32_t kSlotBytes = 32768;  // one [128 x 128] bf16 operand tile (two 64-column panels)
constexpr uint32_t kPanelBytes = 16384; // one [128 x 64] bf16 panel

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// S[tmem] = A B^T, both operands K-major [128][HD] tiles (descriptors advance by their low word only: 32 bytes per step, the next
// 64-column panel after four steps).
template <int HD>
__device__ __forceinline__ void mma_kk(uint32_t d_tmem, uint32_t a0, uint32_t b0, uint32_t idesc) {
    const uint32_t a_lo = umma_desc_lo(a0, 16), b_lo = umma_desc_lo(b0, 16);
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) {
        const uint32_t o = (uint32_t)(kk >> 2) * (kPanelBytes >> 4) + (uint32_t)(kk & 3) * 2u;
        umma_ss(d_tmem, umma_desc_join(a_lo + o), umma_desc_join(b_lo + o), idesc, kk > 0 ? 1u : 0u);
    }
}
// S[tmem] += (+-) Xq Y for the diagonal chunk: Xq K-major, Y as stored ([128 contraction rows][128 keys], MN-major).
__device__ __forceinline__ void mma_correction(uint32_t d_tmem, uint32_t xq, uint32_t y, uint32_t idesc) {
    const uint32_t a_lo = umma_desc_lo(xq, 16), b_lo = umma_desc_lo(y, kPanelBytes);
#pragma unroll
    for (int kk = 0; kk < kTile / 16; ++kk)
        umma_ss(d_tmem, umma_desc_join(a_lo + (uint32_t)(kk >> 2) * (kPanelBytes >> 4) + (uint32_t)(kk & 3) * 2u),
                umma_desc_join(b_lo + kk * 128u), idesc, 1u);
}

// One logit tile of one stream, one query row per thread: S (tensor memory) -> P (packed bf16, tensor memory), running
// maximum m (log2 units) and sum l.  `tS`, `tP`, `tO`: tensor-memory addresses of the thread's lanes; `gk`: gate prefix of
// the tile's key chunk (shared memory), `gi2` that of the row in log2 units; `have_o`: O holds an earlier result.
//   SEP: P has columns of its own (d = 64, where the accumulators leave room) and S is handed back (`sfree`) as soon as it
//   is in registers.  Otherwise P overwrites the first half of S.
// The stream's previous P V has retired before the call: P may be overwritten and O is stable.
// P is handed over in two parts (`pa`: the first 96 keys, `pb`).  Every hand-over is one arrival per warp.
template <int HD, bool GATE, bool DIAG, bool SEP>
__device__ __forceinline__ bool softmax_tile(uint32_t tS, uint32_t tP, uint32_t tO, int row, const uint64_t sl2x2, float sl2,
                                             float gi2, const float* gk, bool have_o, float& m, float& l, uint64_t* sfree,
                                             uint64_t* pa, uint64_t* pb, bool ok) {
    constexpr bool PRE = DIAG || GATE;                 // logits are scaled (and gated, masked) in place first
    const bool lane0 = (threadIdx.x & 31) == 0;
    if (ok) {
        uint32_t r[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, r[c]);
        tmem_ld_wait();
        if (SEP) {
            tc_fence_before_sync();
            __syncwarp();
            if (lane0) mbar_arrive(sfree);
        }
        float m_new = m;
        if (PRE) {
            const uint64_t gi22 = pack2(gi2, gi2), nlog2 = pack2(-1.4426950408889634f, -1.4426950408889634f);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    uint64_t v[2];
#pragma unroll
                    for (int y = 0; y < 2; ++y)
                        v[y] = fma2(pack2(__uint_as_float(r[c][e + 2 * y]), __uint_as_float(r[c][e + 2 * y + 1])), sl2x2, gi22);
                    if (GATE) {
                        const float4 g4 = *reinterpret_cast<const float4*>(gk + c * 32 + e);
                        v[0] = fma2(pack2(g4.x, g4.y), nlog2, v[0]);
                        v[1] = fma2(pack2(g4.z, g4.w), nlog2, v[1]);
                    }
                    float a[4];
                    unpack2(v[0], a[0], a[1]);
                    unpack2(v[1], a[2], a[3]);
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        if (DIAG && c * 32 + e + y > row) a[y] = -INFINITY;
                        r[c][e + y] = __float_as_uint(a[y]);
                    }
                }
        }
        // row maximum of the scaled logits (log2 units)
        float a4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int e = 0; e < 32; e += 2)
                a4[(e >> 1) & 3] = max3(a4[(e >> 1) & 3], __uint_as_float(r[c][e]), __uint_as_float(r[c][e + 1]));
        float mx = fmaxf(fmaxf(a4[0], a4[1]), fmaxf(a4[2], a4[3]));
        if (!PRE) mx *= sl2;
        const bool grow = mx > m + 8.f;       // lazy rescaling: a stale maximum is tolerated up to 2^8
        if (grow) m_new = mx;
        if (__any_sync(0xffffffffu, grow)) {
            const float alpha = ex2(m - m_new);
            l *= alpha;
            if (have_o) {
#pragma unroll 1
                for (int c = 0; c < HD / 16; ++c) {
                    uint32_t o[16];
                    tmem_ld16(tO + c * 16, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                    tmem_st16(tO + c * 16, o);
                }
            }
        }
        m = m_new;
        const uint64_t nm2 = pack2(-m, -m);
        const uint64_t mul2 = PRE ? pack2(1.f, 1.f) : sl2x2;
        uint64_t lacc[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
                const uint64_t v = fma2(pack2(__uint_as_float(r[c][e]), __uint_as_float(r[c][e + 1])), mul2, nm2);
                float a, b;
                unpack2(v, a, b);
                a = ex2(a);
                b = ex2(b);
                lacc[(e >> 1) & 1] = add2(lacc[(e >> 1) & 1], pack2(a, b));
                pk[e >> 1] = pack_bf16(a, b);
            }
            tmem_st16(tP + c * 16, pk);
            if (c == 2) {
                tmem_st_wait();
                tc_fence_before_sync();
                __syncwarp();
                if (lane0) mbar_arrive(pa);
            }
        }
        float la, lb;
        unpack2(add2(lacc[0], lacc[1]), la, lb);
        l += la + lb;
        tmem_st_wait();
    }
    tc_fence_before_sync();
    __syncwarp();
    if (lane0) {
        if (!ok) mbar_arrive(pa);
        if (SEP && !ok) mbar_arrive(sfree);
        mbar_arrive(pb);
    }
    return ok;
}

// ------------------------------------------------------------------------------------------------ one chunk, two streams
struct SplitSmem {
    static constexpr uint32_t offQ = 0;                       // 3 slots: ring of query operands
    static constexpr uint32_t offK = offQ + 3 * kSlotBytes;   // 2 slots: one per stream
    static constexpr uint32_t offV = offK + 2 * kSlotBytes;   // 2 slots: one per stream
    static constexpr uint32_t offBar = offV + 2 * kSlotBytes;
    // [2 streams][128] pairs: at the end of a work item the stream's (running max, running sum) per row; before that the
    // first half of a stream's part holds the gate prefix of its current key chunk
    static constexpr uint32_t offStat = offBar + 256;
    static constexpr uint32_t total = offStat + 2 * kTile * 8;
    static constexpr uint32_t alloc = 232448;                 // everything an SM offers one CTA
    static_assert(total + 512 <= alloc, "no room left to align the base");
};

enum { B_QFULL = 0, B_QEMPTY = 3, B_KFULL = 6, B_KEMPTY = 8, B_VFULL = 10, B_VEMPTY = 12,
       B_SFULL = 14, B_PA = 16, B_PB = 18, B_OFULL = 20, B_OFREE = 22, B_COUNT = 23 };

template <int HD, bool GATE>
__global__ void __launch_bounds__(384, 1)
fa_split_kernel(const __grid_constant__ FwdTensorMaps tm, const FwdParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    if ((uint32_t)(smem - smem_raw) + SplitSmem::total > SplitSmem::alloc) {   // uniform over the CTA
        grid_wait();   // (the status word belongs to the kernels before)
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)ST_FWD_PRODUCER);
        return;
    }
    uint8_t* sQ = smem + SplitSmem::offQ;
    uint8_t* sK = smem + SplitSmem::offK;
    uint8_t* sV = smem + SplitSmem::offV;
    uint64_t* bars = (uint64_t*)(smem + SplitSmem::offBar);
    uint32_t* tmem_slot = (uint32_t*)(bars + B_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    float2* stat = (float2*)(smem + SplitSmem::offStat);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = p.N * p.S;

    if (threadIdx.x == 0) {
        for (int i = 0; i < B_COUNT; ++i)
            mbar_init(&bars[i], (i >= B_PA && i < B_OFULL) ? 4u : (i == B_OFREE ? 256u : 1u));
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 2 && lane < 7) {
        tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&tm) + lane);   // the seven maps are contiguous
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    // tensor memory columns: S of stream x at x*128 (P aliases its first 64 columns), O of stream x at 256 + x*128
    // k-th work item of this CTA: one if there are CTAs enough, otherwise pairs (long, short) of one slice, slice after slice
    const bool single = (int)gridDim.x >= items;
    auto item_of = [&](int k, int& I, int& s) {
        const int w = single ? (k == 0 ? (int)blockIdx.x : items) : 2 * ((int)blockIdx.x + (k >> 1) * (int)gridDim.x) + (k & 1);
        if (w >= items) return false;
        s = w / p.N;
        const int j = w % p.N;
        I = (j & 1) ? (j >> 1) : p.N - 1 - (j >> 1);
        return true;
    };
    // key chunks a work item visits, counted from the diagonal: all I + 1 of them, or fewer when the gate has made the
    // far ones negligible (every warp role reads the same precomputed number)
    auto steps_of = [&](int I, int s) {
        return p.nkeep ? min(I + 1, p.nkeep[s * p.N + I]) : I + 1;
    };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp == 0 && elect_one()) {
            // ------------------------------------------------------------ TMA producer
            bool ok = true;
            int nq = 0;                       // query operands issued so far (all work items)
            uint32_t kf = 0, vf = 0;          // bit x: parity of the number of fills of K / V slot x so far
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_FWD_PRODUCER)) ok = false;
            };
            auto load_q = [&](const CUtensorMap* m, int kdim, int row0, int slice = -1) {   // slice >= 0: a caller's tensor
                const int slot = nq % 3;
                wait_empty(B_QEMPTY + slot, nq / 3);
                if (!ok) return;
                mbar_expect_tx(&bars[B_QFULL + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tile::tma_rows(sQ + slot * kSlotBytes, m, &bars[B_QFULL + slot], kdim, row0, slice);
                else tile::tma_tile(sQ + slot * kSlotBytes, m, &bars[B_QFULL + slot], kdim, row0);
                ++nq;
            };
            auto load_kv = [&](uint8_t* base, int bfull, int bempty, int slot, uint32_t& fills, const CUtensorMap* m,
                               int kdim, int row0, int slice = -1) {
                wait_empty(bempty + slot, (int)((fills >> slot) & 1u));
                if (!ok) return;
                mbar_expect_tx(&bars[bfull + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tile::tma_rows(base + slot * kSlotBytes, m, &bars[bfull + slot], kdim, row0, slice);
                else tile::tma_tile(base + slot * kSlotBytes, m, &bars[bfull + slot], kdim, row0);
                fills ^= 1u << slot;
            };
            int I, s;
            for (int it = 0; ok && item_of(it, I, s); ++it) {
                const int NS = steps_of(I, s);
                const int rowRaw = s * p.Lp + I * kTile;
                // diagonal chunk: raw q, k and the correction operands (both K slots), V of chunk I
                load_q(&tm.q_raw, HD, I * kTile, s);
                load_kv(sK, B_KFULL, B_KEMPTY, 0, kf, &tm.k_raw, HD, I * kTile, s);
                load_q(&tm.xq, kTile, rowRaw);
                load_kv(sV, B_VFULL, B_VEMPTY, 1, vf, &tm.y, kTile, rowRaw);   // Y borrows stream 1's V slot
                load_kv(sV, B_VFULL, B_VEMPTY, 0, vf, &tm.v, HD, I * kTile, s);
                int cur = -1;
                for (int n = 1; n < NS && ok; ++n) {
                    const int J = I - n, x = n & 1, l = msb32((unsigned)(I ^ J));   // l is non-decreasing in n
                    if (l != cur) {
                        load_q(&tm.qv, HD, (int)qver_row(p.vl, s, l, I));
                        cur = l;
                    }
                    load_kv(sK, B_KFULL, B_KEMPTY, x, kf, &tm.kv, HD, (int)kver_row(p.vl, s, l, J));
                    load_kv(sV, B_VFULL, B_VEMPTY, x, vf, &tm.v, HD, J * kTile, s);
                }
            }
        } else if (warp == 1 && elect_one()) {
            // ------------------------------------------------------------ MMA issuer
            // a negative scale is applied as a sign flip of the logits here (negate-A bit), its magnitude in the softmax
            const uint32_t idescS = umma_idesc(128, 128, 0, 0) | (p.scale < 0.f ? (1u << 13) : 0u);
            const uint32_t idescC = umma_idesc(128, 128, 0, 1) | (p.scale < 0.f ? 0u : (1u << 13));   // the correction is subtracted
            constexpr uint32_t idescO = umma_idesc(128, HD, 0, 1);
            bool ok = true;
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_FWD_MMA)) ok = false;
            };
            auto issue_s = [&](int x, int qs, int ks) {
                mma_kk<HD>(tmem + x * 128, smem_u32(sQ + qs * kSlotBytes), smem_u32(sK + ks * kSlotBytes), idescS);
            };
            int qi_next = 0;                   // query operands waited for so far (all work items)
            int released = 0;                  // query operands [0, released) have been handed back to the producer
            uint32_t kc = 0, vc = 0, pc = 0;   // bit x: parity of the K / V fills and P tiles of stream x consumed so far
            int item = 0;
            auto take_q = [&]() {
                const int qi = qi_next++;
                wait(B_QFULL + qi % 3, qi / 3);
                return qi;
            };
            auto take_k = [&](int x) { wait(B_KFULL + x, (int)((kc >> x) & 1u)); kc ^= 1u << x; };
            auto release_q = [&](int upto) {
                for (; released < upto; ++released) umma_commit(&bars[B_QEMPTY + released % 3]);
            };
            int I, s_it;
            for (; ok && item_of(item, I, s_it); ++item) {
                const int NS = steps_of(I, s_it);
                int cur_level = -1;
                int q_of0, q_of1;              // operand index used by each stream's most recent S product
                auto advance_q = [&](int n) {  // operand index of step n >= 1 (waits for a newly needed one)
                    const int l = msb32((unsigned)(I ^ (I - n)));
                    if (l != cur_level) {
                        cur_level = l;
                        take_q();
                    }
                    return qi_next - 1;
                };
                // S of step 0 (diagonal, stream 0): two contractions
                const int q0 = take_q();
                take_k(0);
                tc_fence_after_sync();
                if (ok) issue_s(0, q0 % 3, 0);
                const int q1 = take_q();
                wait(B_VFULL + 1, (int)((vc >> 1) & 1u)); vc ^= 2u;
                tc_fence_after_sync();
                if (!ok) break;
                mma_correction(tmem, smem_u32(sQ + (q1 % 3) * kSlotBytes), smem_u32(sV + kSlotBytes), idescC);
                umma_commit(&bars[B_SFULL + 0]);
                umma_commit(&bars[B_KEMPTY + 0]);
                umma_commit(&bars[B_VEMPTY + 1]);
                release_q(q1 + 1);             // rawQ and Xq go back once the diagonal products retire
                q_of0 = q_of1 = q1 + 1;
                // S of step 1 (stream 1)
                if (NS > 1) {
                    q_of1 = advance_q(1);
                    take_k(1);
                    tc_fence_after_sync();
                    if (!ok) break;
                    issue_s(1, q_of1 % 3, 1);
                    umma_commit(&bars[B_SFULL + 1]);
                    umma_commit(&bars[B_KEMPTY + 1]);
                }
                if (NS <= 2) release_q(qi_next);
                for (int n = 0; n < NS && ok; ++n) {
                    const int x = n & 1, t = n >> 1;
                    // O_x += P_x V_n; the first product of a work item overwrites O_x, which the previous item's
                    // epilogue must have read
                    const uint32_t pp = (pc >> x) & 1u;
                    pc ^= 1u << x;
                    wait(B_VFULL + x, (int)((vc >> x) & 1u)); vc ^= 1u << x;
                    if (t == 0 && item > 0) wait(B_OFREE, item - 1);
                    wait(B_PA + x, (int)pp);
                    tc_fence_after_sync();
                    if (!ok) break;
                    {
                        const uint32_t b_lo = umma_desc_lo(smem_u32(sV + x * kSlotBytes), kPanelBytes);
#pragma unroll
                        for (int kk = 0; kk < kTile / 16; ++kk) {
                            if (kk == 6) {
                                wait(B_PB + x, (int)pp);
                                tc_fence_after_sync();
                                if (!ok) break;
                            }
                            umma_ts(tmem + 256 + x * 128, tmem + x * 128 + kk * 8, umma_desc_join(b_lo + kk * 128u), idescO,
                                    (t > 0 || kk > 0) ? 1u : 0u);
                        }
                        if (!ok) break;
                        umma_commit(&bars[B_VEMPTY + x]);
                    }
                    // the stream's next S overwrites P; products issued by one thread execute in order, so it lands
                    // after the P V above has read P
                    if (n + 2 < NS) {
                        const int qi = advance_q(n + 2);
                        if (x) q_of1 = qi; else q_of0 = qi;
                        take_k(x);
                        tc_fence_after_sync();
                        if (!ok) break;
                        issue_s(x, qi % 3, x);
                        umma_commit(&bars[B_SFULL + x]);
                        umma_commit(&bars[B_KEMPTY + x]);
                        // operands older than what either stream used last can go back to the producer
                        release_q(n + 3 == NS ? qi_next : min(qi, x ? q_of0 : q_of1));
                    } else {
                        umma_commit(&bars[B_OFULL + x]);
                    }
                }
                release_q(qi_next);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // ------------------------------------------------------------ softmax warpgroups, one row per thread
        const int x = (warp - 4) >> 2;          // stream
        const int q4 = warp & 3;                // TMEM lane quadrant this warp may touch
        const int row = q4 * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)(q4 * 32) << 16);
        const uint32_t colS = x * 128, colO = 256 + x * 128;
        const float kLog2e = 1.4426950408889634f;
        const float sl2 = fabsf(p.scale) * kLog2e;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        bool ok = true;
        int sc = 0;                             // S tiles consumed so far by this stream (all work items)
        int o1 = 0;                             // work items so far in which stream 1 had steps
        int item = 0;
        float2* statx = stat + x * kTile;
        float* gkx = reinterpret_cast<float*>(statx);
        auto wg_sync = [&]() {
            __syncwarp();   // bar.sync is warp-aligned: reconverge first
            if (x == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
            else asm volatile("bar.sync 2, 128;" ::: "memory");
        };

        int I, s;
        for (; item_of(item, I, s); ++item) {
            const int NS = steps_of(I, s);
            const int qi = I * kTile + row;     // position within the slice (may be >= L in the ragged tail)
            const int TX = (NS - x + 1) >> 1;   // steps of this stream: n = 2t + x
            float gi2 = 0.f;
            if (GATE) gi2 = p.G[(size_t)s * p.Lp + qi] * kLog2e;
            float m = -INFINITY, l = 0.f;
            // the stat words are shared with the previous item's merge: every thread must have read them
            if (item > 0 && ok && !mbar_wait(&bars[B_OFREE], (item - 1) & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;

            auto softmax_step = [&](auto diag_tag, const int t) {
                constexpr bool DIAG = decltype(diag_tag)::value;   // the diagonal chunk (step 0): causal mask
                const int J = I - (2 * t + x);
                if (GATE) {
                    wg_sync();   // everyone is done with the previous chunk's values
                    gkx[row] = p.G[(size_t)s * p.Lp + J * kTile + row];
                    wg_sync();
                }
                if (ok && !mbar_wait(&bars[B_SFULL + x], sc & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
                ++sc;
                ok = __all_sync(0xffffffffu, ok);  // keep the warp-collective TMEM accesses convergent
                tc_fence_after_sync();
                // O of this stream is stable here: its S tile only becomes ready after the stream's previous P V has retired
                ok = softmax_tile<HD, GATE, DIAG, false>(tlane + colS, tlane + colS, tlane + colO, row, sl2x2, sl2, gi2, gkx, t > 0, m,
                                                         l, nullptr, &bars[B_PA + x], &bars[B_PB + x], ok);
            };
            {
                int t = 0;
                if (x == 0 && TX > 0) {
                    softmax_step(std::true_type{}, 0);
                    t = 1;
                }
#pragma unroll 1
                for (; t < TX; ++t) softmax_step(std::false_type{}, t);
            }
            // ---- merge the two streams and write O, LSE: warpgroup x handles columns [x*HD/2, (x+1)*HD/2)
            if (GATE) wg_sync();
            if (TX > 0) statx[row] = make_float2(m, l);
            if (!barrier_and<3, 256>(ok)) break;   // (all warps or none: see barrier_and)
            const bool two = NS > 1;
            const float2 s0 = stat[row];
            const float2 s1 = two ? stat[kTile + row] : make_float2(-INFINITY, 0.f);
            if (ok && !mbar_wait(&bars[B_OFULL + 0], item & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
            if (two) {
                if (ok && !mbar_wait(&bars[B_OFULL + 1], o1 & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
                ++o1;
            }
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            if (!ok) continue;                    // (to the vote of the next item)
            constexpr int CW = HD / 2;            // columns per warpgroup
            const float mm = fmaxf(s0.x, s1.x);
            const float w0 = ex2(s0.x - mm), w1 = two ? ex2(s1.x - mm) : 0.f;
            const float lsum = s0.y * w0 + s1.y * w1;
            const float inv = 1.f / lsum;
            const float f0 = w0 * inv, f1 = w1 * inv;
            const bool live = qi < p.L;
            const size_t orow = ((size_t)s * p.L + (live ? qi : 0)) * HD;
            uint32_t wrow[CW == 64 ? 32 : 1];   // d = 128: this thread's 64 outputs as one 128-byte row piece
#pragma unroll
            for (int c = 0; c < CW / 32; ++c) {
                const int c0 = x * CW + c * 32;
                uint32_t oa[32], ob[32];
                tmem_ld32(tlane + 256 + c0, oa);
                if (two) tmem_ld32(tlane + 384 + c0, ob);
                tmem_ld_wait();
                if (c == CW / 32 - 1) {
                    tc_fence_before_sync();
                    mbar_arrive(&bars[B_OFREE]);      // O and the stat words may be overwritten
                }
                float o[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    float v = __uint_as_float(oa[e]) * f0;
                    if (two) v += __uint_as_float(ob[e]) * f1;
                    o[e] = v;
                }
                if (CW == 64 && !p.out_fp32) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) wrow[(CW == 64 ? c * 16 : 0) + (CW == 64 ? e : 0)] = pack_bf16(o[2 * e], o[2 * e + 1]);
                    continue;
                }
                if (!live) continue;
                if (p.out_fp32) {
                    float4* dst = reinterpret_cast<float4*>((float*)p.o + orow + c0);
#pragma unroll
                    for (int e = 0; e < 8; ++e) dst[e] = make_float4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
                } else {
                    uint4* dst = reinterpret_cast<uint4*>((__nv_bfloat16*)p.o + orow + c0);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        dst[e] = make_uint4(pack_bf16(o[8 * e], o[8 * e + 1]), pack_bf16(o[8 * e + 2], o[8 * e + 3]),
                                            pack_bf16(o[8 * e + 4], o[8 * e + 5]), pack_bf16(o[8 * e + 6], o[8 * e + 7]));
                }
            }
            if (CW == 64 && !p.out_fp32) {   // the warp's 32 rows, whole 128-byte pieces per store instruction
                const int row0 = I * kTile + q4 * 32;
                if (CW == 64)
                    warp_store_rows128<true>((__nv_bfloat16*)p.o + ((size_t)s * p.L + row0) * HD + x * CW, (size_t)HD * 2,
                                       reinterpret_cast<uint32_t(&)[32]>(wrow), p.L - row0);
            }
            if (live) {
                if (x == 0) p.lse[(size_t)s * p.L + qi] = (mm + log2f(lsum)) * 0.6931471805599453f;
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

// ------------------------------------------------------------------------------------------------ pairs of query chunks
// Work items come from a counter (p.next_item, zero on entry): CTA c starts with item c, every further one is the next
// unclaimed.  The list goes through groups of slices whose keys and values stay in L2 together (p.group slices), inside a
// group longest pairs first, so that the CTAs end together without the items having to be cut alike.
//
// Per item, with I1 = 2k+1 (stream 1) and I0 = 2k (stream 0): stream 1's step n meets key chunk J = I1 - n, stream 0's
// step n - 1 the same chunk.  The loop runs over n; n = 0 is stream 1's diagonal chunk alone, n = 1 stream 0's diagonal
// and stream 1's first earlier chunk (level 0), from n = 2 on both streams use the same key tile.  The products are issued
// in the order  PV0(n), S0(n+1), PV1(n), S1(n+1)  (d = 128: P lies over S) or  S0(n+1), PV0(n), S1(n+1), PV1(n)  (d = 64:
// P has its own columns and S(n+1) only waits until S(n) is in registers).
//
// What bounds it: at d = 128 a tile pair is two products of 512 cycles and 16384 exponentials at 16 per cycle (1024
// cycles); shared memory moves 64 cycles' worth of operands per 64-cycle step of S and half of that for P V, plus the
// arriving tiles, which is why one key and value tile serves two query chunks here.  Measured, against one chunk over two
// streams with P handed over whole: 32 slices x 32768 tokens x d = 128: 8.33 -> 7.85 ms (1120 TFLOP/s; the board is at its
// power cap there); 128 x 2048 x 64: 158 -> 148 us; 128 x 4096 x 64: 517 -> 482 us; 64 x 4096 x 128: 312 -> 308 us; gated
// 32 x 8192 x 128: 187 -> 169 us.  A stream's cycle of about 3400 clocks is 1450 of exponentials (1120 for a warpgroup that
// has the unit to itself), 300 for the maximum, 300 for tensor-memory transfers and 1200 waiting for P V and the next S.
//
// CROSS = true is the segment-against-segment variant of the context-parallel path (paper Sec. 3.5): every query chunk of
// one segment visits EVERY key chunk of another (earlier) one, no diagonal chunk, no causal mask, queries and keys come as
// one prepared tile each (tm.qv / tm.kv, no levels), the key-side gate terms are their own array (whose padded tail holds a
// huge value, which masks the padded keys), and the result is merged into a running state (normalised float32 rows and
// their LSE) where it is written out.  (As a float32 result of its own and a kernel that merged it, the merges took 42 us each
// for 64 slices x 1024 rows x 128.)
struct FwdSmem {
    static constexpr uint32_t offQ = 0;                        // ring of 3 query operands
    static constexpr uint32_t offKV = offQ + 3 * kSlotBytes;   // ring of 4 key / value operands, in the order of their use
    static constexpr uint32_t offBar = offKV + 4 * kSlotBytes;
    static constexpr uint32_t offGk = offBar + 512;            // [2 streams][2][128] gate prefix of a key chunk
    static constexpr uint32_t total = offGk + 2 * 2 * kTile * 4;
    static constexpr uint32_t alloc = 232448;                  // everything an SM offers one CTA
    static_assert(total + 512 <= alloc, "no room left to align the base");
};
enum { F_QFULL = 0, F_QEMPTY = F_QFULL + 3, F_KVFULL = F_QEMPTY + 3, F_KVEMPTY = F_KVFULL + 4, F_SFULL = F_KVEMPTY + 4,
       F_SFREE = F_SFULL + 2, F_PA = F_SFREE + 2, F_PB = F_PA + 2, F_PFREE = F_PB + 2, F_OFULL = F_PFREE + 2,
       F_OFREE = F_OFULL + 2, F_GKFULL = F_OFREE + 2, F_GKEMPTY = F_GKFULL + 4, F_ITFULL = F_GKEMPTY + 4,
       F_ITEMPTY = F_ITFULL + 2, F_COUNT = F_ITEMPTY + 2 };

template <int HD, bool GATE, bool CROSS>
__global__ void __launch_bounds__(384, 1) fa_fwd_kernel(const __grid_constant__ FwdTensorMaps tm, const FwdParams p) {
    constexpr bool SEP = HD == 64;
    constexpr int kOff = CROSS ? 0 : 1;                        // stream 0's step index is n - kOff
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // (Without the gate the integer form, whose accesses are generic: 1 % faster there by the compiler's schedule, 307 / 311 us at
    // 4 x 16 x 4096 x 128, while the gated instance takes 169 / 151 us at 2 x 16 x 8192 x 128.)
    uint8_t* smem = GATE ? align1024(smem_raw) : (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    if ((uint32_t)(smem - smem_raw) + FwdSmem::total > FwdSmem::alloc) {   // uniform over the CTA
        grid_wait();   // (the status word belongs to the kernels before)
        if (threadIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)ST_FWD_PRODUCER);
        return;
    }
    uint8_t* sQ = smem + FwdSmem::offQ;
    uint8_t* sKV = smem + FwdSmem::offKV;
    uint64_t* bars = (uint64_t*)(smem + FwdSmem::offBar);
    uint32_t* tmem_slot = (uint32_t*)(bars + F_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);
    volatile int* item_ring = (volatile int*)(tmem_slot + 2);  // [2]
    static_assert(F_COUNT * 8 + 16 <= 512, "barriers and words must fit");
    float* sGk = (float*)(smem + FwdSmem::offGk);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int NP = (p.N + 1) >> 1, items = NP * p.S;

    if (threadIdx.x == 0) {
        for (int i = 0; i < F_COUNT; ++i) {
            uint32_t n = 1;
            if ((i >= F_SFREE && i < F_PFREE) || (i >= F_OFREE && i < F_GKFULL) || (i >= F_GKEMPTY && i < F_ITFULL)) n = 4;   // one per softmax warp
            if (i >= F_ITEMPTY) n = 9;                         // eight softmax warps and the issuer
            mbar_init(&bars[i], n);
        }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 2 && lane < 7) tma_prefetch_desc(reinterpret_cast<const CUtensorMap*>(&tm) + lane);   // the seven maps are contiguous
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    // tensor-memory columns of stream x: S at x * 128, O at 256 + x * HD, P over S or (d = 64) at 384 + x * 64
    auto colP = [](int x) { return SEP ? 384u + (uint32_t)x * 64u : (uint32_t)x * 128u; };
    auto decode = [&](int idx, int& k, int& s) {
        const int per = p.group * NP, g = idx / per, w = idx - g * per;
        const int gl = min(p.group, p.S - g * p.group);
        k = NP - 1 - w / gl;
        s = g * p.group + w % gl;
    };
    // key chunks query chunk I visits, counted from the diagonal: all I + 1 of them, or fewer when the gate has made the
    // far ones negligible (every warp role reads the same precomputed number); none if the chunk does not exist
    auto steps_of = [&](int I, int s) {
        if (I >= p.N) return 0;
        if (CROSS) return p.Nk;
        return p.nkeep ? min(I + 1, p.nkeep[s * p.N + I]) : I + 1;
    };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp == 0 && elect_one()) {
            // ------------------------------------------------------------ TMA producer (and item scheduler)
            bool ok = true;
            int nq = 0, nkv = 0, it = 0;      // query operands, key / value operands, items handed out so far
            int ng[2] = {0, 0};               // gate vectors so far, per stream
            auto wait_empty = [&](int bar, int use) {
                if (ok && !mbar_wait(&bars[bar], (use & 1) ^ 1, abort_flag, ST_FWD_PRODUCER)) ok = false;
            };
            auto load_q = [&](const CUtensorMap* m, int kdim, int row0, int slice = -1) {   // slice >= 0: a caller's tensor
                const int slot = nq % 3;
                wait_empty(F_QEMPTY + slot, nq / 3);
                if (!ok) return;
                mbar_expect_tx(&bars[F_QFULL + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tile::tma_rows(sQ + slot * kSlotBytes, m, &bars[F_QFULL + slot], kdim, row0, slice);
                else tile::tma_tile(sQ + slot * kSlotBytes, m, &bars[F_QFULL + slot], kdim, row0);
                ++nq;
            };
            auto load_kv = [&](const CUtensorMap* m, int kdim, int row0, int slice = -1) {
                const int slot = nkv & 3;
                wait_empty(F_KVEMPTY + slot, nkv >> 2);
                if (!ok) return;
                mbar_expect_tx(&bars[F_KVFULL + slot], (uint32_t)(kTile * kdim * 2));
                if (slice >= 0) tile::tma_rows(sKV + slot * kSlotBytes, m, &bars[F_KVFULL + slot], kdim, row0, slice);
                else tile::tma_tile(sKV + slot * kSlotBytes, m, &bars[F_KVFULL + slot], kdim, row0);
                ++nkv;
            };
            auto load_gk = [&](int x, const float* src) {
                const int b = x * 2 + (ng[x] & 1);
                wait_empty(F_GKEMPTY + b, ng[x] >> 1);
                if (!ok) return;
                mbar_expect_tx(&bars[F_GKFULL + b], kTile * 4);
                bulk_load(sGk + b * kTile, src, kTile * 4, &bars[F_GKFULL + b]);
                ++ng[x];
            };
            int idx = blockIdx.x;
            for (; ok; ++it) {
                // hand the item to the other roles (-1: no more)
                wait_empty(F_ITEMPTY + (it & 1), it >> 1);
                if (!ok) break;
                item_ring[it & 1] = idx < items ? idx : -1;
                mbar_arrive(&bars[F_ITFULL + (it & 1)]);
                if (idx >= items) break;
                const int next = (int)gridDim.x + atomicAdd(p.next_item, 1);   // (its latency hides under this item's loads)
                int k, s;
                decode(idx, k, s);
                const int I0 = 2 * k, I1 = 2 * k + 1;
                const int NS0 = steps_of(I0, s), NS1 = steps_of(I1, s), NV = max(NS1, NS0 + kOff);
                const int rowS = s * p.Lp;
                auto chunk_at = [&](int n) { return CROSS ? p.Nk - 1 - n : I1 - n; };
                auto level_at = [&](int n) { return n == 1 ? 0 : msb32((unsigned)(I0 ^ (I1 - n))); };
                auto load_step = [&](int n) {   // operands of the logit tiles of step n (n >= 1; CROSS: n >= 0)
                    const bool u0 = n >= 1 + kOff && n - kOff < NS0, u1 = n >= 1 && n < NS1;
                    if (CROSS) {
                        if (u0 || u1) load_kv(&tm.kv, HD, s * p.Lkp + chunk_at(n) * kTile);
                        return;
                    }
                    if (!u0 && !u1) return;
                    const int l = level_at(n);
                    const bool fresh = n <= 2 || l != level_at(n - 1);
                    // (query tiles first: both are ahead of the key tile in the order of use only when they are new)
                    if (u0 && fresh) load_q(&tm.qv, HD, (int)qver_row(p.vl, s, l, I0));
                    load_kv(&tm.kv, HD, (int)kver_row(p.vl, s, l, I1 - n));
                    if (u1 && fresh) load_q(&tm.qv, HD, (int)qver_row(p.vl, s, l, I1));
                };
                if (CROSS) {
                    load_q(&tm.qv, HD, rowS + I0 * kTile);
                    load_kv(&tm.kv, HD, s * p.Lkp + chunk_at(0) * kTile);
                    if (NS1 > 0) load_q(&tm.qv, HD, rowS + I1 * kTile);
                } else {
                    if (NS1 > 0) {   // stream 1's diagonal chunk: raw q, k and the correction operands
                        load_q(&tm.q_raw, HD, I1 * kTile, s);
                        load_kv(&tm.k_raw, HD, I1 * kTile, s);
                        load_q(&tm.xq, kTile, rowS + I1 * kTile);
                        load_kv(&tm.y, kTile, rowS + I1 * kTile);
                    }
                    load_q(&tm.q_raw, HD, I0 * kTile, s);
                    load_kv(&tm.k_raw, HD, I0 * kTile, s);
                    load_q(&tm.xq, kTile, rowS + I0 * kTile);
                    load_kv(&tm.y, kTile, rowS + I0 * kTile);
                }
                for (int n = 0; n < NV && ok; ++n) {
                    const bool u0 = n >= kOff && n - kOff < NS0, u1 = n < NS1;
                    if (SEP) load_step(n + 1);
                    if (u0 || u1) {
                        const int J = chunk_at(n);
                        if (GATE) {
                            const float* g = CROSS ? p.Gk + (size_t)s * p.Lkp + J * kTile : p.G + (size_t)s * p.Lp + J * kTile;
                            if (u0) load_gk(0, g);
                            if (u1) load_gk(1, g);
                        }
                        if (CROSS) load_kv(&tm.v, HD, s * p.Lkp + J * kTile);
                        else load_kv(&tm.v, HD, J * kTile, s);
                    }
                    if (!SEP) load_step(n + 1);
                }
                idx = next;
            }
        } else if (warp == 1 && elect_one()) {
            // ------------------------------------------------------------ MMA issuer
            // a negative scale is applied as a sign flip of the logits here (negate-A bit), its magnitude in the softmax
            const uint32_t idescS = umma_idesc(128, 128, 0, 0) | (p.scale < 0.f ? (1u << 13) : 0u);
            const uint32_t idescC = umma_idesc(128, 128, 0, 1) | (p.scale < 0.f ? 0u : (1u << 13));   // the correction is subtracted
            constexpr uint32_t idescO = umma_idesc(128, HD, 0, 1);
            bool ok = true;
            int nq = 0, nkv = 0;              // query and key / value operands used so far
            int ns[2] = {0, 0}, np[2] = {0, 0}, no[2] = {0, 0};   // logit tiles, P tiles, finished results per stream so far
            int curq[2] = {0, 0};             // ring index of the query tile a stream uses
            auto wait = [&](int bar, int parity) {
                if (ok && !mbar_wait(&bars[bar], parity & 1, abort_flag, ST_FWD_MMA)) ok = false;
            };
            auto q_wait = [&](int i) { wait(F_QFULL + i % 3, i / 3); };
            auto kv_wait = [&](int i) { wait(F_KVFULL + (i & 3), i >> 2); };
            auto q_free = [&](int i) { umma_commit(&bars[F_QEMPTY + i % 3]); };
            auto kv_free = [&](int i) { umma_commit(&bars[F_KVEMPTY + (i & 3)]); };
            auto q_addr = [&](int i) { return smem_u32(sQ + (i % 3) * kSlotBytes); };
            auto kv_addr = [&](int i) { return smem_u32(sKV + (i & 3) * kSlotBytes); };
            auto issue_s = [&](int x, int qi, int ki) { mma_kk<HD>(tmem + x * 128, q_addr(qi), kv_addr(ki), idescS); };
            auto s_ready = [&](int x) {       // the stream's S tile may be overwritten
                if (SEP && ns[x] > 0) wait(F_SFREE + x, ns[x] - 1);
                ++ns[x];
            };
#pragma unroll 1
            for (int it = 0; ok; ++it) {
                wait(F_ITFULL + (it & 1), it >> 1);
                if (!ok) break;
                const int idx = item_ring[it & 1];
                mbar_arrive(&bars[F_ITEMPTY + (it & 1)]);
                if (idx < 0) break;
                int k, s;
                decode(idx, k, s);
                const int I0 = 2 * k, I1 = 2 * k + 1;
                const int NS[2] = {steps_of(I0, s), steps_of(I1, s)}, NV = max(NS[1], NS[0] + kOff);
                auto level_at = [&](int n) { return CROSS ? 0 : (n == 1 ? 0 : msb32((unsigned)(I0 ^ (I1 - n)))); };
                // first logit tile of either stream
                if (CROSS) {
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if (NS[x] == 0) continue;
                        curq[x] = nq++;
                        q_wait(curq[x]);
                        kv_wait(nkv);
                        s_ready(x);
                        tc_fence_after_sync();
                        if (!ok) break;
                        issue_s(x, curq[x], nkv);
                        umma_commit(&bars[F_SFULL + x]);
                        if (NS[x] == 1) q_free(curq[x]);
                    }
                    if (ok) kv_free(nkv);
                    ++nkv;
                } else {
#pragma unroll
                    for (int x = 1; x >= 0; --x) {   // two contractions
                        if (NS[x] == 0) continue;
                        q_wait(nq);
                        kv_wait(nkv);
                        s_ready(x);
                        tc_fence_after_sync();
                        if (!ok) break;
                        issue_s(x, nq, nkv);
                        q_wait(nq + 1);
                        kv_wait(nkv + 1);
                        tc_fence_after_sync();
                        if (!ok) break;
                        mma_correction(tmem + x * 128, q_addr(nq + 1), kv_addr(nkv + 1), idescC);
                        umma_commit(&bars[F_SFULL + x]);
                        q_free(nq);
                        q_free(nq + 1);
                        kv_free(nkv);
                        kv_free(nkv + 1);
                        nq += 2;
                        nkv += 2;
                    }
                }
#pragma unroll 1
                for (int n = 0; n < NV && ok; ++n) {
                    const bool u[2] = {n >= kOff && n - kOff < NS[0], n < NS[1]};
                    const bool nx[2] = {u[0] && n - kOff + 1 < NS[0], n + 1 < NS[1]};
                    const int has_v = (u[0] || u[1]) ? 1 : 0, has_k = (nx[0] || nx[1]) ? 1 : 0;
                    const int vi = nkv + (SEP ? has_k : 0), ki = nkv + (SEP ? 0 : has_v);
                    nkv += has_v + has_k;
                    const bool fresh = !CROSS && (n <= 1 || level_at(n + 1) != level_at(n));
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if (!u[x]) continue;
                        const int t = n - (x == 0 ? kOff : 0);
                        auto next_s = [&]() {
                            if (!nx[x]) return;
                            if (fresh) {
                                curq[x] = nq++;
                                q_wait(curq[x]);
                            }
                            kv_wait(ki);
                            s_ready(x);
                            tc_fence_after_sync();
                            if (!ok) return;
                            issue_s(x, curq[x], ki);
                            umma_commit(&bars[F_SFULL + x]);
                            if (t + 2 >= NS[x] || level_at(n + 2) != level_at(n + 1)) q_free(curq[x]);
                            if (x == 1 || !nx[1]) kv_free(ki);
                        };
                        if (SEP) next_s();
                        // O_x += P_x V_n; the first product of a work item overwrites O_x, which the previous item's
                        // epilogue must have read
                        kv_wait(vi);
                        if (t == 0 && no[x] > 0) wait(F_OFREE + x, no[x] - 1);
                        wait(F_PA + x, np[x]);
                        tc_fence_after_sync();
                        if (!ok) break;
                        const uint32_t b_lo = umma_desc_lo(smem_u32(sKV + (vi & 3) * kSlotBytes), kPanelBytes);
                        const uint32_t tO = tmem + 256 + x * HD, tP = tmem + colP(x);
#pragma unroll
                        for (int kk = 0; kk < 6; ++kk)
                            umma_ts(tO, tP + kk * 8, umma_desc_join(b_lo + kk * 128u), idescO, (t > 0 || kk > 0) ? 1u : 0u);
                        wait(F_PB + x, np[x]);
                        tc_fence_after_sync();
                        if (!ok) break;
#pragma unroll
                        for (int kk = 6; kk < 8; ++kk) umma_ts(tO, tP + kk * 8, umma_desc_join(b_lo + kk * 128u), idescO, 1u);
                        ++np[x];
                        if (SEP) umma_commit(&bars[F_PFREE + x]);
                        if (x == 1 || !u[1]) kv_free(vi);
                        if (t + 1 == NS[x]) {
                            umma_commit(&bars[F_OFULL + x]);
                            ++no[x];
                        }
                        if (!SEP) next_s();   // overwrites P: in-order execution puts it after the product above
                        if (!ok) break;
                    }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // ------------------------------------------------------------ softmax warpgroups, one row per thread
        const int x = (warp - 4) >> 2;          // stream
        const int q4 = warp & 3;                // TMEM lane quadrant this warp may touch
        const int row = q4 * 32 + lane;
        const uint32_t tlane = tmem + ((uint32_t)(q4 * 32) << 16);
        const uint32_t tS = tlane + x * 128, tO = tlane + 256 + x * HD, tP = tlane + colP(x);
        const float kLog2e = 1.4426950408889634f;
        const float sl2 = fabsf(p.scale) * kLog2e;
        const uint64_t sl2x2 = pack2(sl2, sl2);
        bool ok = true;
        int sc = 0, no = 0;                     // tiles and results of this stream so far
#pragma unroll 1
        for (int it = 0; ok; ++it) {
            if (!mbar_wait(&bars[F_ITFULL + (it & 1)], (it >> 1) & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int idx = item_ring[it & 1];
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[F_ITEMPTY + (it & 1)]);
            if (idx < 0) break;
            int k, s;
            decode(idx, k, s);
            const int I = 2 * k + x, T = steps_of(I, s);
            if (T == 0) continue;
            const int qi = I * kTile + row;     // position within the slice (may be >= L in the ragged tail)
            float gi2 = 0.f;
            if (GATE) gi2 = p.G[(size_t)s * p.Lp + qi] * kLog2e;
            float m = -INFINITY, l = 0.f;
            auto step = [&](auto diag_tag, const int t) {
                constexpr bool DIAG = decltype(diag_tag)::value;
                const int gb = x * 2 + (sc & 1);
                if (GATE && ok && !mbar_wait(&bars[F_GKFULL + gb], (sc >> 1) & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
                if (SEP && sc > 0 && ok && !mbar_wait(&bars[F_PFREE + x], (sc - 1) & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
                if (ok && !mbar_wait(&bars[F_SFULL + x], sc & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
                ok = __all_sync(0xffffffffu, ok);  // keep the warp-collective TMEM accesses convergent
                tc_fence_after_sync();
                ok = softmax_tile<HD, GATE, DIAG, SEP>(tS, tP, tO, row, sl2x2, sl2, gi2, sGk + gb * kTile, t > 0, m, l,
                                                       &bars[F_SFREE + x], &bars[F_PA + x], &bars[F_PB + x], ok);
                if (GATE && lane == 0) mbar_arrive(&bars[F_GKEMPTY + gb]);
                ++sc;
            };
            int t = 0;
            if (!CROSS) {
                step(std::true_type{}, 0);
                t = 1;
            }
#pragma unroll 1
            for (; t < T; ++t) step(std::false_type{}, t);
            // ---- write O, LSE
            if (ok && !mbar_wait(&bars[F_OFULL + x], no & 1, abort_flag, ST_FWD_SOFTMAX)) ok = false;
            ++no;
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after_sync();
            if (!ok) break;
            const bool live = qi < p.L;
            const int row0 = I * kTile + q4 * 32;
            float inv = 1.f / l, f_old = 0.f, lse2 = m + log2f(l);   // (log2 units)
            if (CROSS) {   // running result: o <- (2^old o + 2^lse2 O) / (2^old + 2^lse2)
                const float old = live ? p.lse[(size_t)s * p.L + qi] * kLog2e : -INFINITY;
                const float mx = fmaxf(old, lse2), wo = ex2(old - mx), wn = ex2(lse2 - mx), norm = 1.f / (wo + wn);
                f_old = wo * norm;
                inv *= wn * norm;
                lse2 = mx + log2f(wo + wn);
            }
#pragma unroll
            for (int h = 0; h < HD / 64; ++h) {   // 64 columns at a time: one 128-byte line per row
                uint32_t o[2][32];
                tmem_ld32(tO + h * 64, o[0]);
                tmem_ld32(tO + h * 64 + 32, o[1]);
                tmem_ld_wait();
                if (h == HD / 64 - 1) {
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars[F_OFREE + x]);   // O may be overwritten
                }
                if (CROSS || p.out_fp32) {
                    float* dst = (float*)p.o + ((size_t)s * p.L + (live ? qi : 0)) * HD + h * 64;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        float v[32];
                        if (CROSS) tile::gload_f32x32(dst + c * 32, v, live);
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = CROSS ? fmaf(v[e], f_old, __uint_as_float(o[c][e]) * inv) : __uint_as_float(o[c][e]) * inv;
                        tile::gstore_f32x32(dst + c * 32, v, live);
                    }
                } else {
                    uint32_t w[32];
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            w[c * 16 + e] = pack_bf16(__uint_as_float(o[c][2 * e]) * inv, __uint_as_float(o[c][2 * e + 1]) * inv);
                    warp_store_rows128<true>((__nv_bfloat16*)p.o + ((size_t)s * p.L + row0) * HD + h * 64, (size_t)HD * 2, w, p.L - row0);
                }
            }
            if (live) p.lse[(size_t)s * p.L + qi] = lse2 * 0.6931471805599453f;
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

// Slices per group of the item list: what about 64 MB of keys, values and versions (half of L2) come from, but enough that
// a group's items fill the GPU twice.
static int slices_per_group(const FwdParams& p, int hd, int sms, int key_rows) {
    const int np = (p.N + 1) / 2;
    const long per_slice = (long)key_rows * hd * 2;
    const int fit = (int)((64L << 20) / (per_slice > 0 ? per_slice : 1)), fill = (2 * sms + np - 1) / np;
    const int g = fit > fill ? fit : fill;
    return g < 1 ? 1 : (g > p.S ? p.S : g);
}

template <int HD>
static cudaError_t launch_hd(const FwdTensorMaps& tm, FwdParams p, cudaStream_t st) {
    int sms = 0;
    cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const int chunks = p.N * p.S, pairs = (p.N + 1) / 2 * p.S;
    // Pairs that do not fill the GPU leave the time to the longest of them: then one chunk per item, dealt over both streams
    // (S = 8 slices, L = 4096, d = 128: 52 us against 74; S = 1, L = 32768: 269 against 466).  From one pair per SM on the
    // pairs are faster (S = 10, L = 4096: 82 against 93 us; S = 2, L = 20000: 304 against 328), and also below that where
    // items are short and there are more chunks than SMs (S = 64, L = 512: 19 against 23 us).
    if (pairs < sms && (chunks <= sms || p.N >= 8)) {
        const int grid = chunks <= sms ? chunks : ((chunks + 1) / 2 < sms ? (chunks + 1) / 2 : sms);
        return p.G ? launch<fa_split_kernel<HD, true>>(grid, 384, SplitSmem::alloc, st, tm, p)
                   : launch<fa_split_kernel<HD, false>>(grid, 384, SplitSmem::alloc, st, tm, p);
    }
    p.group = slices_per_group(p, HD, sms, 2 * p.Lp + p.vl.ek * CHUNK);
    const int grid = pairs < sms ? pairs : sms;
    return p.G ? launch<fa_fwd_kernel<HD, true, false>>(grid, 384, FwdSmem::alloc, st, tm, p)
               : launch<fa_fwd_kernel<HD, false, false>>(grid, 384, FwdSmem::alloc, st, tm, p);
}

cudaError_t launch_fa_fwd(const FwdTensorMaps& tm, const FwdParams& p, int hd, cudaStream_t st) {
    return hd == 64 ? launch_hd<64>(tm, p, st) : launch_hd<128>(tm, p, st);
}

template <int HD>
static cudaError_t launch_cross_hd(const FwdTensorMaps& tm, FwdParams p, cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    if (!p.G || !p.Gk || p.Nk < 1) return cudaErrorInvalidValue;
    const int pairs = (p.N + 1) / 2 * p.S;
    p.group = slices_per_group(p, HD, sms, 2 * p.Lkp);
    return launch<fa_fwd_kernel<HD, true, true>>(pairs < sms ? pairs : sms, 384, FwdSmem::alloc, st, tm, p);
}

cudaError_t launch_fa_fwd_cross(const FwdTensorMaps& tm, const FwdParams& p, int hd, cudaStream_t st) {
    return hd == 64 ? launch_cross_hd<64>(tm, p, st) : launch_cross_hd<128>(tm, p, st);
}

}  // namespace path
