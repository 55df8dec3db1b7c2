// Per-chunk compact representation of the Householder product (paper Sec. 3.1 UT transform) and the
// boundary-adjusted queries / keys and chunk product built from it (Sec. 3.3), fused into one kernel.
//
// With W, Q, K the rows of one 128-token chunk and D = diag(beta):
//   Gm = W W^T,  Xq = lower(Q W^T),  Xk = strictLower(W K^T)
//   T~ = (I + strictLower(D Gm))^-1 D        (16 x 16 blocks by float32 substitution, merged by warp-level products: tri_inverse)
//   U = T~ W,  Y = T~ Xk
//   Qleft = Q - Xq U,  Kright = K - Y^T W,  P = I - W^T U
// Xq and Y are also the bf16 operands of the diagonal-chunk correction -Xq Y of the attention sweep.
//
// The products are 128 x 128 x {64,128} tcgen05 MMAs whose operands sit in shared memory as row-major
// 128-byte-swizzled tiles; whether a tile enters as X, X^T, on the left or on the right is only a matter of
// the descriptor's major-ness, so nothing is ever transposed in memory.  Accumulators live in tensor memory and
// are read back one row per thread.  T~ is kept as a bf16 pair (hi + lo) because everything downstream
// depends on it; the other intermediates are rounded to bf16 once, like the tiles the attention sweep consumes.
//
// The kernel is persistent: one CTA per SM walks over chunks.  Eight worker warps do the element-wise work (the
// triangular inverse, accumulator read-outs, conversions); one lane of a ninth warp issues the TMA loads and stores and
// every product as soon as its operands are published, so the products run underneath the workers' next phase and the
// first product of the next chunk is already finished when the workers get there.  Every result leaves by a TMA store from
// the tile that the workers have written anyway (or write for that): no worker touches global memory but for beta.
//
// What bounds it: the chain of dependent phases of one chunk (its seven tiles and four accumulators fill the SM, so there is
// one chunk per SM at a time) and, in the backward's instance, bursts of stores: 416 KB per chunk against about 23 bytes per
// cycle and SM of memory bandwidth.  Cycles per chunk at B=4, H=16, L=4096, d=128 (backward's instance) / 32 x 32768 x 128
// (forward's): 29 k / 25 k, of which the inverse 9.7 k, 116 product steps 7.5 k (mostly underneath), E1 1.9 k, Xk and Xq
// 3 k, U and Y 1.8 k, P, Q<- and K-> 3.9 k, the rest waits.  With the inverse in float32 loops plus one tcgen05 level and
// rows stored and fetched by the workers: 43.5 k / 33.9 k.  Time 352 -> 243 us and 1240 -> 940 us; 128 x 2048 x 64: 278 -> 206.
#include <type_traits>
#include "tileops.cuh"

namespace path {
using namespace tc5;

namespace {

using namespace tile;

// Seven 32 KB tile slots.  0: W.  1, 2: N hi, lo -> (I + N)^-1 -> T~ -> U -> Q, K once more.  3: K -> Xq hi -> P lo.
// 4: Q -> Xq lo -> P hi.  5: Xk hi -> Y hi -> Q<-.  6: Xk lo -> Y lo -> K->.  The four results of a chunk wait in slots 3 - 6
// for their TMA stores to read them while the next chunk's triangular inverse runs in slots 1, 2 and in registers; its Q and K
// arrive meanwhile.
struct PrepSmem {
    static constexpr uint32_t offBar = 7 * kTileB;
    static constexpr uint32_t offBeta = offBar + 256;                                      // [128] float
    static constexpr uint32_t total = offBeta + kT * 4;
    static constexpr uint32_t alloc = total + 1024;
};

// mbarriers.  Issuer -> workers: one per group of products (and the TMA load, which only the issuer waits for).
// Workers -> issuer (256 arrivals): operands published / accumulators drained.  Each completes once per chunk.
enum { B_LOAD = 0, B_LOADQK, B_GM, B_XQK, B_U, B_Y, B_G3A, B_G3B, B_ST, B_LOADR, R_TT, R_XK, R_XQ, R_U, R_Y, R_P, R_E3, B_COUNT };
constexpr int kWorkers = 256, kThreads = 384;   // warps 8..11: the issuer's warpgroup (one active lane)

// Barriers over the eight worker warps.  bar.sync / bar.red are warp-aligned instructions: a warp whose lanes left a
// loop at different times must reconverge first, or the part that runs ahead is taken for the whole warp.
__device__ __forceinline__ void wsync() {
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
}
__device__ __forceinline__ bool wsync_and(bool ok) { return barrier_and<1, 256>(ok); }

// ------------------------------------------------------------------------------------------------ triangular inverse
// In place in the two slots of a bf16 pair of swizzled tiles (aH, aL):  N strictly lower -> T~ = (I + N)^-1 D.  The two 64 x 64
// diagonal blocks of N arrive in float32, in the 16 KB that their pair takes up later (fel below); the 64 x 64 block C under the
// diagonal as a pair, and zeros above it.  16 x 16 diagonal blocks by float32 forward substitution, then three merge levels
// [[A,0],[C,B]]^-1 = [[A^-1,0],[-B^-1 C A^-1, B^-1]]  of 16-, 32- and 64-row blocks as warp-level products.  A warp owns a
// 16-row strip of B^-1 C: its accumulators are the A fragments of the second product, so nothing goes through memory in between.
//
// Precision.  The first two levels read and write float32, their products split every operand into two tf32 numbers (mma.sync
// m16n8k8, lo x lo left out: 2^-22 of a product).  The last level takes bf16 pairs (m16n8k16), the form T~ is kept in
// afterwards, and the blocks on the diagonal are scaled by D in float32 before they become one.  Relative error of T~ against
// float64 over 128 chunks, d = 64 / 128, with N and all levels in bf16 pairs -> like this, which is what float32 loops for
// the first two levels give (rounding the exact T~ to a pair: 2.3e-6): random unit w 5.1e-6 / 3.8e-6 -> 4.0e-6 / 3.2e-6; beta = 2
// and w around one direction 1.7e-4 / 1.6e-4 -> 8.4e-5 / 8.2e-5; beta = 2 and four directions 7.7e-5 / 6.2e-5 -> 1.5e-5 / 1.5e-5.
//
// Time: 9.7 thousand cycles (substitution 2.0, merges 0.9, 2.2, 3.3, the change to pairs 0.7, scaling 0.6), 8 with pairs throughout;
// float32 loops up to 64 rows plus one tcgen05 level took 14.  The merges are bound by the rate of mma.sync, about 20 cycles
// each and scheduler for either shape (dependent products in three separate accumulators changed nothing).
// Why not tcgen05: its smallest tile has 64 rows and every product costs a round trip through tensor memory, a shared
// memory tile and two hand-overs (about 1500 cycles each, measured); here the blocks are 16 to 64 rows and dependent.
__device__ __forceinline__ uint32_t frag_addr(uint32_t tile_, int r0, int c0, int lane) {
    const int rr = r0 + (lane & 15), c = c0 + (lane >> 4) * 8;
    return tile_ + (uint32_t)(c >> 6) * kPanelB + sw128_off((uint32_t)rr, (uint32_t)((c & 63) >> 3));
}
__device__ __forceinline__ void ldsm4(uint32_t (&f)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&f)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma1688(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d[16 x 16] += (ah + al) (bh + bl) without al bl
__device__ __forceinline__ void mma_pair(float (&d)[2][4], const uint32_t (&ah)[4], const uint32_t (&al)[4], const uint32_t (&bh)[4],
                                         const uint32_t (&bl)[4]) {
#pragma unroll
    for (int n = 0; n < 2; ++n) mma16816(d[n], ah, bh[2 * n], bh[2 * n + 1]);
#pragma unroll
    for (int n = 0; n < 2; ++n) mma16816(d[n], ah, bl[2 * n], bl[2 * n + 1]);
#pragma unroll
    for (int n = 0; n < 2; ++n) mma16816(d[n], al, bh[2 * n], bh[2 * n + 1]);
}
__device__ __forceinline__ uint32_t split_pair(float a, float b, uint32_t& l) {   // packed hi, l = packed lo
    const uint32_t h = pack_bf16(a, b);
    l = pack_bf16(a - __uint_as_float(h << 16), b - __uint_as_float(h & 0xffff0000u));
    return h;
}
// hi (x cut off), l = lo (the rest, rounded: 11 + 11 bits and a sign).  Plain integer operations: cvt.rna.tf32 took 4 % longer.
__device__ __forceinline__ uint32_t split_tf32(float x, uint32_t& l) {
    const uint32_t h = __float_as_uint(x) & 0xffffe000u;
    l = (__float_as_uint(x - __uint_as_float(h)) + 0x1000u) & 0xffffe000u;
    return h;
}
// Element (r, c) of the float32 diagonal block b (64 x 64): rows 0 - 31 where the block's hi tile goes later, rows 32 - 63 at its lo
// tile.  Columns are permuted in groups of four so that fragment loads (8 rows x 8 columns, rows 2t and 2t + 1) and row-wise
// 16-byte accesses are free of bank conflicts.
__device__ __forceinline__ float* fel(uint8_t* aH, uint8_t* aL, int b, int r, int c) {
    const int f = (((r & 3) ^ ((r >> 2) & 1)) << 3) | (r & 4);
    return reinterpret_cast<float*>((r & 32 ? aL : aH) + b * (kPanelB + 8192)) + (r & 31) * 64 + (c ^ f);
}
// Fragments of float32 blocks for m16n8k8.  Slots t and t + 4 of the contraction stand for columns 2t and 2t + 1 of A and
// rows 2t and 2t + 1 of B, which makes an accumulator tile of one product an A fragment of the next as it is.
struct Tf32A { uint32_t h[4], l[4]; };
__device__ __forceinline__ Tf32A tf32_a(uint8_t* aH, uint8_t* aL, int b, int r0, int c0, int lane) {
    const float2 x = *reinterpret_cast<const float2*>(fel(aH, aL, b, r0 + (lane >> 2), c0 + 2 * (lane & 3)));
    const float2 y = *reinterpret_cast<const float2*>(fel(aH, aL, b, r0 + 8 + (lane >> 2), c0 + 2 * (lane & 3)));
    Tf32A a;
    a.h[0] = split_tf32(x.x, a.l[0]); a.h[1] = split_tf32(y.x, a.l[1]);
    a.h[2] = split_tf32(x.y, a.l[2]); a.h[3] = split_tf32(y.y, a.l[3]);
    return a;
}
__device__ __forceinline__ Tf32A tf32_a(const float (&d)[4]) {
    Tf32A a;
    a.h[0] = split_tf32(d[0], a.l[0]); a.h[1] = split_tf32(d[2], a.l[1]);
    a.h[2] = split_tf32(d[1], a.l[2]); a.h[3] = split_tf32(d[3], a.l[3]);
    return a;
}
// d[16 x 8] += A B, B the 8 x 8 block at (r0, c0)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const Tf32A& a, uint8_t* aH, uint8_t* aL, int b, int r0, int c0, int lane) {
    uint32_t h[2], l[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) h[x] = split_tf32(*fel(aH, aL, b, r0 + 2 * (lane & 3) + x, c0 + (lane >> 2)), l[x]);
    mma1688(d, a.h, h[0], h[1]);
    mma1688(d, a.h, l[0], l[1]);
    mma1688(d, a.l, h[0], h[1]);
}
// One merge level of blocks of NBK 16-row strips (1, 2) inside the float32 blocks.  NBK = 1: four pairs, the two warps of a pair take
// 8 columns of the result each; NBK = 2: a warp takes 16 x 16, the two warps that share a scheduler (w, w + 4) a long and a
// short strip (B^-1 is lower triangular: strip rb needs its first rb + 1 blocks).
template <int NBK>
__device__ __forceinline__ void merge_f32(uint8_t* aH, uint8_t* aL, int warp, int lane) {
    constexpr int NT = NBK;                       // 8-column tiles of the result per warp
    const int hw = warp >> 2, w4 = warp & 3;
    const int b = NBK == 1 ? w4 >> 1 : w4 & 1, rb = NBK == 1 ? 0 : ((w4 >> 1) ^ hw);
    const int base_a = NBK == 1 ? (w4 & 1) * 32 : 0, base_b = base_a + NBK * 16, row0 = base_b + rb * 16;
    const int k_lo = NBK == 1 ? 0 : hw, col0 = base_a + hw * NBK * 8;   // A^-1 is lower triangular: columns col0.. need no earlier block
    float m[NT][4], p1[NBK][2][4];
#pragma unroll
    for (int k = 0; k < NBK; ++k)
#pragma unroll
        for (int x = 0; x < 8; ++x) p1[k][x >> 2][x & 3] = 0.f;
#pragma unroll
    for (int x = 0; x < 4 * NT; ++x) m[x >> 2][x & 3] = 0.f;
#pragma unroll
    for (int j = 0; j < NBK; ++j)
#pragma unroll
        for (int k8 = 0; k8 < 2; ++k8) {
            if (j > rb) continue;
            const Tf32A a = tf32_a(aH, aL, b, row0, base_b + j * 16 + k8 * 8, lane);
#pragma unroll
            for (int kb = 0; kb < NBK; ++kb) {
                if (kb < k_lo) continue;
#pragma unroll
                for (int n = 0; n < 2; ++n) mma_tf32(p1[kb][n], a, aH, aL, b, base_b + j * 16 + k8 * 8, base_a + kb * 16 + n * 8, lane);
            }
        }
#pragma unroll
    for (int kb = 0; kb < NBK; ++kb) {
        if (kb < k_lo) continue;
#pragma unroll
        for (int k8 = 0; k8 < 2; ++k8) {
            const Tf32A a = tf32_a(p1[kb][k8]);
#pragma unroll
            for (int n = 0; n < NT; ++n) mma_tf32(m[n], a, aH, aL, b, base_a + kb * 16 + k8 * 8, col0 + n * 8, lane);
        }
    }
    wsync();   // the other warps of the pair read C as well
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int y = 0; y < 2; ++y)
            *reinterpret_cast<float2*>(fel(aH, aL, b, row0 + (lane >> 2) + 8 * y, col0 + n * 8 + 2 * (lane & 3))) =
                make_float2(-m[n][2 * y], -m[n][2 * y + 1]);
}
// The last level, on the pairs: strips of 64 x 64 blocks, the result scaled by D.
__device__ __forceinline__ void merge_pairs(uint8_t* aH, uint8_t* aL, const float* bt, int warp, int lane) {
    constexpr int NBK = 4, CBN = 2;               // 16-row strips per block, 16-column blocks of the result per warp
    const uint32_t tH = smem_u32(aH), tL = smem_u32(aL);
    const int hw = warp >> 2, w4 = warp & 3, rb = hw ? 3 - w4 : w4, cb0 = hw * CBN, row0 = 64 + rb * 16;
    float m[CBN][2][4], p1[NBK][2][4];
#pragma unroll
    for (int k = 0; k < NBK; ++k)
#pragma unroll
        for (int x = 0; x < 8; ++x) p1[k][x >> 2][x & 3] = 0.f;
#pragma unroll
    for (int k = 0; k < CBN; ++k)
#pragma unroll
        for (int x = 0; x < 8; ++x) m[k][x >> 2][x & 3] = 0.f;
#pragma unroll 1
    for (int j = 0; j <= rb; ++j) {
        uint32_t ah[4], al[4];
        ldsm4(ah, frag_addr(tH, row0, 64 + j * 16, lane));
        ldsm4(al, frag_addr(tL, row0, 64 + j * 16, lane));
#pragma unroll
        for (int kb = 0; kb < NBK; ++kb) {
            if (kb < cb0) continue;       // A^-1 is lower triangular: columns cb0.. need no earlier block
            uint32_t bh[4], bl[4];
            ldsm4t(bh, frag_addr(tH, 64 + j * 16, kb * 16, lane));
            ldsm4t(bl, frag_addr(tL, 64 + j * 16, kb * 16, lane));
            mma_pair(p1[kb], ah, al, bh, bl);
        }
    }
#pragma unroll
    for (int kb = 0; kb < NBK; ++kb) {
        if (kb < cb0) continue;
        uint32_t ah[4], al[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) ah[x] = split_pair(p1[kb][x >> 1][(x & 1) * 2], p1[kb][x >> 1][(x & 1) * 2 + 1], al[x]);
#pragma unroll
        for (int i = 0; i < CBN; ++i) {
            if (kb < cb0 + i) continue;
            uint32_t bh[4], bl[4];
            ldsm4t(bh, frag_addr(tH, kb * 16, (cb0 + i) * 16, lane));
            ldsm4t(bl, frag_addr(tL, kb * 16, (cb0 + i) * 16, lane));
            mma_pair(m[i], ah, al, bh, bl);
        }
    }
    wsync();   // the other strips read C as well
#pragma unroll
    for (int i = 0; i < CBN; ++i)
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int col = (cb0 + i) * 16 + n * 8 + 2 * (lane & 3);
            const float s0 = -bt[col], s1 = -bt[col + 1];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const int rr = row0 + (lane >> 2) + 8 * y;
                uint32_t l;
                const uint32_t h = split_pair(s0 * m[i][n][2 * y], s1 * m[i][n][2 * y + 1], l);
                const uint32_t off = (uint32_t)(col >> 6) * kPanelB + sw128_off((uint32_t)rr, (uint32_t)((col & 63) >> 3)) + (col & 7) * 2;
                *reinterpret_cast<uint32_t*>(aH + off) = h;
                *reinterpret_cast<uint32_t*>(aL + off) = l;
            }
        }
}
__device__ __forceinline__ void tri_inverse(uint8_t* aH, uint8_t* aL, const float* bt, int warp, int lane, int row, int half) {
    {   // diagonal block `warp`: lane j (and its copy j + 16) keeps column j in registers
        const int b = warp >> 2, o = (warp & 3) * 16, j = lane & 15;
        float x[16];
#pragma unroll
        for (int g = 0; g < 4; ++g) {   // four rows at a time: their loads are issued together, ahead of the dependent sums
            float4 f[4][4];
#pragma unroll
            for (int y = 0; y < 4; ++y)
#pragma unroll
                for (int c = 0; c <= g; ++c) f[y][c] = *reinterpret_cast<const float4*>(fel(aH, aL, b, o + 4 * g + y, o + 4 * c));
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int rr = 4 * g + y;
                float acc[4] = {rr == j ? 1.f : 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int c = 0; c < g; ++c) {
                    acc[0] -= f[y][c].x * x[4 * c];
                    acc[1] -= f[y][c].y * x[4 * c + 1];
                    acc[2] -= f[y][c].z * x[4 * c + 2];
                    acc[3] -= f[y][c].w * x[4 * c + 3];
                }
                float a = (acc[0] + acc[1]) + (acc[2] + acc[3]);
                if (y > 0) a -= f[y][g].x * x[4 * g];
                if (y > 1) a -= f[y][g].y * x[4 * g + 1];
                if (y > 2) a -= f[y][g].z * x[4 * g + 2];
                x[rr] = rr >= j ? a : 0.f;
            }
        }
        __syncwarp();
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) *fel(aH, aL, b, o + rr + (lane >> 4) * 8, o + j) = lane < 16 ? x[rr] : x[rr + 8];
    }
    wsync();
    merge_f32<1>(aH, aL, warp, lane);
    wsync();
    merge_f32<2>(aH, aL, warp, lane);
    wsync();
    // the diagonal blocks become pairs, in the same place; this thread's 32 entries stay in registers until they are scaled
    float d[32];
    const int cb = (row & 64) + half * 32;
#pragma unroll
    for (int x = 0; x < 32; x += 4) {
        const float4 v = *reinterpret_cast<const float4*>(fel(aH, aL, row >> 6, row & 63, half * 32 + x));
        d[x] = v.x; d[x + 1] = v.y; d[x + 2] = v.z; d[x + 3] = v.w;
    }
    wsync();
    uint32_t hi[16], lo[16];
    split32(d, hi, lo);
    tile_store_w16(aH, row, cb, hi);
    tile_store_w16(aL, row, cb, lo);
    wsync();
    merge_pairs(aH, aL, bt, warp, lane);   // (from its barrier on nobody reads the diagonal blocks any more)
#pragma unroll
    for (int x = 0; x < 32; x += 4) {
        const float4 v = *reinterpret_cast<const float4*>(bt + cb + x);
        d[x] *= v.x; d[x + 1] *= v.y; d[x + 2] *= v.z; d[x + 3] *= v.w;
    }
    split32(d, hi, lo);
    tile_store_w16(aH, row, cb, hi);
    tile_store_w16(aL, row, cb, lo);
}

// MODE: PREP_FWD = everything the forward needs; PREP_SAVE = also keeps the tiles of the chain rule (the backward's instance);
// PREP_KEYS = the key side only (prompt key cache: Kright and the chunk products; no query is involved, so Xq, Xq U,
// Qleft and the diagonal-correction operands are left out and q is not even loaded).
template <int HD, int MODE>
__global__ void __launch_bounds__(kThreads, 1) chunk_prep_kernel(const __grid_constant__ PrepTensorMaps tm, const PrepParams p,
                                                                      const int nchunks) {
    constexpr bool SAVE = MODE == PREP_SAVE, KEYS = MODE == PREP_KEYS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    auto slot = [&](int i) { return smem + i * kTileB; };
    uint8_t* sW = slot(0);
    float* bt = (float*)(smem + PrepSmem::offBeta);
    uint64_t* bars = (uint64_t*)(smem + PrepSmem::offBar);
    uint32_t* tmem_slot = (uint32_t*)(bars + B_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane;       // accumulator row (TMEM lane) of a worker thread
    const int half = (warp >> 2) & 1;             // which half of the accumulator's columns

    if (tid == 0) {
        for (int i = 0; i < B_COUNT; ++i) mbar_init(&bars[i], i >= R_TT ? (uint32_t)kWorkers : 1u);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    auto beta_of = [&](int chunk_) {   // beta of this thread's row (tid < 128); 0 past the sequence's end
        const int pos = (chunk_ % p.N) * kT + tid;
        return pos < p.L ? p.beta[(size_t)(chunk_ / p.N) * p.L + pos] : 0.f;
    };
    if (HD == 64) {  // second panel of W must read as zeros when W^T is used with M = 128
        for (int i = tid; i < (int)(kPanelB / 16); i += kThreads) reinterpret_cast<uint4*>(sW + kPanelB)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    if (p.clear && blockIdx.x == 0 && tid < 64) p.status[tid] = 0u;   // the workspace's status block (256 bytes)
    if (tid < kT && (int)blockIdx.x < nchunks) bt[tid] = beta_floor(beta_of(blockIdx.x));
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t base_ = smem_u32(smem);
    constexpr int KS = HD / 16;  // k-steps over the head dimension
    // tensor-memory columns:  0: Gm -> U   128: Xq -> W^T U   256: Xk -> Xq U   384: Y -> Y^T W

    if (warp >= kWorkers / 32) {
        // ------------------------------------------------------------------ issuer
        asm volatile("setmaxnreg.dec.sync.aligned.u32 96;");
        if (warp == kWorkers / 32 && elect_one()) {
            auto wait = [&](int b, uint32_t par) { return mbar_wait(&bars[b], par, abort_flag, ST_PREP); };
            auto fetch = [&](const CUtensorMap* m, int i, int b, int chunk_) {
                tma_rows(slot(i), m, &bars[b], HD, (chunk_ % p.N) * kT, chunk_ / p.N);
            };
            auto load_w = [&](int chunk_) {
                mbar_expect_tx(&bars[B_LOAD], kT * HD * 2);
                fetch(&tm.w, 0, B_LOAD, chunk_);
            };
            auto load_qk = [&](int chunk_) {
                mbar_expect_tx(&bars[B_LOADQK], (KEYS ? 1 : 2) * kT * HD * 2);
                if (!KEYS) fetch(&tm.q, 4, B_LOADQK, chunk_);
                fetch(&tm.k, 3, B_LOADQK, chunk_);
            };
            auto store = [&](const CUtensorMap* m, int i, int ncols, int row0) {
                for (int h = 0; h < ncols / 64; ++h) tma_store_2d(m, slot(i) + h * kPanelB, h * 64, row0);
            };
            int chunk = blockIdx.x;
            bool ok = chunk < nchunks;
            if (ok) {
                load_w(chunk);
                load_qk(chunk);
                ok = wait(B_LOAD, 0);
                if (ok) {
                    tc_fence_after_sync();
                    mma<OP_K, OP_K, KS, 128>(tmem + 0, base_, base_, false);
                    umma_commit(&bars[B_GM]);
                }
            }
            for (uint32_t it = 0; ok && chunk < nchunks; ++it, chunk += gridDim.x) {
                const uint32_t par = it & 1;
                const int r0 = chunk * kT, next = chunk + (int)gridDim.x;
                // (the tiles' address is made opaque once per chunk: otherwise every descriptor of every product is
                // hoisted out of this loop and the thread's small register allotment spills)
                uint32_t a0 = base_;
                asm volatile("" : "+r"(a0));
                auto t = [&](int i) { return a0 + i * kTileB; };
                // Xq, Xk: their columns' previous contents have been read (R_P, R_E3 at the end of the previous chunk)
                if (!(ok = wait(B_LOADQK, par))) break;
                tc_fence_after_sync();
                if (!KEYS) mma<OP_K, OP_K, KS, 128>(tmem + 128, t(4), t(0), false);
                mma<OP_K, OP_K, KS, 128>(tmem + 256, t(0), t(3), false);
                tma_store_wait_read();   // the previous chunk's Q<- and K-> tiles: Xk goes over them
                umma_commit(&bars[B_XQK]);
                // U = T~ W  (lo x lo terms are dropped everywhere).  In the backward's instance the tiles kept for the chain
                // rule leave through TMA stores, straight from the operand slots.
                if (!(ok = wait(R_TT, par))) break;
                tc_fence_after_sync();
                if (SAVE) {
                    store(&tm.th, 1, kT, r0);
                    store(&tm.tl, 2, kT, r0);
                    tma_store_commit();
                }
                mma<OP_K, OP_MN, 8, HD>(tmem + 0, t(1), t(0), false);
                mma<OP_K, OP_MN, 8, HD>(tmem + 0, t(2), t(0), true);
                umma_commit(&bars[B_U]);
                // Y = T~ Xk
                if (!(ok = wait(R_XK, par))) break;
                tc_fence_after_sync();
                if (SAVE) {
                    store(&tm.xk, 5, kT, r0);
                    tma_store_commit();
                }
                mma<OP_K, OP_MN, 8, 128>(tmem + 384, t(1), t(5), false);
                mma<OP_K, OP_MN, 8, 128>(tmem + 384, t(2), t(5), true);
                mma<OP_K, OP_MN, 8, 128>(tmem + 384, t(1), t(6), true);
                // B_Y lets the workers overwrite T~ (with U) and Xk (with Y): the stores must have read them
                if (SAVE) tma_store_wait_read();
                umma_commit(&bars[B_Y]);
                if (!KEYS) {
                    if (!(ok = wait(R_XQ, par))) break;
                    store(&tm.xq, 3, kT, r0);
                    tma_store_commit();
                }
                // Xq U and W^T U
                if (!(ok = wait(R_U, par))) break;
                tc_fence_after_sync();
                tma_store_wait_read();   // Xq: the workers' next tile goes over it when this group has retired
                if (SAVE) {
                    store(&tm.u, 1, HD, r0);
                    tma_store_commit();
                }
                if (!KEYS) {
                    mma<OP_K, OP_MN, 8, HD>(tmem + 256, t(3), t(1), false);
                    mma<OP_K, OP_MN, 8, HD>(tmem + 256, t(4), t(1), true);
                    mma<OP_K, OP_MN, 8, HD>(tmem + 256, t(3), t(2), true);
                }
                mma<OP_MN, OP_MN, 8, HD>(tmem + 128, t(0), t(1), false);
                mma<OP_MN, OP_MN, 8, HD>(tmem + 128, t(0), t(2), true);
                umma_commit(&bars[B_G3A]);
                // Y^T W
                if (!(ok = wait(R_Y, par))) break;
                tc_fence_after_sync();
                if (!KEYS) {
                    store(&tm.y, 5, kT, r0);
                    tma_store_commit();
                }
                mma<OP_MN, OP_MN, 8, HD>(tmem + 384, t(5), t(0), false);
                mma<OP_MN, OP_MN, 8, HD>(tmem + 384, t(6), t(0), true);
                umma_commit(&bars[B_G3B]);
                // U's slots take the Q and K rows once more (from L2), for the sums that finish Q<- and K->
                if (!(ok = wait(B_G3A, par))) break;
                mbar_expect_tx(&bars[B_LOADR], (KEYS ? 1 : 2) * kT * HD * 2);
                fetch(&tm.k, 2, B_LOADR, chunk);
                tma_store_wait_read();
                mbar_arrive(&bars[B_ST]);
                if (!KEYS) fetch(&tm.q, 1, B_LOADR, chunk);
                // W's slot is free once this chunk's last product has retired: the next chunk's Gram matrix is ready before
                // the workers have written the last results of this one
                if (next < nchunks) {
                    if (!(ok = wait(B_G3B, par))) break;
                    load_w(next);
                }
                if (!(ok = wait(R_P, par))) break;
                store(&tm.ph, 4, HD, chunk * HD);
                store(&tm.pl, 3, HD, chunk * HD);
                tma_store_commit();
                if (next < nchunks) {
                    if (!(ok = wait(B_LOAD, par ^ 1))) break;
                    tc_fence_after_sync();
                    mma<OP_K, OP_K, KS, 128>(tmem + 0, t(0), t(0), false);
                    umma_commit(&bars[B_GM]);
                    tma_store_wait_read();
                    load_qk(next);
                }
                if (!(ok = wait(R_E3, par))) break;
                if (!KEYS) store(&tm.ql, 5, HD, r0);
                store(&tm.kr, 6, HD, r0);
                tma_store_commit();
            }
            tma_store_wait_all();
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ workers
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        bool ok = true;
        uint32_t r[32];
        float v[32];
        uint32_t hi[16], lo[16];
        // lane 0 of every warp waits; the vote that follows is also the barrier that releases the other lanes
        auto wwait = [&](int b, uint32_t par) {
            bool good = ok;
            if (lane == 0 && good) good = mbar_wait(&bars[b], par, abort_flag, ST_PREP);
            good = wsync_and(good);
            tc_fence_after_sync();
            return good;
        };
        int chunk = blockIdx.x;
        for (uint32_t it = 0; chunk < nchunks; ++it, chunk += gridDim.x) {
            const uint32_t par = it & 1;
            if (!(ok = wwait(B_GM, par))) break;

            // ---- E1: N = strictLower(D Gm) into slots 1, 2 as tri_inverse wants it: the two diagonal blocks in float32, the rest (and
            // the zeros above the diagonal) as a bf16 pair
            uint8_t* aH = slot(1);
            uint8_t* aL = slot(2);
            for (int c = 0; c < 2; ++c) {
                const int c0 = half * 64 + c * 32;
                tmem_ld32(tl + 0 + c0, r);
                tmem_ld_wait();
                const float b = bt[row];
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = (c0 + x < row) ? b * __uint_as_float(r[x]) : 0.f;
                if ((row >> 6) == half) {
#pragma unroll
                    for (int x = 0; x < 32; x += 4)
                        *reinterpret_cast<float4*>(fel(aH, aL, half, row & 63, c * 32 + x)) = make_float4(v[x], v[x + 1], v[x + 2], v[x + 3]);
                } else {
                    split32(v, hi, lo);
                    tile_store_w16(aH, row, c0, hi);
                    tile_store_w16(aL, row, c0, lo);
                }
            }
            wsync();
            tri_inverse(aH, aL, bt, warp, lane, row, half);   // -> T~ = (I + N)^-1 D
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_TT]);

            if (!(ok = wwait(B_XQK, par))) break;
            // ---- E1b: Xk = strictLower(.) -> bf16 hi / lo tiles (slots 5, 6), then Xq = lower(.) (slots 3, 4)
            for (int c = 0; c < 2; ++c) {
                const int c0 = half * 64 + c * 32;
                tmem_ld32(tl + 256 + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = (c0 + x < row) ? __uint_as_float(r[x]) : 0.f;
                split32(v, hi, lo);
                tile_store_w16(slot(5), row, c0, hi);
                tile_store_w16(slot(6), row, c0, lo);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_XK]);
            for (int c = 0; c < (KEYS ? 0 : 2); ++c) {
                const int c0 = half * 64 + c * 32;
                tmem_ld32(tl + 128 + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = (c0 + x <= row) ? __uint_as_float(r[x]) : 0.f;
                split32(v, hi, lo);
                tile_store_w16(slot(3), row, c0, hi);
                tile_store_w16(slot(4), row, c0, lo);
            }
            if (!KEYS) {
                fence_proxy_async_smem();
                tc_fence_before_sync();
                mbar_arrive(&bars[R_XQ]);
            }

            // ---- E2: U -> hi / lo tiles over T~ (slots 1, 2) once Y = T~ Xk has retired; Y -> hi / lo tiles over Xk
            // (slots 5, 6)
            if (!(ok = wwait(B_U, par))) break;
            uint32_t uh[HD / 64][16], ul[HD / 64][16];
#pragma unroll
            for (int c = 0; c < HD / 64; ++c) {
                const int c0 = half * (HD / 2) + c * 32;
                tmem_ld32(tl + 0 + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r[x]);
                split32(v, uh[c], ul[c]);
            }
            if (!(ok = wwait(B_Y, par))) break;
#pragma unroll
            for (int c = 0; c < HD / 64; ++c) {
                const int c0 = half * (HD / 2) + c * 32;
                tile_store_w16(slot(1), row, c0, uh[c]);
                tile_store_w16(slot(2), row, c0, ul[c]);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_U]);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int c0 = half * 64 + c * 32;
                tmem_ld32(tl + 384 + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r[x]);
                split32(v, hi, lo);
                tile_store_w16(slot(5), row, c0, hi);
                tile_store_w16(slot(6), row, c0, lo);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_Y]);

            // ---- E3: P = I - W^T U, Qleft = Q - Xq U, Kright = K - Y^T W; the Q and K rows arrive in U's slots meanwhile
            const int next = chunk + (int)gridDim.x;
            float next_beta = 0.f;
            if (tid < kT && next < nchunks) next_beta = beta_of(next);
            if (!(ok = wwait(B_G3A, par))) break;
#pragma unroll
            for (int c = 0; c < HD / 64; ++c) {   // P: hi over Xq lo, lo over Xq hi
                const int c0 = half * (HD / 2) + c * 32;
                tmem_ld32(tl + 128 + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = ((c0 + x == row) ? 1.f : 0.f) - __uint_as_float(r[x]);
                split32(v, hi, lo);
                tile_store_w16(slot(4), row, c0, hi);
                tile_store_w16(slot(3), row, c0, lo);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_P]);
            if (!(ok = wwait(B_G3B, par))) break;
            // (a wait that runs out here ends everyone's loop at the next worker barrier)
            if (!mbar_wait(&bars[B_LOADR], par, abort_flag, ST_PREP) || !mbar_wait(&bars[B_ST], par, abort_flag, ST_PREP)) ok = false;
            if (!KEYS) {   // Qleft, over Y hi, which has been stored
#pragma unroll
                for (int c = 0; c < HD / 64; ++c) {
                    const int c0 = half * (HD / 2) + c * 32;
                    float in[32];
                    tmem_ld32(tl + 256 + c0, r);
                    tmem_ld_wait();
                    tile_load32(slot(1), row, c0, in);
#pragma unroll
                    for (int x = 0; x < 32; ++x) v[x] = in[x] - __uint_as_float(r[x]);
                    tile_store32(slot(5), row, c0, v);
                }
            }
#pragma unroll
            for (int c = 0; c < HD / 64; ++c) {   // Kright, over Y lo
                const int c0 = half * (HD / 2) + c * 32;
                float in[32];
                tmem_ld32(tl + 384 + c0, r);
                tmem_ld_wait();
                tile_load32(slot(2), row, c0, in);
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = in[x] - __uint_as_float(r[x]);
                tile_store32(slot(6), row, c0, v);
            }
            fence_proxy_async_smem();
            if (tid < kT) bt[tid] = beta_floor(next_beta);   // read again only after the next chunk's first wait (a worker barrier)
            tc_fence_before_sync();
            mbar_arrive(&bars[R_E3]);
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0u, *abort_flag);
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace

cudaError_t launch_chunk_prep(const PrepTensorMaps& tm, const PrepParams& p, int hd, int mode, int nchunks,
                              cudaStream_t st) {
    int sms = 0;
    const cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const int grid = nchunks < sms ? nchunks : sms;
    auto go = [&](auto which) { return launch<decltype(which)::value>(grid, kThreads, PrepSmem::alloc, st, tm, p, nchunks); };
#define PREP(HD, MODE) go(std::integral_constant<decltype(&chunk_prep_kernel<HD, MODE>), &chunk_prep_kernel<HD, MODE>>{})
    if (mode == PREP_KEYS) return hd == 64 ? PREP(64, PREP_KEYS) : PREP(128, PREP_KEYS);
    if (hd == 64) return mode == PREP_SAVE ? PREP(64, PREP_SAVE) : PREP(64, PREP_FWD);
    return mode == PREP_SAVE ? PREP(128, PREP_SAVE) : PREP(128, PREP_FWD);
#undef PREP
}

}  // namespace path
