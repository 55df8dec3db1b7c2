// Per-chunk compact representation of the Householder product (paper Sec. 3.1 UT transform) and the
// boundary-adjusted queries / keys and chunk product built from it (Sec. 3.3), fused into one kernel.
//
// With W, Q, K the rows of one 128-token chunk and D = diag(beta):
//   Gm = W W^T,  Xq = lower(Q W^T),  Xk = strictLower(W K^T)
//   T~ = (I + strictLower(D Gm))^-1 D        (see invert_diagonal)
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
// The kernel is persistent: one CTA per SM walks over chunks, and two chunks are in work at a time.  Eight warps compute the
// triangular inverse of a chunk while eight others still turn the accumulators of the chunk before into operands and results.  One
// thread issues the products as soon as their operands are published, one the two products inside the inverse, one requests and
// stores tiles.  They meet at mbarriers only.  Every result leaves by a TMA store from the tile that the workers have written anyway
// (or write for that): no worker touches global memory but for beta.
//
// What bounds it.  d = 64: the inverse, of which its merges take 7 k cycles (mma.sync shares the tensor pipe
// with the products: 2.6 k when nothing else runs); a chunk takes 19 k.  d = 128: shared memory, which moves about 2 MB per chunk (operand reads of the
// products 1 MB, tiles in and out 0.4, the workers 0.6) = 16 k of 20 k cycles.  Both streams of code together have to fit the
// instruction caches as well: warps went without instructions for 2.3 cycles per issue until the operand group was one loop, 0.7
// since.  And the registers of each role have to do: a few spilled ones cost as much as anything here (shared memory leaves no L1),
// 13 - 18 % of the kernel at d = 64 and 2 % at d = 128.  Times, before with one group of warps and one chunk at a time / now: 2 x 16 x 8192 x 128,
// forward's instance 226 / 175 us, backward's 245 / 197; 32 x 32768 x 128 880 / 630; 128 x 2048 x 64 192 / 135 and 206 / 151.
// Tried: 32 x 32 blocks by substitution and a merge in float32 arithmetic (rows broadcast from shared memory: 4.3 k and 5.7 k
// cycles, the loads' 128 bytes per cycle bound them); T~ from tensor memory at d = 128 too (Gm of the next chunk has to be ready
// before T~: its W arrives too late, 750 -> 880 us).
#include <type_traits>
#include "tileops.cuh"

namespace path {
using namespace tc5;

namespace {

using namespace tile;

// Seven 32 KB tile slots.  0: W.  1, 2: N -> T~ (hi, lo).  3, 4: Xk -> Y (hi, lo) -> Q, K once more -> Q<-, K->.  5, 6: Q, K ->
// the next chunk's W (5) and Xq hi for its store (6) -> U (hi, lo) -> P (hi, lo).  At d = 64 a tile of the head dimension takes one
// 16 KB panel: slot 0 holds the W of two chunks by turns, slot 5 the pair of Xq's panels, then U, then P, slot 6 Q and K.
struct PrepSmem {
    static constexpr uint32_t offBar = 7 * kTileB;
    static constexpr uint32_t offBeta = offBar + 256;                                      // [2][128] float
    static constexpr uint32_t total = offBeta + 2 * kT * 4;
    static constexpr uint32_t alloc = total + 1024;
};

// mbarriers, each completing once per chunk.  L_*: tiles have arrived.  M_*: a group of products has retired.  S_*: stores have
// read their tiles, which may be written again.  R_*: workers (256 arrivals) have published operands or drained accumulators.
enum { L_W = 0, L_QK, L_WN, L_ROW, M_GM, M_IX, M_IT, M_XQK, M_U, M_Y, M_GA, M_GB, S_T, S_XQ, S_XK, S_U, S_E3,
       R_GM, R_ID, R_IX, R_TT, R_XQ, R_XK, R_U, R_Y, R_P, R_E3, B_COUNT };
static_assert(B_COUNT * 8 + 8 <= 256, "");
constexpr int kWorkers = 256;               // per group: warps 0 - 7 invert, warps 8 - 15 turn accumulators into operands and results
constexpr int kThreads = 640;               // one thread each of warp 16: issues products, 17: moves tiles, 18: products of the inverse

// Barriers over the eight warps that invert.  bar.sync / bar.red are warp-aligned instructions: a warp whose lanes left a
// loop at different times must reconverge first, or the part that runs ahead is taken for the whole warp.
__device__ __forceinline__ void wsync() {
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
}
__device__ __forceinline__ bool wsync_and(bool ok) { return barrier_and<1, 256>(ok); }

// ------------------------------------------------------------------------------------------------ triangular inverse
// In place in the two slots of a bf16 pair of swizzled tiles (aH, aL):  N strictly lower -> T~ = (I + N)^-1 D.  The two 64 x 64
// diagonal blocks of N arrive in float32, in the 16 KB that their pair takes up later (fel below); the 64 x 64 block C under them
// as a pair, and zeros above.  16 x 16 diagonal blocks by float32 forward substitution, two float32 merges
// [[A,0],[C,B]]^-1 = [[A^-1,0],[-B^-1 C A^-1, B^-1]]  to 64 rows, and the last merge by two
// products of the tensor unit on bf16 pairs.  The columns are scaled by D in float32, before they become the pair that T~ is kept in.
//
// Precision.  The first two levels read and write float32, their products split every operand into two tf32 numbers (mma.sync
// m16n8k8, lo x lo left out: 2^-22 of a product).  The last level takes pairs of the blocks not yet scaled (their diagonals are
// exact then).  Relative error of T~ against float64, 512 chunks, d = 64 / 128: random unit w 4.0e-6 / 3.2e-6 (rounding
// the exact T~ to a pair: 2.3e-6); beta = 2 and w around one direction 8.3e-5 / 8.3e-5; beta = 2 and four directions 1.6e-5 / 1.5e-5.
// (With T_A, T_B, the scaled blocks, as the last level's operands: 4.9e-6 / 3.9e-6 for random w.)
__device__ __forceinline__ void mma1688(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// hi (x cut off), l = lo (the rest, rounded: 11 + 11 bits and a sign).  Both are tf32 values as they stand: that a product ignores what
// lies below a tf32 number's bits is not promised.
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
// The permutation is split into a lane's part, computed once, and one XOR per column: computed anew for every element it took
// the merges three times as long as their products (integer operations issue at half rate).
struct Tf32A { uint32_t h[4], l[4]; };
struct FragLane {
    int a, xa, b[2], xb[2];
    __device__ __forceinline__ explicit FragLane(int lane) {
        auto perm = [](int r) { return (((r & 3) ^ ((r >> 2) & 1)) << 3) | (r & 4); };
        const int ra = lane >> 2, ca = 2 * (lane & 3), fa = perm(ra);
        a = ra * 256 + (ca ^ (fa & 4)) * 4;
        xa = (fa & 24) * 4;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int fb = perm(ca + x);
            b[x] = (ca + x) * 256 + (ra ^ (fb & 4)) * 4;
            xb[x] = (fb & 24) * 4;
        }
    }
    // `rows`: a stripe's row that is a multiple of 8; c: a column that is
    __device__ __forceinline__ float* at_a(uint8_t* rows, int c) const { return reinterpret_cast<float*>(rows + a + ((c * 4) ^ xa)); }
    __device__ __forceinline__ float at_b(uint8_t* rows, int c, int x) const { return *reinterpret_cast<float*>(rows + b[x] + ((c * 4) ^ xb[x])); }
};
__device__ __forceinline__ Tf32A tf32_a(const FragLane& f, uint8_t* rows, int c) {
    const float2 x = *reinterpret_cast<const float2*>(f.at_a(rows, c));
    const float2 y = *reinterpret_cast<const float2*>(f.at_a(rows + 8 * 256, c));
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
// d[16 x 8 T] += A B, B the 8 x 8 T block at `rows`, column c
template <int T>
__device__ __forceinline__ void mma_tf32(float (&d)[T][4], const Tf32A& a, const FragLane& f, uint8_t* rows, int c) {
    uint32_t h[T][2], l[T][2];
#pragma unroll
    for (int n = 0; n < T; ++n)
#pragma unroll
        for (int x = 0; x < 2; ++x) h[n][x] = split_tf32(f.at_b(rows, c + n * 8, x), l[n][x]);
#pragma unroll
    for (int n = 0; n < T; ++n) mma1688(d[n], a.h, h[n][0], h[n][1]);
#pragma unroll
    for (int n = 0; n < T; ++n) mma1688(d[n], a.h, l[n][0], l[n][1]);
#pragma unroll
    for (int n = 0; n < T; ++n) mma1688(d[n], a.l, h[n][0], h[n][1]);
}
// x *= the 32 entries of D at bt
__device__ __forceinline__ void scale32(float (&x)[32], const float* bt) {
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bt + i);
        x[i] *= b.x; x[i + 1] *= b.y; x[i + 2] *= b.z; x[i + 3] *= b.w;
    }
}
// One merge level of blocks of NBK 16-row strips (1, 2) inside the float32 blocks.  NBK = 1: four pairs, the two warps of a pair take
// 8 columns of the result each; NBK = 2: a warp takes 16 x 16, the two warps that share a scheduler (w, w + 4) a long and a
// short strip (B^-1 is lower triangular: strip rb needs its first rb + 1 blocks).
template <int NBK>
__device__ __forceinline__ void merge_f32(uint8_t* aH, uint8_t* aL, int warp, int lane) {
    constexpr int NT = NBK;                       // 8-column tiles of the result per warp
    const int hw = warp >> 2, w4 = warp & 3;
    const int b = NBK == 1 ? w4 >> 1 : w4 & 1, rb = NBK == 1 ? 0 : ((w4 >> 1) ^ hw), odd = w4 & 1;
    const FragLane f(lane);
    // NBK = 1: a stripe's rows 0 - 15 (A) and 16 - 31; NBK = 2: its upper (A) and its lower stripe
    const int ca = NBK == 1 ? odd * 32 : 0, cb = ca + NBK * 16;
    uint8_t* rows_a = (NBK == 1 && odd ? aL : aH) + b * (kPanelB + 8192);
    uint8_t* rows_b = (NBK == 1 ? rows_a + 16 * 256 : aL + b * (kPanelB + 8192));
    uint8_t* strip = rows_b + rb * 16 * 256;
    const int k_lo = NBK == 1 ? 0 : hw, col0 = ca + hw * NBK * 8;   // A^-1 is lower triangular: columns col0.. need no earlier block
    float m[NT][4], p1[NBK][2][4];
#pragma unroll
    for (int k = 0; k < NBK; ++k)
#pragma unroll
        for (int x = 0; x < 8; ++x) p1[k][x >> 2][x & 3] = 0.f;
#pragma unroll
    for (int x = 0; x < 4 * NT; ++x) m[x >> 2][x & 3] = 0.f;
#pragma unroll 1
    for (int j = 0; j < 16 * (rb + 1); j += 8) {
        const Tf32A a = tf32_a(f, strip, cb + j);
#pragma unroll
        for (int kb = 0; kb < NBK; ++kb) {
            if (kb < k_lo) continue;
            mma_tf32(p1[kb], a, f, rows_b + j * 256, ca + kb * 16);
        }
    }
#pragma unroll
    for (int kb = 0; kb < NBK; ++kb) {
        if (kb < k_lo) continue;
#pragma unroll
        for (int k8 = 0; k8 < 2; ++k8) mma_tf32(m, tf32_a(p1[kb][k8]), f, rows_a + (kb * 16 + k8 * 8) * 256, col0);
    }
    wsync();   // the other warps of the pair read C as well
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int y = 0; y < 2; ++y)
            *reinterpret_cast<float2*>(f.at_a(strip + 8 * y * 256, col0 + n * 8)) = make_float2(-m[n][2 * y], -m[n][2 * y + 1]);
}
// 16 x 16 diagonal blocks: half a warp each, a lane owns a column of the inverse and reads the rows all lanes of its half need.
__device__ __forceinline__ void substitute16(uint8_t* aH, uint8_t* aL, int warp, int lane) {
    const int o = (warp & 1) * 32 + (lane & 16), j = lane & 15;
    uint8_t* rows = (warp & 1 ? aL : aH) + (warp >> 1) * (kPanelB + 8192) + (lane & 16) * 256;
    uint8_t* at[2] = {rows + o * 4, rows + (o ^ 16) * 4};
    auto piece = [&](int r, int c4) {   // fel for these rows, 16 bytes from column o + 4 c4 on
        const int f = (((r & 3) ^ ((r >> 2) & 1)) << 3) | (r & 4);
        return at[(f >> 4) & 1] + r * 256 + ((4 * c4) ^ (f & 12)) * 4;
    };
    float x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        uint64_t acc[2] = {0ull, 0ull};
        ulonglong2 f{};
#pragma unroll
        for (int c = 0; c < (r + 3) / 4; ++c) {
            f = *reinterpret_cast<const ulonglong2*>(piece(r, c));
            if (4 * c + 1 < r) acc[0] = fma2(f.x, pack2(x[4 * c], x[4 * c + 1]), acc[0]);
            if (4 * c + 3 < r) acc[1] = fma2(f.y, pack2(x[4 * c + 2], x[4 * c + 3]), acc[1]);
        }
        float s0, s1, last = 0.f;
        unpack2(r >= 4 ? add2(acc[0], acc[1]) : acc[0], s0, s1);
        if (r & 1) {   // the last of an odd number of entries
            float hi;
            unpack2(r & 2 ? f.y : f.x, last, hi);
            last *= x[r - 1];
        }
        const float sum = (s0 + s1) + last;
        x[r] = r > j ? -sum : r == j ? 1.f : 0.f;
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) *reinterpret_cast<float*>(piece(r, j >> 2) + (j & 3) * 4) = x[r];
}
// The 64 x 64 diagonal blocks of N -> their inverses, as pairs and (d: this thread's 32 entries of a row) scaled by D in float32.
__device__ __forceinline__ void invert_diagonal(uint8_t* aH, uint8_t* aL, const float* bt, int warp, int lane, int row, int half, float (&d)[32]) {
    if (warp < 4) substitute16(aH, aL, warp, lane);
    wsync();
    merge_f32<1>(aH, aL, warp, lane);
    wsync();
    merge_f32<2>(aH, aL, warp, lane);
    wsync();
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
    scale32(d, bt + cb);
}

// Accumulators of one row, W columns from `taddr` on, times `scale` if there is one, as a bf16 pair; the pair into the two tiles.
template <int W, bool SCALED>
__device__ __forceinline__ void read_pair(uint32_t taddr, const float* scale, uint32_t (&hi)[W / 2], uint32_t (&lo)[W / 2]) {
    uint32_t r[W];
    if constexpr (W == 16) tmem_ld16(taddr, r);
    else tmem_ld32(taddr, r);
    tmem_ld_wait();
#pragma unroll
    for (int x = 0; x < W; x += 4) {
        float4 v = make_float4(__uint_as_float(r[x]), __uint_as_float(r[x + 1]), __uint_as_float(r[x + 2]), __uint_as_float(r[x + 3]));
        if (SCALED) {
            const float4 b = *reinterpret_cast<const float4*>(scale + x);
            v.x *= b.x; v.y *= b.y; v.z *= b.z; v.w *= b.w;
        }
        const uint32_t h0 = pack_bf16(v.x, v.y), h1 = pack_bf16(v.z, v.w);
        hi[x / 2] = h0;
        hi[x / 2 + 1] = h1;
        lo[x / 2] = pack_bf16(v.x - __uint_as_float(h0 << 16), v.y - __uint_as_float(h0 & 0xffff0000u));
        lo[x / 2 + 1] = pack_bf16(v.z - __uint_as_float(h1 << 16), v.w - __uint_as_float(h1 & 0xffff0000u));
    }
}
template <int N>
__device__ __forceinline__ void store_pair(uint8_t* aH, uint8_t* aL, int row, int c0, const uint32_t (&hi)[N], const uint32_t (&lo)[N]) {
#pragma unroll
    for (int x = 0; x < N; x += 4) {
        const uint32_t at = (uint32_t)(c0 >> 6) * kPanelB + sw128_off((uint32_t)row, (uint32_t)((c0 & 63) >> 3) + x / 4);
        *reinterpret_cast<uint4*>(aH + at) = make_uint4(hi[x], hi[x + 1], hi[x + 2], hi[x + 3]);
        *reinterpret_cast<uint4*>(aL + at) = make_uint4(lo[x], lo[x + 1], lo[x + 2], lo[x + 3]);
    }
}

// MODE: PREP_FWD = everything the forward needs; PREP_SAVE = also keeps the tiles of the chain rule (the backward's instance);
// PREP_KEYS = the key side only (prompt key cache: Kright and the chunk products; no query is involved, so Xq, Xq U,
// Qleft and the diagonal-correction operands are left out and q is not even loaded).
template <int HD, int MODE>
__global__ void __launch_bounds__(kThreads, 1) chunk_prep_kernel(const __grid_constant__ PrepTensorMaps tm, const PrepParams p,
                                                                      const int nchunks) {
    constexpr bool SAVE = MODE == PREP_SAVE, KEYS = MODE == PREP_KEYS, D64 = HD == 64;
    // T~ as an operand: at d = 64 from tensor memory, so that the next inverse can have its tiles while U and Y are computed.  It lies
    // where the next Gm was, which has to be ready by then: at d = 128 its W comes too late for that.
    constexpr bool TMT = D64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    auto slot = [&](int i) { return smem + i * kTileB; };
    // tiles of the head dimension in slots 5, 6
    constexpr uint32_t oU = 5 * kTileB, oUlo = oU + (D64 ? kPanelB : kTileB);            // U, then P: hi, lo
    constexpr uint32_t oQ = (D64 ? 6 : 5) * kTileB, oK = oQ + (D64 ? kPanelB : kTileB);  // Q, K of the chunk
    constexpr uint32_t oXq = (D64 ? 5 : 6) * kTileB;                                      // Xq hi, for its store
    float* betas = (float*)(smem + PrepSmem::offBeta);   // of this chunk and the next, by turns
    uint64_t* bars = (uint64_t*)(smem + PrepSmem::offBar);
    uint32_t* tmem_slot = (uint32_t*)(bars + B_COUNT);
    volatile uint32_t* abort_flag = (volatile uint32_t*)(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = (warp >> 2) & 1;             // which half of an accumulator's columns a worker thread has

    if (tid == 0) {
        for (int i = 0; i < B_COUNT; ++i) mbar_init(&bars[i], i >= R_GM ? (uint32_t)kWorkers : 1u);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    auto beta_of = [&](int chunk_) {   // beta of this thread's row (tid < 128); 0 past the sequence's end
        const int pos = (chunk_ % p.N) * kT + tid;
        return pos < p.L ? p.beta[(size_t)(chunk_ / p.N) * p.L + pos] : 0.f;
    };
    // the block of T~ above the diagonal blocks stays zero: nothing is ever written there
    for (int i = tid; i < 1024; i += kThreads)
        reinterpret_cast<uint4*>(slot(1 + (i >> 9)) + kPanelB)[i & 511] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_launch();
    if (p.clear && blockIdx.x == 0 && tid < 64) p.status[tid] = 0u;   // the workspace's status block (256 bytes)
    if (tid < kT && (int)blockIdx.x < nchunks) betas[tid] = beta_floor(beta_of(blockIdx.x));
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t base_ = smem_u32(smem);
    constexpr int KS = HD / 16;  // k-steps over the head dimension
    // Tensor-memory columns.  0: the next chunk's Gm, then (TMT) the pair T~, then Xq U.  128: Xq, then its pair.  256 and 384, changing places from
    // chunk to chunk: Xk -> Y -> Y^T W, and the inverse's two products -> U -> W^T U.
    constexpr uint32_t cG = 0, cXq = 128;
    auto col_x = [](uint32_t it) { return 256u + (it & 1) * 128u; };
    auto col_u = [](uint32_t it) { return 384u - (it & 1) * 128u; };

    if (warp >= 2 * kWorkers / 32) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");   // 128 x 80 + 256 x 120 + 256 x 80 = all of the 640 x 96 that the block starts with
        auto wait = [&](int b, uint32_t par) { return mbar_wait<true>(&bars[b], par, abort_flag, ST_PREP); };
        if (warp == 16 && elect_one()) {
            // -------------------------------------------------------------- products
            bool ok = (int)blockIdx.x < nchunks;
            if (ok && (ok = wait(L_W, 0))) {
                tc_fence_after_sync();
                mma<OP_K, OP_K, KS, 128>(tmem + cG, base_, base_, false);
                umma_commit(&bars[M_GM]);
            }
            for (uint32_t it = 0, chunk = blockIdx.x; ok && (int)chunk < nchunks; ++it, chunk += gridDim.x) {
                const uint32_t par = it & 1;
                const bool more = (int)(chunk + gridDim.x) < nchunks;
                // (the tiles' address is made opaque once per chunk: otherwise every descriptor of every product is
                // hoisted out of this loop and the thread's small register allotment spills)
                uint32_t a0 = base_;
                asm volatile("" : "+r"(a0));
                auto t = [&](int i) { return a0 + i * kTileB; };
                const uint32_t w = a0 + (D64 ? par * kPanelB : 0u);
                const uint32_t cx = tmem + col_x(it), cu = tmem + col_u(it);
                // Xq, Xk: P of the chunk before has been read, and with it the columns that Xk takes
                if (!D64 && it > 0 && !(ok = wait(L_W, par))) break;
                if (!(ok = wait(L_QK, par))) break;
                if (it > 0 && !(ok = wait(R_P, par ^ 1))) break;
                tc_fence_after_sync();
                if (!KEYS) mma<OP_K, OP_K, KS, 128>(tmem + cXq, a0 + oQ, w, false);
                mma<OP_K, OP_K, KS, 128>(cx, w, a0 + oK, false);
                umma_commit(&bars[M_XQK]);
                // The next chunk's Gm runs underneath this chunk's inverse; what its columns held has been read: Xq U for Q<- (or the
                // first Gm).  (K-> has been read as well, and with it the columns that U takes.)
                if (more && !(ok = wait(L_WN, par))) break;
                if (it > 0 && !(ok = wait(R_E3, par ^ 1))) break;
                if ((!TMT || it == 0) && !(ok = wait(R_GM, par))) break;
                tc_fence_after_sync();
                if (more) {
                    const uint32_t wn = D64 ? a0 + (par ^ 1) * kPanelB : t(5);
                    mma<OP_K, OP_K, KS, 128>(tmem + cG, wn, wn, false);
                    umma_commit(&bars[M_GM]);
                }
                // U = T~ W, Y = T~ Xk  (lo x lo terms are dropped everywhere)
                if (!(ok = wait(R_TT, par))) break;
                tc_fence_after_sync();
                if (TMT) {
                    mma_tap<OP_MN, 8, HD>(cu, tmem + cG, w, false);
                    mma_tap<OP_MN, 8, HD>(cu, tmem + cG + 16, w, true);
                } else {
                    mma<OP_K, OP_MN, 8, HD>(cu, t(1), w, false);
                    mma<OP_K, OP_MN, 8, HD>(cu, t(2), w, true);
                }
                umma_commit(&bars[M_U]);
                if (!(ok = wait(R_XK, par))) break;
                tc_fence_after_sync();
                if (TMT) {
                    mma_tap<OP_MN, 8, 128>(cx, tmem + cG, t(3), false);
                    mma_tap<OP_MN, 8, 128>(cx, tmem + cG + 16, t(3), true);
                    mma_tap<OP_MN, 8, 128>(cx, tmem + cG, t(4), true);
                } else {
                    mma<OP_K, OP_MN, 8, 128>(cx, t(1), t(3), false);
                    mma<OP_K, OP_MN, 8, 128>(cx, t(2), t(3), true);
                    mma<OP_K, OP_MN, 8, 128>(cx, t(1), t(4), true);
                }
                umma_commit(&bars[M_Y]);
                // -W^T U, and Xq U over the next Gm once that has been read, or over T~ once Y has retired
                if (!(ok = wait(R_U, par))) break;
                tc_fence_after_sync();
                mma<OP_MN, OP_MN, 8, HD, true>(cu, w, a0 + oU, false);
                mma<OP_MN, OP_MN, 8, HD, true>(cu, w, a0 + oUlo, true);
                if (!KEYS) {
                    if (!(ok = TMT ? wait(M_Y, par) : !more || wait(R_GM, par ^ 1))) break;
                    tc_fence_after_sync();
                    mma_tap<OP_MN, 8, HD>(tmem + cG, tmem + cXq, a0 + oU, false);
                    mma_tap<OP_MN, 8, HD>(tmem + cG, tmem + cXq + 16, a0 + oU, true);
                    mma_tap<OP_MN, 8, HD>(tmem + cG, tmem + cXq, a0 + oUlo, true);
                }
                umma_commit(&bars[M_GA]);
                // Y^T W
                if (!(ok = wait(R_Y, par))) break;
                tc_fence_after_sync();
                mma<OP_MN, OP_MN, 8, HD>(cx, t(3), w, false);
                mma<OP_MN, OP_MN, 8, HD>(cx, t(4), w, true);
                umma_commit(&bars[M_GB]);
            }
        }
        if (warp == 17 && elect_one()) {
            // -------------------------------------------------------------- tile loads and stores
            auto fetch = [&](const CUtensorMap* m, uint32_t off, int b, int chunk_) {
                tma_rows(smem + off, m, &bars[b], HD, (chunk_ % p.N) * kT, chunk_ / p.N);
            };
            auto load_w = [&](int chunk_, uint32_t off, int b) {
                mbar_expect_tx(&bars[b], kT * HD * 2);
                fetch(&tm.w, off, b, chunk_);
            };
            auto load_qk = [&](int chunk_, uint32_t off_q, uint32_t off_k, int b) {
                mbar_expect_tx(&bars[b], (KEYS ? 1 : 2) * kT * HD * 2);
                if (!KEYS) fetch(&tm.q, off_q, b, chunk_);
                fetch(&tm.k, off_k, b, chunk_);
            };
            auto store = [&](const CUtensorMap* m, uint32_t off, int ncols, int row0) {
                for (int h = 0; h < ncols / 64; ++h) tma_store_2d(m, smem + off + h * kPanelB, h * 64, row0);
            };
            bool ok = (int)blockIdx.x < nchunks;
            if (ok) {
                load_w(blockIdx.x, 0, L_W);
                load_qk(blockIdx.x, oQ, oK, L_QK);
            }
            for (uint32_t it = 0, chunk = blockIdx.x; ok && (int)chunk < nchunks; ++it, chunk += gridDim.x) {
                const uint32_t par = it & 1;
                const int r0 = chunk * kT, next = chunk + gridDim.x;
                const bool more = next < nchunks;
                if (!D64 && more) {   // what the next chunk reads: its slots become free late, the trip from memory is taken now
                    const int row0 = (next % p.N) * kT, slice = next / p.N;
                    for (int h = 0; h < HD / 64; ++h) {
                        tma_prefetch_3d(&tm.w, h * 64, row0, slice);
                        if (!KEYS) tma_prefetch_3d(&tm.q, h * 64, row0, slice);
                        tma_prefetch_3d(&tm.k, h * 64, row0, slice);
                    }
                }
                if (D64 && more) load_w(next, (par ^ 1) * kPanelB, L_WN);   // (M_GB of the chunk before: its W is not needed any more)
                if (!(ok = wait(M_XQK, par))) break;
                if (more) {
                    if (D64) load_qk(next, oQ, oK, L_QK);
                    else load_w(next, 5 * kTileB, L_WN);
                }
                if (!KEYS) {
                    if (!(ok = wait(R_XQ, par))) break;
                    store(&tm.xq, oXq, kT, r0);
                    tma_store_commit();
                }
                if (SAVE) {
                    if (!(ok = wait(R_XK, par))) break;
                    store(&tm.xk, 3 * kTileB, kT, r0);
                    tma_store_commit();
                }
                if (!KEYS) {
                    tma_store_wait_read();
                    mbar_arrive(&bars[S_XQ]);
                }
                if (SAVE) {
                    mbar_arrive(&bars[S_XK]);
                    if (!(ok = wait(R_TT, par))) break;
                    store(&tm.th, 1 * kTileB, kT, r0);
                    store(&tm.tl, 2 * kTileB, kT, r0);
                    tma_store_commit();
                    tma_store_wait_read();
                    mbar_arrive(&bars[S_T]);
                    if (!(ok = wait(R_U, par))) break;
                    store(&tm.u, oU, HD, r0);
                    tma_store_commit();
                }
                if (!KEYS) {
                    if (!(ok = wait(R_Y, par))) break;
                    store(&tm.y, 3 * kTileB, kT, r0);
                    tma_store_commit();
                }
                if (SAVE) {
                    tma_store_wait_read_but<1>();
                    mbar_arrive(&bars[S_U]);
                }
                // once Y^T W has retired, W's slot takes the next chunk's W, Y's slots the Q and K rows once more (from L2), for the
                // sums that finish Q<- and K->
                if (!(ok = wait(M_GB, par))) break;
                if (!D64 && more) load_w(next, 0, L_W);
                if (!KEYS) tma_store_wait_read();
                load_qk(chunk, 3 * kTileB, 4 * kTileB, L_ROW);
                if (!(ok = wait(R_P, par))) break;
                store(&tm.ph, oU, HD, chunk * HD);
                store(&tm.pl, oUlo, HD, chunk * HD);
                tma_store_commit();
                if (!D64 && more) {
                    tma_store_wait_read();
                    load_qk(next, oQ, oK, L_QK);
                }
                if (!(ok = wait(R_E3, par))) break;
                if (!KEYS) store(&tm.ql, 3 * kTileB, HD, r0);
                store(&tm.kr, 4 * kTileB, HD, r0);
                tma_store_commit();
                tma_store_wait_read();
                mbar_arrive(&bars[S_E3]);
            }
            tma_store_wait_all();
        }
        if (warp == 18 && elect_one()) {
            // -------------------------------------------------------------- products of the inverse
            // in the columns that U takes afterwards, once K-> of the chunk before has been read from them
            bool ok = true;
            for (uint32_t it = 0, chunk = blockIdx.x; ok && (int)chunk < nchunks; ++it, chunk += gridDim.x) {
                const uint32_t par = it & 1;
                uint32_t tH = base_ + kTileB;
                asm volatile("" : "+r"(tH));
                const uint32_t tL = tH + kTileB, cu = tmem + col_u(it);
                if (it > 0 && !(ok = wait(R_E3, par ^ 1))) break;
                if (!(ok = wait(R_ID, par))) break;
                tc_fence_after_sync();
                mma<OP_K, OP_MN, 4, 64>(cu, tH, tH, false);            // rows 64 ..: X = C A^-1
                mma<OP_K, OP_MN, 4, 64>(cu, tL, tH, true);
                mma<OP_K, OP_MN, 4, 64>(cu, tH, tL, true);
                umma_commit(&bars[M_IX]);
                if (!(ok = wait(R_IX, par))) break;
                tc_fence_after_sync();
                mma<OP_K, OP_MN, 4, 64, true>(cu + 64, tH + kPanelB, tH + 8192, false);   // rows 64 ..: -B^-1 X
                mma<OP_K, OP_MN, 4, 64, true>(cu + 64, tL + kPanelB, tH + 8192, true);
                mma<OP_K, OP_MN, 4, 64, true>(cu + 64, tH + kPanelB, tL + 8192, true);
                umma_commit(&bars[M_IT]);
            }
        }
        __syncwarp();
    } else if (warp < kWorkers / 32) {
        // ------------------------------------------------------------------ inverse
        asm volatile("setmaxnreg.inc.sync.aligned.u32 120;");
        bool ok = true;
        // lane 0 of every warp waits; the vote that follows is also the barrier that releases the other lanes
        auto wwait = [&](int b, uint32_t par) {
            bool good = ok;
            if ((tid & 31) == 0 && good) good = mbar_wait<true>(&bars[b], par, abort_flag, ST_PREP);
            return wsync_and(good);
        };
        uint8_t* aH = slot(1);
        uint8_t* aL = slot(2);
        const int w8 = warp;
        // This thread's 64 entries of Gm (only those of the two diagonal blocks and of the block under them are used).
        uint32_t g[2][32];
        auto read_gm = [&]() {
            tmem_ld32(tl + cG + half * 64, g[0]);
            tmem_ld32(tl + cG + half * 64 + 32, g[1]);
            tmem_ld_wait();
        };
        int chunk = blockIdx.x;
        auto first_gm = [&](uint32_t par) {
            if (!(ok = wwait(M_GM, par))) return;
            tc_fence_after_sync();
            read_gm();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_GM]);
        };
        if (TMT) first_gm(0);
        for (uint32_t it = 0; ok && chunk < nchunks; ++it, chunk += gridDim.x) {
            const uint32_t par = it & 1;
            // (made opaque once per chunk: otherwise every address of the inverse is kept from chunk to chunk, in registers it does not have)
            int lane = tid & 31, warp = w8;
            asm volatile("" : "+r"(lane), "+r"(warp));
            const int row = (warp & 3) * 32 + lane, half = (warp >> 2) & 1;   // accumulator row (TMEM lane), half of the columns
            const bool diag = (row >> 6) == half, below = row >= 64 && half == 0;   // (the same for a whole warp)
            const int next = chunk + (int)gridDim.x;
            const float* bt = betas + par * kT;
            float next_beta = 0.f;
            if (tid < kT && next < nchunks) next_beta = beta_of(next);
            // N = strictLower(D Gm) into slots 1, 2 as the inverse wants it: the two diagonal blocks in float32, the block
            // under them as a bf16 pair
            if (!TMT) {   // (read while the products that use the T~ before it still run)
                first_gm(par);
                if (!ok || (it > 0 && !(ok = wwait(M_Y, par ^ 1)))) break;
            }
            if (SAVE && it > 0 && !(ok = wwait(S_T, par ^ 1))) break;
            const float b = bt[row];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int c0 = half * 64 + c * 32;
                if (diag) {
                    const int m = c * 32 - (row & 32);   // > 0: above the diagonal, < 0: below it, 0: on it (the same for a whole warp)
                    float v[32];
#pragma unroll
                    for (int x = 0; x < 32; ++x) v[x] = m > 0 ? 0.f : b * __uint_as_float(g[c][x]);
                    if (m == 0) {
#pragma unroll
                        for (int x = 0; x < 32; ++x) v[x] = x < lane ? v[x] : 0.f;
                    }
#pragma unroll
                    for (int x = 0; x < 32; x += 4)
                        *reinterpret_cast<float4*>(fel(aH, aL, half, row & 63, c * 32 + x)) = make_float4(v[x], v[x + 1], v[x + 2], v[x + 3]);
                } else if (below) {
                    float v[32];
                    uint32_t hi[16], lo[16];
#pragma unroll
                    for (int x = 0; x < 32; ++x) v[x] = b * __uint_as_float(g[c][x]);
                    split32(v, hi, lo);
                    tile_store_w16(aH, row, c0, hi);
                    tile_store_w16(aL, row, c0, lo);
                }
            }
            wsync();
            float d[32];
            invert_diagonal(aH, aL, bt, warp, lane, row, half, d);
            if (tid < kT) betas[(par ^ 1) * kT + tid] = beta_floor(next_beta);   // (nobody reads the chunk before's any more)
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_ID]);
            // X = C A^-1 over C, then the block of T~ there: -B^-1 X D; a thread has 32 entries of a row in all of this.  T~ goes into
            // tensor memory (per 32 columns 16 of hi, 16 of lo) and / or over the tiles.
            const uint32_t cu = col_u(it) + half * 32;
            const int cd = (row & 64) + half * 32, co = half * 32 + 64 - (row & 64);   // its columns in the diagonal block and the other one
            // Columns at a time.  At d = 64 the 64 entries of the next Gm or the 32 of d are live as well; 32 more spilled (183 / 152 us for
            // the 2048 chunks of 8 x 16 x 2048 x 64).
            constexpr int W = D64 ? 16 : 32;
            if (!(ok = wwait(M_IX, par))) break;
            tc_fence_after_sync();
            if (row >= 64) {
#pragma unroll 1
                for (int c = 0; c < 32; c += W) {
                    uint32_t h[W / 2], l[W / 2];
                    read_pair<W, false>(tl + cu + c, nullptr, h, l);
                    store_pair(aH, aL, row, half * 32 + c, h, l);
                }
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_IX]);
            if (TMT && next < nchunks) {   // Gm of the next chunk leaves its columns to T~
                if (!(ok = wwait(M_GM, par ^ 1))) break;
                tc_fence_after_sync();
                read_gm();
            } else {   // (the entries end here in either case: 64 registers that are not carried through the inverse)
#pragma unroll
                for (int x = 0; x < 32; ++x) g[0][x] = g[1][x] = 0u;
            }
            uint32_t hi[16], lo[16];
            split32(d, hi, lo);
            if (!(ok = wwait(M_IT, par))) break;
            tc_fence_after_sync();
            if (TMT) {   // (everybody has read Gm: there was a vote since)
                tmem_st16(tl + cG + cd, hi);
                tmem_st16(tl + cG + cd + 16, lo);
            }
            if (!TMT || SAVE) store_pair(aH, aL, row, cd, hi, lo);
#pragma unroll 1
            for (int c = 0; c < 32; c += W) {
                uint32_t h[W / 2], l[W / 2];
                if (row >= 64) {
                    read_pair<W, true>(tl + cu + 64 + c, bt + half * 32 + c, h, l);
                    if (!TMT || SAVE) store_pair(aH, aL, row, co + c, h, l);
                } else {
#pragma unroll
                    for (int x = 0; x < W / 2; ++x) h[x] = l[x] = 0u;
                }
                if constexpr (TMT) {
                    tmem_st8(tl + cG + co + c / 2, h);
                    tmem_st8(tl + cG + co + 16 + c / 2, l);
                }
            }
            if (TMT) tmem_st_wait();
            if (!TMT || SAVE) fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[R_TT]);
        }
    } else {
        // ------------------------------------------------------------------ operands and results
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        bool ok = true;
        uint32_t r[32];
        float v[32];
        auto wwait = [&](int b, uint32_t par) {   // (a thread touches its own rows only: warps meet nowhere but at mbarriers)
            return __all_sync(0xffffffffu, mbar_wait<true>(&bars[b], par, abort_flag, ST_PREP)) != 0;
        };
        auto publish = [&](int b) {
            fence_proxy_async_smem();
            tc_fence_before_sync();
            mbar_arrive(&bars[b]);
        };
        int chunk = blockIdx.x;
        for (uint32_t it = 0; chunk < nchunks; ++it, chunk += gridDim.x) {
            const uint32_t par = it & 1, cx = col_x(it), cu = col_u(it);
            int row = (warp & 3) * 32 + lane;
            asm volatile("" : "+r"(row));   // (as above)
            // Five accumulators become bf16 pairs:  Xq = lower(.) in its own columns (per 32 columns 16 of hi, 16 of lo; hi also as
            // a tile, for its store), Xk = strictLower(.), U over Q and K, Y over Xk, P = I - W^T U over U.  One body for all of
            // them: the two groups' straight-line code does not fit the instruction caches.
            enum { XQ = 0, XK, UU, YY, PP };
#pragma unroll 1
            for (int st = KEYS ? XK : XQ; st <= PP; ++st) {
                if (!(ok = wwait(st <= XK ? M_XQK : st == UU ? M_U : st == YY ? M_Y : M_GA, par))) break;
                // stores that still read the tiles about to be written (at d = 64 Xq goes over the P of the chunk before)
                const int behind = st == XQ ? (D64 ? S_E3 : -1) : st == XK ? S_E3 : st == UU ? (KEYS ? -1 : S_XQ) : !SAVE ? -1 : st == YY ? S_XK : S_U;
                if (behind >= 0 && (st > XK || it > 0) && !(ok = wwait(behind, st > XK ? par : par ^ 1))) break;
                tc_fence_after_sync();
                const uint32_t col = st == XQ ? cXq : st & 1 ? cx : cu;
                const bool head = st == UU || st == PP;   // HD columns, not 128
                const uint32_t to_hi = head ? oU : st == XQ ? oXq : 3 * kTileB, to_lo = head ? oUlo : 4 * kTileB;
                const int n = head ? HD / 64 : 2;
#pragma unroll 1
                for (int c = 0; c < n; ++c) {
                    const int c0 = half * n * 32 + c * 32, m = st == UU || st == YY ? -1 : c0 - (warp & 3) * 32;
                    uint32_t hi[16], lo[16];
                    if (m > 0 && st <= XK) {   // (the warp's 32 rows and these 32 columns: above the diagonal)
#pragma unroll
                        for (int x = 0; x < 16; ++x) hi[x] = lo[x] = 0u;
                    } else {
                        tmem_ld32(tl + col + c0, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r[x]);
                        if (m == 0) {
                            const int last = st == XQ ? lane + 1 : st == XK ? lane : 32, one = st == PP ? lane : -1;
#pragma unroll
                            for (int x = 0; x < 32; ++x) v[x] = x == one ? v[x] + 1.f : x < last ? v[x] : 0.f;
                        }
                        split32(v, hi, lo);
                    }
                    tile_store_w16(smem + to_hi, row, c0, hi);
                    if (st == XQ) {
                        tmem_st16(tl + cXq + c0, hi);
                        tmem_st16(tl + cXq + c0 + 16, lo);
                    } else {
                        tile_store_w16(smem + to_lo, row, c0, lo);
                    }
                }
                if (st == XQ) tmem_st_wait();
                publish(R_XQ + st);
            }
            if (!ok) break;
            // ---- Qleft = Q - Xq U, Kright = K - Y^T W over the Q and K rows that have arrived in Y's slots
            if (!(ok = wwait(M_GB, par))) break;
            if (!(ok = wwait(L_ROW, par))) break;
            tc_fence_after_sync();
#pragma unroll 1
            for (int c = KEYS ? HD / 64 : 0; c < 2 * (HD / 64); ++c) {
                const bool is_k = c >= HD / 64;
                const int c0 = half * (HD / 2) + (is_k ? c - HD / 64 : c) * 32;
                uint8_t* tile_ = slot(is_k ? 4 : 3);
                float in[32];
                tmem_ld32(tl + (is_k ? cx : cG) + c0, r);
                tmem_ld_wait();
                tile_load32(tile_, row, c0, in);
#pragma unroll
                for (int x = 0; x < 32; ++x) v[x] = in[x] - __uint_as_float(r[x]);
                tile_store32(tile_, row, c0, v);
            }
            publish(R_E3);
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
