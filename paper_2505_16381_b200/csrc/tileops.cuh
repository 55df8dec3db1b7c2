// Building blocks of the per-chunk kernels: every matrix of the chunk-level algebra is a 128-row
// bf16 tile in shared memory (row-major, 64-column panels, 128-byte swizzle), every product a tcgen05 MMA into
// tensor memory issued by one thread, every result read back one row per thread (with 256 worker threads two share a row, each
// taking half of the columns; with the 512 of the chain rule four).
#pragma once
#include "common.cuh"
#include "tc5.cuh"

namespace path {
namespace tile {
using namespace tc5;

constexpr int kT = 128;
constexpr uint32_t kTileB = 32768, kPanelB = 16384;

// K view: contraction over the tile's columns.  MN view: contraction over the tile's rows.
enum { OP_K = 0, OP_MN = 1 };

// beta as the per-chunk kernels use it: kept away from zero, so that the chain rule can divide by it (T~ = Ainv D is kept, and
// Ainv is T~ with its columns divided by beta).  2^-80 of a unit transition is far below every rounding.
__device__ __forceinline__ float beta_floor(float b) { return fabsf(b) < 0x1p-80f ? copysignf(0x1p-80f, b) : b; }

// D[128 x N] (+)= (+-) op(A) op(B), KSTEPS steps of 16 along the contraction.  One thread issues all of them (elect_one), so
// the instructions between two tcgen05.mma count: everything but the tiles' addresses is a compile-time constant, the loop is
// unrolled, and only the low word of a descriptor changes from step to step (the start address; the strides and the swizzle
// mode sit in the high word).  Against a rolled loop in a function of its own, behind `lane == 0`: the chain rule took 302
// instead of 342 us at B=4, H=16, L=4096, d=128 and 246 instead of 306 us at B=8, H=16, L=2048, d=64.
template <int AOP, int BOP, int KSTEPS, int N, bool NEG = false>
__device__ __forceinline__ void mma(uint32_t d_tmem, uint32_t a_tile, uint32_t b_tile, bool acc) {
    constexpr uint32_t idesc = umma_idesc(128, N, AOP, BOP) | (NEG ? (1u << 13) : 0u);
    const uint32_t a_lo = umma_desc_lo(a_tile, AOP == OP_K ? 16u : kPanelB);
    const uint32_t b_lo = umma_desc_lo(b_tile, BOP == OP_K ? 16u : kPanelB);
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) {
        // K view: 32 bytes per step, the next 64-column panel after four; MN view: 2048 bytes per step
        const uint32_t ko = (uint32_t)(kk >> 2) * (kPanelB >> 4) + (uint32_t)(kk & 3) * 2u, mo = (uint32_t)kk * 128u;
        umma_ss(d_tmem, umma_desc_join(a_lo + (AOP == OP_K ? ko : mo)), umma_desc_join(b_lo + (BOP == OP_K ? ko : mo)), idesc,
                (acc || kk > 0) ? 1u : 0u);
    }
}

// The same with A in tensor memory: packed bf16, 8 columns per step, from column `a_tmem` on.
template <int BOP, int KSTEPS, int N>
__device__ __forceinline__ void mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_tile, bool acc) {
    constexpr uint32_t idesc = umma_idesc(128, N, OP_K, BOP);
    const uint32_t b_lo = umma_desc_lo(b_tile, BOP == OP_K ? 16u : kPanelB);
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) {
        const uint32_t ko = (uint32_t)(kk >> 2) * (kPanelB >> 4) + (uint32_t)(kk & 3) * 2u, mo = (uint32_t)kk * 128u;
        umma_ts(d_tmem, a_tmem + kk * 8, umma_desc_join(b_lo + (BOP == OP_K ? ko : mo)), idesc, (acc || kk > 0) ? 1u : 0u);
    }
}

// The same with A as half of a bf16 pair that lies where its float32 accumulator was: per 32 elements of the contraction 16 columns
// of hi, then 16 of lo (`a_tmem` = first column of the half).
template <int BOP, int KSTEPS, int N>
__device__ __forceinline__ void mma_tap(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_tile, bool acc) {
    constexpr uint32_t idesc = umma_idesc(128, N, OP_K, BOP);
    const uint32_t b_lo = umma_desc_lo(b_tile, BOP == OP_K ? 16u : kPanelB);
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) {
        const uint32_t ko = (uint32_t)(kk >> 2) * (kPanelB >> 4) + (uint32_t)(kk & 3) * 2u, mo = (uint32_t)kk * 128u;
        umma_ts(d_tmem, a_tmem + (kk >> 1) * 32 + (kk & 1) * 8, umma_desc_join(b_lo + (BOP == OP_K ? ko : mo)), idesc, (acc || kk > 0) ? 1u : 0u);
    }
}

// Stores columns c0 .. c0+31 of `row` of a swizzled bf16 tile.
__device__ __forceinline__ void tile_store32(uint8_t* t, int row, int c0, const float (&v)[32]) {
    uint8_t* panel = t + (c0 >> 6) * kPanelB;
    const int ch0 = (c0 & 63) >> 3;
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        *reinterpret_cast<uint4*>(panel + sw128_off((uint32_t)row, (uint32_t)(ch0 + ch))) =
            make_uint4(pack_bf16(v[8 * ch], v[8 * ch + 1]), pack_bf16(v[8 * ch + 2], v[8 * ch + 3]),
                       pack_bf16(v[8 * ch + 4], v[8 * ch + 5]), pack_bf16(v[8 * ch + 6], v[8 * ch + 7]));
}
// Row transfers between registers and global memory.  Lane L of a warp owns one row segment (32 consecutive values
// starting at its own pointer).  All 32 lanes must call together: the lanes of a group first swap 32-byte pieces so
// that one instruction covers whole rows (full 128- or 64-byte runs) instead of 32 scattered 16-byte pieces.
// `valid` = false: the lane's row is not written / reads as zero.  CALLER: the row lies in a caller's tensor (16-byte aligned),
// not in a workspace (see st_global_32).
__device__ __forceinline__ void ld_global_v8(const void* p, uint32_t (&v)[8]) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p)
                 : "memory");
}
template <bool CALLER = false>
__device__ __forceinline__ void gstore_f32x32(float* dst, const float (&v)[32], bool valid = true) {
    const int j = threadIdx.x & 3;
    uint32_t w[32];
#pragma unroll
    for (int x = 0; x < 32; ++x) w[x] = __float_as_uint(v[x]);
    rot4_pieces(w, j);
    const unsigned long long mine = (unsigned long long)dst;
#pragma unroll
    for (int r = 0; r < 4; ++r) {   // piece j of the row of lane (L ^ r)
        uint32_t d[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) d[x] = r == 0 ? w[x] : __shfl_xor_sync(0xffffffffu, w[8 * r + x], r);
        const unsigned long long ptr = r == 0 ? mine : __shfl_xor_sync(0xffffffffu, mine, r);
        const bool ok = r == 0 ? valid : (bool)__shfl_xor_sync(0xffffffffu, (int)valid, r);
        if (ok) st_global_32<CALLER>((uint8_t*)ptr + 32 * j, d);
    }
}
__device__ __forceinline__ void gload_f32x32(const float* src, float (&v)[32], bool valid = true) {
    const int j = threadIdx.x & 3;
    uint32_t d[4][8], w[32];
    const unsigned long long mine = (unsigned long long)src;
    unsigned long long ptr[4];
    bool ok[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        ptr[r] = r == 0 ? mine : __shfl_xor_sync(0xffffffffu, mine, r);
        ok[r] = r == 0 ? valid : (bool)__shfl_xor_sync(0xffffffffu, (int)valid, r);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {   // all four loads are in flight together
#pragma unroll
        for (int x = 0; x < 8; ++x) d[r][x] = 0u;
        if (ok[r]) ld_global_v8((const uint8_t*)ptr[r] + 32 * j, d[r]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int x = 0; x < 8; ++x) w[8 * r + x] = r == 0 ? d[r][x] : __shfl_xor_sync(0xffffffffu, d[r][x], r);
    rot4_pieces(w, j);
#pragma unroll
    for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(w[x]);
}
// 32 bf16 = 64 bytes per row: pairs of lanes.  `w`: the row segment as 16 packed words.
template <bool CALLER = false>
__device__ __forceinline__ void gstore_bf16_w16(__nv_bfloat16* dst, const uint32_t (&w)[16], bool valid = true) {
    const bool odd = threadIdx.x & 1;
    uint32_t first[8], second[8];   // halves [32 * odd, +32) of the even lane's row and of the odd lane's row
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, odd ? w[x] : w[8 + x], 1);
        first[x] = odd ? recv : w[x];
        second[x] = odd ? w[8 + x] : recv;
    }
    const unsigned long long mine = (unsigned long long)dst, other = __shfl_xor_sync(0xffffffffu, mine, 1);
    const bool ovalid = (bool)__shfl_xor_sync(0xffffffffu, (int)valid, 1);
    if (odd ? ovalid : valid) st_global_32<CALLER>((uint8_t*)(odd ? other : mine) + 32 * (int)odd, first);
    if (odd ? valid : ovalid) st_global_32<CALLER>((uint8_t*)(odd ? mine : other) + 32 * (int)odd, second);
}
// The load, in two halves, so that a caller can put other work between the request and the first use of the data: 32-byte pieces go to the lanes of a pair so that an instruction covers 64 bytes of each row it touches.
__device__ __forceinline__ void gload_bf16_issue(const __nv_bfloat16* src, uint32_t (&d)[2][8]) {
    const bool odd = threadIdx.x & 1;
    const unsigned long long mine = (unsigned long long)src, other = __shfl_xor_sync(0xffffffffu, mine, 1);
    ld_global_v8((const uint8_t*)(odd ? other : mine) + 32 * (int)odd, d[0]);   // of the even lane's row
    ld_global_v8((const uint8_t*)(odd ? mine : other) + 32 * (int)odd, d[1]);   // of the odd lane's row
}
__device__ __forceinline__ void gload_bf16_finish(const uint32_t (&d)[2][8], uint32_t (&w)[16]) {
    const bool odd = threadIdx.x & 1;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, odd ? d[0][x] : d[1][x], 1);   // the other half of this lane's row
        w[x] = odd ? recv : d[0][x];
        w[8 + x] = odd ? d[1][x] : recv;
    }
}
__device__ __forceinline__ void pack32(const float (&v)[32], uint32_t (&w)[16]) {
#pragma unroll
    for (int x = 0; x < 16; ++x) w[x] = pack_bf16(v[2 * x], v[2 * x + 1]);
}
template <bool CALLER = false>
__device__ __forceinline__ void gstore_bf16x32(__nv_bfloat16* dst, const float (&v)[32], bool valid = true) {
    uint32_t w[16];
    pack32(v, w);
    gstore_bf16_w16<CALLER>(dst, w, valid);
}
// t = hi + lo with hi = bf16(t) and lo = bf16(t - hi), both packed two per word.
__device__ __forceinline__ void split32(const float (&t)[32], uint32_t (&hi)[16], uint32_t (&lo)[16]) {
#pragma unroll
    for (int x = 0; x < 16; ++x) {
        const uint32_t h = pack_bf16(t[2 * x], t[2 * x + 1]);
        hi[x] = h;
        lo[x] = pack_bf16(t[2 * x] - __uint_as_float(h << 16), t[2 * x + 1] - __uint_as_float(h & 0xffff0000u));
    }
}
// Packed counterpart of tile_store32.
__device__ __forceinline__ void tile_store_w16(uint8_t* t, int row, int c0, const uint32_t (&w)[16]) {
    uint8_t* panel = t + (c0 >> 6) * kPanelB;
    const int ch0 = (c0 & 63) >> 3;
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        *reinterpret_cast<uint4*>(panel + sw128_off((uint32_t)row, (uint32_t)(ch0 + ch))) =
            make_uint4(w[4 * ch], w[4 * ch + 1], w[4 * ch + 2], w[4 * ch + 3]);
}
__device__ __forceinline__ void unpack_bf16x32(const uint4 (&u4)[4], float (&v)[32]) {
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const uint32_t w[4] = {u4[x].x, u4[x].y, u4[x].z, u4[x].w};
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[y]));
            v[8 * x + 2 * y] = f.x;
            v[8 * x + 2 * y + 1] = f.y;
        }
    }
}
// Columns c0 .. c0+31 of `row` of a swizzled bf16 tile.
__device__ __forceinline__ void tile_load32(const uint8_t* t, int row, int c0, float (&v)[32]) {
    const uint8_t* panel = t + (c0 >> 6) * kPanelB;
    uint4 u[4];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        u[ch] = *reinterpret_cast<const uint4*>(panel + sw128_off((uint32_t)row, (uint32_t)(((c0 & 63) >> 3) + ch)));
    unpack_bf16x32(u, v);
}
__device__ __forceinline__ void tmem_row32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    tmem_ld32(taddr, r);
    tmem_ld_wait();
#pragma unroll
    for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r[x]);
}
// The same from a caller's tensor [slices][L][ncols]: rows row .. row + 127 of a slice, zeros past its end.
__device__ __forceinline__ void tma_rows(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int ncols, int row, int slice) {
    for (int h = 0; h < ncols / 64; ++h) tma_load_3d(dst + h * kPanelB, m, bar, h * 64, row, slice);
}
// TMA load of a [128 x ncols] bf16 tile (ncols = 64 or 128) whose first row is `row0` of the mapped matrix.
__device__ __forceinline__ void tma_tile(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int ncols, int row0) {
    for (int h = 0; h < ncols / 64; ++h) tma_load_2d(dst + h * kPanelB, m, bar, h * 64, row0);
}

}  // namespace tile
}  // namespace path
