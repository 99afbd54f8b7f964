// pack (offline reorder), standalone dequant, the plain FP32-FMA GEMM and the Split-K
// reduce kernel.
#pragma once

#include "common.cuh"

namespace w4a16 {

// The three kernels below work on whole blocks (64 columns x 128 k), numbered with the column tile fastest, so that the
// CTAs that run together touch neighbouring columns of the same rows.
constexpr int kBlockKernelThreads = 128;
struct BlockPos {
    int t, g;        // column tile, k block
    size_t blk;      // position in the packed buffers
    __device__ __forceinline__ BlockPos(int b, int T, int G) : t(b % T), g(b / T), blk((size_t)t * G + g) {}
};

// Programmatic dependent launch: the kernel behind this one may be set up while this one runs, and this one was set up while
// the kernel in front of it ran.  Every CTA of a kernel launched that way waits, also one without work: what comes behind
// counts on this grid not ending before the one in front of it.  (Their inputs are read past the L1 cache: the kernel in front
// may have written them while this one was already on the SM.)
__device__ __forceinline__ void next_launch_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_launch_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------ pack
// Raw word (nibble i = k + i) -> packed word (even k in the low half, odd k in the high half, ascending).
__device__ __forceinline__ uint32_t pack_word(uint32_t r) {
    const uint32_t e = r & 0x0f0f0f0fu, o = (r >> 4) & 0x0f0f0f0fu;
    return __byte_perm(e | (e >> 4), o | (o >> 4), 0x6420);
}

// One warp per half block (32 columns x 128 k).  A lane reads four consecutive k-words of one column (32 columns: 128 bytes a
// row) and writes them as the column's 16-byte chunk: eight columns make up a 128-byte line.  Scales and zero points of the
// half block go along in the same launch, half a warp per row.  The launch is latency: a warp's loads, all of them ahead of its first
// store.  us, K = 11008 / N = 4096, a row of calls / one by itself: a warp per block, plain launch 12.4 / 15.2, in groups of 32
// 12.4 / 15.8; half a block, the rows of scales one after the other behind the words 10.6 / 16.2 and 12.7 / 18.2; this form
// 9.6 / 14.7 and 10.6 / 16.0 (HBM floor 7.2).
__global__ void __launch_bounds__(kBlockKernelThreads)
pack_kernel(const uint32_t* __restrict__ Wq_raw, const uint16_t* __restrict__ S_raw, const uint8_t* __restrict__ Z_raw,
            uint32_t* __restrict__ Wq, uint16_t* __restrict__ S, uint8_t* __restrict__ Z, int N, int G, int sg, int blocks, bool release) {
    if (release) next_launch_may_start();
    wait_for_launch_before();            // (every warp: see there)
    const int i = blockIdx.x * (kBlockKernelThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int b = i >> 1, h = i & 1;
    if (b >= blocks) return;
    const BlockPos pos(b, N / kTileN, G);
    const uint32_t* src = Wq_raw + (size_t)pos.g * (kGroup / 8) * N + (size_t)pos.t * kTileN + 32 * h + lane;
    uint32_t r[16];
#pragma unroll
    for (int kw = 0; kw < 16; ++kw) r[kw] = __ldcg(src + (size_t)kw * N);
    // Half a warp per row of scales / zero points: rows lane / 16 and that + 2.  Positions 32 h + 2 p, + 1 (p = lane & 15) of a
    // row belong to columns c0, c0 + 8 (sz_perm).
    const int p = lane & 15, c0 = 32 * h + (p >> 1) + (p & 1) * 16;
    uint32_t s[2], z[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int j = (lane >> 4) + 2 * i;
        if (j < sg) {
            const size_t in = (size_t)(pos.g * sg + j) * N + (size_t)pos.t * kTileN + c0;
            s[i] = (uint32_t)__ldcg(S_raw + in) | ((uint32_t)__ldcg(S_raw + in + 8) << 16);
            if (Z_raw != nullptr) z[i] = (__ldcg(Z_raw + in) & 15u) | ((uint32_t)__ldcg(Z_raw + in + 8) << 4);
        }
    }
    __syncwarp();                        // (all loads stay ahead of the first store)
    uint4* dst = reinterpret_cast<uint4*>(Wq + pos.blk * kBlockWords);
#pragma unroll
    for (int q = 0; q < 4; ++q)          // k-words 4 q .. 4 q + 3
        dst[block_word_index(32 * h + lane, 4 * q) / 4] =
            make_uint4(pack_word(r[4 * q]), pack_word(r[4 * q + 1]), pack_word(r[4 * q + 2]), pack_word(r[4 * q + 3]));
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int j = (lane >> 4) + 2 * i;
        if (j < sg) {
            const size_t row = pos.blk * sg + j;
            reinterpret_cast<uint32_t*>(S + row * kSBlockHalves)[16 * h + p] = s[i];
            if (Z_raw != nullptr) Z[row * (kZBlockWords * 4) + 16 * h + p] = (uint8_t)z[i];
        }
    }
}

// Scale (16-bit pattern) and zero point of column `col` for the k-word kw (0..15) of block blk.
__device__ __forceinline__ void load_sz(const uint16_t* __restrict__ S, const uint32_t* __restrict__ Z, size_t blk,
                                        int sg, int col, int kw, uint16_t& s, uint32_t& z) {
    const int j = (kw * 8) / (kGroup / sg);
    const size_t row = blk * sg + j;
    const int p = sz_perm(col);
    s = S[row * kSBlockHalves + p];
    z = Z == nullptr ? (uint32_t)kSymZero : ((Z[row * kZBlockWords + (p >> 3)] >> (4 * (p & 7))) & 15u);
}

// ------------------------------------------------------------------ quantize (the step before the path)
// Eq. 1, x_q = round(x / s) + z, per group of `group` consecutive k of one column.  Asymmetric:
// s = (max - min) / 15 rounded to the 16-bit format, z = clamp(round(-min / s), 0, 15); symmetric:
// s = max|x| / 7, z = 8; a zero or non-finite s becomes 1; q = clamp(round(x / s) + z, 0, 15), ties to
// even.  Every operation is one IEEE binary32 operation in this order, because the results are
// integers decided by floating point.  Output in the raw layout that w4a16_pack consumes.
template <bool BF>
__device__ __forceinline__ float group_scale(float num, float den, uint16_t& bits) {
    bits = cast_out<BF>(__fdiv_rn(num, den));
    float s = widen<BF>(bits);
    if (!(s > 0.0f) || isinf(s)) {
        s = 1.0f;
        bits = cast_out<BF>(1.0f);
    }
    return s;
}

template <bool BF>
__device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr (BF) asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("min.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
template <bool BF>
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
    uint32_t r;
    if constexpr (BF) asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    else asm("max.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// One code of the definition above, and eight of a column as a raw word (out of line: groups whose scale has no normal
// reciprocal hardly ever come, and in line the divisions were four fifths of the kernel's code).
__device__ __forceinline__ uint32_t quantize_exact(float x, float s, int z) {
    const float r = __fadd_rn(rintf(__fdiv_rn(x, s)), (float)z);
    return (uint32_t)(r < 0.0f ? 0 : r > 15.0f ? 15 : (int)r);
}
template <bool BF>
__device__ __noinline__ uint32_t quantize_word_exact(const uint16_t* x, int N, float s, int z) {
    uint32_t w = 0u;
#pragma unroll 1
    for (int i = 0; i < 8; ++i) w |= quantize_exact(widen<BF>(__ldcg(x + (size_t)i * N)), s, z) << (4 * i);
    return w;
}

// Two FP32 operations in one instruction.
__device__ __forceinline__ uint64_t pair_f32(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// One CTA per 64 columns x 128 k, each of its four warps 32 k: a lane keeps its two columns' 32 rows in registers (128
// bytes a row and warp, every weight read once), warps of the same group exchange minimum and maximum through shared
// memory.  Codes without a division: u = x * (1 / s) + 768 in one FMA is the quotient rounded to a multiple of 2^-14 (where it is below
// 256), and that has the same nearest integer, ties to even, as the definition's
// fl(x / s): x = X 2^a and s = T 2^b have 11-bit significands, so x - h s for a half-integer h is zero or at least
// 2^min(a, b - 1), which with |h| >= 1/2 (hence a >= b - 2) is more than 2^-13 of s.  The reciprocal, the FMA and the
// definition's own division are off by less than 2^-19, the grid by at most 2^-15: a tie lands on the half exactly,
// anything else stays on its side of it.  (Scales whose reciprocal is not a normal number take the divisions.)  The clamp to
// 0 .. 15 comes first, on the 16-bit weights, two at a time: x between -z s and (15 - z) s, each rounded to 16 bits.  Those
// bounds are within 2^-9 of themselves, so their own codes are 0 and 15, and what lies beyond them has no other code.
// What bounds it: memory while a CTA loads, instructions while it computes (13 a pair of weights), overlapped only between
// CTAs.  K = 11008 / N = 4096: a thread per (group, column), two passes and a division per weight 96 us; FP32 clamps, one
// column at a time and the divisions in line (25 % of the warp time went into fetching instructions, now 7) 28.9; this form 23.4
// (HBM floor 17.4).  Held to 48 registers for ten CTAs an SM it spills.
template <bool BF>
__global__ void __launch_bounds__(kBlockKernelThreads)
quantize_kernel(const uint16_t* __restrict__ W16, uint32_t* __restrict__ Wq, uint16_t* __restrict__ S,
                uint8_t* __restrict__ Z, int N, int G, int sg, int symmetric) {
    __shared__ uint32_t part_lo[4][32], part_hi[4][32];
    const BlockPos pos(blockIdx.x, N / kTileN, G);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    next_launch_may_start();
    wait_for_launch_before();
    const size_t n = (size_t)pos.t * kTileN + 2 * lane;
    const uint16_t* src = W16 + (size_t)(pos.g * kGroup + warp * 32) * N + n;
    uint32_t v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __ldcg(reinterpret_cast<const uint32_t*>(src + (size_t)k * N));
    uint32_t lo = BF ? 0x7f807f80u : 0x7c007c00u, hi = lo | 0x80008000u;     // +inf, -inf
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        lo = min2<BF>(lo, v[k]);
        hi = max2<BF>(hi, v[k]);
    }
    const int wpg = 4 / sg, first = warp / wpg * wpg;    // warps that share a group, the first of them
    part_lo[warp][lane] = lo;
    part_hi[warp][lane] = hi;
    __syncthreads();
    for (int i = 0; i < wpg; ++i) {
        lo = min2<BF>(lo, part_lo[first + i][lane]);
        hi = max2<BF>(hi, part_hi[first + i][lane]);
    }
    constexpr float kGrid = 768.0f;                      // 1.5 * 2^9: neighbours 2^-14 apart
    constexpr float kMagic = 12582912.0f;                // 1.5 * 2^23, bits 0x4b400000: neighbours 1 apart
    uint16_t sb[2];
    float s[2], rinv[2];
    uint32_t least = 0u, most = 0u;
    int z[2];
    bool slow[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float l = widen<BF>((uint16_t)(lo >> (16 * c))), h = widen<BF>((uint16_t)(hi >> (16 * c)));
        if (symmetric) {
            s[c] = group_scale<BF>(fmaxf(fabsf(l), fabsf(h)), 7.0f, sb[c]);
            z[c] = kSymZero;
        } else {
            s[c] = group_scale<BF>(__fsub_rn(h, l), 15.0f, sb[c]);
            const float zf = rintf(__fdiv_rn(-l, s[c]));
            z[c] = zf < 0.0f ? 0 : zf > 15.0f ? 15 : (int)zf;
        }
        rinv[c] = __frcp_rn(s[c]);
        least |= (uint32_t)cast_out<BF>(-(float)z[c] * s[c]) << (16 * c);          // codes 0 and 15
        most |= (uint32_t)cast_out<BF>((float)(15 - z[c]) * s[c]) << (16 * c);
        slow[c] = !(s[c] > 1e-30f && s[c] < 1e30f);
    }
    const size_t out = (size_t)(pos.g * sg + warp / wpg) * N + n;
    if (warp == first) {
        *reinterpret_cast<uint32_t*>(S + out) = (uint32_t)sb[0] | ((uint32_t)sb[1] << 16);
        if (Z != nullptr) *reinterpret_cast<uint16_t*>(Z + out) = (uint16_t)(z[0] | (z[1] << 8));
    }
    const uint64_t rinv2 = pair_f32(rinv[0], rinv[1]), grid2 = pair_f32(kGrid, kGrid), magic2 = pair_f32(kMagic - kGrid, kMagic - kGrid);
    const uint32_t zw[2] = {((uint32_t)z[0] - 0x4b400000u) * 0x11111111u, ((uint32_t)z[1] - 0x4b400000u) * 0x11111111u};
    uint32_t* dst = Wq + (size_t)(pos.g * (kGroup / 8) + warp * 4) * N + n;
#pragma unroll
    for (int kw = 0; kw < 4; ++kw) {
        uint32_t w[2] = {0u, 0u};
#pragma unroll
        for (int i = 7; i >= 0; --i) {
            const uint32_t x = min2<BF>(max2<BF>(v[8 * kw + i], least), most);
            const uint64_t u = fma_f32x2(pair_f32(widen<BF>((uint16_t)x), widen<BF>((uint16_t)(x >> 16))), rinv2, grid2);
            const uint64_t y = add_f32x2(u, magic2);     // low bits: round(x / s)
            w[0] = w[0] * 16u + (uint32_t)y;
            w[1] = w[1] * 16u + (uint32_t)(y >> 32);
        }
        // + z in each digit, the constant's copies out again
        w[0] += zw[0];
        w[1] += zw[1];
        if (slow[0]) w[0] = quantize_word_exact<BF>(src + (size_t)(8 * kw) * N, N, s[0], z[0]);
        if (slow[1]) w[1] = quantize_word_exact<BF>(src + (size_t)(8 * kw) * N + 1, N, s[1], z[1]);
        *reinterpret_cast<uint2*>(dst + (size_t)kw * N) = make_uint2(w[0], w[1]);
    }
}

// ------------------------------------------------------------------ dequant
// Algorithm 1, Phase 1 as a standalone kernel: w16 = rn((q - z) * s) in the 16-bit format: (q - z) is formed exactly and
// multiplied by s with one multiply (round-to-nearest-even, subnormals kept).  Z == nullptr: symmetric format, z = 8.
// One CTA per block, a warp for 32 k of it: a lane takes 8 neighbouring columns x 8 k (a word of each column), swaps the halves
// of neighbouring columns' registers and stores 16 bytes of a row at a time, eight lanes one 128-byte line of the row.  The
// packed words come through shared memory, 16 bytes a load: fetched word by word a warp's load touches eight lines, and the
// L1 was the busiest unit (75 %; it still is, 73 % of a shorter time, the stores' part).  The 256-byte sub-blocks lie 272 bytes apart, so that the words a warp reads at a time come from
// 32 banks.  Bound by HBM, most of it the stores.  us, a thread per word with 2-byte stores / word loads, plain launch / this form:
// K = N = 8192 68 / 31.2 / 28.5 (HBM floor 26.3, a device copy of as many bytes 28.8), K = 11008 / N = 4096 - / 22.8 / 19.7 (17.6).
template <bool BF>
__global__ void __launch_bounds__(kBlockKernelThreads)
dequant_kernel(const uint32_t* __restrict__ Wq, const uint16_t* __restrict__ S, const uint32_t* __restrict__ Z,
               uint16_t* __restrict__ W16, int N, int G, int sg) {
    constexpr int kSub = 64, kSubStride = 68;           // words
    __shared__ __align__(16) uint32_t packed[kBlockWords / kSub * kSubStride];
    next_launch_may_start();
    wait_for_launch_before();
    const BlockPos pos(blockIdx.x, N / kTileN, G);
    const int kq = threadIdx.x >> 5, kw = (threadIdx.x >> 3) & 3, rb = threadIdx.x & 7;   // columns 8 rb .. + 7, k = 32 kq + 8 kw .. + 7
    const uint4* src = reinterpret_cast<const uint4*>(Wq + pos.blk * kBlockWords) + threadIdx.x;
    const uint4 lo = __ldcg(src), hi = __ldcg(src + kBlockKernelThreads);
    const size_t row = pos.blk * sg + kq * sg / 4;
    // column 8 rb + c sits at position p0 + 4 c of a row of scales / zero points
    const int p0 = sz_perm(8 * rb);
    uint4 zz = make_uint4(0u, 0u, 0u, 0u);
    if (Z != nullptr) zz = __ldcg(reinterpret_cast<const uint4*>(Z + row * kZBlockWords) + (p0 >> 5));
    const uint32_t zw[4] = {zz.x, zz.y, zz.z, zz.w};
    uint32_t s2[8], zlo[8], zhi[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) s2[c] = (uint32_t)__ldcg(S + row * kSBlockHalves + p0 + 4 * c) * 0x00010001u;
    uint4* dst4 = reinterpret_cast<uint4*>(packed) + threadIdx.x + threadIdx.x / (kSub / 4);    // (a sub-block is 16 pieces, 17 with its gap)
    dst4[0] = lo;
    dst4[kBlockKernelThreads / (kSub / 4) * (kSubStride / 4)] = hi;
    __syncthreads();
    uint32_t w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int at = block_word_index(c, 4 * kq) + kw;       // of column c; sub-block rb of that half is rb further
        w[c] = packed[(at / kSub + rb) * kSubStride + at % kSub];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint32_t z = Z == nullptr ? (uint32_t)kSymZero : ((zw[c >> 1] >> (16 * (c & 1) + 4 * (p0 & 3))) & 15u);
        zlo[c] = zconst_lo<BF>(z);
        zhi[c] = zconst_hi<BF>(z);
    }
    uint16_t* dst = W16 + (size_t)(pos.g * kGroup + 32 * kq + 8 * kw) * N + (size_t)pos.t * kTileN + 8 * rb;
    Pack8 f[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) f[c] = dequant_word<BF>(w[c], zlo[c], zhi[c], s2[c]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint16_t* p = dst + (size_t)(2 * j) * N;
        *reinterpret_cast<uint4*>(p) = make_uint4(__byte_perm(f[0].h[j], f[1].h[j], 0x5410), __byte_perm(f[2].h[j], f[3].h[j], 0x5410),
                                                  __byte_perm(f[4].h[j], f[5].h[j], 0x5410), __byte_perm(f[6].h[j], f[7].h[j], 0x5410));
        *reinterpret_cast<uint4*>(p + N) = make_uint4(__byte_perm(f[0].h[j], f[1].h[j], 0x7632), __byte_perm(f[2].h[j], f[3].h[j], 0x7632),
                                                      __byte_perm(f[4].h[j], f[5].h[j], 0x7632), __byte_perm(f[6].h[j], f[7].h[j], 0x7632));
    }
}

// ------------------------------------------------------------------ plain GEMM
// Correct-first kernel: one thread per output column of a 64-column tile, kSimpleMB batch
// rows per thread, FP32 FMA over this CTA's K-slice.  Grid: (N/64,
// ceil(M/kSimpleMB), split_k).  With split_k == 1 it writes C, else FP32 partials
// ws[split][M][N] (Algorithm 1, Phase 2) for splitk_reduce_kernel.
constexpr int kSimpleMB = 4;

__device__ __forceinline__ void slice_of(int G, int split_k, int sp, int& g0, int& ng) {
    int base = G / split_k, rem = G % split_k;
    g0 = sp * base + min(sp, rem);
    ng = base + (sp < rem ? 1 : 0);
}

template <bool BF>
__global__ void __launch_bounds__(64)
gemm_simple_kernel(const uint16_t* __restrict__ A, const uint32_t* __restrict__ Wq, const uint16_t* __restrict__ S,
                   const uint32_t* __restrict__ Z, uint16_t* __restrict__ C, float* __restrict__ ws, int M, int N,
                   int K, int G, int sg, int split_k, Epilogue epi) {
    const int t = blockIdx.x, m0 = blockIdx.y * kSimpleMB, sp = blockIdx.z;
    const int col = threadIdx.x;  // column inside the tile
    int g0, ng;
    slice_of(G, split_k, sp, g0, ng);

    float acc[kSimpleMB];
#pragma unroll
    for (int i = 0; i < kSimpleMB; ++i) acc[i] = 0.f;

    for (int g = g0; g < g0 + ng; ++g) {
        const size_t blk = (size_t)t * G + g;
        const uint32_t* wb = Wq + blk * kBlockWords;
        for (int kw = 0; kw < kGroup / 8; ++kw) {
            uint16_t sb;
            uint32_t z;
            load_sz(S, Z, blk, sg, col, kw, sb, z);
            const float s = widen<BF>(sb);
            const uint32_t w = wb[block_word_index(col, kw)];
            const int k0 = g * kGroup + kw * 8;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const int off = 2 * (p & 3) + (p >> 2);
                const int q = (int)((w >> (4 * p)) & 15u);
                // (q - z) * s is exact in FP32; one rounding to the 16-bit format, as in Phase 1
                const float w16 = widen<BF>(cast_out<BF>((float)(q - (int)z) * s));
#pragma unroll
                for (int mm = 0; mm < kSimpleMB; ++mm) {
                    if (m0 + mm < M)
                        acc[mm] = fmaf(widen<BF>(A[(size_t)(m0 + mm) * K + k0 + off]), w16, acc[mm]);
                }
            }
        }
    }
    const int n = t * kTileN + col;
#pragma unroll
    for (int mm = 0; mm < kSimpleMB; ++mm) {
        if (m0 + mm < M) {
            if (split_k == 1)
                C[(size_t)(m0 + mm) * N + n] = finish<BF>(acc[mm], n, epi);
            else
                ws[((size_t)sp * M + m0 + mm) * N + n] = acc[mm];
        }
    }
}

// Algorithm 1, Phase 3: C = rn16(sum_{i<S} C_i), ascending i, FP32.
template <bool BF>
__global__ void splitk_reduce_kernel(const float* __restrict__ ws, uint16_t* __restrict__ C, size_t MN, int N,
                                     int split_k, Epilogue epi) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MN) return;
    float acc = ws[i];
    for (int s = 1; s < split_k; ++s) acc += ws[(size_t)s * MN + i];
    C[i] = finish<BF>(acc, (int)(i % (size_t)N), epi);
}

// Algorithm 1, Phase 3 for the tcgen05 kernels whose partial tiles went to the workspace (FP32, [batch row in tile][128
// columns]; the first segment of chunk c in slot 2 c, its continuation into a later tile in slot 2 c + 1): this kernel,
// launched behind, sums them in ascending K, applies the optional bias / activation and rounds once.  A thread takes four
// neighbouring columns of one batch row, a block eight rows of one tile.  Inside the GEMM kernel the same sum was a chain of
// L2 round trips in the one CTA per tile that finished last (5 to 10 us of a 32 us launch at M = 256); here the whole GPU
// does it at once.
struct TileReduce {
    int M, N, G, mt, n_tiles;
    int split_k;                 // S >= 2: S slices per tile; 0: balanced chunks
    int nchunks, bal_q, bal_r;   // balanced: units = bal_q nchunks + bal_r
    FastDiv div_mt, div_ntiles;
    Epilogue epi;
};
template <bool BF>
__global__ void __launch_bounds__(256)
tile_splitk_reduce_kernel(const float* __restrict__ ws, uint16_t* __restrict__ C, const TileReduce p) {
    __shared__ int chunks[3];                           // first and last contributor, slot of the first
    // the next kernel of the stream may start its prologue; the partial tiles are the previous kernel's output
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5);   // (tiles * mt < 2^31: gemm_plan)
    const int T = fast_div(r, p.div_mt);                // tile = batch tile * n_tiles + column tile; mt % 16 == 0: one per block
    if (threadIdx.x == 0) {
        if (p.split_k > 0) {
            chunks[0] = T * p.split_k;
            chunks[1] = chunks[0] + p.split_k - 1;
            chunks[2] = 2 * chunks[0];
        } else {
            const long long units = (long long)p.bal_q * p.nchunks + p.bal_r, u0 = (long long)T * p.G;
            const int c0 = (int)(((u0 + 1) * p.nchunks - 1) / units);
            chunks[0] = c0;
            chunks[1] = (int)(((u0 + p.G) * p.nchunks - 1) / units);
            chunks[2] = 2 * c0 + ((long long)c0 * p.bal_q + (long long)c0 * p.bal_r / p.nchunks == u0 ? 0 : 1);
        }
    }
    __syncthreads();
    const int c_first = chunks[0], c_last = chunks[1];
    // Every CTA waits, also one without work: the launch behind this kernel counts on this grid not ending before the GEMM.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (c_first == c_last) return;                      // one chunk has the whole tile and has written it
    const int m_local = r - T * p.mt;
    const int mt_i = fast_div(T, p.div_ntiles), nt = T - mt_i * p.n_tiles;
    const int m = mt_i * p.mt + m_local, n = nt * 128 + (int)(threadIdx.x & 31) * 4;
    if (m >= p.M || n >= p.N) return;
    const size_t slot = (size_t)p.mt * 128, step = 2 * slot;   // floats of a slot; between the first segments of neighbouring chunks
    const float* base = ws + (size_t)m_local * 128 + (threadIdx.x & 31) * 4;
    float4 acc = __ldcg(reinterpret_cast<const float4*>(base + (size_t)chunks[2] * slot));
    const float* src = base + (size_t)(c_first + 1) * step;
    int c = c_first + 1;
    for (; c + 2 <= c_last; c += 3, src += 3 * step) {  // three contributors' loads in flight, added in order
        const float4 x0 = __ldcg(reinterpret_cast<const float4*>(src));
        const float4 x1 = __ldcg(reinterpret_cast<const float4*>(src + step));
        const float4 x2 = __ldcg(reinterpret_cast<const float4*>(src + 2 * step));
        acc.x += x0.x; acc.y += x0.y; acc.z += x0.z; acc.w += x0.w;
        acc.x += x1.x; acc.y += x1.y; acc.z += x1.z; acc.w += x1.w;
        acc.x += x2.x; acc.y += x2.y; acc.z += x2.z; acc.w += x2.w;
    }
    for (; c <= c_last; ++c, src += step) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(src));
        acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
    }
    const uint32_t lo = (uint32_t)finish<BF>(acc.x, n, p.epi) | ((uint32_t)finish<BF>(acc.y, n + 1, p.epi) << 16);
    const uint32_t hi = (uint32_t)finish<BF>(acc.z, n + 2, p.epi) | ((uint32_t)finish<BF>(acc.w, n + 3, p.epi) << 16);
    *reinterpret_cast<uint2*>(C + (size_t)m * p.N + n) = make_uint2(lo, hi);
}

// Activations from page-locked host memory into the staging buffer, ahead of the GEMM (w4a16_gemm_host).  The copy engine
// would need a semaphore each way and 5.5 us of host time a call; a kernel reads the same bytes over PCIe, and the GEMM
// behind it starts its prologue and weight requests meanwhile (programmatic dependent launch).
constexpr int kStageThreads = 128;       // at most
__global__ void __launch_bounds__(kStageThreads)
stage_activations_kernel(const uint4* __restrict__ host, uint4* __restrict__ dev, int n16) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the staging buffer may still be read, and the host buffer written, by what comes before on the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += gridDim.x * blockDim.x) dev[i] = __ldcv(host + i);
}

// Diagnostic: one warp waits on a barrier that nobody ever arrives on, with a limit of `limit_ns`.  The wait
// runs out, records kStatusMbarTimeout in the status word and the kernel returns normally: the same exit
// every GEMM kernel takes when one of its waits gives up, exercised without any fault.
__global__ void wait_timeout_probe_kernel(unsigned long long limit_ns, int* gave_up) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0u, limit_ns);
    if (threadIdx.x == 0 && gave_up != nullptr) *gave_up = ok ? 0 : 1;
}

}  // namespace w4a16
