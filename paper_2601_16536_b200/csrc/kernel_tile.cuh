// Tensor-core tile kernel of the W4A16 GEMM: tcgen05.mma with the accumulator in tensor memory.
//
// The product is computed transposed, C^T[n, m] = sum_k W16[k, n] A[m, k], so that the
// DEQUANTIZED WEIGHTS are the MMA's 128-row A operand and live only in tensor memory:
//
//   HBM --128-bit loads--> registers (packed nibbles, scale, zero)    16 dequant warps,
//   registers: unpack, (q - z) exact, * s in FP16                      one column n per thread
//   registers --tcgen05.st--> TMEM (A operand, one column n per lane, k packed along columns)
//   HBM --TMA tensor (128B swizzle)--> shared (activation tile, MT rows m x 64 k): B operand
//   tcgen05.mma.kind::f16  D[128 n x MT m] (FP32, TMEM) += A(TMEM) . B(shared)   one elected lane
//   TMEM --tcgen05.ld--> registers -> FP16 C, or FP32 partial tile (Split-K)
//
// so packed weights go from HBM straight to registers, dequantized weights never touch shared or
// global memory (Algorithm 1's Phase 1 output stays on chip), and the activation tile is re-used
// by all 128 columns of the CTA tile.
//
// Work is counted in units: one unit = 128 columns x one group (128 k) of one batch tile, numbered
// U = (batch tile * NT + column tile) * G + group.  The unit range is cut into chunks, each CTA of
// the persistent grid walks its chunk(s) front to back:
//   - balanced (split_k == 0): as many chunks as CTAs, equal to within one unit; a chunk may start
//     and end inside a tile's K range and may cover several whole tiles in between;
//   - classic Split-K (split_k = S): every tile's K range is cut into S slices of whole groups
//     (Algorithm 1, Phase 2), chunks dealt round-robin.
// The part of a chunk inside one tile is a segment: the accumulator is zeroed at its first MMA and
// drained after its last.  A segment that covers a whole tile is cast to FP16 and stored; any other
// segment leaves as an FP32 partial tile in the workspace, for the kernel launched behind this one that adds them in
// ascending K order (Phase 3, tile_splitk_reduce_kernel).  No warp ever waits for another CTA, and the order of the sum is
// fixed, so results are bit-identical from run to run.
//
// Batch tiles of up to 256 rows, a run-time multiple of 16 (MT; which shapes come here and which go to kernel_mid.cuh is
// the host's choice by cost).  One pipeline stage is half a group (64 k, four MMAs).
// A ring of R slots holds, per slot, the stage's activation box in shared memory and its dequantized weights in tensor
// memory (32 columns; eight slots fit beside the accumulator).  Four sets of four dequant warps take stages round-robin;
// inside a set warp w owns TMEM lanes 32 (w % 4) .. + 31.  Each thread keeps the packed words of its next two stages in
// registers (loads issued that far ahead, pointers stepped, no register copies).  The packed weights do not depend on the
// previous kernel in the stream: under programmatic dependent launch the dequant warps load and
// convert weights until the TMEM ring is full before anything waits for that kernel; only
// activations, C and the workspace are touched after griddepcontrol.wait.
// The producer and issuer warps run warp-uniform loops and elect one lane per instruction, which
// keeps descriptors in uniform registers.  All waits are bounded mbarrier waits; a wait that runs
// out records a status code and the CTA drains and exits (TMEM is always released).
//
// Which schedule a shape gets when the caller leaves split_k open is the host's choice (api.cu):
// partial tiles are dear (FP32 store, reload; in mid-chunk they also stall the pipeline), so
// balanced chunks are used only where the SMs left idle by whole slices or whole tiles cost more.
#pragma once


#include "common.cuh"

namespace w4a16 {

constexpr int kTileCols = 128;                      // n per CTA tile = UMMA M
constexpr int kTileBoxK = 64;                       // k per activation TMA box (one 128-byte swizzle row)
constexpr int kTileStageK = 64;                     // k per pipeline stage
constexpr int kTileSPU = kGroup / kTileStageK;      // stages per unit
constexpr int kTileDequantWarps = 16;               // four sets of four (one warp per TMEM lane quarter)
constexpr int kTileSets = kTileDequantWarps / 4;
constexpr int kTileThreads = (2 + kTileDequantWarps) * 32;   // producer, issuer, dequant / epilogue warps
constexpr int kTileMaxStages = 8;                   // ring slots: activation box + stage_k / 2 TMEM columns each
// TMEM columns: the accumulator first, then the operand ring
constexpr int kTileACol = 256;
constexpr int kTileSlots = (512 - kTileACol) / (kTileStageK / 2);
constexpr int kTilePrefetch = 2;                    // stages of packed words a dequant thread holds in registers
constexpr int kTileBarBytes = 1024;

__host__ __device__ constexpr int tile_stage_bytes(int mt) { return mt * kTileStageK * 2; }

struct TileParams {
    const uint32_t* Wq;
    const uint16_t* S;
    const uint32_t* Z;   // nullptr: symmetric format, zero point 8
    uint16_t* C;
    float* ws;       // partial tiles: [2 * nchunks slots][MT][128] FP32
    int M, N, K, G;
    int mt;          // batch rows of a tile: multiple of 16, at most 256
    int n_tiles;     // NT = ceil(N / 128)
    int m_tiles;     // ceil(M / MT)
    int split_k;     // 0: balanced chunks; S >= 1: classic Split-K
    int nchunks;
    int stages;
    // chunk arithmetic, prepared by the host (tile_fill_chunk_math); units = m_tiles n_tiles G < 2^31
    FastDiv div_G, div_split, div_nchunks, div_ntiles;
    int slice_base, slice_rem;   // classic: G / split_k, G % split_k
    int bal_q, bal_r;            // balanced: units / nchunks, units % nchunks
    Epilogue epi;
};

inline void tile_fill_chunk_math(TileParams& p) {
    p.div_G = fast_div_make((uint32_t)p.G);
    p.div_split = fast_div_make((uint32_t)(p.split_k > 0 ? p.split_k : 1));
    p.div_nchunks = fast_div_make((uint32_t)p.nchunks);
    p.div_ntiles = fast_div_make((uint32_t)p.n_tiles);
    p.slice_base = p.split_k > 0 ? p.G / p.split_k : 0;
    p.slice_rem = p.split_k > 0 ? p.G % p.split_k : 0;
    const long long units = (long long)p.m_tiles * p.n_tiles * p.G;
    p.bal_q = (int)(units / p.nchunks);
    p.bal_r = (int)(units % p.nchunks);
}

// ------------------------------------------------------------------ tcgen05 / TMA wrappers
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) { tc_commit(smem_u32(bar)); }
// D(tmem) (+)= A(tmem) . B(shared descriptor); `accumulate` == 0 overwrites D.
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The same with the descriptor as two words, of which only the low one (the address) changes from one MMA to the next.
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 16 consecutive 32-bit TMEM columns of this thread's lane <- registers.
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tc_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major operand tile stored as 128-byte rows with the
// 128-byte swizzle (what the activation TMA writes): 8-row groups are 1024 B apart, the
// leading-dimension offset is unused for a tile one swizzle atom wide, descriptor version 1,
// layout code 2 = 128-byte swizzle.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                    // leading byte offset (ignored for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;          // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                    // descriptor version
    d |= (uint64_t)2 << 61;                    // SWIZZLE_128B
    return d;
}

// kind::f16 instruction descriptor: FP32 accumulator, A and B both FP16 or both BF16, both K-major,
// M = 128, N = mt.
__host__ __device__ constexpr uint32_t tile_idesc(int mt, bool bf) {
    return (1u << 4) | (bf ? ((1u << 7) | (1u << 10)) : 0u) | ((uint32_t)(mt >> 3) << 17) |
           ((uint32_t)(kTileCols >> 4) << 24);
}

// ------------------------------------------------------------------ chunk schedule
// First unit of chunk i (i == nchunks gives the end of the last chunk).  Multiply-and-shift divisions with the
// host's constants: every role's walk starts here, ahead of its first request, and with real divisions (two of
// them 64-bit) this was the larger part of the kernel's code and a good microsecond of every launch.
__device__ __forceinline__ int tile_chunk_begin(const TileParams& p, int i) {
    // balanced: floor(i units / nchunks) = i q + floor(i r / nchunks), units = q nchunks + r  (i r < nchunks^2)
    if (p.split_k == 0) return i * p.bal_q + fast_div(i * p.bal_r, p.div_nchunks);
    const int t = fast_div(i, p.div_split), s = i - t * p.split_k;
    return t * p.G + s * p.slice_base + min(s, p.slice_rem);
}
// Where chunk ci (or the next non-empty one of this CTA, stepping by `stride`) starts.
struct ChunkStart {
    int ci;        // the chunk found (>= nchunks: none left)
    int t;         // tile = batch tile * NT + column tile
    int g0;        // first group inside the tile
    int len;       // units of the chunk
};
__device__ __forceinline__ ChunkStart tile_chunk_start(const TileParams& p, int ci, int stride) {
    ChunkStart c;
    int u0 = 0, len = 0;
    while (ci < p.nchunks) {
        u0 = tile_chunk_begin(p, ci);
        len = tile_chunk_begin(p, ci + 1) - u0;
        if (len > 0) break;
        ci += stride;
    }
    c.ci = ci;
    c.len = len;
    c.t = fast_div(u0, p.div_G);
    c.g0 = u0 - c.t * p.G;
    return c;
}

// Walks the segments of this CTA's chunks in order (a segment = the part of a chunk inside one
// tile).  Every role of the CTA runs its own copy and sees the same sequence.  A warp runs dependent
// scalar code at only one instruction every several clocks, and the producer and MMA warps sit on
// the critical path of every stage: so all per-stage work of the roles is a plain counted loop over
// the segment's 2 * units stages, and the chunk arithmetic happens here, once per chunk.
struct SegWalk {
    const TileParams& p;
    int ci;            // current chunk
    int t;             // tile = batch tile * NT + column tile
    int g0;            // first group of the segment inside the tile
    int units;         // groups in the segment
    int left;          // units of the chunk after this segment
    bool first;        // first segment of its chunk
    uint32_t n0;       // stages of this CTA before the segment (ring positions derive from it)
    __device__ __forceinline__ explicit SegWalk(const TileParams& p_)
        : p(p_), ci((int)blockIdx.x), t(0), g0(0), units(0), left(0), first(true), n0(0) {
        load_chunk();
    }
    __device__ __forceinline__ void load_chunk() {
        const ChunkStart c = tile_chunk_start(p, ci, (int)gridDim.x);
        ci = c.ci;
        if (ci >= p.nchunks) return;
        t = c.t;
        g0 = c.g0;
        units = min(c.len, p.G - g0);
        left = c.len - units;
        first = true;
    }
    __device__ __forceinline__ bool valid() const { return ci < p.nchunks; }
    __device__ __forceinline__ void next() {
        n0 += (uint32_t)(kTileSPU * units);
        if (left == 0) {
            ci += (int)gridDim.x;
            load_chunk();
            return;
        }
        ++t;
        g0 = 0;
        units = min(left, p.G);
        left -= units;
        first = false;
    }
    // (batch tile and column tile: asked once per segment, and two registers fewer than kept)
    __device__ __forceinline__ int mt_i() const { return fast_div(t, p.div_ntiles); }
    __device__ __forceinline__ int nt() const { return t - mt_i() * p.n_tiles; }
    __device__ __forceinline__ int stages_in_seg() const { return kTileSPU * units; }
    __device__ __forceinline__ bool whole_tile() const { return g0 == 0 && units == p.G; }
};

// Position in the ring of R slots: slot = n % R, turn = n / R, phase = turn & 1, kept incrementally.
struct RingPos {
    int slot;
    uint32_t ph;
    uint32_t turn;
    __device__ __forceinline__ void advance(int d, int R) {
        slot += d;
        while (slot >= R) { slot -= R; ph ^= 1u; ++turn; }
    }
};

// "The MMAs that read this slot have retired" has TWO barriers per slot, used by alternate ring turns.
// A parity wait tells a phase from the one before it, not from the one two back, so whoever waits on
// a barrier must see every one of its phases.  The producer does (it walks every stage).  A dequant
// set takes every fourth stage, and with six slots it comes back to a slot only every second turn;
// with one barrier per slot it would skip a phase each time, and nothing but a single in-order issuer
// would keep the skipped phase from still being open.  With one barrier per slot and turn parity the
// set meets the same barrier on every visit and that barrier completes exactly one phase in between.  (The stage in slot s of
// turn t commits to retired[(t & 1) * kTileMaxStages + s]: the issuer steps through them.)
// Until the stage that used r's slot one ring turn earlier has retired (r.turn >= 1)
__device__ __forceinline__ bool wait_slot_free(uint64_t* retired, const RingPos& r) {
    const uint32_t t = r.turn - 1u;
    return mbar_wait(retired + (t & 1u) * kTileMaxStages + r.slot, (t >> 1) & 1u);
}

// Packed words, scales and zero points of one thread's column for one stage of 32 * NW k (NR
// quantization groups).
template <int NW, int NR>
struct StageRegs {
    uint4 w[NW];        // w[i]: k = 32 i .. 32 i + 31 of the stage
    uint32_t s[NR];     // 16-bit scale patterns
    uint32_t zw[NR];    // zero-point words that hold the column's nibble
};

// SG = scale / zero-point rows per 128-k block (quantization group 128 / SG);
// BF = BF16 instead of FP16 activations, scales, weights and output; SYM = symmetric format (zero point 8,
// no Z buffer); EPI = bias / activation fused into the final cast.  (Both compiled in: decided at run time
// they cost 9 % at M = 256.)
template <int SG, bool BF, bool SYM, bool EPI>
__global__ void __launch_bounds__(kTileThreads, 1)
gemm_tile_kernel(const __grid_constant__ CUtensorMap tmap_a, const TileParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment of the stage buffers (the swizzle atom) regardless of where the
    // dynamic segment starts
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int mt = p.mt;
    const int stage_bytes = tile_stage_bytes(mt);
    constexpr int kStageK = kTileStageK;                 // k per ring slot
    constexpr int kSPU = kTileSPU;
    constexpr int kSlotCols = kStageK / 2;               // TMEM columns of one operand slot
    constexpr int kACol = kTileACol;
    constexpr int kNW = kStageK / 32;                    // 16-byte chunks of a thread's column per stage
    constexpr int kPF = kTilePrefetch;
    constexpr int kNR = SG / kSPU > 0 ? SG / kSPU : 1;   // scale rows one stage touches
    constexpr bool sym = SYM;

    uint64_t* full = reinterpret_cast<uint64_t*>(smem);          // [R]  activation box landed AND operand stored in TMEM
    uint64_t* retired = full + kTileMaxStages;                   // [2][R]  the stage's MMAs retired: slot free
    uint64_t* d_full = retired + 2 * kTileMaxStages;             // accumulator complete
    uint64_t* d_empty = d_full + 1;                              // accumulator drained by the epilogue
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(d_empty + 1);
    int* flags = reinterpret_cast<int*>(tmem_slot + 1);          // [0] a bounded wait ran out, [1] stages issued
    unsigned char* stage0 = smem + kTileBarBytes;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = p.stages;

    if (threadIdx.x == 0) {
        for (int i = 0; i < R; ++i) {
            mbar_init(&full[i], 1 + 4);      // the producer's arrive.expect_tx + one arrival per warp of a dequant set
            mbar_init(&retired[i], 1);
            mbar_init(&retired[kTileMaxStages + i], 1);
        }
        mbar_init(d_full, 1);
        mbar_init(d_empty, kTileDequantWarps);
        flags[0] = 0;
        flags[1] = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        // whole tensor memory of the SM: 512 columns (one CTA per SM by shared-memory size)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    volatile int* abort_flag = flags;
    // the next kernel in the stream may start its own prologue and weight prefetch
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------ producer: activation boxes
        if (elect_one()) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_a) : "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");   // activations may come from the previous kernel
        bool ok = true;
        RingPos r{0, 0u, 0u};
        uint32_t n = 0;
        for (SegWalk w(p); w.valid() && ok; w.next()) {
            int kb = w.g0 * (kGroup / kTileBoxK);            // 64-k box index along K
            const int m = w.mt_i() * mt;
            const int nst = w.stages_in_seg();
            for (int j = 0; j < nst; ++j) {
                if (r.turn != 0u && !wait_slot_free(retired, r)) { ok = false; break; }
                if (elect_one()) {
                    mbar_expect_tx(&full[r.slot], (uint32_t)stage_bytes);
                    tma_load_2d(stage0 + r.slot * stage_bytes, &tmap_a, kb * kTileBoxK, m, &full[r.slot]);
                }
                __syncwarp();
                kb += kStageK / kTileBoxK;
                ++n;
                r.advance(1, R);
            }
        }
        if (lane == 0) {
            flags[1] = (int)n;
            if (!ok) *abort_flag = 1;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // What the loop needs of a stage steps by constants and is kept as 32-bit shared addresses, tensor-memory columns and
        // the low word of the box's descriptor: the warp's own scalar code, not the tensor pipe, sets the time of a stage.
        // With barriers as 64-bit pointers and the ring position worked out for each stage the issuer always found its stage
        // ready and took 620 clocks for it with 208 rows and 680 with 256; the MMAs alone take 419 and 514.  us, that form /
        // this one one stage at a time / two at a time: M = 777, K = 4096 / N = 22016 117 / 110 / 109; M = 1024, K = N = 8192
        // 100.1 / 99.0 / 98.7, M = 4096 368 / 368 / 362; M = 300, K = N = 4096 24.8 / 23.2 / 23.5.  Not faster: both stages'
        // waits ahead of the first MMA (112.5 at M = 777), the next stage's barrier tested ahead of this one's MMAs (112.6).
        const uint32_t idesc = tile_idesc(mt, BF);
        const uint32_t full0 = smem_u32(full), full_end = full0 + 8u * R, retired0 = smem_u32(retired);
        const uint32_t d_full_a = smem_u32(d_full), d_empty_a = smem_u32(d_empty);
        const uint64_t box0 = smem_desc_sw128(smem_u32(stage0));
        const uint32_t box_lo0 = (uint32_t)box0, box_hi = (uint32_t)(box0 >> 32), box_step = (uint32_t)stage_bytes >> 4;
        uint32_t bar = full0, ret = retired0, box = box_lo0, a_t = tmem_base + kACol, ph = 0u;
        auto half_unit = [&](uint32_t a, uint32_t b, uint32_t first) {
#pragma unroll
            for (int kk = 0; kk < kStageK / 16; ++kk)            // 16 k: 8 TMEM columns of A, 32 bytes along B's swizzled rows
                tc_mma_ts(tmem_base, a + kk * 8, b + kk * 2, box_hi, idesc, kk == 0 ? first : 1u);
        };
        uint32_t n_seg = 0;
        bool ok = true;
        for (SegWalk w(p); w.valid() && ok; w.next(), ++n_seg) {
            // the epilogue of the segment before must have drained the accumulator
            if (!mbar_wait(d_empty_a, (n_seg & 1u) ^ 1u)) { ok = false; break; }
            uint32_t acc = 0u;                                   // the segment's first MMA overwrites
            for (int left = w.units; left > 0; --left) {
                // Two stages a turn (a unit; the ring has an even number of slots): their MMAs in one go if the second one
                // is there already, as it mostly is.
                if (!mbar_wait(bar, ph)) { ok = false; break; }
                // (by vote: the other warps may complete the barrier between the answers of two lanes)
                const bool both = __all_sync(0xffffffffu, mbar_test(bar + 8u, ph));
                tc_fence_after();
                if (elect_one()) {
                    half_unit(a_t, box, acc);
                    tc_commit(ret);
                    if (both) {
                        half_unit(a_t + kSlotCols, box + box_step, 1u);
                        tc_commit(ret + 8u);
                        if (left == 1) tc_commit(d_full_a);
                    }
                }
                __syncwarp();
                if (!both) {
                    if (!mbar_wait(bar + 8u, ph)) { ok = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        half_unit(a_t + kSlotCols, box + box_step, 1u);
                        tc_commit(ret + 8u);
                        if (left == 1) tc_commit(d_full_a);
                    }
                    __syncwarp();
                }
                acc = 1u;
                bar += 16u;
                ret += 16u;
                box += 2u * box_step;
                a_t += 2u * kSlotCols;
                if (bar == full_end) {                           // next turn (t & 1 = ph): the other set of "retired" barriers
                    ph ^= 1u;
                    bar = full0;
                    ret = retired0 + ph * (8u * kTileMaxStages);
                    box = box_lo0;
                    a_t = tmem_base + kACol;
                }
            }
        }
        if (!ok && lane == 0) *abort_flag = 1;
    } else {
        // ------------------------------------------------------------ dequant + epilogue warps
        const int set = (warp - 2) >> 2;       // takes the stages whose index in this CTA is = set (mod 4)
        const int quarter = warp & 3;          // TMEM lanes this warp may touch
        const int row = quarter * 32 + lane;   // column n inside the CTA tile = TMEM lane
        const int half = row >> 6, col = row & 63;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        // 16-byte index of this thread's two chunks inside a block's 64-k half
        const int wo0 = (col >> 3) * 16 + (col & 7);
        const int wo1 = (col >> 3) * 16 + 8 + (((col & 7) + 4) & 7);
        const int zp = sz_perm(col);         // position of this column's scale / zero point inside a row
        const int zsh = 4 * (zp & 7);

        // this set's first stage inside a segment
        auto first_own = [&](const SegWalk& w) { return (int)(((uint32_t)set - w.n0) & 3u); };
        // Load cursor: runs kPF of this set's stages ahead of the compute loop.  Inside a segment this
        // set's stages are kTileSets apart, so its position steps; it is recomputed only when the cursor enters a new
        // segment.  (One 32-bit position instead of three pointers: the loop runs at the register limit.)
        static_assert(kSPU == 2, "a stage is one 64-k half of a packed block");
        SegWalk wl(p);
        int jl = 0;
        bool l_in = false;                      // this thread's column exists (not past the matrix edge)
        uint32_t hb = 0u;                       // 64-k half block: 2 * packed block + half
        auto point = [&]() {                    // cursor entered a new segment: settle on a stage, set pointers
            while (wl.valid()) {
                jl = first_own(wl);
                if (jl < wl.stages_in_seg()) break;
                wl.next();
            }
            if (!wl.valid()) return;
            const int t64 = 2 * wl.nt() + half;   // 64-column packed tile
            l_in = t64 * kTileN < p.N;
            hb = 2u * (uint32_t)(t64 * p.G + wl.g0) + (uint32_t)jl;
        };
        // load the cursor's stage (zeros past the matrix edge) and advance the cursor
        auto fetch = [&](StageRegs<kNW, kNR>& r) {
            if (!wl.valid()) return;
            if (l_in) {
                const uint4* w = reinterpret_cast<const uint4*>(p.Wq) + (size_t)hb * (kBlockWords / 8);
                r.w[0] = __ldg(w + wo0);
                r.w[1] = __ldg(w + wo1);
                // first scale row of the stage: a 64-k half of a block with SG >= 2 rows starts at row (SG / 2) * half
                const size_t sr = SG >= 2 ? (size_t)hb * (SG / 2) : (size_t)(hb >> 1);
#pragma unroll
                for (int i = 0; i < kNR; ++i) {
                    r.s[i] = __ldg(p.S + (sr + i) * kSBlockHalves + zp);
                    r.zw[i] = sym ? 0u : __ldg(p.Z + (sr + i) * kZBlockWords + (zp >> 3));
                }
            } else {
#pragma unroll
                for (int i = 0; i < kNW; ++i) r.w[i] = make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int i = 0; i < kNR; ++i) { r.s[i] = 0; r.zw[i] = 0; }
            }
            jl += kTileSets;
            if (jl < wl.stages_in_seg()) {
                hb += kTileSets;
            } else {
                wl.next();
                point();
            }
        };
        point();
        // register ring of prefetched stages, written out so that no slot is ever copied
        static_assert(kPF == 2, "the ring below has two slots");
        StageRegs<kNW, kNR> pf0, pf1;
        fetch(pf0);
        fetch(pf1);
        // Converting weights into the TMEM ring touches nothing the previous kernel may still be writing,
        // so it starts at once and runs until the ring is full; the dependency wait comes before this
        // warp's first write to global memory (the first epilogue).
        bool dep_waited = false;

        uint32_t n_seg = 0, n_prev = 0;
        int pi = 0;                             // ring slot that holds the next stage to convert
        RingPos rp{0, 0u, 0u};
        bool ok = true;
        // one stage of this thread's column -> kSlotCols TMEM columns of the ring slot
        auto convert = [&](const StageRegs<kNW, kNR>& cur, uint32_t n) -> bool {
            uint32_t s2[kNR], zlo[kNR], zhi[kNR];
#pragma unroll
            for (int i = 0; i < kNR; ++i) {
                const uint32_t z = sym ? (uint32_t)kSymZero : ((cur.zw[i] >> zsh) & 15u);
                s2[i] = cur.s[i] * 0x00010001u;
                zlo[i] = zconst_lo<BF>(z);
                zhi[i] = zconst_hi<BF>(z);
            }
            // the MMAs that read this slot one ring turn ago must have retired
            if (rp.turn != 0u && !wait_slot_free(retired, rp)) return false;
            tc_fence_after();
            const uint32_t a_t = tmem_base + lane_addr + kACol + rp.slot * kSlotCols;
#pragma unroll
            for (int c = 0; c < kNW; ++c) {      // 32 k -> 16 TMEM columns at a time
                const uint32_t ww[4] = {cur.w[c].x, cur.w[c].y, cur.w[c].z, cur.w[c].w};
                constexpr int kRowDiv = 4 / SG > 0 ? 4 / SG : 1;   // 32-k chunks per scale row (group / 32)
                const int ri = (c / kRowDiv) < kNR ? (c / kRowDiv) : kNR - 1;
                uint32_t regs[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const Pack8 f = dequant_word<BF>(ww[i], zlo[ri], zhi[ri], s2[ri]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) regs[4 * i + q] = f.h[q];
                }
                tc_st16(a_t + 16 * c, regs);
            }
            return true;
        };
        for (SegWalk w(p); w.valid() && ok; w.next(), ++n_seg) {
            const int nst = w.stages_in_seg();
            for (int j = first_own(w); j < nst; j += kTileSets) {
                const uint32_t n = w.n0 + (uint32_t)j;
                rp.advance((int)(n - n_prev), R);
                n_prev = n;
                // convert ring slot pi, then refill it with the stage kPF ahead
                if (pi == 0) { ok = convert(pf0, n); fetch(pf0); pi = 1; }
                else { ok = convert(pf1, n); fetch(pf1); pi = 0; }
                if (!ok) break;
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[rp.slot]);
            }
            if (!ok) break;

            // ---------------------------------------------------- epilogue of this segment
            if (!mbar_wait(d_full, n_seg & 1u)) { ok = false; break; }
            tc_fence_after();
            if (!dep_waited) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                dep_waited = true;
            }
            const int n = w.nt() * kTileCols + row;
            const int m_base = w.mt_i() * mt;
            const uint32_t d_t = tmem_base + lane_addr;
            const bool has_bias = EPI && p.epi.bias != nullptr;
            const float bias = has_bias && n < p.N ? widen<BF>(p.epi.bias[n]) : 0.f;
            const bool whole = w.whole_tile();
            // first segment of a chunk -> slot 2 ci, its continuation into a later tile -> 2 ci + 1
            float* part = p.ws + ((size_t)(2 * w.ci + (w.first ? 0 : 1)) * mt) * kTileCols + row;
            constexpr int kStep = 16;
#pragma unroll 1
            for (int cc = kStep * set; cc < mt; cc += kStep * kTileSets) {      // rows 16 at a time to the sets
                uint32_t v[kStep];
                tc_ld16(d_t + cc, v);
                tc_wait_ld();
                if (whole) {
                    uint16_t c[kStep];
                    finish_column<BF>(v, c, has_bias, bias, EPI ? p.epi.act : kActNone);
                    const int rows = n < p.N ? p.M - (m_base + cc) : 0;
                    uint16_t* dst = p.C + (size_t)(m_base + cc) * p.N + n;
#pragma unroll
                    for (int q = 0; q < kStep; ++q, dst += p.N)
                        if (q < rows) *dst = c[q];
                } else {
#pragma unroll
                    for (int q = 0; q < kStep; ++q) part[(size_t)(cc + q) * kTileCols] = __uint_as_float(v[q]);
                }
            }
            // accumulator drained: a later segment's first MMA may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(d_empty);
        }
        if (!ok && lane == 0) *abort_flag = 1;
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (*abort_flag != 0 && threadIdx.x == 0) {
        // some wait ran out: before the CTA's shared memory goes away, give the copies still in
        // flight a (bounded) chance to land -- the last use of every ring slot.  (The phase may lack
        // the dequant warps' arrivals and then runs into the limit; the wait is bounded either way.)
        const uint32_t issued = (uint32_t)flags[1];
        for (uint32_t back = 0; back < (uint32_t)R && back < issued; ++back) {
            const uint32_t ns = issued - 1 - back;
            mbar_wait(&full[ns % R], (ns / R) & 1u);
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

}  // namespace w4a16
