// tcgen05 kernel for batch tiles of up to 64 or 128 rows (M = 9 to a few hundred; the host chooses by cost): two small CTAs
// per SM, Split-K inside a thread-block cluster.
//
// Same product as kernel_tile.cuh (transposed, C^T = W16^T . A^T, dequantized weights as the 128-row A operand in
// tensor memory, FP32 accumulator in tensor memory).  What bounds these calls is neither HBM nor the tensor pipe
// but serial latency: the start of a launch, the hand-offs of a stage (convert, barrier, issue, MMAs, commit,
// barrier) and the exchange of partial tiles at the end.  Hence
//   - two CTAs per SM, each with half of the tensor memory (256 columns: the accumulator and a ring of operand
//     slots), so that one CTA's hand-offs and epilogue overlap the other's work, and so that the next launch's
//     CTAs find room beside the last ones of this launch (programmatic dependent launch);
//   - packed weights through a shared-memory ring filled by TMA bulk copies, 2 units (2 x 128 k) of the tile's two
//     64-column blocks per stage, six copies by a warp of its own: the eight dequant warps issue no global loads and
//     keep no addresses (21.0 M warp instructions for K = 28672 / N = 8192, the conversion itself is 12 M of them);
//   - ten warps and not eleven, so that 96 registers a thread fit twice on an SM: at 80 the stage loop spends a
//     quarter of its instructions on moving and re-making addresses (39.1 against 33.5 us at M = 32 on that shape);
//   - S slices of a tile's K range as a cluster of S CTAs.  Every CTA finishes 1 / S of the tile's batch rows: it
//     gets the other CTAs' partial sums of those rows through distributed shared memory and adds them in ascending
//     slice order (Algorithm 1, Phase 3), so the exchange is one hop of 1 / S of a tile per pair instead of a
//     workspace round trip, a fence, a ticket and a reload by the last CTA to arrive.
// Measured (us, four-stage ring in registers, one 672-thread CTA per SM and a ticket exchange / this kernel): M = 32:
// K = N = 4096 8.5 / 7.1, K = 11008 / N = 4096 12.9 / 11.0, K = 4096 / N = 22016 22.1 / 18.7, K = 28672 / N = 8192 40.9 / 33.7;
// M = 64: 10.9 / 8.8, 16.5 / 12.4, 26.4 / 21.0, 49.0 / 38.3; K = 4096 / N = 12288 16.2 / 14.2.  A unit takes a CTA 0.42 to
// 0.53 us whether it has the SM to itself or shares it, of which the conversion's own instructions are two thirds.
// Slices that do not fit a cluster (an explicit split_k above kMidMaxCluster) leave FP32 partial tiles in the
// workspace for tile_splitk_reduce_kernel, launched behind this kernel.
//
// Warps: 0-7 dequant and epilogue (set 0 = warps 0-3, set 1 = warps 4-7; warp w owns TMEM lanes 32 (w % 4) .. + 31,
// one column n per lane; set s converts unit s of every weight stage), 8 weight producer, 9 MMA issuer and
// activation copies.  All waits are bounded mbarrier waits.
#pragma once

#include "common.cuh"
#include "kernel_tile.cuh"

namespace w4a16 {

constexpr int kMidDequantWarps = 8;
constexpr int kMidThreads = (kMidDequantWarps + 2) * 32;   // (an eleventh warp would cost the dequant warps 16 registers)
constexpr int kMidWUnits = 2;              // units (128 k) of a weight stage: one per dequant set
constexpr int kMidTmemCols = 256;          // half of the SM's tensor memory
constexpr int kMidMaxWStages = 4;
constexpr int kMidMaxCluster = 8;          // largest cluster every device places
constexpr int kMidBarBytes = 256;
// Batch rows of a CTA tile are a run-time multiple of 16 up to MTC; an operand slot holds stage_k of the unit.
__host__ __device__ constexpr int mid_stage_k(int mtc) { return mtc <= 64 ? 128 : 64; }
__host__ __device__ constexpr int mid_slots(int mtc) { return (kMidTmemCols - mtc) / (mid_stage_k(mtc) / 2); }
__host__ __device__ constexpr int mid_wdata_bytes(int sg) {
    return 2 * kMidWUnits * (kBlockBytes + sg * kSBlockHalves * 2 + sg * kZBlockWords * 4);
}
__host__ __device__ constexpr int mid_wstage_bytes(int sg) {
    // (data, then the stage's two barriers: their addresses are the stage's plus a constant)
    return mid_wdata_bytes(sg) + 128;
}
// Partial sums a CTA of a cluster of S receives: S - 1 slots of its share of the rows, in groups of four rows.
__host__ __device__ inline int mid_xch_slot_bytes(int mt, int S) { return (mt / 4 + S - 1) / S * (kTileCols * 16); }
// Up to 64 rows they have a buffer of their own; above, they lie on top of the (by then idle) rings.
inline int mid_xch_bytes(int mtc, int mt, int S) { return mtc <= 64 && S > 1 ? (S - 1) * mid_xch_slot_bytes(mt, S) : 0; }
inline int mid_smem_bytes(int mtc, int mt, int sg, int wstages, int cluster) {
    return 1024 + mid_slots(mtc) * mt * mid_stage_k(mtc) * 2 + wstages * mid_wstage_bytes(sg) + mid_xch_bytes(mtc, mt, cluster) +
           kMidBarBytes;
}

struct MidParams {
    const uint32_t* Wq;
    const uint16_t* S;
    const uint32_t* Z;   // nullptr: symmetric format, zero point 8
    uint16_t* C;
    float* ws;           // deferred reduce: partial tiles [2 * chunk][mt][128] FP32
    int M, N, K, G;
    int n_tiles;         // ceil(N / 128)
    int mt;              // batch rows of a tile: multiple of 16
    int split_k;         // slices per tile
    int nchunks;         // tiles * split_k
    int wstages;         // weight ring
    int cluster;         // 1: the slices of a tile are one cluster and every CTA has one chunk
    FastDiv div_split, div_ntiles;
    int slice_base, slice_rem;   // G / split_k, G % split_k
    Epilogue epi;
};

// Chunk ci = slice ci % S of tile ci / S.
struct MidChunk {
    int nt, mt_i, g0, units, slice, T;
    __device__ __forceinline__ MidChunk(const MidParams& p, int ci) {
        T = fast_div(ci, p.div_split);
        slice = ci - T * p.split_k;
        mt_i = fast_div(T, p.div_ntiles);
        nt = T - mt_i * p.n_tiles;
        g0 = slice * p.slice_base + min(slice, p.slice_rem);
        units = p.slice_base + (slice < p.slice_rem ? 1 : 0);
    }
};

template <int MTC, int SG, bool BF, bool SYM>
__global__ void __launch_bounds__(kMidThreads, 2)
gemm_mid_kernel(const __grid_constant__ CUtensorMap tmap_a, const MidParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // (the swizzle atom of the activation boxes wants 1024-byte alignment)
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int kStageK = mid_stage_k(MTC);
    constexpr int kSPU = kGroup / kStageK;            // operand slots per unit
    constexpr int R = mid_slots(MTC);
    // A set does not visit every ring turn of a slot (three slots, two sets; odd segments), so its wait for "retired" may
    // skip a phase, and a parity wait cannot tell a phase from the one two turns back.  That one is over all the same: the
    // one issuer's commits complete in order, the set's stage before this one (at most kSPU + 1 stages back) has waited for
    // that commit or a later one, and earlier segments' commits are behind the epilogue's wait for d_full.
    static_assert(R >= kSPU + 1, "a slot's retired barrier");
    constexpr int kSlotCols = kStageK / 2;
    constexpr bool kOverlay = MTC > 64;               // exchange buffer on top of the rings
    constexpr int kWStage = mid_wstage_bytes(SG);
    constexpr int kWS = 2 * kMidWUnits * kBlockBytes;                       // scale rows of a weight stage
    constexpr int kWZ = kWS + 2 * kMidWUnits * SG * kSBlockHalves * 2;      // zero-point rows
    const int mt = p.mt;
    const int abytes = mt * kStageK * 2;              // activation slot

    // All shared memory by 32-bit address: [activation slots][weight stages, each with its barriers][exchange][barriers]
    constexpr uint32_t kWFull = (uint32_t)mid_wdata_bytes(SG), kWEmpty = kWFull + 8u;   // inside a weight stage
    const uint32_t act0 = smem_u32(smem);
    const uint32_t w0 = act0 + (uint32_t)(R * abytes);
    const uint32_t w_end = (uint32_t)(p.wstages * kWStage);                 // ring size in bytes
    const uint32_t xch = kOverlay ? act0 : w0 + w_end;
    const int xslot = mid_xch_slot_bytes(mt, p.split_k);
    // slot i: full (activation box landed, operand stored) at bars + 16 i, retired (the MMAs that read it) 8 further
    const uint32_t bars = w0 + w_end + (uint32_t)(!kOverlay && p.cluster ? (p.split_k - 1) * xslot : 0);
    const uint32_t d_full = bars + 16u * R, d_empty = d_full + 8u, xbar = d_full + 16u;   // xbar: the other slices' sums have landed
    unsigned char* misc = smem + (bars - act0) + 16 * R + 24;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc);
    volatile int* flags = reinterpret_cast<int*>(misc + 4);   // [0] a wait ran out, [1] slots, [2] weight stages requested

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < R; ++i) {
            mbar_init(bars + 16u * i, 1 + 4);         // activation copy + the four warps of a dequant set
            mbar_init(bars + 16u * i + 8u, 1);
        }
        for (int i = 0; i < p.wstages; ++i) {
            mbar_init(w0 + i * kWStage + kWFull, 1);
            mbar_init(w0 + i * kWStage + kWEmpty, kMidDequantWarps);
        }
        mbar_init(d_full, 1);
        mbar_init(d_empty, kMidDequantWarps);
        mbar_init(xbar, (uint32_t)((p.split_k - 1) * kMidDequantWarps > 0 ? (p.split_k - 1) * kMidDequantWarps : 1));
        flags[0] = 0;
        flags[1] = 0;
        flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == kMidDequantWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // Every CTA of a cluster must be running, its barriers initialised, before anyone writes to its shared memory: all
    // threads arrive here and each waits once, later, where the guarantee is needed.
    // (With the exchange on top of the rings the guarantee needed is that every CTA has done with its rings: they arrive
    // when they have.)
    bool cl_arrived = p.cluster == 0, cl_waited = p.cluster == 0;
    if (!kOverlay && p.cluster) {
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        cl_arrived = true;
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == kMidDequantWarps) {
        // ------------------------------------------------------------ weight producer (one thread)
        if (lane == 0) {
            int n = 0;
            uint32_t woff = 0u, ph = 0u;
            bool ok = true;
            for (int ci = blockIdx.x; ci < p.nchunks && ok; ci += gridDim.x) {
                const MidChunk c(p, ci);
                const int t64 = 2 * c.nt;
                const int halves = (t64 + 1) * kTileN < p.N ? 2 : 1;      // 64-column blocks this tile really has
                size_t blk = (size_t)t64 * p.G + c.g0;
                for (int left = c.units; left > 0; left -= kMidWUnits, blk += kMidWUnits, ++n) {
                    const uint32_t st = w0 + woff;
                    if (n >= p.wstages && !mbar_wait_inline(st + kWEmpty, ph ^ 1u)) { ok = false; break; }
                    const int gc = min(left, kMidWUnits);
                    mbar_expect_tx(st + kWFull, (uint32_t)(halves * gc * (kBlockBytes + SG * kSBlockHalves * 2 + (SYM ? 0 : SG * kZBlockWords * 4))));
                    for (int h = 0; h < halves; ++h) {
                        const size_t b = blk + (size_t)h * p.G;
                        bulk_g2s(st + h * (kMidWUnits * kBlockBytes), p.Wq + b * kBlockWords, (uint32_t)(gc * kBlockBytes), st + kWFull);
                        bulk_g2s(st + kWS + h * (kMidWUnits * SG * kSBlockHalves * 2), p.S + b * (SG * kSBlockHalves),
                                 (uint32_t)(gc * SG * kSBlockHalves * 2), st + kWFull);
                        if (!SYM)
                            bulk_g2s(st + kWZ + h * (kMidWUnits * SG * kZBlockWords * 4), p.Z + b * (SG * kZBlockWords),
                                     (uint32_t)(gc * SG * kZBlockWords * 4), st + kWFull);
                    }
                    woff += kWStage;
                    if (woff == w_end) { woff = 0u; ph ^= 1u; }
                }
            }
            flags[2] = n;
            if (!ok) flags[0] = 1;
        }
        __syncwarp();
    } else if (warp == kMidDequantWarps + 1) {
        // ------------------------------------------------------------ MMA issuer and activation copies (warp-uniform,
        // one elected lane).  The copy for a slot goes out behind the MMAs of the stage after the one that frees it:
        // by then that one has retired, so the wait for it costs nothing, and the copy is R - 1 stages ahead of its use.
        bool ok = true;
        int a_ci = blockIdx.x, a_left = 0, a_kb = 0, a_m = 0, a_slot = 0, a_n = 0;
        auto next_act = [&]() {
            if (a_left == 0) {
                if (a_ci >= p.nchunks) return;
                const MidChunk c(p, a_ci);
                a_ci += gridDim.x;
                a_m = c.mt_i * mt;
                a_kb = c.g0 * (kGroup / kTileBoxK);
                a_left = c.units * kSPU;
            }
            if (elect_one()) {
                const uint32_t bar = bars + 16u * a_slot;
                mbar_expect_tx(bar, (uint32_t)abytes);
                if constexpr (kStageK == kTileBoxK) tma_load_2d(act0 + a_slot * abytes, &tmap_a, a_kb * kTileBoxK, a_m, bar);
                else tma_load_3d(act0 + a_slot * abytes, &tmap_a, 0, a_m, a_kb, bar);
            }
            __syncwarp();
            a_kb += kStageK / kTileBoxK;
            --a_left;
            ++a_n;
            if (++a_slot == R) a_slot = 0;
        };
        if (elect_one()) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_a) : "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");       // activations may come from the previous kernel
        for (int i = 0; i < R; ++i) next_act();
        int slot = 0;
        uint32_t ph = 0u, seg = 0;
        uint32_t prev = 0u, prev_ph = 0u;                        // barrier of the stage before this one (0: none yet)
        const uint32_t idesc = tile_idesc(mt, BF);
        const uint32_t box_step = (uint32_t)(mt * 128 / 16);     // the next 64-k box, in descriptor units
        for (int ci = blockIdx.x; ci < p.nchunks && ok; ci += gridDim.x, ++seg) {
            const MidChunk c(p, ci);
            if (seg != 0 && !mbar_wait_inline(d_empty, (seg - 1u) & 1u)) { ok = false; break; }
            tc_fence_after();
            const int nst = c.units * kSPU;
            for (int j = 0; j < nst; ++j) {
                const uint32_t bar = bars + 16u * slot;
                if (!mbar_wait_inline(bar, ph)) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t bdesc = smem_desc_sw128(act0 + (uint32_t)(slot * abytes));
                    const uint32_t a_t = tmem_base + MTC + slot * kSlotCols;
#pragma unroll
                    for (int kk = 0; kk < kStageK / 16; ++kk) {
                        const uint64_t bd = bdesc + (uint64_t)((uint32_t)(kk / 4) * box_step + (kk % 4) * 2);
                        tc_mma_ts(tmem_base, a_t + kk * 8, bd, idesc, (kk == 0 && j == 0) ? 0u : 1u);
                    }
                    tc_commit(bar + 8u);
                    if (j + 1 == nst) tc_commit(d_full);
                }
                __syncwarp();
                if (prev != 0u) {
                    if (!mbar_wait_inline(prev + 8u, prev_ph)) { ok = false; break; }
                    next_act();
                }
                prev = bar;
                prev_ph = ph;
                if (++slot == R) { slot = 0; ph ^= 1u; }
            }
        }
        if (lane == 0) {
            flags[1] = a_n;
            if (!ok) flags[0] = 1;
        }
    } else {
        // ------------------------------------------------------------ dequant + epilogue warps
        const int set = warp >> 2;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;   // column n inside the tile = TMEM lane
        const int half = row >> 6, col = row & 63;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        // byte offsets of this thread's column inside a weight stage (unit `set` of it)
        const uint32_t w_a = w0 + (uint32_t)(half * (kMidWUnits * kBlockBytes) + set * kBlockBytes + (col >> 3) * 256);
        const uint32_t w_a0 = w_a + (uint32_t)((col & 7) * 16), w_a1 = w_a + 128u + (uint32_t)((((col & 7) + 4) & 7) * 16);
        const int zp = sz_perm(col);
        const uint32_t zsh = (uint32_t)(4 * (zp & 7));
        const uint32_t s_a = w0 + (uint32_t)(kWS + half * (kMidWUnits * SG * 128) + set * (SG * 128) + zp * 2);
        const uint32_t z_a = w0 + (uint32_t)(kWZ + half * (kMidWUnits * SG * 32) + set * (SG * 32) + (zp >> 3) * 4);
        const uint32_t a_t0 = tmem_base + lane_addr + MTC;

        int n0 = 0;                            // operand slots before the segment
        uint32_t woff = 0u, wph = 0u, seg = 0;
        bool ok = true, dep_waited = false;
        for (int ci = blockIdx.x; ci < p.nchunks && ok; ci += gridDim.x, ++seg) {
            const MidChunk c(p, ci);
            // this set's first operand slot and the ring turn it is used in
            int slot = (n0 + set * kSPU) % R;
            uint32_t turn = (uint32_t)((n0 + set * kSPU) / R);
            for (int own = (c.units + 1 - set) / kMidWUnits; own > 0; --own) {
                if (!mbar_wait(w0 + woff + kWFull, wph)) { ok = false; break; }
                uint4 w[4];
                uint32_t s[SG], zw[SG];
                w[0] = lds128<0>(w_a0 + woff);
                w[1] = lds128<0>(w_a1 + woff);
                w[2] = lds128<2048>(w_a0 + woff);
                w[3] = lds128<2048>(w_a1 + woff);
#pragma unroll
                for (int i = 0; i < SG; ++i) {
                    asm volatile("{\n\t.reg .b16 t;\n\tld.shared.u16 t, [%1];\n\tcvt.u32.u16 %0, t;\n\t}"
                                 : "=r"(s[i]) : "r"(s_a + woff + i * 128) : "memory");
                    if (SYM) zw[i] = 0;
                    else asm volatile("ld.shared.u32 %0, [%1];" : "=r"(zw[i]) : "r"(z_a + woff + i * 32) : "memory");
                }
                __syncwarp();
                mbar_arrive_lane0(w0 + woff + kWEmpty, lane);
                woff += kWStage;
                if (woff == w_end) { woff = 0u; wph ^= 1u; }
                uint32_t s2[SG], zlo[SG], zhi[SG];
#pragma unroll
                for (int i = 0; i < SG; ++i) {
                    const uint32_t z = SYM ? (uint32_t)kSymZero : ((zw[i] >> zsh) & 15u);
                    s2[i] = s[i] * 0x00010001u;
                    zlo[i] = zconst_lo<BF>(z);
                    zhi[i] = zconst_hi<BF>(z);
                }
#pragma unroll
                for (int h = 0; h < kSPU; ++h) {
                    // the MMAs that read this slot one ring turn ago must have retired
                    const uint32_t bar = bars + 16u * slot;
                    if (turn != 0u && !mbar_wait(bar + 8u, (turn - 1u) & 1u)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a_t = a_t0 + slot * kSlotCols;
#pragma unroll
                    for (int cc = 0; cc < kStageK / 32; ++cc) {
                        const int q = h * (kStageK / 32) + cc;             // 32-k chunk of the unit
                        const int ri = q * SG / 4;                        // its scale row
                        const uint32_t ww[4] = {w[q].x, w[q].y, w[q].z, w[q].w};
                        uint32_t regs[16];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const Pack8 f = dequant_word<BF>(ww[i], zlo[ri], zhi[ri], s2[ri]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) regs[4 * i + e] = f.h[e];
                        }
                        tc_st16(a_t + 16 * cc, regs);
                    }
                    tc_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0(bar, lane);
                    slot += (h + 1 < kSPU) ? 1 : kSPU * (kMidWUnits - 1) + 1;
                    if (slot >= R) { slot -= R; ++turn; }
                }
                if (!ok) break;
            }
            if (!ok) break;
            if (set == 1 && (c.units & 1)) {       // the last stage holds set 0's unit only
                if (!mbar_wait(w0 + woff + kWFull, wph)) { ok = false; break; }
                mbar_arrive_lane0(w0 + woff + kWEmpty, lane);
                woff += kWStage;
                if (woff == w_end) { woff = 0u; wph ^= 1u; }
            }
            n0 += c.units * kSPU;

            // ---------------------------------------------------- epilogue of this segment
            if (!mbar_wait(d_full, seg & 1u)) { ok = false; break; }
            tc_fence_after();
            if (!dep_waited) {
                asm volatile("griddepcontrol.wait;" ::: "memory");   // C and the workspace may still be in use
                dep_waited = true;
            }
            const int n = c.nt * kTileCols + row;
            const int m_base = c.mt_i * mt;
            const uint32_t d_t = tmem_base + lane_addr;
            const bool has_bias = p.epi.bias != nullptr;
            const float bias = has_bias && n < p.N ? widen<BF>(p.epi.bias[n]) : 0.f;
            if (!p.cluster) {
                float* part = p.ws + ((size_t)(2 * ci) * mt) * kTileCols + row;
#pragma unroll 1
                for (int c0 = 16 * set; c0 < mt; c0 += 32) {
                    uint32_t v[16];
                    tc_ld16(d_t + c0, v);
                    tc_wait_ld();
                    if (p.split_k == 1) {
                        uint16_t y[16];
                        finish_column<BF>(v, y, has_bias, bias, p.epi.act);
                        const int rows = n < p.N ? p.M - (m_base + c0) : 0;
                        uint16_t* dst = p.C + (size_t)(m_base + c0) * p.N + n;
#pragma unroll
                        for (int q = 0; q < 16; ++q, dst += p.N)
                            if (q < rows) *dst = y[q];
                    } else {
#pragma unroll
                        for (int q = 0; q < 16; ++q) part[(size_t)(c0 + q) * kTileCols] = __uint_as_float(v[q]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                mbar_arrive_lane0(d_empty, lane);
                continue;
            }
            // Cluster: rows 4 q .. 4 q + 3 are finished by CTA owner(q); quads = mt / 4 in S equal runs (the last may
            // be shorter).  Slot of slice s at CTA d: s - (s > d).
            if (kOverlay) {
                asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
                cl_arrived = true;
            }
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            cl_waited = true;
            const int S = p.split_k, rank = c.slice;
            const int per = (mt / 4 + S - 1) / S;
#pragma unroll 1
            for (int c0 = 16 * set; c0 < mt; c0 += 32) {
                uint32_t v[16];
                tc_ld16(d_t + c0, v);
                tc_wait_ld();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int q = c0 / 4 + k;
                    int d = 0;
                    while ((d + 1) * per <= q) ++d;
                    if (d == rank) continue;
                    const uint32_t local = xch + (uint32_t)((rank - (rank > d ? 1 : 0)) * xslot + ((q - d * per) * kTileCols + row) * 16);
                    uint32_t remote;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(d));
                    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(remote), "r"(v[4 * k]), "r"(v[4 * k + 1]),
                                 "r"(v[4 * k + 2]), "r"(v[4 * k + 3])
                                 : "memory");
                }
            }
            __syncwarp();
            if (lane < S && lane != rank) {
                uint32_t remote;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(xbar), "r"(lane));
                asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
            }
            __syncwarp();
            if (!mbar_wait_cluster(xbar, 0u)) { ok = false; break; }
            const int q_end = min((rank + 1) * per, mt / 4);
#pragma unroll 1
            for (int q = rank * per + set; q < q_end; q += 2) {
                uint32_t own[4];
                tc_ld4(d_t + 4 * q, own);
                tc_wait_ld();
                float4 acc;
                const uint32_t src = xch + (uint32_t)(((q - rank * per) * kTileCols + row) * 16);
                for (int s = 0; s < S; ++s) {
                    uint4 x = make_uint4(own[0], own[1], own[2], own[3]);
                    if (s != rank) x = lds128<0>(src + (uint32_t)((s - (s > rank ? 1 : 0)) * xslot));
                    if (s == 0) {
                        acc = make_float4(__uint_as_float(x.x), __uint_as_float(x.y), __uint_as_float(x.z), __uint_as_float(x.w));
                    } else {
                        acc.x += __uint_as_float(x.x); acc.y += __uint_as_float(x.y);
                        acc.z += __uint_as_float(x.z); acc.w += __uint_as_float(x.w);
                    }
                }
                const uint32_t a[4] = {__float_as_uint(acc.x), __float_as_uint(acc.y), __float_as_uint(acc.z), __float_as_uint(acc.w)};
                uint16_t y[4];
                finish_column<BF>(a, y, has_bias, bias, p.epi.act);
                const int rows = n < p.N ? p.M - (m_base + 4 * q) : 0;
                uint16_t* dst = p.C + (size_t)(m_base + 4 * q) * p.N + n;
#pragma unroll
                for (int e = 0; e < 4; ++e, dst += p.N)
                    if (e < rows) *dst = y[e];
            }
        }
        if (!ok && lane == 0) flags[0] = 1;
    }
    __syncwarp();
    if (!cl_arrived) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (!cl_waited) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (flags[0] != 0) {
        // some wait ran out: before the CTA's shared memory goes away, give the copies still in flight a (bounded)
        // chance to land, and stay until the other CTAs of the cluster have left too (each of their waits is bounded)
        if (threadIdx.x == 0) {
            for (int b = 0; b < R && b < flags[1]; ++b) {
                const int ns = flags[1] - 1 - b;
                mbar_wait(bars + 16u * (ns % R), (uint32_t)(ns / R) & 1u);
            }
            for (int b = 0; b < p.wstages && b < flags[2]; ++b) {
                const int ns = flags[2] - 1 - b;
                mbar_wait(w0 + (ns % p.wstages) * kWStage + kWFull, (uint32_t)(ns / p.wstages) & 1u);
            }
        }
        __syncthreads();
        if (p.cluster) {
            asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        }
    }
    if (warp == kMidDequantWarps + 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem_base) : "memory");
    }
}

}  // namespace w4a16
