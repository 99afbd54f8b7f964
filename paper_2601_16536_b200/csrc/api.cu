// C ABI of the library (declared in include/w4a16.h): argument validation, per-shape
// kernel and Split-K selection, launches.  Every step of the computation runs in the
// kernels included below; this file only marshals arguments.
#include "w4a16.h"

#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>
#include <string.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels_basic.cuh"
#include "kernel_tables.h"
#include "pack_order.cuh"

using namespace w4a16;

namespace {

constexpr int kMaxDevices = 64;
constexpr size_t kWsHeaderBytes = 16384;  // zeroed ticket counters ahead of the FP32 partials
constexpr long kMaxTickets = kWsHeaderBytes / sizeof(int);

struct DeviceState {
    bool probed = false;
    bool is_sm100 = false;
    int sm_count = 148;
    int max_smem_optin = 0;
    void* ws = nullptr;
    size_t ws_bytes = 0;
    bool decode_attr_set[3][2][3][2][2][2] = {};   // [mb][cluster exchange][log2 SG][bf16][symmetric][tensor-copy rows]
    int mid_clusters[16] = {};         // mid_max_clusters, 0 = not asked yet
    bool mid_attr_set[2][3][2][2] = {};   // [64 / 128 rows][log2 SG][bf16][symmetric]
    bool tile_attr_set[3][2][2][2] = {};   // [log2 SG][bf16][symmetric][epilogue]
    PackOrder order;          // which GEMM launches may overlap the kernel in front of them
    bool cluster_ok = true;   // cleared when a cluster launch is refused (fewer SMs than usual, MPS limits ...)
};
DeviceState g_dev[kMaxDevices];
// One lock for the per-device records above (workspace registration, attribute flags, stream table):
// the entry points may be called from several host threads.
std::mutex g_mu;

int current_device(DeviceState** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    DeviceState& d = g_dev[dev];
    if (!d.probed) {
        int major = 0, sms = 0, smem = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
            cudaGetLastError();
            return W4A16_ERR_CUDA;
        }
        d.is_sm100 = (major == 10);
        d.sm_count = sms > 0 ? sms : 148;
        d.max_smem_optin = smem;
        d.probed = true;
    }
    *out = &d;
    return W4A16_OK;
}

// The capture that `st` is in; 0 = none.
unsigned long long capture_of(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) {
        cudaGetLastError();    // (the default stream while another one is captured: the launch will be refused)
        return ~0ull;
    }
    return status == cudaStreamCaptureStatusNone ? 0 : id;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_weight_shape(int N, int K, int group) {
    if (!group_ok(group)) return W4A16_ERR_SHAPE;
    if (K <= 0 || N <= 0 || K % kGroup != 0 || N % kTileN != 0) return W4A16_ERR_SHAPE;
    return W4A16_OK;
}
int log2_sg(int sg) { return sg == 1 ? 0 : sg == 2 ? 1 : 2; }
bool flags_ok(int flags) { return (flags & ~(W4A16_FLAG_SYMMETRIC | W4A16_FLAG_BF16)) == 0; }

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// What the schedules are planned for.  Made once per call and passed on: asking for the device costs 30 ns each time.
struct Chip {
    int sms;
    bool clusters;               // a launch with clusters has not been refused
    const int* max_clusters;     // [size]: clusters of two-per-SM CTAs that run at the same time
};
const int* mid_max_clusters(DeviceState* d);
Chip chip_of(DeviceState* d) { return {d->sm_count, d->cluster_ok, mid_max_clusters(d)}; }
// For the size and schedule queries, which also answer on a host without a device.
Chip chip_or_default() {
    DeviceState* d = nullptr;
    if (current_device(&d) == W4A16_OK) return chip_of(d);
    return {148, true, mid_max_clusters(nullptr)};
}
Chip without_clusters(Chip chip) { chip.clusters = false; return chip; }

// f(2), f(3) ... with the sizes as constants.
template <int kFrom, int kTo, typename F>
void for_each_size(const F& f) {
    if constexpr (kFrom <= kTo) {
        f(std::integral_constant<int, kFrom>{});
        for_each_size<kFrom + 1, kTo>(f);
    }
}

// ---- decode-path launch geometry ------------------------------------------------
int decode_mb(int M) { return M <= 8 ? 1 : 2; }

// The decode kernel is persistent: `ctas` CTAs per batch chunk (9 warps, about 100 KiB of shared
// memory), `nchunks` chunks of work units dealt to them.  Two CTAs per SM: three, with a two-stage ring
// and 72 registers, are behind everywhere but at K = 4096 / N = 12288, by 3 % (33.8 against 34.8 us at
// K = 28672 / N = 8192, 15.0 against 15.8 at N = 22016).
constexpr int kDecCtasPerSm = 2;
struct DecodeGeom {
    int mb, mchunks, stages, smem_bytes, ctas, nchunks;
    int stage_bytes;   // ring stride for the batch rows a CTA has
    int prefetch;      // stages whose weights are requested before the wait for the previous kernel
    bool a_box;        // activation rows of a stage as one tensor copy (kernel_decode.cuh)
    long cost;     // ns by the cost model (automatic schedules)
    bool cluster;  // one thread-block cluster of split_k CTAs per tile: partial tiles meet in shared memory
    int split_k;   // what the kernel runs: 0 = balanced chunks, S >= 1 = S slices per tile
};

// From how many batch rows per CTA on a stage's activation rows come as one tensor copy instead of one bulk
// copy per row.  Measured (us, bulk copies per row / one tensor copy), K = 11008 / N = 4096: M = 2 9.28 / 9.09,
// M = 4 9.60 / 9.09, M = 8 10.5 / 9.34, M = 16 13.0 / 11.1; K = 4096 / N = 4096, M = 3: 5.57 / 5.38.  With one
// row the two are within 1 % (9.15 / 9.09 there, 32.6 / 32.8 at K = 28672 / N = 8192, 14.9 / 15.2 at K = 4096 /
// N = 22016: the box takes 8 KiB of a slot whatever M is, and long shapes want the ring stage that costs).
constexpr int kDecABoxMinRows = 2;

DecodeGeom decode_geom(int M, int N, int G, int split_k, const Chip& chip, int sg) {
    DecodeGeom g;
    g.mb = decode_mb(M);
    g.mchunks = (M + 8 * g.mb - 1) / (8 * g.mb);
    const int T = N / kTileN;
    const long units = (long)T * G;
    const bool allow_cluster = chip.clusters;
    const long slots = (long)kDecCtasPerSm * chip.sms;
    g.cost = 0;
    if (split_k == 0) {
        // How the unit range is cut when the caller leaves it open.  Balanced chunks use every CTA slot, but a chunk that
        // crosses a tile boundary goes through the workspace exchange in mid-stream.  S slices per tile keep every chunk
        // inside one tile, and their exchange is cheaper: none at S = 1, through the cluster for S <= 6 (if that many
        // clusters run at once: a second wave doubles the time), through the workspace at the end of the stream otherwise.
        // Costs in ns: a unit takes a CTA 288 with 8 rows and 330 with 16 (two CTAs on some SM set the pace whatever the
        // count: 64 units of 134 whole tiles 17.8 us, of 160 18.6), the rest is what a launch shows beside its units; 500
        // more with nine tenths of the slots taken, because then the next launch cannot start before this one ends; 80 per four
        // rows for every chunk of a tile that the last one to arrive adds (16 rows, four tiles of K = 7296 in 8 / 16 / 24 / 57
        // slices: 7.9 / 9.8 / 13.5 / 23.6 us, six in a cluster 5.0).
        // us, measured: K = 8192 / N = 8576 two slices 11.3, whole tiles 17.8, balanced 14.9; N = 10240 (320 slices do not
        // fit) balanced 16.5, whole 18.6; K = 4096 / N = 12288 whole 10.2, balanced 12.1; K = 11008 / N = 4096 four slices
        // 8.6, three 10.5; K = 23168 / N = 4416 four 15.0, three 18.0; K = 6144 / N = 1536 six in a cluster 4.3, twelve
        // through the workspace 6.5; K = 28672 / N = 8192 two 31.2, balanced 32.4; K = 4096 / N = 22016 (344 whole tiles on
        // 296 CTAs, whose pairs share the SM's issue slots: 15 % over the mean, with 16 rows 30) 14.4, balanced 18.4.
        const long unit_ns = g.mb == 1 ? 288 : 330, wide = g.mb == 1 ? 0 : 700, add_ns = ((M < 8 * g.mb ? M : 8 * g.mb) + 3) / 4 * 80;
        const int* max_clusters = chip.max_clusters;
        auto take = [&](int s, long cost) {
            if (g.cost == 0 || cost < g.cost) { g.cost = cost; split_k = s; }
        };
        // (several batch chunks, which only a forced path has, fill the SMs as few rows do)
        const bool few = g.mb == 1 || g.mchunks > 1;
        if (T > slots) take(1, few ? 1500 + wide + unit_ns * ((units * 23 / 20 + slots - 1) / slots) : 4000 + unit_ns * units * 13 / (10 * slots));
        else take(1, 1500 + wide + unit_ns * G);
        if (allow_cluster && g.mchunks == 1) {
            // The last clusters that fit find a place late, while the launch in front still holds its SMs: from 7/8 or 8/9 of them
            // on with 5 or 3 CTAs (us, M = 8, K = 7296: 48 / 49 / 50 / 52 tiles in five 5.8 / 6.2 / 8.5 / 9.2, in four 6.7; 82 / 84 /
            // 86 / 90 in three 8.1 / 8.6 / 11.5 / 12.8, in two 9.8), a few tiles before the end with 4 and 6 (K = 2048: 66 / 68 /
            // 69 / 70 in four 4.0 / 4.4 / 4.9 / 5.1, in two 4.2; 41 / 42 / 43 / 44 in six 3.8 / 4.0 / 4.4 / 4.8, in five 3.5), not
            // with 2.  A long launch hardly notices (K = 28672: 50 in five 14.9; K = 10880: 42 in six 7.0, in five 7.7).  Of equal
            // slices the even count is ahead (20 tiles of K = 3200, M = 16: 4.4 in six, 4.9 in five).
            for_each_size<2, kDecMaxCluster>([&](auto size) {
                constexpr int s = decltype(size)::value;
                const int room = max_clusters[s];
                // Every place for pairs (us, M = 4, 147 tiles: K = 2048 5.0, whole tiles 6.1; K = 7168 10.3, balanced 14.4; K = 14336
                // 17.5 and 21.5; 148: 10.3 and 12.4, but one whole tile per SM 4.95 to 5.0 at K = 2048, M = 16 5.9 to 6.2).  Of the
                // larger ones the last two cost the time below and more (M = 4, K = 7168: 72 in four 10.7, in three 8.0).
                if (s > G || T + (s > 2 ? 2 : G < 24 ? 1 : 0) > room) return;
                const int u = (G + s - 1) / s, ctas = T * s;
                long wait = 0;
                if (s == 3 || s == 5) {
                    const int over = s == 3 ? T - room * 8 / 9 : T - room * 7 / 8;
                    if (over >= 0 && s == 5) wait = over == 0 ? 800 - 40 * u : 2000L * over;
                    if (over >= (g.mb == 1 ? 0 : -1) && s == 3) wait = g.mb == 1 ? 960L * over - 450 : 1500L * (over + 2);   // (M = 16, K = 4096: 80 tiles 6.9, 82 9.8)
                    if (wait > 5000 - 60 * u) wait = 5000 - 60 * u;
                    if (10 * ctas > 9 * slots && wait < 3500) wait = 3500;
                } else if (s == 4 || s == 6) {
                    const int over = T + 4 - room;
                    if (over > 0) wait = s == 4 ? 500 * over - 15 * u : 700 * over - 45 * u;
                }
                if (wait < 0) wait = 0;
                take(s, (s == 2 ? 1700 : 2150) + (s % 2 != 0 && u > 3 ? 150 : 0) + wide * 7 / 4 + unit_ns * u + (10 * ctas > 9 * slots ? 500 : 0) + wait);
            });
        }
        const int s0 = (int)(slots * 7 / 8 / T < G ? slots * 7 / 8 / T : G);
        if (s0 > kDecMaxCluster || (s0 >= 2 && !(allow_cluster && g.mchunks == 1)))
            take(s0, 4000 + wide + add_ns * s0 + unit_ns * ((G + s0 - 1) / s0));
        const long share = slots / T > 3 ? slots / T - 3 : 0;      // (contributors of a tile, beyond what the constant holds)
        take(0, (g.mb == 1 ? 5700 : 7500) + add_ns * share + unit_ns * ((units * 27 / 25 + slots - 1) / slots));
    }
    g.split_k = split_k;
    if (split_k == 0) {
        // balanced chunks, one per CTA; no more CTAs than stages' worth of units
        long want = (units + kDecUnitsPerStage - 1) / kDecUnitsPerStage;
        g.ctas = (int)(want < slots ? want : slots);
        if (g.ctas < 1) g.ctas = 1;
        g.nchunks = g.ctas;
    } else {
        g.nchunks = T * split_k;
        g.ctas = (int)((long)g.nchunks < slots ? (long)g.nchunks : slots);
    }
    // S slices per tile, every slice on a CTA of its own, one batch chunk: the S CTAs of a tile form a
    // cluster and exchange their partial tiles through distributed shared memory
    g.cluster = allow_cluster && split_k >= 2 && split_k <= kDecMaxCluster && g.nchunks == g.ctas && g.mchunks == 1;
    const int budget = (227 * 1024) / kDecCtasPerSm - 1024;   // per CTA
    const int xs = g.cluster ? split_k : 0;   // slices that meet in the exchange buffer
    const int rows = M < 8 * g.mb ? M : 8 * g.mb;   // batch rows of a CTA (the last chunk of a large M may have fewer)
    // (the box is 8 chunks of 64 k long: K >= 512)
    g.a_box = rows >= kDecABoxMinRows && G >= kDecUnitsPerStage;
    g.stage_bytes = decode_stage_bytes(rows, sg, g.a_box);
    int st = kDecMaxStages;
    while (st > 2 && decode_smem_bytes(g.mb, rows, sg, st, xs, g.a_box) > budget) --st;
    g.stages = st;
    // Weights do not depend on the previous kernel of the stream, so they may be requested before the wait
    // for it.  With K slices that pays only for about as many bytes as HBM delivers during that wait (about
    // 1 us, 6.5 MB over the whole grid): requests beyond that take bandwidth from the previous kernel's last
    // CTAs and stand in the copy queue in front of this kernel's activation rows.  Measured, stages requested
    // early = 1 / 2 / whole ring: K = 11008 / N = 4096 (256 CTAs), M = 1: 9.15 / 9.4 / 10.4 us; K = 16384 /
    // N = 4096: 11.7 / 12.0 / 12.9; K = 6144 / N = 1536 (144 CTAs), M = 8: 5.7 / 5.25 / 5.25.  Whole tiles
    // (wide N, split_k = 1) gain 2 to 4 % from the whole ring (K = 4096 / N = 22016: 15.45 / 15.2 / 14.9 us).
    {
        const long stage_w = (long)kDecUnitsPerStage * (kBlockBytes + sg * (kSBlockHalves * 2 + kZBlockWords * 4));
        long pf = 6500000L / ((long)g.ctas * g.mchunks * stage_w);
        if (pf < 1) pf = 1;
        if (pf > st || split_k == 1) pf = st;
        g.prefetch = (int)pf;
    }
    g.smem_bytes = decode_smem_bytes(g.mb, rows, sg, g.stages, xs, g.a_box);
    return g;
}

// Nominal split factor of the balanced schedule: how many CTAs share one column tile's K range.
int choose_split_decode(int M, int N, int G, const Chip& chip, int sg) {
    DecodeGeom g = decode_geom(M, N, G, 0, chip, sg);
    if (g.split_k >= 1) return g.split_k;
    const int T = N / kTileN;
    int s = (g.ctas + T - 1) / T;
    if (s < 1) s = 1;
    if (s > G) s = G;
    return s;
}

// ---- tile-path launch geometry ----------------------------------------------------
// The unit range (batch tile x column tile x group) is cut into `nchunks` chunks for `ctas` persistent CTAs: balanced
// chunks, one per CTA, when the caller leaves split_k open and slices would leave too many SMs idle; S slices per tile or
// whole tiles otherwise.
struct TileGeom {
    int mt, m_tiles, n_tiles, split_k, nchunks, stages, smem_bytes, ctas;
    long tiles, cost;
};

constexpr size_t kWsFullHeaderBytes = W4A16_WORKSPACE_HEADER_BYTES;   // (the small-M kernel's tickets, the rest reserved)

// Activation ring of a CTA: beyond about 200 KiB of shared memory the L1 that the weight loads pass through gets too small
// (148 whole tiles of K = 16384, 208 rows: eight slots 120 us, six 100; 256 rows have six either way).
constexpr int kTileSmem = 200 * 1024;

// What the host needs to issue a GEMM and the kernel that sums its slices, in ns: no shorter schedule is worth them.
constexpr long kTwoLaunches = 6300;

// What a launch costs, in ns, and how its units are cut.  Here and below the constants are least-squares fits of the relative
// error to calls timed back to back, 12,700 schedules of 840 shapes drawn over M = 17 to 1500 (FP16, groups of 128): 3 to 6 %
// off; the schedules they choose take 1.4 % longer than the best ones timed.  (Fitted before the issuer's loop of kernel_tile.cuh took
// 5 to 20 % off a unit of that kernel.  Timed again with it, 90 shapes drawn over M = 65 to 1500, with and without bias and SiLU:
// the choice is 0.9 % behind the best by the geometric mean and 5 to 13 % in seven of them, mostly where few column tiles would now
// rather go to that kernel: M = 96, K = 9472 / N = 1408, eight of its slices 9.9 us, eleven of the other kernel's 11.2.)  A unit took
// a CTA 0.50 us with 80 rows and 0.57 with 256 while few SMs are busy (the ring's hand-offs) and up to 0.79 with all of them (the L2
// that brings the activations); the rest is what a launch shows beside its units, the epilogue's rows among it, and for slices the
// second kernel, the partial tiles and 79 ns for every slice that it adds.
TileGeom tile_geom_rows(int mt, int M, int N, int G, int split_k, int sms) {
    TileGeom g;
    g.mt = mt;
    g.m_tiles = (M + mt - 1) / mt;
    g.n_tiles = (N + kTileCols - 1) / kTileCols;
    g.tiles = (long)g.m_tiles * g.n_tiles;
    g.cost = 0;
    if (split_k == 0) {
        // Balanced chunks use every SM to the end, but a chunk that starts or ends inside a tile leaves an FP32 partial tile
        // behind, whose store stalls the pipeline in mid-stream; dearer from two waves on (the CTAs no longer read the same
        // activations at the same time) and never from three (M = 2787, K = 4224 / N = 13824 332 us, in waves 275; but 2.2 waves of
        // 256 rows, M = 1454, K = 13056 / N = 6912 227 us, in waves 270).  S slices per tile (tiles <= SMs)
        // or whole tiles in waves (tiles > SMs) avoid that at the price of idle SMs.
        // us after a second of load (power-capped), slices or waves / balanced: M = 256: K = 16384 / N = 4096 31.1 / 33.5, K = N =
        // 8192 34.7 / 38.0; M = 600, K = N = 8192 93.8 / 81.6; M = 777, K = 4096 / N = 22016 137 / 160; M = 1024, K = N = 8192
        // 119 / 129; M = 256, K = 8192 / N = 20480 (160 tiles) 107 / 83.
        auto take = [&](int s, long cost) {
            if (g.cost == 0 || cost < g.cost) { g.cost = cost; split_k = s; }
        };
        const long balanced = (g.tiles * G + sms - 1) / sms;
        // percent; activations of half the L2 and more do not stay in it when the CTAs read different parts of them (M = 2509,
        // K = 22144 / N = 3392, 111 MB: 397 us, in waves 370)
        const int dearer = ((long)M * G * (2 * kGroup) > (56l << 20) ? 113 : 100) * (g.tiles < 2 * sms ? 100 : 113) / 100;
        if (g.tiles <= sms) {
            const int tiles = (int)g.tiles;
            take(1, 1965 + 12 * mt + tiles * 149 / 20 + (long)G * (476 + mt * (400 + 3 * tiles) / 1000));
            auto slices = [&](int s) {
                const int ctas = tiles * s, above = ctas > 48 ? ctas - 48 : 0;
                const long cost = 3800 + 8 * mt + ctas * (440 + 62 * mt / 10) / 100 + 79 * s +
                                  (G + s - 1) / s * (451L + mt * 6 / 10 + above * (31 + mt * 4 / 10) / 100);
                take(s, cost > kTwoLaunches ? cost : kTwoLaunches);
            };
            // as many as there are SMs, or as many as pay for being added
            const int most = sms / tiles < G ? sms / tiles : G;
            if (most >= 2) slices(most);
            if (most > 2) {
                const int s = (int)(sqrtf((float)G * (451 + mt * 6 / 10) / (79 + tiles * (440 + 62 * mt / 10) / 100)) + 0.5f);
                if (s >= 2 && s < most) slices(s);
            }
            if (8 * tiles >= sms) take(0, (6000 + 26 * mt + balanced * (466 + mt * 11 / 10)) * dearer / 100);     // (fewer: slices do as well)
        } else {
            const long waves = (g.tiles + sms - 1) / sms;
            take(1, 1350 - mt + waves * (981 + 10 * mt) + waves * G * (398 + mt / 2) + g.tiles * G / sms * (96 + mt * 4 / 10));
            if (g.tiles < 3 * sms) take(0, (5540 + 61 * mt + balanced * (459 + mt)) * dearer / 100);
        }
    }
    g.split_k = split_k;
    if (split_k == 0) {
        const long units = g.tiles * G;
        long n = units / 2;                      // at least two units (four stages) per chunk
        if (n < 1) n = 1;
        if (n > sms) n = sms;
        g.nchunks = (int)n;
    } else {
        g.nchunks = (int)(g.tiles * split_k);
    }
    g.ctas = g.nchunks < sms ? g.nchunks : sms;
    int st = (kTileSmem - kTileBarBytes - 1024) / tile_stage_bytes(mt);   // (barrier block + alignment slack)
    if (st > kTileMaxStages) st = kTileMaxStages;
    if (st > kTileSlots) st = kTileSlots;               // the ring also lives in tensor memory
    // parity waits tell a barrier phase only from its neighbour: every dequant set has to come back to a slot on
    // every turn or every second one, and the issuer takes two slots a turn of its loop (kernel_tile.cuh)
    st -= st % 2;
    g.stages = st;
    g.smem_bytes = kTileBarBytes + 1024 + st * tile_stage_bytes(mt);
    // each CTA takes the SM's whole tensor memory: ask for enough shared memory that two never share an SM (beside
    // one of the kernel for small batch tiles its allocation waits until that one ends: see w4a16_device_status in the header)
    if (g.smem_bytes < 120 * 1024) g.smem_bytes = 120 * 1024;
    return g;
}

// Batch rows per tile (the MMA's N): M in equal parts of at most 256 rows, rounded up to 16 -- the fewest parts, or one or
// two more where that fills the last wave of tiles better.  M = 777, K = 4096 / N = 22016, us
// after a second of load: 4 x 208 rows 131, 4 x 256 152, 5 x 160 139.
TileGeom tile_geom(int M, int N, int G, int split_k, int sms) {
    const int least = (M + 255) / 256;
    TileGeom best = {};
    for (int parts = least; parts < least + 3; ++parts) {
        const TileGeom g = tile_geom_rows(((M + parts - 1) / parts + 15) / 16 * 16, M, N, G, 0, sms);
        if (parts == least || g.cost < best.cost) best = g;
    }
    return split_k == 0 ? best : tile_geom_rows(best.mt, M, N, G, split_k, sms);
}

// ---- two-CTAs-per-SM tcgen05 kernel (kernel_mid.cuh): launch geometry --------------
constexpr int kMidSmemBudget = (228 * 1024) / 2 - 1024;   // dynamic shared memory of one of two CTAs of an SM

struct MidGeom {
    int mtc, mt, m_tiles, n_tiles, split_k, nchunks, wstages, smem_bytes, ctas;
    long tiles, cost;
    bool cluster;
};

// Clusters of `size` CTAs of that kernel (two per SM) that run at the same time.  The SMs of a GPC hold whole clusters
// only, so this is less than slots / size, and which SMs a GPC has differs from chip to chip: ask, once per device.
// (The runtime counts one CTA per SM for any kernel that allocates tensor memory, so it is asked about a kernel of the
// same launch shape without it, which is never launched.  On the chip measured it says 148 / 93 / 71 / 56 / 45 / 37 / 33
// for 2 .. 8, and calls with one tile more than that take a second wave: 92 tiles in three slices 8.5 us, 96 12.9;
// 70 in four 7.1, 74 11.4; 32 in eight 6.4, 34 9.8, at K = 2048.)
__global__ void __launch_bounds__(kMidThreads, 2) mid_shape_probe_kernel(float* out) {
    extern __shared__ float probe_smem[];
    out[threadIdx.x] = probe_smem[threadIdx.x];
}
const int* mid_max_clusters(DeviceState* d) {     // [size]
    static const int without_device[kMidMaxCluster + 1] = {0, 296, 148, 93, 71, 56, 45, 37, 33};   // (size queries on a host)
    if (d == nullptr || !d->is_sm100) return without_device;
    if (d->mid_clusters[1] != 0) return d->mid_clusters;
    const bool ok = cudaFuncSetAttribute(mid_shape_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         d->max_smem_optin) == cudaSuccess;
    for (int size = 2; size <= kMidMaxCluster; ++size) {
        int n = 0;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(size * d->sm_count), 1, 1);
        cfg.blockDim = dim3(kMidThreads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)kMidSmemBudget;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (!ok || cudaOccupancyMaxActiveClusters(&n, mid_shape_probe_kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        d->mid_clusters[size] = n;
    }
    d->mid_clusters[1] = 2 * d->sm_count;
    return d->mid_clusters;
}

// mtc: most batch rows of a tile, 64 or 128.  Cost model in ns, fitted like the wide-tile kernel's.  A unit takes a CTA of the
// 64-row build 0.34 us with 16 rows and 0.40 with 64 while it has the SM to itself, 0.50 and 0.52 where two share it (whole
// tiles from the first on: 1 / 16 / 32 / 64 of 16 rows 0.34 / 0.39 / 0.44 / 0.47; clusters from 56 CTAs on), more with
// three quarters of the slots taken (64 rows: 256 / 280 / 296 CTAs 0.57 / 0.62 / 0.66).  The exchange inside a cluster grows with
// the rows that a CTA finishes and with the CTAs at it; sizes that are not a power of two and slices of a single unit cost
// a little more, the last cluster that fits finds its place late (16 rows, K = 5120: 91 / 92 / 93 tiles in three slices
// 11.3 / 11.4 / 12.4 us).  Slices beyond a cluster pay for the second kernel and 63 ns each (K = 24960, two tiles, 32 rows: eight
// slices 12.2 us, 16 / 24 / 32 / 74 through the workspace 9.9 / 9.4 / 8.8 / 11.9).
// Measured (us), M = 32: K = N = 4096 four slices 7.09, eight 7.44; K = 11008 / N = 4096 8 / 6 / 4 slices 11.0 / 11.6 /
// 13.8; K = 18432 / N = 7168 5 / 4 21.8 / 22.9; K = 4096 / N = 12288 2 / 1 12.2 / 17.3, three no longer fit at once: 17.5;
// K = 4096 / N = 22016 1 / 2 18.7 / 22.6; K = 1024 / N = 3136 4 / 8 4.18 / 5.10.
// Whole tiles that leave SMs free take one SM each, by asking for more than half of its shared memory: beside the CTAs of the
// launch in front, which are still there when this one starts early, they would come to sit in pairs, and a pair takes 0.45 to
// 0.53 us a unit instead of 0.35 to 0.41.  us in pairs / spread, 32 rows: K = 4096: 64 tiles 17.6 / 14.6, 114 18.5 / 15.0, 140
// 18.6 / 15.3, 148 15.6 / 15.6; K = 1280: 75 6.9 / 6.6, 130 7.5 / 7.1, 148 6.8 / 7.4; K = 640: 130 5.0 / 5.3 (the next launch
// cannot start beside this one).  With one CTA per SM and the kernel before this one: 75 tiles of K = 1280, 64 rows, 7.3.
bool mid_spread(long tiles, int G, int sms) { return tiles <= sms - 8 && G >= 8; }

MidGeom mid_geom(int mtc, int M, int N, int G, int split_k, const Chip& chip, int sg) {
    MidGeom g;
    const int sms = chip.sms;
    const bool allow_cluster = chip.clusters;
    g.mtc = mtc;
    g.m_tiles = (M + g.mtc - 1) / g.mtc;
    g.mt = ((M + g.m_tiles - 1) / g.m_tiles + 15) / 16 * 16;
    g.n_tiles = (N + kTileCols - 1) / kTileCols;
    g.tiles = (long)g.m_tiles * g.n_tiles;
    const int slots = 2 * sms;
    auto fits = [&](int s) { return mid_smem_bytes(g.mtc, g.mt, sg, 2, s) <= kMidSmemBudget; };
    g.cost = 0;
    if (split_k == 0) {
        const int* max_clusters = chip.max_clusters;
        const bool wide = mtc > 64;
        const int mt = g.mt, tiles = (int)(g.tiles < slots ? g.tiles : slots);
        auto take = [&](int s, long cost) {
            if (g.cost == 0 || cost < g.cost) { g.cost = cost; split_k = s; }
        };
        const int rows_ns = sg / 2;     // more scale rows a unit: felt where two CTAs share an SM
        auto sharing = [](int ctas) { return ctas <= 56 ? 0 : ctas >= 104 ? 48 : ctas - 56; };        // of 48
        auto crowd = [&](int ctas) { return ctas > slots * 3 / 4 ? ctas - slots * 3 / 4 : 0; };      // of 74
        if (g.tiles > slots) {
            const long waves = (g.tiles + slots - 1) / slots;
            take(1, wide ? 39 * mt - 670 + waves * (3300 + G * (800L + mt * 4 / 10)) : 600 + waves * (2900 + G * 520L));
        } else if (mid_spread(g.tiles, G, sms)) {
            take(1, wide ? 1620 + 23 * mt + tiles * 285 / 100 + G * (677L - mt / 2 + mt * 3 * tiles / 1000)
                         : 1850 + 16 * mt + tiles * 555 / 100 + G * (330L + mt * 11 / 10 + mt * 7 * tiles / 1000 + 14 * rows_ns * sharing(tiles) / 48));
        } else {
            const int pairs = tiles < 80 ? tiles : 80;
            take(1, wide ? 1740 + 22 * mt + tiles * 514 / 100 + G * (587L + mt * 4 / 10 + 161 * sharing(tiles) / 48)
                         : 1900 + 22 * mt + 2 * tiles + G * (320L + mt * 13 / 10 + (170 - mt * 8 / 10 + 34 * rows_ns) * pairs / 80 + crowd(tiles) * mt * 14 / 740));
        }
        auto cluster = [&](auto size) {        // (sizes as constants: three divisions by each)
            constexpr int s = decltype(size)::value;
            if (s > G || tiles > max_clusters[s] || !fits(s)) return;
            const int ctas = tiles * s, rows = (mt / 4 + s - 1) / s, u = (G + s - 1) / s;
            const bool odd = (s & (s - 1)) != 0, last = s > 2 && tiles == max_clusters[s];
            take(s, wide ? 2230 + 33 * mt + ctas * (15 * mt - 104) / 100 + 99 * s + 26 * rows + u * (644L + 164 * sharing(ctas) / 48 - crowd(ctas) * mt * 9 / 740) +
                               (odd ? 201 : 0) + (last ? 1613 : 0)
                         : 2550 + 17 * mt + ctas * (280 + 55 * mt / 10) / 100 + 63 * s + 96 * rows +
                               u * (316L + mt * 15 / 10 + (109 + 34 * rows_ns) * sharing(ctas) / 48 + crowd(ctas) * (178 - mt * 3 / 4 + 50 * rows_ns) / 100) +
                               (odd ? 107 : 0) + (last ? 513 : 0) + (u == 1 ? 493 : 0) +
                               (sg > 1 && mt < 64 && mid_smem_bytes(mtc, mt, sg, 3, s) > kMidSmemBudget ? 400 : 0));   // (two-stage weight ring)
        };
        if (allow_cluster) for_each_size<2, kMidMaxCluster>(cluster);
        // through the workspace: as many slices as there are SMs or slots, or as many as pay for being added
        // (with few slices only where their exchange buffer leaves no room for a cluster: groups of 32, 64 rows)
        if (3 * tiles <= slots * 7 / 8) {
            const int unit = wide ? 697 + mt / 2 : 224 + mt * 29 / 10, more = wide ? 19 * mt - 364 : 15 * mt - 234;
            const int add = (wide ? 62 : 63) + tiles * more / 100;
            const int pays = (int)(sqrtf((float)G * unit / (add > 20 ? add : 20)) + 0.5f);
            for (int cap : {sms / tiles, slots * 7 / 8 / tiles}) {
                int s = cap < pays ? cap : pays;
                if (s > G) s = G;
                if (s < 2 || (s <= kMidMaxCluster && allow_cluster && fits(s))) continue;
                const int ctas = tiles * s;
                const long cost = (wide ? 4350 + mt : 5200 - 13 * mt) + ctas * more / 100 + (wide ? 62 : 63) * s +
                                  (G + s - 1) / s * (unit + (wide ? -23L : 104L + 28 * rows_ns) * sharing(ctas) / 48);
                take(s, cost > kTwoLaunches ? cost : kTwoLaunches);
            }
        }
        // (large activations, which every column tile reads again, do not stay in L2: M = 1968, K = 15616 / N = 2432 174 us)
        if ((long)M * G * (2 * kGroup) > (40l << 20)) g.cost += g.cost / 4;
    }
    g.split_k = split_k;
    g.cluster = allow_cluster && split_k >= 2 && split_k <= kMidMaxCluster && fits(split_k);
    g.nchunks = (int)(g.tiles * split_k);
    g.ctas = g.cluster || g.nchunks < slots ? g.nchunks : slots;
    int st = kMidMaxWStages;
    while (st > 2 && mid_smem_bytes(g.mtc, g.mt, sg, st, g.cluster ? split_k : 0) > kMidSmemBudget) --st;
    g.wstages = st;
    g.smem_bytes = mid_smem_bytes(g.mtc, g.mt, sg, st, g.cluster ? split_k : 0);
    // A CTA takes half of the SM's tensor memory: ask for enough shared memory that no third one, and no CTA of the
    // wide-tile kernel (which takes all of it), ever shares the SM, so that the allocation never has to wait.
    if (g.smem_bytes < 108 * 1024) g.smem_bytes = 108 * 1024;
    if (split_k == 1 && mid_spread(g.tiles, G, sms) && g.smem_bytes < 120 * 1024) g.smem_bytes = 120 * 1024;
    return g;
}
size_t mid_workspace_bytes(const MidGeom& g) {
    if (g.split_k == 1) return 0;
    return round256((size_t)2 * g.nchunks * g.mt * kTileCols * sizeof(float));
}

// Partial-tile slots of the tile path: two per chunk.  Nothing when every chunk is a whole tile.
size_t tile_workspace_bytes(const TileGeom& g) {
    if (g.split_k == 1) return 0;
    return round256((size_t)2 * g.nchunks * g.mt * kTileCols * sizeof(float));
}

// The tcgen05 path's kernel for a shape: up to 64 rows the 64-row build of kernel_mid.cuh; above, the cheapest by the cost
// models of it (several batch tiles), its 128-row build and kernel_tile.cuh.  us in that order, after a second of load: M = 128:
// K = N = 4096 14.2 / 20.2 / 15.0, K = 11008 / N = 4096 16.9 / 19.6 / 17.7, K = N = 8192 24.3 / 24.4 / 24.7, K = 4096 / N = 22016
// 36.4 / 31.4 / 32.8; M = 256: K = N = 2048 8.4 / 13.4 / 9.5, K = 16384 / N = 4096 46.5 / 41.7 / 35.4; M = 300, K = 4096 / N =
// 12288 45.6 / 34.4 / 43.7; M = 512 69.6 / 66.7 / 48.1; M = 1024, K = N = 8192 181 / 132 / 110.
struct WidePlan {
    bool use_mid;
    MidGeom mid;
    TileGeom tile;
    size_t workspace_bytes() const { return use_mid ? mid_workspace_bytes(mid) : tile_workspace_bytes(tile); }
};
WidePlan wide_plan(int M, int N, int G, int split_k, const Chip& chip, int sg, bool epi) {
    WidePlan w;
    w.use_mid = true;
    if (M <= 64) {
        w.mid = mid_geom(64, M, N, G, split_k, chip, sg);
        return w;
    }
    w.mid = mid_geom(64, M, N, G, 0, chip, sg);
    const MidGeom m128 = mid_geom(128, M, N, G, 0, chip, sg);
    if (m128.cost < w.mid.cost) w.mid = m128;
    w.tile = tile_geom(M, N, G, 0, chip.sms);
    // (bias and SiLU in that kernel's own epilogue: K = 512 / N = 12288, 80 / 208 rows 1.9 / 2.9 us more, bias and ReLU 0.7 / 0.8;
    // in the other one 1.2 / 2.1 and 0.4 / 0.6)
    if (epi && w.tile.split_k == 1) w.tile.cost += (w.tile.tiles + chip.sms - 1) / chip.sms * (1200 + 8 * w.tile.mt);
    w.use_mid = w.mid.cost < w.tile.cost;
    if (split_k != 0) {
        if (w.use_mid) w.mid = mid_geom(w.mid.mtc, M, N, G, split_k, chip, sg);
        else w.tile = tile_geom(M, N, G, split_k, chip.sms);
    }
    return w;
}

// 9 to 16 rows with path and split_k left open: the warp-MMA kernel runs its 16-row build, which converts every weight for
// two MMAs; the two-CTA tcgen05 kernel is ahead on long shapes and level on short ones (calls of less than 4.6 us are the host's, and
// its own is shorter).  us, warp-MMA / tcgen05, M = 16: K = 28672 / N = 8192 38.6 / 32.1, K = 18432 / N = 7168 26.4 / 21.3, K = 4096 /
// N = 12288 12.7 / 11.1, K = 8192 / N = 8192 13.3 / 12.5, K = 27648 / N = 1024 15.2 / 10.5, K = 1024 / N = 3136 5.0 / 3.9, K = 11008 /
// N = 4096 10.9 / 10.4; K = N = 4096 6.1 / 6.8, K = 2048 / N = 8192 5.9 / 6.5, K = 6144 / N = 1536 6.0 / 6.0.
bool small_batch_takes_mid(const DecodeGeom& d, int M, int N, int G, const Chip& chip, int sg, MidGeom* mid) {
    if (M < 9 || M > 16 || d.cost < 4600) return false;
    *mid = mid_geom(64, M, N, G, 0, chip, sg);
    // Whole tiles, and more of them than CTA slots: level by itself, but in front of or behind another launch, as between a
    // block's projections, some SMs get four (us, K = 4096 / N = 22016: 18.8 / 18.5, and with K = N = 4096 in front 30.2 / 25.4).
    // Groups of 32 cost this kernel more (18.9 / 21.1 by itself): by cost, like balanced chunks (K = 8192 / N = 20224 31.4 / 35.1
    // and 40.7 / 43.7).
    if (sg < 4 && d.split_k == 1 && N / kTileN >= 2 * chip.sms + 8) return true;
    // (with an SM to itself a CTA of the warp-MMA kernel is faster than its model says: 256 columns of K = 13952 6.8 us)
    const long dec = d.cluster && d.nchunks <= 36 ? d.cost - 100 * ((G + d.split_k - 1) / d.split_k) : d.cost;
    return mid->cost * 100 < dec * 93;
}

// Nominal split factor of the tcgen05 path's schedule: how many chunks share one tile's K range.
int nominal_split(const WidePlan& w, int G) {
    if (w.use_mid) return w.mid.split_k;
    if (w.tile.split_k >= 1) return w.tile.split_k;
    long s = (w.tile.nchunks + w.tile.tiles - 1) / w.tile.tiles;
    if (s < 1) s = 1;
    if (s > G) s = G;
    return (int)s;
}

// cuTensorMapEncodeTiled, resolved through the runtime so that libcuda is not a link dependency.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
        else
            cudaGetLastError();
    }
    return fn;
}

// Activations A [M, K] 16-bit row-major as a 2-D tensor (k innermost), box = 64 k x mt rows, 128-byte swizzle; rows past
// M read as zero.  With stage_k = 128 one copy brings the stage's two boxes.
bool make_act_tensor_map(CUtensorMap* map, const void* A, int M, int K, int mt, int stage_k) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    if (stage_k == kTileBoxK) {     // one box per stage: plain 2-D tensor, k innermost
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
        const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
        const cuuint32_t box[2] = {(cuuint32_t)kTileBoxK, (cuuint32_t)mt};
        const cuuint32_t estr[2] = {1, 1};
        return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(A), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    // A[M][K] seen as [K / 64][M][64]: one copy brings a stage's 64-k boxes one after the other
    const cuuint64_t dims[3] = {(cuuint64_t)kTileBoxK, (cuuint64_t)M, (cuuint64_t)(K / kTileBoxK)};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)kTileBoxK * 2};
    const cuuint32_t box[3] = {(cuuint32_t)kTileBoxK, (cuuint32_t)mt, (cuuint32_t)(stage_k / kTileBoxK)};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(A), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same activations for the warp-MMA kernel's tensor copy: [K / 64][M][64], box = the 8 chunks of a
// stage x 8 mb rows x 64 k.
bool make_decode_tensor_map(CUtensorMap* map, const void* A, int M, int K, int mb) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    const cuuint64_t dims[3] = {64, (cuuint64_t)M, (cuuint64_t)(K / 64)};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 2, 128};
    const cuuint32_t box[3] = {64, (cuuint32_t)(8 * mb), (cuuint32_t)kDecABoxChunks};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(A), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Path taken when the caller does not force one: up to 16 batch rows the warp-MMA kernel (with 9 to 16, long shapes go to
// the tcgen05 kernel all the same: small_batch_takes_mid), above that the tcgen05 kernels; the warp-MMA kernel would need a
// second pass over the weights (M = 24, when that was measured: 22.5 us against 12.8 and 75.8 against 42.2 at K = 11008 /
// N = 4096 and K = 28672 / N = 8192).
int resolve_path(int M, int path) {
    if (path != W4A16_PATH_AUTO) return path;
    return M <= 16 ? W4A16_PATH_DECODE : W4A16_PATH_TILE;
}

// FP32 partials of the two-kernel reduce used by the plain path: [split_k][M][N].
size_t simple_partial_bytes(int M, int N, int split_k) {
    return round256((size_t)split_k * (size_t)M * (size_t)N * sizeof(float));
}
// Partial-tile slots of the decode kernel: [m chunk][2 * nchunks][8 mb][64] FP32.
size_t decode_partial_bytes(const DecodeGeom& g) {
    return round256((size_t)g.mchunks * 2 * (size_t)g.nchunks * (8 * g.mb) * kTileN * sizeof(float));
}

// Workspace that the warp-MMA kernel's schedule asks for, given the caller's split_k.
size_t decode_scratch(const DecodeGeom& g, int split_k) {
    return g.split_k == 1 || (split_k == 0 && g.cluster) ? 0 : decode_partial_bytes(g);
}

// Can the warp-MMA kernel number this launch's batch chunks and tickets?
bool decode_runs(const DecodeGeom& g, int N) { return g.mchunks <= 65535 && (long)g.mchunks * (N / kTileN) <= kMaxTickets; }

// What a GEMM call runs: kernel, schedule and the workspace behind the header that it asks for (0: none).  The entry points
// and the queries all come here, with the group's scale rows per block (sg): whether a cluster's exchange buffer fits, and
// with it the number of slices, depends on them.
struct GemmPlan {
    int rc;              // W4A16_OK, or why the kernel cannot run the shape
    int kernel;          // W4A16_KERNEL_*
    int split_simple;
    DecodeGeom dec;
    WidePlan wide;
    size_t workspace;
};
// An explicit split_k > 1 asks for its workspace on every kernel, used or not.  With split_k == 0 slices that meet in a cluster
// ask for none, and balanced chunks, which cross tile boundaries, give way to whole tiles where `ws_bytes` does not hold them.
GemmPlan gemm_plan(int M, int N, int G, int sg, int split_k, int path_asked, bool epi, const Chip& chip, size_t ws_bytes) {
    GemmPlan p;
    p.rc = W4A16_OK;
    const int path = resolve_path(M, path_asked);
    if (path == W4A16_PATH_SIMPLE) {
        p.kernel = W4A16_KERNEL_SIMPLE;
        p.split_simple = split_k == 0 ? choose_split_decode(M, N, G, chip, sg) : split_k;
        p.workspace = p.split_simple > 1 ? simple_partial_bytes(M, N, p.split_simple) : 0;
        if ((M + kSimpleMB - 1) / kSimpleMB > 65535) p.rc = W4A16_ERR_PATH;
        return p;
    }
    if (path == W4A16_PATH_DECODE) {
        p.kernel = W4A16_KERNEL_DECODE;
        p.dec = decode_geom(M, N, G, split_k, chip, sg);
        p.wide.use_mid = path_asked == W4A16_PATH_AUTO && split_k == 0 && small_batch_takes_mid(p.dec, M, N, G, chip, sg, &p.wide.mid);
        if (!p.wide.use_mid) {
            p.workspace = decode_scratch(p.dec, split_k);
            if (p.workspace > ws_bytes && p.dec.split_k == 0) {
                p.dec = decode_geom(M, N, G, 1, chip, sg);
                p.workspace = 0;
            }
            if (!decode_runs(p.dec, N)) p.rc = W4A16_ERR_PATH;
            return p;
        }
    } else {
        p.wide = wide_plan(M, N, G, split_k, chip, sg, epi);
    }
    p.kernel = !p.wide.use_mid ? W4A16_KERNEL_TILE : p.wide.mid.mtc <= 64 ? W4A16_KERNEL_MID64 : W4A16_KERNEL_MID128;
    p.workspace = split_k == 0 && p.wide.use_mid && p.wide.mid.cluster ? 0 : p.wide.workspace_bytes();
    if (p.workspace > ws_bytes && !p.wide.use_mid && p.wide.tile.split_k == 0) {
        p.wide.tile = tile_geom(M, N, G, 1, chip.sms);
        p.workspace = 0;
    }
    // 32-bit arithmetic: the kernels count units and chunks, the kernel that sums slices the rows of all tiles
    const bool mid = p.wide.use_mid;
    const long long tiles = mid ? p.wide.mid.tiles : p.wide.tile.tiles;
    const bool summed = mid ? p.wide.mid.split_k != 1 && !p.wide.mid.cluster : p.wide.tile.split_k != 1;
    const int units = mid ? p.wide.mid.split_k : G, rows = !summed ? 0 : mid ? p.wide.mid.mt : p.wide.tile.mt;
    if (tiles * (units > rows ? units : rows) >= (1ll << 31)) p.rc = W4A16_ERR_SHAPE;
    return p;
}

// Quantizer, pack and dequantization: set up while the kernel in front runs, and ordered behind it by the kernels themselves (in a row, as a
// model load calls them, a gap between two launches costs about 2 us).  In a graph plain launches, with a pack that releases nothing.
template <typename... P, typename... A>
int launch_block_kernel(void (*kern)(P...), unsigned blocks, cudaStream_t st, bool early, A... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks, 1, 1);
    cfg.blockDim = dim3(kBlockKernelThreads, 1, 1);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    return W4A16_OK;
}

// ---- built-in scratch for w4a16_gemm_static_ws -------------------------------------
// Lives in the library's device image: every GPU that loads the library holds these bytes until
// the process exits.  In host code `g_static_ws` is only a handle for cudaGetSymbolAddress; the
// device address is looked up once per device (below) and that is what the kernel receives.
static __device__ __align__(256) unsigned char g_static_ws[W4A16_STATIC_WS_BYTES];
unsigned char* g_static_ws_addr[kMaxDevices] = {};

}  // namespace

// =====================================================================================
extern "C" {

const char* w4a16_strerror(int code) {
    switch (code) {
        case W4A16_OK: return "ok";
        case W4A16_ERR_NULL: return "null pointer argument";
        case W4A16_ERR_SHAPE: return "unsupported shape or option (need group in {32, 64, 128}, K % 128 == 0, N % 64 == 0, M >= 1)";
        case W4A16_ERR_ALIGN: return "buffer not 16-byte aligned (workspace: 256-byte)";
        case W4A16_ERR_SPLITK: return "split_k out of range for this shape / path";
        case W4A16_ERR_WORKSPACE: return "split-K workspace missing or too small (w4a16_set_workspace)";
        case W4A16_ERR_CUDA: return "CUDA runtime call failed";
        case W4A16_ERR_ARCH: return "current device is not sm_100";
        case W4A16_ERR_DEVICE_STATUS: return "a kernel gave up on a bounded wait";
        case W4A16_ERR_PATH: return "requested kernel path does not support this shape";
        default: return "unknown error code";
    }
}

size_t w4a16_packed_wq_bytes(int N, int K, int group) {
    if (check_weight_shape(N, K, group) != W4A16_OK) return 0;
    return (size_t)K * (size_t)N / 2;
}
size_t w4a16_packed_s_bytes(int N, int K, int group) {
    if (check_weight_shape(N, K, group) != W4A16_OK) return 0;
    return (size_t)(K / group) * (size_t)N * 2;
}
size_t w4a16_packed_z_bytes(int N, int K, int group) {   // asymmetric formats; a symmetric one has no Z buffer
    if (check_weight_shape(N, K, group) != W4A16_OK) return 0;
    return (size_t)(K / group) * (size_t)N / 2;
}

int w4a16_choose_split_k_ex(int M, int N, int K, int group, int path) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (check_weight_shape(N, K, group) != W4A16_OK || M < 1 || path < W4A16_PATH_AUTO || path > W4A16_PATH_TILE || path == W4A16_PATH_SIMPLE) return 1;
    const int G = K / kGroup, sg = kGroup / group;
    const Chip chip = chip_or_default();
    const GemmPlan p = gemm_plan(M, N, G, sg, 0, path, false, chip, SIZE_MAX);
    return p.kernel == W4A16_KERNEL_DECODE ? choose_split_decode(M, N, G, chip, sg) : nominal_split(p.wide, G);
}
int w4a16_choose_path(int M, int N, int K, int group) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (check_weight_shape(N, K, group) != W4A16_OK || M < 1) return W4A16_ERR_SHAPE;
    const GemmPlan p = gemm_plan(M, N, K / kGroup, kGroup / group, 0, W4A16_PATH_AUTO, false, chip_or_default(), SIZE_MAX);
    return p.kernel == W4A16_KERNEL_DECODE ? W4A16_PATH_DECODE : W4A16_PATH_TILE;
}
int w4a16_choose_split_k(int M, int N, int K, int group) {
    return w4a16_choose_split_k_ex(M, N, K, group, W4A16_PATH_AUTO);
}

size_t w4a16_workspace_bytes(int M, int N, int K, int group, int split_k) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (check_weight_shape(N, K, group) != W4A16_OK || M < 1 || split_k < 0 || split_k > K / kGroup) return 0;
    if (split_k == 1) return 0;
    // enough for whichever path w4a16_gemm / w4a16_gemm_ex may take with this split_k, on a device that places clusters
    // and on one that refused them (the schedule differs)
    const int G = K / kGroup, sg = kGroup / group;
    Chip chip = chip_or_default();
    chip.clusters = true;
    size_t need = simple_partial_bytes(M, N, split_k == 0 ? choose_split_decode(M, N, G, chip, sg) : split_k);
    const size_t whole = decode_partial_bytes(decode_geom(M, N, G, split_k, chip, sg));   // (asked for by whole tiles too)
    if (whole > need) need = whole;
    for (const Chip& c : {chip, without_clusters(chip)})
        for (bool epi : {false, true})
            for (int path : {W4A16_PATH_AUTO, W4A16_PATH_SIMPLE, W4A16_PATH_DECODE, W4A16_PATH_TILE}) {
                const size_t n = gemm_plan(M, N, G, sg, split_k, path, epi, c, SIZE_MAX).workspace;
                if (n > need) need = n;
            }
    return kWsFullHeaderBytes + need;
}

int w4a16_gemm_plan(int M, int N, int K, int group, int split_k, int path, int with_epilogue, w4a16_plan* out) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!out) return W4A16_ERR_NULL;
    const int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (M < 1) return W4A16_ERR_SHAPE;
    if (split_k < 0 || split_k > K / kGroup) return W4A16_ERR_SPLITK;
    if (path < W4A16_PATH_AUTO || path > W4A16_PATH_TILE) return W4A16_ERR_PATH;
    const GemmPlan g = gemm_plan(M, N, K / kGroup, kGroup / group, split_k, path, with_epilogue != 0, chip_or_default(), SIZE_MAX);
    if (g.rc != W4A16_OK) return g.rc;
    out->kernel = g.kernel;
    out->workspace_bytes = g.workspace == 0 ? 0 : kWsFullHeaderBytes + g.workspace;
    switch (g.kernel) {
        case W4A16_KERNEL_SIMPLE: out->tile_rows = kSimpleMB; out->split_k = g.split_simple; out->cluster = 0; break;
        case W4A16_KERNEL_DECODE: out->tile_rows = 8 * g.dec.mb; out->split_k = g.dec.split_k; out->cluster = g.dec.cluster ? 1 : 0; break;
        case W4A16_KERNEL_TILE: out->tile_rows = g.wide.tile.mt; out->split_k = g.wide.tile.split_k; out->cluster = 0; break;
        default: out->tile_rows = g.wide.mid.mt; out->split_k = g.wide.mid.split_k; out->cluster = g.wide.mid.cluster ? 1 : 0;
    }
    return W4A16_OK;
}

int w4a16_set_workspace(void* dev_ptr, size_t bytes) {
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState* d = nullptr;
    int rc = current_device(&d);
    if (rc != W4A16_OK) return rc;
    if (dev_ptr == nullptr || bytes == 0) {
        d->ws = nullptr;
        d->ws_bytes = 0;
        return W4A16_OK;
    }
    if ((reinterpret_cast<uintptr_t>(dev_ptr) & 255u) != 0) return W4A16_ERR_ALIGN;
    if (bytes < kWsFullHeaderBytes) return W4A16_ERR_WORKSPACE;
    // the ticket counters start at zero (and are zero again after every call)
    if (cudaMemset(dev_ptr, 0, kWsFullHeaderBytes) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    d->ws = dev_ptr;
    d->ws_bytes = bytes;
    return W4A16_OK;
}

int w4a16_quantize(const uint16_t* W16, uint32_t* Wq_raw, uint16_t* S_raw, uint8_t* Z_raw, int N, int K, int group,
                   int flags, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!flags_ok(flags)) return W4A16_ERR_SHAPE;
    const bool sym = (flags & W4A16_FLAG_SYMMETRIC) != 0, bf = (flags & W4A16_FLAG_BF16) != 0;
    if (!W16 || !Wq_raw || !S_raw || (!sym && !Z_raw)) return W4A16_ERR_NULL;
    int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (!aligned16(W16) || !aligned16(Wq_raw) || !aligned16(S_raw) || (!sym && !aligned16(Z_raw))) return W4A16_ERR_ALIGN;
    DeviceState* d = nullptr;
    if ((rc = current_device(&d)) != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    const int G = K / kGroup, sg = kGroup / group;
    const unsigned blocks = (unsigned)((long long)G * (N / kTileN));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* z = sym ? nullptr : Z_raw;
    return launch_block_kernel(bf ? quantize_kernel<true> : quantize_kernel<false>, blocks, st, PackOrder::may_release(capture_of(st)), W16, Wq_raw, S_raw, z, N, G, sg, sym ? 1 : 0);
}

int w4a16_pack_fmt(const uint32_t* Wq_raw, const uint16_t* S_raw, const uint8_t* Z_raw, void* Wq, void* S, void* Z,
                   int N, int K, int group, int flags, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!flags_ok(flags)) return W4A16_ERR_SHAPE;
    const bool sym = (flags & W4A16_FLAG_SYMMETRIC) != 0;
    if (!Wq_raw || !S_raw || !Wq || !S) return W4A16_ERR_NULL;
    if (!sym && (!Z_raw || !Z)) return W4A16_ERR_NULL;
    int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (!aligned16(Wq_raw) || !aligned16(S_raw) || !aligned16(Wq) || !aligned16(S)) return W4A16_ERR_ALIGN;
    if (!sym && (!aligned16(Z_raw) || !aligned16(Z))) return W4A16_ERR_ALIGN;
    DeviceState* d = nullptr;
    if ((rc = current_device(&d)) != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int G = K / kGroup, sg = kGroup / group;
    const int blocks = (int)((long long)G * (N / kTileN)), per = kBlockKernelThreads / 64;   // half a block a warp
    const bool early = PackOrder::may_release(capture_of(st));
    d->order.pack_issued();
    return launch_block_kernel(pack_kernel, (unsigned)((blocks + per - 1) / per), st, early, Wq_raw, S_raw, sym ? nullptr : Z_raw,
                               static_cast<uint32_t*>(Wq), static_cast<uint16_t*>(S), sym ? nullptr : static_cast<uint8_t*>(Z), N, G, sg, blocks, early);
}

int w4a16_pack(const uint32_t* Wq_raw, const uint16_t* S_raw, const uint8_t* Z_raw, void* Wq, void* S, void* Z,
               int N, int K, int group, w4a16_stream_t stream) {
    if (!Z_raw || !Z) return W4A16_ERR_NULL;
    return w4a16_pack_fmt(Wq_raw, S_raw, Z_raw, Wq, S, Z, N, K, group, 0, stream);
}

int w4a16_dequant_fmt(const void* Wq, const void* S, const void* Z, uint16_t* W16, int N, int K, int group, int flags,
                      w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!flags_ok(flags)) return W4A16_ERR_SHAPE;
    const bool sym = (flags & W4A16_FLAG_SYMMETRIC) != 0, bf = (flags & W4A16_FLAG_BF16) != 0;
    if (!Wq || !S || !W16 || (!sym && !Z)) return W4A16_ERR_NULL;
    int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (!aligned16(Wq) || !aligned16(S) || (!sym && !aligned16(Z)) || !aligned16(W16)) return W4A16_ERR_ALIGN;
    DeviceState* d = nullptr;
    if ((rc = current_device(&d)) != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    const unsigned blocks = (unsigned)((long long)(K / kGroup) * (N / kTileN));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_block_kernel(bf ? dequant_kernel<true> : dequant_kernel<false>, blocks, st, PackOrder::may_release(capture_of(st)),
                               static_cast<const uint32_t*>(Wq), static_cast<const uint16_t*>(S),
                               sym ? nullptr : static_cast<const uint32_t*>(Z), W16, N, K / kGroup, kGroup / group);
}

int w4a16_dequant(const void* Wq, const void* S, const void* Z, uint16_t* W16, int N, int K, int group,
                  w4a16_stream_t stream) {
    if (!Z) return W4A16_ERR_NULL;
    return w4a16_dequant_fmt(Wq, S, Z, W16, N, K, group, 0, stream);
}

}  // extern "C"

namespace {

// ---- kernel tables: the instantiations live in the inst_*.cu units --------------------------------
DecodeKernel decode_kernel(int mb, bool cluster, int sg, bool bf, bool sym, bool a_box) {
    return bf ? decode_kernel_bf16(mb, cluster, sg, sym, a_box) : decode_kernel_f16(mb, cluster, sg, sym, a_box);
}
TileKernel tile_kernel(int sg, bool bf, bool sym, bool epi) {
    if (bf) return sg == 1 ? tile_kernel_bf16_sg1(sym, epi) : sg == 2 ? tile_kernel_bf16_sg2(sym, epi)
                                                                                : tile_kernel_bf16_sg4(sym, epi);
    return sg == 1 ? tile_kernel_f16_sg1(sym, epi) : sg == 2 ? tile_kernel_f16_sg2(sym, epi)
                                                                       : tile_kernel_f16_sg4(sym, epi);
}

// Launches a GEMM kernel.  Programmatic dependent launch where the order allows it: its prologue and its requests for packed weights
// overlap the tail of the previous kernel of the stream, and it orders itself with griddepcontrol.wait.
// `cluster` CTAs with consecutive blockIdx.x form a thread-block cluster.
template <typename Params>
bool launch_gemm_kernel(DeviceState* d, cudaLaunchConfig_t cfg, int cluster, void (*kern)(CUtensorMap, Params), const CUtensorMap& tmap, const Params& p) {
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (cluster > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = (unsigned)cluster;
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    return d->order.launch(reinterpret_cast<uintptr_t>(cfg.stream), [&] { return capture_of(cfg.stream); }, [&](bool overlap) {
        if (overlap) {
            attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
            ++n_attr;
        }
        cfg.attrs = attr;
        cfg.numAttrs = n_attr;
        if (cudaLaunchKernelEx(&cfg, kern, tmap, p) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    });
}

// Split-K sum behind a tcgen05 kernel that stored its partial tiles: S slices per tile, or (split_k == 0) balanced chunks.
int launch_tile_reduce(const float* parts, uint16_t* C, int M, int N, int G, int mt, int n_tiles, long tiles, int split_k,
                       int nchunks, bool bf, const Epilogue& epi, cudaStream_t st) {
    TileReduce p;
    p.M = M; p.N = N; p.G = G;
    p.mt = mt;
    p.n_tiles = n_tiles;
    p.split_k = split_k;
    p.nchunks = nchunks;
    p.bal_q = (int)((long long)tiles * G / nchunks);
    p.bal_r = (int)((long long)tiles * G % nchunks);
    p.div_mt = fast_div_make((uint32_t)mt);
    p.div_ntiles = fast_div_make((uint32_t)n_tiles);
    p.epi = epi;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // always behind the GEMM kernel just launched on this stream
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * mt / 8), 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = bf ? cudaLaunchKernelEx(&cfg, tile_splitk_reduce_kernel<true>, parts, C, p)
                             : cudaLaunchKernelEx(&cfg, tile_splitk_reduce_kernel<false>, parts, C, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    return W4A16_OK;
}

constexpr size_t kStageMaxBytes = 4u << 20;   // (w4a16_gemm_host)

// Can kernels reach all `bytes` of this host memory, by the same address?  Not if it is pageable, or page-locked in part: a
// copy call then deals with it or refuses it.  The driver tells the extent of one registration, so neighbouring ones are
// walked; 50 ns each.
bool device_reaches(const void* host, size_t bytes) {
    typedef CUresult (*GetAttributesFn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    static const GetAttributesFn get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &qr) != cudaSuccess || qr != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<GetAttributesFn>(f);
    }();
    if (get == nullptr || !aligned16(host)) return false;
    CUdeviceptr at = reinterpret_cast<CUdeviceptr>(host);
    const CUdeviceptr end = at + bytes;
    while (at < end) {
        unsigned int type = 0, managed = 0;
        CUdeviceptr dev = 0, start = 0;
        size_t size = 0;
        CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                      CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
        void* out[] = {&type, &managed, &dev, &start, &size};
        if (get(5, what, out, at) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed != 0 || dev != at || start > at || start + size <= at)
            return false;
        at = start + size;
    }
    return true;
}

int stage_activations(const void* host, void* dev, int n16, cudaStream_t st) {
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState* d = nullptr;
    const int rc = current_device(&d);
    if (rc != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    // Larger copies as single warps, so that the reads in flight are spread over more SMs: us a call, K = 11008 / N = 4096,
    // 128 / 32 threads: M = 8 (11,008 pieces of 16 bytes) 27.1 / 22.6, M = 16 34.4 / 25.5; M = 1 (1,376) 18.0 / 18.8, and
    // K = 4096 (512) 11.1 / 12.7.
    const int threads = n16 < 8192 ? kStageThreads : 32;
    const int want = (n16 + threads - 1) / threads;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(want < 4 * d->sm_count ? want : 4 * d->sm_count), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.stream = st;
    cfg.attrs = attr;
    // (behind a pack a plain launch: the GEMM that follows asks for packed weights while this kernel runs)
    cfg.numAttrs = d->order.may_overlap(reinterpret_cast<uintptr_t>(st), [&] { return capture_of(st); }) ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, stage_activations_kernel, static_cast<const uint4*>(host), static_cast<uint4*>(dev), n16) != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    return W4A16_OK;
}

// The body of every GEMM entry point; the caller holds g_mu.
int gemm_locked(const uint16_t* A, const void* Wq, const void* S, const void* Z, const uint16_t* bias, uint16_t* C,
                int M, int N, int K, int group, int split_k, int path, int flags, int act, w4a16_stream_t stream) {
    if (!flags_ok(flags)) return W4A16_ERR_SHAPE;
    const bool sym = (flags & W4A16_FLAG_SYMMETRIC) != 0, bf = (flags & W4A16_FLAG_BF16) != 0;
    if (!A || !Wq || !S || !C || (!sym && !Z)) return W4A16_ERR_NULL;
    int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (M < 1) return W4A16_ERR_SHAPE;
    if (act < W4A16_ACT_NONE || act > W4A16_ACT_SILU) return W4A16_ERR_SHAPE;
    if (!aligned16(A) || !aligned16(Wq) || !aligned16(S) || (!sym && !aligned16(Z)) || !aligned16(C))
        return W4A16_ERR_ALIGN;
    const int G = K / kGroup, sg = kGroup / group;
    if (split_k < 0 || split_k > G) return W4A16_ERR_SPLITK;
    if (path < W4A16_PATH_AUTO || path > W4A16_PATH_TILE) return W4A16_ERR_PATH;
    DeviceState* d = nullptr;
    if ((rc = current_device(&d)) != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;

    if (split_k > 65535) return W4A16_ERR_SPLITK;
    // registered workspace: [small-M tickets and reserve: the documented header][partial results]
    unsigned char* ws_body = d->ws ? static_cast<unsigned char*>(d->ws) + kWsFullHeaderBytes : nullptr;
    const size_t ws_body_bytes = d->ws_bytes > kWsFullHeaderBytes ? d->ws_bytes - kWsFullHeaderBytes : 0;
    const GemmPlan plan = gemm_plan(M, N, G, sg, split_k, path, bias != nullptr || act != W4A16_ACT_NONE, chip_of(d), ws_body_bytes);
    if (plan.rc != W4A16_OK) return plan.rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t* Zw = sym ? nullptr : static_cast<const uint32_t*>(Z);
    Epilogue epi;
    epi.bias = bias;
    epi.act = act;
    if (plan.kernel == W4A16_KERNEL_SIMPLE) {
        split_k = plan.split_simple;
        if (ws_body_bytes < plan.workspace) return W4A16_ERR_WORKSPACE;
        int mchunks = (M + kSimpleMB - 1) / kSimpleMB;
        float* partials = reinterpret_cast<float*>(ws_body);
        dim3 grid(N / kTileN, mchunks, split_k);
        if (bf)
            gemm_simple_kernel<true><<<grid, 64, 0, st>>>(A, static_cast<const uint32_t*>(Wq),
                                                          static_cast<const uint16_t*>(S), Zw, C, partials, M, N, K, G, sg,
                                                          split_k, epi);
        else
            gemm_simple_kernel<false><<<grid, 64, 0, st>>>(A, static_cast<const uint32_t*>(Wq),
                                                           static_cast<const uint16_t*>(S), Zw, C, partials, M, N, K, G, sg,
                                                           split_k, epi);
        if (cudaGetLastError() != cudaSuccess) return W4A16_ERR_CUDA;
        if (split_k > 1) {
            size_t MN = (size_t)M * N;
            const unsigned blocks = (unsigned)((MN + 255) / 256);
            if (bf) splitk_reduce_kernel<true><<<blocks, 256, 0, st>>>(partials, C, MN, N, split_k, epi);
            else splitk_reduce_kernel<false><<<blocks, 256, 0, st>>>(partials, C, MN, N, split_k, epi);
            if (cudaGetLastError() != cudaSuccess) return W4A16_ERR_CUDA;
        }
        return W4A16_OK;
    }

    if (plan.kernel == W4A16_KERNEL_MID64 || plan.kernel == W4A16_KERNEL_MID128) {
        const MidGeom& g = plan.wide.mid;
        if (g.smem_bytes > d->max_smem_optin) return W4A16_ERR_PATH;
        if (ws_body_bytes < plan.workspace) return W4A16_ERR_WORKSPACE;
        CUtensorMap tmap;
        if (!make_act_tensor_map(&tmap, A, M, K, g.mt, mid_stage_k(g.mtc))) return W4A16_ERR_CUDA;
        MidParams p;
        p.Wq = static_cast<const uint32_t*>(Wq);
        p.S = static_cast<const uint16_t*>(S);
        p.Z = Zw;
        p.C = C;
        p.ws = reinterpret_cast<float*>(ws_body);
        p.M = M; p.N = N; p.K = K; p.G = G;
        p.n_tiles = g.n_tiles;
        p.mt = g.mt;
        p.split_k = g.split_k;
        p.nchunks = g.nchunks;
        p.wstages = g.wstages;
        p.cluster = g.cluster ? 1 : 0;
        p.div_split = fast_div_make((uint32_t)g.split_k);
        p.div_ntiles = fast_div_make((uint32_t)g.n_tiles);
        p.slice_base = G / g.split_k;
        p.slice_rem = G % g.split_k;
        p.epi = epi;
        MidKernel kern = bf ? mid_kernel_bf16(g.mtc, sg, sym) : mid_kernel_f16(g.mtc, sg, sym);
        bool& attr_set = d->mid_attr_set[g.mtc <= 64 ? 0 : 1][log2_sg(sg)][bf ? 1 : 0][sym ? 1 : 0];
        if (!attr_set) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, d->max_smem_optin) != cudaSuccess) {
                cudaGetLastError();
                return W4A16_ERR_CUDA;
            }
            attr_set = true;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g.ctas, 1, 1);
        cfg.blockDim = dim3(kMidThreads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)g.smem_bytes;
        cfg.stream = st;
        if (!launch_gemm_kernel(d, cfg, g.cluster ? g.split_k : 1, kern, tmap, p)) {   // (the slices of a tile are one cluster)
            if (g.cluster) {   // (see the warp-MMA kernel below)
                d->cluster_ok = false;
                return gemm_locked(A, Wq, S, Z, bias, C, M, N, K, group, split_k, path, flags, act, stream);
            }
            return W4A16_ERR_CUDA;
        }
        if (g.split_k > 1 && !g.cluster)
            return launch_tile_reduce(p.ws, C, M, N, G, g.mt, g.n_tiles, g.tiles, g.split_k, g.nchunks, bf, epi, st);
        return W4A16_OK;
    }

    if (plan.kernel == W4A16_KERNEL_TILE) {
        const TileGeom& g = plan.wide.tile;
        if (g.smem_bytes > d->max_smem_optin) return W4A16_ERR_PATH;
        if (ws_body_bytes < plan.workspace) return W4A16_ERR_WORKSPACE;
        CUtensorMap tmap;
        if (!make_act_tensor_map(&tmap, A, M, K, g.mt, kTileStageK)) return W4A16_ERR_CUDA;
        TileParams p;
        p.Wq = static_cast<const uint32_t*>(Wq);
        p.S = static_cast<const uint16_t*>(S);
        p.Z = Zw;
        p.C = C;
        p.ws = reinterpret_cast<float*>(ws_body);
        p.M = M; p.N = N; p.K = K; p.G = G;
        p.mt = g.mt;
        p.n_tiles = g.n_tiles;
        p.m_tiles = g.m_tiles;
        p.split_k = g.split_k;
        p.nchunks = g.nchunks;
        p.stages = g.stages;
        tile_fill_chunk_math(p);
        p.epi = epi;
        // Partial tiles are summed (and get the optional bias / activation) by a second, GPU-wide kernel behind this one
        // (kernels_basic.cuh).  Measured (us, in the kernel / second kernel), M = 256: K = 10240 / N = 4608 (four slices)
        // 31.9 / 24.6, K = 16384 / N = 4096 39.2 / 32.9, K = N = 8192 (two slices) 34.1 / 33.3.
        const bool has_epi = g.split_k < 2 && (bias != nullptr || act != W4A16_ACT_NONE);
        TileKernel kern = tile_kernel(sg, bf, sym, has_epi);
        bool& attr_set = d->tile_attr_set[log2_sg(sg)][bf ? 1 : 0][sym ? 1 : 0][has_epi ? 1 : 0];
        if (!attr_set) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, d->max_smem_optin) !=
                cudaSuccess) {
                cudaGetLastError();
                return W4A16_ERR_CUDA;
            }
            attr_set = true;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g.ctas, 1, 1);
        cfg.blockDim = dim3(kTileThreads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)g.smem_bytes;
        cfg.stream = st;
        if (!launch_gemm_kernel(d, cfg, 1, kern, tmap, p)) return W4A16_ERR_CUDA;
        if (g.split_k != 1)
            return launch_tile_reduce(p.ws, C, M, N, G, g.mt, g.n_tiles, g.tiles, g.split_k, g.nchunks, bf, epi, st);
        return W4A16_OK;
    }

    // W4A16_KERNEL_DECODE
    const DecodeGeom& g = plan.dec;
    if (g.smem_bytes > d->max_smem_optin) return W4A16_ERR_PATH;
    if (ws_body_bytes < plan.workspace) return W4A16_ERR_WORKSPACE;
    DecodeParams p;
    p.A = A;
    p.Wq = static_cast<const uint32_t*>(Wq);
    p.S = static_cast<const uint16_t*>(S);
    p.Z = Zw;
    p.C = C;
    p.ws = reinterpret_cast<float*>(ws_body);
    p.tickets = static_cast<int*>(d->ws);
    p.M = M; p.N = N; p.K = K; p.G = G; p.T = N / kTileN;
    p.split_k = g.split_k;
    p.nchunks = g.nchunks;
    p.stages = g.stages;
    p.stage_bytes = g.stage_bytes;
    p.prefetch = g.prefetch;
    decode_fill_chunk_math(p);
    p.epi = epi;
    CUtensorMap tmap_a;
    if (g.a_box) {
        if (!make_decode_tensor_map(&tmap_a, A, M, K, g.mb)) return W4A16_ERR_CUDA;
    } else {
        memset(&tmap_a, 0, sizeof(tmap_a));
    }
    DecodeKernel kern = decode_kernel(g.mb, g.cluster, sg, bf, sym, g.a_box);
    bool& attr_set = d->decode_attr_set[g.mb][g.cluster ? 1 : 0][log2_sg(sg)][bf ? 1 : 0][sym ? 1 : 0][g.a_box ? 1 : 0];
    if (!attr_set) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, d->max_smem_optin) !=
            cudaSuccess) {
            cudaGetLastError();
            return W4A16_ERR_CUDA;
        }
        attr_set = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.ctas, g.mchunks, 1);
    cfg.blockDim = dim3(kDecThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)g.smem_bytes;
    cfg.stream = st;
    if (!launch_gemm_kernel(d, cfg, g.cluster ? g.split_k : 1, kern, tmap_a, p)) {   // (the split_k CTAs of a column tile are one cluster)
        if (g.cluster) {
            // the device would not place the clusters: from now on the workspace exchange (and the path
            // rule that goes with it), starting with this call
            d->cluster_ok = false;
            return gemm_locked(A, Wq, S, Z, bias, C, M, N, K, group, split_k, path, flags, act, stream);
        }
        return W4A16_ERR_CUDA;
    }
    return W4A16_OK;
}
}  // namespace

extern "C" {

int w4a16_gemm_fmt(const uint16_t* A, const void* Wq, const void* S, const void* Z, const uint16_t* bias, uint16_t* C,
                   int M, int N, int K, int group, int split_k, int path, int flags, int act, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (bias != nullptr && (reinterpret_cast<uintptr_t>(bias) & 1u)) return W4A16_ERR_ALIGN;
    return gemm_locked(A, Wq, S, Z, bias, C, M, N, K, group, split_k, path, flags, act, stream);
}

int w4a16_gemm_ex(const uint16_t* A, const void* Wq, const void* S, const void* Z, uint16_t* C, int M, int N, int K,
                  int group, int split_k, int path, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!Z) return W4A16_ERR_NULL;
    return gemm_locked(A, Wq, S, Z, nullptr, C, M, N, K, group, split_k, path, 0, W4A16_ACT_NONE, stream);
}

int w4a16_gemm(const uint16_t* A, const void* Wq, const void* S, const void* Z, uint16_t* C, int M, int N, int K,
               int group, int split_k, w4a16_stream_t stream) {
    return w4a16_gemm_ex(A, Wq, S, Z, C, M, N, K, group, split_k, W4A16_PATH_AUTO, stream);
}

int w4a16_gemm_host(const uint16_t* A_host, uint16_t* A_dev, const void* Wq, const void* S, const void* Z,
                    uint16_t* C_dev, uint16_t* C_host, int M, int N, int K, int group, int split_k,
                    w4a16_stream_t stream) {
    if (!A_host || !A_dev || !C_dev || !C_host) return W4A16_ERR_NULL;
    if (M < 1 || K < 1 || N < 1) return W4A16_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // Page-locked host memory that the device can address: the kernels read and write it themselves (each element of C is
    // written once, by whoever finishes its sum), which saves two copies, their runtime calls and the waits between copy
    // engine and SMs.  Anything else goes through the staging buffers and the copy engine; so do activations of more than
    // kStageMaxBytes.  us a call on one stream, K = 11008 / N = 4096, copy engine / kernel: M = 1 25.4 / 17.7, 8 34.9 / 22.4,
    // 64 68 / 55, 190 143 / 138, 256 182 / 182: bound by PCIe there, so the SMs are left alone.
    const size_t a_bytes = (size_t)M * K * 2;
    if (a_bytes <= kStageMaxBytes && a_bytes % 16 == 0 && aligned16(A_dev) && device_reaches(A_host, a_bytes)) {
        const int rc = stage_activations(A_host, A_dev, (int)(a_bytes / 16), st);
        if (rc != W4A16_OK) return rc;
    } else if (cudaMemcpyAsync(A_dev, A_host, a_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    const bool c_direct = device_reaches(C_host, (size_t)M * N * 2);
    int rc = w4a16_gemm(A_dev, Wq, S, Z, c_direct ? C_host : C_dev, M, N, K, group, split_k, stream);
    if (rc != W4A16_OK) return rc;
    if (!c_direct && cudaMemcpyAsync(C_host, C_dev, (size_t)M * N * 2, cudaMemcpyDeviceToHost, st) != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    return W4A16_OK;
}

int w4a16_gemm_static_ws(const uint16_t* A, const void* Wq, const void* S, const void* Z, uint16_t* C, int M, int N,
                         int K, int group, int split_k, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!A || !Wq || !S || !Z || !C) return W4A16_ERR_NULL;
    int rc = check_weight_shape(N, K, group);
    if (rc != W4A16_OK) return rc;
    if (M < 1) return W4A16_ERR_SHAPE;
    if (!aligned16(A) || !aligned16(Wq) || !aligned16(S) || !aligned16(Z) || !aligned16(C)) return W4A16_ERR_ALIGN;
    const int G = K / kGroup, sg = kGroup / group;
    if (split_k < 0 || split_k > G) return W4A16_ERR_SPLITK;
    DeviceState* d = nullptr;
    if ((rc = current_device(&d)) != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return W4A16_ERR_CUDA;

    DecodeGeom g = decode_geom(M, N, G, split_k, without_clusters(chip_of(d)), sg);   // no clusters here: this entry point keeps the path it was built with
    // (balanced chunks give way to whole tiles, as in gemm_plan)
    if (g.split_k == 0 && kWsHeaderBytes + decode_partial_bytes(g) > (size_t)W4A16_STATIC_WS_BYTES)
        g = decode_geom(M, N, G, 1, without_clusters(chip_of(d)), sg);
    if (!decode_runs(g, N)) return W4A16_ERR_PATH;
    if (g.smem_bytes > d->max_smem_optin) return W4A16_ERR_PATH;
    // the whole scratch need of this shape must fit the built-in array, or nothing is launched (a schedule of
    // whole tiles, split_k == 1, leaves no partial tiles and draws no tickets: it needs none)
    if (g.split_k != 1 && kWsHeaderBytes + decode_partial_bytes(g) > (size_t)W4A16_STATIC_WS_BYTES)
        return W4A16_ERR_WORKSPACE;

    // first call on this device: resolve the array's device address (this device is current)
    if (g_static_ws_addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_ws) != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return W4A16_ERR_CUDA;
        }
        g_static_ws_addr[dev] = static_cast<unsigned char*>(p);
    }
    unsigned char* ws = g_static_ws_addr[dev];
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the array keeps whatever the previous call left; the ticket counters must start at zero
    if (cudaMemsetAsync(ws, 0, kWsHeaderBytes, st) != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    DecodeParams p;
    p.A = A;
    p.Wq = static_cast<const uint32_t*>(Wq);
    p.S = static_cast<const uint16_t*>(S);
    p.Z = static_cast<const uint32_t*>(Z);
    p.C = C;
    p.ws = reinterpret_cast<float*>(ws + kWsHeaderBytes);
    p.tickets = reinterpret_cast<int*>(ws);
    p.M = M; p.N = N; p.K = K; p.G = G; p.T = N / kTileN;
    p.split_k = g.split_k;
    p.nchunks = g.nchunks;
    p.stages = g.stages;
    p.stage_bytes = g.stage_bytes;
    p.prefetch = g.prefetch;
    decode_fill_chunk_math(p);
    CUtensorMap tmap_a;
    if (g.a_box) {
        if (!make_decode_tensor_map(&tmap_a, A, M, K, g.mb)) return W4A16_ERR_CUDA;
    } else {
        memset(&tmap_a, 0, sizeof(tmap_a));
    }
    p.epi.bias = nullptr;
    p.epi.act = kActNone;
    DecodeKernel kern = decode_kernel(g.mb, false, sg, false, false, g.a_box);
    bool& attr_set = d->decode_attr_set[g.mb][0][log2_sg(sg)][0][0][g.a_box ? 1 : 0];
    if (!attr_set) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, d->max_smem_optin) !=
            cudaSuccess) {
            cudaGetLastError();
            return W4A16_ERR_CUDA;
        }
        attr_set = true;
    }
    kern<<<dim3(g.ctas, g.mchunks, 1), kDecThreads, g.smem_bytes, st>>>(tmap_a, p);
    return cudaGetLastError() == cudaSuccess ? W4A16_OK : W4A16_ERR_CUDA;
}

int w4a16_selftest_wait_timeout(unsigned limit_us, w4a16_stream_t stream) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (limit_us < 1 || limit_us > 100000) return W4A16_ERR_SHAPE;
    DeviceState* d = nullptr;
    int rc = current_device(&d);
    if (rc != W4A16_OK) return rc;
    if (!d->is_sm100) return W4A16_ERR_ARCH;
    wait_timeout_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>((unsigned long long)limit_us * 1000ull,
                                                                               nullptr);
    return cudaGetLastError() == cudaSuccess ? W4A16_OK : W4A16_ERR_CUDA;
}

int w4a16_device_status(int* status_out) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!status_out) return W4A16_ERR_NULL;
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return W4A16_ERR_CUDA;
    }
    // every translation unit that holds kernels has a status word of its own
    const int words[] = {status_take_this_unit(),     status_take_decode_f16(),   status_take_decode_bf16(),
                         status_take_mid_f16(),        status_take_mid_bf16(),
                         status_take_tile_f16_sg1(),  status_take_tile_f16_sg2(), status_take_tile_f16_sg4(),
                         status_take_tile_bf16_sg1(), status_take_tile_bf16_sg2(), status_take_tile_bf16_sg4()};
    int v = 0;
    for (int w : words) {
        if (w < 0) return W4A16_ERR_CUDA;
        v |= w;
    }
    *status_out = v;
    if (v != 0) {
        // a kernel that gave up returned before it drew its tickets: the counters of the registered
        // workspace may be non-zero, and the next call would take a tile for complete too early
        DeviceState* d = nullptr;
        if (current_device(&d) == W4A16_OK && d->ws != nullptr &&
            (cudaMemset(d->ws, 0, kWsFullHeaderBytes) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)) {
            cudaGetLastError();
            return W4A16_ERR_CUDA;
        }
    }
    return v == 0 ? W4A16_OK : W4A16_ERR_DEVICE_STATUS;
}

}  // extern "C"
