// Launch shapes of the CPDP kernels: how many blocks a launch gets and, per
// reconcile variant, the rows per load chunk, the resident blocks per SM it is
// compiled for and when it loads the anchor and velocity. Kept apart from the C
// ABI's host code because, with the kernels in cpdp_kernels.cuh, these decide
// what each launch does on the GPU.
#pragma once

#include <cstdint>
#include <type_traits>

#include "cpdp_kernels.cuh"

namespace cpdp {

constexpr int kLocalUnroll = 2;  // float4 vectors per thread per iteration in the local step

// The local step's vectors per thread run along the warp (each warp streams
// 1 KB of every array) for AdamW with bf16 gradients: 7,157 against 7,035 GB/s
// (ViT-S N, W = 8, back-to-back launches; 7,118 against 7,002 at the ResNet-50
// N). The other variants measured the same or up to 1 % slower that way and
// keep a block-wide spacing.
template <int OPT, typename G>
struct LocalWarpRuns {
    static constexpr bool value = OPT == kOptAdamW && !std::is_same<G, float>::value;
};

// The local step's gradients leave L2 first (SGD) while the state (8 bytes an
// element with either gradient type) is larger than L2 keeps beside them and
// small enough for a part that matters to stay from one step to the next.
// Periods of 2 and 4 steps, 1 to 16 workers, time without / with, geometric
// mean (and the worst), float32 and bf16 gradients: W * N = 4 M elements 1.005
// (0.965) and 0.988 (0.966), 5.4 M 1.04 (0.97) and 1.00 (0.97), 6.6 M 1.07 (1.00)
// and 1.016 (0.99), 8.5 M 1.07 (1.00) and 1.04 (1.00), 13 M 1.03 and 1.03, 20 M 1.014
// and 1.010, 32 M 1.004 and 1.004, 45 M 0.998 and 0.997; 95 M (ResNet-50, 4 workers)
// 0.99. AdamW gains 0.6 % at best; the reconcile, which reads fewer gradients per
// state byte, 1 % at best.
constexpr int64_t kOnceMinElements = 6'000'000, kOnceMaxElements = int64_t(1) << 25;

// Whether a context's launches alternate their walk direction (walk_block):
// not where a sync step's arrays (replicas, optimizer states, gradients; for
// CPDP the anchor and velocity too) are few enough for L2 to keep them from one
// launch to the next whatever else it holds. There a run of sync steps loses by
// it, as a block's columns move to another SM each time (the likely cost: lines
// that come from the other die's half of L2). N a multiple of 4, one direction
// over alternating, geometric means over the variants and 1 to 64 workers, sync
// steps in a row on one state / periods of 2 and 4 steps: 1 to 10 MB 0.95-0.98 /
// 0.998-1.01, 24 MB 0.992 / 0.998, 30 to 60 MB 0.995-1.006 / 0.996-1.001, 72 MB 0.986 /
// 0.996, 83 MB 0.994 / 1.009, 91 MB 1.036 / 1.034, 103 MB 1.07 / 1.07, 118 MB 1.13 / 1.10,
// 149 MB 1.17 / 1.13. Where several states share L2 it gains from less: three of
// 2 workers and 2^20 columns in turn (34 MB a step) take 13.77 us a period walking
// one way and 13.61 alternating.
constexpr int64_t kAlternateMinBytes = 30'000'000;
inline bool walks_alternate(int64_t W, int64_t N, bool adamw, bool cpdp_method, int grad_bytes) {
    return W * N * ((adamw ? 12 : 8) + grad_bytes) + (cpdp_method ? 8 * N : 0) >= kAlternateMinBytes;
}
constexpr int64_t kMaxGrid = 0x7fffffff;

// Blocks for `work_items` items at `per_block` items per block (kernels loop
// over any remainder beyond the grid limit).
inline unsigned grid_for(int64_t work_items, int64_t per_block) {
    int64_t blocks = (work_items + per_block - 1) / per_block;
    if (blocks < 1) blocks = 1;
    if (blocks > kMaxGrid) blocks = kMaxGrid;
    return static_cast<unsigned>(blocks);
}

// Threads per block of a reconcile's column kernels (they are compiled for up
// to kThreads, and for the registers of that many). An SM holds the same warps
// either way, but with few blocks a small one leaves fewer SMs with one block
// more than the others, and its barrier-free warps retire one by one: 64
// threads against 256, time ratio, at N = 20,000 to 320,000 1.00-1.15 (W = 8,
// N = 60,000 3.9 -> 3.4 us), 700,000 1.00-1.10, 1 to 3 million 1.00-1.05. Above
// 4 million columns the two are within 0.4 % (64 slower), except where they
// favour 64: state-reconciling AdamW (ViT-S, W = 8 1.010, W = 32 1.027) and CPDP
// at odd N (W = 4, 23.7 M: bf16 SGD 1.014, AdamW 1.012).
// The GPU starts about one block per ns, and a block shorter than that bounds
// the launch, so past kThreadsSmallColumns a block gets at least
// kBlockElements elements of each array (rows times columns: 9 to 25 KB in
// all). State in L2, sync step, time ratio to 256 threads, geometric means
// (and the worst) over the variants: W = 1, 4 columns per thread, N = 790,000
// 64 threads 0.90 (0.70), 1.8 M 0.72 (0.53); W = 2, 1.8 M 0.96 (0.76), 128
// threads 1.02 (0.98); W = 3 64 threads 1.02-1.05 from 490,000 on. One worker
// at N = 2^26, DDP SGD: 170 us, with 64 threads 264.
constexpr int kThreadsSmall = 64;
constexpr int64_t kThreadsSmallColumns = 65'536;
constexpr int kBlockElements = 768;
inline int reconcile_threads(int method, int opt, bool state_sync, int W, int64_t N, int columns_per_thread) {
    const bool always = (opt == kOptAdamW && state_sync) || (method == kMethodCPDP && (N & 1) != 0);
    if (!always && N > int64_t(1) << 22) return kThreads;
    int threads = kThreadsSmall;
    if (N > kThreadsSmallColumns)
        while (threads < kThreads && int64_t(threads) * columns_per_thread * W < kBlockElements) threads *= 2;
    return threads;
}

// Rows per load chunk of the vectorised reconcile, the resident blocks per SM it
// is compiled for (3 blocks of 256 threads: 80 registers; 4 blocks: 64),
// whether theta_ref and v are loaded after the rows (late) to free registers,
// and whether its offsets are 32-bit where the sizes allow (narrow), which
// frees more. Each entry is the fastest measured (ResNet-50 or ViT-S shape,
// W = 8, TB/s).
// SGD, float32 gradients: 4 rows, 3 blocks, early (7.00; late 6.95; narrow
// offsets make no difference).
// SGD, bf16: 2 rows, 4 blocks, late (6.84; 3 rows / 3 blocks early 6.73; narrow
// 0.8 % slower).
// SGD with state reconciliation (two more running sums): 1 row, 4 blocks, late
// (7.00; early 6.97; 2 rows / 3 blocks 6.25; narrow 1 % slower).
// AdamW carries a third state row per worker. With 64-bit offsets its 2-row
// shape at 4 blocks spilled 24-32 bytes; narrow offsets remove the spill:
// 2 rows, 4 blocks, late, narrow for every AdamW variant (CPDP and DDP without
// state reconciliation now take the gradient-chunk shapes below). Isolated launches at
// the ViT-S N (GB/s, against the best 64-bit shape): bf16 gradients 6,818
// (6,605), float32 6,785 (6,730 at 1 row, early), with state reconciliation
// 6,541 (6,467, bf16) and 6,427 (6,337, float32); at W = 16 +2 to +3 %.
template <int OPT, typename G, bool SS>
struct ReconcileShape {
    static constexpr int rows = 2, min_blocks = 4;
    static constexpr bool late = true, narrow = true;
};
template <>
struct ReconcileShape<kOptSGD, float, false> {
    static constexpr int rows = 4, min_blocks = 3;
    static constexpr bool late = false, narrow = false;
};
template <>
struct ReconcileShape<kOptSGD, bf16_bits, false> {
    static constexpr int rows = 2, min_blocks = 4;
    static constexpr bool late = true, narrow = false;
};
template <typename G>
struct ReconcileShape<kOptSGD, G, true> {
    static constexpr int rows = 1, min_blocks = 4;
    static constexpr bool late = true, narrow = false;
};

// Two workers: 2-row chunks fill every slot, and the freed registers allow 4
// resident blocks. Measured at N = 2^26 (TB/s, against the shapes above):
// SGD float32 7.03 (6.67), AdamW float32 6.79 late (6.43), SGD with state
// reconciliation 7.00 early (6.34), AdamW with state reconciliation 5.96 late
// (5.64); the bf16 SGD and AdamW shapes above already use 2 rows.
template <int OPT, typename G, bool SS>
struct ReconcileShapeW2 {
    static constexpr int rows = 2, min_blocks = 4;
    static constexpr bool late = OPT == kOptAdamW || (!SS && !std::is_same<G, float>::value);
    static constexpr bool narrow = OPT == kOptAdamW;
};

// Three to six workers: the general shapes, except SGD with bf16 gradients,
// where 3-row chunks at 3 blocks with early anchor loads measured fastest
// (N = 2^25, TB/s against 2 rows: W = 3 6.75 / 6.14, W = 4 6.63 / 6.55,
// W = 5 6.88 / 6.38, W = 6 6.95 / 6.64; from W = 7 on the 2-row shape is as
// fast or faster).
template <int OPT, typename G, bool SS>
struct ReconcileShapeFew : ReconcileShape<OPT, G, SS> {};
template <>
struct ReconcileShapeFew<kOptSGD, bf16_bits, false> {
    static constexpr int rows = 3, min_blocks = 3;
    static constexpr bool late = false, narrow = false;
};

// Three-row chunks at 4 resident blocks (late anchor, narrow offsets) for
// worker counts they divide or nearly divide, where they measured at least 2 %
// faster than the shapes above (20 back-to-back launches at N = 2^25, GB/s
// against the shape used before). W = 3: CPDP SGD bf16 6,593 (6,376), CPDP
// SGD with state reconciliation f32 6,562 (5,923) and bf16 6,187 (5,594), DDP
// SGD f32 7,113 (6,680); CPDP AdamW bf16 also measured faster there (6,211
// against 6,096) and now takes the gradient-chunk shape below. W = 5: DDP SGD
// f32 7,081 (6,765). W = 6: CPDP SGD with state reconciliation f32 6,989 (6,867)
// and bf16 6,768 (6,610), DDP SGD f32 7,090 (6,949). Through the library
// (N = 2^25, K = 2, sync-step GB/s) the W = 3 entries gained 1.5-12 % and the
// W = 5 DDP entry 2.6 %; DDP AdamW bf16 at W = 3, which the launch-by-launch
// probe also favoured, lost 2.9 % there and keeps the one-pass kernel.
template <int METHOD, int OPT, bool SS, typename G, int W>
struct ReconcileThreeRows {
    static constexpr bool use = false;
    static constexpr int rows = 3, min_blocks = 4;
    static constexpr bool late = true, narrow = true;
};
#define CPDP_THREE_ROWS(M, O, SS, G, W)                      \
    template <>                                              \
    struct ReconcileThreeRows<M, O, SS, G, W> {              \
        static constexpr bool use = true;                    \
        static constexpr int rows = 3, min_blocks = 4;       \
        static constexpr bool late = true, narrow = true;    \
    };
CPDP_THREE_ROWS(kMethodCPDP, kOptSGD, false, bf16_bits, 3)
CPDP_THREE_ROWS(kMethodCPDP, kOptSGD, true, float, 3)
CPDP_THREE_ROWS(kMethodCPDP, kOptSGD, true, bf16_bits, 3)
CPDP_THREE_ROWS(kMethodDDP, kOptSGD, false, float, 3)
CPDP_THREE_ROWS(kMethodDDP, kOptSGD, false, float, 5)
CPDP_THREE_ROWS(kMethodCPDP, kOptSGD, true, float, 6)
CPDP_THREE_ROWS(kMethodCPDP, kOptSGD, true, bf16_bits, 6)
CPDP_THREE_ROWS(kMethodDDP, kOptSGD, false, float, 6)
#undef CPDP_THREE_ROWS

// Gradient-row chunks, for AdamW and for SGD with bf16 gradients (CPDP and
// DDP without state reconciliation; CPDP AdamW with state reconciliation at 3
// to 5 workers): the gradient rows in chunks of 8 (bf16) or 4 (float32) held
// as raw words, the first state chunk loaded together with the first gradient
// chunk, then the state rows in chunks (narrow offsets, late anchor). The
// results are bit-identical to those of the other shapes. Isolated launches
// at the ViT-S N (W = 32 at N / 2), GB/s against the shape used before:
// AdamW from 2 workers (CPDP; float32 gradients at W = 2 keep the one-pass
// kernel, within 0.4 %; DDP from 5, where the one-pass kernel does not take
// W = 2-4), 2-row state chunks at 4 blocks up to 7 workers and 3-row chunks at
// 3 blocks from 8. CPDP bf16 gradients W = 2 (N = 2^26) 6,987 (6,772; one-pass
// 6,765), W = 3 6,922 (6,600, three-row shape), W = 4 7,008 (6,782), W = 5
// 6,963 (6,600), W = 6 6,965 (6,809),
// W = 7 6,967 (6,904), W = 8 6,979 (6,931; 2-row 6,966), W = 12 6,941 (6,859;
// 2-row 6,911), W = 16 6,917 (6,852), W = 32 6,838 (6,791); float32 gradients
// W = 3 6,997 (6,569), W = 4 7,067 (6,934), W = 5 6,979 (6,755), W = 6 6,998
// (6,928), W = 7 7,004 (6,882), W = 8 7,021 (6,926; 2-row 7,011), W = 12 6,995
// (6,888), W = 16 6,948 (6,853), W = 32 6,899 (6,833); DDP +1 to +6 % at
// W = 5-16. DDP at W = 3-4 measured within 1.3 % of its one-pass kernel.
// AdamW with state reconciliation (CPDP), 2-row chunks at 4 blocks for 3 to 5
// workers: bf16 gradients W = 3 6,496 (6,155), W = 4 6,758 (6,561), W = 5
// 6,665 (6,380); float32 W = 3 6,729 (6,344), W = 4 6,871 (6,777), W = 5 6,703
// (6,570); from W = 6 the shapes above measured as fast or faster.
// SGD with bf16 gradients, 4-row state chunks at 3 blocks, CPDP from 7
// workers (W = 7 7,007 (6,773), W = 8 7,031 (6,913), W = 12 6,976 (6,783),
// W = 16 6,969 (6,886), W = 32 6,891 (6,847); at W = 5-6 within 0.3 %), DDP
// from 5 (W = 5 +5.8 %, W = 6 +1.6 %, W = 8 +4.5 %, W = 16 +5.4 %). With
// float32 gradients the SGD shapes gain at most 0.2 % (CPDP) and 0.6 % (DDP),
// and with state reconciliation nothing, so those keep their shapes.
// The same row traffic in a plain local step walked column by column (no
// sums, no dependency between the rows) peaks at 6,999 GB/s at W = 8 (4-row
// chunks, 2 blocks; 6,930 at 2 rows and 4 blocks), against 7,155 for the flat
// local step: the W = 8 AdamW shape is within 0.3 % of that floor.
// MANY selects the shape from kGradChunksManyWorkers workers on; the other
// one covers min_workers to max_workers (below kGradChunksManyWorkers).
constexpr int kGradChunksManyWorkers = 8;
template <int METHOD, int OPT, bool SS, typename G, bool MANY>
struct ReconcileGradChunks {
    static constexpr bool use = false;
};
template <int METHOD, typename G, bool MANY>
struct ReconcileGradChunks<METHOD, kOptAdamW, false, G, MANY> {
    static constexpr bool use = METHOD != kMethodLocalSGD;
    static constexpr int min_workers = METHOD == kMethodDDP ? 5 : 2, max_workers = kGradChunksManyWorkers - 1;
    static constexpr int rows = MANY ? 3 : 2, min_blocks = MANY ? 3 : 4;
    static constexpr int grad_rows = std::is_same<G, float>::value ? 4 : 8;
    static constexpr bool late = true, narrow = true, overlap = true;
};
template <typename G, bool MANY>
struct ReconcileGradChunks<kMethodCPDP, kOptAdamW, true, G, MANY> {
    static constexpr bool use = !MANY;
    static constexpr int min_workers = 3, max_workers = 5;
    static constexpr int rows = 2, min_blocks = 4, grad_rows = std::is_same<G, float>::value ? 4 : 8;
    static constexpr bool late = true, narrow = true, overlap = true;
};
template <int METHOD, bool MANY>
struct ReconcileGradChunks<METHOD, kOptSGD, false, bf16_bits, MANY> {
    static constexpr bool use = METHOD != kMethodLocalSGD;
    static constexpr int min_workers = METHOD == kMethodDDP ? 5 : 7, max_workers = kGradChunksManyWorkers - 1;
    static constexpr int rows = 4, min_blocks = 3, grad_rows = 8;
    static constexpr bool late = true, narrow = true, overlap = true;
};

// Gradient rows per chunk and overlap of a shape: its own where it states
// them, else the state-row chunk and no overlap.
template <typename S, typename = void>
struct GradChunkOf {
    static constexpr int rows = S::rows;
    static constexpr bool overlap = false;
};
template <typename S>
struct GradChunkOf<S, std::void_t<decltype(S::grad_rows)>> {
    static constexpr int rows = S::grad_rows;
    static constexpr bool overlap = S::overlap;
};

// N not a multiple of 4 (reconcile_scalar_kernel): V = 2 elements per load where
// N is even, else 1. The row bytes are the same as for any N; what a
// one-column-per-thread kernel lacks is bytes in flight per thread, and past
// that the narrow loads cost instructions and, at odd N, a fifth 32-byte
// sector per 128-byte row segment. So a thread owns 4 columns in 4 / V loads
// (a warp covers kRaggedColumns of a row) and loads rows in chunks as the
// vector kernel does. Sync-step GB/s at N = 23.7 M, W = 8, before (one column
// per thread, one row at a time) and now, N odd / N = 2 mod 4: CPDP SGD f32
// 5,264 -> 6,872 / 5,256 -> 7,039; SGD bf16 5,023 -> 6,422 / 5,000 -> 6,979;
// AdamW f32 5,499 -> 6,725 / 5,488 -> 6,952; AdamW bf16 5,306 -> 6,493 /
// 5,302 -> 6,938; with state reconciliation 6,040-6,504 -> 6,568-6,757 (SGD)
// and 5,446-5,687 -> 6,430-6,909 (AdamW). Eight shapes were swept at W = 1 to
// 16: gradient chunks overlapped with the first state chunk win where the loads
// are pairs, and for SGD f32 at odd N; the other odd-N variants are
// short of registers and take plain 2-row or 1-row chunks.
constexpr int kRaggedColumns = 128;
template <int V, int OPT, bool SS, typename G, bool MANY>
struct RaggedShape {
    static constexpr bool f32 = std::is_same<G, float>::value;
    static constexpr bool overlap = V == 2 ? !(SS && OPT == kOptAdamW) : !SS && OPT == kOptSGD && f32;
    static constexpr bool three = overlap && OPT == kOptAdamW && MANY;
    static constexpr int rows = three ? 3 : V == 1 && SS && (OPT == kOptAdamW || f32) ? 1 : 2;
    static constexpr int min_blocks = three ? 3 : 4;
    static constexpr int grad_rows = !overlap ? rows : f32 ? 4 : 8;
    static constexpr bool late = true;
};

// Few columns: at 4 columns per thread N = 300,000 leaves an SM half of the warps
// it can hold, so up to ragged_narrow_columns a thread owns one load's columns
// instead and 4-row chunks keep it busy (W = 8, N = 100,001, us, one column and
// one row at a time / 4 columns / this: CPDP SGD f32 5.15 / 5.87 / 4.29;
// N = 300,002 AdamW bf16 15.1 / 16.2 / 12.7). The lines are where the two cross
// (geometric means over method and gradient type, time of a kernel with one
// column and one row per thread over: this shape, 4 columns). SGD, odd N, sync
// steps in a row: W = 3 to 6 N = 200,000 to 260,000 1.02-1.12, 1.08-1.17, 260,000 to
// 330,000 0.95-1.09, 1.04-1.15, 330,000 to 430,000 1.07-1.26, 1.07-1.14; in periods of 2
// and 4 steps (CPDP and LocalSGD, W = 3 to 16) this shape has 0.97-1.09 from 229,000 to
// 249,000, 4 columns 0.77-0.96 from 259,000 to 325,000 and 1.0-1.1 above. W = 2 from
// 260,000 0.99, 1.10. AdamW, odd N, W = 3 to 6, 260,000 to 330,000 0.95-1.07, 0.84-0.93,
// 330,000 to 430,000 1.02-1.12, 0.90-0.98, W = 3, 410,000, periods 0.93, 0.99.
// State-reconciling SGD stores nothing inside its row loop and holds little
// per column, so 1-row chunks at 8 blocks of single columns are as good as any
// up to 700,000 odd columns below 24 workers (W = 8, N = 300,001 10.4 us; at 6
// blocks 12.0; W = 141, N = 351,435 249, the wide shape 209) and beat pairs up to
// kRaggedSinglesColumns even ones. LocalSGD with bf16 gradients loads a
// gradient row with each state row and wants 4 of them in flight (against one
// column and one row per thread, to 60,000, 150,000, 205,000, 560,000 columns,
// W = 6 to 14: 1-row chunks 0.90 0.94 0.93 1.00, 4-row chunks at 5 blocks 1.06 0.96
// 1.23 1.00). State-reconciling AdamW is short of registers for the overlapped
// chunk and takes 5 blocks without it (W = 8, N = 300,001 15.2 and 14.0 us for
// float32 and bf16 gradients, overlapped at 4 blocks 15.9 and 14.5).
constexpr int64_t kRaggedSinglesColumns = 200'000;
template <int METHOD, int V, int OPT, bool SS>
inline int64_t ragged_narrow_columns(int W) {
    if (W == 1) return V == 2 ? 450'000 : 150'000;
    if (V == 2) return OPT == kOptAdamW || SS ? 1'500'000 : 500'000;
    if (W == 2) return OPT == kOptAdamW ? 450'000 : 260'000;
    if (OPT == kOptAdamW) return 400'000;
    return SS && W < 24 ? 700'000 : METHOD == kMethodDDP ? 250'000 : 330'000;
}
template <int METHOD, int V, int OPT, bool SS, typename G>
struct RaggedShapeNarrow {
    static constexpr bool f32 = std::is_same<G, float>::value;
    static constexpr bool row_loads = METHOD == kMethodLocalSGD && SS && OPT == kOptSGD && !f32;
    static constexpr bool one_row = SS && OPT == kOptSGD && !row_loads;
    static constexpr bool plain_chunks = row_loads || (V == 1 && SS && OPT == kOptAdamW);
    static constexpr bool overlap = !one_row && !plain_chunks;
    static constexpr int rows = one_row ? 1 : 4;
    static constexpr int min_blocks = plain_chunks ? 5 : V == 1 && one_row ? 8 : 4;
    static constexpr int grad_rows = one_row || row_loads ? rows : f32 ? 4 : 8;
    static constexpr bool late = true;
};

// Two workers, few columns: both rows of everything in one trip. Time of a
// kernel with one column and one row per thread over: the narrow shape above,
// this one. N = 40,000, 130,000, 180,000, 230,000, odd: state-reconciling SGD 0.93 0.96
// 1.03 1.02, 1.02 0.91 1.15 1.13; SGD 1.13 1.12 0.93 0.87, 1.16 1.12 1.21 1.21; AdamW
// 1.04 1.06 0.93 0.90, 1.00 1.05 1.22 1.18; state-reconciling AdamW 1.00 0.90 1.17
// 0.89, 1.01 0.93 1.19 1.18. N = 2 mod 4, to 1.05 M: 0.91-1.22, 0.92-1.43.
struct RaggedShapeW2 {
    static constexpr int rows = 2, min_blocks = 6, grad_rows = 2;
    static constexpr bool late = true, overlap = true;
};

// One worker: all rows of a column in one round trip (N = 23.7 M, SGD f32
// 4,244 -> 6,681 GB/s at odd N, 4,251 -> 6,656 at N = 2 mod 4; AdamW bf16
// 4,579 -> 6,609 and 4,582 -> 6,616). State reconciliation at odd N keeps one
// column per thread without it between 150,000 and kRaggedW1Columns (one column
// and one row per thread over 4 columns / this: AdamW N = 180,000 0.81 / 0.97,
// 290,000 0.91 / 0.98; SGD 180,000 0.95 / 1.06, 240,000 0.92 / 1.04).
struct RaggedShapeW1 {
    static constexpr int rows = 1, min_blocks = 4, grad_rows = 1;
    static constexpr bool late = false, overlap = true;
};
constexpr int64_t kRaggedW1Columns = 330'000;
struct RaggedShapeW1States {
    static constexpr int rows = 1, min_blocks = 8, grad_rows = 1;
    static constexpr bool late = true, overlap = false;
};

// One round trip for few workers (reconcile_onepass_kernel: every row of a
// column loaded before any is used). Where it is used, and at how many
// resident blocks, per method, optimizer, state reconciliation and gradient
// type: each entry measured at least 2 % faster than the shapes above at
// N = 2^26 (GB/s, against the vec4 kernel). Entries not listed keep the vec4
// kernel.
// One worker, every variant: 1 row, 4 blocks. CPDP SGD f32 6,788 (5,620),
// SGD bf16 6,483 (5,385), AdamW f32 6,866 (5,814), AdamW bf16 6,653 (5,642);
// LocalSGD and DDP 6,004-6,848 (4,411-6,005); state reconciliation 3,967-5,603
// (3,519-4,189).
struct OnePassW1 {
    static constexpr bool use = true;
    static constexpr int wmax = 1, min_blocks = 4;
};
template <int METHOD, int OPT, bool SS, typename G>
struct OnePassW2 {
    static constexpr bool use = false;
    static constexpr int wmax = 2, min_blocks = 4;
};
// Two workers. CPDP: SGD f32 7,064 (6,792), SGD bf16 6,979 (5,958), AdamW f32
// 7,023 (6,422); with state reconciliation SGD f32 6,344 (6,116), SGD bf16
// 6,768 (5,197), AdamW f32 6,018 (5,364), AdamW bf16 at 3 blocks 5,411
// (5,073). DDP: SGD f32 7,059 (6,694), SGD bf16 6,945 (6,023), AdamW f32 at 3
// blocks 6,901 (6,748), AdamW bf16 6,960 (6,152). CPDP AdamW bf16 without state
// reconciliation and LocalSGD measured as fast or faster with the vec4 kernel.
#define CPDP_ONEPASS(NAME, M, O, SS, G, BLOCKS)          \
    template <>                                         \
    struct NAME<M, O, SS, G> {                          \
        static constexpr bool use = true;               \
        static constexpr int wmax = NAME##Max, min_blocks = BLOCKS; \
    };
constexpr int OnePassW2Max = 2;
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptSGD, false, float, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptSGD, false, bf16_bits, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptAdamW, false, float, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptSGD, true, float, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptSGD, true, bf16_bits, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptAdamW, true, float, 4)
CPDP_ONEPASS(OnePassW2, kMethodCPDP, kOptAdamW, true, bf16_bits, 3)
CPDP_ONEPASS(OnePassW2, kMethodDDP, kOptSGD, false, float, 4)
CPDP_ONEPASS(OnePassW2, kMethodDDP, kOptSGD, false, bf16_bits, 4)
CPDP_ONEPASS(OnePassW2, kMethodDDP, kOptAdamW, false, float, 3)
CPDP_ONEPASS(OnePassW2, kMethodDDP, kOptAdamW, false, bf16_bits, 4)

// Three workers (4-row chunk, the kernel skips the fourth). CPDP SGD f32
// 7,075 (6,731); LocalSGD SGD bf16 6,972 (6,666); DDP SGD bf16 6,985 (6,255),
// AdamW f32 7,018 (6,358), AdamW bf16 at 2 blocks 6,207 (5,974).
template <int METHOD, int OPT, bool SS, typename G>
struct OnePassW3 {
    static constexpr bool use = false;
    static constexpr int wmax = 4, min_blocks = 3;
};
constexpr int OnePassW3Max = 4;
CPDP_ONEPASS(OnePassW3, kMethodCPDP, kOptSGD, false, float, 3)
CPDP_ONEPASS(OnePassW3, kMethodLocalSGD, kOptSGD, false, bf16_bits, 3)
CPDP_ONEPASS(OnePassW3, kMethodDDP, kOptSGD, false, bf16_bits, 3)
CPDP_ONEPASS(OnePassW3, kMethodDDP, kOptAdamW, false, float, 3)
CPDP_ONEPASS(OnePassW3, kMethodDDP, kOptAdamW, false, bf16_bits, 2)

// Four workers. CPDP SGD bf16 at 2 blocks 6,803 (6,258); LocalSGD SGD bf16
// 7,005 (6,705); DDP SGD bf16 7,004 (6,174), AdamW f32 6,992 (6,749), AdamW
// bf16 at 2 blocks 6,758 (6,419).
template <int METHOD, int OPT, bool SS, typename G>
struct OnePassW4 {
    static constexpr bool use = false;
    static constexpr int wmax = 4, min_blocks = 3;
};
constexpr int OnePassW4Max = 4;
CPDP_ONEPASS(OnePassW4, kMethodCPDP, kOptSGD, false, bf16_bits, 2)
CPDP_ONEPASS(OnePassW4, kMethodLocalSGD, kOptSGD, false, bf16_bits, 3)
CPDP_ONEPASS(OnePassW4, kMethodDDP, kOptSGD, false, bf16_bits, 3)
CPDP_ONEPASS(OnePassW4, kMethodDDP, kOptAdamW, false, float, 3)
CPDP_ONEPASS(OnePassW4, kMethodDDP, kOptAdamW, false, bf16_bits, 2)
#undef CPDP_ONEPASS

}  // namespace cpdp
