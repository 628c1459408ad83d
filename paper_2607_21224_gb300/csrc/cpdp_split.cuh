// The reconcile with the worker rows of a column split across the warps of a
// block, for many workers over few columns.
//
// What bounds the column kernels there: one thread walks all W rows of its
// columns, a chunk at a time, so a launch takes about W / 2 dependent trips to
// memory however few columns there are, on N / 256 blocks of 2 warps (W = 64,
// N = 60,000: 235). Here a block owns the columns of 32 loads (64 at even N, 32
// at odd) and its 4 to 16 warps take every R-th row, so a column's rows are
// loaded by R warps at once and N / 64 (N / 32) blocks run. The values to be
// averaged pass through shared memory, where one thread per column adds them
// in worker order: the sums are those of the other kernels bit for bit (partial
// sums per warp measured the same within 10 %, but in another order). Sync step,
// us, column kernel -> this one, CPDP SGD f32, state from DRAM: W = 64,
// N = 60,000 30.6 -> 15.6 (5.0 TB/s; the bytes take 11.4 at the copy rate);
// W = 16, N = 23,000 8.3 -> 3.5; W = 200, N = 23,000 86.5 -> 23.9; AdamW bf16
// W = 64, N = 24,000 45 -> 11. State in L2: W = 64, N = 61,000 17.6 -> 11.1; W = 16,
// N = 23,000 4.4 -> 2.5. What bounds it now is the trips that are left, two to
// six per 64 rows, and the barriers between them.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cpdp_kernels.cuh"
#include "cpdp_launch.cuh"

namespace cpdp {

constexpr int kSplitMaxWarps = 16;

// Where it is used. From 9 workers: up to 8 the column kernels need at most
// four trips. Above these sizes the column kernels have blocks enough, and
// their longer row segments win. Sync steps in a row, time of the column kernel
// (64-thread blocks) over this one's, geometric means over worker counts with
// the state in L2 and out of it; N a multiple of 4 / N = 2 mod 4, whose column
// kernel has twice the threads. W = 9 to 12, N = 64,000: SGD 1.23-1.56 / 1.01-1.64, AdamW
// 1.38-1.80 / 1.04-1.38; 85,000: SGD 0.77-1.38 / 0.78-1.50. W = 16 to 24, 110,000:
// AdamW 1.22-1.46 / 0.93-1.24, SGD f32 1.0-1.17 / 1.03-1.15, bf16 0.91-1.25 / 0.92-1.21,
// state-reconciling SGD 0.85-1.17 / 0.89-1.11; 140,000: 0.91-1.38 / 0.86-1.14. W = 32 and
// more, 140,000: 0.98-1.53 / 0.82-1.32; 180,000: 0.87-1.25 / 0.91-1.44. In a period
// of 2 or 4 steps, where the local steps leave other lines in L2, it is further
// ahead (N a multiple of 4): W = 20, N = 91,000 to 134,000, state-reconciling CPDP SGD
// 1.23-1.27, W = 32, N = 154,000 1.16, W = 200, N = 108,000 1.35, state-reconciling AdamW
// W = 24 to 48, N = 103,000 to 126,000 1.4-2.0.
// Odd rows cost the column kernels more, as a row is more of 4-byte loads, and
// this kernel holds 8 of them at once (split_deep), so its range is longer
// at odd N: float32 gradients, SGD from 24 workers to 300,001 1.0-1.4 for
// CPDP and LocalSGD; DDP from 9 workers 1.0-2.0, at 9 to 23 workers to 250,001
// (W = 12 to 20, 150,000 to 235,000 0.98-1.45, with the state in L2 0.86-1.33; 292,000
// 0.83); AdamW from 24 workers to 420,001 1.0-1.5 for DDP and
// LocalSGD, for CPDP to 110,001 1.0-1.2 and from 100 workers to 300,001
// 1.0-1.3; bf16 from 48 workers to 110,001 1.0-1.2. State reconciliation from
// 100 workers to 300,001, AdamW and LocalSGD: 1.0-1.4; CPDP SGD 0.9-1.1, so it
// keeps 64,000. Its offsets are 32-bit: W rows of N / V loads stay below 2^31.
inline bool split_takes(const ReconcileCall& c) {
    const int64_t units = (c.N & 1) == 0 ? c.N >> 1 : c.N;
    if (c.W < 9 || c.W * units >= int64_t(1) << 31) return false;
    if ((c.N & 1) == 0) return c.N <= (c.W < 16 ? 64'000 : 160'000);
    const bool sgd = c.opt == kOptSGD, cpdp_method = c.method == kMethodCPDP;
    int64_t limit = c.W < 24 ? 24'000 : 64'000;
    if (c.state_sync) {
        if (c.W >= 100 && (!sgd || !cpdp_method)) limit = 300'000;
    } else if (c.bf16) {
        if (c.W >= 48) limit = 110'000;
    } else if (sgd && (c.method == kMethodDDP || c.W >= 24)) {
        limit = c.W < 24 ? 250'000 : 300'000;
    } else if (!sgd && c.W >= 24 && !cpdp_method) {
        limit = 420'000;
    } else if (!sgd && c.W >= 100) {
        limit = 300'000;
    } else if (c.W >= 16 && (!sgd || !cpdp_method)) {
        limit = 110'000;
    }
    return c.N <= limit;
}

// Warps per block over `tiles` blocks: more while the launch stays within
// about one resident wave (152 SMs x 27 warps) and a warp keeps 3 rows or more
// (CPDP SGD f32, state in L2, us at 4 / 8 / 16 warps: W = 16, N = 32,000 2.57 / 2.91 /
// 4.65; W = 64, N = 32,000 6.15 / 5.66 / 6.84; W = 200, N = 8,000 13.3 / 9.8 / 8.5).
inline int split_warps(int W, int64_t tiles) {
    int warps = 4;
    while (warps < kSplitMaxWarps && tiles * warps * 2 <= 4096 && W >= 3 * warps * 2) warps *= 2;
    return warps;
}

// Whether a warp has rows enough for deeper chunks than 4 rows: 8 gradient rows
// for float32 pairs (SGD), 8 gradient and 8 state rows at odd N, where a row is
// one register. Sync step, us, 4-row chunks -> these: CPDP SGD f32 W = 64,
// N = 60,000 15.6 -> 14.9, N = 60,001 23.1 -> 16.2; W = 200, N = 13,215 21.7 ->
// 16.3; state-reconciling SGD f32 W = 64, N = 120,000 32.3 -> 28.3; DDP SGD f32
// W = 64, N = 60,001 18.9 -> 15.4; AdamW bf16 W = 200, N = 60,001 75.1 -> 72.3. With
// fewer rows per warp the deeper chunks are mostly empty and 5 to 20 % slower
// (W = 16, N = 20,001 2.8 -> 3.4; 16 warps, W = 64, N = 5,001 3.6 -> 4.0), as is
// state-reconciling SGD at 8 warps and odd N (W = 64, N = 13,215 6.3 -> 7.0).
constexpr int64_t kSplitManyTiles = 1000;
inline bool split_deep(int W, int warps, int64_t tiles) {
    return warps <= 8 && (W >= 64 || (W >= 24 && tiles >= kSplitManyTiles));
}

// V consecutive columns of one row.
template <int V>
struct Slice {
    float v[V];
};

template <int V>
struct SliceIO;
template <>
struct SliceIO<2> {
    static __device__ __forceinline__ Slice<2> load(const float* p, int32_t u) {
        const float2 x = reinterpret_cast<const float2*>(p)[u];
        return {x.x, x.y};
    }
    static __device__ __forceinline__ void store(float* p, int32_t u, const Slice<2>& x) {
        reinterpret_cast<float2*>(p)[u] = make_float2(x.v[0], x.v[1]);
    }
    static __device__ __forceinline__ float2 words(const float* g, int32_t u) {
        float2 x;
        GradLoad<float>::pair(g, u, x.x, x.y);
        return x;
    }
    static __device__ __forceinline__ uint32_t words(const bf16_bits* g, int32_t u) {
        return GradLoad<bf16_bits>::pair(g, u);
    }
    static __device__ __forceinline__ Slice<2> widen(const float2& x) { return {x.x, x.y}; }
    static __device__ __forceinline__ Slice<2> widen(uint32_t x) {
        return {__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)};
    }
};
template <>
struct SliceIO<1> {
    static __device__ __forceinline__ Slice<1> load(const float* p, int32_t u) { return {p[u]}; }
    static __device__ __forceinline__ void store(float* p, int32_t u, const Slice<1>& x) { p[u] = x.v[0]; }
    template <typename G>
    static __device__ __forceinline__ float words(const G* g, int32_t u) {
        return GradLoad<G>::one(g, u);
    }
    static __device__ __forceinline__ Slice<1> widen(float x) { return {x}; }
};

// Rows of one round: their values pass through shared memory, where one
// thread per column adds them in worker order.
template <bool STATE_SYNC>
struct SplitRows {
    static constexpr int value = STATE_SYNC ? 32 : 64;
};

// s + rows[0][column] + ... + rows[n - 1][column], in that order.
template <int C>
__device__ __forceinline__ float add_rows(float s, const float (*rows)[C], int n, int column) {
#pragma unroll 8
    for (int r = 0; r < n; ++r) s += rows[r][column];
    return s;
}

// A block owns C = 32 * V columns; its warp w of R takes rows w, w + R, ... of
// them. `units` is N / V.
template <int METHOD, int OPT, bool STATE_SYNC, typename G, int V, int CH, int GCH>
__global__ void __launch_bounds__(32 * kSplitMaxWarps, 2)
reconcile_split_kernel(float* __restrict__ params, float* __restrict__ mom, float* __restrict__ sq,
                       const G* __restrict__ grads, float* __restrict__ anchor, float* __restrict__ slow_v,
                       int W, int32_t units, SyncArgs a) {
    static_assert(!(STATE_SYNC && METHOD == kMethodDDP), "DDP's states are identical across workers");
    using IO = SliceIO<V>;
    constexpr int C = 32 * V, B = SplitRows<STATE_SYNC>::value;
    __shared__ __align__(8) float rows_t[B][C];  // the gradients, then the stepped parameters
    __shared__ __align__(8) float rows_b[STATE_SYNC ? B : 1][C];
    __shared__ __align__(8) float rows_s[STATE_SYNC && OPT == kOptAdamW ? B : 1][C];
    __shared__ __align__(8) float mean[3][C];  // what the columns' threads hand back to the warps
    pdl_wait_then_release();
    const int R = blockDim.x / 32, w = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int32_t u = (int32_t)blockIdx.x * 32 + lane;
    const bool in = u < units;  // lanes past the last column only take part in the barriers
    // the thread that adds column t of the block
    const int t = threadIdx.x;
    const int32_t column = (int32_t)blockIdx.x * C + t, columns = units * V;
    const bool adds = t < C && column < columns;
    auto at = [&](int row) { return CPDP_IDX(row * units + u, W * units); };
    auto put = [&](float (*rows)[C], int r, const Slice<V>& x) {
#pragma unroll
        for (int e = 0; e < V; ++e) rows[r][lane * V + e] = x.v[e];
    };
    auto get = [&](const float* row) {
        Slice<V> x;
#pragma unroll
        for (int e = 0; e < V; ++e) x.v[e] = row[lane * V + e];
        return x;
    };

    Slice<V> th[CH], bu[CH], sv[CH], gw[CH];
    auto load_state = [&](int i0, int end) {
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int row = i0 + k * R;
            if (in && row < end) {
                th[k] = IO::load(params, at(row));
                bu[k] = IO::load(mom, at(row));
                if (OPT == kOptAdamW) sv[k] = IO::load(sq, at(row));
                if (METHOD == kMethodLocalSGD) gw[k] = IO::widen(IO::words(grads, at(row)));
            }
        }
    };
    load_state(w, min(B, W));
    float ref = 0.f, vel = 0.f;
    if (METHOD == kMethodCPDP && adds) {
        ref = anchor[CPDP_IDX(column, columns)];
        vel = slow_v[CPDP_IDX(column, columns)];
    }

    // 1. gradient mean (eq. 2)
    Slice<V> gbar = {};
    if (METHOD != kMethodLocalSGD) {
        float gsum = 0.f;
        for (int base = 0; base < W; base += B) {
            const int end = min(base + B, W);
            for (int i0 = base + w; i0 < end; i0 += GCH * R) {
                decltype(IO::words(grads, 0)) gv[GCH];
#pragma unroll
                for (int k = 0; k < GCH; ++k)
                    if (in && i0 + k * R < end) gv[k] = IO::words(grads, at(i0 + k * R));
#pragma unroll
                for (int k = 0; k < GCH; ++k)
                    if (in && i0 + k * R < end) put(rows_t, i0 + k * R - base, IO::widen(gv[k]));
            }
            __syncthreads();
            if (adds) gsum = add_rows<C>(gsum, rows_t, end - base, t);
            if (end == W && t < C) mean[0][t] = gsum / a.workers;
            __syncthreads();
        }
        gbar = get(mean[0]);
    }

    // 2-3. optimizer step on the warp's workers (eq. 6), and the mean of the stepped replicas (eq. 7)
    float tsum = 0.f, bsum = 0.f, ssum = 0.f;
    for (int base = 0; base < W; base += B) {
        const int end = min(base + B, W);
        for (int i0 = base + w; i0 < end; i0 += CH * R) {
            if (i0 != w) load_state(i0, end);
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                const int row = i0 + k * R;
                if (in && row < end) {
#pragma unroll
                    for (int e = 0; e < V; ++e)
                        opt_step<OPT>(METHOD == kMethodLocalSGD ? gw[k].v[e] : gbar.v[e], th[k].v[e], bu[k].v[e],
                                      sv[k].v[e], a.step);
                    if (STATE_SYNC) {
                        put(rows_b, row - base, bu[k]);
                        if (OPT == kOptAdamW) put(rows_s, row - base, sv[k]);
                    } else {
                        IO::store(mom, at(row), bu[k]);
                        if (OPT == kOptAdamW) IO::store(sq, at(row), sv[k]);
                    }
                    if (METHOD == kMethodDDP)
                        IO::store(params, at(row), th[k]);
                    else
                        put(rows_t, row - base, th[k]);
                }
            }
        }
        if (METHOD == kMethodDDP) continue;
        __syncthreads();
        if (adds) {
            tsum = add_rows<C>(tsum, rows_t, end - base, t);
            if (STATE_SYNC) {
                bsum = add_rows<C>(bsum, rows_b, end - base, t);
                if (OPT == kOptAdamW) ssum = add_rows<C>(ssum, rows_s, end - base, t);
            }
            if (end == W) {
                float tn = tsum / a.workers;
                if (METHOD == kMethodCPDP) {  // 4. SlowMo (eqs. 8-10)
                    const float vn = fmaf(a.beta, vel, tn - ref);
                    tn = fmaf(a.alpha, vn, ref);
                    anchor[CPDP_IDX(column, columns)] = tn;
                    slow_v[CPDP_IDX(column, columns)] = vn;
                }
                mean[0][t] = tn;
                if (STATE_SYNC) {
                    mean[1][t] = bsum / a.workers;
                    if (OPT == kOptAdamW) mean[2][t] = ssum / a.workers;
                }
            }
        }
        __syncthreads();
    }
    if (METHOD == kMethodDDP || !in) return;

    // 5. write-back to every replica (eqs. 11-12), and of the averaged state
    const Slice<V> tn = get(mean[0]);
    for (int i = w; i < W; i += R) IO::store(params, at(i), tn);
    if (STATE_SYNC) {
        const Slice<V> bmean = get(mean[1]);
        for (int i = w; i < W; i += R) IO::store(mom, at(i), bmean);
        if (OPT == kOptAdamW) {
            const Slice<V> smean = get(mean[2]);
            for (int i = w; i < W; i += R) IO::store(sq, at(i), smean);
        }
    }
}

}  // namespace cpdp
