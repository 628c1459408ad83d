// What the translation units of libcpdp share on the host: how a kernel is
// launched, and the arguments of a reconcile whose kernels are compiled in a
// file of their own.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cpdp_kernels.cuh"

namespace cpdp {

// Launch `kernel` with `block` threads per block on `s`. With programmatic
// dependent launch on, the launch may begin while the previous grid on the
// stream drains; every kernel waits for that grid's completion itself before
// touching memory (pdl_wait_then_release).
template <typename... KArgs, typename... Args>
cudaError_t launch_shaped(bool pdl, void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem,
                          cudaStream_t s, Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One reconcile: the kernel variant (method, optimizer, state reconciliation,
// gradient type), the arrays and the scalars.
struct ReconcileCall {
    bool pdl;
    int method, opt;
    bool state_sync, bf16;
    int W;
    int64_t N;
    float *params, *mom, *sq;
    const void* grads;
    float *anchor, *slow_v;
    SyncArgs args;
    int backwards;
    cudaStream_t stream;
};

// N not a multiple of 4 (cpdp_ragged.cu).
cudaError_t launch_reconcile_ragged(const ReconcileCall& c);
// Many workers over few columns (cpdp_split.cu).
cudaError_t launch_reconcile_split(const ReconcileCall& c);

// The call's variant as compile-time constants: f.template run<METHOD, OPT, SS, G>().
template <typename F, int METHOD, int OPT, bool SS>
cudaError_t dispatch_grads(const ReconcileCall& c, const F& f) {
    return c.bf16 ? f.template run<METHOD, OPT, SS, bf16_bits>() : f.template run<METHOD, OPT, SS, float>();
}
template <typename F, int METHOD, int OPT>
cudaError_t dispatch_state(const ReconcileCall& c, const F& f) {
    if constexpr (METHOD != kMethodDDP)  // DDP's states are identical across workers: nothing to reconcile
        if (c.state_sync) return dispatch_grads<F, METHOD, OPT, true>(c, f);
    return dispatch_grads<F, METHOD, OPT, false>(c, f);
}
template <typename F, int METHOD>
cudaError_t dispatch_opt(const ReconcileCall& c, const F& f) {
    return c.opt == kOptAdamW ? dispatch_state<F, METHOD, kOptAdamW>(c, f) : dispatch_state<F, METHOD, kOptSGD>(c, f);
}
template <typename F>
cudaError_t dispatch_reconcile(const ReconcileCall& c, const F& f) {
    if (c.method == kMethodLocalSGD) return dispatch_opt<F, kMethodLocalSGD>(c, f);
    if (c.method == kMethodDDP) return dispatch_opt<F, kMethodDDP>(c, f);
    return dispatch_opt<F, kMethodCPDP>(c, f);
}

// The index-checked debug build counts bad indices per translation unit; each
// file's counter, read and set to 0 (current device, after a synchronization).
cudaError_t take_bad_indices_ragged(unsigned long long* count);
cudaError_t take_bad_indices_split(unsigned long long* count);

}  // namespace cpdp
