// The reconcile of many workers over few columns, in a translation unit of its
// own (it compiles beside the vector kernels).
#include "cpdp_kernels.cuh"
#include "cpdp_launch.cuh"
#include "cpdp_split.cuh"

#include <type_traits>

namespace cpdp {
namespace {

struct Split {
    const ReconcileCall& c;

    template <int METHOD, int OPT, bool SS, typename G, int V, int CH, int GCH>
    cudaError_t shaped(int64_t units, int64_t tiles, int warps) const {
        return launch_shaped(c.pdl, reconcile_split_kernel<METHOD, OPT, SS, G, V, CH, GCH>,
                             static_cast<unsigned>(tiles), 32u * warps, 0, c.stream, c.params, c.mom, c.sq,
                             static_cast<const G*>(c.grads), c.anchor, c.slow_v, c.W, static_cast<int32_t>(units),
                             c.args);
    }
    template <int METHOD, int OPT, bool SS, typename G, int V>
    cudaError_t columns() const {
        constexpr bool f32 = std::is_same<G, float>::value;
        const int64_t units = c.N / V, tiles = (units + 31) / 32;
        const int warps = split_warps(c.W, tiles);
        if (split_deep(c.W, warps, tiles)) {
            if constexpr (V == 1) {
                if (!(SS && warps == 8) && (f32 || warps == 8 || tiles >= kSplitManyTiles))
                    return shaped<METHOD, OPT, SS, G, 1, 8, 8>(units, tiles, warps);
            } else if constexpr (OPT == kOptSGD && f32) {
                return shaped<METHOD, OPT, SS, G, 2, 4, 8>(units, tiles, warps);
            }
        }
        return shaped<METHOD, OPT, SS, G, V, 4, f32 ? 4 : 8>(units, tiles, warps);
    }
    template <int METHOD, int OPT, bool SS, typename G>
    cudaError_t run() const {
        return (c.N & 1) == 0 ? columns<METHOD, OPT, SS, G, 2>() : columns<METHOD, OPT, SS, G, 1>();
    }
};

}  // namespace

cudaError_t launch_reconcile_split(const ReconcileCall& c) { return dispatch_reconcile(c, Split{c}); }

#ifdef CPDP_CHECKED
cudaError_t take_bad_indices_split(unsigned long long* count) {
    const unsigned long long zero = 0;
    const cudaError_t e = cudaMemcpyFromSymbol(count, bad_index_count, sizeof *count);
    return e != cudaSuccess ? e : cudaMemcpyToSymbol(bad_index_count, &zero, sizeof zero);
}
#endif

}  // namespace cpdp
