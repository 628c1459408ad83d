// The reconcile for N not a multiple of 4: rows that start off a vector
// boundary. Kept in a translation unit of its own so that it compiles beside
// the vector kernels.
#include "cpdp_kernels.cuh"
#include "cpdp_launch.cuh"
#include "cpdp_shapes.cuh"

#include <type_traits>

namespace cpdp {
namespace {

// V elements per load and U loads per thread and row, in launch shape Shape,
// with offsets of type Idx.
template <typename Shape, int METHOD, int OPT, bool SS, typename G, int V, int U, typename Idx>
cudaError_t launch_shape(const ReconcileCall& c) {
    const int64_t units = c.N / V;
    const int threads = reconcile_threads(METHOD, OPT, SS, c.W, c.N, U * V);
    const unsigned grid = grid_for((units + 32 * U - 1) / (32 * U), threads / 32);
    return launch_shaped(c.pdl,
                         reconcile_scalar_kernel<METHOD, OPT, SS, G, V, U, Shape::rows, Shape::min_blocks, Shape::late, Idx,
                                                 Shape::grad_rows, Shape::overlap && METHOD != kMethodLocalSGD>,
                         grid, threads, 0, c.stream, c.params, c.mom, c.sq, static_cast<const G*>(c.grads), c.anchor,
                         c.slow_v, c.W, static_cast<Idx>(units), c.args, c.backwards);
}

struct Ragged {
    const ReconcileCall& c;

    template <int METHOD, int OPT, bool SS, typename G, int V>
    cudaError_t shaped() const {
        if (c.W == 1) {
            if constexpr (V == 1 && SS)
                if (c.N > ragged_narrow_columns<METHOD, V, OPT, SS>(1) && c.N <= kRaggedW1Columns)
                    return launch_shape<RaggedShapeW1States, METHOD, OPT, SS, G, V, 1, int32_t>(c);
            return by_size<RaggedShapeW1, RaggedShapeW1, METHOD, OPT, SS, G, V>();
        }
        if (c.W == 2) return by_size<RaggedShapeW2, RaggedShape<V, OPT, SS, G, false>, METHOD, OPT, SS, G, V>();
        using Narrow = RaggedShapeNarrow<METHOD, V, OPT, SS, G>;
        using Few = RaggedShape<V, OPT, SS, G, false>;
        using Many = RaggedShape<V, OPT, SS, G, true>;
        if constexpr (Many::rows != Few::rows)
            if (c.W >= kGradChunksManyWorkers) return by_size<Narrow, Many, METHOD, OPT, SS, G, V>();
        return by_size<Narrow, Few, METHOD, OPT, SS, G, V>();
    }
    // one load per thread and row for few columns, kRaggedColumns / 32 columns per thread for more
    template <typename Narrow, typename Wide, int METHOD, int OPT, bool SS, typename G, int V>
    cudaError_t by_size() const {
        if (c.N <= ragged_narrow_columns<METHOD, V, OPT, SS>(c.W) && static_cast<int64_t>(c.W) * c.N < (int64_t(1) << 30))
            return launch_shape<Narrow, METHOD, OPT, SS, G, V, 1, int32_t>(c);
        constexpr int U = kRaggedColumns / (32 * V);
        // the largest offset formed is below W rows plus one grid-wide step
        const int64_t step = (c.N / kRaggedColumns + kThreads) * (kRaggedColumns / V);
        if (static_cast<int64_t>(c.W) * (c.N / V) + step < (int64_t(1) << 31))
            return launch_shape<Wide, METHOD, OPT, SS, G, V, U, int32_t>(c);
        return launch_shape<Wide, METHOD, OPT, SS, G, V, U, int64_t>(c);
    }
    template <int METHOD, int OPT, bool SS, typename G>
    cudaError_t run() const {
        const bool singles = SS && OPT == kOptSGD && c.W > 1 && c.N <= kRaggedSinglesColumns;
        return (c.N & 1) == 0 && !singles ? shaped<METHOD, OPT, SS, G, 2>() : shaped<METHOD, OPT, SS, G, 1>();
    }
};

}  // namespace

cudaError_t launch_reconcile_ragged(const ReconcileCall& c) { return dispatch_reconcile(c, Ragged{c}); }

#ifdef CPDP_CHECKED
cudaError_t take_bad_indices_ragged(unsigned long long* count) {
    const unsigned long long zero = 0;
    const cudaError_t e = cudaMemcpyFromSymbol(count, bad_index_count, sizeof *count);
    return e != cudaSuccess ? e : cudaMemcpyToSymbol(bad_index_count, &zero, sizeof zero);
}
#endif

}  // namespace cpdp
