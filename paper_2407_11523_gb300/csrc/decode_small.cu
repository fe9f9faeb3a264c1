// The small-batch kernels (decode_small.cuh) by variant and lanes per node.
#include "decode_small.cuh"

namespace bpq {

namespace {

template <int V>
SmallKernelFn pick_lanes(int lanes) {
    return lanes == 4 ? dk::decode_small_kernel<V, 4> : lanes == 2 ? dk::decode_small_kernel<V, 2>
                                                                  : dk::decode_small_kernel<V, 1>;
}

}  // namespace

SmallKernelFn pick_small(int variant, int lanes) {
    switch (variant) {
        case BPQ_PLAIN: return pick_lanes<BPQ_PLAIN>(lanes);
        case BPQ_MOMENTUM: return pick_lanes<BPQ_MOMENTUM>(lanes);
        case BPQ_ADAGRAD: return pick_lanes<BPQ_ADAGRAD>(lanes);
        case BPQ_EWAINIT:
        case BPQ_AEWA: return pick_lanes<BPQ_EWAINIT>(lanes);
    }
    return nullptr;
}

}  // namespace bpq
