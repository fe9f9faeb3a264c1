// Bounds-checked copies of the one-code decode kernels (one and two shots per
// thread and small batches; plain, Momentum, AdaGrad and EWAInit BP; one or two
// nodes per thread; every table layout), compiled with BPQ_DEBUG into namespace
// bpq::dk_debug.  bpq_set_debug_checks selects them.
#define BPQ_DEBUG 1
#define dk dk_debug
#include "decode_kernel.cuh"
#include "decode_pair.cuh"
#include "decode_small.cuh"
#undef dk

namespace bpq {

namespace {

template <int V, int NPT>
DecodeKernelFn pick_debug_one(int layout) {
    switch (layout) {
        case 2: return dk_debug::decode_kernel<V, NPT, false, true, true>;
        case 1: return dk_debug::decode_kernel<V, NPT, false, true, false>;
        default: return dk_debug::decode_kernel<V, NPT, false, false, false>;
    }
}

template <int V, bool FULL>
DecodeKernelFn pick_debug_pair(int mode) {
    return mode == kPairOne     ? dk_debug::decode_pair_kernel<V, FULL, kPairOne>
           : mode == kPairWarps ? dk_debug::decode_pair_kernel<V, FULL, kPairWarps>
                                : dk_debug::decode_pair_kernel<V, FULL, kPairGroups>;
}

template <int V>
DecodeKernelFn pick_debug_v(int npt, bool pairs, int mode, int layout) {
    if (pairs) return layout == 2 ? pick_debug_pair<V, true>(mode) : layout == 1 ? pick_debug_pair<V, false>(mode) : nullptr;
    return npt == 1 ? pick_debug_one<V, 1>(layout) : npt == 2 ? pick_debug_one<V, 2>(layout) : nullptr;
}

}  // namespace

DecodeKernelFn pick_debug(int variant, int npt, bool pairs, int mode, int layout) {
    switch (variant) {
        case BPQ_PLAIN: return pick_debug_v<BPQ_PLAIN>(npt, pairs, mode, layout);
        case BPQ_MOMENTUM: return pick_debug_v<BPQ_MOMENTUM>(npt, pairs, mode, layout);
        case BPQ_ADAGRAD: return pick_debug_v<BPQ_ADAGRAD>(npt, pairs, mode, layout);
        case BPQ_EWAINIT: return pick_debug_v<BPQ_EWAINIT>(npt, pairs, mode, layout);
    }
    return nullptr;
}

namespace {

template <int V>
SmallKernelFn pick_debug_lanes(int lanes) {
    return lanes == 4   ? dk_debug::decode_small_kernel<V, 4>
           : lanes == 2 ? dk_debug::decode_small_kernel<V, 2>
                        : dk_debug::decode_small_kernel<V, 1>;
}

}  // namespace

SmallKernelFn pick_debug_small(int variant, int lanes) {
    switch (variant) {
        case BPQ_PLAIN: return pick_debug_lanes<BPQ_PLAIN>(lanes);
        case BPQ_MOMENTUM: return pick_debug_lanes<BPQ_MOMENTUM>(lanes);
        case BPQ_ADAGRAD: return pick_debug_lanes<BPQ_ADAGRAD>(lanes);
        case BPQ_EWAINIT: return pick_debug_lanes<BPQ_EWAINIT>(lanes);
    }
    return nullptr;
}

}  // namespace bpq
