// Bounds-checked copies of the one-code decode kernels (one and two shots per
// thread; plain, Momentum, AdaGrad and EWAInit BP; one or two nodes per
// thread; every table layout), compiled with BPQ_DEBUG into namespace
// bpq::dk_debug.  bpq_set_debug_checks selects them.
#define BPQ_DEBUG 1
#define dk dk_debug
#include "decode_kernel.cuh"
#include "decode_pair.cuh"
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

template <int V>
DecodeKernelFn pick_debug_v(int npt, bool pairs, bool one, int layout) {
    if (pairs) {
        if (layout == 2) return one ? dk_debug::decode_pair_kernel<V, true, true> : dk_debug::decode_pair_kernel<V, true, false>;
        if (layout == 1) return one ? dk_debug::decode_pair_kernel<V, false, true> : dk_debug::decode_pair_kernel<V, false, false>;
        return nullptr;
    }
    return npt == 1 ? pick_debug_one<V, 1>(layout) : npt == 2 ? pick_debug_one<V, 2>(layout) : nullptr;
}

}  // namespace

DecodeKernelFn pick_debug(int variant, int npt, bool pairs, bool one, int layout) {
    switch (variant) {
        case BPQ_PLAIN: return pick_debug_v<BPQ_PLAIN>(npt, pairs, one, layout);
        case BPQ_MOMENTUM: return pick_debug_v<BPQ_MOMENTUM>(npt, pairs, one, layout);
        case BPQ_ADAGRAD: return pick_debug_v<BPQ_ADAGRAD>(npt, pairs, one, layout);
        case BPQ_EWAINIT: return pick_debug_v<BPQ_EWAINIT>(npt, pairs, one, layout);
    }
    return nullptr;
}

}  // namespace bpq
