// Kernels for d = 2, precision PMIXFW (mixed, SFU sincos), phase kind hypradon (q in {2,3,4,5,6,8}).
#include "bf_inst.cuh"

namespace bfl {

const PassFns *fns_d2_sfuw_hypradon(int q, int node_kind)
{
    switch (q) {
    case 2: return fns_for<2, 2, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    case 3: return fns_for<2, 3, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    case 4: return fns_for<2, 4, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    case 5: return fns_for<2, 5, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    case 6: return fns_for<2, 6, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    case 8: return fns_for<2, 8, bfk::PMIXFW, bfk::KIND_HYPRADON>(node_kind);
    default: return nullptr;
    }
}

}  // namespace bfl
