// Kernels for d = 3, precision PMIXFW (mixed, SFU sincos), phase kind genradon (q in {2,3,4}).
#include "bf_inst.cuh"

namespace bfl {

const PassFns *fns_d3_sfuw_genradon(int q, int node_kind)
{
    switch (q) {
    case 2: return fns_for<3, 2, bfk::PMIXFW, bfk::KIND_GENRADON>(node_kind);
    case 3: return fns_for<3, 3, bfk::PMIXFW, bfk::KIND_GENRADON>(node_kind);
    case 4: return fns_for<3, 4, bfk::PMIXFW, bfk::KIND_GENRADON>(node_kind);
    default: return nullptr;
    }
}

}  // namespace bfl
