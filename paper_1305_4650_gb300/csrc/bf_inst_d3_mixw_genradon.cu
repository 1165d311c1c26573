// Kernels for d = 3, precision PMIXW, phase kind genradon (q in {2,3,4}).
#include "bf_inst.cuh"

namespace bfl {

const PassFns *fns_d3_mixw_genradon(int q, int node_kind)
{
    switch (q) {
    case 2: return fns_for<3, 2, bfk::PMIXW, bfk::KIND_GENRADON>(node_kind);
    case 3: return fns_for<3, 3, bfk::PMIXW, bfk::KIND_GENRADON>(node_kind);
    case 4: return fns_for<3, 4, bfk::PMIXW, bfk::KIND_GENRADON>(node_kind);
    default: return nullptr;
    }
}

}  // namespace bfl
