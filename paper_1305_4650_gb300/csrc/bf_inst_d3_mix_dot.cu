// Kernels for d = 3, precision PMIX, phase kind dot (q in {2,3,4}).
#include "bf_inst.cuh"

namespace bfl {

const PassFns *fns_d3_mix_dot(int q, int node_kind)
{
    switch (q) {
    case 2: return fns_for<3, 2, bfk::PMIX, bfk::KIND_DOT>(node_kind);
    case 3: return fns_for<3, 3, bfk::PMIX, bfk::KIND_DOT>(node_kind);
    case 4: return fns_for<3, 4, bfk::PMIX, bfk::KIND_DOT>(node_kind);
    default: return nullptr;
    }
}

}  // namespace bfl
