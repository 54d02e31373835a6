// Symmetric force (and potential) instantiations.
#include "cn_sym.cuh"

namespace cn {
namespace {

// the guarded form (eps2 = 0) holds two particles per thread
template <bool POT>
using ForceTable = SymTable<SymForcePolicy<2, POT, false>, SymForcePolicy<4, POT, false>, SymForcePolicy<8, POT, false>,
                            SymForcePolicy<2, POT, true>>;

}  // namespace

SymOps sym_force_ops(bool pot) { return pot ? ForceTable<true>::ops(8) : ForceTable<false>::ops(8); }

}  // namespace cn
