// Symmetric force (and potential) instantiations.
#include "cn_sym.cuh"

namespace cn {
namespace {

// The guarded form (eps2 = 0) holds two particles per thread. Steps per trip
// of the sweep, measured at N = 131072 (4 / 8 / 16): force 4172 / 4058 / 4005
// us, with the potential 5279 / 5235 / 5187, but 792 / 788 / 806 at 50001.
template <bool POT>
using ForceTable = SymTable<SymForcePolicy<2, POT, false, POT ? 8 : 16>, SymForcePolicy<4, POT, false, POT ? 8 : 16>,
                            SymForcePolicy<8, POT, false, POT ? 8 : 16>, SymForcePolicy<2, POT, true, 4>>;

}  // namespace

SymOps sym_force_ops(bool pot) { return pot ? ForceTable<true>::ops(8) : ForceTable<false>::ops(8); }

}  // namespace cn
