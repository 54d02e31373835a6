// Symmetric force (and potential) of an ensemble: every cluster's unordered
// pairs once, all clusters' rows on one cost line (a table in the plan).
#include "cn_sym.cuh"

namespace cn {
namespace {

// Ensembles with a zero softening keep the one-sided kernel: no guarded form.
// Steps per trip (4 / 8 / 16), 512 clusters of 256 .. 16384: force 4989 / 4855
// / 4996 us, with the potential 6198 / 6352 / 8142.
template <bool POT>
using BatchedTable = SymTable<SymForcePolicy<2, POT, false, POT ? 4 : 8>, SymForcePolicy<4, POT, false, POT ? 4 : 8>,
                              SymForcePolicy<8, POT, false, POT ? 4 : 8>, SymForcePolicy<2, POT, false, POT ? 4 : 8>, true>;

}  // namespace

SymOps sym_batched_ops(bool pot) { return pot ? BatchedTable<true>::ops(8) : BatchedTable<false>::ops(8); }

}  // namespace cn
