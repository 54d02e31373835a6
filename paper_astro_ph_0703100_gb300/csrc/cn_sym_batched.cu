// Symmetric force (and potential) of an ensemble: every cluster's unordered
// pairs once, all clusters' rows on one cost line (a table in the plan).
#include "cn_sym.cuh"

namespace cn {
namespace {

// Ensembles with a zero softening keep the one-sided kernel: no guarded form.
// Steps per trip (4 / 8 / 16), 512 clusters of 256 .. 16384: force 4989 / 4855
// / 4996 us, with the potential 6198 / 6352 / 8142. Sums are folded every 128
// records: in clusters of a few thousand particles one register chain is a
// large part of a sum (500 of 300 .. 3000: error 1.5e-7 with 512, 9.4e-8 with
// 256, 6.2e-8 with 128, one-sided 8.0e-8), for 2% of the time.
template <bool POT, int K>
using BatchedPolicy = SymForcePolicy<K, POT, false, POT ? 4 : 8, 128>;
template <bool POT>
using BatchedTable =
    SymTable<BatchedPolicy<POT, 2>, BatchedPolicy<POT, 4>, BatchedPolicy<POT, 8>, BatchedPolicy<POT, 2>, true>;

}  // namespace

SymOps sym_batched_ops(bool pot) { return pot ? BatchedTable<true>::ops(8) : BatchedTable<false>::ops(8); }

}  // namespace cn
