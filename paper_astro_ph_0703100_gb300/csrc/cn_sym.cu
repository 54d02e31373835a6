// Symmetric force (and potential) instantiations and the dispatch over forms.
#include "cn_sym.cuh"

namespace cn {
namespace {

template <class F>
auto by_policy(SymForm form, int k, bool guard, F&& f) {
  // the guarded form (eps2 = 0) holds two particles per thread
  if (form == kSymForcePot) {
    if (guard) return f(SymForcePolicy<2, true, true>{});
    if (k >= 8) return f(SymForcePolicy<8, true, false>{});
    if (k >= 4) return f(SymForcePolicy<4, true, false>{});
    return f(SymForcePolicy<2, true, false>{});
  }
  if (guard) return f(SymForcePolicy<2, false, true>{});
  if (k >= 8) return f(SymForcePolicy<8, false, false>{});
  if (k >= 4) return f(SymForcePolicy<4, false, false>{});
  return f(SymForcePolicy<2, false, false>{});
}

}  // namespace

int sym_sums(SymForm form) {
  return by_policy(form, 2, false, [](auto pol) { return decltype(pol)::kSumsI; });
}

size_t sym_smem_bytes(SymForm form, int threads, int k, int chunk, int stages) {
  return by_policy(form, k, false, [&](auto pol) { return sym_smem_of<decltype(pol)>(threads, chunk, stages); });
}

cudaError_t occupancy_sym(SymForm form, int k, bool guard, int threads, size_t smem, int* ctas) {
  return by_policy(form, k, guard, [&](auto pol) { return occupancy_sym_of<decltype(pol)>(threads, smem, ctas); });
}

cudaError_t launch_sym(SymForm form, const SymArgs& a, const SymMerge& m, int k, bool guard, int threads, size_t smem,
                       cudaStream_t s) {
  return by_policy(form, k, guard, [&](auto pol) { return launch_sym_of<decltype(pol)>(a, m, threads, smem, s); });
}

}  // namespace cn
