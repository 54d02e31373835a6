// rows_kernel: plain and per-particle-softening instantiations.
#include "cn_rows.cuh"

namespace cn {

namespace {

bool pot_form(RowForm f) { return f & 1; }

const void* select(RowForm form, int k) {
  switch (form) {
    case kRowForce: return rows_fn<false, false>(k);
    case kRowForcePot: return rows_fn<true, false>(k);
    case kRowEpsI: return rows_fn<false, true>(k);
    default: return rows_fn<true, true>(k);
  }
}

}  // namespace

size_t rows_smem_bytes(RowForm form, int k, int chunk, int stages) {
  return 256 + static_cast<size_t>(2) * (pot_form(form) ? 4 : 3) * kRowThreads * k * sizeof(float) +
         static_cast<size_t>(stages) * chunk * 16;
}

cudaError_t occupancy_rows(RowForm form, int k, size_t smem, int* ctas) {
  const void* f = select(form, k);
  const cudaError_t e = prepare_kernel(f, smem);
  return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, f, kRowThreads, smem);
}

cudaError_t launch_rows(RowForm form, int k, const RowArgs& a, size_t smem, cudaStream_t s) {
  const void* f = select(form, k);
  cudaError_t e = prepare_kernel(f, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<RowArgs*>(&a)};
  e = launch_pdl(f, dim3(static_cast<unsigned>(a.grid)), dim3(kRowThreads), args, smem, s);
  if (e != cudaSuccess) return e;
  const int sums = pot_form(form) ? 4 : 3;
  const void* m = pot_form(form) ? reinterpret_cast<const void*>(&rows_merge_kernel<4>)
                                 : reinterpret_cast<const void*>(&rows_merge_kernel<3>);
  return launch_pdl(m, dim3(static_cast<unsigned>(a.grid), static_cast<unsigned>((sums * a.tile + 255) / 256)),
                    dim3(256), args, 0, s);
}

}  // namespace cn
