// Step kernels for one storage type (__half); see step_impl.cuh.
#define LBM_TABLE_PAIRS  // this unit holds its type's constant table
#include "step_impl.cuh"
#include "step_multi.cuh"

namespace lbm {

cudaError_t launch_step_dev_f16(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                              int block, int variant) {
  return launch_step_dev_t<__half>(L, src, dst, st, block, variant);
}

cudaError_t launch_step_batch_f16(const BatchList &bl, int parity, cudaStream_t st, int block,
                                  int variant, const int *limits, int k) {
  return launch_step_batch_t<__half>(bl, parity, st, block, variant, limits, k);
}

cudaError_t upload_batch_consts_f16(const BatchEntry *ents, int n, int pbase, void *stage,
                                   cudaStream_t st) {
  return upload_consts_t<__half>(ents, n, pbase, stage, st);
}

cudaError_t launch_batch_resident_f16(const BatchEntry *ents, const int *idx, int nres,
                                      int nents, long long nodes, int parity, long steps,
                                      const int *limits, cudaStream_t st) {
  return launch_resident_t<__half>(ents, idx, nres, nents, nodes, parity, steps, limits, st);
}

cudaError_t launch_rows_f16(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                            int steps) {
  return launch_rows_t<__half>(L, src, dst, st, steps);
}

cudaError_t launch_rows_batch_f16(const BatchList &bl, int parity, cudaStream_t st,
                                  const int *limits, int k) {
  return launch_rows_batch_t<__half>(bl, parity, st, limits, k);
}

cudaError_t launch_tile_f16(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                            int steps, const float *forced, int sx, int sy) {
  return launch_tile_t<__half>(L, src, dst, st, steps, forced, sx, sy);
}

unsigned bounds_word_step_f16(bool reset) { return bounds::read_word(reset); }

}  // namespace lbm
