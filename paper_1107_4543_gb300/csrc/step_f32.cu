// Step kernels for one storage type (float); see step_impl.cuh.
#define LBM_TABLE_DEV  // this unit holds its type's constant table
#include "step_impl.cuh"
#include "step_multi.cuh"

namespace lbm {

cudaError_t launch_step_dev_f32(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                              int block, int variant) {
  return launch_step_dev_t<float>(L, src, dst, st, block, variant);
}

cudaError_t launch_step_batch_f32(const BatchList &bl, int parity, cudaStream_t st, int block,
                                  int variant, const int *limits, int k) {
  return launch_step_batch_t<float>(bl, parity, st, block, variant, limits, k);
}

cudaError_t upload_batch_consts_f32(const BatchEntry *ents, int n, int pbase, void *stage,
                                    cudaStream_t st) {
  return upload_consts_t<float>(ents, n, pbase, stage, st);
}

cudaError_t launch_batch_resident_f32(const BatchEntry *ents, const int *idx, int nres,
                                      int nents, long long nodes, int parity, long steps,
                                      const int *limits, cudaStream_t st) {
  return launch_resident_t<float>(ents, idx, nres, nents, nodes, parity, steps, limits, st);
}

cudaError_t launch_rows_f32(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                            int steps) {
  return launch_rows_t<float>(L, src, dst, st, steps);
}

cudaError_t launch_rows_batch_f32(const BatchList &bl, int parity, cudaStream_t st,
                                  const int *limits, int k) {
  return launch_rows_batch_t<float>(bl, parity, st, limits, k);
}

cudaError_t launch_tile_f32(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                            int steps, const float *forced, int sx, int sy) {
  return launch_tile_t<float>(L, src, dst, st, steps, forced, sx, sy);
}

unsigned bounds_word_step_f32(bool reset) { return bounds::read_word(reset); }

}  // namespace lbm
