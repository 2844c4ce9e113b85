// Launch dispatch of the element kernels: dg_element.cu is built per number of
// points per direction and part.
#include "dg_kernels.cuh"

namespace dgk {

#define DG_OPS(p) elem_ops_2_##p, elem_ops_3_##p, elem_ops_4_##p, elem_ops_5_##p, elem_ops_6_##p, elem_ops_7_##p
extern const ElemOps DG_OPS(0);
extern const ElemOps DG_OPS(1);
extern const ElemOps DG_OPS(2);

namespace {
// parts of dg_element.cu: 0 the stage phases, 1 the Navier-Stokes volume
// phase, one-shot maps and mass solves, 2 the adjoint
const ElemOps& ops(int n, int part) {
  static const ElemOps* const all[3][6] = {
      {&elem_ops_2_0, &elem_ops_3_0, &elem_ops_4_0, &elem_ops_5_0, &elem_ops_6_0, &elem_ops_7_0},
      {&elem_ops_2_1, &elem_ops_3_1, &elem_ops_4_1, &elem_ops_5_1, &elem_ops_6_1, &elem_ops_7_1},
      {&elem_ops_2_2, &elem_ops_3_2, &elem_ops_4_2, &elem_ops_5_2, &elem_ops_6_2, &elem_ops_7_2}};
  return *all[part][n < 2 ? 0 : (n > kMaxn ? kMaxn - 2 : n - 2)];
}
int points_of(int nQ) {
  int n = 2;
  while (n * n * n < nQ) ++n;
  return n;
}
template <class F>
void each_n(unsigned mask, int part, F f) {
  for (int n = 2; n <= kMaxn; ++n)
    if ((mask >> n) & 1u) f(ops(n, part));
}
}  // namespace

void launch_element(const Ctx& c, int mode, const StageArgs& a, const Sched& s, bool balanced, int grid, int wpb,
                    cudaStream_t st) {
  const bool stage = mode == kFwd || mode == kBwdRhs || mode == kBwdRk || mode == kBwdRkFwd;
  each_n(c.nmask, stage ? 0 : 1, [&](const ElemOps& o) { o.element(c, mode, a, s, balanced, grid, wpb, st); });
}

void launch_vjp(const Ctx& c, int phase, const VjpArgs& va, int64_t nelem, int wpb, cudaStream_t st) {
  each_n(c.nmask, 2, [&](const ElemOps& o) { o.vjp(c, phase, va, nelem, wpb, st); });
}

cudaError_t launch_moving_mass(const Ctx& c, const int64_t* list, int64_t n_slots, const double* in, double* out,
                               const double* x0, const double* tau, int weight, int max_nM, int max_nQ, int grid,
                               cudaStream_t st, int nblk, int64_t blk_stride, float* fac_out, const float* fac_in) {
  return ops(points_of(c.nQmax), 1).mass(c, list, n_slots, in, out, x0, tau, weight, max_nM, max_nQ, grid, st, nblk,
                                      blk_stride, fac_out, fac_in);
}

cudaError_t element_kernel_attributes(int nQmax, int wpb, int* blocks_per_sm, bool curved, bool split) {
  const int n = points_of(nQmax);
  cudaError_t e = face_kernel_attributes();
  for (int part = 2; part > 0 && e == cudaSuccess; --part) e = ops(n, part).attributes(wpb, blocks_per_sm, curved, split);
  if (e != cudaSuccess) return e;
  return ops(n, 0).attributes(wpb, blocks_per_sm, curved, split);
}

cudaError_t element_kernel_attributes_ns(int nQmax, int wpb, int* blocks_per_sm, bool curved) {
  return ops(points_of(nQmax), 1).attributes(wpb, blocks_per_sm, curved, false);
}

}  // namespace dgk
