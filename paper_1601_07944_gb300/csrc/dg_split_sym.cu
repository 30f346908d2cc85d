/*
 * dg_split_sym.cu -- the split-product float64 element kernel (dg_split.cuh) for
 * the fully symmetric volume rules, in a translation unit of its own.
 */
#include "dg_split.cuh"

namespace dg {

int split_tables_sym(dg_mesh *m) {
#define CALL(P, NE) split_tables_pq<P, NE, sym_points(P)>(m)
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaSuccess;
}

int launch_split_sym(const dg_mesh *m, const double *c, const double *u0, double *out, double *trace_out,
                     const double *fhat, const StageUpdate &su, int mode, double *copy, void *stream, int64_t e0,
                     int64_t e1) {
  cudaStream_t s = (cudaStream_t)stream;
#define CALL(P, NE) run_split<P, NE, sym_points(P)>(m, c, u0, out, trace_out, fhat, su, mode, copy, s, e0, e1)
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

}  // namespace dg
