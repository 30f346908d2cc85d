/*
 * dg_split.cu -- the split-product float64 element kernel (dg_split.cuh) for the
 * collapsed volume grid, and the choice of the meshes that take it.
 */
#include "dg_split.cuh"

namespace dg {

int split_tables(dg_mesh *m) {
  if (small_rk_fits(m)) return (int)cudaSuccess;
  if (m->rule == DG_RULE_SYMMETRIC) return split_tables_sym(m);
#define CALL(P, NE) split_tables_pq<P, NE, 0>(m)
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaSuccess;
}

int launch_split(const dg_mesh *m, const double *c, const double *u0, double *out, double *trace_out,
                 const double *fhat, const StageUpdate &su, int mode, double *copy, void *stream, int64_t e0,
                 int64_t e1) {
  cudaStream_t s = (cudaStream_t)stream;
  if (m->rule == DG_RULE_SYMMETRIC)
    return launch_split_sym(m, c, u0, out, trace_out, fhat, su, mode, copy, stream, e0, e1);
#define CALL(P, NE) run_split<P, NE, 0>(m, c, u0, out, trace_out, fhat, su, mode, copy, s, e0, e1)
  if (m->p == 1 && m->ne == 2) return CALL(1, 2);
  if (m->p == 2 && m->ne == 3) return CALL(2, 3);
  if (m->p == 3 && m->ne == 4) return CALL(3, 4);
  if (m->p == 3 && m->ne == 3) return CALL(3, 3);
  if (m->p == 4 && m->ne == 5) return CALL(4, 5);
  if (m->p == 5 && m->ne == 6) return CALL(5, 6);
#undef CALL
  return (int)cudaErrorInvalidValue;
}

int split_wave(const dg_mesh *m) { return m->num_sms * split_groups(m->p); }

}  // namespace dg
