// FP64 gradient partial sums of nets and lattices (kernels of qk_grad.cuh).
#include "qk_grad.cuh"

namespace qk {

int launch_grad_partials_f64(const ColJob &job, uint32_t nrhs, const double *u, double *partial, cudaStream_t st,
                             bool pairs, const double *pcol) {
  if (job.family == QK_SI) {  // differences do not depend on the shift: one set of factors for all vectors
    const uint32_t nper = job.nr * nrhs;
    switch (job.alpha) {
      case 1: return launch_grad64<1, 1>(job, nullptr, 1, nper, u, pairs, pcol, partial, st);
      case 2: return launch_grad64<1, 2>(job, nullptr, 1, nper, u, pairs, pcol, partial, st);
      default: return fail(QK_EINVAL, "SI smoothness must be 1 or 2");
    }
  }
  switch (job.alpha) {
    case 1: return launch_grad64<0, 1>(job, job.Ct, job.nr, nrhs, u, 0, pcol, partial, st);
    case 2: return launch_grad64<0, 2>(job, job.Ct, job.nr, nrhs, u, 0, pcol, partial, st);
    case 3: return launch_grad64<0, 3>(job, job.Ct, job.nr, nrhs, u, 0, pcol, partial, st);
    case 4: return launch_grad64<0, 4>(job, job.Ct, job.nr, nrhs, u, 0, pcol, partial, st);
    default: return fail(QK_EINVAL, "DSI order must be 1..4");
  }
}

}  // namespace qk
