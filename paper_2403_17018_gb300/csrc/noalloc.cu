// henry_residual_jacobian_noalloc: henry_residual_jacobian for callers that
// cannot allocate device memory during a call (see henry.h). The evaluation
// needs no scratch memory; the entry point keeps its documented batch limit.
#include <cuda_runtime.h>

#include <string>

#include "../../include/henry.h"
#include "solver.h"

namespace henry {
cudaError_t launch_residual_jacobian(const Phys& P, const Geom& G, double tau, int B,
                                     const double* phi, const double* K, const double* qin,
                                     const double* p, const double* c, const double* c_old,
                                     double* R, double* J, cudaStream_t s);
}  // namespace henry

namespace {

constexpr size_t kNoAllocCells = 209715;   // largest B nx ny accepted

int fail(int code, const std::string& msg) {
  henry::set_last_error(msg);
  return code;
}

}  // namespace

extern "C" int henry_residual_jacobian_noalloc(const henry_config* cfg, int nx, int ny, double tau,
                                               int B, const double* phi, const double* K,
                                               const double* qin, const double* p,
                                               const double* c, const double* c_old, double* R,
                                               double* J, void* stream) {
  if (!cfg) return fail(HENRY_E_INVALID, "config is NULL");
  if (nx < 2 || ny < 1 || B < 0 || B > HENRY_MAX_BATCH || !(tau > 0))
    return fail(HENRY_E_INVALID, "bad sizes (nx >= 2, ny >= 1, 0 <= B <= 65535, tau > 0)");
  if (B == 0) return HENRY_OK;
  if (!phi || !K || !qin || !p || !c || !c_old || !R) return fail(HENRY_E_INVALID, "NULL argument");
  const size_t cells = (size_t)B * (size_t)nx * (size_t)ny;
  if (cells > kNoAllocCells)
    return fail(HENRY_E_INVALID, "henry_residual_jacobian_noalloc: B*nx*ny = " + std::to_string(cells) +
                                     " exceeds the maximum of " + std::to_string(kNoAllocCells) + " cells");
  henry::Phys P{cfg->rho0, cfg->rho1 - cfg->rho0, cfg->mu, cfg->g, cfg->D, cfg->K0, cfg->phi0,
                cfg->q0, cfg->Lx, cfg->Ly};
  henry::Geom G{nx, ny, cfg->Lx / nx, cfg->Ly / ny};
  const cudaError_t e = henry::launch_residual_jacobian(P, G, tau, B, phi, K, qin, p, c, c_old, R, J,
                                                        (cudaStream_t)stream);
  if (e != cudaSuccess) return fail(HENRY_E_CUDA, std::string("launch: ") + cudaGetErrorString(e));
  return HENRY_OK;
}
