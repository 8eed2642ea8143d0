// k_ros4 for teams of 4 warps in the latency form (n <= 24, few reactors).
#include "ck_ros4.cuh"

namespace ck {

cudaError_t launch_ros4_w4_lat(const HostMech& hm, int64_t n, const double* p, double* y, const double* dt, double* h_io,
                           const SolverParams& sp, int32_t* steps, int32_t* status, int32_t* queue,
                           cudaStream_t st, const LaunchCfg& cfg, double* scratch, size_t scratch_bytes,
                           bool may_alloc) {
  return launch_ros4_team<128, 4>(hm, n, p, y, dt, h_io, sp, steps, status, queue, st, cfg, scratch, scratch_bytes,
                                  may_alloc);
}

}  // namespace ck
