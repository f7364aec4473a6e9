// Host-side declarations shared by the C-ABI layer (api.cu) and the kernel files.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "lbm_device.cuh"

namespace lbm {

constexpr int kResidualMaxBlocks = 2048;  // partial-sum slots of the residual reduction

int record_error(int code, const char* msg);

// Launch of a kernel that begins with wait_prerequisites(): it may be scheduled while the kernel
// before it on the stream still runs.  Such a kernel has no __restrict__ parameter (other than tables that
// only the host writes) and reads what an earlier kernel may write by ordinary loads: a promise that the
// memory does not change would let the compiler move the load up before the wait.
template <class... P, class... A>
inline cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
}  // namespace lbm
struct lbm_config;
namespace lbm {
int validate_config(const ::lbm_config* c);
void params_from_config(const ::lbm_config& k, int prec, int pitch, int64_t plane, StepParams& P);
// The fields that differ between the lattices of a batch whose lattices share rho0, s_e, s_q and
// the storage scale (the batched per-item step then takes everything else from one lattice's
// parameters passed by value, in the kernel's constant bank, instead of staging the whole set).
struct BatchRec {
  const void* src;
  void* dst;
  const float* phi;
  const float* K;
  const float* uw;
  int64_t plane;
  int nx, ny, pitch, bc_x, bc_y, forch;
  float nu, s_v, ax, ay;
};

int64_t batch_items(int nx, int ny, int bc_y, int nt, int flat);
cudaError_t launch_step_batch_shared(const StepParams& U, const BatchRec* R, const StepParams* Pd, const int64_t* item_start,
                                     const int* item_lattice, int64_t total, int prec, int nt, int flat, bool graph, cudaStream_t s);
int batch_max_ctas_per_sm(int prec, int nt);
cudaError_t launch_step_batch(const StepParams* Pd, const int64_t* item_start, const int* item_lattice, int n, int64_t total, int prec,
                              int nt, int grid, int flat, cudaStream_t s);
cudaError_t launch_step(const StepParams& P, int prec, bool het, bool thermal, cudaStream_t s);
int sm_count();  // SMs of the current device
constexpr uint64_t kMarchBytes = 100ull << 20;  // FP32 state (both buffers) from which steps are taken in pairs
bool march_shape(const StepParams& P, int prec, bool het, bool thermal);
bool march_takes(const StepParams& P, int prec, bool het, bool thermal);
int march_kernels(const StepParams& P, int prec, bool het, bool thermal);
// A warp's work in the batched pair kernels: rows [ya, yb) (none if equal) of a strip of a lattice.
struct MarchItem {
  int lattice, strip, ya, yb, strips, wrap;
};
void march_items(const StepParams& P, int lattice, std::vector<MarchItem>& side, std::vector<MarchItem>& main);
cudaError_t launch_march_batch(const StepParams* Pd, const MarchItem* side, int n_side, const MarchItem* main, int n_main, bool pressure,
                               cudaStream_t s);  // pressure: a lattice has pressure columns
int tile_steps(const StepParams& P, int prec, bool het, bool thermal);
cudaError_t launch_tile(const StepParams& P, int prec, bool het, bool thermal, int steps, cudaStream_t s);
cudaError_t launch_march(const StepParams& P, int prec, bool het, bool thermal, cudaStream_t s);
cudaError_t launch_step_inplace(const StepParams& P, int prec, bool het, bool thermal, cudaStream_t s);
int64_t inplace_items(int nx, int ny, int bc_x, int bc_y);
cudaError_t launch_step_batch_inplace(const StepParams* Pd, const int64_t* item_start, const int* item_lattice, int64_t total, int prec,
                                      int parity, cudaStream_t s);
cudaError_t launch_put_inplace(const StepParams& P, int prec, bool het, const float* f, const float* g, bool flow, bool temp,
                               float p0, float ux0, float uy0, int phip_uniform, float T_init, cudaStream_t s);
cudaError_t launch_medium(const float* eps, const float* K, float phi_u, float K_u, int nx, int ny, int pitch, float* phi_out,
                          float* K_out, unsigned int* err, int log_k, cudaStream_t s);
cudaError_t launch_viscous_rate(const float* J, int nx, int ny, int pitch, float nu, float* sv, unsigned int* err, cudaStream_t s);
cudaError_t launch_init(const StepParams& P, int prec, bool het, bool thermal, float p0, float ux0, float uy0, int phip_uniform,
                        float T_init, bool flow, bool temp, cudaStream_t s);
cudaError_t launch_import(const StepParams& P, int prec, const float* f, const float* g, cudaStream_t s);
cudaError_t launch_export(const StepParams& P, int prec, bool het, bool thermal, float* f, float* g, cudaStream_t s);
cudaError_t launch_macros(const StepParams& P, int prec, bool het, bool thermal, float* p, float* ux, float* uy, float* T,
                          cudaStream_t s);
cudaError_t launch_copy_small(float* dst, const float* src, int n, cudaStream_t s);
cudaError_t launch_probe(const StepParams& P, int prec, bool het, bool thermal, int x, int y, float* out, cudaStream_t s);
int residual_blocks(int nx, int ny);
cudaError_t launch_residual(const StepParams& P, int prec, bool het, bool thermal, const void* prev, const void* gprev,
                            const float* uprev, double* partial, int nblocks, double* out, cudaStream_t s);
cudaError_t launch_nusselt(const StepParams& P, int prec, int side, double* out, cudaStream_t s);

cudaError_t launch_adj_seed(const StepParams& P, int prec, bool het, float* nu_out, float* g_l, float* g_phi, int kind,
                            const float* tux, const float* tuy, double* partial, int nblocks, double* loss_out, cudaStream_t s);
cudaError_t launch_adj_wall(const StepParams& P, int prec, bool het, const void* buf, float* nu, float* g_l, float* g_phi,
                            cudaStream_t s);
cudaError_t launch_adj_nee(const StepParams& P, int prec, bool het, const void* buf, float* nu, float* g_l, float* g_phi,
                           cudaStream_t s);
cudaError_t launch_adj_step(const StepParams& P, int prec, bool het, const void* buf, const float* nu_in, float* nu_out, float* g_l,
                            float* g_phi, cudaStream_t s);
cudaError_t launch_adj_init(const StepParams& P, bool het, const float* nu, float* g_phi, float p0, float ux0, float uy0,
                            int phip_uniform, cudaStream_t s);
cudaError_t launch_adj_fold(float* l32, float* p32, double* l64, double* p64, int64_t n, cudaStream_t s);

}  // namespace lbm
