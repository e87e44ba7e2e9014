// Shared by the sweep translation units (sweep.cu, wavefront.cu) and dsa.cu: launch arguments, vector loads, shared-memory
// grants.
#pragma once
#include <atomic>

#include "dfloat.cuh"
#include "internal.h"

namespace rte {

struct SweepArgs {
  const InstInfo* inst;
  const UDir* udir;
  const SweepTask* tasks;
  int ntasks;
  const void* linv;     // compute type: cell inverses, or the FP32 tables that launch_wave puts here
  const void* sig_s;    // compute type, [B][R]; null: no Sigma_s scaling of the input
  const void* src;      // input type, scalar vector
  int with_bc;
  int inflow_mask;      // faces carrying the inflow: 1 x-low, 2 x-high, 4 y-low, 8 y-high
  void* partial;        // compute type, [tasks_per_inst * off_b + t * N_b + i]
  int tasks_per_inst;
  void* psi;            // compute type, angular vector, or null
  int ndir, nu, R, rx, ry;
  const int* active;    // [B] or null
  int smem_per_warp;    // elements of the compute type
  int psi_unique;       // angular output: 0 = all N_Omega directions, 1 = one block per unique direction
};

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
  __device__ static void load(const float* p, float& a, float& b, float& c, float& d) {
    float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x; b = v.y; c = v.z; d = v.w;
  }
  __device__ static void store(float* p, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
  }
};
template <>
struct Vec4<double> {
  __device__ static void load(const double* p, double& a, double& b, double& c, double& d) {
    double2 v0 = reinterpret_cast<const double2*>(p)[0];
    double2 v1 = reinterpret_cast<const double2*>(p)[1];
    a = v0.x; b = v0.y; c = v1.x; d = v1.y;
  }
  __device__ static void store(double* p, double a, double b, double c, double d) {
    reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
    reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
  }
};

template <>
struct Vec4<dfloat> {
  __device__ static void load(const dfloat* p, dfloat& a, dfloat& b, dfloat& c, dfloat& d) {
    const float4 v0 = reinterpret_cast<const float4*>(p)[0];
    const float4 v1 = reinterpret_cast<const float4*>(p)[1];
    a = dfloat(v0.x, v0.y); b = dfloat(v0.z, v0.w); c = dfloat(v1.x, v1.y); d = dfloat(v1.z, v1.w);
  }
  __device__ static void store(dfloat* p, dfloat a, dfloat b, dfloat c, dfloat d) {
    reinterpret_cast<float4*>(p)[0] = make_float4(a.hi, a.lo, b.hi, b.lo);
    reinterpret_cast<float4*>(p)[1] = make_float4(c.hi, c.lo, d.hi, d.lo);
  }
};

// Dynamic shared memory above the 48 KB default must be granted per kernel with cudaFuncSetAttribute, which
// acts on the current device only; granted[dev] remembers the size already granted on each device (zero-
// initialised statics), so a process that drives several GPUs grants it on each of them.
constexpr int kMaxDevices = 64;
template <typename K>
static int grant_smem(K kern, size_t smem, std::atomic<size_t>* granted) {
  if (smem <= 48 * 1024) return RTE_OK;
  int dev = 0;
  RTE_CHECK_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("sweep: device ordinal beyond the supported range");
    return RTE_ERR_UNSUPPORTED;
  }
  if (smem > granted[dev].load(std::memory_order_acquire)) {
    RTE_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    granted[dev].store(smem, std::memory_order_release);
  }
  return RTE_OK;
}

// wavefront.cu: the operator's sweeps (no angular output) on 2D meshes with cross sections per region.  in64: the input
// vector is FP64 (FP32 otherwise; double-float sweeps read pairs).  wave_smem gives a shape's shared memory,
// wave_shape_ok whether it is built and fits the problem.
size_t wave_smem(const rte_problem* p, int prec, WaveShape s);
bool wave_shape_ok(const rte_problem* p, int prec, WaveShape s);
// the shapes a cost estimate ranks first for the problem, best first, at most `keep`
std::vector<WaveShape> wave_shapes(const rte_problem* p, int prec, int keep);
// the shape it ranks first with D directions per task and one row per lane
WaveShape wave_shape_for(const rte_problem* p, int prec, int D);
int launch_wave(const rte_problem* p, int prec, WaveShape s, bool in64, const SweepArgs& a, cudaStream_t st);

}  // namespace rte
