// Host build of the cluster solve's plans and launches (cgcluster.cuh) over a stand-in for the three CUDA calls they make:
// the shared-memory limit of each kernel as the process keeps it, and what a launch then may ask for.
#include <cuda_runtime.h>

#include <map>

namespace fake {
std::map<const void*, int> limit;  // per kernel, for the whole process (48 KB until it is set)
int before_launch[2] = {0, 0};     // box that another thread plans just before a launch (rows, columns)
long long rejected = 0, launched = 0;
int allowed(const void* f) {
  const auto i = limit.find(f);
  return i == limit.end() ? 48 * 1024 : i->second;
}
template <class F>
cudaError_t set_attribute(F* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[(const void*)f] = v;
  return cudaSuccess;
}
template <class F>
cudaError_t max_clusters(int* n, F* f, const cudaLaunchConfig_t* c) {
  *n = (int)c->dynamicSmemBytes <= allowed((const void*)f) ? 9 : 0;
  return cudaSuccess;
}
void other_thread();
template <class F, class A>
cudaError_t launch(const cudaLaunchConfig_t* c, F* f, const A&) {
  other_thread();
  ++launched;
  if ((int)c->dynamicSmemBytes <= allowed((const void*)f)) return cudaSuccess;
  ++rejected;
  return cudaErrorInvalidValue;
}
}  // namespace fake
#define cudaFuncSetAttribute fake::set_attribute
#define cudaOccupancyMaxActiveClusters fake::max_clusters
#define cudaLaunchKernelEx fake::launch
#include "cgcluster.cuh"

void fake::other_thread() {
  if (before_launch[0]) mcrt::cg_plan(before_launch[0], before_launch[1], 1000);
}

// A solve of a box of rows x w, while another thread plans a box of rows2 x w2 between this one's plan and its launch.
// 0: launched, -1: no plan, 1: the launch was rejected
extern "C" int host_cg_solve(int rows, int w, int rows2, int w2) {
  const mcrt::CgPlan L = mcrt::cg_plan(rows, w, 1000);
  if (!L.nc) return -1;
  fake::before_launch[0] = rows2;
  fake::before_launch[1] = w2;
  mcrt::CgBox B = {};
  const cudaError_t e = mcrt::cg_solve(B, L, nullptr);
  fake::before_launch[0] = 0;
  return e == cudaSuccess ? 0 : 1;
}

// box of the cells with mask 2, and whether a box of its size has a plan
extern "C" int host_cg_box(const signed char* mask, int nr, int nt, int* box) {
  mcrt::cg_box(mask, nr, nt, box);
  return mcrt::cg_plan(box[1] - box[0], box[3] - box[2], 1000).nc;
}
