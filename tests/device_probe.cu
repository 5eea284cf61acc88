// Device functions of the library that no entry point exposes by themselves,
// for the tests: built with nvcc by tests/test_gpu_device.py.
#include <cstddef>
#include <type_traits>

#include "cg_common.cuh"
#include "cg_noise.h"

using namespace cgf;

namespace {

// One SC_BB reduction of given thread sums: ||b||^2 of the state.
template <typename T>
__global__ void k_reduce(const double* hi, const double* lo, double* partial, CgState* st, int seg,
                         int shares) {
  __shared__ double red[32];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  Acc<T> acc;
  if constexpr (std::is_same<T, float>::value) {
    acc.hi = (float)hi[i];
    acc.lo = (float)lo[i];
  } else if constexpr (std::is_same<T, df>::value) {
    acc.s = df((float)hi[i], (float)lo[i]);
  } else {
    acc.s = hi[i] + lo[i];
  }
  grid_reduce(red, partial, st, SC_BB, gridDim.x, blockIdx.x, blockDim.x / seg,
              [&](double* out) {
                __shared__ typename Acc<T>::total_t buf[512];
                segment_partials(acc.total(), buf, out, seg, shares);
              });
}

__global__ void k_normals(const double* tab, const uint4* words, int n, double2* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) normals_of(tab, words[i], out[i].x, out[i].y);
}

}  // namespace

// Normals of n Philox outputs; tab: device room for probe_noise_entries() doubles.
extern "C" int probe_normals(double* tab, const void* words, int n, void* out, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const std::vector<double> t = noise_tables();
  cudaError_t e = cudaMemcpy(tab, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return (int)e;
  k_normals<<<(n + 127) / 128, 128, 0, s>>>(tab, (const uint4*)words, n, (double2*)out);
  return (int)cudaGetLastError();
}
extern "C" int probe_noise_entries() { return kNoiseEntries; }

extern "C" int probe_reduce(int type, int ncta, int nthr, int seg, int shares,
                            const double* hi, const double* lo, double* partial, void* state, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  CgState* st = (CgState*)state;
  if (type == 0)
    k_reduce<float><<<ncta, nthr, 0, s>>>(hi, lo, partial, st, seg, shares);
  else if (type == 1)
    k_reduce<df><<<ncta, nthr, 0, s>>>(hi, lo, partial, st, seg, shares);
  else
    k_reduce<double><<<ncta, nthr, 0, s>>>(hi, lo, partial, st, seg, shares);
  return (int)cudaGetLastError();
}

extern "C" int probe_state_bytes() { return (int)sizeof(CgState); }
extern "C" int probe_bb_offset() { return (int)offsetof(CgState, bb); }
