// Device functions of the library that no entry point exposes by themselves,
// for the tests: built with nvcc by tests/test_gpu_device.py.
#include <cstddef>
#include <type_traits>

#include "cg_common.cuh"

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

}  // namespace

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
