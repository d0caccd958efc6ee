// Internal launcher table: one entry per (storage precision, species count).
#pragma once
#include <cuda_runtime.h>
#include "device.cuh"

namespace pslbm {

// SMs of the device (152 on a whole GB300).
inline int device_sms() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
      cudaGetLastError();
      v = 152;
    }
    return v;
  }();
  return n;
}

struct Launchers {
  // work: the VOP chunks of a batch (null for one simulation); nwork: their number
  void (*vop)(cudaStream_t, const DevInst*, const Work* work, int nwork);
  void (*amend)(cudaStream_t, int ninst, const DevInst*);
  // both in one launch, a block an instance
  void (*vop_amend)(cudaStream_t, int ninst, const DevInst*);
  void (*init)(cudaStream_t, DevInst*, const uint8_t*, const double*, const double*, const double*, long long N);
  void (*fields)(cudaStream_t, const DevInst*, long long N, double*, double*, double*, double*, double*, uint8_t*);
  // out: NBUD doubles, then the step count and the status (64-bit words)
  void (*budget)(cudaStream_t, const DevInst*, double* part, double* out);
  // potentials and collide-stream kernels, a warp per work entry: parts
  // of the fluid list (the first nstream entries of one simulation), then chunks
  // of 32 reservoir nodes
  void (*pot)(cudaStream_t, const Work*, int nwork, int nstream, const DevInst*, const DevInst& Ik, int mode);
  void (*move)(cudaStream_t, const Work*, int nwork, int nstream, const DevInst*, const DevInst& Ik, int mode);
};

// prec: 0 FP64, 1 FP32, 2 FP32 + half solutes, 3 FP32 + bfloat16 solutes; ns 0..MAXS
const Launchers* launchers(int prec, int ns);

}  // namespace pslbm
