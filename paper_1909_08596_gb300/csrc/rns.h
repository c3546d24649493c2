// FP64 matrix products on the 16-bit tensor cores through residues (rns.cu): the launch interface.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "internal.h"

namespace dmet {

// Device scratch of the residue products of one stream, and what its bounded waits report to.
struct RnsCtx {
  void* scratch = nullptr;
  size_t bytes = 0;
  int sms = 0;
  unsigned int* err = nullptr;
  unsigned long long wait_ns = 0;
  int withhold_loads = 0;  // test hook (tc::TcCtl)
};

// Whether a product of this shape is faster through residues than on the FP64 pipe (and fits the
// scratch); the launches return the number of kernels in *launches.
bool rns_takes_zgemm(const ZgemmArgs& a, const RnsCtx& c);
bool rns_takes_dsyrk(const DsyrkArgs& a, const RnsCtx& c);
cudaError_t rns_zgemm(const ZgemmArgs& a, int a_layout, bool conj_a, int b_layout, const RnsCtx& c, cudaStream_t s,
                      int* launches);
cudaError_t rns_dsyrk(const DsyrkArgs& a, const RnsCtx& c, cudaStream_t s, int* launches);

// Scratch in bytes with which a product runs in one chunk (less runs it in several).
size_t rns_need(const ZgemmArgs& a);
size_t rns_need(const DsyrkArgs& a);

}  // namespace dmet
