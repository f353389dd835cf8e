// Host-only run of an operator's workspace with a fake CUDA runtime whose k-th
// allocation fails. Prints one line per k: the status of the call that failed and
// how many parts are missing after a smaller call that succeeded. Compiled and
// read by tests/test_growth_cpu.py.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <map>

namespace fake {
int count = 0, fail_at = -1;
std::map<void*, int> live;
cudaError_t alloc(void** p, size_t n) {
  *p = nullptr;
  if (++count == fail_at) return cudaErrorMemoryAllocation;
  *p = std::calloc(1, n ? n : 1);
  live[*p] = 1;
  return cudaSuccess;
}
cudaError_t release(void* p) {
  live.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t fill(void* p) { return p ? cudaSuccess : cudaErrorInvalidValue; }
}  // namespace fake

#define cudaMalloc(p, n) fake::alloc((void**)(p), n)
#define cudaFree(p) fake::release((void*)(p))
#define cudaMallocHost(p, n) fake::alloc((void**)(p), n)
#define cudaFreeHost(p) fake::release((void*)(p))
#define cudaMemset(p, v, n) fake::fill((void*)(p))
#define cudaEventCreate(p) fake::alloc((void**)(p), 1)
#define cudaEventCreateWithFlags(p, f) fake::alloc((void**)(p), 1)
#define cudaEventDestroy(p) fake::release((void*)(p))
#define cudaStreamCreateWithFlags(p, f) fake::alloc((void**)(p), 1)
#define cudaStreamDestroy(p) fake::release((void*)(p))
#define cudaGetLastError() cudaSuccess

#include "ascg_api.cu"

static int missing(const Workspace& w) {
  int m = 0;
  for (const void* p : {(const void*)w.Y, (const void*)w.Y2, (const void*)w.q, (const void*)w.partials, (const void*)w.expp,
                        (const void*)w.emax_part, (const void*)w.counter, (const void*)w.G, (const void*)w.coords,
                        (const void*)w.params, (const void*)w.scal, (const void*)w.spec, (const void*)w.shifts,
                        (const void*)w.bst, (const void*)w.cgs, (const void*)w.res_hist, (const void*)w.ab_hist,
                        (const void*)w.h_bst, (const void*)w.h_seq, (const void*)w.h_cgs, (const void*)w.h_scal,
                        (const void*)w.ev_gram, (const void*)w.side, (const void*)w.ev[7], (const void*)w.ev_x[1]})
    m += p == nullptr;
  return m;
}

int main() {
  for (int grown = 0; grown < 2; ++grown)
    for (int k = 1; k < 200; ++k) {
      ascg_op op = new ascg_op_s();
      op->n = 1000;
      fake::fail_at = -1;
      if (grown && ensure(op, 9, 50) != ASCG_OK) return 2;  // a smaller workspace is there already
      fake::fail_at = fake::count + k;
      const ascg_status st = ensure(op, 17, 100);
      fake::fail_at = -1;
      const ascg_status again = ensure(op, 9, 50);
      std::printf("grown %d k %d status %d again %d missing %d\n", grown, k, (int)st, (int)again, missing(op->ws));
      op->ws.release();
      delete op;
      if (st == ASCG_OK) break;
    }
  std::printf("leaked %zu\n", fake::live.size());
  return 0;
}
