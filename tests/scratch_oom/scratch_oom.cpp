// Test-only program, no GPU: csrc/capi.cu over a stand-in for the allocator that fails once, at
// allocation argv[1] of the implicit scratch. The same request is then made again. Prints
//   <first status> <second status> <arrays missing after the second> <allocations in all>
#include <cstdio>
#include <cstdlib>
#include "../../paper_2304_09485_gb300/csrc/capi.cu"

namespace hgks {
thread_local int64_t g_launches = 0;
}
namespace {
int g_count = 0, g_fail = -1;
}

extern "C" {
cudaError_t cudaMalloc(void **p, size_t) {
  if (g_count++ == g_fail) return cudaErrorMemoryAllocation;
  *p = std::malloc(64);                   // never touched: the addresses only have to differ from null
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "no memory"; }
}

int main(int, char **argv) {
  const bool hex = std::atoi(argv[2]) != 0, mixed = std::atoi(argv[3]) != 0, fd = std::atoi(argv[4]) != 0;
  Mesh m;
  m.N = 1000;
  m.F = 2500;
  m.d.hex = hex;
  if (ensure_scratch(m, 0, false)) return 1;
  const int before = g_count, first_fail = std::atoi(argv[1]);
  if (first_fail >= 0) g_fail = before + first_fail;
  auto request = [&] {
    hgks_status st = ensure_scratch(m, 10, true, mixed);
    return st || !fd ? st : ensure_fd(m);
  };
  const hgks_status a = request(), b = request();
  const Scratch &s = m.s;
  const void *need[] = {s.jv64, s.dval, s.dinv, s.R, s.Gnew, s.dQ, s.w, s.t, s.hs, s.gram, s.z[0], s.z[1]};
  const void *need32[] = {s.jv32, s.dval32, s.dinv32, s.w32, s.t32, s.t232, s.red32, s.V32};
  const void *needfd[] = {s.Qp, s.Rp};
  int missing = mixed ? 0 : s.V == nullptr;
  for (const void *p : need) missing += p == nullptr;
  if (mixed)
    for (const void *p : need32) missing += p == nullptr;
  if (fd)
    for (const void *p : needfd) missing += p == nullptr;
  std::printf("%d %d %d %d\n", (int)a, (int)b, missing, g_count - before);
  return 0;
}
