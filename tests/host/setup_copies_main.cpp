// Set-up copies of the mesh builder, with the weakest order that the CUDA
// runtime promises them: a host-to-device copy is staged when cudaMemcpy returns
// and reaches the "device" only with the next copy back to the host.  Prints, for
// a plain mesh and a union of two, how many copies were still on their way when
// the builder returned, and whether the union's segment bounds are on the device.
// Test infrastructure only.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "chns_internal.h"

namespace {
struct Copy {
  void *dst;
  std::vector<char> data;
};
std::vector<Copy> pending;
void land() {
  for (const Copy &c : pending) std::memcpy(c.dst, c.data.data(), c.data.size());
  pending.clear();
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = std::calloc(n ? n : 1, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind kind) {
  if (kind == cudaMemcpyHostToDevice) {
    const char *b = static_cast<const char *>(s);
    pending.push_back({d, std::vector<char>(b, b + n)});
  } else {
    land();
    std::memcpy(d, s, n);
  }
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  land();
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "host stand-in"; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFreeHost(void *) { return cudaSuccess; }
}

namespace chns {
chns_status build_mesh(int dim, int64_t n, const uint8_t *level, const uint32_t *anchor, int max_level,
                       const double lo[3], const double hi[3], chns_mesh *m);
chns_status build_union(const std::vector<const chns_mesh *> &ms, chns_mesh *u);
chns_status build_gather(chns_mesh *m);
}  // namespace chns

int main() {
  std::vector<const chns_mesh *> ms;
  for (int level = 1; level <= 2; ++level) {  // uniform 2D meshes of 4 and 16 leaves, Morton order
    std::vector<uint8_t> lv;
    std::vector<uint32_t> an;
    for (uint32_t k = 0; k < (1u << (2 * level)); ++k) {
      uint32_t a[2] = {0, 0};
      for (int b = 0; b < level; ++b)
        for (int d = 0; d < 2; ++d) a[d] |= ((k >> (2 * b + d)) & 1u) << b;
      lv.push_back(uint8_t(level));
      an.push_back(a[0]);
      an.push_back(a[1]);
    }
    chns_mesh *m = new chns_mesh;
    if (chns::build_mesh(2, int64_t(lv.size()), lv.data(), an.data(), level, nullptr, nullptr, m) != CHNS_OK ||
        chns::build_gather(m) != CHNS_OK)
      return 2;
    std::printf("mesh %zu\n", pending.size());
    land();
    ms.push_back(m);
  }
  chns_mesh *u = new chns_mesh;
  if (chns::build_union(ms, u) != CHNS_OK || chns::build_gather(u) != CHNS_OK) return 2;
  std::printf("union %zu\n", pending.size());
  bool same = u->inst_dof != nullptr;
  for (int q = 0; same && q <= u->n_inst; ++q) same = u->inst_dof[q] == u->inst_node_start[size_t(q)] * u->nf;
  std::printf("bounds %d\n", int(same));
  return 0;
}
