// Host-only harness for csrc/dev_mem.h over a fake device of a few bytes: every CUDA call that the
// header makes is defined here.  Reads commands from stdin, one answer a line:
//   device TOTAL        a new, empty device         -> ok
//   alloc N             DevMem::alloc               -> free bytes | nomem
//   optional N SPARE    DevMem::optional            -> free bytes | none
//   between LEAST WANT SPARE                        -> got free | nomem
//   release             the last allocation         -> free bytes
//   error               cudaGetLastError            -> code
//   drop                end of the DevMem           -> free bytes
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <string>

#include "dev_mem.h"

static size_t g_total = 0, g_used = 0;
static std::map<void *, size_t> g_size;
static cudaError_t g_last = cudaSuccess;

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
  if (g_used + n > g_total) return g_last = cudaErrorMemoryAllocation;
  *p = std::malloc(1);
  g_size[*p] = n;
  g_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  g_used -= g_size[p];
  g_size.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
  *f = g_total - g_used;
  *t = g_total;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
}

int main() {
  auto mem = std::make_unique<bd::DevMem>();
  char c[32];
  size_t a, b, s;
  while (std::scanf("%31s", c) == 1) {
    const std::string cmd = c;
    try {
      if (cmd == "device") {
        if (std::scanf("%zu", &a) != 1) return 1;
        mem = std::make_unique<bd::DevMem>();
        g_total = a;
        std::printf("ok\n");
      } else if (cmd == "alloc") {
        if (std::scanf("%zu", &a) != 1) return 1;
        mem->alloc<unsigned char>(a);
        std::printf("%zu\n", g_total - g_used);
      } else if (cmd == "optional") {
        if (std::scanf("%zu %zu", &a, &s) != 2) return 1;
        if (mem->optional<unsigned char>(a, s)) std::printf("%zu\n", g_total - g_used);
        else std::printf("none\n");
      } else if (cmd == "between") {
        if (std::scanf("%zu %zu %zu", &a, &b, &s) != 3) return 1;
        size_t got = 0;
        mem->between(a, b, s, &got);
        std::printf("%zu %zu\n", got, g_total - g_used);
      } else if (cmd == "release") {
        mem->release(mem->ptrs.back());
        std::printf("%zu\n", g_total - g_used);
      } else if (cmd == "error") {
        std::printf("%d\n", (int)cudaGetLastError());
      } else if (cmd == "drop") {
        mem.reset();
        std::printf("%zu\n", g_total - g_used);
        mem = std::make_unique<bd::DevMem>();
      }
    } catch (const bd::Status &e) {
      std::printf(e.code == BD_ERR_NOMEM ? "nomem\n" : "status %d\n", e.code);
    }
  }
  return 0;
}
