// Device memory of a handle, and the status that a failing CUDA call becomes (host only).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <stdexcept>
#include <string>
#include <vector>

#include "bidomain.h"

namespace bd {

struct Status : std::runtime_error {
  int code;
  Status(int c, const std::string &m) : std::runtime_error(m), code(c) {}
};

inline void ck(cudaError_t e, const char *what) {
  if (e == cudaErrorMemoryAllocation) throw Status(BD_ERR_NOMEM, what);
  if (e != cudaSuccess) throw Status(BD_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

struct DevMem {
  std::vector<void *> ptrs;
  template <class X>
  X *alloc(size_t n) {
    X *p = attempt<X>(n);
    if (!p) throw Status(BD_ERR_NOMEM, "cudaMalloc");
    return p;
  }
  // for what a handle can do without: nullptr when it would leave less than `spare` bytes
  template <class X>
  X *optional(size_t n, size_t spare) {
    size_t free_b = 0, total = 0;
    ck(cudaMemGetInfo(&free_b, &total), "cudaMemGetInfo");
    if (free_b < spare || free_b - spare < std::max<size_t>(n, 1) * sizeof(X)) return nullptr;
    return attempt<X>(n);
  }
  // `want` bytes, a half, a quarter, ... that leave `spare`; `least` whatever they leave
  unsigned char *between(size_t least, size_t want, size_t spare, size_t *got) {
    for (size_t b = want; b > least; b /= 2)
      if (unsigned char *p = optional<unsigned char>(b, spare)) {
        *got = b;
        return p;
      }
    *got = least;
    return alloc<unsigned char>(least);
  }
  void release(void *p) {
    auto it = std::find(ptrs.begin(), ptrs.end(), p);
    if (it == ptrs.end()) return;
    ptrs.erase(it);
    cudaFree(p);
  }
  template <class X>
  X *upload(const std::vector<X> &v, cudaStream_t s) {
    X *p = alloc<X>(v.size());
    if (!v.empty()) ck(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(X), cudaMemcpyHostToDevice, s), "upload");
    return p;
  }
  ~DevMem() {
    for (void *p : ptrs) cudaFree(p);
  }

 private:
  template <class X>
  X *attempt(size_t n) {
    void *p = nullptr;
    const cudaError_t e = cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(X));
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();  // reported here: later checks of this thread must not find it again
      return nullptr;
    }
    ck(e, "cudaMalloc");
    ptrs.push_back(p);
    return static_cast<X *>(p);
  }
};

}  // namespace bd
