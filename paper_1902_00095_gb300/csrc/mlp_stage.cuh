// Device and pinned buffers of a network's batches (internal header).
#pragma once
#include "learned.cuh"

namespace tp {

struct MlpStage {
  static constexpr size_t kBatchBytes = sizeof(float) * kMlpIn + 3 * sizeof(double) + sizeof(int);
  int cap = 0;              // samples that every buffer below holds
  float* X = nullptr;
  char* batch = nullptr;    // device copy of a training batch, kBatchBytes per sample
  char* hbatch = nullptr;   // pinned image of it, made at the first batch from host memory
  float* O = nullptr;
  float* partials = nullptr;
  Pool pool;

  MlpStage() = default;
  ~MlpStage() {
    if (hbatch) cudaFreeHost(hbatch);
  }
  // Room for n samples. `cap` counts only buffers that are all there: a growth
  // that runs out of memory gives back what it had and leaves none.
  void ensure(int n) {
    if (n <= cap) return;
    cap = 0;
    if (hbatch) cudaFreeHost(hbatch);
    hbatch = nullptr;
    pool.release();
    try {
      X = pool.alloc<float>((size_t)n * kMlpIn);
      batch = pool.alloc<char>((size_t)n * kBatchBytes);
      O = pool.alloc<float>((size_t)n * kMlpOut);
      partials = pool.alloc<float>(((size_t)n + 15) / 16 * kMlpPartial);
    } catch (...) {
      pool.free_all();
      throw;
    }
    cap = n;
  }
  char* host_image() {
    if (!hbatch && cudaMallocHost(&hbatch, (size_t)cap * kBatchBytes) != cudaSuccess) {
      cudaGetLastError();
      hbatch = nullptr;
      fail(TP_ENOMEM, "pinned memory for a training batch");
    }
    return hbatch;
  }
};

}  // namespace tp
