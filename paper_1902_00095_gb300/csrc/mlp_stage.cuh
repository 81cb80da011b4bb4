// Device and pinned buffers of a network's batches (internal header).
#pragma once
#include "learned.cuh"

namespace tp {

struct MlpStage {
  static constexpr size_t kBatchBytes = sizeof(float) * kMlpIn + 3 * sizeof(double) + sizeof(int);
  // Batches from host memory go over in one copy from a pinned image up to this
  // many samples, and array by array straight from the caller's memory above it,
  // where writing the image costs more than the four copies it saves. A training
  // step with the image and without: 256 samples 45 and 45 us, 1024 51 and 56,
  // 3072 64 and 68, 4096 72 and 71, 8192 123 and 89, 20000 276 and 154.
  static constexpr int kImageMax = 3072;
  int cap = 0;              // samples that every buffer below holds
  char* batch = nullptr;    // device copy of a training batch, kBatchBytes per sample
  float* X = nullptr;       // that of inference inputs, in the same place
  char* hbatch = nullptr;   // pinned image of it, made at the first batch that uses one
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
      batch = pool.alloc<char>((size_t)n * kBatchBytes);
      X = reinterpret_cast<float*>(batch);
      O = pool.alloc<float>((size_t)n * kMlpOut);
      partials = pool.alloc<float>(((size_t)n + 15) / 16 * kMlpPartial);
    } catch (...) {
      pool.free_all();
      throw;
    }
    cap = n;
  }
  // room for min(cap, kImageMax) samples
  char* host_image() {
    const size_t n = cap < kImageMax ? cap : kImageMax;
    if (!hbatch && cudaMallocHost(&hbatch, n * kBatchBytes) != cudaSuccess) {
      cudaGetLastError();
      hbatch = nullptr;
      fail(TP_ENOMEM, "pinned memory for a training batch");
    }
    return hbatch;
  }
};

}  // namespace tp
