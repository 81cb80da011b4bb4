// Two pieces of work on two streams, each by its own host thread (internal header).
#pragma once
#include <exception>
#include <system_error>
#include <thread>
#include "common.cuh"

namespace tp {

// on_s(s) by this thread and on_s2(s2) by a second one. Both see what was
// enqueued on s before the call, and s waits for what either enqueued, whether
// they return or throw: the caller may free, rewind or rewrite after an exception
// what the other side's kernels still use. This thread's exception goes first.
// Without a second thread to be had, one after the other.
template <class FA, class FB>
void fork_join(int device, cudaStream_t s, cudaStream_t s2, cudaEvent_t fork, cudaEvent_t join,
               FA on_s, FB on_s2) {
  TP_CUDA_TRY(cudaEventRecord(fork, s));
  TP_CUDA_TRY(cudaStreamWaitEvent(s2, fork, 0));
  std::exception_ptr ea, eb;
  auto second = [&]() {
    try {
      TP_CUDA_TRY(cudaSetDevice(device));
      on_s2(s2);
    } catch (...) {
      eb = std::current_exception();
    }
  };
  std::thread th;
  try {
    th = std::thread(second);
  } catch (const std::system_error&) {
  }
  try {
    on_s(s);
  } catch (...) {
    ea = std::current_exception();
  }
  if (th.joinable()) th.join();
  else second();
  cudaError_t e = cudaEventRecord(join, s2);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, join, 0);
  if (ea) std::rethrow_exception(ea);
  if (eb) std::rethrow_exception(eb);
  TP_CUDA_TRY(e);
}

}  // namespace tp
