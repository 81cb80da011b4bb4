// Host logic of the library's headers against a fake CUDA runtime (no GPU):
// compiled and run by test_host_state.py, one check per argument. A check that
// fails prints its line and exits with 1.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>

#include "fork_join.cuh"
#include "in_place.cuh"
#include "mlp_stage.cuh"
#include "per_device.cuh"
#include "planes.cuh"

// ---------------------------------------------------------------- fake runtime
static size_t g_device_limit = ~size_t(0), g_device_used = 0;
static std::map<char*, size_t> g_device, g_pinned;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_device_used + n > g_device_limit) return cudaErrorMemoryAllocation;
  static char* next = reinterpret_cast<char*>(size_t(1) << 40);  // addresses only
  *p = next;
  next += n + 4096;
  g_device[static_cast<char*>(*p)] = n;
  g_device_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  g_device_used -= g_device.at(static_cast<char*>(p));
  g_device.erase(static_cast<char*>(p));
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = std::malloc(n);
  g_pinned[static_cast<char*>(*p)] = n;
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void* p) {
  g_pinned.erase(static_cast<char*>(p));
  std::free(p);
  return cudaSuccess;
}
static int g_dev = 0, g_attributes = 0;
cudaError_t cudaGetDeviceCount(int* n) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = g_dev;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) {
  *v = 100 + d;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
  if (bytes < 0) return cudaErrorInvalidValue;
  ++g_attributes;
  return cudaSuccess;
}
static const char* g_where[8];  // what s and s2 were made to wait for, in order
static int g_waits = 0;
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  g_where[g_waits++ & 7] = reinterpret_cast<size_t>(s) == 1
                               ? (reinterpret_cast<size_t>(e) == 4 ? "s:join" : "s:fork")
                               : (reinterpret_cast<size_t>(e) == 3 ? "s2:fork" : "s2:join");
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
}

#define CHECK(x)                                             \
  do {                                                       \
    if (!(x)) {                                              \
      std::printf("%s:%d: %s\n", __FILE__, __LINE__, #x);    \
      std::exit(1);                                          \
    }                                                        \
  } while (0)

// [p, p + n) lies in one live allocation
static bool inside(const std::map<char*, size_t>& m, const void* p, size_t n) {
  const char* c = static_cast<const char*>(p);
  for (const auto& a : m)
    if (c >= a.first && c + n <= a.first + a.second) return true;
  return false;
}

// a growth of a network's batch buffers that runs out of memory at any of them
// leaves nothing that a later, smaller batch could run past
static void mlp_growth() {
  for (size_t limit = 8u << 20; limit < (1700u << 20); limit += 8u << 20) {
    tp::MlpStage st;
    g_device_limit = ~size_t(0);
    st.ensure(64);
    st.host_image();
    g_device_limit = limit;
    bool failed = false;
    try {
      st.ensure(1000000);
    } catch (const tp::Error& e) {
      failed = e.code == TP_ENOMEM;
    }
    CHECK(failed == (st.cap == 0));
    g_device_limit = ~size_t(0);
    const size_t n = 5000;
    st.ensure((int)n);
    CHECK(inside(g_device, st.X, n * tp::kMlpIn * sizeof(float)));
    CHECK(inside(g_device, st.batch, n * tp::MlpStage::kBatchBytes));
    CHECK(inside(g_device, st.O, n * tp::kMlpOut * sizeof(float)));
    CHECK(inside(g_device, st.partials, (n + 15) / 16 * tp::kMlpPartial * sizeof(float)));
    CHECK(inside(g_pinned, st.host_image(),
                 tp::MlpStage::kImageMax * tp::MlpStage::kBatchBytes));
  }
  CHECK(g_device.empty() && g_pinned.empty());
}

// memory for one plane but not for two: neither is there, now and when asked
// again, and both once there is room after a build
static void coupling_planes() {
  for (size_t N : {size_t(1001), size_t(1000001)}) {
    tp::CouplingPlanes p;
    tp::Pool shared;
    shared.alloc<char>(1);
    if (N < 5000) shared.alloc<char>(shared.reserved() - 7 * N * sizeof(double) - 512);
    g_device_limit = g_device_used + 7 * N * sizeof(double);
    if (N < 5000) g_device_limit = g_device_used;
    CHECK(!p.ensure(N, shared) && !p.ApT && !p.ATp);
    g_device_limit = ~size_t(0);
    CHECK(!p.ensure(N, shared) && !p.ApT && !p.ATp);
    p.refused = false;
    CHECK(p.ensure(N, shared));
    CHECK(inside(g_device, p.ApT, 7 * N * sizeof(double)));
    CHECK(inside(g_device, p.ATp, 7 * N * sizeof(double)));
    CHECK(p.ATp >= p.ApT + 7 * N && p.owned() == (N > 5000));
  }
  CHECK(g_device.empty());
}

// what a pointer query would say: one allocation of 4096 bytes at 1 << 40
static CUmemorytype g_type;
static int g_owner;
static CUresult fake_query(unsigned n, CUpointer_attribute* what, void** to, CUdeviceptr) {
  for (unsigned k = 0; k < n; ++k) {
    if (what[k] == CU_POINTER_ATTRIBUTE_MEMORY_TYPE) *static_cast<CUmemorytype*>(to[k]) = g_type;
    if (what[k] == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR)
      *static_cast<CUdeviceptr*>(to[k]) = CUdeviceptr(1) << 40;
    if (what[k] == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *static_cast<size_t*>(to[k]) = 4096;
    if (what[k] == CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL) *static_cast<int*>(to[k]) = g_owner;
  }
  return CUDA_SUCCESS;
}

// a kernel takes only aligned memory of its own device, inside one allocation
static void in_place() {
  const char* base = reinterpret_cast<char*>(size_t(1) << 40);
  auto usable = [&](int device, size_t byte, size_t n) {
    return tp::usable_in_place(fake_query, 2, device, reinterpret_cast<const double*>(base + byte), n);
  };
  g_type = CU_MEMORYTYPE_DEVICE;
  g_owner = 1;
  CHECK(usable(1, 0, 512) && usable(1, 8, 511) && usable(1, 4088, 1));
  CHECK(!usable(0, 0, 512));                         // another GPU's
  CHECK(!usable(1, 8, 512) && !usable(1, 0, 513));   // past the end
  CHECK(!usable(1, 4, 1));                           // unaligned
  g_owner = 0;
  CHECK(usable(0, 0, 512) && !usable(1, 0, 512));
  const double* p = reinterpret_cast<const double*>(base);
  CHECK(tp::usable_in_place(fake_query, 1, 0, p, 512) && !tp::usable_in_place(fake_query, 1, 0, p, 513));
  g_type = CU_MEMORYTYPE_HOST;
  CHECK(!usable(0, 0, 1) && !tp::usable_in_place(fake_query, 1, 0, p, 1));
  CHECK(!tp::usable_in_place<double>(nullptr, 1, 0, nullptr, 1));
}

// the first stream waits for the second's work however the two sides end, and
// an exception of either leaves the call after both are done
static void fork_join() {
  const auto s = reinterpret_cast<cudaStream_t>(1), s2 = reinterpret_cast<cudaStream_t>(2);
  const auto fork = reinterpret_cast<cudaEvent_t>(3), join = reinterpret_cast<cudaEvent_t>(4);
  for (int fail = 0; fail < 4; ++fail) {
    g_waits = 0;
    int done = 0, code = 0, waits_on_s = -1, waits_on_s2 = -1;
    try {
      tp::fork_join(
          0, s, s2, fork, join,
          [&](cudaStream_t t) {
            CHECK(t == s);
            waits_on_s = g_waits;
            if (fail & 1) tp::fail(TP_ENOMEM, "first");
          },
          [&](cudaStream_t t) {
            CHECK(t == s2);
            waits_on_s2 = g_waits;
            done = 1;
            if (fail & 2) tp::fail(TP_SETUP_FAILED, "second");
          });
    } catch (const tp::Error& e) {
      code = e.code;
    }
    CHECK(done && waits_on_s == 1 && waits_on_s2 == 1);  // s2 waits for s before either
    CHECK(code == (fail & 1 ? TP_ENOMEM : fail & 2 ? TP_SETUP_FAILED : 0));
    CHECK(g_waits == 2 && !std::strcmp(g_where[0], "s2:fork") && !std::strcmp(g_where[1], "s:join"));
  }
}

// a kernel's shared memory is allowed once on every device it is launched on,
// and what a device answers is that device's
static void per_device() {
  static tp::PerDevice<bool> allowed;
  const void* kernel = &g_dev;
  for (int round = 0; round < 3; ++round)
    for (g_dev = 0; g_dev < 4; ++g_dev) {
      tp::allow_smem(allowed, kernel, 100 << 10);
      CHECK(g_attributes == (round ? 4 : g_dev + 1));
      CHECK(tp::device_sms() == 100 + g_dev);
    }
  static tp::PerDevice<bool> failing;
  g_dev = 1;
  bool threw = false;
  try {
    tp::allow_smem(failing, kernel, size_t(-1));
  } catch (const tp::Error&) {
    threw = true;
  }
  tp::allow_smem(failing, kernel, 1 << 10);  // tried again
  CHECK(threw && g_attributes == 5);
}

int main(int, char** argv) {
  const struct {
    const char* name;
    void (*run)();
  } checks[] = {{"mlp_growth", mlp_growth}, {"coupling_planes", coupling_planes},
                {"in_place", in_place},
                {"fork_join", fork_join},
                {"per_device", per_device}};
  for (const auto& c : checks)
    if (std::strcmp(argv[1], c.name) == 0) {
      c.run();
      return 0;
    }
  std::printf("no such check\n");
  return 1;
}
