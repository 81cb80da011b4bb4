// Memory of the coupling blocks stored by grid direction (internal header).
#pragma once
#include "common.cuh"

namespace tp {

// A_pT and A_Tp by grid direction ([7][N] each, launch_coupling_planes). They
// make the preconditioner's two products faster and cost 112 bytes per cell; the
// CSR planes hold the same values, so without memory for them there are none.
struct CouplingPlanes {
  double *ApT = nullptr, *ATp = nullptr;
  bool refused = false;  // no memory when last asked for (cleared by a build)
  Pool pool;
  // planes of up to this many bytes come from the context's pool and stay there
  // (an allocation of their own takes some 50 us of a new context's first build)
  static constexpr size_t kShared = size_t(4) << 20;

  // both planes of N cells, or neither (false)
  bool ensure(size_t N, Pool& shared) {
    if (ApT) return true;
    if (refused) return false;
    const size_t each = (7 * N + 31) / 32 * 32;
    try {
      Pool& from = 2 * each * sizeof(double) <= kShared ? shared : pool;
      double* p = from.alloc<double>(2 * each);
      ApT = p;
      ATp = p + each;
    } catch (const Error& e) {
      if (e.code != TP_ENOMEM) throw;
      refused = true;
      return false;
    }
    return true;
  }
  // memory of their own, which give_back() frees for an allocation that cannot be
  // done without; nothing may be reading them
  bool owned() const { return pool.reserved() > 0; }
  void give_back() {
    ApT = ATp = nullptr;
    refused = true;
    pool.free_all();
  }
};

}  // namespace tp
