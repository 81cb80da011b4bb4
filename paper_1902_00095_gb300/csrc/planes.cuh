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

  // both planes of N cells, or neither (false)
  bool ensure(size_t N) {
    if (ApT) return true;
    if (refused) return false;
    const size_t each = (7 * N + 31) / 32 * 32;
    try {
      double* p = pool.alloc<double>(2 * each);
      ApT = p;
      ATp = p + each;
    } catch (const Error& e) {
      if (e.code != TP_ENOMEM) throw;
      refused = true;
      return false;
    }
    return true;
  }
  // for an allocation that cannot be done without; nothing may be reading them
  void give_back() {
    ApT = ATp = nullptr;
    refused = true;
    pool.free_all();
  }
};

}  // namespace tp
