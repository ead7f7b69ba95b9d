// plans.cu -- cuFFT plans that outlive a context.
//
// Making a 64^3 FP64 plan takes the host 350-500 us and destroying one 60, so
// a run that makes a context for one gradient (two plans) spent 0.9 ms of its
// 5.6 on them.  A context takes its plans from a pool and gives them back when
// it is destroyed; between the two they are its own, and the stream is set
// before each use.  The pool is bounded: it keeps at most kMostPlans idle plans
// without a work area of more than kMostWork bytes.  A plan belongs to one driver
// context of one device (a device that was reset gets a new one): it is given out
// in that context only, and destroyed only by a call in that context, beyond the
// bound the oldest of the context's own, or the plan that comes where all those
// kept are others' (IdleList).  Plans of a context that is gone went with it; what
// is left of them in the list is a few words each.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cufft.h>

#include <mutex>

#include "idle_list.h"
#include "plans.h"

namespace flame {
namespace {

constexpr int kMostPlans = 8;
constexpr size_t kMostWork = 8u << 20;

struct Key {
  unsigned long long ctx;
  int device, type, nx, ny, nz;
  bool operator==(const Key& k) const {
    return ctx == k.ctx && device == k.device && type == k.type && nx == k.nx && ny == k.ny && nz == k.nz;
  }
};

// The current driver context's id, unique for the life of the process; false
// where it cannot be had (then plans are not pooled).
bool context_id(unsigned long long* id) {
  using Fn = CUresult(CUDAAPI*)(CUcontext, unsigned long long*);
  static const Fn get = [] {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &q);
    return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<Fn>(fn) : nullptr;
  }();
  return get && get(nullptr, id) == CUDA_SUCCESS;
}

struct Pool {
  std::mutex mu;
  IdleList<Key, cufftHandle, kMostPlans> idle;
};
// never destroyed: contexts may be released during the process's exit, after
// static objects are gone
Pool& pool() {
  static Pool* p = new Pool;
  return *p;
}

Key key_of(const FftPlan& f, const Grid& g) { return Key{f.ctx, f.device, (int)f.type, g.nx, g.ny, g.nz}; }

}  // namespace

cufftResult plan_take(const Grid& g, cufftType type, FftPlan* f) {
  f->type = type;
  f->pooled = cudaGetDevice(&f->device) == cudaSuccess && context_id(&f->ctx);
  cufftResult r = CUFFT_SUCCESS;
  if (f->pooled) {
    Pool& p = pool();
    std::lock_guard<std::mutex> lock(p.mu);
    if (p.idle.take(key_of(*f, g), &f->handle)) {
      f->live = true;
      return r;
    }
  }
  r = cufftPlan3d(&f->handle, g.nz, g.ny, g.nx, type);
  f->live = r == CUFFT_SUCCESS;
  return r;
}

void plan_give(const Grid& g, FftPlan* f) {
  if (!f->live) return;
  f->live = false;
  size_t work = 0;
  if (!f->pooled || cufftGetSize(f->handle, &work) != CUFFT_SUCCESS || work > kMostWork) {
    cufftDestroy(f->handle);
    return;
  }
  Pool& p = pool();
  cufftHandle old = 0;
  bool drop = false;
  {
    std::lock_guard<std::mutex> lock(p.mu);
    drop = p.idle.give(key_of(*f, g), f->handle, &old);
  }
  if (drop) cufftDestroy(old);
}

}  // namespace flame
