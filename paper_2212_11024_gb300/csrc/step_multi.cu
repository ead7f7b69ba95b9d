// step_multi.cu -- several steps of a small lattice in one launch.
//
// A lattice whose sites or pairs fit the GPU's resident threads takes 2-5 us
// a step, less than the 6.2 us that launching a step costs the host.  A
// cooperative launch keeps all blocks resident; each thread steps its site
// (the one-site kernel's body) or pair (the pair kernel's), and a barrier across
// the grid separates the steps.  A step reads what other SMs wrote in the one
// before, so populations are loaded from L2, past L1.  What is left is the
// latency of one site's loads, collision and barrier.  us a step of
// flame_step(10), single launches -> one launch: FP32 16^3 6.15 -> 3.1, 32^3
// 6.16 -> 3.7, 40^3 7.2 -> 5.3; FP16 32^3 6.16 -> 4.1, 48^3 8.2 -> 6.1, 52^3 9.2 ->
// 7.5.  512 threads per SM bound the lattices that take this (77,824 sites or
// pairs): with 768, FP32 48^3 ran at 8.5 against 8.2.  Lattices of the automatic
// choice take their pairs here whatever tiling single steps have (the same bits);
// a forced tiling (flame_params.kernel 2 and 3) is kept, a launch per step.
#include "step_row.cuh"
#include "step_site.cuh"

namespace flame {
namespace {

// 512 threads per SM at 128 registers: sites in blocks of 256, pairs of 128 (us a
// step: FP32 42^3 5.6 against 6.3 in blocks of 128, FP16 32^3 4.1 against 4.9 in
// blocks of 256; fewer blocks meet at the barrier, more hide a tail).
constexpr int kSiteThreads = 256, kMultiPairThreads = 128;
// polls of the barrier's counter before a wait is given up (seconds)
constexpr unsigned kBarrierTries = 1u << 22;

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All blocks of the grid (which are resident together) arrive at sync[0];
// false if some did not within the limit.  `target`: arrivals up to and with
// this barrier.
__device__ __forceinline__ bool grid_barrier(unsigned* sync, unsigned target) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(sync, 1u);
    unsigned n = 0;
    while (load_acquire(sync) < target)
      if (++n == kBarrierTries) {
        ok = 0;
        break;
      }
  }
  return __syncthreads_and(ok) != 0;
}

// The last block to leave clears the counters for the next launch.
__device__ __forceinline__ void grid_leave(unsigned* sync) {
  if (threadIdx.x == 0 && atomicAdd(sync + 1, 1u) == gridDim.x - 1) {
    sync[0] = 0u;
    sync[1] = 0u;
    __threadfence();
  }
}

template <class Even, class Odd>
__device__ __forceinline__ void steps(int odd, int n, unsigned* flag, unsigned* sync, const Even& even_step,
                                      const Odd& odd_step) {
  for (int i = 0; i < n; ++i) {
    if ((odd ^ i) & 1) odd_step();
    else even_step();
    if (i + 1 < n && !grid_barrier(sync, (unsigned)(i + 1) * gridDim.x)) {
      if (threadIdx.x == 0) atomicOr(flag, 2u);
      break;
    }
  }
  grid_leave(sync);
}

template <class T, int VAR>
__global__ void __launch_bounds__(kSiteThreads, 2)
    step_sites_kernel(Slots<T> P, Grid g, StepConsts k, unsigned* flag, unsigned* sync, int odd, int n,
                      Reciprocals rc) {
  auto each = [&](auto&& f) {
    for (int p = blockIdx.x * kSiteThreads + threadIdx.x; p < (int)g.n3i; p += gridDim.x * kSiteThreads) {
      const int r = quotient(p, g.nx, rc.x), zz = quotient(r, g.ny, rc.y);
      f(p - r * g.nx, r - zz * g.ny, zz + g.z0);
    }
  };
  steps(
      odd, n, flag, sync,
      [&] { each([&](int x, int y, int z) { step_site<T, false, VAR, true>(P, P, g, k, flag, nullptr, x, y, z); }); },
      [&] { each([&](int x, int y, int z) { step_site<T, true, VAR, true>(P, P, g, k, flag, nullptr, x, y, z); }); });
}

template <class T, int VAR>
__global__ void __launch_bounds__(kMultiPairThreads, 4)
    step_pairs_kernel(Grid g, StepConsts k, unsigned* flag, const __grid_constant__ SlotBases<T> bases, unsigned* sync,
                      int odd, int n, Reciprocals rc) {
  const int total = (g.nx / 2) * g.ny * g.nzi, stride = gridDim.x * kMultiPairThreads;
  const int first = blockIdx.x * kMultiPairThreads + threadIdx.x;
  steps(
      odd, n, flag, sync,
      [&] {
        for (int p = first; p < total; p += stride) step_pair<T, false, VAR, true>(g, k, flag, nullptr, bases, rc, p);
      },
      [&] {
        for (int p = first; p < total; p += stride) step_pair<T, true, VAR, true>(g, k, flag, nullptr, bases, rc, p);
      });
}

// Blocks of a cooperative launch over `threads` threads' work; 0 blocks where
// they would not all be resident with one item per thread.
template <auto Kern>
cudaError_t multi_grid(long long items, int threads, int* grid) {
  int slots = 0;
  const cudaError_t e = persistent_grid<Kern>(threads, 0, 1ll << 30, &slots);
  const long long want = (items + threads - 1) / threads;
  *grid = e == cudaSuccess && want <= slots ? (int)want : 0;
  return e;
}

template <class T, int VAR>
cudaError_t sites_go(const MultiCall& c, bool* taken) {
  int grid = 0;
  cudaError_t e = multi_grid<&step_sites_kernel<T, VAR>>(c.g.n3i, kSiteThreads, &grid);
  *taken = grid > 0;
  if (e != cudaSuccess || grid == 0 || c.n == 0) return e;
  Slots<T> P = make_slots<T>(c.pop, c.g);
  Grid g = c.g;
  StepConsts k = c.k;
  unsigned *flag = c.flag, *sync = c.sync;
  int odd = c.odd, n = c.n;
  Reciprocals rc = reciprocals(c.g);
  void* args[] = {&P, &g, &k, &flag, &sync, &odd, &n, &rc};
  return cudaLaunchCooperativeKernel(step_sites_kernel<T, VAR>, dim3(grid), dim3(kSiteThreads), args, 0, c.s);
}

template <class T, int VAR>
cudaError_t pairs_go(const MultiCall& c, bool* taken) {
  int grid = 0;
  cudaError_t e = multi_grid<&step_pairs_kernel<T, VAR>>((long long)(c.g.nx / 2) * c.g.ny * c.g.nzi, kMultiPairThreads, &grid);
  *taken = grid > 0;
  if (e != cudaSuccess || grid == 0 || c.n == 0) return e;
  SlotBases<T> bases;
  for (int sl = 0; sl < kPop; ++sl) bases.p[sl] = static_cast<T*>(c.pop) + (size_t)sl * (size_t)c.g.n3;
  Grid g = c.g;
  StepConsts k = c.k;
  unsigned *flag = c.flag, *sync = c.sync;
  int odd = c.odd, n = c.n;
  Reciprocals rc = reciprocals(c.g);
  void* args[] = {&g, &k, &flag, &bases, &sync, &odd, &n, &rc};
  return cudaLaunchCooperativeKernel(step_pairs_kernel<T, VAR>, dim3(grid), dim3(kMultiPairThreads), args, 0, c.s);
}

template <class T>
cudaError_t multi_variant(const MultiCall& c, bool pairs, bool* taken) {
  if constexpr (sizeof(T) == 2) {
    if (pairs) switch (c.variant) {
        case kVarFlame: return pairs_go<T, kVarFlame>(c, taken);
        case kVarBgkFluid: return pairs_go<T, kVarBgkFluid>(c, taken);
        case kVarEmhd: return pairs_go<T, kVarEmhd>(c, taken);
      }
  }
  switch (c.variant) {
    case kVarFlame: return sites_go<T, kVarFlame>(c, taken);
    case kVarBgkFluid: return sites_go<T, kVarBgkFluid>(c, taken);
    case kVarEmhd: return sites_go<T, kVarEmhd>(c, taken);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_steps(const MultiCall& c, bool* taken) {
  *taken = false;
  if (c.variant == kVarFdCurrent) return cudaSuccess;  // its pre-pass is a step's second phase
  const bool pairs = step_row_supported(c.g, c.storage, c.variant, c.pop, c.kernel);
  // the caller asked for staged rows, which have no several-step form
  if (pairs && (c.kernel == 2 || c.kernel == 3)) return cudaSuccess;
  switch (c.storage) {
    case 1: return multi_variant<float>(c, pairs, taken);
    case 2: return multi_variant<__half>(c, pairs, taken);
    case 3: return multi_variant<__nv_bfloat16>(c, pairs, taken);
  }
  return cudaErrorInvalidValue;
}

}  // namespace flame
