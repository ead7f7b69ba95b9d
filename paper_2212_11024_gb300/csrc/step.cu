// step.cu -- the fused FLAME collide-and-stream step, one thread per site,
// AA in-place streaming over the 48-slot population state: the kernel for
// FP32 storage, and for 16-bit storage where the row kernel of step_row.cuh
// (the same algebra and variants, two sites per thread) does not apply.
// launch_step chooses between the two; the finite-difference current's B
// pre-pass (bfield_kernel) serves both.
#include "pdl.cuh"
#include "step_site.cuh"

namespace flame {
namespace {

// Step launch: 256 threads per block (a whole 256-site x row at 256^3) and
// at most 80 registers per thread (3 resident blocks per SM); the block
// shape and register budget were chosen by timing at 256^3.  Where nx is
// not a multiple of 32 a block of x rows leaves lanes idle (33 sites: 64
// threads); where that is 10 % or more of them, and more often with 16-bit
// storage (step_shape), the blocks cover consecutive sites instead (flat; a
// separate instantiation, so the row blocks keep their registers).  GLUPS on
// ~8M-site lattices, FP32 / FP16 row blocks -> flat: 33 12.2 -> 15.6 / 13.5 ->
// 22.4, 65 14.1 -> 15.4 / 16.8 -> 22.4, 100 14.8 -> 15.6 / 20.1 -> 22.6 (24.0-24.5
// since the sites are numbered without divisions); flat runs at ~15.7 FP32 at any
// length, row blocks with little waste stay ahead (250: 16.3, 255: 16.4, 256: 17.3).
constexpr int kStepThreads = 256;
constexpr int kStepMinBlocks = 3;

// The site of this thread; false where it has none.
template <class T, bool FLAT>
__device__ __forceinline__ bool site_of(const Grid& g, const Reciprocals& rc, int& x, int& y, int& z) {
  if constexpr (FLAT) {
    // consecutive sites of the updated planes (N3 < 2^31)
    const int p = blockIdx.x * kStepThreads + threadIdx.x;
    if (p >= (int)g.n3i) return false;
    // (FP32 storage waits for HBM either way: 0.5 % slower by quotient)
    const int r = sizeof(T) == 2 ? quotient(p, g.nx, rc.x) : p / g.nx;
    x = p - r * g.nx;
    const int zz = sizeof(T) == 2 ? quotient(r, g.ny, rc.y) : r / g.ny;
    y = r - zz * g.ny;
    z = zz + g.z0;
  } else {
    x = blockIdx.x * blockDim.x + threadIdx.x;
    y = blockIdx.y * blockDim.y + threadIdx.y;
    z = blockIdx.z + g.z0;
    if (x >= g.nx || y >= g.ny) return false;
  }
  return true;
}

template <class T, bool ODD, int VAR, bool FLAT = false>
__global__ void __launch_bounds__(kStepThreads, kStepMinBlocks)
    step_kernel(Slots<T> P, Grid g, StepConsts k, unsigned* __restrict__ flag, const T* __restrict__ Bfd,
                Reciprocals rc) {
  if constexpr (kChained<VAR>) {
    next_kernel_may_come();
    after_previous_kernel();
  }
  int x, y, z;
  if (!site_of<T, FLAT>(g, rc, x, y, z)) return;
  step_site<T, ODD, VAR, false>(P, P, g, k, flag, Bfd, x, y, z);
}

// The step from one state buffer to another, for a run that keeps its states:
// bound by memory like the step in place, and the state is read and written
// once where a copy and a step in place do it twice.  Copy + step -> this, us:
// FP32 33 x 40 x 40 10.3 -> 5.6, 64^3 27.6 -> 14.8, 128^3 246.8 -> 124.0 (6.5
// TB/s), FP16 65 x 64 x 64 20.5 -> 12.5.
template <class T, bool ODD, bool FLAT>
__global__ void __launch_bounds__(kStepThreads, kStepMinBlocks)
    step_between_kernel(const __grid_constant__ Slots<T> P, const __grid_constant__ Slots<T> O, Grid g, StepConsts k,
                        unsigned* __restrict__ flag, Reciprocals rc) {
  next_kernel_may_come();
  after_previous_kernel();
  int x, y, z;
  if (!site_of<T, FLAT>(g, rc, x, y, z)) return;
  step_site<T, ODD, kVarFlame, false>(P, O, g, k, flag, nullptr, x, y, z);
}

// B - B_ref of the pre-collision populations at every site, in the storage's
// element type, for the finite-difference current variant.
template <class T, bool ODD>
__global__ void bfield_kernel(Slots<T> P, Grid g, T* __restrict__ Bfd) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x >= g.nx || y >= g.ny) return;
  const int site = (z * g.ny + y) * g.nx + x;
  const Nbr nb = make_nbr(x, y, z, g);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    float v = 0.f;
#pragma unroll
    for (int i = 0; i < kM; ++i)
      v += (i == 0 ? 0.25f : 0.125f) *
           Codec<T>::dec(P.p[mslot(b, ODD ? opp7(i) : i)][site + src_off<ODD>(nb, mx7(i), my7(i), mz7(i))]);
    Bfd[(long long)b * g.n3 + site] = Codec<T>::enc(v);
  }
}

// The same for 16-bit storage and even nx, two sites (x0, x0 + 1), x0 even,
// per thread: the pair of a slot whose source is not shifted along x is one
// 32-bit load, the x-shifted sources (D3Q7 +-x on odd steps) two 16-bit
// loads, and the pair of B values one 32-bit store.  The sums run in the
// order of bfield_kernel, so both give the same B.
template <class T, bool ODD>
__global__ void bfield2_kernel(Slots<T> P, Grid g, T* __restrict__ Bfd) {
  const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z + g.z0;
  if (x0 >= g.nx || y >= g.ny) return;
  const int s0 = (z * g.ny + y) * g.nx + x0;
  const Nbr n0 = make_nbr(x0, y, z, g), n1 = make_nbr(x0 + 1, y, z, g);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    float v0 = 0.f, v1 = 0.f;
#pragma unroll
    for (int i = 0; i < kM; ++i) {
      const T* p = P.p[mslot(b, ODD ? opp7(i) : i)];
      const float w = i == 0 ? 0.25f : 0.125f;
      float a, c;
      if (!ODD || mx7(i) == 0) {
        // y and z offsets only: the same for both sites, and even
        const float2 v = dec2(p + s0 + src_off<ODD>(n0, 0, my7(i), mz7(i)));
        a = v.x;
        c = v.y;
      } else {
        a = Codec<T>::dec(p[s0 + src_off<ODD>(n0, mx7(i), 0, 0)]);
        c = Codec<T>::dec(p[s0 + 1 + src_off<ODD>(n1, mx7(i), 0, 0)]);
      }
      v0 += w * a;
      v1 += w * c;
    }
    enc2(Bfd + (long long)b * g.n3 + s0, v0, v1);
  }
}

template <class T>
cudaError_t bfield_t(int odd, const void* pop, Grid g, void* Bfd_, cudaStream_t s) {
  T* Bfd = static_cast<T*>(Bfd_);
  const Slots<T> P = make_slots<T>(pop, g);
  if constexpr (sizeof(T) == 2) {
    if (g.nx % 2 == 0) {
      const int pairs = g.nx / 2;
      const int bx = pairs >= 128 ? 128 : ((pairs + 31) / 32) * 32;
      const int by = 128 / bx < g.ny ? 128 / bx : g.ny;
      const dim3 bb(bx, by, 1), gb((pairs + bx - 1) / bx, (g.ny + by - 1) / by, g.nzi);
      if (odd)
        bfield2_kernel<T, true><<<gb, bb, 0, s>>>(P, g, Bfd);
      else
        bfield2_kernel<T, false><<<gb, bb, 0, s>>>(P, g, Bfd);
      return cudaGetLastError();
    }
  }
  const dim3 bb = site_block(g, 128), gb = site_grid(g, bb);
  if (odd)
    bfield_kernel<T, true><<<gb, bb, 0, s>>>(P, g, Bfd);
  else
    bfield_kernel<T, false><<<gb, bb, 0, s>>>(P, g, Bfd);
  return cudaGetLastError();
}

template <class T, int VAR>
cudaError_t step_launch(int odd, const Slots<T>& P, Grid g, const StepConsts& k, unsigned* flag, const T* Bfd, dim3 gr,
                 dim3 b, bool flat, cudaStream_t s) {
  auto go = [&](auto kern) {
    if constexpr (kChained<VAR>) return launch_chained(kern, gr, b, 0, s, P, g, k, flag, Bfd, reciprocals(g));
    kern<<<gr, b, 0, s>>>(P, g, k, flag, Bfd, reciprocals(g));
    return cudaGetLastError();
  };
  if (flat) return odd ? go(step_kernel<T, true, VAR, true>) : go(step_kernel<T, false, VAR, true>);
  return odd ? go(step_kernel<T, true, VAR>) : go(step_kernel<T, false, VAR>);
}

// Blocks and grid of the one-site kernels: flat blocks (true) where blocks of x
// rows leave a tenth of the lanes idle, and with 16-bit storage wherever they
// leave any, but for the BGK fluid, whose flat blocks spill (GLUPS FP16, ~4M sites,
// row blocks / flat: 63 23.6 / 24.3, 159 22.8 / 24.4, 191 23.4 / 24.4, 255 23.7 / 24.2,
// 287 20.0 / 24.3, 1023 23.9 / 24.5; electron MHD alike, the FD current but for 191,
// 1 % behind; BGK 191 23.4 / 22.4, 255 23.5 / 21.9).
template <class T>
bool step_shape(const Grid& g, int variant, dim3* b, dim3* gr) {
  const int padded = (g.nx + 31) / 32 * 32;
  const bool flat = g.nx < padded && ((sizeof(T) == 2 && variant != kVarBgkFluid) || (double)g.nx / padded < 0.9);
  *b = flat ? dim3(kStepThreads, 1, 1) : site_block(g, kStepThreads);
  *gr = flat ? dim3((unsigned)((g.n3i + kStepThreads - 1) / kStepThreads), 1, 1) : site_grid(g, *b);
  return flat;
}

template <class T>
cudaError_t between_t(int odd, const void* from, void* to, Grid g, const StepConsts& k, unsigned* flag, cudaStream_t s) {
  dim3 b, gr;
  const bool flat = step_shape<T>(g, kVarFlame, &b, &gr);
  const Slots<T> P = make_slots<T>(from, g), O = make_slots<T>(to, g);
  auto go = [&](auto kern) { return launch_chained(kern, gr, b, 0, s, P, O, g, k, flag, reciprocals(g)); };
  if (flat) return odd ? go(step_between_kernel<T, true, true>) : go(step_between_kernel<T, false, true>);
  return odd ? go(step_between_kernel<T, true, false>) : go(step_between_kernel<T, false, false>);
}

template <class T>
cudaError_t step_t(int odd, void* pop, Grid g, const StepConsts& k, unsigned* flag, int variant, void* Bfd,
                   cudaStream_t s) {
  dim3 b, gr;
  const bool flat = step_shape<T>(g, variant, &b, &gr);
  const Slots<T> P = make_slots<T>(pop, g);
  switch (variant) {
    case kVarFlame: return step_launch<T, kVarFlame>(odd, P, g, k, flag, nullptr, gr, b, flat, s);
    case kVarBgkFluid: return step_launch<T, kVarBgkFluid>(odd, P, g, k, flag, nullptr, gr, b, flat, s);
    case kVarEmhd: return step_launch<T, kVarEmhd>(odd, P, g, k, flag, nullptr, gr, b, flat, s);
    case kVarFdCurrent: {
      if (!Bfd) return cudaErrorInvalidValue;
      const cudaError_t e = bfield_t<T>(odd, pop, g, Bfd, s);
      if (e != cudaSuccess) return e;
      return step_launch<T, kVarFdCurrent>(odd, P, g, k, flag, static_cast<const T*>(Bfd), gr, b, flat, s);
    }
  }
  return cudaErrorInvalidValue;
}


}  // namespace

cudaError_t launch_bfield(int storage, int odd, const void* pop, Grid g, void* Bfd, cudaStream_t s) {
  if (!Bfd) return cudaErrorInvalidValue;
  switch (storage) {
    case 1: return bfield_t<float>(odd, pop, g, Bfd, s);
    case 2: return bfield_t<__half>(odd, pop, g, Bfd, s);
    case 3: return bfield_t<__nv_bfloat16>(odd, pop, g, Bfd, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_step(int storage, int odd, void* pop, Grid g, const StepConsts& k, unsigned* flag,
                        cudaStream_t s, int variant, void* Bfd, int kernel) {
  if (step_row_supported(g, storage, variant, pop, kernel)) {
    if (variant == kVarFdCurrent) {
      const cudaError_t e = launch_bfield(storage, odd, pop, g, Bfd, s);
      if (e != cudaSuccess) return e;
    }
    return launch_step_row(storage, odd, pop, g, k, flag, s, variant, Bfd, 0, kernel);
  }
  switch (storage) {
    case 1: return step_t<float>(odd, pop, g, k, flag, variant, Bfd, s);
    case 2: return step_t<__half>(odd, pop, g, k, flag, variant, Bfd, s);
    case 3: return step_t<__nv_bfloat16>(odd, pop, g, k, flag, variant, Bfd, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_step_between(int storage, int odd, const void* from, void* to, Grid g, const StepConsts& k,
                                unsigned* flag, cudaStream_t s, int kernel) {
  if (step_row_supported(g, storage, kVarFlame, to, kernel)) {
    const size_t bytes = (size_t)kPop * (size_t)g.n3 * (storage == 1 ? 4 : 2);
    const cudaError_t e = cudaMemcpyAsync(to, from, bytes, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    return launch_step_row(storage, odd, to, g, k, flag, s, kVarFlame, nullptr, 0, kernel);
  }
  switch (storage) {
    case 1: return between_t<float>(odd, from, to, g, k, flag, s);
    case 2: return between_t<__half>(odd, from, to, g, k, flag, s);
    case 3: return between_t<__nv_bfloat16>(odd, from, to, g, k, flag, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace flame
