// step_row.cu -- the row kernel (step_row.cuh) for the paper's scheme, and
// the host side shared by all variants: tensor maps, where the row kernel is
// used, the launch entry and the pre-capture configuration.
#include "step_row.cuh"

namespace flame {

// Tensor maps of a state (16-bit values), cached for the last state seen by
// this thread.  The encoder comes from the driver through the runtime, so the
// library links no driver library.
cudaError_t row_maps(const void* pop, const Grid& g, RowMaps* out) {
  thread_local const void* last_pop = nullptr;
  thread_local Grid last_g{};
  thread_local RowMaps last{};
  if (pop == last_pop && g.nx == last_g.nx && g.ny == last_g.ny && g.nz == last_g.nz) {
    *out = last;
    return cudaSuccess;
  }
  // looked up once (thread-safe initialisation of a function-local static)
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    const cudaError_t e =
        cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn)
                                                                : nullptr;
  }();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)kPop};
  const cuuint64_t strides[3] = {(cuuint64_t)g.nx * 2, (cuuint64_t)g.nx * g.ny * 2, (cuuint64_t)g.n3 * 2};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  RowMaps m;
  for (int w = 0; w < 2; ++w) {
    const cuuint32_t box[4] = {(cuuint32_t)g.nx, 1, 1, w == 0 ? (cuuint32_t)kPop : 3u};
    CUresult r = encode(w == 0 ? &m.all : &m.run, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<void*>(pop), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  last_pop = pop;
  last_g = g;
  last = m;
  *out = m;
  return cudaSuccess;
}

cudaError_t step_row_flame(const RowCall& c) { return row_call<kVarFlame>(c); }

// The automatic choice among the packed kernels, from sweeps with FP16 storage
// on ~4M-site lattices (nx x m x m, graph replay, GLUPS).  The unstaged pair
// kernel runs at 25.6-26.3 at every even length (24.6-25.4 while it numbered its
// pairs by 64-bit divisions, when the lines below were drawn); the staged kernel's
// whole rows run at 26-32 at most multiples of 8 (64 28.1, 128 31.3, 192 31.1, 256
// 32.1, 320 28.7, 384 29.8, 448 28.6, 512 30.2, 768 26.7, 1024 30.2) and lose to it
// where a block is under 48 threads (72-96: 17.8-23.4), where three stages of padded
// rows fit few blocks (136-152: 20.3-22.6), where a block of 260-320 threads fits
// once per SM (520-648: 18.6-23.0, half rows 21.3-25.5) and at 776-792 (23.1-23.5).
// Behind the faster pairs, but left as they were: whole rows at 160-168 (23.7-24.8),
// 264-280, 328-352, 656-728 and 800-840 (23.4-25.5), half rows at 608-640 (24.5-25.5).
// Odd row lengths take the one-site kernel.  Even lengths that are no multiple of 8
// are staged as windows where window_pays, else they take the pair kernel.
//
// Windows run a block of whole warps per row at 128 registers, 512 threads'
// worth per SM.  They are ahead of the pairs where at least 448 threads (of one
// block, 480) are resident and 95.5 % of them hold a pair (GLUPS: 246 26.4, 254
// 27.2, 306 26.1, 318 27.0, 430 26.2, 446 27.1, 486 26.4, 510 27.3, 948 26.6, 1022
// 27.8, and behind at 242 26.0, 298 25.5, 378 25.2, 382 25.5, 422 25.8, 474 25.8, 766
// 25.2, 894 25.4, 900 25.4).  Where the pitch is fixed at compile time
// (window_pitch_fixed) 86.5 % are enough (218 25.7, 222 26.1, 230 27.0, 250 27.9, 190
// 26.2; where it is not, 96-thread blocks stay behind: 190 24.4);
// with the FD current, whose B reads the pairs hide better, 94 % (windows / pairs: 222
// 18.6 / 19.6, 230 19.1 / 19.7, 250 20.0 / 19.8; 182 19.3 / 19.7 FP16, 19.2 / 19.0
// BF16).  At run-time pitches it has the line of the others: FP16 windows / pairs 246
// 19.3 / 19.6, 250 19.5 / 19.7, 306 19.4 / 19.5, 430 19.5 / 19.6, 446 20.1 / 19.8, 1022
// 20.1 / 19.7, BF16 ahead at all of them (246 19.2 / 19.0, 1022 19.9 / 19.0).
static bool window_pays(int nx, long long n3, int variant) {
  if (nx % 2 != 0 || nx % 8 == 0 || nx < 176 || nx > 1024) return false;
  const int pairs = nx / 2, threads = (pairs + 31) / 32 * 32, resident = 512 / threads * threads;
  if (resident < (threads > 256 ? 480 : 448)) return false;
  if (window_pitch_fixed(nx, n3)) return 1000 * pairs >= (variant == kVarFdCurrent ? 940 : 865) * threads;
  return threads >= 128 && 1000 * pairs >= 955 * threads;
}

int row_auto_segments(int nx, long long n3, int variant) {
  if (window_pays(nx, n3, variant)) return kWindows;
  if (nx % 8 != 0 || nx < 64 || nx > 1024) return 0;
  if ((nx > 64 && nx < 104) || (nx > 128 && nx < 160) || (nx >= 776 && nx <= 792)) return 0;
  if (nx > 512 && nx <= 648) return nx >= 608 && nx % 16 == 0 ? 2 : 0;
  return 1;
}

// Row lengths the row kernel stages: whole 16-byte units per row (up to 256
// sites by tensor-map boxes of runs placed at 128-byte aligned offsets,
// longer rows by bulk copies).
static bool row_length_ok(int nx) { return nx % 8 == 0; }

// The pair kernel: 16-bit storage, any even row length, a 4-byte aligned
// state (pairs are 32-bit accesses).
static bool pair_ok(Grid g, int storage, int variant, const void* pop) {
  return variant >= kVarFlame && variant <= kVarFdCurrent && (storage == 2 || storage == 3) && g.nx % 2 == 0 &&
         (reinterpret_cast<uintptr_t>(pop) & 3u) == 0;
}

// The staged tilings: 64 <= nx <= 1024, nx a multiple of 8, a 16-byte
// aligned state.
static bool staged_ok(Grid g, int storage, int variant, const void* pop) {
  return variant >= kVarFlame && variant <= kVarFdCurrent && (storage == 2 || storage == 3) && g.nx >= 64 &&
         g.nx <= 2 * kRowMaxThreads && row_length_ok(g.nx) && (reinterpret_cast<uintptr_t>(pop) & 15u) == 0;
}

bool step_row_supported(Grid g, int storage, int variant, const void* pop, int kernel) {
  switch (kernel) {
    case 1: return false;
    case 2: return staged_ok(g, storage, variant, pop);
    case 3: return staged_ok(g, storage, variant, pop) && g.nx > kBoxMaxX && g.nx % 16 == 0;
    case 4: return pair_ok(g, storage, variant, pop);
  }
  // automatic: the pair kernel or a staged tiling for every even row length
  if (!pair_ok(g, storage, variant, pop)) return false;
  switch (row_auto_segments(g.nx, g.n3, variant)) {
    case 0: return true;
    case kWindows: return (reinterpret_cast<uintptr_t>(pop) & 15u) == 0;
  }
  return staged_ok(g, storage, variant, pop);
}

int row_segments(const Grid& g, int kernel, int variant) {
  return kernel == 4 ? 0 : kernel == 3 ? 2 : kernel == 2 ? 1 : row_auto_segments(g.nx, g.n3, variant);
}

bool step_row_staged(Grid g, int storage, int variant, const void* pop, int kernel) {
  return step_row_supported(g, storage, variant, pop, kernel) && row_segments(g, kernel, variant) != 0;
}

namespace {
cudaError_t row_variant(int variant, const RowCall& c) {
  switch (variant) {
    case kVarFlame: return step_row_flame(c);
    case kVarBgkFluid: return step_row_bgk(c);
    case kVarEmhd: return step_row_emhd(c);
    case kVarFdCurrent: return step_row_fd(c);
  }
  return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t launch_step_row(int storage, int odd, void* pop, Grid g, const StepConsts& k, unsigned* flag,
                            cudaStream_t s, int variant, const void* Bfd, unsigned stall_tries, int kernel) {
  const RowWait wt{stall_tries ? stall_tries : kWaitTries, stall_tries ? 1 : 0};
  return row_variant(variant, RowCall{storage, odd, row_segments(g, kernel, variant), pop, g, k, flag, Bfd, s, true, wt});
}

cudaError_t prepare_step(int storage, const void* pop, Grid g, int variant, int kernel) {
  if (!step_row_supported(g, storage, variant, pop, kernel)) return cudaSuccess;
  // a placeholder field: only the configuration is settled, nothing is read
  static const unsigned no_field = 0u;
  for (int odd = 0; odd < 2; ++odd) {
    const cudaError_t e = row_variant(variant, RowCall{storage, odd, row_segments(g, kernel, variant), const_cast<void*>(pop),
                                                       g, StepConsts{}, nullptr, &no_field, nullptr, false,
                                                       RowWait{kWaitTries, 0}});
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace flame
