// aa.cuh -- addressing of the in-place AA streaming pattern over the
// 48-slot structure-of-arrays population state, shared by the step, the
// diagnostics and the adjoint kernels.
#pragma once

#include "flame_internal.h"
#include "lattice.cuh"

namespace flame {

// p / d for 0 <= p < 2^31, with r = floor(2^32 / d) (2^32 - 1 for d = 1): p r / 2^32
// is at most p / d and less than one below it, so that its floor is the quotient
// or one less.  A division by a run-time int takes some 20 instructions and a
// reciprocal's latency, one of 64-bit ints four times that; where threads or tiles
// are numbered through the lattice they stand before everything else.
// FP16, us per step: one-site kernel in flat blocks 129 x 127 x 131 98.96 -> 90.1,
// 65 x 248 x 248 181.2 -> 165.5; pairs (64-bit before) 100 x 200 x 200 160.8 ->
// 154.1, 256 x 128 x 128 167.2 -> 159.2; several steps in one launch 32^3 3.92 ->
// 3.70.
__device__ __forceinline__ int quotient(int p, int d, unsigned r) {
  const int q = (int)__umulhi((unsigned)p, r);
  return p - q * d >= d ? q + 1 : q;
}

// A load past L1 of what another SM may have written since this thread last read
// the place, in a kernel whose blocks wait for one another.  volatile and "memory":
// the compiler neither takes an earlier load's value for this one nor moves it
// across the wait (the built-in load of a 16-bit value promises neither).
template <class T>
__device__ __forceinline__ T load_l2(const T* p) {
  if constexpr (sizeof(T) == 2) {
    unsigned short v;
    asm volatile("ld.global.cg.b16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return *reinterpret_cast<const T*>(&v);
  } else if constexpr (sizeof(T) == 4) {
    unsigned v;
    asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return *reinterpret_cast<const T*>(&v);
  } else {
    static_assert(sizeof(T) == 8, "16, 32 or 64 bits");
    unsigned long long v;
    asm volatile("ld.global.cg.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return *reinterpret_cast<const T*>(&v);
  }
}

// Site-index offsets of the periodic neighbours.
struct Nbr {
  int xm, xp, ym, yp, zm, zp;
  __device__ __forceinline__ int operator()(int cx, int cy, int cz) const {
    return (cx < 0 ? xm : (cx > 0 ? xp : 0)) + (cy < 0 ? ym : (cy > 0 ? yp : 0)) +
           (cz < 0 ? zm : (cz > 0 ? zp : 0));
  }
};

__device__ __forceinline__ Nbr make_nbr(int x, int y, int z, const Grid& g) {
  Nbr n;
  const int plane = g.nx * g.ny;
  n.xm = x == 0 ? g.nx - 1 : -1;
  n.xp = x == g.nx - 1 ? -(g.nx - 1) : 1;
  n.ym = y == 0 ? (g.ny - 1) * g.nx : -g.nx;
  n.yp = y == g.ny - 1 ? -(g.ny - 1) * g.nx : g.nx;
  n.zm = z == 0 ? (g.nz - 1) * plane : -plane;
  n.zp = z == g.nz - 1 ? -(g.nz - 1) * plane : plane;
  return n;
}

// AA pattern.  Pre-collision population on velocity c of a site:
//   even parity: same site, own slot;  odd: site - c, opposite slot.
// Post-collision population on velocity c:
//   even: same site, opposite slot;    odd: site + c, own slot.
template <bool ODD>
__device__ __forceinline__ long long src27(int i, int site, const Nbr& nb, long long n3) {
  return ODD ? (long long)phys(opp27(i)) * n3 + site + nb(-cx27(i), -cy27(i), -cz27(i))
             : (long long)phys(i) * n3 + site;
}
template <bool ODD>
__device__ __forceinline__ long long dst27(int i, int site, const Nbr& nb, long long n3) {
  return ODD ? (long long)phys(i) * n3 + site + nb(cx27(i), cy27(i), cz27(i))
             : (long long)phys(opp27(i)) * n3 + site;
}
template <bool ODD>
__device__ __forceinline__ long long src7(int b, int i, int site, const Nbr& nb, long long n3) {
  return ODD ? (long long)phys(mslot(b, opp7(i))) * n3 + site + nb(-mx7(i), -my7(i), -mz7(i))
             : (long long)phys(mslot(b, i)) * n3 + site;
}
template <bool ODD>
__device__ __forceinline__ long long dst7(int b, int i, int site, const Nbr& nb, long long n3) {
  return ODD ? (long long)phys(mslot(b, i)) * n3 + site + nb(mx7(i), my7(i), mz7(i))
             : (long long)phys(mslot(b, opp7(i))) * n3 + site;
}

// Base pointers of the 48 populations in natural slot order (natural slot
// q starts at phys(q) * N3), passed as kernel parameters so that each access
// is one index computation on a parameter.
template <class T>
struct Slots {
  T* p[kPop];
};
template <class T>
inline Slots<T> make_slots(const void* pop, const Grid& g) {
  Slots<T> P;
  for (int q = 0; q < kPop; ++q)
    P.p[q] = const_cast<T*>(static_cast<const T*>(pop)) + (size_t)phys(q) * (size_t)g.n3;
  return P;
}

// Site offset of the source (pre-collision) and destination
// (post-collision) of the population on velocity (cx, cy, cz), and the
// slot used there, for the two AA parities.
template <bool ODD>
__device__ __forceinline__ int src_off(const Nbr& nb, int cx, int cy, int cz) {
  return ODD ? nb(-cx, -cy, -cz) : 0;
}
template <bool ODD>
__device__ __forceinline__ int dst_off(const Nbr& nb, int cx, int cy, int cz) {
  return ODD ? nb(cx, cy, cz) : 0;
}

// Block of `threads` threads: x-rows of up to `threads` sites, several
// rows per block when nx is small.
inline dim3 site_block(const Grid& g, int threads = 128) {
  int bx = g.nx >= threads ? threads : ((g.nx + 31) / 32) * 32;
  int by = threads / bx;
  if (by > g.ny) by = g.ny;
  if (by < 1) by = 1;
  return dim3(bx, by, 1);
}

// One grid z-layer per updated plane (z = blockIdx.z + g.z0).
inline dim3 site_grid(const Grid& g, dim3 b) { return dim3((g.nx + b.x - 1) / b.x, (g.ny + b.y - 1) / b.y, g.nzi); }

}  // namespace flame
