// plans.h -- cuFFT plans shared by successive contexts (plans.cu).
#pragma once

#include <cufft.h>

#include "flame_internal.h"

namespace flame {

// A context's plan, taken from the pool or made, its own until it gives it back.
struct FftPlan {
  cufftHandle handle;
  cufftType type;
  unsigned long long ctx;  // the driver context and device it was made in
  int device;
  bool pooled, live;
};

// A 3-D plan of the lattice; f->live tells whether there is one.
cufftResult plan_take(const Grid& g, cufftType type, FftPlan* f);
// Gives a live plan back, once no work of it is in flight.
void plan_give(const Grid& g, FftPlan* f);

}  // namespace flame
