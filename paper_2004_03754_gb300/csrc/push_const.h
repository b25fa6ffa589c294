// push_const.h -- constants of the push of particles in FP32 fields (pair_push.cuh),
// formed once on the host: h = q dt/2m, and 1/h^2 as two FP32 values.
#pragma once
#include "fpbits.cuh"   // PIC_HD

namespace pic {

struct PushConst {
  double h = 0.0;
  float ih2_hi = 0.0f, ih2_lo = 0.0f;
};

PIC_HD PushConst push_const(double qm, double dt) {
  PushConst k;
  k.h = 0.5 * qm * dt;
  const double ih2 = 1.0 / (k.h * k.h);
  if (ih2 > 1e-30 && ih2 < 1e30) {   // zero otherwise: every rotation takes the FP64 push
    k.ih2_hi = (float)ih2;
    k.ih2_lo = (float)(ih2 - (double)k.ih2_hi);
  }
  return k;
}

}  // namespace pic
