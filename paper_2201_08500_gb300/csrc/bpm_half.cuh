// One envelope's half of the coupling, for marches that hold the envelopes in
// different threads: own <- a own + b c' other, c' = c for E0 (env 0) and conj(c) for
// Eh, in the operations of couple_cell and couple3d.
#pragma once

#include "bpm_fft.cuh"
#include "bpm_internal.h"

namespace bpm {

struct HalfCoef {
  float2 ah, al;
  float bx, r1, py, r2;
};
BPM_DEV HalfCoef half_coef(const ChannelCoef& cf, int env) {
  const float2 b = env ? cf.bm : cf.bp;
  HalfCoef h;
  h.ah = cf.a_hi;
  h.al = cf.a_lo;
  h.bx = b.x;
  h.r1 = env ? b.y : -b.y;
  h.py = env ? b.y : b.x;
  h.r2 = env ? -b.x : b.y;
  return h;
}
BPM_DEV float2 half_cell(float2 p, float2 o, float2 c, const HalfCoef& h, int env) {
  const float2 bc = make_float2(fmaf(h.bx, c.x, h.r1 * c.y),
                                fmaf(h.py, env ? c.x : c.y, h.r2 * (env ? c.y : c.x)));
  return make_float2(
      fmaf(h.ah.x, p.x, fmaf(-h.ah.y, p.y, fmaf(bc.x, o.x, fmaf(-bc.y, o.y,
                                                          fmaf(h.al.x, p.x, -h.al.y * p.y))))),
      fmaf(h.ah.x, p.y, fmaf(h.ah.y, p.x, fmaf(bc.x, o.y, fmaf(bc.y, o.x,
                                                         fmaf(h.al.x, p.y, h.al.y * p.x))))));
}

}  // namespace bpm
