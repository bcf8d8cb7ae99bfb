// Host-plan sizes for the tests: built with host_plan.cpp into a small library, no GPU needed.
#include <string>

#include "host_plan.h"

// out: gather bands, gather shared memory (bytes), the largest band's pupil-edge terms.
extern "C" int host_plan_gather(const tomo_geometry *g, int cluster_size, int transforms, long long *out) {
  tomo::HostPlan P;
  std::string err;
  const int st = tomo::build_host_plan(g, &P, &err, cluster_size, transforms);
  if (st != TOMO_OK) return st;
  out[0] = P.gather_bands;
  out[1] = P.smem_gather;
  out[2] = 0;
  for (const auto &s : P.tt_seg) {
    const long long n = P.tt_beg[s.y] - P.tt_beg[s.x];
    if (n > out[2]) out[2] = n;
  }
  return TOMO_OK;
}

// out[0..n_layers): side of the block that one CTA of a layer's cluster finishes.
extern "C" int host_plan_coarse(const tomo_geometry *g, int cluster_size, int transforms, long long *out) {
  tomo::HostPlan P;
  std::string err;
  const int st = tomo::build_host_plan(g, &P, &err, cluster_size, transforms);
  if (st != TOMO_OK) return st;
  for (size_t l = 0; l < P.layers.size(); ++l) out[l] = P.layers[l].coarse;
  return TOMO_OK;
}

// out[0]: CTAs of one forward launch (tiles of the sensors, chunks of the tip/tilt-only ones).
extern "C" int host_plan_forward(const tomo_geometry *g, int cluster_size, int transforms, long long *out) {
  tomo::HostPlan P;
  std::string err;
  const int st = tomo::build_host_plan(g, &P, &err, cluster_size, transforms);
  if (st == TOMO_OK) out[0] = static_cast<long long>(P.fwd_items.size());
  return st;
}

// CTAs up to which a forward launch takes the small form.
extern "C" int host_plan_forward_small() { return tomo::kFwdSmallLaunch; }
