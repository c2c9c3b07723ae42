// Modelled times of the launch shapes that a call of s-steps chooses from (host arithmetic, no CUDA).
#pragma once

namespace gempic {

// Slice times that n marches over nz slices take, P of them in flight: march i starts `lag` slices
// after march i - 1 and not before march i - P has ended, so that march a P + b (b < P) starts at
// a max(P lag, nz) + b lag.
inline double wavefront_slices(int n, int P, int nz, double lag) {
  if (n < 1 || P < 1) return 0.0;
  const double wave = P * lag > nz ? P * lag : (double)nz;
  return (double)((n - 1) / P) * wave + (double)((n - 1) % P) * lag + nz;
}

}  // namespace gempic
