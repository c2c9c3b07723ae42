// Modelled times of the launch shapes that a call of s-steps chooses from (host arithmetic, no
// CUDA).  The cycles are those of one GB300 at its clock of 2.07 GHz; only their ratios decide.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace gempic {

// What decides the time of one slice of a march
struct SliceWork {
  int nx, ny, ppc;                 // transverse grid, particles per cell of all species
  int eb;                          // bytes per real
  int C, split;                    // CTAs per slice; 2-D: CTAs that share its particles
  int dense;                       // two CTAs per SM (FP32 128 x 128)
  int smem_bytes;                  // shared memory per CTA
};

// 2-D: cycles of one slice on S CTAs, fitted to lone marches of 64 to 1024 cells: the push (FP64
// bound by the SM's two lanes, FP32 by issue) divides, transforms and solve do not, and each
// further CTA adds to the cluster barriers and to the sum over the CTAs.  FP64, 128 cells, 4 per
// cell on 1, 2, 4, 8 CTAs: 140, 90, 72, 71 k; FP32, 512 cells: 39, 31, 27, 30 k.
inline double slice_cycles_2d(const SliceWork& w) {
  const int S = w.split;
  const double np = (double)w.nx * w.ppc / S;
  if (w.eb == 8) return 200.0 * np + 18000.0 + 140.0 * w.nx + 2500.0 * (S - 1);
  return 10.0 * np + 8500.0 + 28.0 * w.nx + (S > 1 ? 900.0 + 1200.0 * (S - 1) : 0.0);
}

// 128 x 128 FP32, k cycles of a slice with 1, 2, 4, 8, 16 per cell (one species or two; a bunch
// adds the same share to all): 40, 48, 65, 100, 169 with 512 threads and an SM to each CTA; 256
// threads with two CTAs on some SM 57, 72, 101, 165, 307, with an SM each 49, 61, 83, 129, 230
inline double slice_cycles_128(const SliceWork& w, bool shared) {
  if (!w.dense) return 30600.0 + 8600.0 * w.ppc;
  // (quadratic: the particles of the marches in flight outgrow the L2)
  return shared ? 43400.0 + (13800.0 + 167.0 * w.ppc) * w.ppc : 36500.0 + 12000.0 * w.ppc;
}

// other 3-D grids, fitted (to 15 %) to lone marches of 16 x 16 to 512 x 8 on 1 to 16 CTAs with 1 to
// 16 particles per cell: cells and particles of a CTA; in FP32 what spilled registers cost where a
// CTA's shared memory leaves the L1 little, and the exchange of rows of 256 and more.  64 x 64 FP32
// on 4, 8, 16 CTAs, 2 per cell: 64, 34, 27 k cycles, 8 per cell: 122, 83, 45 k; 128 x 64 on 8 and
// 16, 2 per cell: 63, 36 k; 32 x 32 FP64 on 2, 4, 8, 16, 4 per cell: 685, 358, 214, 143 k.
inline double slice_cycles_3d(const SliceWork& w) {
  const double c = (double)w.nx * w.ny / w.C, np = c * w.ppc;
  if (w.eb == 8) return 60000.0 + 22.5 * std::log2((double)w.nx * w.ny) * c + 249.0 * np;
  const double l1 = w.smem_bytes > 212000 ? 13600.0 : w.smem_bytes > 200000 ? 10000.0 : 0.0;
  const double rows = w.nx >= 256 ? 700.0 * w.C : 0.0;
  return 19800.0 + 11.9 * c + 10.0 * np + l1 + rows;
}

// shared: while more marches are in flight than have an SM to each CTA
inline double slice_cycles(const SliceWork& w, bool shared = true) {
  if (w.ny == 1) return slice_cycles_2d(w);
  return w.eb == 4 && w.nx == 128 && w.ny == 128 ? slice_cycles_128(w, shared) : slice_cycles_3d(w);
}

// Slice times that n marches over nz slices take, P of them in flight: march i starts `lag` slices
// after march i - 1 and not before march i - P has ended, so that march a P + b (b < P) starts at
// a max(P lag, nz) + b lag.
inline double wavefront_slices(int n, int P, int nz, double lag) {
  if (n < 1 || P < 1) return 0.0;
  const double wave = std::max(P * lag, (double)nz);
  return (double)((n - 1) / P) * wave + (double)((n - 1) % P) * lag + nz;
}

// Levels that a ring of s-levels may have for the sake of a deeper wavefront than was always taken
// (7 marches of 128 x 128, 16 elsewhere): 16 GiB, and a sixteenth of the memory that is free, so
// that one simulation of many, or on a full device, does not take room that the next one needs.
inline int ring_levels(double level_bytes, double free_bytes) {
  const double most = std::min(17179869184.0, free_bytes / 16.0);
  return (int)std::min(128.0, most / level_bytes);
}

struct ShapeTime {
  double cycles;                   // of one slice
  int maxcl;                       // marches in flight at most
  double alone;                    // of one slice with an SM to each CTA,
  int alone_cl;                    // which at most so many marches in flight have
};

// Modelled cycles of n marches over nz slices, P in flight.  Marches that share SMs hold up those
// behind them, so all go at the shared pace while more than alone_cl are in flight: not in the
// first alone_cl lags, the last ones, or a last wave of few.
inline double march_cycles(const ShapeTime& t, int n, int P, int nz, double lag) {
  const double total = wavefront_slices(n, P, nz, lag);
  if (P <= t.alone_cl) return total * t.alone;
  const bool few_last = n > P && (n - 1) % P + 1 <= t.alone_cl;
  const double alone = std::min(total, 2.0 * t.alone_cl * lag + (few_last ? nz : 0));
  return total * t.cycles - alone * (t.cycles - t.alone);
}
struct Pick {
  int shape;                       // index, -1: none can march
  int in_flight, count;            // marches in flight; s-steps of this launch
};

// The shape that n s-steps of nz slices take the least modelled time in.  depth: marches in flight
// at most, 0: no limit.  whole: the launch may take only the first `count` s-steps, whole waves of
// its shape, and leave a last wave that would be nearly empty to a launch of another shape.
inline Pick pick_shape(const std::vector<ShapeTime>& shapes, int n, int nz, double lag, int depth,
                       bool whole) {
  const auto in_flight = [&](int i, int m) {
    const int P = std::min(m, shapes[i].maxcl);
    return depth > 0 ? std::min(P, depth) : P;
  };
  const auto time = [&](int i, int m) {
    const int P = in_flight(i, m);
    return P < 1 ? -1.0 : march_cycles(shapes[i], m, P, nz, lag);
  };
  const auto shortest = [&](int m, int* which) {
    double t0 = -1.0;
    *which = -1;
    for (int i = 0; i < (int)shapes.size(); ++i) {
      const double t = time(i, m);
      if (t >= 0 && (t0 < 0 || t < t0)) {
        t0 = t;
        *which = i;
      }
    }
    return t0;
  };
  Pick r{-1, 0, n};
  double t = shortest(n, &r.shape);
  for (int i = 0; whole && i < (int)shapes.size(); ++i) {
    const int P = in_flight(i, n);
    if (P < 1 || n % P == 0) continue;
    int rest = -1;
    const double tc = time(i, n - n % P) + shortest(n % P, &rest);
    if (tc < 0.98 * t) {
      t = tc;
      r.shape = i;
      r.count = n - n % P;
    }
  }
  if (r.shape >= 0) r.in_flight = in_flight(r.shape, r.count);
  return r;
}

}  // namespace gempic
