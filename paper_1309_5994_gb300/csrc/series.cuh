// Stopping rule of the FP32 inner series (App. C), shared by the host loop and the check kernel.  Plain C++, so
// that it compiles without the CUDA headers too.
#pragma once

#ifdef __CUDACC__
#define SERIES_HD __host__ __device__
#else
#define SERIES_HD
#endif

namespace dyson_detail {

// a relative update above this (or not finite) counts as divergence
constexpr double kDivergedGrowth = 1e200;

// The update first grows (the transient of the real-time series), falls factorially after its peak, then
// settles at the FP32 rounding level of the partial sums: the series stops at its target, or once it
// sits kStallDrop below its peak and has not improved for kStallSweeps sweeps
// (improvement counted from the latest peak, never during the growth).
constexpr double kStallDrop = 1e-4;
constexpr int kStallSweeps = 4;
// The same floor seen earlier: on its FP32 floor the update fluctuates, so new minima
// keep resetting the count above, while the decay itself has stopped.  The series also
// stops once the update, kStallDrop below its peak, fell by less than a factor
// kFlatRatio over the last kStallSweeps sweeps (the decay after the peak is factorial:
// a factor 3 to 10 over four sweeps until the floor).
constexpr double kFlatRatio = 0.8;
// Where the transient amplifies the rounding, the floor can lie above kStallDrop of the peak,
// and both rules above would let the series run through its whole budget on it.  It also stops
// after kPlateauSweeps sweeps without a new minimum once it has come below kPlateauDrop of the
// peak.  An oscillating update can rest and fall again (disorder, 10x10, Nc = 256: twelve sweeps without a new
// minimum at 9e-3 of the peak, then four more decades), so a refinement that stopped here and gained less than
// kPlateauGain is the last one that may (plateau_served).
constexpr int kPlateauSweeps = 16;
constexpr double kPlateauDrop = 1e-2;
constexpr double kPlateauGain = 0.1;                     // (twelve refinements of a digit each reach any tolerance)

enum {
  SERIES_RUNNING = 0,
  SERIES_STOPPED,                      // target, or floor below kStallDrop of the peak
  SERIES_PLATEAU,                      // floor below kPlateauDrop of the peak
  SERIES_EXHAUSTED,
  SERIES_ABORTED,                      // the peak passed abort_peak
  SERIES_NOT_FINITE
};

struct SeriesState {
  double best, peak, last;
  double hist[kStallSweeps];           // the last kStallSweeps updates (ring)
  int since_best, since_peak, sweeps;
  int plateau;                         // 1: the plateau rule applies
  int run;                             // 1 while the series goes on (read by the fused sweep)
  int outcome;
};

SERIES_HD inline SeriesState series_start(bool plateau) {
  SeriesState S = {};
  S.best = 1e300;
  S.plateau = plateau;
  S.run = 1;
  return S;
}

// one more sweep, with the relative update upd (infinite where a norm was not a number)
SERIES_HD inline void series_step(SeriesState& S, double upd, int max_sweeps, double target, double abort_peak) {
  const int sweep = ++S.sweeps;
  S.last = upd;
  if (!(upd < kDivergedGrowth)) {
    S.outcome = SERIES_NOT_FINITE;
    S.run = 0;
    return;
  }
  if (upd > S.peak) {                                    // the stall is judged on the decay after the latest peak
    S.peak = upd;
    S.best = upd;
    S.since_best = 0;
    S.since_peak = 0;
  } else {
    ++S.since_peak;
    if (upd < S.best) {
      S.best = upd;
      S.since_best = 0;
    } else {
      ++S.since_best;
    }
  }
  const double ago = S.hist[sweep % kStallSweeps];       // the update kStallSweeps sweeps ago
  S.hist[sweep % kStallSweeps] = upd;
  if (S.peak > abort_peak)
    S.outcome = SERIES_ABORTED;
  else if ((upd <= target && (upd < S.peak || upd == 0.0)) ||   // on the decay, not before the peak
           (S.since_best >= kStallSweeps && S.best < kStallDrop * S.peak) ||
           (S.since_peak >= kStallSweeps && upd < kStallDrop * S.peak && upd > kFlatRatio * ago))
    S.outcome = SERIES_STOPPED;
  else if (S.plateau && S.since_best >= kPlateauSweeps && S.best < kPlateauDrop * S.peak)
    S.outcome = SERIES_PLATEAU;
  else if (sweep >= max_sweeps)
    S.outcome = SERIES_EXHAUSTED;
  if (S.outcome != SERIES_RUNNING) S.run = 0;
}

// whether a refinement that ended on a plateau gained enough for the next one to end there too; res and prev_res:
// relative residuals after it and before it (infinite before the first, whose solution is zero)
inline bool plateau_served(double res, double prev_res) { return res <= kPlateauGain * (prev_res < 1.0 ? prev_res : 1.0); }

// Observables amplify the residual.  The double occupancy D = (Re (G(t) - G(t - dt)) / dt - eps n - E_kin) / U has
// up to 2 / (dt |U|) of it from the difference quotient and (|eps| + 4 |J|) / |U| from the rest (errors of G of the
// residual's size).  An inner solve after the first aims at a tenth of the tolerance (kInnerSlack), but the first
// refinement aims at no tolerance and may end just below a loose one; so at tolerances of kLooseTol and above (no
// first refinement reaches lower ones) one more refinement follows unless the residual is below accept_share
// of the tolerance.
constexpr double kLooseTol = 1e-8;
inline double accept_share(double dt, double u_min, double eps_max, double j_max) {
  const double amplification = u_min > 0.0 ? (2.0 / dt + eps_max + 4.0 * j_max) / u_min : 1e300;
  return amplification > 1.0 ? 1.0 / amplification : 1.0;
}
inline bool refine_once_more(double res, double tol, double prev_res, double share, bool last) {
  return res <= tol && tol >= kLooseTol && res > share * tol && prev_res > tol && !last;
}

}  // namespace dyson_detail
