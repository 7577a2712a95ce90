// Launch-shape autotuner (host side).
//
// A kernel family offers several launch variants that compute identical results (the same
// arithmetic per entry, split differently and under different CTA shapes and register budgets). The first call for a
// problem key (lattice volume and system count) times every variant on that call's own data
// with CUDA events on the call's stream, keeps the fastest and uses it from then on; the
// choices are kept per device for the life of the process. Only idempotent launches are tuned
// (each variant overwrites the same output from unchanged inputs).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>

namespace tmamg {

bool autotune_on();
// the variant every tuned family is held to (tmamg_autotune_force), or -1
int tune_forced();
// the variant chosen for (family, key) on the current device, or -1 if not tuned yet
int tune_lookup(const char* family, int64_t key);
// times variants 0..nvar-1 (launch(v) enqueues variant v on st; one warm-up and two timed launches
// each), records the fastest for (family, key) and returns it
int tune_run(const char* family, int64_t key, int nvar, const std::function<void(int)>& launch, cudaStream_t st);

// the variant to use: the forced one, else the one tuned on first use when tuning is on; tuning (which
// runs every variant on this call's data) only when `may_tune`, i.e. when the launch is repeatable. untuned():
// the family's variant for this call where nothing was tuned
template <class Untuned>
int tune_variant(const char* family, int64_t key, int nvar, Untuned untuned, bool may_tune,
                 const std::function<void(int)>& launch, cudaStream_t st) {
  const int f = tune_forced();
  if (f >= 0) return f < nvar ? f : 0;
  if (!autotune_on() || nvar < 2) return untuned();
  const int v = tune_lookup(family, key);
  if (v >= 0) return v;
  return may_tune ? tune_run(family, key, nvar, launch, st) : untuned();
}

// the variant that a launch would use now without tuning first, or -1 if it would tune
template <class Untuned>
int tune_peek(const char* family, int64_t key, int nvar, Untuned untuned) {
  const int f = tune_forced();
  if (f >= 0) return f < nvar ? f : 0;
  return autotune_on() ? tune_lookup(family, key) : untuned();
}

// largest divisor of nt that keeps a CTA of bx x ty threads at <= maxthreads threads
inline int pick_ty(int nt, int bx, int maxthreads) {
  int best = 1;
  for (int d = 1; d * bx <= maxthreads && d <= nt; ++d)
    if (nt % d == 0) best = d;
  return best;
}

}  // namespace tmamg
