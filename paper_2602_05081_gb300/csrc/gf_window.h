// gf_window.h -- the windows [ta, te) in which the scattering renderer works through a
// ray (host and device code).
//
// A window holds at most a fixed number of points and chords; one that holds more is
// halved, down to kWindowMin of its place.  Windows are a function of the ray and the
// field alone: what a lane did before does not enter, so kappa's fixed-point unit (from
// the largest peak of the window) and with it every decision is the same alone and among
// other rays.
//
// Bound: a window that is kept is at least half of kWindowMin (1 + |ta|) long, and
// halving ends after log2(span / kWindowMin) steps.
#pragma once
#include <math.h>

#ifndef GF_HD
#ifdef __CUDACC__
#define GF_HD __host__ __device__ __forceinline__
#else
#define GF_HD inline
#endif
#endif

namespace gf {

constexpr float kWindowMin = 1e-6f;

// shortest window at t: beyond the spacing of floats there, so that windows advance
GF_HD float window_floor(float t) { return kWindowMin * (1.0f + fabsf(t)); }

struct Window {
  float ta, te;
  float step;  // length of the next windows
};

// the end of the span belongs to the last window
GF_HD float window_end(float te, float t1) { return te >= t1 ? t1 * (1.0f + 1e-7f) + 1e-30f : te; }

// First window of a ray that spans [t0, t1]: 0.3 of the span when tracking (delta tracking
// mostly ends there), all of it for the transmittance of a next-event ray, but not a
// length `lim` that would hold too many chords on average (a 16th of the span at least,
// whatever the average); lim comes back as later windows need it.  Without lim, and with
// it: 120 and 67 ms (12 mixed requests on two fields of a render server), 7.5 and 6.1 ms
// (step through 96x64 3-bounce paths, 200k kernels), the same where windows hold all
// their chords.  Shares of 0.25, 0.3, 0.35 and 0.5: 194.9, 193.5, 191.0 and 197.2 ms
// (1024x1024, 8 samples, 1M kernels, one-cone masks), 94.5, 92.0, 92.2 and 98.4 ms (512x512,
// 16 samples, 100k kernels, every cone).
GF_HD Window window_first(bool tracking, float t0, float t1, float& lim) {
  const float len = t1 - t0;
  lim = fmaxf(fminf(lim, len), 0.0625f * len);
  Window w;
  w.ta = t0;
  w.step = fmaxf(tracking ? fminf(0.3f * len, lim) : lim, window_floor(t0));
  w.te = window_end(w.step < len ? fminf(t1, t0 + w.step) : t1, t1);
  return w;
}

// half of a window that held too much; false when it cannot be halved
GF_HD bool window_halve(Window& w) {
  const float len = w.te - w.ta;
  if (len <= window_floor(w.ta)) return false;
  w.step = 0.5f * len;
  w.te = w.ta + w.step;
  return true;
}

// the window behind w; for a next-event ray twice as long as the last one, up to lim
GF_HD void window_next(Window& w, bool tracking, float lim, float t1) {
  if (!tracking) w.step = fminf(2.0f * w.step, fmaxf(lim, w.step));
  w.ta = w.te;
  w.te = window_end(fminf(t1, w.ta + fmaxf(w.step, window_floor(w.ta))), t1);
}

}  // namespace gf
