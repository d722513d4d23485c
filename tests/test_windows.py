"""The scattering renderer's window rule (csrc/gf_window.h, host code), on the CPU.

Rays over spans from one float spacing to 1e4, near and far, through blocks that more
kernels cover than a window can hold: windows advance, join up and reach the end of the
span, a ray that meets an over-dense block gives up after a number of windows that does
not depend on what was traced before it, and rays elsewhere take the windows of an empty
scene.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "gf_window.h"

// The windows of one ray; blocks [a, b) hold too much.  Returns the number of windows, or
// -1 when they do not join up or never end; gave_up when the ray could not go on.
struct Block { float a, b; };
static int run(bool tracking, float t0, float t1, float lim, const std::vector<Block>& blocks,
               bool& gave_up, int limit) {
  gf::Window w = gf::window_first(tracking, t0, t1, lim);
  gave_up = false;
  float reached = t0;
  for (int k = 1; k <= limit; ++k) {
    if (w.ta != reached || !(w.te > w.ta)) return -1;
    bool full = false;
    for (const Block& b : blocks) full = full || (b.a < w.te && b.b > w.ta);
    if (full) {
      if (!gf::window_halve(w)) {
        gave_up = true;
        return k;
      }
      continue;
    }
    if (w.te >= t1) return k;
    reached = w.te;
    gf::window_next(w, tracking, lim, t1);
  }
  return -1;
}

int main() {
  int bad = 0;
  const float t0s[] = {0.f, 1e-6f, 0.5f, 3.f, 31.f, 33.f, 1000.f, 1e6f};
  // average lengths that a window can hold: any, some, hardly any, none (flat scenes), NaN
  const float lims[] = {INFINITY, 0.2f, 1e-5f, 0.f, NAN};
  for (int track = 0; track < 2; ++track)
    for (float lim : lims)
      for (float t0 : t0s)
        for (int e = -24; e <= 13; ++e) {
          // spans of 2^e, down to one float spacing at t0
          float t1 = t0 + ldexpf(1.f, e);
          if (!(t1 > t0)) t1 = nextafterf(t0, INFINITY);
          bool up = false;
          // an empty scene: 1 / 0.3 windows, or one of NEE; 16 at most however dense it is
          const int n = run(track, t0, t1, lim, {}, up, 1000), most = lim == INFINITY ? 4 : 17;
          if (n < 1 || n > most || up) { printf("empty: track %d lim %g t0 %g t1 %g: %d\n", track, lim, t0, t1, n); ++bad; }
          // an over-dense block in the middle: halvings from the span down to 1e-6 of the
          // place, at most one window kept after each, and those before the block
          const float m = t0 + 0.5f * (t1 - t0);
          const int d = run(track, t0, t1, lim, {{m, t1}}, up, 1 << 20);
          if (d < 1 || d > 17 + 2 * 48 || !up) { printf("dense: track %d lim %g t0 %g t1 %g: %d\n", track, lim, t0, t1, d); ++bad; }
          // the next ray, past no block: as in the empty scene
          if (run(track, t0, t1, lim, {}, up, 1000) != n || up) { printf("state kept\n"); ++bad; }
        }
  printf(bad ? "bad\n" : "ok\n");
  return bad != 0;
}
"""


def test_windows_advance_and_end(tmp_path):
    src = tmp_path / "windows.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "windows"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2602_05081_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
