// Host check of csrc/image_ring.cuh: the kernel's sequence of requests, waits and steps on modelled
// barriers, with one wait that expires, then the last waits. Nothing may be open afterwards, and
// without an expired wait no wait of settle_images may find anything open.
#include <cstdio>
#include <initializer_list>

#include "../../paper_1404_3773_gb300/csrc/image_ring.cuh"

using namespace cs;

// A barrier in phase `done` (phases completed), with `armed` phases requested. A wait on a parity
// other than the current phase's returns at once; on the current phase's it lets what is open land.
struct Barrier {
  int done = 0, armed = 0;
  bool wait(uint32_t parity) {
    if ((uint32_t)(done & 1) != parity) return false;
    if (done < armed) ++done;
    return true;
  }
  bool open() const { return done < armed; }
};

enum { NONE, IMAGE, MMA };

// `total` steps; the wait `what` of step `at` expires, and the CTA stops at the next step's start
bool run(int total, int what, int at) {
  Barrier img[2], mma;
  int step = 0, issued = 0;
  auto issue = [&] { ++img[image_slot(issued++)].armed; };
  issue();
  bool good = true;
  for (int i = 0; i < total && good; ++i) {
    if (i + 1 < total) issue();
    Barrier& b = img[image_slot(step)];
    if (what == IMAGE && i == at) {
      good = false;
    } else {
      // the wait of a step names the phase that its image completes
      if (b.done != (step >> 1) || !b.wait(image_parity(step))) return false;
    }
    ++mma.armed;
    if (what == MMA && i == at) {
      good = false;
    } else if (mma.done != step || !mma.wait(mma_parity(step))) {
      return false;
    }
    ++step;
  }
  int waited_open = 0;
  settle_images(
      step, issued,
      [&](int sl, uint32_t p) {
        waited_open += img[sl].open() && (uint32_t)(img[sl].done & 1) == p;
        img[sl].wait(p);
      },
      [&](uint32_t p) {
        waited_open += mma.open() && (uint32_t)(mma.done & 1) == p;
        mma.wait(p);
      });
  if (what == NONE && waited_open) return false;
  return !img[0].open() && !img[1].open() && !mma.open();
}

// The phi pass of the three-pass block: tile i's rows are copied one tile ahead, and each tile has
// two MMA groups, the next tile's first one started before this tile ends.
bool run_tiles(int total, int what, int at) {
  Barrier rows, mma;
  uint32_t ph_f = 0, ph_mma = 0;
  int nf = 0, nm = 0;
  // wait number n of a barrier: false when it is the one that expires, or a wait that names
  // another phase than its own
  auto wait = [&](Barrier& b, uint32_t& parity, int n, int kind) {
    const bool ok = !(what == kind && n == at) && b.done == n && b.wait(parity);
    parity ^= 1u;
    return ok;
  };
  ++rows.armed;
  auto start = [&](int tile) {
    if (!wait(rows, ph_f, nf++, IMAGE)) {
      ph_f = given_up(ph_f);
      return false;
    }
    if (tile + 1 < total) ++rows.armed;
    ++mma.armed;
    return true;
  };
  bool ok = start(0);
  for (int i = 0; i < total && ok; ++i) {
    for (int group = 0; group < 2 && ok; ++group) {  // synthesis, quadrature
      if (group) ++mma.armed;
      ok = wait(mma, ph_mma, nm++, MMA);
    }
    if (!ok) break;
    if (i + 1 < total) ok = start(i + 1);
  }
  if (!ok) {
    mma.wait(given_up(ph_mma));
    rows.wait(ph_f);
  }
  const int waits = what == MMA ? 2 * total : total;
  if (ok != (what == NONE || at >= waits)) return false;
  return !rows.open() && !mma.open();
}

int main() {
  int bad = 0;
  for (int total = 1; total <= 6; ++total)
    for (int what : {NONE, IMAGE, MMA})
      for (int at = 0; at < 2 * total; ++at)
        if (!run_tiles(total, what, at))
          ++bad, printf("%d tiles, wait %d of step %d expired\n", total, what, at);
  for (int total = 0; total <= 9; ++total) {
    if (total && !run(total, NONE, 0)) ++bad, printf("%d steps, no expired wait\n", total);
    for (int what : {IMAGE, MMA})
      for (int at = 0; at < total; ++at)
        if (!run(total, what, at))
          ++bad, printf("%d steps, wait %d of step %d expired\n", total, what, at);
  }
  return bad != 0;
}
