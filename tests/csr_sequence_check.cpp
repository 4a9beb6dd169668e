// Drives csr_enqueue with a fake device whose launches and clears fail on
// demand.  The fake runs its calls as a stream would: a binning adds to the
// counters, a work kernel whose launch succeeded clears them, and a binning that
// finds them standing is the fault under test.
#include <cstdio>

#include "csr_sequence.h"

namespace {
enum { OK = 0, FAILED = 7 };
struct Fake {
  int counters = 0;
  bool fail_prepare = false, fail_bin = false, bin_enqueued_all_the_same = false, fail_work = false, fail_clear = false;
  bool spoiled = false;
  int prepare() { return fail_prepare ? FAILED : OK; }
  int clear() {
    if (fail_clear) return FAILED;
    counters = 0;
    return OK;
  }
  int bin() {
    if (fail_bin && !bin_enqueued_all_the_same) return FAILED;
    spoiled = spoiled || counters != 0;
    counters += 5;
    return fail_bin ? FAILED : OK;
  }
  int work() {
    if (fail_work) return FAILED;
    counters = 0;
    return OK;
  }
};
}  // namespace

int main() {
  int bad = 0, runs = 0;
  // every combination of failures in one run, then of clears in the next, then a run where all goes well
  for (int f = 0; f < 32; ++f)
    for (int again = 0; again < 2; ++again) {
      Fake d;
      bool dirty = false;
      d.fail_prepare = f & 1;
      d.fail_bin = f & 2;
      d.bin_enqueued_all_the_same = f & 4;
      d.fail_work = f & 8;
      d.fail_clear = f & 16;
      const int e = hp::csr_enqueue(d, &dirty, static_cast<int>(OK));
      bad += (e == OK) != !(d.fail_prepare || d.fail_bin || d.fail_work);
      d.fail_prepare = d.fail_bin = d.fail_work = false;
      if (!again) d.fail_clear = false;
      const int e2 = hp::csr_enqueue(d, &dirty, static_cast<int>(OK));
      d.fail_clear = false;
      const int e3 = hp::csr_enqueue(d, &dirty, static_cast<int>(OK));
      // a run that could not clear what an earlier one left reports it instead of binning
      bad += d.spoiled || d.counters != 0 || dirty || e3 != OK || (e2 != OK && !(again && (f & 16)));
      ++runs;
    }
  std::printf("%s %d\n", bad ? "bad" : "ok", runs);
  return bad != 0;
}
