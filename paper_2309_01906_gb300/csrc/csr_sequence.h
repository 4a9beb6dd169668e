// csr_sequence.h — the host order of a CSR run, apart from CUDA so that its
// failures can be tested without a GPU.
//
// The binning adds to device counters that the work kernel's last CTA clears
// again.  A binning that is enqueued without its work kernel would leave them
// standing, and the next run would place its rows past the ends of the row lists.
#pragma once

namespace hp {

// Dev: prepare() (everything that can fail before a launch), bin(), work() (launches) and clear()
// (zeroes the counters on the run's stream).  Each returns a status that is 0 on success.
// *dirty: the counters could not be cleared; the next run has to do it before its binning.
template <class Dev, class Status>
Status csr_enqueue(Dev& d, bool* dirty, Status ok) {
  Status e = d.prepare();
  if (e != ok) return e;
  if (*dirty) {
    if ((e = d.clear()) != ok) return e;
    *dirty = false;
  }
  // a launch that reports an error may be an earlier call's and have been enqueued all the same
  e = d.bin();
  if (e == ok) e = d.work();
  if (e != ok) *dirty = d.clear() != ok;
  return e;
}

}  // namespace hp
