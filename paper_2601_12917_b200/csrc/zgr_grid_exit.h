// Last step of a grid whose CTAs meet at barriers with a time limit: which status the launch reports.
#ifndef ZGR_GRID_EXIT_H_
#define ZGR_GRID_EXIT_H_

#ifdef __CUDACC__
#define ZGR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ZGR_HOST_DEVICE inline
#endif

namespace zgr {

// Called once per CTA.  Returns true for the one that leaves last, with the launch's status in `status`: -1 if any CTA gave up at
// a barrier (the last one may have passed it, late, after all others had given up), else its own.
// `words`: count_out(n) counts the CTAs that have left and is true for the n-th, which also puts the count back to zero;
// fail() marks the launch as failed; take_failed() reads the mark and clears it.
template <typename Words>
ZGR_HOST_DEVICE bool leave_grid(Words& words, unsigned n, int& status) {
  if (status < 0) words.fail();
  if (!words.count_out(n)) return false;
  if (words.take_failed()) status = -1;
  return true;
}

}  // namespace zgr
#endif  // ZGR_GRID_EXIT_H_
