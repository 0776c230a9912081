// What the issuing thread of k_elem_tc does around the bounded wait for the
// constant operand's copy into shared memory, apart from the PTX (so that the
// host can run it too).
#pragma once

#ifdef __CUDACC__
#define SWE_HD __host__ __device__ __forceinline__
#else
#define SWE_HD inline
#endif

namespace swedg {

// One tile: mma() (the MMAs and their commit) once the copy has landed and
// nothing has failed; otherwise arrive(), which completes the phase of the
// barrier that the block then waits on, so that no MMA reads an operand that is
// not there and no thread runs its wait out.  wait() runs until it has succeeded once.
template <typename Wait, typename Mma, typename Arrive>
SWE_HD bool tc_issue(bool ok, bool& landed, Wait&& wait, Mma&& mma, Arrive&& arrive) {
  if (!landed) landed = wait();
  if (ok && landed) {
    mma();
    return true;
  }
  arrive();
  return false;
}

// Before the block gives its shared memory back: a copy that had not landed
// when the block gave up is waited for once more.
template <typename Wait>
SWE_HD void tc_drain(bool landed, Wait&& wait) {
  if (!landed) wait();
}

}  // namespace swedg
