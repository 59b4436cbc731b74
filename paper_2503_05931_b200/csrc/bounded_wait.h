// The one polling loop behind every wait in the device code (mbarrier phases, arrival counters of other thread
// blocks).  A wait never spins for ever: it ends when the condition holds, when another party of the same block
// has already given up (the abort word is set), or when `limit` ticks of the caller's clock have passed, in which
// case it sets the abort word itself.  The caller then stops issuing work, lets its own copies land, frees what
// it holds and returns, and the host later reads the sticky error word as AED_ERR_TIMEOUT.
//
// A wait belongs to one party, which is a whole warp on the device.  Its lanes poll together, and each decision to leave is put
// to all of them (`all`: true if p is true in every lane): a lane that sees the phase complete while another sees the abort word
// must not return with another result, because what follows a wait are operations of the whole warp (elect.sync, tensor-memory
// loads, named barriers), which are undefined and may hang when lanes are missing.
//
// The loop is plain C++ with the condition, the clock and the vote passed in, so the same source compiles for the host
// (steady clock, threads instead of warps or lanes), which is how its give-up path is tested without a GPU.
#pragma once

#if defined(__CUDACC__)
#define AED_WAIT_FN __device__ __forceinline__
#else
#define AED_WAIT_FN inline
#endif

namespace aed {

template <class Ready, class Now, class All>
AED_WAIT_FN bool bounded_poll(Ready ready, Now now, long long limit, volatile int *abort_flag, All all)
{
    if (all(ready())) return true;
    const long long start = now();
    while (true) {
        if (all(ready())) return true;
        if (!all(*abort_flag == 0)) return false;
        if (!all(now() - start <= limit)) { *abort_flag = 1; return false; }
    }
}

}  // namespace aed
