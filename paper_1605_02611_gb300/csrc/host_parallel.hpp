// Loops over the host threads.
#pragma once
#include <functional>

namespace gbdmrg {

// f(0) .. f(n - 1) on the host threads, each index once in no fixed order; work: an estimate of
// the steps in all (a thread costs about 20 us, so few of them run in the calling thread alone).
// The first exception of f is thrown on to the caller after every thread has ended; where threads or
// the memory for them cannot be had, those there are do it all.
void host_parallel(long n, long work, const std::function<void(long)>& f);

}  // namespace gbdmrg
