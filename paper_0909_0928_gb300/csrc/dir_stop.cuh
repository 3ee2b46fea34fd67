// dir_stop.cuh -- the stop test of Sec. 2.4 as a device function: l(t) =
// sum|du| / sum|u| (or the correlation coefficient); the level stops after
// iteration t when |l(t) - l(t - window)| <= eps.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "dir_launch.h"

namespace dirk {

// Whether the level has stopped by iteration q.iter; writer: this thread records
// l(t) and the stop.  Any number of threads may ask at the same time: what the
// writer stores is what they would find.
__device__ __forceinline__ bool stop_test(const StopTest& q, bool writer) {
    // loads first, so that they take one latency (l of the window is in the level's
    // rows; not used where the window reaches before them)
    const int stopped = *q.stop_iter, tw = max(q.t - q.window, q.level_first);
    const double B = q.red[3 * q.t + 2], A = q.red[3 * q.t + 1], lw = q.lhist[tw];
    if (stopped < q.iter) return true;
    const double l = q.corr ? correlation_from_sums(q.red[3 * q.t], q.corr + 4 * q.t, q.n)
                            : (B > 0.0 ? A / B : nan(""));
    if (writer) q.lhist[q.t] = l;
    if (q.iter < q.window || q.t - q.window < q.level_first) return false;
    const bool stop = !isnan(l) && !isnan(lw) && fabs(l - lw) <= q.eps;
    if (stop && writer) *q.stop_iter = q.iter;
    return stop;
}

// The same for a block of any shape (every thread calls it; one barrier)
__device__ __forceinline__ bool block_stop_test(const StopTest& q, bool first_block) {
    __shared__ int stop;
    if (threadIdx.x == 0 && threadIdx.y == 0) stop = stop_test(q, first_block);
    __syncthreads();
    return stop != 0;
}

}  // namespace dirk
