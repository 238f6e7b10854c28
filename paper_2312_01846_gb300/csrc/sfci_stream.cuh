// The streamed output of sigma's reductions (the bucket merge and the row
// gather): entries with |u| >= a threshold leave the kernel, and the threshold
// rises while it runs so that the stream stays within its buffer.
#pragma once

#include "sfci_internal.cuh"

namespace sfci {

__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// Called by every thread of the CTA that holds A.lock: the highest histogram
// bin b whose streamed entries at or above it number >= nkeep (counts read
// while other CTAs still add, so they only undercount: the threshold is never
// too high), then tau = max(tau, lower edge of b) and the next mark halfway
// between out_n and out_cap; releases the lock.
template <int kMT, class Args>
__device__ __noinline__ void raise_threshold(const Args &A, int tid, int *s_bin,
                                             unsigned long long *part) {
    constexpr int per = kHistBins / kMT;  // bins per thread, thread 0 owns the top ones
    unsigned long long sum = 0;
    const int top = kHistBins - 1 - tid * per;
    for (int q = 0; q < per; ++q) sum += *(volatile unsigned long long *)&A.hist[top - q];
    part[tid] = sum;
    __syncthreads();
    if (tid == 0) {  // exclusive prefix from the top (kMT values)
        unsigned long long run = 0;
        for (int t = 0; t < kMT; ++t) {
            const unsigned long long v = part[t];
            part[t] = run;
            run += v;
        }
    }
    __syncthreads();
    const unsigned long long need = (unsigned long long)(A.nkeep > 0 ? A.nkeep : 1);
    unsigned long long run = part[tid];
    if (run < need && run + sum >= need) {
        // re-read: counts only grow, so a bin found with fresher counts is still
        // one with >= nkeep streamed entries at or above it
        for (int q = 0; q < per; ++q) {
            run += *(volatile unsigned long long *)&A.hist[top - q];
            if (run >= need) {
                *s_bin = top - q;
                break;
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        const int b = *s_bin;
        if (b > 0) atomicMax(A.tau_bits, (unsigned long long)b << kHistShift);
        const unsigned long long on = *(volatile unsigned long long *)A.out_n;
        const unsigned long long cap = (unsigned long long)(A.out_cap > 0 ? A.out_cap : 0);
        *(volatile unsigned long long *)A.mark = on < cap ? on + (cap - on) / 2 : cap;
        __threadfence();
        atomicExch(A.lock, 0);
    }
    __syncthreads();
}

}  // namespace sfci
