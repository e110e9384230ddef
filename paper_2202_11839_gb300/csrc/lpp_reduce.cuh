// Warp-segmented shell reduction and compensated accumulators (internal).
#pragma once

#include "lpp_internal.h"

namespace lpp {

template <typename T> struct Owned;
template <> struct Owned<float> {
    // compensated sum (Knuth two-sum) in two floats
    static __device__ __forceinline__ void add(float* hi, float* lo, float v) {
        const float s = *hi + v;
        const float bp = s - *hi;
        const float err = (*hi - (s - bp)) + (v - bp);
        *hi = s;
        *lo += err;
    }
    static __device__ __forceinline__ double value(const float* hi, const float* lo) {
        return (double)*hi + (double)*lo;
    }
    static constexpr int words = 2;
};
template <> struct Owned<double> {
    static __device__ __forceinline__ void add(double* hi, double*, double v) { *hi += v; }
    static __device__ __forceinline__ double value(const double* hi, const double*) { return *hi; }
    static constexpr int words = 1;
};

// Segmented inclusive scans over lanes with equal shells, the shells monotone along the warp
// (equal shells form one contiguous run).  The steps that add (bit s: lane >= 2^s and the lane
// 2^s below is in the same shell) and whether the lane ends its segment are the same for every
// value of an item and computed once.
struct SegMask {
    unsigned add;   // bit s set: add the value shuffled up by 2^s
    bool last;      // the lane holds its segment's sum after the scan
};

// key: the lane's segment (equal keys contiguous along the warp), e.g. its shell label
__device__ __forceinline__ SegMask seg_mask(int key) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    SegMask m;
    m.add = 0u;
#pragma unroll
    for (int s = 0, d = 1; d < 32; d <<= 1, ++s) {
        const int ok = __shfl_up_sync(full, key, d);
        if (lane >= d && ok == key) m.add |= 1u << s;
    }
    const int nk = __shfl_down_sync(full, key, 1);
    m.last = (lane == 31) || (nk != key);
    return m;
}

// The segmented sums added to the warp's own accumulators own[words][E] (complex, interleaved)
// in shared memory.  Equal shells form one segment (bins monotone along the warp), so no two
// lanes add to the same accumulator.
template <typename T>
__device__ __forceinline__ void warp_own_add(T re, T im, int bin, const SegMask& m, T* own, int E) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int s = 0, d = 1; d < 32; d <<= 1, ++s) {
        const T ore = __shfl_up_sync(full, re, d);
        const T oim = __shfl_up_sync(full, im, d);
        if ((m.add >> s) & 1u) {
            re += ore;
            im += oim;
        }
    }
    if (m.last && bin >= 0) {
        Owned<T>::add(own + 2 * bin, own + E + 2 * bin, re);
        Owned<T>::add(own + 2 * bin + 1, own + E + 2 * bin + 1, im);
    }
    __syncwarp();   // another lane may add to the same shell next
}

}  // namespace lpp
