// hd_units.h -- integer arithmetic of the persistent launch, for host and
// device (plain C++: nothing here needs CUDA).
#pragma once
#ifdef __CUDACC__
#define HD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HD_HOST_DEVICE inline
#endif

namespace hd {

// Barriers that a step of the persistent launch passes at most: three for a
// list rebuild, after the sweep, between the closing update and the chain,
// before the closing scale, at the end; and one before the first step.
constexpr int PERSIST_BARRIERS = 7, PERSIST_BARRIERS_0 = 1;

// Steps that one persistent launch may take where a replica has at most `nc`
// CTAs.  Its barrier counts arrivals in 32 bits, from zero at each launch:
// past 2^32 - 1 of them the target would wrap, every wait would end at once,
// and the carry would reach the half that says a list is due.  (608 CTAs, the
// most that 152 SMs hold at four each: a million steps.)
HD_HOST_DEVICE int persist_steps_max(int nc) {
    const unsigned long long passes = 0xffffffffull / (unsigned)(nc > 1 ? nc : 1);
    const unsigned long long n = (passes - PERSIST_BARRIERS_0) / PERSIST_BARRIERS;
    return n > 0x7fffffffull ? 0x7fffffff : (int)n;
}

// Atoms of unit k of a tile of n atoms from slot `start` on, cut into units of
// `width`.  A ragged tile leaves its last units short or empty; an empty one
// starts at the tile's first atom, which its threads may load.
struct UnitSpan {
    int first, n;
};
HD_HOST_DEVICE UnitSpan unit_span(int start, int n, int width, int k) {
    const int left = n - k * width;
    if (left <= 0) return {start, 0};
    return {start + k * width, left < width ? left : width};
}

}  // namespace hd
