// hd_units.h -- integer arithmetic of the launches: how rows are shared, and
// the persistent launch's units and steps; for host and device (plain C++:
// nothing here needs CUDA).
#pragma once
#ifdef __CUDACC__
#define HD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HD_HOST_DEVICE inline
#endif

namespace hd {

// Lanes that share a row of the pair sweep (4 or 1), of `natom` atoms in all,
// `natom3` of them in 3-D replicas.  152 SMs have 608 schedulers; with a lane a
// row that is 608 x 32 = 19,456 rows with one warp each.
//
// Four lanes shorten the wait for a row's gathers, at the price of sums that
// meet in a tree and of work per atom that each lane repeats.  From ~8 warps an
// SM on (38,912 atoms) there is nothing left to shorten.  Below that, a step (or
// FIRE iteration) with 1 lane and with 4:
//   - rows of 2-D replicas (~15 entries) are too short to be cut beyond 9,728
//     atoms: split form, 20,208 atoms in one launch 16.7 and 20.9 us; FP64,
//     38,732 atoms with the bias 165 and 221 us, 10,104 atoms 78.1 and 77.6;
//   - 3-D, split form: 8 x 1,983 atoms 26.8 and 20.0 us a sweep;
//   - 3-D, FP64: a scheduler's warps share its FP64 pipe, so what counts is how
//     many rows the fullest one gets, in quarters: 14,272 atoms 220 and 181 us
//     (4 and 3 quarters), 15,864 atoms 224 and 243 (4 and 4), 19,830 atoms 346
//     and 270 (8 and 5), 37,677 atoms 367 and 405 (8 and 8).  The persistent
//     launch has 608 CTAs for units of 32 atoms; where many of them have a
//     second one, four lanes lose: 19,830 atoms 327 and 237 us, 23,796 atoms
//     335 and 371, 28,544 atoms 367 and 406.
HD_HOST_DEVICE int row_lanes(long long natom, long long natom3, bool fp64, bool persistent) {
    const long long one = 608 * 32;
    if (natom >= 2 * one) return 1;
    if (2 * natom3 < natom) return 2 * natom <= one ? 4 : 1;
    if (!fp64) return 4;
    if ((4 * natom + one - 1) / one >= 4 * ((natom + one - 1) / one)) return 1;
    return persistent && natom > 640 * 32 ? 1 : 4;
}

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
