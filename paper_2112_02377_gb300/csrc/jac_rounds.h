// The staged rounds in which a block of the allocation-free sweep copies its
// rows' entries: positions [p0, p1) of the caller's arrays, at most CAP a round,
// one round at least (a block of empty rows still writes its rows).  Positions
// reach INT32_MAX, so no position past p1 is ever formed: a round is its first
// entry and a count, taken from what is left.  Plain C++, checked on the CPU.
#ifndef JAC_ROUNDS_H
#define JAC_ROUNDS_H

#ifdef __CUDACC__
#define JAC_HD __host__ __device__ __forceinline__
#else
#define JAC_HD inline
#endif

namespace jac {

template <int CAP, class F>
JAC_HD void for_each_round(int p0, int p1, F&& round)
{
    for (int first = p0;; first += CAP) {
        const int left = p1 - first;
        if (left <= CAP) {
            round(first, left);
            return;
        }
        round(first, CAP);
    }
}

// The part of a row [kb, ke) that a round holds: `len` entries from entry `from`
// of the round.
JAC_HD int row_part(int kb, int ke, int first, int count, int& from)
{
    const int end = first + count;                  // at most p1
    const int lo = kb > first ? kb : first, hi = ke < end ? ke : end;
    from = lo - first;
    return hi > lo ? hi - lo : 0;
}

}  // namespace jac

#endif
