// How a CTA leaves when a bounded wait for its bulk copies runs out.
//
// A wait is made by every thread for itself, and each may find its budget exhausted at another moment;
// yet all must leave after the same row, since the row's barrier is one they meet at together. So a
// thread that gives up in row r raises a flag before the row's barrier, and all read it after. One
// flag for every row would not do where a row has only that one barrier: a fast thread that gives
// up in row r + 1 could raise it before a slow one has read it for row r, and the two would part. The
// flag of row r is raised again in row r + 2 at the earliest, after the barrier of row r + 1, which
// nobody passes before having read the flag of row r: two flags are enough.
// Host code as well: the CPU tests walk through the interleavings.
#pragma once

#if defined(__CUDACC__)
#define SGS_HD __host__ __device__ __forceinline__
#else
#define SGS_HD inline
#endif

namespace sgs {

struct GiveUp {
  volatile int* flag;    // two, in the CTA's shared memory
  SGS_HD void clear() const { flag[0] = flag[1] = 0; }                // one thread, before the first row
  SGS_HD void raise(int row) const { flag[row & 1] = 1; }             // before the row's barrier
  SGS_HD bool raised(int row) const { return flag[row & 1] != 0; }    // between it and the next one
};

// Clock cycles that a CTA which gave up waits for its copies (or its tensor-core work) still in flight
// before it reuses their shared memory or exits: the caller's budget, but at least about a
// millisecond, hundreds of times what a copy takes. Shared memory of a CTA that has exited may
// belong to another one by the time a late copy lands.
constexpr long long DRAIN_CYCLES = 1LL << 21;
SGS_HD long long drain_cycles(long long budget) { return budget > DRAIN_CYCLES ? budget : DRAIN_CYCLES; }

}  // namespace sgs
