// Steps through [p, end) up to the largest counts that a call accepts (2^31 - 1
// nonzeros, rows, fibers): sums of a position and a step are taken unsigned, so
// that those past the end stay past it.  No argument is negative.  Also
// compiled for the host.
#pragma once

#ifdef __CUDACC__
#define SLNR_HD __host__ __device__ __forceinline__
#else
#define SLNR_HD inline
#endif

namespace slnr {

// Item i of those that begin at p.
SLNR_HD unsigned item(int p, int i) { return (unsigned)p + (unsigned)i; }

// Whether it lies before end.
SLNR_HD bool inside(int p, int i, int end) { return item(p, i) < (unsigned)end; }

// End of a step of at most n items from p, not past end (p <= end).
SLNR_HD int step_end(int p, int n, int end) { return inside(p, n, end) ? p + n : end; }

// Pieces of at most n items that `count` items make.
SLNR_HD int pieces(int count, int n) { return count > 0 ? (count - 1) / n + 1 : 0; }

}  // namespace slnr
