// Which pieces of a split head a merge may read (host and device code, no CUDA needed).
#pragma once
#ifdef __CUDACC__
#define TRJ_HOST_DEVICE __host__ __device__
#else
#define TRJ_HOST_DEVICE
#endif

namespace trj {

// (first, last): the streams that the main kernel recorded as the first and the last to work on a head; `streams` of them were
// launched.  True if there are pieces of several streams to merge.  A stream whose wait ran out leaves without a record, so what
// stands there may be anything: only a range of streams that exist keeps the merge inside the workspace and its loop short.
TRJ_HOST_DEVICE inline bool pieces_to_merge(int first, int last, int streams) { return first >= 0 && first < last && last < streams; }

}  // namespace trj
