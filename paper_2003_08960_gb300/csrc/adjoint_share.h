// How the streamed adjoint row pass shares its work out, on host and device.
#pragma once

namespace ssoct {

// (band of rows, frame) pairs i = band * nt + t, an equal, contiguous share of
// them per CTA.  Q is held as partial sums of `chunk` frames, as rows_adj_kernel
// leaves them: FP32 sums no longer than that, however many frames a CTA takes.
// A chunk that a share's end falls into is summed by the two CTAs beside it (a
// share is no shorter than a chunk): its slot is zeroed before the pass and takes
// both parts by atomic additions, whose order changes nothing for two addends.
struct RowsAdjShare {
  int bands, nt, ctas, chunk;
  __host__ __device__ long long pairs() const { return (long long)bands * nt; }
  __host__ __device__ int first(int c) const { return (int)(pairs() * c / ctas); }  // first pair of CTA c
  __host__ __device__ int band(int i) const { return i / nt; }
  __host__ __device__ int slot(int i) const { return i % nt / chunk; }  // partial sum that pair i goes to
  __host__ __device__ int begin(int i) const { return i - i % nt % chunk; }
  __host__ __device__ int end(int i) const {
    const int e = begin(i) + chunk, last = (band(i) + 1) * nt;
    return e < last ? e : last;
  }
  // whether pair i is the last of its chunk in the share [lo, hi), and whether the chunk lies in it whole
  __host__ __device__ bool closes(int i, int hi) const { return i + 1 == hi || i + 1 == end(i); }
  __host__ __device__ bool whole(int i, int lo, int hi) const { return begin(i) >= lo && end(i) <= hi; }
  // whether the first pair of CTA c lies inside a chunk (its slot is then zeroed)
  __host__ __device__ bool splits(int c) const { return first(c) != begin(first(c)); }
  // no chunk falls to more than two CTAs
  __host__ __device__ bool fits() const { return ctas > 0 && pairs() / ctas >= chunk; }
};

}  // namespace ssoct
