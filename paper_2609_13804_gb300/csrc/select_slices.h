// How an episode's candidates are dealt to the CTAs of its cluster, and what
// each CTA sends its peers in a round whose exchange is counted in bytes
// (select_gram.cu, one token a round).  Plain C++ on the host, too.
#pragma once

#if defined(__CUDACC__)
#define SP_HOSTDEV __host__ __device__ __forceinline__
#else
#define SP_HOSTDEV inline
#endif

namespace sp {

struct Slice {
  int n_loc;  // candidates of a full slice
  int j0;     // first candidate (past the last one where the slice is empty)
  int nl;     // candidates
  int words;  // words sent to every CTA in a round: slots j0 .. j0 + words of its key buffer
};

// An empty slice sends one word all the same, into a slot past the candidates
// that nobody reads (j0 >= n): a round then ends only when every CTA has sent,
// and a CTA sends only after it has read the round before, so none can be two
// rounds ahead of another and write into a buffer that is still being read.
SP_HOSTDEV Slice slice_of(int n, int C, int rank) {
  Slice s;
  s.n_loc = (n + C - 1) / C;
  s.j0 = rank * s.n_loc;
  const int end = s.j0 + s.n_loc < n ? s.j0 + s.n_loc : n;
  s.nl = end > s.j0 ? end - s.j0 : 0;
  s.words = s.nl > 0 ? s.nl : 1;
  return s;
}

// Words that a CTA receives in a round: the candidates and one per empty slice.
SP_HOSTDEV int words_of_round(int n, int C) {
  const int n_loc = (n + C - 1) / C;
  return n + C - (n + n_loc - 1) / n_loc;
}

}  // namespace sp
