// Places of the block sums of a team-wide reduction.
//
// A reduction has every block of a team store its sums, pass a barrier, and
// add the sums of all blocks.  Nothing stands between those reads and the
// stores of a reduction that follows: a block without cells in the pass
// between them goes straight from one to the other while a slow block still
// reads.  So the sums lie in two halves, taken by turns: a reduction stored
// after `gen` barriers uses half gen & 1.  A later store into the same half is
// made after at least gen + 2 barriers (one more would be the other half), and
// a block passes barrier gen + 2 only when every block has arrived there, past
// its reads after barrier gen + 1.
#pragma once
#ifdef __CUDACC__
#define LBEH_PART_HD __host__ __device__ __forceinline__
#else
#define LBEH_PART_HD inline
#endif

namespace lbeh {

constexpr int kPartSums = 3;  // values per block of a reduction, at most

// doubles that a team of nb blocks needs
LBEH_PART_HD long long part_doubles(int nb) { return 2ll * kPartSums * nb; }
// place of value m of block b in a reduction stored after gen barriers
LBEH_PART_HD int part_at(unsigned long long gen, int m, int nb, int b) {
  return (int(gen & 1) * kPartSums + m) * nb + b;
}

}  // namespace lbeh
