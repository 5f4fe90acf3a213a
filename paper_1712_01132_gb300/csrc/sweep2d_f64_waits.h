// sweep2d_f64_waits.h -- what the warps of a CTA of the 2D FP64 sweep (sweep2d_f64.cu) wait for before they read or
// overwrite what another warp wrote or reads.  Plain functions, so that the CPU model of the waits in tests/ runs
// through the orders that they allow with the kernel's own figures.
//
// Progress words: col[w], steps that sweeping warp w has finished (a step is a column of its lower row; with rpw = 2
// the upper row is a column behind); rec[p], blocks of columns whose records unit p has; mom[w], blocks of warp w
// whose moments are done with.  Rings of h and of records hold two blocks of B columns, group sums and their count
// are kept for two blocks (parity).  Each function gives the value that has to be reached.
#pragma once

#ifdef __CUDACC__
#define DVM_WAIT __host__ __device__ constexpr
#else
#define DVM_WAIT constexpr
#endif

namespace dvm {
namespace f64waits {

constexpr int kBlk = 16;   // columns of a block

// Bound of these waits, ns, from that of a wait on the band below: a block of columns is up to 16 of those waits away.
// (A bound near the type's largest value stays there.)
DVM_WAIT long long inner_bound(long long timeout_ns) {
    return timeout_ns > (0x7fffffffffffffffLL >> 6) ? 0x7fffffffffffffffLL : 64 * timeout_ns;
}

// Sweeping warp at the start of block k >= 2, which overwrites block k - 2 of its ring of h:
DVM_WAIT int records_of_block(int k) { return k + 1; }                          // rec of its unit (k >= 0)
DVM_WAIT int own_moments(int k) { return k - 1; }                               // mom of itself
template <int B = kBlk> DVM_WAIT int rows_above(int k) { return (k - 1) * B; }  // col of the warps that read its h
// Sweeping warp before the step of column c: col of the warp below (its top row has swept the column)
DVM_WAIT int row_below(int c, int rpw) { return c + rpw; }
// Record warp before it overwrites block k - 2 with block k >= 2: col of the unit's warps
template <int B = kBlk> DVM_WAIT int record_readers(int k, int rpw) { return (k - 1) * B + rpw; }
// Moment warp before it sums block k of a sweeping warp: col of that warp
template <int B = kBlk> DVM_WAIT int swept(int k, int n1, int rpw) { return ((k + 1) * B < n1 ? (k + 1) * B : n1) + rpw - 1; }
// Moment warp before it writes a group's sum of block k >= 2 over that of block k - 2 and counts it: mom of every
// group of the unit.  Blocks k - 2 of all groups are then summed, counted and, by the warp that came last, added: it
// moves its own mom on only afterwards.  The waits above do not give this: at the end of a row no block follows whose
// records would hold the groups together, so that a group may be done with block k while another's block k - 2 is
// still to be summed.
DVM_WAIT int group_moments(int k) { return k - 1; }

}  // namespace f64waits
}  // namespace dvm
