// Arithmetic on key positions, exact over the whole int range: a segment may end at the largest int, a query may stand
// there, and a block or a chunk that contains that position ends one past it.  (Plain C++ apart from the qualifiers.)
#pragma once

#ifdef __CUDACC__
#define KVD_HD __host__ __device__ __forceinline__
#else
#define KVD_HD inline
#endif

namespace kvd {

// First key position that a query at qp sees (window > 0: the last `window` positions up to its own).
KVD_HD int first_visible(int qp, int window) { return window > 0 && qp >= window ? qp - window + 1 : 0; }

// Whether the positions pos .. pos + n - 1 all lie inside the segment first .. first + len - 1 (which ends before the largest
// int; 0 <= n).  (64-bit sums: decode attention is as fast with them as with sums that overflow, an FP8 step over 4096 rows 35.2
// us; with differences, or unsigned sums, it took 35.5.)
KVD_HD bool segment_holds(int first, int len, int pos, int n) { return first <= pos && static_cast<long long>(pos) + n <= first + len; }
// Whether the last of them, pos + n - 1, is at most `last`.
KVD_HD bool ends_by(int pos, int n, int last) { return static_cast<long long>(pos) + n - 1 <= last; }

// Of the 64 positions from pos0 on, those in [a, b) counted from pos0, as bits.
KVD_HD unsigned long long slots64(int a, int b) {
  a = a < 0 ? 0 : a;
  b = b > 64 ? 64 : b;
  return b > a ? (b - a == 64 ? ~0ull : ((1ull << (b - a)) - 1ull) << a) : 0ull;
}
// ... those inside the segment first .. first + len - 1.
KVD_HD unsigned long long segment_slots(int first, int len, int pos0) { return slots64(first - pos0, first + len - pos0); }
// ... those that a query at qp sees which sees nothing before lo (0 <= lo).
KVD_HD unsigned long long visible_slots(int lo, int qp, int pos0) {
  return qp < pos0 ? 0ull : slots64(lo - pos0, qp - pos0 < 63 ? qp - pos0 + 1 : 64);
}

}  // namespace kvd
