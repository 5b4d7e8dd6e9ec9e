// Ranking by splitting (see msd.cu): constants, arguments and host entry.
#pragma once

#include "assign.cuh"
#include "common.cuh"
#include "fft.cuh"  // FftProfile, prof_begin/prof_end, ProfKind
#include "keys.cuh"
#include "sort.cuh"

namespace amber {

constexpr int kMsdSpans = 512;                // equal spans of the key range ...
constexpr int kMsdKnots = 2048;               // ... that share the knots of the distribution map
constexpr int kMsdMaxFine = 5;                // a span has up to 2^5 counters, and at most as many knots
// log2 counters per span: the map kernel's CTAs clear and add them all, 6 us of
// a 64^3 solve's 96 with 2^5; fewer cells need fewer for the same balance
inline int msd_fine(int64_t n) { return n < 1 << 18 ? 3 : n < 1 << 25 ? 4 : kMsdMaxFine; }
constexpr int kMsdMaxDigits = 1024;           // buckets one split can write
// Tiles of a split: 4096 cells (two CTAs per SM), or 10240 (one) where there are
// so many buckets that a small tile's runs would be short: with 529 buckets
// (1024^3) 8.1 against 7.1 ms a split, with 187 (512^3) 0.75 against 0.89.
constexpr int kMsdTileA = 4096, kMsdTileB = 10240;
constexpr uint32_t kMsdManyDigits = 320;
constexpr int kMsdLocalThreads = 512;
constexpr int kMsdLocalItems = 9;
constexpr int kMsdCap = kMsdLocalThreads * kMsdLocalItems;  // most cells of a final bucket
constexpr int kMsdAvg = kMsdCap * 5 / 6;                    // cells per final bucket aimed at,
constexpr int kMsdMinAvg = 320;                             // fewer where that leaves SMs idle
constexpr int kMsdSub = 8192;                               // sub-buckets of a final bucket

// Fields of so many cells with more heavy spans than this, but too few for equal
// knots, reach down to zero through dozens of octaves.  There the transforms'
// rounding leaves thousands of cells with one and the same intensity (multiples of
// 2^-22; 1024^3 4276 cells at l = 1, 1177 at l = 1.5), which no map can spread
// over buckets: they take the digit passes at once, before anything is split.
// (Heavy spans at 512^3: 33 at l = 2, 59 at 1, 78 at 0.5; at 1024^3: 47 at 2, 68
// at 1.5, 84 at 1.  Smaller fields leave no such ties.)
constexpr int64_t kMsdTieCells = 1 << 26, kMsdTieCells2 = 1 << 28;
constexpr uint32_t kMsdTieSpans = 64, kMsdTieSpans2 = 50;

// Words between the first split's bucket counters.  With 4096-cell tiles every tile
// adds to nearly all of them, and 187 side by side (512^3) lie in six lines, whose
// adds come one after another, the dearer the more buckets a tile reaches.  A sector
// each: the passes of a 512^3 ranking 2.78, 2.88 and 2.99 ms (l = 10, 5, 3) -> 2.68,
// 2.71 and 2.80; side by side from a line's start 2.68, 2.73, 2.82, a line each 2.70,
// 2.74, 2.83.  Where there are many, larger tiles add less often and the local sort
// sums more of them: side by side (a 1024^3 solve with a sector each 49.3 ms, 49.1).
constexpr uint32_t kMsdCnt1Step = 8;
__host__ __device__ constexpr uint32_t msd_cnt1_step(uint32_t nb1) { return nb1 <= kMsdManyDigits ? kMsdCnt1Step : 1u; }

// Device control block; zero when created, left clean by every ranking.
struct MsdCtrl {
  uint32_t overflow;  // bit 0: a first-split bucket outgrew its region (or given_up), bit 1: a second-split bucket did
  uint32_t done;      // CTAs of the map kernel that finished
  uint32_t bar;       // grid barrier of the fallback
  uint32_t given_up;  // by the map: ties that no map can spread
  uint32_t pad[60];
  uint32_t hist[kMsdSpans << kMsdMaxFine];
  uint32_t map[kMsdKnots + 4];
  int32_t span[kMsdSpans];  // knot of key k in a span: (k >> (span & 31)) + (span >> 5)
  int32_t equal;            // >= 0: all knots are 2^equal keys wide
  alignas(256) uint32_t cnt1[kMsdManyDigits * kMsdCnt1Step];  // of bucket d: [d msd_cnt1_step(nb1)]
  static_assert(kMsdManyDigits * kMsdCnt1Step >= kMsdMaxDigits, "side by side they fit too");
};

struct MsdArgs {
  const float* J;
  const float* mass;   // or null
  int64_t n;
  uint2* kv1;          // first split: nb1 regions of cap1 (key, cell) pairs (final ones if nb2 is 1)
  float* mass1;
  uint2* kv2;          // second split (nb2 > 1): nb1 nb2 regions of kMsdCap
  float* mass2;
  uint32_t cap1, nb1, nb2;
  int idx_shift;         // cell index << idx_shift fills 32 bits
  int fine;              // log2 counters per span
  unsigned long long scale;  // (2^32 - 1) 2^32 / n
  int digit_bits;        // for the pass count reported
  SortCtrl* ctrl;
  MsdCtrl* mc;
  uint32_t* cnt2;      // nb1 nb2 counts
  unsigned long long* cta_mass;  // per CTA of the first split: exact 128-bit mass sum
  uint32_t* order;     // the ranking, or null
  float* mass_out;     // masses in rank order, or null
  unsigned int* status;
  // matching in the local sort (SCAN)
  unsigned char* actrl;          // assign control block, cleared by the map kernel
  unsigned long long* state;     // scan look-back words, one per final bucket (cleared there too)
  const uint32_t* fb_order[2];   // the fallback's ranking by parity of its passes
  const float* fb_mass[2];
};

struct MsdPlan {
  uint32_t nb1, nb2, cap1;
  int idx_shift, fine;
  int64_t kv1, m1, kv2, m2;  // words of the sets (kv: 2 per cell)
};
MsdPlan msd_plan(int64_t n, bool with_mass, int num_sms);
// No ranking of up to n cells makes more final buckets.
inline int64_t msd_most_buckets(int64_t n) {
  const int64_t nb = (n + kMsdAvg - 1) / kMsdAvg;
  if (nb <= kMsdMaxDigits) return kMsdMaxDigits;
  int64_t r = 1;
  while (r * r < nb) ++r;
  return r * r;
}
int msd_split_ctas(int64_t n, const MsdPlan& p, int num_sms);

// Arguments of the other ranking (digit passes in one cooperative launch),
// which runs when a bucket overflowed.
struct FallbackArgs {
  MsdCtrl* mc;
  HistArgs hist;
  PassArgs pass[4];
  int64_t tiles;
  // second-split overflow: intensities (and masses) kept in workspace were
  // overwritten by then and are put back from the first split's regions
  float* J_restore;
  float* mass_restore;
  const uint2* kv1;
  const float* mass1;
  uint32_t nb1, cap1;
  int fine;
};
cudaError_t sort_fallback(const FallbackArgs& f, bool with_mass, int num_sms, cudaStream_t s);

// Enqueue the ranking of a.J, to a.order (and a.mass_out); with sa (and masses)
// the local sort also matches and stores each redshift in its place (ta:
// thresholds, with cta_mass as partial sums).
cudaError_t msd_run(const MsdArgs& a, const FallbackArgs& f, int num_sms, const ThreshArgs* ta, const ScanArgs* sa,
                    cudaStream_t s, FftProfile* prof);

// Several rankings of one size (one or two splits over 4096-cell tiles), matched
// in place: one launch per stage, a row of CTAs per ranking.  args, scans and
// fallback are device arrays of M, those of the mass weighting (Mg[0]) first.
struct MsdMulti {
  int M, Mg[2];
  const MsdArgs* args;
  const ScanArgs* scans;
  const FallbackArgs* fallback;
  int split_ctas, buckets, fine;
  bool two_splits;
  int64_t tiles;  // sort tiles of one ranking
};
cudaError_t msd_multi(const MsdMulti& m, int num_sms, cudaStream_t s);  // up to the fallback
void msd_multi_match(const MsdMulti& m, cudaStream_t s);                // local sorts with the matching
cudaError_t sort_fallback_multi(const FallbackArgs* f, int M, int64_t tiles, int num_sms, cudaStream_t s);

// Spans are 2^L keys wide and aligned to them, and so are their counters and
// knots, so that none straddles two octaves of the intensity (a float's keys are
// half as dense per unit value in the next octave, which would bend the
// distribution inside a knot); kbase is the smallest key rounded down to a span.
struct MsdRange {
  uint32_t kbase;
  int L;  // fine <= L <= 23
};
__device__ __forceinline__ MsdRange msd_range(const SortCtrl* ctrl, int fine) {
  const uint32_t lo = (uint32_t)ctrl->kmin, hi = (uint32_t)ctrl->kmax;
  const int bits = 32 - __clz((int)(hi - lo));
  int L = fine + max(bits - 9 - fine, 0);
  if ((hi - (lo >> L << L)) >> L >= (uint32_t)kMsdSpans) ++L;
  return {lo >> L << L, L};
}

}  // namespace amber
