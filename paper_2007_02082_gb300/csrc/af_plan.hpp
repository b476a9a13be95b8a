// Layout of the force solve by a thread-block cluster (af_cluster.cuh) and the
// rule that gives a problem to it or to the loop of launches.  Plain C++, so that
// the host decides at set-up with the numbers that the kernel uses.
#pragma once

#include <algorithm>
#include <cstdint>

#if defined(__CUDACC__)
#define AFC_HD __host__ __device__
#else
#define AFC_HD
#endif

namespace ibg {

constexpr int AFC_THREADS = 1024;
constexpr int AFC_RPT = 2;                  // rows per thread at most (x stays in registers)
constexpr int AFC_UNITS = 128;              // 32-row units of a problem that exchanges their sums
constexpr int AFC_MAX = 16;                 // CTAs per cluster at most
constexpr int AFC_SMEM = 218 * 1024;        // dynamic shared memory asked for (with the static part below 227 KB)
static_assert(AFC_UNITS == 128, "16 blocks of 256 rows at most");

// bytes of shared memory per row: p (four values), r with 1/diag, q and the row's first entry
template <typename T>
AFC_HD constexpr int afc_row_bytes() { return 11 * int(sizeof(T)) + 4; }

// Padded rows of a problem that a cluster of cl CTAs takes at most.
template <typename T>
AFC_HD constexpr int64_t afc_max_rows(int cl) { return int64_t(cl) * (sizeof(T) == 4 ? 2048 : 384); }
static_assert(2048 <= AFC_THREADS * AFC_RPT, "x of a CTA's rows is kept in registers");

// How the n rows (whole blocks of 256) of a problem lie in a cluster of cl CTAs.
// Rows per CTA: FP32 whole units of 32 rows where the problem's units fit the
// exchange, else whole blocks of 256 (so that a CTA holds whole blocks
// of the sums); FP64 units of 32.
struct AfcShape {
  bool units;   // every 32 rows' sums are exchanged
  int rper;     // rows per CTA (fewer in the last ones)
  int ubytes;   // shared memory of the units' sums
  int room;     // shared memory left for the others' p and the cached part of S
  int window;   // the others' rows a CTA may need on either side to keep a window of p: half the room at most
};
template <typename T>
AFC_HD constexpr AfcShape afc_shape(int n, int cl) {
  const bool units = sizeof(T) == 4 && n <= 32 * AFC_UNITS;
  const int gran = sizeof(T) == 8 || units ? 32 : 256;
  const int rper = (n / gran + cl - 1) / cl * gran;
  const int ubytes = units ? 12 * (n / 32) * int(sizeof(T)) : 0;
  const int room = AFC_SMEM - 64 - ubytes - rper * afc_row_bytes<T>();
  return AfcShape{units, rper, ubytes, room, room / int(16 * sizeof(T))};
}
// Entries of S a CTA keeps beside a window of `others` rows.
template <typename T>
AFC_HD constexpr int afc_cached(const AfcShape& s, int others) {
  return (s.room - others * int(4 * sizeof(T))) / int(sizeof(T) + 2) / 2 * 2;
}

// Time of an iteration in picoseconds as measured (whole numbers: the same choice on
// the host and on the device).  A cluster pays for its barriers and scalars, for rows,
// for entries in shared memory, for entries that did not fit (read again every
// iteration by 16 SMs) and, where a CTA's columns reach too far for a window
// (points that are not listed along the wall), for reading every foreign p from its
// owner and for a third barrier (a foreign p costs more the larger their part, as then all
// CTAs read from all); its slowest CTA counts.  The loop of launches uses the whole GPU and
// pays for its launches, beyond some rows also for rows.
// Measured, FP32, us an iteration, cluster against loop.  Points along the wall, 34
// entries a row: 8160 rows 9.6 / 18.8, 12,000 12.0 / 19.0, 16,000 18.5 / 19.0, 20,000 23.2 /
// 21.5, 32,000 37.2 / 25.5; 9 entries a row: 32,000 13.8 / 22.0.  Points in random order, 34
// entries: 2000 6.6 / 19.5, 4000 29 / 20, 8160 86 / 21, 32,000 255 / 32.
// FP64, 34 entries: 2000 rows 11.5 / 23.9, 6000 24.6 / 28.4; random order 2000 25.5 / 24.4, 6000 95 / 29.
// A tube's points followed by those of a sac on it (some CTAs without a window, a tenth of
// their entries foreign): 6837 rows of 16 entries 10.9 / 18.0, 15,234 of 18 16.1 / 19.5.
// Over some 250 systems the choice cost at most 17 % against the faster side.

// The CTA with rows r0 .. r0 + s.rper of n, `ne` entries, `nf` of them in columns of other
// CTAs, columns lo .. hi (from the problem's first row; lo > hi: no entries).
template <typename T>
AFC_HD constexpr int64_t afc_cta_ps(const AfcShape& s, int n, int r0, int ne, int nf, int lo, int hi) {
  constexpr bool f32 = sizeof(T) == 4;
  constexpr int64_t base = f32 ? 4600000 : 5100000, row = f32 ? 2400 : 11400, hit = f32 ? 210 : 1180,
                    miss = f32 ? 550 : 2000, own = f32 ? 210 : 1000, third = 1500000,
                    foreign = f32 ? 1600 : 2500, crowd = f32 ? 2900 : 3500;
  const int r1 = r0 + s.rper < n ? r0 + s.rper : n;
  const int below = lo <= hi && lo < r0 ? r0 - lo : 0, above = lo <= hi && hi >= r1 ? hi - r1 + 1 : 0;
  const int need = below > above ? below : above;
  int64_t t = base + row * s.rper;
  if (need > s.window) return t + third + own * (ne - nf) + foreign * nf + crowd * nf * nf / ne;   // ne > 0
  const int w0 = r0 > need ? r0 - need : 0, w1 = r1 + need < n ? r1 + need : n;
  const int room = afc_cached<T>(s, w1 - w0 - (r1 - r0)), cap = ne < room ? ne : room;
  return t + hit * cap + miss * (ne - cap);
}
// (The loop was measured at 17.5 to 21 us in FP32 below 16,000 rows; the cluster's estimate
// is some 10 % high for dense rows near the line, so the line lies at the upper end.)
template <typename T>
AFC_HD constexpr int64_t afc_loop_ps(int n) {
  return sizeof(T) == 4 ? 20500000 + (n > 16000 ? int64_t(300) * (n - 16000) : 0)
                        : 22500000 + (n > 4500 ? int64_t(2000) * (n - 4500) : 0);
}

// Whether a cluster of cl CTAs solves the problem of n rows whose slowest CTA
// takes `ps`.  By the problem's own rows and the device's cluster size alone, so that its
// bits do not depend on the batch it runs in.
template <typename T>
AFC_HD constexpr bool afc_takes(int64_t n, int cl, int64_t ps) {
  return cl > 0 && n > 0 && n <= afc_max_rows<T>(cl) && ps <= afc_loop_ps<T>(int(n));
}
// ps from rowptr ([n + 1], any base) and the problem's first entry of col, whose first
// row has number row0 there.  Where no cluster takes n rows: 0.
template <typename T>
inline int64_t afc_cluster_ps(const int32_t* rowptr, const int32_t* col, int32_t row0, int64_t n, int cl) {
  int64_t worst = 0;
  if (cl <= 0 || n > afc_max_rows<T>(cl)) return 0;
  const AfcShape s = afc_shape<T>(int(n), cl);
  for (int r0 = 0; r0 < n; r0 += s.rper) {
    const int r1 = int(std::min<int64_t>(n, r0 + s.rper));
    const int32_t *e0 = col + (rowptr[r0] - rowptr[0]), *e1 = col + (rowptr[r1] - rowptr[0]);
    int lo = int(n), hi = -1, nf = 0;
    for (const int32_t* e = e0; e < e1; ++e) {
      const int k = *e - row0;
      lo = std::min(lo, k);
      hi = std::max(hi, k);
      nf += k < r0 || k >= r1;
    }
    worst = std::max(worst, afc_cta_ps<T>(s, int(n), r0, int(e1 - e0), nf, lo, hi));
  }
  return worst;
}

}  // namespace ibg
