// finalize_routes.h -- which of two kernels with the same results a smoothing
// pass takes, where the line between them is a measurement (host code, no CUDA:
// also compiled by the CPU tests).
#ifndef PSC_FINALIZE_ROUTES_H
#define PSC_FINALIZE_ROUTES_H

namespace psc {

// The axial pass of planes whose bins are not a multiple of 4: tiles on padded
// planes, or the pass that loads its rows directly.  A tile reads its rows once,
// and each output's 2 K + 1 taps from shared memory, where the direct pass moves a
// register window; but a CTA sets up barriers, a row table and its copies first,
// and a tile has one thread for two columns.  So tiles pay for wide windows and
// where there are many columns (segments x bins of a plane) to hide the set-up.
// So the line is a number of columns for each window, form of the epilogue (a
// normalisation or its division is one more load an output) and length of the segments
// (tiles of 37 rows and more are half as wide, those of 90 leave room for few).  Time of the
// whole call with tiles over that with the direct pass, 8 to 90 rings, planes of 45 to 140,000 bins:
//   radius 25 - 32: 0.16 - 0.9 everywhere (direct: a load per tap)
//   radius 13 - 24: 0.4 - 0.95 above the line, 0.9 - 1.9 below
//   radius 9 - 12: 0.7 - 0.95 and 1.0 - 2.1
//   radius 3 - 8: 0.8 - 0.98 and 1.0 - 2.2
//   radius 0 - 2: 0.95 - 1.0 and 1.0 - 1.6; with a normalisation 0.87 - 0.99 and 1.0 - 2.3
enum AxialForm { kAxialPlain = 0, kAxialNorm = 1, kAxialDivide = 2 };

inline bool padded_tiles_pay(int radius, AxialForm form, int n_rings, long long columns) {
  if (radius > 24) return true;
  constexpr long long kNever = 1LL << 62;
  if (n_rings == 1) return radius > 2;
  // columns from which tiles pay: form, window (radius 0 - 2, 3 - 8, 9 - 12, 13 - 16, 17 - 24), and up
  // to 8, 36, 48, 64 and more rings
  constexpr long long kLeast[3][5][5] = {
      {{6000000, 6000000, kNever, kNever, kNever},
       {250000, 500000, 800000, 900000, kNever},
       {150000, 300000, 500000, 450000, 450000},
       {80000, 150000, 300000, 200000, 110000},
       {50000, 90000, 155000, 155000, 50000}},
      {{700000, 700000, 1500000, kNever, kNever},
       {350000, 550000, 1000000, kNever, kNever},
       {250000, 400000, 650000, 800000, kNever},
       {150000, 220000, 275000, 275000, 220000},
       {80000, 110000, 160000, 160000, 220000}},
      {{kNever, kNever, kNever, kNever, kNever},
       {400000, 1900000, 5000000, kNever, kNever},
       {200000, 300000, 600000, 600000, kNever},
       {150000, 220000, 275000, 275000, 220000},
       {80000, 110000, 160000, 160000, 220000}}};
  const int window = radius <= 2 ? 0 : radius <= 8 ? 1 : radius <= 12 ? 2 : radius <= 16 ? 3 : 4;
  const int rows = n_rings <= 8 ? 0 : n_rings <= 36 ? 1 : n_rings <= 48 ? 2 : n_rings <= 64 ? 3 : 4;
  return columns >= kLeast[form][window][rows];
}

// The radial pass: whole lines staged in shared memory, or a column a thread.
// A column's neighbours lie T bins apart, so with few TOF bins a column's loads waste
// sectors: up to 4 bins lines always pay (448 x 45, radius 8: 1 bin 1798 -> 572 us, 3 bins
// 2088 -> 1737, 4 bins 0.97 - 0.99 of the whole call).  Above that the column pass is the better one
// once its columns (planes x views x TOF bins) keep the chip busy; below 200,000 that is so
// only where its CTAs of 256 columns, each of which walks whole lines, just fill one wave
// (4 CTAs an SM, 5 up to radius 3, on 152 SMs), for narrow windows without factors (lines load
// a sensitivity or normalisation together with the counts).  Time of the whole call with
// lines over that with columns, 40 to 448 crystals, 5 to 60 TOF bins, 1533 calls:
//   radius up to 8, no factor, one wave filled to more than 0.6: 0.86 - 1.20, 1.03 on average (100 x
//     10, 27 TOF bins: 109 against 131 us; 300 x 10, 9 bins: 316 against 353)
//   the others: 0.41 - 1.14, 0.82 on average (more than 1.03 in 34 of 1379)
inline bool radial_lines_pay(int T, long long planes, int views, int radius, bool factors) {
  const long long columns = planes * views * T;
  if (T <= 4) return true;
  if (columns > 200000) return false;
  if (factors || radius > 8) return true;
  const long long wave = 152 * (radius <= 3 ? 5 : 4), ctas = planes * ((views * T + 255) / 256);
  return ctas > wave || 5 * columns <= 3 * 256 * wave;
}

}  // namespace psc

#endif
