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
// Time of the whole call with tiles over that with the direct pass (8 to 90 rings, planes of
// 45 to 140,000 bins):
//   radius 25 - 32: 0.16 - 0.9 everywhere (direct: a load per tap)
//   radius 16: 0.7 on average above 275,000 columns, 1.3 (up to 1.8) below
//   radius 9 - 12: 0.8 above 700,000, 1.3 below; with a normalisation or its division (one
//     more load an output, fewer tiles of more than 48 rows at once) 1.05 - 1.2 at 64 and 90 rings
//   radius 3 - 8: 0.9 above 700,000 and up to 64 rings (48 with a normalisation), 1.1 - 1.4 below
//     or at 90 rings; the division 1.1 - 1.6 everywhere
//   radius 0 - 2: 1.0 at best; with a normalisation 0.9 above 700,000 and up to 48 rings
enum AxialForm { kAxialPlain, kAxialNorm, kAxialDivide };

inline bool padded_tiles_pay(int radius, AxialForm form, int n_rings, long long columns) {
  if (radius > 24) return true;
  if (radius > 12) return columns >= 275000;
  if (form == kAxialDivide && radius <= 8) return false;
  if (form == kAxialPlain && radius <= 2) return false;
  return columns >= 700000 && n_rings <= (form != kAxialPlain ? 48 : radius > 8 ? 96 : 64);
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
