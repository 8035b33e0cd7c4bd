// postproc.cu -- post-processing of int64 fixed-point sinograms: mashing of
// views and TOF bins (Sec. 4 names it as a way to need fewer counts and less
// smoothing time) and the sum over the scanner's rotational symmetries
// (Sec. 2.2.4 averages the sensitivity sinograms over them).  Both are exact
// integer sums, so their results do not depend on summation order.
//
// Layout of a sinogram: [plane = ring_a * n_rings + ring_b][view][rad][tof],
// with the integer LOR formula of the binning: for crystals a < b, f = a + b
// (f -= n and s = -1 when f >= n, else s = +1), view = f >> 1, radial
// s (n/2 - (b - a)) + n/2 - 1 less the centred clip offset.
#include <algorithm>

#include "psc_internal.h"

namespace psc {

namespace {

// out[p][v / vf][r][t / tf] = sum of the vf x tf block; grid (ceil(R T2 /
// 256), V2, planes).  Mashing of TOF bins, or of many views; else the kernel below.
// Bound by memory.  Whole TOF axes: eight views' loads go out together.  Blocks of TOF
// bins: a bin's neighbours lie in the sectors that its first load brought into L1, so
// a thread walks a view's bins, four loads a turn, and the views one by one (more in
// flight asked L2 for the same sectors again: 3 bins to 1 605 -> 1070 us).  As two plain loops that
// the compiler unrolled as it chose, 288 x 16 scanner, 27 TOF bins: 3 to 1 707 -> 605 us,
// with pairs of views 537 -> 441; TOF kept and 16 views to one 836 -> 416.
template <bool kWholeTof>
__global__ void __launch_bounds__(256) mash_kernel(const long long* __restrict__ in, long long* __restrict__ out, int V,
                                                   int R, int T, int vf, int tf) {
  const int V2 = V / vf, T2 = T / tf;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;  // r * T2 + t2
  if (c >= R * T2) return;
  const int r = c / T2, t2 = c - r * T2;
  const int v2 = blockIdx.y;
  const long long p = blockIdx.z;
  const long long* row = in + ((p * V + (long long)v2 * vf) * R + r) * T + (long long)t2 * tf;
  const long long vstride = (long long)R * T;
  long long sum = 0;
  if (kWholeTof) {
#pragma unroll 8
    for (int j = 0; j < vf; ++j) sum += __ldg(row + j * vstride);
  } else {
#pragma unroll 1
    for (int j = 0; j < vf; ++j, row += vstride) {
#pragma unroll 4
      for (int u = 0; u < tf; ++u) sum += __ldg(row + u);
    }
  }
  out[((p * V2 + v2) * R + r) * T2 + t2] = sum;
}

// The same for VF views and whole TOF axes: bound by memory, so a thread
// keeps the loads of kRows output rows (8 or so) in flight at once; with one
// output's it waited on each (5 TOF bins, 45 rings, views by 2: 3411 -> 1660 us,
// 7.3 TB/s).
// grid (ceil(R T / 256), ceil(V2 / kRows), planes)
template <int VF>
__global__ void __launch_bounds__(256) mash_views_kernel(const long long* __restrict__ in, long long* __restrict__ out,
                                                         int V, int row) {
  constexpr int kRows = VF == 1 ? 8 : VF == 2 ? 4 : VF <= 4 ? 2 : 1;
  const int V2 = V / VF;
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= row) return;
  const int v0 = blockIdx.y * kRows;
  const long long* src = in + ((long long)blockIdx.z * V + (long long)v0 * VF) * row + c;
  long long* dst = out + ((long long)blockIdx.z * V2 + v0) * row + c;
  long long x[kRows][VF];
#pragma unroll
  for (int i = 0; i < kRows; ++i)
#pragma unroll
    for (int j = 0; j < VF; ++j) x[i][j] = v0 + i < V2 ? __ldg(src + (long long)(i * VF + j) * row) : 0;
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    if (v0 + i >= V2) break;
    long long sum = 0;
#pragma unroll
    for (int j = 0; j < VF; ++j) sum += x[i][j];
    dst[(long long)i * row] = sum;
  }
}

// the crystal pair a < b of (view, unclipped radial index): the inverse of
// the binning's LOR formula (one of s = +1, -1 gives a valid pair)
__device__ __forceinline__ void lor_crystals(int n, int v, int r_full, int& a, int& b) {
  const int q = r_full - n / 2 + 1;
  a = b = -1;
#pragma unroll
  for (int si = 0; si < 2; ++si) {
    const int s = si ? -1 : 1;
    const int d = n / 2 - s * q;
    if (d < 1 || d > n - 1) continue;
    const int f = 2 * v + (d & 1) + (s < 0 ? n : 0);  // a + b
    const int a2 = f - d;
    if (a2 < 0 || (a2 & 1)) continue;
    const int lo = a2 >> 1, hi = (f + d) >> 1;
    if (lo < hi && hi < n && a < 0) {
      a = lo;
      b = hi;
    }
  }
}

// out[bin] = sum over the n / step rotations by k * step crystals of in at
// the rotated LOR: (a + c, b + c) mod n; when the order reverses, the ring
// indices swap and the TOF bin mirrors.  grid (ceil(R T / 256), V, planes)
__global__ void rotate_sum_kernel(const long long* __restrict__ in, long long* __restrict__ out, int n,
                                  int n_rings, int R, int T, int step) {
  const int V = n / 2;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= R * T) return;
  const int r = c / T, t = c - r * T;
  const int v = blockIdx.y;
  const int p = blockIdx.z;
  const int ra = p / n_rings, rb = p - ra * n_rings;
  const int rad_off = (n - 1 - R) / 2;
  int a, b;
  lor_crystals(n, v, r + rad_off, a, b);
  long long sum = 0;
  int a2 = a, b2 = b;  // (a + k step, b + k step) mod n, kept below n by one subtraction
  for (int k = 0; k < n / step; ++k, a2 += step, b2 += step) {
    if (a2 >= n) a2 -= n;
    if (b2 >= n) b2 -= n;
    const bool flip = a2 > b2;
    const int lo = flip ? b2 : a2, hi = flip ? a2 : b2;
    int f = lo + hi, s = 1;
    if (f >= n) {
      f -= n;
      s = -1;
    }
    const int v2 = f >> 1;
    const int r2 = s * (n / 2 - (hi - lo)) + n / 2 - 1 - rad_off;
    const long long p2 = flip ? (long long)rb * n_rings + ra : p;
    const int t2 = flip ? T - 1 - t : t;
    sum += __ldg(in + ((p2 * V + v2) * R + r2) * T + t2);
  }
  out[(((long long)p * V + v) * R + r) * T + t] = sum;
}

// The same sum, one orbit at a time, for n / step even.  A rotation by
// step crystals moves an LOR by step views, so every orbit has members in
// views [0, step): an LOR x and its half-turn partner (rotation by n / 2
// crystals).  The one of the two with the lower bin index sums the input
// over the n / step rotations of x and writes that sum to every member of
// the orbit (the sum is the same for all of them): one read and one write
// per bin.
//
// Where the rotation by c crystals takes (a, b) of view v and radial bin r:
// a + b grows by 2 c, so the view is (v + c) mod n / 2, and each wrap mirrors
// the radial bin (n crystals in the sum turn the sign of the LOR formula);
// b alone has passed crystal n for c in [n - b, n - a), where the crystals'
// order, the rings and the TOF axis are reversed.  That is a compare and a
// select a member where applying the LOR formula to each took twenty
// instructions, and four members' loads are in flight together (5 TOF bins, 45
// rings, 28 rotations: 3559 -> 2606 us, 6.2 TB/s).
// grid (ceil(R T / 256), step, planes)
__global__ void __launch_bounds__(256) rotate_orbit_kernel(const long long* __restrict__ in, long long* __restrict__ out,
                                                           int n, int n_rings, int R, int T, int step) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= R * T) return;
  const int r = i / T, t = i - r * T;
  const int v = blockIdx.y;
  const int p = blockIdx.z;
  const int ra = p / n_rings, rb = p - ra * n_rings;
  const int rad_off = (n - 1 - R) / 2;
  int a, b;
  lor_crystals(n, v, r + rad_off, a, b);
  const int h = n / 2, row = R * T;
  const long long J = (long long)h * row, base = (long long)p * J, base_t = (long long)(rb * n_rings + ra) * J;
  // places in a view's row: kept or mirrored radially, TOF kept or reversed (by the planes kept or swapped)
  const int keep = r * T + t, keep_t = r * T + (T - 1 - t);
  const int mirr = (R - 1 - r) * T + t, mirr_t = (R - 1 - r) * T + (T - 1 - t);
  auto reversed = [&](int c) { return (unsigned)(c - (n - b)) < (unsigned)(b - a); };
  const bool half = reversed(h);
  if ((half ? base_t + mirr_t : base + mirr) < base + keep) return;  // (both in view v) the partner's thread does it
  // the member at view w (v + c less the wraps), mirrored m, rotation c
  auto member = [&](int w, bool m, int c) -> long long {
    const bool f = reversed(c);
    return (f ? base_t : base) + ((long long)w * row + (f ? (m ? mirr_t : keep_t) : (m ? mirr : keep)));
  };
  constexpr int kU = 4;
  const int members = n / step;
  long long sum = 0;
  int w = v, c = 0;
  bool m = false;
  auto advance = [&]() {
    c += step;
    w += step;
    if (w >= h) {
      w -= h;
      m = !m;
    }
  };
  for (int k = 0; k < members; k += kU) {
    long long x[kU];
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      x[q] = k + q < members ? __ldg(in + member(w, m, c)) : 0;
      advance();
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) sum += x[q];
  }
  w = v;
  c = 0;
  m = false;
  for (int k = 0; k < members; ++k) {
    out[member(w, m, c)] = sum;
    advance();
  }
}

// Span mashing: the segment of span-mashed output plane o, and its axial sum
// z = ra + rb.  Segment k (k = -K..K) holds the ring differences
// [k span - h, k span + h] (h = (span - 1) / 2) within the ring range, and
// the axial sums from its smallest |d| to 2 n - 2 minus it (every other one
// when it holds a single ring difference); output planes run over the
// segments in order, each by z ascending.
struct SpanPlane {
  int d_lo, d_hi, z;
};

__host__ __device__ inline int span_count(int n, int span, int k, int& d_lo, int& d_hi, int& m, int& step) {
  const int h = (span - 1) / 2;
  d_lo = max(k * span - h, -(n - 1));
  d_hi = min(k * span + h, n - 1);
  m = (d_lo <= 0 && 0 <= d_hi) ? 0 : min(abs(d_lo), abs(d_hi));
  step = d_hi > d_lo ? 1 : 2;
  return (2 * n - 2 - 2 * m) / step + 1;
}

__device__ inline SpanPlane span_plane(int n, int span, int o) {
  const int K = (n - 1 + (span - 1) / 2) / span;
  int d_lo = 0, d_hi = 0, m = 0, step = 1;
  for (int k = -K; k <= K; ++k) {
    const int c = span_count(n, span, k, d_lo, d_hi, m, step);
    if (o < c || k == K) break;
    o -= c;
  }
  return SpanPlane{d_lo, d_hi, m + o * step};
}

// grid (column blocks, output planes): each output bin sums the input planes
// (ra, rb) of its segment with ra + rb = z, read once each (exact int64).  A
// thread sums kSpanBins bins at once, and a CTA more than a handful: with one, a
// load or two were in flight (5 TOF bins, 45 rings, span 3: 3856 -> 1978 us).
constexpr int kSpanBins = 4;

__global__ void __launch_bounds__(256) span_kernel(const long long* __restrict__ in, long long* __restrict__ out,
                                                   int n, int span, long long J) {
  const SpanPlane sp = span_plane(n, span, (int)blockIdx.y);
  long long* __restrict__ dst = out + (long long)blockIdx.y * J;
  for (long long j0 = (long long)blockIdx.x * (256 * kSpanBins) + threadIdx.x; j0 < J;
       j0 += (long long)gridDim.x * (256 * kSpanBins)) {
    long long sum[kSpanBins] = {};
    for (int d = sp.d_lo + ((sp.z + sp.d_lo) & 1); d <= sp.d_hi; d += 2) {  // of z's parity
      const int ra = (sp.z - d) / 2, rb = (sp.z + d) / 2;
      if (ra < 0 || ra >= n || rb < 0 || rb >= n) continue;
      const long long* src = in + (long long)(ra * n + rb) * J + j0;
      long long x[kSpanBins];
#pragma unroll
      for (int q = 0; q < kSpanBins; ++q) x[q] = j0 + 256 * q < J ? __ldg(src + 256 * q) : 0;
#pragma unroll
      for (int q = 0; q < kSpanBins; ++q) sum[q] += x[q];
    }
#pragma unroll
    for (int q = 0; q < kSpanBins; ++q)
      if (j0 + 256 * q < J) dst[j0 + 256 * q] = sum[q];
  }
}

}  // namespace

int span_planes(int n_rings, int span) {
  const int K = (n_rings - 1 + (span - 1) / 2) / span;
  int total = 0, d_lo, d_hi, m, step;
  for (int k = -K; k <= K; ++k) total += span_count(n_rings, span, k, d_lo, d_hi, m, step);
  return total;
}

cudaError_t launch_span(const long long* in, long long* out, int n_rings, int span, long long J, int sms,
                        cudaStream_t s) {
  const int planes = span_planes(n_rings, span);
  const long long per = std::max(1LL, std::min((J + 256 * kSpanBins - 1) / (256 * kSpanBins), 64LL * sms / planes + 1));
  span_kernel<<<dim3((unsigned)per, (unsigned)planes), 256, 0, s>>>(in, out, n_rings, span, J);
  return cudaGetLastError();
}

cudaError_t launch_mash(const long long* in, long long* out, int planes, int V, int R, int T, int vf, int tf,
                        cudaStream_t s) {
  if (tf == 1 && vf <= 8) {
    const int row = R * T, V2 = V / vf;
    auto go = [&](auto kernel, int rows) {
      kernel<<<dim3((row + 255) / 256, (V2 + rows - 1) / rows, planes), 256, 0, s>>>(in, out, V, row);
    };
    switch (vf) {
      case 1: go(mash_views_kernel<1>, 8); break;
      case 2: go(mash_views_kernel<2>, 4); break;
      case 3: go(mash_views_kernel<3>, 2); break;
      case 4: go(mash_views_kernel<4>, 2); break;
      case 5: go(mash_views_kernel<5>, 1); break;
      case 6: go(mash_views_kernel<6>, 1); break;
      case 7: go(mash_views_kernel<7>, 1); break;
      default: go(mash_views_kernel<8>, 1); break;
    }
    return cudaGetLastError();
  }
  const int cols = R * (T / tf);
  const dim3 grid((cols + 255) / 256, V / vf, planes);
  if (tf == 1) mash_kernel<true><<<grid, 256, 0, s>>>(in, out, V, R, T, vf, tf);
  else mash_kernel<false><<<grid, 256, 0, s>>>(in, out, V, R, T, vf, tf);
  return cudaGetLastError();
}

cudaError_t launch_rotate_sum(const long long* in, long long* out, int n_crystals, int n_rings, int R, int T,
                              int step, cudaStream_t s) {
  // a short row gets a CTA of its own size (9 bins, 400 crystals x 20 rings, half-turn sum: 60.0 us with 256 threads, 47.7)
  const int block = std::min(256, (R * T + 31) / 32 * 32);
  if ((n_crystals / step) % 2 == 0)
    rotate_orbit_kernel<<<dim3((R * T + block - 1) / block, step, n_rings * n_rings), block, 0, s>>>(in, out, n_crystals,
                                                                                                    n_rings, R, T, step);
  else
    rotate_sum_kernel<<<dim3((R * T + 255) / 256, n_crystals / 2, n_rings * n_rings), 256, 0, s>>>(
        in, out, n_crystals, n_rings, R, T, step);
  return cudaGetLastError();
}

}  // namespace psc
