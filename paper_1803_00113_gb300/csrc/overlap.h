// The part of a neighbour's patch that lies in a run of an own patch's pixels:
// index arithmetic of the rendered backgrounds, for host and device (no CUDA
// types, so that it can be enumerated on the host).
#pragma once

#ifdef __CUDACC__
#define CELESTE_HD __host__ __device__ __forceinline__
#else
#define CELESTE_HD inline
#endif

namespace celeste {

// Pixels begin..end - 1 (row-major) of a rectangle w columns wide whose corner
// is column x, row y of the own patch.
struct Overlap {
  int x, y, w, begin, end;
};

CELESTE_HD int overlap_clamp(int v, int hi) { return v < 0 ? 0 : (v > hi ? hi : v); }

// Own pixels c0..c1 - 1 (c0 < c1, row-major) of a patch w wide against a
// neighbour's nw x nh patch, (nx, ny) from the own patch's frame to the
// neighbour's: the overlap in the rows of the run, without what the run's
// first and last row have before and after it.  Empty: end <= begin.
CELESTE_HD Overlap chunk_overlap(int c0, int c1, int w, int nx, int ny, int nw, int nh) {
  const int r0 = c0 / w, r1 = (c1 - 1) / w + 1;
  Overlap o;
  o.x = nx < 0 ? -nx : 0;
  o.w = (w < nw - nx ? w : nw - nx) - o.x;
  o.y = r0 > -ny ? r0 : -ny;
  const int h = (r1 < nh - ny ? r1 : nh - ny) - o.y;
  o.begin = o.end = 0;
  if (o.w <= 0 || h <= 0) return o;
  if (o.y == r0) o.begin = overlap_clamp(c0 - r0 * w - o.x, o.w);
  o.end = o.w * h;
  if (o.y + h == r1) o.end -= overlap_clamp(o.x + o.w - (c1 - (r1 - 1) * w), o.w);
  return o;
}

}  // namespace celeste
