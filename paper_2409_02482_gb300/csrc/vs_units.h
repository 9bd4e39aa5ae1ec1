// Sizes of the raster's work units: rules on the sizes of meshes, images and
// the launch, in plain C++ (no CUDA), so that the host can be tested alone.
//
// A unit costs about 5 ns of the words that all warps share, whatever its
// size (its number and its completion are atomics on them), and its triangles
// run 32 at a time, one after the other.  So a launch wants enough units that
// every warp finds some and none lasts long, and no more.
#pragma once

namespace vsu {

// A raster unit of a batch is cut, down to kLeastTris triangles, while its
// shell's triangles would cover more than kUnitPixels pixels if the shell
// filled the image: the units of a shell of 10 k triangles are then about as
// long as those of one with 1 M, and the shading of a view does not wait for
// its last few coarse units.  Fused step over 8 objects with 10 k to 1 M
// triangles per shell: 7.32 ms with equal units, 4.72 at 32 triangles at
// least, 4.56 at 8, the same at 1.  kUnitPixels = 1024 halves the units of a
// 4K view of 9 x 2 M triangles, 10.34 -> 10.70 ms; 1400 to 4096 are within
// 0.3 % of each other there and at 800^2.
constexpr int kUnitPixels = 2048, kLeastTris = 8;

// Units of fewer pixels than this are not cut to give each warp several.  16
// views of 5 x 20 k triangles at 100 x 1000, where the few triangles of the
// strip have all its pixels: 550 us at 512, 618 at 1024, 783 uncut.  12 fitting
// views of 5 x 10 k at 200^2: 425 us at 512, 371 at 1024 and uncut.
constexpr int kSharePixels = 600;

struct RasterUnits {
  int tris;   // triangles per unit
  int lg;     // a unit of one triangle is shared by 2^lg units
};

// Raster units of an item in a launch over n items of `tris` triangles
// together, run by `warps` resident warps: units of the asked size while
// every warp finds one, else smaller.  A batch stops at 32 triangles, one per
// lane; a launch of one item goes down to one triangle, which 2, 4 .. 64 warps
// then share: at 256^2, 3 x 1224 triangles took 253 us in units of 32 (115
// warps busy) and take 7 us one by one.  The items of a batch count together,
// because they run beside one another: with a quarter of the warps for each
// item by itself, 64 fitting views of 3 x 2 k triangles at 64^2 had 12 k units
// of 32 and took 326 us, and take 251 with 3 k units of 128.
inline RasterUnits raster_units(long long tris, int asked, int n, int warps) {
  RasterUnits u = {asked, 0};
  const int least = n > 1 ? 32 : 1;
  while (u.tris > least && tris / u.tris < warps) u.tris /= 2;
  while (u.tris == 1 && u.lg < 6 && (tris << (u.lg + 1)) <= warps) ++u.lg;
  return u;
}

// Triangles per raster unit of one shell (`tris` triangles, image of `pixels`)
// in a batch of n items with batch_tris triangles, from the item's `unit`: cut
// to kUnitPixels; and, where several items run, while fewer units than n / 4
// (at most 4) per warp would be left, to kSharePixels, so that warps with short
// units take others' work.
inline int shell_unit(int unit, int tris, long long pixels, long long batch_tris, int n, int warps) {
  while (unit > kLeastTris && unit * pixels > (long long)kUnitPixels * tris) unit /= 2;
  if (n > 1) {
    const long long enough = (long long)warps * (n < 16 ? n : 16) / 4;
    while (unit > 32 && unit * pixels > (long long)kSharePixels * tris && batch_tris / unit < enough) unit /= 2;
  }
  return unit;
}

}  // namespace vsu
