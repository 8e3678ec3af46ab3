// How one launch of k_residual shares out its work (also compiled by the host's
// compiler alone: no CUDA names).
#pragma once

#ifdef __CUDACC__
#define PS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define PS_HOST_DEVICE inline
#endif

namespace ps {

struct ResidualSplit {
  bool wide;             // work items of 1024 cells, else of 256
  int items_per_plane;
  int items;             // of all active planes; block b takes items b, b + grid, ..
  int waiting;           // blocks without an item whose arrival the retirement awaits
};

// nact planes of bpp 256-cell pieces on a grid of `grid` blocks and `sms` SMs.
// With many cells active the per-item reduction, fence and arrival count are paid
// once per 1024 cells; with few planes, or where that leaves fewer than two blocks
// an SM, items of 256 cells spread a plane's FP64 work over more SMs (17 planes of
// 32 x 32 cells, FP64: 8.2 us, 14.2 with 17 blocks).
//
// A launch's last arrival rewrites the count of active planes, and nothing but
// that arrival orders it after a block that the launch starts late.  Such a block
// must find no item with the smaller count either.  Small items are fewer the
// fewer planes are active, so a block beyond them stays idle; but below the line
// small items take over from large ones and are four times as many, so with large
// items the idle blocks arrive as well and none can be late (their arrivals take
// no time that shows: 17 to 513 planes of 32 x 32 to 512 x 512 cells within 3 %).
PS_HOST_DEVICE ResidualSplit residual_split(int nact, int bpp, int grid, int sms) {
  ResidualSplit s;
  s.wide = nact >= 16 && nact * bpp >= 4 * 2 * sms;
  s.items_per_plane = s.wide ? (bpp + 3) / 4 : bpp;
  s.items = nact * s.items_per_plane;
  s.waiting = s.wide && s.items < grid ? grid - s.items : 0;
  return s;
}

}  // namespace ps
