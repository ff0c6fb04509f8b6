// Host rules that choose how a call runs (no CUDA types, so that they can be
// compiled and checked without a device).
#pragma once

namespace fw2 {

// Sources of a 2D pipelined context: inside the half steps (one warp of each
// block adds those of its half tiles) or by a kernel of their own after each
// half step.  Inside, a block's warp takes about 1.5 us for a half tile with
// sources, 9 ns more for each of its targets and a memory latency (0.6 us) for
// each further entry of a target, one after the other; kernels of their own,
// with a launch per half step, cost about 16 us a step more.  The line is
// where the two meet, at ten half tiles per SM: 2048 x 1024 (N = 4, float)
// with every cell a source took 223 us a step inside and takes 104 apart, a
// quarter of the cells 123 and 96, one in 64 100 and 94; 512 x 512 with every
// cell 25 either way, with a quarter of them 19 inside.  It also keeps what a
// block adds within a few ms, far below the limit of the waits that the other
// blocks spend on it.
// half_tiles: half tiles with sources, targets: cells fed, extra: entries
// beyond the first of a target, each summed over the fields.
inline bool sources_apart(long long half_tiles, long long targets, long long extra, int n_sm) {
  return (double)half_tiles + (double)targets / 170.0 + 0.4 * (double)extra > 10.0 * n_sm;
}

// Recording of a 2D pipelined context: inside a launch of many steps (each
// group summed by one thread in the following half step, while the others of
// its warp wait), or by a kernel of its own after launches of one step.
// Inside, a long group costs 55 to 80 ns a cell that the whole grid waits for
// (35 to 50 in its own kernel), with a limit on that wait of 2 s; launches of
// one step cost 3 to 7 us a step and the kernel 4.  512 x 512 and 2048 x 1024
// (N = 4), groups of 256 cells: 31 and 111 us a step inside; of 512: 46 and
// 126 apart; of 10000: 554 and 844 inside, 350 and 594 apart.  Many sensors:
// every cell of 2048 x 1024 140 inside and 107 apart, a quarter 95 and 96.
// longest: cells of the longest group, cells: of all groups.
inline bool record_apart(long long longest, long long cells) { return longest > 384 || cells > (1ll << 19); }

// Field copies between a context and a caller's device buffer: by a kernel
// where the context's device is current and holds the buffer, else by the copy
// calls, which reach any device from any other (a kernel would be launched on
// the current device and follow the pointers of another).
// buf_device: device of the buffer, -1 where it is not device memory.
inline bool copy_by_kernel(int ctx_device, int current_device, int buf_device, bool aligned) {
  return aligned && buf_device >= 0 && buf_device == ctx_device && current_device == ctx_device;
}

}  // namespace fw2
