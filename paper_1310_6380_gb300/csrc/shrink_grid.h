// Launches that need all their blocks resident at once (grid barriers), for
// kernels that are right with any number of blocks.  How many fit is not known
// beforehand: the process may be given fewer SMs than the device has (a client
// limit, a partition), and then the launch of a full grid is refused.
#pragma once

// launch(grid) until it is not refused as too large: grid, grid / 2, ... 1.
// Returns the last launch's status.
template <typename Status, typename Launch>
Status bs_shrink_grid(int grid, Status too_large, Launch launch) {
  for (;;) {
    const Status e = launch(grid);
    if (e != too_large || grid <= 1) return e;
    grid /= 2;
  }
}
