// Size buckets of the mixed-precision forward: which engine takes a row of order m.
// Written by paper_1710_10899_gb300/tune.py from forward times measured on a GB300 (the
// measurements are listed below); rows of order m <= kTunedSmallMaxM go to the small engine
// (working set in shared memory, 16 x 8 warp tiles of mma.sync), rows with
// kTunedSmallMaxM < m <= kTunedSyncMaxM to the mma.sync engine (64 x 64 tiles, cp.async
// pipeline), the rest to the tcgen05 engine (128 x 96 tiles in TMEM, TMA pipeline).
// Device: NVIDIA GB300; p = 2; 7296 rows of one order per case; ms per forward
// (median):
//     m        small      sync   tcgen05
//     8        1.806     4.832     3.745
//    16        1.823     4.978     3.874
//    24        2.115     5.206     4.234
//    32        2.265     5.398     4.360
//    48            -     6.325     5.252
//    64            -     6.827     6.324
//    96            -    16.404     8.414
//   128            -    18.568    11.695
#pragma once
namespace submat {
constexpr int kTunedSmallMaxM = 32;
constexpr int kTunedSyncMaxM = 0;
}  // namespace submat
