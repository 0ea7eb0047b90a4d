// Launch shapes of collision_kernel<T, N, W>: thread-block cluster size, plane groups per CTA and the
// CTAs per SM the registers are sized for.  DGFS_SHAPE3: VHS batches (paper_1903_03056_gb300/tune.py writes
// these lines); DGFS_WIDE: the shape of small VHS batches where they use one of their own; DGFS_VSS: VSS plans.
// Grids up to N = 12 have CTAs of one to five warps: sized for one CTA an SM they held 4 to 10 warps (FP32, VHS,
// 8000 two-species nodes, M = 12: N = 6 1181 -> 827 us, 8 1688 -> 1390, 12 14.7 -> 7.8 ms; VSS 2000 nodes:
// 653 -> 426 us, 810 -> 738, 8.2 -> 4.1 ms).
#pragma once

DGFS_SHAPE3(float, 4, 1, 4, 16)
DGFS_SHAPE3(float, 6, 1, 6, 8)
DGFS_SHAPE3(float, 8, 1, 8, 6)
DGFS_SHAPE3(float, 12, 1, 12, 3)
DGFS_SHAPE3(float, 16, 1, 8, 4)
DGFS_SHAPE3(float, 24, 1, 8, 2)
DGFS_SHAPE3(float, 32, 2, 4, 3)
DGFS_SHAPE3(float, 48, 4, 4, 2)
DGFS_SHAPE3(double, 4, 1, 4, 1)
DGFS_SHAPE3(double, 6, 1, 6, 1)
DGFS_SHAPE3(double, 8, 1, 8, 1)
DGFS_SHAPE3(double, 12, 1, 12, 1)
DGFS_SHAPE3(double, 16, 1, 8, 1)
DGFS_SHAPE3(double, 24, 6, 4, 1)
DGFS_SHAPE3(double, 32, 4, 4, 2)
DGFS_SHAPE3(double, 48, 4, 1, 1)

// ... and how many times longer the wide shape takes per radial node on a full device (measured:
// N = 16 7.16 / 4.72 ms, 24 15.2 / 10.6, 32 14.1 / 12.4, 48 13.9 / 10.8; FP64 8 6.70 / 3.25,
// 12 10.7 / 9.47, 16 12.7 / 11.2)
DGFS_WIDE(float, 16, 8, 2, 1, 1.5)
DGFS_WIDE(float, 24, 6, 4, 5, 1.43)
DGFS_WIDE(float, 32, 8, 4, 3, 1.14)
DGFS_WIDE(float, 48, 8, 6, 1, 1.29)
DGFS_WIDE(double, 8, 4, 2, 1, 2.06)
DGFS_WIDE(double, 12, 6, 2, 1, 1.13)
DGFS_WIDE(double, 16, 8, 2, 1, 1.13)

// VSS plans (W = 2).  N = 32: 8-CTA clusters, 60 one-species nodes of 9 radial nodes 1395 (2, 4, 3) -> 561 us,
// 200 two-species nodes 23.6 -> 21.9 ms; N = 16 (2, 8, 4) -> (1, 16, 2) 600 two-species nodes 3.61 -> 3.49 ms
DGFS_VSS(float, 4, 1, 4, 1)
DGFS_VSS(float, 6, 1, 6, 8)
DGFS_VSS(float, 8, 1, 8, 8)
DGFS_VSS(float, 12, 1, 12, 3)
DGFS_VSS(float, 16, 1, 16, 2)
DGFS_VSS(float, 24, 1, 8, 2)
DGFS_VSS(float, 32, 8, 4, 4)
DGFS_VSS(float, 48, 8, 2, 4)
DGFS_VSS(double, 4, 1, 4, 1)
DGFS_VSS(double, 6, 1, 6, 1)
DGFS_VSS(double, 8, 1, 8, 1)
DGFS_VSS(double, 12, 1, 12, 2)
DGFS_VSS(double, 16, 1, 8, 1)
DGFS_VSS(double, 24, 6, 4, 1)
DGFS_VSS(double, 32, 4, 4, 2)
DGFS_VSS(double, 48, 4, 1, 1)
