// Launch shapes of vhs_kernel<T, N, W>: thread-block cluster size, plane groups per CTA and the CTAs
// per SM the registers are sized for; DGFS_VHS_WIDE where small batches use a shape of their own
#pragma once

DGFS_VHS_SHAPE(float, 4, 1, 4, 1)
DGFS_VHS_SHAPE(float, 6, 1, 6, 1)
DGFS_VHS_SHAPE(float, 8, 1, 8, 1)
DGFS_VHS_SHAPE(float, 12, 1, 12, 1)
DGFS_VHS_SHAPE(float, 16, 1, 8, 4)
DGFS_VHS_SHAPE(float, 24, 1, 8, 2)
DGFS_VHS_SHAPE(float, 32, 2, 4, 3)
DGFS_VHS_SHAPE(float, 48, 4, 4, 2)
DGFS_VHS_SHAPE(double, 4, 1, 4, 1)
DGFS_VHS_SHAPE(double, 6, 1, 6, 1)
DGFS_VHS_SHAPE(double, 8, 1, 8, 1)
DGFS_VHS_SHAPE(double, 12, 1, 12, 1)
DGFS_VHS_SHAPE(double, 16, 1, 8, 1)
DGFS_VHS_SHAPE(double, 24, 6, 4, 1)
DGFS_VHS_SHAPE(double, 32, 4, 4, 2)
DGFS_VHS_SHAPE(double, 48, 4, 1, 1)

// ... and how many times longer the wide shape takes per radial node on a full device (measured:
// N = 16 7.16 / 4.72 ms, 24 15.2 / 10.6, 32 14.1 / 12.4, 48 13.9 / 10.8; FP64 8 6.70 / 3.25,
// 12 10.7 / 9.47, 16 12.7 / 11.2)
DGFS_VHS_WIDE(float, 16, 8, 2, 1, 1.5)
DGFS_VHS_WIDE(float, 24, 6, 4, 5, 1.43)
DGFS_VHS_WIDE(float, 32, 8, 4, 3, 1.14)
DGFS_VHS_WIDE(float, 48, 8, 6, 1, 1.29)
DGFS_VHS_WIDE(double, 8, 4, 2, 1, 2.06)
DGFS_VHS_WIDE(double, 12, 6, 2, 1, 1.13)
DGFS_VHS_WIDE(double, 16, 8, 2, 1, 1.13)
