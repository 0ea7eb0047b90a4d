// Radix schedule of the register line transform per (precision, N): the decimal digits of the
// code, first stage first (442 = radix 4, 4, then 2).  paper_1903_03056_gb300/tune.py --radix times the
// orders on the device and writes these lines.
// FP32 lines of N points run as transforms of N / 2, so the FP32 entry of N / 2 serves grid size N.
// Where the orders' times agree within 1 %, the one with the smallest error against 64 bits is kept:
// 16 takes 44 (N = 32: 1.32e-6 -> 1.21e-6 of ||Q|| on 8 two-species nodes, 28 measured 145.5 ms against
// 146.0), 24 takes 243 (N = 48: 1.45e-6 -> 1.23e-6, 38 35.8 ms against 36.1); radix 3 last is the better
// order throughout.
#pragma once

DGFS_RADIX(float, 4, 4)
DGFS_RADIX(float, 6, 23)
DGFS_RADIX(float, 8, 42)
DGFS_RADIX(float, 12, 43)
DGFS_RADIX(float, 16, 44)
DGFS_RADIX(float, 24, 243)
DGFS_RADIX(float, 32, 228)
DGFS_RADIX(float, 48, 344)
DGFS_RADIX(double, 4, 4)
DGFS_RADIX(double, 6, 23)
DGFS_RADIX(double, 8, 42)
DGFS_RADIX(double, 12, 43)
DGFS_RADIX(double, 16, 44)
DGFS_RADIX(double, 24, 423)
DGFS_RADIX(double, 32, 442)
DGFS_RADIX(double, 48, 443)
