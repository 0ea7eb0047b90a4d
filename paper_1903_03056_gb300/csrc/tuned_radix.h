// Radix schedule of the register line transform per (precision, N): the decimal digits of the
// code, first stage first (442 = radix 4, 4, then 2).  paper_1903_03056_gb300/tune.py --radix times the
// orders on the device and writes these lines.
// FP32 lines of N points run as transforms of N / 2, so the FP32 entry of N / 2 serves grid size N.
// Where the orders' times agree within 2 %, the one with the smallest error against 64 bits is kept (64
// nodes, 2-norm): 16 takes 44 (N = 32: 1.10e-6 of ||Q||, 149.8 ms; 82 1.23e-6, 148.1), 24 takes 243 (N = 48:
// 9.80e-7, 296.3 ms; 38 1.23e-6, 294.2), 12 takes 43 (N = 24: 8.9e-7; 34 1.06e-6, the same time).
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
