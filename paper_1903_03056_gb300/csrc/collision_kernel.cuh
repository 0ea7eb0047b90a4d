// Persistent collision kernel: one thread-block cluster per work item (node b, task), on real
// transforms.
//
// Only Re Q is wanted, and for VHS (alpha = 1) the gain weight F(k, rho) and the loss weight G^-(k) are real
// and even in k, so Q_ij = IDFT(sum_rho w F DFT(Re P_rho)) - f_i IDFT(G^- f_hat_j) holds with the
// real part of the products alone:
//
//     Re P = sum_e w_e (Re a_e Re b_e - Im a_e Im b_e).
//
// f is real, so the shifted copies a_e, b_e would be real too but for the unpaired modes at index
// N/2 of an axis: there the phase e^{i theta k} has no conjugate partner and leaves
// c + i t = cos - i sin of theta N / 2.  Write the shift along one axis as R + i t Pi, R the
// real shift (phase c at the unpaired mode) and Pi the projection on that mode, an alternating
// sequence.  The product over the three axes gives
//
//     Re a = RxRyRz f - ty tz RxPyPz f - tx tz PxRyPz f - tx ty PxPyRz f
//     Im a = tx PxRyRz f + ty RxPyRz f + tz RxRyPz f - tx ty tz PxPyPz f.
//
// Every term but the first lives on faces or edges of the mode cube, so a shifted copy costs one
// real 3D transform and two real 2D ones (the faces k_x = N/2 and k_y = N/2; the face k_z = N/2
// falls out of the y pass, see below) instead of a complex 3D transform: half the arithmetic and
// half the workspace.
//
// Layouts.  A spectrum keeps columns c = 0..N/2-1 of the z modes; column 0 holds
// X(k_z = 0) + i X(k_z = N/2) ("C form": every x and y pass is linear and maps each part to
// itself, so the pair travels as one complex line).  Rows of N complex values hold two such half
// rows: role 0 (species i, shift +) and role 1 (species j, shift -).  After the inverse y pass
// column 0 is (a(k_z = 0), a(k_z = N/2)), two real numbers.  The product's spectrum splits column
// 0 over k_y instead ("N form", row r of column 0: r = 1..N/2-1 is (k_y = r, k_z = 0), N/2 + r is
// (k_y = r, k_z = N/2), row 0 holds X(0,0) + i X(N/2,0) and row N/2 holds X(0,N/2) + i X(N/2,N/2)),
// since there the weights of the two parts differ.
//
// Per radial node the phases run as a pipeline over sigma_x groups: phase 0 transforms the faces of
// all entries and runs step A of group 0; phase k runs step A of group k and step B of group
// k - 1; one cluster barrier each.
//   step A  x pass of both roles' half spectra (one thread per pencil, coalesced)
//   step B  per plane x and entry: y phases, y pass of N/2 columns of either role (one line per
//           thread), transpose through shared memory, z phases and the real z transform of both
//           roles (one row per thread), and the product into P, N real values per thread
//   step C  after the last group: P -> spectrum, Q_hat_ij += F_ij P_hat (and Q_hat_ji for a cross pair)
//
// VSS (alpha != 1, W = 2): F depends on sigma and is complex, so every entry's product, now complex
// (Im a Re b + Re a Im b beside the real part), is transformed forward by itself in step B, and step C
// runs two phases behind step A, entry by entry, on the half space of its Hermitian part (vss_step_c).
// Groups hold one or two entries.
//
// The finish transforms gain and loss back, whose rounding every result keeps: FP32 carries it along
// there (VGeo::FINE_Z).
//
// Measured on the GB300 against the complex-transform kernel this one replaced: 4096 nodes of N = 32
// FP32 285 -> 151 ms, 3001 of N = 24 74.9 -> 37.7, 8192 of N = 16 28.6 -> 16.7, 61 three-species nodes
// of N = 48 86.0 -> 35.9, 61 nodes of N = 32 FP64 184 (201 on another device) -> 83, VSS 37 three-species
// nodes of N = 48 (M = 32) 339 -> 146 ms.  What bounds it: FP64 the FP64 pipe (79 % of its cycles); FP32 latency -- the
// FMA pipes run half their cycles (N = 16: the L1 data path three quarters), the stalls are L2 loads
// of the x-passed spectra, whose workspaces together exceed L2 from N = 24 on.
#pragma once

#include <algorithm>
#include <cmath>

#include <cuda_runtime.h>

#include "dd_line.cuh"
#include "dgfs_internal.h"
#include "group_sync.cuh"
#include "launch_plan.h"
#include "real_line.cuh"
#include "tcgen05.cuh"

namespace dgfs {

// Launch shape per (precision, N, W): cluster size, plane groups per CTA, CTAs per SM the registers
// are sized for.  W = 0 serves batches that fill the device; W = 1, where it differs, spreads one
// work item over more SMs for small batches (one plane per group, clusters of 4 to 8 CTAs).
template <typename T, int N, int W> struct VShape : VShape<T, N, 0> {};
template <typename T, int N> struct HasWide {
  static constexpr bool value = false;
  static constexpr double slow = 1.0;
};
#define DGFS_SHAPE3(TT, NN, CC, GG, MB)   \
  template <> struct VShape<TT, NN, 0> {     \
    static constexpr int cluster = CC;       \
    static constexpr int groups = GG;        \
    static constexpr int min_blocks = MB;    \
  };
#define DGFS_VSS(TT, NN, CC, GG, MB)   \
  template <> struct VShape<TT, NN, 2> {     \
    static constexpr int cluster = CC;       \
    static constexpr int groups = GG;        \
    static constexpr int min_blocks = MB;    \
  };
#define DGFS_WIDE(TT, NN, CC, GG, MB, SLOW)    \
  template <> struct VShape<TT, NN, 1> {     \
    static constexpr int cluster = CC;       \
    static constexpr int groups = GG;        \
    static constexpr int min_blocks = MB;    \
  };                                         \
  template <> struct HasWide<TT, NN> {       \
    static constexpr bool value = true;      \
    static constexpr double slow = SLOW;     \
  };
#include "tuned_shapes.h"
#undef DGFS_SHAPE3
#undef DGFS_WIDE
#undef DGFS_VSS

template <typename T, int N, int W>
struct VGeo {
  static constexpr int h = N / 2;
  static constexpr int N2 = N * N, HN2 = N * h;
  static constexpr size_t N3 = size_t(N) * N * N, HN3 = size_t(N) * HN2;
  static constexpr int PITCH = N + 1;
  static constexpr int CL = VShape<T, N, W>::cluster;
  static constexpr int GP = VShape<T, N, W>::groups;
  static constexpr int MINB = VShape<T, N, W>::min_blocks;
  static constexpr int THREADS = GP * N;
  static constexpr int PLANES = N / CL;  // planes, and rows of pencils, per CTA
  static_assert(N % CL == 0 && PLANES % GP == 0, "planes must split evenly over the cluster and its plane groups");
  // P of a plane stays in the row's thread (FP64 N = 48: in shared memory, its line alone fills
  // the registers); with one plane per group it lives there for the whole radial node, otherwise
  // it is parked in the workspace between sigma_x groups
  static constexpr bool PSM = sizeof(T) == 8 && N >= 48 && W != 2;
  // W = 2: VSS (sigma-dependent weights).  Groups hold one or two entries; each entry's product is
  // complex and transformed forward by itself
  static constexpr bool VSS = W == 2;
  static constexpr bool KEEP = PLANES == GP;
  // L2 prefetch of a group's next plane one plane ahead (measured: N = 32 -1.8 %, 48 -0.8 %, smaller
  // grids, whose workspaces mostly stay in L2, +0.5 to 1.4 %)
  static constexpr bool PF = sizeof(T) == 4 && N >= 32;
  // Tensor memory (FP32): each thread owns a lane, TMEM holds its raw line of the current plane (read
  // once per sigma_x group, used by every entry of it) and the parked P of its planes.  Neither then
  // goes through L2 or the L1 data path again.  Used while the CTAs an SM holds fit its 512 columns.
  static constexpr int PPG = PLANES / GP;
  static constexpr int SETS = (THREADS + 127) / 128;  // warps that share a lane quarter
  static constexpr int alloc_of(int cols) { return cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512; }
  static constexpr bool fits(int cols) { return cols > 0 && cols <= 512 && MINB * alloc_of(cols) <= 512; }
  static constexpr bool TMOK = sizeof(T) == 4 && N % 8 == 0 && N >= 16 && N <= 32 && THREADS % 32 == 0 && W == 0;
  static constexpr int P_COLS = KEEP ? 0 : PPG * N;
  static constexpr bool TMP = TMOK && !KEEP && fits(SETS * P_COLS);
  static constexpr bool TMR = TMOK && fits(SETS * (2 * N + (TMP ? P_COLS : 0)));
  static constexpr int TM_SET = (TMR ? 2 * N : 0) + (TMP ? P_COLS : 0);  // columns of a thread
  static constexpr int TM_ALLOC = TM_SET > 0 ? alloc_of(SETS * TM_SET) : 0;
  // FP32: passes of the finish whose sums carry their rounding errors along (dd_line.cuh).  Gain and loss
  // are larger than their difference, so the rounding of these last transforms is in every result; real
  // transforms alone round more than the complex ones they replaced (a complex transform of real data leaves
  // half its error in the part that is dropped): 2-norm error 1.04 to 1.19 times theirs, N = 48 0.84 to 0.96.
  // These are the fewest passes that bring it below theirs (N = 6 to 32: 0.78 to 0.99; VSS needs y at N = 6
  // alone).  Measured: 4096 nodes of N = 32 145.2 -> 149.9 ms, 3001 of N = 24 36.6 -> 37.5, 8192 of N = 16
  // 16.3 -> 16.7, one N = 16 relaxation step 144 -> 155 us; in FP64 the same passes took 3 to 5 times that.
  static constexpr bool FINE_Z = sizeof(T) == 4 && (N <= 16 || N == 32 || (N == 24 && !VSS));
  static constexpr bool FINE_Y = FINE_Z && (VSS ? N == 6 : N != 24);
  static constexpr bool FINE_X = FINE_Y && N <= 8 && !VSS;
  static constexpr bool CALL = sizeof(T) == 4 && W == 0 && (N == 24 || N == 32);  // add_parts
  static constexpr int QU = W == 1 || N <= 12 ? 8 : CALL || sizeof(T) == 8 ? 4 : 2;
  // shared memory per group: one padded plane, the entry's row of the k_y face, P if PSM
  // (FP32: the groups' stride is 2 N words modulo 32, so that the lanes of a warp that spans two
  // groups hit distinct banks: N = 24)
  static constexpr size_t GROUP_BASE = (size_t(N) * PITCH + N) * sizeof(C<T>) + (PSM ? N2 * sizeof(T) : 0);
  static constexpr size_t GROUP_BYTES =
      GROUP_BASE + (sizeof(T) == 4 ? size_t((2 * N + 32 - int(GROUP_BASE / 4 % 32)) % 32) * 4 : 0);
  static_assert(GROUP_BYTES % 16 == 0, "16-byte accesses");
  static constexpr size_t SMEM = GP * GROUP_BYTES;
  // phase block of an entry (complex values): x [h][role], y [h][role], z [role][h] (role 1 times
  // w_e), then (w_e, 0) and a pad.  Mode 0 needs no phase: its slot holds c + i t, the unpaired mode's
  static constexpr int PB = 3 * N + 2;
  // workspace per cluster (complex values): f_hat of both species, NBH buffers of x-passed
  // half spectra of both roles, one more for the group with sigma_x = 0, P_hat, two gain accumulators, parked P; then per entry the two faces
  // and the k_x-face's k_z = N/2 line.  The same for every W of (T, N).
  static constexpr bool SPLIT = CL > 1 && (sizeof(T) == 8 || N >= 48) && !VSS;
  static constexpr int NBH = SPLIT ? 3 : 2;
  // VSS: complex product spectra [x][k_y][k_z] of up to two entries a group, double buffered, and
  // accumulators (total and current part of the radial nodes) per k_x: pencils [k_y][0..N/2], then
  // (k_y = N/2, k_z = N/2+1..N-1)
  static constexpr size_t PVN = VSS ? 4 * N3 : HN3;
  static constexpr int QROW = VSS ? N * (h + 1) + h - 1 : HN2;
  static constexpr size_t QN = VSS ? (size_t(N) * QROW + 1) / 2 * 2 : HN3;
  static constexpr size_t SLOT = VSS ? (2 + 2) * N3 + PVN + 4 * QN : (2 + 3) * N3 + 4 * HN3;
  static constexpr size_t FACE = 2 * N2 + N;
};

// v[n] *= e^{i theta k_n}, ph[2 n] the phase of mode n: mode -n (entry N - n) takes its conjugate, the
// unpaired mode the real factor c, mode 0 none
template <typename T, int N>
__device__ __forceinline__ void shift_line(C<T> (&v)[N], const C<T>* ph) {
  v[N / 2] = scale<T>(v[N / 2], ph[0].x);
#pragma unroll
  for (int n = 1; n < N / 2; ++n) {
    const C<T> f = ph[2 * n], a = v[n], b = v[N - n];
    v[n] = mk<T>(a.x * f.x - a.y * f.y, a.x * f.y + a.y * f.x);
    v[N - n] = mk<T>(b.x * f.x + b.y * f.y, b.y * f.x - b.x * f.y);
  }
}

// whether an entry (phase block pe) has a shift along x, and with it a k_x face
template <typename T> __device__ __forceinline__ bool has_face(const C<T>* pe) { return pe[0].y != T(0) || pe[1].y != T(0); }

// two neighbouring complex values (index i even) with one 16-byte access
__device__ __forceinline__ void load_two(const float2* p, float2& a, float2& b) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void load_two(const double2* p, double2& a, double2& b) {
  a = p[0];
  b = p[1];
}

// Real rows of both roles of a plane.  In FP32 the roles run packed, one register pair per value:
// the two transforms share every twiddle, so one instruction serves both.
template <typename T, int N> struct Rows {
  T a[N], b[N];
  // a_z, b_z
  __device__ __forceinline__ C<T> at(int z) const { return mk<T>(a[z], b[z]); }
};
template <int N> struct Rows<float, N> {
  F2 v[N];
  __device__ __forceinline__ float2 at(int z) const { return unpack2(v[z]); }
};

// z transform of a row of both roles (row: role 0, row + N/2: role 1) with the z phases phz (null:
// none), x0 and xh the values (role 0, role 1) of modes 0 and N/2
template <int N>
__device__ __forceinline__ void rows_c2r(const float2* row, const float2* phz, float2 x0, float2 xh, Rows<float, N>& y) {
  constexpr int h = N / 2;
  C2 x[h];
  float2 fa[2], fb[2];
#pragma unroll
  for (int k = 1; k < h; ++k) {
    float2 a = row[k], b = row[h + k];
    if (phz != nullptr) {
      if constexpr (h % 2 == 0) {  // the phases two at a time (every block starts on 16 bytes)
        if (k == 1 || k % 2 == 0) {
          load_two(phz + (k & ~1), fa[0], fa[1]);
          load_two(phz + h + (k & ~1), fb[0], fb[1]);
        }
        a = cmul<float>(a, fa[k & 1]);
        b = cmul<float>(b, fb[k & 1]);
      } else {
        a = cmul<float>(a, phz[k]);
        b = cmul<float>(b, phz[h + k]);
      }
    }
    x[k].x = pack2(a.x, b.x);
    x[k].y = pack2(a.y, b.y);
  }
  c2r_line<F2, N>(x, pack2(x0.x, x0.y), pack2(xh.x, xh.y), y.v);
}
template <int N>
__device__ __forceinline__ void rows_c2r(const double2* row, const double2* phz, double2 x0, double2 xh,
                                         Rows<double, N>& y) {
  constexpr int h = N / 2;
  // a shift of zero along z leaves role 0 as it is and scales role 1 by its weight (bound by the FP64
  // pipe: half the multiplications of those rows)
  const bool plain = phz == nullptr || (phz[0].y == 0.0 && phz[h].y == 0.0);
  double2 x[h];
  if (plain) {
#pragma unroll
    for (int k = 1; k < h; ++k) x[k] = row[k];
  } else {
#pragma unroll
    for (int k = 1; k < h; ++k) x[k] = cmul<double>(row[k], phz[k]);
  }
  c2r_line<double, N>(x, x0.x, xh.x, y.a);
  if (plain) {
    const double w = phz != nullptr ? phz[h].x : 1.0;
#pragma unroll
    for (int k = 1; k < h; ++k) x[k] = scale<double>(row[h + k], w);
  } else {
#pragma unroll
    for (int k = 1; k < h; ++k) x[k] = cmul<double>(row[h + k], phz[h + k]);
  }
  c2r_line<double, N>(x, x0.y, xh.y, y.b);
}

// the last z pass of a row (gain in row, loss in row + N/2): out[z] = gain - f loss
template <int N>
__device__ __forceinline__ void dd_finish_row(const float2* row, const float* f, float (&out)[N]) {
  constexpr int h = N / 2;
  CDD<F2> x[h];
  DD<F2> y[N];
#pragma unroll
  for (int k = 1; k < h; ++k) x[k] = dd_of(pack2(row[k].x, row[h + k].x), pack2(row[k].y, row[h + k].y));
  const float2 g0 = row[0], l0 = row[h];
  c2r_line<DD<F2>, N>(x, dd_of(pack2(g0.x, l0.x)), dd_of(pack2(g0.y, l0.y)), y);
#pragma unroll
  for (int z = 0; z < N; ++z) {
    const float2 hi = unpack2(y[z].hi), lo = unpack2(y[z].lo);
    const float fz = __ldg(f + z);
    out[z] = fmaf(-fz, hi.y, hi.x) + fmaf(-fz, lo.y, lo.x);
  }
}

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// (s u + t w) + m in both halves
__device__ __forceinline__ float2 face_sum(float s, float2 u, float t, float2 w, float2 m) {
  return unpack2(fma2(pack2(s, s), pack2(u.x, u.y), fma2(pack2(t, t), pack2(w.x, w.y), pack2(m.x, m.y))));
}
__device__ __forceinline__ double2 face_sum(double s, double2 u, double t, double2 w, double2 m) {
  return make_double2(fma(s, u.x, fma(t, w.x, m.x)), fma(s, u.y, fma(t, w.y, m.y)));
}
__device__ __forceinline__ float2 mul_each(float2 s, float2 v) { return unpack2(pack2(s.x, s.y) * pack2(v.x, v.y)); }
__device__ __forceinline__ double2 mul_each(double2 s, double2 v) { return make_double2(s.x * v.x, s.y * v.y); }

// Gain of one mode: Q_hat (+)= F P_hat.  A work item split over its radial nodes adds them up later
// with these operations in the same order, so it gives the same bits.
template <typename T>
__device__ __forceinline__ C<T> add_gain(C<T> acc, T f, C<T> v, bool first) {
  return first ? scale<T>(v, f) : mk<T>(fma_(v.x, f, acc.x), fma_(v.y, f, acc.y));
}
// a mode of two real pencils held as one, p_0 + i p_h with weights fa, fh: v its value, m that of -k_x
template <typename T>
__device__ __forceinline__ C<T> add_gain_pair(C<T> acc, T fa, T fh, C<T> v, C<T> m, bool first) {
  const T fp = T(0.5) * (fa + fh), fm = T(0.5) * (fa - fh);
  const C<T> w = mk<T>(fma_(fm, m.x, fp * v.x), fma_(-fm, m.y, fp * v.y));
  return first ? w : add<T>(w, acc);
}

// n consecutive TMEM columns of the thread's lane (n a multiple of 8; every thread of the warp takes
// part).  A load waits for its data inside its asm statement; a store is waited for at once, since the
// next access of these columns may come soon.
template <int n>
__device__ __forceinline__ void tm_load(uint32_t ta, float* v) {
  if constexpr (n >= 32) {
    tc::tmem_ld32w(ta, v);
    if constexpr (n > 32) tm_load<n - 32>(ta + 32, v + 32);
  } else if constexpr (n >= 16) {
    tc::tmem_ld16w(ta, v);
    if constexpr (n > 16) tm_load<n - 16>(ta + 16, v + 16);
  } else {
    tc::tmem_ld8w(ta, v);
  }
}
template <int n>
__device__ __forceinline__ void tm_store_part(uint32_t ta, const float* v) {
  if constexpr (n >= 16) {
    tc::tmem_st16p(ta, v);
    if constexpr (n > 16) tm_store_part<n - 16>(ta + 16, v + 16);
  } else {
    tc::tmem_st8(ta, v);
  }
}
template <int n>
__device__ __forceinline__ void tm_store(uint32_t ta, const float* v) {
  tm_store_part<n>(ta, v);
  tc::tmem_wait_st();
}

// Step C of one VSS entry: x pass of its complex product spectrum P_hat and Q_hat += F P_hat.  Only the
// real part of IDFT(Q_hat) is wanted, that is Herm(Q_hat)(k) = (Q_hat(k) + conj Q_hat(-k)) / 2, so the half
// space k_z = 0..N/2 is enough.  F(-k) = conj F(k) except where k has an unpaired mode N/2: a pencil
// (k_y, k_z) off those faces needs Herm(P_hat) alone, adds its partner (-k_y, -k_z) before the transform,
// and weights only its element k_x = N/2 apart (two alternating sums over x).  The pencils with k_y or
// k_z = N/2 keep Q_hat itself, partner included, until the finish.
template <typename T, int N, int W>
__device__ __forceinline__ void vss_step_c(const KernelParams& p, const TaskDesc& tk, int q, int e, bool first,
                                           const C<T>* PV, C<T>* QA, C<T>* QB, int plane0, int tid) {
  using G = VGeo<T, N, W>;
  using CT = C<T>;
  constexpr int h = G::h, N2 = G::N2, QS = G::QROW, HP = h + 1;
  const int c0 = p.ent_m[2 * (tk.ent_off + e)], c1 = p.ent_m[2 * (tk.ent_off + e) + 1];
  const bool self_sum = tk.i == tk.j && c1 >= 0;
  const int own = G::PLANES * HP;
  const int all = own + (plane0 <= h && h < plane0 + G::PLANES ? h - 1 : 0);
  for (int u = tid; u < all; u += G::THREADS) {
    const int r = u < own ? plane0 + u / HP : h, kz = u < own ? u % HP : HP + u - own;
    const int at = u < own ? r * HP + kz : N * HP + u - own;
    const int rm = r == 0 ? 0 : N - r, km = kz == 0 ? 0 : N - kz;
    const bool inner = kz < h && r != h;
    const CT* const pv = PV + r * N + kz;
    const CT* const pm = PV + rm * N + km;
    CT v[N];
    CT av = mk<T>(0, 0), am = mk<T>(0, 0);
    if (inner) {
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const CT a = ld2<T>(pv + n * N2), m = ld2<T>(pm + n * N2);
        const T s = (n & 1) ? T(-1) : T(1);
        av = mk<T>(fma_(s, a.x, av.x), fma_(s, a.y, av.y));
        am = mk<T>(fma_(s, m.x, am.x), fma_(s, m.y, am.y));
        v[n] = mk<T>(T(0.5) * (a.x + m.x), T(0.5) * (a.y - m.y));
      }
    } else {
#pragma unroll
      for (int n = 0; n < N; ++n) v[n] = ld2<T>(pv + n * N2);
    }
    line_fft<T, N, -1>(v);
    for (int o = 0; o < 2; ++o) {
      const int pair = o == 0 ? tk.out0 : tk.out1;
      if (pair < 0) break;
      // the slot of the output's direction, conjugated where it holds the antipode's weight; a halved
      // self pair takes F(sigma) + F(-sigma) (FP32 tables hold the sum)
      const int code = o == 0 ? c0 : c1;
      const CT* const F = static_cast<const CT*>(p.Fv) + ((size_t(pair) * p.n_rho + q) * p.n_fslot + (code >> 1)) * G::N3;
      auto weight = [&](int n, int row, int col) {
        const CT f = __ldg(F + n * N2 + row * N + col);
        if (sizeof(T) == 8 && self_sum) return mk<T>(f.x + f.x, T(0));
        return mk<T>(f.x, (code & 1) ? -f.y : f.y);
      };
      CT* const acc = (o == 0 ? QA : QB) + at;
      // Bound by the latency of these loads.  VU weights and accumulators are loaded before the first is
      // used: one at a time 37 three-species nodes of N = 48 took 163 ms against 147, FP64 16 nodes 1975
      // against 1915 (VU = 4 152 ms, 12 to 24 146 to 147).
      constexpr int VU = N % 8 == 0 ? 8 : N % 6 == 0 ? 6 : 4;
#pragma unroll
      for (int n0 = 0; n0 < N; n0 += VU) {
        CT f[VU], old[VU];
#pragma unroll
        for (int d = 0; d < VU; ++d) f[d] = weight(n0 + d, r, kz);
#pragma unroll
        for (int d = 0; d < VU; ++d) old[d] = first ? mk<T>(0, 0) : ld2<T>(acc + (n0 + d) * QS);
#pragma unroll
        for (int d = 0; d < VU; ++d) {
          const int n = n0 + d;
          CT val = cmul<T>(v[n], f[d]);
          if (n == h && inner) {
            const CT x = cmul<T>(f[d], av), z = cmul<T>(weight(h, rm, km), am);
            val = mk<T>(T(0.5) * (x.x + z.x), T(0.5) * (x.y - z.y));
          }
          if (!first) val = add<T>(val, old[d]);
          st2<T>(acc + n * QS, val);
        }
      }
    }
  }
}

// VSS: total += part (or its copy), both accumulators, this CTA's pencils.  A radial sum is the sum, in
// order, of the sums of at most kVssParts parts of the radial nodes, whether one cluster runs them all or
// several run some each: a node's bits do not depend on how its item was split.  (Out of line, so that its
// pointers and loads cost the inner loops no registers.)
template <typename T, int N, int W>
__device__ __noinline__ void vss_add_part(C<T>* total, const C<T>* part, bool copy, bool both, int plane0, int tid) {
  using G = VGeo<T, N, W>;
  constexpr int HP = G::h + 1, own = G::PLANES * HP;
  const int all = own + (plane0 <= G::h && G::h < plane0 + G::PLANES ? G::h - 1 : 0);
  for (int o = 0; o < (both ? 2 : 1); ++o) {
#pragma unroll 4
    for (int v0 = tid; v0 < N * all; v0 += G::THREADS) {
      const int n = v0 / all, u = v0 % all;
      const size_t at = size_t(o) * G::QN + n * G::QROW + (u < own ? plane0 * HP + u : N * HP + u - own);
      C<T> v = ld2<T>(part + at);
      if (!copy) v = add<T>(ld2<T>(total + at), v);
      st2<T>(total + at, v);
    }
  }
}

// Gain of a split work item from its stored products PT [rho][k_x][pencil], this CTA's pencils, QU radial
// nodes of loads in flight per thread.  It runs once per split item, but inside the kernel its pointers
// and loads cost the inner loops registers, so the batch shapes trade: N = 24 and 32 call it out of line
// with QU = 4 (45 nodes of N = 24 0.80 ms; inline 8: 0.81, but batches 36.6 -> 37.2 ms), N = 16 and 48
// inline it with QU = 2 (batches 16.3 and 35.6 ms; out of line 16.6 and 36.7).
template <typename T, int N, int W>
__device__ __forceinline__ void add_parts(const C<T>* PT, const T* Fp, C<T>* QA, C<T>* QB, int out0, int out1, int n_rho,
                                       int plane0, int tid) {
  using G = VGeo<T, N, W>;
  using CT = C<T>;
  constexpr int h = G::h, N2 = G::N2, HN2 = G::HN2, NT = G::THREADS;
  constexpr size_t N3 = G::N3, HN3 = G::HN3;
  // (bound by L2 latency: one cluster reads all products and weights of the item)
  constexpr int total = N * G::PLANES * h, QU = G::QU;
  const T* const F0 = Fp + size_t(out0) * n_rho * N3;
  const T* const F1 = Fp + size_t(out1 >= 0 ? out1 : out0) * n_rho * N3;
#pragma unroll 1
  for (int u = tid; u < total; u += NT) {
    const int n = u / (G::PLANES * h), pp = plane0 * h + u % (G::PLANES * h);
    const int r = pp / h, cc = pp % h;
    if (cc == 0 && (r == 0 || r == h)) continue;  // the pencils that hold two real ones, below
    const int at = n * HN2 + pp;
    const int fo = n * N2 + (cc == 0 && r >= h ? (r - h) * N + h : r * N + cc);
    CT a0 = mk<T>(0, 0), a1 = mk<T>(0, 0);
#pragma unroll 1
    for (int q = 0; q < n_rho; q += QU) {
      CT v[QU];
      T wa[QU], wb[QU];
#pragma unroll
      for (int j = 0; j < QU; ++j)
        if (q + j < n_rho) {
          v[j] = ld2<T>(PT + (q + j) * HN3 + at);
          wa[j] = __ldg(F0 + (q + j) * N3 + fo);
          wb[j] = __ldg(F1 + (q + j) * N3 + fo);
        }
#pragma unroll
      for (int j = 0; j < QU; ++j)
        if (q + j < n_rho) {
          a0 = add_gain<T>(a0, wa[j], v[j], q + j == 0);
          a1 = add_gain<T>(a1, wb[j], v[j], q + j == 0);
        }
    }
    st2<T>(QA + at, a0);
    if (out1 >= 0) st2<T>(QB + at, a1);
  }
  for (int u = tid; u < 2 * N; u += NT) {  // the pencils (0, 0) and (N/2, 0)
    const int n = u >> 1, pp = (u & 1) * h * h;
    if (pp / h < plane0 || pp / h >= plane0 + G::PLANES) continue;
    const CT* const pv = PT + n * HN2 + pp;
    const CT* const pm = PT + (n == 0 ? 0 : N - n) * HN2 + pp;
    for (int o = 0; o < 2; ++o) {
      const int pair = o == 0 ? out0 : out1;
      if (pair < 0) break;
      const T* const Fw = Fp + size_t(pair) * n_rho * N3 + n * N2 + (u & 1) * h;
      CT acc = mk<T>(0, 0);
#pragma unroll 4
      for (int q = 0; q < n_rho; ++q)
        acc = add_gain_pair<T>(acc, __ldg(Fw + q * N3), __ldg(Fw + q * N3 + h * N), ld2<T>(pv + q * HN3),
                               ld2<T>(pm + q * HN3), q == 0);
      st2<T>((o == 0 ? QA : QB) + n * HN2 + pp, acc);
    }
  }
}

template <typename T, int N, int W>
__device__ __noinline__ void add_parts_call(const C<T>* PT, const T* Fp, C<T>* QA, C<T>* QB, int out0, int out1, int n_rho,
                                            int plane0, int tid) {
  add_parts<T, N, W>(PT, Fp, QA, QB, out0, out1, n_rho, plane0, tid);
}

template <typename T, int N, int W>
__global__ void __launch_bounds__(VGeo<T, N, W>::THREADS, VGeo<T, N, W>::MINB) collision_kernel(const KernelParams p) {
  using G = VGeo<T, N, W>;
  using CT = C<T>;
  constexpr int h = G::h, N2 = G::N2, HN2 = G::HN2, CL = G::CL, GP = G::GP, NT = G::THREADS, PITCH = G::PITCH;
  constexpr int PB = G::PB;
  constexpr size_t N3 = G::N3, HN3 = G::HN3;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x;
  const int grp = tid / N;  // plane group
  const int t = tid % N;    // line within the group: column (role, c) in y passes, row in z passes
  const int role = t / h, c = t % h;
  unsigned char* const gsm = smem_raw + size_t(grp) * G::GROUP_BYTES;
  CT* const tb = reinterpret_cast<CT*>(gsm);  // padded plane; the pad column of rows 0, 1 carries a corner value
  CT* const uyb = tb + N * PITCH;             // the entry's row of the k_y face
  T* const pb = reinterpret_cast<T*>(uyb + N);
  CT* const phs = reinterpret_cast<CT*>(smem_raw + G::SMEM);  // phase block of the current (task, rho)
  const bool ph_smem = p.phase_smem != 0;

  // TMEM: warp 0 allocates the CTA's columns; warp w reaches lanes 32 (w % 4) .. + 31
  __shared__ uint32_t s_tmem;
  uint32_t tm_raw = 0, tm_p = 0;
  if constexpr (G::TM_ALLOC > 0) {
    if (tid < 32) {
      tc::tmem_alloc(&s_tmem, G::TM_ALLOC);
      tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    tm_raw = s_tmem + (uint32_t(32 * ((tid / 32) & 3)) << 16) + uint32_t((tid / 128) * G::TM_SET);
    tm_p = tm_raw + (G::TMR ? 2 * N : 0);
  }

  const int rank = CL == 1 ? 0 : int(cluster_rank());
  const int cid = blockIdx.x / CL;
  CT* const scr = reinterpret_cast<CT*>(p.scratch) + size_t(cid) * p.slot;
  CT* const FS = scr;               // f_hat [k_x][k_y][species 0 | 1][c]
  CT* const H0 = FS + N3;           // x-passed half spectra [x][k_y][role][c], NBH buffers
  CT* const HZ = H0 + G::NBH * N3;  // the same for the group with sigma_x = 0, kept for all radial nodes
  CT* const PV = HZ + N3;       // product spectrum [x][row][c] (N form)
  CT* const QA = PV + G::PVN;          // gain accumulators [k_x][row][c] (N form)
  CT* const QB = QA + G::QN;
  T* const PS = reinterpret_cast<T*>(QB + HN3);  // parked P [x][z][y]
  CT* const FC = scr + G::SLOT;     // faces per entry: X [z][y], Y [x][z], line [y]; values (role 0, role 1)
  const int plane0 = rank * G::PLANES;
  const T inv_n3 = T(1) / T(N3);

  // Work items (task, node, chunk of radial nodes) come from a counter: thread 0 of the rank-0 CTA
  // takes the next item after the first barrier of the current one, when every CTA has read the
  // current value.  Tasks are in order of falling cost, so the last items are the short ones.
  __shared__ int s_next_item;
  __shared__ int s_last;
  const int n_items = p.batch * p.n_tasks * p.chunks;
  if (rank == 0 && tid == 0) s_next_item = int(atomicAdd(p.work_counter, 1u));
  cluster_sync<CL>();
  for (int item = CL == 1 ? s_next_item : ld_rank0(&s_next_item); item < n_items;
       item = CL == 1 ? s_next_item : ld_rank0(&s_next_item)) {
    const int chunk = item % p.chunks;
    const int whole = item / p.chunks;
    const int b = whole % p.batch;
    const int task = whole / p.batch;
    const bool split = p.chunks > 1;
    // VSS: the chunk is a range of the plan's parts of the radial nodes
    const int n_part = G::VSS ? vss_parts(p.n_rho) : p.chunks;
    int part = G::VSS ? chunk * n_part / p.chunks : chunk;
    const int part_end = G::VSS ? (chunk + 1) * n_part / p.chunks : chunk + 1;
    const int q0 = part * p.n_rho / n_part, q1 = part_end * p.n_rho / n_part;
    int part_q0 = q0;
    // split items: P_hat of every radial node; VSS: both accumulators of every part
    CT* const PT = static_cast<CT*>(p.parts) + (G::VSS ? size_t(whole) * n_part * 2 * G::QN : size_t(whole) * p.n_rho * HN3);
    const TaskDesc tk = p.tasks[task];
    const T* fb = reinterpret_cast<const T*>(p.f) + size_t(b) * p.s * N3;
    const bool self = tk.i == tk.j;

    // ---- step 0: f_hat = N^-3 DFT(f) of species i (and j), half spectra in C form -----------
    for (int xl = grp; xl < G::PLANES; xl += GP) {
      const int x = plane0 + xl;
      for (int sp = 0; sp < (self ? 1 : 2); ++sp) {
        const T* src = fb + size_t(sp == 0 ? tk.i : tk.j) * N3 + size_t(x) * N2 + t * N;
        T y[N];
        CT z[h];
#pragma unroll
        for (int n = 0; n < N; ++n) y[n] = __ldg(src + n);
        r2c_line<T, N>(y, z);
#pragma unroll
        for (int k = 0; k < h; ++k) tb[t * PITCH + sp * h + k] = z[k];
      }
      group_sync<N, GP>();
      if (!self || role == 0) {
        CT v[N];
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = tb[r * PITCH + t];
        line_fft<T, N, -1>(v);
#pragma unroll
        for (int r = 0; r < N; ++r) st2<T>(FS + size_t(x) * N2 + r * N + t, v[r]);
        // without a shift along x the x passes there and back cancel
        if (tk.any_zero) {
#pragma unroll
          for (int r = 0; r < N; ++r) st2<T>(HZ + size_t(x) * N2 + r * N + t, scale<T>(v[r], T(1) / T(N2)));
        }
      }
      group_sync<N, GP>();
    }
    cluster_sync<CL>();
    if (rank == 0 && tid == 0) s_next_item = int(atomicAdd(p.work_counter, 1u));
    if (!self || role == 0) {
      for (int xl = grp; xl < G::PLANES; xl += GP) {
        CT* const vol = FS + (plane0 + xl) * N + t;
        CT v[N];
#pragma unroll
        for (int n = 0; n < N; ++n) v[n] = ld2<T>(vol + n * N2);
        line_fft<T, N, -1>(v);
#pragma unroll
        for (int n = 0; n < N; ++n) st2<T>(vol + n * N2, scale<T>(v[n], inv_n3));
      }
    }
    cluster_sync<CL>();
    const CT* const Fr = FS + (self ? c : t);     // this thread's column of f_hat
    const CT fe = ld2<T>(Fr + h * N2 + h * N);    // its value on the edge k_x = k_y = N/2

    // ---- gain ---------------------------------------------------------------------------------
    T P[G::PSM || G::VSS ? 1 : N];
    auto part_acc = [&]() { return split ? PT + size_t(part) * 2 * G::QN : QB + G::QN; };
    for (int q = q0; q < q1; ++q) {
      const CT* const phq = static_cast<const CT*>(p.phase) + (size_t(task) * p.n_rho + q) * p.max_ent * PB;
      if (ph_smem) {
        for (int u = tid; u < tk.n_ent * PB; u += NT) phs[u] = __ldg(phq + u);
        __syncthreads();
      }
      const CT* const phb = ph_smem ? phs : phq;

      // faces of the entries whose shift along the face's axis is not zero, spread over the
      // cluster's CTAs first; code 2 e + kind.  kind 0: k_x = N/2 (y and z shifted), kind 1:
      // k_y = N/2 (x and z shifted)
      for (int f0 = 0; f0 < tk.n_face; f0 += CL * GP) {
        // groups that share a barrier run the same number of rounds: one without a face of its own
        // repeats the last and stores nothing
        const int f = f0 + grp * CL + rank;
        const bool live = f < tk.n_face;
        if (N % 32 == 0 && !live) break;
        const int code = p.faces[tk.face_off + (live ? f : tk.n_face - 1)];
        const int e = code >> 1, kind = code & 1;
        const CT* const pe = phb + e * PB;
        CT* const fc = FC + size_t(e) * G::FACE;
        {
          const CT* const src = Fr + (kind == 0 ? h * N2 : h * N);
          const int step = kind == 0 ? N : N2;
          CT v[N];
#pragma unroll
          for (int r = 0; r < N; ++r) v[r] = ld2<T>(src + r * step);
          shift_line<T, N>(v, pe + (kind == 0 ? N : 0) + role);
          line_fft<T, N, +1>(v);
          group_sync<N, GP>();
#pragma unroll
          for (int r = 0; r < N; ++r) tb[r * PITCH + t] = v[r];
          group_sync<N, GP>();
        }
        const CT* const row = tb + t * PITCH;
        const CT cta = pe[2 * N], ctb = pe[2 * N + h];
        const CT a0 = row[0], b0 = row[h];
        Rows<T, N> y;
        rows_c2r<N>(row, pe + 2 * N, mk<T>(a0.x, pe[3 * N].x * b0.x), mk<T>(cta.x * a0.y, ctb.x * b0.y), y);
        const CT sc = mk<T>(pe[kind == 0 ? 0 : N].y, pe[kind == 0 ? 1 : N + 1].y);
        if (!live) {
        } else if (kind == 0) {
#pragma unroll
          for (int z = 0; z < N; ++z) st2<T>(fc + z * N + t, mul_each(sc, y.at(z)));
          st2<T>(fc + 2 * N2 + t, mk<T>(sc.x * a0.y, sc.y * b0.y));
        } else {
#pragma unroll
          for (int z = 0; z < N; ++z) st2<T>(fc + N2 + t * N + z, mul_each(sc, y.at(z)));
        }
      }

      for (int k = 0; k <= tk.n_grp + (G::VSS ? 1 : 0); ++k) {
        // step A of group k: x pass of this thread's pencils with the group's x phases
        if (k < tk.n_grp && !p.groups[tk.grp_off + k].zero) {
          const GroupDesc gd = p.groups[tk.grp_off + k];
          CT* const dst = H0 + size_t(k % G::NBH) * N3;
          const CT* const phx = phb + gd.first * PB + role;
          for (int xl = grp; xl < G::PLANES; xl += GP) {
            const int r = plane0 + xl;
            CT v[N];
#pragma unroll
            for (int n = 0; n < N; ++n) v[n] = ld2<T>(Fr + n * N2 + r * N);
            shift_line<T, N>(v, phx);
            line_fft<T, N, +1>(v);
#pragma unroll
            for (int n = 0; n < N; ++n) st2<T>(dst + n * N2 + r * N + t, v[n]);
          }
        }
        // split barrier: step B of group k - 1 covers the other CTAs' lag in step A of group k
        const bool halves = G::SPLIT && k > 0 && k < tk.n_grp;
        if (halves) cluster_arrive();
        // step B of group k - 1: this group's planes
        if (k > 0 && k <= tk.n_grp) {
          const GroupDesc gd = p.groups[tk.grp_off + k - 1];
          const bool zero = gd.zero != 0;
          const CT* const src = zero ? HZ : H0 + size_t((k - 1) % G::NBH) * N3;
          const int col = zero && self ? c : t;  // (a self pair's roles share the unshifted columns)
          const bool fresh = k == 1, last = k == tk.n_grp;
          for (int xl = grp; xl < G::PLANES; xl += GP) {
            const int x = plane0 + xl;
            if constexpr (G::PF) {
              if (t == 0 && xl + GP < G::PLANES) prefetch_l2(src + size_t(x + GP) * N2, N2 * sizeof(CT));
            }
            const T sgx = (x & 1) ? T(-1) : T(1), sgy = (t & 1) ? T(-1) : T(1);
            if constexpr (G::VSS) {
              // no sum over the entries
            } else if constexpr (G::PSM) {
              if (fresh || !G::KEEP) {
#pragma unroll
                for (int z = 0; z < N; ++z) pb[z * N + t] = fresh ? T(0) : __ldcg(PS + size_t(x) * N2 + z * N + t);
              }
            } else {
              if (fresh) {
#pragma unroll
                for (int z = 0; z < N; ++z) P[z] = T(0);
              } else if constexpr (G::TMP) {
                __syncwarp();
                tm_load<N>(tm_p + uint32_t((xl / GP) * N), reinterpret_cast<float*>(P));
              } else if constexpr (!G::KEEP) {
#pragma unroll
                for (int z = 0; z < N; ++z) P[z] = __ldcg(PS + size_t(x) * N2 + z * N + t);
              }
            }
            for (int e = gd.first; e < gd.first + gd.count; ++e) {
              const CT* const pe = phb + e * PB;
              const CT* const fc = FC + size_t(e) * G::FACE;
              // a shift of zero along an axis has no face there
              const T txa = pe[0].y, txb = pe[1].y, tya = pe[N].y, tyb = pe[N + 1].y;
              const bool has_x = has_face<T>(pe), has_y = tya != T(0) || tyb != T(0);
              const CT uy = has_y ? __ldca(fc + N2 + x * N + t) : mk<T>(0, 0);
              const CT en = has_x ? __ldca(fc + 2 * N2 + t) : mk<T>(0, 0);
              {
                CT v[N];
                if (!G::TMR || e == gd.first) {
#pragma unroll
                  for (int r = 0; r < N; ++r) v[r] = ld2<T>(src + size_t(x) * N2 + r * N + col);
                  if constexpr (G::TMR) {
                    if (gd.count > 1) {
                      __syncwarp();
                      tm_store<2 * N>(tm_raw, reinterpret_cast<const float*>(v));
                    }
                  }
                } else if constexpr (G::TMR) {
                  __syncwarp();
                  tm_load<2 * N>(tm_raw, reinterpret_cast<float*>(v));
                }
                const T corner = v[h].y;  // of column 0: f on the edge k_y = k_z = N/2
                // (a shift of zero has phase 1 throughout; measured: skipping it N = 32 -2.3 %, FP64 N = 32 -1 %,
                // N = 16, 24, 48 +0.7 to 3 %)
                if (!(sizeof(T) == 8 || N == 32) || has_y) shift_line<T, N>(v, pe + N + role);
                const T w = sgx * (role == 0 ? txa * tya : txb * tyb);
                v[h] = mk<T>(v[h].x - w * fe.x, v[h].y - w * fe.y);
                line_fft<T, N, +1>(v);
                group_sync<N, GP>();  // the previous entry's rows have been read
#pragma unroll
                for (int r = 0; r < N; ++r) tb[r * PITCH + t] = v[r];
                uyb[t] = uy;
                if (c == 0) tb[role * PITCH + N] = mk<T>(corner, T(0));
                group_sync<N, GP>();
              }
              const CT* const row = tb + t * PITCH;
              const CT cta = pe[2 * N], ctb = pe[2 * N + h];
              const CT a0 = row[0], b0 = row[h];
              const CT m = mk<T>(cta.y * a0.y, ctb.y * b0.y);
              Rows<T, N> y;
              rows_c2r<N>(row, pe + 2 * N, mk<T>(a0.x, pe[3 * N].x * b0.x),
                          mk<T>(cta.x * a0.y - cta.y * (sgx * en.x + sgy * tya * tb[N].x),
                                ctb.x * b0.y - ctb.y * (sgx * en.y + sgy * tyb * tb[PITCH + N].x)),
                          y);
              if constexpr (G::VSS) {
                // the product is complex; forward z and y transforms, all N columns
                CT pr[N];
#pragma unroll
                for (int z = 0; z < N; z += 2) {
                  CT uz[2];
                  load_two(uyb + z, uz[0], uz[1]);
#pragma unroll
                  for (int d = 0; d < 2; ++d) {
                    // read by every plane of the CTA: through L1
                    const CT ux = has_x ? __ldca(fc + (z + d) * N + t) : mk<T>(0, 0);
                    const CT im = face_sum(sgx, ux, sgy, uz[d], d ? mk<T>(-m.x, -m.y) : m);
                    const CT re = y.at(z + d);
                    pr[z + d] = mk<T>(fma_(-im.x, im.y, re.x * re.y), fma_(re.x, im.y, im.x * re.y));
                  }
                }
                line_fft<T, N, -1>(pr);
                group_sync<N, GP>();
#pragma unroll
                for (int z = 0; z < N; ++z) tb[t * PITCH + z] = pr[z];
                group_sync<N, GP>();
#pragma unroll
                for (int r = 0; r < N; ++r) pr[r] = tb[r * PITCH + t];
                line_fft<T, N, -1>(pr);
                CT* const dst = PV + size_t(2 * ((k - 1) & 1) + e - gd.first) * N3 + size_t(x) * N2 + t;
#pragma unroll
                for (int r = 0; r < N; ++r) st2<T>(dst + r * N, pr[r]);
              } else {
#pragma unroll
                for (int z = 0; z < N; z += 2) {
                  CT uz[2];
                  load_two(uyb + z, uz[0], uz[1]);
#pragma unroll
                  for (int d = 0; d < 2; ++d) {
                    // read by every plane of the CTA: through L1
                    const CT ux = has_x ? __ldca(fc + (z + d) * N + t) : mk<T>(0, 0);
                    const CT im = face_sum(sgx, ux, sgy, uz[d], d ? mk<T>(-m.x, -m.y) : m);
                    const CT re = y.at(z + d);
                    if constexpr (G::PSM) pb[(z + d) * N + t] = fma_(-im.x, im.y, fma_(re.x, re.y, pb[(z + d) * N + t]));
                    else P[z + d] = fma_(-im.x, im.y, fma_(re.x, re.y, P[z + d]));
                  }
                }
              }
            }
            if constexpr (G::VSS) {
              // done entry by entry
            } else if (last) {
              group_sync<N, GP>();
              {
                CT z[h];
                T y[N];
#pragma unroll
                for (int n = 0; n < N; ++n) {
                  if constexpr (G::PSM) y[n] = pb[n * N + t]; else y[n] = P[n];
                }
                r2c_line<T, N>(y, z);
#pragma unroll
                for (int kz = 0; kz < h; ++kz) tb[t * PITCH + kz] = z[kz];
              }
              group_sync<N, GP>();
              if (role == 0) {
                CT v[N];
#pragma unroll
                for (int r = 0; r < N; ++r) v[r] = tb[r * PITCH + t];
                line_fft<T, N, -1>(v);
                CT* const dst = PV + size_t(x) * HN2 + c;
                if (c != 0) {
#pragma unroll
                  for (int r = 0; r < N; ++r) st2<T>(dst + r * h, v[r]);
                } else {  // C form -> N form
                  st2<T>(dst, mk<T>(v[0].x, v[h].x));
                  st2<T>(dst + h * h, mk<T>(v[0].y, v[h].y));
#pragma unroll
                  for (int r = 1; r < h; ++r) {
                    const CT m = conj_<T>(v[N - r]);
                    const CT d = sub<T>(v[r], m);
                    st2<T>(dst + r * h, scale<T>(add<T>(v[r], m), T(0.5)));
                    st2<T>(dst + (h + r) * h, mk<T>(T(0.5) * d.y, T(-0.5) * d.x));
                  }
                }
              }
            } else if constexpr (G::TMP) {
              __syncwarp();
              tm_store<N>(tm_p + uint32_t((xl / GP) * N), reinterpret_cast<const float*>(P));
            } else if constexpr (!G::KEEP) {
#pragma unroll
              for (int z = 0; z < N; ++z) {
                T val;
                if constexpr (G::PSM) val = pb[z * N + t]; else val = P[z];
                __stcg(PS + size_t(x) * N2 + z * N + t, val);
              }
            }
          }
        }
        if constexpr (G::VSS) {
          if (k >= 2) {
            const GroupDesc gd = p.groups[tk.grp_off + k - 2];
            for (int j = 0; j < gd.count; ++j)
              vss_step_c<T, N, W>(p, tk, q, gd.first + j, q == part_q0 && gd.first + j == 0,
                                  PV + size_t(2 * (k & 1) + j) * N3, part_acc(), part_acc() + G::QN, plane0, tid);
          }
        }
        if (halves) cluster_wait(); else cluster_sync<CL>();
      }
      if constexpr (G::VSS) {
        if (q + 1 == (part + 1) * p.n_rho / n_part) {  // the part's last
          if (!split) vss_add_part<T, N, W>(QA, part_acc(), part == 0, tk.out1 >= 0, plane0, tid);
          ++part;
          part_q0 = q + 1;
        }
        continue;
      }

      // step C: x pass of the product spectrum, weights, accumulation
      for (int u = tid; u < G::PLANES * h; u += NT) {
        const int r = plane0 + u / h, cc = u % h;
        const size_t pp = size_t(r) * h + cc;
        CT v[N];
#pragma unroll
        for (int n = 0; n < N; ++n) v[n] = ld2<T>(PV + n * HN2 + pp);
        line_fft<T, N, -1>(v);
        // modes of the pencil (N form): column 0 holds k_z = 0 in rows 1..N/2-1 and k_z = N/2 above
        // them; rows 0 and N/2 hold two real pencils, k_y = 0 and N/2, as one
        const bool pair_row = cc == 0 && (r == 0 || r == h);
        const int ky = cc == 0 && r >= h ? r - h : r;
        const int kz = cc == 0 && r >= h ? h : cc;
        if (split) {
#pragma unroll
          for (int n = 0; n < N; ++n) st2<T>(PT + q * HN3 + n * HN2 + pp, v[n]);
          continue;
        }
        for (int o = 0; o < 2; ++o) {
          const int pair = o == 0 ? tk.out0 : tk.out1;
          if (pair < 0) break;
          const T* const Fw = static_cast<const T*>(p.Fw) + (size_t(pair) * p.n_rho + q) * N3 + ky * N + kz;
          CT* const acc = (o == 0 ? QA : QB) + pp;
          if (!pair_row) {
#pragma unroll
            for (int n = 0; n < N; ++n) {
              const CT old = q > 0 ? ld2<T>(acc + n * HN2) : mk<T>(0, 0);
              st2<T>(acc + n * HN2, add_gain<T>(old, __ldg(Fw + n * N2), v[n], q == 0));
            }
          } else {
#pragma unroll
            for (int n = 0; n < N; ++n) {
              const CT old = q > 0 ? ld2<T>(acc + n * HN2) : mk<T>(0, 0);
              st2<T>(acc + n * HN2, add_gain_pair<T>(old, __ldg(Fw + n * N2), __ldg(Fw + n * N2 + h * N), v[n],
                                                     v[(N - n) % N], q == 0));
            }
          }
        }
      }
    }
    if (split) {
      // the cluster that stores the last of the item's products adds them up and finishes the item
      __threadfence();
      cluster_sync<CL>();
      if (rank == 0 && tid == 0) {
        unsigned* const done = p.work_counter + kDoneWord + whole;
        s_last = atomicAdd(done, 1u) + 1 == unsigned(p.chunks) ? 1 : 0;
        if (s_last) *done = 0;  // ready for the next launch
        __threadfence();
      }
      cluster_sync<CL>();
      if ((CL == 1 ? s_last : ld_rank0(&s_last)) == 0) {
        cluster_sync<CL>();  // s_last has been read
        continue;
      }
      __threadfence();
      if constexpr (G::VSS) {
        for (int j = 0; j < n_part; ++j)
          vss_add_part<T, N, W>(QA, PT + size_t(j) * 2 * G::QN, j == 0, tk.out1 >= 0, plane0, tid);
      } else if constexpr (G::CALL)
        add_parts_call<T, N, W>(PT, static_cast<const T*>(p.Fw), QA, QB, tk.out0, tk.out1, p.n_rho, plane0, tid);
      else
        add_parts<T, N, W>(PT, static_cast<const T*>(p.Fw), QA, QB, tk.out0, tk.out1, p.n_rho, plane0, tid);
    }
    if constexpr (G::VSS) cluster_sync<CL>(); else __syncthreads();

    // ---- finish: Q_ij = IDFT(Q_hat) - f_i IDFT(G^- f_hat_j); role 0 the gain, role 1 the loss ----
    for (int o = 0; o < 2; ++o) {
      const int pair = o == 0 ? tk.out0 : tk.out1;
      if (pair < 0) break;
      const int io = o == 0 ? tk.i : tk.j;
      const int jo = o == 0 ? tk.j : tk.i;
      const CT* const acc = o == 0 ? QA : QB;
      const CT* const Fj = FS + (jo == tk.i ? 0 : h);
      const T* const Gm = static_cast<const T*>(p.Gm) + size_t(pair) * N3;
      for (int xl = grp; xl < G::PLANES; xl += GP) {
        const int r = plane0 + xl;
        CT v[N];
        if (role == 0 && G::VSS) {  // the Hermitian part, in C form
          constexpr int HP = h + 1;
          auto at = [&](int n, int row, int kz) {
            return ld2<T>(acc + n * G::QROW + (kz <= h ? row * HP + kz : N * HP + kz - HP));
          };
          auto herm = [](CT a, CT m) { return mk<T>(T(0.5) * (a.x + m.x), T(0.5) * (a.y - m.y)); };
          const int rm = r == 0 ? 0 : N - r;
          for (int n = 0; n < N; ++n) {
            const int nm = n == 0 ? 0 : N - n;
            CT a = at(n, r, c);
            if (r == h) a = herm(a, at(nm, h, c == 0 ? 0 : N - c));
            if (c == 0) {
              const CT d = herm(at(n, r, h), at(nm, rm, h));
              a = mk<T>(a.x - d.y, a.y + d.x);
            }
            st2<T>(H0 + n * N2 + r * N + t, a);
          }
#pragma unroll
          for (int n = 0; n < N; ++n) v[n] = ld2<T>(H0 + n * N2 + r * N + t);
        } else if (role == 0) {
#pragma unroll
          for (int n = 0; n < N; ++n) v[n] = ld2<T>(acc + n * HN2 + r * h + c);
        } else if (c != 0) {
#pragma unroll
          for (int n = 0; n < N; ++n) v[n] = scale<T>(ld2<T>(Fj + n * N2 + r * N + c), __ldg(Gm + n * N2 + r * N + c));
        } else {  // C form: the two parts of column 0 have weights of their own
          const int rm = r == 0 ? 0 : N - r;
#pragma unroll
          for (int n = 0; n < N; ++n) {
            const T ga = __ldg(Gm + n * N2 + r * N), gh = __ldg(Gm + n * N2 + r * N + h);
            const T gp = T(0.5) * (ga + gh), gm = T(0.5) * (ga - gh);
            const CT a = ld2<T>(Fj + n * N2 + r * N), m = ld2<T>(Fj + ((N - n) % N) * N2 + rm * N);
            v[n] = mk<T>(gp * a.x + gm * m.x, gp * a.y - gm * m.y);
          }
        }
        if constexpr (G::FINE_X) dd_line_fft<N, +1>(v); else line_fft<T, N, +1>(v);
#pragma unroll
        for (int n = 0; n < N; ++n) st2<T>(H0 + n * N2 + r * N + t, v[n]);
      }
      cluster_sync<CL>();
      T* const Qout = reinterpret_cast<T*>(p.Q) + ((size_t(b) * p.s + io) * p.s + jo) * N3;
      const T* const fi = fb + size_t(io) * N3;
      for (int xl = grp; xl < G::PLANES; xl += GP) {
        const int x = plane0 + xl;
        const CT* const src = H0 + size_t(x) * N2;
        {
          CT v[N];
          if (t != 0 || G::VSS) {
#pragma unroll
            for (int r = 0; r < N; ++r) v[r] = ld2<T>(src + r * N + t);
          } else {  // N form -> C form
            const CT a = ld2<T>(src), d = ld2<T>(src + h * N);
            v[0] = mk<T>(a.x, d.x);
            v[h] = mk<T>(a.y, d.y);
#pragma unroll
            for (int r = 1; r < h; ++r) {
              const CT al = ld2<T>(src + r * N), be = ld2<T>(src + (h + r) * N);
              v[r] = mk<T>(al.x - be.y, al.y + be.x);
              v[N - r] = mk<T>(al.x + be.y, be.x - al.y);
            }
          }
          if constexpr (G::FINE_Y) dd_line_fft<N, +1>(v); else line_fft<T, N, +1>(v);
          group_sync<N, GP>();
#pragma unroll
          for (int r = 0; r < N; ++r) tb[r * PITCH + t] = v[r];
          group_sync<N, GP>();
        }
        // stage the row through shared memory for a coalesced store
        T* const rb = reinterpret_cast<T*>(tb);
        const T* const fr = fi + size_t(x) * N2 + t * N;
        if constexpr (G::FINE_Z) {
          T y[N];
          dd_finish_row<N>(tb + t * PITCH, fr, y);
          group_sync<N, GP>();
#pragma unroll
          for (int z = 0; z < N; ++z) rb[t * PITCH + z] = y[z];
        } else {
          const CT g0 = tb[t * PITCH], l0 = tb[t * PITCH + h];
          Rows<T, N> y;
          rows_c2r<N>(tb + t * PITCH, static_cast<const CT*>(nullptr), mk<T>(g0.x, l0.x), mk<T>(g0.y, l0.y), y);
          group_sync<N, GP>();
#pragma unroll
          for (int z = 0; z < N; ++z) {
            const CT gl = y.at(z);
            rb[t * PITCH + z] = gl.x - __ldg(fr + z) * gl.y;
          }
        }
        group_sync<N, GP>();
#pragma unroll
        for (int r = 0; r < N; ++r) Qout[size_t(x) * N2 + r * N + t] = rb[r * PITCH + t];
        group_sync<N, GP>();
      }
      cluster_sync<CL>();
    }
  }
  if constexpr (G::TM_ALLOC > 0) {
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid < 32) tc::tmem_dealloc(s_tmem, G::TM_ALLOC);
  }
  // no CTA leaves while another may still read its shared memory (the last item index)
  if constexpr (CL > 1) cluster_sync<CL>();
  // every cluster has taken its last item once all have come here: the last one readies the counter
  // for the next launch
  if (rank == 0 && tid == 0 && atomicAdd(p.work_counter + kExitWord, 1u) + 1 == gridDim.x / CL) {
    p.work_counter[0] = 0;
    p.work_counter[kExitWord] = 0;
  }
}

// dynamic shared memory of a shape: the plane buffers and, while MINB CTAs still fit, the phase block
// of the current (task, rho)
template <typename T, int N, int W>
size_t kernel_smem(const Plan& pl, KernelShape& s) {
  using G = VGeo<T, N, W>;
  const size_t limit = size_t(226) * 1024 / G::MINB - 2048;  // per CTA while MINB CTAs still fit
  const size_t ph_bytes = (size_t(pl.max_ent) * G::PB + 1) / 2 * 2 * sizeof(C<T>);
  s.phase_smem = G::SMEM + ph_bytes <= limit ? 1 : 0;
  const size_t used = G::SMEM + (s.phase_smem ? ph_bytes : 0);
  return used;
}

// raise a kernel's dynamic shared memory limit to `smem` (never lower it: plans of one shape share the
// kernel, and their phase blocks differ)
template <typename K>
bool allow_smem(K kern, size_t smem) {
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return false;
  if (fa.maxDynamicSharedSizeBytes >= int(smem)) return true;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) == cudaSuccess;
}

inline void launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cluster, int clusters, const KernelShape& s,
                       cudaStream_t st) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(clusters * cluster);
  cfg.blockDim = dim3(s.threads);
  cfg.dynamicSmemBytes = s.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

template <typename T, int N, int W>
int configure_shape(Plan& pl) {
  using G = VGeo<T, N, W>;
  auto kern = collision_kernel<T, N, W>;
  KernelShape& s = pl.shapes[W == 2 ? 0 : W];
  s.threads = G::THREADS;
  s.smem = kernel_smem<T, N, W>(pl, s);
  if (!allow_smem(kern, s.smem)) return DGFS_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  launch_config(cfg, attr, G::CL, 1, s, nullptr);
  if (cudaOccupancyMaxActiveClusters(&s.clusters, kern, &cfg) != cudaSuccess || s.clusters <= 0) {
    cudaGetLastError();
    return DGFS_ERR_CUDA;
  }
  if constexpr (G::TM_ALLOC > 0) {
    // The occupancy calculator grants a kernel that allocates tensor memory one CTA per SM; the
    // device co-schedules what registers, shared memory and threads allow.
    cudaFuncAttributes fa;
    int dev = 0, sms = 0;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return DGFS_ERR_CUDA;
    if (G::CL > 1) {
      // A CTA that waits for columns inside a cluster must not wait for another waiting cluster:
      // each CTA asks for at least its columns' share of the SM's shared memory, so whatever mix of
      // such kernels an SM holds, their columns fit.  (A kernel without clusters waits for nobody
      // once it has its columns.)
      const size_t least = (size_t(228) * 1024 * G::TM_ALLOC + 511) / 512 - 1024 - fa.sharedSizeBytes;
      if (s.smem < least) s.smem = least;
      if (!allow_smem(kern, s.smem)) return DGFS_ERR_CUDA;
    }
    const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;
    int most = 65536 / (regs_warp * ((G::THREADS + 31) / 32));
    const int by_smem = int(size_t(228) * 1024 / (s.smem + fa.sharedSizeBytes + 1024));
    if (by_smem < most) most = by_smem;
    if (2048 / G::THREADS < most) most = 2048 / G::THREADS;
    if (512 / G::TM_ALLOC < most) most = 512 / G::TM_ALLOC;
    if (most < 1) return DGFS_ERR_CUDA;
    const int cap = most * sms / G::CL;
    if (cap > s.clusters) s.clusters = cap;
  }
  return DGFS_OK;
}

// Fewer clusters where their workspaces would pass 16 GB: the faces grow with the sphere rule (a
// thousand directions at N = 32: 17 MB a cluster), and rules of any size stay accepted.
inline void cap_clusters(Plan& pl, size_t slot_bytes) {
  const size_t cap = (size_t(16) << 30) / slot_bytes;
  for (KernelShape& s : pl.shapes)
    if (size_t(s.clusters) > cap) s.clusters = cap > 0 ? int(cap) : 1;
}

template <typename T, int N>
int vhs_configure_impl(Plan& pl) {
  using G = VGeo<T, N, 0>;
  if (int rc = configure_shape<T, N, 0>(pl)) return rc;
  if constexpr (HasWide<T, N>::value) {
    if (int rc = configure_shape<T, N, 1>(pl)) return rc;
  }
  pl.shape.slot = G::SLOT + size_t(pl.max_ent) * G::FACE;
  // one workspace per cluster of either shape, then the products of split items
  cap_clusters(pl, pl.shape.slot * sizeof(C<T>));
  pl.part_slots = kPartsPerCluster * std::max(pl.shapes[0].clusters, pl.shapes[1].clusters);
  pl.part_size = G::HN3;
  size_workspace(pl);
  return DGFS_OK;
}

template <typename T, int N>
int vss_configure_impl(Plan& pl) {
  using G = VGeo<T, N, 2>;
  if (int rc = configure_shape<T, N, 2>(pl)) return rc;
  pl.shape.slot = G::SLOT + size_t(pl.max_ent) * G::FACE;
  cap_clusters(pl, pl.shape.slot * sizeof(C<T>));
  pl.part_slots = kVssPartsPerCluster * pl.shapes[0].clusters;
  pl.part_size = 2 * G::QN;
  size_workspace(pl);
  return DGFS_OK;
}

template <typename T, int N, int W>
int launch_shape(const Plan& pl, KernelParams& kp, int items, int limit, cudaStream_t st) {
  using G = VGeo<T, N, W>;
  const KernelShape& s = pl.shapes[W == 2 ? 0 : W];
  kp.phase_smem = s.phase_smem;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  launch_config(cfg, attr, G::CL, items < limit ? items : limit, s, st);
  return cudaLaunchKernelEx(&cfg, collision_kernel<T, N, W>, kp) == cudaSuccess ? DGFS_OK : DGFS_ERR_CUDA;
}

inline KernelParams kernel_params(const Plan& pl, const void* f, void* Q, int batch, int ws) {
  KernelParams kp{};
  kp.f = f;
  kp.Q = Q;
  kp.batch = batch;
  kp.s = pl.s;
  kp.n_tasks = int(pl.tasks.size());
  kp.n_rho = pl.N_rho;
  kp.max_ent = pl.max_ent;
  kp.tasks = pl.d_tasks;
  kp.groups = pl.d_groups;
  kp.faces = pl.d_faces;
  kp.phase = pl.d_phase;
  kp.Fw = pl.d_Fwf ? static_cast<const void*>(pl.d_Fwf) : static_cast<const void*>(pl.d_Fw);
  kp.Fv = pl.d_Fvf ? static_cast<const void*>(pl.d_Fvf) : static_cast<const void*>(pl.d_Fv);
  kp.Gm = pl.d_Gmf ? static_cast<const void*>(pl.d_Gmf) : static_cast<const void*>(pl.d_Gm);
  kp.ent_m = pl.d_ent_m;
  kp.n_fslot = pl.n_fslot;
  kp.scratch = pl.scratch_of(ws);
  kp.slot = pl.shape.slot;
  kp.work_counter = pl.counter_of(ws);
  kp.chunks = 1;
  return kp;
}

template <typename T, int N>
int vss_launch_impl(const Plan& pl, const void* f, void* Q, int batch, cudaStream_t st, int ws) {
  KernelParams kp = kernel_params(pl, f, Q, batch, ws);
  kp.parts = static_cast<C<T>*>(pl.scratch_of(ws)) + pl.part_off;
  const int n = int(pl.shapes[0].clusters * pl.shape.share), limit = n < 1 ? 1 : n;
  const int items = batch * kp.n_tasks;
  kp.chunks = vss_chunks(items, pl.N_rho, limit, task_load(pl), pl.part_slots_of(ws));
  return launch_shape<T, N, 2>(pl, kp, items * kp.chunks, limit, st);
}

template <typename T, int N>
int vhs_launch_impl(const Plan& pl, const void* f, void* Q, int batch, cudaStream_t st, int ws) {
  KernelParams kp = kernel_params(pl, f, Q, batch, ws);
  kp.parts = static_cast<C<T>*>(pl.scratch_of(ws)) + pl.part_off;
  auto share_of = [&](int clusters) {
    const int n = int(clusters * pl.shape.share);
    return n < 1 ? 1 : n;
  };
  const int items = batch * kp.n_tasks;
  const int c0 = share_of(pl.shapes[0].clusters), c1 = pl.shapes[1].clusters > 0 ? share_of(pl.shapes[1].clusters) : 0;
  const LaunchPlan run = plan_launch(items, pl.N_rho, c0, c1, HasWide<T, N>::slow, task_load(pl),
                                     pl.part_slots_of(ws));
  kp.chunks = run.chunks;
  if constexpr (HasWide<T, N>::value) {
    if (run.wide) return launch_shape<T, N, 1>(pl, kp, items * run.chunks, c1, st);
  }
  return launch_shape<T, N, 0>(pl, kp, items * run.chunks, c0, st);
}

}  // namespace dgfs
