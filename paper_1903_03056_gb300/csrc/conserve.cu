// Conservation projection and species sum, applied after the collision kernel.
//
// A block is a self pair Q_ii (5 constraint rows: 1, v_x, v_y, v_z, |v|^2) or a stacked cross pair
// [Q_ij; Q_ji] (6 rows: the two masses, m_i w_ij v + m_j w_ji v, m_i w_ij |v|^2 + m_j w_ji |v|^2),
// the discrete laws of Eq. consv.  The projection replaces Q by Q - C^T lambda,
// lambda = (C C^T)^-1 C Q, the nearest vector (in L2) that satisfies the laws exactly.
//
// conserve_kernel: one cluster of CTAs per (node, block).  The moment sums are FP64 and bound by
// the FP64 pipe (two multiply-adds a cycle and SM), so each thread keeps one pair of v_z nodes and
// walks over the (x, y) rows: eight FP64 operations and one integer division per pair of values instead
// of nine operations and two 64-bit divisions per value, and the cluster spreads a block over up to 8 SMs.  The CTAs read each
// other's partial sums through distributed shared memory, in rank order, so the result does not
// depend on the batch.  Then each CTA subtracts C^T lambda from its rows (APPLY), or rank 0 stores
// lambda for the species sum.  Measured (GB300): one N = 16 node 79 us -> 7 us, 45 nodes of N = 24
// 230 us -> 21 us.
//
// species_sum_kernel: Q_i = sum_j kappa_ij Q_ij (Eq. NMBE right-hand side, kappa = 1/Kn).  With the
// projection it subtracts sum_j kappa_ij C^T lambda_ij, a polynomial in v of five coefficients per
// (node, i), so the projected operators are never written.
#include "dgfs_internal.h"
#include "group_sync.cuh"

namespace dgfs {

namespace {

constexpr int kConsThreads = 256;
constexpr int kMaxN = 48;

// CTAs per (node, block): about 64 rows of N values each, at most 8 (a portable cluster)
int cons_cluster(int N) { return N <= 8 ? 1 : N == 12 ? 2 : N == 16 ? 4 : 8; }

__device__ __forceinline__ double2 load_pair(const float* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  return make_double2(double(v.x), double(v.y));
}
__device__ __forceinline__ double2 load_pair(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ void store_pair(float* p, double a, double b) {
  *reinterpret_cast<float2*>(p) = make_float2(float(a), float(b));
}
__device__ __forceinline__ void store_pair(double* p, double a, double b) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

__device__ __forceinline__ double ld_cluster(const double* local, unsigned rank) {
  const unsigned addr = static_cast<unsigned>(__cvta_generic_to_shared(local));
  unsigned remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the threads of a CTA as pairs of v_z nodes times rows: thread t owns pair t % (N / 2) and the rows
// t / (N / 2) + k (threads of a multiple of N / 2)
__device__ __forceinline__ int rows_per_round(int N) { return kConsThreads / (N / 2); }

template <typename T, bool APPLY>
__global__ void __launch_bounds__(kConsThreads) conserve_kernel(T* Q, int s, int N, double L, const ConsBlock* blocks,
                                                                int n_blocks, int cl, double* lam_out) {
  __shared__ double vt[kMaxN];                // grid velocities
  __shared__ double red[10][kConsThreads];
  __shared__ double part[10];                 // this CTA's sums, read by the whole cluster
  __shared__ double tot[10];
  __shared__ double lam[6];
  const int tid = threadIdx.x;
  const unsigned rank = blockIdx.x % cl;
  const int work = blockIdx.x / cl;
  const int b = work / n_blocks;
  const ConsBlock& cb = blocks[work % n_blocks];
  const bool cross = cb.rows == 6;
  const int N2 = N * N, h = N / 2;
  T* const x1 = Q + ((size_t(b) * s + cb.i) * s + cb.j) * N2 * N;
  T* const x2 = Q + ((size_t(b) * s + cb.j) * s + cb.i) * N2 * N;  // == x1 for a self pair
  if (tid < N) vt[tid] = -L + (tid + 0.5) * (2.0 * L / N);
  __syncthreads();

  const int rpr = rows_per_round(N);
  const int z = 2 * (tid % h);
  const int row0 = int(rank) * N2 / cl, row1 = (int(rank) + 1) * N2 / cl;
  const int first = tid / h < rpr ? row0 + tid / h : row1;
  const double vz0 = vt[z], vz1 = vt[z + 1];

  // per half: sums of the two v_z nodes' values, and of their sum times vx, vy, vx^2 + vy^2
  double acc[10] = {};
  auto take = [&](const T* q, int r, double* a) {
    const int ix = r / N, iy = r - ix * N;
    const double2 v = load_pair(q + size_t(r) * N + z);
    const double vx = vt[ix], vy = vt[iy], sum = v.x + v.y;
    a[0] += v.x;
    a[1] += v.y;
    a[2] += sum * vx;
    a[3] += sum * vy;
    a[4] += sum * (vx * vx + vy * vy);
  };
  for (int r = first; r < row1; r += rpr) {
    take(x1, r, acc);
    if (cross) take(x2, r, acc + 5);
  }
  // 1, vx, vy, vz, |v|^2
#pragma unroll
  for (int k = 0; k < 10; k += 5) {
    const double a0 = acc[k], a1 = acc[k + 1];
    red[k][tid] = a0 + a1;
    red[k + 1][tid] = acc[k + 2];
    red[k + 2][tid] = acc[k + 3];
    red[k + 3][tid] = a0 * vz0 + a1 * vz1;
    red[k + 4][tid] = acc[k + 4] + a0 * (vz0 * vz0) + a1 * (vz1 * vz1);
  }
  __syncthreads();
  {
    const int k = tid / 16, j = tid % 16;  // 160 threads: 16 per sum, 16 values each
    double v = 0.0;
    if (k < 10)
      for (int i = 0; i < kConsThreads / 16; ++i) v += red[k][j + 16 * i];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
    if (k < 10 && j == 0) part[k] = v;
  }
  if (cl > 1) cluster_barrier(); else __syncthreads();
  if (tid < 10) {
    double v = 0.0;
    if (cl > 1)
      for (int r = 0; r < cl; ++r) v += ld_cluster(&part[tid], unsigned(r));
    else
      v = part[tid];
    tot[tid] = v;
  }
  __syncthreads();
  if (tid < cb.rows) {
    double v = 0.0;
    for (int c = 0; c < cb.rows; ++c) {
      double cq;
      if (!cross) cq = tot[c];
      else if (c < 2) cq = tot[5 * c];
      else cq = cb.a * tot[c - 1] + cb.b * tot[c + 4];
      v += cb.minv[tid * cb.rows + c] * cq;
    }
    lam[tid] = v;
    if (!APPLY && rank == 0) lam_out[size_t(work) * 6 + tid] = v;
  }
  if constexpr (APPLY) {
    __syncthreads();
    // Q <- Q - C^T lambda: a polynomial l0 + w (l vx + l vy + l vz + l |v|^2) per half
    auto give = [&](T* q, int r, double l0, double w, const double* l) {
      const int ix = r / N, iy = r - ix * N;
      const double vx = vt[ix], vy = vt[iy];
      const double base = l0 + w * (l[0] * vx + l[1] * vy + l[3] * (vx * vx + vy * vy));
      const double2 v = load_pair(q + size_t(r) * N + z);
      store_pair(q + size_t(r) * N + z, v.x - (base + w * (l[2] * vz0 + l[3] * (vz0 * vz0))),
                 v.y - (base + w * (l[2] * vz1 + l[3] * (vz1 * vz1))));
    };
    for (int r = first; r < row1; r += rpr) {
      if (cross) {
        give(x1, r, lam[0], cb.a, lam + 2);
        give(x2, r, lam[1], cb.b, lam + 2);
      } else {
        give(x1, r, lam[0], 1.0, lam + 1);
      }
    }
  }
  if (cl > 1) cluster_barrier();  // no CTA leaves while another may read its sums
}

// one CTA per (node, species) and slab of rows (grid.x); lam != null: subtract the projection
template <typename T>
__global__ void __launch_bounds__(kConsThreads) species_sum_kernel(const T* __restrict__ Qfull, T* __restrict__ Qsum,
                                                                   int batch, int s, int N, double L,
                                                                   const double* __restrict__ kappa,
                                                                   const ConsBlock* __restrict__ blocks, int n_blocks,
                                                                   const double* __restrict__ lam) {
  __shared__ double vt[kMaxN];
  __shared__ double coef[5];  // 1, vx, vy, vz, |v|^2
  const int tid = threadIdx.x;
  const int N2 = N * N, h = N / 2;
  const int rpr = rows_per_round(N);
  const int z = 2 * (tid % h);
  const int row0 = int(blockIdx.x) * N2 / int(gridDim.x), row1 = (int(blockIdx.x) + 1) * N2 / int(gridDim.x);
  const int first = tid / h < rpr ? row0 + tid / h : row1;
  if (tid < N) vt[tid] = -L + (tid + 0.5) * (2.0 * L / N);
  for (int bi = blockIdx.y; bi < batch * s; bi += gridDim.y) {
    const int b = bi / s, i = bi % s;
    __syncthreads();  // vt written, the previous coefficients read
    if (tid < 5) {
      double c = 0.0;
      if (lam != nullptr) {
        for (int k = 0; k < n_blocks; ++k) {
          const ConsBlock& cb = blocks[k];
          const double* const l = lam + (size_t(b) * n_blocks + k) * 6;
          if (cb.rows == 5) {
            if (cb.i == i) c += kappa[i * s + i] * l[tid];
          } else {
            if (cb.i == i) c += kappa[i * s + cb.j] * (tid == 0 ? l[0] : cb.a * l[tid + 1]);
            if (cb.j == i) c += kappa[i * s + cb.i] * (tid == 0 ? l[1] : cb.b * l[tid + 1]);
          }
        }
      }
      coef[tid] = c;
    }
    __syncthreads();
    const double vz0 = vt[z], vz1 = vt[z + 1];
    const double pz0 = coef[3] * vz0 + coef[4] * (vz0 * vz0), pz1 = coef[3] * vz1 + coef[4] * (vz1 * vz1);
    const T* const q = Qfull + size_t(bi) * s * N2 * N + z;
    T* const out = Qsum + size_t(bi) * N2 * N + z;
    for (int r = first; r < row1; r += rpr) {
      double a0 = 0.0, a1 = 0.0;
      for (int j = 0; j < s; ++j) {
        const double2 v = load_pair(q + (size_t(j) * N2 + r) * N);
        a0 += kappa[i * s + j] * v.x;
        a1 += kappa[i * s + j] * v.y;
      }
      if (lam != nullptr) {
        const int ix = r / N, iy = r - ix * N;
        const double vx = vt[ix], vy = vt[iy];
        const double base = coef[0] + coef[1] * vx + coef[2] * vy + coef[4] * (vx * vx + vy * vy);
        a0 -= base + pz0;
        a1 -= base + pz1;
      }
      store_pair(out + size_t(r) * N, a0, a1);
    }
  }
}

template <typename T, bool APPLY>
int run_conserve(const Plan& p, void* Q, int batch, double* lam, cudaStream_t st) {
  const int nb = int(p.cons.size()), cl = cons_cluster(p.N);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(unsigned(batch) * nb * cl);
  cfg.blockDim = dim3(kConsThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const ConsBlock* const blocks = p.d_cons;
  return cudaLaunchKernelEx(&cfg, conserve_kernel<T, APPLY>, static_cast<T*>(Q), p.s, p.N, p.L, blocks, nb, cl, lam) ==
                 cudaSuccess
             ? DGFS_OK
             : (cudaGetLastError(), DGFS_ERR_CUDA);
}

template <typename T>
int run_species_sum(const Plan& p, const void* Qfull, void* Qsum, int batch, const double* lam, cudaStream_t st) {
  // slabs of about 4 rounds of rows, fewer where the nodes alone fill the device
  const int rounds = (p.N * p.N + kConsThreads / (p.N / 2) - 1) / (kConsThreads / (p.N / 2));
  const unsigned gx = unsigned((rounds + 3) / 4);
  const unsigned gy = unsigned(batch) * p.s < 65535u ? unsigned(batch) * p.s : 65535u;
  species_sum_kernel<T><<<dim3(gx, gy), kConsThreads, 0, st>>>(static_cast<const T*>(Qfull), static_cast<T*>(Qsum), batch,
                                                              p.s, p.N, p.L, p.d_kappa, p.d_cons, int(p.cons.size()), lam);
  return cudaPeekAtLastError() == cudaSuccess ? DGFS_OK : (cudaGetLastError(), DGFS_ERR_CUDA);
}

}  // namespace

int launch_conserve(const Plan& p, void* Q, int batch, double* lam, cudaStream_t st) {
  if (p.cons.empty() || batch == 0) return DGFS_OK;
  if (p.f32io()) return lam ? run_conserve<float, false>(p, Q, batch, lam, st) : run_conserve<float, true>(p, Q, batch, lam, st);
  return lam ? run_conserve<double, false>(p, Q, batch, lam, st) : run_conserve<double, true>(p, Q, batch, lam, st);
}

int launch_species_sum(const Plan& p, const void* Qfull, void* Qsum, int batch, const double* lam, cudaStream_t st) {
  if (batch == 0) return DGFS_OK;
  return p.f32io() ? run_species_sum<float>(p, Qfull, Qsum, batch, lam, st)
                   : run_species_sum<double>(p, Qfull, Qsum, batch, lam, st);
}

}  // namespace dgfs
