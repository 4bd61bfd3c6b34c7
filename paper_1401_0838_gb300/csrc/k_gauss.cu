// Charge-conservation diagnostic: the residual of Gauss's law div E - F rho on the integer nodes.
//
// The Esirkepov deposit (cited in Sec. 2) makes the current satisfy the discrete continuity equation
// with the charge density rho of the particles' own shapes, and the Yee E update subtracts the
// filtered current F J, so div E - F rho keeps its initial value (zero for the neutral beam) up to
// rounding. These kernels compute that residual in FP64 from the live state: rho deposited from the
// particle bins with the B-spline of the run's shape order, filtered by the current filter's taps
// (the separable stencil kernel in FP64), then reduced node by node.
#include "common.cuh"
#include "launch.h"

namespace picgb {

constexpr int RHO_THREADS = 256;
constexpr int GR_THREADS = 256;
constexpr int GR_BLOCKS = 4 * 152;

// Weights of the nodes base, base + 1, ... for offset o in [0, 1) inside the cell: order 1 on the
// cell's two nodes (base = cell), order 3 the cubic B-spline on four nodes (base = cell - 1).
template <int ORDER>
__device__ __forceinline__ void node_weights(double o, double (&w)[ORDER + 1]) {
  if constexpr (ORDER == 3) {
    const double p = 1.0 - o;
    w[0] = p * p * p / 6.0;
    w[1] = (4.0 - 6.0 * o * o + 3.0 * o * o * o) / 6.0;
    w[2] = (4.0 - 6.0 * p * p + 3.0 * p * p * p) / 6.0;
    w[3] = o * o * o / 6.0;
  } else {
    w[0] = 1.0 - o;
    w[1] = o;
  }
}

__device__ __forceinline__ int wrap_any(int g, int n) {
  g %= n;
  return g < 0 ? g + n : g;
}

// rho += q w S(x - x_node) / dV for every particle. lpc lanes per cell, a power of two: one where the cells
// alone fill the GPU, so that every lane of an FP64 instruction works (that pipe bounds this kernel: a
// warp per cell left half to three quarters of the lanes idle). A lane sums its particles' weights in
// registers, the cell's lanes add up, and one lane adds each node once instead of once per particle:
// 331 -> 95 us on 301 x 517 cells of 2 x 8 particles. Cells that hold far more particles than their
// neighbours (bunches) would keep a warp on one lane: past a limit the whole warp takes a cell's
// particles together (3000 more in each of eight cells of 300 x 300, cubic: the residual in 0.7 ms, 12 ms
// on the cells' own lanes).
template <typename T, int NDIM, int ORDER>
__global__ void __launch_bounds__(RHO_THREADS) k_rho(const __grid_constant__ RunDev<T> r, int lpc, double inv_dv,
                                                     double* __restrict__ rho) {
  constexpr int NN = ORDER + 1, NY = NDIM == 3 ? NN : 1, LO = ORDER == 3 ? -1 : 0;
  const int lane = threadIdx.x & 31;
  const long long step = (long long)gridDim.x * RHO_THREADS / lpc;
  // every lane of a warp runs the same trips: the lanes past the last cell take part in the sums with nothing
  for (long long c0 = ((long long)blockIdx.x * RHO_THREADS + (threadIdx.x & ~31)) / lpc; c0 < r.ncell; c0 += step) {
    const long long own = c0 + lane / lpc;
    const bool in = own < r.ncell;
    const int own0 = in ? min(r.in[0].cnt[own], r.cap) : 0, own1 = in ? min(r.in[1].cnt[own], r.cap) : 0;
    // slots per species that the cell's own lanes take: all, or what leaves clearly fewer rounds of the warp (a
    // round of the lanes' own cells, or 32 slots of a crowded one, which also costs two for its sums)
    const int most = __reduce_max_sync(0xffffffffu, max(own0, own1));
    int limit = most;
    unsigned more = 0;
    if (lpc < 32 && most > 16 * lpc) {
      int best = 3 * ((most + lpc - 1) / lpc) / 2;  // a quarter less than all of them
      for (int l = 8 * lpc; l < most; l *= 2) {
        const int x = max(own0 - l, 0), y = max(own1 - l, 0);
        const int extra = lane % lpc == 0 && (x | y) != 0 ? (x + 31) / 32 + (y + 31) / 32 + 2 : 0;
        const int rounds = 2 * (l / lpc) + __reduce_add_sync(0xffffffffu, extra);
        if (rounds < best) {
          best = rounds;
          limit = l;
        }
      }
      more = __ballot_sync(0xffffffffu, lane % lpc == 0 && max(own0, own1) > limit);
    }
    int lanes = lpc, first = 0;
    bool on = in;
    long long cell = own;
    int n0 = min(own0, limit), n1 = min(own1, limit);
    for (;;) {
      const int sub = lane & (lanes - 1);
      double acc[NN * NY * NN] = {};
#pragma unroll 1
      for (int s = 0; s < 2; ++s) {
        const SpeciesBuf<T>& b = s ? r.in[1] : r.in[0];
        const int n = s ? n1 : n0;
        const double q = s ? inv_dv : -inv_dv;
        for (int slot = first + sub; slot < n; slot += lanes) {
          const long long o = cell * r.cap + slot;
          const double qw = q * (b.w ? (double)b.w[o] : (double)r.wconst);
          double wx[NN], wy[NN], wz[NN];
          const PartVals<T> v = part_get(b, NDIM, o);
          node_weights<ORDER>((double)v.ox, wx);
          if constexpr (NDIM == 3) node_weights<ORDER>((double)v.oy, wy);
          node_weights<ORDER>((double)v.oz, wz);
#pragma unroll
          for (int c = 0; c < NN; ++c)
#pragma unroll
            for (int bb = 0; bb < NY; ++bb) {
              const double wyz = NDIM == 3 ? qw * wy[bb] * wz[c] : qw * wz[c];
#pragma unroll
              for (int a = 0; a < NN; ++a) acc[(c * NY + bb) * NN + a] = fma(wyz, wx[a], acc[(c * NY + bb) * NN + a]);
            }
        }
      }
      int d = lanes >> 1;
      while (d >= most && d > 0) d >>= 1;  // the lanes past the fullest cell's slots hold nothing
      for (; d > 0; d >>= 1)
#pragma unroll
        for (int e = 0; e < NN * NY * NN; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], d);
      if (on && sub == 0) {
        const int ci = (int)cell, i = ci % r.nx, j = ci / r.nx % r.ny, k = ci / r.nx / r.ny;
#pragma unroll
        for (int c = 0; c < NN; ++c) {
          const long long kz = wrap_any(k + LO + c, r.nz);
#pragma unroll
          for (int bb = 0; bb < NY; ++bb) {
            const long long jy = NDIM == 3 ? wrap_any(j + LO + bb, r.ny) : 0;
#pragma unroll
            for (int a = 0; a < NN; ++a) {
              const double v = acc[(c * NY + bb) * NN + a];
              if (v != 0.0) atomicAdd(rho + (kz * r.ny + jy) * r.nx + wrap_any(i + LO + a, r.nx), v);
            }
          }
        }
      }
      if (more == 0) break;
      const int src = __ffs(more) - 1;  // the next crowded cell, past its lanes' share
      more &= more - 1;
      lanes = 32;
      first = limit;
      on = true;
      cell = c0 + src / lpc;
      n0 = __shfl_sync(0xffffffffu, own0, src);
      n1 = __shfl_sync(0xffffffffu, own1, src);
    }
  }
}

// (max, sum, max) of the block's values, in thread 0.
__device__ __forceinline__ void block_max_sum_max(double& m0, double& s, double& m1) {
  __shared__ double red[3][GR_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m0 = fmax(m0, __shfl_xor_sync(0xffffffffu, m0, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
    m1 = fmax(m1, __shfl_xor_sync(0xffffffffu, m1, o));
  }
  __syncthreads();  // the sums of an earlier call are read
  if (lane == 0) {
    red[0][w] = m0;
    red[1][w] = s;
    red[2][w] = m1;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int q = 1; q < GR_THREADS / 32; ++q) {
      m0 = fmax(m0, red[0][q]);
      s += red[1][q];
      m1 = fmax(m1, red[2][q]);
    }
}

// Node residual res = div E - rho_f (FP64 from the stored precision). Per thread: max |res|, sum
// res^2, max |rho_f|; per block: tree into scratch[3 * block + r]; the last block to finish combines
// the partials in a fixed order (all its threads: one thread's walk over 608 blocks took 120 of 129 us)
// and writes out = (max |res|, rms res, max |rho_f|).
template <typename T>
__global__ void __launch_bounds__(GR_THREADS) k_gauss_residual(const T* __restrict__ ex, const T* __restrict__ ey,
                                                               const T* __restrict__ ez,
                                                               const double* __restrict__ rhof, int nx, int ny,
                                                               int nz, double idx, double idy, double idz,
                                                               double* scratch, double* out) {
  const long long nxy = (long long)nx * ny, n = nxy * nz;
  double mres = 0.0, ssq = 0.0, mrho = 0.0;
  for (long long c = blockIdx.x * (long long)GR_THREADS + threadIdx.x; c < n; c += (long long)gridDim.x * GR_THREADS) {
    const int i = (int)(c % nx), j = (int)((c / nx) % ny), k = (int)(c / nxy);
    const long long im = c - i + (i == 0 ? nx - 1 : i - 1);
    const long long jm = c + ((j == 0 ? ny - 1 : j - 1) - j) * (long long)nx;
    const long long km = c + ((k == 0 ? nz - 1 : k - 1) - k) * nxy;
    const double dive = ((double)ex[c] - (double)ex[im]) * idx + ((double)ey[c] - (double)ey[jm]) * idy +
                        ((double)ez[c] - (double)ez[km]) * idz;
    const double res = dive - rhof[c];
    mres = fmax(mres, fabs(res));
    ssq += res * res;
    mrho = fmax(mrho, fabs(rhof[c]));
  }
  __shared__ bool last;
  block_max_sum_max(mres, ssq, mrho);
  if (threadIdx.x == 0) {
    scratch[3 * blockIdx.x + 0] = mres;
    scratch[3 * blockIdx.x + 1] = ssq;
    scratch[3 * blockIdx.x + 2] = mrho;
    __threadfence();
    last = atomicAdd(reinterpret_cast<unsigned*>(scratch + 3 * GR_BLOCKS), 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  mres = ssq = mrho = 0.0;
  for (unsigned q = threadIdx.x; q < gridDim.x; q += GR_THREADS) {
    mres = fmax(mres, __ldcg(scratch + 3 * q + 0));
    ssq += __ldcg(scratch + 3 * q + 1);
    mrho = fmax(mrho, __ldcg(scratch + 3 * q + 2));
  }
  block_max_sum_max(mres, ssq, mrho);
  if (threadIdx.x == 0) {
    out[0] = mres;
    out[1] = sqrt(ssq / (double)n);
    out[2] = mrho;
    *reinterpret_cast<unsigned*>(scratch + 3 * GR_BLOCKS) = 0u;
  }
}

size_t gauss_scratch_bytes() { return sizeof(double) * (3 * GR_BLOCKS + 2); }

template <typename T>
cudaError_t launch_rho(const RunDev<T>& r, int order, double inv_dv, double* rho, cudaStream_t st) {
  // lanes per cell: until the cells give each of the 152 SMs four warps, one per scheduler, or a warp has one
  // cell. The residual on 64x64 cubic cells of 2 x 8 takes 123 us (with 8 warps per SM 140, with 16 191)
  int lpc = 1;
  while (lpc < 32 && r.ncell * lpc < 152ll * 128) lpc *= 2;
  const long long want = (r.ncell * lpc + RHO_THREADS - 1) / RHO_THREADS;
  const int blocks = (int)(want < 8 * 152 ? (want < 1 ? 1 : want) : 8 * 152);
  if (r.ndim == 3 && order == 3)
    k_rho<T, 3, 3><<<blocks, RHO_THREADS, 0, st>>>(r, lpc, inv_dv, rho);
  else if (r.ndim == 3)
    k_rho<T, 3, 1><<<blocks, RHO_THREADS, 0, st>>>(r, lpc, inv_dv, rho);
  else if (order == 3)
    k_rho<T, 2, 3><<<blocks, RHO_THREADS, 0, st>>>(r, lpc, inv_dv, rho);
  else
    k_rho<T, 2, 1><<<blocks, RHO_THREADS, 0, st>>>(r, lpc, inv_dv, rho);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gauss_residual(const T* ex, const T* ey, const T* ez, const double* rhof, int nx, int ny, int nz,
                                  double idx, double idy, double idz, double* scratch, double* out, cudaStream_t st) {
  const long long n = (long long)nx * ny * nz;
  const long long want = (n + GR_THREADS - 1) / GR_THREADS;
  const int blocks = (int)(want < GR_BLOCKS ? (want < 1 ? 1 : want) : GR_BLOCKS);
  k_gauss_residual<T><<<blocks, GR_THREADS, 0, st>>>(ex, ey, ez, rhof, nx, ny, nz, idx, idy, idz, scratch, out);
  return cudaGetLastError();
}

template cudaError_t launch_rho<float>(const RunDev<float>&, int, double, double*, cudaStream_t);
template cudaError_t launch_rho<double>(const RunDev<double>&, int, double, double*, cudaStream_t);
template cudaError_t launch_gauss_residual<float>(const float*, const float*, const float*, const double*, int, int,
                                                  int, double, double, double, double*, double*, cudaStream_t);
template cudaError_t launch_gauss_residual<double>(const double*, const double*, const double*, const double*, int,
                                                   int, int, double, double, double, double*, double*, cudaStream_t);

}  // namespace picgb
