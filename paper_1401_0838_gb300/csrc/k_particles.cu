// Particle kernels: fused gather + Boris + move + Esirkepov deposition + rebin, beam
// initialisation, state import (binning) and export (compaction).
//
// Particle storage: per species, per cell, a bin of `cap` slots (SpeciesBuf). The push kernel
// reads the input buffer and writes every particle straight into its destination cell's bin of
// the output buffer (a counting-sort rebin fused into the push), so particles stay sorted by
// cell at no extra HBM pass. Positions are cell-relative offsets in [0,1); momenta are stored
// relative to the drift u0 z_hat so that FP32 keeps the thermal spread (u0 = 130, spread 1e-4).
#include "common.cuh"
#include "launch.h"
#include "push_tile.cuh"

namespace picgb {

// One tile per block.
template <typename T, int NDIM, int SCHEME, int LPC>
__global__ void __launch_bounds__(PushThreads<T, NDIM>::value, PushMinBlocks<T, NDIM>::value)
    k_push(const __grid_constant__ RunDev<T> r) {
  pdl_wait();
  push_tile<T, NDIM, SCHEME, LPC>(r, blockIdx.x);
}

// Persistent form for many runs: each block takes (run, tile) work items from a global counter
// (items grouped by run, so a block mostly stays on one run) and copies the run's descriptor into
// shared memory when the run changes. Work-list counter reset: the caller zeroes *queue before the
// launch.
template <typename T, int NDIM, int SCHEME, int LPC>
__global__ void __launch_bounds__(PushThreads<T, NDIM>::value, PushMinBlocks<T, NDIM>::value)
    k_push_batch(const RunDev<T>* __restrict__ runs, const int2* __restrict__ items, int nitems, int* queue) {
  pdl_wait();
  __shared__ RunDev<T> rs;
  __shared__ int cur, cur_run;
  if (threadIdx.x == 0) cur_run = -1;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) cur = atomicAdd(queue, 1);
    __syncthreads();
    const int it = cur;
    if (it >= nitems) break;
    const int2 w = items[it];
    if (w.x != cur_run) {  // warp 0 copies the descriptor as 32-bit words
      __syncthreads();
      constexpr int NW = (int)(sizeof(RunDev<T>) / 4);
      const int* src = reinterpret_cast<const int*>(runs + w.x);
      int* dst = reinterpret_cast<int*>(&rs);
      for (int k = threadIdx.x; k < NW; k += PushThreads<T, NDIM>::value) dst[k] = src[k];
      __syncthreads();
      if (threadIdx.x == 0) cur_run = w.x;
    }
    __syncthreads();
    push_tile<T, NDIM, SCHEME, LPC>(rs, w.y);
  }
}

// Lanes per cell from the expected particles per cell (both species): packs of 4 per lane.
static int lanes_per_cell(int ndim, int ppc_total) {
  const int packs = 2 * ((ppc_total / 2 + 3) / 4);  // packs of 4 per species
  // 2D: four lanes per cell up to 8 packs (two packs per lane halve the per-cell reduction cost;
  // measured 3 % faster than eight lanes at 16 particles/cell/species on GB300)
  // 3D up to 4 packs: two lanes per cell (a lane's two packs halve the per-cell reduction and
  // Galerkin loads per particle; measured 5 % faster than four lanes at 8 particles/cell/species)
  if (ndim == 3 && packs <= 4) return 2;
  if (packs <= 4 || (ndim == 2 && packs <= 8)) return 4;
  if (packs <= 8) return 8;
  return 16;
}

template <typename T, int NDIM, int SCHEME>
static cudaError_t launch_push_t(const RunDev<T>& r, int lpc, cudaStream_t st) {
  using S = PushSmem<T, NDIM>;
  const size_t sm = S::bytes();
  const int ntiles = r.ntx * r.nty * r.ntz;
  auto go = [&](void (*kern)(const RunDev<T>)) -> cudaError_t {
    cudaError_t e = ensure_dynamic_smem((const void*)kern, sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(ntiles), dim3(PushThreads<T, NDIM>::value), sm, st, r);
  };
  if constexpr (NDIM == 3) {
    if (lpc == 2) return go(k_push<T, NDIM, SCHEME, 2>);
  }
  if (lpc == 4) return go(k_push<T, NDIM, SCHEME, 4>);
  if (lpc == 8) return go(k_push<T, NDIM, SCHEME, 8>);
  return go(k_push<T, NDIM, SCHEME, 16>);
}

template <typename T>
cudaError_t launch_push(const RunDev<T>& r, int ppc_total, cudaStream_t st) {
  if (!tiles_fit<PTile>(r)) return cudaErrorInvalidValue;
  const int lpc = lanes_per_cell(r.ndim, ppc_total);
  if (r.ndim == 2)
    return r.scheme == 0 ? launch_push_t<T, 2, 0>(r, lpc, st) : launch_push_t<T, 2, 1>(r, lpc, st);
  return r.scheme == 0 ? launch_push_t<T, 3, 0>(r, lpc, st) : launch_push_t<T, 3, 1>(r, lpc, st);
}
template cudaError_t launch_push<float>(const RunDev<float>&, int, cudaStream_t);

template <typename T, int NDIM, int SCHEME>
static cudaError_t launch_push_batch_t(const RunDev<T>* runs, const int2* items, int nitems, int* queue, int lpc,
                                       int blocks, cudaStream_t st) {
  using S = PushSmem<T, NDIM>;
  const size_t sm = S::bytes();
  auto go = [&](void (*kern)(const RunDev<T>*, const int2*, int, int*)) -> cudaError_t {
    cudaError_t e = ensure_dynamic_smem((const void*)kern, sm);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(queue, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(blocks), dim3(PushThreads<T, NDIM>::value), sm, st, runs, items, nitems, queue);
  };
  if (lpc == 4) return go(k_push_batch<T, NDIM, SCHEME, 4>);
  if (lpc == 8) return go(k_push_batch<T, NDIM, SCHEME, 8>);
  return go(k_push_batch<T, NDIM, SCHEME, 16>);
}

template <typename T>
cudaError_t launch_push_batch(const RunDev<T>* runs, const int2* items, int nitems, int* queue, int ndim, int scheme,
                              int lpc, int blocks, cudaStream_t st) {
  if (ndim == 2)
    return scheme == 0 ? launch_push_batch_t<T, 2, 0>(runs, items, nitems, queue, lpc, blocks, st)
                       : launch_push_batch_t<T, 2, 1>(runs, items, nitems, queue, lpc, blocks, st);
  return scheme == 0 ? launch_push_batch_t<T, 3, 0>(runs, items, nitems, queue, lpc, blocks, st)
                     : launch_push_batch_t<T, 3, 1>(runs, items, nitems, queue, lpc, blocks, st);
}
template cudaError_t launch_push_batch<float>(const RunDev<float>*, const int2*, int, int*, int, int, int, int,
                                              cudaStream_t);
template cudaError_t launch_push_batch<double>(const RunDev<double>*, const int2*, int, int*, int, int, int, int,
                                               cudaStream_t);

// The batched kernel is built for 4, 8 and 16 lanes per cell.
int push_lanes_per_cell(int ndim, int ppc_total) {
  const int l = lanes_per_cell(ndim, ppc_total);
  return l < 4 ? 4 : l;
}

template <typename T>
int push_max_blocks_per_sm(int ndim, int scheme, int lpc) {
  int n = 0;
  size_t sm = ndim == 2 ? PushSmem<T, 2>::bytes() : PushSmem<T, 3>::bytes();
  const void* k = nullptr;
  if (ndim == 2)
    k = scheme == 0 ? (lpc == 4 ? (const void*)k_push_batch<T, 2, 0, 4> : lpc == 8 ? (const void*)k_push_batch<T, 2, 0, 8> : (const void*)k_push_batch<T, 2, 0, 16>)
                    : (lpc == 4 ? (const void*)k_push_batch<T, 2, 1, 4> : lpc == 8 ? (const void*)k_push_batch<T, 2, 1, 8> : (const void*)k_push_batch<T, 2, 1, 16>);
  else
    k = scheme == 0 ? (lpc == 4 ? (const void*)k_push_batch<T, 3, 0, 4> : lpc == 8 ? (const void*)k_push_batch<T, 3, 0, 8> : (const void*)k_push_batch<T, 3, 0, 16>)
                    : (lpc == 4 ? (const void*)k_push_batch<T, 3, 1, 4> : lpc == 8 ? (const void*)k_push_batch<T, 3, 1, 8> : (const void*)k_push_batch<T, 3, 1, 16>);
  if (ensure_dynamic_smem(k, sm) != cudaSuccess) return 1;
  const int nt = ndim == 2 ? PushThreads<T, 2>::value : PushThreads<T, 3>::value;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, nt, sm) != cudaSuccess || n < 1) return 1;
  return n;
}
template int push_max_blocks_per_sm<float>(int, int, int);
template int push_max_blocks_per_sm<double>(int, int, int);
template cudaError_t launch_push<double>(const RunDev<double>&, int, cudaStream_t);

// The compile-time tile TL of the working precision T.
template <template <typename, int> class TL, typename T>
static void tile_of(int ndim, int te[3]) {
  if (ndim == 2) {
    te[0] = TL<T, 2>::TX;
    te[1] = 1;
    te[2] = TL<T, 2>::TZ;
  } else {
    te[0] = TL<T, 3>::TX;
    te[1] = TL<T, 3>::TY;
    te[2] = TL<T, 3>::TZ;
  }
}

void push_tiles(int ndim, int es, bool ho, int nx, int ny, int nz, int spread, int nt[3], int te[3]) {
  const int n[3] = {nx, ndim == 3 ? ny : 1, nz};
  int full[3];
  if (es == 4) ho ? tile_of<HoTile, float>(ndim, full) : tile_of<PTile, float>(ndim, full);
  else ho ? tile_of<HoTile, double>(ndim, full) : tile_of<PTile, double>(ndim, full);
  auto set = [&](int ex, int ey, int ez) {
    te[0] = ex;
    te[1] = ey;
    te[2] = ez;
    long long t = 1;
    for (int d = 0; d < 3; ++d) {
      nt[d] = (n[d] + te[d] - 1) / te[d];
      t *= nt[d];
    }
    return t;
  };
  set(full[0], full[1], full[2]);
  if (spread <= 0) return;
  // the resident blocks, and a tile's fixed cost (prologue and epilogue) in cells
  const int per_sm = es == 8 ? 1 : (ndim == 2 ? 2 : (ho ? 1 : 3));
  const long long slots = (long long)spread * per_sm;
  const int fixed = es == 4 ? 40 : 6;
  // a warp's cell group takes whole rows of the full tile's width, however narrow the tile is
  auto cost_of = [&](long long tiles) {
    return (double)((tiles + slots - 1) / slots) * ((double)full[0] * te[1] * te[2] + fixed);
  };
  const long long all = set(full[0], full[1], full[2]);
  if (per_sm > 1 && all > slots) return;  // several waves: the partners of a late block speed it up
  double best = 0.97 * cost_of(all);  // full tiles unless others gain 3 %
  int b[3] = {full[0], full[1], full[2]};
  for (int ey = full[1]; ey >= 4 || ey == full[1]; ey /= 2)
    for (int ez = full[2]; ez >= 4 || ez == full[2]; --ez) {
      const double cost = cost_of(set(full[0], ey, ez));
      if (cost < best * (1 - 1e-9)) {
        best = cost;
        b[1] = ey;
        b[2] = ez;
      }
    }
  // half the width where the tiles still fill one wave: the same rows, on twice as many SMs
  if (full[0] >= 8 && set(full[0] / 2, b[1], b[2]) <= slots) return;
  set(b[0], b[1], b[2]);
}

// ---------------------------------------------------------------------------------------------
// Migrate: insert the particles that left their tile in this step (leaver list of the push
// kernel) into their destination bins, then zero the other parity's list counter for the next
// step's push.
// ---------------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void migrate_body(const RunDev<T>& r, int* other_count, int bid, int nblk) {
  const long long n = min((long long)*r.lv_count, r.lv_cap);
  const int lane = threadIdx.x & 31;
  // whole warps iterate together (leavers of one source cell are consecutive and mostly share their
  // destination, so one atomic per destination group reserves their slots)
  const long long stride = (long long)nblk * blockDim.x;
  for (long long base = bid * (long long)blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
    const long long i = base + lane;
    const bool valid = i < n;
    int key = -1 - lane;
    T ox = T(0), oy = T(0), oz = T(0), ux = T(0), uy = T(0), uz = T(0), w = T(0);
    unsigned id = 0;
    if (valid) {
      key = r.lv.key[i];
      ox = r.lv.ox[i];
      if (r.ndim == 3) oy = r.lv.oy[i];
      oz = r.lv.oz[i];
      ux = r.lv.dux[i];
      uy = r.lv.duy[i];
      uz = r.lv.duz[i];
      if (r.lv.w) w = r.lv.w[i];
      if (r.lv.id) id = r.lv.id[i];
    }
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    const int rank = __popc(peers & ((1u << lane) - 1u));
    const int s = key & 1;
    const long long cell = key >> 1;
    const SpeciesBuf<T> b = s ? r.out[1] : r.out[0];
    int j0 = 0;
    if (valid && lane == leader) j0 = atomicAdd(b.cnt + cell, __popc(peers));
    j0 = __shfl_sync(0xffffffffu, j0, leader);
    // a full bin: the particle goes to the spill list, which the next step pushes from (the count
    // keeps the excess, so the host sees how large the bin has to grow)
    const bool full = valid && j0 + rank >= r.cap;
    const unsigned fmask = __ballot_sync(0xffffffffu, full);
    long long so = 0;
    if (fmask) {
      const int fl = __ffs(fmask) - 1;
      int sb = 0;
      if (lane == fl) {
        sb = atomicAdd(r.sp_out, __popc(fmask));
        atomicAdd(r.sp_total, (unsigned long long)__popc(fmask));
      }
      sb = __shfl_sync(0xffffffffu, sb, fl);
      so = (long long)sb + __popc(fmask & ((1u << lane) - 1u));
    }
    if (!valid) continue;
    if (full) {
      if (so < r.sp_cap) list_put(r.sp, so, key, ox, oy, oz, ux, uy, uz, w, id);
      else flag_error(r.err, ERR_OVERFLOW);
      continue;
    }
    const int j = j0 + rank;
    const long long o = cell * r.cap + j;
    part_put(b, r.ndim, o, ox, oy, oz, ux, uy, uz);
    if (b.w) b.w[o] = w;
    if (b.id) b.id[o] = id;
  }
  if (bid == 0 && threadIdx.x == 0) *other_count = 0;
}

template <typename T>
__global__ void k_migrate(const __grid_constant__ RunDev<T> r, int* other_count) {
  pdl_wait();
  migrate_body<T>(r, other_count, blockIdx.x, gridDim.x);
}

template <typename T>
__global__ void k_migrate_batch(const RunDev<T>* __restrict__ runs) {
  pdl_wait();
  const RunDev<T>& r = runs[blockIdx.y];
  migrate_body<T>(r, r.lv_other, blockIdx.x, gridDim.x);
}

template <typename T>
cudaError_t launch_migrate(const RunDev<T>& r, int* other_count, cudaStream_t st) {
  return launch_pdl(k_migrate<T>, dim3(152 * 4), dim3(256), 0, st, r, other_count);
}

template <typename T>
cudaError_t launch_migrate_batch(const RunDev<T>* runs, int nruns, cudaStream_t st) {
  dim3 grid(4 * 152 / (nruns < 4 ? 1 : nruns / 4) + 1, (unsigned)nruns);
  return launch_pdl(k_migrate_batch<T>, grid, dim3(256), 0, st, runs);
}
template cudaError_t launch_migrate_batch<float>(const RunDev<float>*, int, cudaStream_t);
template cudaError_t launch_migrate_batch<double>(const RunDev<double>*, int, cudaStream_t);
template cudaError_t launch_migrate<float>(const RunDev<float>&, int*, cudaStream_t);
template cudaError_t launch_migrate<double>(const RunDev<double>&, int*, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Insert one particle of species s into its cell bin of the input buffers (used by init and
// import) at slot j of the bin, reserved by the caller; past a full bin it goes to the spill list that the
// next step pushes from.
// ---------------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void insert_at(const RunDev<T>& r, const SpeciesBuf<T>& b, int s, long long cell, int j,
                                          T ox, T oy, T oz, T ux, T uy, T uz, T w, unsigned id) {
  const int cap = r.cap;
  if (j >= cap) {
    const long long o = atomicAdd(r.sp_in, 1);
    atomicAdd(r.sp_total, 1ull);
    if (o < r.sp_cap) list_put(r.sp, o, (int)(cell * 2 + s), ox, oy, oz, ux, uy, uz, w, id);
    else flag_error(r.err, ERR_OVERFLOW);
    return;
  }
  const long long o = cell * cap + j;
  part_put(b, r.ndim, o, ox, oy, oz, ux, uy, uz);
  if (b.w) b.w[o] = w;
  if (b.id) b.id[o] = id;
}
template <typename T>
__device__ __forceinline__ void insert_particle(const RunDev<T>& r, int s, long long cell, T ox, T oy, T oz, T ux,
                                                T uy, T uz, T w, unsigned id) {
  const SpeciesBuf<T>& b = s ? r.in[1] : r.in[0];
  insert_at(r, b, s, cell, atomicAdd(b.cnt + cell, 1), ox, oy, oz, ux, uy, uz, w, id);
}

// Fold a position (cell index per direction + offset, offset possibly outside [0,1)) into range.
template <typename T>
__device__ __forceinline__ void fold(int& i, T& o, int n) {
  T f = dev_floor(o);
  i += (int)f;
  o -= f;
  if (o >= T(1)) { o = T(0); i += 1; }
  if (o < T(0)) o = T(0);
  i = wrapi(i, n);
}

// ---------------------------------------------------------------------------------------------
// Seeded beam: one thread per lattice point p (cell-major, ppc points per cell on an lx x ly x lz
// lattice at offsets (l + 1/2) / n). Philox4x32-10 keyed by the seed with counter (p, 0, 0, 0) gives
// the position jitter, uniform in +-jitter cells per coordinate; counter (p, 1 + s, 0, 0) gives
// species s's two Box-Muller pairs for the thermal momenta (spread u_th per component, relative to
// the drift). The electron and the positron of a point share its position, and with transverse
// Gaussian weights w = w0 exp(-r_perp^2 / (2 sigma^2)) about the box axis. All random numbers and
// the derived positions and momenta are computed in FP64 and rounded once.
// ---------------------------------------------------------------------------------------------
struct BeamDev {
  int ppc, lx, ly, lz;
  double u0, w0, jitter, u_th, sigma_perp;
  uint32_t k0, k1;
};

__device__ __forceinline__ double u01(uint32_t r) { return ((double)r + 0.5) * (1.0 / 4294967296.0); }

template <typename T>
__global__ void k_init_beam(const __grid_constant__ RunDev<T> r, BeamDev b, long long npoints) {
  long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= npoints) return;
  const long long nxy = (long long)r.nx * r.ny;
  long long cell = p / b.ppc;
  int l = (int)(p - cell * b.ppc);
  int i = (int)(cell % r.nx), j = (int)((cell / r.nx) % r.ny), k = (int)(cell / nxy);
  int lx = l % b.lx, ly = (l / b.lx) % b.ly, lz = l / (b.lx * b.ly);
  u32x4 c = {{(uint32_t)((unsigned long long)p & 0xffffffffu), (uint32_t)((unsigned long long)p >> 32), 0u, 0u}};
  u32x4 rr = philox10(c, b.k0, b.k1);
  double ox = (lx + 0.5) / b.lx + b.jitter * (2.0 * u01(rr.v[0]) - 1.0);
  double oy = r.ndim == 3 ? (ly + 0.5) / b.ly + b.jitter * (2.0 * u01(rr.v[1]) - 1.0) : 0.0;
  double oz = (lz + 0.5) / b.lz + b.jitter * (2.0 * u01(rr.v[2]) - 1.0);
  double w = b.w0;
  if (b.sigma_perp > 0) {
    double X = i + ox, Y = r.ndim == 3 ? j + oy : 0.0;
    X = X - r.nx * floor(X / r.nx);
    if (r.ndim == 3) Y = Y - r.ny * floor(Y / r.ny);
    double rx = X - 0.5 * r.nx, ry = r.ndim == 3 ? Y - 0.5 * r.ny : 0.0;
    w = b.w0 * exp(-(rx * rx + ry * ry) / (2.0 * b.sigma_perp * b.sigma_perp));
  }
  // fold in FP64, then round the offsets
  double fxd = floor(ox), fyd = floor(oy), fzd = floor(oz);
  int ci = wrapi(i + (int)fxd, r.nx), cj = r.ndim == 3 ? wrapi(j + (int)fyd, r.ny) : 0, ck = wrapi(k + (int)fzd, r.nz);
  T tox = (T)(ox - fxd), toy = (T)(oy - fyd), toz = (T)(oz - fzd);
  if (tox >= T(1)) { tox = T(0); ci = wrapi(ci + 1, r.nx); }
  if (r.ndim == 3 && toy >= T(1)) { toy = T(0); cj = wrapi(cj + 1, r.ny); }
  if (toz >= T(1)) { toz = T(0); ck = wrapi(ck + 1, r.nz); }
  long long dcell = (long long)ck * nxy + (long long)cj * r.nx + ci;
  const double two_pi = 6.283185307179586476925286766559;
  for (int s = 0; s < 2; ++s) {
    c.v[2] = (uint32_t)(1 + s);
    u32x4 t = philox10(c, b.k0, b.k1);
    double ra = sqrt(-2.0 * log(u01(t.v[0]))), ta = two_pi * u01(t.v[1]);
    double rb = sqrt(-2.0 * log(u01(t.v[2]))), tb = two_pi * u01(t.v[3]);
    T ux = (T)(b.u_th * ra * cos(ta));
    T uy = (T)(b.u_th * ra * sin(ta));
    T uz = (T)(b.u_th * rb * cos(tb));
    insert_particle(r, s, dcell, tox, toy, toz, ux, uy, uz, (T)w, (unsigned)(p * 2 + s));
  }
}

template <typename T>
cudaError_t launch_init_beam(const RunDev<T>& r, int ppc, const int lat[3], double u0, double w0, double jitter,
                             double u_th, double sigma_perp, unsigned long long seed, cudaStream_t st) {
  BeamDev b;
  b.ppc = ppc;
  b.lx = lat[0];
  b.ly = lat[1];
  b.lz = lat[2];
  b.u0 = u0;
  b.w0 = w0;
  b.jitter = jitter;
  b.u_th = u_th;
  b.sigma_perp = sigma_perp;
  b.k0 = (uint32_t)(seed & 0xffffffffull);
  b.k1 = (uint32_t)(seed >> 32);
  long long np = r.ncell * ppc;
  int threads = 256;
  long long blocks = (np + threads - 1) / threads;
  if (blocks > 0) k_init_beam<T><<<(unsigned)blocks, threads, 0, st>>>(r, b, np);
  return cudaGetLastError();
}
template cudaError_t launch_init_beam<float>(const RunDev<float>&, int, const int*, double, double, double, double,
                                             double, unsigned long long, cudaStream_t);
template cudaError_t launch_init_beam<double>(const RunDev<double>&, int, const int*, double, double, double, double,
                                              double, unsigned long long, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Import: flat particle arrays (device) -> cell bins of the input buffers.
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void k_import(const __grid_constant__ RunDev<T> r, const __grid_constant__ FlatDev<T> f) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  bool valid = p < f.np;
  int s = 0;
  long long cell = 0;
  T ox = T(0), oy = T(0), oz = T(0);
  if (valid) {
    s = f.species[p];
    cell = f.cell[p];
    ox = f.ox[p];
    if (r.ndim == 3 && f.oy) oy = f.oy[p];
    oz = f.oz[p];
    const T lim = T(1 << 20);
    if ((s != 0 && s != 1) || cell < 0 || cell >= r.ncell ||
        !(ox > -lim && ox < lim && oy > -lim && oy < lim && oz > -lim && oz < lim)) {
      flag_error(r.err, ERR_IMPORT);
      valid = false;
    }
  }
  int key = -1 - lane;  // unique per lane when there is nothing to insert
  if (valid) {
    const long long nxy = (long long)r.nx * r.ny;
    int i = (int)(cell % r.nx), j = (int)((cell / r.nx) % r.ny), k = (int)(cell / nxy);
    fold(i, ox, r.nx);
    if (r.ndim == 3) fold(j, oy, r.ny);
    fold(k, oz, r.nz);
    cell = (long long)k * nxy + (long long)j * r.nx + i;
    key = (int)(cell * 2 + s);  // cells < 2^30
  }
  // neighbouring particles mostly share a cell (a saved state lists them by cell): one reservation for
  // the lanes of a cell and species (one atomic per particle took 262 us for 16.8M particles)
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int leader = __ffs(peers) - 1;
  const SpeciesBuf<T>& b = s ? r.in[1] : r.in[0];
  int j0 = 0;
  if (valid && lane == leader) j0 = atomicAdd(b.cnt + cell, __popc(peers));
  j0 = __shfl_sync(0xffffffffu, j0, leader) + __popc(peers & ((1u << lane) - 1u));
  if (!valid) return;
  const T w = f.w ? f.w[p] : r.wconst;
  insert_at(r, b, s, cell, j0, ox, oy, oz, f.dux[p], f.duy[p], f.duz[p], w, f.id ? f.id[p] : (unsigned)p);
}

template <typename T>
cudaError_t launch_import(const RunDev<T>& r, const FlatDev<T>& f, cudaStream_t st) {
  if (f.np <= 0) return cudaSuccess;
  int threads = 256;
  long long blocks = (f.np + threads - 1) / threads;
  k_import<T><<<(unsigned)blocks, threads, 0, st>>>(r, f);
  return cudaGetLastError();
}
template cudaError_t launch_import<float>(const RunDev<float>&, const FlatDev<float>&, cudaStream_t);
template cudaError_t launch_import<double>(const RunDev<double>&, const FlatDev<double>&, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Export: bins -> flat arrays, species 0 first, cells in order. One block per 256 cells and species:
// `bsum` holds the species' particles before each block's cells and `total` the species' numbers
// (launch_count_prefix); the block scans its own cells' counts and copies its particles in flat order, so
// the stores of every array are contiguous. Arrays that the caller does not want are null.
// ---------------------------------------------------------------------------------------------
constexpr int PFX = 256;  // cells per block

// Exclusive scan of v over the block's 256 threads; *sum: the total.
__device__ __forceinline__ int block_scan(int v, int* sum) {
  __shared__ int ws[PFX / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int q = 0; q < PFX / 32; ++q) {
    if (q < w) before += ws[q];
    all += ws[q];
  }
  *sum = all;
  return before + x - v;
}

template <typename T>
__global__ void __launch_bounds__(PFX) k_export(const __grid_constant__ RunDev<T> r, const long long* __restrict__ bsum,
                                                long long nb, const long long* __restrict__ total,
                                                const __grid_constant__ FlatDev<T> f) {
  __shared__ int first[PFX];
  const int s = blockIdx.y;
  const SpeciesBuf<T>& b = s ? r.in[1] : r.in[0];  // constant indices: no local copy of r
  const long long cell0 = blockIdx.x * (long long)PFX, c = cell0 + threadIdx.x;
  int n;
  first[threadIdx.x] = block_scan(c < r.ncell ? min(b.cnt[c], r.cap) : 0, &n);
  __syncthreads();
  const long long base = bsum[s * nb + blockIdx.x] + (s ? total[0] : 0);
  for (int q = threadIdx.x; q < n; q += PFX) {
    int lo = 0;  // the last cell whose first particle is at or before q
#pragma unroll
    for (int h = PFX / 2; h > 0; h >>= 1)
      if (first[lo + h] <= q) lo += h;
    const long long src = (cell0 + lo) * r.cap + (q - first[lo]), d = base + q;
    if (d >= f.np) return;
    const PartVals<T> v = part_get(b, r.ndim, src);
    if (f.cell) f.cell[d] = (int)(cell0 + lo);
    if (f.species) f.species[d] = s;
    if (f.ox) f.ox[d] = v.ox;
    if (f.oy) f.oy[d] = v.oy;
    if (f.oz) f.oz[d] = v.oz;
    if (f.dux) f.dux[d] = v.ux;
    if (f.duy) f.duy[d] = v.uy;
    if (f.duz) f.duz[d] = v.uz;
    if (f.w) f.w[d] = b.w ? b.w[src] : r.wconst;
    if (f.id) f.id[d] = b.id ? b.id[src] : 0u;
  }
}

template <typename T>
cudaError_t launch_export(const RunDev<T>& r, const long long* bsum, const long long* total, const FlatDev<T>& f,
                          cudaStream_t st) {
  const long long nb = count_prefix_blocks(r.ncell);
  if (nb > 0) k_export<T><<<dim3((unsigned)nb, 2), PFX, 0, st>>>(r, bsum, nb, total, f);
  return cudaGetLastError();
}
template cudaError_t launch_export<float>(const RunDev<float>&, const long long*, const long long*,
                                          const FlatDev<float>&, cudaStream_t);
template cudaError_t launch_export<double>(const RunDev<double>&, const long long*, const long long*,
                                           const FlatDev<double>&, cudaStream_t);

// Spill list entries [0, n) -> flat arrays at [base, base + n) (cell and species from the key).
template <typename T>
__global__ void k_spill_export(const __grid_constant__ RunDev<T> r, long long n, long long base,
                               const __grid_constant__ FlatDev<T> f) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n || base + i >= f.np) return;
  const long long d = base + i;
  const int key = r.sp.key[i];
  f.cell[d] = key >> 1;
  f.species[d] = key & 1;
  f.ox[d] = r.sp.ox[i];
  if (f.oy) f.oy[d] = r.ndim == 3 ? r.sp.oy[i] : T(0);
  f.oz[d] = r.sp.oz[i];
  f.dux[d] = r.sp.dux[i];
  f.duy[d] = r.sp.duy[i];
  f.duz[d] = r.sp.duz[i];
  if (f.w) f.w[d] = r.sp.w ? r.sp.w[i] : r.wconst;
  if (f.id) f.id[d] = r.sp.id ? r.sp.id[i] : 0u;
}

template <typename T>
cudaError_t launch_spill_export(const RunDev<T>& r, long long n, long long base, const FlatDev<T>& f,
                                cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_spill_export<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(r, n, base, f);
  return cudaGetLastError();
}
template cudaError_t launch_spill_export<float>(const RunDev<float>&, long long, long long, const FlatDev<float>&,
                                                cudaStream_t);
template cudaError_t launch_spill_export<double>(const RunDev<double>&, long long, long long,
                                                 const FlatDev<double>&, cudaStream_t);

// Largest insertion count over the cells of two count arrays (counts keep every insertion, the
// spilled ones too) into *out, which the caller zeroes.
__global__ void k_max_count(const int* __restrict__ c0, const int* __restrict__ c1, long long ncell, int* out) {
  int m = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell; c += (long long)gridDim.x * blockDim.x)
    m = max(m, max(c0[c], c1[c]));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

cudaError_t launch_max_count(const int* c0, const int* c1, long long ncell, int* out, cudaStream_t st) {
  if (ncell <= 0) return cudaSuccess;
  long long blocks = (ncell + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_max_count<<<(unsigned)blocks, 256, 0, st>>>(c0, c1, ncell, out);
  return cudaGetLastError();
}

// Exclusive prefix of min(cnt, cap) over blocks of 256 cells, both species: block sums, then one block per
// species scans them, 1024 threads over contiguous runs (one thread walking them took 0.8 ms on 32768
// blocks).
__global__ void __launch_bounds__(PFX) k_count_blocks(const int* __restrict__ c0, const int* __restrict__ c1,
                                                      long long ncell, int cap, long long* bsum) {
  __shared__ int ws[PFX / 32];
  const int* cnt = blockIdx.y ? c1 : c0;
  const long long c = blockIdx.x * (long long)PFX + threadIdx.x;
  const int t = __reduce_add_sync(0xffffffffu, c < ncell ? min(cnt[c], cap) : 0);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long a = 0;
    for (int w = 0; w < PFX / 32; ++w) a += ws[w];
    bsum[blockIdx.y * (long long)gridDim.x + blockIdx.x] = a;
  }
}

__global__ void __launch_bounds__(1024) k_scan_blocks(long long* bsum, long long nb, long long* total) {
  __shared__ long long ws[32];
  long long* v = bsum + blockIdx.x * nb;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long per = (nb + 1023) / 1024, b0 = min(threadIdx.x * per, nb), b1 = min(b0 + per, nb);
  long long sum = 0;
  for (long long b = b0; b < b1; ++b) sum += v[b];
  long long x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  long long acc = x - sum;
  for (int q = 0; q < w; ++q) acc += ws[q];
  if (threadIdx.x == 1023) total[blockIdx.x] = acc + sum;
  for (long long b = b0; b < b1; ++b) {
    const long long t = v[b];
    v[b] = acc;
    acc += t;
  }
}

cudaError_t launch_count_prefix(const int* c0, const int* c1, long long ncell, int cap, long long* bsum,
                                long long* total, cudaStream_t st) {
  const long long nb = count_prefix_blocks(ncell);
  if (nb == 0) return cudaSuccess;
  k_count_blocks<<<dim3((unsigned)nb, 2), PFX, 0, st>>>(c0, c1, ncell, cap, bsum);
  k_scan_blocks<<<2, 1024, 0, st>>>(bsum, nb, total);
  return cudaGetLastError();
}

long long count_prefix_blocks(long long ncell) { return (ncell + PFX - 1) / PFX; }

}  // namespace picgb
