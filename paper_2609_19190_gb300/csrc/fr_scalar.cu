// fr_scalar.cu -- scalar extraction: the 93 features of the whole VOI (the
// paper's other extraction mode, "Software design and extraction modes"; a
// map value equals it wherever the window covers the VOI).
//
// The whole VOI is one region, so the work is a set of grid-wide counts
// instead of per-voxel windows: histograms, co-occurrence and run-length
// counts per direction (privatised in shared memory where they fit), the
// 26-connected zones by a lock-free union-find over the volume, zone (level,
// size) pairs in an open-addressing hash table.  Counts are exact integers;
// the features are then taken in FP64 by a few small kernels (MCC in FP32 by
// the warp eigen-solver of the map path in shared memory), one block per direction.
#include <cfloat>
#include <climits>
#include <cstdint>

#include "fr_device.cuh"
#include "fr_internal.h"
#include "fr_voxel.cuh"

namespace fr {

constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kScThreads = 256;
constexpr int kMiscThreads = 1024;
// threads of the counting blocks that keep a private copy of the counts: the
// copies are sized by the plan's level cap (83 and 130 KB at 255 levels, two
// blocks and one an SM), so the warps in flight come from wide blocks
constexpr int kCountThreads = 1024;
// dynamic shared memory of the neighbourhood kernel, for levels 0..ngc:
// ngacc [27] u64, gldm [27] u32, hlev u32, ngn u32
static __host__ __device__ constexpr int neigh_smem(int ngc) {
  return (ngc + 1) * (27 * 8 + 27 * 4 + 4 + 4);
}

__device__ __forceinline__ bool sc_failed(const FrScalarArgs& a) {
  return *(const volatile int32_t*)&a.state->status != 0;
}

__device__ __forceinline__ void sc_zyx(const FrScalarArgs& a, int lin, int& z, int& y, int& x) {
  x = lin % a.nx;
  const int t = lin / a.nx;
  y = t % a.ny;
  z = t / a.ny;
}

// Gray level at (z, y, x); 0 outside the volume or the VOI.
__device__ __forceinline__ int sc_level(const FrScalarArgs& a, int z, int y, int x) {
  if ((unsigned)z >= (unsigned)a.nz || (unsigned)y >= (unsigned)a.ny ||
      (unsigned)x >= (unsigned)a.nx)
    return 0;
  return (int)(a.packed[((size_t)z * a.ny + y) * a.px + x] & 0xFFu);
}

// Sum over the block of K doubles (fixed order: deterministic).  sh holds
// K * 32 doubles; every thread gets the totals.
template <int K>
__device__ void block_sum(double (&v)[K], double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k * 32 + warp] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double x = lane < nw ? sh[k * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
      if (lane == 0) sh[k * 32] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = sh[k * 32];
  __syncthreads();
}

template <int K>
__device__ void block_sum_u64(unsigned long long (&v)[K], unsigned long long* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k * 32 + warp] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      unsigned long long x = lane < nw ? sh[k * 32 + lane] : 0ull;
#pragma unroll
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
      if (lane == 0) sh[k * 32] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = sh[k * 32];
  __syncthreads();
}

// Fixed-point terms for sums whose order of addition varies between runs
// (the zone table's slot order depends on thread timing): x >= 0 times 2^fb,
// truncated to an unsigned 128-bit integer.  Integer sums do not depend on
// the order of addition, so the total is the same on every run.  The caller
// keeps x < 2^(127 - fb).
__device__ __forceinline__ unsigned __int128 sc_fixed(double x, int fb) {
  if (!(x > 0.0)) return 0;
  int e;
  const double m = frexp(x, &e);  // x = m 2^e, 0.5 <= m < 1
  const unsigned long long mi = (unsigned long long)ldexp(m, 53);  // exact
  const int sh = e - 53 + fb;
  if (sh >= 0) return (unsigned __int128)mi << sh;
  if (sh <= -64) return 0;
  return (unsigned __int128)(mi >> (-sh));
}
__device__ __forceinline__ double sc_unfixed(unsigned __int128 v, int fb) {
  const double hi = (double)(unsigned long long)(v >> 64), lo = (double)(unsigned long long)v;
  return ldexp(hi, 64 - fb) + ldexp(lo, -fb);
}

// Block sum of K unsigned 128-bit integers (exact); sh holds K * 32 values.
template <int K>
__device__ void block_sum_u128(unsigned __int128 (&v)[K], unsigned __int128* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto shfl = [](unsigned __int128 x, int o) {
    const unsigned long long lo = __shfl_xor_sync(kFull, (unsigned long long)x, o);
    const unsigned long long hi = __shfl_xor_sync(kFull, (unsigned long long)(x >> 64), o);
    return ((unsigned __int128)hi << 64) | lo;
  };
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] += shfl(v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k * 32 + warp] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      unsigned __int128 x = lane < nw ? sh[k * 32 + lane] : (unsigned __int128)0;
#pragma unroll
      for (int o = 16; o; o >>= 1) x += shfl(x, o);
      if (lane == 0) sh[k * 32] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = sh[k * 32];
  __syncthreads();
}

__device__ __forceinline__ double sc_ent(double p) { return p > 0.0 ? -p * log2(p) : 0.0; }
__device__ __forceinline__ double sc_div(double a, double b) {
  return b == 0.0 ? __longlong_as_double(0x7ff8000000000000ll) : a / b;
}

// ---------------------------------------------------------------- counting

// The union-find forest starts as runs along x: each voxel points up to eight
// voxels back along its run (a bounded walk; finds follow the steps), so the
// unions below have one per pair of touching runs left to make.
__global__ void sc_init_kernel(const __grid_constant__ FrScalarArgs a) {
  if (sc_failed(a)) return;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int lin = a.voi[k];
    int z, y, x;
    sc_zyx(a, lin, z, y, x);
    const int g = sc_level(a, z, y, x);
    int back = 0;
    while (back < 8 && sc_level(a, z, y, x - back - 1) == g) ++back;
    a.parent[lin] = lin - back;
  }
}

// Per VOI voxel: raw / level histograms, GLDM dependence (equal 26-neighbours),
// NGTDM n_i and |i k - sum|, and the zone unions with the 13 forward
// neighbours of equal level.  Bound by the latency of the neighbour reads and
// of the unions; a block clears and adds only the levels in use (200k voxels, from
// single-voxel trees and a union per pair: 288 us; from runs along x, a union per
// pair of runs: 227 us).
__global__ void __launch_bounds__(kCountThreads) sc_neigh_kernel(const __grid_constant__ FrScalarArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int rows = sc_failed(a) ? 0 : a.state->ng + 1, cells = rows * 27;
  unsigned long long* s_acc = (unsigned long long*)sm;  // [rows][27]
  uint32_t* s_gldm = (uint32_t*)(s_acc + cells);        // [rows][27]
  uint32_t* s_hlev = s_gldm + cells;                    // [rows]
  uint32_t* s_ngn = s_hlev + rows;                      // [rows]
  for (int i = threadIdx.x; i < cells; i += blockDim.x) {
    s_acc[i] = 0ull;
    s_gldm[i] = 0u;
  }
  for (int i = threadIdx.x; i < rows; i += blockDim.x) s_hlev[i] = s_ngn[i] = 0u;
  __syncthreads();
  if (!sc_failed(a)) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
         k += (int64_t)gridDim.x * blockDim.x) {
      const int lin = a.voi[k];
      int z, y, x;
      sc_zyx(a, lin, z, y, x);
      const uint32_t w = a.packed[((size_t)z * a.ny + y) * a.px + x];
      const int g = (int)(w & 0xFFu);
      const int raw = (int)(w >> 8) - 32768;
      atomicAdd(&a.hraw[raw + 32768], 1u);
      atomicAdd(&s_hlev[g], 1u);
      int cnt = 0, sum = 0, eq = 0;
      const bool left = sc_level(a, z, y, x - 1) == g;
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
          const bool ahead = dz > 0 || (dz == 0 && dy > 0);
          bool before = false;  // the neighbour to the left of the next one is of level g
          for (int dx = -1; dx <= 1; ++dx) {
            if (!dz && !dy && !dx) continue;
            const int b = sc_level(a, z + dz, y + dy, x + dx);
            const bool same = b == g;
            if (b) {
              ++cnt;
              sum += b;
              eq += same;
            }
            // two runs along x are joined where the pair one step to the left
            // is not of the level, not at every pair
            if (ahead && same) {
              if (dx < 0) before = left && sc_level(a, z + dz, y + dy, x - 2) == g;
              if (!(left && before))
                uf_unite(a.parent, lin, ((z + dz) * a.ny + (y + dy)) * a.nx + (x + dx));
            }
            before = same;
          }
        }
      atomicAdd(&s_gldm[g * 27 + eq], 1u);
      if (cnt) {
        atomicAdd(&s_ngn[g], 1u);
        const int dev = g * cnt - sum;
        atomicAdd(&s_acc[g * 27 + cnt], (unsigned long long)(dev < 0 ? -dev : dev));
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cells; i += blockDim.x) {
    if (s_acc[i]) atomicAdd(&a.ngacc[i], s_acc[i]);
    if (s_gldm[i]) atomicAdd(&a.gldm[i], s_gldm[i]);
  }
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    if (s_hlev[i]) atomicAdd(&a.hlev[i], s_hlev[i]);
    if (s_ngn[i]) atomicAdd(&a.ngn[i], s_ngn[i]);
  }
}

// Co-occurrence pairs (u, u + delta d) of direction blockIdx.y, as packed
// upper-triangle counts over levels (a shared-memory copy per block).
__global__ void __launch_bounds__(kCountThreads) sc_glcm_kernel(const __grid_constant__ FrScalarArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  if (sc_failed(a)) return;
  uint32_t* s = (uint32_t*)sm;
  // the levels in use fill the leading triangle of the block's copy
  const int ng = a.state->ng, np = ng * (ng + 1) / 2, ngc = a.ngc, d = blockIdx.y;
  for (int i = threadIdx.x; i < np; i += blockDim.x) s[i] = 0u;
  __syncthreads();
  const int oz = c_dirs[d][0] * a.delta, oy = c_dirs[d][1] * a.delta, ox = c_dirs[d][2] * a.delta;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
       k += (int64_t)gridDim.x * blockDim.x) {
    int z, y, x;
    sc_zyx(a, a.voi[k], z, y, x);
    const int g = sc_level(a, z, y, x);
    const int b = sc_level(a, z + oz, y + oy, x + ox);
    if (!b) continue;
    atomicAdd(&s[pk(ng, min(g, b) - 1, max(g, b) - 1)], 1u);
  }
  __syncthreads();
  uint32_t* dst = a.glcm + (size_t)d * (ngc * (ngc + 1) / 2);
  for (int t = threadIdx.x; t < ng * ng; t += blockDim.x) {
    const int i = t / ng, j = t - i * ng;
    if (j < i) continue;
    const uint32_t c = s[pk(ng, i, j)];
    if (c) atomicAdd(&dst[pk(ngc, i, j)], c);
  }
}

// Runs of direction blockIdx.y: a voxel whose predecessor (u - d) is not of
// its level starts a run, measured by walking forward.
__global__ void __launch_bounds__(kScThreads) sc_glrlm_kernel(const __grid_constant__ FrScalarArgs a) {
  if (sc_failed(a)) return;
  const int d = blockIdx.y;
  const int dz = c_dirs[d][0], dy = c_dirs[d][1], dx = c_dirs[d][2];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
       k += (int64_t)gridDim.x * blockDim.x) {
    int z, y, x;
    sc_zyx(a, a.voi[k], z, y, x);
    const int g = sc_level(a, z, y, x);
    if (sc_level(a, z - dz, y - dy, x - dx) == g) continue;
    int len = 1, zz = z + dz, yy = y + dy, xx = x + dx;
    while (sc_level(a, zz, yy, xx) == g) {
      ++len;
      zz += dz;
      yy += dy;
      xx += dx;
    }
    atomicAdd(&a.glrlm[((size_t)d * a.ngc + (g - 1)) * a.lmax + (len - 1)], 1u);
  }
}

// Zone size at each root (the unions are complete).
__global__ void sc_flatten_kernel(const __grid_constant__ FrScalarArgs a) {
  if (sc_failed(a)) return;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int r = uf_find((volatile int*)a.parent, a.voi[k]);
    atomicAdd(&a.zsize[r], 1);
  }
}

// 64-bit mix (MurmurHash3's finaliser) for the zone-key table.
__device__ __forceinline__ unsigned long long sc_mix(unsigned long long k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

// One entry per zone (at its root): zones per level, per size, and per
// (level, size) in the hash table (linear probing; at least half empty).
__global__ void sc_zone_kernel(const __grid_constant__ FrScalarArgs a) {
  if (sc_failed(a)) return;
  const unsigned long long mask = (unsigned long long)a.hcap - 1ull;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n_voi;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int lin = a.voi[k];
    if (a.parent[lin] != lin) continue;
    int z, y, x;
    sc_zyx(a, lin, z, y, x);
    const int g = sc_level(a, z, y, x);
    const int size = a.zsize[lin];
    atomicAdd(&a.zrow[g], 1u);
    atomicAdd(&a.zcol[size], 1u);
    const unsigned long long key = ((unsigned long long)g << 32) | (unsigned)size;
    unsigned long long slot = sc_mix(key) & mask;
    for (int64_t probe = 0; probe < a.hcap; ++probe) {
      const unsigned long long prev = atomicCAS(&a.hkey[slot], kEmptyKey, key);
      if (prev == kEmptyKey || prev == key) {
        atomicAdd(&a.hcnt[slot], 1u);
        break;
      }
      slot = (slot + 1ull) & mask;
    }
  }
}

// ---------------------------------------------------------------- features

// (1 + d) ln(1 + d) - d >= 0 for d >= -1 (the value at -1 is 1).
__device__ __forceinline__ double sc_bregman(double d) {
  if (d <= -1.0) return 1.0;
  if (fabs(d) < 1e-3) return d * d * (0.5 + d * (-1.0 / 6.0 + d * (1.0 / 12.0 + d * (-1.0 / 20.0))));
  return (1.0 + d) * log1p(d) - d;
}

// The t-th cell (i <= j) of the upper triangle of n levels, rows r and
// n - 1 - r side by side: t < (n + 1) / 2 * (n + 1); false for the middle
// row's second half (n odd).
__device__ __forceinline__ bool sc_cell(int t, int n, int& i, int& j) {
  const int r = t / (n + 1), c = t - r * (n + 1);
  if (c < n - r) {
    i = r;
    j = r + c;
    return true;
  }
  i = n - 1 - r;
  j = i + c - (n - r);
  return i > r;
}

// GLCM features of direction blockIdx.x (or of the merged matrix), written to
// dirf[blockIdx.x][0..23] (and the IBSI sum variance and dissimilarity at
// [40..41]).  Counts C(i, j): n for i != j, 2n on the diagonal.
//
// Bound by the FP64 pipe (one warp instruction in 16 cycles of an SM) and by
// chains of dependent FP64 instructions: what depends on |i - j| or i + j
// alone is taken from the difference and sum bins (ng and 2 ng terms instead
// of ng^2), sums of integers stay integers, a cell of the triangle stands for
// both entries, and one warp solves the MCC in shared memory meanwhile.
// 200k voxels, FBW 25: 1147 -> 195 us, now one warp's solve (its
// cells in eight blocks a direction: 218 us).
__global__ void __launch_bounds__(kScThreads) sc_glcm_feat_kernel(const __grid_constant__ FrScalarArgs a) {
  __shared__ unsigned long long s_marg[256];
  __shared__ unsigned long long s_sbin[512];
  __shared__ unsigned long long s_dbin[256];
  __shared__ double s_rs[256];
  __shared__ double s_red[15 * 32];
  __shared__ unsigned long long s_ured[32];
  // the solve: 64 rows, then a tridiagonal and factors of up to 255
  __shared__ float4 s_room[(64 * 64 * 4 + 256 * 24) / 16];
  __shared__ unsigned long long s_max;
  __shared__ int s_present;
  __shared__ float s_mcc;
  const int d = blockIdx.x, tid = threadIdx.x;
  double* f = a.dirf + d * kScalarDirF;
  const double kNaN = __longlong_as_double(0x7ff8000000000000ll);
  if (sc_failed(a)) {
    if (tid < 24) f[tid] = kNaN;
    if (tid < 2) f[40 + tid] = kNaN;
    return;
  }
  const bool merged = a.agg == 1;
  const int ng = a.state->ng, ngc = a.ngc, np = ngc * (ngc + 1) / 2;
  auto cnt = [&](int i, int j) -> unsigned long long {  // pair count, 0-based levels i <= j
    const size_t t = (size_t)pk(ngc, i, j);
    if (!merged) return a.glcm[(size_t)d * np + t];
    unsigned long long s = 0;
#pragma unroll
    for (int q = 0; q < kNumDirs; ++q) s += a.glcm[(size_t)q * np + t];
    return s;
  };
  for (int i = tid; i < 512; i += blockDim.x) s_sbin[i] = 0ull;
  for (int i = tid; i < 256; i += blockDim.x) s_dbin[i] = s_marg[i] = 0ull;
  if (tid == 0) {
    s_max = 0ull;
    s_present = 0;
    s_mcc = 0.f;
  }
  __syncthreads();
  const int cells = (ng + 1) / 2 * (ng + 1);
  unsigned long long ij[1] = {0ull};  // sum of (i + 1)(j + 1) C
  {
    unsigned long long mx = 0ull;
    for (int t = tid; t < cells; t += blockDim.x) {
      int i, j;
      if (!sc_cell(t, ng, i, j)) continue;
      const unsigned long long n = cnt(i, j);
      if (!n) continue;
      const unsigned long long C = i == j ? 2ull * n : n;
      atomicAdd(&s_marg[i], C);
      if (i != j) atomicAdd(&s_marg[j], C);
      atomicAdd(&s_sbin[i + j + 2], 2ull * n);
      atomicAdd(&s_dbin[j - i], 2ull * n);
      ij[0] += 2ull * n * (unsigned)((i + 1) * (j + 1));
      mx = max(mx, C);
    }
    if (mx) atomicMax(&s_max, mx);
  }
  block_sum_u64<1>(ij, s_ured);
  unsigned long long T = 0;
  for (int i = 0; i < ng; ++i) T += s_marg[i];
  if (T == 0) {
    if (tid < 24) f[tid] = kNaN;
    if (tid < 2) f[40 + tid] = kNaN;
    return;
  }
  const double dT = (double)T, iT = 1.0 / dT;
  double u[4] = {0.0, 0.0, 0.0, 0.0};  // mean, HX, difference average, sum average
  for (int i = tid; i < 2 * ng + 1; i += blockDim.x) {
    if (i < ng) {
      const unsigned long long mi = s_marg[i];
      s_rs[i] = mi ? 1.0 / sqrt((double)mi) : 0.0;
      if (mi) atomicAdd(&s_present, 1);
      const double p = (double)mi / dT;
      u[0] += (i + 1) * p;
      u[1] += sc_ent(p);
      u[2] += i * ((double)s_dbin[i] / dT);
    }
    u[3] += i * ((double)s_sbin[i] / dT);
  }
  block_sum<4>(u, s_red);
  const double mu = u[0], hx = u[1], da = u[2], sa = u[3];
  // MCC: spectral radius of S - u u^T over the levels (absent levels: zero rows)
  float* S = a.mcc_s + (size_t)d * ngc * ngc;
  for (int t = tid; t < cells; t += blockDim.x) {
    int i, j;
    if (!sc_cell(t, ng, i, j)) continue;
    const unsigned long long mi = s_marg[i], mj = s_marg[j];
    const unsigned long long C = (i == j ? 2ull : 1ull) * cnt(i, j);
    const long long num = (long long)C * (long long)T - (long long)(mi * mj);
    const float val = (float)((double)num * (s_rs[i] * s_rs[j]) * iT);
    S[(size_t)i * ngc + j] = val;
    S[(size_t)j * ngc + i] = val;
  }
  __syncthreads();
  double v[15];
  for (int k = 0; k < 15; ++k) v[k] = 0.0;
  if (tid < 32) {
    if (s_present >= 2) {
      const float mcc = warp_rho(S, ngc, ng, nullptr, 0.f, (char*)s_room, (int)sizeof(s_room));
      if (tid == 0) s_mcc = mcc;
    }
  } else {
    for (int t = tid - 32; t < cells; t += blockDim.x - 32) {
      int i, j;
      if (!sc_cell(t, ng, i, j)) continue;
      const unsigned long long mi = s_marg[i], mj = s_marg[j];
      if (!mi || !mj) continue;
      const double w = i == j ? 1.0 : 2.0;
      const unsigned long long C = (i == j ? 2ull : 1ull) * cnt(i, j);
      // mutual information, nats: sum of q g(p / q - 1) >= 0 over all present pairs
      const long long num = (long long)C * (long long)T - (long long)(mi * mj);
      const double mm = (double)mi * (double)mj;
      v[0] += w * (mm * (iT * iT)) * sc_bregman((double)num / mm);
      if (!C) continue;
      const double p = (double)C / dT;
      v[1] += w * (p * p);       // joint energy
      v[2] += w * sc_ent(p);     // joint entropy
    }
    const double ngd = (double)ng;
    for (int k = tid - 32; k < 2 * ng + 1; k += blockDim.x - 32) {
      if (k < ng) {
        v[3] += ((k + 1) - mu) * ((k + 1) - mu) * ((double)s_marg[k] / dT);  // sum of squares
        const unsigned long long c = s_dbin[k];
        if (c) {
          const double p = (double)c / dT, dd = k;
          v[4] += dd * dd * p;                          // contrast
          v[5] += p / (1.0 + dd * dd);                  // Idm
          v[6] += p / (1.0 + dd * dd / (ngd * ngd));    // Idmn
          v[7] += p / (1.0 + dd);                       // Id
          v[8] += p / (1.0 + dd / ngd);                 // Idn
          if (k) v[9] += p / (dd * dd);                 // inverse variance
          v[10] += sc_ent(p);                           // difference entropy
          v[11] += (dd - da) * (dd - da) * p;           // difference variance
        }
      }
      const unsigned long long c = s_sbin[k];
      if (c) {
        const double p = (double)c / dT, tt = k - 2.0 * mu, t2 = tt * tt;
        v[12] += t2 * t2 * p;  // cluster prominence
        v[13] += t2 * tt * p;  // cluster shade
        v[14] += t2 * p;       // cluster tendency
      }
    }
  }
  // (the bin 2 ng of the sums is the last: two levels ng)
  block_sum<15>(v, s_red);
  double e[2] = {0.0, 0.0};  // sum entropy, sum variance
  for (int k = tid; k < 2 * ng + 1; k += blockDim.x) {
    const double p = (double)s_sbin[k] / dT;
    e[0] += sc_ent(p);
    e[1] += (k - sa) * (k - sa) * p;
  }
  block_sum<2>(e, s_red);
  if (tid == 0) {
    f[40] = e[1];
    f[41] = da;
    const double mi_bits = v[0] * 1.4426950408889634, ac = (double)ij[0] / dT;
    f[0] = ac;
    f[1] = mu;
    f[2] = v[12];
    f[3] = v[13];
    f[4] = v[14];
    f[5] = v[4];
    f[6] = sc_div(ac - mu * mu, v[3]);
    f[7] = da;
    f[8] = v[10];
    f[9] = v[11];
    f[10] = v[1];
    f[11] = v[2];
    f[12] = sc_div(-mi_bits, hx);
    f[13] = sqrt(fmax(0.0, -expm1(-2.0 * mi_bits)));
    f[14] = v[5];
    f[15] = v[6];
    f[16] = v[7];
    f[17] = v[8];
    f[18] = v[9];
    f[19] = (double)s_max / dT;
    f[20] = sa;
    f[21] = e[0];
    f[22] = v[3];
    f[23] = s_present >= 2 ? (double)s_mcc : kNaN;
  }
}

// The eleven sums over a (gray level I, size J) matrix's cells of share p
// (short and long, low and high emphases, variances, entropy): two
// reciprocals instead of seven divisions, which are what a cell costs.
__device__ __forceinline__ void sc_size_terms(double p, double I, double J, double mui, double muj,
                                              double (&v)[11]) {
  const double i2 = I * I, j2 = J * J, ri = 1.0 / i2, rj = 1.0 / j2, pi = p * i2, qi = p * ri;
  v[0] += p * rj;
  v[1] += p * j2;
  v[2] += (I - mui) * (I - mui) * p;
  v[3] += (J - muj) * (J - muj) * p;
  v[4] += sc_ent(p);
  v[5] += qi;
  v[6] += pi;
  v[7] += qi * rj;
  v[8] += pi * rj;
  v[9] += qi * j2;
  v[10] += pi * j2;
}

// GLRLM features of direction blockIdx.x (or of the merged matrix), written to
// dirf[blockIdx.x][24..39].
__global__ void __launch_bounds__(kScThreads) sc_glrlm_feat_kernel(const __grid_constant__ FrScalarArgs a) {
  __shared__ double s_red[13 * 32];
  __shared__ unsigned long long s_ured[3 * 32];
  const int d = blockIdx.x, tid = threadIdx.x;
  double* f = a.dirf + d * kScalarDirF + 24;
  const double kNaN = __longlong_as_double(0x7ff8000000000000ll);
  if (sc_failed(a)) {
    if (tid < 16) f[tid] = kNaN;
    return;
  }
  const bool merged = a.agg == 1;
  const int ng = a.state->ng, L = a.lmax;
  auto R = [&](int i, int l) -> unsigned long long {
    if (!merged) return a.glrlm[((size_t)d * a.ngc + i) * L + l];
    unsigned long long s = 0;
    for (int q = 0; q < kNumDirs; ++q) s += a.glrlm[((size_t)q * a.ngc + i) * L + l];
    return s;
  };
  // totals, row and column sums of squares: a warp per level, a thread per length
  unsigned long long u[3] = {0ull, 0ull, 0ull};  // N, sum_i rows^2, sum_l cols^2
  for (int i = tid >> 5; i < ng; i += blockDim.x >> 5) {
    unsigned long long r = 0;
    for (int l = tid & 31; l < L; l += 32) r += R(i, l);
#pragma unroll
    for (int o = 16; o; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
    if ((tid & 31) == 0) {
      u[0] += r;
      u[1] += r * r;
    }
  }
  for (int l = tid; l < L; l += blockDim.x) {
    unsigned long long c = 0;
#pragma unroll 8
    for (int i = 0; i < ng; ++i) c += R(i, l);
    u[2] += c * c;
  }
  block_sum_u64<3>(u, s_ured);
  if (u[0] == 0) {
    if (tid < 16) f[tid] = kNaN;
    return;
  }
  const double N = (double)u[0];
  double m[2] = {0.0, 0.0};
  for (int t = tid; t < ng * L; t += blockDim.x) {
    const int i = t / L, l = t - i * L;
    const unsigned long long c = R(i, l);
    if (!c) continue;
    m[0] += (i + 1) * (double)c;
    m[1] += (l + 1) * (double)c;
  }
  block_sum<2>(m, s_red);
  const double mui = m[0] / N, muj = m[1] / N;
  double v[11];
  for (int k = 0; k < 11; ++k) v[k] = 0.0;
  for (int t = tid; t < ng * L; t += blockDim.x) {
    const int i = t / L, l = t - i * L;
    const unsigned long long c = R(i, l);
    if (!c) continue;
    const double p = (double)c / N, I = i + 1, J = l + 1;
    sc_size_terms(p, I, J, mui, muj, v);
  }
  block_sum<11>(v, s_red);
  if (tid == 0) {
    const double nv = (double)a.n_voi * (merged ? kNumDirs : 1);
    f[0] = v[0];
    f[1] = v[1];
    f[2] = (double)u[1] / N;
    f[3] = (double)u[1] / (N * N);
    f[4] = (double)u[2] / N;
    f[5] = (double)u[2] / (N * N);
    f[6] = N / nv;
    f[7] = v[2];
    f[8] = v[3];
    f[9] = v[4];
    f[10] = v[5];
    f[11] = v[6];
    f[12] = v[7];
    f[13] = v[8];
    f[14] = v[9];
    f[15] = v[10];
  }
}

// First order (block 0), GLDM (block 1) and NGTDM (block 2), written to
// out[0..17], out[74..92] and their extras out[93..95], out[98..100].  Bound
// by latency and the FP64 pipe of one SM: the histogram is read in rows of the
// block (all loads of a pass in flight), and after the first pass between the
// smallest and largest intensity only.
// 200k voxels: 1250 us with the zones here, on one SM each -> 68 us.
__global__ void __launch_bounds__(kMiscThreads) sc_misc_feat_kernel(const __grid_constant__ FrScalarArgs a) {
  __shared__ double s_red[12 * 32];
  __shared__ unsigned long long s_ured[4 * 32];
  __shared__ unsigned long long s_rank[10];
  __shared__ double s_pct[5];
  __shared__ long long s_p100[5];
  __shared__ int s_val[10];
  __shared__ int s_mm[2];
  __shared__ double s_si[256];
  const int tid = threadIdx.x;
  const double kNaN = __longlong_as_double(0x7ff8000000000000ll);
  double* out = a.out;
  if (sc_failed(a)) {
    if (blockIdx.x == 0 && tid < 18) out[tid] = kNaN;
    if (blockIdx.x == 0 && tid < 3) out[kFirstExtra + tid] = kNaN;
    if (blockIdx.x == 0 && tid == 0) out[kScalarStd] = kNaN;
    if (blockIdx.x == 1 && tid < 14) out[74 + tid] = kNaN;
    if (blockIdx.x == 1 && tid < 3) out[kGldmExtra + tid] = kNaN;
    if (blockIdx.x == 2 && tid < 5) out[88 + tid] = kNaN;
    return;
  }
  const int ng = a.state->ng;
  if (blockIdx.x == 0) {
    // ---- first order from the raw histogram
    unsigned long long u[3] = {0ull, 0ull, 0ull};  // N, sum x (offset), sum x^2
    long long s1 = 0;
    int lo = INT_MAX, hi = INT_MIN;
#pragma unroll 16
    for (int b = tid; b < 65536; b += kMiscThreads) {
      const unsigned c = a.hraw[b];
      const long long xv = b - 32768;
      u[0] += c;
      s1 += (long long)c * xv;
      u[2] += (unsigned long long)c * (unsigned long long)(xv * xv);
      if (c) {
        lo = min(lo, b);
        hi = max(hi, b);
      }
    }
    u[1] = (unsigned long long)s1;  // two's complement sums add exactly
    if (tid < 2) s_mm[tid] = tid == 0 ? INT_MAX : INT_MIN;
    __syncthreads();
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if ((tid & 31) == 0) {
      atomicMin(&s_mm[0], lo);
      atomicMax(&s_mm[1], hi);
    }
    block_sum_u64<3>(u, s_ured);  // contains __syncthreads
    const unsigned long long n = u[0];
    const long long S1 = (long long)u[1];
    const unsigned long long S2 = u[2];
    lo = s_mm[0];  // bins of the smallest and largest intensity
    hi = s_mm[1];
    if (n == 0) lo = 32768, hi = 32767;  // no bins
    // order statistics at the ranks of P10, P25, P50, P75, P90 (k and k + 1)
    const int qs[5] = {10, 25, 50, 75, 90};
    if (tid < 10) {
      const unsigned long long k =
          (n - 1) * (unsigned long long)qs[tid >> 1] / 100 + (unsigned)(tid & 1);
      s_rank[tid] = min(k, n - 1);
    }
    {
      // each thread some consecutive bins, between the counts before and after
      const int per = (hi - lo + kMiscThreads) / kMiscThreads;
      const int b0 = lo + tid * per, b1 = min(b0 + per, hi + 1);
      unsigned long long own = 0;
      for (int b = b0; b < b1; ++b) own += a.hraw[b];
      unsigned long long inc = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, inc, o);
        if ((tid & 31) >= o) inc += t;
      }
      if ((tid & 31) == 31) s_ured[tid >> 5] = inc;
      __syncthreads();
      unsigned long long run = inc - own;
      for (int w = 0; w < (tid >> 5); ++w) run += s_ured[w];
      if (own)
        for (int r = 0; r < 10; ++r) {
          const unsigned long long k = s_rank[r];
          if (k < run || k >= run + own) continue;
          unsigned long long at = run;
          int b = b0;
          while (k >= at + a.hraw[b]) at += a.hraw[b++];
          s_val[r] = b - 32768;
        }
    }
    __syncthreads();
    const double N = (double)n, mean = (double)S1 / N;
    if (tid < 5) {
      const unsigned long long num = (n - 1) * (unsigned long long)qs[tid];
      const long long rem = (long long)(num % 100);
      const long long xk = s_val[2 * tid], xk1 = s_val[2 * tid + 1];
      s_pct[tid] = rem == 0 ? (double)xk : xk + (rem / 100.0) * (double)(xk1 - xk);
      // 100 * P_q exactly, for the robust subset P10 <= x <= P90
      s_p100[tid] = 100 * xk + (rem ? rem * (xk1 - xk) : 0);
    }
    __syncthreads();
    auto pct = [&](int qi) -> double { return s_pct[qi]; };
    const long long r10 = s_p100[0], r90 = s_p100[4];
    const double med = pct(2);
    double m[7] = {0, 0, 0, 0, 0, 0, 0};  // m2 m3 m4 mad, robust count, robust sum, |x - median|
    for (int b = lo + tid; b <= hi; b += kMiscThreads) {
      const unsigned c = a.hraw[b];
      if (!c) continue;
      const double xv = b - 32768, dv = xv - mean, dc = (double)c;
      m[0] += dc * dv * dv;
      m[1] += dc * dv * dv * dv;
      m[2] += dc * dv * dv * dv * dv;
      m[3] += dc * fabs(dv);
      m[6] += dc * fabs(xv - med);
      const long long x100 = 100ll * (b - 32768);
      if (x100 >= r10 && x100 <= r90) {
        m[4] += dc;
        m[5] += dc * xv;
      }
    }
    block_sum<7>(m, s_red);
    const double rmean = m[5] / m[4];
    double rm[1] = {0.0};
    for (int b = lo + tid; b <= hi; b += kMiscThreads) {
      const unsigned c = a.hraw[b];
      if (!c) continue;
      const long long x100 = 100ll * (b - 32768);
      if (x100 >= r10 && x100 <= r90) rm[0] += (double)c * fabs((b - 32768) - rmean);
    }
    block_sum<1>(rm, s_red);
    // discretised entropy and uniformity
    double e[2] = {0.0, 0.0};
    for (int g = tid + 1; g <= ng; g += blockDim.x) {
      const double p = (double)a.hlev[g] / N;
      e[0] += sc_ent(p);
      e[1] += p * p;
    }
    block_sum<2>(e, s_red);
    if (tid == 0) {
      const double m2 = m[0] / N, m3 = m[1] / N, m4 = m[2] / N;
      out[0] = (double)S2;
      out[1] = a.voxel_volume * (double)S2;
      out[2] = e[0];
      out[3] = (double)(lo - 32768);
      out[4] = pct(0);
      out[5] = pct(4);
      out[6] = (double)(hi - 32768);
      out[7] = mean;
      out[8] = pct(2);
      out[9] = pct(3) - pct(1);
      out[10] = (double)(hi - lo);
      out[11] = m[3] / N;
      out[12] = rm[0] / m[4];
      out[13] = sqrt((double)S2 / N);
      out[14] = m2 == 0.0 ? kNaN : m3 / pow(m2, 1.5);
      out[15] = m2 == 0.0 ? kNaN : m4 / (m2 * m2) - (a.kurt_excess ? 3.0 : 0.0);
      out[16] = m2;
      out[17] = e[1];
      // IBSI extras: median absolute deviation, coefficient of variation,
      // quartile coefficient of dispersion
      const double p25 = pct(1), p75 = pct(3);
      out[kFirstExtra] = m[6] / N;
      out[kFirstExtra + 1] = sc_div(sqrt(m2), mean);
      out[kFirstExtra + 2] = sc_div(p75 - p25, p75 + p25);
      // standard deviation (population), the scalar-only statistic
      out[kScalarStd] = sqrt(m2);
    }
  } else if (blockIdx.x == 1) {
    // ---- GLDM from [level][equal neighbours] counts
    // N, sum rows^2, sum cols^2, sum of squared cells
    unsigned long long u[4] = {0ull, 0ull, 0ull, 0ull};
    for (int g = tid + 1; g <= ng; g += blockDim.x) {
      unsigned long long r = 0;
      for (int j = 0; j < 27; ++j) {
        const unsigned long long c = a.gldm[g * 27 + j];
        r += c;
        u[3] += c * c;
      }
      u[0] += r;
      u[1] += r * r;
    }
    if (tid < 27) {
      unsigned long long c = 0;
      for (int g = 1; g <= ng; ++g) c += a.gldm[g * 27 + tid];
      u[2] += c * c;
    }
    block_sum_u64<4>(u, s_ured);
    const double N = (double)u[0];
    double m[2] = {0.0, 0.0};
    for (int t = tid; t < ng * 27; t += blockDim.x) {
      const int g = t / 27 + 1, j = t % 27;
      const double c = (double)a.gldm[g * 27 + j];
      m[0] += g * c;
      m[1] += (j + 1) * c;
    }
    block_sum<2>(m, s_red);
    const double mui = m[0] / N, muj = m[1] / N;
    double v[11];
    for (int k = 0; k < 11; ++k) v[k] = 0.0;
    for (int t = tid; t < ng * 27; t += blockDim.x) {
      const int g = t / 27 + 1, j = t % 27;
      const unsigned c = a.gldm[g * 27 + j];
      if (!c) continue;
      const double p = (double)c / N, I = g, J = j + 1;
      sc_size_terms(p, I, J, mui, muj, v);
    }
    block_sum<11>(v, s_red);
    if (tid == 0) {
      double* f = out + 74;
      if (u[0] == 0) {
        for (int k = 0; k < 14; ++k) f[k] = kNaN;
      } else {
        f[0] = v[0];
        f[1] = v[1];
        f[2] = (double)u[1] / N;
        f[3] = (double)u[2] / N;
        f[4] = (double)u[2] / (N * N);
        f[5] = v[2];
        f[6] = v[3];
        f[7] = v[4];
        f[8] = v[5];
        f[9] = v[6];
        f[10] = v[7];
        f[11] = v[8];
        f[12] = v[9];
        f[13] = v[10];
      }
      // IBSI extras: normalised gray level non-uniformity, dependence count
      // percentage, dependence count energy
      double* e = out + kGldmExtra;
      if (u[0] == 0) {
        for (int k = 0; k < 3; ++k) e[k] = kNaN;
      } else {
        e[0] = (double)u[1] / (N * N);
        e[1] = N / (double)a.n_voi;
        e[2] = (double)u[3] / (N * N);
      }
    }
  } else {
    // ---- NGTDM: n_i, s_i = sum_k acc[i][k] / k
    double w[4] = {0, 0, 0, 0};  // Nvp, sum n_i s_i, sum s_i, levels present
    for (int g = tid; g < 256; g += blockDim.x) {
      double si = 0.0;
      if (g >= 1 && g <= ng)
        for (int k = 1; k <= 26; ++k) si += (double)a.ngacc[g * 27 + k] / (double)k;
      s_si[g] = si;
    }
    __syncthreads();
    for (int g = tid + 1; g <= ng; g += blockDim.x) {
      const double ni = (double)a.ngn[g], si = s_si[g];
      w[0] += ni;
      w[1] += ni * si;
      w[2] += si;
      w[3] += ni > 0.0 ? 1.0 : 0.0;
    }
    block_sum<4>(w, s_red);
    const double Nvp = w[0], sum_ps = w[1] / Nvp, sum_s = w[2], ngp = w[3];
    // c1, busy den, complexity, strength: symmetric, and 0 for i = j
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    for (int t = tid; t < (ng + 1) / 2 * (ng + 1); t += blockDim.x) {
      int i, j;
      if (!sc_cell(t, ng, i, j) || i == j) continue;
      ++i;
      ++j;
      const double ni = (double)a.ngn[i], nj = (double)a.ngn[j];
      if (ni == 0.0 || nj == 0.0) continue;
      const double si = s_si[i], sj = s_si[j];
      const double dd = (double)(j - i);
      x[0] += ni * nj * (dd * dd);
      x[1] += fabs((double)i * ni - (double)j * nj);
      x[2] += dd * (ni * si + nj * sj) / (ni + nj);
      x[3] += (ni + nj) * (dd * dd);
    }
    block_sum<4>(x, s_red);
    x[0] *= 2.0 / (Nvp * Nvp);
    x[1] *= 2.0 / Nvp;
    x[2] *= 2.0;
    x[3] *= 2.0 / Nvp;
    if (tid == 0) {
      double* h = out + 88;
      if (Nvp == 0.0) {
        for (int k = 0; k < 5; ++k) h[k] = kNaN;
      } else {
        h[0] = sc_div(1.0, sum_ps);
        h[1] = ngp == 1.0 ? 0.0 : (x[0] / (ngp * (ngp - 1.0))) * (sum_s / Nvp);
        h[2] = sc_div(sum_ps, x[1]);
        h[3] = x[2] / Nvp;
        h[4] = sc_div(x[3], sum_s);
      }
    }
  }
}

// GLSZM from the zones per level, per size and per (level, size).  The table
// of the last is read by the whole chip; a block packs its occupied slots
// first, so that the FP64 terms run on full warps (a few zones in a thousand
// slots), and adds its sums in fixed point: integers, so that neither the slot
// order of the table nor the order of the blocks changes the result.  The last
// block writes out[58..73].  524k slots: 31 us.
constexpr int kZoneSlots = 8 * kScThreads;
__global__ void __launch_bounds__(kScThreads) sc_zone_feat_kernel(const __grid_constant__ FrScalarArgs a) {
  __shared__ unsigned long long s_ured[3 * 32];
  __shared__ unsigned __int128 s_qred[11 * 32];
  __shared__ int s_slot[kZoneSlots];
  __shared__ int s_n;
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  double* f = a.out + 58;
  const double kNaN = __longlong_as_double(0x7ff8000000000000ll);
  if (sc_failed(a)) {
    if (blockIdx.x == 0 && tid < 16) f[tid] = kNaN;
    return;
  }
  const int ng = a.state->ng;
  unsigned long long u[3] = {0ull, 0ull, 0ull};  // N zones, sum rows^2, sum of levels
  for (int g = tid + 1; g <= ng; g += blockDim.x) {
    const unsigned long long r = a.zrow[g];
    u[0] += r;
    u[1] += r * r;
    u[2] += (unsigned)g * r;
  }
  block_sum_u64<3>(u, s_ured);
  if (u[0] == 0) {
    if (blockIdx.x == 0 && tid < 16) f[tid] = kNaN;
    return;
  }
  // the sizes add up to the VOI
  const double N = (double)u[0], mui = (double)u[2] / N, muj = (double)a.n_voi / N;
  unsigned long long c2[1] = {0ull};  // sum cols^2
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + tid + 1; j <= a.n_voi;
       j += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long c = a.zcol[j];
    c2[0] += c * c;
  }
  // bits after the point per sum, from its bound (I <= 255, J < 2^31, sum p =
  // 1): <= 1 -> 120; <= 255^2 -> 110; <= 2^62 -> 64; <= 2^78 -> 48
  constexpr int kFb[11] = {120, 64, 110, 64, 120, 120, 110, 120, 110, 64, 48};
  unsigned __int128 q[11];
  for (int k = 0; k < 11; ++k) q[k] = 0;
  for (int64_t t0 = (int64_t)blockIdx.x * kZoneSlots; t0 < a.hcap; t0 += (int64_t)gridDim.x * kZoneSlots) {
    if (tid == 0) s_n = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kZoneSlots / kScThreads; ++k) {
      const int64_t t = t0 + k * kScThreads + tid;
      if (t < a.hcap && a.hkey[t] != kEmptyKey) s_slot[atomicAdd(&s_n, 1)] = k * kScThreads + tid;
    }
    __syncthreads();
    for (int e = tid; e < s_n; e += blockDim.x) {
      const int64_t t = t0 + s_slot[e];
      const unsigned long long key = a.hkey[t];
      const double I = (double)(key >> 32), J = (double)(key & 0xffffffffull);
      double tv[11] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      sc_size_terms((double)a.hcnt[t] / N, I, J, mui, muj, tv);
#pragma unroll
      for (int k = 0; k < 11; ++k) q[k] += sc_fixed(tv[k], kFb[k]);
    }
    __syncthreads();
  }
  block_sum_u64<1>(c2, s_ured);
  block_sum_u128<11>(q, s_qred);
  if (tid < 11) {
    // 128-bit sums as two words, the carry passed on by the addition that wraps
    const unsigned __int128 own = s_qred[tid * 32];
    const unsigned long long lo = (unsigned long long)own;
    const unsigned long long was = atomicAdd(&a.zsum[2 * tid], lo);
    atomicAdd(&a.zsum[2 * tid + 1], (unsigned long long)(own >> 64) + (was + lo < was ? 1ull : 0ull));
  }
  if (tid == 11) atomicAdd(&a.zsum[22], c2[0]);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&a.zsum[23], 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid == 0) {
    double v[11];
#pragma unroll
    for (int k = 0; k < 11; ++k)
      v[k] = sc_unfixed(((unsigned __int128)__ldcg(&a.zsum[2 * k + 1]) << 64) | __ldcg(&a.zsum[2 * k]), kFb[k]);
    const double cols2 = (double)__ldcg(&a.zsum[22]);
    f[0] = v[0];
    f[1] = v[1];
    f[2] = (double)u[1] / N;
    f[3] = (double)u[1] / (N * N);
    f[4] = cols2 / N;
    f[5] = cols2 / (N * N);
    f[6] = N / (double)a.n_voi;
    f[7] = v[2];
    f[8] = v[3];
    f[9] = v[4];
    f[10] = v[5];
    f[11] = v[6];
    f[12] = v[7];
    f[13] = v[8];
    f[14] = v[9];
    f[15] = v[10];
  }
}

// Direction averages (NaN skipped), then the selected features in id order.
__global__ void sc_final_kernel(const __grid_constant__ FrScalarArgs a, double* user_out,
                                const int16_t* __restrict__ row_of_dev) {
  const double kNaN = __longlong_as_double(0x7ff8000000000000ll);
  const int ndir = a.agg == 1 ? 1 : kNumDirs;
  const bool bad = sc_failed(a);
  for (int k = threadIdx.x; k < kScalarDirF; k += blockDim.x) {
    double s = 0.0;
    int c = 0;
    for (int d = 0; d < ndir; ++d) {
      const double v = a.dirf[d * kScalarDirF + k];
      if (isnan(v)) continue;
      s += v;
      ++c;
    }
    a.out[k < 24 ? 18 + k : k < 40 ? 42 + (k - 24) : kGlcmExtra + (k - 40)] = c ? s / c : kNaN;
  }
  __syncthreads();
  for (int f = threadIdx.x; f < kNumScalarFeatures; f += blockDim.x) {
    const int row = row_of_dev[f];
    if (row >= 0) user_out[row] = bad ? kNaN : a.out[f];
  }
}

// ---------------------------------------------------------------- host side

static int sc_grid(int64_t n, int threads, int cap) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

cudaError_t fr_scalar_configure(int ngc) {
  cudaError_t e = cudaFuncSetAttribute(sc_neigh_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       neigh_smem(255));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(sc_glcm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              255 * 256 / 2 * 4);
}

// Every kernel of one scalar extraction, after discretisation and the
// zeroing of the count buffers.
cudaError_t fr_scalar_launch(const FrScalarArgs& a, double* user_out, const int16_t* row_of_dev,
                             int sms, cudaStream_t s) {
  const int grid = sc_grid(a.n_voi, kScThreads, 8 * sms);
  sc_init_kernel<<<grid, kScThreads, 0, s>>>(a);
  sc_neigh_kernel<<<sc_grid(a.n_voi, kCountThreads, 2 * sms), kCountThreads, neigh_smem(a.ngc), s>>>(a);
  // one wave of blocks at the largest level cap, whose copy leaves one a SM
  // (200k voxels: 66 us with 312 blocks of 256 threads -> 19 us)
  const int gx = sc_grid(a.n_voi, kCountThreads * 4, sms / kNumDirs > 0 ? sms / kNumDirs : 1);
  const int np = a.ngc * (a.ngc + 1) / 2;
  sc_glcm_kernel<<<dim3(gx, kNumDirs), kCountThreads, np * 4, s>>>(a);
  sc_glrlm_kernel<<<dim3(sc_grid(a.n_voi, kScThreads, (8 * sms) / kNumDirs + 1), kNumDirs),
                    kScThreads, 0, s>>>(a);
  sc_flatten_kernel<<<grid, kScThreads, 0, s>>>(a);
  sc_zone_kernel<<<grid, kScThreads, 0, s>>>(a);
  const int ndir = a.agg == 1 ? 1 : kNumDirs;
  sc_glcm_feat_kernel<<<ndir, kScThreads, 0, s>>>(a);
  sc_glrlm_feat_kernel<<<ndir, kScThreads, 0, s>>>(a);
  sc_zone_feat_kernel<<<sc_grid(a.hcap, kZoneSlots, 2 * sms), kScThreads, 0, s>>>(a);
  sc_misc_feat_kernel<<<3, kMiscThreads, 0, s>>>(a);
  sc_final_kernel<<<1, 128, 0, s>>>(a, user_out, row_of_dev);
  return cudaGetLastError();
}

}  // namespace fr
