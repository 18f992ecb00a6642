// k_surface.cu — surface reconstruction (Sec. 3.3): the particles' signed
// distance field on a sampling grid (Sec. 3.3.1), marching cubes over it and
// inverse-area-weighted vertex normals (Sec. 3.3.2).  C ABI: include/flip_surface.h.
//
// Pipeline of flip_surface_sdf (all on the surface's stream):
//   k_sbin_count    particle -> bin of edge R/2 over the corner box grown by R;
//                   the histogram atomic returns its rank in the bin
//   scan            exclusive scan of the bin counts (tile scan below)
//   k_sbin_scatter  positions into bin order as float4
//   k_sdf           one warp per 2 x 2 x 2 corners: the bin rows that meet their balls of
//                   radius R, read as coalesced particle ranges; kernel sums of k and
//                   k (x_i - x), phi = |sum k d| / sum k - r
// Pipeline of flip_surface_mesh:
//   k_mc_classify   every corner's crossing / case code and the tiles' counts, packed as
//                   (vertices on the corner's 3 outgoing edges) + (triangles of the cube it
//                   is the lowest corner of) << 32
//   k_tile_scan     exclusive scan of the tiles' counts; their total goes to the host, which
//                   grows the mesh's arrays
//   k_mc_vertices   vertices, and the offsets of the corners that have any
//   k_mc_triangles  triangles and their weighted normals n / A
//   k_mc_normals    the weights gathered per vertex from the four cubes around its edge in a
//                   fixed order (deterministic sums)
// A call of 4.2 M corners and 53 thousand vertices, with its field set and its results read,
// 258 -> 180 us (174 to 185 from run to run).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/flip_surface.h"
#include "flip_kernels.cuh"

void flip_set_last_error_(const std::string& msg);

using namespace flipk;

namespace {

int sfail(int code, const std::string& msg) {
  flip_set_last_error_(msg);
  return code;
}

int scuda(cudaError_t e, const char* what) {
  const int code = (e == cudaErrorMemoryAllocation) ? FLIP_E_OOM : FLIP_E_CUDA;
  return sfail(code, std::string(what) + ": " + cudaGetErrorName(e));
}

#define SURF_CUDA(call)                            \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return scuda(e_, #call); \
  } while (0)

// ------------------------------------------------------------------ case table
//
// Local cube numbering: corner c has offset (c & 1, (c >> 1) & 1, c >> 2).  Edge
// e runs along axis a = e / 4 from the corner with bit a clear; its bits on the
// other two axes (ascending) are e & 1 and (e >> 1) & 1.
constexpr int MC_MAXT = 12;

struct McTable {
  uint8_t ntri[256];
  uint8_t tri[256][MC_MAXT][3];
};

// In global memory, not constant: lanes look up different cases, which constant reads serve one
// after the other.
__device__ McTable c_mc;

int edge_of(int c0, int c1) {
  const int d = c0 ^ c1;
  const int a = (d == 1) ? 0 : (d == 2) ? 1 : 2;
  const int lo = (a == 0) ? 1 : 0, hi = (a == 2) ? 1 : 2;
  return 4 * a + ((c0 >> lo) & 1) + 2 * ((c0 >> hi) & 1);
}

void edge_ends(int e, int& c0, int& c1) {
  const int a = e / 4;
  const int lo = (a == 0) ? 1 : 0, hi = (a == 2) ? 1 : 2;
  c0 = ((e & 1) << lo) | (((e >> 1) & 1) << hi);
  c1 = c0 | (1 << a);
}

bool build_table(McTable& T) {
  std::memset(&T, 0, sizeof(T));
  for (int cs = 0; cs < 256; ++cs) {
    auto in = [&](int c) { return (cs >> c) & 1; };
    // face segments: each crossing edge gets one partner per face it lies on
    int partner[12][2];
    int np_[12] = {0};
    for (int f = 0; f < 6; ++f) {
      const int a = f / 2, s = f % 2;
      const int u = (a == 0) ? 1 : 0, v = (a == 2) ? 1 : 2;
      int P[4];
      const int cyc[4][2] = {{0, 0}, {1, 0}, {1, 1}, {0, 1}};
      for (int q = 0; q < 4; ++q) P[q] = (s << a) | (cyc[q][0] << u) | (cyc[q][1] << v);
      int E[4], X[4], nx = 0;
      for (int q = 0; q < 4; ++q) {
        E[q] = edge_of(P[q], P[(q + 1) & 3]);
        X[q] = in(P[q]) != in(P[(q + 1) & 3]);
        nx += X[q];
      }
      auto link = [&](int e0, int e1) {
        partner[e0][np_[e0]++] = e1;
        partner[e1][np_[e1]++] = e0;
      };
      if (nx == 2) {
        int k0 = -1, k1 = -1;
        for (int q = 0; q < 4; ++q)
          if (X[q]) (k0 < 0 ? k0 : k1) = q;
        link(E[k0], E[k1]);
      } else if (nx == 4) {
        for (int q = 0; q < 4; ++q)
          if (in(P[q])) link(E[(q + 3) & 3], E[q]);  // cut off each inside corner
      }
    }
    bool used[12] = {false};
    int nt = 0;
    for (int e0 = 0; e0 < 12; ++e0) {
      if (np_[e0] == 0 || used[e0]) continue;
      if (np_[e0] != 2) return false;
      int loop[12], len = 0, prev = -1, cur = e0;
      do {
        if (len == 12) return false;
        loop[len++] = cur;
        used[cur] = true;
        const int nxt = (partner[cur][0] != prev) ? partner[cur][0] : partner[cur][1];
        prev = cur;
        cur = nxt;
      } while (cur != e0);
      if (len < 3) return false;
      // winding: Newell normal of the edge midpoints against inside -> outside
      double N[3] = {0, 0, 0}, D[3] = {0, 0, 0}, M[12][3];
      for (int q = 0; q < len; ++q) {
        int c0, c1;
        edge_ends(loop[q], c0, c1);
        for (int d = 0; d < 3; ++d) {
          const double p0 = (c0 >> d) & 1, p1 = (c1 >> d) & 1;
          M[q][d] = 0.5 * (p0 + p1);
          D[d] += in(c0) ? (p1 - p0) : (p0 - p1);
        }
      }
      for (int q = 0; q < len; ++q) {
        const double* A = M[q];
        const double* B = M[(q + 1) % len];
        N[0] += (A[1] - B[1]) * (A[2] + B[2]);
        N[1] += (A[2] - B[2]) * (A[0] + B[0]);
        N[2] += (A[0] - B[0]) * (A[1] + B[1]);
      }
      const double nd = N[0] * D[0] + N[1] * D[1] + N[2] * D[2];
      if (std::fabs(nd) < 1e-9) return false;
      if (nd < 0) std::reverse(loop, loop + len);
      // fan apex: the lowest edge on no face the loop crosses twice (a face holding
      // four of its edges); a fan from there puts no triangle inside a cube face
      int on_face[6] = {0, 0, 0, 0, 0, 0};
      auto faces_of = [](int e, int& f0, int& f1) {
        const int a = e / 4;
        const int lo = (a == 0) ? 1 : 0, hi = (a == 2) ? 1 : 2;
        f0 = 2 * lo + (e & 1);
        f1 = 2 * hi + ((e >> 1) & 1);
      };
      for (int q = 0; q < len; ++q) {
        int f0, f1;
        faces_of(loop[q], f0, f1);
        ++on_face[f0];
        ++on_face[f1];
      }
      int r0 = -1;
      for (int q = 0; q < len; ++q) {
        int f0, f1;
        faces_of(loop[q], f0, f1);
        if (on_face[f0] < 4 && on_face[f1] < 4 && (r0 < 0 || loop[q] < loop[r0])) r0 = q;
      }
      if (r0 < 0) r0 = (int)(std::min_element(loop, loop + len) - loop);
      std::rotate(loop, loop + r0, loop + len);
      for (int q = 1; q + 1 < len; ++q) {
        if (nt == MC_MAXT) return false;
        T.tri[cs][nt][0] = (uint8_t)loop[0];
        T.tri[cs][nt][1] = (uint8_t)loop[q];
        T.tri[cs][nt][2] = (uint8_t)loop[q + 1];
        ++nt;
      }
    }
    T.ntri[cs] = (uint8_t)nt;
  }
  return true;
}

// The table is generated once per process and uploaded to each device that
// creates a surface object (a device variable has a copy on each).
std::mutex g_table_mutex;
bool g_table_built = false, g_table_ok = false;
McTable g_table;
std::vector<int> g_table_devices;

int ensure_table() {
  std::lock_guard<std::mutex> lock(g_table_mutex);
  if (!g_table_built) {
    g_table_ok = build_table(g_table);
    g_table_built = true;
  }
  if (!g_table_ok) return sfail(FLIP_E_CUDA, "marching-cubes table generation failed");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return scuda(e, "cudaGetDevice");
  if (std::find(g_table_devices.begin(), g_table_devices.end(), dev) != g_table_devices.end())
    return FLIP_OK;
  e = cudaMemcpyToSymbol(c_mc, &g_table, sizeof(g_table));
  if (e != cudaSuccess) return scuda(e, "cudaMemcpyToSymbol(case table)");
  g_table_devices.push_back(dev);
  return FLIP_OK;
}

// ------------------------------------------------------------------ geometry

struct SGrid {
  int n[3];           // cells per axis
  int c[3];           // corners per axis (n + 1)
  long long ncorners;
  float o[3];         // origin
  float h;
  float iso;
};

struct SBins {
  int nb[3];
  long long nbins;
  float o[3];         // bin-grid origin (corner origin - R)
  float b;            // bin edge
  float inv_b;
  float R, R2, inv_R2, r;
};

__device__ __forceinline__ void corner_ijk(const SGrid& g, long long c, int& i, int& j, int& k) {
  // at most 1025^3 corners: 32-bit divisions, which are several times cheaper
  const unsigned int x = (unsigned int)c, t = x / (unsigned)g.c[0];
  i = (int)(x - t * (unsigned)g.c[0]);
  k = (int)(t / (unsigned)g.c[1]);
  j = (int)(t - (unsigned)k * (unsigned)g.c[1]);
}

// ------------------------------------------------------------------ tile scan
//
// An exclusive scan over n items of a per-item count computed by a functor:
// pass 1 reduces tiles of SC_TILE items, pass 2 (one CTA) scans the tile sums,
// pass 3 recomputes the counts, scans them within the tile and hands each item
// its exclusive prefix.  The counts are never stored.
constexpr int SC_THREADS = 256;
constexpr int SC_ROWS = 8;
constexpr int SC_TILE = SC_THREADS * SC_ROWS;
typedef unsigned long long u64;

__device__ __forceinline__ u64 block_excl_scan(u64 v, u64& total, u64* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) sm[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    u64 w = (lane < SC_THREADS / 32) ? sm[lane] : 0ull;
    u64 wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    if (lane < SC_THREADS / 32) sm[32 + lane] = wi - w;
    if (lane == SC_THREADS / 32 - 1) sm[64] = wi;
  }
  __syncthreads();
  total = sm[64];
  return sm[32 + warp] + incl - v;
}

template <class F>
__global__ void __launch_bounds__(SC_THREADS) k_tile_reduce(F f, long long n, u64* tile_sum) {
  __shared__ u64 sm[72];
  const long long base = (long long)blockIdx.x * SC_TILE;
  u64 s = 0;
#pragma unroll
  for (int r = 0; r < SC_ROWS; ++r) {
    const long long i = base + r * SC_THREADS + threadIdx.x;
    if (i < n) s += f.count(i);
  }
  u64 tot;
  block_excl_scan(s, tot, sm);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

// Bound by latency: 4 sums a thread, so that 4096 tiles take one round (2038 tiles 8.5 ->
// 4.5 us against 256 a round).
constexpr int TS_THREADS = 1024;
__global__ void __launch_bounds__(TS_THREADS) k_tile_scan(u64* tile_sum, long long ntiles,
                                                          u64* total) {
  __shared__ u64 sm[TS_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 carry = 0;
  for (long long b = 0; b < ntiles; b += 4 * TS_THREADS) {
    const long long i = b + 4 * (long long)threadIdx.x;
    u64 v[4], own = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = i + q < ntiles ? tile_sum[i + q] : 0ull;
      own += v[q];
    }
    u64 incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) sm[warp] = incl;
    __syncthreads();
    const u64 w = sm[lane];  // every warp scans the warps' sums
    u64 wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    u64 run = carry + __shfl_sync(0xffffffffu, wi - w, warp) + incl - own;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (i + q < ntiles) tile_sum[i + q] = run;
      run += v[q];
    }
    carry += __shfl_sync(0xffffffffu, wi, 31);
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

template <class F>
__global__ void __launch_bounds__(SC_THREADS) k_tile_apply(F f, long long n, const u64* tile_off) {
  __shared__ u64 sm[72];
  const long long base = (long long)blockIdx.x * SC_TILE;
  u64 run = tile_off[blockIdx.x];
  for (int r = 0; r < SC_ROWS; ++r) {
    const long long i = base + r * SC_THREADS + threadIdx.x;
    const u64 c = (i < n) ? f.count(i) : 0ull;
    u64 tot;
    const u64 ex = block_excl_scan(c, tot, sm);
    if (i < n) f.apply(i, run + ex);
    run += tot;
  }
}

template <class F>
void tile_scan(const F& f, long long n, u64* tile_sum, u64* total, cudaStream_t s) {
  const long long ntiles = (n + SC_TILE - 1) / SC_TILE;
  k_tile_reduce<F><<<(unsigned)ntiles, SC_THREADS, 0, s>>>(f, n, tile_sum);
  k_tile_scan<<<1, TS_THREADS, 0, s>>>(tile_sum, ntiles, total);
  k_tile_apply<F><<<(unsigned)ntiles, SC_THREADS, 0, s>>>(f, n, tile_sum);
}

// ------------------------------------------------------------------ binning + SDF

__device__ __forceinline__ int bin_coord(float x, const SBins& B, int a) {
  const float t = floorf((x - B.o[a]) * B.inv_b);
  return (t >= 0.0f && t < (float)B.nb[a]) ? (int)t : -1;
}

__global__ void k_sbin_count(const PartView p, long long np, const SBins B,
                             unsigned int* __restrict__ count, int* __restrict__ pbin,
                             unsigned int* __restrict__ prank) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= np) return;
  const int bx = bin_coord(p.x[i], B, 0), by = bin_coord(p.y[i], B, 1),
            bz = bin_coord(p.z[i], B, 2);
  int b = -1;
  if (bx >= 0 && by >= 0 && bz >= 0) {
    b = bx + B.nb[0] * (by + B.nb[1] * bz);
    prank[i] = atomicAdd(count + b, 1u);
  }
  pbin[i] = b;
}

// Scans nbins + 1 items so that start[nbins] is the total.
struct BinScan {
  const unsigned int* cnt;
  unsigned int* start;
  long long nbins;
  __device__ u64 count(long long i) const { return i < nbins ? cnt[i] : 0u; }
  __device__ void apply(long long i, u64 ex) const { start[i] = (unsigned int)ex; }
};

__global__ void k_fill(float* __restrict__ p, long long n, float v) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

__global__ void k_sbin_scatter(const PartView p, long long np, const int* __restrict__ pbin,
                               const unsigned int* __restrict__ prank,
                               const unsigned int* __restrict__ start, float4* __restrict__ pos) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= np) return;
  const int b = pbin[i];
  if (b < 0) return;
  pos[start[b] + prank[i]] = make_float4(p.x[i], p.y[i], p.z[i], 0.0f);
}

// One warp per group of 2 PX x GY x GZ corners (sdf_launch has the lines between them).  With
// bins of edge R/2 the balls' extent along y or z is at most 5.98 bins, which meets at most 7
// (8 with roundings), so at most 64 bin rows (fixed y, z bin): lane r finds the particle
// ranges of rows r and r + 32 (a row's bins within the balls' x extent are one contiguous
// range; a bin whose nearest point is R or farther from the corners holds no particle closer
// than R and is skipped), the nonempty rows are packed into a per-warp list, and the warp's
// four groups of eight lanes take a row each, eight particles (128 bytes) at a time.  Each
// particle is tested against all the group's corners, whose sums stay in registers until a
// reduction that halves the values with every step.  The eight warps of a CTA take
// neighbouring groups (2 x 2 x 2 of them), so that most of a CTA's particle reads hit L1.
//
// With e the offset particle minus corner, 1 - |e|^2 / R^2 is taken axis by axis: the two
// values of 1 - ez^2 / R^2 and the four with y are shared by the corners, so that a corner's
// weight costs one FMA more.
//
// Bound by issue.  A whole flip_surface_sdf of 42 M particles at 257^3 corners takes 4.04 ms,
// of 2.1 M at 129^3 0.358; with 2 x 2 x 1 corners a warp 4.81 and 0.414 (about 50 instructions
// per particle and four corners; a wider group tests more particles, but shares more of their
// arithmetic); with one warp per 4 corners along x, whose lanes walked one flat range over all
// rows, 6.80 and 0.555.  With t from 1 - |p|^2 / R^2 about the group's centre plus terms linear
// in p 4.16 and 0.366, at twice the rounding error; 16 lanes a row 4.40; 4 CTAs per SM 4.40.
constexpr int SDF_THREADS = 256;
constexpr int SDF_WARPS = SDF_THREADS / 32;
constexpr int SDF_ROW_LANES = 8;
constexpr int SDF_ROWS = 64;
// On a grid of few groups the lanes of a warp share every row from this many particles a row
// on, instead of a row per eight lanes.  Such a grid's balls can meet few rows of up to
// thousands of particles each: 2^3 cells over 32 thousand particles, R = 4 h, 1010 -> 345 us,
// 10^3 cells, R = 4, 6 and 8 h, 252, 366 and 508 -> 189, 241 and 260 (with lanes that walk one
// flat range over the rows of 4 corners along x 401, 186, 281 and 353).  From 32 on, rows that
// do not fill the lanes cost more (64^3 cells, R = 2 h, 132 -> 162 us).
constexpr unsigned int SDF_LONG = 64;
// A corner whose sum of weights is below this is summed again with the ball's edge taken
// exactly.  A particle at distance R or more has a rounded 1 - d^2 / R^2 of up to 2^-23, a
// weight of 2^-69: nothing beside this sum, but all there is at a corner that no particle is
// closer to than R.
constexpr float SDF_THIN = 0x1p-30f;

template <int PX, int GY, int GZ, bool FEW>
__global__ void __launch_bounds__(SDF_THREADS) k_sdf(const SGrid g, const SBins B,
                                                     const unsigned int* __restrict__ start,
                                                     const float4* __restrict__ pos,
                                                     float* __restrict__ phi) {
  constexpr int GX = 2 * PX, NP = PX * GY * GZ;  // pairs along x
  static_assert((GY == 1 || GY == 2) && (GZ == 1 || GZ == 2) && NP <= 4, "offsets in pairs");
  __shared__ uint2 s_row[SDF_WARPS][SDF_ROWS];  // {first particle, end} of the nonempty rows
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // a CTA's groups: 2 x 2 x 2
  constexpr int CX = 2 * GX, CY = 2 * GY, CZ = 2 * GZ;
  const int tx = (g.c[0] + CX - 1) / CX, ty = (g.c[1] + CY - 1) / CY, tz = (g.c[2] + CZ - 1) / CZ;
  const long long ntiles = (long long)tx * ty * tz;
  constexpr float Rb = 2.0f;  // R in bins (the bin edge is R/2)
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (int)(tile % tx) * CX + (wid & 1) * GX;
    const int j0 = (int)((tile / tx) % ty) * CY + ((wid >> 1) & 1) * GY;
    const int k0 = (int)(tile / ((long long)tx * ty)) * CZ + (wid >> 2) * GZ;
    if (i0 >= g.c[0] || j0 >= g.c[1] || k0 >= g.c[2]) continue;
    const float x0 = g.o[0] + g.h * (float)i0, x1 = g.o[0] + g.h * (float)(i0 + GX - 1);
    const float y0 = g.o[1] + g.h * (float)j0, y1 = g.o[1] + g.h * (float)(j0 + GY - 1);
    const float z0 = g.o[2] + g.h * (float)k0, z1 = g.o[2] + g.h * (float)(k0 + GZ - 1);
    const float ry0 = (y0 - B.o[1]) * B.inv_b, ry1 = (y1 - B.o[1]) * B.inv_b;
    const float rz0 = (z0 - B.o[2]) * B.inv_b, rz1 = (z1 - B.o[2]) * B.inv_b;
    const int by0 = max(0, (int)floorf(ry0 - Rb)), by1 = min(B.nb[1] - 1, (int)floorf(ry1 + Rb));
    const int bz0 = max(0, (int)floorf(rz0 - Rb)), bz1 = min(B.nb[2] - 1, (int)floorf(rz1 + Rb));
    const int nyr = max(by1 - by0 + 1, 1);
    const int nrows = min(nyr * (bz1 - bz0 + 1), SDF_ROWS);
    int nrow = 0;
    unsigned int npart = 0;
    __syncwarp();  // the last group's reads of the list are done
    for (int r0 = 0; r0 < nrows; r0 += 32) {
      const int r = r0 + lane;
      unsigned int p0 = 0, p1 = 0;
      if (r < nrows) {
        const int by = by0 + r % nyr, bz = bz0 + r / nyr;
        const float dy = fmaxf(fmaxf(B.o[1] + B.b * by - y1, y0 - (B.o[1] + B.b * (by + 1))), 0.0f);
        const float dz = fmaxf(fmaxf(B.o[2] + B.b * bz - z1, z0 - (B.o[2] + B.b * (bz + 1))), 0.0f);
        const float dyz = dy * dy + dz * dz;
        if (dyz < B.R2) {
          const float rx = sqrtf(B.R2 - dyz) * B.inv_b;
          const int bx0 = max(0, (int)floorf((x0 - B.o[0]) * B.inv_b - rx));
          // (a bin that begins at the balls' end holds nothing closer than R)
          const int bx1 = min(B.nb[0] - 1, (int)ceilf((x1 - B.o[0]) * B.inv_b + rx) - 1);
          if (bx0 <= bx1) {
            const long long row = (long long)B.nb[0] * (by + (long long)B.nb[1] * bz);
            p0 = start[row + bx0];
            p1 = start[row + bx1 + 1];
          }
        }
      }
      const unsigned int some = __ballot_sync(0xffffffffu, p0 < p1);
      if (p0 < p1) s_row[wid][nrow + __popc(some & ((1u << lane) - 1u))] = make_uint2(p0, p1);
      nrow += __popc(some);
      npart += p1 - p0;
    }
    __syncwarp();
    // the rows a lane walks and its particles of each
    int row0 = lane / SDF_ROW_LANES, rows = 32 / SDF_ROW_LANES;
    unsigned int part0 = lane % SDF_ROW_LANES, parts = SDF_ROW_LANES;
    if (FEW && __reduce_add_sync(0xffffffffu, npart) >= SDF_LONG * (unsigned int)nrow)
      row0 = 0, rows = 1, part0 = (unsigned int)lane, parts = 32u;
    // minus the corners' coordinates (P.x + (-x) rounds as P.x - x); packed operations round
    // like the scalar ones
    float2 mx[PX];
#pragma unroll
    for (int p = 0; p < PX; ++p)
      mx[p] = make_float2(-(g.o[0] + g.h * (float)(i0 + 2 * p)),
                          -(g.o[0] + g.h * (float)(i0 + 2 * p + 1)));
    const float2 my = make_float2(-y0, -y1), mz = make_float2(-z0, -z1);
    const float2 nr = make_float2(-B.inv_R2, -B.inv_R2);
    // per corner: sum k and sum k e; corners (2 p, y, z) and (2 p + 1, y, z) are the two lanes
    float2 sk[NP], sx[NP], sy[NP], sz[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) sk[q] = sx[q] = sy[q] = sz[q] = make_float2(0.0f, 0.0f);
    for (int r = row0; r < nrow; r += rows) {
      const uint2 row = s_row[wid][r];
      unsigned int f = row.x + part0;
      float4 next = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (f < row.y) next = pos[f];
      for (; f < row.y; f += parts) {
        const float4 P = next;  // the next particle's load is in flight during this one's sums
        if (f + parts < row.y) next = pos[f + parts];
        const float2 ey = __fadd2_rn(make_float2(P.y, P.y), my);
        const float2 ez = __fadd2_rn(make_float2(P.z, P.z), mz);
        const float2 fy = __fmul2_rn(ey, nr);
        float2 ex[PX], fx[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
          ex[p] = __fadd2_rn(make_float2(P.x, P.x), mx[p]);
          fx[p] = __fmul2_rn(ex[p], nr);
        }
        const float2 wz = __ffma2_rn(ez, __fmul2_rn(ez, nr), make_float2(1.0f, 1.0f));
#pragma unroll
        for (int z = 0; z < GZ; ++z) {
          const float e2 = z ? ez.y : ez.x;
#pragma unroll
          for (int y = 0; y < GY; ++y) {
            const float e1 = y ? ey.y : ey.x;
            const float w = __fmaf_rn(e1, y ? fy.y : fy.x, z ? wz.y : wz.x);
#pragma unroll
            for (int p = 0; p < PX; ++p) {
              const int q = p + PX * (y + GY * z);
              // k = max(0, 1 - d^2 / R^2)^3 (saturating: d^2 >= 0), at d >= R to rounding
              // (SDF_THIN)
              const float2 t = make_float2(__saturatef(__fmaf_rn(ex[p].x, fx[p].x, w)),
                                           __saturatef(__fmaf_rn(ex[p].y, fx[p].y, w)));
              const float2 kk = __fmul2_rn(__fmul2_rn(t, t), t);
              sk[q] = __fadd2_rn(sk[q], kk);
              sx[q] = __ffma2_rn(kk, ex[p], sx[q]);
              sy[q] = __ffma2_rn(kk, make_float2(e1, e1), sy[q]);
              sz[q] = __ffma2_rn(kk, make_float2(e2, e2), sz[q]);
            }
          }
        }
      }
    }
    // reduction: with every step a lane keeps half of its values and adds its partner's
    // halves of them; then lane l holds value l % 4 of corner l / 4 (modulo the corners)
    constexpr int NV = 8 * NP;
    float v[NV];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      v[8 * q] = sk[q].x;
      v[8 * q + 1] = sx[q].x;
      v[8 * q + 2] = sy[q].x;
      v[8 * q + 3] = sz[q].x;
      v[8 * q + 4] = sk[q].y;
      v[8 * q + 5] = sx[q].y;
      v[8 * q + 6] = sy[q].y;
      v[8 * q + 7] = sz[q].y;
    }
#pragma unroll
    for (int n = NV / 2; n >= 1; n >>= 1) {
      const bool hi = lane & n;
#pragma unroll
      for (int q = 0; q < n; ++q) {
        const float send = hi ? v[q] : v[q + n];
        const float keep = hi ? v[q + n] : v[q];
        v[q] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, n));
      }
    }
    // lanes equal modulo NV hold partial sums of the same value
    float s = v[0];
#pragma unroll
    for (int n = NV; n < 32; n <<= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, n));
    float a = __shfl_sync(0xffffffffu, s, 4 * lane);  // lane c < corners: corner c's sums
    float b0 = __shfl_sync(0xffffffffu, s, 4 * lane + 1);
    float b1 = __shfl_sync(0xffffffffu, s, 4 * lane + 2);
    float b2 = __shfl_sync(0xffffffffu, s, 4 * lane + 3);
    const int i = i0 + lane % GX, j = j0 + lane / GX % GY, k = k0 + lane / (GX * GY);
    const bool in = lane < 2 * NP && i < g.c[0] && j < g.c[1] && k < g.c[2];
    // (few: no measurable time)
    for (unsigned int thin = __ballot_sync(0xffffffffu, in && a > 0.0f && a < SDF_THIN); thin;
         thin &= thin - 1u) {
      const int c = __ffs(thin) - 1;
      float2 m = mx[0];
      if (PX > 1 && c % GX >= 2) m = mx[PX - 1];
      const float cx = -(c & 1 ? m.y : m.x), cy = c / GX % GY ? y1 : y0, cz = c / (GX * GY) ? z1 : z0;
      float w = 0.0f, wx = 0.0f, wy = 0.0f, wz = 0.0f;
      for (int r = row0; r < nrow; r += rows) {
        const uint2 row = s_row[wid][r];
        for (unsigned int f = row.x + part0; f < row.y; f += parts) {
          const float4 P = pos[f];
          const float ex = P.x - cx, ey = P.y - cy, ez = P.z - cz;
          const float dd = __fmaf_rn(ex, ex, __fmaf_rn(ez, ez, __fmul_rn(ey, ey)));
          const float t = dd < B.R2 ? fmaxf(__fmaf_rn(dd, -B.inv_R2, 1.0f), 0.0f) : 0.0f;
          const float kk = t * t * t;
          w += kk;
          wx = __fmaf_rn(kk, ex, wx);
          wy = __fmaf_rn(kk, ey, wy);
          wz = __fmaf_rn(kk, ez, wz);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        w += __shfl_xor_sync(0xffffffffu, w, o);
        wx += __shfl_xor_sync(0xffffffffu, wx, o);
        wy += __shfl_xor_sync(0xffffffffu, wy, o);
        wz += __shfl_xor_sync(0xffffffffu, wz, o);
      }
      if (lane == c) a = w, b0 = wx, b1 = wy, b2 = wz;
    }
    if (in) {
      const float d = (a > 0.0f) ? sqrtf(b0 * b0 + b1 * b1 + b2 * b2) / a - B.r : B.R - B.r;
      phi[i + (long long)g.c[0] * (j + (long long)g.c[1] * k)] = d;
    }
  }
}

// 2 x 2 x 2 corners share most of their bins and, up to corners 1.98 bins apart (R a little
// over h), their rows fit a warp's list; wider grids take 4 x 1 x 1, whose rows do not grow
// with h.  A 128^3 pool at R = 1.9, 1.4, 1.05 and 0.9, 0.7 and 0.5 h: 658, 530, 547 us and
// 617, 762, 1293; with 2 x 1 x 1 from R < 2 h on 1063, 823, 802 and 835, 999, 1515; with
// lanes that walk one flat range over the rows of 4 corners along x 962, 699, 653 and 701,
// 871, 1488.
// A grid of few groups (of less than four rounds of resident warps: 14592 on 152 SMs) takes
// 2 x 2 x 1 ones, twice as many, to even out the chip's last rounds, and a CTA per tile, which
// the device hands out as CTAs end: 40^3 cells (9261 groups), R = 2, 4 and 8 h, 79, 233 and
// 1200 -> 70, 149 and 678 us; 32^3 (4913) 140, 640 and 3650 -> 129, 577 and 3020, and with
// 2 x 2 x 2 corners 140, 659 and 3120.  With fewer groups than resident warps it takes pairs:
// 32 x 25 x 16 cells (1989 groups), R = 1.2, 2, 4 and 8 h, 282, 667, 3319 and 13918 -> 241,
// 611, 3152 and 13955 us, but 32^3 94, 129, 577 and 3020 -> 91, 130, 614 and 3550.  More groups
// do not gain by a CTA per tile (256^3 cells 4.01 -> 4.41 ms), nor by the smaller ones (26
// thousand 72-103 us with 2 x 2 x 2 corners, 77-109 with 2 x 2 x 1).
using SdfKernel = void (*)(const SGrid, const SBins, const unsigned int*, const float4*, float*);

struct SdfLaunch {
  SdfKernel kernel = nullptr;
  int ctas = 0;
};

// Once per surface object, on its device.
cudaError_t sdf_launch(const SGrid& g, const SBins& B, int sms, SdfLaunch* out) {
  int per = 0;
  const bool wide = g.h > 1.98f * B.b;
  SdfKernel k = wide ? k_sdf<2, 1, 1, false> : k_sdf<1, 2, 2, false>;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, SDF_THREADS, 0);
  const long long held = (long long)sms * std::max(per, 1);  // CTAs
  const auto over = [&](int a, int n) { return (long long)((g.c[a] + n - 1) / n); };
  const long long groups =
      wide ? over(0, 4) * g.c[1] * g.c[2] : over(0, 2) * over(1, 2) * over(2, 2);
  out->ctas = (int)held;
  if (groups < 4 * SDF_WARPS * held) {  // four rounds of warps
    const bool pairs = !wide && groups < SDF_WARPS * held;
    k = wide ? k_sdf<2, 1, 1, true> : pairs ? k_sdf<1, 1, 1, true> : k_sdf<1, 2, 1, true>;
    out->ctas = (int)(over(0, wide ? 8 : 4) * over(1, wide || pairs ? 2 : 4) * over(2, 2));
  }
  out->kernel = k;
  return e;
}

// ------------------------------------------------------------------ marching cubes

// Corners of a tile by 32-bit arithmetic: the tile's first corner once, then offsets from it.
struct TileCorner {
  unsigned int i, j, k;
  __device__ __forceinline__ TileCorner(const SGrid& g, long long base) {
    int a, b, c;
    corner_ijk(g, base, a, b, c);
    i = a, j = b, k = c;
  }
  // the corner `off` (< SC_TILE) places on
  __device__ __forceinline__ void at(const SGrid& g, unsigned int off, int (&ijk)[3]) const {
    const unsigned int x = i + off, y = j + x / (unsigned)g.c[0];
    ijk[0] = (int)(x % (unsigned)g.c[0]);
    ijk[1] = (int)(y % (unsigned)g.c[1]);
    ijk[2] = (int)(k + y / (unsigned)g.c[1]);
  }
};

// Triangles per case, in shared memory (lanes look up different cases).  CTA-uniform.
__device__ __forceinline__ void load_ntri(uint8_t (&s)[256]) {
  for (int t = threadIdx.x; t < 256; t += blockDim.x) s[t] = c_mc.ntri[t];
  __syncthreads();
}

// Every corner's code (bits 0..2: crossing edges along x, y, z; bits 8..15: the case of the
// cube it is the lowest corner of, 0 where there is none) and the tiles' counts, vertices +
// (triangles << 32).  A thread compares the four corners of its x, all its tile's loads in
// flight at once; its right neighbour's come through shared memory.  Bound by issue (135 instructions per 32
// corners, the ALU pipe at 72 %): 4.2 M corners 25 us from a cold cache; the counts alone, with
// eight loads and 64-bit divisions per corner, took 28, and the codes came with the vertices.
__global__ void __launch_bounds__(SC_THREADS) k_mc_classify(const SGrid g,
                                                            const float* __restrict__ phi,
                                                            uint16_t* __restrict__ code,
                                                            u64* __restrict__ tile_sum) {
  __shared__ u64 sm[72];
  __shared__ uint8_t s_ntri[256];
  load_ntri(s_ntri);
  const long long base = (long long)blockIdx.x * SC_TILE;
  const long long sy = g.c[0], sz = (long long)g.c[0] * g.c[1];
  __shared__ uint8_t s_col[SC_TILE + 1];
  // Bits 0, 2, 4, 6 of a column: the corners (0, 0), (1, 0), (0, 1), (1, 1) in (y, z) inside;
  // bits 1, 3, 5: the corner has a neighbour in x, y, z.  (Where it has none, its own value
  // stands in and nobody looks at it.)
  const auto column = [&](long long c, const int (&ijk)[3]) {
    const bool x = ijk[0] < g.n[0], y = ijk[1] < g.n[1], z = ijk[2] < g.n[2];
    const float* p = phi + c;
    const float a = p[0], b = p[y ? sy : 0], d = p[z ? sz : 0], e = p[(y ? sy : 0) + (z ? sz : 0)];
    return (unsigned)(a < g.iso) | (unsigned)(b < g.iso) << 2 | (unsigned)(d < g.iso) << 4 |
           (unsigned)(e < g.iso) << 6 | (unsigned)x << 1 | (unsigned)y << 3 | (unsigned)z << 5;
  };
  // the thread's corners are SC_THREADS apart: a step of (di, dj, dk) with carries
  const TileCorner tc(g, base);
  int ijk[3];
  tc.at(g, threadIdx.x, ijk);
  const int plane = (int)min(sz, 2ll * SC_THREADS);  // (a larger one gives the same step)
  const int dk = SC_THREADS / plane, dj = SC_THREADS % plane / g.c[0],
            di = SC_THREADS % plane % g.c[0];
  unsigned int col[SC_ROWS];
#pragma unroll
  for (int r = 0; r < SC_ROWS; ++r) {
    const long long c = base + r * SC_THREADS + threadIdx.x;
    col[r] = c < g.ncorners ? column(c, ijk) : 0u;
    ijk[0] += di;
    ijk[1] += dj;
    ijk[2] += dk;
    if (ijk[0] >= g.c[0]) ijk[0] -= g.c[0], ++ijk[1];
    if (ijk[1] >= g.c[1]) ijk[1] -= g.c[1], ++ijk[2];
  }
#pragma unroll
  for (int r = 0; r < SC_ROWS; ++r) s_col[r * SC_THREADS + threadIdx.x] = (uint8_t)col[r];
  if (threadIdx.x == 0) {
    tc.at(g, SC_TILE, ijk);
    s_col[SC_TILE] = base + SC_TILE < g.ncorners ? column(base + SC_TILE, ijk) : 0u;
  }
  __syncthreads();
  u64 sum = 0;
#pragma unroll
  for (int r = 0; r < SC_ROWS; ++r) {
    const unsigned int off = r * SC_THREADS + threadIdx.x;
    if (base + off >= g.ncorners) break;
    const unsigned int m = s_col[off], mx = s_col[off + 1];
    const bool x = m & 2u, y = m & 8u, z = m & 32u;
    unsigned int flags = 0;
    if (x && ((m ^ mx) & 1u)) flags |= 1u;
    if (y && ((m ^ (m >> 2)) & 1u)) flags |= 2u;
    if (z && ((m ^ (m >> 4)) & 1u)) flags |= 4u;
    const unsigned int cs = (x && y && z) ? (m & 0x55u) | ((mx & 0x55u) << 1) : 0u;
    code[base + off] = (uint16_t)(flags | (cs << 8));
    sum += (u64)__popc(flags) | ((u64)s_ntri[cs] << 32);
  }
  u64 tot;
  block_excl_scan(sum, tot, sm);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

// A thread's eight consecutive corners' codes (corners past the end: 0).
__device__ __forceinline__ void load_codes(const uint16_t* code, long long c, long long n,
                                           unsigned int (&v)[8]) {
  if (c + 8 <= n) {
    const uint4 t = *reinterpret_cast<const uint4*>(code + c);
    const unsigned int w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = (w[q / 2] >> (16 * (q & 1))) & 0xffffu;
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = c + q < n ? code[c + q] : 0u;
  }
}

// The vertices, and the offsets of the corners that have any vertex or triangle (nobody reads
// the others').  Most corners have none: a thread looks at eight, one scan per tile does, and
// each warp lists its own that have any, so that its lanes share them evenly.
// 4.2 M corners, 53 thousand vertices: 14 us, of 61 with a scan per 256 corners, the
// classification again and every offset written.
__global__ void __launch_bounds__(SC_THREADS) k_mc_vertices(const SGrid g,
                                                            const float* __restrict__ phi,
                                                            const uint16_t* __restrict__ code,
                                                            const u64* __restrict__ tile_off,
                                                            unsigned int* __restrict__ voff,
                                                            unsigned int* __restrict__ toff,
                                                            float* __restrict__ vert,
                                                            long long* __restrict__ vedge,
                                                            unsigned int parts) {
  static_assert(SC_ROWS == 8, "eight corners a thread");
  __shared__ u64 sm[72];
  __shared__ uint8_t s_ntri[256];
  __shared__ ushort4 s_item[SC_THREADS / 32][256];  // {corner, code, vertices, triangles before}
  load_ntri(s_ntri);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned int tile = blockIdx.x / parts, part = blockIdx.x % parts;
  const long long base = (long long)tile * SC_TILE;
  unsigned int cd[8];
  load_codes(code, base + 8 * threadIdx.x, g.ncorners, cd);
  u64 own = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q)
    own += (u64)__popc(cd[q] & 7u) | ((u64)s_ntri[cd[q] >> 8] << 32);
  u64 tot;
  const u64 off = tile_off[tile], ex = block_excl_scan(own, tot, sm);
  // the tile's own counts (at most 3 and 12 a corner) fit 16 bits
  unsigned int nv = (unsigned int)(ex & 0xffffffffull), nt = (unsigned int)(ex >> 32);
  int n = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const unsigned int t = s_ntri[cd[q] >> 8], v = __popc(cd[q] & 7u);
    const unsigned int some = __ballot_sync(0xffffffffu, v + t != 0u);
    if (v + t != 0u)
      s_item[warp][n + __popc(some & ((1u << lane) - 1u))] =
          make_ushort4((unsigned short)(8 * threadIdx.x + q), (unsigned short)cd[q],
                       (unsigned short)nv, (unsigned short)nt);
    n += __popc(some);
    nv += v;
    nt += t;
  }
  __syncwarp();
  if (n == 0) return;
  const TileCorner tc(g, base);
  const long long st[3] = {1, g.c[0], (long long)g.c[0] * g.c[1]};
  for (int m = (int)part * 32 + lane; m < n; m += 32 * (int)parts) {
    const ushort4 it = s_item[warp][m];
    const long long c = base + it.x;
    unsigned int v = (unsigned int)(off & 0xffffffffull) + it.z;
    voff[c] = v;
    toff[c] = (unsigned int)(off >> 32) + it.w;
    if (!(it.y & 7u)) continue;
    int ijk[3];
    tc.at(g, it.x, ijk);
    const float pa = phi[c];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (!((it.y >> a) & 1u)) continue;
      const float pb = phi[c + st[a]];
      const float t = (g.iso - pa) / (pb - pa);
#pragma unroll
      for (int d = 0; d < 3; ++d)
        vert[3 * (size_t)v + d] = g.o[d] + g.h * ((float)ijk[d] + (d == a ? t : 0.0f));
      vedge[v] = 3 * c + a;
      ++v;
    }
  }
}

__device__ __forceinline__ unsigned int vertex_of_edge(const SGrid& g, long long c, int e,
                                                       const unsigned int* voff,
                                                       const uint16_t* code) {
  const int a = e >> 2;
  const int lo = (a == 0) ? 1 : 0, hi = (a == 2) ? 1 : 2;
  int off[3] = {0, 0, 0};
  off[lo] = e & 1;
  off[hi] = (e >> 1) & 1;
  const long long cc = c + off[0] + (long long)g.c[0] * (off[1] + (long long)g.c[1] * off[2]);
  const int fl = code[cc] & 7;
  return voff[cc] + __popc(fl & ((1 << a) - 1));
}

// n / A for a triangle of unit normal n and area A: 2 (e1 x e2) / |e1 x e2|^2.
__device__ __forceinline__ void tri_weight(const float* __restrict__ vert, const int (&t)[3],
                                           float* __restrict__ tw) {
  const float* a = vert + 3 * (size_t)t[0];
  const float* b = vert + 3 * (size_t)t[1];
  const float* c = vert + 3 * (size_t)t[2];
  const float ax = a[0], ay = a[1], az = a[2];
  const float e1x = b[0] - ax, e1y = b[1] - ay, e1z = b[2] - az;
  const float e2x = c[0] - ax, e2y = c[1] - ay, e2z = c[2] - az;
  const float nx = e1y * e2z - e1z * e2y, ny = e1z * e2x - e1x * e2z, nz = e1x * e2y - e1y * e2x;
  const float l2 = nx * nx + ny * ny + nz * nz;
  const float s = (l2 > 0.0f) ? 2.0f / l2 : 0.0f;
  tw[0] = s * nx;
  tw[1] = s * ny;
  tw[2] = s * nz;
}

// Triangles and their weights.  A warp looks at 256 corners, eight a lane, and lists those
// whose cube has triangles; then four lanes take a cube.  4.2 M corners, 106 thousand triangles:
// 14 us, of 22 with a thread per corner and the weights in a pass of their own.
__global__ void __launch_bounds__(SC_THREADS) k_mc_triangles(const SGrid g,
                                                             const unsigned int* __restrict__ voff,
                                                             const unsigned int* __restrict__ toff,
                                                             const uint16_t* __restrict__ code,
                                                             const float* __restrict__ vert,
                                                             int* __restrict__ tri,
                                                             float* __restrict__ tw,
                                                             unsigned int parts) {
  __shared__ uint16_t s_cube[SC_THREADS / 32][256];
  __shared__ uint8_t s_ntri[256];
  load_ntri(s_ntri);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned int tile = blockIdx.x / parts, part = blockIdx.x % parts;
  const long long c0 = (long long)tile * SC_TILE + 256 * warp;
  unsigned int cd[8];
  load_codes(code, c0 + 8 * lane, g.ncorners, cd);
  int n = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const bool any = s_ntri[cd[q] >> 8] != 0;
    const unsigned int some = __ballot_sync(0xffffffffu, any);
    if (any) s_cube[warp][n + __popc(some & ((1u << lane) - 1u))] = (uint16_t)(8 * lane + q);
    n += __popc(some);
  }
  __syncwarp();
  for (int m = (int)part * 8 + (lane >> 2); m < n; m += 8 * (int)parts) {
    const long long c = c0 + s_cube[warp][m];
    const int cs = code[c] >> 8;
    const unsigned int t0 = toff[c];
    for (int t = lane & 3; t < s_ntri[cs]; t += 4) {
      int v[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) v[q] = (int)vertex_of_edge(g, c, c_mc.tri[cs][t][q], voff, code);
      const size_t o = 3 * ((size_t)t0 + t);
#pragma unroll
      for (int q = 0; q < 3; ++q) tri[o + q] = v[q];
      tri_weight(vert, v, tw + o);
    }
  }
}

// The weights of the triangles at a vertex, gathered from the four cubes around its edge by
// four lanes, a cube each, and added in the cubes' order.  Bound by latency (a cube's offsets,
// its triangles, their weights): 53 thousand vertices 8 us, of 19.5 with a
// thread per vertex.
__global__ void k_mc_normals(const SGrid g, long long nv,
                             const long long* __restrict__ vedge,
                             const unsigned int* __restrict__ toff,
                             const uint16_t* __restrict__ code, const int* __restrict__ tri,
                             const float* __restrict__ tw, float* __restrict__ nrm) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long v = t >> 2;
  const int q = (int)(t & 3);
  float sx = 0.0f, sy = 0.0f, sz = 0.0f;
  if (v < nv) {
    const long long e = vedge[v];
    const long long c = e / 3;
    const int a = (int)(e - 3 * c);
    int ijk[3];
    corner_ijk(g, c, ijk[0], ijk[1], ijk[2]);
    const long long st[3] = {1, g.c[0], (long long)g.c[0] * g.c[1]};
    const int iu = (a == 0) ? ijk[1] : ijk[0], iw = (a == 2) ? ijk[1] : ijk[2];
    const int nu = (a == 0) ? g.n[1] : g.n[0], nw = (a == 2) ? g.n[1] : g.n[2];
    const long long su = (a == 0) ? st[1] : st[0], sw = (a == 2) ? st[1] : st[2];
    const int bu = q & 1, bw = q >> 1;
    if (iu - bu >= 0 && iw - bw >= 0 && iu - bu < nu && iw - bw < nw) {
      const long long cc = c - bu * su - bw * sw;
      const unsigned int t0 = toff[cc];
      const int nt = c_mc.ntri[code[cc] >> 8];
      for (int n = 0; n < nt; ++n) {
        const size_t o = 3 * ((size_t)t0 + n);
        const float wx = tw[o], wy = tw[o + 1], wz = tw[o + 2];
        if (tri[o] == (int)v || tri[o + 1] == (int)v || tri[o + 2] == (int)v) {
          sx += wx;
          sy += wy;
          sz += wz;
        }
      }
    }
  }
  const int l0 = threadIdx.x & 28;
  float s[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    s[0] += __shfl_sync(0xffffffffu, sx, l0 + k);
    s[1] += __shfl_sync(0xffffffffu, sy, l0 + k);
    s[2] += __shfl_sync(0xffffffffu, sz, l0 + k);
  }
  if (v >= nv || q != 0) return;
  const float l = sqrtf(s[0] * s[0] + s[1] * s[1] + s[2] * s[2]);
  const float f = (l > 0.0f) ? 1.0f / l : 0.0f;
  nrm[3 * v] = s[0] * f;
  nrm[3 * v + 1] = s[1] * f;
  nrm[3 * v + 2] = s[2] * f;
}

// CTAs per tile in the passes over lists, each with its part of every warp's list: few tiles
// leave most of the chip idle while a warp has a list of up to 256 corners.  Up to eight CTAs
// per SM in all: flip_surface_mesh of random fields on 32^3 cells (18 tiles, every corner
// crosses) 112 -> 71 us, on 16^3 105 -> 67, of a field with a surface around single particles
// on 150 x 40 x 90 (275 tiles) 99 -> 78 (two per SM 99, four 82, sixteen 79); with a thread
// per corner 105, 96 and 93.
unsigned int mc_parts(long long ntiles, int sms) {
  unsigned int parts = 1;
  while (parts < 8u && 2 * parts * ntiles <= 8ll * sms) parts *= 2;
  return parts;
}

unsigned int blocks_for(long long n, int threads) {
  return (unsigned int)std::max<long long>(1, (n + threads - 1) / threads);
}

}  // namespace

// ------------------------------------------------------------------ object

struct flip_surface {
  flip_surface_params prm{};
  SGrid g{};
  SBins B{};
  SdfLaunch sdf;
  int sms = 0;  // of its device
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float* phi = nullptr;
  // bins (grow with the particle count)
  unsigned int* bin_count = nullptr;
  unsigned int* bin_start = nullptr;
  long long part_cap = 0;
  int* pbin = nullptr;
  unsigned int* prank = nullptr;
  float4* pos = nullptr;
  // marching cubes
  unsigned int* voff = nullptr;
  unsigned int* toff = nullptr;
  uint16_t* code = nullptr;
  u64* tile = nullptr;       // tile sums + the total
  long long tile_cap = 0;
  long long vcap = 0, tcap = 0;
  float* vert = nullptr;
  float* nrm = nullptr;
  long long* vedge = nullptr;
  int* tri = nullptr;
  float* tw = nullptr;
  long long nv = 0, nt = 0;
  u64* htotal = nullptr;     // pinned
};

namespace {

void sfree(void* p) {
  if (p) cudaFree(p);
}

// Replaces p by a fresh device array of n (>= 1) elements.
template <class T>
int realloc_n(T*& p, long long n) {
  sfree(p);
  p = nullptr;
  SURF_CUDA(cudaMalloc(reinterpret_cast<void**>(&p), sizeof(T) * (size_t)std::max<long long>(n, 1)));
  return FLIP_OK;
}

}  // namespace

namespace flipk {
bool handle_particles(flip_handle* h, PartView* p, long long* np, cudaStream_t* s);
}

extern "C" {

void flip_surface_default_params(const flip_params* p, flip_surface_params* out) {
  if (!out) return;
  std::memset(out, 0, sizeof(*out));
  if (!p) return;
  for (int a = 0; a < 3; ++a) {
    out->n[a] = p->n[a];
    out->origin[a] = 0.0;
  }
  out->h = p->dx;
  out->radius = 0.5 * p->dx;
  out->search_radius = 2.0 * p->dx;
  out->iso = 0.0;
}

int flip_surface_create(const flip_surface_params* sp, void* stream, flip_surface** out) {
  if (!sp || !out) return sfail(FLIP_E_ARG, "params or out is NULL");
  *out = nullptr;
  for (int a = 0; a < 3; ++a)
    if (sp->n[a] < 1 || sp->n[a] > 1024) return sfail(FLIP_E_ARG, "n must be in [1, 1024]");
  if (!(sp->h > 0.0) || !std::isfinite(sp->h)) return sfail(FLIP_E_ARG, "h must be > 0");
  if (!(sp->search_radius > 0.0) || !std::isfinite(sp->search_radius))
    return sfail(FLIP_E_ARG, "search_radius must be > 0");
  if (!(sp->radius >= 0.0) || !(sp->radius < sp->search_radius))
    return sfail(FLIP_E_ARG, "radius must be in [0, search_radius)");
  if (!std::isfinite(sp->iso)) return sfail(FLIP_E_ARG, "iso must be finite");
  for (int a = 0; a < 3; ++a)
    if (!std::isfinite(sp->origin[a])) return sfail(FLIP_E_ARG, "origin must be finite");
  {
    // particle bins (edge search_radius / 2) are indexed in 32 bits
    const double bb = (double)(0.5f * (float)sp->search_radius);  // the bin edge used below
    double nbins = 1.0;
    for (int a = 0; a < 3; ++a)
      nbins *= std::ceil((sp->n[a] * sp->h + 2.0 * sp->search_radius) / bb) + 1.0;
    if (!(nbins <= 2147483647.0))
      return sfail(FLIP_E_ARG, "bin grid too large (over 2^31 bins): search_radius is too small "
                               "for the sampling grid");
  }
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0)
    return sfail(FLIP_E_NOGPU, "no CUDA device");
  if (int rc = ensure_table()) return rc;
  flip_surface* s = new (std::nothrow) flip_surface;
  if (!s) return sfail(FLIP_E_OOM, "host allocation failed");
  s->prm = *sp;
  SGrid& g = s->g;
  for (int a = 0; a < 3; ++a) {
    g.n[a] = sp->n[a];
    g.c[a] = sp->n[a] + 1;
    g.o[a] = (float)sp->origin[a];
  }
  g.ncorners = (long long)g.c[0] * g.c[1] * g.c[2];
  g.h = (float)sp->h;
  g.iso = (float)sp->iso;
  SBins& B = s->B;
  B.R = (float)sp->search_radius;
  B.R2 = B.R * B.R;
  B.inv_R2 = 1.0f / B.R2;
  B.r = (float)sp->radius;
  B.b = 0.5f * B.R;
  B.inv_b = 1.0f / B.b;
  B.nbins = 1;
  for (int a = 0; a < 3; ++a) {
    B.o[a] = g.o[a] - B.R;
    B.nb[a] = (int)std::ceil((sp->n[a] * sp->h + 2.0 * sp->search_radius) / B.b) + 1;
    B.nbins *= B.nb[a];
  }
  int rc = FLIP_OK;
  auto step = [&](cudaError_t e, const char* what) {
    if (rc == FLIP_OK && e != cudaSuccess) rc = scuda(e, what);
  };
  if (stream) {
    s->stream = static_cast<cudaStream_t>(stream);
  } else {
    step(cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking), "cudaStreamCreate");
    s->own_stream = rc == FLIP_OK;
  }
  int dev = 0;
  step(cudaGetDevice(&dev), "cudaGetDevice");
  step(cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
  step(sdf_launch(g, B, s->sms, &s->sdf), "scalar field launch shape");
  const long long nc = g.ncorners;
  step(cudaMalloc(&s->phi, sizeof(float) * nc), "cudaMalloc(phi)");
  step(cudaMalloc(&s->voff, sizeof(unsigned int) * nc), "cudaMalloc(voff)");
  step(cudaMalloc(&s->toff, sizeof(unsigned int) * nc), "cudaMalloc(toff)");
  step(cudaMalloc(&s->code, sizeof(uint16_t) * nc), "cudaMalloc(code)");
  step(cudaMalloc(&s->bin_count, sizeof(unsigned int) * B.nbins), "cudaMalloc(bins)");
  step(cudaMalloc(&s->bin_start, sizeof(unsigned int) * (B.nbins + 1)), "cudaMalloc(bins)");
  step(cudaMallocHost(&s->htotal, sizeof(u64)), "cudaMallocHost");
  if (rc == FLIP_OK) {
    const long long ntiles = (std::max(nc, B.nbins + 1) + SC_TILE - 1) / SC_TILE;
    rc = realloc_n(s->tile, ntiles + 1);
    if (rc == FLIP_OK) s->tile_cap = ntiles + 1;
  }
  if (rc == FLIP_OK) {
    // corners start outside: phi = R - r until a field is computed or set
    k_fill<<<blocks_for(nc, 256), 256, 0, s->stream>>>(s->phi, nc, B.R - B.r);
    step(cudaGetLastError(), "k_fill");
    step(cudaStreamSynchronize(s->stream), "cudaStreamSynchronize");
  }
  if (rc != FLIP_OK) {
    flip_surface_destroy(s);
    return rc;
  }
  *out = s;
  return FLIP_OK;
}

int flip_surface_case_table(uint8_t ntri[256], uint8_t* tri) {
  if (!ntri || !tri) return sfail(FLIP_E_ARG, "NULL output");
  static_assert(MC_MAXT == FLIP_SURF_MAX_TRI, "table width");
  McTable T;
  if (!build_table(T)) return sfail(FLIP_E_CUDA, "marching-cubes table generation failed");
  std::memcpy(ntri, T.ntri, sizeof(T.ntri));
  std::memcpy(tri, T.tri, sizeof(T.tri));
  return FLIP_OK;
}

void flip_surface_destroy(flip_surface* s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  for (void* p : {(void*)s->phi, (void*)s->bin_count, (void*)s->bin_start, (void*)s->pbin,
                  (void*)s->prank, (void*)s->pos, (void*)s->voff, (void*)s->toff,
                  (void*)s->code, (void*)s->tile, (void*)s->vert, (void*)s->nrm,
                  (void*)s->vedge, (void*)s->tri, (void*)s->tw})
    sfree(p);
  if (s->htotal) cudaFreeHost(s->htotal);
  if (s->own_stream) cudaStreamDestroy(s->stream);
  delete s;
}

int flip_surface_sdf(flip_surface* s, flip_handle* h) {
  if (!s || !h) return sfail(FLIP_E_ARG, "surface or handle is NULL");
  PartView P;
  long long np = 0;
  cudaStream_t hs = nullptr;
  if (!handle_particles(h, &P, &np, &hs)) return sfail(FLIP_E_ARG, "bad handle");
  // order after the handle's queued work
  cudaEvent_t ev;
  SURF_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  SURF_CUDA(cudaEventRecord(ev, hs));
  SURF_CUDA(cudaStreamWaitEvent(s->stream, ev, 0));
  cudaEventDestroy(ev);
  if (np > s->part_cap) {
    s->part_cap = 0;
    if (int rc = realloc_n(s->pbin, np)) return rc;
    if (int rc = realloc_n(s->prank, np)) return rc;
    if (int rc = realloc_n(s->pos, np)) return rc;
    s->part_cap = np;
  }
  const cudaStream_t st = s->stream;
  SURF_CUDA(cudaMemsetAsync(s->bin_count, 0, sizeof(unsigned int) * s->B.nbins, st));
  if (np > 0) {
    k_sbin_count<<<blocks_for(np, 256), 256, 0, st>>>(P, np, s->B, s->bin_count, s->pbin,
                                                      s->prank);
  }
  BinScan bs{s->bin_count, s->bin_start, s->B.nbins};
  tile_scan(bs, s->B.nbins + 1, s->tile, s->tile + s->tile_cap - 1, st);
  if (np > 0) {
    k_sbin_scatter<<<blocks_for(np, 256), 256, 0, st>>>(P, np, s->pbin, s->prank, s->bin_start,
                                                        s->pos);
  }
  s->sdf.kernel<<<s->sdf.ctas, SDF_THREADS, 0, st>>>(s->g, s->B, s->bin_start, s->pos, s->phi);
  SURF_CUDA(cudaGetLastError());
  return FLIP_OK;
}

int flip_surface_set_field(flip_surface* s, const float* phi, int32_t src_is_device) {
  if (!s || !phi) return sfail(FLIP_E_ARG, "surface or phi is NULL");
  SURF_CUDA(cudaMemcpyAsync(s->phi, phi, sizeof(float) * s->g.ncorners,
                            src_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                            s->stream));
  SURF_CUDA(cudaStreamSynchronize(s->stream));
  return FLIP_OK;
}

int flip_surface_mesh(flip_surface* s, int64_t* n_vertices, int64_t* n_triangles) {
  if (!s) return sfail(FLIP_E_ARG, "surface is NULL");
  const cudaStream_t st = s->stream;
  const long long nc = s->g.ncorners;
  const long long ntiles = (nc + SC_TILE - 1) / SC_TILE;
  u64* total = s->tile + s->tile_cap - 1;
  k_mc_classify<<<(unsigned)ntiles, SC_THREADS, 0, st>>>(s->g, s->phi, s->code, s->tile);
  k_tile_scan<<<1, TS_THREADS, 0, st>>>(s->tile, ntiles, total);
  SURF_CUDA(cudaMemcpyAsync(s->htotal, total, sizeof(u64), cudaMemcpyDeviceToHost, st));
  SURF_CUDA(cudaStreamSynchronize(st));
  // Vertices (crossing edges, at most 3 per corner) never exceed 2^32, so the low
  // word is exact.  Each crossing edge is a vertex of one fan polygon in each of at
  // most 4 cubes, and a k-gon gives k - 2 triangles, so triangles <= 4 * vertices:
  // below 2^31 vertices / 4 the high word cannot have wrapped either.
  const long long nv = (long long)(*s->htotal & 0xffffffffull);
  const long long nt = (long long)(*s->htotal >> 32);
  if (4 * nv >= (1ll << 31) || nt >= (1ll << 31))
    return sfail(FLIP_E_SIZE, "mesh too large for int32 indices (2^29 vertices or more)");
  if (nv > s->vcap) {
    s->vcap = 0;
    s->nv = 0;
    if (int rc = realloc_n(s->vert, 3 * nv)) return rc;
    if (int rc = realloc_n(s->nrm, 3 * nv)) return rc;
    if (int rc = realloc_n(s->vedge, nv)) return rc;
    s->vcap = nv;
  }
  if (nt > s->tcap) {
    s->tcap = 0;
    s->nt = 0;
    if (int rc = realloc_n(s->tri, 3 * nt)) return rc;
    if (int rc = realloc_n(s->tw, 3 * nt)) return rc;
    s->tcap = nt;
  }
  if (nv > 0) {  // (a triangle has vertices)
    const unsigned int parts = mc_parts(ntiles, s->sms), ctas = (unsigned int)ntiles * parts;
    k_mc_vertices<<<ctas, SC_THREADS, 0, st>>>(s->g, s->phi, s->code, s->tile, s->voff, s->toff,
                                               s->vert, s->vedge, parts);
    if (nt > 0)
      k_mc_triangles<<<ctas, SC_THREADS, 0, st>>>(s->g, s->voff, s->toff, s->code, s->vert,
                                                  s->tri, s->tw, parts);
    k_mc_normals<<<blocks_for(4 * nv, 256), 256, 0, st>>>(s->g, nv, s->vedge, s->toff, s->code,
                                                          s->tri, s->tw, s->nrm);
  }
  SURF_CUDA(cudaGetLastError());
  SURF_CUDA(cudaStreamSynchronize(st));
  s->nv = nv;
  s->nt = nt;
  if (n_vertices) *n_vertices = nv;
  if (n_triangles) *n_triangles = nt;
  return FLIP_OK;
}

size_t flip_surface_bytes(const flip_surface* s, flip_surface_field which) {
  if (!s) return 0;
  switch (which) {
    case FLIP_SURF_FIELD: return sizeof(float) * (size_t)s->g.ncorners;
    case FLIP_SURF_VERTICES: case FLIP_SURF_NORMALS: return 12 * (size_t)s->nv;
    case FLIP_SURF_TRIANGLES: return 12 * (size_t)s->nt;
    case FLIP_SURF_VERTEX_EDGE: return 8 * (size_t)s->nv;
    default: return 0;
  }
}

int flip_surface_read(flip_surface* s, flip_surface_field which, void* dst, size_t bytes,
                      int32_t dst_is_device) {
  if (!s) return sfail(FLIP_E_ARG, "surface is NULL");
  if (which < FLIP_SURF_FIELD || which > FLIP_SURF_VERTEX_EDGE)
    return sfail(FLIP_E_ARG, "unknown field");
  const size_t need = flip_surface_bytes(s, which);
  if (bytes != need) return sfail(FLIP_E_SIZE, "bytes must be " + std::to_string(need));
  if (need == 0) return FLIP_OK;
  if (!dst) return sfail(FLIP_E_ARG, "dst is NULL");
  const void* src = nullptr;
  switch (which) {
    case FLIP_SURF_FIELD: src = s->phi; break;
    case FLIP_SURF_VERTICES: src = s->vert; break;
    case FLIP_SURF_NORMALS: src = s->nrm; break;
    case FLIP_SURF_TRIANGLES: src = s->tri; break;
    case FLIP_SURF_VERTEX_EDGE: src = s->vedge; break;
  }
  SURF_CUDA(cudaMemcpyAsync(dst, src, bytes,
                            dst_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                            s->stream));
  SURF_CUDA(cudaStreamSynchronize(s->stream));
  return FLIP_OK;
}

}  // extern "C"
