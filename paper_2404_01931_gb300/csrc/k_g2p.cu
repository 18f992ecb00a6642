// k_g2p.cu — grid-to-particle transfer with the PIC/FLIP blend (Sec. 2.1.4,
// 3.1.8), forward-Euler advection and the wall clamp (Sec. 3.1.3), fused with
// the histogram of the next step's binning.
//
// One CTA takes one active 8x8x8 brick at a time (its particles are one
// contiguous range after binning; they stream into shared memory by bulk copies,
// see below).  It first stages in shared memory the
// pressure of the brick plus a one-cell halo, then, for every component, the
// face nodes any of the brick's particles can reach (the 9x10x10 tile P2G also
// uses): U = u_new (Eq. 5 with gravity and walls, face_unew's arithmetic) and
// dU = u_new - u_old.  Each face value is so computed once per brick instead of
// once per particle that touches it.  Then one thread per particle interpolates
// (U, dU) with P2G's weights and applies
//     v <- r (v + interp(dU)) + (1 - r) interp(U)
//     x <- clamp(x + dt v, skin, n dx - skin)      (or dt interp(U), grid advection)
// and computes the key of the cell it moved to and its rank there.  Ranks come
// from one histogram atomic per distinct key in a warp (lanes with the same key
// take consecutive ranks), which is all the next step's counting sort needs.
//
// The pressure slab of a brick (the 10 x 10 x 10 cells [b - 1, b + 8] per axis)
// is staged by one TMA tensor copy (cp.async.bulk.tensor) when the handle has a
// tensor map of its pressure (row pitches a multiple of 16 bytes): the copy starts
// at x = b0 - XOFF so that its first coordinate is 16-byte aligned, rows are SPX
// cells wide, and cells outside the grid arrive as 0.  Otherwise, and in the
// batched kernel, the same tile is filled with plain loads.
#include <cudaTypedefs.h>

#include <cstring>

#include "flip_kernels.cuh"

namespace flipk {

constexpr int G2P_THREADS = 256;
constexpr unsigned int G2P_MAX_SPLIT = 8;
constexpr int G2P_TILE = 904;     // >= 9 * 10 * 10 face nodes per component

template <int D>
struct FaceTile {
  static constexpr int X = (D == 0) ? 9 : 10;
  static constexpr int Y = (D == 1) ? 9 : 10;
  static constexpr int Z = (D == 2) ? 9 : 10;
  static constexpr int N = X * Y * Z;
};

// The staged pressure tile: element type (the float pair of mixed mode, or FP32),
// row width SPX and the x offset XOFF of its first cell from the brick origin, so
// that XOFF * sizeof(T) and SPX * sizeof(T) are multiples of 16 bytes.
template <bool PAIR>
struct PTile;
template <>
struct PTile<true> {
  using T = float2;
  static constexpr int SPX = 12, XOFF = 2;
};
template <>
struct PTile<false> {
  using T = float;
  static constexpr int SPX = 16, XOFF = 4;
};
template <bool PAIR>
constexpr int PTILE_N = 10 * 10 * PTile<PAIR>::SPX;

// ---------------------------------------------------------------- bulk copies
// Particles stream into shared memory in chunks of G2P_THREADS (one per thread)
// by cp.async.bulk (the Blackwell/Hopper bulk-copy engine), double-buffered and
// tracked by an mbarrier per buffer, so a chunk's loads are in flight while the
// previous chunk is processed.  A bulk copy starts and ends on 16-byte
// boundaries: a chunk [q0, q1) is copied as [q0 & ~3, (q1 + 3) & ~3), which stays
// inside its array (every array of the arena is padded to 256 bytes).
constexpr int G2P_CHUNK_PAD = G2P_THREADS + 8;
// After a wait has given up (StepConsts::wait_ns), the copies still in flight are
// waited for once more, up to this limit, before the CTA leaves: its shared memory
// must not be handed to another CTA while the copy engine still writes into it.
constexpr unsigned long long G2P_DRAIN_NS = 1000000000ull;

__device__ __forceinline__ unsigned int smem_u32(const void* p) {
  return (unsigned int)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned int parity) {
  unsigned int ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for phase `parity` of the barrier; false after limit_ns.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned int parity,
                                          unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_timer_ns() - t0 > limit_ns) return false;
  return true;
}

// One 3-D tiled tensor copy of the box at (x, y, z) into dst, completing on bar.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned int bytes,
                                         unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// One thread: copy particles [q0, q1) of x, y, z, u, v, w into `dst` (the
// buffer then starts at particle q0 rounded down to 4), completing on `bar`.
__device__ __forceinline__ void issue_chunk(const PartView& P, unsigned int q0, unsigned int q1,
                                            float (*dst)[G2P_CHUNK_PAD],
                                            unsigned long long* bar) {
  const unsigned int a0 = q0 & ~3u, a1 = (q1 + 3u) & ~3u;
  const unsigned int bytes = 4u * (a1 - a0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  mbar_expect_tx(bar, 6u * bytes);
  const float* src[6] = {P.x, P.y, P.z, P.u, P.v, P.w};
#pragma unroll
  for (int a = 0; a < 6; ++a) bulk_g2s(dst[a], src[a] + a0, bytes, bar);
}

// Pressure difference p(+) - p(-) in the arithmetic of face_unew.
__device__ __forceinline__ float pdiff(float2 hp, float2 hm) {
  return __fadd_rn(__fsub_rn(hp.x, hm.x), __fsub_rn(hp.y, hm.y));
}
__device__ __forceinline__ float pdiff(float hp, float hm) { return __fsub_rn(hp, hm); }

// Stages component D's face tile: node (a, b, c) with a in [o0, o0 + X) etc.,
// o = brick origin on the own axis and origin - 1 on the others.  Nodes outside
// the face grid are never interpolated (the clamped weights keep every node in
// range) and are set to 0.
template <int D, bool PAIR>
__device__ __forceinline__ void stage_faces(const Grid& g, const StepConsts& K, int b0, int b1,
                                            int b2, const float* __restrict__ uo,
                                            const typename PTile<PAIR>::T* sp, float2* sud) {
  constexpr int TX = FaceTile<D>::X, TY = FaceTile<D>::Y, N = FaceTile<D>::N;
  const int o0 = (D == 0) ? b0 : b0 - 1, o1 = (D == 1) ? b1 : b1 - 1, o2 = (D == 2) ? b2 : b2 - 1;
  const int FX = g.nx + (D == 0), FY = g.ny + (D == 1), FZ = g.nz + (D == 2);
  const int nmax = (D == 0) ? g.nx : (D == 1) ? g.ny : g.nz;
  for (int t = threadIdx.x; t < N; t += G2P_THREADS) {
    const int ta = t % TX, tb = (t / TX) % TY, tc = t / (TX * TY);
    const int a = o0 + ta, b = o1 + tb, c = o2 + tc;
    float un = 0.0f, du = 0.0f;
    if (a >= 0 && b >= 0 && c >= 0 && a < FX && b < FY && c < FZ) {
      const float uov = __ldg(uo + (a + FX * (b + FY * c)));
      const int nd = (D == 0) ? a : (D == 1) ? b : c;
      if (nd != 0 && nd != nmax) {
        // pressure tile cell of (a, b, c) is (a - b0 + XOFF, b - b1 + 1, c - b2 + 1);
        // the minus cell is one step down along D
        constexpr int SPX = PTile<PAIR>::SPX, XOFF = PTile<PAIR>::XOFF;
        const int pc = (a - b0 + XOFF) + SPX * ((b - b1 + 1) + 10 * (c - b2 + 1));
        const int pm = pc - ((D == 0) ? 1 : (D == 1) ? SPX : 10 * SPX);
        const float dp = pdiff(sp[pc], sp[pm]);
        un = __fsub_rn(__fadd_rn(uov, K.gdt[D]), __fmul_rn(K.pscale, dp));
      }
      du = __fsub_rn(un, uov);
    }
    sud[t] = make_float2(un, du);
  }
}

// floor(v) for |v| < 2^22 by an addition rounded down, and the integer in its low bits: the
// conversion units have a fraction of the FP32 rate.
constexpr float FLOOR_MAGIC = 12582912.0f;  // 1.5 * 2^23
__device__ __forceinline__ float floor_small(float v, int& i) {
  const float m = __fadd_rd(v, FLOOR_MAGIC);
  i = __float_as_int(m) - __float_as_int(FLOOR_MAGIC);
  return __fsub_rn(m, FLOOR_MAGIC);
}

// cell_of for an x inside the domain (the same integer: both floors are exact).
__device__ __forceinline__ int cell_in(float x, float inv, int n) {
  const float p = __fmul_rn(x, inv);
  const float e = __fmaf_rn(x, inv, -p);
  int i;
  const float f = floor_small(p, i);
  if (p == f && e < 0.0f) --i;
  return min(max(i, 0), n - 1);
}

// One axis of a particle's interpolation, both kinds of nodes: the two nodes of the tile
// (lower index, two weights).  The weights are axis_weights', bit for bit: past the two
// roundings of x/dx and x/dx - 1/2 every difference is exact.  A position that the first
// takes to the end of its cell may stand at a node of weight 1 as the lower or as the
// upper of the two; the other's weight is 0 and the interpolant the same.
struct NodeW {
  int i;
  float w0, w1;
};
struct AxisG {
  NodeW face, cen;
};

// The faces are the tile's nodes 0 .. 8 (of the brick's eight cells), the centres (from one
// below the brick on) its nodes 0 .. 9, of which those outside the domain are not reached:
// centre 0 at the least, n - 1 at the most.  lo, hi: those centres, or the ends of what the
// brick's particles reach (b0 - 1, b0 + 7.5), which keep the indices in range.
__device__ __forceinline__ AxisG axis_g(float x, float inv, int b0, float lo, float hi) {
  constexpr float BELOW_8 = 7.9999995f;
  const float g = __fmul_rn(x, inv);
  const float p = fminf(fmaxf(__fsub_rn(g, (float)b0), 0.0f), 8.0f);
  const float c = fminf(fmaxf(__fsub_rn(g, 0.5f), lo), hi);
  AxisG a;
  a.face.w1 = __fsub_rn(p, floor_small(fminf(p, BELOW_8), a.face.i));
  a.face.w0 = __fsub_rn(1.0f, a.face.w1);
  a.cen.w1 = __fsub_rn(c, floor_small(c, a.cen.i));
  a.cen.w0 = __fsub_rn(1.0f, a.cen.w1);
  a.cen.i += 1 - b0;
  return a;
}

// Interpolates component D of (U, dU) from the staged tile: one packed two-lane FMA per
// node, each lane rounded like __fmaf_rn.
template <int D>
__device__ __forceinline__ float2 interp_tile(const AxisG& ax, const AxisG& ay, const AxisG& az,
                                              const float2* sud) {
  constexpr int TX = FaceTile<D>::X, TY = FaceTile<D>::Y;
  const NodeW& nx = (D == 0) ? ax.face : ax.cen;
  const NodeW& ny = (D == 1) ? ay.face : ay.cen;
  const NodeW& nz = (D == 2) ? az.face : az.cen;
  const float2* t = sud + (nx.i + TX * (ny.i + TY * nz.i));
  const float wy[2] = {ny.w0, ny.w1}, wz[2] = {nz.w0, nz.w1};
  float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int dz = 0; dz < 2; ++dz)
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const float wyz = __fmul_rn(wy[dy], wz[dz]);
      const float w0 = __fmul_rn(nx.w0, wyz), w1 = __fmul_rn(nx.w1, wyz);
      s = __ffma2_rn(make_float2(w0, w0), t[TX * (dy + TY * dz)], s);
      s = __ffma2_rn(make_float2(w1, w1), t[TX * (dy + TY * dz) + 1], s);
    }
  return s;
}

// Shared memory of a G2P CTA: the brick's staged tiles and the particle buffers.
template <bool PAIR>
struct G2pShared {
  __align__(128) typename PTile<PAIR>::T sp[PTILE_N<PAIR>];  // the pressure slab
  float2 sud[3][G2P_TILE];  // (u_new, u_new - u_old) per face node
  __align__(16) float pbuf[2][6][G2P_CHUNK_PAD];
  __align__(8) unsigned long long bar[3];  // particle buffers 0, 1; the pressure slab
  unsigned long long empty[2];             // ... the buffers' readers, one arrival per warp
  int abort;
};

// A CTA's streaming state, kept across bricks (and across scenes in a batched launch), a bit
// per barrier: their phases, and (thread 0) which have a copy that nobody has waited for, the
// readers' phases, and which buffers have had readers; the buffer of the next chunk.
struct G2pCta {
  unsigned int phase = 0u, inflight = 0u, empty = 0u, used = 0u, kbuf = 0u;
};

template <bool PAIR>
__device__ __forceinline__ void g2p_init(G2pShared<PAIR>& sh) {
  if (threadIdx.x == 0) {
    mbar_init(&sh.bar[0], 1);
    mbar_init(&sh.bar[1], 1);
    mbar_init(&sh.bar[2], 1);
    mbar_init(&sh.empty[0], G2P_THREADS / 32);
    mbar_init(&sh.empty[1], G2P_THREADS / 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sh.abort = 0;
  }
  __syncthreads();
}

// Thread 0: particles [q0, q1) into the next buffer, once its readers have left it; false if
// they have not within the limit.
template <bool PAIR>
__device__ __forceinline__ bool g2p_issue(const PartView& P, unsigned int q0, unsigned int q1,
                                          unsigned long long wait_ns, G2pShared<PAIR>& sh,
                                          G2pCta& cs) {
  const unsigned int k = cs.kbuf, bit = 1u << k;
  if (cs.used & bit) {
    if (!mbar_wait(&sh.empty[k], (cs.empty >> k) & 1u, wait_ns)) return false;
    cs.empty ^= bit;
  }
  cs.used |= bit;
  issue_chunk(P, q0, q1, sh.pbuf[k], &sh.bar[k]);
  cs.inflight |= bit;
  return true;
}

// One brick of one scene (pmap: the tensor map of the scene's pressure, or
// nullptr for plain loads).  CTA-uniform; returns false once a wait has given up
// (DEV_TIMEOUT set in the scene's status), after which the CTA takes no more bricks.
template <bool PAIR, bool ORDERED>
__device__ __forceinline__ bool g2p_brick(const Grid& g, const StepConsts& K, const PartView& P,
                                          const BinView& B, const float* __restrict__ uo0,
                                          const float* __restrict__ uo1,
                                          const float* __restrict__ uo2,
                                          const float* __restrict__ p32,
                                          const float2* __restrict__ pff, DevStats* st,
                                          const CUtensorMap* pmap, unsigned int brick,
                                          unsigned int part, unsigned int split,
                                          G2pShared<PAIR>& sh, G2pCta& cs, float& speed2) {
  using PT = typename PTile<PAIR>::T;
  const int lane = threadIdx.x & 31;
  const int b0 = (int)(brick % (unsigned)g.bx) * BRICK;
  const int b1 = (int)((brick / (unsigned)g.bx) % (unsigned)g.by) * BRICK;
  const int b2 = (int)(brick / ((unsigned)g.bx * (unsigned)g.by)) * BRICK;
  unsigned int bstart = B.brick_start[brick], bend = B.brick_start[brick + 1];
  if (split > 1) {  // the part's whole chunks
    const unsigned int chunks = (bend - bstart + G2P_THREADS - 1) / G2P_THREADS;
    const unsigned int per = (chunks + split - 1) / split * G2P_THREADS;
    const unsigned int first = min(bend, bstart + part * per);
    bend = min(bend, first + per);
    bstart = first;
    if (bstart == bend) return true;
  }
  // the brick's first chunk streams in while the tiles are staged
  if (threadIdx.x == 0 && bstart < bend &&
      !g2p_issue(P, bstart, min(bend, bstart + G2P_THREADS), K.wait_ns, sh, cs)) {
    atomicOr(&st->status, DEV_TIMEOUT);
    sh.abort = 1;
  }
  // pressure of cells [b0 - XOFF, b0 - XOFF + SPX) x [b1 - 1, b1 + 9) x [b2 - 1, b2 + 9)
  // (0 outside the grid: never used)
  constexpr int SPX = PTile<PAIR>::SPX, XOFF = PTile<PAIR>::XOFF;
  if (pmap) {
    if (threadIdx.x == 0) {
      // the tile's readers of the previous brick passed the __syncthreads that
      // ended it; order their generic-proxy reads before the async-proxy write
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(&sh.bar[2], (unsigned)sizeof(sh.sp));
      tma_load_3d(sh.sp, pmap, b0 - XOFF, b1 - 1, b2 - 1, &sh.bar[2]);
      cs.inflight |= 4u;
    }
    if (mbar_wait(&sh.bar[2], cs.phase >> 2, K.wait_ns)) {
      cs.phase ^= 4u;
      cs.inflight &= ~4u;
    } else {
      atomicOr(&st->status, DEV_TIMEOUT);
      sh.abort = 1;
    }
  } else {
    for (int t = threadIdx.x; t < PTILE_N<PAIR>; t += G2P_THREADS) {
      const int i = b0 - XOFF + t % SPX, j = b1 - 1 + (t / SPX) % 10, k = b2 - 1 + t / (10 * SPX);
      PT v{};
      if (i >= 0 && j >= 0 && k >= 0 && i < g.nx && j < g.ny && k < g.nz) {
        const int c = i + g.nx * (j + g.ny * k);
        if constexpr (PAIR) v = pff[c];
        else v = p32[c];
      }
      sh.sp[t] = v;
    }
  }
  __syncthreads();
  if (sh.abort) return false;
  stage_faces<0, PAIR>(g, K, b0, b1, b2, uo0, sh.sp, sh.sud[0]);
  stage_faces<1, PAIR>(g, K, b0, b1, b2, uo1, sh.sp, sh.sud[1]);
  stage_faces<2, PAIR>(g, K, b0, b1, b2, uo2, sh.sp, sh.sud[2]);
  __syncthreads();
  // A particle's rank in its new cell is what the histogram's atomic returns, with its place
  // among the warp's lanes of that cell; it is written a chunk later, so that the atomic's
  // round trip passes under the next chunk's arithmetic.
  unsigned int first = 0u, rank_ofs = 0u, rank_q = ~0u;
  int rank_lead = 0;
  const auto put_ranks = [&]() {
    const unsigned int f = __shfl_sync(0xffffffffu, first, rank_lead);
    if (rank_q != ~0u) B.rank[rank_q] = f + rank_ofs;
    rank_q = ~0u;
  };
  // chunk loop: warp-uniform trip count, so every lane takes part in the key match; the warps
  // run apart by up to the buffers' depth, or (ORDERED) meet after every chunk, so that a
  // chunk's atomics come before the next one's
  for (unsigned int c0 = bstart; c0 < bend; c0 += G2P_THREADS) {
    const unsigned int cur = cs.kbuf;
    cs.kbuf ^= 1u;
    const unsigned int n0 = c0 + G2P_THREADS;
    bool ok = true;
    if (threadIdx.x == 0 && n0 < bend)
      ok = g2p_issue(P, n0, min(bend, n0 + G2P_THREADS), K.wait_ns, sh, cs);
    // a warp with a wait that gave up reads nothing of the chunk; one whose waits
    // succeeded saw the whole chunk land
    if (ok && mbar_wait(&sh.bar[cur], (cs.phase >> cur) & 1u, K.wait_ns)) {
      cs.phase ^= 1u << cur;
      cs.inflight &= ~(1u << cur);
    } else {
      ok = false;
      atomicOr(&st->status, DEV_TIMEOUT);
      sh.abort = 1;
    }
    if (!__all_sync(0xffffffffu, ok)) {
      if (ORDERED) (void)__syncthreads_or(1);  // the others meet there, and leave too
      break;
    }
    const float(*pb)[G2P_CHUNK_PAD] = sh.pbuf[cur];
    const unsigned int q = c0 + threadIdx.x;
    const bool valid = q < bend;
    const unsigned int o = min(q, bend - 1u) - (c0 & ~3u);
    float x = pb[0][o], y = pb[1][o], z = pb[2][o];
    const float vp[3] = {pb[3][o], pb[4][o], pb[5][o]};
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.empty[cur]);
    unsigned int key = 0xffffffffu;
    if (valid) {
      // the particle lies in this brick (its key was taken from the same coordinates); the
      // clamps only keep the shared-memory indices in range
      const auto axis = [&](float p, int b, int n) {
        return axis_g(p, g.inv_dx, b, (float)max(b - 1, 0), fminf((float)(n - 1), (float)b + 7.5f));
      };
      const AxisG ax = axis(x, b0, g.nx), ay = axis(y, b1, g.ny), az = axis(z, b2, g.nz);
      const float2 ud[3] = {interp_tile<0>(ax, ay, az, sh.sud[0]),
                            interp_tile<1>(ax, ay, az, sh.sud[1]),
                            interp_tile<2>(ax, ay, az, sh.sud[2])};
      const float r = K.flip_ratio, r1 = 1.0f - K.flip_ratio;
      float vn[3], adv[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        vn[d] = __fadd_rn(__fmul_rn(r, __fadd_rn(vp[d], ud[d].y)), __fmul_rn(r1, ud[d].x));
        adv[d] = K.advect_grid ? ud[d].x : vn[d];
      }
      x = fminf(fmaxf(__fmaf_rn(K.dt, adv[0], x), g.skin), g.hi[0]);
      y = fminf(fmaxf(__fmaf_rn(K.dt, adv[1], y), g.skin), g.hi[1]);
      z = fminf(fmaxf(__fmaf_rn(K.dt, adv[2], z), g.skin), g.hi[2]);
      P.x[q] = x;
      P.y[q] = y;
      P.z[q] = z;
      P.u[q] = vn[0];
      P.v[q] = vn[1];
      P.w[q] = vn[2];
      speed2 = fmaxf(speed2, vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
      key = brick_key(g, cell_in(x, g.inv_dx, g.nx), cell_in(y, g.inv_dx, g.ny),
                      cell_in(z, g.inv_dx, g.nz));
    }
    if (valid) B.key[q] = key;
    put_ranks();
    // one histogram atomic per distinct key of the warp
    const unsigned int same = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(same) - 1;
    if (valid && lane == leader) first = atomicAdd(B.cell_count + key, (unsigned)__popc(same));
    rank_lead = leader;
    rank_ofs = (unsigned)__popc(same & ((1u << lane) - 1u));
    rank_q = valid ? q : ~0u;
    if (ORDERED && __syncthreads_or(0)) break;
  }
  put_ranks();
  __syncthreads();
  return !sh.abort;
}

// After an abort, thread 0 drains the copies it issued and nobody waited for
// (the chunk whose wait gave up, the one issued after it), boundedly; the CTA's
// shared memory stays allocated until thread 0 leaves.
template <bool PAIR>
__device__ __forceinline__ void g2p_drain(G2pShared<PAIR>& sh, const G2pCta& cs) {
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if ((cs.inflight >> k) & 1u)
        (void)mbar_wait(&sh.bar[k], (cs.phase >> k) & 1u, G2P_DRAIN_NS);
}

// The largest particle speed a CTA saw in a scene, into the scene's statistics.
// CTA-uniform (every warp takes part).
__device__ __forceinline__ void g2p_flush_speed(float& speed2, DevStats* st) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) speed2 = fmaxf(speed2, __shfl_xor_sync(0xffffffffu, speed2, o));
  if ((threadIdx.x & 31) == 0 && speed2 > 0.0f)
    atomicMax(&st->max_speed_bits, __float_as_uint(sqrtf(speed2)));
  speed2 = 0.0f;
}

// Parts per brick: a brick's chunks are a serial chain, so few bricks are shared out over the
// launch's CTAs, each staging the tiles for itself.  The stage at 16 bricks (32^3 dam break)
// 37 -> 16 us, at 150 (64^3) 42 -> 25.  Not with reseeding (ORDERED), where the ranks decide
// which of a crowded cell's particles are dropped: a brick's particles then take theirs in the
// order of its chunks, on one CTA that meets after every chunk.
__device__ __forceinline__ unsigned int g2p_split(unsigned int nact, unsigned int ctas) {
  unsigned int split = 1;
  while (split < G2P_MAX_SPLIT && nact * 2u * split <= ctas) split *= 2;
  return split;
}

// Bound by latency (the tiles' loads, the histogram's atomics) and by shared-memory accesses:
// at 256^3 (42.3 M particles, 2.4 GB) the stage takes 0.703 ms of the 0.34 that the bytes do.
// It took 0.745 with conversions to integers in the weights and cells, ranks written in the
// same chunk, a CTA barrier per chunk, and the barriers' state in a stack array.  One value
// per node, u_new - r u_old, would give the blend as r v + interp(u_new - r u_old) with half
// the shared-memory traffic (0.648), but rounds it otherwise than the interpolants of u_new
// and u_new - u_old: a position's last bit is any change of the velocity of a face that only
// vanishing weights reach.
template <bool PAIR, bool ORDERED>
__global__ void __launch_bounds__(G2P_THREADS, 5) k_g2p(const Grid g, const StepConsts K0,
                                                     const PartView P, const BinView B,
                                                     const float* __restrict__ uo0,
                                                     const float* __restrict__ uo1,
                                                     const float* __restrict__ uo2,
                                                     const float* __restrict__ p32,
                                                     const float2* __restrict__ pff,
                                                     DevStats* st,
                                                     const __grid_constant__ CUtensorMap pmap,
                                                     int use_tma) {
  __shared__ G2pShared<PAIR> sh;
  const StepConsts K = step_consts(K0);
  const unsigned int nact = st->n_active;
  g2p_init(sh);
  G2pCta cs;
  float speed2 = 0.0f;
  const CUtensorMap* map = use_tma ? &pmap : nullptr;
  const unsigned int split = ORDERED ? 1u : g2p_split(nact, gridDim.x);
  for (unsigned int bi = blockIdx.x; bi < nact * split; bi += gridDim.x)
    if (!g2p_brick<PAIR, ORDERED>(g, K, P, B, uo0, uo1, uo2, p32, pff, st, map, B.active[bi / split],
                         bi % split, split, sh, cs, speed2))
      break;
  g2p_drain(sh, cs);
  g2p_flush_speed(speed2, st);
}

// All scenes' active bricks as one list (L.first from k_active_prefix): the CTAs
// share every scene's bricks evenly.  A CTA that gives up on a wait marks every
// scene whose bricks it leaves undone.  4 CTAs per SM (5 spill: 16 scenes 3.65 against
// 3.62 ms per step).
template <bool PAIR>
__global__ void __launch_bounds__(G2P_THREADS, 4) k_g2p_batch(const BatchLaunch L) {
  __shared__ G2pShared<PAIR> sh;
  g2p_init(sh);
  G2pCta cs;
  float speed2 = 0.0f;
  int cur = -1;
  const unsigned int g0 = L.first[0], g1 = L.first[L.n];
  const unsigned int split = g2p_split(g1 - g0, gridDim.x), n = (g1 - g0) * split;
  unsigned int q = blockIdx.x;
  for (; q < n; q += gridDim.x) {
    const unsigned int gb = g0 + q / split;
    const int s = batch_scene(L, gb);
    const SceneDev& S = L.scenes[s];
    if (s != cur) {
      if (cur >= 0) g2p_flush_speed(speed2, L.scenes[cur].st);
      cur = s;
    }
    if (!g2p_brick<PAIR, false>(S.g, step_consts(S.K), S.dst, S.B, S.uo[0], S.uo[1], S.uo[2], S.x32,
                         S.pff, S.st, nullptr, S.B.active[gb - L.first[s]], q % split, split, sh, cs,
                         speed2))
      break;
  }
  g2p_drain(sh, cs);
  if (cur >= 0) g2p_flush_speed(speed2, L.scenes[cur].st);
  if (q < n && threadIdx.x == 0)  // aborted: the scenes of the bricks left undone
    for (q += gridDim.x; q < n; q += gridDim.x)
      atomicOr(&L.scenes[batch_scene(L, g0 + q / split)].st->status, DEV_TIMEOUT);
}

int g2p_blocks(int sm_count) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_g2p<true, false>, G2P_THREADS, 0) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  return sm_count * per_sm;
}

void launch_g2p_batch(const BatchLaunch& L, unsigned int ctas, bool pair, cudaStream_t s) {
  if (!ctas) return;
  if (pair) k_g2p_batch<true><<<ctas, G2P_THREADS, 0, s>>>(L);
  else k_g2p_batch<false><<<ctas, G2P_THREADS, 0, s>>>(L);
}

void launch_g2p(const Grid& g, const StepConsts& k, const PartView& p, const BinView& b,
                const float* const uo[3], const float* p32, const float2* pff, DevStats* st,
                long long np, int nblocks, const CUtensorMap* pmap, bool keep_order,
                cudaStream_t s) {
  if (np <= 0) return;
  CUtensorMap none;
  std::memset(&none, 0, sizeof(none));
  const CUtensorMap& m = pmap ? *pmap : none;
  const int tma = pmap ? 1 : 0;
  const auto kernel = pff ? (keep_order ? k_g2p<true, true> : k_g2p<true, false>)
                          : (keep_order ? k_g2p<false, true> : k_g2p<false, false>);
  kernel<<<nblocks, G2P_THREADS, 0, s>>>(g, k, p, b, uo[0], uo[1], uo[2], p32, pff, st, m, tma);
}

bool encode_pressure_map(const Grid& g, void* base, bool pair, CUtensorMap* out) {
  // row and plane pitches must be multiples of 16 bytes; the box (SPX x 10 x 10)
  // must fit the grid
  const size_t elem = pair ? 8 : 4;
  const int spx = pair ? PTile<true>::SPX : PTile<false>::SPX;
  if (!base || (reinterpret_cast<uintptr_t>(base) & 15u) || ((size_t)g.nx * elem) % 16 != 0 ||
      g.nx < spx || g.ny < 10 || g.nz < 10)
    return false;
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    cudaDriverEntryPointQueryResult q;
    void* f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      encode = (PFN_cuTensorMapEncodeTiled_v12000)f;
    cudaGetLastError();
    looked_up = true;
  }
  if (!encode) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
  const cuuint64_t strides[2] = {(cuuint64_t)g.nx * elem, (cuuint64_t)g.nx * g.ny * elem};
  const cuuint32_t box[3] = {(cuuint32_t)spx, 10u, 10u};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return encode(out, pair ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace flipk
