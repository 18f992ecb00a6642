// k_mg.cu — conjugate gradient on A p = b (Sec. 3.1.7) preconditioned by one
// multigrid V-cycle per iteration, whose smoother is the red-black Gauss-Seidel
// the paper runs on the GPU (Sec. 3.2.3).  One persistent cooperative kernel
// per solve, like the Jacobi version in k_pcg.cu.
//
// Hierarchy: level 0 is the cell grid; level l+1 has ceil(n_l/2) cells per axis
// and a coarse cell is fluid when any of its children is; coarsening stops when
// the largest extent is <= 4.  Level l carries the 7-point operator with scale
// dt/(rho (2^l dx)^2).  V-cycle from a zero guess at every level: nu
// (red, black) half-sweep pairs, restriction of the residual b_{l+1} =
// (1/16) sum over fluid children (Galerkin scaling for piecewise-constant
// prolongation), the coarse cycle, correction x += omega x_{l+1}(parent), nu
// (black, red) pairs; the coarsest level does MG_COARSE_SWEEPS pairs each way.
// The cycle is a symmetric positive-definite operator, as CG requires.
//
// Layout and work split.  The grid-wide levels (l < lgrid) are stored
// colour-split (see MgLevel): a half-sweep reads and writes contiguous runs of
// one colour and its six neighbour runs of the other colour, so it moves half
// the bytes of a natural-layout sweep, every access coalesced.  Work is a list
// of active segments per level (64 cells of a row that meet a block holding
// fluid), found at the start of every solve, each CTA a contiguous slice of it.
// Per cell one 16-bit code carries the fluid neighbours and the neighbour
// count, so value loads never wait on flags.  A level takes one of three forms
// by its size per CTA: with many segments, a warp takes four of them, a lane
// four slots (sweep_split_q); with fewer, a lane takes one slot and a warp loads
// several segments before it computes; with few blocks holding fluid, a CTA
// smooths whole 8x8x8 blocks with a halo in shared memory, everything before the
// coarse cycle (restriction included) in one pass and everything after it in
// another (block_pass).  The small coarsest levels (at most MG_CTA_CELLS cells
// together) run inside CTA 0 from shared memory, in registers (cta_cycle_tiled)
// or over lists; the others use grid barriers between passes.
//
// In the passes over segments the correction is never written: the first
// post-smoothing half-sweep (black) reads its red neighbours plus omega times
// their parents' values, and the red half-sweep that follows overwrites the red
// cells anyway.  The first red
// half-sweep from zero only needs the residual, so it is fused into the pass
// that produces it: at level 0 the CG phase that updates r, at a grid-wide
// coarse level the restriction.  The last black and the last red half-sweeps of
// level 0 also accumulate r.z.
#include "pcg_common.cuh"

namespace flipk {

// Solve trace, in builds with -DFLIP_SOLVE_TRACE only (compiled out otherwise):
// thread 0 of the team's first CTA stamps the global timer after each phase of
// a solve into flip_trace_ns[slot] (slots below), each stamp taken after the grid
// barrier that ends its phase; flip_solve_trace copies them to the host.
#ifdef FLIP_SOLVE_TRACE
__device__ unsigned long long flip_trace_ns[64];
#define SOLVE_TRACE(slot) trace_stamp(slot)
#else
#define SOLVE_TRACE(slot) ((void)0)
#endif

enum TraceSlot {
  TR_ENTRY = 0,       // kernel entry
  TR_TABLES = 1,      // shared tables loaded
  TR_BFLAG = 2,       // block flags cleared
  TR_FLAGS = 2,       // + 1: fluid flags of all levels built
  TR_SEG_COUNT = 14,  // active segments counted (large grids)
  TR_SEG_WRITE = 15,  // active-segment lists written
  TR_CODES = 16,      // neighbour codes built
  TR_SEG_CACHE = 17,  // segment slices cached
  TR_CTA_LISTS = 18,  // CTA-local lists built (CTA 0)
  TR_START = 19,      // start pass (r, z, b) done
  TR_ITER = 20,       // + 3 i, + 1, + 2: V-cycle, phase A, phase B of iteration i (i < 3)
  TR_LOOP_END = 29,   // CG loop left
  TR_END = 30,        // solution written
  TR_EXIT = 31,       // kernel exit
  TR_V_PRE1 = 32,     // the V-cycle's pieces (the last V-cycle of the solve):
  TR_V_PRE = 33,      //   level-0 pre-smoothing (first black, the rest),
  TR_V_RESTRICT = 34, //   restriction 0 -> 1,
  TR_V_DOWN = 34,     //   + l: level l's pre-smoothing and restriction (l = 1 .. 11),
  TR_V_CTA = 46,      //   the CTA-local levels,
  TR_V_UP = 46,       //   + l: level l's correction and post-smoothing (l = 1 .. 11),
  TR_V_CORRECT = 58,  //   level-0 correction and first black half-sweep,
  TR_V_POST = 59,     //   the rest of level 0's post-smoothing but the last red
  TR_REFINE = 60      // + 0, 1, 2: the first refinement's start, x += d, residual
};

namespace {

#ifdef FLIP_SOLVE_TRACE
__device__ __forceinline__ void trace_stamp(int slot) {
  if (team_rank() == 0 && threadIdx.x == 0) flip_trace_ns[slot] = global_timer_ns();
}
#endif

constexpr unsigned int CODE_SELF = 64u;
constexpr unsigned int CODE_FULL = 0x67fu;  // fluid, six fluid neighbours, count 6
// Both cells of a slot pair's codes (16 bits each) are CODE_FULL.
__device__ __forceinline__ bool pair_full(unsigned int code2) {
  return code2 == (CODE_FULL | (CODE_FULL << 16));
}
constexpr int SEG_SLOTS = 32;  // slots of one colour per segment (a warp)

// Gauss-Seidel coefficients per level, copied to shared memory at kernel start:
// s_inv_scnt[l][n] = 1 / (s_l n), s_inv_cnt[n] = 1 / n.
// s_gs[l][n] holds both (0, 0 for n = 0), for the passes that need the pair.
__shared__ float s_inv_scnt[MG_MAX_LEVELS][8];
__shared__ float s_inv_cnt[8];
__shared__ float2 s_gs[MG_MAX_LEVELS][8];

__device__ __forceinline__ void load_tables(const MgArgs& M) {
  if (threadIdx.x < MG_MAX_LEVELS * 8) {
    const int l = threadIdx.x >> 3, n = threadIdx.x & 7;
    s_inv_scnt[l][n] = l < M.nlev ? M.lv[l].inv_scnt[n] : 0.0f;
    s_gs[l][n] = make_float2(l < M.nlev ? M.lv[l].inv_scnt[n] : 0.0f, M.inv_cnt[n]);
  }
  if (threadIdx.x < 8) s_inv_cnt[threadIdx.x] = M.inv_cnt[threadIdx.x];
  __syncthreads();
}

// Each CTA's slice of a level's active segments is the same in every pass of a
// solve, so after the lists are built the CTA copies its slices into shared
// memory (as many levels as SEG_CACHE holds, level 0 first): the first load of
// every item of a pass, the segment, is then a shared-memory read.  s_segc[l] is
// the copy of level l's slice (nullptr: read the list in global memory) and
// s_segb[l] the index of its first segment.
constexpr int SEG_CACHE = 4096;
__shared__ const unsigned int* s_segc[MG_MAX_LEVELS];
__shared__ int s_segb[MG_MAX_LEVELS];
// A level's number of active segments and this CTA's slice of them.
__shared__ int s_nseg[MG_MAX_LEVELS];
__shared__ int2 s_slice[MG_MAX_LEVELS];

// One thread: the slice of a level with n active segments.
__device__ __forceinline__ void set_slice(int l, int n) {
  const int per = (n + (int)team_size() - 1) / (int)team_size();
  const int q0 = min(n, (int)team_rank() * per);
  s_nseg[l] = n;
  s_slice[l] = make_int2(q0, min(n, q0 + per));
}

// Levels whose smoothing runs blocked (block_pass): their number of blocks holding
// fluid, 0 for the levels swept pass by pass.  s_z0 and s_q0 are the arrays that hold
// level 0's z after a V-cycle and A p: z in lv[0].x and A p in q0, or the other way
// round when level 0 is blocked (a blocked post-smoothing writes to a second array).
__shared__ int s_nblk[MG_MAX_LEVELS];
__shared__ float* s_z0;
__shared__ float* s_q0;

// The fields of a colour-split level a pass uses, read once into registers at
// the start of the pass (the level descriptions live in parameter or shared
// memory and would otherwise be re-read through generic pointers per cell).
// Segment t of the level is seg[t - seg_base].
struct SV {
  float* x;
  float* b;
  uint16_t* code;
  const unsigned int* seg;
  int seg_base;
  int nx, ny, hx, half, margin, pl;
  float s;
};

__device__ __forceinline__ SV sview(const MgLevel& L) {
  const unsigned int* c = s_segc[L.lvl];
  return SV{L.x, L.b, L.code16, c ? c : L.seg, c ? s_segb[L.lvl] : 0, L.nx, L.ny, L.hx,
            L.half, L.margin, L.hx * L.ny, L.s};
}

// The same for the level whose x a correction reads (colour-split or natural).
struct PV {
  const float* x;
  int split, nx, ny, nz, hx, half, margin;
};

__device__ __forceinline__ PV pview(const MgLevel& C) {
  return PV{s_nblk[C.lvl] > 0 ? C.x2 : C.x, C.split, C.nx, C.ny, C.nz, C.hx, C.half, C.margin};
}

// Runs items first, first + stride, ... < end in batches of U: pre(e, ok)
// returns a state with the item's first loads, load(state) adds the loads that
// depend on them, apply(state) computes and stores.  All loads of a batch come
// before its first store.  Items past the end are handed to pre() as 'first'
// with ok = false (valid addresses; apply must skip them).
template <int U, class Pre, class Load, class Apply>
__device__ __forceinline__ void run_batched(unsigned int first, unsigned int end,
                                            unsigned int stride, Pre&& pre, Load&& load,
                                            Apply&& apply) {
  using S = decltype(pre(0u, false));
  for (unsigned int e0 = first; e0 < end; e0 += (unsigned)U * stride) {
    S s[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned int e = e0 + (unsigned)u * stride;
      const bool ok = e < end;
      s[u] = pre(ok ? e : e0, ok);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) load(s[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) apply(s[u]);
  }
}

// ---------------------------------------------------------------- indexing

// Index of cell (i, j, k) of a level in its storage (colour-split or natural).
__device__ __forceinline__ int level_index(const PV& C, int i, int j, int k) {
  if (C.split) return ((i + j + k) & 1) * C.half + C.margin + C.hx * (j + C.ny * k) + (i >> 1);
  return i + C.nx * (j + C.ny * k);
}

// A slot of a colour-split level: cell (i, j, k) of row r = j + ny k, its
// storage index and the base index of its neighbours in the other colour.
struct SCell {
  int i, j, k, r;
  int idx, ob;
  int par;  // i & 1
  bool ok;
};

// A segment {segment in row, j, k}: 5, 11 and 11 bits (extents up to 2048 cells).
__device__ __forceinline__ unsigned int seg_pack(int w, int j, int k) {
  return (unsigned)w | (unsigned)j << 5 | (unsigned)k << 16;
}

// {row, segment in row, j, k} of a segment of a level with ny rows per plane.
__device__ __forceinline__ int4 seg_unpack(unsigned int v, int ny) {
  const int j = (int)((v >> 5) & 2047u), k = (int)(v >> 16);
  return make_int4(j + ny * k, (int)(v & 31u), j, k);
}

// Lane 'lane' of colour c in segment v.
template <class LV>
__device__ __forceinline__ SCell scell(const LV& L, unsigned int v, int c, int lane) {
  const int4 sg = seg_unpack(v, L.ny);
  SCell e;
  const int s = sg.y * SEG_SLOTS + lane;
  e.j = sg.z;
  e.k = sg.w;
  e.r = sg.x;
  e.par = (c + e.j + e.k) & 1;
  e.i = 2 * s + e.par;
  e.ok = s < L.hx && e.i < L.nx;
  e.idx = c * L.half + L.margin + L.hx * e.r + min(s, L.hx - 1);
  e.ob = e.idx + (1 - 2 * c) * L.half;
  return e;
}

// Storage indices of the six neighbours (-x, +x, -y, +y, -z, +z), all in the
// other colour's half; addresses of neighbours off the grid are valid but their
// values are never used (the code bit is clear).
template <class LV>
__device__ __forceinline__ void snbr(const LV& L, const SCell& e, int (&nb)[6]) {
  const int pl = L.hx * L.ny;
  nb[0] = e.ob - 1 + e.par;
  nb[1] = e.ob + e.par;
  nb[2] = e.ob - L.hx;
  nb[3] = e.ob + L.hx;
  nb[4] = e.ob - pl;
  nb[5] = e.ob + pl;
}

// This CTA's slice [q0, q1) of a level's active segments.
__device__ __forceinline__ int2 seg_slice(const MgLevel& L) { return s_slice[L.lvl]; }

// Items (segment, colour) of this CTA for ncol colours: item t is segment
// t / ncol, colour t % ncol (ncol = 2) or the pass's colour (ncol = 1).  Each
// warp takes items first, first + PCG_WARPS, ...
struct Items {
  unsigned int first, end;
};

__device__ __forceinline__ Items seg_items(const MgLevel& L, int ncol) {
  const int2 q = seg_slice(L);
  return Items{(unsigned)(q.x * ncol + (int)(threadIdx.x >> 5)), (unsigned)(q.y * ncol)};
}

// Vectorised passes: a warp takes two segments (lanes 0-15 and 16-31), a lane two
// adjacent slots s, s + 1 of one colour (s even), read and written as 8-byte
// pairs.  Items are (segment pair, colour); item t is pair t / ncol.
__device__ __forceinline__ Items pair_items(int2 q, int ncol) {
  const int npairs = (q.y - q.x + 1) >> 1;
  return Items{(unsigned)(threadIdx.x >> 5), (unsigned)(npairs * ncol)};
}

// The two cells of a lane: slots s and s + 1 of colour c in one row.
struct PCell {
  int j, k, r, s, par;
  int iA;         // x of the first cell (the second is iA + 2)
  int idx, ob;    // storage index of slot s (even) and of slot s in the other colour
  bool okA, okB;  // inside the grid (and the lane's segment exists)
};

template <class LV>
__device__ __forceinline__ PCell pcell(const LV& L, int2 q, unsigned int pair, int c, int lane) {
  int sq = q.x + 2 * (int)pair + (lane >> 4);
  const bool seg_ok = sq < q.y;
  if (!seg_ok) sq = q.x;
  const int4 sg = seg_unpack(L.seg[sq - L.seg_base], L.ny);
  PCell e;
  e.j = sg.z;
  e.k = sg.w;
  e.r = sg.x;
  e.s = sg.y * SEG_SLOTS + 2 * (lane & 15);
  e.par = (c + e.j + e.k) & 1;
  e.iA = 2 * e.s + e.par;
  const bool s_ok = seg_ok && e.s < L.hx;
  e.okA = s_ok && e.iA < L.nx;
  e.okB = s_ok && e.iA + 2 < L.nx;
  e.idx = c * L.half + L.margin + L.hx * e.r + min(e.s, L.hx - 2);
  e.ob = e.idx + (1 - 2 * c) * L.half;
  return e;
}

// Passes over four slots per lane: a warp takes four segments (eight lanes each), a lane
// the slots s .. s + 3 of one colour (s a multiple of 4), read and written as 16 bytes.
// Item t is segments 4 (t / ncol) .., colour t % ncol.
__device__ __forceinline__ Items quad_items(int2 q, int ncol) {
  const int n = (q.y - q.x + 3) >> 2;
  return Items{(unsigned)(threadIdx.x >> 5), (unsigned)(n * ncol)};
}

struct QCell {
  int j, k, s, par;  // par: x of slot s is 2 s + par
  int idx, ob;       // storage index of slot s and of slot s in the other colour
  bool ok;           // the lane's segment exists and slot s lies in its row
};

template <class LV>
__device__ __forceinline__ QCell qcell(const LV& L, int2 q, unsigned int quad, int c, int lane) {
  const int sq = q.x + 4 * (int)quad + (lane >> 3);
  QCell e;
  e.ok = sq < q.y;
  const int4 sg = seg_unpack(L.seg[(e.ok ? sq : q.x) - L.seg_base], L.ny);
  e.j = sg.z;
  e.k = sg.w;
  e.s = sg.y * SEG_SLOTS + 4 * (lane & 7);
  e.par = (c + e.j + e.k) & 1;
  e.ok = e.ok && e.s < L.hx;
  e.idx = c * L.half + L.margin + L.hx * sg.x + e.s;
  e.ob = e.idx + (1 - 2 * c) * L.half;
  return e;
}

// Count of neighbours in the grid (0: not fluid) of slot s + h, from the four codes.
__device__ __forceinline__ int quad_cnt(uint2 code4, int h) {
  return (int)((h < 2 ? code4.x : code4.y) >> (h & 1 ? 24 : 8)) & 7;
}

// ---------------------------------------------------------------- natural levels

struct Cell {
  int i, j, k, c;
  bool ok;
};

struct Part {
  int begin, end, stride;
};

// Slots of a level owned by this thread: a contiguous slice per CTA (grid-wide
// levels) or all slots by CTA 0's threads (CTA-local levels).
__device__ __forceinline__ Part level_part(int n, bool cta_local) {
  if (cta_local) return Part{(int)threadIdx.x, n, PCG_THREADS};
  int per = (n + (int)team_size() - 1) / (int)team_size();
  per = (per + 31) & ~31;
  const int b = min(n, (int)team_rank() * per);
  return Part{b + (int)threadIdx.x, min(n, b + per), PCG_THREADS};
}

__device__ __forceinline__ Cell cell_at(const MgLevel& L, int c) {
  return Cell{c % L.nx, (c / L.nx) % L.ny, c / (L.nx * L.ny), c, true};
}

// Neighbour code of cell (i, j, k) from natural fluid flags fl (value 1 = fluid):
// bits 0..5 fluid neighbours inside the grid, bit 6 the cell itself, bits 8..10
// the number of neighbours inside the grid; 0 for a cell that is not fluid.
__device__ __forceinline__ unsigned int make_code(const MgLevel& L, const uint8_t* fl, int i, int j,
                                                  int k) {
  const int c = i + L.nx * (j + L.ny * k);
  const int sy = L.nx, sz = L.nx * L.ny;
  const bool in[6] = {i > 0, i < L.nx - 1, j > 0, j < L.ny - 1, k > 0, k < L.nz - 1};
  const int off[6] = {-1, 1, -sy, sy, -sz, sz};
  if (fl[c] != 1) return 0u;
  unsigned int code = CODE_SELF;
  int cnt = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    cnt += in[q];
    if (in[q] && fl[c + off[q]] == 1) code |= 1u << q;
  }
  return code | ((unsigned)cnt << 8);
}

// ---------------------------------------------------------------- arithmetic

enum SweepMode { FIRST = 0, NORMAL = 1, CORRECT = 2 };

__device__ __forceinline__ int code_cnt(unsigned int code) { return (int)((code >> 8) & 7u); }

// One Gauss-Seidel update of a cell of level l: x_c = b_c / (s_l n_c) + (sum of
// fluid neighbours' x) / n_c, with n_c the count of neighbours inside the grid.
__device__ __forceinline__ float gs_first(int l, int cnt, float bc) {
  return __fmul_rn(bc, s_inv_scnt[l][cnt]);
}

__device__ __forceinline__ float gs_sum(int l, int cnt, unsigned int code, float bc,
                                        const float (&xv)[6]) {
  const float base = __fmul_rn(bc, s_inv_scnt[l][cnt]);
  float sum = 0.0f;
#pragma unroll
  for (int q = 0; q < 6; ++q) sum += ((code >> q) & 1u) ? xv[q] : 0.0f;
  return __fmaf_rn(sum, s_inv_cnt[cnt], base);
}

// Residual b - A x of a fluid cell, A x in difference form
// s (sum_fluid (x_c - x_n) + n_air x_c).
__device__ __forceinline__ float resid(float s, int cnt, unsigned int code, float bc, float xc,
                                       const float (&xv)[6]) {
  float d = 0.0f;
  int nfl = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const bool f = (code >> q) & 1u;
    d += f ? __fsub_rn(xc, xv[q]) : 0.0f;
    nfl += f;
  }
  return __fsub_rn(bc, __fmul_rn(s, __fmaf_rn((float)(cnt - nfl), xc, d)));
}

// resid for a cell whose six neighbours are all fluid (code CODE_FULL): the same
// operations without the masks (cnt - nfl = 0).
__device__ __forceinline__ float resid_full(float s, float bc, float xc, const float (&xv)[6]) {
  float d = 0.0f;
#pragma unroll
  for (int q = 0; q < 6; ++q) d = __fadd_rn(d, __fsub_rn(xc, xv[q]));
  return __fsub_rn(bc, __fmul_rn(s, __fmaf_rn(0.0f, xc, d)));
}

// ---------------------------------------------------------------- sweeps

// Parents on level C of the six neighbours of cell (i, j, k) of a level with
// extents (nx, ny, nz); a neighbour off the grid is replaced by the cell itself
// (its value is unused).
__device__ __forceinline__ void parent_values(const PV& C, int nx, int ny, int nz, int i, int j,
                                              int k, float (&pv)[6]) {
  const int pi[6] = {max(i - 1, 0), min(i + 1, nx - 1), i, i, i, i};
  const int pj[6] = {j, j, max(j - 1, 0), min(j + 1, ny - 1), j, j};
  const int pk[6] = {k, k, k, k, max(k - 1, 0), min(k + 1, nz - 1)};
#pragma unroll
  for (int q = 0; q < 6; ++q) pv[q] = C.x[level_index(C, pi[q] >> 1, pj[q] >> 1, pk[q] >> 1)];
}

// Half-sweep of one colour over colour-split level l (description L).  With RZ, returns
// b x over the updated cells.  A level's x is 0 where there is no fluid cell (zero_near
// before the solve, and these sweeps store 0 there) and the neighbours beyond a row's or a
// plane's end, which the storage wraps to other rows, are not read, so the sum of the six
// neighbours needs no masks: gs_sum's values.  (A grid-wide level never sweeps from zero
// here: its first red half-sweep is made by the pass that produces its right-hand side.)
//
// Bound by issue: the index arithmetic is the larger part of an item (a version that loaded
// next to nothing took three quarters of the time), so a lane takes four slots.  A level-0
// half-sweep at 256^3 with its barrier 11.2 -> 8.2 us, against two slots a lane, masks, and
// a second path without masks that a segment at a wall always defeats (every pair of a
// 256-cell row has one); solves 5.17 -> 4.50 ms at 256^3, 1.46 -> 1.30 at 128^3.
template <bool RZ>
__device__ __noinline__ FF sweep_split_q(const MgLevel& L, int l, int colour) {
  const int lane = threadIdx.x & 31;
  const SV v = sview(L);
  const int2 q = seg_slice(L);
  const Items it = quad_items(q, 1);
  const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  FF acc;
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const QCell e = qcell(v, q, t, colour, lane);
    if (!e.ok) continue;
    const float* xo = v.x + e.ob;
    const uint2 code4 = *reinterpret_cast<const uint2*>(v.code + e.idx);
    const float4 b = *reinterpret_cast<const float4*>(v.b + e.idx);
    const float4 m = *reinterpret_cast<const float4*>(xo);
    const float4 zm = *reinterpret_cast<const float4*>(xo - v.pl);
    const float4 zp = *reinterpret_cast<const float4*>(xo + v.pl);
    const float4 ym = e.j > 0 ? *reinterpret_cast<const float4*>(xo - v.hx) : zero;
    const float4 yp = e.j < v.ny - 1 ? *reinterpret_cast<const float4*>(xo + v.hx) : zero;
    // the slot beyond the four, before (par 0) or after (par 1)
    const float ex = (e.par ? e.s + 4 < v.hx : e.s > 0) ? xo[5 * e.par - 1] : 0.0f;
    const float4 o = e.par ? make_float4(m.y, m.z, m.w, ex) : make_float4(ex, m.x, m.y, m.z);
    float2 s0 = __fadd2_rn(make_float2(m.x, m.y), make_float2(o.x, o.y));
    float2 s1 = __fadd2_rn(make_float2(m.z, m.w), make_float2(o.z, o.w));
    s0 = __fadd2_rn(s0, make_float2(ym.x, ym.y));
    s1 = __fadd2_rn(s1, make_float2(ym.z, ym.w));
    s0 = __fadd2_rn(s0, make_float2(yp.x, yp.y));
    s1 = __fadd2_rn(s1, make_float2(yp.z, yp.w));
    s0 = __fadd2_rn(s0, make_float2(zm.x, zm.y));
    s1 = __fadd2_rn(s1, make_float2(zm.z, zm.w));
    s0 = __fadd2_rn(s0, make_float2(zp.x, zp.y));
    s1 = __fadd2_rn(s1, make_float2(zp.z, zp.w));
    float out[4];
    const float sum[4] = {s0.x, s0.y, s1.x, s1.y}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int cnt = quad_cnt(code4, h);
      const float2 gs = s_gs[l][cnt];
      out[h] = cnt ? __fmaf_rn(sum[h], gs.y, __fmul_rn(bv[h], gs.x)) : 0.0f;
      if (RZ) acc.add_prod(cnt ? bv[h] : 0.0f, out[h]);
    }
    *reinterpret_cast<float4*>(v.x + e.idx) = make_float4(out[0], out[1], out[2], out[3]);
  }
  return acc;
}

// Four consecutive cells x = I .. I + 3 (I a multiple of 4) of a row of colour-split level
// C, base being the row's slot I / 2 of colour 0: two pairs, one of each colour.
__device__ __forceinline__ float4 coarse4(const PV& C, int base, int J, int K) {
  const int even = ((J + K) & 1) * C.half, odd = C.half - even;
  const float2 a = *reinterpret_cast<const float2*>(C.x + even + base);
  const float2 b = *reinterpret_cast<const float2*>(C.x + odd + base);
  return make_float4(a.x, b.x, a.y, b.y);
}

// The half-sweep that makes the coarse correction on the fly (C is level l+1, colour-split):
// black cells from their red neighbours plus omega times those' parents.  The twenty-four
// neighbours of a lane's four cells have thirteen parents: the four own ones and the one
// beyond them in the cells' coarse row, and four each in the coarse row and plane next to
// it that the y and z neighbours outside the own parents lie in.  At 256^3 18.5 -> 15.6 us
// against two slots and seven parents a lane, whose indexes cost more than the loads.
template <bool RZ>
__device__ __noinline__ FF correct_split_q(const MgArgs& M, const MgLevel& L, const MgLevel& Cl,
                                           int l, int colour) {
  const int lane = threadIdx.x & 31;
  const SV v = sview(L);
  const PV C = pview(Cl);
  const float omega = M.omega;
  const int2 q = seg_slice(L);
  const Items it = quad_items(q, 1);
  FF acc;
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const QCell e = qcell(v, q, t, colour, lane);
    if (!e.ok) continue;
    const float* xo = v.x + e.ob;
    const uint2 code4 = *reinterpret_cast<const uint2*>(v.code + e.idx);
    const float4 b4 = *reinterpret_cast<const float4*>(v.b + e.idx);
    const float4 m = *reinterpret_cast<const float4*>(xo);
    const float4 ym = *reinterpret_cast<const float4*>(xo - v.hx);
    const float4 yp = *reinterpret_cast<const float4*>(xo + v.hx);
    const float4 zm = *reinterpret_cast<const float4*>(xo - v.pl);
    const float4 zp = *reinterpret_cast<const float4*>(xo + v.pl);
    const float ex = xo[5 * e.par - 1];
    const int J = e.j >> 1, K = e.k >> 1;
    // (off the grid: clamped, the values are not used)
    const int Jy = min(max(e.j & 1 ? J + 1 : J - 1, 0), C.ny - 1);
    const int Kz = min(max(e.k & 1 ? K + 1 : K - 1, 0), C.nz - 1);
    const int col = C.margin + (e.s >> 1);
    const float4 po = coarse4(C, col + C.hx * (J + C.ny * K), J, K);
    const float4 py = coarse4(C, col + C.hx * (Jy + C.ny * K), Jy, K);
    const float4 pz = coarse4(C, col + C.hx * (J + C.ny * Kz), J, Kz);
    const float pe = C.x[level_index(C, min(max(e.par ? e.s + 4 : e.s - 1, 0), C.nx - 1), J, K)];
    // the cells' own parents are also those of the x neighbour on the side of par
    const float xo4[4] = {m.x, m.y, m.z, m.w}, pv4[4] = {po.x, po.y, po.z, po.w};
    const float xl[6] = {ex, m.x, m.y, m.z, m.w, ex};    // par 0: slot h - 1 is xl[h]
    const float pl[6] = {pe, po.x, po.y, po.z, po.w, pe};  // par 1: slot h + 1 is xl[h + 2]
    const float yl[4] = {ym.x, ym.y, ym.z, ym.w}, yh[4] = {yp.x, yp.y, yp.z, yp.w};
    const float zl[4] = {zm.x, zm.y, zm.z, zm.w}, zh[4] = {zp.x, zp.y, zp.z, zp.w};
    const float py4[4] = {py.x, py.y, py.z, py.w}, pz4[4] = {pz.x, pz.y, pz.z, pz.w};
    const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
    float out[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const unsigned int code = ((h < 2 ? code4.x : code4.y) >> (16 * (h & 1))) & 0xffffu;
      const float own = __fmaf_rn(omega, pv4[h], xo4[h]);
      const float oth = e.par ? __fmaf_rn(omega, pl[h + 2], xl[h + 2])
                              : __fmaf_rn(omega, pl[h], xl[h]);
      const float c[6] = {e.par ? own : oth,
                          e.par ? oth : own,
                          __fmaf_rn(omega, e.j & 1 ? pv4[h] : py4[h], yl[h]),
                          __fmaf_rn(omega, e.j & 1 ? py4[h] : pv4[h], yh[h]),
                          __fmaf_rn(omega, e.k & 1 ? pv4[h] : pz4[h], zl[h]),
                          __fmaf_rn(omega, e.k & 1 ? pz4[h] : pv4[h], zh[h])};
      float sum = 0.0f;
#pragma unroll
      for (int u = 0; u < 6; ++u)
        if ((code >> u) & 1u) sum = __fadd_rn(sum, c[u]);
      const float2 gs = s_gs[l][code_cnt(code)];
      out[h] = code ? __fmaf_rn(sum, gs.y, __fmul_rn(bv[h], gs.x)) : 0.0f;
      if (RZ) acc.add_prod(code ? bv[h] : 0.0f, out[h]);
    }
    *reinterpret_cast<float4*>(v.x + e.idx) = make_float4(out[0], out[1], out[2], out[3]);
  }
  return acc;
}

// Scalar forms: a lane takes one slot (levels with few segments per CTA, where
// more items in flight matter more than wider loads).
template <int MODE>
__device__ __noinline__ FF sweep_split_s(const MgArgs& M, const MgLevel& L, const MgLevel& C,
                                         int l, int colour, bool rz) {
  static_assert(MODE != FIRST, "grid-wide levels start from the fused first half-sweep");
  constexpr int U = (MODE == CORRECT) ? 1 : 2;
  const int lane = threadIdx.x & 31;
  const SV v = sview(L);
  const PV cv = pview(C);
  const int nz = L.nz;
  const float omega = M.omega;
  const Items it = seg_items(L, 1);
  struct S {
    int idx;
    unsigned int code;            // 0: not fluid, or no item
    float b;
    float xv[6];
    float pv[MODE == CORRECT ? 6 : 1];  // the neighbours' parents on the coarser level
  };
  FF acc;
  run_batched<U>(
      it.first, it.end, PCG_WARPS,
      [&](unsigned int t, bool ok) {
        const SCell e = scell(v, v.seg[t - v.seg_base], colour, lane);
        S st;
        st.idx = e.idx;
        st.code = e.ok && ok ? (unsigned int)v.code[e.idx] : 0u;
        st.b = v.b[e.idx];
        int nb[6];
        snbr(v, e, nb);
#pragma unroll
        for (int q = 0; q < 6; ++q) st.xv[q] = v.x[nb[q]];
        if constexpr (MODE == CORRECT)
          parent_values(cv, v.nx, v.ny, nz, min(e.i, v.nx - 1), e.j, e.k, st.pv);
        return st;
      },
      [&](S&) {},
      [&](S& st) {
        if (!st.code) return;
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          float x = st.xv[q];
          if constexpr (MODE == CORRECT) x = __fmaf_rn(omega, st.pv[q], x);
          sum += (st.code >> q) & 1u ? x : 0.0f;
        }
        const float2 gs = s_gs[l][code_cnt(st.code)];
        const float x = __fmaf_rn(sum, gs.y, __fmul_rn(st.b, gs.x));
        v.x[st.idx] = x;
        if (rz) acc.add_prod(st.b, x);
      });
  return acc;
}

// Levels with many segments per CTA take the wide forms (fewer instructions per cell); the
// others the scalar form (more items in flight).  Solves at 256^3 (level 0: 519 segments
// per CTA, level 1: 65) and 128^3 (66) with the line at 256 and at 64: 5.17 -> 5.09 and
// 1.46 -> 1.42 ms.
constexpr int VEC_SEGS_PER_CTA = 64;

__device__ __forceinline__ bool use_wide(const MgLevel& L) {
  return s_nseg[L.lvl] >= VEC_SEGS_PER_CTA * (int)team_size();
}

template <int MODE>
__device__ __forceinline__ FF sweep_split(const MgArgs& M, const MgLevel& L, const MgLevel& C,
                                          int l, int colour, bool rz) {
  if (!use_wide(L) || (MODE == CORRECT && !C.split))
    return sweep_split_s<MODE>(M, L, C, l, colour, rz);
  // the r.z accumulation only where asked (it costs registers)
  if constexpr (MODE == CORRECT)
    return rz ? correct_split_q<true>(M, L, C, l, colour)
              : correct_split_q<false>(M, L, C, l, colour);
  else return rz ? sweep_split_q<true>(L, l, colour) : sweep_split_q<false>(L, l, colour);
}

// ---------------------------------------------------------------- restriction

// Residual of the red child (dy, dz) of coarse cell (I, J, K) on the
// colour-split fine level F.  The child's x offset dx makes its colour red:
// 2I+dx + 2J+dy + 2K+dz even, so its red slot is I.
struct ChildIn {
  bool ok;
  unsigned int code;
  float b, xc;
  float xv[6];
};

__device__ __forceinline__ void child_load(const SV& F, int fnz, int I, int J, int K, int dy,
                                           int dz, ChildIn& s) {
  const int dx = (dy + dz) & 1;
  const int i = 2 * I + dx, j = 2 * J + dy, k = 2 * K + dz;
  s.ok = i < F.nx && j < F.ny && k < fnz;
  const int jj = min(j, F.ny - 1), kk = min(k, fnz - 1);
  const int idx = F.margin + F.hx * (jj + F.ny * kk) + min(I, F.hx - 1);
  const int ob = idx + F.half;
  s.code = F.code[idx];
  s.b = F.b[idx];
  s.xc = F.x[idx];
  const int nb[6] = {ob - 1 + dx, ob + dx, ob - F.hx, ob + F.hx, ob - F.pl, ob + F.pl};
#pragma unroll
  for (int q = 0; q < 6; ++q) s.xv[q] = F.x[nb[q]];
}

// b_C(I,J,K) = (1/16) sum over fluid children of the fine residual.  The
// restriction follows the pre-smoothing, whose last half-sweep is black: a black
// cell's update solves its own equation against the red neighbours it read, so
// its residual is exactly zero and only the red children contribute.  The four
// red children are loaded two at a time and summed in the order (dy, dz) =
// (0,0), (1,0), (0,1), (1,1).
__device__ __forceinline__ float restrict_sum(const SV& F, int fnz, int I, int J, int K) {
  float sum = 0.0f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    ChildIn ch[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) child_load(F, fnz, I, J, K, q, h, ch[q]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const ChildIn& c = ch[q];
      if (!c.ok || !(c.code & CODE_SELF)) continue;
      sum = __fadd_rn(sum, resid(F.s, code_cnt(c.code), c.code, c.b, c.xc, c.xv));
    }
  }
  return __fmul_rn(sum, 0.0625f);
}

// Colour-split F -> colour-split C, over C's active segments; a warp takes half a
// segment, 32 cells in x order (so the fine red slots it reads are contiguous).
// The pass also makes C's first red half-sweep from zero, x = b / (s_C n) on C's
// red fluid cells, which needs only the b it has just computed: C's
// pre-smoothing then starts with the black half-sweep, and the cycle meets one
// grid barrier fewer per level (the values are those the separate half-sweep
// computes; the slots of C's non-fluid cells, never read unmasked, are left).
// Bound by latency (two rounds of 18 loads a lane, about four items a warp at 256^3).  Half
// segments rather than whole ones even out the last round; two children a lane, the upper
// plane's on the upper half-warp, took 23.4 us instead of 16.6 (half the slots per request).
__device__ __noinline__ void restrict_split(const MgLevel& Fl, const MgLevel& Cl) {
  const int lane = threadIdx.x & 31;
  const SV F = sview(Fl), C = sview(Cl);
  const int fnz = Fl.nz;
  const int lc = Cl.lvl;
  const Items it = seg_items(Cl, 2);
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const int4 sg = seg_unpack(C.seg[(int)(t >> 1) - C.seg_base], C.ny);
    const int J = sg.z, K = sg.w, h = (int)(t & 1u);
    {
      // every lane takes part (a lane past the row's end on its last cell, whose
      // result it drops), so that a warp can vote
      const int I = sg.y * (2 * SEG_SLOTS) + h * 32 + lane;
      const bool in = I < C.nx;
      const int Ic = in ? I : C.nx - 1;
      const int red = ((Ic + J + K) & 1) == 0;
      const int ci = (1 - red) * C.half + C.margin + C.hx * sg.x + (Ic >> 1);
      const unsigned int code = C.code[ci];
      // restrict_sum's sum over the red children; a pair of children that is all
      // interior fluid cells in every lane is added without the masks
      float sum = 0.0f;
#pragma unroll
      for (int hz = 0; hz < 2; ++hz) {
        ChildIn ch[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) child_load(F, fnz, Ic, J, K, q, hz, ch[q]);
        const bool full = ch[0].ok && ch[1].ok && ch[0].code == CODE_FULL && ch[1].code == CODE_FULL;
        if (__all_sync(0xffffffffu, full)) {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            sum = __fadd_rn(sum, resid_full(F.s, ch[q].b, ch[q].xc, ch[q].xv));
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const ChildIn& c = ch[q];
            if (!c.ok || !(c.code & CODE_SELF)) continue;
            sum = __fadd_rn(sum, resid(F.s, code_cnt(c.code), c.code, c.b, c.xc, c.xv));
          }
        }
      }
      if (!in || !(code & CODE_SELF)) continue;
      const float bc = __fmul_rn(sum, 0.0625f);
      C.b[ci] = bc;
      if (red) C.x[ci] = gs_first(lc, code_cnt(code), bc);
    }
  }
}

// Colour-split F -> natural-layout C (the first CTA-local level, in global
// memory), over all of C's cells.
__device__ __noinline__ void restrict_split_nat(const MgLevel& Fl, const MgLevel& Cl) {
  const SV F = sview(Fl);
  const int fnz = Fl.nz;
  const int nx = Cl.nx, ny = Cl.ny;
  float* cb = Cl.b;
  const uint8_t* code = Cl.code;
  const Part p = level_part(Cl.ncells, false);
  for (int c = p.begin; c < p.end; c += p.stride) {
    if (!(code[c] & CODE_SELF)) continue;
    const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
    cb[c] = restrict_sum(F, fnz, i, j, k);
  }
}

// ---------------------------------------------------------------- barriers

// Out of line: one copy of it stays in the instruction cache for an iteration's ~30
// barriers.
__device__ __noinline__ bool gsync(const PcgArgs& A) {
  return grid_barrier(A.bar, A.status, team_size(), A.timeout_ns);
}

__device__ __forceinline__ void garrive(const PcgArgs& A) { grid_arrive(A.bar); }

__device__ __forceinline__ bool gwait(const PcgArgs& A) {
  return grid_wait(A.bar, A.status, team_size(), A.timeout_ns);
}

// ---------------------------------------------------------------- blocked smoothing
//
// On a level with few cells per CTA a half-sweep is all latency: a grid barrier
// (~1.5 us) and a round trip to L2 for a few hundred cells.  There the whole
// pre-smoothing with the restriction, and the whole correction with the
// post-smoothing, run as one pass each: a CTA takes an 8^3 block with a halo of
// TILE_H = 4 cells into registers and shared memory and makes all the half-sweeps there,
// between CTA barriers, on the cells that the block's own still depend on (those within
// L1 distance 3, 2, 1, 0 of the block).  Every cell gets gs_sum's operations on the same
// values in its order, so the results are those of the pass-by-pass form.
//
// The tile (16^3 cells) is colour-split like the level: cell (tx, ty, tz) of colour c
// is slot tx >> 1 of row (ty, tz).  Thread t owns slot s = t & 7 of row y = (t >> 3) & 15
// in the planes 2 g and 2 g + 1, g = t >> 7, of both colours, in registers, as one float2
// per colour.  Of a cell's six neighbours one along x and one along z are then its own
// thread's; the others come from the shared copy, along y both planes at a time.  The
// other x neighbour is slot s - 1 in one plane and s + 1 in the other.  Cells that are not
// fluid hold 0, with 0 coefficients, so nothing is masked; cells farther out than a
// half-sweep's results are needed get values nobody uses.  The neighbour codes of each
// thread's cells are laid out once per solve (MgLevel::tab), so a pass loads them, and the
// cells they mark, without index or bounds logic.
//
// Bound by latency (one block per CTA: 4.5-5 us a pass with its 1.5 us grid barrier, against
// four or five passes of 3.3 us) and, from two blocks on, by issue (2 us per further block).
// What counts is that nothing spills: 1024 threads have 64 registers each, and a spilled
// value costs every warp a trip to L1.  With four planes per thread and two 512-thread
// tiles side by side (68-140 bytes of spills) a pass took 6.2-6.7 us, with one plane twice
// and scalar shared loads 7.1-8.8.  Solve per step, pass by pass -> four planes -> this:
// 64^3 double dam (mixed) 1.20 -> 0.77 -> 0.61 ms, 128^3 dam break (FP32) 1.55 -> 1.12 ->
// 1.00, 101 x 67 x 83 pool 2.06 -> 1.37 -> 1.20, 256^3 pool 6.13 -> 5.43 -> 5.24.
constexpr int TILE_H = 4;
constexpr int TILE_W = 8 + 2 * TILE_H;
constexpr int TILE_PLANE = TILE_W * 8;        // threads (and slots of a colour) per plane
static_assert(MG_BLK_MAX_NU == TILE_H / 2, "the halo's depth");
static_assert(TILE_PLANE * TILE_W / 2 == PCG_THREADS && PCG_THREADS == MG_BLK_THREADS,
              "a thread per slot and two planes");

struct MgTile {
  float2 x[2][PCG_THREADS];  // by colour
};

__device__ __forceinline__ MgTile& mg_tile();

// Distance of a tile coordinate from the block's own [TILE_H, TILE_H + 8).
__device__ __forceinline__ int tile_dist(int t) {
  return max(max(TILE_H - t, t - (TILE_H + 7)), 0);
}

// A thread's place in its tile.
struct TilePos {
  int s, y, g;    // slot, row, pair of planes
  int wdist;      // smallest L1 distance of the warp's rows from the block
  bool own;       // the thread's cells are the block's own
};

__device__ __forceinline__ TilePos tile_pos() {
  TilePos p;
  p.s = (int)threadIdx.x & 7;
  p.y = ((int)threadIdx.x >> 3) & 15;
  p.g = (int)threadIdx.x >> 7;
  const int y0 = p.y & ~3;  // the warp's rows y0 .. y0 + 3
  p.wdist = (y0 == 0 || y0 == 12) + min(tile_dist(2 * p.g), tile_dist(2 * p.g + 1));
  p.own = p.s >= 2 && p.s < 6 && p.y >= 4 && p.y < 12 && p.g >= 2 && p.g < 6;
  return p;
}

// The block's first cell, and a thread's first red slot (plane 2 g) in the level.
struct BlkPos {
  int b0, b1, b2, gi;
};

__device__ __forceinline__ BlkPos blk_pos(const SV& v, const TilePos& p, int e) {
  BlkPos q;
  q.b0 = (e & 255) * 8;
  q.b1 = ((e >> 8) & 255) * 8;
  q.b2 = (e >> 16) * 8;
  const int j = q.b1 - TILE_H + p.y, k = q.b2 - TILE_H + 2 * p.g;
  q.gi = v.margin + v.hx * (j + v.ny * k) + (q.b0 >> 1) - TILE_H / 2 + p.s;
  return q;
}

// A thread's four codes in a word: the counts of the red cells and of the black ones (a digit
// each, plane 0 first; 0 where there is no fluid cell), and the red cells' fluid neighbours (a
// byte each), which the residual needs.  At 8 bytes a thread (the codes themselves) the
// tables took twice the memory; a pass is no slower.
__device__ __forceinline__ unsigned int blk_pack(const unsigned int (&red)[2],
                                                 const unsigned int (&black)[2]) {
  unsigned int w = 0u;
#pragma unroll
  for (int z = 0; z < 2; ++z)
    w |= (red[z] >> 8 & 7u) << (4 * z) | (black[z] >> 8 & 7u) << (8 + 4 * z) |
         (red[z] & 63u) << (16 + 8 * z);
  return w;
}

// Count of plane z (0 or 1 of the thread's two), colour c; fluid neighbours of a red cell.
__device__ __forceinline__ int blk_cnt(unsigned int w, int z, int c) {
  return (int)(w >> (8 * c + 4 * z)) & 7;
}
__device__ __forceinline__ unsigned int blk_nbr(unsigned int w, int z) {
  return w >> (16 + 8 * z);
}

__device__ __forceinline__ float& plane(float2& a, int z) { return z == 0 ? a.x : a.y; }

// The sum of the six neighbours in colour o of a thread's two cells of the other colour:
// (-x) + (+x), -y, +y, -z, +z.  zprev and znext are the planes below and above the two.
__device__ __forceinline__ float2 tile_sum(const float2 own, const float2* t, int d, float zprev,
                                           float znext) {
  float2 s = __fadd2_rn(own, make_float2(t[d].x, t[-d].y));
  s = __fadd2_rn(s, t[-8]);
  s = __fadd2_rn(s, t[8]);
  s = __fadd2_rn(s, make_float2(zprev, own.x));
  return __fadd2_rn(s, make_float2(own.y, znext));
}

// One half-sweep of colour c (compile-time) over the tile: x = inv (sum of the six
// neighbours) + base.
template <int c>
__device__ __forceinline__ void tile_sweep(MgTile& T, const TilePos& p, float2 (&x)[2],
                                           const float2 (&inv)[2], const float2 (&base)[2]) {
  if (p.y == 0 || p.y == TILE_W - 1) return;  // the outermost rows are never updated
  const float2* t = T.x[1 - c] + threadIdx.x;
  const float zprev = p.g > 0 ? t[-TILE_PLANE].y : 0.0f;
  const float znext = p.g < TILE_W / 2 - 1 ? t[TILE_PLANE].x : 0.0f;
  const float2 s = tile_sum(x[1 - c], t, ((c + p.y) & 1) ? 1 : -1, zprev, znext);
  x[c] = __ffma2_rn(s, inv[c], base[c]);
  T.x[c][threadIdx.x] = x[c];
}

struct PassSum {  // a pass's dot product, and whether its barrier held
  FF sum;
  bool ok;
};

// Blocked pre-smoothing and restriction (POST false: level l's b -> its x and level
// l + 1's b), or blocked correction and post-smoothing (POST true: x and level l + 1's
// final x -> xout; RZ: returns b x over the CTA's cells).  With `wait`, the grid barrier
// before it has only been arrived at (garrive): the CTA loads what does not depend on the
// pass before (the tables; for the post-smoothing b and x too), then waits.  ok is false if
// the barrier failed.  The caller meets a grid barrier after it.
template <bool POST, bool RZ>
__device__ __noinline__ PassSum block_pass(const PcgArgs& A, int l, bool wait) {
  const MgArgs& M = A.mg;
  MgTile& T = mg_tile();
  const MgLevel& L = M.lv[l];
  const MgLevel& Cl = M.lv[l + 1];
  const SV v = sview(L);
  const PV C = pview(Cl);
  float* xout = POST ? (l == 0 ? s_z0 : L.x2) : v.x;
  const int n = s_nblk[l];
  const TilePos p = tile_pos();
  FF acc;
  int q = (int)team_rank();
  int e = 0;
  unsigned int w = 0u;
  float2 r[2];  // the right-hand side
  float2 x0;    // POST: the red cells' x
  auto load = [&](const BlkPos& bp) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int z = 0; z < 2; ++z)
        plane(r[c], z) = blk_cnt(w, z, c) ? v.b[c * v.half + bp.gi + z * v.pl] : 0.0f;
    if constexpr (POST) {
#pragma unroll
      for (int z = 0; z < 2; ++z)
        plane(x0, z) = blk_cnt(w, z, 0) ? v.x[bp.gi + z * v.pl] : 0.0f;
    }
  };
  if (q < n) {
    e = L.blk[q];
    w = L.tab[(size_t)q * PCG_THREADS + threadIdx.x];
    if (POST) load(blk_pos(v, p, e));
  }
  if (wait && !gwait(A)) return PassSum{FF(), false};
  for (; q < n; q += (int)team_size()) {
    const BlkPos bp = blk_pos(v, p, e);
    float2 x[2], inv[2], base[2];
    if (!POST) load(bp);
    const int I = (bp.b0 >> 1) - TILE_H / 2 + p.s, J = (bp.b1 - TILE_H + p.y) >> 1,
              K = (bp.b2 - TILE_H + 2 * p.g) >> 1;  // the two red cells' parent
    if constexpr (POST) {
      const float px = (w & 0x77u) ? C.x[level_index(C, I, J, K)] : 0.0f;
#pragma unroll
      for (int z = 0; z < 2; ++z)
        plane(x[0], z) = blk_cnt(w, z, 0) ? __fmaf_rn(M.omega, px, plane(x0, z)) : 0.0f;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const int cnt = blk_cnt(w, z, c);  // 0 where there is no fluid cell
        plane(inv[c], z) = s_inv_cnt[cnt];
        plane(base[c], z) = __fmul_rn(plane(r[c], z), s_inv_scnt[l][cnt]);
      }
    if constexpr (!POST) x[0] = base[0];
    x[1] = make_float2(0.0f, 0.0f);
    __syncthreads();  // the last block's readers are done
    T.x[0][threadIdx.x] = x[0];
    __syncthreads();
    int reach = 2 * M.nu - 1;
#pragma unroll 1
    for (int h = 0; h < M.nu; ++h) {
      if (p.wdist <= reach) tile_sweep<1>(T, p, x, inv, base);
      __syncthreads();
      --reach;
      if (POST || h + 1 < M.nu) {
        if (p.wdist <= reach) tile_sweep<0>(T, p, x, inv, base);
        --reach;
        if (!POST || h + 1 < M.nu) __syncthreads();
      }
    }
    if (p.own) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int z = 0; z < 2; ++z)
          if (blk_cnt(w, z, c)) {
            xout[c * v.half + bp.gi + z * v.pl] = plane(x[c], z);
            if constexpr (RZ) acc.add_prod(plane(r[c], z), plane(x[c], z));
          }
    }
    if constexpr (!POST) {
      if (p.wdist == 0) {
        // residuals of the red cells (0 where there is no fluid cell)
        const float2* t = T.x[1] + threadIdx.x;
        const int d = (p.y & 1) ? 1 : -1;
        const float2 other = make_float2(t[d].x, t[-d].y), ym = t[-8], yp = t[8];
        const float zprev = t[-TILE_PLANE].y, znext = t[TILE_PLANE].x;
        const bool low = (p.y & 1) == 0;  // plane 0: the other slot is the -x neighbour
        const float xv0[6] = {low ? other.x : x[1].x, low ? x[1].x : other.x, ym.x, yp.x, zprev,
                              x[1].y};
        const float xv1[6] = {low ? x[1].y : other.y, low ? other.y : x[1].y, ym.y, yp.y, x[1].x,
                              znext};
        const int c0 = blk_cnt(w, 0, 0), c1 = blk_cnt(w, 1, 0);
        float r0 = resid(v.s, c0, blk_nbr(w, 0), r[0].x, x[0].x, xv0);
        float r1 = resid(v.s, c1, blk_nbr(w, 1), r[0].y, x[0].y, xv1);
        r0 = c0 ? r0 : 0.0f;
        r1 = c1 ? r1 : 0.0f;
        // b of the coarse cell: restrict_sum's sum over the red children in order, the
        // (dy = 1) children being the next row's, eight lanes on
        const float q0 = __shfl_down_sync(0xffffffffu, r0, 8);
        const float q1 = __shfl_down_sync(0xffffffffu, r1, 8);
        if (p.own && (p.y & 1) == 0 && I < C.nx && J < C.ny && K < C.nz) {
          const int ci = level_index(C, I, J, K);
          const unsigned int cd = C.split ? (unsigned int)Cl.code16[ci] : (unsigned int)Cl.code[ci];
          if (cd & CODE_SELF) {
            const float bv =
                __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(r0, q0), r1), q1), 0.0625f);
            Cl.b[ci] = bv;
            // the coarse level's first red half-sweep, as in restrict_split
            if (C.split && ((I + J + K) & 1) == 0) Cl.x[ci] = gs_first(Cl.lvl, code_cnt(cd), bv);
          }
        }
      }
    }
    if (q + (int)team_size() < n) {
      e = L.blk[q + team_size()];
      w = L.tab[(size_t)(q + team_size()) * PCG_THREADS + threadIdx.x];
      if (POST) load(blk_pos(v, p, e));
    }
  }
  return PassSum{acc, true};
}

// ---------------------------------------------------------------- cycle pieces

// Pre-smoothing from zero and restriction, colour-split level l -> l+1.  The
// first red half-sweep from zero was made by the restriction into level l
// (restrict_split), behind the barrier that followed it.  Ends arrived at a barrier.
__device__ __forceinline__ bool down_split(const PcgArgs& A, int l) {
  const MgArgs& M = A.mg;
  const MgLevel& L = M.lv[l];
  const MgLevel& C = M.lv[l + 1];
  sweep_split<NORMAL>(M, L, C, l, 1, false);
  if (!gsync(A)) return false;
  for (int s = 1; s < M.nu; ++s) {
    sweep_split<NORMAL>(M, L, C, l, 0, false);
    if (!gsync(A)) return false;
    sweep_split<NORMAL>(M, L, C, l, 1, false);
    if (!gsync(A)) return false;
  }
  if (C.split) restrict_split(L, C);
  else restrict_split_nat(L, C);
  garrive(A);
  return true;
}

// Coarse correction from level l+1 and post-smoothing, colour-split level l.  Ends arrived
// at a barrier.
__device__ __forceinline__ bool up_split(const PcgArgs& A, int l) {
  const MgArgs& M = A.mg;
  const MgLevel& L = M.lv[l];
  const MgLevel& C = M.lv[l + 1];
  sweep_split<CORRECT>(M, L, C, l, 1, false);
  if (!gsync(A)) return false;
  sweep_split<NORMAL>(M, L, C, l, 0, false);
  for (int s = 1; s < M.nu; ++s) {
    if (!gsync(A)) return false;
    sweep_split<NORMAL>(M, L, C, l, 1, false);
    if (!gsync(A)) return false;
    sweep_split<NORMAL>(M, L, C, l, 0, false);
  }
  garrive(A);
  return true;
}

// ---------------------------------------------------------------- CTA-local levels in tiles
//
// Up to three CTA-local levels (their extents are then at most 16, 8 and 4 cells: all
// but long thin grids) run in the manner of block_pass's tiles, whole level and no halo:
// the 16^3 level on warps 0..15, the 8^3 level on warps 16 and 17, the 4^3 level on
// warp 18, each thread with a slot's eight cells in four planes in registers, as float2 a
// (planes 4 g, 4 g + 2) and b (4 g + 1, 4 g + 3), and the neighbours in shared memory.  A half-sweep waits only for its own level's warps, and the levels hand over
// by barriers of the two levels' warps.  The values are those of the list form below,
// sum for sum.
//
// Bound by latency: 22 dependent half-sweeps and residuals, and by instruction fetch,
// since one SM runs this code once per V-cycle: all levels share one copy of it (15 KB),
// with the level's shape in registers.  With its grid barrier 8.5 us at 64^3 and 11.1 at
// 256^3, where the solve's other code takes more of the instruction cache; a copy per
// level with constant shapes (37 KB) took 9.2 and 17.7, the list form 14 and 17-19.
constexpr int CT_THREADS = 512 + 64 + 8;

// The tile of each level's threads: 8 >> v slots, 16 >> v rows, 4 >> v plane groups; the
// entries of the arrays below are thread numbers (level v's from ct_first(v)).
struct CtaTiles {
  uint4 tab[CT_THREADS];                           // codes
  float2 a[2][CT_THREADS], b[2][CT_THREADS];       // x by colour (planes 4 g, 4 g + 2; 4 g + 1,
                                                   // 4 g + 3)
  float2 ra[2][CT_THREADS], rb[2][CT_THREADS];     // right-hand side, in the same form
};

__device__ __forceinline__ CtaTiles& cta_tiles();

__device__ __forceinline__ bool cta_tiled(const MgArgs& M) { return M.nlev - M.lgrid <= 3; }

__device__ __forceinline__ int ct_first(int v) { return v == 0 ? 0 : v == 1 ? 512 : 576; }

// A thread's level v (0: up to 16^3 cells, 1: 8^3, 2: 4^3; 3: none) and place in its tile.
struct CtPos {
  int v, ns, ny, ng;  // slots, rows, plane groups
  int s, y, g;
  bool live;          // owns cells (of the 4^3 level's warp only eight threads do)
};

__device__ __forceinline__ CtPos ct_pos() {
  const int id = (int)threadIdx.x;
  CtPos p;
  p.v = id < 512 ? 0 : id < 576 ? 1 : id < 608 ? 2 : 3;
  p.ns = 8 >> p.v;
  p.ny = 16 >> p.v;
  p.ng = 4 >> p.v;
  const int t = id - ct_first(p.v);
  p.s = t & (p.ns - 1);
  p.y = (t >> (3 - p.v)) & (p.ny - 1);
  p.g = t >> (7 - 2 * p.v);
  p.live = id < CT_THREADS;
  return p;
}

// Barrier of level v's warps, or (hand) of the warps of levels v and v + 1.
__device__ __forceinline__ void ct_sync(int v) {
  asm volatile("bar.sync %0, %1;" ::"r"(3 + v), "r"(v == 0 ? 512 : v == 1 ? 64 : 32) : "memory");
}
__device__ __forceinline__ void ct_hand(int v) {
  asm volatile("bar.sync %0, %1;" ::"r"(6 + v), "r"(v == 0 ? 512 + 64 : 64 + 32) : "memory");
}

// Code of plane z (0..3 in the thread's group), colour c.
__device__ __forceinline__ unsigned int tab_code(const uint4& w, int z, int c) {
  const unsigned int v = z == 0 ? w.x : z == 1 ? w.y : z == 2 ? w.z : w.w;
  return c ? v >> 16 : v & 0xffffu;
}

__device__ __forceinline__ float& plane(float2& a, float2& b, int z) {
  return z == 0 ? a.x : z == 1 ? b.x : z == 2 ? a.y : b.y;
}

// The float of plane z (0..3) of a pair of arrays at entry t.
__device__ __forceinline__ float& pair_at(float2* a, float2* b, int t, int z) {
  float2& v = (z & 1) ? b[t] : a[t];
  return (z & 2) ? v.y : v.x;
}

// The neighbours in colour o's arrays of a thread's cells of colour 1 - o, but for those
// that are its own cells: along x (oa, ob), y (ma, mb below, pa, pb above), and the
// plane before and after its four.  Beyond the tile's faces they are 0.
struct CtNbr {
  float2 oa, ob, ma, mb, pa, pb;
  float zprev, znext;
};

__device__ __forceinline__ CtNbr ct_nbr(const CtaTiles& S, const CtPos& p, int o) {
  const float2 zero = make_float2(0.0f, 0.0f);
  const float2* ta = S.a[o] + threadIdx.x;
  const float2* tb = S.b[o] + threadIdx.x;
  const bool up = (1 - o + p.y) & 1;  // the a planes' other x neighbour is the next slot
  const bool lo = p.s > 0, hi = p.s < p.ns - 1;
  const int pl = p.ns * p.ny;
  CtNbr n;
  n.oa = (up ? hi : lo) ? ta[up ? 1 : -1] : zero;
  n.ob = (up ? lo : hi) ? tb[up ? -1 : 1] : zero;
  n.ma = p.y > 0 ? ta[-p.ns] : zero;
  n.mb = p.y > 0 ? tb[-p.ns] : zero;
  n.pa = p.y < p.ny - 1 ? ta[p.ns] : zero;
  n.pb = p.y < p.ny - 1 ? tb[p.ns] : zero;
  n.zprev = p.g > 0 ? tb[-pl].y : 0.0f;
  n.znext = p.g < p.ng - 1 ? ta[pl].x : 0.0f;
  return n;
}

// The same sums as tile_sum, in the same order.
template <int c>
__device__ __forceinline__ void ct_sweep(CtaTiles& S, const CtPos& p, float2 (&xa)[2],
                                         float2 (&xb)[2], const float2 (&ia)[2],
                                         const float2 (&ib)[2], const float2 (&ba)[2],
                                         const float2 (&bb)[2]) {
  constexpr int o = 1 - c;
  if (!p.live) return;
  const CtNbr n = ct_nbr(S, p, o);
  float2 sa = __fadd2_rn(xa[o], n.oa), sb = __fadd2_rn(xb[o], n.ob);
  sa = __fadd2_rn(sa, n.ma);
  sb = __fadd2_rn(sb, n.mb);
  sa = __fadd2_rn(sa, n.pa);
  sb = __fadd2_rn(sb, n.pb);
  sa = __fadd2_rn(sa, make_float2(n.zprev, xb[o].x));
  sb = __fadd2_rn(sb, xa[o]);
  sa = __fadd2_rn(sa, xb[o]);
  sb = __fadd2_rn(sb, make_float2(xa[o].y, n.znext));
  xa[c] = __ffma2_rn(sa, ia[c], ba[c]);
  xb[c] = __ffma2_rn(sb, ib[c], bb[c]);
  S.a[c][threadIdx.x] = xa[c];
  S.b[c][threadIdx.x] = xb[c];
}

// Levels [lgrid, nlev) inside CTA 0 in tile form, from level lgrid's global b to its
// global x, as cta_cycle.
__device__ __noinline__ void cta_cycle_tiled(const MgArgs& M) {
  const CtPos p = ct_pos();
  const int l = M.nlev - 3 + p.v;  // the thread's level
  if (p.v == 3 || l < M.lgrid) return;
  CtaTiles& S = cta_tiles();
  const MgLevel& L = M.lv[l];
  const bool top = l == M.lgrid, coarsest = p.v == 2;
  const uint4 w = p.live ? S.tab[threadIdx.x] : make_uint4(0u, 0u, 0u, 0u);
  const int nat = L.nx * (p.y + L.ny * 4 * p.g) + 2 * p.s, nsl = L.nx * L.ny;  // natural index
  float2 xa[2], xb[2], ia[2], ib[2], ba[2], bb[2], ra[2], rb[2];
  if (top) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int z = 0; z < 4; ++z)
        plane(ra[c], rb[c], z) =
            tab_code(w, z, c) ? L.b[nat + z * nsl + ((c + p.y + z) & 1)] : 0.0f;
  } else {
    ct_hand(p.v - 1);  // the finer level's restriction is done
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float2 zero = make_float2(0.0f, 0.0f);
      ra[c] = p.live ? S.ra[c][threadIdx.x] : zero;
      rb[c] = p.live ? S.rb[c][threadIdx.x] : zero;
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const int cnt = code_cnt(tab_code(w, z, c));  // 0 where there is no fluid cell
      plane(ia[c], ib[c], z) = s_inv_cnt[cnt];
      plane(ba[c], bb[c], z) = __fmul_rn(plane(ra[c], rb[c], z), s_inv_scnt[l][cnt]);
    }
  xa[0] = ba[0];
  xb[0] = bb[0];
  xa[1] = xb[1] = make_float2(0.0f, 0.0f);
  const int cfirst = ct_first(p.v + 1), cns = p.ns >> 1, cny = p.ny >> 1;  // the coarser tile
  const int I = p.s, J = p.y >> 1;  // the red cells' parents: (I, J, 2 g) and (I, J, 2 g + 1)
#pragma unroll 1
  for (int post = 0;; ++post) {
    if (p.live) {
      S.a[0][threadIdx.x] = xa[0];
      S.b[0][threadIdx.x] = xb[0];
    }
    ct_sync(p.v);
    // the coarsest level: MG_COARSE_SWEEPS (red, black) pairs from zero, then as many
    // (black, red) pairs, as one alternating sequence (see coarsest_cta)
    const int pairs = coarsest ? 2 * MG_COARSE_SWEEPS - 1 : M.nu;
#pragma unroll 1
    for (int h = 0; h < pairs; ++h) {
      ct_sweep<1>(S, p, xa, xb, ia, ib, ba, bb);
      ct_sync(p.v);
      if (!coarsest && post == 0 && h + 1 == pairs) break;
      ct_sweep<0>(S, p, xa, xb, ia, ib, ba, bb);
      ct_sync(p.v);
    }
    if (coarsest || post == 1) break;
    // residuals of the red cells and the coarser level's right-hand side (restrict_cta)
    float r[4], r1[4];
    {
      CtNbr n = ct_nbr(S, p, 1);
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const unsigned int cd = tab_code(w, z, 0);
        const float own = plane(xa[1], xb[1], z), other = plane(n.oa, n.ob, z);
        const bool low = ((z + p.y) & 1) == 0;  // the other slot is the -x neighbour
        const float xv[6] = {low ? other : own,
                             low ? own : other,
                             plane(n.ma, n.mb, z),
                             plane(n.pa, n.pb, z),
                             z == 0 ? n.zprev : plane(xa[1], xb[1], z > 0 ? z - 1 : 0),
                             z == 3 ? n.znext : plane(xa[1], xb[1], z < 3 ? z + 1 : 3)};
        const float rr = resid(L.s, code_cnt(cd), cd, plane(ra[0], rb[0], z),
                               plane(xa[0], xb[0], z), xv);
        r[z] = cd ? rr : 0.0f;
      }
    }
#pragma unroll
    for (int z = 0; z < 4; ++z) r1[z] = __shfl_down_sync(0xffffffffu, r[z], p.ns);
    int pt[2], pz[2];  // the parents' entries and planes
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int K = 2 * p.g + h;
      pt[h] = cfirst + ((K >> 2) * cny + J) * cns + (I >> 1) + ((I + J + K) & 1) * CT_THREADS;
      pz[h] = K & 3;
    }
    if ((p.y & 1) == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float sum = __fadd_rn(__fadd_rn(__fadd_rn(r[2 * h], r1[2 * h]), r[2 * h + 1]),
                                    r1[2 * h + 1]);
        pair_at(S.ra[0], S.rb[0], pt[h], pz[h]) = __fmul_rn(sum, 0.0625f);
      }
    }
    ct_hand(p.v);  // to the coarser level
    ct_hand(p.v);  // and back
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      float& x = plane(xa[0], xb[0], z);
      const float px = pair_at(S.a[0], S.b[0], pt[z >> 1], pz[z >> 1]);
      x = tab_code(w, z, 0) ? __fmaf_rn(M.omega, px, x) : 0.0f;
    }
  }
  if (top) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (tab_code(w, z, c))
          L.x[nat + z * nsl + ((c + p.y + z) & 1)] = plane(xa[c], xb[c], z);
  } else {
    ct_hand(p.v - 1);  // x is in shared memory for the finer level
  }
}

// Once per solve, after build_levels: CTA 0's codes, code bits plus the count of
// neighbours inside the grid, 0 where there is no fluid cell; x starts as 0.
__device__ __noinline__ void cta_tiles_init(const MgArgs& M) {
  const CtPos p = ct_pos();
  const int l = M.nlev - 3 + p.v;
  if (!p.live || l < M.lgrid) return;
  CtaTiles& S = cta_tiles();
  const MgLevel& L = M.lv[l];
  unsigned int cd[4];
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    cd[z] = 0u;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = 2 * p.s + ((c + p.y + z) & 1), j = p.y, k = 4 * p.g + z;
      if (i >= L.nx || j >= L.ny || k >= L.nz) continue;
      const unsigned int code = L.code[i + L.nx * (j + L.ny * k)];
      const int cnt = (i > 0) + (i < L.nx - 1) + (j > 0) + (j < L.ny - 1) + (k > 0) +
                      (k < L.nz - 1);
      if (code & CODE_SELF) cd[z] |= (code | (unsigned)cnt << 8) << (16 * c);
    }
  }
  S.tab[threadIdx.x] = make_uint4(cd[0], cd[1], cd[2], cd[3]);
}

// ---------------------------------------------------------------- CTA-local levels by lists

// The CTA-local levels [lgrid, nlev) live in CTA 0's (dynamic) shared memory:
// x, b and the neighbour codes of every such level (MG_CTA_CELLS cells in all),
// and per level and colour the list of its fluid cells, each as the packed
// coordinates i | j << bx | k << (bx + by) with bx, by the bits of nx - 1 and
// ny - 1 (at most 16 bits, since a CTA-local level has fewer than 2^13 cells).
// A half-sweep then visits exactly the fluid cells of its colour, with no
// divisions and no idle slots.
struct CtaMg {
  float x[MG_CTA_CELLS];
  float b[MG_CTA_CELLS];
  uint8_t code[MG_CTA_CELLS];
  uint16_t list[MG_CTA_CELLS];
  int off[MG_MAX_LEVELS][3];   // list of level l: colour 0 [off0, off1), colour 1 [off1, off2)
  int base[MG_MAX_LEVELS];     // first cell of level l in x, b, code
  int nx[MG_MAX_LEVELS], ny[MG_MAX_LEVELS], nz[MG_MAX_LEVELS];
  int bx[MG_MAX_LEVELS], by[MG_MAX_LEVELS];
  float s[MG_MAX_LEVELS];
};

// CTA 0's CTA-local levels sit at the start of the kernel's dynamic shared memory;
// reached through this (not a pointer argument) the compiler addresses them as
// shared memory.
__device__ __forceinline__ CtaMg& cta_mg() {
  extern __shared__ __align__(16) unsigned char mg_dyn[];
  return *reinterpret_cast<CtaMg*>(mg_dyn);
}

// The tile form's arrays lie in the same place.
__device__ __forceinline__ CtaTiles& cta_tiles() {
  static_assert(sizeof(CtaTiles) <= sizeof(CtaMg), "shares the list form's memory");
  extern __shared__ __align__(16) unsigned char mg_dyn[];
  return *reinterpret_cast<CtaTiles*>(mg_dyn);
}

__device__ __forceinline__ int bits_for(int n) {  // bits of n - 1 (0 for n = 1)
  return n > 1 ? 32 - __clz(n - 1) : 0;
}

struct CtaCell {
  int i, j, k, c;
};

__device__ __forceinline__ CtaCell cta_cell(const CtaMg& sm, int l, unsigned int e) {
  const int bx = sm.bx[l], by = sm.by[l];
  CtaCell r;
  r.i = (int)(e & ((1u << bx) - 1u));
  r.j = (int)((e >> bx) & ((1u << by) - 1u));
  r.k = (int)(e >> (bx + by));
  r.c = r.i + sm.nx[l] * (r.j + sm.ny[l] * r.k);
  return r;
}

// Half-sweep of one colour over CTA-local level l (parents on level l + 1).
template <int MODE>
__device__ __noinline__ void sweep_cta(float omega, int l, int colour) {
  static_assert(MODE != FIRST, "the first half-sweep of a CTA-local level comes with its b");
  CtaMg& sm = cta_mg();
  const int nx = sm.nx[l], ny = sm.ny[l], nz = sm.nz[l], sy = nx, sz = nx * ny;
  float* x = sm.x + sm.base[l];
  const float* b = sm.b + sm.base[l];
  const uint8_t* code = sm.code + sm.base[l];
  const int e1 = sm.off[l][colour + 1];
  for (int e = sm.off[l][colour] + (int)threadIdx.x; e < e1; e += PCG_THREADS) {
    const CtaCell p = cta_cell(sm, l, sm.list[e]);
    const int cnt = (p.i > 0) + (p.i < nx - 1) + (p.j > 0) + (p.j < ny - 1) + (p.k > 0) +
                    (p.k < nz - 1);
    const unsigned int cd = code[p.c];
    const int off[6] = {-1, 1, -sy, sy, -sz, sz};
    float xv[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) xv[q] = ((cd >> q) & 1u) ? x[p.c + off[q]] : 0.0f;
    if constexpr (MODE == CORRECT) {
      const float* px = sm.x + sm.base[l + 1];
      const int pnx = sm.nx[l + 1], pny = sm.ny[l + 1];
      const int di[6] = {-1, 1, 0, 0, 0, 0}, dj[6] = {0, 0, -1, 1, 0, 0}, dk[6] = {0, 0, 0, 0, -1, 1};
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if ((cd >> q) & 1u) {
          const int pi = (p.i + di[q]) >> 1, pj = (p.j + dj[q]) >> 1, pk = (p.k + dk[q]) >> 1;
          xv[q] = __fmaf_rn(omega, px[pi + pnx * (pj + pny * pk)], xv[q]);
        }
    }
    x[p.c] = gs_sum(l, cnt, cd, b[p.c], xv);
  }
}

// b_{l+1} = (1/16) sum of the red fluid children's residuals, over level l+1's
// fluid cells (both colours), and the first red half-sweep of level l+1 from
// zero: x = gs_first(b) on its red cells.  Four consecutive lanes take the four
// red children of one coarse cell, and the group's first lane adds their
// residuals in child order.
__device__ __noinline__ void restrict_cta(int l) {
  CtaMg& sm = cta_mg();
  const int nx = sm.nx[l], ny = sm.ny[l], nz = sm.nz[l], sy = nx, sz = nx * ny;
  const int cnx = sm.nx[l + 1], cny = sm.ny[l + 1], cnz = sm.nz[l + 1];
  const float* x = sm.x + sm.base[l];
  const float* b = sm.b + sm.base[l];
  const uint8_t* code = sm.code + sm.base[l];
  float* cb = sm.b + sm.base[l + 1];
  float* cx = sm.x + sm.base[l + 1];
  const float sl = sm.s[l];
  const int e0 = sm.off[l + 1][0], ered = sm.off[l + 1][1];
  const int n4 = 4 * (sm.off[l + 1][2] - e0);
  const int lane = threadIdx.x & 31;
  for (int e4 = (int)threadIdx.x; e4 - lane < n4; e4 += PCG_THREADS) {  // warp-uniform bound
    const bool live = e4 < n4;
    float r = 0.0f;
    bool has = false;
    CtaCell P = {0, 0, 0, 0};
    if (live) {
      P = cta_cell(sm, l + 1, sm.list[e0 + (e4 >> 2)]);
      const int q = e4 & 3, dy = q & 1, dz = q >> 1, dx = (dy + dz) & 1;
      const int i = 2 * P.i + dx, j = 2 * P.j + dy, k = 2 * P.k + dz;
      if (i < nx && j < ny && k < nz) {
        const int fc = i + nx * (j + ny * k);
        const unsigned int cd = code[fc];
        if (cd & CODE_SELF) {
          const int off[6] = {-1, 1, -sy, sy, -sz, sz};
          float xv[6];
#pragma unroll
          for (int u = 0; u < 6; ++u) xv[u] = ((cd >> u) & 1u) ? x[fc + off[u]] : 0.0f;
          const int cnt = (i > 0) + (i < nx - 1) + (j > 0) + (j < ny - 1) + (k > 0) + (k < nz - 1);
          r = resid(sl, cnt, cd, b[fc], x[fc], xv);
          has = true;
        }
      }
    }
    const unsigned int hm = __ballot_sync(0xffffffffu, has) >> (lane & ~3);
    const float r1 = __shfl_down_sync(0xffffffffu, r, 1);
    const float r2 = __shfl_down_sync(0xffffffffu, r, 2);
    const float r3 = __shfl_down_sync(0xffffffffu, r, 3);
    if (live && (e4 & 3) == 0) {
      float sum = 0.0f;
      if (hm & 1u) sum = __fadd_rn(sum, r);
      if (hm & 2u) sum = __fadd_rn(sum, r1);
      if (hm & 4u) sum = __fadd_rn(sum, r2);
      if (hm & 8u) sum = __fadd_rn(sum, r3);
      const float bc = __fmul_rn(sum, 0.0625f);
      cb[P.c] = bc;
      if (e0 + (e4 >> 2) < ered) {
        const int cnt = (P.i > 0) + (P.i < cnx - 1) + (P.j > 0) + (P.j < cny - 1) + (P.k > 0) +
                        (P.k < cnz - 1);
        cx[P.c] = gs_first(l + 1, cnt, bc);
      }
    }
  }
}

// Points the shared level descriptions at the shared arrays, loads the codes and
// builds the fluid-cell lists (once per solve, after build_levels).  CTA 0 only.
__device__ __noinline__ void cta_levels_init(const MgArgs& M) {
  CtaMg& sm = cta_mg();
  __shared__ unsigned int s_wc[PCG_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    int off = 0;
    for (int l = M.lgrid; l < M.nlev; ++l) {
      sm.base[l] = off;
      sm.nx[l] = M.lv[l].nx;
      sm.ny[l] = M.lv[l].ny;
      sm.nz[l] = M.lv[l].nz;
      sm.bx[l] = bits_for(M.lv[l].nx);
      sm.by[l] = bits_for(M.lv[l].ny);
      sm.s[l] = M.lv[l].s;
      off += M.lv[l].ncells;
    }
  }
  __syncthreads();
  // Per level: each thread takes a contiguous run of cells, counts its fluid cells
  // of each colour (the two counts packed in one word: a level has fewer than 2^16
  // cells), a block-wide exclusive scan gives each run its place, and the runs
  // write their entries: colour 0's list then colour 1's, each in cell order.
  __shared__ unsigned int s_scan[PCG_WARPS];
  int pos = 0;  // next free list entry (same value in every thread)
  for (int l = M.lgrid; l < M.nlev; ++l) {
    const int n = M.lv[l].ncells, nx = sm.nx[l], ny = sm.ny[l], bl = sm.base[l];
    for (int c = threadIdx.x; c < n; c += PCG_THREADS) sm.code[bl + c] = M.lv[l].code[c];
    __syncthreads();
    const int per = (n + PCG_THREADS - 1) / PCG_THREADS;
    const int c0 = min(n, (int)threadIdx.x * per), c1 = min(n, c0 + per);
    unsigned int mine = 0;  // colour 0 in the low half, colour 1 in the high half
    for (int c = c0; c < c1; ++c) {
      const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
      if (sm.code[bl + c] & CODE_SELF) mine += ((i + j + k) & 1) ? 0x10000u : 1u;
    }
    unsigned int inc = mine;  // inclusive scan over the warp, then over the warps
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned int v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (lane == 31) s_scan[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const unsigned int t = lane < PCG_WARPS ? s_scan[lane] : 0u;
      unsigned int w = t;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned int v = __shfl_up_sync(0xffffffffu, w, d);
        if (lane >= d) w += v;
      }
      if (lane < PCG_WARPS) s_scan[lane] = w - t;  // exclusive, per warp
      const unsigned int tot = __shfl_sync(0xffffffffu, w, 31);
      if (lane == 0) s_wc[0] = tot;
    }
    __syncthreads();
    const unsigned int before = s_scan[warp] + inc - mine, tot = s_wc[0];
    const int n0 = (int)(tot & 0xffffu), n1 = (int)(tot >> 16);
    int p0 = pos + (int)(before & 0xffffu), p1 = pos + n0 + (int)(before >> 16);
    for (int c = c0; c < c1; ++c) {
      if (!(sm.code[bl + c] & CODE_SELF)) continue;
      const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
      const uint16_t e = (uint16_t)(i | (j << sm.bx[l]) | (k << (sm.bx[l] + sm.by[l])));
      if ((i + j + k) & 1) sm.list[p1++] = e;
      else sm.list[p0++] = e;
    }
    if (threadIdx.x == 0) {
      sm.off[l][0] = pos;
      sm.off[l][1] = pos + n0;
      sm.off[l][2] = pos + n0 + n1;
    }
    pos += n0 + n1;
    __syncthreads();
  }
}

// The same cycle pieces as for the grid-wide levels, inside CTA 0.  The first
// red half-sweep of a level (from zero) is done where its b is made: in the
// copy-in for level lgrid, in the restriction for the levels below.
__device__ __forceinline__ void down_cta(const MgArgs& M, int l) {
  sweep_cta<NORMAL>(M.omega, l, 1);
  __syncthreads();
  for (int s = 1; s < M.nu; ++s) {
    sweep_cta<NORMAL>(M.omega, l, 0);
    __syncthreads();
    sweep_cta<NORMAL>(M.omega, l, 1);
    __syncthreads();
  }
  restrict_cta(l);
  __syncthreads();
}

__device__ __forceinline__ void up_cta(const MgArgs& M, int l) {
  sweep_cta<CORRECT>(M.omega, l, 1);
  __syncthreads();
  sweep_cta<NORMAL>(M.omega, l, 0);
  __syncthreads();
  for (int s = 1; s < M.nu; ++s) {
    sweep_cta<NORMAL>(M.omega, l, 1);
    __syncthreads();
    sweep_cta<NORMAL>(M.omega, l, 0);
    __syncthreads();
  }
}

// The coarsest level: MG_COARSE_SWEEPS (red, black) pairs from zero, then as many
// (black, red) pairs, run as one alternating sequence: the second of the two black
// half-sweeps in the middle would repeat the first on the same red values.
__device__ __forceinline__ void coarsest_cta(const MgArgs& M, int l) {
  for (int h = 1; h < 4 * MG_COARSE_SWEEPS - 1; ++h) {  // black, red, ..., red
    sweep_cta<NORMAL>(M.omega, l, h & 1);
    __syncthreads();
  }
}

// Levels [lgrid, nlev) inside CTA 0, from the right-hand side that the grid-wide
// restriction left in level lgrid's global b; leaves level lgrid's x in global
// memory for the correction of level lgrid - 1.
__device__ __noinline__ void cta_cycle(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  CtaMg& sm = cta_mg();
  const int lg = M.lgrid;
  const int n = M.lv[lg].ncells;
  const float* gb = M.lv[lg].b;
  float* gx = M.lv[lg].x;
  // b of level lgrid (all loads of a thread before its stores), and the first red
  // half-sweep of level lgrid from zero on the same values
  constexpr int U = 4;
  float* sb = sm.b + sm.base[lg];
  for (int c0 = threadIdx.x; c0 < n; c0 += U * PCG_THREADS) {
    float v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int c = c0 + u * PCG_THREADS;
      v[u] = c < n ? gb[c] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int c = c0 + u * PCG_THREADS;
      if (c < n) sb[c] = v[u];
    }
  }
  {
    const int nx = sm.nx[lg], ny = sm.ny[lg], nz = sm.nz[lg];
    float* sx = sm.x + sm.base[lg];
    const int e1 = sm.off[lg][1];
    for (int e = sm.off[lg][0] + (int)threadIdx.x; e < e1; e += PCG_THREADS) {
      const CtaCell p = cta_cell(sm, lg, sm.list[e]);
      const int cnt = (p.i > 0) + (p.i < nx - 1) + (p.j > 0) + (p.j < ny - 1) + (p.k > 0) +
                      (p.k < nz - 1);
      sx[p.c] = gs_first(lg, cnt, gb[p.c]);
    }
  }
  __syncthreads();
  for (int l = lg; l < M.nlev - 1; ++l) down_cta(M, l);
  coarsest_cta(M, M.nlev - 1);
  for (int l = M.nlev - 2; l >= lg; --l) up_cta(M, l);
  for (int c = threadIdx.x; c < n; c += PCG_THREADS) gx[c] = sm.x[sm.base[lg] + c];
}

// z = V(r), given that the first red half-sweep of level 0 (from zero) has been
// done in the phase that produced r, and that a grid barrier has passed since.
// Returns r.z over the CTA's cells, from the last black and the last red half-sweeps of
// level 0 (the caller publishes it and meets the next barrier); ok is false if a barrier
// failed.
__device__ __noinline__ PassSum vcycle_rest(const PcgArgs& A) {
  PassSum V{FF(), false};
  const MgArgs& M = A.mg;
  const MgLevel& L0 = M.lv[0];
  if (M.nlev == 1) {  // level 0 is the coarsest level
    // rest of the pre pairs (red, black) after the fused first red half-sweep
    for (int s = 0; s < MG_COARSE_SWEEPS; ++s) {
      sweep_split<NORMAL>(M, L0, L0, 0, 1, false);
      if (!gsync(A)) return V;
      if (s + 1 < MG_COARSE_SWEEPS) {
        sweep_split<NORMAL>(M, L0, L0, 0, 0, false);
        if (!gsync(A)) return V;
      }
    }
    // post pairs (black, red); the last black and the last red give r.z
    for (int s = 0; s < MG_COARSE_SWEEPS; ++s) {
      V.sum = sweep_split<NORMAL>(M, L0, L0, 0, 1, s + 1 == MG_COARSE_SWEEPS);
      if (!gsync(A)) return V;
      if (s + 1 < MG_COARSE_SWEEPS) {
        sweep_split<NORMAL>(M, L0, L0, 0, 0, false);
        if (!gsync(A)) return V;
      }
    }
    V.sum.add(sweep_split<NORMAL>(M, L0, L0, 0, 0, true));
    V.ok = true;
    return V;
  }
  const MgLevel& L1 = M.lv[1];
  const bool blocked0 = s_nblk[0] > 0;
  if (blocked0) {
    if (!block_pass<false, false>(A, 0, false).ok) return V;
  } else {
    sweep_split<NORMAL>(M, L0, L1, 0, 1, false);
    if (!gsync(A)) return V;
    SOLVE_TRACE(TR_V_PRE1);
    for (int s = 1; s < M.nu; ++s) {
      sweep_split<NORMAL>(M, L0, L1, 0, 0, false);
      if (!gsync(A)) return V;
      sweep_split<NORMAL>(M, L0, L1, 0, 1, false);
      if (!gsync(A)) return V;
    }
    SOLVE_TRACE(TR_V_PRE);
    if (L1.split) restrict_split(L0, L1);
    else restrict_split_nat(L0, L1);
  }
  garrive(A);  // from here to level 0, every pass waits for the barrier before it
  for (int l = 1; l < M.lgrid; ++l) {
    if (s_nblk[l] > 0) {
      if (!block_pass<false, false>(A, l, true).ok) return V;
      SOLVE_TRACE(l == 1 ? TR_V_RESTRICT : TR_V_DOWN + min(l - 1, 11));
      garrive(A);
    } else {
      if (!gwait(A)) return V;
      SOLVE_TRACE(l == 1 ? TR_V_RESTRICT : TR_V_DOWN + min(l - 1, 11));
      if (!down_split(A, l)) return V;
    }
  }
  if (!gwait(A)) return V;
  SOLVE_TRACE(M.lgrid == 1 ? TR_V_RESTRICT : TR_V_DOWN + min(M.lgrid - 1, 11));
  if (team_rank() == 0) {
    if (cta_tiled(M)) cta_cycle_tiled(M);
    else cta_cycle(A);
  }
  garrive(A);
  for (int l = M.lgrid - 1; l >= 1; --l) {
    if (s_nblk[l] > 0) {
      if (!block_pass<true, false>(A, l, true).ok) return V;
      SOLVE_TRACE(l == M.lgrid - 1 ? TR_V_CTA : TR_V_UP + min(l + 1, 11));
      garrive(A);
    } else {
      if (!gwait(A)) return V;
      SOLVE_TRACE(l == M.lgrid - 1 ? TR_V_CTA : TR_V_UP + min(l + 1, 11));
      if (!up_split(A, l)) return V;
    }
  }
  if (blocked0) return block_pass<true, true>(A, 0, true);
  if (!gwait(A)) return V;
  SOLVE_TRACE(M.lgrid == 1 ? TR_V_CTA : TR_V_UP + 1);
  V.sum = sweep_split<CORRECT>(M, L0, L1, 0, 1, M.nu == 1);
  if (!gsync(A)) return V;
  SOLVE_TRACE(TR_V_CORRECT);
  for (int s = 1; s < M.nu; ++s) {
    sweep_split<NORMAL>(M, L0, L1, 0, 0, false);
    if (!gsync(A)) return V;
    V.sum = sweep_split<NORMAL>(M, L0, L1, 0, 1, s + 1 == M.nu);
    if (!gsync(A)) return V;
  }
  SOLVE_TRACE(TR_V_POST);
  V.sum.add(sweep_split<NORMAL>(M, L0, L1, 0, 0, true));  // the last red half-sweep
  V.ok = true;
  return V;
}

// ---------------------------------------------------------------- level-0 passes

// Phase A with z from the V-cycle: p_new = z + beta p_old (recomputed for the
// neighbours), q = A p_new in difference form, partial p.q.  Both colours; a lane takes two
// slots, the pair's and its neighbour pairs' operations packed.
__device__ __noinline__ FF phase_a_v(const PcgArgs& A, const float* pold, float* pnew, float beta) {
  const MgArgs& M = A.mg;
  const SV v = sview(M.lv[0]);
  const float* z = s_z0;
  float* q0 = s_q0;
  const float s_a = A.s;
  const int lane = threadIdx.x & 31;
  const int2 q = seg_slice(M.lv[0]);
  const Items it = pair_items(q, 2);
  const float2 beta2 = make_float2(beta, beta);
  FF acc;
  auto p_at = [&](int i) {  // p_new of a pair of slots
    return __ffma2_rn(beta2, *reinterpret_cast<const float2*>(pold + i),
                      *reinterpret_cast<const float2*>(z + i));
  };
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const PCell e = pcell(v, q, t >> 1, (int)(t & 1u), lane);
    const unsigned int code2 = *reinterpret_cast<const unsigned int*>(v.code + e.idx);
    const float2 pc = p_at(e.idx), m = p_at(e.ob);
    const float2 ym = p_at(e.ob - v.hx), yp = p_at(e.ob + v.hx);
    const float2 zm = p_at(e.ob - v.pl), zp = p_at(e.ob + v.pl);
    const int ei = e.ob - 1 + 3 * e.par;  // slot s - 1 (par 0) or s + 2 (par 1)
    const float ex = __fmaf_rn(beta, pold[ei], z[ei]);
    const float2 xm = e.par ? m : make_float2(ex, m.x);
    const float2 xp = e.par ? make_float2(m.y, ex) : m;
    const float2 n[6] = {xm, xp, ym, yp, zm, zp};
    const unsigned int cA = e.okA ? code2 & 0xffffu : 0u, cB = e.okB ? code2 >> 16 : 0u;
    float dA = 0.0f, dB = 0.0f;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const float2 d = __fadd2_rn(pc, make_float2(-n[u].x, -n[u].y));
      if ((cA >> u) & 1u) dA = __fadd_rn(dA, d.x);
      if ((cB >> u) & 1u) dB = __fadd_rn(dB, d.y);
    }
    const float nA = (float)(code_cnt(cA) - __popc(cA & 63u));  // neighbours in air
    const float nB = (float)(code_cnt(cB) - __popc(cB & 63u));
    const float2 pn = make_float2(cA ? pc.x : 0.0f, cB ? pc.y : 0.0f);
    const float2 qn = make_float2(cA ? __fmul_rn(s_a, __fmaf_rn(nA, pc.x, dA)) : 0.0f,
                                  cB ? __fmul_rn(s_a, __fmaf_rn(nB, pc.y, dB)) : 0.0f);
    acc.add_prod(pn.x, qn.x);
    acc.add_prod(pn.y, qn.y);
    if (e.okA || e.okB) {
      *reinterpret_cast<float2*>(pnew + e.idx) = pn;
      *reinterpret_cast<float2*>(q0 + e.idx) = qn;
    }
  }
  return acc;
}

// Phase B: d += alpha p, r -= alpha q, partial r.r, and the next V-cycle's first
// red half-sweep (from zero) z = r / (s n) on red cells.  Both colours, four slots a lane.
__device__ __noinline__ FF phase_b_q(const PcgArgs& A, const float* pnew, float alpha) {
  const MgArgs& M = A.mg;
  const SV v = sview(M.lv[0]);
  float* d0 = M.d0;
  const float* q0 = s_q0;
  const bool first_red = s_nblk[0] == 0;  // a blocked level 0 makes it from r itself
  const int lane = threadIdx.x & 31;
  const int2 q = seg_slice(M.lv[0]);
  const Items it = quad_items(q, 2);
  FF acc;
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const int c = (int)(t & 1u);
    const QCell e = qcell(v, q, t >> 1, c, lane);
    if (!e.ok) continue;
    const uint2 code4 = *reinterpret_cast<const uint2*>(v.code + e.idx);
    const float4 d4 = *reinterpret_cast<const float4*>(d0 + e.idx);
    const float4 p4 = *reinterpret_cast<const float4*>(pnew + e.idx);
    const float4 q4 = *reinterpret_cast<const float4*>(q0 + e.idx);
    const float4 r4 = *reinterpret_cast<const float4*>(v.b + e.idx);
    const float dd[4] = {d4.x, d4.y, d4.z, d4.w}, pp[4] = {p4.x, p4.y, p4.z, p4.w};
    const float qq[4] = {q4.x, q4.y, q4.z, q4.w}, rr[4] = {r4.x, r4.y, r4.z, r4.w};
    float dn[4], rn[4], zn[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int cnt = quad_cnt(code4, h);  // 0: not fluid
      const float rc = __fmaf_rn(-alpha, qq[h], rr[h]);
      dn[h] = cnt ? __fmaf_rn(alpha, pp[h], dd[h]) : dd[h];
      rn[h] = cnt ? rc : rr[h];
      zn[h] = cnt ? gs_first(0, cnt, rc) : 0.0f;
      const float rs = cnt ? rc : 0.0f;
      acc.add_prod(rs, rs);
    }
    *reinterpret_cast<float4*>(d0 + e.idx) = make_float4(dn[0], dn[1], dn[2], dn[3]);
    *reinterpret_cast<float4*>(v.b + e.idx) = make_float4(rn[0], rn[1], rn[2], rn[3]);
    if (first_red && c == 0)
      *reinterpret_cast<float4*>(v.x + e.idx) = make_float4(zn[0], zn[1], zn[2], zn[3]);
  }
  return acc;
}

// Phase A with z from the V-cycle: p_new = z + beta p_old (recomputed for the
// neighbours), q = A p_new in difference form, partial p.q.  Both colours.
__device__ __noinline__ FF phase_a_s(const PcgArgs& A, const float* pold, float* pnew, float beta) {
  const MgArgs& M = A.mg;
  const SV v = sview(M.lv[0]);
  const float* z = s_z0;
  float* q0 = s_q0;
  const float s_a = A.s;
  const int lane = threadIdx.x & 31;
  const Items it = seg_items(M.lv[0], 2);
  struct S {
    int idx;
    bool ok;
    unsigned int code;
    float zc, pc;
    float zv[6], pv[6];
  };
  FF acc;
  run_batched<1>(
      it.first, it.end, PCG_WARPS,
      [&](unsigned int t, bool ok) {
        const SCell e = scell(v, v.seg[(int)(t >> 1) - v.seg_base], (int)(t & 1u), lane);
        S s;
        s.idx = e.idx;
        s.ok = e.ok && ok;
        s.code = v.code[e.idx];
        s.zc = z[e.idx];
        s.pc = pold[e.idx];
        int nb[6];
        snbr(v, e, nb);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          s.zv[q] = z[nb[q]];
          s.pv[q] = pold[nb[q]];
        }
        return s;
      },
      [&](S&) {},
      [&](S& s) {
        if (!s.ok || !(s.code & CODE_SELF)) return;
        const int cnt = code_cnt(s.code);
        const float pc = __fmaf_rn(beta, s.pc, s.zc);
        float d = 0.0f;
        int nfl = 0;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          const bool f = (s.code >> q) & 1u;
          d += f ? __fsub_rn(pc, __fmaf_rn(beta, s.pv[q], s.zv[q])) : 0.0f;
          nfl += f;
        }
        const float qc = __fmul_rn(s_a, __fmaf_rn((float)(cnt - nfl), pc, d));
        pnew[s.idx] = pc;
        q0[s.idx] = qc;
        acc.add_prod(pc, qc);
      });
  return acc;
}

// Phase B: d += alpha p, r -= alpha q, partial r.r, and the next V-cycle's first
// red half-sweep (from zero) z = r / (s n) on red cells.  Both colours.
__device__ __noinline__ FF phase_b_s(const PcgArgs& A, const float* pnew, float alpha) {
  const MgArgs& M = A.mg;
  const SV v = sview(M.lv[0]);
  float* d0 = M.d0;
  const float* q0 = s_q0;
  const bool first_red = s_nblk[0] == 0;  // a blocked level 0 makes it from r itself
  const int lane = threadIdx.x & 31;
  const Items it = seg_items(M.lv[0], 2);
  struct S {
    int idx, c;
    bool ok;
    unsigned int code;
    float d, p, q, r;
  };
  FF acc;
  run_batched<2>(
      it.first, it.end, PCG_WARPS,
      [&](unsigned int t, bool ok) {
        const SCell e = scell(v, v.seg[(int)(t >> 1) - v.seg_base], (int)(t & 1u), lane);
        S s;
        s.idx = e.idx;
        s.c = (int)(t & 1u);
        s.ok = e.ok && ok;
        s.code = v.code[e.idx];
        s.d = d0[e.idx];
        s.p = pnew[e.idx];
        s.q = q0[e.idx];
        s.r = v.b[e.idx];
        return s;
      },
      [&](S&) {},
      [&](S& s) {
        if (!s.ok || !(s.code & CODE_SELF)) return;
        d0[s.idx] = __fmaf_rn(alpha, s.p, s.d);
        const float rc = __fmaf_rn(-alpha, s.q, s.r);
        v.b[s.idx] = rc;
        if (first_red && s.c == 0) v.x[s.idx] = gs_first(0, code_cnt(s.code), rc);
        acc.add_prod(rc, rc);
      });
  return acc;
}

__device__ __forceinline__ FF phase_a(const PcgArgs& A, const float* pold, float* pnew,
                                      float beta) {
  return use_wide(A.mg.lv[0]) ? phase_a_v(A, pold, pnew, beta) : phase_a_s(A, pold, pnew, beta);
}

__device__ __forceinline__ FF phase_b(const PcgArgs& A, const float* pnew, float alpha) {
  return use_wide(A.mg.lv[0]) ? phase_b_q(A, pnew, alpha) : phase_b_s(A, pnew, alpha);
}

// One pass over this thread's fluid cells of level 0, both colours (start of the
// solve, the refinements and the end: not batched).  f(e, code, n) gets the slot,
// its code and the natural index n of the cell.
template <class F>
__device__ __forceinline__ void for_fluid0(const PcgArgs& A, F&& f) {
  const MgLevel& L0 = A.mg.lv[0];
  const SV v0 = sview(L0);
  const int lane = threadIdx.x & 31;
  const Items it = seg_items(L0, 2);
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const SCell e = scell(v0, v0.seg[(int)(t >> 1) - v0.seg_base], (int)(t & 1u), lane);
    if (!e.ok) continue;
    const unsigned int code = L0.code16[e.idx];
    if (!(code & CODE_SELF)) continue;
    f(e, code, e.i + L0.nx * e.r);
  }
}

// Residual b - A x of one level-0 cell with x and b as float pairs (split
// layout); the arithmetic is residual_pair_cell's.
__device__ __forceinline__ float2 residual_pair(const SV& v, const float2* x2, const float2* b2,
                                                const SCell& e, unsigned int code, float s_hi,
                                                float s_lo) {
  int nb[6];
  snbr(v, e, nb);
  const float2 xc = x2[e.idx];
  float2 xn[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) xn[q] = x2[nb[q]];
  return residual_pair_cell(b2[e.idx], xc, xn, code & 63u, code_cnt(code), s_hi, s_lo);
}

// ---------------------------------------------------------------- set-up

// Whether segment g (flat: row g / nw, segment g % nw) of split level L meets a
// block holding fluid; sg receives the packed segment.  Level 0 reads
// the binning's brick fluid counts.
__device__ __forceinline__ bool seg_active(const PcgArgs& A, const MgLevel& L, int l, int g,
                                           unsigned int& sg) {
  const int r = g / L.nw, w = g - r * L.nw;
  const int j = r % L.ny, k = r / L.ny;
  sg = seg_pack(w, j, k);
  const int by = j >> 3, bz = k >> 3;
  const int b0 = w * 8, b1 = min(L.nbx, b0 + 8);
  bool any = false;
  for (int bx = b0; bx < b1; ++bx) {
    const int bi = bx + L.nbx * (by + L.nby * bz);
    any |= (l == 0) ? (A.brick_fluid[bi] > 0u) : (L.bflag[bi] != 0);
  }
  return any;
}

// Whether a level with n blocks holding fluid is smoothed blocked.  The line: a block
// takes ~2 us of a CTA, a pass-by-pass half-sweep ~3.3 us plus the cells' own time.  Solves
// with the limit at 3, 6, 10 and 16 blocks per CTA: 128^3 dam break (3.4 blocks) 1.03, 1.00,
// 1.00, 0.98 ms; 128^3 pool (8.7 blocks) 1.52, 1.52, 1.79, 1.80; 256^3 pool (level 1: 8.4
// blocks) 5.29, 5.29, 5.55, 5.54; 101 x 67 x 83 pool 1.28, 1.20, 1.21, 1.23.
// A small team's barriers are cheaper, so its line is lower: a batch of 16 scenes (teams of 2
// to 27 CTAs) at 2, 3, 4 and 6 blocks per CTA 3.37, 3.33, 3.34, 3.45 ms per step.
__device__ __forceinline__ bool blocked(const MgArgs& M, unsigned int n) {
  const int most = team_size() < (unsigned)MG_WIDE_TEAM ? MG_BLK_PER_CTA_TEAM : MG_BLK_PER_CTA;
  return M.nlev > 1 && M.nu <= MG_BLK_MAX_NU && n > 0u && n <= (unsigned)most * team_size();
}

// The grid-wide levels' lists of blocks holding fluid.  Level 0's follows the
// binning's active list, so the sums that blocks of one CTA share keep their order; on
// the coarser levels the order decides nothing and blocks append as they come.
__device__ __forceinline__ void block_lists(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  {
    const MgLevel& L = M.lv[0];
    const unsigned int n = *A.n_active;
    if (blocked(M, n)) {
      const Part p = level_part((int)n, false);
      for (int c = p.begin; c < p.end; c += p.stride) {
        const int b = (int)A.active[c];
        L.blk[c] = b % L.nbx | ((b / L.nbx) % L.nby) << 8 | (b / (L.nbx * L.nby)) << 16;
      }
    }
  }
  for (int l = 1; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const Part p = level_part(L.nbx * L.nby * L.nbz, false);
    for (int c = p.begin; c < p.end; c += p.stride)
      if (L.bflag[c])
        L.blk[atomicAdd(L.nblk, 1u)] =
            c % L.nbx | ((c / L.nbx) % L.nby) << 8 | (c / (L.nbx * L.nby)) << 16;
  }
}

// The codes that each thread of a block's tile works with (MgLevel::tab): those of its
// four cells within L1 distance TILE_H of the block, 0 elsewhere, off the grid and where
// there is no fluid.  A thread's cells lie in one of the 27 blocks around, and codes are
// this solve's only where that block holds fluid.
__device__ __noinline__ void block_tables(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  const TilePos p = tile_pos();
  const int nbx = ((p.s + 2) >> 2) - 1, nby = ((p.y + 4) >> 3) - 1, nbz = ((p.g + 2) >> 2) - 1;
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const SV v = sview(L);
    const int nz = L.nz;
    for (int q = (int)team_rank(); q < s_nblk[l]; q += (int)team_size()) {
      const int e = L.blk[q];
      const BlkPos bp = blk_pos(v, p, e);
      const int x = (e & 255) + nbx, y = ((e >> 8) & 255) + nby, z = (e >> 16) + nbz;
      bool any = x >= 0 && y >= 0 && z >= 0 && x < L.nbx && y < L.nby && z < L.nbz;
      if (any) {
        const int b = x + L.nbx * (y + L.nby * z);
        any = l == 0 ? A.brick_fluid[b] > 0u : L.bflag[b] != 0;
      }
      const int j = bp.b1 - TILE_H + p.y;
      unsigned int red[2] = {0u, 0u}, black[2] = {0u, 0u};
      if (any && j < v.ny) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = bp.b2 - TILE_H + 2 * p.g + u;
          const int dyz = tile_dist(p.y) + tile_dist(2 * p.g + u);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int tx = 2 * p.s + ((c + p.y + u) & 1), i = bp.b0 - TILE_H + tx;
            if (k < nz && i < v.nx && tile_dist(tx) + dyz <= TILE_H) {
              const unsigned int code = v.code[c * v.half + bp.gi + u * v.pl];
              if (code & CODE_SELF) (c ? black : red)[u] = code;
            }
          }
        }
      }
      L.tab[(size_t)q * PCG_THREADS + threadIdx.x] = blk_pack(red, black);
    }
  }
}

// After build_levels: which levels are smoothed blocked, and level 0's arrays.
__device__ __forceinline__ void block_rule(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  if (threadIdx.x < MG_MAX_LEVELS) {
    const int l = threadIdx.x;
    const unsigned int n = l >= M.lgrid ? 0u : l == 0 ? *A.n_active : *M.lv[l].nblk;
    s_nblk[l] = blocked(M, n) ? (int)n : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s_z0 = s_nblk[0] > 0 ? M.q0 : M.lv[0].x;
    s_q0 = s_nblk[0] > 0 ? M.lv[0].x : M.q0;
  }
  __syncthreads();
}

// The active segments of large grids: counted per CTA, then written in segment order into
// the levels' lists.  Ends with a grid barrier.
__device__ __noinline__ bool seg_lists(const PcgArgs& A, Shared& sh) {
  const MgArgs& M = A.mg;
  __shared__ unsigned int s_wsum[PCG_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const int nsegs = L.nw * L.ny * L.nz;
    const int per = (nsegs + (int)team_size() - 1) / (int)team_size();
    const int g0 = min(nsegs, (int)team_rank() * per), g1 = min(nsegs, g0 + per);
    unsigned int cnt = 0;
    for (int g = g0 + (int)threadIdx.x; g < g1; g += PCG_THREADS) {
      unsigned int sg;
      cnt += seg_active(A, L, l, g, sg);
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) s_wsum[warp] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned int tot = 0;
      for (int w = 0; w < PCG_WARPS; ++w) tot += s_wsum[w];
      M.segcount[l * team_size() + team_rank()] = tot;
    }
    __syncthreads();
  }
  if (!gsync(A)) return false;
  SOLVE_TRACE(TR_SEG_COUNT);
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const int nsegs = L.nw * L.ny * L.nz;
    const int per = (nsegs + (int)team_size() - 1) / (int)team_size();
    const int g0 = min(nsegs, (int)team_rank() * per), g1 = min(nsegs, g0 + per);
    // this CTA's offset: the counts of the CTAs before it
    if (warp == 0) {
      unsigned int before = 0, total = 0;
      for (unsigned int t = lane; t < team_size(); t += 32) {
        const unsigned int v = M.segcount[l * team_size() + t];
        total += v;
        before += (t < team_rank()) ? v : 0u;
      }
      before = __reduce_add_sync(0xffffffffu, before);
      total = __reduce_add_sync(0xffffffffu, total);
      if (lane == 0) {
        sh.dscal[0] = (double)before;
        set_slice(l, (int)total);
      }
    }
    __syncthreads();
    unsigned int base = (unsigned int)sh.dscal[0];
    __syncthreads();
    for (int g00 = g0; g00 < g1; g00 += PCG_THREADS) {
      const int g = g00 + (int)threadIdx.x;
      unsigned int sg = 0u;
      const bool act = g < g1 && seg_active(A, L, l, g, sg);
      const unsigned int bal = __ballot_sync(0xffffffffu, act);
      if (lane == 0) s_wsum[warp] = __popc(bal);
      __syncthreads();
      unsigned int off = 0, tot = 0;
      for (int w = 0; w < PCG_WARPS; ++w) {
        off += (w < warp) ? s_wsum[w] : 0u;
        tot += s_wsum[w];
      }
      if (act) L.seg[base + off + __popc(bal & ((1u << lane) - 1u))] = sg;
      base += tot;
      __syncthreads();
    }
  }
  return gsync(A);
}

// Copies this CTA's slice of each grid-wide level's segment list into the
// shared-memory cache, level 0 first, while it fits (after build_levels).
__device__ __noinline__ void seg_cache_fill(const MgArgs& M, unsigned int* cache) {
  int used = 0;
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const int2 q = s_slice[l];
    const int n = q.y - q.x;
    const bool fits = used + n <= SEG_CACHE;
    if (fits)
      for (int i = threadIdx.x; i < n; i += PCG_THREADS) cache[used + i] = L.seg[q.x + i];
    if (threadIdx.x == 0) {
      s_segc[l] = fits ? cache + used : nullptr;
      s_segb[l] = q.x;
    }
    if (fits) used += n;
  }
  __syncthreads();
}

// The fluid flags of levels 1.. (a coarse cell is fluid when any child is) and their block
// flags and segment masks, all of them straight from the binning's active bricks, a warp
// per brick: lane l has rows 2 (l & 3) and the next of plane l >> 2 of the brick's cells as
// bits; the rows, planes and bits that share a coarse cell are or-ed.  From level 3 on a
// brick lies in one cell.  All flags start clear.
__device__ __noinline__ void level_flags(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  const MgLevel& L0 = M.lv[0];
  const int lane = threadIdx.x & 31;
  const int n = (int)*A.n_active;
  for (int q = (int)team_rank() * PCG_WARPS + (int)(threadIdx.x >> 5); q < n;
       q += (int)team_size() * PCG_WARPS) {
    const int b = (int)A.active[q];
    const int bx = b % L0.nbx, by = (b / L0.nbx) % L0.nby, bz = b / (L0.nbx * L0.nby);
    const int k = bz * 8 + (lane >> 2);
    unsigned int m = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = by * 8 + 2 * (lane & 3) + h;
      if (j >= L0.ny || k >= L0.nz) continue;
      const uint8_t* row = A.type + bx * 8 + L0.nx * (j + L0.ny * k);
      if (bx * 8 + 8 <= L0.nx && (reinterpret_cast<uintptr_t>(row) & 7u) == 0) {
        const unsigned long long v = *reinterpret_cast<const unsigned long long*>(row);
#pragma unroll
        for (int x = 0; x < 8; ++x) m |= ((unsigned)(v >> (8 * x)) & 255u) == 1u ? 1u << x : 0u;
      } else {
        for (int x = 0; x < 8 && bx * 8 + x < L0.nx; ++x) m |= row[x] == 1 ? 1u << x : 0u;
      }
    }
    m |= __shfl_xor_sync(0xffffffffu, m, 4);
    if (M.nlev > 1 && (lane & 4) == 0) {
      const MgLevel& L = M.lv[1];
      const int j = by * 4 + (lane & 3), kk = bz * 4 + (lane >> 3);
      if (j < L.ny && kk < L.nz) {
        // the brick's four cells of the row: one word where it is aligned
        uint8_t* t = L.t + bx * 4 + L.nx * (j + L.ny * kk);
        const unsigned int c = m | m >> 1;
        if (bx * 4 + 4 <= L.nx && (reinterpret_cast<uintptr_t>(t) & 3u) == 0) {
          *reinterpret_cast<unsigned int*>(t) = (c & 1u) | (c >> 2 & 1u) << 8 |
                                                (c >> 4 & 1u) << 16 | (c >> 6 & 1u) << 24;
        } else {
#pragma unroll
          for (int x = 0; x < 4; ++x)
            if ((c >> (2 * x)) & 1u) t[x] = 1;
        }
      }
    }
    m |= __shfl_xor_sync(0xffffffffu, m, 1);
    m |= __shfl_xor_sync(0xffffffffu, m, 8);
    if (M.nlev > 2 && (lane & 13) == 0) {
      const MgLevel& L = M.lv[2];
      const int j = by * 2 + ((lane >> 1) & 1), kk = bz * 2 + (lane >> 4);
      if (j < L.ny && kk < L.nz)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if ((m >> (4 * x)) & 15u) L.t[bx * 2 + x + L.nx * (j + L.ny * kk)] = 1;
    }
    if (lane >= 1 && lane < M.nlev) {
      const MgLevel& L = M.lv[lane];
      if (lane >= 3) {
        const int sh = lane - 3;
        L.t[(bx >> sh) + L.nx * ((by >> sh) + L.ny * (bz >> sh))] = 1;
      }
      if (L.split) L.bflag[(bx >> lane) + L.nbx * ((by >> lane) + L.nby * (bz >> lane))] = 1;
    }
    if (lane < M.lgrid) {
      const MgLevel& L = M.lv[lane];
      atomicOr(L.segmask + (by >> lane) + L.nby * (bz >> lane), 1u << (bx >> lane >> 3));
    }
  }
}

// Block-rows (the 8 x 8 rows of cells of blocks (*, J, K)) of level 0 up to which every CTA
// finds its own slices by itself.
constexpr int SEG_ROWS_PER_THREAD = 8;

// This CTA's slice of each level's active segments, found by every CTA for itself: each
// counts the segments of all block-rows (MgLevel::segmask: which segments of a row meet a
// block holding fluid, the same for its 64 rows), scans the counts, and writes those of its
// own slice, row by row, into the shared-memory cache while the slices fit, else into its
// part of the level's list.  No CTA reads another's slice, so no grid barrier follows
// (counting per CTA and writing in segment order took two).
__device__ __noinline__ void seg_slices(const PcgArgs& A, unsigned int* cache) {
  const MgArgs& M = A.mg;
  constexpr int ROUND = 256;  // block-rows written at a time
  __shared__ int s_scan[PCG_WARPS + 1], s_ra, s_rb, s_at[ROUND];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int used = 0;
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const int nr = L.nby * L.nbz, per_thread = (nr + PCG_THREADS - 1) / PCG_THREADS;
    const int r0 = (int)threadIdx.x * per_thread;
    int cnt = 0;
    for (int u = 0; u < per_thread && r0 + u < nr; ++u) {
      const int J = (r0 + u) % L.nby, K = (r0 + u) / L.nby;
      cnt += __popc(L.segmask[r0 + u]) * min(8, L.ny - 8 * J) * min(8, L.nz - 8 * K);
    }
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    __syncthreads();
    if (lane == 31) s_scan[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const int t = s_scan[lane];
      int w = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += x;
      }
      s_scan[lane] = w - t;
      if (lane == 31) {
        const int per = (w + (int)team_size() - 1) / (int)team_size();
        const bool fits = used + per <= SEG_CACHE;
        set_slice(l, w);
        s_segc[l] = fits ? cache + used : nullptr;
        s_segb[l] = s_slice[l].x;
        s_scan[PCG_WARPS] = fits ? per : 0;
        s_ra = nr;
        s_rb = 0;
      }
    }
    __syncthreads();
    const int2 q = s_slice[l];
    unsigned int* dst = s_segc[l] ? cache + used - q.x : L.seg;
    used += s_scan[PCG_WARPS];
    // the block-rows that the slice meets are consecutive: [s_ra, s_rb)
    const int at0 = s_scan[warp] + inc - cnt;
    const bool mine = cnt > 0 && at0 < q.y && at0 + cnt > q.x;
    if (mine) {
      atomicMin(&s_ra, r0);
      atomicMax(&s_rb, min(nr, r0 + per_thread));
    }
    __syncthreads();
    const int ra = s_ra, rb = s_rb;
    for (int base = ra; base < rb; base += ROUND) {
      if (mine) {
        int at = at0;
        for (int u = 0; u < per_thread && r0 + u < nr; ++u) {
          const int J = (r0 + u) % L.nby, K = (r0 + u) / L.nby, r = r0 + u - base;
          if (r >= 0 && r < ROUND) s_at[r] = at;
          at += __popc(L.segmask[r0 + u]) * min(8, L.ny - 8 * J) * min(8, L.nz - 8 * K);
        }
      }
      __syncthreads();
      for (int r = warp; r < min(ROUND, rb - base); r += PCG_WARPS) {  // a warp per block-row
        const int J = (base + r) % L.nby, K = (base + r) / L.nby;
        const unsigned int mask = L.segmask[base + r];
        const int nw = __popc(mask), nj = min(8, L.ny - 8 * J);
        const int n = nw * nj * min(8, L.nz - 8 * K), at = s_at[r];
        for (int i = max(0, q.x - at) + lane; i < min(n, q.y - at); i += 32) {
          const int row = i / nw;
          dst[at + i] = seg_pack(__fns(mask, 0, i - row * nw + 1), 8 * J + row % nj,
                                 8 * K + row / nj);
        }
      }
      __syncthreads();
    }
  }
}

// x = 0 on the rows of every block-row within one of a block-row that holds fluid, so that
// the sweeps read 0 from neighbours that are not fluid (what an earlier solve left there).
// Level 0 only where it will be swept pass by pass: a blocked level masks what it loads.
__device__ __noinline__ void zero_near(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool skip0 = A.precond != PRECOND_RBGS && blocked(M, *A.n_active);
  for (int l = skip0 ? 1 : 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const int rows = 64 * L.nby * L.nbz;
    for (int r = (int)team_rank() * PCG_WARPS + warp; r < rows; r += (int)team_size() * PCG_WARPS) {
      const int J = (r >> 6) % L.nby, K = (r >> 6) / L.nby;
      const int j = 8 * J + (r & 7), k = 8 * K + ((r >> 3) & 7);
      if (j >= L.ny || k >= L.nz) continue;
      const int dj = J + lane % 3 - 1, dk = K + lane / 3 - 1;
      const bool near = lane < 9 && dj >= 0 && dk >= 0 && dj < L.nby && dk < L.nbz &&
                        L.segmask[dj + L.nby * dk] != 0u;
      if (!__any_sync(0xffffffffu, near)) continue;
      float* x = L.x + L.margin + L.hx * (j + L.ny * k);
      for (int c = 0; c < 2; ++c)
        for (int s = 2 * lane; s < L.hx; s += 64)
          *reinterpret_cast<float2*>(x + c * L.half + s) = make_float2(0.0f, 0.0f);
    }
  }
}

// Builds, once per solve: the fluid flags of levels 1.. with their block flags, the
// active-segment slices and the block lists of the colour-split levels, the codes of every
// level.  Ends with a grid barrier.  All latency: three barriers instead of one per level
// and five more took the set-up up to the start pass from 41 to 25 us at 64^3, from 155 to
// 84 us at 256^3 (of which the codes 34 and the flags 20).
__device__ __noinline__ bool build_levels(const PcgArgs& A, Shared& sh, unsigned int* cache) {
  const MgArgs& M = A.mg;
  // flags start clear (16 bytes at a time: the arrays are padded to 256)
  for (int l = 1; l < M.nlev; ++l) {
    const MgLevel& L = M.lv[l];
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const Part p = level_part((L.ncells + 15) / 16, false);
    for (int c = p.begin; c < p.end; c += p.stride) reinterpret_cast<uint4*>(L.t)[c] = zero;
    if (L.split) {
      const Part pb = level_part((L.nbx * L.nby * L.nbz + 15) / 16, false);
      for (int c = pb.begin; c < pb.end; c += pb.stride) reinterpret_cast<uint4*>(L.bflag)[c] = zero;
      if (team_rank() == 0 && threadIdx.x == 0) *L.nblk = 0u;
    }
  }
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const Part p = level_part(L.nby * L.nbz, false);
    for (int c = p.begin; c < p.end; c += p.stride) L.segmask[c] = 0u;
  }
  if (!gsync(A)) return false;
  SOLVE_TRACE(TR_BFLAG);
  level_flags(A);
  if (!gsync(A)) return false;
  SOLVE_TRACE(TR_FLAGS + 1);
  block_lists(A);
  const int lane = threadIdx.x & 31;
  if (M.lv[0].nby * M.lv[0].nbz <= SEG_ROWS_PER_THREAD * PCG_THREADS) {
    seg_slices(A, cache);
  } else {
    if (!seg_lists(A, sh)) return false;
    seg_cache_fill(M, cache);
  }
  SOLVE_TRACE(TR_SEG_WRITE);
  zero_near(A);
  // codes: split levels over their active segments, CTA-local levels over all cells
  for (int l = 0; l < M.lgrid; ++l) {
    const MgLevel& L = M.lv[l];
    const SV v = sview(L);
    const Items it = seg_items(L, 2);
    for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
      const SCell e = scell(v, v.seg[(int)(t >> 1) - v.seg_base], (int)(t & 1u), lane);
      if (e.ok) v.code[e.idx] = (uint16_t)make_code(L, L.t, e.i, e.j, e.k);
    }
  }
  for (int l = M.lgrid; l < M.nlev; ++l) {
    const MgLevel& L = M.lv[l];
    const Part p = level_part(L.ncells, false);
    for (int c = p.begin; c < p.end; c += p.stride) {
      const Cell cl = cell_at(L, c);
      L.code[c] = (uint8_t)(make_code(L, L.t, cl.i, cl.j, cl.k) & 0x7fu);
    }
  }
  const bool ok = gsync(A);
  SOLVE_TRACE(TR_CODES);
  return ok;
}

// The shared-memory cache of the segment slices sits after the CTA-local levels
// in the kernel's dynamic shared memory, the tile of the blocked smoothing after it.
constexpr size_t MG_DYN_CTA = (sizeof(CtaMg) + 15) / 16 * 16;
constexpr size_t MG_DYN_TILE = MG_DYN_CTA + sizeof(unsigned int) * SEG_CACHE;
constexpr size_t MG_DYN_BYTES = MG_DYN_TILE + sizeof(MgTile);
// one carve-out step up (132 KB) would take L1 from the level-0 passes; beside the dynamic
// memory lie the arguments and the sums (3.4 KB), the level tables, slices and the set-up's
// scratch (3 KB; the kernel's own variables are 6432 bytes in all), and 1 KB of every CTA's
constexpr size_t MG_STATIC_BYTES = sizeof(PcgArgs) + sizeof(Shared) + 4096;
static_assert(MG_DYN_BYTES + MG_STATIC_BYTES + 1024 <= 100 * 1024,
              "the kernel stays in the 100 KB carve-out");

__device__ __forceinline__ unsigned int* seg_cache_of(unsigned char* dyn) {
  return reinterpret_cast<unsigned int*>(dyn + MG_DYN_CTA);
}

__device__ __forceinline__ MgTile& mg_tile() {
  extern __shared__ __align__(16) unsigned char mg_dyn[];
  return *reinterpret_cast<MgTile*>(mg_dyn + MG_DYN_TILE);
}

// The mixed mode's refinement, over level 0's slot pairs with two items in flight
// per warp (the per-cell arithmetic of the single-slot form, so the same values).
// refine_update: x += d as float pairs on fluid cells, d = 0 there.
__device__ __noinline__ void refine_update(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  const SV v = sview(M.lv[0]);
  float* d0 = M.d0;
  float2* x2 = M.x2;
  const int lane = threadIdx.x & 31;
  const int2 q = seg_slice(M.lv[0]);
  const Items it = pair_items(q, 2);
  struct S {
    PCell e;
    unsigned int code2;
    float2 d;
    float4 x;  // the two slots' (hi, lo)
  };
  run_batched<2>(
      it.first, it.end, PCG_WARPS,
      [&](unsigned int t, bool ok) {
        S st;
        st.e = pcell(v, q, t >> 1, (int)(t & 1u), lane);
        st.e.okA &= ok;
        st.e.okB &= ok;
        st.code2 = *reinterpret_cast<const unsigned int*>(v.code + st.e.idx);
        st.d = *reinterpret_cast<const float2*>(d0 + st.e.idx);
        st.x = *reinterpret_cast<const float4*>(x2 + st.e.idx);
        return st;
      },
      [&](S&) {},
      [&](S& st) {
        if (!(st.e.okA || st.e.okB)) return;
        const bool fa = st.e.okA && (st.code2 & CODE_SELF);
        const bool fb = st.e.okB && ((st.code2 >> 16) & CODE_SELF);
        const float2 ta = two_sum(st.x.x, st.d.x), tb = two_sum(st.x.z, st.d.y);
        const float2 xa = fast_two_sum(ta.x, __fadd_rn(ta.y, st.x.y));
        const float2 xb = fast_two_sum(tb.x, __fadd_rn(tb.y, st.x.w));
        *reinterpret_cast<float4*>(x2 + st.e.idx) =
            make_float4(fa ? xa.x : st.x.x, fa ? xa.y : st.x.y, fb ? xb.x : st.x.z,
                        fb ? xb.y : st.x.w);
        *reinterpret_cast<float2*>(d0 + st.e.idx) =
            make_float2(fa ? 0.0f : st.d.x, fb ? 0.0f : st.d.y);
      });
}

// refine_residual: r = b - A x in float pairs (residual_pair_cell) on fluid cells,
// the next V-cycle's first red half-sweep z = r / (s n) on red ones, and r.r.
__device__ __noinline__ FF refine_residual(const PcgArgs& A) {
  const MgArgs& M = A.mg;
  const MgLevel& L0 = M.lv[0];
  const SV v = sview(L0);
  const float2* x2 = M.x2;
  const float2* b2 = M.b2;
  float* r = L0.b;
  float* z = L0.x;
  const float s_hi = A.s, s_lo = A.s_lo;
  const int lane = threadIdx.x & 31;
  const int2 q = seg_slice(L0);
  const Items it = pair_items(q, 2);
  FF acc;
  for (unsigned int t = it.first; t < it.end; t += PCG_WARPS) {
    const int c = (int)(t & 1u);
    const PCell e = pcell(v, q, t >> 1, c, lane);
    const unsigned int code2 = *reinterpret_cast<const unsigned int*>(v.code + e.idx);
    const float4 bb = *reinterpret_cast<const float4*>(b2 + e.idx);
    const float4 xc = *reinterpret_cast<const float4*>(x2 + e.idx);
    // the other colour around the pair: slots s, s + 1 of this row, the one beyond
    // (s - 1 or s + 2), and the pairs in the rows and planes next door
    const float4 m = *reinterpret_cast<const float4*>(x2 + e.ob);
    const float2 ex = x2[e.ob - 1 + 3 * e.par];
    const float4 ym = *reinterpret_cast<const float4*>(x2 + e.ob - v.hx);
    const float4 yp = *reinterpret_cast<const float4*>(x2 + e.ob + v.hx);
    const float4 zm = *reinterpret_cast<const float4*>(x2 + e.ob - v.pl);
    const float4 zp = *reinterpret_cast<const float4*>(x2 + e.ob + v.pl);
    // a warp whose cells are all fluid with six fluid neighbours: the same cell
    // function with the mask and the count known
    const bool full = __all_sync(0xffffffffu, pair_full(code2) && e.okA && e.okB);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned int code = h == 0 ? (code2 & 0xffffu) : (code2 >> 16);
      if (!full && (!(h == 0 ? e.okA : e.okB) || !(code & CODE_SELF))) continue;
      const float2 m0 = make_float2(m.x, m.y), m1 = make_float2(m.z, m.w);
      float2 xn[6];
      if (h == 0) {
        xn[0] = e.par ? m0 : ex;
        xn[1] = e.par ? m1 : m0;
        xn[2] = make_float2(ym.x, ym.y);
        xn[3] = make_float2(yp.x, yp.y);
        xn[4] = make_float2(zm.x, zm.y);
        xn[5] = make_float2(zp.x, zp.y);
      } else {
        xn[0] = e.par ? m1 : m0;
        xn[1] = e.par ? ex : m1;
        xn[2] = make_float2(ym.z, ym.w);
        xn[3] = make_float2(yp.z, yp.w);
        xn[4] = make_float2(zm.z, zm.w);
        xn[5] = make_float2(zp.z, zp.w);
      }
      const float2 bc = h == 0 ? make_float2(bb.x, bb.y) : make_float2(bb.z, bb.w);
      const float2 xcc = h == 0 ? make_float2(xc.x, xc.y) : make_float2(xc.z, xc.w);
      const float2 rp = full ? residual_pair_cell(bc, xcc, xn, 63u, 6, s_hi, s_lo)
                             : residual_pair_cell(bc, xcc, xn, code & 63u, code_cnt(code), s_hi,
                                                  s_lo);
      const float r32 = __fadd_rn(rp.x, rp.y);
      r[e.idx + h] = r32;
      if (c == 0) z[e.idx + h] = gs_first(0, full ? 6 : code_cnt(code), r32);
      acc.add_prod(r32, r32);
    }
  }
  return acc;
}

struct SolveState {
  int iters = 0;
  int refinements = 0;
  bool conv = false;
  bool ok = true;
  double rel = 0.0;
  double bnorm = 0.0;
};

// Partial-sum slots (float pairs): 0 = p.q (phase A), 1 = r.r (phase B),
// 3 = r.z (end of the V-cycle), 4 and 5 = ||b||^2 and ||r_0||^2 (start), 5 = the
// recomputed residual's norm (refinement).  A slot's readers always pass another barrier before the slot
// is written again.
template <bool MIXED>
__device__ void solve_mg(const PcgArgs& A, Shared& sh, unsigned int* segc, SolveState& S) {
  const MgArgs& M = A.mg;
  const MgLevel& L0 = M.lv[0];
  float* d = M.d0;
  float* z = L0.x;
  float* r = L0.b;
  if (!build_levels(A, sh, segc)) { S.ok = false; return; }
  block_rule(A);
  SOLVE_TRACE(TR_SEG_CACHE);
  block_tables(A);  // visible to the V-cycles after the start pass's barrier
  if (M.nlev > 1 && team_rank() == 0) {
    if (cta_tiled(M)) cta_tiles_init(M);
    else cta_levels_init(M);
  }
  SOLVE_TRACE(TR_CTA_LISTS);
  // ---- start: r = b (cold) or b - A x0 (warm start from the last solve's x),
  // p_old = 0, first red half-sweep of the V-cycle; mixed mode: b as a float pair,
  // the correction d = 0, and x = 0 unless warm
  const bool warm = A.warm_start != 0;
  {
    FF bb, rr0;
    const SV v0 = sview(L0);
    const float s_a = A.s;
    if (warm && MIXED) {  // b as a pair first: the residual pass below reads it
      for_fluid0(A, [&](const SCell& e, unsigned int, int n) {
        const double b64 = A.b64[n];
        const float bh = __double2float_rn(b64);
        M.b2[e.idx] = make_float2(bh, __double2float_rn(b64 - (double)bh));
      });
      if (!gsync(A)) { S.ok = false; return; }
    }
    for_fluid0(A, [&](const SCell& e, unsigned int code, int n) {
      float bc, rc;
      if constexpr (MIXED) {
        if (warm) {
          bc = M.b2[e.idx].x;
          const float2 rp = residual_pair(v0, M.x2, M.b2, e, code, s_a, A.s_lo);
          rc = __fadd_rn(rp.x, rp.y);
        } else {
          const double b64 = A.b64[n];
          bc = __double2float_rn(b64);
          M.b2[e.idx] = make_float2(bc, __double2float_rn(b64 - (double)bc));
          M.x2[e.idx] = make_float2(0.0f, 0.0f);
          rc = bc;
        }
        d[e.idx] = 0.0f;
      } else {
        bc = A.b32[n];
        rc = bc;
        if (warm) {
          int nb[6];
          snbr(v0, e, nb);
          float xv[6];
#pragma unroll
          for (int q = 0; q < 6; ++q) xv[q] = d[nb[q]];
          rc = resid(s_a, code_cnt(code), code, bc, d[e.idx], xv);
        } else {
          d[e.idx] = 0.0f;
        }
      }
      r[e.idx] = rc;
      M.pa0[e.idx] = 0.0f;
      if (e.idx < L0.half) z[e.idx] = gs_first(0, code_cnt(code), rc);
      bb.add_prod(bc, bc);
      rr0.add_prod(rc, rc);
    });
    F2 v[2] = {f2_of(bb), f2_of(rr0)};
    publish<2>(A, 4, v, sh);
  }
  if (!gsync(A)) { S.ok = false; return; }
  SOLVE_TRACE(TR_START);
  // thread 0's, in shared memory to keep every thread's registers free
  double &rz = sh.dscal[0], &bnorm = sh.dscal[1], &rnorm = sh.dscal[2], &rmax = sh.dscal[3];
  const double target = MIXED ? A.ir_tol : A.tol;
  {
    double s0[2];
    gather<2>(A, 4, s0, sh);
    if (threadIdx.x == 0) {
      bnorm = sqrt(fmax(s0[0], 0.0));
      rnorm = rmax = sqrt(fmax(s0[1], 0.0));
      sh.flag = (bnorm == 0.0 || rnorm <= target * bnorm) ? 1 : 0;
    }
  }
  __syncthreads();
  int it = 0, refinements = 0;
  bool conv = sh.flag == 1, first = true;
  float* pold = M.pa0;
  float* pnew = M.pb0;
  while (!conv) {
    const PassSum V = vcycle_rest(A);
    if (!V.ok) { S.ok = false; return; }
    {
      F2 v[1] = {f2_of(V.sum)};
      publish<1>(A, 3, v, sh);
    }
    if (!gsync(A)) { S.ok = false; return; }
    if (it < 3) SOLVE_TRACE(TR_ITER + 3 * it);
    {
      double s[1];
      gather<1>(A, 3, s, sh);
      if (threadIdx.x == 0) {
        sh.beta = first ? 0.0f : (float)(s[0] / rz);
        rz = s[0];
        if (sh.flag == 0 && it >= A.max_iter) sh.flag = 3;
      }
    }
    __syncthreads();
    if (sh.flag == 1) { conv = true; break; }
    if (sh.flag == 3) break;
    first = false;
    ++it;
    const float beta = sh.beta;
    // ---- phase A
    const FF pq = phase_a(A, pold, pnew, beta);
    {
      F2 v[1] = {f2_of(pq)};
      publish<1>(A, 0, v, sh);
    }
    if (!gsync(A)) { S.ok = false; return; }
    if (it <= 3) SOLVE_TRACE(TR_ITER + 3 * (it - 1) + 1);
    {
      double s[1];
      gather<1>(A, 0, s, sh);
      if (threadIdx.x == 0) sh.alpha = (float)(rz / s[0]);
    }
    __syncthreads();
    const float alpha = sh.alpha;
    // ---- phase B (+ the next V-cycle's first red half-sweep)
    const FF rr = phase_b(A, pnew, alpha);
    {
      F2 v[1] = {f2_of(rr)};
      publish<1>(A, 1, v, sh);
    }
    if (!gsync(A)) { S.ok = false; return; }
    if (it <= 3) SOLVE_TRACE(TR_ITER + 3 * (it - 1) + 2);
    {
      double s[1];
      gather<1>(A, 1, s, sh);
      if (threadIdx.x == 0) {
        rnorm = sqrt(fmax(s[0], 0.0));
        int f = 0;  // 0 continue, 1 converged, 2 refine
        if (rnorm <= target * bnorm) f = MIXED ? 2 : 1;
        else if (MIXED && rnorm <= A.tol * rmax) f = 2;
        sh.flag = f;
      }
    }
    __syncthreads();
    float* t = pold; pold = pnew; pnew = t;
    if constexpr (MIXED) {
      if (sh.flag == 2) {
        // ---- refinement: x += d, d = 0; r = b - A x in float pairs (+ first red
        // half-sweep)
        if (refinements == 0) SOLVE_TRACE(TR_REFINE);
        refine_update(A);
        if (!gsync(A)) { S.ok = false; return; }
        if (refinements == 0) SOLVE_TRACE(TR_REFINE + 1);
        const FF rr64 = refine_residual(A);
        {
      F2 v[1] = {f2_of(rr64)};
      publish<1>(A, 5, v, sh);
    }
        if (!gsync(A)) { S.ok = false; return; }
        if (refinements == 0) SOLVE_TRACE(TR_REFINE + 2);
        double s[1];
      gather<1>(A, 5, s, sh);
        ++refinements;
        if (threadIdx.x == 0) {
          rnorm = sqrt(fmax(s[0], 0.0));
          rmax = rnorm;
          if (rnorm <= target * bnorm) sh.flag = 1;
          else if (refinements >= A.ir_max_iter) sh.flag = 3;
          else sh.flag = 0;
        }
        __syncthreads();
        if (sh.flag == 1) { conv = true; break; }
        if (sh.flag == 3) break;
        continue;  // the refinement's barrier has made the fused red half-sweep visible
      }
    }
    if (sh.flag == 1) { conv = true; break; }
  }
  SOLVE_TRACE(TR_LOOP_END);
  // ---- the solution in natural layout: the FP32 pressure, or the float pair
  // (for G2P) and its FP64 value
  if constexpr (MIXED) {
    for_fluid0(A, [&](const SCell& e, unsigned int, int n) {
      float2 xp = M.x2[e.idx];
      if (!conv) {
        const float2 t = two_sum(xp.x, d[e.idx]);
        xp = fast_two_sum(t.x, __fadd_rn(t.y, xp.y));
        d[e.idx] = 0.0f;
      }
      A.pff[n] = xp;
      A.x64[n] = (double)xp.x + (double)xp.y;
    });
  } else {
    for_fluid0(A, [&](const SCell& e, unsigned int, int n) { A.x32[n] = d[e.idx]; });
  }
  SOLVE_TRACE(TR_END);
  S.iters = it;
  S.refinements = refinements;
  S.conv = conv;
  if (threadIdx.x == 0) {
    S.rel = bnorm > 0.0 ? rnorm / bnorm : 0.0;
    S.bnorm = bnorm;
  }
}

// The paper's GPU solver (Sec. 3.2.3): red-black Gauss-Seidel sweeps on A p = b
// from p = 0 (FP32), on the colour-split level-0 storage with the smoother's
// half-sweeps, until ||b - A p|| <= tol ||b||; the residual is taken every
// RBGS_CHECK sweep pairs and the sweep pairs are capped at max_iter.
constexpr int RBGS_CHECK = 8;

__device__ __noinline__ void solve_rbgs(const PcgArgs& A, Shared& sh, unsigned int* segc, SolveState& S) {
  const MgArgs& M = A.mg;
  const MgLevel& L0 = M.lv[0];
  const MgLevel& L1 = M.nlev > 1 ? M.lv[1] : M.lv[0];
  float* z = L0.x;
  float* r = L0.b;
  if (!build_levels(A, sh, segc)) { S.ok = false; return; }
  {
    FF bb;
    for_fluid0(A, [&](const SCell& e, unsigned int, int n) {
      const float bc = A.b32[n];
      r[e.idx] = bc;
      z[e.idx] = 0.0f;
      bb.add_prod(bc, bc);
    });
    F2 v[1] = {f2_of(bb)};
    publish<1>(A, 4, v, sh);
  }
  if (!gsync(A)) { S.ok = false; return; }
  double bnorm = 0.0, rnorm = 0.0;
  {
    double s0[1];
    gather<1>(A, 4, s0, sh);
    if (threadIdx.x == 0) {
      bnorm = sqrt(fmax(s0[0], 0.0));
      rnorm = bnorm;
      sh.flag = (bnorm == 0.0) ? 1 : 0;
    }
  }
  __syncthreads();
  bool conv = sh.flag == 1;
  int it = 0;
  while (!conv) {
    for (int k = 0; k < RBGS_CHECK; ++k) {
      sweep_split<NORMAL>(M, L0, L1, 0, 0, false);
      if (!gsync(A)) { S.ok = false; return; }
      sweep_split<NORMAL>(M, L0, L1, 0, 1, false);
      if (!gsync(A)) { S.ok = false; return; }
    }
    it += RBGS_CHECK;
    FF rr;
    const SV v0 = sview(L0);
    for_fluid0(A, [&](const SCell& e, unsigned int code, int) {
      int nb[6];
      snbr(v0, e, nb);
      float xv[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) xv[q] = z[nb[q]];
      const float rc = resid(A.s, code_cnt(code), code, r[e.idx], z[e.idx], xv);
      rr.add_prod(rc, rc);
    });
    {
      F2 v[1] = {f2_of(rr)};
      publish<1>(A, 5, v, sh);
    }
    if (!gsync(A)) { S.ok = false; return; }
    {
      double s[1];
      gather<1>(A, 5, s, sh);
      if (threadIdx.x == 0) {
        rnorm = sqrt(fmax(s[0], 0.0));
        if (rnorm <= A.tol * bnorm) sh.flag = 1;
        else if (it >= A.max_iter) sh.flag = 3;
        else sh.flag = 0;
      }
    }
    __syncthreads();
    if (sh.flag == 1) conv = true;
    if (sh.flag == 3) break;
  }
  for_fluid0(A, [&](const SCell& e, unsigned int, int n) { A.x32[n] = z[e.idx]; });
  S.iters = it;
  S.conv = conv;
  S.rel = bnorm > 0.0 ? rnorm / bnorm : 0.0;
  S.bnorm = bnorm;
}

template <bool MIXED>
__device__ void solve_scene_mg(const PcgArgs& A, Shared& sh, unsigned char* dyn) {
  unsigned int* segc = seg_cache_of(dyn);
  if (threadIdx.x < MG_MAX_LEVELS) {
    s_segc[threadIdx.x] = nullptr;  // no cache until filled
    s_nblk[threadIdx.x] = 0;        // no blocked level until block_rule
  }
  __syncthreads();
  const long long ncells = (long long)A.g.nx * A.g.ny * A.g.nz;
  const bool singular = A.check_singular && ((long long)A.stats->n_fluid == ncells);
  SolveState S;
  if (!singular) {
    if (!MIXED && A.precond == PRECOND_RBGS) solve_rbgs(A, sh, segc, S);
    else solve_mg<MIXED>(A, sh, segc, S);
  }
  if (team_rank() == 0 && threadIdx.x == 0) {
    int st = 0;
    if (singular) st |= DEV_SINGULAR;
    else if (S.ok && !S.conv) st |= DEV_NOT_CONVERGED;
    if (st) atomicOr(A.status, st);
    A.stats->cg_iters = S.iters;
    A.stats->ir_iters = S.refinements;
    A.stats->cg_iters_total += S.iters;
    A.stats->ir_iters_total += S.refinements;
    A.stats->rel_res = S.rel;
    A.stats->bnorm = S.bnorm;
  }
}

template <bool MIXED>
__global__ void __launch_bounds__(PCG_THREADS, 1) k_pcg_mg(const __grid_constant__ PcgArgs A) {
  __shared__ Shared sh;
  extern __shared__ __align__(16) unsigned char mg_dyn[];
  team_enter(blockIdx.x, gridDim.x);
  SOLVE_TRACE(TR_ENTRY);
  load_args(A);
  load_tables(s_args.mg);
  SOLVE_TRACE(TR_TABLES);
  solve_scene_mg<MIXED>(s_args, sh, mg_dyn);
  SOLVE_TRACE(TR_EXIT);
}

// Several scenes in one launch: CTA b works on scene block_scene[b], in the team
// of CTAs team_first[s] .. team_first[s+1]-1.
template <bool MIXED>
__global__ void __launch_bounds__(PCG_THREADS, 1) k_pcg_mg_batch(const __grid_constant__ PcgBatch B) {
  __shared__ Shared sh;
  extern __shared__ __align__(16) unsigned char mg_dyn[];
  const int s = B.block_scene[blockIdx.x];
  team_enter(blockIdx.x - B.team_first[s], B.team_first[s + 1] - B.team_first[s]);
  load_args(B.args[s]);
  load_tables(s_args.mg);
  solve_scene_mg<MIXED>(s_args, sh, mg_dyn);
}

}  // namespace

int mg_level_dims(int nx, int ny, int nz, int dims[MG_MAX_LEVELS][3]) {
  int n[3] = {nx, ny, nz};
  int L = 0;
  for (;;) {
    for (int a = 0; a < 3; ++a) dims[L][a] = n[a];
    ++L;
    const int m = n[0] > n[1] ? (n[0] > n[2] ? n[0] : n[2]) : (n[1] > n[2] ? n[1] : n[2]);
    if (m <= 4 || L == MG_MAX_LEVELS) break;
    for (int a = 0; a < 3; ++a) n[a] = (n[a] + 1) / 2;
  }
  return L;
}

cudaError_t launch_pcg_mg(const PcgArgs& a, bool mixed, int nblocks, cudaStream_t s) {
  void* args[] = {const_cast<PcgArgs*>(&a)};
  if (mixed)
    return cudaLaunchCooperativeKernel((const void*)k_pcg_mg<true>, dim3(nblocks),
                                       dim3(PCG_THREADS), args, MG_DYN_BYTES, s);
  return cudaLaunchCooperativeKernel((const void*)k_pcg_mg<false>, dim3(nblocks),
                                     dim3(PCG_THREADS), args, MG_DYN_BYTES, s);
}

cudaError_t launch_pcg_mg_batch(const PcgBatch& b, bool mixed, int nblocks, cudaStream_t s) {
  void* args[] = {const_cast<PcgBatch*>(&b)};
  if (mixed)
    return cudaLaunchCooperativeKernel((const void*)k_pcg_mg_batch<true>, dim3(nblocks),
                                       dim3(PCG_THREADS), args, MG_DYN_BYTES, s);
  return cudaLaunchCooperativeKernel((const void*)k_pcg_mg_batch<false>, dim3(nblocks),
                                     dim3(PCG_THREADS), args, MG_DYN_BYTES, s);
}

// Opts the kernels in to the dynamic shared memory of the CTA-local levels and
// checks that one CTA per SM fits.
cudaError_t pcg_mg_check_occupancy() {
  const void* fns[4] = {(const void*)k_pcg_mg<false>, (const void*)k_pcg_mg<true>,
                        (const void*)k_pcg_mg_batch<false>, (const void*)k_pcg_mg_batch<true>};
  for (const void* f : fns) {
    cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MG_DYN_BYTES);
    if (e != cudaSuccess) return e;
    int a = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, f, PCG_THREADS, MG_DYN_BYTES);
    if (e != cudaSuccess) return e;
    if (a < 1) return cudaErrorInvalidConfiguration;
  }
  return cudaSuccess;
}

}  // namespace flipk

#ifdef FLIP_SOLVE_TRACE
// The stamps of the last solve (nanoseconds of the global timer; slots of
// flipk::TraceSlot; 0 where no stamp was taken since the library was loaded).
extern "C" int flip_solve_trace(unsigned long long* out, int n) {
  if (!out || n < 1 || n > 64) return 1;
  return cudaMemcpyFromSymbol(out, flipk::flip_trace_ns, sizeof(unsigned long long) * (size_t)n) ==
                 cudaSuccess
             ? 0
             : 3;
}
#endif
